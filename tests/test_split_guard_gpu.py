"""FP64 products whose operands the tensor-core split does not take: by the SIMT kernel behind."""
import numpy as np
import pytest

from test_gemm_gpu import _rand

pytestmark = pytest.mark.gpu


def _cholqr(S):
    import torch

    from paper_2601_19650_gb300 import _cbc as c
    d = torch.from_numpy(S).to("cuda").contiguous()
    c.cbc_cholqr2(c.CBC_C128 if np.iscomplexobj(S) else c.CBC_F64, S.shape[1], S.shape[2],
                  S.shape[0], d.data_ptr())
    return d.cpu().numpy()


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("nb", [2, 5])
def test_a_problem_does_not_send_its_neighbours(nb, cplx):
    """The Gram products of a batch in which one matrix has 40 tiny entries in every
    row: bit for bit the others' results of a batch without it."""
    rng = np.random.default_rng([nb, cplx])
    S = _rand(rng, (nb, 16, 64), cplx)
    T = S.copy()
    T[1, :, :40] *= 2.0 ** -60
    Q, R = _cholqr(S), _cholqr(T)
    for b in range(nb):
        if b != 1:
            assert np.array_equal(Q[b], R[b])


def _bound(A, B):
    """K eps |A||B| (sqrt 2 more per complex product), as for any FP64 sum."""
    return 4 * (A.shape[1] + 2) * 2.0 ** -53 * (np.abs(A) @ np.abs(B))


def _check(A, B):
    from test_gemm_gpu import _run
    C, _ = _run(0, 0, A, B)
    long = np.clongdouble if np.iscomplexobj(A) else np.longdouble
    # of large products the first and last rows and columns of tiles
    rows = [i for i in range(len(A)) if len(A) < 70 or i % 64 in (0, 63) or i == len(A) - 1]
    cols = [j for j in range(B.shape[1]) if B.shape[1] < 70 or j % 32 in (0, 31) or j == B.shape[1] - 1]
    a, b = A[rows], B[:, cols]
    err = np.abs(C[np.ix_(rows, cols)] - a.astype(long) @ b.astype(long))
    assert np.all(err <= _bound(a, b)), (err / _bound(a, b)).max()


def _alternate(K, r, up):
    w = np.ones(K)
    w[int(up)::2] = 2.0 ** -r
    return w


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("shape", [(128, 64, 32), (40, 300, 64), (65, 33, 257), (16, 20, 2049)])
@pytest.mark.parametrize("r", [0, 4, 8, 12, 20, 30, 36, 45])
@pytest.mark.parametrize("how", ["slope", "alternate", "half", "one", "rows"])
def test_opposite_grading(how, r, shape, cplx):
    """A graded along K and B the other way, so that large entries meet small ones: the plain
    bound of an FP64 sum, entry by entry."""
    rng = np.random.default_rng([r, shape[2], cplx])
    M, N, K = shape
    A, B = _rand(rng, (M, K), cplx), _rand(rng, (K, N), cplx)
    if how == "slope":
        w = 2.0 ** -np.linspace(0, r, K)
        wb = w[::-1]
    elif how == "alternate":
        w, wb = _alternate(K, r, True), _alternate(K, r, False)
    elif how == "half":
        w = np.where(np.arange(K) < K // 2, 1.0, 2.0 ** -r)
        wb = w[::-1]
    else:  # one large entry, in the same place or, "rows", in one row and column only
        w = np.where(np.arange(K) == 3, 1.0, 2.0 ** -r)
        wb = np.where(np.arange(K) == 4, 1.0, 2.0 ** -r)
    if how == "rows":
        A[-1], B[:, -1] = A[-1] * w, B[:, -1] * wb
    else:
        A, B = A * w, B * wb[:, None]
    _check(A, B)


@pytest.mark.parametrize("r", [3, 6, 9, 20])
def test_equal_digits(r):
    """Terms whose dropped digits all add up: equal entries 2^-r below one large one."""
    rng = np.random.default_rng(r)
    M, N, K = 40, 40, 512
    A = np.full((M, K), (1 - 2.0 ** -9 + 2.0 ** -40) * 2.0 ** -r / 1.5)
    B = np.full((K, N), (1 - 2.0 ** -10 - 2.0 ** -41) * 2.0 ** -r / 1.5)
    A[:, 0], B[1] = rng.uniform(1, 2, M), rng.uniform(1, 2, N)
    _check(A, B)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("kind", ["zero_rows", "sparse", "identity", "subnormal", "ends"])
def test_forms(kind, cplx):
    """Rows of zeros, mostly zeros, a permutation, and the ends of the exponent range."""
    rng = np.random.default_rng(3)
    M, N, K = 70, 45, 130
    A, B = _rand(rng, (M, K), cplx), _rand(rng, (K, N), cplx)
    if kind == "zero_rows":
        A[::3], B[:, 1::4] = 0, 0
    elif kind == "sparse":
        A, B = A * (rng.random(A.shape) < 0.05), B * (rng.random(B.shape) < 0.2)
    elif kind == "identity":
        A = np.eye(M, K) * (1 + 1j if cplx else 1)
        B = B * 2.0 ** -rng.integers(0, 50, B.shape).astype(float)
    elif kind == "subnormal":
        A = A * 2.0 ** -1030
        B = B * 2.0 ** 1000
    else:
        A, B = A * 2.0 ** 1000, B * 2.0 ** -1000
    _check(A, B)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("shape", [(300, 200, 1100), (129, 65, 64), (257, 64, 2049), (20, 20, 28)])
@pytest.mark.parametrize("r", [2, 4, 6, 9, 14, 22])
def test_one_entry_below_the_line(r, shape, cplx):
    """Half of every row small, in the same places in A and B, and then the last row and column
    graded against each other besides, which one entry of the last tile shows."""
    rng = np.random.default_rng([r, shape[0], cplx])
    M, N, K = shape
    A, B = _rand(rng, (M, K), cplx), _rand(rng, (K, N), cplx)
    h = np.where(rng.random(K) < 0.5, 1.0, 2.0 ** -12)
    A, B = A * h, B * h[:, None]
    _check(A, B)
    A[-1] *= np.where(h == 1.0, 2.0 ** -r, 1.0)
    A[-1, 5] = 2.0
    B[:, -1] *= np.where(h == 1.0, 2.0 ** -r, 1.0)
    B[7, -1] = 2.0
    _check(A, B)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("shape", [(64, 64, 8192), (33, 45, 300), (65, 130, 255), (64, 64, 256),
                                   (31, 33, 40), (700, 1900, 30), (1300, 1040, 33)])
def test_products_turned_down(shape, cplx):
    """Operands graded against each other: few and many tiles of either size, split along K
    (sums added into the zeros that the tensor-core kernel leaves) and not."""
    rng = np.random.default_rng([*shape, cplx])
    M, N, K = shape
    w = 2.0 ** -np.linspace(0, 45, K)
    _check(_rand(rng, (M, K), cplx) * w, _rand(rng, (K, N), cplx) * w[::-1][:, None])


def test_error_of_products_turned_down():
    """Equal positive terms, whose roundings add up along a partial sum: the split of K keeps
    them as short as on the SIMT kernel alone (3 parts of 344 terms: 344 / 2 roundings at most
    of half a unit of the running sum, which is half of the whole on average, and one for each
    part)."""
    from test_gemm_gpu import _run
    M, N, K = 501, 777, 1030
    A = np.full((M, K), 1 / 3.0) + 0j
    B = np.full((K, N), 1 / 7.0) + 0j
    C, _ = _run(0, 0, A, B)
    ref = float(K * (np.longdouble(1 / 3.0) * np.longdouble(1 / 7.0)))
    assert np.abs(C - ref).max() <= (344 / 4 + 3) * 2.0 ** -53 * ref
