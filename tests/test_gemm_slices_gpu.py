"""Operand slicing of the split products at the edges of its tiles: row blocks of 32, K tiles
of 64 packed values, shares of up to 4 tiles per CTA and 8 CTAs along K, both read patterns."""
import numpy as np
import pytest

from test_gemm_gpu import _rand, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("trans", [(False, False), (True, True)])
@pytest.mark.parametrize("K", [1, 31, 33, 64, 65, 127, 129, 256, 257, 513, 1023, 1025, 2049])
def test_slicing_edges(K, trans, cplx):
    rng = np.random.default_rng(K)
    M, N, S = 130, 33, 4
    A = _rand(rng, (K, M) if trans[0] else (M, K), cplx) * np.exp(rng.uniform(-9, 9))
    B = _rand(rng, (N, K) if trans[1] else (K, N), cplx)
    C, ref = _run(1, S, A, B, trans[0], False, trans[1], cplx)
    a, b = (A.T if trans[0] else A), (B.T if trans[1] else B)
    # an element is off by at most 2^(e-8S) (e: the exponent of its row's or column's
    # maximum); the dropped levels add at most S^2/2 2^(e_a+e_b-8S) per term
    ea = 2.0 ** (np.floor(np.log2(np.abs(np.stack([a.real, a.imag])).max(axis=(0, 2)))) + 1)
    eb = 2.0 ** (np.floor(np.log2(np.abs(np.stack([b.real, b.imag])).max(axis=(0, 1)))) + 1)
    bound = (2 if cplx else 1) * K * np.outer(ea, eb) * 2.0 ** (-8 * S) * (3 + S * S / 2)
    assert np.all(np.abs(C - ref) <= bound)


def _fp64_case(rng, M, N, K, cplx, grade=None):
    A, B = _rand(rng, (M, K), cplx), _rand(rng, (K, N), cplx)
    if grade is not None:  # entries of a row fall by 2^-grade along K
        A = A * 2.0 ** (-np.linspace(0, grade, K))[None, :]
    return A, B


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("shape", [(128, 64, 28), (1, 1, 8), (33, 31, 127), (129, 33, 129),
                                   (256, 40, 1025), (65, 300, 4097)])
@pytest.mark.parametrize("grade", [None, 20, 80])
def test_fp64_split(shape, grade, cplx):
    """FP64 products on the tensor cores and, for rows that span too much, behind them: the
    componentwise bound K eps |A||B| of an FP64 sum (sqrt 2 more per complex product), in
    80-bit arithmetic; split operands add at most 2^(e_a+e_b) K 2^-58."""
    rng = np.random.default_rng(5)
    M, N, K = shape
    A, B = _fp64_case(rng, M, N, K, cplx, grade)
    C, _ = _run(0, 0, A, B)
    wide = np.clongdouble if cplx else np.longdouble
    ref = A.astype(wide) @ B.astype(wide)
    eps = 2.0 ** -53
    bound = 4 * (K + 2) * eps * (np.abs(A) @ np.abs(B))
    if grade != 80:
        bound = bound + K * 2.0 ** -55 * np.outer(np.abs(A).max(1), np.abs(B).max(0))
    assert np.all(np.abs(C - ref) <= bound)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_fp64_nonfinite_passes_through(bad):
    """Inf and NaN go through an FP64 product as through any sum."""
    rng = np.random.default_rng(9)
    A, B = _fp64_case(rng, 70, 40, 64, False)
    A[3, 5] = bad
    C, ref = _run(0, 0, A, B)
    assert np.array_equal(np.isnan(C), np.isnan(ref)) and np.array_equal(np.isinf(C), np.isinf(ref))
    assert np.abs(np.delete(C, 3, 0) - np.delete(ref, 3, 0)).max() <= 1e-12


@pytest.mark.parametrize("prec", [0, 1])
def test_operands_on_odd_doubles(prec):
    """Complex operands whose storage starts on an odd double (8-byte aligned only)."""
    import torch

    from paper_2601_19650_gb300 import _cbc
    rng = np.random.default_rng(4)
    M, N, K = 70, 45, 130
    A, B = _rand(rng, (M, K), True), _rand(rng, (K, N), True)

    def shifted(x):
        buf = torch.zeros(2 * x.size + 1, dtype=torch.float64, device="cuda")
        buf[1:] = torch.from_numpy(np.ascontiguousarray(x).view(np.float64).reshape(-1)).to("cuda")
        return buf, buf.data_ptr() + 8

    (ka, pa), (kb, pb) = shifted(A), shifted(B)
    kc, pc = shifted(np.zeros((M, N), dtype=np.complex128))
    _cbc.cbc_gemm(prec, 5, _cbc.CBC_C128, M, N, K, pa, K, False, False, pb, N, False, False, pc, N)
    C = kc[1:].cpu().numpy().view(np.complex128).reshape(M, N)
    # 5 slices: K terms, each off by at most 16 2^(e_a+e_b-40) with entries below 2^3
    assert np.abs(C - A @ B).max() <= (1e-12 if prec == 0 else 2 * K * 16 * 2.0 ** (6 - 40))


def _digits(x, e, S):
    """The balanced base-256 digits q_0 .. q_{S-1} of x 2^(7-e), rounded to nearest, ties to
    even, in Python integers."""
    from fractions import Fraction
    n = round(Fraction(float(x)) * Fraction(2) ** (7 - e + 8 * (S - 1)))
    q = [0] * S
    for s in range(S - 1, 0, -1):
        hi = (n + 128) >> 8
        q[s], n = n - (hi << 8), hi
    q[0] = n
    return q


def _planes(rows, S):
    e = np.frexp(np.abs(rows).max(axis=1))[1]
    q = np.array([[_digits(x, int(ei), S) for x in r] for r, ei in zip(rows, e)], dtype=object)
    return q, e


@pytest.mark.parametrize("ties", [False, True])
@pytest.mark.parametrize("S", [4, 5])
@pytest.mark.parametrize("cplx,conj", [(False, False), (True, False), (True, True)])
def test_split_product_bits(cplx, conj, S, ties):
    """The split product bit for bit: exact integer sums of the digits' products of the first
    S levels, rounded once.  Digits of -x are not the negated digits of x where one is -128;
    `ties`: half of the entries lie halfway between two last digits."""
    rng = np.random.default_rng([S, cplx, ties])
    M, N, K = 40, 20, 48
    def draw(shape):
        top = 2 ** (7 + 8 * (S - 1))
        n = rng.integers(-top + 1, top - 1, shape).astype(float)
        n[0, :], n[:, 0] = 0.75 * top, 0.75 * top  # every row and column: exponent 0
        f = 0.5 * rng.integers(0, 2, shape) if ties else rng.integers(0, 8, shape) / 8 + 1 / 16
        return (n + f) * 2.0 ** (-7 - 8 * (S - 1))
    A, B = draw((M, K)), draw((K, N))
    if cplx:
        A, B = A + 1j * draw((M, K)), B + 1j * draw((K, N))
    C, _ = _run(1, S, A, B, False, False, False, conj)
    b = B.conj() if conj else B
    if cplx:
        ra = np.stack([A.real, A.imag], axis=2).reshape(M, 2 * K)
        rb = np.stack([np.stack([b.real, -b.imag], 1).reshape(2 * K, N),
                       np.stack([b.imag, b.real], 1).reshape(2 * K, N)], 2).reshape(2 * K, 2 * N).T
    else:
        ra, rb = A, b.T
    (qa, ea), (qb, eb) = _planes(ra, S), _planes(rb, S)
    want = np.zeros((len(ra), len(rb)))
    for i in range(len(ra)):
        for j in range(len(rb)):
            t = sum(int((qa[i, :, s] * qb[j, :, g - s]).sum()) << (8 * (S - 1 - g))
                    for g in range(S) for s in range(g + 1))
            want[i, j] = np.ldexp(float(t), int(ea[i] + eb[j]) - 14 - 8 * (S - 1))
    got = np.stack([C.real, C.imag], axis=2).reshape(M, 2 * N) if cplx else C
    assert np.array_equal(got, want)
