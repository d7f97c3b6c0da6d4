"""The reductions to tridiagonal form at the edges of their ranges, through cbc_heev: sizes
around the columns per thread (256) and the rows per CTA, reflectors that are the identity
(diagonal, block-diagonal and low-rank matrices), and matrices of very small or large norm."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _check(a, kmax=None, nb=1, mixed=False):
    import torch

    from paper_2601_19650_gb300 import _cbc as c
    m = a.shape[0]
    k = kmax or m
    cplx = np.iscomplexobj(a)
    dt = torch.complex128 if cplx else torch.float64
    A = torch.from_numpy(np.ascontiguousarray(np.stack([a] * nb))).to("cuda", dt)
    lam = torch.zeros(nb, m, dtype=torch.float64, device="cuda")
    U = torch.zeros(nb, m, k, dtype=dt, device="cuda")
    c.cbc_heev(c.CBC_C128 if cplx else c.CBC_F64, m, k, nb, A.data_ptr(), lam.data_ptr(),
               U.data_ptr(), mixed)
    ref = np.linalg.eigvalsh(a)[::-1][:k]
    scale = max(np.abs(ref).max(), np.finfo(float).tiny)
    # backward stable: a few hundred roundings of 2^-53 (2^-46 in double-float) per entry
    tol = (2.0 ** -46 if mixed else 2.0 ** -53) * 300 * max(1.0, m / 64) ** 0.5
    for b in range(nb):
        u, l = U[b].cpu().numpy(), lam[b, :k].cpu().numpy()
        assert np.abs(l - ref).max() <= tol * scale
        assert np.linalg.norm(a @ u - u * l, axis=0).max() <= 10 * tol * scale
        assert np.abs(u.conj().T @ u - np.eye(k)).max() <= 40 * tol


def _random(m, cplx, seed=1):
    r = np.random.default_rng([m, seed])
    x = r.standard_normal((m, 3 * m)) + (1j * r.standard_normal((m, 3 * m)) if cplx else 0)
    return x @ x.conj().T / (3 * m)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("m", [1, 2, 3, 5, 31, 33, 64, 65, 255, 256, 257, 511, 513, 700])
def test_lone_sizes(m, cplx):
    _check(_random(m, cplx), kmax=max(1, m // 3))


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("nb,mixed", [(1, False), (3, False), (3, True)])
@pytest.mark.parametrize("kind", ["diagonal", "blocks", "rank", "tiny", "huge"])
def test_special_matrices(kind, nb, mixed, cplx):
    m = 48
    a = _random(m, cplx)
    if kind == "diagonal":  # every reflector is the identity
        a = np.diag(np.linspace(1.0, 2.0, m)).astype(a.dtype)
    elif kind == "blocks":  # a column that is already zero below the first off-diagonal entry
        a[:20, 20:] = 0
        a[20:, :20] = 0
    elif kind == "rank":    # rank 5 next to a part of full rank
        a[20:, :] = 0
        a[:, 20:] = 0
        x = _random(28, cplx, 2)[:, :5]
        a[20:, 20:] = x @ x.conj().T
        a += 0.5 * np.diag(np.linspace(0.0, 1.0, m))
    elif kind == "tiny":
        a = a * (1e-60 if not mixed else 1e-12)
    elif kind == "huge":
        a = a * (1e60 if not mixed else 1e12)
    _check(a, kmax=m // 2, nb=nb, mixed=mixed)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("m", [48, 63, 64, 65, 127, 128, 129, 193])
def test_back_transformation_blocks(m, cplx):
    """Batches large enough for the back transformation by products, around its blocks of 64
    reflectors (two halves of 32) and a last block that is short."""
    k = m // 2 + 1
    nb = int(4e6 / (m * m * k)) + 1
    _check(_random(m, cplx), kmax=k, nb=nb)


@pytest.mark.parametrize("nb", [1, 3])
@pytest.mark.parametrize("m", [2, 33, 64, 257])
def test_estimates_bits(m, nb):
    """The eigenvalue estimates beyond kmax are points of the FP32 bisection's grid between
    Gershgorin's bounds in FP64: bit for bit on diagonal matrices, whose counts are exact."""
    import torch

    from paper_2601_19650_gb300 import _cbc as c
    f = np.float32
    dg = np.random.default_rng(m).standard_normal(m)
    A = torch.from_numpy(np.stack([np.diag(dg)] * nb)).cuda()
    lam = torch.zeros(nb, m, dtype=torch.float64, device="cuda")
    U = torch.zeros(nb, m, 1, dtype=torch.float64, device="cuda")
    c.cbc_heev(c.CBC_F64, m, 1, nb, A.data_ptr(), lam.data_ptr(), U.data_ptr(), False)
    span = np.abs(dg).max()
    d32, want = dg.astype(f), np.zeros(m)
    for j in range(1, m):
        lo, hi = f(dg.min() - 1e-6 * span), f(dg.max() + 1e-6 * span)
        for _ in range(12):
            step = (hi - lo) * np.arange(1, 33, dtype=f)
            # fma(step, 1 / 33, lo): one rounding
            x = (lo.astype(np.float64) + step.astype(np.float64) * np.float64(f(1) / f(33))).astype(f)
            n = int(sum((d32 < v).sum() <= m - 1 - j for v in x))
            lo, hi = (x[n - 1] if n else lo), (x[n] if n < 32 else hi)
            if hi - lo <= f(2e-7) * max(abs(lo), abs(hi)):
                break
        want[j] = f(0.5) * (lo + hi)
    for b in range(nb):
        assert np.array_equal(lam[b, 1:].cpu().numpy(), want[1:])
