"""Inverse iteration with idle lanes: warps whose members (two lanes each) do not fill them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _with_spectrum(spec, cplx, seed):
    rng = np.random.default_rng(seed)
    m = len(spec)
    q, _ = np.linalg.qr(rng.standard_normal((m, m)) + (1j * rng.standard_normal((m, m)) if cplx else 0))
    a = (q * spec) @ q.conj().T
    return (a + a.conj().T) / 2


def _heev(a, k, nb):
    import torch

    from paper_2601_19650_gb300 import _cbc as c
    m, cplx = a.shape[0], np.iscomplexobj(a)
    dt = torch.complex128 if cplx else torch.float64
    A = torch.from_numpy(np.stack([a] * nb)).to("cuda", dt).contiguous()
    lam = torch.zeros(nb, m, dtype=torch.float64, device="cuda")
    U = torch.zeros(nb, m, k, dtype=dt, device="cuda")
    c.cbc_heev(c.CBC_C128 if cplx else c.CBC_F64, m, k, nb, A.data_ptr(), lam.data_ptr(),
               U.data_ptr(), False)
    return lam.cpu().numpy(), U.cpu().numpy()


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("m", [41, 64, 129])
def test_members_do_not_depend_on_idle_lanes(m, cplx):
    """30 copies of a matrix: 1, 3 and up to 16 members per warp for 1, 6 and 40 candidates.
    T, the shifts and every member's operations are the same, so the eigenvalues are too."""
    a = _with_spectrum(np.linspace(2.0, 1.0, m), cplx, m)
    full, _ = _heev(a, 40, 30)
    for k in (1, 3, 6, 17):
        lam, _ = _heev(a, k, 30)
        assert np.array_equal(lam[:, :k], full[:, :k])
        assert np.array_equal(lam[:, :k], np.broadcast_to(lam[0, :k], (30, k)))


@pytest.mark.parametrize("m,k", [(701, 60), (1001, 31)])
def test_clusters_on_part_of_a_warp(m, k):
    """Clusters of 8 where shared memory holds 7 and 5 members at a time: the vectors span the
    invariant subspace (40 sums of m roundings of 2^-53, and inverse iteration's own)."""
    base = np.linspace(2.0, 1.0, (m + 7) // 8)
    spec = (np.repeat(base, 8) - np.tile(np.arange(8) * 1e-9, len(base)))[:m]
    a = _with_spectrum(spec, False, m)
    k -= k % 8
    lam, U = _heev(a, k, 1)
    u = U[0]
    assert np.abs(u.T @ u - np.eye(k)).max() < 1e-11
    h = u.T @ a @ u
    assert np.linalg.norm(a @ u - u @ h, axis=0).max() < 1e-11
    assert np.abs(np.sort(np.linalg.eigvalsh(h))[::-1] - np.sort(spec)[::-1][:k]).max() < 1e-11
