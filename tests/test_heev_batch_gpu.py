"""Matrices of a batch don't touch one another: one that is not finite, or zero, spoils nothing
but its own outputs, on both ways of the back transformation."""
import numpy as np
import pytest

from test_invit_gpu import _with_spectrum

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("m,k,nb", [(40, 20, 6),     # one reflector at a time
                                    (64, 32, 40),    # products: one block of reflectors
                                    (130, 65, 7)])   # products: three blocks
@pytest.mark.parametrize("bad", [np.nan, np.inf, 0.0])
def test_bad_matrix_stays_alone(bad, m, k, nb, cplx, mixed):
    import torch

    from paper_2601_19650_gb300 import _cbc as c
    mats = [_with_spectrum(np.linspace(3.0, 1.0, m), cplx, s) for s in range(nb)]
    at = nb // 2
    if bad == 0.0:
        mats[at] = np.zeros_like(mats[at])
    else:
        mats[at][m // 2, m // 3] = mats[at][m // 3, m // 2] = bad
    dt = torch.complex128 if cplx else torch.float64
    A = torch.from_numpy(np.stack(mats)).to("cuda", dt).contiguous()
    lam = torch.zeros(nb, m, dtype=torch.float64, device="cuda")
    U = torch.zeros(nb, m, k, dtype=dt, device="cuda")
    c.cbc_heev(c.CBC_C128 if cplx else c.CBC_F64, m, k, nb, A.data_ptr(), lam.data_ptr(),
               U.data_ptr(), mixed)
    l, u = lam.cpu().numpy(), U.cpu().numpy()
    tol = 2.0 ** -46 * 300 if mixed else 2.0 ** -53 * 300
    want = np.linspace(3.0, 1.0, m)[:k]
    for b in range(nb):
        if b == at:
            continue
        assert np.abs(l[b, :k] - want).max() <= 3 * tol
        assert np.linalg.norm(mats[b] @ u[b] - u[b] * l[b, :k], axis=0).max() <= 30 * tol
        assert np.abs(u[b].conj().T @ u[b] - np.eye(k)).max() <= 40 * tol
    if bad != 0.0:  # NaN or Inf in, nothing that looks like a result out
        assert not np.isfinite(u[at]).all()
