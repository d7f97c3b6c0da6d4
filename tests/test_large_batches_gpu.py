"""Batches whose blocks of 64 rows are more than one product call takes (65535 problems): the
solve and the back transformation go the way without products."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NB = 33000  # two blocks each


def _base(shape, seed=3):
    import torch
    return torch.from_numpy(np.random.default_rng(seed).standard_normal((8, *shape))).cuda()


def test_cholqr2():
    import torch

    from paper_2601_19650_gb300 import _cbc as c
    m, n = 65, 100
    b = _base((m, n))
    S = b.repeat(NB // 8, 1, 1).contiguous()
    c.cbc_cholqr2(c.CBC_F64, m, n, NB, S.data_ptr())
    eye = torch.eye(m, dtype=torch.float64, device="cuda")
    for at in (0, NB // 2, NB - 8):
        Q = S[at:at + 8]
        R = b.roll(-(at % 8), 0) @ Q.mT
        assert (Q @ Q.mT - eye).abs().max() < 1e-13
        assert (b.roll(-(at % 8), 0) - R @ Q).abs().max() < 1e-12 and R.triu(1).abs().max() < 1e-12


def test_heev():
    import torch

    from paper_2601_19650_gb300 import _cbc as c
    m, k = 65, 2
    b = _base((m, m))
    b = b + b.mT
    A = b.repeat(NB // 8, 1, 1).contiguous()
    lam = torch.zeros(NB, m, dtype=torch.float64, device="cuda")
    U = torch.zeros(NB, m, k, dtype=torch.float64, device="cuda")
    c.cbc_heev(c.CBC_F64, m, k, NB, A.data_ptr(), lam.data_ptr(), U.data_ptr(), False)
    ref = torch.linalg.eigvalsh(b.cpu()).flip(-1)[:, :k].cuda()
    for at in (0, NB // 2, NB - 8):
        s, l, u = at % 8, lam[at:at + 8, :k], U[at:at + 8]
        assert (l - ref.roll(-s, 0)).abs().max() < 1e-11
        assert (b.roll(-s, 0) @ u - u * l[:, None]).abs().max() < 1e-10
