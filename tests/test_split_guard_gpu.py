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
