"""The Cholesky factor of CholeskyQR2 at the edges of its kernels, through cbc_cholqr2: sizes
around a pair of columns and the rows per CTA, batches that take clusters of 16, 4 and 2 CTAs
and one CTA each, a row far smaller than the others (the rows are scaled to unit norm before), and rows that repeat an
earlier one; and the triangular solve by products (batches with enough work) at the edges of
its blocks of 64 rows and their halves, nearly dependent rows among them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _run(S):
    import torch

    from paper_2601_19650_gb300 import _cbc as c
    nb, m, n = S.shape
    d = torch.from_numpy(np.ascontiguousarray(S)).to("cuda")
    c.cbc_cholqr2(c.CBC_C128 if np.iscomplexobj(S) else c.CBC_F64, m, n, nb, d.data_ptr())
    return d.cpu().numpy()


def _random(nb, m, cplx):
    r = np.random.default_rng([nb, m, cplx])
    shape = (nb, m, 2 * m + 3)
    return r.standard_normal(shape) + (1j * r.standard_normal(shape) if cplx else 0)


def _check(S, Q):
    # two passes leave a few roundings of sums of up to 800 terms: well below 1e-13
    for s, q in zip(S, Q):
        m = len(s)
        assert np.abs(q @ q.conj().T - np.eye(m)).max() < 1e-13
        # S = R Q row by row (the rows' norms may differ), R lower triangular, diagonal > 0
        norm = np.linalg.norm(s, axis=1, keepdims=True)
        R = (s / norm) @ q.conj().T
        assert np.linalg.norm(s / norm - R @ q, axis=1).max() < 1e-12
        assert np.abs(np.triu(R, 1)).max() < 1e-12
        dg = np.diag(R)
        assert np.all(dg.real > 0) and np.abs(dg.imag).max() < 1e-12


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("m,nb", [(1, 1), (2, 1), (3, 1), (4, 1), (5, 1), (17, 1), (31, 3),
                                  (33, 1), (63, 1), (65, 3), (129, 1), (200, 1), (257, 1),
                                  (400, 1), (33, 20), (64, 20), (65, 70), (7, 100), (130, 100)])
def test_sizes_and_batches(m, nb, cplx):
    S = _random(nb, m, cplx)
    _check(S, _run(S))


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("row", [0, 3, 4, 11])
def test_tiny_row(row, cplx):
    S = _random(1, 12, cplx)
    S[0, row] *= 2.0 ** -516  # its squared norm is denormal
    _check(S, _run(S))


@pytest.mark.parametrize("nb", [1, 20])
@pytest.mark.parametrize("pair", [(3, 7), (0, 1), (6, 7), (7, 8), (5, 39)])
def test_repeated_row_is_reported(pair, nb):
    from paper_2601_19650_gb300 import _cbc as c
    S = np.random.default_rng(3).standard_normal((nb, 40, 200))
    S[nb - 1, pair[1]] = S[nb - 1, pair[0]]
    with pytest.raises(c.CBCError) as ei:
        _run(S)
    assert ei.value.code == 4


@pytest.mark.parametrize("m,n,nb,cplx", [(33, 70, 200, True), (40, 41, 240, True),
                                         (64, 64, 60, True), (65, 131, 56, True),
                                         (97, 195, 24, True), (130, 261, 12, True),
                                         (128, 130, 32, False), (128, 130, 64, False),
                                         (129, 300, 40, False)])
def test_solve_by_products(m, n, nb, cplx):
    # by products where m^2 n nb (times 4 if complex) is 6e7 or more per block of 64 rows: all
    # of these but the 32 of 128 x 130, which lie below the line
    r = np.random.default_rng([m, n, nb])
    S = r.standard_normal((nb, m, n)) + (1j * r.standard_normal((nb, m, n)) if cplx else 0)
    S[:, 5] = S[:, 4] + 1e-5 * S[:, 5]
    S[:, m - 1] = S[:, 0] + 1e-5 * S[:, m - 1]
    S[:, 7] *= 2.0 ** -300
    _check(S, _run(S))
