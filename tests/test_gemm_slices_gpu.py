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
