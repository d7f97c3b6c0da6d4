"""Split products of operands whose rows are wholly subnormal."""
import numpy as np
import pytest

from test_gemm_gpu import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("S", [2, 3, 4, 5])
@pytest.mark.parametrize("bits", [1, 10, 36, 37, 38, 39, 45, 46, 52])
def test_subnormal_rows(bits, S, cplx):
    """Rows of integers below 2^bits times 2^-1074: each operand is off by 2^-8S of its row's
    maximum, the dropped levels by S^2 / 2 of that (the exponent of a subnormal row may be one
    above its maximum's)."""
    rng = np.random.default_rng([bits, S])
    M, N, K = 33, 20, 40

    def ints():
        x = rng.integers(0, 2 ** bits, (M, K)).astype(float) * rng.choice([-1.0, 1.0], (M, K))
        x[:, 0] = 2.0 ** bits - 1
        return x
    a = ints() + (1j * ints() if cplx else 0)
    B = rng.standard_normal((K, N)) + (1j * rng.standard_normal((K, N)) if cplx else 0)
    B = B * 2.0 ** 200
    C, _ = _run(1, S, a * 2.0 ** -1074, B)
    ref = a @ B
    eb = 2.0 ** (np.frexp(np.abs(np.stack([B.real, B.imag])).max(axis=(0, 1)))[1])
    bound = (2 if cplx else 1) * K * 2.0 ** (bits + 1) * eb * 2.0 ** (-8 * S) * (3 + S * S / 2)
    assert np.all(np.abs(C * 2.0 ** 800 - ref * 2.0 ** -274) <= bound * 2.0 ** -274 + 2.0 ** -40 * np.abs(ref * 2.0 ** -274))
