"""Products whose K is so long that the sums of four groups pass 64 bits (digit products near the largest
with one sign over millions of elements), and the longest K below that, bit for bit against the oracle."""
import numpy as np
import pytest

from gpu_util import rand_complex
from oracle import c_oracle as co

pytestmark = pytest.mark.gpu

X127 = sum(127.0 / 256.0 ** (i + 1) for i in range(6))      # leading balanced digits all 127


def _operands(k):
    A, B = np.full((2, k), X127 * (1 - 1j)), np.full((k, 2), X127 * (1 + 1j))
    A[1] = rand_complex(1, k, 21)[0]
    B[:, 1] = rand_complex(k, 1, 22)[:, 0]
    return A, B


# groups 4..7 of the constant row and column: (5 2^24 + 6 2^16 + ...) 127^2 2 k, above 2^63 for the longer K
@pytest.mark.parametrize("k", [3_200_000, 3_600_001])
@pytest.mark.parametrize("S", [8, 9, 10])
def test_sums_beyond_64_bits(ozk_mod, handle, S, k):
    A, B = _operands(k)
    # group weights of the constant pair: digits 127 six times, then zeros
    top = sum(min(g + 1, 11 - g) * 256 ** (7 - g) for g in range(4, 8)) * 127 ** 2 * 2 * k
    assert (top >= 2 ** 63) == (k > 3_400_000)
    dA, dB = ozk_mod.colmajor_cuda(A), ozk_mod.colmajor_cuda(B)
    C = ozk_mod.colmajor_cuda(np.zeros((2, 2), dtype=np.complex128))
    ozk_mod.ozaki_zgemm(handle, dA, dB, C, S=S)
    assert handle.status() == 0
    want = co.zgemm(A, B, S)
    assert np.array_equal(ozk_mod.to_numpy(C), want)
    if S == 8:                                               # subtracted from C too
        C0 = rand_complex(2, 2, 23)
        C = ozk_mod.colmajor_cuda(C0)
        ozk_mod.ozaki_zgemm(handle, dA, dB, C, S=S, alpha=-1.0, beta=1.0)
        assert np.array_equal(ozk_mod.to_numpy(C), C0 - want)
