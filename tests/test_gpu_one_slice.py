"""Products with one slice (S = 1: one group of accumulators, whose second part is empty), bit for bit
against the oracle: CTAs that run several tiles of one K-block or of several exactness chunks (512
elements of K each), stored and subtracted from C, with warps that have no output in their tile."""
import numpy as np
import pytest

from gpu_util import rand_complex
from oracle import c_oracle as co

pytestmark = pytest.mark.gpu


# (m, n): 128 x 64 stacked tiles -- 352 of them on at most 152 SMs, the last columns 4 wide; 3 of which
# 3 slabs of 16 columns are idle; 200 of them for the longest K
@pytest.mark.parametrize("m,n,k", [(2000, 674, 8), (2000, 674, 5), (300, 3, 1600), (40, 33, 2100), (900, 770, 1030)])
@pytest.mark.parametrize("pairs", ["tri", "full"])
def test_one_slice(ozk_mod, handle, m, n, k, pairs):
    mode = ozk_mod.OZK_PAIRS_TRI if pairs == "tri" else ozk_mod.OZK_PAIRS_FULL
    A, B, C0 = rand_complex(m, k, 500 + k, 0.5), rand_complex(k, n, 600 + k, 0.5), rand_complex(m, n, 700 + k, 0.5)
    dA, dB, dC = ozk_mod.colmajor_cuda(A), ozk_mod.colmajor_cuda(B), ozk_mod.colmajor_cuda(C0)
    want = co.zgemm(A, B, 1)
    ozk_mod.ozaki_zgemm(handle, dA, dB, dC, S=1, pair_mode=mode)
    assert handle.status() == 0
    assert np.array_equal(ozk_mod.to_numpy(dC), want)
    dC = ozk_mod.colmajor_cuda(C0)
    ozk_mod.ozaki_zgemm(handle, dA, dB, dC, S=1, alpha=-1.0, beta=1.0, pair_mode=mode)
    assert handle.status() == 0
    assert np.array_equal(ozk_mod.to_numpy(dC), C0 - want)
