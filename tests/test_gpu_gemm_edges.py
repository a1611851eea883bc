"""Edges of the digit planes and of the slice GEMM's epilogue, bit for bit against the oracle: K
tails (a last K-block of 1..8 elements, packed into one half up to 4), row and column remainders of
the 128 x 64 tiles and of the 32-row split blocks, row blocks shared by a cluster, accumulators
above 2^22 (the corrected fold), exponents at the ends of the binary64 range, and batches whose
problems have their own K."""
import numpy as np
import pytest

from gpu_util import rand_complex, stored
from oracle import c_oracle as co

pytestmark = pytest.mark.gpu


def _product(ozk, h, A, B, S, ta="N", tb="N"):
    C = ozk.colmajor_cuda(np.zeros((A.shape[0], B.shape[1]), dtype=np.complex128))
    ozk.ozaki_zgemm(h, ozk.colmajor_cuda(stored(A, ta)), ozk.colmajor_cuda(stored(B, tb)), C, S=S, transa=ta, transb=tb)
    return ozk.to_numpy(C)


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 7, 8, 9, 12, 13, 63, 65, 72, 73, 145])
@pytest.mark.parametrize("S,ta,tb", [(3, "N", "N"), (5, "T", "C"), (6, "C", "T"), (7, "N", "T"), (8, "T", "N"), (10, "N", "N")])
def test_k_tails(ozk_mod, handle, k, S, ta, tb):
    A, B = rand_complex(35, k, seed=k), rand_complex(k, 33, seed=100 + k)
    assert np.array_equal(_product(ozk_mod, handle, A, B, S, ta, tb), co.zgemm(A, B, S))


@pytest.mark.parametrize("m,n", [(1, 1), (31, 32), (33, 31), (127, 33), (128, 64), (129, 65), (257, 97)])
@pytest.mark.parametrize("S", [4, 6, 7, 8, 9])
def test_row_and_column_remainders(ozk_mod, handle, m, n, S):
    A, B = rand_complex(m, 40, seed=m), rand_complex(40, n, seed=200 + n)
    assert np.array_equal(_product(ozk_mod, handle, A, B, S), co.zgemm(A, B, S))


@pytest.mark.parametrize("k", [129, 520, 1100, 2051])
def test_row_blocks_shared_by_a_cluster(ozk_mod, handle, k):
    A, B = rand_complex(40, k, seed=k), rand_complex(k, 36, seed=300 + k)
    assert np.array_equal(_product(ozk_mod, handle, A, B, 7), co.zgemm(A, B, 7))


@pytest.mark.parametrize("S", [3, 5, 6, 7, 8])
@pytest.mark.parametrize("k", [40, 72, 300])
def test_accumulators_beyond_the_small_range(ozk_mod, handle, S, k):
    """Equal values whose digits are near the largest magnitude in every slice: the group sums pass
    2^22 in some tiles' rows, and stay small in the rows of random values next to them."""
    x = sum(128.0 / 256.0 ** (s + 1) for s in range(7)) * 0.999
    A, B = np.full((70, k), x - 1j * x), np.full((k, 40), x + 1j * x)
    A[::3] = rand_complex(24, k, seed=S)
    B[:, 1::2] *= -1.0
    assert np.array_equal(_product(ozk_mod, handle, A, B, S), co.zgemm(A, B, S))


@pytest.mark.parametrize("S", [3, 4, 7, 8, 10])
@pytest.mark.parametrize("pa,pb", [(-500, -480), (-540, -530), (500, 480), (600, -560), (520, 503), (-1030, 900),
                                   (-1060, 1000), (980, -1050)])
def test_exponents_at_the_ends_of_the_range(ozk_mod, handle, S, pa, pb):
    A, B = rand_complex(37, 20, seed=9), rand_complex(20, 35, seed=10)
    # all but one row and one column (ordinary ones in the same tile)
    A[np.arange(37) != 3] *= 2.0 ** pa
    B[:, np.arange(35) != 5] *= 2.0 ** pb
    assert np.array_equal(_product(ozk_mod, handle, A, B, S), co.zgemm(A, B, S))


@pytest.mark.parametrize("S", [5, 7])
def test_batch_of_different_k(ozk_mod, handle, S):
    sizes = [(33, 20, 1), (130, 37, 12), (64, 64, 8), (5, 70, 100), (128, 33, 73), (1, 1, 3), (40, 129, 145)]
    As = [rand_complex(m, k, seed=i) for i, (m, n, k) in enumerate(sizes)]
    Bs = [rand_complex(k, n, seed=50 + i) for i, (m, n, k) in enumerate(sizes)]
    Cs = [ozk_mod.colmajor_cuda(np.zeros((m, n), dtype=np.complex128)) for m, n, k in sizes]
    _, keep = ozk_mod.ozaki_zgemm_vbatched(handle, [ozk_mod.colmajor_cuda(a) for a in As],
                                           [ozk_mod.colmajor_cuda(b) for b in Bs], Cs, S=S)
    for a, b, c in zip(As, Bs, Cs):
        assert np.array_equal(ozk_mod.to_numpy(c), co.zgemm(a, b, S))
    del keep
