"""Accumulators at and above 2^22 (the second reading of a part, which corrects what the first folded as
small values), bit for bit against the oracle, in every form of the fold: 64-bit sums, two 64-bit halves
(S = 6..8, and S = 5 with a long K), halves of a split K, and the quads of S = 9 and 10; stored and
subtracted from C.  Whether the operands get there is asserted from the oracle's digits."""
import numpy as np
import pytest

from gpu_util import rand_complex
from oracle import c_oracle as co

pytestmark = pytest.mark.gpu

# leading balanced digits all 127
X127 = sum(127.0 / 256.0 ** (i + 1) for i in range(6))


def _operands(m, n, k):
    A, B = np.full((m, k), X127 * (1 - 1j)), np.full((k, n), X127 * (1 + 1j))
    A[1::3] = rand_complex(len(range(1, m, 3)), k, 11)       # small sums beside the large ones
    B[:, 2::3] = rand_complex(k, len(range(2, n, 3)), 12)
    A[2::3] *= -1.0
    return A, B


def _chunk(S):
    return 8 * max(1, 64 // S)                               # elements of K per exactness chunk


def _largest_sum(A, B, S):
    """Largest |group sum| of one chunk at row 0, column 0, from the oracle's digits."""
    k, L = A.shape[1], _chunk(S)
    DA, DB = co.split_left(A[:1], S)[1][:, 0], co.split_right(B[:, :1], S)[1][:, 0]
    best = 0
    for g in range(S):
        P = sum(DA[s] * DB[g - s] for s in range(g + 1))
        P = P[:k] + P[k:]
        best = max(best, max(abs(int(P[c:c + L].sum())) for c in range(0, k, L)))
    return best


@pytest.mark.parametrize("S,k", [(S, 2 * _chunk(S) + 5) for S in range(3, 11)] + [(5, 6600)])
@pytest.mark.parametrize("update", [False, True])
def test_sums_of_a_batch(ozk_mod, handle, S, k, update):
    """Batched products: one unit per tile, chunks one after the other."""
    A, B = _operands(70, 40, k)
    assert 2 ** 22 < _largest_sum(A, B, S) <= 2 ** 24
    C0 = rand_complex(70, 40, 13) if update else np.zeros((70, 40), dtype=np.complex128)
    C = ozk_mod.colmajor_cuda(C0)
    ab = dict(alpha=-1.0, beta=1.0) if update else {}
    _, keep = ozk_mod.ozaki_zgemm_vbatched(handle, [ozk_mod.colmajor_cuda(A)], [ozk_mod.colmajor_cuda(B)], [C], S=S, **ab)
    want = co.zgemm(A, B, S)
    assert np.array_equal(ozk_mod.to_numpy(C), C0 - want if update else want)
    assert handle.status() == 0
    del keep


@pytest.mark.parametrize("S,chunks", [(6, 3), (7, 3), (7, 10), (8, 10), (9, 3), (10, 3), (5, 69)])
@pytest.mark.parametrize("update", [False, True])
def test_sums_of_a_single_product(ozk_mod, handle, S, chunks, update):
    """Single products: K split into up to 8 units of one or more chunks (S <= 8 with sums beyond 64 bits)."""
    k = (chunks - 1) * _chunk(S) + 5
    A, B = _operands(70, 40, k)
    assert 2 ** 22 < _largest_sum(A, B, S) <= 2 ** 24
    C0 = rand_complex(70, 40, 14) if update else np.zeros((70, 40), dtype=np.complex128)
    C = ozk_mod.colmajor_cuda(C0)
    ozk_mod.ozaki_zgemm(handle, ozk_mod.colmajor_cuda(A), ozk_mod.colmajor_cuda(B), C, S=S,
                        **(dict(alpha=-1.0, beta=1.0) if update else {}))
    want = co.zgemm(A, B, S)
    assert np.array_equal(ozk_mod.to_numpy(C), C0 - want if update else want)
    assert handle.status() == 0
