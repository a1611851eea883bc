"""Splits of few row blocks with a long K, whose row maxima are taken by a launch of their own: products
bit for bit against the oracle around the shortest such K (384 blocks of 8 elements), with ragged last
blocks, the largest entry of a row anywhere in it, all three operations, batches whose problems have
their own K, rows at the ends of the exponent range, and non-finite entries."""
import numpy as np
import pytest

from gpu_util import rand_complex, stored
from oracle import c_oracle as co

pytestmark = pytest.mark.gpu


def _operands(m, n, k, seed):
    A, B = rand_complex(m, k, seed, 1.0), rand_complex(k, n, seed + 1, 1.0)
    for r in range(m):                                       # the row's maximum in another CTA's share each time
        A[r, (r * 7919) % k] *= 2.0 ** 20
    for c in range(n):
        B[(k - 1 - c * 104729) % k, c] *= 2.0 ** 17
    return A, B


@pytest.mark.parametrize("m,n", [(1, 1), (32, 33), (70, 20), (250, 256)])
@pytest.mark.parametrize("k", [3064, 3065, 3072, 3073, 3077, 5000])
@pytest.mark.parametrize("S,ta,tb", [(7, "N", "N"), (5, "C", "T"), (10, "T", "C"), (2, "N", "T")])
def test_products(ozk_mod, handle, m, n, k, S, ta, tb):
    A, B = _operands(m, n, k, m + k)
    C = ozk_mod.colmajor_cuda(np.zeros((m, n), dtype=np.complex128))
    for _ in range(2):                                       # the second call finds the first one's maxima cleared
        ozk_mod.ozaki_zgemm(handle, ozk_mod.colmajor_cuda(stored(A, ta)), ozk_mod.colmajor_cuda(stored(B, tb)), C, S=S,
                            transa=ta, transb=tb)
        assert handle.status() == 0
        assert np.array_equal(ozk_mod.to_numpy(C), co.zgemm(A, B, S))
        A, B = A * 2.0 ** -30, B * 2.0 ** -30


@pytest.mark.parametrize("S", [5, 7])
def test_batch_of_different_k(ozk_mod, handle, S):
    sizes = [(33, 20, 4000), (5, 60, 3), (64, 64, 3100), (20, 1, 8)]
    AB = [_operands(m, n, k, 40 + i) for i, (m, n, k) in enumerate(sizes)]
    Cs = [ozk_mod.colmajor_cuda(np.zeros((m, n), dtype=np.complex128)) for m, n, k in sizes]
    _, keep = ozk_mod.ozaki_zgemm_vbatched(handle, [ozk_mod.colmajor_cuda(a) for a, b in AB],
                                           [ozk_mod.colmajor_cuda(b) for a, b in AB], Cs, S=S)
    for (a, b), c in zip(AB, Cs):
        assert np.array_equal(ozk_mod.to_numpy(c), co.zgemm(a, b, S))
    assert handle.status() == 0
    del keep


@pytest.mark.parametrize("S", [7, 10])
def test_exponent_range_and_zero_rows(ozk_mod, handle, S):
    A, B = _operands(40, 24, 3333, 5)
    A[1] *= 2.0 ** -1060
    A[2] = 0.0
    A[3] *= 2.0 ** 900
    B[:, 7] *= 2.0 ** -300
    C = ozk_mod.colmajor_cuda(np.zeros((40, 24), dtype=np.complex128))
    ozk_mod.ozaki_zgemm(handle, ozk_mod.colmajor_cuda(A), ozk_mod.colmajor_cuda(B), C, S=S)
    assert handle.status() == 0
    assert np.array_equal(ozk_mod.to_numpy(C), co.zgemm(A, B, S))


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_entries(ozk_mod, handle, bad):
    """Flagged, and the other rows and columns come out as if the entry's row were another."""
    A, B = _operands(40, 24, 4001, 6)
    want = co.zgemm(A, B, 7)
    A[17, 4000] = bad
    C = ozk_mod.colmajor_cuda(np.zeros((40, 24), dtype=np.complex128))
    ozk_mod.ozaki_zgemm(handle, ozk_mod.colmajor_cuda(A), ozk_mod.colmajor_cuda(B), C, S=7)
    assert handle.status() & (1 << 2)
    got = ozk_mod.to_numpy(C)
    rows = np.arange(40) != 17
    assert np.array_equal(got[rows], want[rows])


def test_replayed_from_a_graph(ozk_mod):
    import torch
    h = ozk_mod.Handle()
    A, B = _operands(33, 40, 3500, 7)
    dA, dB = ozk_mod.colmajor_cuda(A), ozk_mod.colmajor_cuda(B)
    C = ozk_mod.colmajor_cuda(np.zeros((33, 40), dtype=np.complex128))
    ozk_mod.ozaki_zgemm(h, dA, dB, C, S=7)                   # scratch grows before the capture
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        h.set_stream(torch.cuda.current_stream())
        ozk_mod.ozaki_zgemm(h, dA, dB, C, S=7)
    h.set_stream(torch.cuda.current_stream())
    for f in (1.0, 2.0 ** -25):
        dA.copy_(ozk_mod.colmajor_cuda(A * f))
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(ozk_mod.to_numpy(C), co.zgemm(A * f, B, 7))
    h.close()
