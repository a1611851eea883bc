"""Selector kernels at the sizes where their work is dealt differently: more vectors than one pass of the
features' cluster, many chunks of a probe product, and both forms of the perceptron."""
import numpy as np
import pytest

from gpu_util import rand_complex, stored
from oracle import selector as sel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mnk,ta,tb", [((2049, 5, 33), "N", "N"), ((3, 2300, 17), "N", "T"),
                                       ((3000, 31, 321), "N", "N"), ((47, 1, 2600), "T", "N"),
                                       ((31, 33, 1), "N", "C"), ((1, 1, 1), "N", "N")])
def test_features_over_the_range_of_sizes(ozk_mod, handle, mnk, ta, tb):
    m, n, k = mnk
    A, B = rand_complex(m, k, 51, 2.0), rand_complex(k, n, 52, 2.0)
    if m > 8:
        A[m - 1, :] = 0
        A[5, :] *= 2.0 ** -700                # its power of 4 is below the normal range
    f = ozk_mod.to_numpy(ozk_mod.selector_features(handle, ozk_mod.colmajor_cuda(stored(A, ta)),
                                                   ozk_mod.colmajor_cuda(stored(B, tb)), ta, tb, seed=3))
    want, _, _ = sel.features(A, B, sel.probe_vectors(n, 3))
    assert np.abs(f - want).max() <= 2e-6 * max(1.0, np.abs(want).max())


def test_residual_of_a_product_of_many_chunks(ozk_mod, handle):
    m, n, k = 1300, 1000, 40
    A, B = rand_complex(m, k, 61, 1.0), rand_complex(k, n, 62, 1.0)
    p = np.zeros(sel.NPARAMS, dtype=np.float32)
    p[sel.OFF_B3:] = -30                      # S = 3
    handle.selector_set_params(p)
    handle.selector_configure(tol=1e-1, margin=0.0)
    C = ozk_mod.colmajor_cuda(np.zeros((m, n), dtype=np.complex128))
    ozk_mod.ozaki_zgemm(handle, ozk_mod.colmajor_cuda(A), ozk_mod.colmajor_cuda(B), C, S=0)
    info = handle.selector_last()
    assert info["S_selected"] == 3 and not info["fallback"]
    X = sel.probe_vectors(n, info["probe_seed"])
    z, W = A @ (B @ X), ozk_mod.to_numpy(C) @ X
    r = np.linalg.norm(W - z) / np.linalg.norm(z)
    # binary64 sums of up to 1000 products on both sides: 1000 eps sqrt(1000) is 7e-12
    assert r > 1e-8 and abs(info["residual"] - r) <= 1e-11
    handle.selector_configure()


def test_perceptron_forms_agree(ozk_mod, handle):
    """A sample alone and as one of more samples than there are SMs: the same bits."""
    import torch
    rng = np.random.default_rng(9)
    handle.selector_set_params(rng.normal(0, 0.3, sel.NPARAMS).astype(np.float32))
    F = rng.normal(size=(400, 16)).astype(np.float32)
    many = ozk_mod.to_numpy(ozk_mod.selector_predict(handle, torch.from_numpy(F).cuda()))
    few = [ozk_mod.to_numpy(ozk_mod.selector_predict(handle, torch.from_numpy(F[i:i + 3]).cuda())) for i in (0, 101, 397)]
    for i, got in zip((0, 101, 397), few):
        assert np.array_equal(got, many[i:i + 3])
