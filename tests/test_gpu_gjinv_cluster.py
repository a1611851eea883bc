"""Pivot-block inverses spread over clusters of 8, 4 and 2 CTAs (launches that leave SMs idle): tau_00
of matrices whose pivot blocks need row interchanges, over the orders and batch sizes where the
columns' split is ragged or the cluster size changes, against the full-inverse oracle, and a singular
block, which every CTA of the cluster has to leave together."""
import numpy as np
import pytest

from oracle import c_oracle as co
from oracle import kkr

pytestmark = pytest.mark.gpu


def _matrix(b, w, seed):
    """Order b + 2 w, every block of the elimination dominated by its reversal permutation, zero diagonal."""
    rng = np.random.default_rng(seed)
    n = b + 2 * w
    M = 0.02 * (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    for lo, hi in ((0, b), (b, b + w), (b + w, n)):
        for r in range(hi - lo):
            M[lo + r, hi - 1 - r] += 1.0
    np.fill_diagonal(M, 0.0)
    return M


@pytest.mark.parametrize("b,w", [(2, 2), (3, 9), (4, 20), (1, 33), (8, 64), (5, 65), (16, 96), (16, 112)])
@pytest.mark.parametrize("batch", [1, 20, 40, 80])
def test_orders_and_batch_sizes(ozk_mod, handle, b, w, batch):
    Ms = [_matrix(b, w, i) for i in range(min(batch, 3))]
    t0 = np.eye(b, dtype=np.complex128) * (0.3 + 0.1j)
    dM = [ozk_mod.colmajor_cuda(Ms[i % len(Ms)]) for i in range(batch)]
    dt = [ozk_mod.colmajor_cuda(t0) for _ in range(batch)]
    taus = [ozk_mod.colmajor_cuda(np.zeros((b, b), dtype=np.complex128)) for _ in range(batch)]
    ozk_mod.kkr_tau00_batched(handle, dM, dt, taus, S=8, nb=w)
    assert handle.status() == 0
    # the bound of the row-interchange tests at S >= 7
    for i in range(batch):
        assert kkr.rel_err(ozk_mod.to_numpy(taus[i]), co.tau00_full(Ms[i % len(Ms)], t0)) < 1e-10, i


@pytest.mark.parametrize("batch", [1, 20, 40])
def test_singular_block_of_a_batch(ozk_mod, handle, batch):
    """One singular pivot block sets the status; the other solves of the launch are unaffected."""
    b, w = 16, 48
    M = _matrix(b, w, 7)
    bad = M.copy()
    bad[:, -5] = 0.0
    t0 = np.eye(b, dtype=np.complex128)
    dM = [ozk_mod.colmajor_cuda(bad if i == 0 else M) for i in range(batch)]
    dt = [ozk_mod.colmajor_cuda(t0) for _ in range(batch)]
    taus = [ozk_mod.colmajor_cuda(np.zeros((b, b), dtype=np.complex128)) for _ in range(batch)]
    ozk_mod.kkr_tau00_batched(handle, dM, dt, taus, S=8, nb=w)
    assert handle.status() & (1 << 3)
    want = co.tau00_full(M, t0)
    for i in range(1, batch):
        assert kkr.rel_err(ozk_mod.to_numpy(taus[i]), want) < 1e-10, i


@pytest.mark.parametrize("b,w", [(2, 2), (8, 64), (16, 80), (16, 96)])
@pytest.mark.parametrize("batch", [100, 152])
def test_two_clusters_an_sm(ozk_mod, handle, b, w, batch):
    """More blocks than SM pairs: clusters of two CTAs share SMs up to order 80."""
    Ms = [_matrix(b, w, 7 + i) for i in range(2)]
    t0 = np.eye(b, dtype=np.complex128) * (0.3 + 0.1j)
    dM = [ozk_mod.colmajor_cuda(Ms[i % 2]) for i in range(batch)]
    dt = [ozk_mod.colmajor_cuda(t0) for _ in range(batch)]
    taus = [ozk_mod.colmajor_cuda(np.zeros((b, b), dtype=np.complex128)) for _ in range(batch)]
    ozk_mod.kkr_tau00_batched(handle, dM, dt, taus, S=8, nb=w)
    assert handle.status() == 0
    want = [co.tau00_full(M, t0) for M in Ms]
    for i in range(batch):
        assert kkr.rel_err(ozk_mod.to_numpy(taus[i]), want[i % 2]) < 1e-10, i
