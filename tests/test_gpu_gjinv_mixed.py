"""Launches of more than half as many pivot blocks as SMs, at most one per SM, with a widest block above
order 80: blocks of order 57..64 are inverted in registers, the others in shared memory.  tau_00 of
matrices whose blocks need row interchanges, against the full-inverse oracle and bit for bit the solve by
itself (whose block is spread over a cluster), and a singular block of either kind."""
import numpy as np
import pytest

from oracle import c_oracle as co
from oracle import kkr

pytestmark = pytest.mark.gpu

ORDERS = [96, 57, 64, 60, 56, 65, 33, 63]                    # panels of 96: one pivot block a solve


def _matrix(w, seed):
    """Order 1 + w, its pivot block dominated by the reversal permutation, zero diagonal in the block."""
    rng = np.random.default_rng(seed)
    n = 1 + w
    M = 0.02 * (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    M[0, 0] += 1.0
    for r in range(w):
        M[1 + r, w - r] += 1.0
        if w - r != 1 + r:
            M[1 + r, 1 + r] = 0.0
    return M


def _solve(ozk, h, Ms, nb):
    t0 = np.array([[0.3 + 0.1j]])
    dM = [ozk.colmajor_cuda(M) for M in Ms]
    dt = [ozk.colmajor_cuda(t0) for _ in Ms]
    taus = [ozk.colmajor_cuda(np.zeros((1, 1), dtype=np.complex128)) for _ in Ms]
    ozk.kkr_tau00_batched(h, dM, dt, taus, S=8, nb=nb)
    st = h.status()
    return [ozk.to_numpy(t) for t in taus], [ozk.to_numpy(M) for M in dM], st


@pytest.mark.parametrize("batch", [77, 100, 152])
def test_mixed_orders(ozk_mod, handle, batch):
    Ms = [_matrix(w, i) for i, w in enumerate(ORDERS)]
    taus, outs, st = _solve(ozk_mod, handle, [Ms[i % len(Ms)] for i in range(batch)], 96)
    assert st == 0
    for q, M in enumerate(Ms):
        alone, out, st = _solve(ozk_mod, handle, [M], 96)
        assert st == 0
        # the bound of the row-interchange tests at S >= 7
        assert kkr.rel_err(alone[0], co.tau00_full(M, np.array([[0.3 + 0.1j]]))) < 1e-10, ORDERS[q]
        for i in range(q, batch, len(Ms)):
            assert np.array_equal(taus[i], alone[0]) and np.array_equal(outs[i], out[0]), (i, ORDERS[q])


@pytest.mark.parametrize("order", [60, 96])
def test_singular_block(ozk_mod, handle, order):
    Ms = [_matrix(w, i) for i, w in enumerate(ORDERS)]
    q = ORDERS.index(order)
    bad = Ms[q].copy()
    bad[1:, -5] = 0.0
    taus, _, st = _solve(ozk_mod, handle, [bad if i == q else Ms[i % len(Ms)] for i in range(100)], 96)
    assert st & (1 << 3)
    for i in range(100):
        if i != q:
            want = co.tau00_full(Ms[i % len(Ms)], np.array([[0.3 + 0.1j]]))
            assert kkr.rel_err(taus[i], want) < 1e-10, i
