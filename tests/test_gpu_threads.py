"""Calls of several host threads, each with its own handle and stream, whose kernels are the same but
need different amounts of shared memory: every launch must be accepted, whatever another thread's call
of the same kernel needs in between, and every result be the one of a call by itself."""
import threading

import numpy as np
import pytest

from gpu_util import rand_complex

pytestmark = pytest.mark.gpu


def _run(works, rounds):
    """Each work(i) in a thread of its own, `rounds` times; the first error of any of them."""
    errors, gate = [], threading.Barrier(len(works))

    def loop(work):
        try:
            gate.wait()
            for i in range(rounds):
                if errors:
                    return
                work(i)
        except Exception as ex:                              # noqa: BLE001 (reported by the test)
            errors.append(ex)

    ts = [threading.Thread(target=loop, args=(w,)) for w in works]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    return errors


def _product(ozk, S, mode, n, seed):
    import torch
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        h = ozk.Handle(st)
        A, B = (ozk.colmajor_cuda(rand_complex(n, n, seed + i)) for i in range(2))
        C, want = (ozk.colmajor_cuda(np.zeros((n, n), dtype=np.complex128)) for _ in range(2))
        ozk.ozaki_zgemm(h, A, B, want, S=S, pair_mode=mode)
    st.synchronize()

    def work(i):
        ozk.ozaki_zgemm(h, A, B, C, S=S, pair_mode=mode)
        if i % 50 == 49:
            st.synchronize()
            assert torch.equal(C, want)
    return work, h


def _solve(ozk, nb, b, seed):
    import torch
    n = b + 2 * nb
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        h = ozk.Handle(st)
        M = ozk.colmajor_cuda(np.eye(n) + 0.3 / np.sqrt(n) * rand_complex(n, n, seed, 0.0))
        W = ozk.colmajor_cuda(np.zeros((n, n), dtype=np.complex128))
        t0 = ozk.colmajor_cuda(np.eye(b, dtype=np.complex128))
        tau, want = (ozk.colmajor_cuda(np.zeros((b, b), dtype=np.complex128)) for _ in range(2))
        W.copy_(M)
        ozk.kkr_tau00(h, W, t0, want, S=7, nb=nb)
    st.synchronize()

    def work(i):
        with torch.cuda.stream(st):
            W.copy_(M)
            ozk.kkr_tau00(h, W, t0, tau, S=7, nb=nb)
        if i % 50 == 49:
            st.synchronize()
            assert torch.equal(tau, want)
    return work, h


def _check(made, rounds):
    errors = _run([w for w, _ in made], rounds)
    assert not errors, errors[0]
    for _, h in made:
        assert h.status() == 0
        h.close()


def test_products_of_different_slice_counts(ozk_mod):
    tri, full = ozk_mod.OZK_PAIRS_TRI, ozk_mod.OZK_PAIRS_FULL
    _check([_product(ozk_mod, S, mode, 40, 10 * S) for S, mode in ((2, tri), (2, full), (4, full))], 1500)


def test_solves_of_different_block_orders(ozk_mod):
    _check([_solve(ozk_mod, nb, b, nb) for nb, b in ((112, 16), (16, 16), (104, 52), (48, 48))], 400)
