"""Kernels that start while the one before them in the stream ends: products whose operands the kernels right
before write and whose results and operands the kernels right after read and overwrite, on the default stream,
on another one and replayed from a CUDA graph, against the same calls with the stream drained in between."""
import numpy as np
import pytest

from gpu_util import rand_complex

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [5, 64, 200])
@pytest.mark.parametrize("S", [0, 3, 7, 10])
@pytest.mark.parametrize("where", ["default", "stream", "graph"])
def test_chains_of_products_in_stream_order(ozk_mod, n, S, where):
    import torch
    if S == 0 and where == "graph":
        pytest.skip("S = 0 reads its choice on the host: refused under capture")
    h = ozk_mod.Handle()
    if S == 0:
        h.selector_load()
    A0, B0 = ozk_mod.colmajor_cuda(rand_complex(n, n, 71, 0.5)), ozk_mod.colmajor_cuda(rand_complex(n, n, 72, 0.5))
    A, B, C = (ozk_mod.colmajor_cuda(np.zeros((n, n), dtype=np.complex128)) for _ in range(3))

    def chain(drain):
        A.copy_(A0)
        B.copy_(B0)
        for i in range(6):
            ozk_mod.ozaki_zgemm(h, A, B, C, S=S)
            if drain:
                torch.cuda.synchronize()
            A.copy_(C)                                   # the operand just read, from the result just written
            A.mul_(1.0 / n)
            if drain:
                torch.cuda.synchronize()
            ozk_mod.ozaki_zgemm(h, C, A, B, S=S, alpha=0.25, beta=0.5 + 0.1j)
            if drain:
                torch.cuda.synchronize()
            B.mul_(1.0 / n)
        return ozk_mod.to_numpy(B)

    h.set_stream(torch.cuda.current_stream())
    want = chain(True)
    if where == "default":
        got = chain(False)
    elif where == "stream":
        st = torch.cuda.Stream()
        st.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(st):
            h.set_stream(st)
            got = chain(False)
        st.synchronize()
        h.set_stream(torch.cuda.current_stream())
    else:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            h.set_stream(torch.cuda.current_stream())
            A.copy_(A0)
            B.copy_(B0)
            for i in range(6):
                ozk_mod.ozaki_zgemm(h, A, B, C, S=S)
                A.copy_(C)
                A.mul_(1.0 / n)
                ozk_mod.ozaki_zgemm(h, C, A, B, S=S, alpha=0.25, beta=0.5 + 0.1j)
                B.mul_(1.0 / n)
        h.set_stream(torch.cuda.current_stream())
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        got = ozk_mod.to_numpy(B)
    assert np.all(np.isfinite(want)) and np.array_equal(got, want)
    assert h.status() == 0
    h.close()
