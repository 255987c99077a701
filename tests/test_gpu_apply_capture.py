"""An apply captured into a CUDA graph: replays equal the plain call bit for bit (the same kernel), and read the
caller's frequency array anew, on grids with even and odd rows and in both precisions."""
import ctypes as ct

import numpy as np
import pytest

import fitgen as G
from tests._gpu_util import fitlib, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("shape", [(32, 20, 9), (33, 20, 9)])
def test_captured_apply_replays(prec, shape):
    torch = torch_cuda()
    fit = fitlib()
    case = G.small_random(*shape, seed=3, pec_frac=0.05)
    ws = [2 * np.pi * 3e9, 2 * np.pi * 8e9]
    dt = torch.complex64 if prec == 0 else torch.complex128
    with fit.Grid.from_case(case) as g:
        x = torch.from_numpy(G.random_vector(g.ne, 1)).to(dt).cuda()
        want = []
        for w in ws:  # (the first call also picks the kernel)
            y = torch.empty_like(x)
            g.apply([w], x, y, prec)
            want.append(y)
        om = torch.tensor([ws[0]], dtype=torch.float64).pin_memory()
        out = torch.zeros_like(x)
        graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            st = fit.lib().fit_apply(g.h, 1, ct.c_void_p(om.data_ptr()), x.data_ptr(), out.data_ptr(), prec,
                                     torch.cuda.current_stream().cuda_stream)
        assert st == fit.FIT_OK
        for w, y in zip(ws, want):
            om[0] = w
            out.zero_()
            graph.replay()
            assert fit.fit_sync(g.h) == fit.FIT_OK
            assert torch.equal(out, y)
