"""Applies captured with a list of frequencies, which the binding turns into a temporary array: replays after that
array's scope has ended, and its memory would have been handed out again, equal the plain call bit for bit; the
arrays are let go with the graphs."""
import gc
import time

import numpy as np
import pytest

import fitgen as G
from tests._gpu_util import fitlib, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [1, 3, 20])  # 20: more systems than travel as kernel arguments
@pytest.mark.parametrize("own_stream", [False, True])
def test_capture_with_a_list(nb, own_stream):
    torch = torch_cuda()
    fit = fitlib()
    ws = [2 * np.pi * (3e9 + 1e8 * b) for b in range(nb)]
    with fit.Grid.from_case(G.small_random(33, 20, 9, seed=3, pec_frac=0.05)) as g:
        x = torch.from_numpy(G.random_vector(g.ne * nb, 1)).to(torch.complex64).cuda()
        want, out = torch.empty_like(x), torch.zeros_like(x)
        g.apply(ws, x, want)
        torch.cuda.synchronize()
        before = len(fit._held)
        graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(graph, stream=stream):
            g.apply(list(ws), x, out, stream=torch.cuda.current_stream() if own_stream else None)
        assert any(np.array_equal(a, ws) for a in fit._held.values())
        gc.collect()
        junk = [np.full(nb, 1e3 * k) for k in range(1000)]  # (arrays of the same size take freed memory over)
        for _ in range(2):
            out.zero_()
            graph.replay()
            assert fit.fit_sync(g.h) == fit.FIT_OK
            assert torch.equal(out, want)
        del junk, graph
        gc.collect()
        torch.cuda.synchronize()
        for _ in range(50):  # the runtime reports a destroyed graph from a thread of its own; a capture takes it out
            last, scratch = torch.cuda.CUDAGraph(), torch.cuda.Stream()
            with torch.cuda.graph(last, stream=scratch):
                g.apply(ws, x, out)
            del last
            if len(fit._held) <= before + 1:
                break
            time.sleep(0.1)
        assert len(fit._held) <= before + 1
