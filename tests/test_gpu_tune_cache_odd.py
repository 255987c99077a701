"""FIT_TUNE_CACHE on complex64 grids with an odd nx, whose shape is picked by rule: a recorded choice comes before
the rule, nothing is recorded for a choice by rule, and a shape that does not take such rows gives the generic
kernel's result."""
import numpy as np
import pytest

import fitgen as G
from tests._gpu_util import fitlib, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("choice", [None, -1, 0, 4, 22])
def test_a_recorded_choice_comes_first(tmp_path, monkeypatch, choice):
    torch = torch_cuda()
    fit = fitlib()
    path = tmp_path / "tune.txt"
    dims = (33, 12, 9)
    if choice is not None:
        p = torch.cuda.get_device_properties(0)
        fit.fit_tuning_record(str(path), p.name, p.multi_processor_count, *dims, fit.FIT_C64, 1, choice)
    monkeypatch.setenv("FIT_TUNE_CACHE", str(path))
    with fit.Grid.from_case(G.small_random(*dims, seed=3, pec_frac=0.05)) as g:
        x = torch.from_numpy(G.random_vector(g.ne, 1)).to(torch.complex64).cuda()
        y, want = torch.empty_like(x), torch.empty_like(x)
        g.apply([2e10], x, y)
        got = fit.fit_apply_tuned(g.h, fit.FIT_C64, 1)["choice"]
        assert got == choice if choice is not None else got >= 0
        if choice is None:
            assert not path.exists()
        monkeypatch.setenv("FIT_APPLY_KERNEL", "generic")
        g.apply([2e10], x, want)
        # every kernel sums seven products per edge in FP32
        assert float((y - want).norm() / want.norm()) <= 1e-6
