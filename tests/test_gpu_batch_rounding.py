"""Dot products and norms of a system do not get coarser with the number of systems in the call.

Two iterations (or Arnoldi steps) on 64 copies of one system and on the system alone.  The field is uniform along
x and takes two values along z, so that nearly all terms of a sum are one of two numbers: every thread then
rounds its share the same way, and errors do not average out between threads.  Added one after the other in FP32, the
2048 elements a thread gets with the blocks of one system shared by 64 put x off by 1.2e-5 (COCG on these
two-valued vectors in numpy).  Bound, per solve: sums of at most 8 elements per thread or compensated ones, and a 5-level
shuffle tree, in FP32: 13 roundings of 6e-8 = 8e-7; the first residual's sum, at most 41 nonzero terms per thread: 6e-7;
the apply's own, at most 45 planes per thread: 6e-7 (both from adding equal random values in numpy); together
2e-6, counted for both solves, with coefficients that enter the direction of x by factors of at most one."""
import numpy as np
import pytest

from tests._gpu_util import fitlib, torch_cuda

pytestmark = pytest.mark.gpu

NX, NY, NZ, B = 256, 384, 16, 64


@pytest.mark.parametrize("method", ["cocg", "bicgstab", "fgmres"])
def test_one_of_many_as_alone(method):
    torch = torch_cuda()
    fit = fitlib()
    h = np.ones(NZ), np.ones(NY), np.ones(NX)
    shape = (NZ, NY, NX, 3)
    half = np.arange(NZ)[:, None, None, None] < NZ // 2
    eps = np.broadcast_to(np.where(half, 1.0, 10.0), shape)
    kap = np.broadcast_to(np.where(half, 0.5, 0.9), shape)
    kw = dict(method={"cocg": fit.FIT_COCG, "bicgstab": fit.FIT_BICGSTAB, "fgmres": fit.FIT_FGMRES}[method], restart=2,
              max_iter=2, max_outer=1, inner_tol=1e-12)
    xs = []
    with fit.Grid(NX, NY, NZ, h[2], h[1], h[0]) as g:
        fit.fit_set_material_matrices(g.h, eps, kap, np.ones(shape))
        row = torch.zeros(NX * NY * NZ, 3, dtype=torch.complex128, device="cuda")
        row[:, 0] = 0.7 + 0.3j
        for n in (1, B):
            b = row.reshape(1, -1).repeat(n, 1)
            x = torch.zeros_like(b)
            g.solve([1.0] * n, b, x, 1e-14, **kw)
            xs.append(x[-1].clone())
            del b, x
    assert float(xs[0].abs().max()) > 0
    assert float((xs[1] - xs[0]).norm() / xs[0].norm()) <= 4e-6
