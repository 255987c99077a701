"""Every launch shape on complex64 grids with an odd nx, whose rows of x start on 8-byte boundaries (plain row
copies in place of tensor-map boxes), against the oracle's assembled A; sizes at the edges of the 32-cell
tiles, batches whose vectors start on odd and even values and end on an odd total.  A NaN or an infinity
in x reaches exactly the outputs that it reaches in the untiled kernel: nothing from a neighbouring row,
plane or system leaks into a tile's halo."""
import numpy as np
import pytest

import fitgen as G
from tests._gpu_util import fitlib, oracle_A, relerr, torch_cuda

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (3, 5, 7), (31, 9, 4), (33, 8, 5), (35, 17, 3), (65, 3, 6), (67, 16, 9)]
TOL = 1e-5  # single-precision rounding of 13-term rows, as in the other complex64 parity tests


def _run(fit, torch, g, ws, x):
    xd = torch.from_numpy(x.reshape(-1)).cuda()
    yd = torch.full_like(xd, 7.0)
    fit.fit_apply(g.h, ws, xd, yd, fit.FIT_C64)
    assert fit.fit_sync(g.h) == fit.FIT_OK
    return yd.cpu().numpy().reshape(x.shape)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("nb", [1, 2, 3])
def test_every_variant_on_odd_rows(shape, nb, monkeypatch):
    torch = torch_cuda()
    fit = fitlib()
    case = G.small_random(*shape, seed=sum(shape) + nb, pec_frac=0.06)
    ws = 2 * np.pi * np.array([5e9, 1.5e9, 12e9])[:nb]
    ne = 3 * shape[0] * shape[1] * shape[2]
    x = G.random_vector(ne, 4, np.complex64, batch=nb)
    bad = x.copy()
    bad[0, ne // 2], bad[nb - 1, 0], bad[nb - 1, ne - 1] = np.nan, np.inf, -np.inf
    want = [oracle_A(case, w) for w in ws]
    with fit.Grid.from_case(case) as g:
        monkeypatch.setenv("FIT_APPLY_KERNEL", "generic")
        nan_ref = np.isnan(_run(fit, torch, g, ws, bad))
        for k in range(fit.fit_apply_variant_count(fit.FIT_C64)):
            monkeypatch.setenv("FIT_APPLY_KERNEL", f"fused:{k}")
            y = _run(fit, torch, g, ws, x)
            for b, (A, mask) in enumerate(want):
                yo = A @ x[b].astype(np.complex128)
                assert relerr(y[b], yo) <= TOL, (k, b)
                assert np.array_equal(y[b][mask != 0], x[b][mask != 0]), (k, b)
            assert np.array_equal(np.isnan(_run(fit, torch, g, ws, bad)), nan_ref), k
