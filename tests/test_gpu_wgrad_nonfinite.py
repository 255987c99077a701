"""Infinite and NaN activations in the conv weight gradient reach the taps that read them and no others: a row's
last voxel is read by no output at the taps x - 1, whatever the row's length leaves of its last segment.  Against
the sums in FP64 over the zero-padded input, tap by tap; tolerance as for finite inputs (1e-5 of the result's norm)."""
import pytest

from tests._gpu_util import fitlib, torch_cuda

pytestmark = pytest.mark.gpu

SHAPES = [(16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (64, 32), (32, 16)]


@pytest.mark.parametrize("cin,cout", SHAPES)
@pytest.mark.parametrize("nx", [1, 2, 7, 8, 15, 16, 17, 31, 32, 33, 40, 57, 63, 64, 65, 72, 79, 80, 100, 127])
def test_nonfinite_voxels_at_the_row_end(cin, cout, nx):
    torch = torch_cuda()
    fit = fitlib()
    ny, nz = 3, 2
    g = torch.Generator(device="cuda")
    g.manual_seed(nx + cin + cout)
    x = torch.randn(nz, ny, nx, cin, device="cuda", generator=g).to(torch.bfloat16)
    dy = torch.randn(nz, ny, nx, cout, device="cuda", generator=g).to(torch.bfloat16)
    x[1, 1, nx - 1, 3] = float("inf")
    x[0, 2, nx - 1, cin - 1] = float("nan")
    n = nx * ny * nz
    dw = torch.zeros(27, cout, cin, device="cuda")
    db = torch.zeros(cout, device="cuda")
    fit.fit_unet_conv3_wgrad(nx, ny, nz, cin, cout, x.reshape(n, cin), dy.reshape(n, cout), dw, db)
    for t in range(27):
        dz, dyy, dx = t // 9 - 1, t // 3 % 3 - 1, t % 3 - 1
        # outputs whose tap lies inside the grid
        z, y, v = (slice(max(0, -d), m - max(0, d)) for d, m in ((dz, nz), (dyy, ny), (dx, nx)))
        zs, ys, vs = (slice(max(0, d), m + min(0, d)) for d, m in ((dz, nz), (dyy, ny), (dx, nx)))
        a, b = dy[z, y, v].reshape(-1, cout).double(), x[zs, ys, vs].reshape(-1, cin).double()
        ok = torch.isfinite(b).all(0)  # channels whose voxels are all finite
        want = a.t() @ torch.where(torch.isfinite(b), b, 0.0)
        assert torch.isfinite(dw[t][:, ok]).all(), t
        assert not torch.isfinite(dw[t][:, ~ok]).any(), t
        assert float((dw[t][:, ok] - want[:, ok]).norm()) <= 1e-5 * max(float(want.norm()), 1.0), t
