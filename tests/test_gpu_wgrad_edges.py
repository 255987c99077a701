"""The conv weight gradient at the edges of its row segments (32 and 64 voxels), y-chunks (8 rows) and rings, for
every layer shape, against the sums in FP64; into a dw at a 4-byte offset too (scalar instead of vector
reductions).  Inputs are bf16 with exact products in FP32; the FP32 sums of n terms of unit scale are
within n eps of the FP64 ones at worst, in 2-norm about sqrt(n) eps: 1e-5 of the result's norm is ten times that for
the largest n here."""
import pytest

from tests._gpu_util import fitlib, torch_cuda

pytestmark = pytest.mark.gpu

SHAPES = [(16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (64, 32), (32, 16)]
DIMS = [(1, 1, 1), (3, 2, 5), (31, 9, 3), (33, 8, 2), (64, 17, 4), (65, 7, 3), (100, 33, 2)]


@pytest.mark.parametrize("cin,cout", SHAPES)
@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("offset", [0, 1])
def test_weight_gradient_edges(cin, cout, dims, offset):
    torch = torch_cuda()
    fit = fitlib()
    nx, ny, nz = dims
    n = nx * ny * nz
    g = torch.Generator(device="cuda")
    g.manual_seed(n + cin + cout)
    x = torch.randn(n, cin, device="cuda", generator=g).to(torch.bfloat16)
    dy = torch.randn(n, cout, device="cuda", generator=g).to(torch.bfloat16)
    buf = torch.full((27 * cout * cin + 4,), 7.0, device="cuda")
    dw, db = buf[offset:offset + 27 * cout * cin], torch.full((cout,), 7.0, device="cuda")
    fit.fit_unet_conv3_wgrad(nx, ny, nz, cin, cout, x, dy, dw, db)
    xp = torch.nn.functional.pad(x.double().reshape(nz, ny, nx, cin), (0, 0, 1, 1, 1, 1, 1, 1))
    want = torch.stack([dy.double().t() @ xp[t // 9:t // 9 + nz, t // 3 % 3:t // 3 % 3 + ny, t % 3:t % 3 + nx].reshape(n, cin)
                        for t in range(27)])
    assert float((dw.reshape(27, cout, cin) - want).norm() / want.norm()) <= 1e-5
    assert float((db - dy.double().sum(0)).norm()) <= 1e-5 * float(dy.double().norm()) * n ** 0.5
    assert torch.all(buf[:offset] == 7.0) and torch.all(buf[offset + 27 * cout * cin:] == 7.0)
