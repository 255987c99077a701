"""One FGMRES(m) cycle against the GMRES optimum: the smallest residual over the Jacobi-preconditioned Krylov
space of dimension m, from an Arnoldi process with repeated Gram-Schmidt in FP64 on the oracle's matrix.
m covers the edges of the complex64 passes' vector groups (4 to 32 vectors held in registers, longer bases
read twice), on a grid with an odd number of unknowns and a batch of two."""
import numpy as np
import pytest

import fitgen as G
from tests._gpu_util import fitlib, oracle_A, torch_cuda

pytestmark = pytest.mark.gpu

DIMS = (21, 13, 11)
FREQS = (4e9, 7e9)


def _optimum(A, b, m):
    """min ||b - A D^-1 V y|| / ||b|| over the m-dimensional Krylov space, D = diag(A)."""
    d = 1.0 / A.diagonal()
    V, H = [b / np.linalg.norm(b)], np.zeros((m + 1, m), complex)
    for j in range(m):
        q = A @ (d * V[j])
        for _ in range(2):
            for i in range(j + 1):
                h = np.vdot(V[i], q)
                H[i, j] += h
                q = q - h * V[i]
        H[j + 1, j] = np.linalg.norm(q)
        V.append(q / H[j + 1, j].real)
    e = np.zeros(m + 1, complex)
    e[0] = 1.0
    return np.linalg.norm(e - H @ np.linalg.lstsq(H, e, rcond=None)[0])


@pytest.mark.parametrize("m", [1, 3, 4, 5, 8, 9, 28, 29, 32, 33, 41, 64])
def test_one_cycle_reaches_the_gmres_optimum(m):
    torch = torch_cuda()
    fit = fitlib()
    case = G.small_random(*DIMS, seed=61, pec_frac=0.05)
    ws = 2 * np.pi * np.array(FREQS)
    ne = 3 * DIMS[0] * DIMS[1] * DIMS[2]
    mats = [oracle_A(case, w) for w in ws]
    mask = mats[0][1]
    b = np.stack([G.random_vector(ne, s) * (1 - mask) for s in (7, 8)])
    with fit.Grid.from_case(case) as g:
        bd = torch.from_numpy(b.reshape(-1)).cuda()
        xd = torch.zeros_like(bd)
        g.solve(ws, bd, xd, 1e-12, method=fit.FIT_FGMRES, precond=fit.FIT_PC_JACOBI, restart=m, max_outer=1,
                max_iter=m, inner_tol=1e-12)
        x = xd.cpu().numpy().reshape(2, ne)
    for i, (A, _) in enumerate(mats):
        rr = np.linalg.norm(b[i] - A @ x[i]) / np.linalg.norm(b[i])
        # FP32 Arnoldi: a backward error of about m eps on the preconditioned operator, whose condition
        # number on this lossy grid is below 50: 64 * 6e-8 * 50
        assert abs(rr - _optimum(A.tocsr(), b[i], m)) <= 2e-4, (i, rr)
