"""The field solve against the exact solution of the discrete equation (Fourier modes in x
and y, a tridiagonal solve in z, in 64 bits), on meshes that take the V-cycle and its
exact coarse level through their different branches: coarse slabs of few values (4 per
thread), of many (16 per thread) and of both kinds side by side; one grid-wide level and
several; in float the finest level's first red half-sweep folded into the black one.  The
iteration count is that of a V(2,2) cycle (0.1 per iteration): a node left uncorrected
would show there, since the refinement hides it in the result."""
import numpy as np
import pytest

import paper_1801_00972_gb300 as P
from paper_1801_00972_gb300 import build as B
from paper_1801_00972_gb300 import inputs as I

pytestmark = pytest.mark.gpu
EPS0 = 8.8541878128e-12


def _exact(wl, rho):
    """Potential, and the bound of its error for a residual of 1e-10 of the right-hand side."""
    nx, ny, nz = wl.nx, wl.ny, wl.nz
    f = (rho.astype(np.float64) * (I.QE * wl.weight / wl.dx ** 3 * 2.0 ** -42 / EPS0) * wl.dx ** 2).reshape(nz + 1, ny, nx)
    f = f[1:nz].copy()
    f[0] += wl.v_dc
    norm = np.sqrt((f ** 2).sum())
    g = np.fft.rfft2(f, axes=(1, 2))
    lam = (2 - 2 * np.cos(2 * np.pi * np.arange(ny) / ny))[:, None] + (2 - 2 * np.cos(2 * np.pi * np.arange(nx // 2 + 1) / nx))
    p = np.zeros((nz - 1,) + lam.shape)
    for k in range(nz - 1):
        p[k] = 1.0 / (2.0 + lam - (p[k - 1] if k else 0.0))
        g[k] = p[k] * (g[k] + (g[k - 1] if k else 0.0))
    for k in range(nz - 3, -1, -1):
        g[k] += p[k] * g[k + 1]
    phi = np.zeros((nz + 1, ny, nx))
    phi[0] = wl.v_dc
    phi[1:nz] = np.fft.irfft2(g, s=(ny, nx), axes=(1, 2))
    phi = phi.reshape(-1)
    # |error| <= |residual| / smallest eigenvalue, and the rounding of the two-float potential
    return phi, 1e-10 * norm / (2 - 2 * np.cos(np.pi / nz)) + 1e-13 * np.sqrt((phi ** 2).sum())


MESHES = [(16, 16, 16), (32, 32, 64), (64, 64, 32), (64, 64, 256), (80, 48, 100), (96, 120, 20), (96, 88, 20), (32, 64, 6)]


@pytest.mark.parametrize("mesh,prec", [(m, p) for m in MESHES for p in (P.PIC_MIXED, P.PIC_FP64)] +
                         [((144, 120, 10), P.PIC_MIXED)])   # (its coarse level does not fit a cluster in FP64)
def test_solve_from_zero_matches_the_exact_solution(mesh, prec):
    import torch
    B.build()
    torch.cuda.set_device(0)
    wl = I.small(nx=mesh[0], ny=mesh[1], nz=mesh[2], n_e=20000, n_i=21000, grains=0, v_dc=-50.0)
    run = P.Run(wl, I.sample_particles(wl), prec=prec, stream=torch.cuda.current_stream().cuda_stream)
    phi, bound = _exact(wl, run.rho())
    run.set_phi(np.zeros(wl.nodes))
    it, res = run.solve()
    assert res <= 1e-10 and it <= 10
    assert np.sqrt(((run.phi() - phi) ** 2).sum()) <= bound
    run.close()
