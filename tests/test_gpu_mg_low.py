"""The one-CTA kernel of the small multigrid levels (k_mg_low): hierarchies that
start inside it at once, whose first small level is as large as it takes, with
odd counts, a single level, more than 64 cells in few rows; against the FP64
oracle's solution of the same system.  Both residuals are at most tol, so the
solutions differ by at most ||L^-1|| 2 tol (1e3 bounds the inverse on these
domains, as in test_gpu_mg.py)."""
import numpy as np
import pytest

import oracle
from paper_2402_17337_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(5, 4), (8, 8), (9, 8), (17, 16), (33, 5), (128, 64), (129, 65), (255, 31), (256, 128),
                                   (258, 130), (61, 97), (200, 12)])
def test_small_hierarchies_match_oracle(nx, ny):
    import torch
    from paper_2402_17337_gb300 import Solver, build
    build.build()
    kw = dict(x0=0.0, x1=nx / 32.0, y0=0.0, y1=ny / 32.0, nx=nx, ny=ny, hmin=0.0, dt=1.0)
    o, g = oracle.Sim(**kw), Solver(**kw, precision=2)
    b = W.random_field((ny, nx), seed=nx * ny)
    b -= b.mean()
    tol = 1e-7
    rc, phio, _, _ = o.poisson(b, tol=tol, check=8)
    assert rc == 0
    bd = torch.tensor(b, device="cuda")
    pd = torch.zeros_like(bd)
    torch.cuda.synchronize()
    rc, cycles, res = g.poisson_solve(bd.data_ptr(), pd.data_ptr(), tol, 0, 2000)
    assert rc == 0 and res <= tol and cycles < 200, (rc, cycles, res)
    assert np.abs(pd.cpu().numpy() - phio).max() <= 1e3 * 2 * tol
