"""The residual norm that a solve reports equals the norm of b - L x of the
solution it returns, for rows of every number of lanes (fewer cells than a
warp, a tail, more cells than a CTA), in both precisions, twice on one handle."""
import numpy as np
import pytest

import inputs
from oracle.poisson import apply_poisson

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_05031_gb300 import build
    build.build()
    from paper_2601_05031_gb300 import vsv
    vsv.lib()
    return vsv


# One cycle leaves a residual of 1e-3 .. 1e-1 of b, so numpy's own rounding
# (1e-16 of L x) is < 1e-12 of it.  FP32 residuals: each rounds at 6e-8 of its
# terms, which are < 1e2 r; 1e-5 of the norm covers it.
@pytest.mark.parametrize("shape", [(1, 16, 16), (8, 6, 10), (32, 8, 6), (34, 8, 6), (66, 12, 10),
                                   (130, 4, 6), (258, 4, 4), (600, 4, 4), (256, 32, 16)])
@pytest.mark.parametrize("prec,kind", [("fp64", "mg"), ("fp64", "sor"), ("mixed", "mg")])
def test_reported_residual_is_the_residual(V, shape, prec, kind):
    from paper_2601_05031_gb300.sim import Simulation
    nx, ny, nz = shape
    bc = (True, False, False)
    sim = Simulation(nx, ny, nz, 0.8, V.VSV_FP64 if prec == "fp64" else V.VSV_MIXED)
    sp = sim.solver_params()
    sp.kind = V.VSV_SOLVER_SOR if kind == "sor" else V.VSV_SOLVER_MG
    V.vsv_set_solver(sim.g, sp)
    for seed in (3, 4):
        b = inputs.random_field((nz, ny, nx), seed=seed)
        x, cyc, rr, st = sim.solve_poisson(b, periodic=bc, tol=0.0, max_cycles=1, check=False)
        r = np.linalg.norm(b - apply_poisson(x, 0.8, bc)) / np.linalg.norm(b)
        assert cyc == 1 and r > 1e-5
        assert abs(rr - r) <= (1e-10 if prec == "fp64" else 1e-5) * r
    sim.close()
