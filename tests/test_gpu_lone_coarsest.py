"""A coarsest level whose level above has kernels of its own, on both sides of
every limit of its kernel (register runs, shared-memory loop, one-CTA solve,
launches per colour): the iterates of the per-colour kernels bit for bit."""
import numpy as np
import pytest

import inputs

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


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("shape,bc", [
    ((28, 28, 28), (True, True, False)),      # 7 planes below 14, which no runs cover
    ((36, 30, 22), (True, False, False)),     # 2,970 cells in 11 planes
    ((44, 38, 26), (True, False, False)),     # 5,434: below the FP64 solve's 6,144 cells
    ((44, 38, 30), (False, False, False)),    # 6,270: above
    ((44, 42, 38), (True, False, False)),     # 8,778: the FP64 cycle does not fit
    ((56, 46, 38), (True, False, False)),     # 12,236: below the FP32 solve's 12,288 cells
    ((52, 50, 46), (True, False, False)),     # 14,950: above
    ((60, 54, 46), (True, False, False)),     # 18,630: the FP32 cycle does not fit
])
def test_lone_coarsest_level_bit_identical(V, shape, bc, prec):
    from paper_2601_05031_gb300.sim import Simulation
    nx, ny, nz = shape
    b = inputs.random_field((nz, ny, nx), seed=21)
    out = []
    for variant in (0, 1):
        sim = Simulation(nx, ny, nz, 1.0, V.VSV_MIXED if prec == "mixed" else V.VSV_FP64)
        sp = sim.solver_params()
        sp.variant = variant
        V.vsv_set_solver(sim.g, sp)
        x, _, _, _ = sim.solve_poisson(b, periodic=bc, tol=0.0, max_cycles=2, check=False)
        assert V.vsv_check(sim.g, check=False) == V.VSV_OK
        out.append(x)
        sim.close()
    assert np.all(np.isfinite(out[0])) and np.any(out[0])
    assert np.array_equal(out[0], out[1])
