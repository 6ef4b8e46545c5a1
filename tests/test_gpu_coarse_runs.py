"""Coarsest levels of 3, 5, 6, 9, 10 .. planes, which the one-CTA coarse cycle
holds in register runs of three or five planes (with and without levels above
in it), give the iterates of the per-colour kernels bit for bit."""
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
    ((48, 24, 20), (True, False, False)),
    ((48, 24, 20), (False, True, True)),
    ((60, 20, 10), (False, False, False)),    # odd rows of 15 columns
    ((48, 24, 12), (True, False, True)),
    ((64, 32, 24), (True, False, False)),
    ((56, 44, 30), (True, False, False)),
    ((72, 8, 18), (False, False, False)),
])
def test_runs_of_three_and_five_planes(V, shape, bc, prec):
    from paper_2601_05031_gb300.sim import Simulation
    nx, ny, nz = shape
    b = inputs.random_field((nz, ny, nx), seed=9)
    out = []
    for variant in (0, 2, 1):
        sim = Simulation(nx, ny, nz, 1.0, V.VSV_MIXED if prec == "mixed" else V.VSV_FP64)
        sp = sim.solver_params()
        sp.variant = variant
        V.vsv_set_solver(sim.g, sp)
        x, _, _, _ = sim.solve_poisson(b, periodic=bc, tol=0.0, max_cycles=2, check=False)
        assert V.vsv_check(sim.g, check=False) == V.VSV_OK
        out.append(x)
        sim.close()
    assert np.all(np.isfinite(out[0])) and np.any(out[0])
    assert np.array_equal(out[0], out[2]) and np.array_equal(out[1], out[2])
