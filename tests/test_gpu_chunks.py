"""The z-marching kernels with the short chunks of small levels (two planes in
the transfers, four in the defect, a remainder in the last chunk) give the
iterates of the reference kernels bit for bit."""
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


@pytest.mark.parametrize("shape,bc", [
    ((128, 16, 2), (True, False, False)),
    ((128, 32, 6), (True, False, True)),
    ((256, 16, 38), (True, False, False)),
    ((128, 48, 66), (True, False, False)),
    ((136, 60, 42), (True, False, True)),     # partial edge tiles
    ((384, 96, 34), (True, True, False)),
])
def test_short_chunks_bit_identical(V, shape, bc):
    from paper_2601_05031_gb300.sim import Simulation
    nx, ny, nz = shape
    b = inputs.random_field((nz, ny, nx), seed=7)
    out = []
    for variant in (0, 2, 1):
        sim = Simulation(nx, ny, nz, 1.0, V.VSV_MIXED)
        sp = sim.solver_params()
        sp.variant = variant
        V.vsv_set_solver(sim.g, sp)
        x, _, _, _ = sim.solve_poisson(b, periodic=bc, tol=0.0, max_cycles=2, check=False)
        assert V.vsv_check(sim.g, check=False) == V.VSV_OK
        out.append(x)
        sim.close()
    assert np.all(np.isfinite(out[0])) and np.any(out[0])
    assert np.array_equal(out[0], out[2]) and np.array_equal(out[1], out[2])
