"""The two-sweep passes of the multigrid V-cycle (a level's whole pre- or
post-smoothing in one launch) give the iterates of the per-colour reference
kernels bit for bit at the edges of their 32 x 8 x 8 blocks and of their size
range."""
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


# one block exactly; extents below, just above and several times the block;
# a window that wraps a short axis several times; the largest finest level
# with and without the residual restricted in the pass; a level below 2^18
@pytest.mark.parametrize("shape", [(32, 8, 8), (8, 4, 4), (4, 2, 2), (36, 10, 12), (72, 18, 26),
                                   (24, 40, 6), (64, 48, 40), (64, 64, 64), (128, 64, 16),
                                   (192, 32, 48)])
@pytest.mark.parametrize("bc", [(True, False, False), (True, False, True), (True, True, False)])
def test_two_sweep_passes_bit_identical_to_reference(V, shape, bc):
    from paper_2601_05031_gb300.sim import Simulation
    nx, ny, nz = shape
    b = inputs.random_field((nz, ny, nx), seed=17)
    x0 = inputs.random_field((nz, ny, nx), seed=18)
    out, launches = [], []
    for variant in (0, 1):
        sim = Simulation(nx, ny, nz, 1.0, V.VSV_MIXED)
        sp = sim.solver_params()
        sp.variant = variant
        V.vsv_set_solver(sim.g, sp)
        n0 = sim.kernel_launches()
        x, _, _, _ = sim.solve_poisson(b, x0=x0, periodic=bc, tol=0.0, max_cycles=2, check=False,
                                       shift=0.25)
        launches.append(sim.kernel_launches() - n0)
        assert V.vsv_check(sim.g, check=False) == V.VSV_OK
        out.append(x)
        sim.close()
    assert np.all(np.isfinite(out[0])) and np.any(out[0] != x0)
    assert np.array_equal(out[0], out[1])
    assert launches[0] <= launches[1], launches
