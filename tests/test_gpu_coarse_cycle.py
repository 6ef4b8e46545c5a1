"""The one-CTA coarse cycle gives the iterates of the level-by-level reference
kernels bit for bit, in both precisions, on hierarchies whose levels it holds
in register runs of every length and on those it loops over (odd extents,
walls on every axis, more column pairs than threads, one cell across)."""
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
    ((64, 32, 32), (True, False, True)),      # runs of 8, 1 planes
    ((32, 16, 8), (True, False, False)),      # runs of 2 (from 16 x 8 x 4)
    ((28, 12, 20), (False, False, False)),    # odd extents at the coarsest level, every wall
    ((60, 36, 20), (False, False, True)),     # a walled odd x, periodic z
    ((60, 60, 12), (False, False, False)),    # no even cover: loop, odd rows of 15
    ((80, 80, 4), (True, False, False)),      # more column pairs than threads
    ((24, 12, 20), (True, True, False)),      # periodic x and y
    ((16, 2, 16), (True, False, True)),       # one cell across y below the finest level
    ((1, 24, 32), (True, False, False)),      # no x coupling: transfers that halve two axes
])
def test_coarse_cycle_bit_identical_to_reference(V, shape, bc, prec):
    from paper_2601_05031_gb300.sim import Simulation
    nx, ny, nz = shape
    b = inputs.random_field((nz, ny, nx), seed=5)
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
