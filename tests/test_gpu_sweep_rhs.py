"""FP64 time steps against the oracle on grids whose levels reach
odd extents.  There the per-colour
sweeps see every form of right-hand side (plain, negated with the wall planes)
and a start from zero on rows of every parity."""
import numpy as np
import pytest

import inputs
import oracle

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


# Poisson solves to 1e-13 leave the velocity within 1e-13 times the condition
# of these small grids (< 1e3): 1e-10.
@pytest.mark.parametrize("shape", [(14, 10, 18), (16, 10, 12), (34, 12, 10)])
@pytest.mark.parametrize("kind", ["mg", "sor"])
def test_fp64_steps_vs_oracle(V, shape, kind):
    from paper_2601_05031_gb300.sim import Simulation
    nx, ny, nz = shape
    w = inputs.droplet_duct(nx=nx, ny=ny, nz=nz, radius=3.0, dt=0.01)
    st = oracle.init_state(oracle.params_from_workload(w), w.phi0)
    for _ in range(2):
        oracle.step(st, w.dt)
    sim = Simulation.from_workload(w, V.VSV_FP64)
    sp = sim.solver_params()
    sp.tol, sp.fixed_cycles = 1e-13, 0
    if kind == "sor":
        sp.kind, sp.max_cycles, sp.check_every = V.VSV_SOLVER_SOR, 20000, 10
    V.vsv_set_solver(sim.g, sp)
    sim.set_phi(w.phi0)
    sim.step(2, w.dt)
    got = [sim.field(V.VSV_FIELD_PHI), np.stack([sim.field(V.VSV_FIELD_VEL_X + c) for c in range(3)])]
    want = [st.phi, np.stack(list(oracle.velocity(st)))]
    for a, b in zip(got, want):
        assert np.linalg.norm(a - b) <= 1e-10 * np.linalg.norm(b)
    sim.close()
