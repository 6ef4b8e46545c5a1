"""The observables of the mixed path against the oracle's operators evaluated on
the exported state in FP64: velocity (double words summed by error-free FP32
transforms), in-plane stress, stress profile and diagnostics, on 4-cell groups
and on extents that have none, for walls and periodic z, and a spacing whose
1 / 2h is no power of two."""
import numpy as np
import pytest

import inputs
import oracle
from oracle.diagnostics import velocity_gradient
from oracle.grid import curl

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
@pytest.mark.parametrize("shape,h,flow", [((40, 24, 20), 1.0, inputs.COUETTE),
                                          ((22, 14, 18), 1.0, inputs.POISEUILLE_DUCT),
                                          ((24, 16, 12), 0.7, inputs.POISEUILLE_PLANAR)])
def test_observables_of_the_exported_state(V, shape, h, flow, prec):
    import torch
    from paper_2601_05031_gb300.sim import Simulation
    nx, ny, nz = shape
    w = inputs.droplet_duct(nx=nx, ny=ny, nz=nz, radius=4.0, flow_kind=flow)
    w.h = h
    if flow == inputs.COUETTE:
        w.u_max, w.v_lo, w.v_hi = 0.0, -0.05, 0.07
    p = V.VSV_MIXED if prec == "mixed" else V.VSV_FP64
    sim = Simulation.from_workload(w, p)
    sp = sim.solver_params()
    sp.tol, sp.fixed_cycles = 1e-6, 0
    V.vsv_set_solver(sim.g, sp)
    sim.set_phi(w.phi0)
    st = oracle.init_state(oracle.params_from_workload(w), w.phi0)
    psi = [sim.field(V.VSV_FIELD_PSI_X + c) for c in range(3)]
    st.psi = psi
    vel = curl(psi, st.bf.psi_b, h, w.z_periodic)
    scale = max(np.abs(v).max() for v in vel)
    # the exported psi carries a rounding of 2^-49 of max |psi| per value, of
    # which v takes two differences over 2h; the velocity's own words 2^-48
    u = (4 * 2.0 ** -49 * max(np.abs(a).max() for a in psi) / (2 * h) + 2.0 ** -48 * scale) * 4
    got = []
    for c in range(3):
        d64 = sim.field(V.VSV_FIELD_VEL_X + c)
        d32 = sim.field(V.VSV_FIELD_VEL_X + c, dtype=np.float32)
        dev = sim.field(V.VSV_FIELD_VEL_X + c, torch.float64, on_device=True).cpu().numpy()
        # a destination that a kernel cannot write element by element
        raw = torch.zeros(nx * ny * nz * 8 + 4, dtype=torch.uint8, device="cuda")
        V.vsv_get_field(sim.g, V.VSV_FIELD_VEL_X + c, raw.data_ptr() + 4, V.VSV_DTYPE_F64, 1)
        odd = np.frombuffer(raw.cpu().numpy().tobytes()[4:], dtype=np.float64).reshape(d64.shape)
        assert np.array_equal(d64, dev) and np.array_equal(d64, odd)
        assert np.array_equal(d64.astype(np.float32), d32)
        assert np.max(np.abs(d64 - vel[c])) <= u
        got.append(d64)
    # stress and diagnostics of that velocity: differences over 2h, times eta
    g = velocity_gradient(got, st.bf.vel_b, h, w.z_periodic)
    e = [[g[i][j] + g[j][i] for j in range(3)] for i in range(3)]
    sig = w.eta * np.sqrt(e[0][1] ** 2 + e[1][2] ** 2 + e[0][2] ** 2)
    us = w.eta * 8 * 2.0 ** -44 * scale / h
    f64 = sim.field(V.VSV_FIELD_STRESS_T)
    assert np.max(np.abs(f64 - sig)) <= us + (2.0 ** -24 * sig.max() if prec == "mixed" else 0.0)
    prof = sim.stress_profile()
    ref = w.eta * e[0][1].mean(axis=(0, 2))
    assert np.max(np.abs(prof - ref)) <= w.eta * nx * nz * 2.0 ** -52 * scale / h + us
    d = sim.diagnostics()
    diss = 0.5 * w.eta * h ** 3 * sum(float(np.sum(x * x)) for r in e for x in r)
    # relative rounding of the differences against the strain that carries them
    assert abs(d["dissipation"] - diss) <= 1e-11 * diss
    assert abs(d["max_sigma_t"] - sig.max()) <= 1e-11 * sig.max()
    phi = sim.field(V.VSV_FIELD_PHI)
    wgt = 0.5 * (1.0 - phi)
    xs = [inputs.cell_coords(nx, h, False), inputs.cell_coords(ny, h, True),
          inputs.cell_coords(nz, h, not w.z_periodic)]
    for a, com in enumerate(d["com"]):
        s = [1, 1, 1]
        s[2 - a] = -1
        assert abs(com - np.sum(wgt * xs[a].reshape(s)) / np.sum(wgt)) <= 1e-11 * nx
    sim.close()
