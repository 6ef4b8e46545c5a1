"""The in-plane stress over the range of its type and the precision of the stress
profile: both against the FP64 evaluation of the exported velocity."""
import math

import numpy as np
import pytest

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


def _state(V, shape, prec, flow, vs, eta, h=1.0):
    """A handle whose velocity is of size vs: base flow and a smooth psi'."""
    from paper_2601_05031_gb300.sim import Simulation
    nx, ny, nz = shape
    sim = Simulation(nx, ny, nz, h, V.VSV_MIXED if prec == "mixed" else V.VSV_FP64)
    if flow == "couette":
        V.vsv_set_flow(sim.g, V.VSV_COUETTE, 0.0, -0.3 * vs, 0.7 * vs, eta)
    else:
        V.vsv_set_flow(sim.g, V.VSV_POISEUILLE_DUCT, vs, 0.0, 0.0, eta)
    V.vsv_set_free_energy(sim.g, V.VSV_CAHN_HILLIARD)
    sp = sim.solver_params()
    sp.tol = 1.0   # the flow that is solved for here is replaced: it need not converge
    V.vsv_set_solver(sim.g, sp)
    sim.set_phi(np.ones(sim.shape))
    z, y, x = np.meshgrid(*[(np.arange(n) + 0.5) / n for n in (nz, ny, nx)], indexing="ij")
    for c in range(3):
        p = 0.2 * vs * h * nx * np.sin(2 * np.pi * (x + 0.1 * c)) * np.sin(np.pi * y) ** 2 * np.sin(
            np.pi * (z + 0.05 * c)) ** 2
        sim.set_field(V.VSV_FIELD_PSI_PERT_X + c, p)
    return sim


def _sheared(v, flow, vs, h, eta):
    """eta (d_a v_b + d_b v_a) for (xy, yz, xz) by central differences over 2h,
    no-slip wall values on the wall nodes, in FP64."""
    lo, hi = (-0.3 * vs, 0.7 * vs) if flow == "couette" else (0.0, 0.0)

    def d(a, axis, wall):
        if axis == 2 or (axis == 0 and flow == "couette"):
            return np.roll(a, -1, axis) - np.roll(a, 1, axis)
        w = [np.full_like(np.take(a, [0], axis), x) for x in wall]
        e = np.concatenate([w[0], a, w[1]], axis)
        n = a.shape[axis]
        return np.take(e, range(2, n + 2), axis) - np.take(e, range(n), axis)
    wx = (lo, hi)
    f = eta * (0.5 / h)
    xy = f * (d(v[0], 1, wx) + d(v[1], 2, None))
    yz = f * (d(v[1], 0, (0.0, 0.0)) + d(v[2], 1, (0.0, 0.0)))
    xz = f * (d(v[0], 0, (0.0, 0.0)) + d(v[2], 2, None))
    return xy, yz, xz


@pytest.mark.parametrize("vs,eta", [
    (1.0, 1.0), (1e-20, 1.0), (1e-23, 1e-2), (1e-6, 1e-15), (1e-20, 5e-4), (1e-3, 1e20), (1e22, 1.0),
    (1e25, 1e-3), (1e-32, 1e10), (1e18, 1e18), (1e20, 1e19), (1e-20, 1e-22)])
@pytest.mark.parametrize("shape,flow", [((24, 16, 12), "couette"), ((22, 10, 14), "duct")])
def test_stress_field_over_the_range_of_fp32(V, shape, flow, vs, eta):
    h = 0.7
    sim = _state(V, shape, "mixed", flow, vs, eta, h)
    v = [sim.field(V.VSV_FIELD_VEL_X + c) for c in range(3)]
    with np.errstate(over="ignore", under="ignore"):
        ref = np.sqrt(sum(s * s for s in _sheared(v, flow, vs, h, eta)))
        r32 = ref.astype(np.float32)
    got = sim.field(V.VSV_FIELD_STRESS_T, dtype=np.float32)
    sim.close()
    # the FP64 evaluation rounded once: half an ulp of FP32, and the two FP64
    # evaluations' difference (12 operations of 2^-53 on terms of which at most
    # 2^10 cancel)
    big = np.isinf(r32)
    assert np.array_equal(np.isinf(got), big)
    ulp = np.spacing(np.maximum(r32[~big], np.float32(2.0 ** -126))).astype(np.float64)
    assert np.all(np.abs(got[~big].astype(np.float64) - ref[~big]) <= 0.5 * ulp + 2.0 ** -39 * ref[~big])
    assert np.mean(got != r32) <= 1e-3
    assert np.any(got > 0)


@pytest.mark.parametrize("vs,eta", [(1.0, 1.0), (1e-170, 1e30), (1e160, 1e-20)])
def test_stress_field_over_the_range_of_fp64(V, vs, eta):
    h = 0.7
    sim = _state(V, (24, 16, 12), "fp64", "couette", vs, eta, h)
    v = [sim.field(V.VSV_FIELD_VEL_X + c) for c in range(3)]
    ref = np.sqrt(sum(s * s for s in _sheared(v, "couette", vs, h, eta)))
    got = sim.field(V.VSV_FIELD_STRESS_T)
    sim.close()
    # a dozen operations of 2^-53 on differences of values up to max |v|
    tol = 12 * 2.0 ** -53 * eta * 0.5 / h * max(np.abs(a).max() for a in v) * 4
    assert np.max(np.abs(got - ref)) <= tol and np.max(ref) > 100 * tol


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("shape,flow", [((64, 96, 48), "duct"), ((30, 34, 26), "couette"),
                                        ((128, 128, 96), "duct"), ((32, 8, 256), "duct")])
def test_stress_profile_as_a_sum_of_fp64_differences(V, shape, flow, prec):
    nx, ny, nz = shape
    sim = _state(V, shape, prec, flow, 1.0, 1.3)
    vx = sim.field(V.VSV_FIELD_VEL_X)
    prof = sim.stress_profile()
    sim.close()
    lo, hi = (-0.3, 0.7) if flow == "couette" else (0.0, 0.0)
    e = np.concatenate([np.full((nz, 1, nx), lo), vx, np.full((nz, 1, nx), hi)], axis=1)
    m = nx * nz
    for j in range(ny):
        # the mean of the periodic difference d_x v_y vanishes
        d = e[:, j + 2] - e[:, j]
        ref = 1.3 * math.fsum(d.ravel()) * 0.5 / m
        # a thread adds at most m / 256 differences, then come the block's and the
        # chunks' sums (fewer than 48 additions on any path), each to 2^-53, and
        # the rounding of a difference
        tol = (m / 256 + 48) * 2.0 ** -53 * 1.3 * 0.5 * np.mean(np.abs(d))
        assert abs(prof[j] - ref) <= tol, (j, prof[j], ref, tol)
