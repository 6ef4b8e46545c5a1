"""An FP64 field set on the mixed path is held as (RN(d), RN(d - RN(d))) in
FP32 for every finite d: ties, zeros of both signs, magnitudes on both sides of
the range that the integer split covers, and a Poisson guess and rhs read from
and written to device memory directly and at odd offsets."""
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


def words(n, seed):
    r = np.random.default_rng(seed)
    b = r.integers(0, 1 << 63, n, dtype=np.uint64) << np.uint64(1) | r.integers(0, 2, n, dtype=np.uint64)
    e = r.choice([700, 948, 949, 950, 975, 1000, 1020, 1022, 1023, 1024, 1040, 1149, 1150], n)
    low = r.integers(0, 5, n)
    m = b & np.uint64(0xfffffffffffff)
    tail = np.uint64(0x1fffffff)
    m = np.where(low == 1, m & ~tail, m)                                 # exact in FP32
    m = np.where(low == 2, (m & ~tail) | np.uint64(0x10000000), m)       # ties
    m = np.where(low == 3, (m & ~tail) | np.uint64(0x10000001), m)       # just above
    m = np.where((e == 1150), m & np.uint64(0xbffffffffffff), m)         # below FLT_MAX
    d = ((b & np.uint64(1 << 63)) | (e.astype(np.uint64) << np.uint64(52)) | m).view(np.float64).copy()
    d[:: 7] = 0.0
    d[3:: 11] = -0.0
    return d


@pytest.mark.parametrize("dense", [False, True])
def test_split_and_merge_are_exactly_rounded(V, dense):
    import torch
    w = inputs.droplet_duct(nx=16, ny=12, nz=10, radius=3.5, dt=0.01)
    from paper_2601_05031_gb300.sim import Simulation
    sim = Simulation.from_workload(w, V.VSV_MIXED)
    sim.set_phi(w.phi0)
    n = 16 * 12 * 10
    d = words(n, 1)
    if dense:   # every word in the integer split's range
        d = np.where(np.abs(d) < 1e-20, 0.25, d)
    t = torch.from_numpy(d).cuda()
    fid = V.VSV_FIELD_PSI_PERT_X
    V.vsv_set_field(sim.g, fid, t.data_ptr(), V.VSV_DTYPE_F64, 1)
    got = sim.field(fid, np.float64, on_device=True).cpu().numpy().ravel()
    h = d.astype(np.float32).astype(np.float64)
    want = h + (d - h).astype(np.float32).astype(np.float64)
    np.testing.assert_array_equal(got, want)
    sim.close()


def test_poisson_in_place_on_device_words(V):
    import torch
    from paper_2601_05031_gb300.sim import Simulation
    nx, ny, nz = 32, 16, 10
    n = nx * ny * nz
    b = inputs.random_field((nz, ny, nx), seed=2)
    sim = Simulation(nx, ny, nz, 1.0, V.VSV_MIXED)
    want, _, _, _ = sim.solve_poisson(b, tol=0.0, max_cycles=2, check=False)
    for off in (0, 1):       # whole vectors, and words at an 8-byte offset
        buf = torch.full((2, n + 1), float("nan"), dtype=torch.float64, device="cuda")
        rhs, x = buf[0, off:off + n], buf[1, off:off + n]
        rhs.copy_(torch.from_numpy(b.ravel()))
        x.zero_()
        torch.cuda.synchronize()
        V.vsv_solve_poisson(sim.g, rhs.data_ptr(), x.data_ptr(), V.VSV_DTYPE_F64, 1,
                            (True, False, False), 0.0, 2, check=False)
        np.testing.assert_array_equal(x.cpu().numpy(), want.ravel())
        np.testing.assert_array_equal(rhs.cpu().numpy(), b.ravel())
    sim.close()
