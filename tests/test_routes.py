"""Which kernels the library launches, and what it does on a second device, on
the CPU: the library's object files linked against a CUDA runtime of the host
(tests/fake_cuda.cpp) that records launches and keeps each device's kernel
attributes apart."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2601_05031_gb300 import build, vsv
    build.build()
    out = str(tmp_path_factory.mktemp("fake") / "libvsv_host.so")
    objs = [os.path.join(build.OUT_DIR, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    inc = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include")
    # the runtime's symbols bind inside the library, whatever the process has loaded
    subprocess.run([shutil.which("g++"), "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic",
                    "-I", inc, os.path.join(HERE, "fake_cuda.cpp"), *objs, "-o", out, "-ldl",
                    "-lpthread", "-lrt"], check=True)
    lib = vsv.load(out)
    lib.fake_name.restype = C.c_char_p
    lib.fake_refuse.argtypes = lib.fake_fail.argtypes = [C.c_char_p]
    return lib


def _grid(lib, shape, prec):
    """A handle, and the workspace it lives in."""
    from paper_2601_05031_gb300 import vsv as V
    p = V.VSV_MIXED if prec == "mixed" else V.VSV_FP64
    need = lib.vsv_workspace_bytes(*shape, p)
    buf = np.zeros(need + 256, dtype=np.uint8)
    g = C.c_void_p()
    assert lib.vsv_create(C.byref(g), *shape, 1.0, p, (buf.ctypes.data + 255) // 256 * 256, need,
                          None) == V.VSV_OK
    return g, buf


def _solve(lib, shape, prec, periodic=(1, 0, 0), device=0, refuse=b"", cycles=1):
    """The status of one solve of `cycles` cycles and the kernels it launched."""
    from paper_2601_05031_gb300 import vsv as V
    nx, ny, nz = shape
    lib.fake_device(device)
    lib.fake_refuse(refuse)
    g, buf = _grid(lib, shape, prec)
    rhs, x = np.zeros(nx * ny * nz), np.zeros(nx * ny * nz)
    bc = V.vsv_bc((C.c_int * 3)(*periodic), 0.0)
    cyc, rr = C.c_int(), C.c_double()
    lib.fake_clear()
    st = lib.vsv_solve_poisson(g, rhs.ctypes.data, x.ctypes.data, V.VSV_DTYPE_F64, 1, C.byref(bc), 0.0,
                               cycles, C.byref(cyc), C.byref(rr))
    names = [lib.fake_name(i).decode() for i in range(lib.fake_count())]
    lib.vsv_destroy(g)
    lib.fake_refuse(b"")
    lib.fake_device(0)
    return st, names


def _count(names, part):
    return sum(part in n for n in names)


@pytest.mark.parametrize("shape", [(64, 32, 32), (36, 10, 12)])
def test_passes_opt_in_on_every_device(lib, shape):
    """The shared-memory limit of the two-sweep passes is an attribute of a
    kernel on one device: a second device's solve runs the same kernels."""
    from paper_2601_05031_gb300 import vsv as V
    for device in (0, 1, 0, 100):
        st, names = _solve(lib, shape, "mixed", device=device)
        assert st in (V.VSV_OK, V.VSV_ENOCONV) and _count(names, "k_pre_pass") > 0, device


@pytest.mark.parametrize("shape", [(128, 64, 128), (192, 96, 80)])
def test_tiled_kernels_opt_in_on_every_device(lib, shape):
    """So do the marching kernels of larger levels (tile-aligned and ragged)."""
    from paper_2601_05031_gb300 import vsv as V
    for device in (0, 1, 3):
        st, names = _solve(lib, shape, "mixed", device=device)
        assert st in (V.VSV_OK, V.VSV_ENOCONV), device
        for k in ("k_rbgs_fused", "k_defect_tiled", "k_restrict_tiled"):
            assert _count(names, k) > 0, (device, k, names)


def test_passes_refused_by_the_device_fall_back(lib):
    """A device that refuses the passes' limit gets the separate kernels."""
    from paper_2601_05031_gb300 import vsv as V
    st, names = _solve(lib, (64, 32, 32), "mixed", device=2, refuse=b"k_post_pass")
    assert st in (V.VSV_OK, V.VSV_ENOCONV)
    assert _count(names, "k_pre_pass") == 0 and _count(names, "k_post_pass") == 0
    assert _count(names, "k_rb_sweep") > 0


@pytest.mark.parametrize("offset", [0, 4])
def test_export_reports_the_launch_error_of_its_refresh(lib, offset):
    """mu of a replaced phi is formed by the export; a kernel of it that fails
    to launch is reported for any destination, also one that kernels cannot
    write in place."""
    from paper_2601_05031_gb300 import vsv as V
    g, buf = _grid(lib, (16, 8, 8), "mixed")
    fl, fe = V.vsv_flow_params(V.VSV_COUETTE, 0.0, -0.1, 0.1, 1.0, 0.0), V.vsv_fe_params(
        V.VSV_CAHN_HILLIARD, 1.0, 0.0, 1.0, 1.0, 0.0, 0.0, 0)
    assert lib.vsv_set_flow(g, C.byref(fl)) == V.VSV_OK
    assert lib.vsv_set_free_energy(g, C.byref(fe)) == V.VSV_OK
    phi, out = np.ones(1024), np.zeros(1026)
    assert lib.vsv_set_phi(g, phi.ctypes.data, V.VSV_DTYPE_F64, 0) in (V.VSV_OK, V.VSV_ENOCONV)
    assert lib.vsv_set_field(g, V.VSV_FIELD_PHI, phi.ctypes.data, V.VSV_DTYPE_F64, 1) == V.VSV_OK
    lib.fake_fail(b"k_mu")
    st = lib.vsv_get_field(g, V.VSV_FIELD_MU, out.ctypes.data + offset, V.VSV_DTYPE_F64, 1)
    lib.fake_fail(b"")
    lib.vsv_destroy(g)
    assert st == V.VSV_ECUDA


@pytest.mark.parametrize("shape,prec,kernel", [
    ((36, 30, 22), "mixed", "k_coarse_vcycle"),   # 18 x 15 x 11: no runs cover it, FP32
    ((44, 38, 34), "mixed", "k_coarse_vcycle"),
    ((36, 30, 22), "fp64", "k_coarse_solve"),     # FP64, up to 6,144 cells
    ((28, 28, 28), "fp64", "k_coarse_solve"),
    ((44, 38, 20), "fp64", "k_coarse_vcycle"),    # 22 x 19 x 10: runs of 5 planes
    ((28, 28, 20), "fp64", "k_coarse_vcycle"),
    ((44, 38, 34), "fp64", "k_rb_sweep"),         # 7,106 cells: sweeps on every SM
    ((52, 44, 28), "fp64", "k_rb_sweep"),
])
def test_kernel_of_a_lone_coarsest_level(lib, shape, prec, kernel):
    """A coarsest level below a level with kernels of its own: one CTA holds it
    in register runs; on the FP64 path, where no runs cover it, the one-CTA
    solve over shared memory takes it, or above its size launches per colour."""
    st, names = _solve(lib, shape, prec, cycles=2)
    for k in ("k_coarse_vcycle", "k_coarse_solve"):
        assert _count(names, k) == (2 if k == kernel else 0), (k, names)
    # two cycles: four smoothing sweeps of two colours on the level above, and 24
    # sweeps of the coarsest where it has launches of its own
    if prec == "fp64":
        assert _count(names, "k_rb_sweep") == 2 * (8 + (48 if kernel == "k_rb_sweep" else 0))


# kernel counts of one cycle: (pre-smoothing with, without the restriction; post-
# smoothing with, without the update; one-CTA cycle)
@pytest.mark.parametrize("shape,periodic,counts", [
    ((64, 32, 32), (1, 0, 0), (2, 0, 1, 1, 1)),      # 64 x 32 x 32, 32 x 16 x 16; the cycle from 1,024 cells
    ((128, 64, 16), (1, 0, 1), (2, 0, 1, 1, 1)),     # 2^17 cells: the pass restricts; the cycle from 2,048
    ((128, 48, 24), (1, 0, 0), (2, 1, 1, 2, 1)),     # above: the tiled restriction; a pass at 2,304 cells
    ((128, 64, 32), (1, 0, 0), (2, 1, 1, 2, 1)),     # 2^18 cells
    ((160, 64, 32), (1, 0, 0), (2, 0, 0, 2, 1)),     # above: fused sweeps on the finest level
    ((64, 32, 32), (0, 0, 0), (0, 0, 0, 0, 1)),      # walls in x: no passes
])
def test_passes_run_where_their_sizes_say(lib, shape, periodic, counts):
    st, names = _solve(lib, shape, "mixed", periodic=periodic)
    got = tuple(_count(names, k) for k in ("k_pre_passILb1", "k_pre_passILb0", "k_post_passILb1",
                                           "k_post_passILb0", "k_coarse_vcycleIf"))
    assert got == counts, names
