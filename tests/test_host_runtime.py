"""What the library's host code asks of the CUDA runtime, checked without a GPU:
the built host objects linked with a runtime of two devices that runs nothing
(fake_cudart.cpp)."""
import ctypes
import glob
import os
import shutil
import subprocess

import pytest

from paper_2503_08217_gb300 import binding
from paper_2503_08217_gb300 import build as libbuild

HERE = os.path.dirname(os.path.abspath(__file__))
HAVE_NVCC = shutil.which("nvcc") is not None or os.path.exists("/usr/local/cuda/bin/nvcc")
pytestmark = pytest.mark.skipif(not HAVE_NVCC, reason="nvcc is needed to build")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    libbuild.build()
    objs = [os.path.join(libbuild.BUILD, s.replace(".cu", ".o")) for s in libbuild.SOURCES]
    if not all(map(os.path.exists, objs)):
        libbuild.build(force=True)
    out = str(tmp_path_factory.mktemp("fake") / "libs3r_fake.so")
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(libbuild.nvcc())))
    inc = [f"-I{p}" for p in [os.path.join(cuda, "include"), *glob.glob(os.path.join(cuda, "targets/*/include"))]]
    # -Bsymbolic: the fake's functions, whatever runtime the process has loaded
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", *inc,
                    os.path.join(HERE, "fake_cudart.cpp"), *objs, "-o", out], check=True)
    L = ctypes.CDLL(out)
    L.s3r_last_error.restype = ctypes.c_char_p
    L.s3r_workspace_bytes.restype = L.fake_allocated.restype = ctypes.c_int64
    return L


def _workspace(L, device=0, **kw):
    cap = dict(max_gaussians=1000, max_splats=1000, max_duplicates=8000, max_views=2, max_instances=600,
               max_tiles=64, max_pixels=16384, max_rows=0)
    cap.update(kw)
    h = ctypes.c_void_p()
    assert L.s3r_workspace_create(ctypes.byref(binding.Capacity(**cap)), device, ctypes.byref(h)) == 0
    return h


def _step(L, ws, degree, n_inst):
    """Statuses of project, sort, forward and backward."""
    at = 0x10000
    sc = binding.Scene(n=1000, means=at, log_scales=at, quats=at, opacity_logits=at, sh=at, sh_degree=degree,
                       inst_offsets=at, n_inst=n_inst)
    poses = binding.Poses(quat=at, trans=at)
    cam = binding.Camera(width=64, height=64, fx=50.0, fy=50.0, cx=32.0, cy=32.0, near_z=0.2)
    f = ctypes.c_float
    p = ctypes.c_void_p
    st = [L.s3r_project(ws, ctypes.byref(sc), ctypes.byref(poses), ctypes.byref(cam), 1, f(0.0), p(at), None,
                        f(0.0), None),
          L.s3r_sort(ws, None), L.s3r_render_fwd(ws, p(at), p(at), None)]
    g = binding.Grads(means=at, log_scales=at, quats=at, opacity_logits=at, sh=at, inst_quat=at, inst_trans=at)
    st.append(L.s3r_render_bwd(ws, ctypes.byref(sc), ctypes.byref(poses), p(at), p(at), ctypes.byref(g), None))
    return st, L.s3r_last_error()


@pytest.mark.parametrize("degree", [0, 1, 2, 3])
@pytest.mark.parametrize("n_inst", [0, 600])
def test_one_thread_steps_on_two_devices(lib, degree, n_inst):
    """The rows of SH degree 3 need more shared memory than a function has by
    default, and its limit is a property of the function on one device."""
    spaces = [_workspace(lib, device) for device in (0, 1)]
    for device in (0, 1, 0):
        before = lib.fake_launches(device, b"13k_project_bwdI")   # mangled: the kernel, not its file
        st, message = _step(lib, spaces[device], degree, n_inst)
        assert st == [0, 0, 0, 0], (device, st, message)
        assert lib.fake_launches(device, b"13k_project_bwdI") == before + 1
    for ws in spaces:
        lib.s3r_workspace_destroy(ws)


# small image, 1080p view, seven-camera rig, and a row table larger than the pairs
@pytest.mark.parametrize("cap,most", [
    (dict(max_gaussians=22_000, max_splats=22_000, max_duplicates=1 << 21, max_views=1, max_instances=2,
          max_tiles=240, max_pixels=61_440), 41_404_064),
    (dict(max_gaussians=1_100_000, max_splats=1_100_000, max_duplicates=8_800_000, max_views=1, max_instances=20,
          max_tiles=8160, max_pixels=2_073_600), 424_125_164),
    (dict(max_gaussians=9_000_000, max_splats=18_000_000, max_duplicates=144_000_000, max_views=7, max_instances=80,
          max_tiles=57_600, max_pixels=13_000_000), 6_544_673_372),
    (dict(max_gaussians=300_000, max_splats=300_000, max_duplicates=3_000_000, max_views=2, max_instances=0,
          max_tiles=4000, max_pixels=1_000_000, max_rows=3_000_000), 136_828_636)], ids=["tiny", "mid", "rig", "rows"])
def test_workspaces_stay_within_what_four_byte_rows_took(lib, cap, most):
    """A workspace takes no more device memory than with the row table of four
    bytes a row, and s3r_workspace_bytes is what was allocated."""
    before = lib.fake_allocated()
    ws = _workspace(lib, **cap)
    taken = lib.s3r_workspace_bytes(ws)
    assert taken == lib.fake_allocated() - before
    assert taken <= most
    lib.s3r_workspace_destroy(ws)
