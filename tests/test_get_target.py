"""hrm_get into device memory: a kernel stores straight into the caller's planes only
where they are plain memory of the context's own device at an address of whole
doubles; anything else takes the copy, which also serves memory of another device.
The rule itself is tested on the CPU (there is one GPU to run on), the fields on
the GPU against the same call into host memory."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2208_04488_gb300 import problems as P

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
UNREGISTERED, HOST, DEVICE, MANAGED = 0, 1, 2, 3

HARNESS = """
#include "hrm_target.h"
extern "C" int target(long dst, int got, int type, int owner, long devptr, int device) {
  cudaPointerAttributes a{};
  a.type = (cudaMemoryType)type;
  a.device = owner;
  a.devicePointer = (void*)devptr;
  return hrm::kernel_target((const double*)dst, got != 0, a, device);
}
"""


@pytest.fixture(scope="module")
def target(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    d = tmp_path_factory.mktemp("target")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-fPIC", "-shared", "-I", inc, "-I", os.path.join(ROOT, "paper_2208_04488_gb300", "csrc"),
                    str(d / "h.cpp"), "-o", str(d / "h.so")], check=True)
    f = ctypes.CDLL(str(d / "h.so")).target
    f.argtypes = [ctypes.c_long, ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_long, ctypes.c_int]
    return f


@pytest.mark.parametrize("what,dst,got,kind,owner,device,direct", [
    ("own device", 0x1000, 1, DEVICE, 0, 0, 1),
    ("own device, not the first", 0x1008, 1, DEVICE, 3, 3, 1),
    ("another device", 0x1000, 1, DEVICE, 1, 0, 0),
    ("not whole doubles", 0x1004, 1, DEVICE, 0, 0, 0),
    ("pinned host memory", 0x1000, 1, HOST, 0, 0, 0),
    ("managed memory", 0x1000, 1, MANAGED, 0, 0, 0),
    ("memory CUDA does not know", 0x1000, 1, UNREGISTERED, 0, 0, 0),
    ("attributes refused", 0x1000, 0, DEVICE, 0, 0, 0)])
def test_which_memory_a_kernel_stores_to(target, what, dst, got, kind, owner, device, direct):
    assert target(dst, got, kind, owner, dst, device) == direct


@pytest.fixture(scope="module")
def hrm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2208_04488_gb300 import build, hrm as H
    build.build()
    return H


@pytest.mark.gpu
@pytest.mark.parametrize("pr", [P.shock_tube_1d_baseline(37), P.shock_bubble_2d(45, 21), P.dirichlet_box([11, 9]),
                                P.interface_3d(12)], ids=lambda p: p.name)
@pytest.mark.parametrize("offset", [0, 4], ids=["aligned", "half_a_double_off"])
def test_fields_into_device_memory(hrm, pr, offset):
    """Every field: as into host memory, nothing beyond its planes touched; with
    Dirichlet slices (other strides) and at an address of no whole double too."""
    import torch
    s = hrm.Solver.from_problem(pr, params=hrm.params_default(cfl=0.4, check=0))
    s.step(0.0, 2)
    for field in range(9):
        ref = s.get(field)
        buf = torch.full((ref.size + 2,), -7.0, dtype=torch.float64, device="cuda")
        st = hrm.lib().hrm_get(s.h, field, ctypes.c_void_p(buf.data_ptr() + 8 + offset), 1)
        assert st == hrm.HRM_OK
        torch.cuda.synchronize()
        raw = buf.cpu().numpy().view(np.uint8)
        got = raw[8 + offset:8 + offset + ref.nbytes].copy().view(np.float64).reshape(ref.shape)
        np.testing.assert_array_equal(got, ref)
        rest = np.delete(raw, np.arange(8 + offset, 8 + offset + ref.nbytes))
        assert (rest == np.delete(np.full(buf.numel(), -7.0).view(np.uint8), np.arange(8 + offset, 8 + offset + ref.nbytes))).all()
    s.close()
