"""The integer-pipe FP64 arithmetic (hrm_soft64.cuh): products, quotients and
square roots must be the correctly rounded ones, bit for bit. On the CPU the
functions compile as host C++ and are compared with the machine's FP64
arithmetic for every error that the approximate reciprocals they start from may
have; on the GPU the probe entry point is compared with torch's."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
OPS = ["mul", "div", "sqrt"]

HARNESS = """
#include "hrm_soft64.cuh"
int hrm::soft::rcp_error = 0;
extern "C" void apply(int op, int err, long n, const double* a, const double* b, double* out) {
  hrm::soft::rcp_error = err;
  for (long i = 0; i < n; ++i)
    out[i] = op == 0 ? hrm::soft::mul(a[i], b[i]) : (op == 1 ? hrm::soft::div(a[i], b[i]) : hrm::soft::root(a[i]));
}
"""


def operands(op, n, seed):
    """Any bit patterns; moderate numbers; significands with few bits (exact results, ties of products); significands
    at the ends of the binade; operands whose result lies next to a rounding boundary; specials."""
    rng = np.random.default_rng(seed)
    anything = rng.integers(0, 2**64, size=(2, n), dtype=np.uint64).view(np.float64)
    mid = rng.standard_normal((2, n)) * 10.0 ** rng.uniform(-120, 120, (2, n))
    few = (rng.integers(1, 2**27, (2, n)) * 2.0 ** rng.integers(-60, 60, (2, n))).astype(np.float64)
    ends = (2.0 ** rng.integers(-50, 50, (2, n))) * (1.0 + rng.integers(-4, 5, (2, n)) * 2.0**-52)
    q, d = mid[0], np.where(mid[1] == 0, 1.0, mid[1])
    with np.errstate(all="ignore"):
        near = np.stack([q * d if op == "div" else (np.abs(q) ** 2 if op == "sqrt" else q), d])
    near[0] = np.nextafter(near[0], np.where(rng.random(n) < 0.5, np.inf, -np.inf))
    tiny = np.finfo(np.float64).tiny
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, tiny, -tiny, tiny / 8, 5e-324, 1.0, -1.0, 2.0, 1e308, -1e308,
                        np.nextafter(1.0, 0), np.nextafter(2.0, 0), 3.0, 1e-300])
    pairs = np.stack([np.repeat(special, special.size), np.tile(special, special.size)])
    return np.concatenate([anything, mid, few, ends, near, pairs], axis=1)


def expected(op, a, b):
    with np.errstate(all="ignore"):
        return a * b if op == "mul" else (a / b if op == "div" else np.sqrt(a))


def same(got, ref):
    return np.where(np.isnan(ref), np.isnan(got), got.view(np.uint64) == ref.view(np.uint64))


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("soft64")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-fPIC", "-shared", "-I",
                    os.path.join(ROOT, "paper_2208_04488_gb300", "csrc"), str(d / "h.cpp"), "-o", str(d / "h.so")], check=True)
    return ctypes.CDLL(str(d / "h.so"))


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("err", [-2, -1, 0, 1, 2])
def test_host_results_are_correctly_rounded(host, op, err):
    """err: units of 2^-24 on the reciprocal (mul has none)."""
    x = operands(op, 100_000, 11 + err)
    a, b = np.ascontiguousarray(x[0]), np.ascontiguousarray(x[1])
    out = np.empty_like(a)
    P = ctypes.c_void_p
    host.apply(OPS.index(op), err, ctypes.c_long(a.size), P(a.ctypes.data), P(b.ctypes.data), P(out.ctypes.data))
    ok = same(out, expected(op, a, b))
    assert ok.all(), [(a[i].hex(), b[i].hex(), out[i].hex()) for i in np.flatnonzero(~ok)[:3]]


@pytest.mark.gpu
@pytest.mark.parametrize("op", OPS)
def test_gpu_results_are_correctly_rounded(op):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2208_04488_gb300 import build, hrm
    build.build()
    x = operands(op, 1_000_000, 3)
    # every leading significand that the reciprocal is looked up for, in both parities of the exponent
    lead = (np.arange(2**24, dtype=np.uint64) << np.uint64(29)) + np.uint64(1022 << 52) + np.uint64(0x155)
    lead = lead.view(np.float64)
    x = np.concatenate([x, np.stack([np.roll(lead, 12345), lead] if op == "div" else [lead, np.roll(lead, 12345)])], axis=1)
    a, b = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in x)
    got = hrm.probe_soft64(OPS.index(op), a, b).cpu().numpy()
    assert same(got, expected(op, x[0], x[1])).all()
