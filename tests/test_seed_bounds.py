"""The single-precision seeds of the integer root and reciprocal (csrc/int64math.cuh,
csrc/weno_int.cuh).  Their exponent is dropped, so a seed below 1 or at 2 must
not get through: the seeds' documented errors allow both.

CPU: the host build with the root's seed moved by a unit or two, at arguments
whose true seed is 1 or 2.  With |e| < 2^-21 the series' next term, 5/16 e^3,
stays below 2^-64, so the bounds are those of the unmoved build.
GPU: the hardware's seeds at the ends of the argument range, the same bounds
against extended precision.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2209_15095_gb300", "csrc")
HOST = """
#include <math.h>
static int g_ulps = 0;
static float moved(float x) {
  for (int i = 0; i < (g_ulps < 0 ? -g_ulps : g_ulps); ++i) x = nextafterf(x, g_ulps < 0 ? 0.0f : 4.0f);
  return x;
}
#define sqrtf(x) moved(sqrtf(x))
#include "weno_int.cuh"
extern "C" void set_ulps(int n) { g_ulps = n; }
extern "C" void roots(int n, const double* a, double* s, double* r) {
  for (int i = 0; i < n; ++i) etd::root_pair(a[i], s[i], r[i]);
}
extern "C" unsigned seed(float r) { return etd::seed_bits(r); }
"""
DEVICE = """
#include "weno_int.cuh"
__global__ void k(int n, const double* a, double* s, double* r, const unsigned long long* w, unsigned long long* q) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    etd::root_pair(a[i], s[i], r[i]);
    q[i] = etd::recip_u(w[i]);
  }
}
extern "C" int probe(int n, const double* a, double* s, double* r, const unsigned long long* w, unsigned long long* q) {
  k<<<64, 256>>>(n, a, s, r, w, q);
  return (int)cudaDeviceSynchronize();
}
"""


def _ends():
    """Arguments next to powers of 2: the mantissa's leading bits all ones, or just above the lower end."""
    m = np.concatenate([1.0 + np.arange(64) * 2.0 ** -52, 2.0 - np.arange(1, 65) * 2.0 ** -52,
                        1.0 + np.arange(64) * 2.0 ** -24, 2.0 - np.arange(1, 65) * 2.0 ** -24])
    return np.concatenate([np.ldexp(m, e) for e in (-1022, -501, -2, -1, 0, 1, 7, 500, 1022)])


def _check_roots(a, s, r):
    ref = np.sqrt(a.astype(np.longdouble))
    assert np.max(np.abs(s / ref - 1)) <= 2.0 ** -52.9
    assert np.max(np.abs(r * ref - 1)) <= 2.0 ** -52.9


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("seed")
    (d / "s.cpp").write_text(HOST)
    subprocess.run([cxx, "-O2", "-shared", "-fPIC", "-I" + CSRC, str(d / "s.cpp"), "-o", str(d / "s.so")], check=True)
    lib = ctypes.CDLL(str(d / "s.so"))
    lib.seed.argtypes, lib.seed.restype = [ctypes.c_float], ctypes.c_uint
    return lib


@pytest.mark.parametrize("ulps", [-2, -1, 0, 1, 2])
def test_moved_root_seed(host, ulps):
    a = _ends()
    s, r = np.empty_like(a), np.empty_like(a)
    host.set_ulps(ulps)
    host.roots(a.size, *(x.ctypes.data_as(ctypes.c_void_p) for x in (a, s, r)))
    host.set_ulps(0)
    _check_roots(a, s, r)


def test_seed_ends(host):
    one = np.float32(1)
    assert host.seed(float(np.nextafter(one, np.float32(0)))) == host.seed(1.0) == 1 << 31
    assert host.seed(float(np.float32(1.5))) == 3 << 30
    top = host.seed(2.0)
    assert top == host.seed(float(np.nextafter(np.float32(2), np.float32(3)))) and top >= (1 << 32) - (1 << 10)


@pytest.mark.gpu
def test_hardware_seeds(tmp_path):
    import torch

    from paper_2209_15095_gb300 import build

    (tmp_path / "p.cu").write_text(DEVICE)
    so = str(tmp_path / "p.so")
    subprocess.run([build.nvcc()] + build.ARCH + build.CFLAGS + ["-shared", "-cudart", "shared", str(tmp_path / "p.cu"),
                                                                  "-o", so], check=True)
    a = _ends()
    w = np.concatenate([(1 << 62) + np.arange(a.size // 4, dtype=np.int64), (1 << 62) + (np.arange(a.size // 4) << 38),
                        (1 << 63) - 1 - np.arange(a.size // 4, dtype=np.int64),
                        (1 << 63) - 1 - (np.arange(a.size // 4) << 38)]).astype(np.uint64)
    assert w.size == a.size
    da = torch.tensor(a, device="cuda")
    ds, dr = torch.empty_like(da), torch.empty_like(da)
    dw = torch.tensor(w.astype(np.int64), device="cuda")
    dq = torch.empty_like(dw)
    torch.cuda.synchronize()
    p = [ctypes.c_void_p(t.data_ptr()) for t in (da, ds, dr, dw, dq)]
    assert ctypes.CDLL(so).probe(a.size, *p) == 0
    _check_roots(a, ds.cpu().numpy(), dr.cpu().numpy())
    q = dq.cpu().numpy().astype(np.uint64)
    for wi, qi in zip(w.tolist(), q.tolist()):
        # 2^126 / w to 2^-58 of itself
        assert abs(qi * wi - (1 << 126)) <= 1 << 68
