"""The device helpers that every norm and every error check of the Krylov and Poisson
kernels goes through, by themselves: warp_sum_int and GridSums (csrc/common.cuh)
against exact sums, and the small exponential (small_expm_warp,
csrc/krylov_impl.cuh) against values from high-precision arithmetic.

Bounds.  warp_sum_int adds 32 K values as integers in units u = 2^(e - 56 + KB) with
2^e <= max |v| and KB = ceil(log2 K): half a unit a value, and one rounding; near
the ends of the exponent range K - 1 + 5 FP64 additions.  GridSums: three of these
(a value a lane, a value a warp, 8 values a lane).  The small exponential: 1e-14
of the largest entry; the last entry, which the error estimate is, to 1e-14 of
itself and 1e-17 (the terms cut from the series, 1e-24 each, times the growth of T_k
along the p + 1 coupled rows, k^(2p+2) / ((2p+1)!! (p+1)!) < 1e7 at k = 20).
"""
import ctypes
import math
import subprocess
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SRC = """
#include <cstring>
#include "krylov_impl.cuh"
using namespace etd;
template <int K>
__global__ void warps(int n, const double* v, double* out) {  // a block of one warp per row
  double x[K];
  for (int k = 0; k < K; ++k) x[k] = v[((size_t)blockIdx.x * K + k) * 32 + threadIdx.x];
  out[blockIdx.x * 32 + threadIdx.x] = warp_sum_int<K>(x);
}
extern "C" int probe_warps(int K, int n, const double* v, double* out) {
  if (K == 1) warps<1><<<n, 32>>>(n, v, out);
  else if (K == 3) warps<3><<<n, 32>>>(n, v, out);
  else warps<8><<<n, 32>>>(n, v, out);
  return (int)cudaDeviceSynchronize();
}
constexpr int REP = 3;
__global__ void __launch_bounds__(512, 1) grids(DevStatus* st, double* part, const double* v, double* out) {
  unsigned bar = 0;
  GridSums gs(part);
  const size_t gth = (size_t)gridDim.x * blockDim.x, i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (int r = 0; r < REP; ++r) {
    const double x[3] = {v[i], v[gth + i], (r + 1) * v[2 * gth + i]};
    double t[3];
    if (!gs.sum<3>(st, bar, x, t, 90)) break;
    if (threadIdx.x == blockDim.x - 1)
      for (int q = 0; q < 3; ++q) out[((size_t)r * gridDim.x + blockIdx.x) * 3 + q] = t[q];
  }
  barrier_done(st);
}
extern "C" int probe_blocks() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms < MAX_SUM_BLOCKS ? sms : MAX_SUM_BLOCKS;
}
extern "C" int probe_status_bytes() { return (int)sizeof(DevStatus); }
extern "C" int probe_part_doubles() { return 8 * MAX_BLOCKS; }
extern "C" int probe_grid(int nb, int nt, void* st, double* part, const double* v, double* out) {
  void* args[] = {&st, &part, &v, &out};
  cudaError_t e = cudaLaunchCooperativeKernel((void*)grids, nb, nt, args, 0, 0);
  return e != cudaSuccess ? (int)e : (int)cudaDeviceSynchronize();
}
__global__ void small(int m, int p, double tau, int indef, const double* al, const double* b, double* y) {
  __shared__ Ctl c;
  const int o = blockIdx.x * 64;
  for (int i = threadIdx.x; i < m; i += 32) {
    c.alpha[i] = al[o + i];
    if (i + 1 < m) c.low[i] = c.up[i + 1] = b[o + i];
  }
  __syncwarp();
  small_expm_warp(c, m, p, tau, indef != 0, c.yexp);
  for (int i = threadIdx.x; i < m; i += 32) y[o + i] = c.yexp[i];
}
extern "C" int probe_small(int n, int m, int p, double tau, int indef, const double* al, const double* b, double* y) {
  small<<<n, 32>>>(m, p, tau, indef, al, b, y);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_2209_15095_gb300 import build

    d = tmp_path_factory.mktemp("sums")
    (d / "p.cu").write_text(SRC)
    subprocess.run([build.nvcc()] + build.ARCH + build.CFLAGS + ["-shared", "-cudart", "shared", str(d / "p.cu"), "-o",
                                                                  str(d / "p.so")], check=True)
    lib = ctypes.CDLL(str(d / "p.so"))
    P, I, D = ctypes.c_void_p, ctypes.c_int, ctypes.c_double
    lib.probe_warps.argtypes = [I, I, P, P]
    lib.probe_grid.argtypes = [I, I, P, P, P, P]
    lib.probe_small.argtypes = [I, I, I, D, I, P, P, P]
    return lib


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _p(t):
    return t.data_ptr()


def _exact(v):
    return sum(map(Fraction, np.ravel(v).tolist()))


def _int_bound(v, n_sum):
    """Half a unit a value and the final rounding (v: the values of one sum)."""
    K = max(1, n_sum // 32)
    kb = int(math.ceil(math.log2(K)))
    top = float(np.max(np.abs(v)))
    return 0.5 * n_sum * 2.0 ** (math.frexp(top)[1] - 1 - 56 + kb) if top else 0.0


@pytest.mark.parametrize("K", [1, 3, 8])
def test_warp_sums(probe, K):
    rng = np.random.default_rng(21)
    n = 400
    rows = []
    for i in range(n):
        x = rng.standard_normal((K, 32))
        kind = i % 8
        if kind == 1:  # mixed magnitudes
            x *= 2.0 ** rng.integers(-80, 80, x.shape)
        elif kind == 2:  # cancelling
            f = x.ravel()
            f[1::2] = -f[::2] * (1 + 1e-13 * rng.standard_normal(f[::2].shape))
        elif kind == 3:  # all but one zero, signed zeros among them
            x = np.where(rng.random(x.shape) < 0.04, x, -0.0)
        elif kind == 4:  # the ends of the exponent range: FP64 additions
            x *= 2.0 ** (-1000 if i % 16 < 8 else 990)
        elif kind == 5:  # subnormal numbers alone
            x *= 2.0 ** -1040
        elif kind == 6:  # equal values at a power of 2, and just below
            x = np.full_like(x, 2.0 ** 17 if i % 16 < 8 else np.nextafter(2.0 ** 17, 0.0))
        elif kind == 7:
            x = np.abs(x) * 2.0 ** rng.integers(-300, 300)
        rows.append(x)
    v = np.array(rows)
    v[8, 0, 3] = np.inf
    v[16, 0, 3], v[16, K - 1, 7] = np.inf, -np.inf
    v[24, K - 1, 31] = np.nan
    v[32] = 0.0
    out = torch.empty(n * 32, dtype=torch.float64, device="cuda")
    assert probe.probe_warps(K, n, _p(_dev(v)), _p(out)) == 0
    got = out.cpu().numpy().reshape(n, 32)
    assert all(len({x.tobytes() for x in r}) == 1 for r in got)  # the same bits in every lane
    got = got[:, 0]
    assert got[8] == np.inf and np.isnan(got[16]) and np.isnan(got[24]) and got[32] == 0.0
    for i in range(n):
        if i in (8, 16, 24):
            continue
        ref = _exact(v[i])
        if i % 8 in (4, 5):
            bound = (K + 4) * 2.0 ** -53 * math.fsum(np.abs(v[i]).ravel()) + 2.0 ** -1074
        else:
            bound = _int_bound(v[i], 32 * K) + 2.0 ** -53 * abs(float(ref))
        assert abs(Fraction(got[i]) - ref) <= bound * (1 + 1e-12)


@pytest.mark.parametrize("nt", [128, 512])
@pytest.mark.parametrize("blocks", [1, 5, 0])
def test_grid_sums(probe, blocks, nt):
    nb = blocks or probe.probe_blocks()
    rng = np.random.default_rng(22)
    n = nb * nt
    v = np.stack([rng.standard_normal(n), rng.standard_normal(n) * 2.0 ** rng.integers(-60, 60, n), np.ones(n)])
    v[0, n // 2] = 1e9
    st = torch.zeros(probe.probe_status_bytes() // 8 + 1, dtype=torch.float64, device="cuda")
    part = torch.zeros(probe.probe_part_doubles(), dtype=torch.float64, device="cuda")
    out = torch.zeros(3 * nb * 3, dtype=torch.float64, device="cuda")
    dv = _dev(v)
    for _ in range(2):  # the second launch starts from the barrier that the first one left
        out.zero_()
        torch.cuda.synchronize()
        assert probe.probe_grid(nb, nt, _p(st), _p(part), _p(dv), _p(out)) == 0
        got = out.cpu().numpy().reshape(3, nb, 3)
        assert np.all(got == got[:, :1])  # every block has the same bits
        for q in range(3):
            for r in range(3):
                w = v[q] * (r + 1 if q == 2 else 1)
                # the largest value any stage meets is below sum |w|: units of a lane's,
                # a warp's and a block's sum, and a rounding each
                top = math.fsum(np.abs(w))
                bound = (n + 32 * nb) * 0.5 * 2.0 ** -56 * top + 256 * 0.5 * 2.0 ** -53 * top + 3 * 2.0 ** -53 * top
                assert abs(Fraction(got[r, 0, q]) - _exact(w)) <= bound
        assert np.all(got[:, 0, 2] == [n, 2 * n, 3 * n])


def _small_reference(mp, al, b, p, tau):
    """The first m entries of exp(K) e_{M-1} by its power series: 100 digits after the
    cancellation of terms up to e^|K|."""
    mp.mp.dps = 100 + int(0.5 * tau * (np.max(np.abs(al)) + 2 * np.max(b) + 2))
    m = len(al)
    M = m + p + 1
    t = mp.mpf(tau)
    d = [t * mp.mpf(x) for x in al] + [mp.mpf(0)] * (p + 1)
    o = [t * mp.mpf(x) for x in b]
    x = [mp.mpf(0)] * M
    x[M - 1] = mp.mpf(1)
    acc = list(x)
    k = 0
    big = 1
    while k < 6000:
        k += 1
        y = [d[r] * x[r] for r in range(M)]
        for r in range(m - 1):
            y[r] += o[r] * x[r + 1]
            y[r + 1] += o[r] * x[r]
        y[0] += x[m]
        for r in range(m, M - 1):
            y[r] += x[r + 1]
        x = [v / k for v in y]
        acc = [u + v for u, v in zip(acc, x)]
        big = max(abs(v) for v in x)
        if big < mp.mpf(10) ** -80:
            break
    assert big < mp.mpf(10) ** -80
    return np.array([float(v) for v in acc[:m]])


def _lanczos(rng, lo, hi, m):
    """alpha, beta of m Lanczos steps on a spectrum in [lo, hi] (full orthogonalisation)."""
    lam = np.linspace(lo, hi, 200)
    Q = np.zeros((200, m))
    q = rng.standard_normal(200)
    al, b = np.zeros(m), np.zeros(m)
    for j in range(m):
        Q[:, j] = q / np.linalg.norm(q)
        w = lam * Q[:, j]
        al[j] = Q[:, j] @ w
        for _ in range(2):
            w = w - Q[:, : j + 1] @ (Q[:, : j + 1].T @ w)
        b[j] = np.linalg.norm(w)
        q = w
    return al, b


@pytest.mark.parametrize("p", [0, 2, 3])
@pytest.mark.parametrize("m", [1, 5, 28, 29, 31, 60])
@pytest.mark.parametrize("rho,top", [(0.3, 0.0), (7.0, 0.0), (120.0, 0.0), (400.0, 0.0), (1600.0, 0.0), (60.0, 8.0)])
def test_small_exponential(probe, rho, top, m, p):
    mp = pytest.importorskip("mpmath")
    if m + p + 1 > 64:
        pytest.skip("m + p + 1 <= 64")
    al, b = _lanczos(np.random.default_rng(23), -rho, top, m)
    y = torch.zeros(64, dtype=torch.float64, device="cuda")
    pad = lambda a: _dev(np.concatenate([a, np.zeros(64 - m)]))  # noqa: E731
    da, db = pad(al), pad(b)
    torch.cuda.synchronize()
    assert probe.probe_small(1, m, p, 0.7, int(top > 0), _p(da), _p(db), _p(y)) == 0
    got = y.cpu().numpy()[:m]
    ref = _small_reference(mp, al, b, p, 0.7)
    assert np.max(np.abs(got - ref)) <= 1e-14 * np.max(np.abs(ref))
    assert abs(got[-1] - ref[-1]) <= 1e-14 * abs(ref[-1]) + 1e-17
