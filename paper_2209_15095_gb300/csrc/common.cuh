// Shared device utilities: grid descriptor, node kinds, status flags, the
// bounded grid barrier, deterministic block/grid reductions, FP32
// error-free accumulation.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "int64math.cuh"

namespace etd {

constexpr int MAXD = 4;
constexpr int MAX_M = 61;           // largest Krylov basis (m + p + 1 <= 64)
constexpr int MAX_BLOCKS = 1024;    // partial-sum slots per reduction quantity
constexpr int MAX_SUM_BLOCKS = 256; // CTAs of a launch that uses GridSums

// Unsigned division of n < 2^31 by a divisor d >= 1 fixed at set-up, on the
// integer pipe: with s = ceil(log2 d) and m = floor(2^32 (2^s - d) / d) + 1,
// n / d = (umulhi(m, n) + n) >> s (the round-up method of Granlund &
// Montgomery 1994; the sum cannot overflow for n < 2^31).  A division by a
// runtime divisor otherwise goes through float conversions, which GB300
// issues at its FP64 rate.
struct FastDiv {
  unsigned m;
  int s;
  __host__ __device__ FastDiv() : m(1u), s(0) {}
  __host__ explicit FastDiv(unsigned d) : s(0) {
    while ((1ull << s) < (unsigned long long)d) ++s;
    m = (unsigned)(((1ull << 32) * ((1ull << s) - d)) / d + 1ull);
  }
  __device__ __forceinline__ unsigned div(unsigned n) const { return (__umulhi(m, n) + n) >> s; }
};

struct GridDev {
  int ndim;
  int n[MAXD];
  long long stride[MAXD];
  long long size;
  double lo[MAXD];
  double h;
  FastDiv sdiv[MAXD];  // by stride[d]
  // bit-plane geometry of the level-set work sets (rows along the last axis
  // padded to 32-bit words): by the words per row and by the row strides
  // stride[d] / n[ndim - 1] of the other axes
  FastDiv wdiv, rdiv[MAXD];
};

// Fills the FastDiv members of g from ndim, n and stride (host side).
inline void grid_divisors(GridDev& g) {
  const long long nx = g.n[g.ndim - 1];
  for (int d = 0; d < g.ndim; ++d) {
    g.sdiv[d] = FastDiv((unsigned)g.stride[d]);
    g.rdiv[d] = FastDiv((unsigned)(g.stride[d] / nx > 0 ? g.stride[d] / nx : 1));
  }
  g.wdiv = FastDiv((unsigned)((nx + 31) / 32));
}

// node class in the low two bits of a kind byte
enum : uint8_t { K_OUT = 0, K_GHOST = 1, K_COMP = 2 };

// device status word bits (DevStatus::err)
enum : int {
  ERRF_DOMAIN = 1,     // an inside node within 3 nodes of the box edge
  ERRF_TIMEOUT = 2,    // a bounded device wait gave up
  ERRF_KRYLOV = 4,     // tolerance not met at tau_min
  ERRF_NONFINITE = 8,  // NaN / Inf in a reduction
  ERRF_CAPACITY = 16,  // a list or trace outgrew its buffer
  ERRF_UNSUPPORTED = 32,  // boundary data at a case-3 face with N >= 3
};

struct DevStatus {
  int err;
  int nclamp;           // ghost weights clamped to [0, 1]
  int timeout_site;
  int pad;
  double gersh[2];      // Gershgorin bound of h^2 C per species (max row sum of |h^2 C|)
  unsigned int barrier; // grid-barrier arrival counter (0 between launches, see barrier_done)
  unsigned int done;    // CTAs of the running launch that have ended
  int negb[2];          // per species: the beta field has a negative value
  unsigned long long wait_ns;  // limit of every device wait in ns (0: BARRIER_LIMIT_NS)
};

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void red_release_add_u32(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Grid-wide barrier for a cooperative launch: a monotonically increasing
// arrival counter (0 at the launch, see barrier_done).  Barrier number `k`
// (1-based, identical in every CTA) completes when the counter reaches
// k * gridDim.x.  Ordering: __syncthreads orders the CTA's accesses before
// thread 0's gpu-scope release add; the waiting thread's gpu-scope acquire
// load and the following __syncthreads order them before every later access
// of its CTA.  Every wait is bounded: from the first unsuccessful poll, the
// clock and the status word are checked every 16 polls (every poll when the
// limit is below 1 ms); after st->wait_ns (default BARRIER_LIMIT_NS, ~1 s)
// the status word gets ERRF_TIMEOUT and the call returns false, after which
// the kernel must return.  A CTA that sees another CTA's ERRF_TIMEOUT stops
// waiting too, so every CTA returns.
constexpr unsigned long long BARRIER_LIMIT_NS = 1000000000ull;
constexpr unsigned long long BARRIER_SHORT_NS = 1000000ull;

__device__ __forceinline__ bool grid_barrier(DevStatus* st, unsigned& k, int site) {
  __shared__ int s_ok;
  ++k;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    red_release_add_u32(&st->barrier, 1u);
    // the limit's load is issued before the first poll and has returned by
    // the time that poll's result is known: it adds no latency
    unsigned long long w = *((volatile unsigned long long*)&st->wait_ns);
    const unsigned target = k * gridDim.x;
    unsigned long long t0 = 0;
    unsigned polls = 0;
    while (ld_acquire_u32(&st->barrier) < target) {
      // an opaque update of w: its tests stay after the poll instead of
      // being hoisted above the first one (which would wait for the load)
      asm volatile("" : "+l"(w));
      if (polls == 0) t0 = global_ns();
      ++polls;
      const bool short_limit = w != 0ull && w < BARRIER_SHORT_NS;
      if (short_limit || (polls & 15u) == 0u) {
        if (global_ns() - t0 >= (w != 0ull ? w : BARRIER_LIMIT_NS)) {
          atomicOr(&st->err, ERRF_TIMEOUT);
          atomicExch(&st->timeout_site, site);
          ok = 0;
          break;
        }
        // another CTA gave up: stop waiting for it
        if (*((volatile int*)&st->err) & ERRF_TIMEOUT) { ok = 0; break; }
      }
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// Last action of every CTA of a cooperative kernel, whatever way it ends: the
// last CTA to end puts the arrival counter back to 0 for the next launch (a
// memset before every launch takes 2 to 3 us of the stream's time).  A CTA that
// ends has polled the counter after its own last arrival, so no arrival is
// still on its way.
__device__ __forceinline__ void barrier_done(DevStatus* st) {
  __syncthreads();
  if (threadIdx.x == 0 && atomicAdd(&st->done, 1u) == gridDim.x - 1u) {
    st->barrier = 0u;
    st->done = 0u;
  }
}

// barrier_done at every return of a kernel
struct BarrierDone {
  DevStatus* st;
  __device__ __forceinline__ ~BarrierDone() { barrier_done(st); }
};

// Index of this thread in the node loops: 32-index chunks dealt round-robin
// over the CTAs (chunk j to warp j / gridDim of CTA j % gridDim), a
// bijection onto [0, gridDim * blockDim).  A problem smaller than the grid
// then spreads over every SM instead of filling the first CTAs, whose FP64
// pipes are shared by all of their warps.
__device__ __forceinline__ long long dealt_tid() {
  return (long long)(threadIdx.x & 31) + 32ll * ((long long)blockIdx.x + (long long)gridDim.x * (threadIdx.x >> 5));
}

// ---------------------------------------------------------------- reductions
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum of K values per lane over the warp, the same bits in every lane.  The
// values are aligned to the largest exponent as 64-bit integers (rounded to
// nearest at 2^-(57 - ceil(log2 K)) of the largest, below the rounding of an FP64
// addition for K <= 8) and added exactly by three integer warp reductions: a
// dependent FP64 addition takes about 70 cycles here and a tree of five with
// their shuffles 500, this about 130.  Infinities, NaNs and sums near the ends of
// the exponent range take FP64 additions.
template <int K>
__device__ __forceinline__ double warp_sum_int(const double (&v)[K]) {
  constexpr int KB = K == 1 ? 0 : K == 2 ? 1 : K <= 4 ? 2 : 3;
  static_assert(K <= 8, "too many values");
  unsigned e = 0;
#pragma unroll
  for (int k = 0; k < K; ++k) e = max(e, ((unsigned)__double2hiint(v[k]) >> 20) & 0x7ffu);
  e = __reduce_max_sync(0xffffffffu, e);
  if (e == 0u || e - 200u > 1600u) {
    double x = 0.0;
#pragma unroll
    for (int k = 0; k < K; ++k) x += v[k];
    return e == 0u && !__any_sync(0xffffffffu, x != 0.0) ? 0.0 : warp_sum(x);
  }
  i64 f = 0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const u64 b = (u64)__double_as_longlong(v[k]);
    const int ek = (int)((b >> 52) & 0x7ff);
    const int r = (int)e - ek + 1;  // >= 1: one more bit for the rounding
    u64 m = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << (5 - KB);
    m = ek == 0 || r > 62 ? 0ull : ((m >> (r - 1)) + 1ull) >> 1;
    const i64 sg = (i64)b >> 63;
    f += ((i64)m ^ sg) - sg;
  }
  // |f| < 2^57 in all: 22 + 22 + 14 bits
  const int s0 = __reduce_add_sync(0xffffffffu, (int)(f & 0x3fffff));
  const int s1 = __reduce_add_sync(0xffffffffu, (int)((f >> 22) & 0x3fffff));
  const int s2 = __reduce_add_sync(0xffffffffu, (int)(f >> 44));
  const i64 S = ((i64)s2 << 44) + ((i64)s1 << 22) + (i64)s0;
  // units 2^(e - 1023 - 52 - 5 + KB + 1)
  const double d = (double)S;
  return S == 0 ? 0.0 : __longlong_as_double(__double_as_longlong(d) + ((i64)((int)e - 1023 - 56 + KB) << 52));
}

// Sums over the grid of NQ per-thread values, with a grid barrier: warp sums,
// the CTA's sum by warp q for quantity q, the barrier, and all CTAs' sums by
// warp q again, every CTA alike (the same bits everywhere).  Two sets of sums
// alternate: between two that use the same set every CTA has passed a barrier
// after reading it.  Returns false if the kernel must stop.
struct GridSums {
  double* part;  // 2 sets x 4 quantities x MAX_BLOCKS
  int no;
  __device__ __forceinline__ explicit GridSums(double* p) : part(p), no(0) {}
  template <int NQ>
  __device__ __forceinline__ bool sum(DevStatus* st, unsigned& bar, const double (&v)[NQ], double (&out)[NQ],
                                      int site);
};

template <int NQ>
__device__ __forceinline__ bool GridSums::sum(DevStatus* st, unsigned& bar, const double (&v)[NQ], double (&out)[NQ],
                                              int site) {
  __shared__ double s_w[NQ][32], s_out[NQ];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  double* const w = part + (size_t)(no & 1) * (4 * MAX_BLOCKS) + wid * MAX_BLOCKS;
  ++no;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const double one[1] = {v[q]};
    const double x = warp_sum_int<1>(one);
    if (lane == 0) s_w[q][wid] = x;
  }
  __syncthreads();
  if (wid < NQ) {
    const double one[1] = {lane < nw ? s_w[wid][lane] : 0.0};
    const double x = warp_sum_int<1>(one);
    if (lane == 0) w[blockIdx.x] = x;
  }
  if (!grid_barrier(st, bar, site)) return false;
  if (wid < NQ) {
    constexpr int K = MAX_SUM_BLOCKS / 32;
    double val[K];
#pragma unroll
    for (int k = 0; k < K; ++k) val[k] = 32 * k + lane < (int)gridDim.x ? __ldcg(w + 32 * k + lane) : 0.0;
    const double t = warp_sum_int<K>(val);
    if (lane == 0) s_out[wid] = t;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NQ; ++q) out[q] = s_out[q];
  return true;
}

// Exact widening to FP64.  For a float, normal values are widened on the
// integer pipe (rebias the exponent, shift the mantissa): the hardware
// conversion is an FP64-pipe instruction, which costs as much as an FMA.
// Zero, subnormal, infinite and NaN values take the hardware conversion.
__device__ __forceinline__ double to_f64(double x) { return x; }
__device__ __forceinline__ double to_f64(float x) {
  const unsigned f = __float_as_uint(x);
  const unsigned e = (f >> 23) & 0xffu;
  if (e - 1u < 254u) {
    const unsigned hi = (f & 0x80000000u) | ((e + 896u) << 20) | ((f & 0x7fffffu) >> 3);
    const unsigned lo = (f & 7u) << 29;
    return __hiloint2double((int)hi, (int)lo);
  }
  return (double)x;
}

// Rounding of an FP64 value to FP32, to nearest with ties to even (IEEE
// 754), on the integer pipe where the result is a normal float: the FP32
// exponent is the FP64 one rebiased (1023 -> 127), the 23 mantissa bits are
// the top of the 52, and the 29 bits dropped decide the rounding (above
// half: up; exactly half: up when the kept mantissa is odd).  A carry out
// of the mantissa increments the exponent, and one out of the largest
// exponent gives the infinity bit pattern, as the rounding rule does.
// Results that would be subnormal, zero, infinite or NaN take the hardware
// conversion (an FP64-pipe instruction, as costly as an FMA on this GPU).
__device__ __forceinline__ float to_f32_rn(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned ex = (hi >> 20) & 0x7ffu;
  if (ex - 897u < 254u) {
    const unsigned m = ((hi & 0xfffffu) << 3) | (lo >> 29);
    const unsigned r = lo & 0x1fffffffu;
    const unsigned up = (r > 0x10000000u || (r == 0x10000000u && (m & 1u))) ? 1u : 0u;
    return __uint_as_float((hi & 0x80000000u) | (((ex - 896u) << 23) + m + up));
  }
  return (float)x;
}

// FP32 error-free accumulation of products (TwoProduct via fma + TwoSum,
// Ogita, Rump & Oishi 2005): s + c carries the sum to about twice single
// precision.  Intrinsics keep the compiler from contracting or reassociating.
struct Dot2f {
  float s, c;
  __device__ __forceinline__ Dot2f() : s(0.f), c(0.f) {}
  __device__ __forceinline__ void add(float a, float b) {
    float p = __fmul_rn(a, b);
    float pe = __fmaf_rn(a, b, -p);
    float t = __fadd_rn(s, p);
    float z = __fsub_rn(t, s);
    float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));
    s = t;
    c = __fadd_rn(c, __fadd_rn(e, pe));
  }
  // (a warp without points issues no FP64)
  __device__ __forceinline__ double value() const { return s == 0.f && c == 0.f ? 0.0 : to_f64(s) + to_f64(c); }
};

template <typename T>
struct Acc;
template <>
struct Acc<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double a, double b) { s = fma(a, b, s); }
  __device__ __forceinline__ double value() const { return s; }
};
template <>
struct Acc<float> {
  Dot2f d;
  __device__ __forceinline__ void add(float a, float b) { d.add(a, b); }
  __device__ __forceinline__ double value() const { return d.value(); }
};

}  // namespace etd
