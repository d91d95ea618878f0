// Embedded-boundary Poisson solve (Sec. 2: div(beta grad u) = f with Dirichlet
// data, interior ghost points; Sec. 4.1 applies it to a virus-shaped domain).
//
// At the computational points the discrete problem is C u + b = f, with C the
// matrix-free EB operator (the stencil of the Krylov kernel with dt = 1) and
// b the boundary-data term of the ghost values (per point, the face slots'
// coefficient times the boundary value).  C is symmetric negative definite
// (Sec. 2), so the kernel runs conjugate gradients on A = -C, A u = b - f,
// FP64, as one persistent cooperative kernel.  Up to PS_FUSED_PER points per thread
// an iteration has two grid barriers: the new search direction p = r + beta p_old
// is formed at the point and its 2N neighbours by the pass that applies A to it
// (r and p on the grid, p in two alternating arrays) instead of in a pass of
// its own with a barrier before the stencil reads it, as larger problems do (r
// compact); the last pass updates x and r.  They differ by rounding at most.  Sums
// are deterministic (every CTA forms them alike), so every CTA takes the same
// stopping decision; the iteration's scalars come from one thread (an FP64
// root and two divisions in every warp took an SM 6 us per iteration).
// Problems of at most one point per thread keep the point's index, diagonal
// and face coefficients in registers.  Measured on the virus domain at 321^2
// (28k points, 780 iterations): 14.4 -> 7.5 us per iteration; on a ball of 1.37M
// points 56.1 -> 51.4 (89.7 -> 85.8 with a node field).
#include "common.cuh"
#include "kernels.cuh"

namespace etd {

constexpr int PS_NT = 512;
// Points per thread up to which the search direction is formed at the stencil's points.
// Above, its 2 (2N + 1) loads and 2N + 1 FP64 FMAs a point cost more than a pass and
// a barrier: us per iteration with it / with a pass, constant beta: 3D 2.8 points a
// thread 15.9 / 16.0, 4.5 20.7 / 19.2, 17.5 62.2 / 51.4, 2D 2.4 13.1 / 14.5, 4.9 18.8 /
// 18.4; node field (the means cost more than either): 3D 2.8 18.5 / 20.3, 4.5 26.5 /
// 26.5, 17.5 93.2 / 85.8, 2D 4.9 22.9 / 23.8, 8.1 34.8 / 35.0.
template <int N, bool NODE>
constexpr int PS_FUSED_PER = N == 2 ? (NODE ? 8 : 4) : NODE ? 5 : 3;

// A computational point of the stencil: grid index (-1: none), diagonal and,
// with a node field (NODE), face coefficients.  NODE is a template argument: a
// constant beta's kernel would issue the face means' FP64 instructions predicated
// off, which costs their slots all the same.
template <int N, bool NODE>
struct PsPoint {
  long long p;
  double D, f[NODE ? 2 * N : 1];
};
template <int N, bool NODE>
__device__ __forceinline__ PsPoint<N, NODE> ps_point(const SpeciesDev<double>& S, const GridDev& g, long long k,
                                                     int ncomp) {
  PsPoint<N, NODE> o;
  o.p = -1;
  if (k >= ncomp) return o;
  o.p = __ldg(S.idx + k);
  o.D = __ldg(S.diag + k);
  if constexpr (NODE) {
    const double* const bf = S.beta_field;
    const double bp = __ldg(bf + o.p);
#pragma unroll
    for (int d = 0; d < N; ++d) {
      o.f[2 * d] = 0.5 * (bp + __ldg(bf + o.p - g.stride[d]));
      o.f[2 * d + 1] = 0.5 * (bp + __ldg(bf + o.p + g.stride[d]));
    }
  }
  return o;
}

// (C v)_p for v = val(grid index), with the value at the point itself
template <int N, bool NODE, typename Val>
__device__ __forceinline__ double cstencil(const PsPoint<N, NODE>& o, const GridDev& g, double cfac, double vp,
                                           double bc, Val val) {
  double s = -0.0;  // x + (-0) == x: the first add is free
  if constexpr (NODE) {
#pragma unroll
    for (int d = 0; d < N; ++d) {
      s += o.f[2 * d] * val(o.p - g.stride[d]);
      s += o.f[2 * d + 1] * val(o.p + g.stride[d]);
    }
    return cfac * (s - o.D * vp);
  } else {
#pragma unroll
    for (int d = 0; d < N; ++d) s += val(o.p - g.stride[d]) + val(o.p + g.stride[d]);
    return cfac * (bc * s - o.D * vp);
  }
}

template <int N, bool NODE>
__device__ __forceinline__ void poisson_body(const PoissonArgs& a) {
  const SpeciesDev<double>& S = a.S;
  const GridDev& g = a.g;
  const int ncomp = *S.ncomp;
  const long long gtid = dealt_tid();
  const long long gth = (long long)gridDim.x * blockDim.x;
  const double cfac = a.cfac;
  constexpr int SL = 2 * N * (N == 2 ? 2 : 1);
  unsigned bar = 0;
  GridSums gs(a.part);
  double* const x = S.Yc;             // compact: iterate
  double* const q = (double*)S.V2c;   // compact: A p
  const bool fused = ncomp <= PS_FUSED_PER<N, NODE> * gth;
  double* const r = (double*)(fused ? S.Z[0] : S.V1c);  // residual: grid (zero off the set), or compact
  double* const P[2] = {(double*)S.Yg, (double*)S.W1g};  // grid: search direction (zero off the set)
  __shared__ double s_alpha, s_beta, s_rr, s_stop, s_stop2;
  __shared__ int s_state;  // 0: go on, 1: converged, 2: stop
  const PsPoint<N, NODE> own = ps_point<N, NODE>(S, g, gtid, ncomp);
  // x_0 from the caller's u; P[1] holds x_0 to apply C to it
  for (long long k = gtid; k < ncomp; k += gth) {
    const long long p = __ldg(S.idx + k);
    const double v = a.u[p];
    x[k] = v;
    P[1][p] = v;
  }
  if (!grid_barrier(a.st, bar, 70)) return;
  // r_0 = (b - f) - A x_0 = (b - f) + C x_0;  |r_0|^2, |b - f|^2
  {
    double rr = 0.0, bb = 0.0;
    for (long long k = gtid; k < ncomp; k += gth) {
      const PsPoint<N, NODE> o = k == gtid ? own : ps_point<N, NODE>(S, g, k, ncomp);
      double rhs = -a.f[o.p];
      if (S.bco && S.bval) {
#pragma unroll
        for (int i = 0; i < SL; ++i) {
          const double cf = S.bco[k * SL + i];
          if (cf != 0.0) rhs = fma(cf, S.bval[k * SL + i], rhs);
        }
      }
      const double* const X = P[1];
      const double cx = cstencil<N, NODE>(o, g, cfac, __ldcg(X + o.p), S.beta_c, [&](long long i) { return __ldcg(X + i); });
      const double rk = rhs + cx;
      r[fused ? o.p : k] = rk;
      rr = fma(rk, rk, rr);
      bb = fma(rhs, rhs, bb);
    }
    const double v[2] = {rr, bb};
    double tot[2];
    if (!gs.sum<2>(a.st, bar, v, tot, 71)) return;
    if (threadIdx.x == 0) {
      const double bnorm = sqrt(tot[1]);
      s_stop = a.tol * (bnorm > 0.0 ? bnorm : 1.0);
      s_stop2 = 1.0000001 * s_stop * s_stop;
      s_rr = tot[0];
      s_beta = 0.0;
      s_state = sqrt(tot[0]) <= s_stop ? 1 : 0;
      if (blockIdx.x == 0) a.out[1] = bnorm;
    }
    __syncthreads();
  }
  int it = 0;
  while (s_state == 0 && it < a.max_iter) {
    // p = r + beta p_old, q = A p, <p, q>
    const double* const Po = P[(it & 1) ^ 1];
    double* const Pn = P[fused ? it & 1 : 0];
    const double beta = s_beta;
    const bool first = it == 0;
    double pq = 0.0, p0 = 0.0, q0 = 0.0;
    if (fused) {
      const auto dir = [&](long long i) {
        const double ri = __ldcg(r + i);
        return first ? ri : fma(beta, __ldcg(Po + i), ri);
      };
      for (long long k = gtid; k < ncomp; k += gth) {
        const PsPoint<N, NODE> o = k == gtid ? own : ps_point<N, NODE>(S, g, k, ncomp);
        const double pk = dir(o.p);
        const double qk = -cstencil<N, NODE>(o, g, cfac, pk, S.beta_c, dir);
        Pn[o.p] = pk;
        if (k == gtid) {
          p0 = pk;
          q0 = qk;
        } else {
          q[k] = qk;
        }
        pq = fma(pk, qk, pq);
      }
    } else {
      for (long long k = gtid; k < ncomp; k += gth) {
        const long long p = __ldg(S.idx + k);
        Pn[p] = first ? r[k] : fma(beta, __ldcg(Pn + p), r[k]);
      }
      if (!grid_barrier(a.st, bar, 75)) return;
      for (long long k = gtid; k < ncomp; k += gth) {
        const PsPoint<N, NODE> o = ps_point<N, NODE>(S, g, k, ncomp);
        const double pk = __ldcg(Pn + o.p);
        const double qk = -cstencil<N, NODE>(o, g, cfac, pk, S.beta_c, [&](long long i) { return __ldcg(Pn + i); });
        q[k] = qk;
        pq = fma(pk, qk, pq);
      }
    }
    {
      const double v[1] = {pq};
      double tot[1];
      if (!gs.sum<1>(a.st, bar, v, tot, 73)) return;
      if (threadIdx.x == 0) {
        s_alpha = s_rr / tot[0];
        if (!(tot[0] > 0.0) || !isfinite(tot[0])) {  // A is positive definite: breakdown only on bad data
          atomicOr(&a.st->err, ERRF_NONFINITE);
          s_state = 2;
        }
      }
      __syncthreads();
      if (s_state == 2) return;
    }
    // x += alpha p, r -= alpha q, |r|^2
    const double alpha = s_alpha;
    double rn = 0.0;
    for (long long k = gtid; k < ncomp; k += gth) {
      const bool mine = fused && k == gtid;
      const long long p = mine ? own.p : (long long)__ldg(S.idx + k);
      const long long ri = fused ? p : k;
      x[k] = fma(alpha, mine ? p0 : __ldcg(Pn + p), x[k]);
      const double rk = fma(-alpha, mine ? q0 : q[k], __ldcg(r + ri));
      r[ri] = rk;
      rn = fma(rk, rk, rn);
    }
    {
      const double v[1] = {rn};
      double tot[1];
      if (!gs.sum<1>(a.st, bar, v, tot, 74)) return;
      if (threadIdx.x == 0) {
        // the root only where the squares do not decide
        s_state = tot[0] <= s_stop2 && sqrt(tot[0]) <= s_stop ? 1 : 0;
        s_beta = tot[0] / s_rr;
        s_rr = tot[0];
      }
      __syncthreads();
    }
    ++it;
  }
  // the solution at the computational points; other nodes keep their values
  for (long long k = gtid; k < ncomp; k += gth) a.u[__ldg(S.idx + k)] = x[k];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const double bnorm = a.out[1];
    a.out[0] = (double)it;
    a.out[1] = bnorm > 0.0 ? sqrt(s_rr) / bnorm : sqrt(s_rr);
    if (s_state != 1) atomicOr(&a.st->err, ERRF_KRYLOV);
  }
}

template <int N, bool NODE>
__global__ void __launch_bounds__(PS_NT, 1) poisson_kernel(const __grid_constant__ PoissonArgs a) {
  poisson_body<N, NODE>(a);
  barrier_done(a.st);
}

cudaError_t launch_poisson(const PoissonArgs& a, cudaStream_t stream) {
  void* fn;
  const bool node = a.S.beta_field != nullptr;
  switch (a.g.ndim) {
    case 2: fn = node ? (void*)poisson_kernel<2, true> : (void*)poisson_kernel<2, false>; break;
    case 3: fn = node ? (void*)poisson_kernel<3, true> : (void*)poisson_kernel<3, false>; break;
    case 4: fn = node ? (void*)poisson_kernel<4, true> : (void*)poisson_kernel<4, false>; break;
    default: return cudaErrorInvalidValue;
  }
  int dev = 0, sms = 0, per = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, PS_NT, 0);
  if (e != cudaSuccess) return e;
  if (per < 1) return cudaErrorLaunchOutOfResources;
  PoissonArgs c = a;
  c.cfac = 1.0 / (a.g.h * a.g.h);
  void* args[] = {(void*)&c};
  return cudaLaunchCooperativeKernel(fn, min(sms, MAX_SUM_BLOCKS), PS_NT, args, 0, stream);
}

}  // namespace etd
