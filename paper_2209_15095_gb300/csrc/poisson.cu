// Embedded-boundary Poisson solve (Sec. 2: div(beta grad u) = f with Dirichlet
// data, interior ghost points; Sec. 4.1 applies it to a virus-shaped domain).
//
// At the computational points the discrete problem is C u + b = f, with C the
// matrix-free EB operator (the stencil of the Krylov kernel with dt = 1) and
// b the boundary-data term of the ghost values (per point, the face slots'
// coefficient times the boundary value).  C is symmetric negative definite
// (Sec. 2), so the kernel runs conjugate gradients on A = -C, A u = b - f,
// FP64, as one persistent cooperative kernel with two grid barriers per
// iteration: the new search direction p = r + beta p_old is formed at the
// point and its 2N neighbours by the pass that applies A to it (r and p on the
// grid, p in two alternating arrays) instead of in a pass of its own with a
// barrier before the stencil reads it; the second pass updates x and r.  Sums
// are deterministic (every CTA forms them alike), so every CTA takes the same
// stopping decision; the iteration's scalars come from one thread (an FP64
// root and two divisions in every warp took an SM 6 us per iteration).
// Problems of at most one point per thread keep the point's index, diagonal
// and face coefficients in registers.  Measured on the virus domain at 321^2
// (28k points, 780 iterations): 14.4 -> 7.5 us per iteration.
#include "common.cuh"
#include "kernels.cuh"

namespace etd {

constexpr int PS_NT = 512;

// A computational point of the stencil: grid index (-1: none), diagonal and
// face coefficients.
template <int N>
struct PsPoint {
  long long p;
  double D, f[2 * N];
};
template <int N>
__device__ __forceinline__ PsPoint<N> ps_point(const SpeciesDev<double>& S, const GridDev& g, long long k, int ncomp) {
  PsPoint<N> o;
  o.p = -1;
  if (k >= ncomp) return o;
  o.p = __ldg(S.idx + k);
  o.D = __ldg(S.diag + k);
  const double* const bf = S.beta_field;
  const double bp = bf ? __ldg(bf + o.p) : 0.0;
#pragma unroll
  for (int d = 0; d < N; ++d) {
    o.f[2 * d] = bf ? 0.5 * (bp + __ldg(bf + o.p - g.stride[d])) : S.beta_c;
    o.f[2 * d + 1] = bf ? 0.5 * (bp + __ldg(bf + o.p + g.stride[d])) : S.beta_c;
  }
  return o;
}

// (C v)_p for v = val(grid index), with the value at the point itself
template <int N, typename Val>
__device__ __forceinline__ double cstencil(const PsPoint<N>& o, const GridDev& g, double cfac, double vp, bool node,
                                           double bc, Val val) {
  double s = -0.0;  // x + (-0) == x: the first add is free
  if (node) {
#pragma unroll
    for (int d = 0; d < N; ++d) {
      s += o.f[2 * d] * val(o.p - g.stride[d]);
      s += o.f[2 * d + 1] * val(o.p + g.stride[d]);
    }
    return cfac * (s - o.D * vp);
  }
#pragma unroll
  for (int d = 0; d < N; ++d) s += val(o.p - g.stride[d]) + val(o.p + g.stride[d]);
  return cfac * (bc * s - o.D * vp);
}

template <int N>
__device__ __forceinline__ void poisson_body(const PoissonArgs& a) {
  const SpeciesDev<double>& S = a.S;
  const GridDev& g = a.g;
  const int ncomp = *S.ncomp;
  const long long gtid = dealt_tid();
  const long long gth = (long long)gridDim.x * blockDim.x;
  const double cfac = a.cfac;
  const bool node = S.beta_field != nullptr;
  constexpr int SL = 2 * N * (N == 2 ? 2 : 1);
  unsigned bar = 0;
  GridSums gs(a.part);
  double* const x = S.Yc;             // compact: iterate
  double* const q = (double*)S.V2c;   // compact: A p
  double* const r = (double*)S.Z[0];  // grid: residual (zero off the set)
  double* const P[2] = {(double*)S.Yg, (double*)S.W1g};  // grid: search direction (zero off the set)
  __shared__ double s_alpha, s_beta, s_rr, s_stop, s_stop2;
  __shared__ int s_state;  // 0: go on, 1: converged, 2: stop
  const PsPoint<N> own = ps_point<N>(S, g, gtid, ncomp);
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
      const PsPoint<N> o = k == gtid ? own : ps_point<N>(S, g, k, ncomp);
      double rhs = -a.f[o.p];
      if (S.bco && S.bval) {
#pragma unroll
        for (int i = 0; i < SL; ++i) {
          const double cf = S.bco[k * SL + i];
          if (cf != 0.0) rhs = fma(cf, S.bval[k * SL + i], rhs);
        }
      }
      const double* const X = P[1];
      const double cx = cstencil<N>(o, g, cfac, __ldcg(X + o.p), node, S.beta_c, [&](long long i) { return __ldcg(X + i); });
      const double rk = rhs + cx;
      r[o.p] = rk;
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
    // p = r + beta p_old at the stencil's points, q = A p, <p, q>
    const double* const Po = P[(it & 1) ^ 1];
    double* const Pn = P[it & 1];
    const double beta = s_beta;
    const bool first = it == 0;
    const auto dir = [&](long long i) {
      const double ri = __ldcg(r + i);
      return first ? ri : fma(beta, __ldcg(Po + i), ri);
    };
    double pq = 0.0, p0 = 0.0, q0 = 0.0;
    for (long long k = gtid; k < ncomp; k += gth) {
      const PsPoint<N> o = k == gtid ? own : ps_point<N>(S, g, k, ncomp);
      const double pk = dir(o.p);
      const double qk = -cstencil<N>(o, g, cfac, pk, node, S.beta_c, dir);
      Pn[o.p] = pk;
      if (k == gtid) {
        p0 = pk;
        q0 = qk;
      } else {
        q[k] = qk;
      }
      pq = fma(pk, qk, pq);
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
      const bool mine = k == gtid;
      const long long p = mine ? own.p : (long long)__ldg(S.idx + k);
      x[k] = fma(alpha, mine ? p0 : Pn[p], x[k]);
      const double rk = fma(-alpha, mine ? q0 : q[k], __ldcg(r + p));
      r[p] = rk;
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

template <int N>
__global__ void __launch_bounds__(PS_NT, 1) poisson_kernel(const __grid_constant__ PoissonArgs a) {
  poisson_body<N>(a);
  barrier_done(a.st);
}

cudaError_t launch_poisson(const PoissonArgs& a, cudaStream_t stream) {
  void* fn;
  switch (a.g.ndim) {
    case 2: fn = (void*)poisson_kernel<2>; break;
    case 3: fn = (void*)poisson_kernel<3>; break;
    case 4: fn = (void*)poisson_kernel<4>; break;
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
