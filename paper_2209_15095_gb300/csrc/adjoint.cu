// Adjoint of the ETD2 step on a frozen domain: pointwise combination of the
// phi-function actions, the ETD2 right-hand vectors at a quadrature time, and
// the face contraction that gives the gradient with respect to a node field
// beta.  The phi-function actions themselves come from the Krylov kernel.
//
// With lambda = dL/du_{n+1}, Phi_k = phi_k(dt C) lambda (C symmetric):
//   dL/du_n      = Phi_0 + dt F'(u_n) (Phi_1 + Phi_2) + (contribution of the later step)
//   dL/du_{n-1} += -dt F'(u_{n-1}) Phi_2
//   dL/dalpha   += dt <Phi_1 + Phi_2, dF/dalpha(u_n)> - dt <Phi_2, dF/dalpha(u_{n-1})>
// and, for beta, d(mu^T C y)/d beta_f = -h^-2 (mu_p - mu_q)(y_p - y_q) on a face
// between computational points, -h^-2 (1 - w_f) mu_p y_p on a face to a ghost
// point, half of it to each end node (beta_f is the mean of the two nodes).
#include "common.cuh"
#include "kernels.cuh"

namespace etd {

constexpr int ADJ_NT = 256;
constexpr int ADJ_BLOCKS = 608;

// F, F' and dF/dalpha of the single-species reactions
__device__ __forceinline__ void reaction_terms(int kind, const double* rp, double u, double& F, double& dF,
                                               double& dFa) {
  switch (kind) {
    case 1:
      F = u * (1.0 - u);
      dF = 1.0 - 2.0 * u;
      dFa = 0.0;
      break;
    case 2:
      F = rp[0] * u * (1.0 - u / rp[1]);
      dF = rp[0] * (1.0 - 2.0 * u / rp[1]);
      dFa = u * (1.0 - u / rp[1]);
      break;
    default:
      F = 0.0;
      dF = 0.0;
      dFa = 0.0;
  }
}

// part[blockIdx.x] = sum of v over the block, in a fixed order: warp 0 sums the staged
// values (lane-strided, then a warp tree), so that the FP64 additions run on one
// warp instead of every warp's shuffle tree.
__device__ __forceinline__ void block_partial(double v, double* part) {
  __shared__ double st[ADJ_NT];
  st[threadIdx.x] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    double x0 = 0.0, x1 = 0.0;
    for (int t = threadIdx.x; t < ADJ_NT; t += 64) {
      x0 += st[t];
      if (t + 32 < ADJ_NT) x1 += st[t + 32];
    }
    const double x = warp_sum(x0 + x1);
    if (threadIdx.x == 0) part[blockIdx.x] = x;
  }
}

__global__ void __launch_bounds__(ADJ_NT) adjoint_combine_kernel(const AdjointArgs a) {
  double part = 0.0;
  const long long G = a.g.size;
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < G; p += (long long)gridDim.x * blockDim.x) {
    if ((a.kind[p] & 3) != K_COMP) {
      a.lam[p] = 0.0;
      a.acc[p] = 0.0;
      continue;
    }
    double F, dFn, dFan, dFm, dFam;
    reaction_terms(a.reaction, a.rp, a.un[p], F, dFn, dFan);
    reaction_terms(a.reaction, a.rp, a.unm1[p], F, dFm, dFam);
    const double p0 = a.P0[p], p1 = a.P1[p], p2 = a.P2[p];
    double lam = p0 + a.dt * dFn * (p1 + p2) + a.acc[p];
    double acc = -a.dt * dFm * p2;
    if (a.first) {  // u_{-1} is u_0
      lam += acc;
      acc = 0.0;
    }
    part += a.dt * (p1 + p2) * dFan - a.dt * p2 * dFam;
    a.lam[p] = lam;
    a.acc[p] = acc;
  }
  block_partial(part, a.part);
}

// Sums the per-block partials in a fixed order (lane-strided, then a warp tree:
// one thread's 608 dependent FP64 additions took 25 us) and adds them to
// grad_params[0].
__global__ void adjoint_alpha_finish_kernel(const double* part, int nblocks, double* grad_params) {
  double s0 = 0.0, s1 = 0.0;
  for (int b = threadIdx.x; b < nblocks; b += 64) {
    s0 += part[b];
    if (b + 32 < nblocks) s1 += part[b + 32];
  }
  const double s = warp_sum(s0 + s1);
  if (threadIdx.x == 0) grad_params[0] += s;
}

cudaError_t launch_adjoint_combine(const AdjointArgs& a, cudaStream_t stream) {
  adjoint_combine_kernel<<<ADJ_BLOCKS, ADJ_NT, 0, stream>>>(a);
  adjoint_alpha_finish_kernel<<<1, 32, 0, stream>>>(a.part, ADJ_BLOCKS, a.grad_params);
  return cudaGetLastError();
}

__global__ void __launch_bounds__(ADJ_NT) adjoint_rhs_kernel(const AdjointArgs a, double s1, double s2, double* v1,
                                                            double* v2) {
  const int ncomp = *a.ncomp;
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < ncomp;
       k += (long long)gridDim.x * blockDim.x) {
    const long long p = a.idx[k];
    double F, Fm, d1, d2;
    reaction_terms(a.reaction, a.rp, a.un[p], F, d1, d2);
    reaction_terms(a.reaction, a.rp, a.unm1[p], Fm, d1, d2);
    v1[p] = s1 * (a.dt * F);
    v2[p] = s2 * (a.dt * (F - Fm));
  }
}

cudaError_t launch_adjoint_rhs(const AdjointArgs& a, double s1, double s2, double* v1, double* v2,
                               cudaStream_t stream) {
  adjoint_rhs_kernel<<<ADJ_BLOCKS, ADJ_NT, 0, stream>>>(a, s1, s2, v1, v2);
  return cudaGetLastError();
}

// All quadrature times at once, in two kernels: the weighted sum over i of the
// face derivative, once per face between computational points (a.face[d] at
// the lower node: four FP64 instructions per time, which bound the kernel),
// then one update per node (and one atomic per ghost face).
template <int N>
__global__ void __launch_bounds__(ADJ_NT) beta_faces_kernel(const AdjointArgs a) {
  const int ncomp = *a.ncomp;
  const int nq = a.nq;
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < ncomp;
       k += (long long)gridDim.x * blockDim.x) {
    const long long p = a.idx[k];
    double f[N];
#pragma unroll
    for (int d = 0; d < N; ++d) f[d] = 0.0;
    for (int i = 0; i < nq; ++i) {
      const double* __restrict__ const mu = a.muq[i];
      const double* __restrict__ const y = a.yq[i];
      const double mp = mu[p], yp = y[p], w = a.wq[i];
#pragma unroll
      for (int d = 0; d < N; ++d) {
        const long long q = p + a.g.stride[d];
        f[d] = fma(w, -(mp - mu[q]) * (yp - y[q]), f[d]);
      }
    }
    // (off the computational set the value is not read)
#pragma unroll
    for (int d = 0; d < N; ++d) a.face[d][p] = f[d];
  }
}

template <int N>
__global__ void __launch_bounds__(ADJ_NT) beta_gather_kernel(const AdjointArgs a, double* grad_beta) {
  const int ncomp = *a.ncomp;
  const double inv_h2 = 1.0 / (a.g.h * a.g.h);
  const int nq = a.nq;
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < ncomp;
       k += (long long)gridDim.x * blockDim.x) {
    const long long p = a.idx[k];
    double own = 0.0;
#pragma unroll
    for (int d = 0; d < N; ++d) {
#pragma unroll
      for (int si = 0; si < 2; ++si) {
        const long long q = p + (si == 0 ? -a.g.stride[d] : a.g.stride[d]);
        if ((a.kind[q] & 3) == K_COMP) {
          own += 0.5 * (a.face[d][si == 0 ? q : p] * inv_h2);
        } else {
          const double gw = a.facew[k * (2 * N) + 2 * d + si];
          double f = 0.0;
          for (int i = 0; i < nq; ++i) f = fma(a.wq[i], -gw * a.muq[i][p] * a.yq[i][p], f);
          const double df = 0.5 * (f * inv_h2);
          own += df;
          atomicAdd(grad_beta + q, df);
        }
      }
    }
    grad_beta[p] += own;
  }
}

template <int N>
static void beta_contract_launch(const AdjointArgs& a, double* grad_beta, cudaStream_t stream) {
  beta_faces_kernel<N><<<ADJ_BLOCKS, ADJ_NT, 0, stream>>>(a);
  beta_gather_kernel<N><<<ADJ_BLOCKS, ADJ_NT, 0, stream>>>(a, grad_beta);
}

cudaError_t launch_beta_contract_multi(const AdjointArgs& a, double* grad_beta, cudaStream_t stream) {
  switch (a.g.ndim) {
    case 2: beta_contract_launch<2>(a, grad_beta, stream); break;
    case 3: beta_contract_launch<3>(a, grad_beta, stream); break;
    case 4: beta_contract_launch<4>(a, grad_beta, stream); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace etd
