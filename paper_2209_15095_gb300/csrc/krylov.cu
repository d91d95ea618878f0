// Launch of the adaptive Krylov kernel (krylov_impl.cuh): picks the
// instantiation by precision and, for FP32, by `wide` (the caller's choice of
// the 768-thread kernel for problems on the 4-node groups), and runs it as a
// cooperative launch (one CTA per SM).
#include "kernels.cuh"

namespace etd {

PhipmKernels phipm_kernels_f64();
PhipmKernels phipm_kernels_f32();
PhipmKernels phipm_kernels_f32w();

namespace {
const PhipmKernels& f64() {
  static const PhipmKernels k = phipm_kernels_f64();
  return k;
}
const PhipmKernels& f32() {
  static const PhipmKernels k = phipm_kernels_f32();
  return k;
}
const PhipmKernels& f32w() {
  static const PhipmKernels k = phipm_kernels_f32w();
  return k;
}

template <typename T>
const PhipmKernels& variant(bool wide) {
  if (sizeof(T) == 8) return f64();
  return wide ? f32w() : f32();
}
}  // namespace

template <typename T>
cudaError_t launch_phipm(const PhipmArgs<T>& a, int nblocks, cudaStream_t stream, bool wide) {
  const PhipmKernels& v = variant<T>(wide);
  const bool adj = a.mode == MODE_ADJ_LAMBDA || a.mode == MODE_ADJ_Y;
  if (a.g.ndim < 2 || a.g.ndim > 4) return cudaErrorInvalidValue;
  void* fn = v.fn[a.g.ndim - 2][adj ? 1 : 0];
  if (nblocks > MAX_SUM_BLOCKS) return cudaErrorInvalidValue;
  void* args[] = {(void*)&a};
  const size_t dsm = adj ? v.adj_smem : 0;
  return cudaLaunchCooperativeKernel(fn, nblocks, v.nt, args, dsm, stream);
}

// CTAs of a launch: one per SM, if every instantiation the context may
// launch (the adjoint ones with their dynamic shared memory, which for the
// 768-thread kernel exceeds the default 48 KB of a block) fits once per SM.
int phipm_max_blocks(int ndim, bool fp32) {
  if (ndim < 2 || ndim > 4) return 0;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const PhipmKernels* vs[2] = {fp32 ? &f32() : &f64(), fp32 ? &f32w() : nullptr};
  int per = 1;
  for (const PhipmKernels* v : vs) {
    if (!v) continue;
    for (int adj = 0; adj < 2; ++adj) {
      void* fn = v->fn[ndim - 2][adj];
      const size_t dsm = adj ? v->adj_smem : 0;
      if (adj && cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dsm) != cudaSuccess)
        return 0;
      int p = 0;
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p, fn, v->nt, dsm) != cudaSuccess) return 0;
      per = min(per, p);
    }
  }
  return min(per * sms, MAX_SUM_BLOCKS);
}

template cudaError_t launch_phipm<double>(const PhipmArgs<double>&, int, cudaStream_t, bool);
template cudaError_t launch_phipm<float>(const PhipmArgs<float>&, int, cudaStream_t, bool);

}  // namespace etd
