// stream.cu -- launch of the streamed propagators (stream.cuh); the kernels are instantiated
// per task kind in stream_inst.cu.
#include "stream.cuh"

namespace ptg {

cudaError_t launch_stream(const StepParams& P, int precision, int ngroups, cudaStream_t stream) {
  StreamKernels ks{nullptr, nullptr};
  switch (P.kind) {
    case KIND_FINE_PRI: ks = stream_select_0(); break;
    case KIND_COARSE_PRI: ks = stream_select_1(); break;
    case KIND_CORRECT_PRI: ks = stream_select_2(); break;
    case KIND_FINE_ADJ: ks = stream_select_3(); break;
    case KIND_COARSE_ADJ: ks = stream_select_4(); break;
    case KIND_CORRECT_ADJ: ks = stream_select_5(); break;
    default: break;
  }
  const StreamKernel k = precision == PTG_FP32_REFINE ? ks.f32 : ks.f64;
  if (!k || ngroups < 1 || ngroups * P.cs > kMaxGrid) return cudaErrorInvalidConfiguration;
  // shared memory of the largest level's rings
  size_t smem = 0;
  for (int l = 0; l + 1 < P.mg_levels; ++l) {
    const int G4 = P.mg[l].W / kGroup;
    const int weights = l == 0 ? kElemWeights : kNodeWeights;
    if (pipe_rows(G4, weights) > 0 && pipe_bytes(G4, weights) > smem) smem = pipe_bytes(G4, weights);
  }
  cudaError_t e = configure_kernel((const void*)k, smem, false);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(P.g_bar, 0, 4 * sizeof(unsigned) * ngroups, stream);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = dim3((unsigned)(ngroups * P.cs), 1, 1);
  cfg.blockDim = dim3((unsigned)kStreamThreads, 1, 1);   // the row rings count on it
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, P);
}

}  // namespace ptg
