// k_f64_net.cu -- the in-loop learned curvature of the double-precision form.
// The network's FP32 epilogues round without fused multiply-add here (this
// unit compiles with --fmad=false, the rest of the FP64 kernels with it): a
// curvature from the network enters the FP64 run with its FP32 rounding, and
// fused it moved such runs by 1e-8 where everything else agrees to 1e-14.
#include "lbf_mlp_kappa.cuh"

namespace lbf {
void mlp_kappa_f64(const Params &p, const void *img, int blocks, cudaStream_t s) {
  k_mlp_kappa<3, double><<<blocks, MLP_THREADS, sizeof(tc::Tile), s>>>(p, (const tc::Image *)img);
}
}  // namespace lbf
