// FP64 instances of the any-size transform kernels.
#include "transformg.cuh"

cudaError_t mf_g_xyf_f64(const void* in, void* spec, const XYArgs& a, cudaStream_t st) {
  return trg::xyf<double>(in, spec, a, st);
}
cudaError_t mf_g_xyi_f64(int mode, const void* spec, void* out, double* partials, const XYArgs& a,
                         const Scalars* sc, cudaStream_t st) {
  return trg::xyi<double>(mode, spec, out, partials, a, sc, st);
}
cudaError_t mf_g_zp_f64(int mode, void* spec, const ZArgs& a, cudaStream_t st) {
  return trg::zp<double>(mode, spec, a, st);
}
