// The projected-operator passes: y = F^-1{ G-hat-star : F{ K : x } }
// (Eq. linequil2ast) and the residual b = -F^-1{ G-hat-star : F{ P - P-bar } }.
//
// Three kernels per application, each one pass over memory:
//   x-y forward : per (z-plane, component c): (K:x)_c or P_c for the plane,
//                 real-to-complex transform along x, then the complex
//                 transform along y; the plane stays in shared memory.
//   z-pass      : per tile of (ky, kx) columns and row group of three
//                 components: forward transform along z, G-hat-star
//                 (Eq. eq:Gnewnew) with the per-component null-frequency
//                 control, inverse along z.
//   x-y inverse : per (z-plane, component): inverse along y, complex-to-real
//                 along x, optionally the CG residual update.
// The fixed-size kernels (transform2.cuh) run on the grids they exist for,
// the any-size ones (transformg.cuh) on the others.  The x-Nyquist coefficient
// is never stored because G-hat-star is zero there.  The 1/N of the forward
// transform is applied once, in the z-pass.
#include "common.cuh"
#include "dw.cuh"

#include "launch.h"

long long g_mf_launches = 0;

namespace {

cudaError_t xyf(bool f32, const void* in, void* spec, const XYArgs& a, cudaStream_t st) {
  if (a.v2) return f32 ? mf_v2_xyf_f32(in, spec, a, st) : mf_v2_xyf_f64(in, spec, a, st);
  return f32 ? mf_g_xyf_f32(in, spec, a, st) : mf_g_xyf_f64(in, spec, a, st);
}

cudaError_t zp(bool f32, int mode, void* spec, const ZArgs& a, cudaStream_t st) {
  if (a.v2) return f32 ? mf_v2_zp_f32(mode, spec, a, st) : mf_v2_zp_f64(mode, spec, a, st);
  return f32 ? mf_g_zp_f32(mode, spec, a, st) : mf_g_zp_f64(mode, spec, a, st);
}

cudaError_t xyi(bool f32, int mode, const void* spec, void* out, double* partials, const XYArgs& a, const Scalars* sc,
                cudaStream_t st) {
  if (a.v2)
    return f32 ? mf_v2_xyi_f32(mode, spec, out, partials, a, sc, st)
               : mf_v2_xyi_f64(mode, spec, out, partials, a, sc, st);
  return f32 ? mf_g_xyi_f32(mode, spec, out, partials, a, sc, st) : mf_g_xyi_f64(mode, spec, out, partials, a, sc, st);
}

}  // namespace

cudaError_t mf_launch_residual(const double* P, void* spec, double* b, double* partials,
                               const XYArgs& xa, const ZArgs& za, bool dw, cudaStream_t st) {
  if (dw) {
    cudaError_t e = mf_v2_xyf_dw(P, spec, xa, st);
    if (e == cudaSuccess) e = mf_v2_zp_dw(spec, za, st);
    if (e == cudaSuccess) e = mf_v2_xyi_dw(spec, b, partials, xa, st);
    return e;
  }
  cudaError_t e = xyf(false, P, spec, xa, st);
  if (e == cudaSuccess) e = zp(false, 1, spec, za, st);
  if (e == cudaSuccess) e = xyi(false, 0, spec, b, partials, xa, nullptr, st);
  return e;
}

namespace {

// FP64 -> FP32 rounded through the double-word split (no FP64 instruction)
__global__ void k_d2f(const double* __restrict__ a, float* __restrict__ b, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const dw d = dw_split(a[i]);
    b[i] = __fadd_rn(d.hi, d.lo);
  }
}

__global__ void k_f2d(const float* __restrict__ a, double* __restrict__ b, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    b[i] = f32_as_f64(a[i]);
}

}  // namespace

cudaError_t mf_launch_residual_f32(const double* P, float* Pf, void* spec, float* bf, double* b,
                                   const XYArgs& xa, const ZArgs& za, cudaStream_t st) {
  if (!xa.v2) return cudaErrorInvalidValue;
  const long long n9 = 9 * xa.N;
  cudaError_t e = cudaSuccess;
  if (P) {
    k_d2f<<<stride_grid(n9), 256, 0, st>>>(P, Pf, n9);
    e = cudaGetLastError();
    g_mf_launches += 1;
  }
  if (e == cudaSuccess) e = mf_v2_xyf_f32(Pf, spec, xa, st);
  if (e == cudaSuccess) e = mf_v2_zp_f32(1, spec, za, st);
  if (e == cudaSuccess) e = mf_v2_xyi_f32(0, spec, bf, nullptr, xa, nullptr, st);
  if (e == cudaSuccess) {
    k_f2d<<<stride_grid(n9), 256, 0, st>>>(bf, b, n9);
    e = cudaGetLastError();
  }
  g_mf_launches += 1;
  return e;
}

cudaError_t mf_launch_project(bool f32, const void* t, void* spec, void* out, int inv_mode,
                              double* partials, const XYArgs& xa, const ZArgs& za,
                              const Scalars* sc, cudaStream_t st) {
  cudaError_t e = xyf(f32, t, spec, xa, st);
  if (e == cudaSuccess) e = zp(f32, 0, spec, za, st);
  if (e == cudaSuccess) e = xyi(f32, inv_mode, spec, out, partials, xa, sc, st);
  return e;
}

cudaError_t mf_launch_project_part(int which, bool f32, const void* t, void* spec, void* r,
                                   double* partials, const XYArgs& xa, const ZArgs& za,
                                   const Scalars* sc, cudaStream_t st) {
  if (which == 0) return xyf(f32, t, spec, xa, st);
  if (which == 1) return zp(f32, 0, spec, za, st);
  return xyi(f32, 3, spec, r, partials, xa, sc, st);
}

bool mf_v2_supported(int nx, int ny, int nz) {
  auto ok = [](int n) { return n == 16 || n == 32 || n == 48 || n == 64 || n == 96 || n == 128 || n == 256; };
  return nx == ny && ok(nx) && ok(nz);
}

bool mf_split_supported(int nx) { return nx == 32 || nx == 256; }
bool mf_persist_supported(int nx) { return nx == 48 || nx == 64 || nx == 96 || nx == 128; }
bool mf_cluster_supported(int nx) { return nx == 128; }

int mf_xy_blocks(int ny, int nz, bool split) { return split ? 9 * nz * (ny / 16) : 9 * nz; }
