// Tangent pass and x transform in one kernel, for x-y planes that the separate
// row and column kernels serve (transform3.cuh, nx = ny = 256): a block takes
// RowVoxels consecutive voxels (whole rows), evaluates t = K : p there (with
// the CG vector updates of k_tangent inside a solve), keeps the nine
// components of t in shared memory as half-length complex rows, transforms
// them and writes the row spectra.  t itself never reaches memory: 72 bytes
// per voxel and application less than a tangent pass and a row pass (the
// operator on a 256^3 cell moved 472 bytes per voxel and is bound by HBM:
// 1584 -> 1444 us).  t and its row spectra have the bits of those two; inside a
// solve p.t is summed over other groups of voxels, so that its last bits (and
// through alpha now and then an FP32 rounding) are its own.
#include "tangent.cuh"
#include "transform3.cuh"

namespace {

constexpr int kThreads = 256;
// Voxels per group: two per thread inside a solve, four for the operator alone,
// which has three of its streams less to load before a group's transform
// (256^3 operator, neo-Hookean 1455 -> 1444 us, SVK 1521 -> 1487; inside a solve
// four are slower: 113.1 -> 115.3 ms for 32 SVK iterations at 256^3)
template <bool CG> struct RowVoxels { static constexpr int value = CG ? 512 : 1024; };
constexpr int kMaxBlocks = 152 * 4;     // resident at once; each walks over groups of rows

template <int NX, bool CG> struct RowsShape {
  static constexpr int H = NX / 2, PX = H + 1, ROWS = RowVoxels<CG>::value / NX, NSEQ = 9 * ROWS;
  static constexpr size_t smem() {
    return (size_t)NSEQ * PX * sizeof(float2) + (size_t)NX * sizeof(float2) + (size_t)H * sizeof(int);
  }
};

template <int NX, int TAN, bool CG>
__global__ void __launch_bounds__(kThreads, 4)
    k_tangent_rows(const float* __restrict__ pin, const float* __restrict__ r, float* __restrict__ pout,
                   float* __restrict__ x, TangentArgs ta, float2* __restrict__ spec, int nz, long long N,
                   const float2* __restrict__ gtw, const int* __restrict__ gpos, double* __restrict__ partials,
                   Scalars* sc) {
  typedef float2 C;
  typedef RowsShape<NX, CG> Sh;
  constexpr int kRowVoxels = RowVoxels<CG>::value;
  constexpr int H = Sh::H, PX = Sh::PX, ROWS = Sh::ROWS, NSEQ = Sh::NSEQ, NY = NX;
  static_assert(kRowVoxels % NX == 0 && NY % ROWS == 0, "whole rows, groups within a plane");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[32];
  C* buf = reinterpret_cast<C*>(smem_raw);   // [9][ROWS][PX]
  C* twx = buf + NSEQ * PX;
  int* posx = reinterpret_cast<int*>(twx + NX);
  for (int i = threadIdx.x; i < NX; i += kThreads) twx[i] = gtw[i];
  for (int i = threadIdx.x; i < H; i += kThreads) posx[i] = gpos[i];
  float beta = 0.f, alpha = 0.f;
  double rr = 0.0;   // thread 0
  bool first = false;
  if (CG) {
    // one reader per block (see k_tangent)
    __shared__ int s_stop, s_its;
    __shared__ float s_beta, s_alpha;
    if (threadIdx.x == 0) {
      s_stop = *(volatile const int*)&sc->stop;
      s_its = *(volatile const int*)&sc->its;
      s_beta = (float)*(volatile const double*)&sc->beta;
      s_alpha = (float)*(volatile const double*)&sc->alpha;
      rr = *(volatile const double*)&sc->rr;
    }
    __syncthreads();
    if (s_stop) return;
    beta = s_beta;
    alpha = s_alpha;
    first = s_its == 0;
  }
  Dot32 acc;
  const int groups = (int)(N / kRowVoxels);
  for (int g = blockIdx.x; g < groups; g += gridDim.x) {
#pragma unroll 1
    for (int k = 0; k < kRowVoxels / kThreads; ++k) {
      const int local = threadIdx.x + k * kThreads;
      const long long v = MF_AT((long long)g * kRowVoxels + local, N);
      float po[9], rv[9], xv[9], h[9], q[9], t[9];
#pragma unroll
      for (int c = 0; c < 9; ++c) {
        po[c] = (CG && first) ? 0.f : pin[c * N + v];
        rv[c] = CG ? r[c * N + v] : 0.f;
        xv[c] = (CG && !first) ? x[c * N + v] : 0.f;
        h[c] = ta.H[c * N + v];
      }
      const int ph = ta.phase[v];
#pragma unroll
      for (int c = 0; c < 9; ++c) {
        if (CG) {
          q[c] = rv[c] + beta * po[c];
          x[c * N + v] = xv[c] + alpha * po[c];
          pout[c * N + v] = q[c];
        } else {
          q[c] = po[c];
        }
      }
      if (TAN == 1) neohooke_apply(h, ta.table[2 * ph], ta.table[2 * ph + 1], q, t);
      else svk_apply(h, ta.table + 36 * ph, q, t);
      const float s = ta.scale ? ta.scale[v] : 1.f;
      const int row = local / NX, xx = local % NX;
#pragma unroll
      for (int c = 0; c < 9; ++c) {
        const float o = s * t[c];
        reinterpret_cast<float*>(buf)[2 * MF_AT((c * ROWS + row) * PX, NSEQ * PX) + xx] = o;
        if (CG) acc.add_prod(q[c], o);
      }
    }
    __syncthreads();
    fft2::forward<C, H, NX, NSEQ, 1, PX, 0, 1>(buf, twx);
    constexpr int NP = H / 2 + 1;
    for (int idx = threadIdx.x; idx < NSEQ * NP; idx += kThreads) {
      const int y = idx % NSEQ, k = idx / NSEQ;
      const int km = (H - k) % H;
      C* rw = buf + y * PX;
      const int pa = posx[k], pb = posx[km];
      const C za = rw[pa], zb = rw[pb];
      if (km != k) rw[pb] = tr2::split_one<float>(zb, za, twx[km]);
      rw[pa] = tr2::split_one<float>(za, zb, twx[k]);
    }
    __syncthreads();
    const int z = g / (NY / ROWS), y0 = (g % (NY / ROWS)) * ROWS;
    for (int idx = threadIdx.x; idx < NSEQ * H; idx += kThreads) {
      const int y = idx / H, j = idx - y * H, c = y / ROWS, row = y % ROWS;
      spec[MF_AT((((long long)c * nz + z) * NY + y0 + row) * H + j, 9LL * nz * NY * H)] = buf[y * PX + j];
    }
    __syncthreads();   // the buffer is refilled by the next group
  }
  if (CG) {
    const double s = block_total(acc.value(), red);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
    double pAp;
    if (last_block_total(partials, &sc->arrive, &pAp) && threadIdx.x == 0) cg_finish_alpha(pAp, rr, sc);
  }
}

template <int NX, int TAN, bool CG>
cudaError_t launch_rows(const float* pin, const float* r, float* pout, float* x, const TangentArgs& ta, void* spec,
                        const XYArgs& a, double* partials, Scalars* sc, cudaStream_t st) {
  const size_t sm = RowsShape<NX, CG>::smem();
  const long long groups = a.N / RowVoxels<CG>::value;
  const int grid = (int)(groups < kMaxBlocks ? groups : kMaxBlocks);
  ++g_mf_launches;
  k_tangent_rows<NX, TAN, CG><<<grid, kThreads, sm, st>>>(pin, r, pout, x, ta, (float2*)spec, a.nz, a.N,
                                                          (const float2*)a.twx, a.xpos, partials, sc);
  return cudaGetLastError();
}

template <int NX>
cudaError_t launch_nx(int tan, bool cg, const float* pin, const float* r, float* pout, float* x, const TangentArgs& ta,
                      void* spec, const XYArgs& a, double* partials, Scalars* sc, cudaStream_t st) {
  if (tan == 1)
    return cg ? launch_rows<NX, 1, true>(pin, r, pout, x, ta, spec, a, partials, sc, st)
              : launch_rows<NX, 1, false>(pin, r, pout, x, ta, spec, a, partials, sc, st);
  return cg ? launch_rows<NX, 2, true>(pin, r, pout, x, ta, spec, a, partials, sc, st)
            : launch_rows<NX, 2, false>(pin, r, pout, x, ta, spec, a, partials, sc, st);
}

}  // namespace

cudaError_t mf_launch_tangent_rows(const void* pin, const void* r, void* pout, void* x, int tan, bool cg,
                                   const TangentArgs& ta, void* spec, const XYArgs& a, double* partials, Scalars* sc,
                                   cudaStream_t st) {
  if (!a.split || (tan != 1 && tan != 2)) return cudaErrorInvalidValue;
  const float *p = (const float*)pin, *rf = (const float*)r;
  float *po = (float*)pout, *xf = (float*)x;
  if (a.nx == 256) return launch_nx<256>(tan, cg, p, rf, po, xf, ta, spec, a, partials, sc, st);
  if (a.nx == 32) return launch_nx<32>(tan, cg, p, rf, po, xf, ta, spec, a, partials, sc, st);
  return cudaErrorInvalidValue;
}
