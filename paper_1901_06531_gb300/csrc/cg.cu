// Conjugate-gradient iteration on the projected tangent operator of
// Eq. (linequil2ast), restructured so that every vector update rides on a
// pass that streams the same data anyway:
//
//   tangent pass : p = r + beta p', x += alpha' p' (alpha', p' of the previous
//                  iteration), t = K : p, partial sums of p . t
//   transforms   : y = G*(t) (x-y forward, z-pass with G-hat-star, x-y inverse)
//   inverse pass : r -= alpha y, partial sums of r . r
//
// p . A p = p . G*(K:p) = p . (K:p) because every CG direction lies in the
// range of the orthogonal projection G* (b does, and A maps into it), so the
// curvature is available before the transforms run.
//
// The tangent K = dP/dF (Eq. eq:lineariz) is either read packed (45 entries
// per voxel) or, in FP32, applied without being stored, from H = F - I and
// the phase's parameters:
//   neo-Hookean   K:q = mu q + lam (G:q) G + (mu - lam ln J) G q^T G, G = F^-T
//   St V.-K.      K:q = q S + F (C : sym(F^T q)),  S = C : E,  E = (H + H^T + H^T H)/2
#include <type_traits>

#include "launch.h"
#include "tangent.cuh"

namespace {

constexpr int kThreads = 256;
constexpr int kTangentBlocks = 152 * 8;   // rows of the table of partial sums the callers provide

// TAN 0: packed tangent K45 of type T; 1: neo-Hookean from H; 2: SVK from H.
// CG true: p = r + beta p', x += alpha' p' first (p' = pin); false: p = pin.
// FIN (with CG): the last block to finish sums the partials of p.t and sets
// alpha (no separate finishing launch).
// Registers: TAN 0 two blocks of 256 an SM (its 45 tangent entries in flight),
// the others four, five without the CG vectors.
template <typename T, int TAN, bool CG, bool FIN>
__global__ void __launch_bounds__(kThreads, TAN == 0 ? 2 : (CG ? 4 : 5)) k_tangent(const T* __restrict__ pin, const T* __restrict__ r,
                                                      T* __restrict__ pout, T* __restrict__ x,
                                                      TangentArgs ta, T* __restrict__ t, long long N,
                                                      double* __restrict__ partials, Scalars* sc) {
  static_assert(!FIN || CG, "the fused finish belongs to the CG pass");
  __shared__ double red[32];
  T beta = (T)0, alpha = (T)0;
  double rr = 0.0;   // thread 0
  pdl_wait();
  bool first = false;   // first CG iteration: p = r, x = 0 (neither previous vector is read)
  if (CG) {
    // the four scalars in one memory latency, read by one thread: the block
    // scalars share an L2 line, which a read per warp turns into a queue
    // (64^3, 8192 warps)
    __shared__ int s_stop, s_its;
    __shared__ T s_beta, s_alpha;
    if (threadIdx.x == 0) {
      const int stop = *(volatile const int*)&sc->stop, its = *(volatile const int*)&sc->its;
      const double b = *(volatile const double*)&sc->beta, a = *(volatile const double*)&sc->alpha;
      if (FIN) rr = *(volatile const double*)&sc->rr;
      s_stop = stop;
      s_its = its;
      s_beta = (T)b;
      s_alpha = (T)a;
    }
    __syncthreads();
    if (s_stop) return;
    beta = s_beta;
    alpha = s_alpha;
    first = s_its == 0;
  }
  double acc64 = 0.0;
  Dot32 acc32;
  // one voxel; FIRST: p = r, x = 0 without loading the previous vectors
  // (the loop is instantiated once per case, so that in each every load of
  // the voxel is issued before any arithmetic)
  auto voxel = [&](long long v, auto first_tag) {
    constexpr bool FIRST = decltype(first_tag)::value;
    v = MF_AT(v, N);   // every access below is c * N + v (c < 9) or t * N + v (t < 45)
    T po[9], rv[9], xv[9];
    float h[9];
    int ph = 0;
    if constexpr (FIRST) {
#pragma unroll
      for (int c = 0; c < 9; ++c) { rv[c] = r[c * N + v]; po[c] = (T)0; xv[c] = (T)0; }
    } else {
#pragma unroll
      for (int c = 0; c < 9; ++c) po[c] = pin[c * N + v];
      if (CG) {
#pragma unroll
        for (int c = 0; c < 9; ++c) { rv[c] = r[c * N + v]; xv[c] = x[c * N + v]; }
      }
    }
    T kv[TAN == 0 ? 45 : 1];
    if (TAN != 0) {
#pragma unroll
      for (int c = 0; c < 9; ++c) h[c] = ta.H[c * N + v];
      ph = ta.phase[v];
    } else {
      const T* K = reinterpret_cast<const T*>(ta.K45);
#pragma unroll
      for (int t = 0; t < 45; ++t) kv[t] = K[t * N + v];
    }
    T q[9];
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
    T o[9];
    if (TAN == 0) {
      // every entry loaded once, each used for its row and its column
#pragma unroll
      for (int a = 0; a < 9; ++a) o[a] = kv[sym45(a, a)] * q[a];
#pragma unroll
      for (int a = 0; a < 9; ++a)
#pragma unroll
        for (int b = a + 1; b < 9; ++b) {
          o[a] += kv[sym45(a, b)] * q[b];
          o[b] += kv[sym45(a, b)] * q[a];
        }
    } else {
      float qf[9], tf[9];
#pragma unroll
      for (int c = 0; c < 9; ++c) qf[c] = (float)q[c];
      if (TAN == 1) neohooke_apply(h, ta.table[2 * ph], ta.table[2 * ph + 1], qf, tf);
      else svk_apply(h, ta.table + 36 * ph, qf, tf);
      const float s = ta.scale ? ta.scale[v] : 1.f;
#pragma unroll
      for (int c = 0; c < 9; ++c) o[c] = (T)(s * tf[c]);
    }
#pragma unroll
    for (int c = 0; c < 9; ++c) {
      t[c * N + v] = o[c];
      if (sizeof(T) == 4) acc32.add_prod((float)q[c], (float)o[c]);
      else acc64 += (double)q[c] * (double)o[c];
    }
  };
  const long long v0 = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long dv = (long long)gridDim.x * blockDim.x;
  if (CG && first) {
    for (long long v = v0; v < N; v += dv) voxel(v, std::true_type{});
  } else {
    for (long long v = v0; v < N; v += dv) voxel(v, std::false_type{});
  }
  if (partials) {
    const double acc = block_total(sizeof(T) == 4 ? acc32.value() : acc64, red);
    if (threadIdx.x == 0) partials[blockIdx.x] = acc;
    if constexpr (FIN) {
      double pAp;
      if (last_block_total(partials, &sc->arrive, &pAp) && threadIdx.x == 0) cg_finish_alpha(pAp, rr, sc);
    }
  }
}

__device__ __forceinline__ double col_sum(const double* partials, int n, double* shm) {
  double s = 0.0;
  for (int b = threadIdx.x; b < n; b += blockDim.x) s += partials[b];
  shm[threadIdx.x] = s;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) shm[threadIdx.x] += shm[threadIdx.x + w];
    __syncthreads();
  }
  const double r = shm[0];
  __syncthreads();
  return r;
}

__global__ void __launch_bounds__(kThreads) k_fin_beta(const double* __restrict__ partials, int n,
                                                       Scalars* sc) {
  __shared__ double shm[kThreads];
  if (*(volatile const int*)&sc->stop) return;
  CgScalars cs;
  cs.load(sc);
  const double rr = col_sum(partials, n, shm);
  if (threadIdx.x == 0) cg_finish_beta(rr, cs, sc);
}

template <typename T>
__global__ void k_axpy_alpha(T* __restrict__ x, const T* __restrict__ p, long long n, const Scalars* sc) {
  const T a = (T)sc->alpha;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    x[i] += a * p[i];
}

// End of a CG body in a graph: keep looping while the solve has not stopped.
__global__ void k_cg_cond(const Scalars* sc, cudaGraphConditionalHandle h) {
  pdl_wait();
  cudaGraphSetConditional(h, *(volatile const int*)&sc->stop ? 0u : 1u);
}

// Final lagging update x += alpha p, with p the direction of the last
// completed iteration (iteration j writes pbuf[(j+1) % 2]).
template <typename T>
__global__ void k_axpy_last(T* __restrict__ x, const T* __restrict__ p0, const T* __restrict__ p1, long long n,
                            const Scalars* sc) {
  const int its = sc->its;
  if (its == 0) {   // no iteration ran (converged at the start, or stopped in the first): x = 0
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
      x[i] = (T)0;
    return;
  }
  const T* p = (its & 1) ? p1 : p0;
  const T a = (T)sc->alpha;
  const long long i0 = blockIdx.x * (long long)blockDim.x + threadIdx.x, di = (long long)gridDim.x * blockDim.x;
  long long head = 0;
  if constexpr (sizeof(T) == 4) {
    // 16-byte accesses where both vectors allow them (the same arithmetic)
    if ((((uintptr_t)x | (uintptr_t)p) & 15) == 0) {
      head = n & ~3LL;
      float4* x4 = reinterpret_cast<float4*>(x);
      const float4* p4 = reinterpret_cast<const float4*>(p);
      for (long long i = i0; i < head / 4; i += di) {
        float4 xv = x4[i];
        const float4 pv = p4[i];
        xv.x += a * pv.x;
        xv.y += a * pv.y;
        xv.z += a * pv.z;
        xv.w += a * pv.w;
        x4[i] = xv;
      }
    }
  }
  for (long long i = head + i0; i < n; i += di) x[i] += a * p[i];
}

// H = F - I in FP32 (the state the matrix-free tangent needs).
__global__ void k_make_H(const double* __restrict__ F, float* __restrict__ H, long long N) {
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < N;
       v += (long long)gridDim.x * blockDim.x) {
#pragma unroll
    for (int c = 0; c < 9; ++c) {
      const double d = (c == 0 || c == 4 || c == 8) ? 1.0 : 0.0;
      H[c * N + v] = (float)(F[c * N + v] - d);
    }
  }
}

}  // namespace

cudaError_t mf_launch_tangent(const void* pin, const void* r, void* pout, void* x, bool f32, int tan,
                              bool cg, const TangentArgs& ta, void* t, long long N, double* partials,
                              int nblk, Scalars* sc, cudaStream_t st, bool fin_alpha, bool pdl) {
  cudaError_t e = cudaSuccess;
  // small cells: blocks of 64 threads, which spread the voxels over the SMs
  // (16^3: 64 blocks instead of 16; with the packed FP64 tangent, bound by the
  // FP64 pipes of the SMs that take part, 9.2 -> 6.2 us, with the FP32 one
  // 3.8 -> 3.0 us; 36^3 16.8 -> 11.4 and 5.0 -> 4.2 us), as long as their
  // partial sums fit the table of kTangentBlocks rows
  int threads = kThreads;
  if (N <= 64LL * kTangentBlocks) {
    threads = 64;
    nblk = (int)((N + 63) / 64);
  }
#define MF_TAN(T, K, CGV, FV)                                                                                 \
  e = launch_k(pdl, k_tangent<T, K, CGV, FV>, dim3(nblk), dim3(threads), 0, st, (const T*)pin, (const T*)r, \
               (T*)pout, (T*)x, ta, (T*)t, N, partials, sc)
#define MF_TAN_CG(T, K)                                       \
  do {                                                        \
    if (!cg) MF_TAN(T, K, false, false);                      \
    else if (fin_alpha && partials) MF_TAN(T, K, true, true); \
    else MF_TAN(T, K, true, false);                           \
  } while (0)
  if (f32) {
    if (tan == 0) MF_TAN_CG(float, 0);
    else if (tan == 1) MF_TAN_CG(float, 1);
    else MF_TAN_CG(float, 2);
  } else {
    MF_TAN_CG(double, 0);
  }
#undef MF_TAN_CG
#undef MF_TAN
  g_mf_launches += 1;
  return e;
}

__global__ void k_cg_batch_init(Scalars* sc, int max_its) {
  sc->its = 0;
  sc->arrive = 0u;
  sc->max_its = max_its;
  sc->stop = (sc->done || sc->flags) ? 1 : 0;
}

cudaError_t mf_launch_cg_batch_init(Scalars* sc, int max_its, cudaStream_t st) {
  k_cg_batch_init<<<1, 1, 0, st>>>(sc, max_its);
  g_mf_launches += 1;
  return cudaGetLastError();
}

cudaError_t mf_launch_fin_beta(const double* partials, int n, Scalars* sc, cudaStream_t st) {
  k_fin_beta<<<1, kThreads, 0, st>>>(partials, n, sc);
  g_mf_launches += 1;
  return cudaGetLastError();
}

cudaError_t mf_launch_axpy_alpha(void* x, const void* p, bool f32, long long n, const Scalars* sc,
                                 cudaStream_t st) {
  const int g = stride_grid(n, kThreads);
  if (f32) k_axpy_alpha<float><<<g, kThreads, 0, st>>>((float*)x, (const float*)p, n, sc);
  else k_axpy_alpha<double><<<g, kThreads, 0, st>>>((double*)x, (const double*)p, n, sc);
  g_mf_launches += 1;
  return cudaGetLastError();
}

cudaError_t mf_launch_make_H(const double* F, float* H, long long N, cudaStream_t st) {
  k_make_H<<<stride_grid(N, kThreads), kThreads, 0, st>>>(F, H, N);
  g_mf_launches += 1;
  return cudaGetLastError();
}

cudaError_t mf_launch_cg_cond(const Scalars* sc, cudaGraphConditionalHandle h, cudaStream_t st, bool pdl) {
  g_mf_launches += 1;
  return launch_k(pdl, k_cg_cond, dim3(1), dim3(1), 0, st, sc, h);
}

cudaError_t mf_launch_axpy_last(void* x, const void* p0, const void* p1, bool f32, long long n,
                                const Scalars* sc, cudaStream_t st) {
  const int g = stride_grid(n, kThreads);
  if (f32) k_axpy_last<float><<<g, kThreads, 0, st>>>((float*)x, (const float*)p0, (const float*)p1, n, sc);
  else k_axpy_last<double><<<g, kThreads, 0, st>>>((double*)x, (const double*)p0, (const double*)p1, n, sc);
  g_mf_launches += 1;
  return cudaGetLastError();
}
