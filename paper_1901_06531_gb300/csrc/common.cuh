// Shared device machinery: complex helpers, per-axis FFT plans, small DFTs
// and the scalar blocks of the solvers.
//
// Transforms are computed in place with mixed-radix stages.  The
// forward transform is decimation in frequency (natural order in, digit-
// reversed order out), the inverse is its exact adjoint, decimation in time
// (digit-reversed in, natural out).  The spectrum therefore never needs a
// reordering pass: the projection is applied in digit-reversed order, with
// each position's frequency read from a small table.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#define MF_MAX_STAGES 10
#define MF_MAX_PASSES 5

// Bounds checks of the debug build (compiled with -DMF_DEBUG; release builds
// compile them away).  MF_AT(i, n) is i when 0 <= i < n; otherwise the
// failure is counted, the first one (source line, index, extent) recorded,
// and element 0 -- in bounds -- is used instead, so that the kernel runs to
// its end and the host reads the record (mf_debug_report) rather than the
// GPU faulting.  Every translation unit has its own record and registers a
// reader and a reset for it with the library at load time.
#ifdef MF_DEBUG
struct MfDebugRecord {
  unsigned long long count;
  long long index, extent;
  int line, pad;
};
void mf_debug_register(void (*read)(MfDebugRecord*), void (*clear)());
static __device__ MfDebugRecord g_mf_debug;
static void mf_debug_read_tu(MfDebugRecord* r) { cudaMemcpyFromSymbol(r, g_mf_debug, sizeof(*r)); }
static void mf_debug_clear_tu() {
  MfDebugRecord z = {0ull, 0, 0, 0, 0};
  cudaMemcpyToSymbol(g_mf_debug, &z, sizeof(z));
}
static const bool g_mf_debug_registered = (mf_debug_register(mf_debug_read_tu, mf_debug_clear_tu), true);
__device__ __forceinline__ long long mf_dbg_check(long long i, long long n, int line) {
  if (i >= 0 && i < n) return i;
  if (atomicAdd(&g_mf_debug.count, 1ull) == 0ull) {
    g_mf_debug.index = i;
    g_mf_debug.extent = n;
    g_mf_debug.line = line;
  }
  return 0;
}
#define MF_AT(i, n) mf_dbg_check((long long)(i), (long long)(n), __LINE__)
#else
#define MF_AT(i, n) (i)
#endif

// Programmatic dependent launch: a kernel launched with the programmatic
// stream-serialization attribute may be scheduled as soon as the blocks of
// its predecessor in the stream have exited, before that grid's completion
// (its memory flush) and the launch that would normally follow it; pdl_wait()
// returns once the predecessor grid has completed and its memory operations
// are visible.  For a kernel launched without the attribute it returns at
// once.  (No kernel here signals its dependents early: measured on the 128^3
// cell, dependents resident during the predecessor's last wave slowed it.)
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Grid of a grid-stride elementwise pass over n items with `threads` per
// block: one item per thread for small passes, at most 8 blocks per SM (152
// SMs) otherwise.
inline int stride_grid(long long n, int threads = 256) {
  const long long b = (n + threads - 1) / threads;
  return (int)(b < 1 ? 1 : (b < 152 * 8 ? b : 152 * 8));
}

// Quotients by a run-time divisor d through m = ceil(2^32 / d) (d > 1).
struct FastDiv {
  int d;
  unsigned m;
};
inline FastDiv fast_div(int d) {
  FastDiv f;
  f.d = d;
  f.m = d > 1 ? (unsigned)((0x100000000ull + (unsigned)d - 1) / (unsigned)d) : 0u;
  return f;
}

// One pass of an any-size transform over memory: a stage of radix r1 and, with
// r2 > 1, the stage of radix r2 after it.
struct AxisPass {
  int r1, r2;
  int tstep1, tstep2;   // twiddle table steps of the two stages
  FastDiv dm;           // by the last stage's sub-transform length / radix
  FastDiv nb;           // by the butterflies of a sequence, n / (r1 r2)
};

// Stages of a transform in decimation-in-frequency order (built by plan.h)
// and their grouping into passes.
struct AxisPlan {
  int n;                        // transform length
  int ntab;                     // length of the twiddle table, a multiple of n
  int nst, npass;
  unsigned char rad[MF_MAX_STAGES];
  AxisPass pass[MF_MAX_PASSES];
};

template <typename T> struct CT;
template <> struct CT<double> { typedef double2 t; };
template <> struct CT<float> { typedef float2 t; };

__device__ __forceinline__ double2 cmake(double a, double b) { return make_double2(a, b); }
__device__ __forceinline__ float2 cmake(float a, float b) { return make_float2(a, b); }
template <typename C> __device__ __forceinline__ C cadd(C a, C b) { a.x += b.x; a.y += b.y; return a; }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { a.x -= b.x; a.y -= b.y; return a; }
#ifndef MF_NO_F32X2
// FP32 complex add and subtract as one packed two-lane instruction (sm_100
// and later: add.f32x2, sub.f32x2), each lane rounded to nearest like the
// scalar pair; the butterflies of the FP32 transforms are mostly these.
__device__ __forceinline__ unsigned long long f2_pack(float2 a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ float2 f2_unpack(unsigned long long r) {
  float2 a;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
  return a;
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_pack(a)), "l"(f2_pack(b)));
  return f2_unpack(r);
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_pack(a)), "l"(f2_pack(b)));
  return f2_unpack(r);
}
#endif
template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
  C r; r.x = a.x * b.x - a.y * b.y; r.y = a.x * b.y + a.y * b.x; return r;
}
// a * conj(b)
template <typename C> __device__ __forceinline__ C cmulc(C a, C b) {
  C r; r.x = a.x * b.x + a.y * b.y; r.y = a.y * b.x - a.x * b.y; return r;
}
// multiply by -i (FWD) or +i (INV)
template <typename C, bool INV> __device__ __forceinline__ C rot90(C a) {
  C r;
  if (INV) { r.x = -a.y; r.y = a.x; } else { r.x = a.y; r.y = -a.x; }
  return r;
}

// Small DFT of length R on registers: y_k = sum_j x_j w^(jk), w = exp(-+2 pi i/R).
template <int R, bool INV, typename C> struct Radix;

template <bool INV, typename C> struct Radix<2, INV, C> {
  static __device__ __forceinline__ void run(C* v) {
    C a = v[0], b = v[1]; v[0] = cadd(a, b); v[1] = csub(a, b);
  }
};

template <bool INV, typename C> struct Radix<4, INV, C> {
  static __device__ __forceinline__ void run(C* v) {
    C t0 = cadd(v[0], v[2]), t1 = csub(v[0], v[2]);
    C t2 = cadd(v[1], v[3]), t3 = rot90<C, INV>(csub(v[1], v[3]));
    v[0] = cadd(t0, t2); v[2] = csub(t0, t2);
    v[1] = cadd(t1, t3); v[3] = csub(t1, t3);
  }
};

template <bool INV, typename C> struct Radix<3, INV, C> {
  static __device__ __forceinline__ void run(C* v) {
    typedef decltype(v[0].x) T;
    const T h = (T)0.5;
    const T s3 = (T)0.86602540378443864676372317075294;   // sin(2 pi / 3)
    C a = v[0];
    C t1 = cadd(v[1], v[2]);
    C d = csub(v[1], v[2]);
    C t2; t2.x = a.x - h * t1.x; t2.y = a.y - h * t1.y;
    // forward: y1 = t2 - i s3 d, y2 = t2 + i s3 d; inverse: signs of i swap
    C t3; t3.x = s3 * d.x; t3.y = s3 * d.y;
    C it3 = rot90<C, INV>(t3);     // -i*t3 forward, +i*t3 inverse
    v[0] = cadd(a, t1);
    v[1] = cadd(t2, it3);
    v[2] = csub(t2, it3);
  }
};

// Index of the packed symmetric 9x9 tangent entry (a, b), a, b in [0, 9).
__host__ __device__ __forceinline__ int sym45(int a, int b) {
  if (a > b) { int t = a; a = b; b = t; }
  return a * 9 - (a * (a - 1)) / 2 + (b - a);
}

// Device-side scalar block shared by the Newton/CG kernels (FP64).
struct Scalars {
  double rr;          // current r.r
  double rr0;         // r.r at CG start
  double pAp;
  double alpha;
  double beta;
  double thr2N;       // CG stop: rr <= thr2N
  double meanF[9];
  double meanP[9];
  double dF2max;      // max_v |dF_v|^2 of the last Newton update
  double meanF_new[9];
  double T[9];        // sum_v P_v F_v^T   (rotation moments, row-major)
  double S[9];        // sum_v F_v F_v^T
  double What[9];     // skew matrix of the last null-rotation projection
  double lin[9];      // FP32 inner solve: sum over its iterations of alpha_k <t_k> (= <K:x>, x = sum alpha_k p_k)
  int flags;          // bit 0: breakdown, bit 1: nonpositive J, bit 2: non-finite
  int done;           // CG converged
  int its;            // CG iterations completed
  int stop;           // CG finished (converged, failed or capped): iteration kernels return at once
  int max_its;
  unsigned arrive;    // blocks of the current pass that have stored their partial sum
};

// Sum of one value per thread over the block (whole warps, at most 32; red:
// 32 shared doubles), in thread 0.  The warps' sums are combined in log2 of
// their number of steps: each dependent FP64 addition is a step of the
// latency chain that ends a CG kernel.
__device__ __forceinline__ double block_total(double v, double* red) {
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  v = 0.0;
  if (threadIdx.x < 32) {
    v = lane < nw ? red[lane] : 0.0;
    for (int o = nw > 16 ? 16 : (nw > 8 ? 8 : (nw > 4 ? 4 : (nw > 2 ? 2 : 1))); o > 0; o >>= 1)
      v += __shfl_xor_sync(0xffffffffu, v, o);
  }
  return v;
}

// Grid-wide sum finished by the last block to arrive: every block's thread 0
// has stored its partial sum in partials[blockIdx.x]; here it counts the
// block in *arrive (one acquire-release operation publishes the partial and,
// in the last block, orders the reads of the others behind it).  The block
// that arrives last adds all partials in a fixed order, leaves the total in
// *total (thread 0), resets the counter and returns true; the others return
// false.  No block waits on another.
__device__ __forceinline__ bool last_block_total(const double* partials, unsigned* arrive, double* total) {
  __shared__ unsigned s_last;
  __shared__ double s_red[32];
  if (threadIdx.x == 0) {
    unsigned before;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(before) : "l"(arrive) : "memory");
    s_last = (before == gridDim.x - 1) ? 1u : 0u;
  }
  __syncthreads();
  if (!s_last) return false;
  double s = 0.0;
  for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x) s += __ldcg(partials + b);
  s = block_total(s, s_red);
  if (threadIdx.x == 0) {
    *total = s;
    *arrive = 0u;
  }
  return true;
}

#define MF_FLAG_BREAKDOWN 1
#define MF_FLAG_NONPOS_J 2
#define MF_FLAG_NONFINITE 4
#define MF_FLAG_TIMEOUT 8     // a bounded device-side wait gave up

// The scalars the updates below need, as the previous kernel left them: the
// fused passes read them when they start, off the chain at their end.
struct CgScalars {
  double rr, thr2N;
  int flags, its, max_its;
  __device__ __forceinline__ void load(const Scalars* sc) {
    rr = sc->rr;
    thr2N = sc->thr2N;
    flags = sc->flags;
    its = sc->its;
    max_its = sc->max_its;
  }
};

// CG scalar updates after the curvature p.Ap and after the new r.r (shared by
// the one-block finishing kernels and the last blocks of fused passes).
__device__ __forceinline__ void cg_finish_alpha(double pAp, double rr, Scalars* sc) {
  sc->pAp = pAp;
  if (!(pAp > 0.0) || !isfinite(pAp)) {
    sc->flags |= MF_FLAG_BREAKDOWN;
    sc->alpha = 0.0;
    sc->stop = 1;
  } else {
    sc->alpha = rr / pAp;
  }
}

__device__ __forceinline__ void cg_finish_beta(double rr, const CgScalars& b, Scalars* sc) {
  int flags = b.flags;
  if (!isfinite(rr)) sc->flags = flags = flags | MF_FLAG_NONFINITE;
  sc->beta = rr / b.rr;
  sc->rr = rr;
  const int done = (rr <= b.thr2N) ? 1 : 0;
  sc->done = done;
  sc->its = b.its + 1;
  sc->stop = (done || flags || b.its + 1 >= b.max_its) ? 1 : 0;
}
