// Transform kernels for any admissible size (nx, ny even, all of the form
// 2^a 3^b), with the sizes as run-time values: the grids the fixed-size
// kernels (transform2.cuh) do not cover.  Three kernels per projected
// operator, like there.
//
// Spectrum layout (per component c and plane z, one contiguous block of
// ny/2 x nx complex values, row q', slot s): two real rows q and q + ny/2 are
// transformed as one complex row, whose split is fused with the first
// (radix-2) stage of the y transform, which combines exactly those two.
//   slot s holds x-frequency kx(s) in [0, nx/2) of parity e(s) -- the
//   x-Nyquist coefficient is never stored because G-hat-star is zero there;
//   row q' holds y-frequency ky = 2 * yk(q') + e(s);
//   plane position p holds z-frequency kz = zk(p) during the z-pass.
//
// A length runs in radix-4, 2 and 3 stages, taken two at a time in registers
// (4 x 4, 4 x 2, 4 x 3, 2 x 3, 3 x 3: at most three shared-memory passes,
// two for every length but a few), the twiddles between the two from the same
// table as between passes: the arithmetic is that of separate stages, value
// for value.  The first pass of a transform reads global memory and the last
// one writes it where the layout allows.  The radices are a switch over
// unrolled butterflies; the index arithmetic that a template constant would
// fold away is two divisions by precomputed reciprocals per butterfly.  What
// bounds them is the work per sample that is not arithmetic, shared-memory
// passes and indices, in FP32, and the FP64 pipe in FP64.  Against one stage
// per pass with hardware divisions, whole planes staged before and after, and
// all nine components in one z-pass block: FP32 operator on 108 x 72 x 54
// 125 -> 52 us, stress and residual in FP64 on 48 x 36 x 18 184 -> 134 us.
#pragma once

#include <atomic>

#include "launch.h"

namespace trg {

// Quotient by a run-time divisor through its reciprocal (exact for t < 2^16
// and d <= 2^15, which bounds every index below).
__device__ __forceinline__ int fdiv(int t, FastDiv f) {
  return f.d == 1 ? t : (int)__umulhi((unsigned)t, f.m);
}

// One pass over nseq sequences: stage radix R1 and (R2 > 1) the radix-R2 stage
// after it, R1 R2 values per thread.  Inputs from ld(q, e), outputs to
// st(q, e, value), e the position along sequence q.  Value i = r R2 + a sits
// at e0 + i m, m the last stage's sub-length: the first stage combines r for
// each a (sub-index j0 + m a), the second a for each r.  SEQFAST: consecutive
// threads take consecutive sequences (else consecutive butterflies of one).
template <typename C, int R1, int R2, bool INV, bool SEQFAST, typename LD, typename ST>
__device__ __forceinline__ void pass_r(const AxisPass& p, int ntab, int nseq, FastDiv dseq, const C* tw, LD ld, ST st) {
  constexpr int R = R1 * R2;
  const int m = p.dm.d, nb = p.nb.d, total = nseq * nb, t1 = p.tstep1, t2 = p.tstep2;
  (void)ntab;
  for (int t = threadIdx.x; t < total; t += blockDim.x) {
    int q, b;
    if (SEQFAST) { b = fdiv(t, dseq); q = t - b * nseq; } else { q = fdiv(t, p.nb); b = t - q * nb; }
    const int blk = fdiv(b, p.dm);
    const int j0 = b - blk * m;
    const int e0 = blk * m * R + j0;
    C v[R];
#pragma unroll
    for (int i = 0; i < R; ++i) v[i] = ld(q, e0 + i * m);
    auto first = [&]() {
#pragma unroll
      for (int a = 0; a < R2; ++a) {
        const int ja = (j0 + m * a) * t1;
        C u[R1];
#pragma unroll
        for (int r = 0; r < R1; ++r) u[r] = v[r * R2 + a];
        if (INV) {
#pragma unroll
          for (int k = 1; k < R1; ++k) u[k] = cmulc(u[k], tw[MF_AT(ja * k, ntab)]);
        }
        Radix<R1, INV, C>::run(u);
        if (!INV) {
#pragma unroll
          for (int k = 1; k < R1; ++k) u[k] = cmul(u[k], tw[MF_AT(ja * k, ntab)]);
        }
#pragma unroll
        for (int r = 0; r < R1; ++r) v[r * R2 + a] = u[r];
      }
    };
    auto second = [&]() {
      if constexpr (R2 > 1) {
#pragma unroll
        for (int r = 0; r < R1; ++r) {
          C* u = v + r * R2;
          if (INV && m > 1) {
#pragma unroll
            for (int k = 1; k < R2; ++k) u[k] = cmulc(u[k], tw[MF_AT(j0 * k * t2, ntab)]);
          }
          Radix<R2, INV, C>::run(u);
          if (!INV && m > 1) {
#pragma unroll
            for (int k = 1; k < R2; ++k) u[k] = cmul(u[k], tw[MF_AT(j0 * k * t2, ntab)]);
          }
        }
      }
    };
    if (!INV) { first(); second(); } else { second(); first(); }
#pragma unroll
    for (int i = 0; i < R; ++i) st(q, e0 + i * m, v[i]);
  }
}

template <typename C, bool INV, bool SEQFAST, typename LD, typename ST>
__device__ __forceinline__ void pass(const AxisPlan& pl, int g, int nseq, FastDiv dseq, const C* tw, LD ld, ST st) {
  const AxisPass& p = pl.pass[g];
  const int nt = pl.ntab;
  switch (8 * p.r1 + p.r2) {
    case 8 * 2 + 1: pass_r<C, 2, 1, INV, SEQFAST>(p, nt, nseq, dseq, tw, ld, st); break;
    case 8 * 3 + 1: pass_r<C, 3, 1, INV, SEQFAST>(p, nt, nseq, dseq, tw, ld, st); break;
    case 8 * 4 + 1: pass_r<C, 4, 1, INV, SEQFAST>(p, nt, nseq, dseq, tw, ld, st); break;
    case 8 * 2 + 3: pass_r<C, 2, 3, INV, SEQFAST>(p, nt, nseq, dseq, tw, ld, st); break;
    case 8 * 3 + 3: pass_r<C, 3, 3, INV, SEQFAST>(p, nt, nseq, dseq, tw, ld, st); break;
    case 8 * 4 + 2: pass_r<C, 4, 2, INV, SEQFAST>(p, nt, nseq, dseq, tw, ld, st); break;
    case 8 * 4 + 3: pass_r<C, 4, 3, INV, SEQFAST>(p, nt, nseq, dseq, tw, ld, st); break;
    default: pass_r<C, 4, 4, INV, SEQFAST>(p, nt, nseq, dseq, tw, ld, st); break;
  }
}

// Row pitch of a plane in shared memory: odd, so that rows fall in different banks.
__host__ __device__ __forceinline__ int pitch(int nx) { return nx | 1; }

template <typename C>
__device__ __forceinline__ void load_tables(C* twx, C* twy, int* posx, const XYArgs& a) {
  const C* gx = reinterpret_cast<const C*>(a.twx);
  const C* gy = reinterpret_cast<const C*>(a.twy);
  for (int i = threadIdx.x; i < a.nx; i += blockDim.x) { twx[i] = gx[i]; posx[i] = a.xpos[i]; }
  for (int i = threadIdx.x; i < a.ny; i += blockDim.x) twy[i] = gy[i];
}

// Forward x-y transform of one (c, z) plane per block.
// Registers: 64 a thread in FP32 (two blocks of 512 an SM; the inverse pass
// spills 80 to 220 bytes for them), 128 in FP64.
template <typename T> __host__ __device__ constexpr int xy_min_blocks() { return sizeof(T) == 4 ? 2 : 1; }

template <typename T>
__global__ void __launch_bounds__(512, xy_min_blocks<T>()) k_xyf(const T* __restrict__ in, typename CT<T>::t* __restrict__ spec, XYArgs a) {
  typedef typename CT<T>::t C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nx = a.nx, ny = a.ny, hy = ny / 2, hx = nx / 2, PX = pitch(nx);
  C* buf = reinterpret_cast<C*>(smem_raw);
  C* twx = buf + hy * PX;
  C* twy = twx + nx;
  int* posx = reinterpret_cast<int*>(twy + ny);
  load_tables(twx, twy, posx, a);   // constant: before the wait for the predecessor
  pdl_wait();
  // the stop flag is read by one thread (a read per warp makes its L2 line a
  // queue) and tested after the first barrier behind the plane's loads
  // (nothing is written before), and the first pass reads its twiddles from
  // global memory: the loads wait neither for the flag nor for the tables
  __shared__ int s_stop;
  if (threadIdx.x == 0) s_stop = a.skip ? *(volatile const int*)a.skip : 0;
  const int c = blockIdx.x % 9, z = blockIdx.x / 9;
  const T* src = in + c * a.N + (long long)z * ny * nx;
  const int ext = hy * PX, half = hy * nx;
  (void)ext;
  // x: rows q and q + ny/2 as one complex row; the first pass reads the two
  // real rows along themselves
  pass<C, false, false>(a.px, 0, hy, a.dhy, reinterpret_cast<const C*>(a.twx),
                        [&](int q, int e) {
                          const int i = MF_AT(q * nx + e, half);
                          return cmake(src[i], src[i + half]);
                        },
                        [&](int q, int e, C v) { buf[MF_AT(q * PX + e, ext)] = v; });
  __syncthreads();
  if (s_stop) return;
  for (int g = 1; g < a.px.npass; ++g) {
    pass<C, false, true>(a.px, g, hy, a.dhy, twx, [&](int q, int e) { return buf[MF_AT(q * PX + e, ext)]; },
                         [&](int q, int e, C v) { buf[MF_AT(q * PX + e, ext)] = v; });
    __syncthreads();
  }
  // split the packed rows into the spectra of rows q and q + ny/2, and apply
  // the first (radix-2) stage of the y transform, which combines those two
  for (int idx = threadIdx.x; idx < hy * hx; idx += blockDim.x) {
    const int k = fdiv(idx, a.dhy), q = idx - k * hy;
    C* row = buf + MF_AT(q * PX, ext - nx + 1);
    const int sa = posx[MF_AT(k, nx)], sb = posx[MF_AT(k == 0 ? hx : nx - k, nx)];
    const C za = row[sa], zb = row[sb];
    C xa, xb;
    if (k == 0) {
      xa = cmake(za.x, (T)0);
      xb = cmake(za.y, (T)0);
    } else {
      xa = cmake((T)0.5 * (za.x + zb.x), (T)0.5 * (za.y - zb.y));
      xb = cmake((T)0.5 * (za.y + zb.y), (T)-0.5 * (za.x - zb.x));
    }
    row[sa] = cadd(xa, xb);
    row[sb] = cmul(csub(xa, xb), twy[MF_AT(q, ny)]);
  }
  __syncthreads();
  // remaining y stages: nx columns of ny/2 samples; the last pass stores the spectrum
  for (int g = 0; g + 1 < a.py.npass; ++g) {
    pass<C, false, true>(a.py, g, nx, a.dnx, twy, [&](int q, int e) { return buf[MF_AT(e * PX + q, ext)]; },
                         [&](int q, int e, C v) { buf[MF_AT(e * PX + q, ext)] = v; });
    __syncthreads();
  }
  C* dst = spec + ((long long)c * a.nz + z) * half;
  pass<C, false, true>(a.py, a.py.npass - 1, nx, a.dnx, twy, [&](int q, int e) { return buf[MF_AT(e * PX + q, ext)]; },
                       [&](int q, int e, C v) { dst[MF_AT(e * nx + q, half)] = v; });
}

// Sum of squares of FP32 values: each square exactly as a product and its
// remainder, summed in three FP32 words with the errors of the first two
// carried on.  After n terms it is within n^3 2^-72 of the exact sum, below
// FP64 accumulation's n 2^-53 for the at most 200 terms of a thread (measured
// over 2 .. 200 terms: 1.1e-16 against 2.2e-15; two words: 2.2e-13), as long as
// the squares stay in range: the caller scales its values to about 1 by a
// power of two and takes FP64 where that fails.  FP64 for every value would
// take its pipe 20 us of a 108^3 cell's CG iteration (inverse pass 76 against
// 55 us; 72^3 24.6 against 14.9).
struct SumSq {
  float s = 0.f, c = 0.f, d = 0.f;
  static __device__ __forceinline__ float two_sum(float& a, float b) {   // a += b, returns the error
    const float t = __fadd_rn(a, b), bb = __fsub_rn(t, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(t, bb)), __fsub_rn(b, bb));
    a = t;
    return e;
  }
  __device__ __forceinline__ void add(float v) {
    const float p = __fmul_rn(v, v);
    const float e1 = two_sum(s, p), e2 = two_sum(c, e1), e3 = two_sum(c, __fmaf_rn(v, v, -p));
    d = __fadd_rn(d, __fadd_rn(e2, e3));
  }
  __device__ __forceinline__ double value() const { return (double)s + ((double)c + (double)d); }
};

// Power of two that brings values of mean square rr / n to about 1 (1 when rr
// is zero or no finite number).
__device__ __forceinline__ float unit_scale(double rr, int n) {
  const int field = (__double2hiint(rr) >> 20) & 0x7ff;
  if (field == 0 || field == 0x7ff) return 1.f;
  int k = -((field - 1023 - (31 - __clz(n))) >> 1);
  k = k < -100 ? -100 : (k > 100 ? 100 : k);
  return __int_as_float((127 + k) << 23);
}
__device__ __forceinline__ double unit_squared_inverse(float unit) {
  return __hiloint2double((1023 - 2 * ((__float_as_int(unit) >> 23) - 127)) << 20, 0);
}

// Inverse x-y transform of one (c, z) plane per block.  MODE 0: out[c] = y.
// MODE 3: out[c] -= alpha y (alpha from sc), partial sum out^2; with a.fin
// the last block to finish sums the partials and updates beta, r.r and the
// stop flag.
template <typename T, int MODE>
__global__ void __launch_bounds__(512, xy_min_blocks<T>()) k_xyi(const typename CT<T>::t* __restrict__ spec, T* __restrict__ out,
                                             double* __restrict__ partials, XYArgs a, Scalars* sc) {
  typedef typename CT<T>::t C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[32];
  const int nx = a.nx, ny = a.ny, hy = ny / 2, hx = nx / 2, PX = pitch(nx);
  C* buf = reinterpret_cast<C*>(smem_raw);
  C* twx = buf + hy * PX;
  C* twy = twx + nx;
  int* posx = reinterpret_cast<int*>(twy + ny);
  load_tables(twx, twy, posx, a);   // constant: before the wait for the predecessor
  pdl_wait();
  // (see k_xyf); alpha is needed at the end
  __shared__ int s_stop;
  __shared__ T s_alpha;
  __shared__ float s_unit;
  __shared__ CgScalars s_cg;
  if (threadIdx.x == 0) {
    s_stop = a.skip ? *(volatile const int*)a.skip : 0;
    if (MODE == 3) {
      s_alpha = (T)sc->alpha;
      if (a.fin) s_cg.load(sc);
      if (sizeof(T) == 4) s_unit = unit_scale(sc->rr, (int)(9 * a.N));   // r has not moved far from the last r.r
    }
  }
  const int c = blockIdx.x % 9, z = blockIdx.x / 9;
  const int ext = hy * PX, half = hy * nx;
  (void)ext;
  T* dst = out + c * a.N + (long long)z * ny * nx;
  const C* src = spec + ((long long)c * a.nz + z) * half;
  if (MODE == 3) {
    // the residual plane is read only at the end: start pulling it into L2 now
    const char* rp = reinterpret_cast<const char*>(dst);
    for (int i = threadIdx.x * 128; i < ny * nx * (int)sizeof(T); i += blockDim.x * 128)
      asm volatile("prefetch.global.L2 [%0];" ::"l"(rp + i));
  }
  // y: the first inverse pass reads the spectrum
  pass<C, true, true>(a.py, a.py.npass - 1, nx, a.dnx, reinterpret_cast<const C*>(a.twy),
                      [&](int q, int e) { return src[MF_AT(e * nx + q, half)]; },
                      [&](int q, int e, C v) { buf[MF_AT(e * PX + q, ext)] = v; });
  __syncthreads();
  if (s_stop) return;
  for (int g = a.py.npass - 2; g >= 0; --g) {
    pass<C, true, true>(a.py, g, nx, a.dnx, twy, [&](int q, int e) { return buf[MF_AT(e * PX + q, ext)]; },
                        [&](int q, int e, C v) { buf[MF_AT(e * PX + q, ext)] = v; });
    __syncthreads();
  }
  for (int idx = threadIdx.x; idx < hy * hx; idx += blockDim.x) {
    const int k = fdiv(idx, a.dhy), q = idx - k * hy;
    C* row = buf + MF_AT(q * PX, ext - nx + 1);
    const int sa = posx[MF_AT(k, nx)], sb = posx[MF_AT(k == 0 ? hx : nx - k, nx)];
    const C y0 = row[sa];
    const C t = cmulc(row[sb], twy[MF_AT(q, ny)]);
    const C xa = cadd(y0, t), xb = csub(y0, t);
    if (k == 0) {
      row[sa] = cmake(xa.x, xb.x);
      row[sb] = cmake((T)0, (T)0);
    } else {
      row[sa] = cmake(xa.x - xb.y, xa.y + xb.x);
      row[sb] = cmake(xa.x + xb.y, xb.x - xa.y);
    }
  }
  __syncthreads();
  for (int g = a.px.npass - 1; g >= 1; --g) {
    pass<C, true, true>(a.px, g, hy, a.dhy, twx, [&](int q, int e) { return buf[MF_AT(q * PX + e, ext)]; },
                        [&](int q, int e, C v) { buf[MF_AT(q * PX + e, ext)] = v; });
    __syncthreads();
  }
  auto sload = [&](int q, int e) { return buf[MF_AT(q * PX + e, ext)]; };
  if (MODE == 3) {
    // the read-modify-write of r in whole rows: a butterfly step of the last
    // pass covers only part of a row
    pass<C, true, true>(a.px, 0, hy, a.dhy, twx, sload, [&](int q, int e, C v) { buf[MF_AT(q * PX + e, ext)] = v; });
    __syncthreads();
    double acc = 0.0;
    SumSq sq;
    float unit = 1.f;
    if constexpr (sizeof(T) == 4) unit = s_unit;
    auto add2 = [&](T v) {
      if constexpr (sizeof(T) == 4) sq.add(unit * v);
      else acc += (double)v * (double)v;
    };
    const T alpha = s_alpha;
    constexpr int kAhead = 4;   // pairs of r in flight per thread
    for (int i0 = threadIdx.x; i0 < half; i0 += kAhead * blockDim.x) {
      T ra[kAhead], rb[kAhead];
#pragma unroll
      for (int k = 0; k < kAhead; ++k) {
        const int i = i0 + k * blockDim.x;
        if (i < half) { ra[k] = dst[i]; rb[k] = dst[i + half]; }
      }
#pragma unroll
      for (int k = 0; k < kAhead; ++k) {
        const int i = i0 + k * blockDim.x;
        if (i < half) {
          const int q = fdiv(i, a.dnx);
          const C v = buf[MF_AT(q * PX + i - q * nx, ext)];
          const T r0 = ra[k] - alpha * v.x, r1 = rb[k] - alpha * v.y;
          dst[i] = r0;
          dst[i + half] = r1;
          add2(r0);
          add2(r1);
        }
      }
    }
    if constexpr (sizeof(T) == 4) {
      acc = sq.value() * unit_squared_inverse(unit);
      if (!(sq.s >= 0x1p-70f && sq.s <= 0x1p127f)) {
        // far from the last r.r (or zero, or no finite number): the same sum in FP64
        acc = 0.0;
        for (int i = threadIdx.x; i < half; i += blockDim.x)
          acc += (double)dst[i] * (double)dst[i] + (double)dst[i + half] * (double)dst[i + half];
      }
    }
    acc = block_total(acc, red);
    if (threadIdx.x == 0) partials[blockIdx.x] = acc;
    if (a.fin) {
      double rr;
      if (last_block_total(partials, &sc->arrive, &rr) && threadIdx.x == 0) cg_finish_beta(rr, s_cg, sc);
    }
  } else {
    pass<C, true, false>(a.px, 0, hy, a.dhy, twx, sload, [&](int q, int e, C v) {
      const int i = MF_AT(q * nx + e, half);
      dst[i] = v.x;
      dst[i + half] = v.y;
    });
  }
}

// z-pass: one row group (components 3g, 3g+1, 3g+2, the three that
// G-hat-star mixes, Eq. eq:Gnewnew) of S consecutive columns per block;
// transform along z, G-hat-star, inverse transform.  MODE 0: operator (with
// a.lin, the null-frequency coefficient / N times *a.lin_alpha added to
// a.lin).  MODE 1: residual (adds a.add at the null frequency and records the
// null-frequency coefficient / N in a.mean_out).  Element (component cl,
// position z, column s) lives at cl * CP + z * ZS + s.
template <typename T> struct ZPad {
  static __host__ __device__ __forceinline__ int zs(int S) { return S + (sizeof(T) == 4 ? 1 : 0); }
  static __host__ __device__ __forceinline__ int cp(int nz, int S) { return nz * zs(S) + 1; }
};

template <typename T, int MODE, int S>
__global__ void __launch_bounds__(256) k_zp(typename CT<T>::t* __restrict__ spec, ZArgs a) {
  typedef typename CT<T>::t C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nx = a.nx, ny = a.ny, nz = a.nz, ncol = (ny / 2) * nx;
  const int ZS = ZPad<T>::zs(S), CP = ZPad<T>::cp(nz, S);
  C* buf = reinterpret_cast<C*>(smem_raw);   // [3][CP]
  C* twz = buf + 3 * CP;
  T* xiz = reinterpret_cast<T*>(twz + nz);   // k_z / n_z (signed) of each position
  int* zk = reinterpret_cast<int*>(xiz + nz);
  const C* gtwz = reinterpret_cast<const C*>(a.twz);
  for (int i = threadIdx.x; i < nz; i += blockDim.x) {
    twz[i] = gtwz[i];
    const int kz = a.zk[i];
    zk[i] = kz;
    xiz[i] = (T)((2 * kz < nz) ? kz : kz - nz) / (T)nz;
  }
  pdl_wait();
  __shared__ int s_stop;   // tested after the first barrier (see k_xyf)
  if (threadIdx.x == 0) s_stop = a.skip ? *(volatile const int*)a.skip : 0;
  const int ntile = (ncol + S - 1) / S;
  const int g = blockIdx.x / ntile;
  const int col0 = (blockIdx.x - g * ntile) * S;
  const int ns = ncol - col0 < S ? ncol - col0 : S;   // columns of the last tile
  const int ext = 3 * CP;
  (void)ext;
  C* gsp = spec + (long long)(3 * g) * nz * ncol + col0;
  // sequence q = cl * S + s; the columns past the last one hold zeros
  auto gld = [&](int q, int z) {
    const int cl = q / S, s = q % S;
    return s < ns ? gsp[((long long)cl * nz + MF_AT(z, nz)) * ncol + s] : cmake((T)0, (T)0);
  };
  auto gst = [&](int q, int z, C v) {
    const int cl = q / S, s = q % S;
    if (s < ns) gsp[((long long)cl * nz + MF_AT(z, nz)) * ncol + s] = v;
  };
  auto sld = [&](int q, int z) { return buf[MF_AT((q / S) * CP + z * ZS + q % S, ext)]; };
  auto sst = [&](int q, int z, C v) { buf[MF_AT((q / S) * CP + z * ZS + q % S, ext)] = v; };
  constexpr int NSEQ = 3 * S;
  const FastDiv dseq = a.dseq;
  pass<C, false, true>(a.pz, 0, NSEQ, dseq, gtwz, gld, sst);
  __syncthreads();
  if (s_stop) return;
  for (int p = 1; p < a.pz.npass; ++p) {
    pass<C, false, true>(a.pz, p, NSEQ, dseq, twz, sld, sst);
    __syncthreads();
  }
  // G-hat-star: a thread keeps one column (the block is a multiple of S)
  const T scale = (T)a.scale;
  const int s = threadIdx.x % S, col = col0 + s;
  if (s < ns) {
    const int row = fdiv(col, a.dnx), slot = col - row * nx;
    const int kx = a.xk[MF_AT(slot, nx)];
    const int ky = 2 * a.yk[MF_AT(row, ny / 2)] + a.xe[MF_AT(slot, nx)];
    const int kys = (ky < ny / 2) ? ky : ky - ny;
    const T xi0 = (T)kx / (T)nx, xi1 = (T)kys / (T)ny;
    for (int p = threadIdx.x / S; p < nz; p += blockDim.x / S) {
      const int kz = zk[p];
      C* e = buf + MF_AT(p * ZS + s, ext - 2 * CP);
      if (2 * ky == ny || 2 * kz == nz) {
#pragma unroll
        for (int cl = 0; cl < 3; ++cl) e[cl * CP] = cmake((T)0, (T)0);
      } else if (kx == 0 && ky == 0 && kz == 0) {
#pragma unroll
        for (int cl = 0; cl < 3; ++cl) {
          const int cc = 3 * g + cl;
          const C X = e[cl * CP];
          if (MODE == 1 && a.mean_out) a.mean_out[cc] = (double)X.x / (double)a.N;
          if (MODE == 0 && a.lin) a.lin[cc] += *a.lin_alpha * ((double)X.x / (double)a.N);
          if (a.mask & (1u << cc)) {
            const T add = (MODE == 1) ? (T)(a.add_dev ? a.add_dev[cc] : a.add[cc]) : (T)0;
            e[cl * CP] = cmake(scale * X.x + add, scale * X.y);
          } else {
            e[cl * CP] = cmake((T)0, (T)0);
          }
        }
      } else {
        const T xi2 = xiz[p];
        const T inv = scale / (xi0 * xi0 + xi1 * xi1 + xi2 * xi2);
        const C A0 = e[0], A1 = e[CP], A2 = e[2 * CP];
        C q;
        q.x = (A0.x * xi0 + A1.x * xi1 + A2.x * xi2) * inv;
        q.y = (A0.y * xi0 + A1.y * xi1 + A2.y * xi2) * inv;
        e[0] = cmake(q.x * xi0, q.y * xi0);
        e[CP] = cmake(q.x * xi1, q.y * xi1);
        e[2 * CP] = cmake(q.x * xi2, q.y * xi2);
      }
    }
  }
  __syncthreads();
  for (int p = a.pz.npass - 1; p >= 1; --p) {
    pass<C, true, true>(a.pz, p, NSEQ, dseq, twz, sld, sst);
    __syncthreads();
  }
  pass<C, true, true>(a.pz, 0, NSEQ, dseq, twz, sld, gst);
}

// ---------------------------------------------------------------- launchers
// Threads of a block of a grid of `blocks`, at most one per butterfly
// (`work`): of the counts that run the grid in the fewest waves of resident
// blocks, the largest.  The phases of a block alternate with barriers, so an
// SM wants several blocks, and a last wave of a few blocks costs a whole one:
// 72^3 in FP32 (648 planes) takes 160 us per CG iteration with 352 threads
// (two blocks an SM, 2.1 waves) and 137 us with 192 (five, one wave), 108^3
// 406 us with 512 and 391 us with 256.
inline int pick_threads(int regs, size_t smem, int blocks, int work, int most) {
  work = ((work + 31) / 32) * 32;
  most = work < 64 ? 64 : (work < most ? work : most);
  const int r8 = ((regs + 7) / 8) * 8;
  int best = 64, fewest = 1 << 30;
  for (int t = 64; t <= most; t += 32) {
    int res = 65536 / (r8 * t);
    const int by_smem = (int)(228 * 1024 / (smem + 1024)), by_warps = 2048 / t;
    if (by_smem < res) res = by_smem;
    if (by_warps < res) res = by_warps;
    if (res > 32) res = 32;
    if (res < 1) continue;
    const int waves = (blocks + 152 * res - 1) / (152 * res);
    if (waves <= fewest) { fewest = waves; best = t; }
  }
  return best;
}

// Registers a thread of kernel K, asked for once (the same on every device
// this code runs on); a query that fails is asked again at the next launch.
template <auto K> int regs_of() {
  static std::atomic<int> known{0};
  int n = known.load(std::memory_order_relaxed);
  if (n == 0) {
    cudaFuncAttributes at;
    if (cudaFuncGetAttributes(&at, K) != cudaSuccess) {
      cudaGetLastError();
      return 128;
    }
    n = at.numRegs;
    known.store(n, std::memory_order_relaxed);
  }
  return n;
}

// Values of a butterfly: eight in plans of paired stages, else four.
inline int xy_work(const XYArgs& a) {
  const bool paired = a.px.npass < a.px.nst || a.py.npass < a.py.nst;
  return a.ny * (a.nx / 2) / (paired ? 8 : 4);
}

template <typename T>
size_t xy_smem(const XYArgs& a) {
  typedef typename CT<T>::t C;
  return (size_t)(a.ny / 2) * pitch(a.nx) * sizeof(C) + (size_t)(a.nx + a.ny) * sizeof(C) + (size_t)a.nx * sizeof(int);
}

// The shared-memory opt-in, at every launch that needs one: it belongs to a
// device, and contexts on several devices of a process, and the residual
// without a context on whichever device its caller has current, run these
// kernels.
// Always at the most a plane of any admissible size takes, so that host
// threads launching different sizes set the same value.  Launches that stay
// within the default 48 KB with the kernels' static part (below 1 KB) need
// none: planes up to 72 x 72 in FP64, 108 x 96 in FP32.
constexpr size_t kSmemMax = 226 * 1024, kSmemDefault = 47 * 1024;
template <auto K>
cudaError_t smem_opt_in(size_t sm) {
  if (sm <= kSmemDefault) return cudaSuccess;
  if (sm > kSmemMax) return cudaErrorInvalidValue;
  return cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
}

template <typename T>
cudaError_t xyf(const void* in, void* spec, const XYArgs& a, cudaStream_t st) {
  typedef typename CT<T>::t C;
  const size_t sm = xy_smem<T>(a);
  const cudaError_t e = smem_opt_in<k_xyf<T>>(sm);
  if (e != cudaSuccess) return e;
  ++g_mf_launches;
  const int t = pick_threads(regs_of<k_xyf<T>>(), sm, 9 * a.nz, xy_work(a), 512);
  return launch_k(a.pdl != 0, k_xyf<T>, dim3(9 * a.nz), dim3(t), sm, st, (const T*)in, (C*)spec, a);
}

template <typename T, int MODE>
cudaError_t xyi_m(const void* spec, void* out, double* partials, const XYArgs& a, const Scalars* sc, cudaStream_t st) {
  typedef typename CT<T>::t C;
  const size_t sm = xy_smem<T>(a);
  const cudaError_t e = smem_opt_in<k_xyi<T, MODE>>(sm);
  if (e != cudaSuccess) return e;
  ++g_mf_launches;
  const int t = pick_threads(regs_of<k_xyi<T, MODE>>(), sm, 9 * a.nz, xy_work(a), 512);
  return launch_k(a.pdl != 0, k_xyi<T, MODE>, dim3(9 * a.nz), dim3(t), sm, st, (const C*)spec, (T*)out, partials, a,
                  const_cast<Scalars*>(sc));
}

template <typename T>
cudaError_t xyi(int mode, const void* spec, void* out, double* partials, const XYArgs& a, const Scalars* sc,
                cudaStream_t st) {
  return mode == 3 ? xyi_m<T, 3>(spec, out, partials, a, sc, st) : xyi_m<T, 0>(spec, out, partials, a, sc, st);
}

template <typename T, int MODE, int S>
cudaError_t zp_s(void* spec, ZArgs a, cudaStream_t st) {
  typedef typename CT<T>::t C;
  const size_t sm = (size_t)3 * ZPad<T>::cp(a.nz, S) * sizeof(C) + (size_t)a.nz * (sizeof(C) + sizeof(T) + sizeof(int));
  const cudaError_t e = smem_opt_in<k_zp<T, MODE, S>>(sm);
  if (e != cudaSuccess) return e;
  const int ncol = a.ny * (a.nx / 2);
  a.dseq = fast_div(3 * S);
  const int blocks = 3 * ((ncol + S - 1) / S);
  const int t = pick_threads(regs_of<k_zp<T, MODE, S>>(), sm, blocks, 3 * S * a.nz / (a.pz.npass < a.pz.nst ? 8 : 4), 256);
  ++g_mf_launches;
  return launch_k(a.pdl != 0, k_zp<T, MODE, S>, dim3(blocks), dim3(t), sm, st, (C*)spec, a);
}

// Tile of 8 columns; of 4 when 8 would leave SMs without a block.
template <typename T, int MODE>
cudaError_t zp_m(void* spec, const ZArgs& a, cudaStream_t st) {
  const int ncol = a.ny * (a.nx / 2);
  if (3 * ((ncol + 7) / 8) < 2 * 152) return zp_s<T, MODE, 4>(spec, a, st);
  return zp_s<T, MODE, 8>(spec, a, st);
}

template <typename T>
cudaError_t zp(int mode, void* spec, const ZArgs& a, cudaStream_t st) {
  return mode == 1 ? zp_m<T, 1>(spec, a, st) : zp_m<T, 0>(spec, a, st);
}

}  // namespace trg
