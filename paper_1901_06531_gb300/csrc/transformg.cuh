// Transform kernels for any admissible size (nx, ny even, all of the form
// 2^a 3^b), with the sizes as run-time values: the grids, or the axes of a
// grid, that the fixed-size kernels (transform2.cuh) do not cover.  Three
// kernels per projected operator, like there, on the same spectrum layout
// (half-length real rows; per (c, z) ny rows in digit-reversed ky order of
// nx/2 slots in digit-reversed kx order), so either kind of z-pass follows
// either kind of x-y pass.
//
// A length runs in as few stages as radices 2, 3, 4, 6, 8, 9, 12 and 16
// allow (one to 16, two up to 144 and for most lengths beyond, three for the
// rest), each butterfly in registers, one shared-memory pass per stage; the
// first stage of a pass reads global memory and the last one writes it.  The
// radix of a stage is a switch over unrolled butterflies; the index
// arithmetic that a template constant would fold away is two divisions by
// precomputed reciprocals per butterfly.  What bounds them is the work per
// sample that is not arithmetic: shared-memory passes and indices (FP32), the
// FP64 pipe (FP64).  Against radix-2/3/4 stages with hardware divisions and
// one pass per stage (108 = 4 x 3 x 3 x 3 took four, 12 x 9 takes two) the
// FP32 operator on 108 x 72 x 54 went from 125.5 to 74.5 us, stress and
// residual in FP64 on 48 x 36 x 18 from 184 to 146 us.
#pragma once

#include "fft2.cuh"
#include "launch.h"

namespace fft2 {

// Radices 6 and 12 by the prime-factor map (coprime factors: no twiddles),
// radix 9 as 3 x 3 with the twiddles W_9^(n2 k1).
template <bool INV, typename C> struct Dft<6, INV, C> {
  static __device__ __forceinline__ void run(C* v) {
    // n = 3 n1 + 2 n2, k = 3 k1 + 4 k2 (mod 6), n1, k1 < 2, n2, k2 < 3
    C a[3] = {v[0], v[2], v[4]}, b[3] = {v[3], v[5], v[1]};
    Dft<3, INV, C>::run(a);
    Dft<3, INV, C>::run(b);
    v[0] = cadd(a[0], b[0]); v[3] = csub(a[0], b[0]);
    v[4] = cadd(a[1], b[1]); v[1] = csub(a[1], b[1]);
    v[2] = cadd(a[2], b[2]); v[5] = csub(a[2], b[2]);
  }
};

template <bool INV, typename C> struct Dft<12, INV, C> {
  static __device__ __forceinline__ void run(C* v) {
    // n = 4 n1 + 3 n2, k = 4 k1 + 9 k2 (mod 12), n1, k1 < 3, n2, k2 < 4
    C t[4][3];
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) {
#pragma unroll
      for (int n1 = 0; n1 < 3; ++n1) t[n2][n1] = v[(4 * n1 + 3 * n2) % 12];
      Dft<3, INV, C>::run(t[n2]);
    }
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) {
      C u[4] = {t[0][k1], t[1][k1], t[2][k1], t[3][k1]};
      Dft<4, INV, C>::run(u);
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) v[(4 * k1 + 9 * k2) % 12] = u[k2];
    }
  }
};

// v * W_9^E (forward) or v * conj(W_9^E) (inverse), E in {1, 2, 4}
template <int E, bool INV, typename C>
__device__ __forceinline__ C tw9(C v) {
  typedef decltype(v.x) T;
  constexpr double c9 = E == 1 ? 0.76604444311897803520 : E == 2 ? 0.17364817766693034885 : -0.93969262078590838405;
  constexpr double s9 = E == 1 ? 0.64278760968653932632 : E == 2 ? 0.98480775301220805937 : 0.34202014332566873304;
  C w;
  w.x = (T)c9;
  w.y = (T)-s9;
  return INV ? cmulc(v, w) : cmul(v, w);
}

template <bool INV, typename C> struct Dft<9, INV, C> {
  static __device__ __forceinline__ void run(C* v) {
    // n = 3 n1 + n2, k = k1 + 3 k2
    C t[3][3];
#pragma unroll
    for (int n2 = 0; n2 < 3; ++n2) {
#pragma unroll
      for (int n1 = 0; n1 < 3; ++n1) t[n2][n1] = v[3 * n1 + n2];
      Dft<3, INV, C>::run(t[n2]);
    }
    t[1][1] = tw9<1, INV>(t[1][1]);
    t[1][2] = tw9<2, INV>(t[1][2]);
    t[2][1] = tw9<2, INV>(t[2][1]);
    t[2][2] = tw9<4, INV>(t[2][2]);
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) {
      C u[3] = {t[0][k1], t[1][k1], t[2][k1]};
      Dft<3, INV, C>::run(u);
#pragma unroll
      for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = u[k2];
    }
  }
};

}  // namespace fft2

namespace trg {

// Quotient by a run-time divisor through its reciprocal (exact for t < 2^16
// and d <= 2^15, which bounds every index below).
__device__ __forceinline__ int fdiv(int t, FastDiv f) {
  return f.d == 1 ? t : (int)__umulhi((unsigned)t, f.m);
}

// One stage of radix R over nseq sequences: inputs from ld(q, e), outputs to
// st(q, e, value), e the position along sequence q.  SEQFAST: consecutive
// threads take consecutive sequences (else consecutive butterflies of one).
template <typename C, int R, bool INV, bool SEQFAST, typename LD, typename ST>
__device__ __forceinline__ void stage_r(const AxisPlan& p, int s, int nseq, FastDiv dseq, const C* tw, LD ld, ST st) {
  const int M = p.m[s], nb = p.nb[s].d, total = nseq * nb, ts = p.tstep[s];
  for (int t = threadIdx.x; t < total; t += blockDim.x) {
    int q, b;
    if (SEQFAST) { b = fdiv(t, dseq); q = t - b * nseq; } else { q = fdiv(t, p.nb[s]); b = t - q * nb; }
    const int blk = fdiv(b, p.dm[s]);
    const int j0 = b - blk * M;
    const int e0 = blk * M * R + j0;
    C v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = ld(q, e0 + r * M);
    if (!INV) {
      fft2::Dft<R, false, C>::run(v);
      if (M > 1) {
#pragma unroll
        for (int k = 1; k < R; ++k) v[k] = cmul(v[k], tw[MF_AT(j0 * k * ts, p.ntab)]);
      }
    } else {
      if (M > 1) {
#pragma unroll
        for (int k = 1; k < R; ++k) v[k] = cmulc(v[k], tw[MF_AT(j0 * k * ts, p.ntab)]);
      }
      fft2::Dft<R, true, C>::run(v);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) st(q, e0 + r * M, v[r]);
  }
}

template <typename C, bool INV, bool SEQFAST, typename LD, typename ST>
__device__ __forceinline__ void stage(const AxisPlan& p, int s, int nseq, FastDiv dseq, const C* tw, LD ld, ST st) {
  switch (p.rad[s]) {
    case 2: stage_r<C, 2, INV, SEQFAST>(p, s, nseq, dseq, tw, ld, st); break;
    case 3: stage_r<C, 3, INV, SEQFAST>(p, s, nseq, dseq, tw, ld, st); break;
    case 4: stage_r<C, 4, INV, SEQFAST>(p, s, nseq, dseq, tw, ld, st); break;
    case 6: stage_r<C, 6, INV, SEQFAST>(p, s, nseq, dseq, tw, ld, st); break;
    case 8: stage_r<C, 8, INV, SEQFAST>(p, s, nseq, dseq, tw, ld, st); break;
    case 9: stage_r<C, 9, INV, SEQFAST>(p, s, nseq, dseq, tw, ld, st); break;
    case 12: stage_r<C, 12, INV, SEQFAST>(p, s, nseq, dseq, tw, ld, st); break;
    default: stage_r<C, 16, INV, SEQFAST>(p, s, nseq, dseq, tw, ld, st); break;
  }
}

// Row pitch of a plane in shared memory: odd, so that rows fall in different banks.
__host__ __device__ __forceinline__ int pitch(int h) { return h | 1; }

// X_k = E_k + W_nx^k O_k, E_k = (Z_k + conj Z_(H-k)) / 2, O_k = (Z_k - conj Z_(H-k)) / 2i
template <typename T, typename C>
__device__ __forceinline__ C split_one(C za, C zb, C w) {
  C e, o;
  e.x = (T)0.5 * (za.x + zb.x); e.y = (T)0.5 * (za.y - zb.y);
  o.x = (T)0.5 * (za.y + zb.y); o.y = (T)-0.5 * (za.x - zb.x);
  return cadd(e, cmul(o, w));
}

// Z_k = E_k + i O_k, E_k = X_k + conj X_(H-k), O_k = (X_k - conj X_(H-k)) conj(W_nx^k)
// (the adjoint of the split, times 2)
template <typename T, typename C>
__device__ __forceinline__ C merge_one(C xa, C xb, C w) {
  C e, d;
  e.x = xa.x + xb.x; e.y = xa.y - xb.y;
  d.x = xa.x - xb.x; d.y = xa.y + xb.y;
  const C o = cmulc(d, w);
  C z;
  z.x = e.x - o.y; z.y = e.y + o.x;
  return z;
}

template <typename C>
__device__ __forceinline__ void load_tables(C* twx, C* twy, int* posx, const XYArgs& a) {
  const C* gx = reinterpret_cast<const C*>(a.twx);
  const C* gy = reinterpret_cast<const C*>(a.twy);
  for (int i = threadIdx.x; i < a.nx; i += blockDim.x) twx[i] = gx[i];
  for (int i = threadIdx.x; i < a.ny; i += blockDim.x) twy[i] = gy[i];
  for (int i = threadIdx.x; i < a.nx / 2; i += blockDim.x) posx[i] = a.xpos[i];
}

// Forward x-y transform of one (c, z) plane per block.  wide: the field is
// aligned to a complex sample (it may be a caller's).
template <typename T>
__global__ void __launch_bounds__(512) k_xyf(const T* __restrict__ in, typename CT<T>::t* __restrict__ spec, XYArgs a,
                                             int wide) {
  typedef typename CT<T>::t C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nx = a.nx, ny = a.ny, H = nx / 2, PX = pitch(H);
  C* buf = reinterpret_cast<C*>(smem_raw);
  C* twx = buf + ny * PX;
  C* twy = twx + nx;
  int* posx = reinterpret_cast<int*>(twy + ny);
  load_tables(twx, twy, posx, a);   // constant: before the wait for the predecessor
  pdl_wait();
  if (a.skip && *(volatile const int*)a.skip) return;
  const int c = blockIdx.x % 9, z = blockIdx.x / 9;
  const T* src1 = in + c * a.N + (long long)z * ny * nx;
  const C* src = reinterpret_cast<const C*>(src1);
  auto gload = [&](int q, int e) {
    const int i = MF_AT(q * H + e, ny * H);
    return wide ? src[i] : cmake(src1[2 * i], src1[2 * i + 1]);
  };
  const int ext = ny * PX;
  (void)ext;
  __syncthreads();   // tables
  // x: rows of H samples; the first stage reads global memory along the rows
  stage<C, false, false>(a.px, 0, ny, a.dny, twx, gload, [&](int q, int e, C v) { buf[MF_AT(q * PX + e, ext)] = v; });
  for (int s = 1; s < a.px.nst; ++s) {
    __syncthreads();
    stage<C, false, true>(a.px, s, ny, a.dny, twx, [&](int q, int e) { return buf[MF_AT(q * PX + e, ext)]; },
                          [&](int q, int e, C v) { buf[MF_AT(q * PX + e, ext)] = v; });
  }
  __syncthreads();
  const int np = H / 2 + 1;
  for (int idx = threadIdx.x; idx < ny * np; idx += blockDim.x) {
    const int k = fdiv(idx, a.dny), y = idx - k * ny;
    const int km = k == 0 ? 0 : H - k;
    C* row = buf + MF_AT(y * PX, ext - H + 1);
    const int pa = posx[MF_AT(k, H)], pb = posx[MF_AT(km, H)];
    const C za = row[pa], zb = row[pb];
    if (km != k) row[pb] = split_one<T>(zb, za, twx[km]);
    row[pa] = split_one<T>(za, zb, twx[k]);
  }
  __syncthreads();
  // y: H columns of ny samples; the last stage stores the spectrum rows
  for (int s = 0; s + 1 < a.py.nst; ++s) {
    stage<C, false, true>(a.py, s, H, a.dh, twy, [&](int q, int e) { return buf[MF_AT(e * PX + q, ext)]; },
                          [&](int q, int e, C v) { buf[MF_AT(e * PX + q, ext)] = v; });
    __syncthreads();
  }
  C* dst = spec + ((long long)c * a.nz + z) * ny * H;
  stage<C, false, true>(a.py, a.py.nst - 1, H, a.dh, twy, [&](int q, int e) { return buf[MF_AT(e * PX + q, ext)]; },
                        [&](int q, int e, C v) { dst[MF_AT(e * H + q, ny * H)] = v; });
}

// Inverse x-y transform of one (c, z) plane per block.  MODE 0: out[c] = y.
// MODE 3: out[c] -= alpha y (alpha from sc), partial sum out^2; with a.fin
// the last block to finish sums the partials and updates beta, r.r and the
// stop flag.
template <typename T, int MODE>
__global__ void __launch_bounds__(512) k_xyi(const typename CT<T>::t* __restrict__ spec, T* __restrict__ out,
                                             double* __restrict__ partials, XYArgs a, Scalars* sc, int wide) {
  typedef typename CT<T>::t C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[32];
  const int nx = a.nx, ny = a.ny, H = nx / 2, PX = pitch(H);
  C* buf = reinterpret_cast<C*>(smem_raw);
  C* twx = buf + ny * PX;
  C* twy = twx + nx;
  int* posx = reinterpret_cast<int*>(twy + ny);
  load_tables(twx, twy, posx, a);   // constant: before the wait for the predecessor
  pdl_wait();
  if (a.skip && *(volatile const int*)a.skip) return;
  const int c = blockIdx.x % 9, z = blockIdx.x / 9;
  const int ext = ny * PX;
  (void)ext;
  T* dst1 = out + c * a.N + (long long)z * ny * nx;
  C* dst = reinterpret_cast<C*>(dst1);
  const C* src = spec + ((long long)c * a.nz + z) * ny * H;
  __syncthreads();   // tables
  // y: the first inverse stage reads the spectrum rows
  stage<C, true, true>(a.py, a.py.nst - 1, H, a.dh, twy, [&](int q, int e) { return src[MF_AT(e * H + q, ny * H)]; },
                       [&](int q, int e, C v) { buf[MF_AT(e * PX + q, ext)] = v; });
  for (int s = a.py.nst - 2; s >= 0; --s) {
    __syncthreads();
    stage<C, true, true>(a.py, s, H, a.dh, twy, [&](int q, int e) { return buf[MF_AT(e * PX + q, ext)]; },
                         [&](int q, int e, C v) { buf[MF_AT(e * PX + q, ext)] = v; });
  }
  __syncthreads();
  const int np = H / 2 + 1;
  for (int idx = threadIdx.x; idx < ny * np; idx += blockDim.x) {
    const int k = fdiv(idx, a.dny), y = idx - k * ny;
    const int km = k == 0 ? 0 : H - k;
    C* row = buf + MF_AT(y * PX, ext - H + 1);
    const int pa = posx[MF_AT(k, H)], pb = posx[MF_AT(km, H)];
    const C xa = row[pa], xb = row[pb];
    if (k == 0) {
      // the x-constant coefficient keeps only its real part and X_H (Nyquist) is zero
      row[pa] = cmake(xa.x, xa.x);
      continue;
    }
    if (km != k) row[pb] = merge_one<T>(xb, xa, twx[km]);
    row[pa] = merge_one<T>(xa, xb, twx[k]);
  }
  __syncthreads();
  for (int s = a.px.nst - 1; s >= 1; --s) {
    stage<C, true, true>(a.px, s, ny, a.dny, twx, [&](int q, int e) { return buf[MF_AT(q * PX + e, ext)]; },
                         [&](int q, int e, C v) { buf[MF_AT(q * PX + e, ext)] = v; });
    __syncthreads();
  }
  // per-thread sums: FP64 for FP64 data; for FP32 data exact FP32 products
  // with Neumaier-compensated FP32 accumulation, combined in FP64 below
  double acc = 0.0;
  float fs = 0.f, fc = 0.f;
  auto fadd = [&](float v) {
    const float tt = fs + v;
    fc += (fabsf(fs) >= fabsf(v)) ? ((fs - tt) + v) : ((v - tt) + fs);
    fs = tt;
  };
  auto fsq = [&](float v) {
    const float p = v * v;
    fadd(p);
    fadd(fmaf(v, v, -p));
  };
  T alpha = (T)0;
  if (MODE == 3) alpha = (T)sc->alpha;
  auto emit = [&](int i, C v) {
    i = MF_AT(i, ny * H);
    if constexpr (MODE == 3) {
      C r = dst[i];
      r.x -= alpha * v.x;
      r.y -= alpha * v.y;
      dst[i] = r;
      if (sizeof(T) == 4) { fsq((float)r.x); fsq((float)r.y); }
      else acc += (double)r.x * (double)r.x + (double)r.y * (double)r.y;
    } else {
      if (wide) dst[i] = v;
      else { dst1[2 * i] = v.x; dst1[2 * i + 1] = v.y; }
    }
  };
  auto sload = [&](int q, int e) { return buf[MF_AT(q * PX + e, ext)]; };
  if (MODE == 3) {
    // the read-modify-write of r in whole rows: a butterfly step of the last
    // stage covers only H / R consecutive samples of a row
    stage<C, true, true>(a.px, 0, ny, a.dny, twx, sload, [&](int q, int e, C v) { buf[MF_AT(q * PX + e, ext)] = v; });
    __syncthreads();
#pragma unroll 4
    for (int idx = threadIdx.x; idx < ny * H; idx += blockDim.x) {
      const int y = fdiv(idx, a.dh);
      emit(idx, buf[MF_AT(y * PX + idx - y * H, ext)]);
    }
    if (sizeof(T) == 4) acc = (double)fs + (double)fc;
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
      double s = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : 0.0;
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (threadIdx.x == 0) partials[blockIdx.x] = s;
    }
    if (a.fin) {
      double rr;
      if (last_block_total(partials, &sc->arrive, &rr) && threadIdx.x == 0) cg_finish_beta(rr, sc);
    }
  } else {
    stage<C, true, false>(a.px, 0, ny, a.dny, twx, sload, [&](int q, int e, C v) { emit(q * H + e, v); });
  }
}

// z-pass: one row group (components 3g, 3g+1, 3g+2, the three that
// G-hat-star mixes, Eq. eq:Gnewnew) of S consecutive (ky, kx) columns per
// block; transform along z, G-hat-star, inverse transform.  MODE 0: operator
// (with a.lin, the null-frequency coefficient / N times *a.lin_alpha added to
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
  const int nz = a.nz, H = a.nx / 2, ncol = a.ny * H;
  const int ZS = ZPad<T>::zs(S), CP = ZPad<T>::cp(nz, S);
  C* buf = reinterpret_cast<C*>(smem_raw);   // [3][CP]
  C* twz = buf + 3 * CP;
  int* zk = reinterpret_cast<int*>(twz + nz);
  const C* gtwz = reinterpret_cast<const C*>(a.twz);
  for (int i = threadIdx.x; i < nz; i += blockDim.x) { twz[i] = gtwz[i]; zk[i] = a.zk[i]; }
  pdl_wait();
  if (a.skip && *(volatile const int*)a.skip) return;
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
  __syncthreads();   // tables
  stage<C, false, true>(a.pz, 0, NSEQ, dseq, twz, gld, sst);
  __syncthreads();
  for (int s = 1; s < a.pz.nst; ++s) {
    stage<C, false, true>(a.pz, s, NSEQ, dseq, twz, sld, sst);
    __syncthreads();
  }
  const T scale = (T)a.scale;
  const T rnx = (T)1 / (T)a.nx, rny = (T)1 / (T)a.ny, rnz = (T)1 / (T)nz;
  for (int idx = threadIdx.x; idx < nz * S; idx += blockDim.x) {
    const int s = idx % S, p = idx / S;
    if (s >= ns) continue;
    const int col = col0 + s, row = fdiv(col, a.dh), slot = col - row * H;
    const int kx = a.xk[MF_AT(slot, H)], ky = a.yk[MF_AT(row, a.ny)], kz = zk[MF_AT(p, nz)];
    C* e = buf + MF_AT(p * ZS + s, ext - 2 * CP);
    if (2 * ky == a.ny || 2 * kz == nz) {
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
      const int kys = (2 * ky < a.ny) ? ky : ky - a.ny;
      const int kzs = (2 * kz < nz) ? kz : kz - nz;
      const T xi0 = (T)kx * rnx, xi1 = (T)kys * rny, xi2 = (T)kzs * rnz;
      const T den = xi0 * xi0 + xi1 * xi1 + xi2 * xi2;
      T inv;
      if constexpr (sizeof(T) == 4) inv = scale * __frcp_rn(den);
      else inv = scale / den;
      const C A0 = e[0], A1 = e[CP], A2 = e[2 * CP];
      C q;
      q.x = (A0.x * xi0 + A1.x * xi1 + A2.x * xi2) * inv;
      q.y = (A0.y * xi0 + A1.y * xi1 + A2.y * xi2) * inv;
      e[0] = cmake(q.x * xi0, q.y * xi0);
      e[CP] = cmake(q.x * xi1, q.y * xi1);
      e[2 * CP] = cmake(q.x * xi2, q.y * xi2);
    }
  }
  __syncthreads();
  for (int s = a.pz.nst - 1; s >= 1; --s) {
    stage<C, true, true>(a.pz, s, NSEQ, dseq, twz, sld, sst);
    __syncthreads();
  }
  stage<C, true, true>(a.pz, 0, NSEQ, dseq, twz, sld, gst);
}

// ---------------------------------------------------------------- launchers
// Threads of an x-y block: about one radix-8 butterfly each, so that small
// planes share an SM.
inline int xy_threads(const XYArgs& a) {
  const int t = ((a.ny * (a.nx / 2) / 8 + 31) / 32) * 32;
  return t < 64 ? 64 : (t > 512 ? 512 : t);
}

template <typename T>
size_t xy_smem(const XYArgs& a) {
  typedef typename CT<T>::t C;
  return (size_t)a.ny * pitch(a.nx / 2) * sizeof(C) + (size_t)(a.nx + a.ny) * sizeof(C) + (size_t)(a.nx / 2) * sizeof(int);
}

// The shared-memory opt-in, once per kernel and process (one process drives
// one device), at the most a plane of any admissible size takes.
constexpr size_t kSmemMax = 226 * 1024;
template <auto K>
cudaError_t smem_once() {
  static const cudaError_t e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
  return e;
}

template <typename T>
cudaError_t xyf(const void* in, void* spec, const XYArgs& a, cudaStream_t st) {
  typedef typename CT<T>::t C;
  const cudaError_t e = smem_once<k_xyf<T>>();
  if (e != cudaSuccess) return e;
  const size_t sm = xy_smem<T>(a);
  if (sm > kSmemMax) return cudaErrorInvalidValue;
  ++g_mf_launches;
  return launch_k(a.pdl != 0, k_xyf<T>, dim3(9 * a.nz), dim3(xy_threads(a)), sm, st, (const T*)in, (C*)spec, a,
                  (int)(((uintptr_t)in & (sizeof(C) - 1)) == 0));
}

template <typename T, int MODE>
cudaError_t xyi_m(const void* spec, void* out, double* partials, const XYArgs& a, const Scalars* sc, cudaStream_t st) {
  typedef typename CT<T>::t C;
  const cudaError_t e = smem_once<k_xyi<T, MODE>>();
  if (e != cudaSuccess) return e;
  const size_t sm = xy_smem<T>(a);
  const int wide = ((uintptr_t)out & (sizeof(C) - 1)) == 0;
  if (sm > kSmemMax || (MODE == 3 && !wide)) return cudaErrorInvalidValue;
  ++g_mf_launches;
  return launch_k(a.pdl != 0, k_xyi<T, MODE>, dim3(9 * a.nz), dim3(xy_threads(a)), sm, st, (const C*)spec, (T*)out,
                  partials, a, const_cast<Scalars*>(sc), wide);
}

template <typename T>
cudaError_t xyi(int mode, const void* spec, void* out, double* partials, const XYArgs& a, const Scalars* sc,
                cudaStream_t st) {
  return mode == 3 ? xyi_m<T, 3>(spec, out, partials, a, sc, st) : xyi_m<T, 0>(spec, out, partials, a, sc, st);
}

template <typename T, int MODE, int S>
cudaError_t zp_s(void* spec, ZArgs a, cudaStream_t st) {
  typedef typename CT<T>::t C;
  const cudaError_t e = smem_once<k_zp<T, MODE, S>>();
  if (e != cudaSuccess) return e;
  const size_t sm = (size_t)3 * ZPad<T>::cp(a.nz, S) * sizeof(C) + (size_t)a.nz * (sizeof(C) + sizeof(int));
  if (sm > kSmemMax) return cudaErrorInvalidValue;
  const int ncol = a.ny * (a.nx / 2);
  a.dseq = fast_div(3 * S);
  int t = ((3 * S * a.nz / 8 + 31) / 32) * 32;   // about one radix-8 butterfly per thread
  t = t < 64 ? 64 : (t > 256 ? 256 : t);
  ++g_mf_launches;
  return launch_k(a.pdl != 0, k_zp<T, MODE, S>, dim3(3 * ((ncol + S - 1) / S)), dim3(t), sm, st, (C*)spec, a);
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
