// Block sums of several FP64 columns.
#pragma once

#include <cuda_runtime.h>

// Warp sums of NC columns, one value per lane and column: each of the five
// steps halves the columns a lane still holds (lanes with the step's bit set
// keep the upper half and send the lower one, the others the reverse), so a
// warp issues about NC + 2 FP64 additions instead of 5 NC of a butterfly per
// column.  FP64 runs at 1/62 of the FP32 rate here (one warp instruction
// occupies an SM's FP64 pipe for about 15 cycles), and five steps over the
// 36 columns of the constitutive pass took that pipe 11 us per block (stress
// and residual of a 128^3 FP32-inner cell: 968 -> 941 us with this form).  The
// additions pair the same lanes in the same order as the butterfly's: the
// sums are bit for bit the same.
// On return v[0 .. kLeft) holds columns first, first + 1, ...; count of them
// are the lane's to store.
template <int NC> struct WarpColumns {
  static __host__ __device__ constexpr int half(int n) { return (n + 1) / 2; }
  static constexpr int kLeft = half(half(half(half(half(NC)))));
  int first = 0, count = NC;

  template <int N, int O>
  __device__ __forceinline__ void step(double* v, int lane) {
    constexpr int HF = half(N);
    const bool up = lane & O;
#pragma unroll
    for (int i = 0; i < HF; ++i) {
      const double lo = v[i], hi = HF + i < N ? v[HF + i < N ? HF + i : 0] : 0.0;
      const double send = up ? lo : hi;
      v[i] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, send, O);
    }
    first += up ? HF : 0;
    count = up ? (count > HF ? count - HF : 0) : (count < HF ? count : HF);
    if constexpr (O > 1) step<HF, O / 2>(v, lane);
  }
  __device__ __forceinline__ WarpColumns(double (&v)[NC], int lane) { step<NC, 16>(v, lane); }
};

// Sum NC columns over the block (whole warps, at most 32): out[col], a
// shared array, for every thread after the call.
template <int NC>
__device__ __forceinline__ void block_sum(double (&v)[NC], double* out) {
  __shared__ double red[NC][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const WarpColumns<NC> w(v, lane);
#pragma unroll
  for (int i = 0; i < WarpColumns<NC>::kLeft; ++i)
    if (i < w.count) red[w.first + i][warp] = v[i];
  __syncthreads();
  if (threadIdx.x < NC) {
    double s = 0.0;
    const int nw = blockDim.x >> 5;
    for (int k = 0; k < nw; ++k) s += red[threadIdx.x][k];
    out[threadIdx.x] = s;
  }
  __syncthreads();
}
