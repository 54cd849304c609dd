// Register and shared-memory FFTs of the kinetic pass, shared by the molecular
// kernels' translation units.
#pragma once

#include "mol_common.cuh"

namespace ms {
namespace {

constexpr int kPad = 0;  // state rows are stored unpadded (one bulk copy per molecule)

template <int NR>
struct FFTShape;
template <>
struct FFTShape<64> {
  static constexpr int N1 = 8, N2 = 8, THREADS = 256;
};
template <>
struct FFTShape<128> {
  static constexpr int N1 = 16, N2 = 8, THREADS = 256;
};
template <>
struct FFTShape<256> {
  static constexpr int N1 = 16, N2 = 16, THREADS = 256;
};

// cos / sin of t*pi/8, t = 0..7 (exact decimal expansions of the constants)
__host__ __device__ constexpr double cos_pi8(int t) {
  return t == 0 ? 1.0
       : t == 1 ? 0.92387953251128675613
       : t == 2 ? 0.70710678118654752440
       : t == 3 ? 0.38268343236508977173
       : t == 4 ? 0.0
       : t == 5 ? -0.38268343236508977173
       : t == 6 ? -0.70710678118654752440
                : -0.92387953251128675613;
}
__host__ __device__ constexpr double sin_pi8(int t) { return t <= 4 ? cos_pi8(4 - t) : cos_pi8(t - 4); }
__host__ __device__ constexpr float hi_of(double v) { return (float)v; }
__host__ __device__ constexpr float lo_of(double v) { return (float)(v - (double)(float)v); }

// multiply by exp(-+ i t pi/8) (forward: minus)
template <int T, bool INV>
__device__ __forceinline__ float2 twiddle16(float2 v) {
  if constexpr (T == 0) {
    return v;
  } else if constexpr (T == 4) {
    return INV ? make_float2(-v.y, v.x) : make_float2(v.y, -v.x);
  } else {
    constexpr float c = (float)cos_pi8(T);
    constexpr float s = INV ? (float)sin_pi8(T) : -(float)sin_pi8(T);
    return make_float2(fmaf(v.x, c, -v.y * s), fmaf(v.x, s, v.y * c));
  }
}

template <int L>
__device__ constexpr int bitrev(int a) {
  int r = 0;
  for (int b = 1, q = L >> 1; b < L; b <<= 1, q >>= 1)
    if (a & b) r |= q;
  return r;
}

// In-register DFT of size L (8 or 16), radix-2 decimation in time.  PACK: the
// butterflies' sums as packed FP32x2 (the same results).
template <int L, bool INV, bool PACK, int H, int J>
__device__ __forceinline__ void dft_stage_j(float2 (&x)[L]) {
  if constexpr (J < H) {
    constexpr int T = J * (16 / (2 * H));
#pragma unroll
    for (int a = J; a < L; a += 2 * H) {
      const float2 u = x[a];
      const float2 v = twiddle16<T, INV>(x[a + H]);
      x[a] = PACK ? add2(u, v) : u + v;
      x[a + H] = PACK ? sub2(u, v) : u - v;
    }
    dft_stage_j<L, INV, PACK, H, J + 1>(x);
  }
}
template <int L, bool INV, bool PACK, int H>
__device__ __forceinline__ void dft_stages(float2 (&x)[L]) {
  if constexpr (H < L) {
    dft_stage_j<L, INV, PACK, H, 0>(x);
    dft_stages<L, INV, PACK, 2 * H>(x);
  }
}
template <int L, bool INV, bool PACK = false>
__device__ __forceinline__ void dft_reg(float2 (&x)[L]) {
#pragma unroll
  for (int a = 0; a < L; ++a) {
    const int b = bitrev<L>(a);
    if (b > a) {
      const float2 t = x[a];
      x[a] = x[b];
      x[b] = t;
    }
  }
  dft_stages<L, INV, PACK, 1>(x);
}

// Four-step FFT pass on all `rows` rows (each NR complex, stride NRP) held
// in shared memory, in place: forward DFT, multiply by kph[k], inverse DFT.
// With kph = (P_k - 1)/NR it produces (T - 1) x; with kph = P_k/NR it
// applies T.  n = n1 + N1 n2, k = k2 + N2 k1.  Step A: per n1, an N2-point
// DFT over n2 and the twiddle exp(-2 pi i n1 k2/NR); step B: per k2, an
// N1-point DFT over n1.  The intermediate y[n1][k2] lives at n1 + N1 k2,
// xor-swizzled within each block of N1 so that step B is conflict free.
// Position of y[n1][k2] of `row` within the row: the xor with (k2 mod N1)
// spreads step B's N2 threads over distinct banks, the xor with CR for odd
// rows keeps the two rows that share a half-warp apart.
template <int N1, int N2>
__device__ __forceinline__ int swz(int n1, int k2, int row) {
  constexpr int CR = N1 > N2 ? N2 : (N1 == N2 && N1 == 8 ? 1 : 0);
  return (n1 ^ (k2 % N1) ^ ((row & 1) * CR)) + N1 * k2;
}

// The rows are read from `in` (st itself for the transform in place) by NT threads.
// The result goes back to st, or, with `take`, to take(row, n1, x): x[n2] at
// point n1 + N1 n2, called for every row by the N1 neighbouring lanes n1, and
// by whole warps together (rows past the end too, with row >= rows).
struct KeepRows {};
template <int NR, int NT = FFTShape<NR>::THREADS, bool PACK = false, class Take = KeepRows>
__device__ __forceinline__ void kinetic_pass(float2* st, const float2* in, int rows, const float2* kph, const float2* tw,
                                             Take take = Take()) {
  using S = FFTShape<NR>;
  constexpr int N1 = S::N1, N2 = S::N2, NRP = NR + kPad;
  const int t = threadIdx.x;
  {  // step A
    constexpr int per = NT / N1;
    const int n1 = t % N1, rsub = t / N1;
    for (int r0 = 0; r0 < rows; r0 += per) {
      const int row = r0 + rsub;
      float2 x[N2];
      if (row < rows) {
#pragma unroll
        for (int n2 = 0; n2 < N2; ++n2) x[n2] = in[row * NRP + n1 + N1 * n2];
      }
      __syncwarp();  // a row's N1 threads sit in one warp
      if (row < rows) {
        dft_reg<N2, false, PACK>(x);
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2)
          st[row * NRP + swz<N1, N2>(n1, k2, row)] = cmul(x[k2], tw[k2 * N1 + n1]);
      }
      __syncwarp();
    }
  }
  __syncthreads();
  {  // step B, the phase, inverse step B (in place per thread)
    constexpr int per = NT / N2;
    const int k2 = t % N2, rsub = t / N2;
    for (int r0 = 0; r0 < rows; r0 += per) {
      const int row = r0 + rsub;
      if (row < rows) {
        float2 x[N1];
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) x[n1] = st[row * NRP + swz<N1, N2>(n1, k2, row)];
        dft_reg<N1, false, PACK>(x);  // x[k1] = X[k2 + N2 k1]
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) x[k1] = cmul(x[k1], kph[k2 + N2 * k1]);
        dft_reg<N1, true, PACK>(x);
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) st[row * NRP + swz<N1, N2>(n1, k2, row)] = x[n1];
      }
    }
  }
  __syncthreads();
  {  // inverse step A
    constexpr int per = NT / N1;
    const int n1 = t % N1, rsub = t / N1;
    for (int r0 = 0; r0 < rows; r0 += per) {
      const int row = r0 + rsub;
      float2 x[N2];
      if (row < rows) {
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) {
          const float2 w = tw[k2 * N1 + n1];
          x[k2] = cmul(st[row * NRP + swz<N1, N2>(n1, k2, row)], make_float2(w.x, -w.y));
        }
        dft_reg<N2, true, PACK>(x);
      }
      __syncwarp();
      if constexpr (!std::is_same_v<Take, KeepRows>) {
        take(row, n1, x);
      } else if (row < rows) {
#pragma unroll
        for (int n2 = 0; n2 < N2; ++n2) st[row * NRP + n1 + N1 * n2] = x[n2];
      }
      __syncwarp();
    }
  }
  __syncthreads();
}

}  // namespace
}  // namespace ms
