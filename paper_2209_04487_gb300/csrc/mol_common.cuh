// Device helpers shared by the molecular kernels' translation units (mol.cu,
// mol_tile.cu, mol_pair.cu, mol_rotor.cu, mol_col.cu).  Everything here has
// internal linkage: each unit holds its own copy.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "ms_internal.cuh"

namespace ms {

// Tensor maps of one species for the tiled R-space kernel: 8-byte elements
// (one complex FP32 value), boxes of TILE radial points by the rows of a
// molecule, at most 256 rows a box (a box dimension's limit): a molecule's
// rows arrive as full boxes (s, d2) and one remainder box (s_r, d2_r).
struct RspaceMaps {
  CUtensorMap s, d2;      // [n_mol * rows][nr], box TILE x min(rows, 256)
  CUtensorMap s_r, d2_r;  // same arrays, box TILE x the remainder rows (rows > 256 only)
  CUtensorMap vd, vh;     // [2 (J + 1)][nr], box TILE x 2 (J + 1)
  CUtensorMap mk;         // [1][nr], box TILE x 1
};

namespace {

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 operator+(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 operator-(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }

// ---- TMA bulk copies (cp.async.bulk) completing on an mbarrier --------------
__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
// 2-D tensor copy global -> shared (box of the map at element (x, y)).
__device__ __forceinline__ void tensor2d_g2s(void* dst, const CUtensorMap* map, int x, int y,
                                             unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}
// Wait for phase `parity` of the barrier, giving up after `limit` polls.
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity, long long limit) {
  for (long long it = 0; it < limit; ++it) {
    unsigned done;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}
constexpr long long kWaitPolls = 1LL << 24;  // far beyond any copy's duration

__device__ __forceinline__ int j_of(int c) { return (int)sqrtf((float)c + 0.5f); }  // c = j^2+j+m

template <int I, int N, class F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>());
    static_for<I + 1, N>(f);
  }
}

// ---- angular coefficients as compile-time constants ------------------------
// square root by Newton's iteration in double precision (x >= 0)
constexpr double c_sqrt(double x) {
  if (x <= 0.0) return 0.0;
  double r = x < 1.0 ? 1.0 : x;
  for (int i = 0; i < 64; ++i) r = 0.5 * (r + x / r);
  return r;
}
constexpr bool ch_valid(int j, int m) { return j >= 0 && m >= -j && m <= j; }
// <j+1, m|cos t|j, m>, -<j+1, m+1|sin t e^{i p}|j, m> and <j-1, m+1|sin t e^{i p}|j, m>
// in the Condon-Shortley phase convention
constexpr double c_ang_a(int j, int m) {
  return c_sqrt(((j + 1.0) * (j + 1) - (double)m * m) / ((2.0 * j + 1) * (2.0 * j + 3)));
}
constexpr double c_ang_b(int j, int m) {
  return -c_sqrt((j + m + 1.0) * (j + m + 2) / ((2.0 * j + 1) * (2.0 * j + 3)));
}
constexpr double c_ang_c(int j, int m) {
  return c_sqrt((j - m) * (j - m - 1.0) / ((2.0 * j - 1) * (2.0 * j + 1)));
}
// Row (j, m) of Z, S+ = sin t e^{ip} and S- = sin t e^{-ip} on the runs (j + 1, .) and (j - 1, .):
// Z from (j +- 1, m), S+ from (j +- 1, m - 1), S- from (j +- 1, m + 1).
constexpr float c_zu(int j, int m) { return (float)c_ang_a(j, m); }
constexpr float c_zd(int j, int m) { return ch_valid(j - 1, m) ? (float)c_ang_a(j - 1, m) : 0.f; }
constexpr float c_pu(int j, int m) { return ch_valid(j + 1, m - 1) ? (float)c_ang_c(j + 1, m - 1) : 0.f; }
constexpr float c_pd(int j, int m) { return ch_valid(j - 1, m - 1) ? (float)c_ang_b(j - 1, m - 1) : 0.f; }
constexpr float c_mu(int j, int m) { return (float)c_ang_b(j, m); }
constexpr float c_md(int j, int m) { return j >= 1 ? (float)c_ang_c(j, m) : 0.f; }



// compensated FP32 accumulation (TwoSum): hi + lo carries ~48 bits
__device__ __forceinline__ void acc2(float& hi, float& lo, float x) {
  const float t = hi + x;
  const float z = t - hi;
  lo += (hi - (t - z)) + (x - z);
  hi = t;
}

// The state's one full-magnitude rounding per step, s' = fl(s + D'), with the
// update D' = D + c s scaled by the previous step's rounding feedback c, and
// the exact residual e = (s + D') - s' of that rounding (TwoSum; the FP32
// operations must stay unfused and unreordered) folded into acc as
// Re(conj(s') e).  The rounding changed sum |s|^2 by -2 sum Re(conj(s') e) to
// first order; the next step's c = sum Re(conj(s') e) / sum |s'|^2 gives that
// back, so the norm carries one step's rounding instead of a random walk.
__device__ __forceinline__ float2 round_update(float2 sv, float2 D, float c, float& acc) {
  const float dx = fmaf(c, sv.x, D.x), dy = fmaf(c, sv.y, D.y);
  const float nx = __fadd_rn(sv.x, dx), ny = __fadd_rn(sv.y, dy);
  const float bx = __fsub_rn(nx, sv.x), by = __fsub_rn(ny, sv.y);
  const float ex = __fadd_rn(__fsub_rn(sv.x, __fsub_rn(nx, bx)), __fsub_rn(dx, bx));
  const float ey = __fadd_rn(__fsub_rn(sv.y, __fsub_rn(ny, by)), __fsub_rn(dy, by));
  acc = fmaf(nx, ex, fmaf(ny, ey, acc));
  return make_float2(nx, ny);
}

// feedback factor for the next step from the summed residual products and the
// summed |s'|^2 of a molecule (0 for an empty state)
__device__ __forceinline__ float rounding_feedback(float res, float norm2) {
  return norm2 > 0.f && isfinite(res) ? res / norm2 : 0.f;
}

// ---- packed FP32x2 arithmetic (one instruction; sign changes and equal constants of both parts are free)
__device__ __forceinline__ float2 lo2(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }
__device__ __forceinline__ float2 dup2(float c) { return make_float2(c, c); }
// round_update on one point held as a (Re, Im) pair, packed: s' = fl(s + D'),
// D' = D + c s, with the exact residual of that rounding folded into acc
// (per part; the two parts are added at the end)
__device__ __forceinline__ float2 round_update2(float2 sv, float2 D, float2 c, float2& acc) {
  const float2 d = fma2(c, sv, D);
  const float2 n = add2(sv, d);
  const float2 b = sub2(n, sv);
  const float2 e = add2(sub2(sv, sub2(n, b)), sub2(d, b));
  acc = fma2(n, e, acc);
  return n;
}
// compensated sums of point pairs (TwoSum per part)
__device__ __forceinline__ void acc2p(float2& hi, float2& lo, float2 x) {
  const float2 t = add2(hi, x);
  const float2 z = sub2(t, hi);
  lo = add2(lo, add2(sub2(hi, sub2(t, z)), sub2(x, z)));
  hi = t;
}



// Terms N of the coupling series exp(iA) ~ sum_{n <= N} (iA)^n / n!, for a
// Hermitian A with |A| <= x (x = theta |E'|).  Truncated after N terms the
// step changes the norm by up to 2 x^(N+1)/(N+1)! when N is odd; when N is
// even the first omitted term (iA)^(N+1) is odd in A and has no real part,
// so the norm changes only by up to 2 x^(N+2)/(N+1)!, while the amplitude
// the omitted terms carry, relative to the first-order term, is x^N/(N+1)!.
// N is the smallest count with a norm change below 1e-11 per step (1e-7 over
// 10^4 steps) and, for even N, an amplitude error below 1e-6.  24 flags a
// field out of range.
__device__ __forceinline__ int coupling_terms(float x) {
  if (!(x > 0.f)) return 0;
  float t = x;  // x^N / N!
  for (int N = 1; N < 24; ++N) {
    const float t1 = t * x / (float)(N + 1);  // x^(N+1) / (N+1)!
    const bool done = (N & 1) ? 2.f * t1 < 1e-11f : (2.f * t1 * x < 1e-11f && t1 < 1e-6f * x);
    if (done) return N;
    t = t1;
  }
  return 24;
}

// A molecule's field record: the local field in the molecule frame scaled by
// theta, (theta E'_z, theta E'_x / 2, theta E'_y / 2), and the number of
// coupling-series terms (coupling_terms).
__device__ __forceinline__ float4 field_record(const SpeciesDev& sp, const MolDev& md, const Grid& g, int prescribed,
                                               int m, int* err) {
  float E[3];
  lab_field(md, g, prescribed, m, E, err);
  const float* O = md.rot + 9 * (long long)m;  // molecule -> lab, row-major
  const float inv_fau = 1.0f / 5.14220674763e11f;
  float Ep[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) Ep[i] = (O[i] * E[0] + O[3 + i] * E[1] + O[6 + i] * E[2]) * inv_fau;
  const float th = (float)sp.theta;
  const float x = th * sqrtf(Ep[0] * Ep[0] + Ep[1] * Ep[1] + Ep[2] * Ep[2]);
  if (!isfinite(x)) atomicOr(err, kErrNonFinite);  // a non-finite local field
  const int nt = coupling_terms(x);
  if (nt >= 24 || x > 4.f) atomicOr(err, kErrCouplingSeries);
  // no field, or one that is not a number: no terms, and factors of zero for the kernels that always take one
  if (nt == 0) return make_float4(0.f, 0.f, 0.f, __int_as_float(0));
  return make_float4(th * Ep[2], 0.5f * th * Ep[0], 0.5f * th * Ep[1], __int_as_float(nt));
}

// Wait for phase `parity`, each try suspending up to hint_ns until the phase
// completes; gives up after `tries` tries (by default about 2 s in all).
__device__ __forceinline__ bool mbar_wait_sleep(unsigned long long* bar, unsigned parity, int tries = 2000,
                                                unsigned hint_ns = 1000000u) {
  for (int it = 0; it < tries; ++it) {
    unsigned done;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3; selp.u32 %0, 1, 0, p; }"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity), "r"(hint_ns)
        : "memory");
    if (done) return true;
  }
  return false;
}

// persistent launch of a tiled kernel: CTA b walks molecules b, b + grid,
// ...; the grid is the plan's resident CTAs per SM (0: as many as fit) times
// the SMs, or one CTA per molecule (cps < 0)
using RspaceKernel = void (*)(SpeciesDev, MolDev, int*, const RspaceMaps);
static void launch_persistent(RspaceKernel k, int nt, int bytes, const SpeciesDev& sp, const MolDev& md, int* err,
                              const RspaceMaps& maps, cudaStream_t s) {
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  int dev = 0, nsm = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, nt, bytes);
  per = std::max(per, 1);
  if (sp.cps > 0) per = std::min(per, sp.cps);
  const long long fit = sp.cps < 0 ? (long long)sp.nmol : (long long)std::max(nsm, 1) * per;
  const int grid = (int)std::min<long long>(sp.nmol, fit);
  k<<<grid, nt, bytes, s>>>(sp, md, err, maps);
}


}  // namespace

// The two-points-a-thread tiled R-space pass (mol_pair.cu): the kernel of the
// species' J at tile width `tile` (and its parity-reduced form for a
// parity-reduced species), launched persistently on stream s.
void launch_rspace_pair(const SpeciesDev& sp, const MolDev& md, int* err, const RspaceMaps& maps, int tile,
                        cudaStream_t s);
// The molecular step on whole rotors, J <= 4, reachable rows (mol_rotor.cu):
// the R-space pass of a streaming species or the whole fused step.
void launch_rotor(const SpeciesDev& sp, const MolDev& md, int* err, cudaStream_t s);
// The R-space pass on columns of the rotor, J = 5..8, reachable rows (mol_col.cu).
void launch_rspace_col(const SpeciesDev& sp, const MolDev& md, int* err, cudaStream_t s);
// uploads the angular tables into mol_pair.cu's copy
cudaError_t upload_triplet_tables_pair(const CouplEntry* dip);
// The one-point-a-thread tiled R-space pass (mol_tile.cu) at tile width
// `tile`, launched persistently on stream s, and its copy of the tables.
void launch_rspace(const SpeciesDev& sp, const MolDev& md, int* err, const RspaceMaps& maps, int tile,
                   cudaStream_t s);
cudaError_t upload_triplet_tables_tile(const CouplEntry* dip);

}  // namespace ms
