// Angular coefficients by channel as device tables, for the kernels that look
// them up per row (mol_tile.cu, mol_pair.cu).  Each unit that includes this
// holds its own copy, which its upload_triplet_tables_* fills; the other
// kernels have the coefficients as immediates (c_zu and the like).
#pragma once

#include "mol_common.cuh"

namespace ms {
namespace {

// Per channel, on the two runs (j + 1, .) and (j - 1, .): .x S+ (from m - 1),
// .y Z (from m), .z S- (from m + 1), .w 0.
static __device__ float4 g_tri_up[kMaxRot], g_tri_dn[kMaxRot];

static cudaError_t upload_triplet_tables_local(const CouplEntry* dip) {
  // dipole slots: 0 Z (j-1, m), 1 Z (j+1, m), 2 S+ (j-1, m-1), 3 S+ (j+1, m-1), 4 S- (j+1, m+1), 5 S- (j-1, m+1)
  std::vector<float4> up(kMaxRot, make_float4(0.f, 0.f, 0.f, 0.f)), dn = up;
  for (int c = 0; c < kMaxRot; ++c) {
    auto cf = [&](int slot) { const CouplEntry& e = dip[c * kMaxCoupl + slot]; return e.nbr >= 0 ? e.coef : 0.f; };
    up[c] = make_float4(cf(3), cf(1), cf(4), 0.f);
    dn[c] = make_float4(cf(2), cf(0), cf(5), 0.f);
  }
  cudaError_t e = cudaMemcpyToSymbol(g_tri_up, up.data(), sizeof(float4) * kMaxRot);
  if (e != cudaSuccess) return e;
  return cudaMemcpyToSymbol(g_tri_dn, dn.data(), sizeof(float4) * kMaxRot);
}

constexpr int kTriGuard = 3;  // zero rows ahead of each term buffer

}  // namespace
}  // namespace ms
