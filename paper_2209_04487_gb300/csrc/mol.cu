// Molecular split-operator step (Eqs. 3-5 with the surfaces of Eqs. 6-7),
// one CTA per molecule, the molecule's whole state resident in shared memory.
//
// The library stores s = T^{-1/2} psi, so that one coupled step is
//   u  = T s                                   (kinetic pass, per channel)
//   s' = Mask V^{1/2} K(E') V^{1/2} u          (R-space pass, per radial point)
// which equals the paper's split-operator step T^{1/2} Mask V^{1/2} K V^{1/2}
// T^{1/2} on psi (T commutes with the angular coupling because the
// transition dipole is R-independent, and is unitary per channel, so
// populations and the dipole can be taken from s').
//
// Norm-preserving FP32 arithmetic: every unit-modulus factor (potential
// phase, kinetic phase, FFT twiddle) is carried as an FP32 hi+lo pair and
// applied with a compensated product, so the factor is exact to ~1e-15 and
// only unbiased output rounding remains.  Every factor of the step is close
// to the identity (|V dtau| and |k^2 dtau/2mu| are a few 1e-2 at one
// molecular step per field step, O(1) under sub-stepping), so the step is
// computed as a correction: d2 = (T - 1) s, u = s + d2,
// d1 = (V - 1) u + V^{1/2} S with S = sum_{n>=1} (i theta sigma_x M)^n/n!
// V^{1/2} u (Taylor series of the coupling exponential, |theta M| << 1), and
// s' = s + (d2 + d1): the full-magnitude state is rounded once per step,
// which turns the FP32 norm error from a drift into a random walk of about
// 1e-8 per step.  That one rounding's exact residual (TwoSum) gives the norm
// it changed; the next step scales its update by the factor that returns it
// (round_update), so the walk of the final roundings does not accumulate:
// what remains is one step's rounding plus the much smaller rounding inside
// the correction.  The coupling is evaluated in the frame turned about
// z that puts E' in the xz plane (a diagonal phase on the correction only),
// where M is real.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <mutex>
#include <type_traits>
#include <vector>

#include "ms_internal.cuh"
#include "mol_common.cuh"
#include "mol_fft.cuh"

namespace ms {

namespace {

// 16-byte asynchronous global -> shared copies (per thread), completed by
// cp.async.wait_group.
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

}  // namespace

// Angular coupling tables, shared by every species (they depend only on the
// channel (j, m), and a species with jmax < kMaxJ ignores entries whose
// neighbour lies beyond its basis).  c_rot: rows of Ex' X + Ez' Z written in
// the frame turned about z so that E'_y = 0 (kind 1: X entry, scaled by
// E_perp; kind 0: Z entry, scaled by E'_z).  c_dip: rows of Z (kind 0),
// S+ = sin(t)e^{ip} (kind 1) and S- (kind 2) for the dipole.
__constant__ CouplEntry c_rot[kMaxRot * kMaxCoupl];
__constant__ CouplEntry c_dip[kMaxRot * kMaxCoupl];

cudaError_t upload_coupling_tables(const CouplEntry* rot, const CouplEntry* dip) {
  cudaError_t e = cudaMemcpyToSymbol(c_rot, rot, sizeof(CouplEntry) * kMaxRot * kMaxCoupl);
  if (e != cudaSuccess) return e;
  return cudaMemcpyToSymbol(c_dip, dip, sizeof(CouplEntry) * kMaxRot * kMaxCoupl);
}

// Local field at molecule m in its own frame (a.u.): fld = (E_perp, E'_z), the
// phases e^{i m' phi_E} (ph[m' + J], m' = -J..J) of the frame turned about z
// so that E'_y = 0, and the number of coupling-series terms (coupling_terms).
// Run by one thread.
__device__ __noinline__ void molecule_field(const MolDev& md, const Grid& g, int prescribed, int m, int J,
                                            double theta, float* fld, float2* ph, int* nterms, int* err) {
  float E[3];
  lab_field(md, g, prescribed, m, E, err);
  const float* O = md.rot + 9 * (long long)m;  // molecule -> lab, row-major
  const float inv_fau = 1.0f / 5.14220674763e11f;
  float Ep[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) Ep[i] = (O[i] * E[0] + O[3 + i] * E[1] + O[6 + i] * E[2]) * inv_fau;
  const float eperp = sqrtf(Ep[0] * Ep[0] + Ep[1] * Ep[1]);
  fld[0] = eperp;
  fld[1] = Ep[2];
  // e^{i phi_E} = (E'_x + i E'_y)/E_perp; e^{i m phi_E} by repeated products
  const float2 e1 = eperp > 0.f ? make_float2(Ep[0] / eperp, Ep[1] / eperp) : make_float2(1.f, 0.f);
  float2 pw = make_float2(1.f, 0.f);
  ph[J] = pw;
  for (int q = 1; q <= J; ++q) {
    pw = cmul(pw, e1);
    ph[J + q] = pw;
    ph[J - q] = make_float2(pw.x, -pw.y);
  }
  const float x = (float)theta * sqrtf(eperp * eperp + Ep[2] * Ep[2]);
  if (!isfinite(x)) atomicOr(err, kErrNonFinite);  // a non-finite local field
  const int nt = coupling_terms(x);
  if (nt >= 24 || x > 4.f) atomicOr(err, kErrCouplingSeries);
  *nterms = nt;
}

constexpr int kChunk = 32;            // widest R-space chunk (one radial point per lane)

// ----------------------------------------------------------------------------
// the coupled molecular step, s = T^{-1/2} psi stored:
//   d2 = (T - 1) s           (kinetic pass, in shared memory)
//   u  = s + d2 = T s        (per radial point)
//   s' = Mask V^{1/2} K(E') V^{1/2} u, computed as s + (d2 + d1)
// ----------------------------------------------------------------------------
// FUSED: the whole state is staged in shared memory and the kinetic pass runs
// in this kernel.  Otherwise (streaming form) d2 = (T - 1) s comes from the
// scratch written by mol_kinetic_kernel and is streamed chunk by chunk with s.
// MAXR bounds the rows a thread owns in the R-space pass.
template <int NR, bool FUSED, int MAXR>
__global__ void __launch_bounds__(FFTShape<NR>::THREADS, FUSED ? 2 : (MAXR <= 4 ? 4 : (MAXR <= 12 ? 2 : 1)))
    mol_step_kernel(SpeciesDev sp, MolDev md, Grid g, int prescribed, int CH, int* err) {
  if (idle_launch(sp)) return;
  // CH radial points per chunk (32 down to 4): a warp covers 32/CH rows of CH points
  constexpr int NT = FFTShape<NR>::THREADS, NRP = NR + kPad, NW = NT / 32;
  extern __shared__ float4 smem4[];
  const int nrot = sp.nrot, rows = 2 * nrot, J = sp.jmax;
  float2* s_tw = reinterpret_cast<float2*>(smem4);      // [N2][N1] twiddles (fused)
  float2* s_kd = s_tw + (FUSED ? NR : 0);                // [NR] kinetic deltas (fused)
  float2* st = s_kd + (FUSED ? NR : 0);                  // [rows][NRP] state, then d2 (fused)
  float2* bY = st + (FUSED ? rows * NRP : 0);            // [rows][CH] Taylor terms / new state
  float2* bZ = bY + rows * CH;                           // [rows][CH] Taylor terms
  // per chunk, double buffered: old state [rows][CH], (streaming: d2
  // [rows][CH]), e^{-iV dtau} - 1 and e^{-iV dtau/2} [2(J+1)][CH] each, and
  // absorber mask [CH].  The half-step phase is read from its exact table:
  // with sub-stepping |V dtau| reaches O(1), where no short series of the
  // full-step delta would keep the coupling correction unitary.
  const int nd = FUSED ? 0 : rows;
  const int cbuf = (rows + nd + 4 * (J + 1) + 1) * CH;
  float2* bC = bZ + rows * CH;
  int2* s_prog = reinterpret_cast<int2*>(bC + 2 * cbuf);  // [nrot][6] (nbr*CH, coupling) this step
  int2* s_dipp = s_prog + nrot * kMaxCoupl;              // [nrot][6] (nbr*CH, dipole coefficient)
  int2* s_rinfo = s_dipp + nrot * kMaxCoupl;             // [rows] (table row, m + J)
  __shared__ __align__(8) unsigned long long s_bar[1];   // the state copy
  __shared__ float s_rot[9];                             // molecule -> lab rotation
  __shared__ double s_mu[3];                             // lab dipole of the previous step
  __shared__ double s_abs[2];                            // absorbed norm so far
  __shared__ float2 s_ph[2 * kMaxJ + 1];                 // e^{+i m phi_E}
  __shared__ float s_fld[2];                             // E_perp, E'_z (a.u.)
  __shared__ int s_nterms;
  __shared__ float2 s_red[NW][8];
  __shared__ float s_fin[8], s_fin_lo[8];

  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int LPR = 32 / CH;                       // row groups per warp
  const int rl = lane & (CH - 1), rg = lane / CH;
  const int row0 = w * LPR + rg, rstep = NW * LPR;
  const int lm = blockIdx.x;
  const int m = sp.mol[lm];
  float2* gs = sp.psi + (long long)lm * rows * NR;

  // chunk copy: old state, potential phases and mask of radial points [r0, r0 + CH)
  // every thread copies 16-byte pieces (cp.async); rows: old state, then
  // the potential deltas, the half-step phases, then the mask
  const float2* gd = FUSED ? nullptr : sp.d2 + (long long)lm * rows * NR;
  const int cp_per_row = CH / 2;                   // 16-byte pieces per chunk row
  const int cp_c2 = 2 * (t % cp_per_row), cp_q0 = t / cp_per_row, cp_qs = NT / cp_per_row;
  auto issue_chunk = [&](int r0, int b) {
    float2* buf = bC + b * cbuf;
    const int nv = 2 * (J + 1), nq = rows + nd + 2 * nv + 1;
    for (int q = cp_q0; q < nq; q += cp_qs) {
      const float2* src;
      if (q < rows) src = gs + (long long)q * NR;
      else if (q < rows + nd) src = gd + (long long)(q - rows) * NR;
      else if (q < rows + nd + nv) src = sp.vdelta + (long long)(q - rows - nd) * NR;
      else if (q < rows + nd + 2 * nv) src = sp.vhalf + (long long)(q - rows - nd - nv) * NR;
      else src = sp.maskw;
      cp_async16(buf + q * CH + cp_c2, src + r0 + cp_c2);
    }
    cp_async_commit();
  };
  if (t == 0) {
    mbar_init(&s_bar[0], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (FUSED && t == 0) {  // the whole (contiguous) state in one bulk copy
    mbar_expect_tx(&s_bar[0], (unsigned)(rows * NR * sizeof(float2)));
    bulk_g2s(st, gs, (unsigned)(rows * NR * sizeof(float2)), &s_bar[0]);
  }
  issue_chunk(0, 0);
  if (t < 9) s_rot[t] = md.rot[9 * (long long)m + t];
  else if (t < 12) s_mu[t - 9] = md.mu[3 * (long long)m + (t - 9)];
  else if (t < 14) s_abs[t - 12] = md.absorbed[2 * (long long)m + (t - 12)];
  if (FUSED) {
    for (int q = t; q < NR; q += NT) {
      s_tw[q] = __ldg(&sp.twiddle[q]);
      s_kd[q] = __ldg(&sp.kdelta[q]);
    }
  }
  for (int q = t; q < rows; q += NT) {
    const int sf = q >= nrot, c = q - sf * nrot, j = j_of(c);
    s_rinfo[q] = make_int2((sf * (J + 1) + j) * CH, c - j * j - j + J);
  }
  for (int q = t; q < nrot * kMaxCoupl; q += NT) {  // dipole rows: slots 0-1 Z, 2-3 S+, 4-5 S-
    const CouplEntry e = c_dip[q];
    const bool ok = (unsigned)e.nbr < (unsigned)nrot;
    s_dipp[q] = make_int2(ok ? e.nbr * CH : 0, __float_as_int(ok ? e.coef : 0.f));
  }

  // ---- local field, rotated into the molecule frame (a.u.)
  if (t == 0) molecule_field(md, g, prescribed, m, J, sp.theta, s_fld, s_ph, &s_nterms, err);
  __syncthreads();
  {  // this step's coupling rows: slots 0-1 Z (times E'_z), 2-5 X (times E_perp)
    const float eperp = s_fld[0], ez = s_fld[1];
    for (int q = t; q < nrot * kMaxCoupl; q += NT) {
      const CouplEntry e = c_rot[q];
      const bool ok = (unsigned)e.nbr < (unsigned)nrot;
      const float cf = ok ? e.coef * ((q % kMaxCoupl) >= 2 ? eperp : ez) : 0.f;
      s_prog[q] = make_int2(ok ? e.nbr * CH : 0, __float_as_int(cf));
    }
  }
  if (FUSED) {
    const bool ok = mbar_wait(&s_bar[0], 0, kWaitPolls);
    if (!__syncthreads_and(ok)) {  // uniform decision; copies still in flight get a second bounded wait
      if (t == 0) atomicOr(err, kErrTimeout);
      if (!ok) mbar_wait(&s_bar[0], 0, kWaitPolls);
      cp_async_wait_all();
      return;
    }
    // ---- kinetic pass: st <- d2 = (T - 1) s
    kinetic_pass<NR>(st, st, rows, s_kd, s_tw);
  } else {
    __syncthreads();
  }

  // ---- R-space pass, CH radial points at a time; thread rows row0 + i*rstep
  const int nterms = s_nterms;
  const float theta = (float)sp.theta;
  const float cfix = md.ncorr[m];  // rounding feedback of the previous step
  float a_hi[7] = {0, 0, 0, 0, 0, 0, 0}, a_lo[7] = {0, 0, 0, 0, 0, 0, 0};
  float rnd = 0.f;
  const int nchunks = NR / CH;
  for (int ck = 0; ck < nchunks; ++ck) {
    const int r0 = ck * CH, r = r0 + rl, b = ck & 1;
    float2* bU = bC + b * cbuf;
    const float2* bD = bU + rows * CH;              // streaming form: d2 of the chunk
    const float2* bV = bD + nd * CH;                // e^{-iV dtau} - 1
    const float2* bH = bV + 2 * (J + 1) * CH;       // e^{-iV dtau/2}
    const float2* bM = bH + 2 * (J + 1) * CH;
    // this chunk's copies (issued one chunk earlier) are complete and
    // visible; the other buffer is free since the previous chunk's barriers
    cp_async_wait_all();
    __syncthreads();
    if (ck + 1 < nchunks) issue_chunk(r0 + CH, b ^ 1);
    // eta = D^dagger V^{1/2} u (rotated frame) into bZ (no coupling work when E' = 0)
    float2 sacc[MAXR];
#pragma unroll
    for (int i = 0; i < MAXR; ++i) sacc[i] = make_float2(0.f, 0.f);
    if (nterms > 0) {
#pragma unroll
      for (int i = 0; i < MAXR; ++i) {
        const int row = row0 + i * rstep;
        if (row < rows) {
          const int2 ri = s_rinfo[row];
          const float2 u = (FUSED ? st[row * NRP + r] : bD[row * CH + rl]) + bU[row * CH + rl];
          bZ[row * CH + rl] = cmul(s_ph[ri.y], cmul(bH[ri.x + rl], u));
        }
      }
      __syncthreads();
    }
    float2* in = bZ;
    float2* out = bY;
    for (int n = 1; n <= nterms; ++n) {
      const float cn = theta / (float)n;
#pragma unroll
      for (int i = 0; i < MAXR; ++i) {
        const int row = row0 + i * rstep;
        if (row < rows) {
          const int sf = row >= nrot, c = row - sf * nrot;
          const float2* src = in + (1 - sf) * nrot * CH + rl;
          const int2* pr = s_prog + c * kMaxCoupl;
          float ax = 0.f, ay = 0.f;
#pragma unroll
          for (int e = 0; e < kMaxCoupl; ++e) {  // unused slots carry a zero coefficient
            const int2 q = pr[e];
            const float cf = __int_as_float(q.y);
            const float2 v = src[q.x];
            ax = fmaf(cf, v.x, ax);
            ay = fmaf(cf, v.y, ay);
          }
          const float2 o = make_float2(-cn * ay, cn * ax);  // i (theta/n) (M_r in)
          out[row * CH + rl] = o;
          sacc[i].x += o.x;
          sacc[i].y += o.y;
        }
      }
      __syncthreads();
      float2* tmp = in;
      in = out;
      out = tmp;
    }
    // d1 = (V - 1) u + V^{1/2} D S_r ; mask ; s' = s + (d2 + d1) + cfix s
    const float mk = bM[rl].x;
    float agf = 0.f, aef = 0.f;
#pragma unroll
    for (int i = 0; i < MAXR; ++i) {
      const int row = row0 + i * rstep;
      if (row < rows) {
        const int2 ri = s_rinfo[row];
        const int sf = row >= nrot;
        const float2 sv = bU[row * CH + rl];
        const float2 d2 = FUSED ? st[row * NRP + r] : bD[row * CH + rl];
        const float2 u = sv + d2;
        const float2 ph = s_ph[ri.y];
        const float2 vd = bV[ri.x + rl];
        const float2 corr = cmul(bH[ri.x + rl], cmul(make_float2(ph.x, -ph.y), sacc[i]));
        float2 d1 = make_float2(fmaf(u.x, vd.x, fmaf(-u.y, vd.y, corr.x)), fmaf(u.x, vd.y, fmaf(u.y, vd.x, corr.y)));
        if (mk < 1.f) {
          const float px = u.x + d1.x, py = u.y + d1.y;
          d1.x = fmaf(mk - 1.f, u.x, mk * d1.x);
          d1.y = fmaf(mk - 1.f, u.y, mk * d1.y);
          const float qx = u.x + d1.x, qy = u.y + d1.y;
          const float dd = fmaf(px, px, py * py) - fmaf(qx, qx, qy * qy);
          if (sf == 0) agf += dd; else aef += dd;
        }
        const float2 sn = round_update(sv, d2 + d1, cfix, rnd);
        gs[(long long)row * NR + r] = sn;
        bY[row * CH + rl] = sn;
        const float b2 = fmaf(sn.x, sn.x, sn.y * sn.y);
        if (sf == 0) acc2(a_hi[0], a_lo[0], b2);  // compensated from the first term on
        else acc2(a_hi[1], a_lo[1], b2);
      }
    }
    acc2(a_hi[2], a_lo[2], agf);
    acc2(a_hi[3], a_lo[3], aef);
    __syncthreads();
    // dipole in the molecule frame: sum_c conj(g_c) (A e)_c for A = Z, S+, S-
    {
      float2 accP = make_float2(0.f, 0.f), accM = accP, accZ = accP;
      for (int c = row0; c < nrot; c += rstep) {
        const float2 gc = bY[c * CH + rl];
        const float2* ee = bY + nrot * CH + rl;
        const int2* pr = s_dipp + c * kMaxCoupl;
        float2 w3[3];
#pragma unroll
        for (int kk = 0; kk < 3; ++kk) {  // slots 0-1 Z, 2-3 S+, 4-5 S- (unused: zero coefficient)
          const int2 q0 = pr[2 * kk], q1 = pr[2 * kk + 1];
          const float c0 = __int_as_float(q0.y), c1 = __int_as_float(q1.y);
          const float2 e0 = ee[q0.x], e1 = ee[q1.x];
          w3[kk] = make_float2(fmaf(c0, e0.x, c1 * e1.x), fmaf(c0, e0.y, c1 * e1.y));
        }
        // conj(gc) * w
        accZ.x += fmaf(gc.x, w3[0].x, gc.y * w3[0].y);
        accZ.y += fmaf(gc.x, w3[0].y, -gc.y * w3[0].x);
        accP.x += fmaf(gc.x, w3[1].x, gc.y * w3[1].y);
        accP.y += fmaf(gc.x, w3[1].y, -gc.y * w3[1].x);
        accM.x += fmaf(gc.x, w3[2].x, gc.y * w3[2].y);
        accM.y += fmaf(gc.x, w3[2].y, -gc.y * w3[2].x);
      }
      acc2(a_hi[4], a_lo[4], accP.x + accM.x);
      acc2(a_hi[5], a_lo[5], accP.y - accM.y);
      acc2(a_hi[6], a_lo[6], 2.f * accZ.x);
    }
    __syncthreads();
  }
  // ---- block reduction (compensated FP32; FP64 only for the final sums)
  {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      float hi = q < 7 ? a_hi[q] : rnd, lo = q < 7 ? a_lo[q] : 0.f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float h2 = __shfl_xor_sync(0xffffffffu, hi, o);
        const float l2 = __shfl_xor_sync(0xffffffffu, lo, o);
        acc2(hi, lo, h2);
        lo += l2;
      }
      if (lane == 0) s_red[w][q] = make_float2(hi, lo);
    }
    __syncthreads();
    if (t < 8) {  // one quantity per thread, compensated over the warps
      float hi = 0.f, lo = 0.f;
      for (int ww = 0; ww < NW; ++ww) {
        acc2(hi, lo, s_red[ww][t].x);
        lo += s_red[ww][t].y;
      }
      s_fin[t] = hi + lo;  // FP32 sum; its rounding is 6e-8 relative
      s_fin_lo[t] = lo - (s_fin[t] - hi);
    }
    __syncthreads();
    if (t < 3) {  // lab dipole component t: mu = O mu', mu' = d dR (Re(S+ + S-), Im(S+ - S-), 2 Re Z)
      const float sc = (float)sp.dipole * sp.dR;
      const float lab = sc * (s_rot[3 * t] * s_fin[4] + s_rot[3 * t + 1] * s_fin[5] + s_rot[3 * t + 2] * s_fin[6]);
      const double nl = (double)lab;
      md.dmu[3 * (long long)m + t] = nl - s_mu[t];
      md.mu[3 * (long long)m + t] = nl;
    } else if (t < 5) {  // populations P_g, P_e
      const double P = ((double)s_fin[t - 3] + (double)s_fin_lo[t - 3]) * (double)sp.dR;
      md.pop[2 * (long long)m + (t - 3)] = P;
      if (!isfinite(P)) atomicOr(err, kErrNonFinite);
    } else if (t < 7) {  // absorbed norm, cumulative
      md.absorbed[2 * (long long)m + (t - 5)] =
          s_abs[t - 5] + ((double)s_fin[t - 3] + (double)s_fin_lo[t - 3]) * (double)sp.dR;
    } else if (t == 7) {  // rounding feedback for the next step
      md.ncorr[m] = rounding_feedback(s_fin[7], s_fin[0] + s_fin[1]);
    }
  }
}


// ----------------------------------------------------------------------------
// R-space pass of the streaming form, tiled: one CTA per molecule at a time,
// TILE = 32 or 16 radial points per tile, every row of the state.  The rows
// (surface, channel) are spread over the warps and stay in registers for a
// tile: s and d2 = (T - 1) s arrive by 2-D tensor copies and the coupling
// series exchanges values between rows through two term buffers in shared
// memory.
//
// Neighbour structure: the angular couplings of channel (j, m) reach the
// channels (j + 1, m - 1 .. m + 1) and (j - 1, m - 1 .. m + 1), two runs of
// three consecutive channels (c + 2j + 1 .. c + 2j + 3 and c - 2j - 1 ..
// c - 2j + 1, c = j^2 + j + m).  A row therefore needs two base offsets and
// six coefficients: for the coupling E_perp X + E'_z Z in the turned frame
// (X = (S+ + S-)/2) and for the dipole (Z, S+, S-).  Coefficients of channels
// outside the basis are zero and their reads land on finite data: kTriGuard
// zero rows precede each buffer, and a missing run points at them.
// ----------------------------------------------------------------------------
// Fills the copies of the angular tables of the kernels that read them.
cudaError_t upload_triplet_tables(const CouplEntry* dip) {
  const cudaError_t e = upload_triplet_tables_tile(dip);
  return e == cudaSuccess ? upload_triplet_tables_pair(dip) : e;
}

// Diagnostic of the bounded wait: one CTA waits on a barrier that nothing
// completes, gives up after `tries` tries of up to 10 us, and records the
// timeout as the molecular kernels do.
__global__ void wait_timeout_probe_kernel(int tries, int* flag) {
  __shared__ __align__(8) unsigned long long bar[1];
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const bool ok = mbar_wait_sleep(&bar[0], 0, tries, 10000u);
  if (!__syncthreads_and(ok) && threadIdx.x == 0) atomicOr(flag, kErrTimeout);
}

// Latches a host-detected launch failure into the error word.
__global__ void flag_error_kernel(int* err, int code) { atomicOr(err, code); }

cudaError_t launch_wait_timeout_probe(int tries, int* flag, cudaStream_t s) {
  wait_timeout_probe_kernel<<<1, 32, 0, s>>>(tries, flag);
  return cudaGetLastError();
}

// ----------------------------------------------------------------------------
// R-space pass of the streaming form, point-resident layout (J <= 4): one CTA
// per molecule, one thread per (radial point, surface).  A thread holds the
// channel vector of its surface at its point in registers, so the angular
// couplings become register arithmetic with indices fixed at compile time;
// the coupling series (sigma_x swaps the surfaces) and the dipole only
// exchange the other surface's vector, through one shared buffer.
// ----------------------------------------------------------------------------
constexpr int ch_j(int c) { return c < 1 ? 0 : (c < 4 ? 1 : (c < 9 ? 2 : (c < 16 ? 3 : (c < 25 ? 4 : -1)))); }
__host__ __device__ constexpr int j_of_c(int c) { return ch_j(c); }
constexpr int ch_m(int c) { return c - ch_j(c) * ch_j(c) - ch_j(c); }
// channel of (j, m), or -1 outside the basis of size J
constexpr int ch_of(int j, int m, int J) { return (j < 0 || j > J || m < -j || m > j) ? -1 : j * j + j + m; }

// The records on their own, where no FFT kernel makes them: for the mixed kinetic
// pass and the fused form (a thread of the fused kernel that makes its molecule's
// record waits for three dependent loads, and its CTA with it: 9.99 against 9.30
// ms for eight steps of 50,000 molecules).
__global__ void mol_field_kernel(SpeciesDev sp, MolDev md, Grid g, int prescribed, int* err) {
  if (idle_launch(sp)) return;
  const int lm = blockIdx.x * blockDim.x + threadIdx.x;
  if (lm < sp.nmol) sp.fld[lm] = field_record(sp, md, g, prescribed, sp.mol[lm], err);
}

// Row layout of a molecule's state.  Full: both surfaces carry every channel
// c = j^2 + j + m, c < (J+1)^2, in channel order.  Parity-reduced: starting
// from j = 0 on the ground surface, the couplings (j -> j +- 1, surfaces
// swapped) only ever populate (ground, even j) and (excited, odd j), so only
// those rows are stored: ground rows are the even-j channels, excited rows
// the odd-j channels, each in channel order.
template <int J, bool PAR>
struct Rows {
  static constexpr int NROT = (J + 1) * (J + 1);
  static constexpr int count(int q) {  // channels of j parity q up to J
    int n = 0;
    for (int j = q; j <= J; j += 2) n += 2 * j + 1;
    return n;
  }
  static constexpr int NG = PAR ? count(0) : NROT;  // ground rows
  static constexpr int NE = PAR ? count(1) : NROT;  // excited rows
  static constexpr int ROWS = NG + NE;
  static constexpr int N(int sf) { return sf ? NE : NG; }
  static constexpr int base(int sf) { return sf ? NG : 0; }  // first row of surface sf
  // channel stored in row r of surface sf
  static constexpr int chan(int sf, int r) {
    if (!PAR) return r;
    for (int j = sf; j <= J; j += 2) {
      if (r < 2 * j + 1) return j * j + r;
      r -= 2 * j + 1;
    }
    return -1;
  }
  // row of surface sf holding channel c (-1: c outside the basis or not stored)
  static constexpr int row(int sf, int c) {
    if (c < 0) return -1;
    if (!PAR) return c;
    const int j = ch_j(c);
    if ((j & 1) != sf) return -1;
    int r = 0;
    for (int jj = sf; jj < j; jj += 2) r += 2 * jj + 1;
    return r + (c - j * j);
  }
};

// i (theta/n) (M in) for row R of either surface, M = E'_z Z + (E'_x - i E'_y)/2 S+
// + (E'_x + i E'_y)/2 S- (the molecule-frame coupling), `in` the other
// surface's rows; f = (theta E'_z, theta E'_x/2, theta E'_y/2)
template <int J, int R, class V>
__device__ __forceinline__ float2 coupling_row(const V& in, float fz, float fx, float fy, float cn) {
  constexpr int j = ch_j(R), mm = ch_m(R);
  float2 az = make_float2(0.f, 0.f), ap = az, am = az;
  auto mac = [&](float2& a, float cf, auto ni) {
    constexpr int q = decltype(ni)::value;
    if constexpr (q >= 0) {
      a.x = fmaf(cf, in[q].x, a.x);
      a.y = fmaf(cf, in[q].y, a.y);
    }
  };
  if constexpr (j < J) {
    mac(az, c_zu(j, mm), std::integral_constant<int, (ch_of(j + 1, mm, J))>());
    mac(ap, c_pu(j, mm), std::integral_constant<int, (ch_of(j + 1, mm - 1, J))>());
    mac(am, c_mu(j, mm), std::integral_constant<int, (ch_of(j + 1, mm + 1, J))>());
  }
  if constexpr (j > 0) {
    mac(az, c_zd(j, mm), std::integral_constant<int, c_zd(j, mm) != 0.f ? (ch_of(j - 1, mm, J)) : -1>());
    mac(ap, c_pd(j, mm),
        std::integral_constant<int, c_pd(j, mm) != 0.f ? (ch_of(j - 1, mm - 1, J)) : -1>());
    mac(am, c_md(j, mm),
        std::integral_constant<int, c_md(j, mm) != 0.f ? (ch_of(j - 1, mm + 1, J)) : -1>());
  }
  // a = fz Z-part + fx (S+ + S-) - i fy (S+ - S-)
  const float bx = ap.x + am.x, by = ap.y + am.y, cx = ap.x - am.x, cy = ap.y - am.y;
  const float ax = fmaf(fz, az.x, fmaf(fx, bx, fy * cy));
  const float ay = fmaf(fz, az.y, fmaf(fx, by, -fy * cx));
  return make_float2(-cn * ay, cn * ax);
}

// Dipole sums of ground rows [R0, R1): sum_c conj(g_c) (A e)_c for A = S+, S-,
// Z (g the ground rows, e the excited rows at one radial point)
template <int J, bool PAR, int R, class V, class W>
__device__ __forceinline__ void dipole_row(const V& gv, const W& ev, float2& accP, float2& accM, float2& accZ) {
  using L = Rows<J, PAR>;
  constexpr int C = L::chan(0, R), j = ch_j(C), mm = ch_m(C);
  float2 wP = make_float2(0.f, 0.f), wZ = wP, wM = wP;
  auto mac = [&](float2& a, float cf, auto ni) {
    constexpr int q = decltype(ni)::value;
    if constexpr (q >= 0) {
      a.x = fmaf(cf, ev[q].x, a.x);
      a.y = fmaf(cf, ev[q].y, a.y);
    }
  };
  if constexpr (j < J) {
    mac(wZ, c_zu(j, mm), std::integral_constant<int, L::row(1, ch_of(j + 1, mm, J))>());
    mac(wP, c_pu(j, mm), std::integral_constant<int, L::row(1, ch_of(j + 1, mm - 1, J))>());
    mac(wM, c_mu(j, mm), std::integral_constant<int, L::row(1, ch_of(j + 1, mm + 1, J))>());
  }
  if constexpr (j > 0) {
    mac(wZ, c_zd(j, mm), std::integral_constant<int, c_zd(j, mm) != 0.f ? L::row(1, ch_of(j - 1, mm, J)) : -1>());
    mac(wP, c_pd(j, mm), std::integral_constant<int, c_pd(j, mm) != 0.f ? L::row(1, ch_of(j - 1, mm - 1, J)) : -1>());
    mac(wM, c_md(j, mm), std::integral_constant<int, c_md(j, mm) != 0.f ? L::row(1, ch_of(j - 1, mm + 1, J)) : -1>());
  }
  const float2 gc = gv[R];
  accZ.x += fmaf(gc.x, wZ.x, gc.y * wZ.y);
  accZ.y += fmaf(gc.x, wZ.y, -gc.y * wZ.x);
  accP.x += fmaf(gc.x, wP.x, gc.y * wP.y);
  accP.y += fmaf(gc.x, wP.y, -gc.y * wP.x);
  accM.x += fmaf(gc.x, wM.x, gc.y * wM.y);
  accM.y += fmaf(gc.x, wM.y, -gc.y * wM.x);
}
template <int J, bool PAR, int R0, int R1, class V, class W>
__device__ __forceinline__ void dipole_rows(const V& gv, const W& ev, float2& accP, float2& accM, float2& accZ) {
  if constexpr (R0 < R1) {
    dipole_row<J, PAR, R0>(gv, ev, accP, accM, accZ);
    dipole_rows<J, PAR, R0 + 1, R1>(gv, ev, accP, accM, accZ);
  }
}

// Point-resident R-space pass (and, FUSED, the kinetic pass) of states with
// every row populated (the reachable rows run on whole rotors, mol_rotor.cu):
// one CTA of 2 N_r threads per molecule, thread = (radial point, surface).
// FUSED (N_r = 128): the state is staged once into D and turned in place into
// d2 = (T - 1) s by the shared-memory FFT, while a second copy of s (an L2
// hit) fills X.  Otherwise d2 comes from the kinetic kernel's scratch.
template <int J, int NR, bool FUSED, bool DIPR = false>
__global__ void __launch_bounds__(2 * NR, NR <= 64 ? 4 : (NR <= 128 ? 2 : 1))
    mol_rpoint_kernel(SpeciesDev sp, MolDev md, int* err) {
  if (idle_launch(sp)) return;
  using L = Rows<J, false>;
  constexpr int ROWS = L::ROWS, NG = L::NG, NT = 2 * NR, NW = NT / 32;
  constexpr int RMAX = L::NG > L::NE ? L::NG : L::NE;
  constexpr unsigned kStateBytes = (unsigned)ROWS * NR * sizeof(float2);  // one molecule's state
  static_assert(!FUSED || NT == FFTShape<NR>::THREADS, "the fused form runs the FFT with every thread");
  extern __shared__ __align__(16) float4 smem4[];
  float2* X = reinterpret_cast<float2*>(smem4);  // [ROWS][NR]: s, then eta and the series terms, then s'
  float2* D = X + ROWS * NR;                     // [ROWS][NR]: d2
  float2* s_tw = D + ROWS * NR;                  // fused: [N2][N1] FFT twiddles
  float2* s_kd = s_tw + NR;                      // fused: [NR] kinetic phase deltas
  __shared__ __align__(8) unsigned long long s_bar[2];
  __shared__ float s_rot[9];
  __shared__ double s_mu[3], s_abs[2];
  __shared__ float s_red[NW][10];
  __shared__ float s_fin[8], s_fin_lo[2];

  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int sf = t >= NR, p = t - sf * NR;  // surface (warp-uniform) and radial point
  const int lm = blockIdx.x;
  const int m = sp.mol[lm];
  const long long mol0 = (long long)lm * sp.mrows * NR;  // first element of this molecule's state
  const int own0 = sf ? NG : 0, oth0 = sf ? 0 : NG;   // first rows of this and the other surface
  float2* gs = sp.psi + mol0 + (long long)own0 * NR + p;
  float2* Xo = X + own0 * NR + p;        // own rows
  const float2* Xt = X + oth0 * NR + p;  // the other surface's rows
  const float2* Do = D + own0 * NR + p;
  const float2* vdp = sp.vdelta + sf * (J + 1) * NR + p;
  const float2* vhp = sp.vhalf + sf * (J + 1) * NR + p;

  // the molecule's state (and d2), one bulk copy each (contiguous in global memory)
  if (t == 0) {
    mbar_init(&s_bar[0], 1);
    mbar_init(&s_bar[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (FUSED) {
      mbar_expect_tx(&s_bar[0], kStateBytes);
      bulk_g2s(D, sp.psi + mol0, kStateBytes, &s_bar[0]);
    } else {
      mbar_expect_tx(&s_bar[0], 2 * kStateBytes);
      bulk_g2s(X, sp.psi + mol0, kStateBytes, &s_bar[0]);
      bulk_g2s(D, sp.d2 + (long long)lm * ROWS * NR, kStateBytes, &s_bar[0]);
    }
  }
  if (FUSED) {
    for (int q = t; q < NR; q += NT) {
      s_tw[q] = __ldg(&sp.twiddle[q]);
      s_kd[q] = __ldg(&sp.kdelta[q]);
    }
  }
  if (t >= 32 && t < 41) s_rot[t - 32] = md.rot[9 * (long long)m + (t - 32)];
  else if (t >= 64 && t < 67) s_mu[t - 64] = md.mu[3 * (long long)m + (t - 64)];
  else if (t >= 67 && t < 69) s_abs[t - 67] = md.absorbed[2 * (long long)m + (t - 67)];
  // theta E' of the molecule, times d(R) / max|d| at this thread's point
  // (1 for a constant dipole)
  float4 f = __ldg(&sp.fld[lm]);
  if constexpr (DIPR) {
    const float dw = __ldg(&sp.dipw[p]);
    f.x *= dw;
    f.y *= dw;
    f.z *= dw;
  }
  const int nterms = __float_as_int(f.w);
  const float mk = sp.maskw[p].x;
  const float cfix = md.ncorr[m];  // rounding feedback of the previous step
  float2 vh[J + 1], vd[J + 1];
#pragma unroll
  for (int j = 0; j <= J; ++j) {
    vd[j] = __ldg(vdp + j * NR);
    vh[j] = __ldg(vhp + j * NR);
  }
  __syncthreads();  // the barrier is initialised
  auto wait_all = [&](int id) -> bool {
    const bool ok = mbar_wait_sleep(&s_bar[id], 0);
    if (__syncthreads_and(ok)) return true;
    if (t == 0) atomicOr(err, kErrTimeout);
    if (!ok) mbar_wait_sleep(&s_bar[id], 0);
    return false;
  };
  if (!wait_all(0)) return;
  if (FUSED) {
    if (t == 0) {  // s again into X (the lines were just read), while the FFT runs on D
      mbar_expect_tx(&s_bar[1], kStateBytes);
      bulk_g2s(X, sp.psi + mol0, kStateBytes, &s_bar[1]);
    }
    kinetic_pass<NR>(D, D, ROWS, s_kd, s_tw);  // D <- d2 = (T - 1) s
    if (!wait_all(1)) return;
  }
  // ---- eta = V^{1/2} u, u = s + d2, over this thread's own rows of the state
  if (nterms > 0)
    static_for<0, L::NROT>([&](auto ri) {
      constexpr int r = decltype(ri)::value, j = ch_j(r);
      Xo[r * NR] = cmul(vh[j], Xo[r * NR] + Do[r * NR]);
    });
  __syncthreads();
  // ---- coupling series: S = sum_n (i theta M sigma_x)^n eta / n!
  float2 sacc[RMAX], in[RMAX];
#pragma unroll
  for (int r = 0; r < RMAX; ++r) sacc[r] = make_float2(0.f, 0.f);
  auto term = [&](float cn, bool store) {
    static_for<0, L::NROT>([&](auto ri) {
      constexpr int r = decltype(ri)::value;
      const float2 o = coupling_row<J, r>(in, f.x, f.y, f.z, cn);
      sacc[r].x += o.x;
      sacc[r].y += o.y;
      if (store) Xo[r * NR] = o;
    });
  };
  for (int n = 1; n <= nterms; ++n) {
#pragma unroll
    for (int r = 0; r < RMAX; ++r) in[r] = Xt[r * NR];
    __syncthreads();  // every thread has its input: the buffer may be overwritten
    const float cn = 1.f / (float)n;
    const bool store = n < nterms;
    term(cn, store);
    if (store) __syncthreads();
  }
  // ---- d1 = (V - 1) u + V^{1/2} S ; mask ; s' = s + (d2 + d1) + cfix s
  float sn2 = 0.f, sn2_lo = 0.f, absd = 0.f, rnd = 0.f;  // |s'|^2 compensated from the first term on
  {
    constexpr int NO = L::NROT;
    // s again (from L2), in two batches each requested in full first; d2 from shared memory
    constexpr int NB = NO > 1 ? (NO + 1) / 2 : 1;
    float2 sb[NB];
    auto fetch = [&](int r0) {
#pragma unroll
      for (int k = 0; k < NB; ++k)
        if (r0 + k < NO) sb[k] = __ldcs(gs + (r0 + k) * NR);
    };
    fetch(0);
    static_for<0, NO>([&](auto ri) {
      constexpr int r = decltype(ri)::value, j = ch_j(r);
      if constexpr (r == NB) fetch(NB);
      const float2 sv = sb[r % NB], dv = Do[r * NR];
      const float2 u = sv + dv;
      float2 d1 = cmul(vd[j], u);
      if (nterms > 0) d1 = d1 + cmul(vh[j], sacc[r]);
      if (mk < 1.f) {
        const float px = u.x + d1.x, py = u.y + d1.y;
        d1.x = fmaf(mk - 1.f, u.x, mk * d1.x);
        d1.y = fmaf(mk - 1.f, u.y, mk * d1.y);
        absd += (1.f - mk * mk) * fmaf(px, px, py * py);
      }
      const float2 s1 = round_update(sv, dv + d1, cfix, rnd);
      __stcs(gs + r * NR, s1);
      acc2(sn2, sn2_lo, fmaf(s1.x, s1.x, s1.y * s1.y));
      sacc[r] = s1;  // the new state of this surface, kept for the dipole
      Xo[r * NR] = s1;
    });
  }
  __syncthreads();
  // ---- dipole in the molecule frame: sum over ground rows of conj(g_c) (A e)_c
  // for A = Z, S+, S-; ground rows [0, NH) on the ground-surface threads, the
  // rest on the excited ones
  float dP = 0.f, dQ = 0.f, dZ = 0.f;
  {
    constexpr int NH = (NG + 1) / 2;
#pragma unroll
    for (int r = 0; r < RMAX; ++r) in[r] = Xt[r * NR];
    float2 accP = make_float2(0.f, 0.f), accM = accP, accZ = accP;
    if (sf == 0) dipole_rows<J, false, 0, NH>(sacc, in, accP, accM, accZ);
    else dipole_rows<J, false, NH, NG>(in, sacc, accP, accM, accZ);
    dP = accP.x + accM.x;
    dQ = accP.y - accM.y;
    dZ = 2.f * accZ.x;
  }
  // ---- block reduction: populations compensated, the rest plain FP32
  {
    float v[8] = {sf ? 0.f : sn2, sf ? sn2 : 0.f, sf ? 0.f : absd, sf ? absd : 0.f, dP, dQ, dZ, rnd};
    float lo[2] = {sf ? 0.f : sn2_lo, sf ? sn2_lo : 0.f};
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const float h2 = __shfl_xor_sync(0xffffffffu, v[k], o);
        const float l2 = __shfl_xor_sync(0xffffffffu, lo[k], o);
        acc2(v[k], lo[k], h2);
        lo[k] += l2;
      }
#pragma unroll
      for (int k = 2; k < 8; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    }
    if (lane == 0) {
#pragma unroll
      for (int k = 0; k < 7; ++k) s_red[w][k] = v[k];
      s_red[w][7] = lo[0];
      s_red[w][8] = lo[1];
      s_red[w][9] = v[7];
    }
    __syncthreads();
    if (t < 8) {
      float hi = 0.f, l = 0.f;
      for (int ww = 0; ww < NW; ++ww) {
        acc2(hi, l, s_red[ww][t < 7 ? t : 9]);
        if (t < 2) l += s_red[ww][7 + t];
      }
      s_fin[t] = hi + l;
      if (t < 2) s_fin_lo[t] = l - (s_fin[t] - hi);
    }
    __syncthreads();
    if (t < 3) {  // lab dipole: mu = O mu', mu' = d dR (Re(S+ + S-), Im(S+ - S-), 2 Re Z)
      if constexpr (!DIPR) {  // with d(R) the dipole is read from T^{1/2} s' by mol_dipole_r_kernel
        const float sc = (float)sp.dipole * sp.dR;
        const float lab = sc * (s_rot[3 * t] * s_fin[4] + s_rot[3 * t + 1] * s_fin[5] + s_rot[3 * t + 2] * s_fin[6]);
        const double nl = (double)lab;
        md.dmu[3 * (long long)m + t] = nl - s_mu[t];
        md.mu[3 * (long long)m + t] = nl;
      }
    } else if (t < 5) {
      const double P = ((double)s_fin[t - 3] + (double)s_fin_lo[t - 3]) * (double)sp.dR;
      md.pop[2 * (long long)m + (t - 3)] = P;
      if (!isfinite(P)) atomicOr(err, kErrNonFinite);
    } else if (t < 7) {
      md.absorbed[2 * (long long)m + (t - 5)] = s_abs[t - 5] + (double)s_fin[t - 3] * (double)sp.dR;
    } else if (t == 7) {
      md.ncorr[m] = rounding_feedback(s_fin[7], s_fin[0] + s_fin[1]);
    }
  }
}

template <int J, int NR, bool FUSED, bool DIPR = false>
static void launch_rpoint_jnd(const SpeciesDev& sp, const MolDev& md, int* err, cudaStream_t s) {
  constexpr int ROWS = Rows<J, false>::ROWS;
  const size_t smem = (size_t)2 * ROWS * NR * sizeof(float2) + (FUSED ? 2 * NR * sizeof(float2) : 0);
  auto k = mol_rpoint_kernel<J, NR, FUSED, DIPR>;
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  k<<<sp.nmol, 2 * NR, smem, s>>>(sp, md, err);
}
template <int J, int NR, bool FUSED>
static void launch_rpoint_jn(const SpeciesDev& sp, const MolDev& md, int* err, cudaStream_t s) {
  if constexpr (NR <= 128) {  // R-dependent dipole: N_r 64 or 128
    if (sp.dipw) {
      launch_rpoint_jnd<J, NR, FUSED, true>(sp, md, err, s);
      return;
    }
  }
  launch_rpoint_jnd<J, NR, FUSED>(sp, md, err, s);
}

template <int NR, bool FUSED = false>
static void launch_rpoint_n(const SpeciesDev& sp, const MolDev& md, int* err, cudaStream_t s) {
  if (sp.par) {
    launch_rotor(sp, md, err, s);
    return;
  }
  switch (sp.jmax) {
    case 0: launch_rpoint_jn<0, NR, FUSED>(sp, md, err, s); break;
    case 1: launch_rpoint_jn<1, NR, FUSED>(sp, md, err, s); break;
    case 2: launch_rpoint_jn<2, NR, FUSED>(sp, md, err, s); break;
    case 3: launch_rpoint_jn<3, NR, FUSED>(sp, md, err, s); break;
    case 4: launch_rpoint_jn<4, NR, FUSED>(sp, md, err, s); break;
  }
}

// Dipole of a species with an R-dependent transition dipole d(R).  The
// stored state is s = T^{-1/2} psi; the populations are the same from s and
// psi (T^{1/2} is unitary per channel), and so is the dipole while d is
// constant (T commutes with d sigma_x (x) R^).  With d(R) it does not, so the
// dipole is taken from psi' = T^{1/2} s' after the step: one CTA per
// molecule stages s', turns it into psi' with the shared-memory FFT and sums
// 2 Re sum_R d(R) g^dagger A e dR for A = S+, S-, Z (threads t < N_r: one
// radial point each), then writes mu and the change over the step.
template <int J, int NR, bool PAR>
__global__ void __launch_bounds__(FFTShape<NR>::THREADS) mol_dipole_r_kernel(SpeciesDev sp, MolDev md, int* err) {
  if (idle_launch(sp)) return;
  using L = Rows<J, PAR>;
  constexpr int ROWS = L::ROWS, NG = L::NG, NE = L::NE, NT = FFTShape<NR>::THREADS, NW = NT / 32;
  constexpr unsigned kStateBytes = (unsigned)ROWS * NR * sizeof(float2);
  extern __shared__ __align__(16) float4 smem4[];
  float2* X = reinterpret_cast<float2*>(smem4);  // [ROWS][NR]: s', then psi'
  float2* s_tw = X + ROWS * NR;
  float2* s_kh = s_tw + NR;
  __shared__ __align__(8) unsigned long long s_bar[1];
  __shared__ float s_red[NW][3];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int lm = blockIdx.x;
  const int m = sp.mol[lm];
  if (t == 0) {
    mbar_init(&s_bar[0], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect_tx(&s_bar[0], kStateBytes);
    bulk_g2s(X, sp.psi + (long long)lm * sp.mrows * NR, kStateBytes, &s_bar[0]);
  }
  for (int q = t; q < NR; q += NT) {
    s_tw[q] = __ldg(&sp.twiddle[q]);
    s_kh[q] = __ldg(&sp.khalf[q]);
  }
  __syncthreads();
  const bool ok = mbar_wait_sleep(&s_bar[0], 0);
  if (!__syncthreads_and(ok)) {
    if (t == 0) atomicOr(err, kErrTimeout);
    if (!ok) mbar_wait_sleep(&s_bar[0], 0);
    return;
  }
  kinetic_pass<NR>(X, X, ROWS, s_kh, s_tw);  // psi' = T^{1/2} s'
  float dP = 0.f, dQ = 0.f, dZ = 0.f;
  if (t < NR) {
    float2 gv[NG], ev[NE > 0 ? NE : 1];  // J = 0, parity-reduced: no excited row
#pragma unroll
    for (int r = 0; r < NG; ++r) gv[r] = X[r * NR + t];
#pragma unroll
    for (int r = 0; r < NE; ++r) ev[r] = X[(NG + r) * NR + t];
    float2 accP = make_float2(0.f, 0.f), accM = accP, accZ = accP;
    dipole_rows<J, PAR, 0, NG>(gv, ev, accP, accM, accZ);
    const float d = (float)sp.dipole * __ldg(&sp.dipw[t]);
    dP = d * (accP.x + accM.x);
    dQ = d * (accP.y - accM.y);
    dZ = d * 2.f * accZ.x;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    dP += __shfl_xor_sync(0xffffffffu, dP, o);
    dQ += __shfl_xor_sync(0xffffffffu, dQ, o);
    dZ += __shfl_xor_sync(0xffffffffu, dZ, o);
  }
  if (lane == 0) {
    s_red[w][0] = dP;
    s_red[w][1] = dQ;
    s_red[w][2] = dZ;
  }
  __syncthreads();
  if (t < 3) {
    float v[3] = {0.f, 0.f, 0.f};
    for (int ww = 0; ww < NW; ++ww)
      for (int k = 0; k < 3; ++k) v[k] += s_red[ww][k];
    const float* O = md.rot + 9 * (long long)m;  // molecule -> lab, row-major
    const double lab = (double)(sp.dR * (O[3 * t] * v[0] + O[3 * t + 1] * v[1] + O[3 * t + 2] * v[2]));
    md.dmu[3 * (long long)m + t] = lab - md.mu[3 * (long long)m + t];
    md.mu[3 * (long long)m + t] = lab;
  }
}

template <int J, int NR>
static void launch_dipole_r_jn(const SpeciesDev& sp, const MolDev& md, int* err, cudaStream_t s) {
  auto run = [&](auto k, int rows) {
    const size_t smem = ((size_t)rows * NR + 2 * NR) * sizeof(float2);
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k<<<sp.nmol, FFTShape<NR>::THREADS, smem, s>>>(sp, md, err);
  };
  if (sp.par) run(mol_dipole_r_kernel<J, NR, true>, Rows<J, true>::ROWS);
  else run(mol_dipole_r_kernel<J, NR, false>, Rows<J, false>::ROWS);
}

template <int NR>
static void launch_dipole_r(const SpeciesDev& sp, const MolDev& md, int* err, cudaStream_t s) {
  switch (sp.jmax) {
    case 0: launch_dipole_r_jn<0, NR>(sp, md, err, s); break;
    case 1: launch_dipole_r_jn<1, NR>(sp, md, err, s); break;
    case 2: launch_dipole_r_jn<2, NR>(sp, md, err, s); break;
    case 3: launch_dipole_r_jn<3, NR>(sp, md, err, s); break;
    case 4: launch_dipole_r_jn<4, NR>(sp, md, err, s); break;
  }
}

// The point-resident kernel runs a species' R-space pass (and, fused, its
// kinetic pass) where it applies (J <= 4; fused only at N_r = 128) unless the
// species' plan names another kernel.
static bool use_point(const SpeciesDev& sp) {
  if (sp.jmax > 4 || (sp.path == MS_MOL_FUSED && sp.nr != 128)) return false;
  return sp.kern == MS_KERN_DEFAULT || sp.kern == MS_KERN_POINT;
}
static bool rspace_ok(int nr, int jmax);
// The tiled kernel runs a streaming species' R-space pass where the point-
// resident one does not and it applies, unless the plan names another kernel.
static bool pair_ok(int nr, int jmax) { return (nr == 64 || nr == 128 || nr == 256) && jmax <= 16; }
// The column kernel runs the reachable rows of a streaming species from J = 5
// to 8: 5.9 to 6.5 ps a row and point at N_r = 128, 5.8 to 6.4 at 256 and 6.6 to 6.9 at 64,
// against 8.0 for the two-points-a-thread kernel.  Below, a thread holds the
// whole rotor; above, half a side's columns no longer fit a thread's registers.
static bool use_col(const SpeciesDev& sp) {
  return sp.path == MS_MOL_STREAMING && sp.par && sp.jmax >= 5 && sp.jmax <= 8;
}
// The two-points-a-thread tiled kernel runs a streaming species' R-space pass
// where the plan names it, and by the static rule from J = 5 on (from J = 9 on
// for the reachable rows).
static bool use_pair(const SpeciesDev& sp) {
  if (sp.path != MS_MOL_STREAMING || sp.dipw || !pair_ok(sp.nr, sp.jmax)) return false;
  if (sp.par) return sp.jmax >= 9;
  return sp.kern == MS_KERN_PAIR || (sp.kern == MS_KERN_DEFAULT && sp.jmax >= 5);
}
static bool use_tile(const SpeciesDev& sp) {
  if (sp.path != MS_MOL_STREAMING || use_point(sp) || use_col(sp) || use_pair(sp) || !rspace_ok(sp.nr, sp.jmax))
    return false;
  return sp.kern == MS_KERN_DEFAULT || sp.kern == MS_KERN_TILE;
}
// its tile width: 8 points from J = 9 on; else the plan's, or 8 points from
// J = 5 on (the nanohole pass 113.7 against 118.3 ms at 16) and 32 below
static int pair_tile(const SpeciesDev& sp) {
  if (sp.jmax >= 9) return 8;
  if (sp.ch == 8 || sp.ch == 16 || sp.ch == 32) return sp.ch;
  return sp.jmax >= 5 ? 8 : 32;
}
}  // namespace ms

// ----------------------------------------------------------------------------
// Eq. 8 readout: psi = T^{1/2} s on the excited surface, then
// <chi_e|R|chi_e> and <chi_e|chi_e> per molecule: a row's sums in FP32 pairs that
// take every rounding of the additions and of r |psi|^2 (about 48 bits), rows in FP64
// ----------------------------------------------------------------------------
namespace ms {

// A CTA takes `mpb` molecules whose excited rows fill an FFT block (one where a
// molecule has more, in blocks of RB rows).  Each row's sums of |psi|^2 and
// r |psi|^2 are taken from the transform's registers, compensated, over the N1
// lanes that share the row, and summed in FP64 per molecule.  With a molecule a
// CTA and psi brought back to shared memory 50,000 molecules at J = 4 (ten
// excited rows) took 1.27 ms.
template <int NR>
constexpr int kObserveRows = 8192 / NR;  // rows of a block at most: 64 KB

template <int NR>
__global__ void __launch_bounds__(FFTShape<NR>::THREADS)
    mol_observe_kernel(SpeciesDev sp, MolDev md, int RB, int mpb, int* err) {
  constexpr int N1 = FFTShape<NR>::N1, N2 = FFTShape<NR>::N2;
  extern __shared__ float4 smem4[];
  float2* s_tw = reinterpret_cast<float2*>(smem4);
  float2* s_kh = s_tw + NR;
  float2* st = s_kh + NR;
  __shared__ __align__(8) unsigned long long s_bar;
  __shared__ double s_row[kObserveRows<NR>][2];
  const int t = threadIdx.x;
  const int ne = sp.rows - sp.rows_g;  // excited rows
  const int l0 = blockIdx.x * mpb, nm = min(mpb, sp.nmol - l0);
  if (t == 0) {
    mbar_init(&s_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int q = t; q < NR; q += blockDim.x) {
    s_tw[q] = __ldg(&sp.twiddle[q]);
    s_kh[q] = __ldg(&sp.khalf[q]);
  }
  double num = 0.0, den = 0.0;
  unsigned phase = 0;
  for (int b0 = 0; b0 < ne; b0 += RB) {  // one pass unless a molecule has more than RB rows (mpb = 1)
    const int nb = mpb > 1 ? nm * ne : min(RB, ne - b0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the last pass's rows before the copy over them
    __syncthreads();  // the barrier is initialised; the rows and sums of the last pass are read
    if (t == 0) {
      mbar_expect_tx(&s_bar, (unsigned)(nb * NR * sizeof(float2)));
      const int per = mpb > 1 ? ne : nb;
      for (int k = 0; k * per < nb; ++k)
        bulk_g2s(st + k * per * NR, sp.psi + ((long long)(l0 + k) * sp.mrows + sp.rows_g + b0) * NR,
                 (unsigned)(per * NR * sizeof(float2)), &s_bar);
    }
    const bool ok = mbar_wait_sleep(&s_bar, phase);
    if (!__syncthreads_and(ok)) {
      if (t == 0) atomicOr(err, kErrTimeout);
      if (!ok) mbar_wait_sleep(&s_bar, phase);
      return;
    }
    phase ^= 1;
    kinetic_pass<NR, FFTShape<NR>::THREADS, false>(st, st, nb, s_kh, s_tw, [&](int row, int n1, float2(&x)[N2]) {
      float dh = 0.f, dl = 0.f, nh = 0.f, nl = 0.f;  // psi = T^{1/2} s
      if (row < nb) {
#pragma unroll
        for (int n2 = 0; n2 < N2; ++n2) {
          const float a = fmaf(x[n2].x, x[n2].x, x[n2].y * x[n2].y), r = __ldg(&sp.r[n1 + N1 * n2]);
          const float p = a * r;
          acc2(dh, dl, a);
          acc2(nh, nl, p);
          nl += fmaf(a, r, -p);
        }
      }
#pragma unroll
      for (int o = N1 / 2; o > 0; o >>= 1) {
        const float dh2 = __shfl_xor_sync(0xffffffffu, dh, o), dl2 = __shfl_xor_sync(0xffffffffu, dl, o);
        const float nh2 = __shfl_xor_sync(0xffffffffu, nh, o), nl2 = __shfl_xor_sync(0xffffffffu, nl, o);
        acc2(dh, dl, dh2);
        acc2(nh, nl, nh2);
        dl += dl2;
        nl += nl2;
      }
      if (row < nb && n1 == 0) {
        s_row[row][0] = (double)nh + (double)nl;
        s_row[row][1] = (double)dh + (double)dl;
      }
    });
    const int per = mpb > 1 ? ne : nb;  // kinetic_pass ends on a barrier
    if (t < (mpb > 1 ? nm : 1))
      for (int k = 0; k < per; ++k) {
        num += s_row[t * per + k][0];
        den += s_row[t * per + k][1];
      }
    if (mpb > 1) break;
  }
  if (t < nm) {
    const int m = sp.mol[l0 + t];
    md.Rnum[m] = num * sp.dR;
    md.Rden[m] = den * sp.dR;
  }
}

// initial condition: the same radial row (ground surface, j = m = 0) for
// every molecule of a species; the rest of the state is already zero
__global__ void broadcast_row_kernel(float2* psi, const float2* row, int nr, size_t per, long long nmol) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= nmol * nr) return;
  const long long m = i / nr;
  const int a = (int)(i - m * nr);
  psi[m * per + a] = row[a];
}

cudaError_t launch_broadcast_row(float2* psi, const float2* row, int nr, size_t per, long long nmol,
                                 cudaStream_t s) {
  if (nmol == 0) return cudaSuccess;
  const long long n = nmol * nr;
  broadcast_row_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(psi, row, nr, per, nmol);
  return cudaGetLastError();
}

// ----------------------------------------------------------------------------
// streaming form, first pass: the molecules' field records, by the first nfld
// blocks (a launch of their own took 4 us a step), and d2 = (T - 1) s for blocks of rows (rows of all
// molecules of a species are independent here); one bulk copy per block, or one
// per molecule that the block touches where the molecules store more rows than
// are processed
// ----------------------------------------------------------------------------
template <int NR>
__global__ void __launch_bounds__(FFTShape<NR>::THREADS)
    mol_kinetic_kernel(SpeciesDev sp, MolDev md, Grid g, int prescribed, int nfld, long long rows_total, int RB,
                       int* err) {
  if (idle_launch(sp)) return;
  if ((int)blockIdx.x < nfld) {
    const int lm = blockIdx.x * FFTShape<NR>::THREADS + threadIdx.x;
    if (lm < sp.nmol) sp.fld[lm] = field_record(sp, md, g, prescribed, sp.mol[lm], err);
    return;
  }
  extern __shared__ float4 smem4[];
  float2* s_tw = reinterpret_cast<float2*>(smem4);
  float2* s_kd = s_tw + NR;
  float2* st = s_kd + NR;
  __shared__ __align__(8) unsigned long long s_bar;
  const long long r0 = ((int)blockIdx.x - nfld) * (long long)RB;
  const int nrows = (int)min((long long)RB, rows_total - r0);
  const int t = threadIdx.x;
  if (t == 0) {
    mbar_init(&s_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (t == 0) {
    mbar_expect_tx(&s_bar, (unsigned)(nrows * NR * sizeof(float2)));
    if (sp.rows == sp.mrows) {
      bulk_g2s(st, sp.psi + r0 * NR, (unsigned)(nrows * NR * sizeof(float2)), &s_bar);
    } else {
      long long m = r0 / sp.rows;
      int k = (int)(r0 - m * sp.rows);
      for (int q = 0; q < nrows; ++m, k = 0) {
        const int len = min(sp.rows - k, nrows - q);
        bulk_g2s(st + q * NR, sp.psi + (m * sp.mrows + k) * NR, (unsigned)(len * NR * sizeof(float2)), &s_bar);
        q += len;
      }
    }
  }
  for (int q = t; q < NR; q += blockDim.x) {
    s_tw[q] = __ldg(&sp.twiddle[q]);
    s_kd[q] = __ldg(&sp.kdelta[q]);
  }
  const bool ok = mbar_wait(&s_bar, 0, kWaitPolls);
  if (!__syncthreads_and(ok)) {
    if (t == 0) atomicOr(err, kErrTimeout);
    if (!ok) mbar_wait(&s_bar, 0, kWaitPolls);
    return;
  }
  kinetic_pass<NR>(st, st, nrows, s_kd, s_tw);
  const float4* s4 = reinterpret_cast<const float4*>(st);
  float4* d4 = reinterpret_cast<float4*>(sp.d2 + r0 * NR);
  for (int q = t; q < nrows * NR / 2; q += blockDim.x) d4[q] = s4[q];
}

size_t mol_state_smem(int nr, int rows) { return (size_t)rows * (nr + kPad) * sizeof(float2); }

static size_t step_smem(int nr, int nrot, int ch, bool fused) {
  const int rows = 2 * nrot;
  const int jm = (int)std::lround(std::sqrt((double)nrot)) - 1;
  const size_t nd = fused ? 0 : rows;
  return (fused ? 2 * (size_t)nr * sizeof(float2) + mol_state_smem(nr, rows) : 0) +
         2 * (size_t)rows * ch * sizeof(float2) +
         2 * (size_t)(rows + nd + 4 * (jm + 1) + 1) * ch * sizeof(float2) +
         2 * (size_t)nrot * kMaxCoupl * sizeof(int2) + (size_t)rows * sizeof(int2);
}

// rows each thread owns at chunk width ch (8 warps; 32/ch row groups per warp)
static int rows_per_thread(int nrot, int ch) {
  const int rstep = 8 * (32 / ch);
  return (2 * nrot + rstep - 1) / rstep;
}

// Launch shape of one species: chunk width, rows-per-thread bound, shared
// memory.  Fused: the widest chunk keeping two CTAs per SM.  Streaming: the
// widest chunk with at most 4 rows per thread (64 registers, four CTAs per
// SM), else at most 12.
struct StepShape {
  int ch, maxr;
  size_t smem;
  bool ok;
};
static StepShape step_shape(int nr, int nrot, bool fused) {
  // k CTAs per SM: k x (dynamic + static (< 800 B) + 1 KB reserved) <= 228 KB
  auto cap = [](int k) { return (size_t)(228 * 1024 / k - 1024 - 800); };
  if (fused) {
    for (int k : {2, 1})
      for (int ch = kChunk; ch >= 8; ch >>= 1)
        if (rows_per_thread(nrot, ch) <= 12 && step_smem(nr, nrot, ch, true) <= cap(k))
          return {ch, 12, step_smem(nr, nrot, ch, true), true};
    return {8, 12, 0, false};
  }
  for (int maxr : {4, 12, 24})
    for (int ch = kChunk; ch >= 4; ch >>= 1)
      if (rows_per_thread(nrot, ch) <= maxr &&
          step_smem(nr, nrot, ch, false) <= cap(maxr == 4 ? 4 : (maxr == 12 ? 2 : 1)))
        return {ch, maxr, step_smem(nr, nrot, ch, false), true};
  return {4, 24, 0, false};
}

bool mol_step_supported(int nr, int nrot, int path) {
  return step_shape(nr, nrot, path == MS_MOL_FUSED).ok;
}

// The chunked kernel's launch shape at a given chunk width (the plan a tuner
// picked), or ok = false where that width does not fit.
static StepShape step_shape_ch(int nr, int nrot, bool fused, int ch) {
  auto cap = [](int k) { return (size_t)(228 * 1024 / k - 1024 - 800); };
  if (ch != 4 && ch != 8 && ch != 16 && ch != 32) return {ch, 12, 0, false};
  if (fused) {
    const size_t sm = step_smem(nr, nrot, ch, true);
    return {ch, 12, sm, ch >= 8 && rows_per_thread(nrot, ch) <= 12 && sm <= cap(1)};
  }
  for (int maxr : {4, 12, 24})
    if (rows_per_thread(nrot, ch) <= maxr && step_smem(nr, nrot, ch, false) <= cap(maxr == 4 ? 4 : (maxr == 12 ? 2 : 1)))
      return {ch, maxr, step_smem(nr, nrot, ch, false), true};
  return {ch, 24, 0, false};
}

// The tiled R-space kernel covers J <= 8 (rows <= 162) at tile widths of 32
// and 16 radial points (N_r 64, 128 and 256 hold an even number of tiles).
// Its static rule: 16-point tiles from J = 5 on (two CTAs per SM), else 32.
static bool rspace_ok(int nr, int jmax) { return (nr == 64 || nr == 128 || nr == 256) && jmax <= 16; }
static int rspace_tile(const SpeciesDev& sp) {
  if (sp.jmax >= 9) return 8;
  if (sp.kern == MS_KERN_TILE && (sp.ch == 16 || sp.ch == 32)) return sp.ch;
  return sp.jmax >= 5 ? 16 : 32;
}

// The plans a species can run: (layout, kernel, chunk width).  Parity-reduced
// and d(R) species follow the rule; the mixed kinetic pass needs the streaming
// layout.  A plan that names a tiled, pair or chunked kernel processes every
// stored row.
int mol_plan_candidates(const SpeciesDev& sp, int (*out)[4], int max) {
  int n = 0;
  auto add = [&](int path, int kern, int ch, int cps = 0) {
    if (n < max) {
      out[n][0] = path;
      out[n][1] = kern;
      out[n][2] = ch;
      out[n][3] = cps;
    }
    ++n;
  };
  if (sp.bloch || sp.par_form || sp.dipw) return 0;
  // from J = 5 on the static rule's kernel, the only one there that processes
  // the reachable rows alone
  if (sp.jmax >= 5) add(MS_MOL_STREAMING, MS_KERN_DEFAULT, 0);
  if (!sp.mixed) {
    if (sp.nr == 128 && sp.jmax <= 4) add(MS_MOL_FUSED, MS_KERN_POINT, 0);
    for (int ch : {32, 16, 8})
      if (step_shape_ch(sp.nr, sp.nrot, true, ch).ok) add(MS_MOL_FUSED, MS_KERN_CHUNK, ch);
  }
  if (sp.jmax <= 4) add(MS_MOL_STREAMING, MS_KERN_POINT, 0);
  if (rspace_ok(sp.nr, sp.jmax)) {  // tile width x grid: as many CTAs as fit, one per SM, one per molecule
    if (sp.jmax >= 9) {
      for (int cps : {0, -1}) add(MS_MOL_STREAMING, MS_KERN_TILE, 8, cps);
    } else {
      for (int tile : {32, 16})
        for (int cps : {0, 1, -1}) add(MS_MOL_STREAMING, MS_KERN_TILE, tile, cps);
    }
  }
  if (pair_ok(sp.nr, sp.jmax)) {  // two points a thread: 32 or 16 for J <= 4, 16 or 8 to J = 8, then 8
    if (sp.jmax >= 9) {
      for (int cps : {0, 1, -1}) add(MS_MOL_STREAMING, MS_KERN_PAIR, 8, cps);
    } else {
      for (int tile : {sp.jmax <= 4 ? 32 : 16, sp.jmax <= 4 ? 16 : 8})
        for (int cps : {0, 1, -1}) add(MS_MOL_STREAMING, MS_KERN_PAIR, tile, cps);
    }
  }
  for (int ch : {32, 16, 8, 4})
    if (step_shape_ch(sp.nr, sp.nrot, false, ch).ok) add(MS_MOL_STREAMING, MS_KERN_CHUNK, ch);
  return n < max ? n : max;
}

// cuTensorMapEncodeTiled, looked up once through the runtime
static PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    else
      cudaGetLastError();
  });
  return fn;
}

// [nrows][nr] array of complex FP32 values (8-byte elements), box tile x box_rows
static bool encode_rows(CUtensorMap* m, const void* base, unsigned long long nr, unsigned long long nrows,
                        unsigned box_rows, unsigned tile) {
  const PFN_cuTensorMapEncodeTiled_v12000 fn = tensor_map_encoder();
  if (!fn || !base) return false;
  const cuuint64_t dims[2] = {nr, nrows};
  const cuuint64_t strides[1] = {nr * sizeof(float2)};
  const cuuint32_t box[2] = {(cuuint32_t)tile, box_rows};
  const cuuint32_t es[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_INT64, 2, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The species' tensor maps, encoded on first use of a given set of arrays
// (a few entries are kept: each handle, and the allocation-free scratch).
static bool rspace_maps(const SpeciesDev& sp, int tile, bool pair, RspaceMaps* out) {
  struct Entry {
    const void *psi, *d2, *vd, *vh, *mk;
    int nmol, nr, rows, mrows, tile;
    RspaceMaps maps;
  };
  static std::mutex mu;
  static std::vector<Entry> cache;
  std::lock_guard<std::mutex> lock(mu);
  // the pair kernel reads the potential and mask tables in its pair layout
  const float2 *vd = pair ? sp.vdelta_pp : sp.vdelta, *vh = pair ? sp.vhalf_pp : sp.vhalf,
               *mk = pair ? sp.maskw_pp : sp.maskw;
  for (const Entry& e : cache)
    if (e.psi == sp.psi && e.d2 == sp.d2 && e.vd == vd && e.vh == vh && e.mk == mk && e.nmol == sp.nmol &&
        e.nr == sp.nr && e.rows == sp.rows && e.mrows == sp.mrows && e.tile == tile) {
      *out = e.maps;
      return true;
    }
  Entry e{sp.psi, sp.d2, vd, vh, mk, sp.nmol, sp.nr, sp.rows, sp.mrows, tile, {}};
  const unsigned rows = sp.rows, nv = 2 * (sp.jmax + 1);  // processed rows a molecule
  const unsigned boxr = rows < 256 ? rows : 256, lastr = rows - (rows + boxr - 1) / boxr * boxr + boxr;
  const unsigned long long nr = sp.nr, nrows = (unsigned long long)sp.nmol * rows,
                           srows = (unsigned long long)sp.nmol * sp.mrows;
  if (!encode_rows(&e.maps.s, sp.psi, nr, srows, boxr, tile) || !encode_rows(&e.maps.d2, sp.d2, nr, nrows, boxr, tile) ||
      !encode_rows(&e.maps.s_r, sp.psi, nr, srows, lastr, tile) ||
      !encode_rows(&e.maps.d2_r, sp.d2, nr, nrows, lastr, tile) ||
      !encode_rows(&e.maps.vd, vd, nr, nv, nv, tile) || !encode_rows(&e.maps.vh, vh, nr, nv, nv, tile) ||
      !encode_rows(&e.maps.mk, mk, nr, 1, 1, tile))
    return false;
  if (cache.size() >= 32) cache.erase(cache.begin());
  cache.push_back(e);
  *out = e.maps;
  return true;
}

bool mol_tensor_maps_available() { return tensor_map_encoder() != nullptr; }

// ---- the rows a species processes -------------------------------------------
// The point-resident kernels and, from J = 5 on, the static rule's kernel work
// on the reachable rows alone: half of a full-form state's bytes and work (its
// other rows are zeros before and after every step).  Plans that name another
// kernel process every row.  A step over every row against one over the
// reachable ones: 22.0 and 9.9 ms with 100,000 molecules at J = 8, N_r = 128
// (streaming), 2.70 and 1.16 ms with 50,000 at J = 4, N_r = 128 (fused).
bool mol_reachable_rows(const SpeciesDev& sp) {
  if (sp.par_form) return true;
  if (sp.all_rows || sp.keep_all) return false;
  return use_point(sp) ||
         (sp.path == MS_MOL_STREAMING && sp.kern == MS_KERN_DEFAULT && sp.jmax >= 5 &&
          (sp.jmax <= 8 || mol_tensor_maps_available()));
}

void mol_set_rows(SpeciesDev& sp, bool reachable) {
  sp.par = reachable ? 1 : 0;
  sp.rows = reachable ? sp.nrot : 2 * sp.nrot;
  sp.rows_g = sp.nrot;
  if (reachable) {
    sp.rows_g = 0;
    for (int j = 0; j <= sp.jmax; j += 2) sp.rows_g += 2 * j + 1;
  }
}

bool mol_both_orders(const SpeciesDev& sp, SpeciesDev v[2]) {
  v[0] = v[1] = sp;
  mol_set_rows(v[0], false);
  v[1].all_rows = 0;
  if (!mol_reachable_rows(v[1])) {  // a plan that names a kernel for every row: the rule's kernel for the reachable ones
    v[1].kern = MS_KERN_DEFAULT;
    v[1].ch = v[1].cps = 0;
  }
  if (!mol_reachable_rows(v[1])) return false;
  mol_set_rows(v[1], true);
  v[0].guard = v[1].guard = 1;
  return true;
}

namespace {
// Channel-order row (surface x n_rot + channel) of row p in the order
// (ground, even j), (excited, odd j), (ground, odd j), (excited, even j).
__device__ __forceinline__ int channel_row(int p, int nrot, int J) {
  for (int run = 0; run < 4; ++run) {
    const int sf = run & 1;
    for (int j = run < 2 ? sf : 1 - sf; j <= J; j += 2) {
      if (p < 2 * j + 1) return sf * nrot + j * j + p;
      p -= 2 * j + 1;
    }
  }
  return 0;
}

constexpr int kOrderPoints = 16;

// A block turns kOrderPoints radial points of one molecule, every row staged in
// shared memory (16 points: 128 contiguous bytes a row, at most 74 KB).  Bound by
// HBM; it runs when a state is saved or loaded or a plan changes, not in a step.
__global__ void order_rows_kernel(float2* psi, int mrows, int nrot, int J, int nr, int reachable_first) {
  extern __shared__ float4 smem4[];
  float2* st = reinterpret_cast<float2*>(smem4);
  float2* g = psi + (long long)blockIdx.x * mrows * nr + blockIdx.y * kOrderPoints;
  const int x = threadIdx.x % kOrderPoints, y0 = threadIdx.x / kOrderPoints, ys = blockDim.x / kOrderPoints;
  for (int p = y0; p < mrows; p += ys) st[p * kOrderPoints + x] = g[(long long)p * nr + x];
  __syncthreads();
  for (int p = y0; p < mrows; p += ys) {
    const int c = channel_row(p, nrot, J);
    const int from = reachable_first ? c : p, to = reachable_first ? p : c;
    g[(long long)to * nr + x] = st[from * kOrderPoints + x];
  }
}

__global__ void find_other_rows_kernel(const float2* psi, int mrows, int nrot, int J, int nr, int* flag) {
  const float2* g = psi + (long long)blockIdx.x * mrows * nr;
  bool found = false;
  for (int q = threadIdx.x; q < nrot * nr; q += blockDim.x) {
    const float2 v = g[(long long)channel_row(nrot + q / nr, nrot, J) * nr + q % nr];
    found = found || !(v.x == 0.f && v.y == 0.f);
  }
  if (__syncthreads_or(found) && threadIdx.x == 0) atomicOr(flag, 1);
}
}  // namespace

cudaError_t launch_order_rows(const SpeciesDev& sp, bool reachable_first, cudaStream_t s) {
  if (sp.nmol == 0) return cudaSuccess;
  const int smem = sp.mrows * kOrderPoints * (int)sizeof(float2);
  const cudaError_t e = cudaFuncSetAttribute(order_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             2 * kMaxRot * kOrderPoints * (int)sizeof(float2));
  if (e != cudaSuccess) return e;
  order_rows_kernel<<<dim3((unsigned)sp.nmol, (unsigned)(sp.nr / kOrderPoints)), 256, smem, s>>>(
      sp.psi, sp.mrows, sp.nrot, sp.jmax, sp.nr, reachable_first ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_find_other_rows(const SpeciesDev& sp, int* flag, cudaStream_t s) {
  if (sp.nmol == 0) return cudaSuccess;
  find_other_rows_kernel<<<(unsigned)sp.nmol, 256, 0, s>>>(sp.psi, sp.mrows, sp.nrot, sp.jmax, sp.nr, flag);
  return cudaGetLastError();
}

// rows per kinetic block: 32 KB of state
static int kinetic_rows(int nr) { return 4096 / nr; }

template <int NR, bool FUSED, int MAXR>
static void launch_step_tt(const SpeciesDev& sp, const MolDev& md, const Grid& g, int prescribed, int* err,
                           const StepShape& sh, cudaStream_t s) {
  auto k = mol_step_kernel<NR, FUSED, MAXR>;
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh.smem);
  k<<<sp.nmol, FFTShape<NR>::THREADS, sh.smem, s>>>(sp, md, g, prescribed, sh.ch, err);
}

// ----------------------------------------------------------------------------
// Mixed form of the kinetic pass: d2 = (K - I) s for every row as a tensor-core
// GEMM on split FP16 operands (x = x_hi + x_lo, three products, FP32
// accumulation in tensor memory).  K is the N_r x N_r circulant of the
// kinetic propagator (symmetric).  Transposed so that the accumulator lanes
// are radial points: D[n][m] = sum_k (K - I)[n][k] s_m[k], A = K - I (resident
// in shared memory, four planes), B = 64 state rows per tile (four planes,
// double buffered), D double-buffered in tensor memory: one tile is staged
// while the previous tile's products run, and written out while the next
// tile's run.  K - I being circulant, its K-slice j (columns 16 j..16 j + 15)
// is slice 0 with the rows shifted by 16 j; A is therefore stored once as
// one 16-column strip of 128 + N_r - 16 rows, and slice j is the window
// starting 16 j rows higher.
// ----------------------------------------------------------------------------
__host__ __device__ inline int tc_kmaj_off(int r, int k, int K) {
  // K-major, no swizzle: 8-row x 16-byte core matrices, 128 B each, row groups outer
  return ((r >> 3) * (K >> 3) + (k >> 3)) * 128 + (r & 7) * 16 + (k & 7) * 2;
}
int mixed_plane_offset(int row, int k, int nr) { return tc_kmaj_off(row, k, 16); }
int mixed_strip_rows(int nr) { return 128 + nr - 16; }
bool mol_mixed_supported(int nr) { return nr == 64 || nr == 128; }

// shared-memory matrix descriptor: start, leading (K-direction) and stride
// (8-row group) byte offsets, no swizzle
__device__ __forceinline__ unsigned long long tc_desc(unsigned addr, unsigned lbo, unsigned sbo) {
  return (unsigned long long)((addr >> 4) & 0x3FFF) | ((unsigned long long)((lbo >> 4) & 0x3FFF) << 16) |
         ((unsigned long long)((sbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}
__device__ __forceinline__ void tc_mma(unsigned d, unsigned long long a, unsigned long long b, unsigned idesc,
                                       int accumulate) {
  asm volatile(
      "{ .reg .pred p; setp.ne.b32 p, %4, 0; tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p; }" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}
__device__ __forceinline__ void tc_ld32(unsigned taddr, unsigned (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
        "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
        "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
}

template <int NR>
struct TcShape {
  static constexpr int MR = 128;                 // accumulator lanes: radial points (>= NR discarded)
  static constexpr int TR = 64;                  // state rows per tile (the MMA's N)
  static constexpr int KS = NR / 16;             // K slices of 16
  static constexpr int SR = MR + NR - 16;        // rows of the circulant strip
  static constexpr int APL = SR * 16 * 2;        // bytes of one strip plane
  static constexpr int BPL = TR * NR * 2;        // bytes of one B plane
  static constexpr int LOADS = TR * NR / (256 * 2);  // 16-byte loads per thread per tile
  static constexpr int SMEM = 4 * APL + 2 * 4 * BPL; // strip + two tile buffers
};

template <int NR>
__global__ void __launch_bounds__(256, 1) mol_kinetic_tc_kernel(SpeciesDev sp, long long rows, int* err) {
  if (idle_launch(sp)) return;
  using S = TcShape<NR>;
  constexpr int TR = S::TR, KS = S::KS, APL = S::APL, BPL = S::BPL, LOADS = S::LOADS;
  constexpr unsigned SBO_A = 2 * 128, SBO_B = (NR / 8) * 128;
  constexpr unsigned kCols = 4 * TR;  // tensor memory: 2 buffers x (Re, Im) x TR rows
  extern __shared__ __align__(1024) uint8_t smem_tc[];
  uint8_t* A = smem_tc;             // (K - I) strip: Re hi, Re lo, Im hi, Im lo
  uint8_t* Bt = smem_tc + 4 * APL;  // two tile buffers, each Re hi, Re lo, Im hi, Im lo
  __shared__ __align__(8) unsigned long long bar[2];  // [0] A staged, [1] products done
  __shared__ unsigned tmem_base;
  __shared__ float s_wmax[8][TR];                       // per warp: row maxima of the tile being staged
  __shared__ int s_rexp[2][TR];                         // per tile buffer: row scale exponents
  const int t = threadIdx.x, w = t >> 5, lane = t & 31;
  const float2* X = sp.psi;
  float2* Y = sp.d2;

  if (t == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect_tx(&bar[0], 4u * APL);
    bulk_g2s(A, sp.kpl, 4u * APL, &bar[0]);
  }
  if (w == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(kCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem = tmem_base;
  auto release = [&]() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (w == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols));
  };
  // a wait on bar[id] phase ph by every thread, uniform outcome; on a timeout
  // the products in flight get a second bounded wait before tensor memory is freed
  auto wait_all = [&](int id, unsigned ph) -> bool {
    const bool ok = mbar_wait_sleep(&bar[id], ph);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (__syncthreads_and(ok)) return true;
    if (t == 0) atomicOr(err, kErrTimeout);
    if (!ok) mbar_wait_sleep(&bar[id], ph);
    release();
    return false;
  };
  if (!wait_all(0, 0)) return;

  // load slot u of a tile: rows 8 q + (lane & 7), points 8 kc + 2 (lane >> 3) (+1)
  auto slot_row = [&](int u) { return 8 * ((w + 8 * u) / (NR / 8)) + (lane & 7); };
  auto slot_k = [&](int u) { return 8 * ((w + 8 * u) % (NR / 8)) + 2 * (lane >> 3); };
  float4 pre[LOADS];
  auto fetch = [&](long long tile) {
#pragma unroll
    for (int u = 0; u < LOADS; ++u) {
      const long long gr = tile * TR + slot_row(u);
      long long xr = gr;  // stored row of processed row gr (fewer than 2^31 rows fit the memory)
      if (sp.rows != sp.mrows) {
        const unsigned m = (unsigned)gr / (unsigned)sp.rows;
        xr = (long long)m * sp.mrows + ((unsigned)gr - m * (unsigned)sp.rows);
      }
      pre[u] = gr < rows ? __ldcs(reinterpret_cast<const float4*>(X + xr * NR + slot_k(u)))
                         : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  // The fetched tile -> four FP16 planes of buffer buf.  Each state row is
  // scaled by 2^e so that its largest |Re|, |Im| lies in [2^14, 2^15) (an
  // exact power-of-two scale, undone on write-out): hi = fp16(x), lo =
  // fp16(x - hi) then carry 22 bits of every element of the row's scale.
  // Row maxima: slot u of every thread lies in row group u / UPQ (rows 8 q +
  // (lane & 7)) whatever the warp, so each thread folds its slots per group,
  // the four lanes sharing a row fold by shuffles, and each warp leaves one
  // value per row; 64 threads then fold the 8 warps' values.
  auto stage = [&](int buf) {
    constexpr int UPQ = LOADS / 8;
    static_assert(LOADS % 8 == 0 && TR == 64, "eight row groups of eight rows per tile");
    uint8_t* B0 = Bt + buf * 4 * BPL;
    float rm[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) rm[q] = 0.f;
#pragma unroll
    for (int u = 0; u < LOADS; ++u)
      rm[u / UPQ] = fmaxf(rm[u / UPQ], fmaxf(fmaxf(fabsf(pre[u].x), fabsf(pre[u].y)),
                                             fmaxf(fabsf(pre[u].z), fabsf(pre[u].w))));
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      rm[q] = fmaxf(rm[q], __shfl_xor_sync(0xffffffffu, rm[q], 8));
      rm[q] = fmaxf(rm[q], __shfl_xor_sync(0xffffffffu, rm[q], 16));
    }
    if (lane < 8) {
#pragma unroll
      for (int q = 0; q < 8; ++q) s_wmax[w][8 * q + lane] = rm[q];
    }
    __syncthreads();
    if (t < TR) {
      float m = 0.f;
#pragma unroll
      for (int ww = 0; ww < 8; ++ww) m = fmaxf(m, s_wmax[ww][t]);
      int ex = 0;
      if (m > 0.f) frexpf(m, &ex);
      s_rexp[buf][t] = m > 0.f ? min(15 - ex, 100) : 0;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < LOADS; ++u) {
      const float sc = __int_as_float((127 + s_rexp[buf][slot_row(u)]) << 23);  // 2^e
      const float re[2] = {pre[u].x * sc, pre[u].z * sc}, im[2] = {pre[u].y * sc, pre[u].w * sc};
      __half rh[2], rl[2], ih[2], il[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        rh[e] = __float2half_rn(re[e]);
        rl[e] = __float2half_rn(re[e] - __half2float(rh[e]));
        ih[e] = __float2half_rn(im[e]);
        il[e] = __float2half_rn(im[e] - __half2float(ih[e]));
      }
      const int off = tc_kmaj_off(slot_row(u), slot_k(u), NR);
      *reinterpret_cast<__half2*>(B0 + 0 * BPL + off) = __halves2half2(rh[0], rh[1]);
      *reinterpret_cast<__half2*>(B0 + 1 * BPL + off) = __halves2half2(rl[0], rl[1]);
      *reinterpret_cast<__half2*>(B0 + 2 * BPL + off) = __halves2half2(ih[0], ih[1]);
      *reinterpret_cast<__half2*>(B0 + 3 * BPL + off) = __halves2half2(il[0], il[1]);
    }
  };
  auto issue = [&](int buf) {  // 2 outputs x 6 split products x KS slices, one thread
    // FP32 accumulator (bit 4), A and B FP16 (format fields at bits 7 and 10 zero), N, M
    constexpr unsigned idp = (1u << 4) | ((unsigned)(TR >> 3) << 17) | ((unsigned)(128 >> 4) << 24);
    constexpr unsigned idn = idp | (1u << 14);  // B negated
    // {A plane, B plane, negate}: Re = Kr Xr - Ki Xi, Im = Kr Xi + Ki Xr, each as hh + hl + lh
    constexpr int blk[2][6][3] = {{{0, 0, 0}, {0, 1, 0}, {1, 0, 0}, {2, 2, 1}, {2, 3, 1}, {3, 2, 1}},
                                  {{0, 2, 0}, {0, 3, 0}, {1, 2, 0}, {2, 0, 0}, {2, 1, 0}, {3, 0, 0}}};
    // slice j: A window starts (NR - 16 - 16 j) rows into the strip, B at column 16 j
    unsigned long long da[4], db[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      da[p] = tc_desc(smem_u32(A + p * APL) + ((NR - 16) / 8) * SBO_A, 128, SBO_A);
      db[p] = tc_desc(smem_u32(Bt + (buf * 4 + p) * BPL), 128, SBO_B);
    }
#pragma unroll
    for (int o = 0; o < 2; ++o) {
      const unsigned d = tmem + (unsigned)(buf * 2 * TR + o * TR);
#pragma unroll
      for (int b = 0; b < 6; ++b)
#pragma unroll
        for (int j = 0; j < KS; ++j)
          tc_mma(d, da[blk[o][b][0]] - (unsigned long long)(j * 2 * SBO_A / 16),
                 db[blk[o][b][1]] + (unsigned long long)(j * 256 / 16), blk[o][b][2] ? idn : idp,
                 (b | j) != 0);
    }
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(&bar[1]))
                 : "memory");
  };
  auto drain = [&](int buf, long long tile) {  // tensor memory -> d2 rows of the tile
    constexpr int H = TR / 2;                       // rows per warp half
    const int n = 32 * (w & 3) + lane, rh = w >> 2;  // radial point, row half
    static_assert(H == 32, "the write-out loads 32 accumulator columns per warp half");
    unsigned re[H], im[H];
    const unsigned ta = tmem + ((unsigned)(32 * (w & 3)) << 16) + (unsigned)(buf * 2 * TR + H * rh);
    tc_ld32(ta, re);
    tc_ld32(ta + TR, im);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    if (n < NR) {
#pragma unroll
      for (int r = 0; r < H; ++r) {
        const long long gr = tile * TR + H * rh + r;
        // undo the row's and the matrix's power-of-two scales
        const float us = __int_as_float((127 - s_rexp[buf][H * rh + r] - sp.kpl_exp) << 23);
        if (gr < rows)
          __stcs(Y + gr * NR + n, make_float2(__uint_as_float(re[r]) * us, __uint_as_float(im[r]) * us));
      }
    }
  };
  auto sync_async = [&]() {  // the staged planes are visible to the tensor cores
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  };

  // tile i: staged into buffer i & 1 while the products of tile i - 1 run
  // (its loads were issued one iteration earlier), issued once those are
  // done; then tile i - 1 is written out while tile i's products run
  const long long ntiles = (rows + TR - 1) / TR;
  long long tile = blockIdx.x;
  if (tile >= ntiles) {
    release();
    return;
  }
  fetch(tile);
  stage(0);
  sync_async();
  if (t == 0) issue(0);
  long long prev = tile;
  tile += gridDim.x;
  if (tile < ntiles) fetch(tile);
  int i = 1;
  for (; tile < ntiles; tile += gridDim.x, ++i) {
    stage(i & 1);  // buffer i & 1 was read by the products of tile i - 2, complete
    if (tile + gridDim.x < ntiles) fetch(tile + gridDim.x);  // in flight until the next stage
    sync_async();
    if (!wait_all(1, (unsigned)((i - 1) & 1))) return;  // products of tile i - 1
    if (t == 0) issue(i & 1);
    drain((i - 1) & 1, prev);  // overlaps the products of tile i
    prev = tile;
  }
  if (!wait_all(1, (unsigned)((i - 1) & 1))) return;
  drain((i - 1) & 1, prev);
  release();
}

// Stage 1 of a species' step: in the streaming form the per-molecule field
// records (point-resident R-space kernel only) and the kinetic pass d2 = (T - 1) s.
// Stage 2: the R-space pass (streaming form) or the whole fused step.
// Each returns the number of kernels it launched.
template <int NR>
static int launch_stage1_t(const SpeciesDev& sp, const MolDev& md, const Grid& g, int prescribed, int* err,
                           cudaStream_t s) {
  if (sp.path == MS_MOL_FUSED) {
    if (!use_point(sp)) return 0;
    mol_field_kernel<<<(sp.nmol + 127) / 128, 128, 0, s>>>(sp, md, g, prescribed, err);
    return 1;
  }
  // the per-molecule frame-field records those kernels read
  const bool records = use_point(sp) || use_col(sp) || use_tile(sp) || use_pair(sp);
  int n = 0;
  if (records && sp.mixed) {
    mol_field_kernel<<<(sp.nmol + 127) / 128, 128, 0, s>>>(sp, md, g, prescribed, err);
    ++n;
  }
  const long long rows_total = (long long)sp.nmol * sp.rows;
  if (sp.mixed) {  // split-FP16 tensor-core GEMM
    if constexpr (NR == 64 || NR == 128) {
      using T = TcShape<NR>;
      int dev = 0, nsm = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
      const long long ntiles = (rows_total + T::TR - 1) / T::TR;
      const int grid = (int)std::min<long long>(ntiles, (long long)(nsm > 0 ? nsm : 1));
      cudaFuncSetAttribute(mol_kinetic_tc_kernel<NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, T::SMEM);
      mol_kinetic_tc_kernel<NR><<<grid, 256, T::SMEM, s>>>(sp, rows_total, err);
    }
    return n + 1;
  }
  const int RB = kinetic_rows(NR);
  const size_t ksmem = 2 * (size_t)NR * sizeof(float2) + (size_t)RB * NR * sizeof(float2);
  cudaFuncSetAttribute(mol_kinetic_kernel<NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ksmem);
  constexpr int NT = FFTShape<NR>::THREADS;
  const int nfld = records ? (sp.nmol + NT - 1) / NT : 0;
  mol_kinetic_kernel<NR><<<(unsigned)(nfld + (rows_total + RB - 1) / RB), NT, ksmem, s>>>(
      sp, md, g, prescribed, nfld, rows_total, RB, err);
  return n + 1;
}

template <int NR>
static int launch_stage2_t(const SpeciesDev& sp, const MolDev& md, const Grid& g, int prescribed, int* err,
                           cudaStream_t s) {
  const bool fused = sp.path == MS_MOL_FUSED;
  const StepShape sh = sp.kern == MS_KERN_CHUNK && sp.ch > 0 ? step_shape_ch(NR, sp.nrot, fused, sp.ch)
                                                             : step_shape(NR, sp.nrot, fused);
  if (fused) {
    if constexpr (NR == 128) {
      if (use_point(sp)) {
        launch_rpoint_n<NR, true>(sp, md, err, s);
        if (sp.dipw) launch_dipole_r<NR>(sp, md, err, s);
        return sp.dipw ? 2 : 1;
      }
    }
    launch_step_tt<NR, true, 12>(sp, md, g, prescribed, err, sh, s);
    return 1;
  }
  if (use_point(sp)) {  // point-resident R-space pass
    launch_rpoint_n<NR>(sp, md, err, s);
    if constexpr (NR <= 128) {
      if (sp.dipw) {
        launch_dipole_r<NR>(sp, md, err, s);
        return 2;
      }
    }
    return 1;
  }
  if (use_col(sp)) {
    launch_rspace_col(sp, md, err, s);
    return 1;
  }
  RspaceMaps maps;
  if (use_pair(sp)) {
    if (rspace_maps(sp, pair_tile(sp), true, &maps)) {
      launch_rspace_pair(sp, md, err, maps, pair_tile(sp), s);
      return 1;
    }
    if (sp.par) {  // no other kernel takes the reachable rows beyond J = 8: report it
      flag_error_kernel<<<1, 1, 0, s>>>(err, kErrLaunch);
      return 1;
    }
  }
  if (use_tile(sp) && rspace_maps(sp, rspace_tile(sp), false, &maps)) {
    launch_rspace(sp, md, err, maps, rspace_tile(sp), s);
    return 1;
  }
  if (sh.maxr == 4) launch_step_tt<NR, false, 4>(sp, md, g, prescribed, err, sh, s);
  else if (sh.maxr == 12) launch_step_tt<NR, false, 12>(sp, md, g, prescribed, err, sh, s);
  else launch_step_tt<NR, false, 24>(sp, md, g, prescribed, err, sh, s);
  return 1;
}

int launch_mol_stage1(const SpeciesDev& sp, const MolDev& md, const Grid& g, int prescribed, int* err,
                      cudaStream_t s) {
  if (sp.nmol == 0 || sp.bloch) return 0;
  switch (sp.nr) {
    case 64: return launch_stage1_t<64>(sp, md, g, prescribed, err, s);
    case 128: return launch_stage1_t<128>(sp, md, g, prescribed, err, s);
    case 256: return launch_stage1_t<256>(sp, md, g, prescribed, err, s);
  }
  return 0;
}

int launch_mol_stage2(const SpeciesDev& sp, const MolDev& md, const Grid& g, int prescribed, int* err,
                      cudaStream_t s) {
  if (sp.nmol == 0) return 0;
  if (sp.bloch) return launch_bloch_step(sp, md, g, prescribed, err, s);
  switch (sp.nr) {
    case 64: return launch_stage2_t<64>(sp, md, g, prescribed, err, s);
    case 128: return launch_stage2_t<128>(sp, md, g, prescribed, err, s);
    case 256: return launch_stage2_t<256>(sp, md, g, prescribed, err, s);
  }
  return 0;
}

template <int NR>
static void launch_observe_t(const SpeciesDev& sp, const MolDev& md, int* err, cudaStream_t s) {
  // as many molecules as fill half a block, or one whose rows go in even blocks
  const int ne = std::max(1, sp.rows - sp.rows_g), most = kObserveRows<NR>;
  const int mpb = std::max(1, most / 2 / ne);
  const int passes = (ne + most - 1) / most, RB = mpb > 1 ? mpb * ne : (ne + passes - 1) / passes;
  const size_t smem = 2 * (size_t)NR * sizeof(float2) + mol_state_smem(NR, RB);
  cudaFuncSetAttribute(mol_observe_kernel<NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  mol_observe_kernel<NR><<<(sp.nmol + mpb - 1) / mpb, FFTShape<NR>::THREADS, smem, s>>>(sp, md, RB, mpb, err);
}

void launch_mol_observe(const SpeciesDev& sp, const MolDev& md, int* err, cudaStream_t s) {
  if (sp.nmol == 0) return;
  if (sp.bloch) {
    launch_bloch_observe(sp, md, s);
    return;
  }
  switch (sp.nr) {
    case 64: launch_observe_t<64>(sp, md, err, s); break;
    case 128: launch_observe_t<128>(sp, md, err, s); break;
    case 256: launch_observe_t<256>(sp, md, err, s); break;
  }
}

}  // namespace ms
