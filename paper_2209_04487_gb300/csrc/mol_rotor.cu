// Molecular step on whole rotors (J <= 4, reachable rows): the kernel and its
// launch.
//
// The reachable rows of a molecule are one vector psi_{j m} over all channels
// (the surface is the parity of j), (J + 1)^2 values at a radial point.  A
// thread holds all of them at one point in registers, so the coupling
// E'.R^ = E'_z Z + S+- parts, which joins (j, m) with (j +- 1, m) and (j +- 1,
// m +- 1), is register arithmetic with compile-time coefficients: no exchange
// through shared memory and no barrier between the terms of the series.  With
// a thread per surface and point instead (the kernel that runs states with
// every row populated), the other surface's rows pass through shared memory
// for every term and its barriers and the idle half of the larger surface's
// threads cost a third of the time.
//
// The coupling's exponential series S = sum_{n=1..N} T_n, T_1 = i theta M eta,
// T_n = (i theta / n) M T_{n-1}, is summed by Horner's rule on T_1: S = P_1, P_n
// = T_1 + (i theta / (n + 1)) M P_{n+1}, P_N = T_1 (on eta itself every step would
// round at eta's size, not at T_1's).  Values are kept as (Re, Im) pairs and
// multiplied by real coefficients as packed FP32x2 products, whose equal
// constants are immediates.
//
// What bounds it: latency.  By registers an SM holds twelve warps.  In the fused
// step at J = 4 an issued instruction costs 5.4 warp cycles: 1 its issue, 0.9
// fixed latency, 1.2 memory (shared and global), 0.6 barriers, 0.5 the FP32 pipe,
// 0.5 another warp's turn, 0.4 instruction fetch; issue slots are 50% and the
// shared-memory pipe 46% busy (142 warp instructions a row and 32 points, the FFT
// included).  Per row and point of the reachable rows: the R-space
// pass at J = 4, N_r = 64 takes 4.36 ps, 5.5 TB/s, against 7.13 for a thread per
// surface; the fused step at J = 4, N_r = 128 6.79 against 12.14 ps.
//
// FUSED (N_r = 128): the kinetic pass runs in the same kernel.  The state
// arrives by one bulk copy and stays in shared memory; the FFT turns it into
// d2 = (T - 1) s beside it.
#include "mol_fft.cuh"

namespace ms {
namespace {

template <int J>
struct RotorDims {
  static constexpr int NROT = (J + 1) * (J + 1);
  // first row of shell j among the reachable rows: ground even shells, then excited odd shells
  static constexpr int shell(int j) {
    int n = 0;
    for (int q = 0; q <= J; ++q)
      if ((q & 1) < (j & 1) || ((q & 1) == (j & 1) && q < j)) n += 2 * q + 1;
    return n;
  }
  static constexpr int row(int j, int m) { return shell(j) + j + m; }
  // register of (j, m): columns m = -J .. J, each by j
  static constexpr int at(int j, int m) {
    int n = 0;
    for (int q = -J; q < m; ++q) n += J + 1 - (q < 0 ? -q : q);
    return n + j - (m < 0 ? -m : m);
  }
};

// calls fn(j, m) for every channel, columns in order
template <int J, class F>
__device__ __forceinline__ void for_channels(F&& fn) {
  static_for<-J, J + 1>([&](auto mc) {
    constexpr int m = decltype(mc)::value;
    static_for<(m < 0 ? -m : m), J + 1>([&](auto jc) { fn(jc, mc); });
  });
}

struct RotorSums {
  float2 hi, lo;  // populations (ground, excited), compensated
  float ab[2];    // absorbed norm
  float2 x, z;    // dipole sums by parts
  float y;
  float2 rnd;     // rounding residual products
};

// The R-space pass at one radial point p of a molecule: gs its state (global,
// at p), ss and ds where s and d2 are read (at p; FUSED: shared memory).
template <int J, int NR, bool FUSED, bool DIPR>
__device__ __forceinline__ void rotor_point(const SpeciesDev& sp, int p, float2* gs, const float2* ss, const float2* ds,
                                            float4 f, float cfix, RotorSums& a) {
  using D = RotorDims<J>;
  constexpr int NROT = D::NROT;
  if constexpr (DIPR) {  // times d(R) / max|d| at this point
    const float dw = __ldg(&sp.dipw[p]);
    f.x *= dw;
    f.y *= dw;
    f.z *= dw;
  }
  const int nterms = max(__float_as_int(f.w), 1);  // no field: one term of zeros
  const float mk = __ldg(&sp.maskw[p]).x;
  auto s_at = [&](int row) { return ss[row * NR]; };
  auto d_at = [&](int row) { return FUSED ? ds[row * NR] : __ldg(ds + row * NR); };
  // potential phases of shell j on the surface of its parity
  auto vh_at = [&](auto jc) {
    constexpr int j = decltype(jc)::value;
    return __ldg(sp.vhalf + ((j & 1) * (J + 1) + j) * NR + p);
  };
  auto vd_at = [&](auto jc) {
    constexpr int j = decltype(jc)::value;
    return __ldg(sp.vdelta + ((j & 1) * (J + 1) + j) * NR + p);
  };

  float2 v[NROT], q[NROT];
  // i (M v) at (j, m); z2, x2 and y the field's factors
  auto coupled = [&](auto jc, auto mc, float2 z2, float2 x2, float y) -> float2 {
    constexpr int j = decltype(jc)::value, m = decltype(mc)::value;
    auto sum2 = [&](auto cf0, auto cf1, auto c2) {  // cf0 (j - 1, c2) + cf1 (j + 1, c2)
      constexpr int cq = decltype(c2)::value, mq = cq < 0 ? -cq : cq;
      constexpr bool lo = j - 1 >= mq, hi = j + 1 <= J && j + 1 >= mq;
      if constexpr (lo && hi)
        return fma2(dup2(cf0()), v[D::at(lo ? j - 1 : j, lo ? cq : m)], mul2(dup2(cf1()), v[D::at(hi ? j + 1 : j, hi ? cq : m)]));
      else if constexpr (lo) return mul2(dup2(cf0()), v[D::at(j - 1, cq)]);
      else if constexpr (hi) return mul2(dup2(cf1()), v[D::at(j + 1, cq)]);
      else return make_float2(0.f, 0.f);
    };
    const float2 az = sum2([] { return c_zd(j, m); }, [] { return c_zu(j, m); }, std::integral_constant<int, m>());
    const float2 ap = sum2([] { return c_pd(j, m); }, [] { return c_pu(j, m); }, std::integral_constant<int, m - 1>());
    const float2 am = sum2([] { return c_md(j, m); }, [] { return c_mu(j, m); }, std::integral_constant<int, m + 1>());
    const float2 r = fma2(z2, az, mul2(x2, add2(ap, am)));
    const float2 d = sub2(ap, am);
    return make_float2(fmaf(y, d.x, -r.y), fmaf(y, d.y, r.x));
  };
  auto eta = [&](auto jc, auto mc) -> float2 {  // V^{1/2} (s + d2)
    constexpr int row = D::row(decltype(jc)::value, decltype(mc)::value);
    return cmul(vh_at(jc), add2(s_at(row), d_at(row)));
  };
  for_channels<J>([&](auto jc, auto mc) { v[D::at(decltype(jc)::value, decltype(mc)::value)] = eta(jc, mc); });
  // ---- S into q
  {
    const float2 z2 = dup2(f.x), x2 = dup2(f.y);
    for_channels<J>([&](auto jc, auto mc) {  // T_1
      q[D::at(decltype(jc)::value, decltype(mc)::value)] = coupled(jc, mc, z2, x2, f.z);
    });
  }
  if (nterms == 2) {
#pragma unroll
    for (int k = 0; k < NROT; ++k) v[k] = q[k];
    const float2 z2 = dup2(0.5f * f.x), x2 = dup2(0.5f * f.y);
    for_channels<J>([&](auto jc, auto mc) {
      constexpr int k = D::at(decltype(jc)::value, decltype(mc)::value);
      q[k] = add2(v[k], coupled(jc, mc, z2, x2, 0.5f * f.z));
    });
  } else if (nterms > 2) {
    float2 t1[NROT];
#pragma unroll
    for (int k = 0; k < NROT; ++k) t1[k] = q[k];
#pragma unroll 1
    for (int n = nterms; n >= 2; --n) {
#pragma unroll
      for (int k = 0; k < NROT; ++k) v[k] = q[k];
      const float cn = 1.f / (float)n;
      const float2 z2 = dup2(f.x * cn), x2 = dup2(f.y * cn);
      for_channels<J>([&](auto jc, auto mc) {
        constexpr int k = D::at(decltype(jc)::value, decltype(mc)::value);
        q[k] = add2(t1[k], coupled(jc, mc, z2, x2, f.z * cn));
      });
    }
  }
  // ---- d1 = (V - 1) u + V^{1/2} S, mask, s' = s + (d2 + d1) + cfix s
  {
    const float2 cf = dup2(cfix);
    const bool masked = mk < 1.f;
    float b2 = 0.f;
    for_channels<J>([&](auto jc, auto mc) {
      constexpr int j = decltype(jc)::value, m = decltype(mc)::value, k = D::at(j, m), row = D::row(j, m), sf = j & 1;
      const float2 S = q[k];
      const float2 s0 = s_at(row), d0 = d_at(row), u = add2(s0, d0), vh = vh_at(jc), vd = vd_at(jc);
      float2 d1 = make_float2(fmaf(vd.x, u.x, fmaf(-vd.y, u.y, fmaf(vh.x, S.x, -vh.y * S.y))),
                              fmaf(vd.x, u.y, fmaf(vd.y, u.x, fmaf(vh.x, S.y, vh.y * S.x))));
      if (masked) {
        const float2 p = add2(u, d1);
        d1 = fma2(dup2(mk - 1.f), u, mul2(dup2(mk), d1));
        a.ab[sf] += (1.f - mk * mk) * fmaf(p.x, p.x, p.y * p.y);
      }
      const float2 sn = round_update2(s0, add2(d0, d1), cf, a.rnd);
      __stcs(gs + row * NR, sn);
      q[k] = sn;
      const float b = fmaf(sn.x, sn.x, sn.y * sn.y);
      if constexpr (sf == 1) acc2p(a.hi, a.lo, make_float2(j > (m < 0 ? -m : m) ? b2 : 0.f, b));  // compensated from the first term on
      else if constexpr (j == J) acc2p(a.hi, a.lo, make_float2(b, 0.f));
      else b2 = b;
    });
  }
  // ---- dipole: over pairs of rows of one column (Z) and of columns m, m + 1 (S+, S-); each pair joins a
  // ground and an excited row, and conj(g) e and conj(e) g give the same Re (P + M), Im (P - M)
  if constexpr (!DIPR) {  // with d(R) the dipole is read from T^{1/2} s' by mol_dipole_r_kernel
    for_channels<J>([&](auto jc, auto mc) {
      constexpr int j = decltype(jc)::value, m = decltype(mc)::value, m1 = m + 1 < 0 ? -m - 1 : m + 1;
      const float2 b = q[D::at(j, m)];
      if constexpr (j < J) a.z = fma2(dup2(c_zu(j, m)), mul2(b, q[D::at(j + 1, m)]), a.z);
      constexpr bool up = j + 1 <= J && j + 1 >= m1, dn = j - 1 >= m1;
      if constexpr (up || dn) {
        float2 r = make_float2(0.f, 0.f);
        if constexpr (up) r = mul2(dup2(c_mu(j, m)), q[D::at(up ? j + 1 : j, up ? m + 1 : m)]);
        if constexpr (up && dn) r = fma2(dup2(c_md(j, m)), q[D::at(dn ? j - 1 : j, dn ? m + 1 : m)], r);
        else if constexpr (dn) r = mul2(dup2(c_md(j, m)), q[D::at(dn ? j - 1 : j, dn ? m + 1 : m)]);
        a.x = fma2(b, r, a.x);
        a.y = fmaf(b.y, r.x, fmaf(-b.x, r.y, a.y));
      }
    });
  }
}

// A molecule's sums over its lanes, populations compensated, the rest plain
// FP32: r[0..7] = P_g, P_e, absorbed, Re(S+ + S-), Im(S+ - S-), 2 Re Z, the
// rounding residuals; l the low parts of the populations.
__device__ __forceinline__ void rotor_warp_sum(const RotorSums& a, float (&r)[8], float (&l)[2]) {
  const float v[8] = {a.hi.x, a.hi.y, a.ab[0], a.ab[1], a.x.x + a.x.y, a.y, 2.f * (a.z.x + a.z.y), a.rnd.x + a.rnd.y};
  l[0] = a.lo.x;
  l[1] = a.lo.y;
#pragma unroll
  for (int k = 0; k < 8; ++k) r[k] = v[k];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float h2 = __shfl_xor_sync(0xffffffffu, r[k], o);
      const float g2 = __shfl_xor_sync(0xffffffffu, l[k], o);
      acc2(r[k], l[k], h2);
      l[k] += g2;
    }
#pragma unroll
    for (int k = 2; k < 8; ++k) r[k] += __shfl_xor_sync(0xffffffffu, r[k], o);
  }
}

// What the closing threads t < 8 of a molecule hold from before its step.
__device__ __forceinline__ double rotor_old(const MolDev& md, int m, int t) {
  return t < 3 ? md.mu[3 * (long long)m + t]
               : (t == 5 || t == 6 ? md.absorbed[2 * (long long)m + (t - 5)] : 0.0);
}

// The molecule's outputs from its sums, by threads t < 8.
template <bool DIPR>
__device__ __forceinline__ void rotor_close(const SpeciesDev& sp, const MolDev& md, int m, int t, double old,
                                            const float* fin, const float* fin_lo, int* err) {
  if (t < 3) {  // lab dipole: mu = O mu', mu' = d dR (Re(S+ + S-), Im(S+ - S-), 2 Re Z)
    if constexpr (!DIPR) {  // with d(R) the dipole is read from T^{1/2} s' by mol_dipole_r_kernel
      const float* O = md.rot + 9 * (long long)m + 3 * t;
      const float lab = (float)sp.dipole * sp.dR * (O[0] * fin[4] + O[1] * fin[5] + O[2] * fin[6]);
      const double nl = (double)lab;
      md.dmu[3 * (long long)m + t] = nl - old;
      md.mu[3 * (long long)m + t] = nl;
    }
  } else if (t < 5) {
    const double P = ((double)fin[t - 3] + (double)fin_lo[t - 3]) * (double)sp.dR;
    md.pop[2 * (long long)m + (t - 3)] = P;
    if (!isfinite(P)) atomicOr(err, kErrNonFinite);
  } else if (t < 7) {
    md.absorbed[2 * (long long)m + (t - 5)] = old + (double)fin[t - 3] * (double)sp.dR;
  } else if (t == 7) {
    md.ncorr[m] = rounding_feedback(fin[7], fin[0] + fin[1]);
  }
}

// The fused step: one CTA of N_r threads a molecule (at J = 3 a fourth CTA an SM is worth 4%).
template <int J, int NR, bool DIPR>
__global__ void __launch_bounds__(NR, J <= 3 ? 4 : 3) mol_rotor_fused_kernel(SpeciesDev sp, MolDev md, int* err) {
  constexpr int NROT = RotorDims<J>::NROT, NW = NR / 32;
  constexpr unsigned kStateBytes = (unsigned)NROT * NR * sizeof(float2);
  if (idle_launch(sp)) return;
  extern __shared__ __align__(16) float4 smem4[];
  float2* Sb = reinterpret_cast<float2*>(smem4);  // [NROT][NR] s
  float2* Db = Sb + NROT * NR;                    // [NROT][NR] d2
  float2* s_tw = Db + NROT * NR;                  // [N2][N1] FFT twiddles
  float2* s_kd = s_tw + NR;                       // [NR] kinetic phase deltas
  __shared__ __align__(8) unsigned long long s_bar[1];
  __shared__ float s_red[NW][10];
  __shared__ float s_fin[8], s_fin_lo[2];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int lm = blockIdx.x, m = sp.mol[lm];
  float2* const gs = sp.psi + (long long)lm * sp.mrows * NR;  // this molecule's state
  if (t == 0) {
    mbar_init(&s_bar[0], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect_tx(&s_bar[0], kStateBytes);
    bulk_g2s(Sb, gs, kStateBytes, &s_bar[0]);
  }
  s_tw[t] = __ldg(&sp.twiddle[t]);
  s_kd[t] = __ldg(&sp.kdelta[t]);
  const float4 f = __ldg(&sp.fld[lm]);  // (theta E'_z, theta E'_x/2, theta E'_y/2, terms)
  const float cfix = md.ncorr[m];       // rounding feedback of the previous step
  const double old = rotor_old(md, m, t);
  __syncthreads();  // the barrier is initialised
  const bool ok = mbar_wait_sleep(&s_bar[0], 0);
  if (!__syncthreads_and(ok)) {
    if (t == 0) atomicOr(err, kErrTimeout);
    if (!ok) mbar_wait_sleep(&s_bar[0], 0);
    return;
  }
  kinetic_pass<NR, NR, true>(Db, Sb, NROT, s_kd, s_tw);  // d2 = (T - 1) s
  RotorSums a = {};
  rotor_point<J, NR, true, DIPR>(sp, t, gs + t, Sb + t, Db + t, f, cfix, a);
  float r[8], l[2];
  rotor_warp_sum(a, r, l);
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < 8; ++k) s_red[w][k] = r[k];
    s_red[w][8] = l[0];
    s_red[w][9] = l[1];
  }
  __syncthreads();
  if (t < 8) {
    float h = 0.f, lo = 0.f;
    for (int ww = 0; ww < NW; ++ww) {
      acc2(h, lo, s_red[ww][t]);
      if (t < 2) lo += s_red[ww][8 + t];
    }
    s_fin[t] = h + lo;
    if (t < 2) s_fin_lo[t] = lo - (s_fin[t] - h);
  }
  __syncthreads();
  rotor_close<DIPR>(sp, md, m, t, old, s_fin, s_fin_lo, err);
}

// The streaming R-space pass: two warps a molecule, each 32 points at a time, so
// that the closing sums (a third of the instructions at J = 1) are paid twice a
// molecule and not once for every 32 points.  Per row and point, against a warp
// for every 32 points: J = 4, N_r = 256 6.56 -> 4.68 ps, J = 1, N_r = 64 7.91 ->
// 6.76 ps; one warp a molecule: 5.13 against 4.42 ps at J = 4, N_r = 64.  The
// blocks asked for an SM set the registers a thread may take, and the order of
// loads that follows from that: at J = 4 five (of which six fit) 4.36, 4.37 and
// 4.15 ps at N_r = 64, 128 and 256, asking for six 4.43, 5.44 and 5.18; at J = 3
// seven 4.45, 4.73 and 4.38 ps, six 4.89, 5.32 and 4.88.
template <int J, int NR, bool DIPR>
__global__ void __launch_bounds__(64, J == 4 ? 5 : (J == 3 ? 7 : 6)) mol_rotor_kernel(SpeciesDev sp, MolDev md, int* err) {
  constexpr int NROT = RotorDims<J>::NROT;
  if (idle_launch(sp)) return;
  __shared__ float s_red[2][10], s_fin[10];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int lm = blockIdx.x, m = sp.mol[lm];
  float2* const gs = sp.psi + (long long)lm * sp.mrows * NR + lane;
  const float2* const ds = sp.d2 + (long long)lm * NROT * NR + lane;
  const float4 f = __ldg(&sp.fld[lm]);  // (theta E'_z, theta E'_x/2, theta E'_y/2, terms)
  const float cfix = md.ncorr[m];       // rounding feedback of the previous step
  const double old = rotor_old(md, m, t);
  RotorSums a = {};
#pragma unroll 1
  for (int p = 32 * w; p < NR; p += 64) rotor_point<J, NR, false, DIPR>(sp, p + lane, gs + p, gs + p, ds + p, f, cfix, a);
  float r[8], l[2];
  rotor_warp_sum(a, r, l);
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < 8; ++k) s_red[w][k] = r[k];
    s_red[w][8] = l[0];
    s_red[w][9] = l[1];
  }
  __syncthreads();
  if (w != 0) return;
  if (lane < 8) {
    float h = s_red[0][lane], lo = lane < 2 ? s_red[0][8 + lane] + s_red[1][8 + lane] : 0.f;
    acc2(h, lo, s_red[1][lane]);
    s_fin[lane] = h + lo;
    if (lane < 2) s_fin[8 + lane] = lo - (s_fin[lane] - h);
  }
  __syncwarp();
  rotor_close<DIPR>(sp, md, m, lane, old, s_fin, s_fin + 8, err);
}

template <int J, int NR, bool DIPR>
static void launch_rotor_fused(const SpeciesDev& sp, const MolDev& md, int* err, cudaStream_t s) {
  constexpr int bytes = (2 * RotorDims<J>::NROT + 2) * NR * (int)sizeof(float2);
  auto k = mol_rotor_fused_kernel<J, NR, DIPR>;
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  k<<<sp.nmol, NR, bytes, s>>>(sp, md, err);
}
template <int J, int NR, bool DIPR>
static void launch_rotor_streaming(const SpeciesDev& sp, const MolDev& md, int* err, cudaStream_t s) {
  mol_rotor_kernel<J, NR, DIPR><<<sp.nmol, 64, 0, s>>>(sp, md, err);
}

template <int J>
static void launch_rotor_j(const SpeciesDev& sp, const MolDev& md, int* err, cudaStream_t s) {
  const bool fused = sp.path == MS_MOL_FUSED;  // N_r = 128
  if (sp.dipw) {                               // d(R): N_r 64 or 128
    if (fused) launch_rotor_fused<J, 128, true>(sp, md, err, s);
    else if (sp.nr == 128) launch_rotor_streaming<J, 128, true>(sp, md, err, s);
    else launch_rotor_streaming<J, 64, true>(sp, md, err, s);
  } else if (fused) launch_rotor_fused<J, 128, false>(sp, md, err, s);
  else if (sp.nr == 64) launch_rotor_streaming<J, 64, false>(sp, md, err, s);
  else if (sp.nr == 128) launch_rotor_streaming<J, 128, false>(sp, md, err, s);
  else launch_rotor_streaming<J, 256, false>(sp, md, err, s);
}

}  // namespace

void launch_rotor(const SpeciesDev& sp, const MolDev& md, int* err, cudaStream_t s) {
  switch (sp.jmax) {
    case 0: launch_rotor_j<0>(sp, md, err, s); break;
    case 1: launch_rotor_j<1>(sp, md, err, s); break;
    case 2: launch_rotor_j<2>(sp, md, err, s); break;
    case 3: launch_rotor_j<3>(sp, md, err, s); break;
    case 4: launch_rotor_j<4>(sp, md, err, s); break;
  }
}

}  // namespace ms
