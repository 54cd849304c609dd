// R-space pass on columns of the rotor (J = 5..8, streaming layout, reachable
// rows): the kernel and its launch.
//
// The reachable rows of a molecule are one vector psi_{j m} over all channels
// (the surface is the parity of j), and the coupling E'.R^ is E'_z Z within a
// column of fixed m plus S+- between neighbouring columns.  For the coupling a
// thread holds whole columns at one radial point in registers: the Z
// neighbours are its own, the S+- neighbours too except at the edges of its
// columns, and the coefficients are immediates of packed FP32x2 products.  A
// thread a row instead reads six neighbours of every row from shared memory,
// whose pipe then bounds the pass.
//
// Four warps take a molecule, 32 radial points at a time (lane = point).  Warps
// 0 and 1 hold the columns m = 0 .. K - 1 and K .. J, warps 2 and 3 the
// mirrored ones, -m: with mu = -m the coupling has the same form with the sign
// of E'_x flipped, so they run the same code.  Column 0 belongs to warp 0 and
// is read by warp 2.  The vector itself stands in shared memory (one array Y,
// rewritten term by term between barriers).
//
// Everything that is not the coupling (eta before it, the update after it) runs
// row by row in loops over Y, shared out evenly over the warps: only about 30
// instructions a row are unrolled.  With every phase unrolled (100 KB of code
// at J = 8) the pass waited for instructions: 8.8 ps a row and point; with the
// rows' loads one at a time for those loads: 12.5 ps.  A thread per row: 8.0 ps;
// now 5.9 to 6.5 at N_r = 128; 3.5 ps is HBM's.  What bounds it is latency, with
// the fifteen warps an SM that registers leave: at J = 8 an issued instruction costs
// 8.0 warp cycles, 1.6 of them global loads, 1.2 fixed latency, 0.9 barriers and
// 0.7 each shared memory, the FP32 pipe and instruction fetch; the shared-memory
// pipe is 71% and issue slots 47% busy.
//
// The coupling's exponential series S = sum_{n=1..N} T_n, T_1 = i theta M eta,
// T_n = (i theta / n) M T_{n-1}, is summed by Horner's rule on T_1: S = P_1, P_n
// = T_1 + (i theta / (n + 1)) M P_{n+1}, P_N = T_1.  On eta itself (S = i theta M
// (eta + (i theta / 2) M (eta + ..))) every step would round at eta's size, not at
// T_1's, which costs 3% in the populations' and dipoles' error against 64 bits.
#include "mol_common.cuh"

namespace ms {
namespace {

template <int J>
struct ColDims {
  static constexpr int len(int m) { return m > J ? 0 : J - m + 1; }  // rows of column m
  static constexpr int rows(int a, int b) {                          // rows of columns [a, b)
    int n = 0;
    for (int m = a; m < b; ++m) n += len(m);
    return n;
  }
  // columns 0 .. K - 1 on the low warps: the split with the smallest larger share, of two such the one with the
  // larger low share (J = 7: 21 and 15 rows took 23.4 ms where 15 and 21 took 23.9)
  static constexpr int split() {
    int best = 2;
    for (int k = 3; k <= J; ++k) {
      const int a = rows(0, k), b = rows(k, J + 1), c = rows(0, best), d = rows(best, J + 1);
      if ((a > b ? a : b) <= (c > d ? c : d)) best = k;
    }
    return best;
  }
  static constexpr int K = split();
  static constexpr int NROT = (J + 1) * (J + 1);
  // first row of shell j among the reachable rows: ground even shells, then excited odd shells
  static constexpr int shell(int j) {
    int n = 0;
    for (int q = 0; q <= J; ++q)
      if ((q & 1) < (j & 1) || ((q & 1) == (j & 1) && q < j)) n += 2 * q + 1;
    return n;
  }
  static constexpr int NG = shell(1);  // ground rows
  // rows whose loads a warp keeps in flight before the coupling, and after it for the ground and the excited rows:
  // few passes over a warp's rows (at J = 8: 21, 12 and 9) with few idle places.  Six throughout took 7.29, 6.97,
  // 7.43 and 6.84 ps a row and point at J = 5, 6, 7 and 8; these 6.07, 5.95, 6.03 and 6.50.
  static constexpr int EB = J == 8 ? 11 : (J == 7 ? 8 : (J == 6 ? 7 : 9));
  static constexpr int GB = J == 5 ? 4 : (J == 8 ? 6 : 7), XB = J == 5 ? 6 : (J == 6 ? 7 : 9);
};

constexpr int kColThreads = 128;

// warps arrive here from different code, so the barrier is named
__device__ __forceinline__ void col_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kColThreads) : "memory"); }

// One warp's columns: LOW 0 .. K - 1 (0 is only read when mirrored), else K .. J.
template <int J, bool LOW>
struct ColWarp {
  using D = ColDims<J>;
  static constexpr int C0 = LOW ? 0 : D::K, C1 = LOW ? D::K : J + 1, N = D::rows(C0, C1);
  static constexpr int ix(int c, int j) { return D::rows(C0, c) + j - c; }
  static constexpr int at(int j) { return D::shell(j) + j; }  // row (j, 0)

  // calls fn(c, j) for the rows of this warp's columns; OWN: those it stores
  template <bool OWN, class F>
  static __device__ __forceinline__ void each(bool mir, F&& fn) {
    static_for<C0, C1>([&](auto cc) {
      constexpr int c = decltype(cc)::value;
      if (OWN && LOW && c == 0 && mir) return;
      static_for<c, J + 1>([&](auto jc) { fn(cc, jc); });
    });
  }

  // Y <- S of the series on Y = eta (at this lane); row(j, c) of Y at Y + 32 (at(j) + sg c)
  static __device__ __forceinline__ void series(float2* Y, bool mir, int nterms, float fz, float fx, float fy) {
    const int sg = mir ? -32 : 32;  // from one column to the next
    float2 v[N], w[N];
    auto load = [&]() {
      each<false>(mir, [&](auto cc, auto jc) {
        constexpr int c = decltype(cc)::value, j = decltype(jc)::value;
        v[ix(c, j)] = (Y + sg * c)[32 * at(j)];
      });
    };
    auto store = [&]() {  // between barriers: every neighbour is read, then everything is written
      col_sync();
      each<true>(mir, [&](auto cc, auto jc) {
        constexpr int c = decltype(cc)::value, j = decltype(jc)::value;
        (Y + sg * c)[32 * at(j)] = w[ix(c, j)];
      });
      col_sync();
    };
    auto get = [&](auto cc, auto jc) -> float2 {
      constexpr int c = decltype(cc)::value, j = decltype(jc)::value;
      if constexpr (c >= C0 && c < C1) return v[ix(c, j)];
      else return (Y + sg * c)[32 * at(j)];
    };
    // i (M v) at row (c, j); z2, x2 and y the field's factors
    auto coupled = [&](auto cc, auto jc, float2 z2, float2 x2, float y) -> float2 {
      constexpr int c = decltype(cc)::value, j = decltype(jc)::value;
      auto sum2 = [&](auto cf0, auto cf1, auto c2) {  // cf0 (c2, j - 1) + cf1 (c2, j + 1)
        constexpr int cq = decltype(c2)::value, mq = cq < 0 ? -cq : cq;
        constexpr bool lo = j - 1 >= mq, hi = j + 1 <= J && j + 1 >= mq;
        using std::integral_constant;
        if constexpr (lo && hi)
          return fma2(dup2(cf0()), get(c2, integral_constant<int, j - 1>()),
                      mul2(dup2(cf1()), get(c2, integral_constant<int, j + 1>())));
        else if constexpr (lo) return mul2(dup2(cf0()), get(c2, integral_constant<int, j - 1>()));
        else if constexpr (hi) return mul2(dup2(cf1()), get(c2, integral_constant<int, j + 1>()));
        else return make_float2(0.f, 0.f);
      };
      const float2 az = sum2([] { return c_zd(j, c); }, [] { return c_zu(j, c); }, std::integral_constant<int, c>());
      const float2 ap = sum2([] { return c_pd(j, c); }, [] { return c_pu(j, c); }, std::integral_constant<int, c - 1>());
      const float2 am = sum2([] { return c_md(j, c); }, [] { return c_mu(j, c); }, std::integral_constant<int, c + 1>());
      const float2 t = fma2(z2, az, mul2(x2, add2(ap, am)));
      const float2 d = sub2(ap, am);
      return make_float2(fmaf(y, d.x, -t.y), fmaf(y, d.y, t.x));
    };
    load();
    each<true>(mir, [&](auto cc, auto jc) {  // T_1
      constexpr int c = decltype(cc)::value, j = decltype(jc)::value;
      w[ix(c, j)] = coupled(cc, jc, dup2(fz), dup2(fx), fy);
    });
    store();
    if (nterms == 2) {
      load();
      const float2 z2 = dup2(0.5f * fz), x2 = dup2(0.5f * fx);
      each<true>(mir, [&](auto cc, auto jc) {
        constexpr int c = decltype(cc)::value, j = decltype(jc)::value;
        w[ix(c, j)] = add2(v[ix(c, j)], coupled(cc, jc, z2, x2, 0.5f * fy));
      });
      store();
    } else if (nterms > 2) {
      float2 t1[N];  // in local memory (an index that the compiler does not know): no registers of the other branch
      int z;
      asm volatile("mov.u32 %0, 0;" : "=r"(z));
      each<true>(mir, [&](auto cc, auto jc) {
        constexpr int k = ix(decltype(cc)::value, decltype(jc)::value);
        t1[k + z] = w[k];
      });
#pragma unroll 1
      for (int n = nterms; n >= 2; --n) {
        load();
        const float cn = 1.f / (float)n;
        const float2 z2 = dup2(fz * cn), x2 = dup2(fx * cn);
        each<true>(mir, [&](auto cc, auto jc) {
          constexpr int k = ix(decltype(cc)::value, decltype(jc)::value);
          w[k] = add2(t1[k + z], coupled(cc, jc, z2, x2, fy * cn));
        });
        store();
      }
    }
  }

  // Dipole sums of Y = s': over pairs of rows of one column (Z) and of columns c, c + 1 (S+, S-); each pair
  // joins a ground and an excited row, and conj(g) e and conj(e) g give the same Re (P + M), Im (P - M).
  // Column 0's pairs with columns 1 and -1 are taken together: what the two have in common (the first-order
  // Im (g* e), much larger than the dipole) cancels before it is rounded in a product.
  static __device__ __forceinline__ void dipole(const float2* Y, bool mir, float2& ax, float& ay, float2& az) {
    const int sg = mir ? -32 : 32;
    float2 v[N];
    each<false>(mir, [&](auto cc, auto jc) {
      constexpr int c = decltype(cc)::value, j = decltype(jc)::value;
      v[ix(c, j)] = (Y + sg * c)[32 * at(j)];
    });
    each<true>(mir, [&](auto cc, auto jc) {
      constexpr int c = decltype(cc)::value, j = decltype(jc)::value;
      if constexpr (j < J) az = fma2(dup2(c_zu(j, c)), mul2(v[ix(c, j)], v[ix(c, j + 1)]), az);
    });
    each<true>(mir, [&](auto cc, auto jc) {
      constexpr int c = decltype(cc)::value, j = decltype(jc)::value;
      if constexpr (c < J) {
        constexpr bool hi = j + 1 <= J, lo = j - 1 >= c + 1;
        auto sum = [&](auto up) {  // over the neighbours (j + 1, c + 1) and (j - 1, c + 1)
          float2 t = make_float2(0.f, 0.f);
          if constexpr (hi) t = mul2(dup2(c_mu(j, c)), up(std::integral_constant<int, j + 1>()));
          if constexpr (lo && hi) t = fma2(dup2(c_md(j, c)), up(std::integral_constant<int, j - 1>()), t);
          else if constexpr (lo) t = mul2(dup2(c_md(j, c)), up(std::integral_constant<int, j - 1>()));
          return t;
        };
        if constexpr (hi || lo) {
          const float2 q = v[ix(c, j)];
          float2 tx, ty;
          if constexpr (c == 0) {  // not mirrored
            static_assert(C1 > 1, "column 1 stands beside column 0");
            auto m1 = [&](auto jq) { return (Y - 32)[32 * at(decltype(jq)::value)]; };
            tx = sum([&](auto jq) { return sub2(v[ix(1, decltype(jq)::value)], m1(jq)); });
            ty = sum([&](auto jq) { return add2(v[ix(1, decltype(jq)::value)], m1(jq)); });
          } else {
            tx = ty = sum([&](auto jq) -> float2 {
              if constexpr (c + 1 < C1) return v[ix(c + 1, decltype(jq)::value)];
              else return (Y + sg * (c + 1))[32 * at(decltype(jq)::value)];
            });
          }
          ax = fma2(q, tx, ax);
          ay = fmaf(q.y, ty.x, fmaf(-q.x, ty.y, ay));
        }
      }
    });
  }
};

template <int J>
__global__ void __launch_bounds__(kColThreads, 4) mol_rspace_col_kernel(SpeciesDev sp, MolDev md, int* err) {
  using D = ColDims<J>;
  constexpr int NROT = D::NROT, NG = D::NG;
  if (idle_launch(sp)) return;
  __shared__ float2 Ys[NROT][32];
  __shared__ int s_vt[NROT];  // row -> its shell's row of the phase table
  __shared__ float s_fin[8], s_fin_lo[2];  // P_g, P_e, Re(S+ + S-), Im(S+ - S-), 2 Re Z, absorbed (2), rounding residuals
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int lm = blockIdx.x, m = sp.mol[lm], NR = sp.nr;
  const float4 f = __ldg(&sp.fld[lm]);  // (theta E'_z, theta E'_x/2, theta E'_y/2, terms)
  const float cfix = md.ncorr[m];       // rounding feedback of the previous step
  const float2 cf = dup2(cfix);
  // what the closing threads add to: the previous dipole, the absorbed norm so far
  const double old = t < 3 ? md.mu[3 * (long long)m + t]
                           : (t == 5 || t == 6 ? md.absorbed[2 * (long long)m + (t - 5)] : 0.0);
  for (int q = t; q < NROT; q += kColThreads) {
    int j = q >= NG, r = q - (j ? NG : 0);
    while (r >= 2 * j + 1 && j + 2 <= J) {
      r -= 2 * j + 1;
      j += 2;
    }
    s_vt[q] = j * NR;
  }
  const int nterms = max(__float_as_int(f.w), 1);  // no field: one term of zeros
  const bool mir = (w & 2) != 0;
  const float fx = mir ? -f.y : f.y;
  float2* const Y = &Ys[0][lane];
  float2 hi = make_float2(0.f, 0.f), lo = hi, ax = hi, az = hi, rnd = hi;  // hi, lo: populations (ground, excited)
  float ab[2] = {0.f, 0.f}, ay = 0.f;

#pragma unroll 1
  for (int r0 = 0; r0 < NR; r0 += 32) {
    float2* const s = sp.psi + (long long)lm * sp.mrows * NR + r0 + lane;
    const float2* const d = sp.d2 + (long long)lm * NROT * NR + r0 + lane;
    const float4* const vt = sp.vcol + r0 + lane;
    const float2 mk = __ldg(&sp.maskw[r0 + lane]);
    __syncthreads();  // the table is built; the last points' dipole has read Y
    // ---- eta = V^{1/2} (s + d2): rows w, w + 4, .., D::EB at a time, their loads in flight together
#pragma unroll 1
    for (int q0 = w; q0 < NROT; q0 += 4 * D::EB) {
      float2 s0[D::EB], d0[D::EB], p[D::EB];
#pragma unroll
      for (int i = 0; i < D::EB; ++i) {
        const int q = min(q0 + 4 * i, NROT - 1);
        s0[i] = s[q * NR];
        d0[i] = __ldg(d + q * NR);
        p[i] = __ldg(reinterpret_cast<const float2*>(vt + s_vt[q]));
      }
#pragma unroll
      for (int i = 0; i < D::EB; ++i)
        if (q0 + 4 * i < NROT) Y[32 * (q0 + 4 * i)] = cmul(p[i], add2(s0[i], d0[i]));
    }
    if (r0 + 32 < NR) {  // the next points' lines towards L2
      for (int q = t; q < 4 * NROT; q += kColThreads) {
        const float2* b = (q & 1 ? d : s) - lane + 32 + (q >> 2) * NR + (q & 2) * 8;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(b));
      }
    }
    __syncthreads();
    // ---- Y <- S
    if (w & 1) ColWarp<J, false>::series(Y, mir, nterms, f.x, fx, f.z);
    else ColWarp<J, true>::series(Y, mir, nterms, f.x, fx, f.z);
    // ---- d1 = (V - 1) u + V^{1/2} S, mask, s' = s + (d2 + d1) + cfix s; a surface at a time
    const bool masked = mk.x < 1.f;
    static_for<0, 2>([&](auto sfc) {
      constexpr int sf = decltype(sfc)::value, q1 = sf ? NROT : NG, UB = sf ? D::XB : D::GB;
      float2 h2 = make_float2(sf ? hi.y : hi.x, 0.f), l2 = make_float2(sf ? lo.y : lo.x, 0.f);
#pragma unroll 1
      for (int q0 = (sf ? NG : 0) + w; q0 < q1; q0 += 4 * UB) {
        float2 s0[UB], d0[UB];
        float4 p[UB];
#pragma unroll
        for (int i = 0; i < UB; ++i) {
          const int q = min(q0 + 4 * i, q1 - 1);
          s0[i] = s[q * NR];
          d0[i] = __ldg(d + q * NR);
          p[i] = __ldg(vt + s_vt[q]);
        }
        float b2 = 0.f;
#pragma unroll
        for (int i = 0; i < UB; ++i) {
          const int q = q0 + 4 * i;
          float b = 0.f;
          if (q < q1) {
            const float2 S = Y[32 * q], u = add2(s0[i], d0[i]);
            float2 d1 = make_float2(fmaf(p[i].z, u.x, fmaf(-p[i].w, u.y, fmaf(p[i].x, S.x, -p[i].y * S.y))),
                                    fmaf(p[i].z, u.y, fmaf(p[i].w, u.x, fmaf(p[i].x, S.y, p[i].y * S.x))));
            if (masked) {
              const float2 z = add2(u, d1);
              d1 = fma2(dup2(mk.x - 1.f), u, mul2(dup2(mk.x), d1));
              ab[sf] += mk.y * fmaf(z.x, z.x, z.y * z.y);
            }
            const float2 sn = round_update2(s0[i], add2(d0[i], d1), cf, rnd);
            __stcs(s + q * NR, sn);
            Y[32 * q] = sn;
            b = fmaf(sn.x, sn.x, sn.y * sn.y);
          }
          if (i & 1) acc2p(h2, l2, make_float2(b2, b));  // compensated from the first term on
          else if (i == UB - 1) acc2p(h2, l2, make_float2(b, 0.f));
          else b2 = b;
        }
      }
      float h = h2.x, l = l2.x + l2.y;
      acc2(h, l, h2.y);
      if (sf) hi.y = h, lo.y = l;
      else hi.x = h, lo.x = l;
    });
    __syncthreads();
    if (w & 1) ColWarp<J, false>::dipole(Y, mir, ax, ay, az);
    else ColWarp<J, true>::dipole(Y, mir, ax, ay, az);
  }
  // ---- block sums: a lane's values of the four warps first, then a tree over the lanes; warp w takes the
  // quantities w and w + 4.  Mirrored columns count E'_x reversed, and what is much larger than the dipole in
  // each (the first-order Im (g* e)) cancels against the other lane by lane: a tree over each warp's own part
  // rounds at that part's size instead (the dipoles' error against 64 bits at J = 8, N_r = 128, with the same in
  // dipole(): 1.75e-7, now 1.31e-7).
  __syncthreads();  // the last points' dipole has read Y
  float* const red = reinterpret_cast<float*>(&Ys[0][0]);
  {
    const float dx = ax.x + ax.y;
    const float v[10] = {hi.x, hi.y, mir ? -dx : dx, ay, 2.f * (az.x + az.y), ab[0], ab[1], rnd.x + rnd.y, lo.x, lo.y};
#pragma unroll
    for (int k = 0; k < 10; ++k) red[k * kColThreads + t] = v[k];
  }
  __syncthreads();
#pragma unroll
  for (int k = w; k < 8; k += 4) {
    float h = 0.f, l = 0.f;
#pragma unroll
    for (int ww = 0; ww < 4; ++ww) {
      acc2(h, l, red[k * kColThreads + 32 * ww + lane]);
      if (k < 2) l += red[(8 + k) * kColThreads + 32 * ww + lane];
    }
    if (k < 2) {  // populations compensated
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float h2 = __shfl_xor_sync(0xffffffffu, h, o), l2 = __shfl_xor_sync(0xffffffffu, l, o);
        acc2(h, l, h2);
        l += l2;
      }
    } else {
      h += l;
      l = 0.f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
    }
    if (lane == 0) {
      s_fin[k] = h + l;
      if (k < 2) s_fin_lo[k] = l - (s_fin[k] - h);
    }
  }
  __syncthreads();
  if (t < 3) {  // lab dipole: mu = O mu', mu' = d dR (Re(S+ + S-), Im(S+ - S-), 2 Re Z)
    const float* O = md.rot + 9 * (long long)m + 3 * t;
    const float lab = (float)sp.dipole * sp.dR * (O[0] * s_fin[2] + O[1] * s_fin[3] + O[2] * s_fin[4]);
    const double nl = (double)lab;
    md.dmu[3 * (long long)m + t] = nl - old;
    md.mu[3 * (long long)m + t] = nl;
  } else if (t < 5) {
    const double P = ((double)s_fin[t - 3] + (double)s_fin_lo[t - 3]) * (double)sp.dR;
    md.pop[2 * (long long)m + (t - 3)] = P;
    if (!isfinite(P)) atomicOr(err, kErrNonFinite);
  } else if (t < 7) {
    md.absorbed[2 * (long long)m + (t - 5)] = old + (double)s_fin[t] * (double)sp.dR;
  } else if (t == 7) {
    md.ncorr[m] = rounding_feedback(s_fin[7], s_fin[0] + s_fin[1]);
  }
}

}  // namespace

void launch_rspace_col(const SpeciesDev& sp, const MolDev& md, int* err, cudaStream_t s) {
  switch (sp.jmax) {
    case 5: mol_rspace_col_kernel<5><<<sp.nmol, kColThreads, 0, s>>>(sp, md, err); break;
    case 6: mol_rspace_col_kernel<6><<<sp.nmol, kColThreads, 0, s>>>(sp, md, err); break;
    case 7: mol_rspace_col_kernel<7><<<sp.nmol, kColThreads, 0, s>>>(sp, md, err); break;
    case 8: mol_rspace_col_kernel<8><<<sp.nmol, kColThreads, 0, s>>>(sp, md, err); break;
  }
}

}  // namespace ms
