// Yee leap-frog kernels for Eq. 1 with the Drude current of Eq. 2, CPML
// along z, periodic x/y, TF/SF plane-wave source and the molecular
// polarization current (section "The domain decomposition methodology for
// FDTD"; coupling section for dP/dt).
//
// Both half steps are stencils bound by HBM (grids beyond L2) or by the loads
// in flight.  A thread marches along z through four neighbouring columns (x to
// x + 3, 16-byte loads), the lanes running over the plane's quads in storage
// order; the z neighbour stays in registers, the x neighbour comes from the
// adjacent lane, the y neighbour through L1/L2.  Rows that are no multiple of
// four cells take the kernels with one column a thread, which issue about 180
// instructions for 32 cells of a plane where these issue about 130 for 128.
#include "ms_internal.cuh"

namespace ms {

// The two half steps march along z: a block owns a tile of 32 x 8 columns
// (i, j) and kKz planes, one thread per column.  Each thread carries the
// plane it shares with the next (previous) cell of its column in registers,
// takes its x neighbour from the adjacent lane by a shuffle (the last lane of
// a warp, and the periodic wrap, load it), and reads its y neighbour through
// L1/L2.  Lanes outside the grid load a valid cell and store nothing.
constexpr int kTx = 32, kTy = 8, kKz = 8;

struct Tile {
  int i, j, s, k0, k1;
  bool in;
};

__device__ __forceinline__ Tile tile_of(const Grid& g, int b) {
  const int tx = (g.nx + kTx - 1) / kTx, ty = (g.ny + kTy - 1) / kTy, tz = (g.nz + kKz - 1) / kKz;
  Tile t;
  const int bx = b % tx;
  b /= tx;
  const int by = b % ty;
  b /= ty;
  const int bz = b % tz;
  t.s = b / tz;
  t.i = bx * kTx + (int)threadIdx.x;
  t.j = by * kTy + (int)threadIdx.y;
  t.k0 = bz * kKz;
  t.k1 = min(t.k0 + kKz, g.nz);
  t.in = t.i < g.nx && t.j < g.ny;
  return t;
}

static int yee_tiles(const Grid& g) {
  return ((g.nx + kTx - 1) / kTx) * ((g.ny + kTy - 1) / kTy) * ((g.nz + kKz - 1) / kKz) * g.nsim;
}

__device__ __forceinline__ long long pml_index(const Grid& g, int s, int k, int j, int i) {
  const int slab = k < g.pml ? 0 : 1;
  const int kk = k < g.pml ? k : k - (g.nz - g.pml);
  return (((long long)(s * 2 + slab) * g.pml + kk) * g.ny + j) * g.nx + i;
}

// Incident line.  Node m of the line sits at z = (ks - 2 + m) dx; only nodes
// inside the numerical light cone of the source (m <= step + 2) can be
// non-zero, so only those are touched.  kAuxBlocks blocks per sim share them:
// with one, a long run waits for its line (at 30,000 steps of the 32 x 32 x 64
// workload a step took 48 us, 21 us of them for the line).
constexpr int kAuxBlocks = 32;

// H half step by block b of a sim's, nt threads each
__device__ void aux_h_block(const Grid& g, int b, int t, int nt) {
  const int s = b / kAuxBlocks;
  const long long n = *g.step;
  const int lim = (int)min((long long)g.aux_len, n + 4);
  float* E1 = g.auxE + (long long)s * (g.aux_len + 1);
  float* H1 = g.auxH + (long long)s * g.aux_len;
  for (int m = (b % kAuxBlocks) * nt + t; m < lim; m += kAuxBlocks * nt) H1[m] -= g.ch * (E1[m + 1] - E1[m]);
}

// E half step, and the new source sample at node 0.
__device__ void aux_e_block(const Grid& g, int b, int t, int nt) {
  const int s = b / kAuxBlocks;
  const long long n = *g.step;
  const int lim = (int)min((long long)g.aux_len, n + 4);
  float* E1 = g.auxE + (long long)s * (g.aux_len + 1);
  const float* H1 = g.auxH + (long long)s * g.aux_len;
  const float ce = g.ce_vac;
  for (int m = 1 + (b % kAuxBlocks) * nt + t; m < lim; m += kAuxBlocks * nt) E1[m] += ce * (0.f - (H1[m] - H1[m - 1]));
  if (b % kAuxBlocks == 0 && t == 0) E1[0] = (float)incident_field(g.src[s], (double)(n + 1) * g.dt);
}

// H^{n-1/2} -> H^{n+1/2}.  Blocks past the tiles step the incident lines
// (they read only the lines; the tiles read only E and one line sample).
// The loads of plane k + 1 are issued before plane k is computed and stored,
// so every warp keeps two planes of loads in flight.
struct HPlane {
  float ez, ex_z, ey_z, ez_y, ex_y, ez_x, ey_x, h0, h1, h2;
};

__global__ void __launch_bounds__(kTx * kTy, 6) yee_h_kernel(Grid g, int ntiles) {
  if ((int)blockIdx.x >= ntiles) {
    aux_h_block(g, (int)blockIdx.x - ntiles, threadIdx.y * kTx + threadIdx.x, kTx * kTy);
    return;
  }
  const Tile t = tile_of(g, blockIdx.x);
  const int i = t.in ? t.i : 0, j = t.in ? t.j : 0;
  const int sxy = g.nx * g.ny;                                   // offsets within one sim (< 2^31 cells)
  const int dx = i + 1 < g.nx ? 1 : 1 - g.nx;                    // to (i + 1) mod nx
  const int dy = j + 1 < g.ny ? g.nx : -(g.ny - 1) * g.nx;       // to (j + 1) mod ny
  const int dzw = -(g.nz - 1) * sxy;                             // top plane -> bottom plane (periodic)
  const bool xsh = threadIdx.x + 1 < kTx && i + 1 < g.nx;        // the next lane holds i + 1
  const long long sb = (long long)t.s * g.ncell_sim;
  const float* __restrict__ Ex = g.E[0] + sb;
  const float* __restrict__ Ey = g.E[1] + sb;
  const float* __restrict__ Ez = g.E[2] + sb;
  float* __restrict__ H0 = g.H[0] + sb;
  float* __restrict__ H1 = g.H[1] + sb;
  float* __restrict__ H2 = g.H[2] + sb;
  const int c0 = t.k0 * sxy + j * g.nx + i;
  // plane k: E on k and k + 1 (zero above a conducting top), the y and x
  // neighbours (x only where no lane holds it), and H
  auto load = [&](int k, int c) {
    HPlane p;
    const bool top = k + 1 >= g.nz, zero_top = top && !g.periodic_z;
    const int cz = c + (top ? dzw : sxy);
    p.ez = Ez[c];
    p.ex_z = zero_top ? 0.f : Ex[cz];
    p.ey_z = zero_top ? 0.f : Ey[cz];
    p.ez_y = Ez[c + dy];
    p.ex_y = Ex[c + dy];
    p.ez_x = xsh ? 0.f : Ez[c + dx];
    p.ey_x = xsh ? 0.f : Ey[c + dx];
    p.h0 = H0[c];
    p.h1 = H1[c];
    p.h2 = H2[c];
    return p;
  };
  float ex = Ex[c0], ey = Ey[c0];  // plane k, carried from the previous iteration
  HPlane nx_ = load(t.k0, c0);
  int c = c0;
  for (int k = t.k0; k < t.k1; ++k, c += sxy) {
    const HPlane p = nx_;
    if (k + 1 < t.k1) nx_ = load(k + 1, c + sxy);
    const float ez_n = __shfl_down_sync(0xffffffffu, p.ez, 1);
    const float ey_n = __shfl_down_sync(0xffffffffu, ey, 1);
    const float ez_x = xsh ? ez_n : p.ez_x;
    const float ey_x = xsh ? ey_n : p.ey_x;
    float dEz_dy = p.ez_y - p.ez;
    float dEy_dz = p.ey_z - ey;
    float dEx_dz = p.ex_z - ex;
    const float dEz_dx = ez_x - p.ez;
    const float dEy_dx = ey_x - ey;
    const float dEx_dy = p.ex_y - ex;
    if (g.pml > 0 && (k < g.pml || k >= g.nz - g.pml)) {
      const float4 co = g.cpml[k];  // (bE, aE, bH, aH); psi stored times dx
      const long long q = pml_index(g, t.s, k, j, i);
      const float px = co.z * g.psiH[0][q] + co.w * dEy_dz;
      const float py = co.z * g.psiH[1][q] + co.w * dEx_dz;
      if (t.in) {
        g.psiH[0][q] = px;
        g.psiH[1][q] = py;
      }
      dEy_dz += px;
      dEx_dz += py;
    }
    float hy_src = 0.f;
    if (k == g.ks - 1) hy_src = g.auxE[(long long)t.s * (g.aux_len + 1) + 2];
    if (t.in) {
      H0[c] = p.h0 - g.ch * (dEz_dy - dEy_dz);
      H1[c] = p.h1 - g.ch * (dEx_dz - dEz_dx) + g.ch * hy_src;
      H2[c] = p.h2 - g.ch * (dEy_dx - dEx_dy);
    }
    ex = p.ex_z;
    ey = p.ey_z;
  }
}

// E^n -> E^{n+1}, with J_D^{n+1/2} and the molecular polarization change.
// Blocks past the tiles step the incident lines and set the new source
// sample (they read only the lines' H; the tiles read one H sample).
// Pipelined over the planes as the H half step.
struct EPlane {
  float hx, hy, hz, hz_y, hx_y, hz_x, hy_x, e0, e1, e2;
  int mat;
};

__global__ void __launch_bounds__(kTx * kTy, 5) yee_e_kernel(Grid g, int ntiles) {
  if ((int)blockIdx.x >= ntiles) {
    aux_e_block(g, (int)blockIdx.x - ntiles, threadIdx.y * kTx + threadIdx.x, kTx * kTy);
    return;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0 && threadIdx.y == 0) *g.step_next = *g.step + 1;
  const Tile t = tile_of(g, blockIdx.x);
  const int i = t.in ? t.i : 0, j = t.in ? t.j : 0;
  const int sxy = g.nx * g.ny;                               // offsets within one sim (< 2^31 cells)
  const int dx = i > 0 ? 1 : 1 - g.nx;                       // from (i - 1) mod nx
  const int dy = j > 0 ? g.nx : -(g.ny - 1) * g.nx;          // from (j - 1) mod ny
  const bool xsh = threadIdx.x > 0 && i > 0;                 // the previous lane holds i - 1
  const long long sb = (long long)t.s * g.ncell_sim;
  const float* __restrict__ Hx = g.H[0] + sb;
  const float* __restrict__ Hy = g.H[1] + sb;
  const float* __restrict__ Hz = g.H[2] + sb;
  float* __restrict__ E0 = g.E[0] + sb;
  float* __restrict__ E1 = g.E[1] + sb;
  float* __restrict__ E2 = g.E[2] + sb;
  const uint8_t* __restrict__ mat = g.mat + sb;
  const int c0 = t.k0 * sxy + j * g.nx + i;
  auto load = [&](int c) {
    EPlane p;
    p.hx = Hx[c];
    p.hy = Hy[c];
    p.hz = Hz[c];
    p.hz_y = Hz[c - dy];
    p.hx_y = Hx[c - dy];
    p.hz_x = xsh ? 0.f : Hz[c - dx];
    p.hy_x = xsh ? 0.f : Hy[c - dx];
    p.e0 = E0[c];
    p.e1 = E1[c];
    p.e2 = E2[c];
    p.mat = mat[c];
    return p;
  };
  // plane k - 1, carried from the previous iteration
  float hx_m = 0.f, hy_m = 0.f;
  if (t.k0 > 0) {
    hx_m = Hx[c0 - sxy];
    hy_m = Hy[c0 - sxy];
  } else if (g.periodic_z) {
    hx_m = Hx[c0 + (g.nz - 1) * sxy];
    hy_m = Hy[c0 + (g.nz - 1) * sxy];
  }  // else: perfect conductor below the bottom plane
  EPlane nx_ = load(c0);
  int c = c0;
  for (int k = t.k0; k < t.k1; ++k, c += sxy) {
    const EPlane p = nx_;
    if (k + 1 < t.k1) nx_ = load(c + sxy);
    const float hz_n = __shfl_up_sync(0xffffffffu, p.hz, 1);
    const float hy_n = __shfl_up_sync(0xffffffffu, p.hy, 1);
    const float hz_x = xsh ? hz_n : p.hz_x;
    const float hy_x = xsh ? hy_n : p.hy_x;
    float dHz_dy = p.hz - p.hz_y;
    float dHy_dz = p.hy - hy_m;
    float dHx_dz = p.hx - hx_m;
    const float dHz_dx = p.hz - hz_x;
    const float dHy_dx = p.hy - hy_x;
    const float dHx_dy = p.hx - p.hx_y;
    hx_m = p.hx;
    hy_m = p.hy;
    if (g.pml > 0 && (k < g.pml || k >= g.nz - g.pml)) {
      const float4 co = g.cpml[k];
      const long long q = pml_index(g, t.s, k, j, i);
      const float px = co.x * g.psiE[0][q] + co.y * dHy_dz;
      const float py = co.x * g.psiE[1][q] + co.y * dHx_dz;
      if (t.in) {
        g.psiE[0][q] = px;
        g.psiE[1][q] = py;
      }
      dHy_dz += px;
      dHx_dz += py;
    }
    float cxv = dHz_dy - dHy_dz;
    const float cyv = dHx_dz - dHz_dx;
    const float czv = dHy_dx - dHx_dy;
    if (k == g.ks) cxv += g.auxH[(long long)t.s * g.aux_len + 1];
    if (t.in) {
      const MaterialCoef mc = g.mc[p.mat];
      float ex = p.e0, ey = p.e1, ez = p.e2;
      float jx = 0.f, jy = 0.f, jz = 0.f;
      if (mc.metal && k >= g.jk0 && k < g.jk1) {
        const long long jj = (((long long)t.s * (g.jk1 - g.jk0) + (k - g.jk0)) * g.ny + j) * g.nx + i;
        jx = mc.alpha * g.J[0][jj] + mc.beta * ex;
        jy = mc.alpha * g.J[1][jj] + mc.beta * ey;
        jz = mc.alpha * g.J[2][jj] + mc.beta * ez;
        g.J[0][jj] = jx;
        g.J[1][jj] = jy;
        g.J[2][jj] = jz;
      }
      ex += mc.ce * cxv - mc.cj * jx;
      ey += mc.ce * cyv - mc.cj * jy;
      ez += mc.ce * czv - mc.cj * jz;
      if (k >= g.mk0 && k < g.mk1) {
        const long long sl = (((long long)t.s * (g.mk1 - g.mk0) + (k - g.mk0)) * g.ny + j) * g.nx + i;
        const int b = g.cell_off[sl], e = g.cell_off[sl + 1];
        if (e > b) {
          double px = 0.0, py = 0.0, pz = 0.0;  // ensemble sum in FP64
          for (int q = b; q < e; ++q) {
            const int m = g.cell_mol[q];
            px += g.dmu[3 * (long long)m + 0];
            py += g.dmu[3 * (long long)m + 1];
            pz += g.dmu[3 * (long long)m + 2];
          }
          ex -= mc.cp * (float)px;
          ey -= mc.cp * (float)py;
          ez -= mc.cp * (float)pz;
        }
      }
      if (!g.periodic_z && k == 0) {
        ex = 0.f;  // tangential E on the bottom conductor
        ey = 0.f;
      }
      E0[c] = ex;
      E1[c] = ey;
      E2[c] = ez;
    }
  }
}

// ---- four columns a thread ---------------------------------------------------
// Phases of a step, H and E half step: 256^3 with a 100 nm film 118 -> 101 us
// (6.0 TB/s) and 144 -> 137 us; 128 x 128 x 192, whose fields stay in L2, 29 ->
// 18 us and 31 -> 21 us; 32 x 32 x 64 10.3 -> 6.6 us and 13.4 -> 9.9 us.
// A thread takes quad q of the plane (row j = q / (nx/4), cells 4 i4 .. 4 i4 + 3)
// and kz planes.  Quads past the plane load the last one and store nothing.
constexpr int kQt = 128;  // threads a block

struct Quad {
  int i, j, s, k0, k1;  // first cell, row, sim, planes
  bool in, last, first; // in the plane; the row's last, first quad
};

__device__ __forceinline__ Quad quad_of(const Grid& g, int b, int kz) {
  const int n4 = g.nx >> 2, np = n4 * g.ny, tq = (np + kQt - 1) / kQt, tz = (g.nz + kz - 1) / kz;
  Quad t;
  int q = (b % tq) * kQt + (int)threadIdx.x;
  b /= tq;
  t.in = q < np;
  q = min(q, np - 1);
  t.j = q / n4;
  const int i4 = q - t.j * n4;
  t.i = 4 * i4;
  t.first = i4 == 0;
  t.last = i4 == n4 - 1;
  t.k0 = (b % tz) * kz;
  t.k1 = min(t.k0 + kz, g.nz);
  t.s = b / tz;
  return t;
}

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ float4 operator-(float4 a, float4 b) {
  return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
}
__device__ __forceinline__ float4 operator+(float4 a, float4 b) {
  return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}
// a x + b y
__device__ __forceinline__ float4 comb4(float a, float4 x, float b, float4 y) {
  return make_float4(a * x.x + b * y.x, a * x.y + b * y.y, a * x.z + b * y.z, a * x.w + b * y.w);
}
// h - c d
__device__ __forceinline__ float4 sub_mul4(float4 h, float c, float4 d) {
  return make_float4(h.x - c * d.x, h.y - c * d.y, h.z - c * d.z, h.w - c * d.w);
}
// the quad moved by one cell: (b, c, d, next quad's a) and (previous quad's d, a, b, c)
__device__ __forceinline__ float4 up_x(float4 v, float edge, bool shuffled) {
  const float n = __shfl_down_sync(0xffffffffu, v.x, 1);
  return make_float4(v.y, v.z, v.w, shuffled ? n : edge);
}
__device__ __forceinline__ float4 down_x(float4 v, float edge, bool shuffled) {
  const float n = __shfl_up_sync(0xffffffffu, v.w, 1);
  return make_float4(shuffled ? n : edge, v.x, v.y, v.z);
}

// H^{n-1/2} -> H^{n+1/2} (the arithmetic of yee_h_kernel)
__global__ void __launch_bounds__(kQt) yee_h4_kernel(Grid g, int ntiles, int kz) {
  if ((int)blockIdx.x >= ntiles) {
    aux_h_block(g, (int)blockIdx.x - ntiles, threadIdx.x, kQt);
    return;
  }
  const Quad t = quad_of(g, blockIdx.x, kz);
  const int sxy = g.nx * g.ny;
  const int dy = t.j + 1 < g.ny ? g.nx : -(g.ny - 1) * g.nx;
  const int dx = t.last ? 4 - g.nx : 4;                      // to the first cell of the next quad of the row
  const bool xsh = (threadIdx.x & 31) < 31 && !t.last;       // the next lane holds it
  const long long sb = (long long)t.s * g.ncell_sim;
  const float* __restrict__ Ex = g.E[0] + sb;
  const float* __restrict__ Ey = g.E[1] + sb;
  const float* __restrict__ Ez = g.E[2] + sb;
  float* __restrict__ H0 = g.H[0] + sb;
  float* __restrict__ H1 = g.H[1] + sb;
  float* __restrict__ H2 = g.H[2] + sb;
  int c = t.k0 * sxy + t.j * g.nx + t.i;
  float4 ex = ld4(Ex + c), ey = ld4(Ey + c);
  for (int k = t.k0; k < t.k1; ++k, c += sxy) {
    const bool top = k + 1 >= g.nz;
    const int cz = c + (top ? -(g.nz - 1) * sxy : sxy);
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const bool zero_top = top && !g.periodic_z;
    const float4 ex_z = zero_top ? z4 : ld4(Ex + cz), ey_z = zero_top ? z4 : ld4(Ey + cz);
    const float4 ez = ld4(Ez + c), ez_y = ld4(Ez + c + dy), ex_y = ld4(Ex + c + dy);
    const float4 h0 = ld4(H0 + c), h1 = ld4(H1 + c), h2 = ld4(H2 + c);
    const float ez_e = xsh ? 0.f : Ez[c + dx], ey_e = xsh ? 0.f : Ey[c + dx];
    const float4 dEz_dy = ez_y - ez, dEx_dy = ex_y - ex;
    float4 dEy_dz = ey_z - ey, dEx_dz = ex_z - ex;
    const float4 dEz_dx = up_x(ez, ez_e, xsh) - ez, dEy_dx = up_x(ey, ey_e, xsh) - ey;
    if (g.pml > 0 && (k < g.pml || k >= g.nz - g.pml)) {
      const float4 co = g.cpml[k];  // (bE, aE, bH, aH); psi stored times dx
      const long long q = pml_index(g, t.s, k, t.j, t.i);
      const float4 px = comb4(co.z, ld4(g.psiH[0] + q), co.w, dEy_dz);
      const float4 py = comb4(co.z, ld4(g.psiH[1] + q), co.w, dEx_dz);
      if (t.in) {
        st4(g.psiH[0] + q, px);
        st4(g.psiH[1] + q, py);
      }
      dEy_dz = dEy_dz + px;
      dEx_dz = dEx_dz + py;
    }
    if (t.in) {
      st4(H0 + c, sub_mul4(h0, g.ch, dEz_dy - dEy_dz));
      float4 n1 = sub_mul4(h1, g.ch, dEx_dz - dEz_dx);
      if (k == g.ks - 1) {
        const float a = g.auxE[(long long)t.s * (g.aux_len + 1) + 2];
        n1 = make_float4(fmaf(g.ch, a, n1.x), fmaf(g.ch, a, n1.y), fmaf(g.ch, a, n1.z), fmaf(g.ch, a, n1.w));
      }
      st4(H1 + c, n1);
      st4(H2 + c, sub_mul4(h2, g.ch, dEy_dx - dEx_dy));
    }
    ex = ex_z;
    ey = ey_z;
  }
}

// E^n -> E^{n+1} (the arithmetic of yee_e_kernel)
__global__ void __launch_bounds__(kQt) yee_e4_kernel(Grid g, int ntiles, int kz) {
  if ((int)blockIdx.x >= ntiles) {
    aux_e_block(g, (int)blockIdx.x - ntiles, threadIdx.x, kQt);
    return;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *g.step_next = *g.step + 1;
  const Quad t = quad_of(g, blockIdx.x, kz);
  const int sxy = g.nx * g.ny;
  const int dy = t.j > 0 ? g.nx : -(g.ny - 1) * g.nx;
  const int dx = t.first ? g.nx - 1 : -1;                    // to the last cell of the previous quad of the row
  const bool xsh = (threadIdx.x & 31) > 0 && !t.first;       // the previous lane holds it
  const long long sb = (long long)t.s * g.ncell_sim;
  const float* __restrict__ Hx = g.H[0] + sb;
  const float* __restrict__ Hy = g.H[1] + sb;
  const float* __restrict__ Hz = g.H[2] + sb;
  float* const E[3] = {g.E[0] + sb, g.E[1] + sb, g.E[2] + sb};
  int c = t.k0 * sxy + t.j * g.nx + t.i;
  float4 hx_m = make_float4(0.f, 0.f, 0.f, 0.f), hy_m = hx_m;  // plane k - 1
  if (t.k0 > 0 || g.periodic_z) {
    const int cm = t.k0 > 0 ? c - sxy : c + (g.nz - 1) * sxy;
    hx_m = ld4(Hx + cm);
    hy_m = ld4(Hy + cm);
  }  // else: perfect conductor below the bottom plane
  for (int k = t.k0; k < t.k1; ++k, c += sxy) {
    const float4 hx = ld4(Hx + c), hy = ld4(Hy + c), hz = ld4(Hz + c), hz_y = ld4(Hz + c - dy), hx_y = ld4(Hx + c - dy);
    const float4 e0 = ld4(E[0] + c), e1 = ld4(E[1] + c), e2 = ld4(E[2] + c);
    const unsigned mats = *reinterpret_cast<const unsigned*>(g.mat + sb + c);
    const float hz_e = xsh ? 0.f : Hz[c + dx], hy_e = xsh ? 0.f : Hy[c + dx];
    const float4 dHz_dy = hz - hz_y, dHx_dy = hx - hx_y;
    float4 dHy_dz = hy - hy_m, dHx_dz = hx - hx_m;
    const float4 dHz_dx = hz - down_x(hz, hz_e, xsh), dHy_dx = hy - down_x(hy, hy_e, xsh);
    hx_m = hx;
    hy_m = hy;
    if (g.pml > 0 && (k < g.pml || k >= g.nz - g.pml)) {
      const float4 co = g.cpml[k];
      const long long q = pml_index(g, t.s, k, t.j, t.i);
      const float4 px = comb4(co.x, ld4(g.psiE[0] + q), co.y, dHy_dz);
      const float4 py = comb4(co.x, ld4(g.psiE[1] + q), co.y, dHx_dz);
      if (t.in) {
        st4(g.psiE[0] + q, px);
        st4(g.psiE[1] + q, py);
      }
      dHy_dz = dHy_dz + px;
      dHx_dz = dHx_dz + py;
    }
    float4 cx = dHz_dy - dHy_dz;
    const float4 cy = dHx_dz - dHz_dx, cz = dHy_dx - dHx_dy;
    if (k == g.ks) {
      const float a = g.auxH[(long long)t.s * g.aux_len + 1];
      cx = cx + make_float4(a, a, a, a);
    }
    if (!t.in) continue;
    float ev[3][4] = {{e0.x, e0.y, e0.z, e0.w}, {e1.x, e1.y, e1.z, e1.w}, {e2.x, e2.y, e2.z, e2.w}};
    const float cv[3][4] = {{cx.x, cx.y, cx.z, cx.w}, {cy.x, cy.y, cy.z, cy.w}, {cz.x, cz.y, cz.z, cz.w}};
    float jv[3][4] = {};
    if (k >= g.jk0 && k < g.jk1) {  // the slab that holds metal cells
      bool any = false;
#pragma unroll
      for (int a = 0; a < 4; ++a) any = any || g.mc[(mats >> (8 * a)) & 255u].metal;
      if (any) {
        const long long jj = (((long long)t.s * (g.jk1 - g.jk0) + (k - g.jk0)) * g.ny + t.j) * g.nx + t.i;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const float4 j0 = ld4(g.J[d] + jj);
          float jo[4] = {j0.x, j0.y, j0.z, j0.w};
#pragma unroll
          for (int a = 0; a < 4; ++a) {
            const MaterialCoef& mc = g.mc[(mats >> (8 * a)) & 255u];
            if (mc.metal) jv[d][a] = jo[a] = mc.alpha * jo[a] + mc.beta * ev[d][a];
          }
          st4(g.J[d] + jj, make_float4(jo[0], jo[1], jo[2], jo[3]));
        }
      }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const MaterialCoef& mc = g.mc[(mats >> (8 * a)) & 255u];
#pragma unroll
      for (int d = 0; d < 3; ++d) ev[d][a] += mc.ce * cv[d][a] - mc.cj * jv[d][a];
    }
    if (k >= g.mk0 && k < g.mk1) {  // the molecular slab
      const long long sl = (((long long)t.s * (g.mk1 - g.mk0) + (k - g.mk0)) * g.ny + t.j) * g.nx + t.i;
      const int4 o4 = *reinterpret_cast<const int4*>(g.cell_off + sl);
      const int off[5] = {o4.x, o4.y, o4.z, o4.w, g.cell_off[sl + 4]};
      if (off[4] > off[0]) {
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          if (off[a + 1] == off[a]) continue;
          double px = 0.0, py = 0.0, pz = 0.0;  // ensemble sum in FP64
          for (int q = off[a]; q < off[a + 1]; ++q) {
            const int m = g.cell_mol[q];
            px += g.dmu[3 * (long long)m + 0];
            py += g.dmu[3 * (long long)m + 1];
            pz += g.dmu[3 * (long long)m + 2];
          }
          const float cp = g.mc[(mats >> (8 * a)) & 255u].cp;
          ev[0][a] -= cp * (float)px;
          ev[1][a] -= cp * (float)py;
          ev[2][a] -= cp * (float)pz;
        }
      }
    }
    if (!g.periodic_z && k == 0) {  // tangential E on the bottom conductor
#pragma unroll
      for (int a = 0; a < 4; ++a) ev[0][a] = ev[1][a] = 0.f;
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) st4(E[d] + c, make_float4(ev[d][0], ev[d][1], ev[d][2], ev[d][3]));
  }
}

// to = from + add: the step counter of a step without an E half step (add = 1),
// or its value in the other slot (add = 0)
__global__ void step_counter_kernel(const long long* from, long long* to, int add) { *to = *from + add; }

// The quad kernels take rows of whole quads and arrays on 16-byte boundaries
// (mat: 4, cell_off: 16); an allocator of the caller may place them anywhere.
static bool quads_ok(const Grid& g) {
  if (g.nx % 4 != 0) return false;
  uintptr_t a = 0;
  for (int c = 0; c < 3; ++c) a |= (uintptr_t)g.E[c] | (uintptr_t)g.H[c] | (uintptr_t)g.J[c];
  if (g.pml > 0)
    for (int c = 0; c < 2; ++c) a |= (uintptr_t)g.psiE[c] | (uintptr_t)g.psiH[c];
  a |= (uintptr_t)g.cell_off | ((uintptr_t)g.mat & 3) << 2;
  return (a & 15) == 0;
}
// Planes a thread: eight where that leaves every SM enough warps (about 64), fewer
// on small grids, whose half steps are as long as one thread's walk.
static int quad_planes(const Grid& g) {
  const long long quads = g.ncell_sim / 4 * g.nsim;
  const long long kz = quads / (152LL * 64 * 32);
  return (int)(kz < 1 ? 1 : (kz > 8 ? 8 : kz));
}
static int quad_tiles(const Grid& g, int kz) {
  return ((g.nx / 4 * g.ny + kQt - 1) / kQt) * ((g.nz + kz - 1) / kz) * g.nsim;
}

void launch_yee_h(const Grid& g, cudaStream_t s) {
  const int aux = g.ks >= 0 ? g.nsim * kAuxBlocks : 0;
  if (quads_ok(g)) {
    const int kz = quad_planes(g), nt = quad_tiles(g, kz);
    yee_h4_kernel<<<nt + aux, kQt, 0, s>>>(g, nt, kz);
    return;
  }
  const int nt = yee_tiles(g);
  yee_h_kernel<<<nt + aux, dim3(kTx, kTy), 0, s>>>(g, nt);
}
void launch_yee_e(const Grid& g, cudaStream_t s) {
  const int aux = g.ks >= 0 ? g.nsim * kAuxBlocks : 0;
  if (quads_ok(g)) {
    const int kz = quad_planes(g), nt = quad_tiles(g, kz);
    yee_e4_kernel<<<nt + aux, kQt, 0, s>>>(g, nt, kz);
    return;
  }
  const int nt = yee_tiles(g);
  yee_e_kernel<<<nt + aux, dim3(kTx, kTy), 0, s>>>(g, nt);
}
// E^n at the cells of listed molecules (the coupled step's gather)
__global__ void record_fields_kernel(Grid g, const int* cell, const long long* ids, int m, float* out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= m) return;
  const long long c = cell[ids[k]];
  out[3 * k] = g.E[0][c];
  out[3 * k + 1] = g.E[1][c];
  out[3 * k + 2] = g.E[2][c];
}
void launch_record_fields(const Grid& g, const int* cell, const long long* ids, int m, float* out,
                          cudaStream_t s) {
  record_fields_kernel<<<(m + 127) / 128, 128, 0, s>>>(g, cell, ids, m, out);
}
// Spectral detection: after the E update of step n (E^{n+1}, H^{n+1/2}),
// every cell of every detector plane adds dt F e^{i omega t} for each
// frequency: Ex, Ey of the plane at t_{n+1}; Hx, Hy averaged over the planes
// z = k - 1/2 and k + 1/2 (indices k - 1 and k) at t_{n+1/2}, into FP64
// accumulators.  Reading and writing those every step took 48 us a step (two
// planes of 128 x 128 cells, 48 frequencies: 201 MB); the FP64 products alone
// need 22 us (two a clock and SM).  So a step only keeps its samples, and one
// launch adds up to kDftBatch kept steps, in their order: every accumulator is
// read and written once a batch and takes the same sums as step by step.  Where a
// call has kDftDirect steps or fewer left, each is added straight from the
// fields: calls of 1, 2 and 3 steps of that workload, half steps included, take
// 90, 180 and 270 us so and 153, 226 and 287 with kept samples (a step more: 90 and
// 63).
constexpr int kDftF = 8;  // frequencies a block

// One step: a block covers 256 cells of one plane and kDftF frequencies.
__global__ void dft_kernel(Grid g, int nfc) {
  __shared__ double2 ph[2][kDftF];  // dt e^{i omega t} at the E and at the H times
  const long long n = *g.step;
  const int d = blockIdx.y / nfc, f0 = (blockIdx.y % nfc) * kDftF, sim = blockIdx.z;
  const int nf = min(kDftF, g.nfreq - f0);
  if (threadIdx.x < 2 * nf) {
    const int f = threadIdx.x % nf, h = threadIdx.x / nf;
    double sn, cs;
    sincos(g.omega[f0 + f] * (h ? (double)n + 0.5 : (double)(n + 1)) * g.dt, &sn, &cs);
    ph[h][f] = make_double2(cs * g.dt, sn * g.dt);
  }
  __syncthreads();
  const long long plane = (long long)g.ny * g.nx;
  const long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (q >= plane) return;
  const long long ck = sim * g.ncell_sim + (long long)g.det_k[d] * plane + q, cm = ck - plane;
  const double v[4] = {g.E[0][ck], g.E[1][ck], 0.5 * ((double)g.H[0][cm] + (double)g.H[0][ck]),
                       0.5 * ((double)g.H[1][cm] + (double)g.H[1][ck])};
  double2* acc = g.dft + (((long long)sim * g.ndet + d) * g.nfreq + f0) * 4 * plane + q;
  for (int f = 0; f < nf; ++f) {  // four independent sums at a time
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const double2 w = ph[c < 2 ? 0 : 1][f];
      double2* a = acc + ((long long)f * 4 + c) * plane;
      double2 x = *a;
      x.x = fma(v[c], w.x, x.x);
      x.y = fma(v[c], w.y, x.y);
      *a = x;
    }
  }
}

__global__ void dft_keep_kernel(Grid g) {
  const long long plane = (long long)g.ny * g.nx, q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (q >= plane) return;
  const long long ck = blockIdx.z * g.ncell_sim + (long long)g.det_k[blockIdx.y] * plane + q, cm = ck - plane;
  const int slot = (int)(*g.step & (kDftBatch - 1));
  float* o = g.dft_ring + (((long long)slot * g.nsim + blockIdx.z) * g.ndet + blockIdx.y) * 6 * plane + q;
  o[0] = g.E[0][ck];
  o[plane] = g.E[1][ck];
  o[2 * plane] = g.H[0][cm];
  o[3 * plane] = g.H[0][ck];
  o[4 * plane] = g.H[1][cm];
  o[5 * plane] = g.H[1][ck];
}

// A block: 256 cells of one plane, kDftF frequencies, every component, the `count` steps before step *done.
__global__ void __launch_bounds__(256) dft_add_kernel(Grid g, int nfc, int count, const long long* done) {
  __shared__ double2 ph[2][kDftF][kDftBatch];  // dt e^{i omega t} at the E and at the H times
  const long long n0 = *done - count;
  const int d = blockIdx.y / nfc, f0 = (blockIdx.y % nfc) * kDftF, sim = blockIdx.z;
  const int nf = min(kDftF, g.nfreq - f0);
  for (int q = threadIdx.x; q < 2 * nf * count; q += blockDim.x) {
    const int b = q % count, f = (q / count) % nf, h = q / (count * nf);
    const long long n = n0 + b;
    double sn, cs;
    sincos(g.omega[f0 + f] * (h ? (double)n + 0.5 : (double)(n + 1)) * g.dt, &sn, &cs);
    ph[h][f][b] = make_double2(cs * g.dt, sn * g.dt);
  }
  __syncthreads();
  const long long plane = (long long)g.ny * g.nx;
  const long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (q >= plane) return;
  const float* ring = g.dft_ring + ((long long)sim * g.ndet + d) * 6 * plane + q;
  const long long slot = (long long)g.nsim * g.ndet * 6 * plane;
  double2* acc = g.dft + (((long long)sim * g.ndet + d) * g.nfreq + f0) * 4 * plane + q;
#pragma unroll 1
  for (int c = 0; c < 4; ++c) {
    double v[kDftBatch];
#pragma unroll
    for (int b = 0; b < kDftBatch; ++b) {
      v[b] = 0.0;
      if (b < count) {
        const float* r = ring + ((n0 + b) & (kDftBatch - 1)) * slot;
        v[b] = c < 2 ? (double)r[c * plane] : 0.5 * ((double)r[(2 * c - 2) * plane] + (double)r[(2 * c - 1) * plane]);
      }
    }
#pragma unroll 1
    for (int f = 0; f < nf; f += 2) {  // two frequencies at a time: four independent chains
      const bool two = f + 1 < nf;
      const double2 *w0 = ph[c < 2 ? 0 : 1][f], *w1 = ph[c < 2 ? 0 : 1][two ? f + 1 : f];
      double2 *a0 = acc + ((long long)f * 4 + c) * plane, *a1 = a0 + (two ? 4 * plane : 0);
      double2 x = *a0, y = *a1;
#pragma unroll
      for (int b = 0; b < kDftBatch; ++b) {
        if (b >= count) break;
        x.x = fma(v[b], w0[b].x, x.x);
        x.y = fma(v[b], w0[b].y, x.y);
        if (two) {
          y.x = fma(v[b], w1[b].x, y.x);
          y.y = fma(v[b], w1[b].y, y.y);
        }
      }
      *a0 = x;
      if (two) *a1 = y;
    }
  }
}

// Poynting flux through detector plane `plane`, one block per (frequency, sim): the cells' Re (Ex conj(Hy) - Ey
// conj(Hx)) in FP64, summed over a thread's cells, then over the block.  Bound by the accumulators' 64 B a cell.
// Copying the accumulators to the host and summing them there took 2.6 ms a plane for 48 frequencies of 128 x 128.
__global__ void __launch_bounds__(512) flux_kernel(Grid g, int plane, double dx2, double* out) {
  __shared__ double part[16];
  const long long cells = (long long)g.ny * g.nx;
  const int f = blockIdx.x, sim = blockIdx.y, t = threadIdx.x;
  const double2* a = g.dft + (((long long)sim * g.ndet + plane) * g.nfreq + f) * 4 * cells;
  double acc = 0.0;
  for (long long q = t; q < cells; q += blockDim.x) {
    const double2 ex = a[q], ey = a[cells + q], hx = a[2 * cells + q], hy = a[3 * cells + q];
    acc += (ex.x * hy.x + ex.y * hy.y) - (ey.x * hx.x + ey.y * hx.y);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((t & 31) == 0) part[t >> 5] = acc;
  __syncthreads();
  if (t == 0) {
    double v = 0.0;
    for (int w = 0; w < 16; ++w) v += part[w];
    out[(long long)sim * g.nfreq + f] = v * dx2;
  }
}

void launch_flux(const Grid& g, int plane, double dx2, double* out, cudaStream_t s) {
  flux_kernel<<<dim3((unsigned)g.nfreq, (unsigned)g.nsim), 512, 0, s>>>(g, plane, dx2, out);
}
static dim3 dft_grid(const Grid& g, int nfc) {
  const long long plane = (long long)g.ny * g.nx;
  return dim3((unsigned)((plane + 255) / 256), (unsigned)(g.ndet * nfc), (unsigned)g.nsim);
}
void launch_dft(const Grid& g, cudaStream_t s) {
  const int nfc = (g.nfreq + kDftF - 1) / kDftF;
  dft_kernel<<<dft_grid(g, nfc), 256, 0, s>>>(g, nfc);
}
void launch_dft_keep(const Grid& g, cudaStream_t s) { dft_keep_kernel<<<dft_grid(g, 1), 256, 0, s>>>(g); }
void launch_dft_add(const Grid& g, int count, const long long* done, cudaStream_t s) {
  const int nfc = (g.nfreq + kDftF - 1) / kDftF;
  dft_add_kernel<<<dft_grid(g, nfc), 256, 0, s>>>(g, nfc, count, done);
}
void launch_step_counter(const long long* from, long long* to, int add, cudaStream_t s) {
  step_counter_kernel<<<1, 1, 0, s>>>(from, to, add);
}

}  // namespace ms
