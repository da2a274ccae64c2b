// lbm_tile.cuh -- one step of one tile of an FP32 domain: 64 columns x R rows,
// worked on by a CTA of R + 3 warps; shared by the small-domain kernel
// (lbm_tile.cu) and the batched one (lbm_batch.cu).
#pragma once

#include "lbm_node.cuh"

namespace lbm_tile {

using lbm_node::add2;
using lbm_node::collide_node2;
using lbm_node::eos_node;
using lbm_node::eos_node2;
using lbm_node::ghost_rule;

constexpr int kW = 64;        // columns per tile: one warp per row, a lane owns columns t and t + 32
constexpr int kH = kW / 2;
constexpr int kWP = kH + 4;   // paired window entries i = -2 .. kH + 1 at index i + 2
constexpr int kWR = kW + 4;   // density window columns c = -2 .. kW + 1 at index c + 2

__device__ __forceinline__ float sum9(const float (&v)[9]) {
  return (((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]))) + v[8];
}

// (psi, psi^2) of column c into a window row: lane 0 of entry c and/or lane 1
// of entry c - kH
__device__ __forceinline__ void put(float2 *ps, float2 *sq, int c, float p, float q) {
  if (c <= kH + 1) {
    ps[c + 2].x = p;
    sq[c + 2].x = q;
  }
  if (c >= kH - 2) {
    ps[c - kH + 2].y = p;
    sq[c - kH + 2].y = q;
  }
}

template <int R>
struct Smem {
  float2 psi[R + 2][kWP], sq[R + 2][kWP];
  float rho[R + 2][kWR];
};

// The tile whose first column and row are x0 and y0, from fin to fout.  Warps
// 0 .. R + 1 each load one row (the tile's and the one above and below), lane t
// columns t and t + kH; the last warp loads the columns beside the tile.  Window
// row w holds row y0 - 1 + w.  ready() returns once the state may be read;
// unstable() reports a density outside (0, rho_max].  MCW, KIND: wetting rule
// and EOS when fixed at compile time, else -1 (read from P).
template <bool UNIT, int MCW, int KIND, int R, class PT, class Ready, class Unstable>
__device__ __forceinline__ void step(const PT &P, int x0, int y0, const float *__restrict__ fin,
                                     float *__restrict__ fout, Smem<R> &M, Ready ready, Unstable unstable) {
  static_assert(2 * (R + 2) + 4 <= 32, "one warp loads the columns beside the tile");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wr = min(kW, P.nx - x0);
  const int nr = min(R, (P.walls ? P.ny - 1 : P.ny) - y0);  // rows of this tile
  const size_t n = (size_t)P.nx * P.ny;
  const bool geo = (MCW < 0 ? P.wetting == LBM_WET_GEOMETRIC : MCW == 0) && P.walls;
  const bool low = geo && y0 == 1, high = geo && y0 + nr == P.ny - 1;  // the tile touches a wall with a ghost row
  bool bad = false;

  // the window row and columns of this thread
  int w = warp, hc = 0;
  bool on = true;
  if (warp == R + 2) {
    const int k = lane - 2 * (R + 2);
    w = lane >> 1;
    hc = lane & 1 ? wr : -1;
    if (k >= 0) {  // densities two columns out, which the ghost values one column out read
      w = k >> 1 ? nr : 1;
      hc = k & 1 ? wr + 1 : -2;
      on = k < 4 && (k >> 1 ? high : low);
    }
  }
  on = on && w <= nr + 1;
  const int v = y0 - 1 + w;                                       // may be -1 or ny in a periodic box
  const bool solid = P.walls && (v == 0 || v == P.ny - 1);
  const int y = v < 0 ? v + P.ny : (v >= P.ny ? v - P.ny : v);
  const int c0 = lane, c1 = lane + kH;
  const bool act0 = c0 < wr, act1 = c1 < wr;  // act1 implies act0
  int gx = x0 + hc;
  gx = gx < 0 ? gx + P.nx : (gx >= P.nx ? gx - P.nx : gx);

  // the wall coefficients of a ghost row, loaded before the densities it waits for
  double k0 = 0.0, k1 = 0.0;
  if (on && solid && geo) {
    const double *coef = P.coef + (P.n_iter > 0 ? 0 : 2 * P.nx) + (v != 0 ? P.nx : 0);
    if (warp < R + 2) {
      if (act0) k0 = coef[x0 + c0];
      if (act1) k1 = coef[x0 + c1];
    } else {
      k0 = coef[gx];
    }
  }
  ready();
  float2 f[9], r = make_float2(0.0f, 0.0f);
  if (on && warp < R + 2) {
    if (!solid) {
      if (act0) {
        const float *q0 = fin + (size_t)y * P.nx + x0 + c0, *q1 = act1 ? q0 + kH : q0;
#pragma unroll
        for (int a = 0; a < 9; ++a) f[a] = make_float2(q0[a * n], q1[a * n]);
        r = add2(add2(add2(add2(f[0], f[1]), add2(f[2], f[3])), add2(add2(f[4], f[5]), add2(f[6], f[7]))), f[8]);
        float2 ps, ps2;
        eos_node2<KIND>(P, r, ps, ps2);
        // unstable unless 0 < rho <= rho_max, tested on the bits
        const unsigned mx = __float_as_uint(P.rho_max);
        bad = (__float_as_uint(r.x) - 1u >= mx) | (__float_as_uint(r.y) - 1u >= mx);
        put(M.psi[w], M.sq[w], c0, ps.x, ps2.x);
        M.rho[w][c0 + 2] = r.x;
        if (act1) {
          put(M.psi[w], M.sq[w], c1, ps.y, ps2.y);
          M.rho[w][c1 + 2] = r.y;
        }
      }
    } else if (!geo) {  // Martys-Chen: psi = U = 0 on the solid rows
      put(M.psi[w], M.sq[w], c0, 0.0f, 0.0f);
      put(M.psi[w], M.sq[w], c1, 0.0f, 0.0f);
    }
  } else if (on) {
    if (!solid) {
      const float *q = fin + (size_t)y * P.nx + gx;
      float g[9];
#pragma unroll
      for (int a = 0; a < 9; ++a) g[a] = q[a * n];
      const float4 e = eos_node<KIND>(P, sum9(g));
      M.rho[w][hc + 2] = e.x;
      put(M.psi[w], M.sq[w], hc, e.y, e.z);
    } else if (!geo) {
      put(M.psi[w], M.sq[w], hc, 0.0f, 0.0f);
    }
  }
  __syncthreads();
  if (low || high) {  // uniform in the CTA
    if (on && solid) {
      // Eqs. 19-21 ghost row: v == 0 from window rows 1, 2; v == ny - 1 from the two rows below it
      const float *r1 = M.rho[v != 0 ? w - 1 : 1], *r2 = M.rho[v != 0 ? w - 2 : 2];
      auto ghost = [&](int c, double k) {
        const float4 e = ghost_rule<KIND>(P, r1[c + 1], r1[c + 2], r1[c + 3], r2[c + 2], (float)k, (float)k);
        put(M.psi[w], M.sq[w], c, e.y, e.z);
      };
      if (warp < R + 2) {
        if (act0) ghost(c0, k0);
        if (act1) ghost(c1, k1);
      } else {
        ghost(hc, k0);
      }
    }
    __syncthreads();
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) unstable();
  if (warp < 1 || warp > nr || !act0) return;

  // collide row y (its populations are in this warp's registers)
  const float2 *pm = M.psi[w - 1], *p0 = M.psi[w], *pp = M.psi[w + 1];
  const float2 *qm = M.sq[w - 1], *q0 = M.sq[w], *qp = M.sq[w + 1];
  const int i = lane + 2;
  const float2 pn[9] = {p0[i], p0[i + 1], pp[i], p0[i - 1], pm[i], pp[i + 1], pp[i - 1], pm[i - 1], pm[i + 1]};
  const float2 qn[9] = {q0[i], q0[i + 1], qp[i], q0[i - 1], qm[i], qp[i + 1], qp[i - 1], qm[i - 1], qm[i + 1]};
  float2 fs[9];
  collide_node2<UNIT, MCW>(P, f, pn, qn, r, y, fs);
  const bool wall_dn = P.walls && y == 1, wall_up = P.walls && y == P.ny - 2;
  const unsigned nx = P.nx, un = (unsigned)n;
  const unsigned ry = (unsigned)y * nx, rym = (unsigned)(y == 0 ? P.ny - 1 : y - 1) * nx,
                 ryp = (unsigned)(y == P.ny - 1 ? 0 : y + 1) * nx;
  float *const o0 = fout, *const o1 = o0 + un, *const o2 = o1 + un, *const o3 = o2 + un, *const o4 = o3 + un;
  float *const o5 = o4 + un, *const o6 = o5 + un, *const o7 = o6 + un, *const o8 = o7 + un;
  // streaming with half-way bounce-back of node x's post-collision populations
  auto push = [&](unsigned x, float f0, float f1, float f2, float f3, float f4, float f5, float f6, float f7,
                  float f8) {
    const unsigned xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
    o0[ry + x] = f0;
    o1[ry + xp] = f1;
    o3[ry + xm] = f3;
    if (wall_up) {
      o4[ry + x] = f2;
      o7[ry + x] = f5;
      o8[ry + x] = f6;
    } else {
      o2[ryp + x] = f2;
      o5[ryp + xp] = f5;
      o6[ryp + xm] = f6;
    }
    if (wall_dn) {
      o2[ry + x] = f4;
      o5[ry + x] = f7;
      o6[ry + x] = f8;
    } else {
      o4[rym + x] = f4;
      o7[rym + xm] = f7;
      o8[rym + xp] = f8;
    }
  };
  push(x0 + c0, fs[0].x, fs[1].x, fs[2].x, fs[3].x, fs[4].x, fs[5].x, fs[6].x, fs[7].x, fs[8].x);
  if (act1) push(x0 + c1, fs[0].y, fs[1].y, fs[2].y, fs[3].y, fs[4].y, fs[5].y, fs[6].y, fs[7].y, fs[8].y);
}

}  // namespace lbm_tile
