// lbm_tile.cuh -- one or two steps of one tile of an FP32 domain: 64 columns x R
// rows, worked on by a CTA of R + 3 warps; shared by the small-domain kernels
// (lbm_tile.cu) and the batched one (lbm_batch.cu).
#pragma once

#include "lbm_node.cuh"

namespace lbm_tile {

using lbm_node::add2;
using lbm_node::collide_node2;
using lbm_node::eos_node;
using lbm_node::eos_node2;
using lbm_node::sqrt0;

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

// A density outside (0, rho_max], tested on the bits: positive floats order like
// their bit patterns, and -0, negatives, +inf and NaN land above rho_max's.
template <class PT>
__device__ __forceinline__ bool outside(const PT &P, float r) {
  return __float_as_uint(r) - 1u >= __float_as_uint(P.rho_max);
}

// Ghost entries (Eqs. 19-21) of columns ca (if on0) and cb (if on1) in window row
// w, row v of the domain: v == 0 from window rows w + 1, w + 2, v == ny - 1 from
// the two below.  k: the wall coefficient of each column.  lbm_node.cuh's
// ghost_rule for both columns in one chain: one after the other they were the
// longest part of a small domain's step (256 x 128: 1.2 of 2.8 us).
template <int KIND, int R, class PT>
__device__ __forceinline__ void ghost_at(const PT &P, Smem<R> &M, int w, int v, int ca, int cb, bool on0, bool on1,
                                         float2 k) {
  const float *r1 = M.rho[v != 0 ? w - 1 : w + 1], *r2 = M.rho[v != 0 ? w - 2 : w + 2];
  const int c[2] = {ca, on1 ? cb : ca};
  const float kk[2] = {k.x, k.y};
  float g[2], aa[2], d[2], ri2[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    aa[j] = r1[c[j] + 3] - r1[c[j] + 1];
    ri2[j] = r2[c[j] + 2];
    d[j] = 2.0f * (ri2[j] - r1[c[j] + 2]);
    g[j] = ri2[j];
  }
  if (P.n_iter <= 0) {
#pragma unroll
    for (int j = 0; j < 2; ++j) g[j] = fmaf(kk[j], fabsf(aa[j]), ri2[j]);
  } else {
    for (int i = 0; i < P.n_iter; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        g[j] = fmaf(kk[j], sqrt0(P, fmaf(aa[j], aa[j], d[j] * d[j])), ri2[j]);
        d[j] = ri2[j] - g[j];
      }
  }
#pragma unroll
  for (int j = 0; j < 2; ++j) g[j] = fminf(fmaxf(g[j], 0.0f), P.ghost_max);
  float2 ps, ps2;
  eos_node2<KIND>(P, make_float2(g[0], g[1]), ps, ps2);
  // psi = U = 0 at rho_max
  if (on0) put(M.psi[w], M.sq[w], ca, g[0] < P.rho_max ? ps.x : 0.0f, g[0] < P.rho_max ? ps2.x : 0.0f);
  if (on1) put(M.psi[w], M.sq[w], cb, g[1] < P.rho_max ? ps.y : 0.0f, g[1] < P.rho_max ? ps2.y : 0.0f);
}

// A thread's place in a tile of `wr` <= kW columns from x0 and `nr` <= R rows
// from y0 (both may lie outside a periodic direction).  Warps 0 .. R + 1 each
// have one window row, w (row y0 - 1 + w), lane t columns t and t + kH of it; the
// last warp has the columns beside the tile (hc).
// WRAP: the tile itself may cross the periodic columns' seam.
template <int MCW, int R, bool WRAP, class PT>
struct Place {
  int nx, ny, walls;  // of the domain (copies: P may lie in shared memory)
  int warp, lane, w, hc, v, y, wr, nr;
  int xa, xb;        // the columns in the domain (a thread of the last warp: xa)
  bool on, solid, act0, act1, geo, low, high;
  __device__ __forceinline__ Place(const PT &P, int x0, int y0, int wr_, int nr_)
      : nx(P.nx), ny(P.ny), walls(P.walls), wr(wr_), nr(nr_) {
    static_assert(2 * (R + 2) + 4 <= 32, "one warp loads the columns beside the tile");
    warp = threadIdx.x >> 5;
    lane = threadIdx.x & 31;
    geo = (MCW < 0 ? P.wetting == LBM_WET_GEOMETRIC : MCW == 0) && walls;
    low = geo && y0 == 1;  // the tile touches a wall with a ghost row
    high = geo && y0 + nr == ny - 1;
    w = warp;
    hc = 0;
    on = true;
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
    v = y0 - 1 + w;
    solid = walls && (v == 0 || v == ny - 1);
    y = v < 0 ? v + ny : (v >= ny ? v - ny : v);
    act0 = lane < wr;
    act1 = lane + kH < wr;  // implies act0
    auto wrap = [&](int x) { return x < 0 ? x + nx : (x >= nx ? x - nx : x); };
    if (WRAP) {
      xa = wrap(x0 + (warp < R + 2 ? lane : hc));
      xb = wrap(x0 + lane + kH);
    } else {
      xa = warp < R + 2 ? x0 + lane : wrap(x0 + hc);
      xb = x0 + lane + kH;
    }
  }
};

// Fills the window from the state fin: psi and psi^2 of every node of the tile
// and around it, ghost rows included; f and r are the populations and densities
// of the thread's nodes.  ready() returns once the state may be read.  Ends with
// a barrier.  True if the thread saw a density outside (0, rho_max].
template <int KIND, int R, bool WRAP, class PT, class PL, class Ready>
__device__ __forceinline__ bool enter(const PT &P, const PL &q, const float *__restrict__ fin, Smem<R> &M,
                                      float2 (&f)[9], float2 &r, Ready ready) {
  const size_t n = (size_t)q.nx * q.ny;
  const int w = q.w, c0 = q.lane, c1 = q.lane + kH;
  bool bad = false;
  // the wall coefficients of a ghost row, loaded before the densities it waits for
  float2 k = make_float2(0.0f, 0.0f);
  const bool g0 = q.on && q.solid && q.geo && (q.warp == R + 2 || q.act0), g1 = g0 && q.warp < R + 2 && q.act1;
  const double *coef = P.coef + (P.n_iter > 0 ? 0 : 2 * q.nx) + (q.v != 0 ? q.nx : 0);
  if (g0) k.x = (float)coef[q.xa];
  if (g1) k.y = (float)coef[q.xb];
  ready();
  r = make_float2(0.0f, 0.0f);
  if (q.on && q.warp < R + 2) {
    if (!q.solid) {
      if (q.act0) {
        const float *p0 = fin + (size_t)q.y * q.nx + q.xa, *p1 = q.act1 ? p0 + (WRAP ? q.xb - q.xa : kH) : p0;
#pragma unroll
        for (int a = 0; a < 9; ++a) f[a] = make_float2(p0[a * n], p1[a * n]);
        r = add2(add2(add2(add2(f[0], f[1]), add2(f[2], f[3])), add2(add2(f[4], f[5]), add2(f[6], f[7]))), f[8]);
        float2 ps, ps2;
        eos_node2<KIND>(P, r, ps, ps2);
        bad = outside(P, r.x) | outside(P, r.y);
        put(M.psi[w], M.sq[w], c0, ps.x, ps2.x);
        M.rho[w][c0 + 2] = r.x;
        if (q.act1) {
          put(M.psi[w], M.sq[w], c1, ps.y, ps2.y);
          M.rho[w][c1 + 2] = r.y;
        }
      }
    } else if (!q.geo) {  // Martys-Chen: psi = U = 0 on the solid rows
      put(M.psi[w], M.sq[w], c0, 0.0f, 0.0f);
      put(M.psi[w], M.sq[w], c1, 0.0f, 0.0f);
    }
  } else if (q.on) {
    if (!q.solid) {
      const float *p = fin + (size_t)q.y * q.nx + q.xa;
      float g[9];
#pragma unroll
      for (int a = 0; a < 9; ++a) g[a] = p[a * n];
      const float4 e = eos_node<KIND>(P, sum9(g));
      M.rho[w][q.hc + 2] = e.x;
      put(M.psi[w], M.sq[w], q.hc, e.y, e.z);
    } else if (!q.geo) {
      put(M.psi[w], M.sq[w], q.hc, 0.0f, 0.0f);
    }
  }
  __syncthreads();
  if (q.low || q.high) {  // uniform in the CTA
    if (g0) ghost_at<KIND>(P, M, w, q.v, q.warp < R + 2 ? c0 : q.hc, c1, true, g1, k);
    __syncthreads();
  }
  return bad;
}

// Post-collision populations fs of the thread's nodes (window row w, row y).
template <bool UNIT, int MCW, int R, class PT>
__device__ __forceinline__ void collide_at(const PT &P, const Smem<R> &M, int w, int lane, int y, const float2 (&f)[9],
                                           float2 r, float2 (&fs)[9]) {
  const float2 *pm = M.psi[w - 1], *p0 = M.psi[w], *pp = M.psi[w + 1];
  const float2 *qm = M.sq[w - 1], *q0 = M.sq[w], *qp = M.sq[w + 1];
  const int i = lane + 2;
  const float2 pn[9] = {p0[i], p0[i + 1], pp[i], p0[i - 1], pm[i], pp[i + 1], pp[i - 1], pm[i - 1], pm[i + 1]};
  const float2 qn[9] = {q0[i], q0[i + 1], qp[i], q0[i - 1], qm[i], qp[i + 1], qp[i - 1], qm[i - 1], qm[i + 1]};
  collide_node2<UNIT, MCW>(P, f, pn, qn, r, y, fs);
}

// Streaming with half-way bounce-back of the thread's nodes (the first if on0, the
// second if on1).
template <class PL>
__device__ __forceinline__ void push(const PL &q, float *__restrict__ fout, bool on0, bool on1, const float2 (&fs)[9]) {
  const int y = q.y;
  const bool wall_dn = q.walls && y == 1, wall_up = q.walls && y == q.ny - 2;
  const unsigned nx = q.nx, un = (unsigned)q.nx * (unsigned)q.ny;
  const unsigned ry = (unsigned)y * nx, rym = (unsigned)(y == 0 ? q.ny - 1 : y - 1) * nx,
                 ryp = (unsigned)(y == q.ny - 1 ? 0 : y + 1) * nx;
  float *const o0 = fout, *const o1 = o0 + un, *const o2 = o1 + un, *const o3 = o2 + un, *const o4 = o3 + un;
  float *const o5 = o4 + un, *const o6 = o5 + un, *const o7 = o6 + un, *const o8 = o7 + un;
  auto node = [&](unsigned x, float f0, float f1, float f2, float f3, float f4, float f5, float f6, float f7,
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
  if (on0) node(q.xa, fs[0].x, fs[1].x, fs[2].x, fs[3].x, fs[4].x, fs[5].x, fs[6].x, fs[7].x, fs[8].x);
  if (on1) node(q.xb, fs[0].y, fs[1].y, fs[2].y, fs[3].y, fs[4].y, fs[5].y, fs[6].y, fs[7].y, fs[8].y);
}

// One step of the tile whose first column and row are x0 and y0, from fin to
// fout.  unstable() reports a density outside (0, rho_max].  MCW, KIND: wetting
// rule and EOS when fixed at compile time, else -1 (read from P).
template <bool UNIT, int MCW, int KIND, int R, class PT, class Ready, class Unstable>
__device__ __forceinline__ void step(const PT &P, int x0, int y0, const float *__restrict__ fin,
                                     float *__restrict__ fout, Smem<R> &M, Ready ready, Unstable unstable) {
  const Place<MCW, R, false, PT> q(P, x0, y0, min(kW, P.nx - x0), min(R, (P.walls ? P.ny - 1 : P.ny) - y0));
  float2 f[9], r, fs[9];
  const bool bad = enter<KIND, R, false>(P, q, fin, M, f, r, ready);
  if (__any_sync(0xffffffffu, bad) && q.lane == 0) unstable();
  if (q.warp < 1 || q.warp > q.nr || !q.act0) return;
  collide_at<UNIT, MCW, R>(P, M, q.w, q.lane, q.y, f, r, fs);
  push(q, fout, true, q.act1, fs);
}

// ---- two steps -----------------------------------------------------------------
// The tile of kPairW columns x R - 4 rows at (xo, yo), two steps ahead.  The first
// step is made on a tile 3 columns and 2 rows larger on every side (a row that a
// wall bounds needs no more), its streamed populations stay in shared memory (F),
// and the second one reads them there.  (3 columns: the ghost row beside a column
// reads the densities beside that, which need the collisions beside those.)

constexpr int kPairW = kW - 6;

template <int R>
struct PairSmem {
  Smem<R> win;
  float F[9][R][kW];
};

template <bool UNIT, int MCW, int KIND, int R, class PT, class Ready, class Unstable>
__device__ __forceinline__ void step_pair(const PT &P, int xo, int yo, const float *__restrict__ fin,
                                          float *__restrict__ fout, PairSmem<R> &S, Ready ready, Unstable unstable) {
  const int wo = min(kPairW, P.nx - xo), end = P.walls ? P.ny - 1 : P.ny;  // columns; end of the fluid rows
  const int ye = min(yo + R - 4, end);                                     // rows [yo, ye)
  const int y0 = P.walls ? max(yo - 2, 1) : yo - 2, y1 = P.walls ? min(ye + 2, end) : ye + 2;
  const Place<MCW, R, true, PT> q(P, xo - 3, y0, wo + 6, y1 - y0);
  Smem<R> &M = S.win;
  float2 f[9], r, fs[9];
  bool bad = enter<KIND, R, true>(P, q, fin, M, f, r, ready);
  const bool row = q.warp >= 1 && q.warp <= q.nr && q.act0;  // a thread with nodes of the larger tile
  const int i = q.w - 1, c0 = q.lane, c1 = q.lane + kH;      // its row and columns there
  if (row) {
    collide_at<UNIT, MCW, R>(P, M, q.w, q.lane, q.y, f, r, fs);
    const bool dn = P.walls && q.y == 1, up = P.walls && q.y == P.ny - 2;
    const bool below = i > 0, above = i + 1 < q.nr;
    auto put9 = [&](int c, float f0, float f1, float f2, float f3, float f4, float f5, float f6, float f7, float f8) {
      const bool left = c > 0, right = c + 1 < q.wr;
      S.F[0][i][c] = f0;
      if (right) S.F[1][i][c + 1] = f1;
      if (left) S.F[3][i][c - 1] = f3;
      if (up) {
        S.F[4][i][c] = f2;
        S.F[7][i][c] = f5;
        S.F[8][i][c] = f6;
      } else if (above) {
        S.F[2][i + 1][c] = f2;
        if (right) S.F[5][i + 1][c + 1] = f5;
        if (left) S.F[6][i + 1][c - 1] = f6;
      }
      if (dn) {
        S.F[2][i][c] = f4;
        S.F[5][i][c] = f7;
        S.F[6][i][c] = f8;
      } else if (below) {
        S.F[4][i - 1][c] = f4;
        if (left) S.F[7][i - 1][c - 1] = f7;
        if (right) S.F[8][i - 1][c + 1] = f8;
      }
    };
    put9(c0, fs[0].x, fs[1].x, fs[2].x, fs[3].x, fs[4].x, fs[5].x, fs[6].x, fs[7].x, fs[8].x);
    if (q.act1) put9(c1, fs[0].y, fs[1].y, fs[2].y, fs[3].y, fs[4].y, fs[5].y, fs[6].y, fs[7].y, fs[8].y);
  }
  __syncthreads();
  // the second step: nodes with all nine populations are the larger tile's without
  // its outermost columns, and rows unless a wall bounds them
  const int ylow = P.walls && y0 == 1 ? y0 : y0 + 1, yhigh = P.walls && y1 == end ? y1 : y1 - 1;  // rows [ylow, yhigh)
  const bool full = row && q.v >= ylow && q.v < yhigh;
  const bool out = row && q.v >= yo && q.v < ye, out0 = out && c0 >= 3 && c0 < wo + 3, out1 = out && c1 < wo + 3;
  if (full) {
#pragma unroll
    for (int a = 0; a < 9; ++a) f[a] = make_float2(S.F[a][i][c0], S.F[a][i][q.act1 ? c1 : c0]);
    r = add2(add2(add2(add2(f[0], f[1]), add2(f[2], f[3])), add2(add2(f[4], f[5]), add2(f[6], f[7]))), f[8]);
    float2 ps, ps2;
    eos_node2<KIND>(P, r, ps, ps2);
    bad |= (out0 && outside(P, r.x)) | (out1 && outside(P, r.y));
    put(M.psi[q.w], M.sq[q.w], c0, ps.x, ps2.x);
    M.rho[q.w][c0 + 2] = r.x;
    if (q.act1) {
      put(M.psi[q.w], M.sq[q.w], c1, ps.y, ps2.y);
      M.rho[q.w][c1 + 2] = r.y;
    }
  }
  const bool low = q.geo && yo == 1, high = q.geo && ye == end;
  if (low || high) {  // uniform in the CTA (the Martys-Chen rows still hold their zeros)
    float2 k = make_float2(0.0f, 0.0f);
    const bool g0 = q.solid && q.warp < R + 2 && q.on && q.act0, g1 = g0 && q.act1;
    const double *coef = P.coef + (P.n_iter > 0 ? 0 : 2 * P.nx) + (q.v != 0 ? P.nx : 0);
    if (g0) k.x = (float)coef[q.xa];
    if (g1) k.y = (float)coef[q.xb];
    __syncthreads();
    if (g0) ghost_at<KIND>(P, M, q.w, q.v, c0, c1, c0 >= 2, g1 && c1 < wo + 4, k);
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) unstable();
  if (!out) return;
  collide_at<UNIT, MCW, R>(P, M, q.w, q.lane, q.y, f, r, fs);
  push(q, fout, out0, out1, fs);
}

}  // namespace lbm_tile
