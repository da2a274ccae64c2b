// lbm_measure.cu -- density field, reductions and the apparent contact-angle
// measurement (the paper reports "measured" angles in Secs. 4.2.1-4.2.2
// without a procedure; the one implemented here is documented in lbm.h).
// Compiled with -fmad=false: with an FP64 state the column sums, crossings
// and heights are bit-identical to a sequential FP64 evaluation.
#include <float.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "lbm_internal.h"

namespace {

// The left-to-right double sum (((0 + f_0) + f_1) + ...) + f_8 of nine
// floats, bit for bit, mostly without FP64 instructions (GB300 issues FP64 at
// a small fraction of its FP32 rate).  When the nonzero terms span at most 26
// binades (exponents emin..emin+25), each term is an integer multiple of
// u = 2^(emin - 150) below 2^49 u, so every partial sum is a multiple of u
// below 9 * 2^49 u < 2^53 u: exactly representable in double.  The double
// additions are then exact, and the sum is the integer total S times u,
// assembled directly as a double (exact cancellation gives +0, as the double
// additions starting from +0 do).  Wider spans and subnormal, infinite or NaN
// terms take the double additions.
__device__ __forceinline__ double sum9(const float (&v)[9]) {
  int emin = 255, emax = 0;
  bool plain = true;
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    const unsigned u = __float_as_uint(v[a]);
    const int e = (int)((u >> 23) & 255u);
    plain &= e != 255 && (e != 0 || (u & 0x7fffffu) == 0u);
    if (e != 0) {
      emin = min(emin, e);
      emax = max(emax, e);
    }
  }
  if (plain && emax - emin <= 25) {
    long long S = 0;
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      const unsigned u = __float_as_uint(v[a]);
      const int e = (int)((u >> 23) & 255u);
      if (e != 0) {
        const long long m = (long long)((u & 0x7fffffu) | 0x800000u) << (e - emin);
        S += (u >> 31) ? -m : m;
      }
    }
    if (S == 0) return 0.0;
    const unsigned long long A = S < 0 ? (unsigned long long)(-S) : (unsigned long long)S;
    const int p = 63 - __clzll((long long)A);  // p <= 52
    const unsigned long long bits = ((unsigned long long)(S < 0) << 63) |
                                    ((unsigned long long)(p + emin - 150 + 1023) << 52) |
                                    ((A << (52 - p)) & 0xfffffffffffffull);
    return __longlong_as_double((long long)bits);
  }
  double r = 0.0;
#pragma unroll
  for (int a = 0; a < 9; ++a) r = r + (double)v[a];
  return r;
}

// rho = sum_a f_a accumulated in double, left to right, at fluid nodes; 0 on
// the solid rows; nodes [i0, i1) of the field.
template <typename R>
__global__ void k_rho64(int nx, int ny, int walls, const R *__restrict__ f, double *__restrict__ rho, size_t i0,
                        size_t i1) {
  size_t n = (size_t)nx * ny;
  size_t i = i0 + (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= i1) return;
  int y = (int)(i / nx);
  if (walls && (y == 0 || y == ny - 1)) {
    rho[i] = 0.0;
    return;
  }
  if (sizeof(R) == sizeof(float)) {
    float v[9];
#pragma unroll
    for (int a = 0; a < 9; ++a) v[a] = (float)f[a * n + i];
    rho[i] = sum9(v);
    return;
  }
  double r = 0.0;
#pragma unroll
  for (int a = 0; a < 9; ++a) r = r + (double)f[a * n + i];
  rho[i] = r;
}

// The same for FP32 states with nx % 4 == 0: four consecutive nodes of one
// row per thread (16-byte loads of each plane, 2 x 16-byte stores); groups of
// four [q0, q1).
__global__ void k_rho64_x4(int nx, int ny, int walls, const float4 *__restrict__ f, double2 *__restrict__ rho,
                           size_t q0, size_t q1) {
  const size_t n4 = (size_t)nx * ny / 4;
  const size_t i = q0 + (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= q1) return;
  const int y = (int)((4 * i) / nx);
  double2 lo = make_double2(0.0, 0.0), hi = lo;
  if (!(walls && (y == 0 || y == ny - 1))) {
    float v0[9], v1[9], v2[9], v3[9];
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      const float4 v = f[a * n4 + i];
      v0[a] = v.x;
      v1[a] = v.y;
      v2[a] = v.z;
      v3[a] = v.w;
    }
    lo = make_double2(sum9(v0), sum9(v1));
    hi = make_double2(sum9(v2), sum9(v3));
  }
  rho[2 * i] = lo;
  rho[2 * i + 1] = hi;
}

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Sum over the block (<= 1024 threads), valid in thread 0; a fixed tree.
__device__ __forceinline__ double block_sum(double s, double *sh) {
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 32) t = warp_sum(threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : 0.0);
  __syncthreads();
  return t;
}

// True in every thread of the block that arrives last of nb at *counter (which
// it leaves at 0): it then sees what the others wrote before arriving.
__device__ __forceinline__ bool arrives_last(unsigned *counter, unsigned nb) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(counter, 1u) == nb - 1u;
    if (last) *counter = 0u;
  }
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// Sum of val(i), i in [i0, i1), in a fixed order: block b sums a contiguous
// chunk, the last block to arrive the chunks' sums.
template <class Val>
__device__ __forceinline__ void sum_range(size_t i0, size_t i1, double *partial, unsigned *counter, double *out,
                                          Val val) {
  __shared__ double sh[32];
  const size_t len = i1 - i0, chunk = (len + gridDim.x - 1) / gridDim.x;
  const size_t b0 = i0 + blockIdx.x * chunk, b1 = min(i1, b0 + chunk);
  double s = 0.0;
  for (size_t i = b0 + threadIdx.x; i < b1; i += blockDim.x) s += val(i);
  s = block_sum(s, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
  if (!arrives_last(counter, gridDim.x)) return;
  s = 0.0;
  for (unsigned i = threadIdx.x; i < gridDim.x; i += blockDim.x) s += __ldcg(partial + i);
  s = block_sum(s, sh);
  if (threadIdx.x == 0) out[0] = s;
}

__global__ void k_sum(const double *__restrict__ v, size_t i0, size_t i1, double *partial, unsigned *counter,
                      double *out) {
  sum_range(i0, i1, partial, counter, out, [&](size_t i) { return v[i]; });
}

// rho = sum_a f_a in double, left to right, at node i.
__device__ __forceinline__ double node_rho64(const float *__restrict__ f, size_t n, size_t i) {
  float v[9];
#pragma unroll
  for (int a = 0; a < 9; ++a) v[a] = f[a * n + i];
  return sum9(v);
}
__device__ __forceinline__ double node_rho64(const double *__restrict__ f, size_t n, size_t i) {
  double r = 0.0;
#pragma unroll
  for (int a = 0; a < 9; ++a) r = r + f[a * n + i];
  return r;
}

// Total mass of the nodes [i0, i1) straight from the populations (the density
// field does not go through memory: 36 bytes a node instead of 52).
template <typename R>
__global__ void k_mass(const R *__restrict__ f, size_t n, size_t i0, size_t i1, double *partial, unsigned *counter,
                       double *out) {
  sum_range(i0, i1, partial, counter, out, [&](size_t i) { return node_rho64(f, n, i); });
}

// The sum of the populations of four nodes, rounded once.  Where all 36 are normal
// numbers within 31 binades, each is an integer below 2^54 times the last place of
// the smallest ones, and the sum of the integers stays below 2^60: one widening
// multiply-add per value.  Otherwise (zeros among them too) the sum of the four
// densities.
__device__ __forceinline__ double sum36(const float4 (&v)[9]) {
  unsigned lo = 0xffffffffu, hi = 0u;
  auto span = [&](float x) {
    const unsigned u = __float_as_uint(x) & 0x7fffffffu;
    lo = min(lo, u);
    hi = max(hi, u);
  };
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    span(v[a].x);
    span(v[a].y);
    span(v[a].z);
    span(v[a].w);
  }
  const int emin = (int)(lo >> 23), emax = (int)(hi >> 23);
  if (emin >= 1 && emax <= 254 && emax - emin <= 30) {
    long long S = 0;
    auto add = [&](float x) {
      const unsigned u = __float_as_uint(x);
      const int m = (int)((u & 0x7fffffu) | 0x800000u);
      S += (long long)((int)u < 0 ? -m : m) * (1 << (((int)(u >> 23) - emin) & 31));
    };
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      add(v[a].x);
      add(v[a].y);
      add(v[a].z);
      add(v[a].w);
    }
    return (double)S * __longlong_as_double((long long)(emin - 150 + 1023) << 52);
  }
  double r = 0.0;
#pragma unroll 1
  for (int k = 0; k < 4; ++k) {
    float q[9];
#pragma unroll
    for (int a = 0; a < 9; ++a) q[a] = k == 0 ? v[a].x : (k == 1 ? v[a].y : (k == 2 ? v[a].z : v[a].w));
    r += sum9(q);
  }
  return r;
}

// Mass of four nodes at once (nx % 4 == 0; groups [q0, q1)): 16-byte loads.
// 4096 x 2048, a call: the densities and their sum in two kernels 161 us, each
// node's density by itself 128, so 75; the populations alone take 45.
__global__ void k_mass_x4(const float4 *__restrict__ f, size_t n4, size_t q0, size_t q1, double *partial,
                          unsigned *counter, double *out) {
  sum_range(q0, q1, partial, counter, out, [&](size_t i) {
    float4 v[9];
#pragma unroll
    for (int a = 0; a < 9; ++a) v[a] = f[a * n4 + i];
    return sum36(v);
  });
}

// Block-wide minimum or maximum of one int, in every thread.
__device__ int block_reduce_int(int v, bool is_max, int *sh) {
  for (int o = 16; o > 0; o >>= 1) {
    int u = __shfl_down_sync(0xffffffffu, v, o);
    v = is_max ? max(v, u) : min(v, u);
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    int nw = blockDim.x >> 5;
    int t = threadIdx.x < nw ? sh[threadIdx.x] : (is_max ? INT_MIN : INT_MAX);
    for (int o = 16; o > 0; o >>= 1) {
      int u = __shfl_down_sync(0xffffffffu, t, o);
      t = is_max ? max(t, u) : min(t, u);
    }
    if (threadIdx.x == 0) sh[32] = t;
  }
  __syncthreads();
  return sh[32];
}

// ---- apparent contact angle ---------------------------------------------------
// The centre column is the one with the largest sum over the wall's half, each
// sum taken bottom to top, one addition after the other: a chain of 35 ns a row.
// In a half of few rows a block takes the sums of 32 columns so, from densities that
// it forms in parallel.  In a higher one the blocks sum chunks of rows in parallel,
// which places every column's sum within a proven distance of the sequential one;
// only columns within twice that distance of the largest still need the sequential
// sum to tell them apart.  Usually that is one column, or two (a droplet with a
// mirror axis between columns): up to four are summed by the last block.  With more
// (a wall without droplets, where all are equal) it leaves the domain undecided, and
// a second pass (k_angle_ties) takes the sums of all columns in parallel.
// us a call, FP32, one block over a density field / this, one column the largest | all
// equal: 300 x 100 49 / 37 | 42 / 35, 400 x 200 50 / 48 | 50 / 50, 512 x 400 73 / 47 |
// 75 / 50, 1001 x 501 122 / 47 | 114 / 97, 4096 x 2048 1365 / 182 | 1360 / 365.  A
// low half ends at 200 rows: at 249 (1001 x 501) its chain costs the call of one
// largest column 58 instead of 47, at 199 nothing (512 x 400).
// Everything else (the boundary row's liquid run, the walk up the centre column)
// reads its densities straight from the populations.  The last block's phases
// follow one another, so they are kept short: comparisons of positive doubles
// are made on their bits (an FP64 instruction of a warp takes 64 cycles), and
// the few divisions and the arc tangent are left to the host.

constexpr int kACols = 32, kALanes = 8, kARows = 64;  // columns, row lanes, rows of a block
constexpr int kAThreads = kACols * kALanes;
constexpr int kALow = 200, kLCols = 8, kLLanes = 32;  // rows of a low half; columns and row lanes of a block there
static_assert(kLCols * kLLanes == kAThreads, "one thread per column and lane");
constexpr int kAFew = 4;                              // columns that the last block may sum from the populations
constexpr int kTThreads = 128;                        // of a block of k_angle_ties

__device__ __forceinline__ long long bits(double v) { return __double_as_longlong(v); }
constexpr long long kInfBits = 0x7ff0000000000000ll;
// v >= lim for lim > 0 (false for NaN): numbers order like their bits, negative
// ones below, NaNs above infinity
__device__ __forceinline__ bool at_least(double v, long long lim) { return bits(v) >= lim && bits(v) <= kInfBits; }

// One copy of the density's code for the last block, which runs through its
// phases once: inlined in each, the instructions had to be fetched anew every
// time (400 x 200: 23 us more).
template <typename R>
__device__ __noinline__ double rho_at(const R *f, size_t n, size_t i) {
  return node_rho64(f, n, i);
}

__device__ __forceinline__ long long block_max_key(long long k, long long *sh) {
  for (int o = 16; o > 0; o >>= 1) k = max(k, __shfl_xor_sync(0xffffffffu, k, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = k;
  __syncthreads();
  for (int j = 0; j < kAThreads / 32; ++j) k = max(k, sh[j]);
  return k;
}

// Rows [lo, hi) of the wall's half.
__host__ __device__ __forceinline__ int half_lo(int ny, int wall) { return wall == 0 ? 1 : ny / 2; }
__host__ __device__ __forceinline__ int half_hi(int ny, int wall) { return wall == 0 ? ny / 2 : ny - 1; }

// Column of the largest sum (the lowest of equal ones) over the block's threads, in
// every thread; INT_MAX where no thread has one.
template <int THREADS>
__device__ __forceinline__ int block_argmax(double best, int x) {
  __shared__ double shv[THREADS / 32];
  __shared__ int shx[THREADS / 32];
  for (int o = 16; o > 0; o >>= 1) {
    const double ov = __shfl_down_sync(0xffffffffu, best, o);
    const int ox = __shfl_down_sync(0xffffffffu, x, o);
    if (ov > best || (ov == best && ox < x)) best = ov, x = ox;
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) shv[threadIdx.x >> 5] = best, shx[threadIdx.x >> 5] = x;
  __syncthreads();
  best = shv[0], x = shx[0];
  for (int j = 1; j < THREADS / 32; ++j)
    if (shv[j] > best || (shv[j] == best && shx[j] < x)) best = shv[j], x = shx[j];
  __syncthreads();
  return x;
}

// The cuts of the contour with the boundary row and the centre column xc, by one block.
template <typename R>
__device__ __forceinline__ void cut_at(const lbm_angle_args &A, int xc) {
  __shared__ int shi[33];
  const int nx = A.nx, ny = A.ny, wall = A.wall, x0 = A.x0, x1 = A.x1;
  const long long mid = bits(A.rho_mid);
  const R *f = (const R *)A.f;
  const size_t n = (size_t)nx * ny;
  auto rho = [&](int y, int x) { return rho_at(f, n, (size_t)y * nx + x); };
  lbm_angle_cut *res = A.res;
  if (xc < x0 || xc >= x1) {  // no column has a sum at all (NaN everywhere)
    if (threadIdx.x == 0) res->contact = 0;
    return;
  }
  const int ylo = half_lo(ny, wall), yhi = half_hi(ny, wall);
  const int base = wall == 0 ? 1 : ny - 2, dir = wall == 0 ? 1 : -1;
  // liquid run of the boundary row containing xc
  int jl = INT_MIN, jr = INT_MAX;
  bool dry = false;
  for (int x = x0 + threadIdx.x; x < x1; x += blockDim.x) {
    const bool vap = !at_least(rho(base, x), mid);
    if (vap && x < xc) jl = max(jl, x);
    if (vap && x > xc) jr = min(jr, x);
    dry |= vap && x == xc;
  }
  // first vapour node walking away from the wall along xc
  const int ymax = wall == 0 ? yhi : ylo - 1;
  const int nwalk = wall == 0 ? (ymax - base - 1) : (base - ymax - 1);
  int kmin = INT_MAX;
  for (int k = 1 + threadIdx.x; k <= nwalk; k += blockDim.x)
    if (!at_least(rho(base + k * dir, xc), mid)) {
      kmin = k;
      break;
    }
  jl = block_reduce_int(jl, true, shi);
  jr = block_reduce_int(jr, false, shi);
  kmin = block_reduce_int(kmin, false, shi);
  if (__syncthreads_or(dry) || jl == INT_MIN || jr == INT_MAX || kmin == INT_MAX) {
    if (threadIdx.x == 0) res->contact = 0;
    return;
  }
  // the six densities around the three crossings
  const int t = threadIdx.x, y = base + (kmin - 1) * dir;
  if (t < 6) res->rho[t] = t < 4 ? rho(base, t < 2 ? jl + t : jr - 3 + t) : rho(y + (t - 4) * dir, xc);
  if (t == 0) {
    res->xl = jl;
    res->xr = jr - 1;
    res->steps = kmin - 1;
    res->contact = 1;
  }
}

// Blocks of a domain: groups of columns x chunks of rows (a low half in one).
struct AngleGrid {
  bool low;
  int groups, chunks;
  __host__ __device__ __forceinline__ AngleGrid(int cols, int half) : low(half <= kALow) {
    groups = low ? (cols + kLCols - 1) / kLCols : (cols + kACols - 1) / kACols;
    chunks = low ? 1 : (half + kARows - 1) / kARows;
  }
};

// The blocks of one domain along x, domains of a table along y (tab == NULL: the one
// in A).
template <typename R>
__global__ void __launch_bounds__(kAThreads) k_angle(lbm_angle_args A, const lbm_angle_args *__restrict__ tab) {
  if (tab) A = tab[blockIdx.y];
  const int nx = A.nx, ny = A.ny, wall = A.wall, x0 = A.x0, x1 = A.x1, cols = x1 - x0;
  const int ylo = half_lo(ny, wall), yhi = half_hi(ny, wall), half = yhi - ylo;
  const AngleGrid G(cols, half);
  const int chunks = G.chunks;
  if ((int)blockIdx.x >= G.groups * chunks) return;

  __shared__ double tile[kALow * kLCols];
  {
    const R *f = (const R *)A.f;
    const size_t n = (size_t)nx * ny;
    const int g = (int)blockIdx.x % G.groups, k = (int)blockIdx.x / G.groups, w = G.low ? kLCols : kACols;
    const int tx = threadIdx.x % w, ty = threadIdx.x / w, c = g * w + tx;
    double s = 0.0;
    if (G.low) {  // the columns' sums in order
      if (c < cols)
#pragma unroll 2
        for (int y = ty; y < half; y += kLLanes) tile[y * kLCols + tx] = node_rho64(f, n, (size_t)(ylo + y) * nx + x0 + c);
      __syncthreads();
      if (ty == 0 && c < cols)
#pragma unroll 8
        for (int y = 0; y < half; ++y) s = s + tile[y * kLCols + tx];
    } else {  // the block's part of them; NaN where a density is negative or not finite
              // (the bound below is for positive terms)
      if (c < cols) {
        const int ya = ylo + k * kARows, yb = min(yhi, ya + kARows);
        bool odd = false;
#pragma unroll 2
        for (int y = ya + ty; y < yb; y += kALanes) {
          const double r = node_rho64(f, n, (size_t)y * nx + x0 + c);
          odd |= (unsigned long long)bits(r) >= (unsigned long long)kInfBits;
          s += r;
        }
        if (odd) s = (double)NAN;
      }
      tile[ty * kACols + tx] = s;
      __syncthreads();
      if (ty == 0 && c < cols)
        for (int j = 1; j < kALanes; ++j) s += tile[j * kACols + tx];
    }
    if (ty == 0 && c < cols) A.partial[(size_t)k * cols + c] = s;
  }
  if (!arrives_last(A.counter, (unsigned)(G.groups * chunks))) return;

  // ---- the last block ----
  double best = -DBL_MAX;
  int xc = INT_MAX;
  if (G.low) {
    for (int c = threadIdx.x; c < cols; c += kAThreads) {
      const double s = __ldcg(A.partial + c);
      if (s > best) best = s, xc = x0 + c;
    }
    cut_at<R>(A, block_argmax<kAThreads>(best, xc));
    return;
  }
  __shared__ long long shk[kAThreads / 32];
  // bits of a column's sum (NaN: above kInfBits)
  auto total = [&](int c) {
    double s = __ldcg(A.partial + c);
    for (int k = 1; k < chunks; ++k) s += __ldcg(A.partial + (size_t)k * cols + c);
    return bits(s);
  };
  long long top = -1;
  for (int c = threadIdx.x; c < cols; c += kAThreads) {
    const long long t = total(c);
    if (t <= kInfBits) top = max(top, t);
  }
  top = block_max_key(top, shk);
  // A sum of m positive terms, in any order, is within m 2^-53 of the true one
  // (relative, to first order), so two sums of a column differ by at most
  // m 2^-52 or m units in the last place; the largest sequential sum is among
  // the columns within twice that of the largest of these (here eight times, as
  // the units halve below a power of two).
  const long long near = top - (8LL * half + 64LL);
  // candidates: their number, and the first few to be found
  __shared__ int found, cand[kAFew];
  if (threadIdx.x == 0) found = 0;
  __syncthreads();
  for (int c = threadIdx.x; c < cols; c += kAThreads)
    if (total(c) >= near) {
      const int k = atomicAdd(&found, 1);
      if (k < kAFew) cand[k] = c;
    }
  __syncthreads();
  if (found > kAFew) {
    if (threadIdx.x == 0) A.res->contact = -1;
    return;
  }
  xc = x0 + cand[0];
  if (found > 1) {
    // one after the other: the densities of 256 rows in parallel, added by one thread
    __shared__ double line[kAThreads];
    xc = INT_MAX;
    for (int j = 0; j < found; ++j) {
      const int x = x0 + cand[j];
      double s = 0.0;
      for (int y = ylo; y < yhi; y += kAThreads) {
        if (y + (int)threadIdx.x < yhi)
          line[threadIdx.x] = rho_at((const R *)A.f, (size_t)nx * ny, (size_t)(y + threadIdx.x) * nx + x);
        __syncthreads();
        if (threadIdx.x == 0)
          for (int k = 0; k < min(kAThreads, yhi - y); ++k) s = s + line[k];
        __syncthreads();
      }
      if (threadIdx.x == 0 && (s > best || (s == best && x < xc))) best = s, xc = x;
    }
    xc = block_argmax<kAThreads>(best, xc);
  }
  cut_at<R>(A, xc);
}

// The same from the densities rho [ny][nx] of the wall's half: every column's sum
// by one thread, sums[] and the largest of them by the last block.
template <typename R>
__global__ void __launch_bounds__(kTThreads) k_angle_ties(lbm_angle_args A, const double *rho, double *sums) {
  const int ylo = half_lo(A.ny, A.wall), half = half_hi(A.ny, A.wall) - ylo, cols = A.x1 - A.x0;
  const int c = blockIdx.x * kTThreads + threadIdx.x;
  if (c < cols) {
    const double *v = rho + (size_t)ylo * A.nx + A.x0 + c;
    double s = 0.0;
#pragma unroll 16
    for (int y = 0; y < half; ++y) s = s + v[(size_t)y * A.nx];
    sums[c] = s;
  }
  if (!arrives_last(A.counter, gridDim.x)) return;
  double best = -DBL_MAX;
  int xc = INT_MAX;
  for (int k = threadIdx.x; k < cols; k += kTThreads) {
    const double s = __ldcg(sums + k);
    if (s > best) best = s, xc = A.x0 + k;
  }
  cut_at<R>(A, block_argmax<kTThreads>(best, xc));
}

inline unsigned nblk(size_t n, int t) { return (unsigned)((n + t - 1) / t); }

// FP32 populations to and from the caller's doubles.
template <typename From, typename To>
__global__ void k_convert(const From *__restrict__ in, To *__restrict__ out, size_t n) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = (To)in[i];
}

}  // namespace

cudaError_t lbm_widen(const lbm_ctx *C, const float *in, double *out, size_t n, unsigned long long *launches) {
  k_convert<<<(unsigned)((n + 255) / 256), 256, 0, C->stream>>>(in, out, n);
  ++*launches;
  return cudaGetLastError();
}
cudaError_t lbm_narrow(const lbm_ctx *C, const double *in, float *out, size_t n, unsigned long long *launches) {
  k_convert<<<(unsigned)((n + 255) / 256), 256, 0, C->stream>>>(in, out, n);
  ++*launches;
  return cudaGetLastError();
}

cudaError_t lbm_rho64_rows(const lbm_ctx *C, const void *f, double *rho, int row0, int row1,
                           unsigned long long *launches) {
  const size_t i0 = (size_t)row0 * C->nx, i1 = (size_t)row1 * C->nx;
  if (i1 <= i0) return cudaSuccess;
  if (C->precision == 64)
    k_rho64<double><<<nblk(i1 - i0, 256), 256, 0, C->stream>>>(C->nx, C->ny, C->walls, (const double *)f, rho, i0,
                                                                i1);
  else if (C->nx % 4 == 0 && ((uintptr_t)f & 15) == 0 && ((uintptr_t)rho & 15) == 0)
    k_rho64_x4<<<nblk((i1 - i0) / 4, 256), 256, 0, C->stream>>>(C->nx, C->ny, C->walls, (const float4 *)f,
                                                                 (double2 *)rho, i0 / 4, i1 / 4);
  else
    k_rho64<float><<<nblk(i1 - i0, 256), 256, 0, C->stream>>>(C->nx, C->ny, C->walls, (const float *)f, rho, i0, i1);
  ++*launches;
  return cudaGetLastError();
}

cudaError_t lbm_rho64(const lbm_ctx *C, const void *f, double *rho, unsigned long long *launches) {
  return lbm_rho64_rows(C, f, rho, 0, C->ny, launches);
}

cudaError_t lbm_reduce_rows(const lbm_ctx *C, const double *v, int row0, int row1, double *res,
                            unsigned long long *launches) {
  k_sum<<<C->red_len, 256, 0, C->stream>>>(v, (size_t)row0 * C->nx, (size_t)row1 * C->nx, C->d_red,
                                           (unsigned *)C->d_flag + 3, res);
  ++*launches;
  return cudaGetLastError();
}

cudaError_t lbm_mass_of(const lbm_ctx *C, const void *f, double *res, unsigned long long *launches) {
  const size_t n = (size_t)C->nx * C->ny, i0 = C->walls ? C->nx : 0, i1 = n - i0;
  unsigned *counter = (unsigned *)C->d_flag + 3;
  const bool x4 = C->precision == 32 && C->nx % 4 == 0 && ((uintptr_t)f & 15) == 0;
  const unsigned g = std::min((unsigned)C->red_len, nblk((i1 - i0) / (x4 ? 4 : 1), 256));
  if (C->precision == 64)
    k_mass<double><<<g, 256, 0, C->stream>>>((const double *)f, n, i0, i1, C->d_red, counter, res);
  else if (x4)
    k_mass_x4<<<g, 256, 0, C->stream>>>((const float4 *)f, n / 4, i0 / 4, i1 / 4, C->d_red, counter, res);
  else
    k_mass<float><<<g, 256, 0, C->stream>>>((const float *)f, n, i0, i1, C->d_red, counter, res);
  ++*launches;
  return cudaGetLastError();
}

lbm_angle_args lbm_make_angle_args(const lbm_ctx *C, int wall, int x0, int x1, void *res) {
  return lbm_angle_args{C->f[C->cur], C->nx, C->ny, wall, x0, x1, C->rho_mid, C->d_rho64, (unsigned *)C->d_flag + 3,
                        (lbm_angle_cut *)res};
}

int lbm_angle_of(const lbm_angle_cut &r, double rho_mid, double *theta, double *H, double *L) {
  if (r.contact <= 0) return LBM_ENOCONTACT;
  const double *q = r.rho;
  const double left = (double)r.xl + (rho_mid - q[0]) / (q[1] - q[0]);
  const double right = (double)r.xr + (q[2] - rho_mid) / (q[2] - q[3]);
  *H = (double)r.steps + (q[4] - rho_mid) / (q[4] - q[5]);
  *L = right - left;
  *theta = 2.0 * atan2(2.0 * *H, *L);
  return LBM_OK;
}

int lbm_angle_blocks(const lbm_angle_args &A) {
  const AngleGrid G(A.x1 - A.x0, half_hi(A.ny, A.wall) - half_lo(A.ny, A.wall));
  return G.groups * G.chunks;
}

cudaError_t lbm_angle(const lbm_ctx *C, const lbm_angle_args &A, unsigned long long *launches) {
  const dim3 g(lbm_angle_blocks(A));
  if (C->precision == 64)
    k_angle<double><<<g, kAThreads, 0, C->stream>>>(A, nullptr);
  else
    k_angle<float><<<g, kAThreads, 0, C->stream>>>(A, nullptr);
  ++*launches;
  return cudaGetLastError();
}

cudaError_t lbm_angle_ties(const lbm_ctx *C, const lbm_angle_args &A, unsigned long long *launches) {
  // the sums go where the density of the lower solid row would be
  cudaError_t e = lbm_rho64_rows(C, A.f, C->d_rho64, half_lo(A.ny, A.wall), half_hi(A.ny, A.wall), launches);
  if (e != cudaSuccess) return e;
  const unsigned g = nblk(A.x1 - A.x0, kTThreads);
  if (C->precision == 64)
    k_angle_ties<double><<<g, kTThreads, 0, C->stream>>>(A, C->d_rho64, C->d_rho64);
  else
    k_angle_ties<float><<<g, kTThreads, 0, C->stream>>>(A, C->d_rho64, C->d_rho64);
  ++*launches;
  return cudaGetLastError();
}

cudaError_t lbm_angle_many(const lbm_angle_args *tab, int first, int count, int blocks, cudaStream_t stream) {
  k_angle<float><<<dim3(blocks, count), kAThreads, 0, stream>>>(lbm_angle_args{}, tab + first);
  return cudaGetLastError();
}
