// Temporally blocked 2D wave step in 64-bit fixed point (fixed64.cuh): the FP64 wave solve of
// 2D problems, second or fourth order, with a constant or two-layer c^2.
//
// The scheme is advanced in its increment form, D^{n+1/2} = D^{n-1/2} + kappa_n (c^2 Delta_h W^n -
// F^n), W^{n+1} = W^n + D^{n+1/2} (kappa_0 = dt^2/2 with D^{-1/2} = 0, else dt^2; eq. WaveSchemeA,
// eq. implicitFirstStep with alpha = 0), W and D as integers in units of the launch's quantum.  A
// step rounds once per point (the product with kappa c^2 / h^2; a second time for the forcing).
// The filter sums q_m = sum_n w_{n,m} W^n (eq. pDefQ) are 64-bit integers too.  The contribution of
// a launch's 8 steps is formed from the weights' and the levels' two 32-bit digits (60 bits of the
// weights): high x high and high x low digits are summed exactly, the weights' low digits times the
// levels' high ones in FP32 (2^-24 of terms below 2^-28 of the largest), low x low is dropped
// (2^-60), and the sum is rounded once to the unit of the sums.  The filter solve is FP64.  The
// forcing of a launch's steps is summed over the frequencies by a kernel before it (k_fx_force),
// once per point, in the same way.
//
// The quantum.  A launch knows the largest |W| and |D| of its input (FxState, left by the launch
// before), and with them bounds every level of its steps: |W^{n+k}| <= gw max |W| + gd max |D| + gf
// kappa sum_m max |f_m|, where gw, gd and gf are the largest absolute row sums of the 8 steps'
// propagators (api.cu).  It takes the quantum that puts this bound just below 2^59, so that the
// neighbour differences (at most 8 times a level) fit 63 bits, and rescales its input by the power
// of two between the two quanta.  The sums' unit follows the largest bound so far, with
// sum_n |w_{n,m}| below 2^wsum weight units: |q_m| < 2^62.
//
// What bounds it.  A point-step of the FP64 form takes five FP64 instructions, 64 cycles each of
// an SM sub-partition, and 15 FP32 instructions per filter sum (float pairs).  Here it is about 13
// integer additions with carry, 4 wide products and 2 shuffles, and 3 multiply-adds per filter sum:
// the kernel is bound by instruction issue and the integer multiplier and, on grids beyond L2, by
// HBM (32 + 16 N_f bytes per point and launch of 8 steps).  N_f = 8, homogeneous, per 8 steps: 76
// us on 1025^2 (111 Gpts/s) against 162 us for the FP64 form (k_tb2d_pipe), 248 us on 2049^2, 26 us
// on 513^2.  Small grids are bound by the latency of a launch: 10.4 us on 65^2, of which 5 with
// nothing stepped and no sums made.  Fourth order, 513^2, N_f = 3: 22.5 us per 4 steps against 4 x
// 12.2 us for the FP64 one-step kernel.
//
// Roles.  A persistent CTA per SM has kFxStep warps that step tiles and kFxTail warps that make
// the filter sums of the tile stepped before, so that the one's loads, stores and barriers
// overlap the other's arithmetic.  (With one role after the other, in one CTA per SM or in two,
// which then run in the same phase, a launch took the sum of the phases' times.)
//
// Tile.  The step warps hold an extended tile of 64 x 4 warps points in registers: lane l has
// columns 2l, 2l + 1, warp w rows 4w .. 4w + 3.  Every step updates all of them except that a warp
// rests once no later step reads its rows; after 8 steps the points 8 or more from the edge are
// exact.  Left and right neighbours come by shuffle, the rows above and below a warp's four
// through shared memory (double buffered: one barrier per step).  An owned point's new value
// is stored per step as two digits in shared memory (64 bytes per owned point, double buffered
// between the roles); a thread of the tail warps takes owned points one by one and forms their N_f
// contributions in registers, with the weights as constant operands.  (All of this for the
// second-order operator; the fourth-order one reaches two points, so a launch makes 4 steps within
// the same halo, the warps exchange all their rows, and its sums of 64 times a level along an axis
// leave the levels 56 bits.)  The sums are laid out tile by tile, [tile][m][owned point], so that
// their addresses are a pointer plus constants and the loop has no index arithmetic or masks (points
// outside the interior have zero levels).
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <type_traits>

#include "fixed64.cuh"
#include "kernels.h"

namespace mfwh {
namespace {

constexpr int kFxT = 8;                          // halo points: 8 steps of reach 1 or 4 of reach 2
constexpr int kFxStep = 12, kFxTail = 8;         // warps of the two roles (step warps: at most)
constexpr int kFxThreads = 32 * (kFxStep + kFxTail);
constexpr int kFxEX = 64, kFxEY = 4 * kFxStep;   // extended tile
constexpr int kFxVX = kFxTileX;                  // owned columns
static_assert(kFxVX == kFxEX - 2 * kFxT && kFxTileY == kFxEY - 2 * kFxT, "tile and halo");

// Coefficients kappa c^2 / h_x^2 and / h_y^2 of one layer and step kind.
struct FxAxes {
  FxCoef x, y;
};

template <int NF>
struct FxArgs {
  FxAxes coef[2][2];         // [first step][upper layer]
  LayerCoef lay[2][2];       // the same steps in FP64 (fallback)
  int n0, steps, forced, last, has_e;
  int warps, wsum;
  int subtract;              // v_out = V (0), v_sub - V (1) or v_sub + V (-1)
  float gw, gd;              // growth of the levels in 8 steps
  const double* vprev;       // V^k
  double binv[NF * NF];      // epilogue V^{k+1} = C q + E V^k
  double emat[NF * NF];
  int wh[kFxT * NF];         // digits of w_{n+1,m} 2^wexp[m] of step s, [s * NF + m]: the high
  float wl[kFxT * NF];       // one, and the low one / 2^32
  int64_t off1[NF], off2[NF];         // the sums' start: the level digits' constant, rounding
  int wexp[NF];
  double wd[kFxT * NF];      // w_{n+1,m} (fallback)
  double fc[kFxT * NF];      // kappa_n cos(omega~_m t^n)
};

// Shared memory: the two buffers of new values, the two of edge rows (2 or 4 per warp).
constexpr size_t fx_hist_bytes(int order) {
  return (size_t)fx_launch_steps(order) * kFxTile * sizeof(int2);
}
constexpr size_t fx_smem_bytes(int order) {
  return 2 * fx_hist_bytes(order) + (size_t)2 * kFxStep * order * kFxEX * 8;
}

// Barriers among part of the CTA's warps (0 is __syncthreads).
__device__ __forceinline__ void fx_bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void fx_bar_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void fx_prefetch(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// The quantum 2^e of a launch from its input's state, the factor 2^shift of the input and the
// unit of the sums.  b: bound of the launch's levels in the input's quanta, which the quantum puts
// just below 2^fx_bits.  In FP32, rounding up: every warp makes it before its first load is used, and
// the few FP64 instructions it would take cost a launch a microsecond (64 cycles a warp each).
struct FxQuantum {
  float b;
  int shift, e, eq;
};
__device__ __forceinline__ FxQuantum fx_quantum(const FxState& st, const FxScale& sc, float gw,
                                                float gd, int wsum, int order) {
  FxQuantum r;
  r.b = __fmaf_ru(gw, __ull2float_ru(st.wmax), __fmul_ru(gd, __ull2float_ru(st.dmax)));
  // (a quantum keeps the forcing's part below 2^59: no overflow; far below the levels it may
  // become 0 in float, and counts one quantum)
  if (sc.fm > 0.0f) r.b = __fadd_ru(r.b, __fadd_ru(ldexpf(sc.fm, sc.fx - st.e), 1.0f));
  r.shift = 0;
  r.eq = st.eq;
  if (r.b > 0.0f) {
    const int ex = (__float_as_int(r.b) >> 23) - 126;   // b < 2^ex (b is normal)
    r.shift = fx_bits(order) - ex;
    r.eq = max(r.eq, ex + st.e + wsum - 62);
  }
  r.e = st.e - r.shift;
  return r;
}

// A global offset clamped into [lo, hi] as a 32-bit local coordinate.
__device__ __forceinline__ int fx_clamp(int64_t v, int lo, int hi) {
  return v < lo ? lo : (v > hi ? hi : (int)v);
}

// The steps of one launch on one tile in FP64, for values that have no quantum (infinities, NaN,
// magnitudes near the ends of the double range): A and B hold W^n and W^{n-1} on the extended
// tile in shared memory, the sums (qi: the tile's) are updated in place in global memory.  The
// arrays hold doubles.
template <int NF, int ORDER>
__device__ __noinline__ void fx_double_steps(double* A, double* B, const FxArrays& in,
                                             const FxArrays& out, const double* f, int64_t* qi,
                                             const FxArgs<NF>& a, const Geom& g, int64_t x0,
                                             int64_t y0) {
  constexpr int T = kFxT;
  const int EY = 4 * a.warps;
  double* q = reinterpret_cast<double*>(qi);
  const int tid = threadIdx.x;
  constexpr int kTileValues = kFxEX * kFxEY;   // of A and of B
  for (int e = tid; e < kFxEX * EY; e += blockDim.x) {
    const int64_t x = x0 + e % kFxEX, y = y0 + e / kFxEX;
    const bool is = x >= 0 && x <= g.nx && y >= 0 && y <= g.ny &&
                    MFWH_IDX(g.fault, y * g.syw + x, g.wpoints);
    if (!MFWH_IDX(g.fault, e, kTileValues)) continue;
    A[e] = is ? __longlong_as_double(in.W[y * g.syw + x]) : 0.0;
    B[e] = (is && a.n0 > 0) ? __longlong_as_double(in.D[y * g.syw + x]) : 0.0;
  }
  __syncthreads();
  for (int s = 0; s < a.steps; ++s) {
    const int first = a.n0 + s == 0;
    for (int e = tid; e < kFxEX * EY; e += blockDim.x) {
      const int lx = e % kFxEX, ly = e / kFxEX;
      const int64_t x = x0 + lx, y = y0 + ly;
      constexpr int H = ORDER / 2;   // reach
      if (lx < H || lx >= kFxEX - H || ly < H || ly >= EY - H || x <= 0 || x >= g.nx || y <= 0 ||
          y >= g.ny)
        continue;
      const LayerCoef& L = a.lay[first][(g.layer_axis == 0 ? x : y) >= g.layer_split];
      const double sx = A[e - 1] + A[e + 1], sy = A[e - kFxEX] + A[e + kFxEX];
      double acc = fma(L.A0, A[e], -B[e]);
      acc = fma(L.Ax, sx, acc);
      acc = fma(L.Ay, sy, acc);
      if constexpr (ORDER == 4) {   // the ghost value beyond the boundary is minus the centre's
        const double tx = (x == 1 ? -A[e] : A[e - 2]) + (x == g.nx - 1 ? -A[e] : A[e + 2]);
        const double ty =
            (y == 1 ? -A[e] : A[e - 2 * kFxEX]) + (y == g.ny - 1 ? -A[e] : A[e + 2 * kFxEX]);
        acc = fma(L.Bx, tx, acc);
        acc = fma(L.By, ty, acc);
      }
      const int64_t p = y * g.sy + x;
      if (!MFWH_IDX(g.fault, p, g.points)) continue;
      if (a.forced)
        for (int m = 0; m < NF; ++m) acc = fma(-a.fc[s * NF + m], f[m * g.points + p], acc);
      B[e] = acc;
      if (lx >= T && lx < kFxEX - T && ly >= T && ly < EY - T) {
        double* qp = q + (ly - T) * kFxVX + lx - T;
        if (!MFWH_IDX(g.fault, (ly - T) * kFxVX + lx - T, kFxTile)) continue;
        for (int m = 0; m < NF; ++m)
          qp[m * kFxTile] = fma(a.wd[s * NF + m], acc, qp[m * kFxTile]);
      }
    }
    __syncthreads();
    double* t = A;
    A = B;
    B = t;
  }
  if (a.last) return;
  for (int e = tid; e < kFxEX * EY; e += blockDim.x) {
    const int lx = e % kFxEX, ly = e / kFxEX;
    const int64_t x = x0 + lx, y = y0 + ly;
    if (lx < T || lx >= kFxEX - T || ly < T || ly >= EY - T || x > g.nx || y > g.ny) continue;
    if (!MFWH_IDX(g.fault, y * g.syw + x, g.wpoints)) continue;
    out.W[y * g.syw + x] = __double_as_longlong(A[e]);
    out.D[y * g.syw + x] = __double_as_longlong(B[e]);
  }
}

// Epilogue of the last launch at one grid point (q: its first sum, offset o in the [points] arrays):
// V^{k+1} = C q + E V^k at interior points, 0 on the boundary.
template <int NF>
__device__ __noinline__ void fx_finish(const int64_t* q, const double* unit, bool is, double* vout,
                                          const double* vsub, const FxArgs<NF>& a,
                                          int64_t points, int64_t o) {
  double qd[NF], vk[NF];
#pragma unroll
  for (int j = 0; j < NF; ++j) {   // unit null: the sums are doubles
    const int64_t v = is ? q[j * kFxTile] : 0;
    qd[j] = unit ? (double)v * unit[j] : __longlong_as_double(v);
    vk[j] = (a.has_e && is) ? a.vprev[j * points + o] : 0.0;   // (v_out may be V^k)
  }
#pragma unroll 1
  for (int m = 0; m < NF; ++m) {
    double acc = 0.0;
#pragma unroll
    for (int j = 0; j < NF; ++j) acc = fma(a.binv[m * NF + j], qd[j], acc);
    if (a.has_e) {
#pragma unroll
      for (int j = 0; j < NF; ++j) acc = fma(a.emat[m * NF + j], vk[j], acc);
    }
    if (a.subtract) acc = a.subtract > 0 ? vsub[m * points + o] - acc : vsub[m * points + o] + acc;
    vout[m * points + o] = is ? acc : 0.0;
  }
}

// Reads W, D (level n0; D is not read when n0 = 0) and writes those of level n0 + steps, with the
// sums updated in place; the last launch writes v_out instead.  state[0]: the input's quantum and
// maxima; state[1]: the output's, its maxima 0 on entry; state[2]: reset to 0.  ISO (second
// order): equal spacings (one product per step instead of two).
template <int NF, bool ISO, bool FORCED, int ORDER>
__global__ void __launch_bounds__(kFxThreads, 1)
k_fx2d(const FxArrays in, const FxArrays out, const double* __restrict__ f,
       const int64_t* force, int64_t* __restrict__ q, double* vout, const double* vsub,
       const __grid_constant__ FxArgs<NF> a, const FxScale* scale,
       const FxState* s_in, FxState* s_out, FxState* s_reset, const Geom g, int tiles_x,
       int tiles) {
  constexpr int T = kFxT, VX = kFxVX, REACH = ORDER / 2, STEPS = fx_launch_steps(ORDER);
  constexpr size_t kHist = fx_hist_bytes(ORDER);
  const int NW = a.warps, EY = 4 * NW, VY = EY - 2 * T;   // step warps, rows of the tile, owned rows
  const int threads = 32 * (NW + kFxTail);
  constexpr int kBarStep = 1, kBarFull = 2, kBarEmpty = 4;   // (and + 1: second buffer)
  extern __shared__ __align__(16) unsigned char fx_smem[];
  __shared__ double s_unit[NF];   // last launch: unit of the sums
  __shared__ int64_t s_off[NF];   // start of the contributions, with half a unit of the sums
  int64_t* edge = reinterpret_cast<int64_t*>(fx_smem + 2 * kHist);   // [2][warp][ORDER][64]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_begin();
  const FxScale sc = *scale;
  if (sc.mode) {   // FP64 steps by the whole CTA
    double* A = reinterpret_cast<double*>(fx_smem);
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
      const int64_t x0 = (int64_t)(tile % tiles_x) * VX - T, y0 = (int64_t)(tile / tiles_x) * VY - T;
      int64_t* qt = q + (int64_t)tile * NF * kFxTile;
      fx_double_steps<NF, ORDER>(A, A + kFxEX * EY, in, out, f, qt, a, g, x0, y0);
      __syncthreads();
      if (!a.last) continue;
      for (int i = tid; i < VX * VY; i += threads) {
        const int64_t x = x0 + T + i % VX, y = y0 + T + i / VX;
        if (x > g.nx || y > g.ny || !MFWH_IDX(g.fault, y * g.sy + x, g.points)) continue;
        const bool is = x > 0 && x < g.nx && y > 0 && y < g.ny;
        fx_finish<NF>(qt + i, nullptr, is, vout, vsub, a, g.points, y * g.sy + x);
      }
    }
    return;
  }
  const FxState st = *s_in;
  const FxQuantum Q = fx_quantum(st, sc, a.gw, a.gd, a.wsum, ORDER);
  const int shift = Q.shift;
  const bool zero = Q.b == 0.0f;   // all levels are 0
  // shifts of the stored sums and of the launch's contributions (units of 2^(e + 64)): eq - e - 64
  // >= wsum + fx_bits - 126 >= 0 as the bound's exponent is e + fx_bits
  const int q_old = Q.eq - st.eq, q_new = Q.eq - Q.e - 64;
  const bool wide = q_new >= 32;   // the contributions' high words only
  if (blockIdx.x == 0 && tid == 0) {
    s_out->e = Q.e;
    s_out->eq = Q.eq;
    s_reset->wmax = s_reset->dmax = 0;
  }
  if (tid < NF) {
    if (a.last) s_unit[tid] = ldexp(1.0, Q.eq - a.wexp[tid]);
    s_off[tid] = a.off1[tid] + (q_new > 0 && q_new < 62 ? (int64_t)1 << (q_new - 1) : 0);
  }
  __syncthreads();
  if (warp < NW) {
    // ---- step warps
    const int lx = 2 * lane, ly = 4 * warp;   // this thread's first point
    const bool owner = lx >= T && lx < T + VX && ly >= T && ly < T + VY;
    int mw = 0, md = 0;                        // largest high words of |W| and |D|
    int it = 0;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++it) {
      int2* hist = reinterpret_cast<int2*>(fx_smem + (it & 1) * kHist);   // [T][kFxTile]
      const int64_t x0 = (int64_t)(tile % tiles_x) * VX - T, y0 = (int64_t)(tile / tiles_x) * VY - T;
      // local bounds of grid rows and of interior points; first local index of the upper layer
      const int ghy = fx_clamp(g.ny - y0, -1, EY - 1);
      const int ilx = fx_clamp(1 - x0, 0, kFxEX), ihx = fx_clamp(g.nx - 1 - x0, -1, kFxEX - 1);
      const int ily = fx_clamp(1 - y0, 0, EY), ihy = fx_clamp(g.ny - 1 - y0, -1, EY - 1);
      const bool lay_x = g.layer_axis == 0;
      const int thr = fx_clamp(g.layer_split - (lay_x ? x0 : y0), 0, kFxEX + EY);
      // the thread's points: interior (bit 2k + c of in_mask), upper layer (of hi_mask)
      unsigned in_mask = 0, hi_mask = 0;
      const unsigned in_x =
          (lx >= ilx && lx <= ihx ? 1u : 0u) | (lx + 1 >= ilx && lx + 1 <= ihx ? 2u : 0u);
      const unsigned hi_x = lay_x ? (lx >= thr ? 1u : 0u) | (lx + 1 >= thr ? 2u : 0u) : 0u;
      int64_t w[4][2], d[4][2];
      const int64_t base = (y0 + ly) * g.syw + x0 + lx;
      // x0 + lx is even and rows are padded: both columns lie in a row of the arrays or none
      const bool col = x0 + lx >= 0 && x0 + lx < g.syw;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int64_t o = base + k * g.syw;
        const bool have = col && y0 + ly + k >= 0 && ly + k <= ghy &&
                          MFWH_IDX(g.fault, o, g.wpoints) && MFWH_IDX(g.fault, o + 1, g.wpoints);
        longlong2 v = make_longlong2(0, 0), u = v;
        if (have) {
          v = *reinterpret_cast<const longlong2*>(in.W + o);
          if (a.n0 > 0) u = *reinterpret_cast<const longlong2*>(in.D + o);
        }
        w[k][0] = v.x;
        w[k][1] = v.y;
        d[k][0] = u.x;
        d[k][1] = u.y;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const unsigned row = ly + k >= ily && ly + k <= ihy ? in_x : 0u;
        in_mask |= row << (2 * k);
        hi_mask |= (lay_x ? hi_x : (ly + k >= thr ? 3u : 0u)) << (2 * k);
        // points outside the interior (boundary, padding) are 0
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const bool is = row >> c & 1u;
          w[k][c] = is ? fx_rescale(w[k][c], shift) : 0;
          d[k][c] = is ? fx_rescale(d[k][c], shift) : 0;
        }
      }
      // the rows a warp shows its neighbours: second order 0 and 3, fourth order all
      auto edge_row = [&](int buf, int wp, int row) {
        const int i = ((buf * kFxStep + wp) * ORDER + (ORDER == 4 ? row : row / 3)) * kFxEX;
        const bool ok = MFWH_IDX(g.fault, i + 2 * lane + 1, 2 * kFxStep * ORDER * kFxEX);
        return reinterpret_cast<longlong2*>(edge + (ok ? i : 0)) + lane;
      };
      auto put_edges = [&](int buf) {
#pragma unroll
        for (int k = 0; k < 4; k += ORDER == 4 ? 1 : 3)
          *edge_row(buf, warp, k) = make_longlong2(w[k][0], w[k][1]);
      };
      // forced: the step's forcing, loaded while the step before ends
      int64_t fs[FORCED ? 4 : 1][2];
      auto load_force = [&](int s) {
        if constexpr (FORCED) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            longlong2 v = make_longlong2(0, 0);
            if ((in_mask >> (2 * k) & 3u) &&
                MFWH_IDX(g.fault, s * g.wpoints + base + k * g.syw + 1, 8 * g.wpoints))
              v = *reinterpret_cast<const longlong2*>(force + s * g.wpoints + base + k * g.syw);
            fs[k][0] = v.x;
            fs[k][1] = v.y;
          }
        }
      };
      // One step of the thread's points from the edge rows of buffer buf.  PLAIN: every point of
      // the warp is interior with one c^2; the values are the same.
      auto step_points = [&](int s, int buf, auto plain_c) {
        constexpr bool PLAIN = decltype(plain_c)::value;
        const int first = a.n0 + s == 0;
        const FxAxes one = a.coef[first][hi_mask & 1u];
        const FxAxes clo = PLAIN ? one : a.coef[first][0], chi = PLAIN ? one : a.coef[first][1];
        // the outermost rows have no neighbour warp: their values are never read
        const int wu = warp > 0 ? warp - 1 : 0, wb = warp < NW - 1 ? warp + 1 : warp;
        const longlong2 up = *edge_row(buf, wu, 3);
        const longlong2 bl = *edge_row(buf, wb, 0);
        const int64_t below[2] = {bl.x, bl.y};
        int64_t dv[2] = {fx_sub(w[0][0], up.x), fx_sub(w[0][1], up.y)};   // W - W_above of the row
        // fourth order: the same of the row above, and the second row below
        int64_t dv2[2] = {0, 0}, below2[2] = {0, 0};
        if constexpr (ORDER == 4) {
          const longlong2 up2 = *edge_row(buf, wu, 2), bl2 = *edge_row(buf, wb, 1);
          dv2[0] = fx_sub(up.x, up2.x);
          dv2[1] = fx_sub(up.y, up2.y);
          below2[0] = bl2.x;
          below2[1] = bl2.y;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int64_t left = __shfl_up_sync(0xffffffffu, w[k][1], 1);
          const int64_t right = __shfl_down_sync(0xffffffffu, w[k][0], 1);
          // W - W_left of columns 0 .. 2, fourth order also -1 and 3
          const int64_t dx[3] = {fx_sub(w[k][0], left), fx_sub(w[k][1], w[k][0]),
                                 fx_sub(right, w[k][1])};
          int64_t dxl = 0, dxr = 0;
          if constexpr (ORDER == 4) {
            dxl = fx_sub(left, __shfl_up_sync(0xffffffffu, w[k][0], 1));
            dxr = fx_sub(__shfl_down_sync(0xffffffffu, w[k][1], 1), right);
          }
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const int64_t dn = fx_sub(k < 3 ? w[k < 3 ? k + 1 : 3][c] : below[c], w[k][c]);
            int64_t dxx = fx_sub(dx[c + 1], dx[c]), dyy = fx_sub(dn, dv[c]);
            if constexpr (ORDER == 4) {
              // 16 times the first neighbours' sum of differences less the second neighbours', which
              // is dxx + (difference two to the right) - (two to the left)
              int64_t ra = c == 0 ? dx[2] : dxr, la = c == 0 ? dxl : dx[0];
              const int64_t w1 = k < 3 ? w[k < 3 ? k + 1 : 3][c] : below[c];
              const int64_t w2 = k < 2 ? w[k < 2 ? k + 2 : 3][c] : (k == 2 ? below[c] : below2[c]);
              int64_t ba = fx_sub(w2, w1), ab = dv2[c];
              if (!PLAIN) {   // a ghost value beyond the boundary is minus the centre's
                if (lx + c == ihx) ra = fx_sub(0, w[k][c]);
                if (lx + c == ilx) la = w[k][c];
                if (ly + k == ihy) ba = fx_sub(0, w[k][c]);
                if (ly + k == ily) ab = w[k][c];
              }
              dxx = fx_sub(fx_mul15(dxx), fx_sub(ra, la));
              dyy = fx_sub(fx_mul15(dyy), fx_sub(ba, ab));
              dv2[c] = dv[c];
            }
            dv[c] = dn;
            const bool upper = !PLAIN && (hi_mask >> (2 * k + c) & 1u);
            const FxAxes& L = upper ? chi : clo;
            int64_t dnew = d[k][c];
            if constexpr (ISO) {
              dnew = fx_mac(dnew, fx_add(dxx, dyy), L.x);
            } else {
              dnew = fx_mac(dnew, dxx, L.x);
              dnew = fx_mac(dnew, dyy, L.y);
            }
            if constexpr (FORCED) dnew = fx_sub(dnew, fs[k][c]);
            int64_t wnew = fx_add(w[k][c], dnew);
            if (!PLAIN && !(in_mask >> (2 * k + c) & 1u)) dnew = wnew = 0;
            d[k][c] = dnew;
            w[k][c] = wnew;
          }
        }
      };
      // (fourth order: not the rows next to the boundary, which have a ghost neighbour)
      const bool plain = __all_sync(0xffffffffu, in_mask == 0xFFu) &&
                         (ORDER == 2 || (y0 + ly > 1 && y0 + ly + 3 < g.ny - 1)) &&
                         (__all_sync(0xffffffffu, hi_mask == 0u) ||
                          __all_sync(0xffffffffu, hi_mask == 0xFFu));
      load_force(0);
      put_edges(0);
      fx_bar_sync(kBarStep, 32 * NW);
      if (it >= 2) fx_bar_sync(kBarEmpty + (it & 1), threads);   // the buffer's sums are made
      for (int s = 0; s < a.steps; ++s) {
        const int r = REACH * (a.steps - 1 - s);   // later steps read the owned points grown by r
        if (ly + 3 >= T - r && ly < T + VY + r) {
          if (plain)
            step_points(s, s & 1, std::true_type{});
          else
            step_points(s, s & 1, std::false_type{});
          if (r > 0) {
            load_force(s + 1);
            put_edges((s + 1) & 1);
          }
          if (owner) {
            const int i = s * kFxTile + (ly - T) * VX + lx - T;
            int2* h = hist + i;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              if (!MFWH_IDX(g.fault, i + k * VX + 1, STEPS * kFxTile)) continue;
              const int2 p = fx_level_digits(w[k][0]), r2 = fx_level_digits(w[k][1]);
              *reinterpret_cast<int4*>(h + k * VX) = make_int4(p.x, p.y, r2.x, r2.y);
            }
          }
        }
        fx_bar_sync(kBarStep, 32 * NW);
      }
      fx_bar_arrive(kBarFull + (it & 1), threads);
      if (owner && !a.last && x0 + lx < g.syw) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int64_t o = base + k * g.syw;
          if (ly + k > ghy || !MFWH_IDX(g.fault, o, g.wpoints) ||
              !MFWH_IDX(g.fault, o + 1, g.wpoints))
            continue;
          *reinterpret_cast<longlong2*>(out.W + o) = make_longlong2(w[k][0], w[k][1]);
          *reinterpret_cast<longlong2*>(out.D + o) = make_longlong2(d[k][0], d[k][1]);
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            mw = max(mw, abs((int)(w[k][c] >> 32)));
            md = max(md, abs((int)(d[k][c] >> 32)));
          }
        }
      }
    }
    // |W| <= (mw + 1) 2^32
    mw = __reduce_max_sync(0xffffffffu, mw);
    md = __reduce_max_sync(0xffffffffu, md);
    if (lane == 0 && !a.last) {
      atomicMax(&s_out->wmax, (unsigned long long)(mw + 1) << 32);
      atomicMax(&s_out->dmax, (unsigned long long)(md + 1) << 32);
    }
    // the sums of the last tiles
    for (int i = it < 2 ? 0 : it - 2; i < it; ++i) fx_bar_sync(kBarEmpty + (i & 1), threads);
  } else {
    // ---- tail warps: the filter sums of the owned points
    const int t0 = tid - 32 * NW;
    constexpr int MG = NF <= 4 ? NF : 4;   // frequencies at a time (registers)
    // Ask L2 for a tile's sums and levels.
    auto prefetch = [&](int tile) {
      const int64_t* qt = q + (int64_t)tile * NF * kFxTile;
      for (int i = t0 * 16; i < NF * kFxTile; i += 32 * kFxTail * 16) if (i % kFxTile < VX * VY) fx_prefetch(qt + i);
      const int64_t x0 = (int64_t)(tile % tiles_x) * VX - T, y0 = (int64_t)(tile / tiles_x) * VY - T;
      for (int i = t0; i < 2 * EY * 4; i += 32 * kFxTail) {
        const int64_t y = y0 + (i >> 2) % EY, x = x0 + (i & 3) * 16;
        if (y >= 0 && y <= g.ny && x >= 0 && x < g.syw)
          fx_prefetch((i < EY * 4 ? in.W : in.D) + y * g.syw + x);
      }
    };
    int it = 0;
    if ((int)blockIdx.x < tiles) prefetch(blockIdx.x);
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++it) {
      const int2* hist = reinterpret_cast<const int2*>(fx_smem + (it & 1) * kHist);
      int64_t* qt = q + (int64_t)tile * NF * kFxTile;
      // the sums are loaded one group of MG frequencies ahead
      int64_t qm[MG], qn[MG];
      auto in_sums = [&](const int64_t* p) {
        return MFWH_IDX(g.fault, p - q, (int64_t)tiles * NF * kFxTile);
      };
      auto load = [&](const int64_t* p, int m0, int64_t* v) {
#pragma unroll
        for (int j = 0; j < MG; ++j)
          if (m0 + j < NF && in_sums(p + (m0 + j) * kFxTile)) v[j] = p[(m0 + j) * kFxTile];
      };
      load(qt + t0, 0, qm);
      if (tile + (int)gridDim.x < tiles) prefetch(tile + (int)gridDim.x);
      fx_bar_sync(kBarFull + (it & 1), threads);
      if (!zero) {
        for (int i = t0; i < VX * VY; i += 32 * kFxTail) {
          int64_t* qi = qt + i;
          const int64_t* qnext = i + 32 * kFxTail < VX * VY ? qi + 32 * kFxTail : qi;
#pragma unroll
          for (int m0 = 0; m0 < NF; m0 += MG) {
            if (m0 + MG < NF)
              load(qi, m0 + MG, qn);
            else
              load(qnext, 0, qn);
            FxSum S[MG];
            float r[MG];   // the weights' low digits times the levels' high ones, / 2^32
#pragma unroll
            for (int j = 0; j < MG; ++j)
              if (m0 + j < NF) {
                S[j] = FxSum{s_off[m0 + j], a.off2[m0 + j]};
                r[j] = 0.0f;
              }
            auto add = [&](int s) {
              if (!MFWH_IDX(g.fault, s * kFxTile + i, STEPS * kFxTile)) return;
              const int2 v = hist[s * kFxTile + i];
              const float vf = (float)v.x;
#pragma unroll
              for (int j = 0; j < MG; ++j)
                if (m0 + j < NF) {
                  const int e = s * NF + m0 + j;
                  fx_madd(S[j], a.wh[e], v);
                  r[j] = fmaf(a.wl[e], vf, r[j]);
                }
            };
            if (a.steps == STEPS) {
#pragma unroll
              for (int s = 0; s < STEPS; ++s) add(s);
            } else {
#pragma unroll 1
              for (int s = 0; s < a.steps; ++s) add(s);
            }
#pragma unroll
            for (int j = 0; j < MG; ++j)
              if (m0 + j < NF) {
                int64_t c = S[j].s1 + (S[j].s2 >> 32) + __float2int_rn(r[j]), v = qm[j];
                if (wide)   // (below half a unit from 62 on)
                  c = q_new < 62 ? (c >> 32) >> (q_new - 32) : 0;
                else
                  c = (int64_t)((uint64_t)(uint32_t)(c >> 32 >> q_new) << 32 |
                                __funnelshift_r((uint32_t)c, (uint32_t)(c >> 32), q_new));
                if (q_old != 0) v = fx_rescale(v, -q_old);
                if (in_sums(qi + (m0 + j) * kFxTile)) qi[(m0 + j) * kFxTile] = fx_add(v, c);
              }
#pragma unroll
            for (int j = 0; j < MG; ++j) qm[j] = qn[j];
          }
        }
      }
      if (a.last) {
        const int64_t x1 = (int64_t)(tile % tiles_x) * VX, y1 = (int64_t)(tile / tiles_x) * VY;
        for (int i = t0; i < VX * VY; i += 32 * kFxTail) {
          const int64_t x = x1 + i % VX, y = y1 + i / VX;
          if (x > g.nx || y > g.ny || !MFWH_IDX(g.fault, y * g.sy + x, g.points) ||
              !in_sums(qt + (NF - 1) * kFxTile + i))
            continue;
          const bool is = x > 0 && x < g.nx && y > 0 && y < g.ny;
          fx_finish<NF>(qt + i, s_unit, is, vout, vsub, a, g.points, y * g.sy + x);
        }
      }
      fx_bar_arrive(kBarEmpty + (it & 1), threads);
    }
  }
}

// A float not below v.
inline float fx_up(double v) {
  const float f = (float)v;
  return (double)f < v ? std::nextafter(f, 3e38f) : f;
}

// Coefficient of f_m in the step from level n.
inline double fx_forcing_coef(const FxHost& h, int n, int nf, int m) {
  return (n == 0 ? 0.5 * h.dt2 : h.dt2) * h.cos_host[(size_t)n * nf + m];
}

// ---- host launchers ------------------------------------------------------------------------

template <int NF, bool ISO, bool FORCED, int ORDER>
void fx_launch(const Geom& g, const FxArrays& in, const FxArrays& out, int64_t* q, double* vout,
               const double* vsub, const FxHost& h, cudaStream_t st) {
  constexpr size_t smem = fx_smem_bytes(ORDER);
  static int sms[64] = {};   // SMs of the device; the attribute is set on first use
  int dev = 0;
  cudaGetDevice(&dev);
  int n = (dev >= 0 && dev < 64) ? sms[dev] : 0;
  if (n == 0) {
    cudaFuncSetAttribute(k_fx2d<NF, ISO, FORCED, ORDER>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)smem);
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1)
      n = 1;
    if (dev >= 0 && dev < 64) sms[dev] = n;
  }
  FxArgs<NF> a;
  for (int i = 0; i < 2; ++i)
    for (int j = 0; j < 2; ++j) {
      a.coef[i][j].x = h.cx[i][j];
      a.coef[i][j].y = h.cy[i][j];
      a.lay[i][j] = h.lay[i][j];
    }
  a.n0 = h.n0;
  a.steps = h.steps;
  a.forced = h.forced;
  a.last = h.last;
  a.gw = fx_up(h.gw);
  a.gd = fx_up(h.gd);
  a.warps = h.warps;
  a.wsum = h.wsum;
  a.subtract = vsub == nullptr ? 0 : (h.add ? -1 : 1);
  a.has_e = h.has_e && h.vprev != nullptr;
  a.vprev = h.vprev;
  for (int m = 0; m < NF; ++m) {
    a.wexp[m] = h.wexp[m];
    for (int j = 0; j < NF; ++j) {
      a.binv[m * NF + j] = h.binv[m * MFWH_MAX_NF + j];
      a.emat[m * NF + j] = h.emat[m * MFWH_MAX_NF + j];
    }
    // the sums start with the constant 2^31 of the level digits times the weights (in units of
    // 2^32: half their sum) and half a unit of 2^64
    int64_t sum = 0;
    for (int s = 0; s < h.steps; ++s) sum += h.wint[(size_t)(h.n0 + s + 1) * NF + m];
    a.off1[m] = sum >> 33;
    a.off2[m] = ((sum >> 1) & 0xFFFFFFFFll) + ((int64_t)1 << 31);
  }
  for (int s = 0; s < kFxT; ++s)
    for (int m = 0; m < NF; ++m) {
      const int k = h.n0 + s, i = s * NF + m;
      const bool is = s < h.steps;
      int lo;
      fx_digits(is ? h.wint[(size_t)(k + 1) * NF + m] : 0, a.wh[i], lo);
      a.wl[i] = (float)lo * 0x1p-32f;
      a.wd[i] = is ? h.wq_host[(size_t)(k + 1) * NF + m] : 0.0;
      a.fc[i] = is && h.forced ? fx_forcing_coef(h, k, NF, m) : 0.0;
    }
  const int64_t tx = (g.nx + kFxVX) / kFxVX, tiles = fx_tiles(g.nx, g.ny, h.warps);
  const int L = h.n0 / fx_launch_steps(ORDER);
  launch_dependent(k_fx2d<NF, ISO, FORCED, ORDER>, dim3((unsigned)(tiles < n ? tiles : n)),
                   dim3(32 * (h.warps + kFxTail)), smem, st, in, out, h.f, h.force, q, vout, vsub, a,
                   h.scale, h.state + L % 3, h.state + (L + 1) % 3, h.state + (L + 2) % 3, g, (int)tx,
                   (int)tiles);
}

template <int NF>
void fx_launch_nf(const Geom& g, const FxArrays& in, const FxArrays& out, int64_t* q, double* vout,
                  const double* vsub, const FxHost& h, cudaStream_t st) {
  auto go = [&](auto iso, auto order) {
    constexpr bool I = decltype(iso)::value;
    constexpr int O = decltype(order)::value;
    if (h.forced)
      fx_launch<NF, I, true, O>(g, in, out, q, vout, vsub, h, st);
    else
      fx_launch<NF, I, false, O>(g, in, out, q, vout, vsub, h, st);
  };
  if (g.order == 4)
    go(std::false_type{}, std::integral_constant<int, 4>{});
  else if (h.iso)
    go(std::true_type{}, std::integral_constant<int, 2>{});
  else
    go(std::false_type{}, std::integral_constant<int, 2>{});
}

}  // namespace

using FxFn = void (*)(const Geom&, const FxArrays&, const FxArrays&, int64_t*, double*,
                      const double*, const FxHost&, cudaStream_t);
FxFn fx_fn_p1(int nf);   // wave_fx_p1.cu: 1-3 frequencies
FxFn fx_fn_p2(int nf);   // wave_fx_p2.cu: 4-6
FxFn fx_fn_p3(int nf);   // wave_fx_p3.cu: 7-8
FxFn fx_fn_p4(int nf);   // wave_fx_p4.cu: 9-11
FxFn fx_fn_p5(int nf);   // wave_fx_p5.cu: 12-14
FxFn fx_fn_p6(int nf);   // wave_fx_p6.cu: 15-16

}  // namespace mfwh
