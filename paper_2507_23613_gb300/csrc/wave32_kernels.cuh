// FP32 MFWH wave solve with compensated filter sums, sm_103a.
//
// The wave levels are FP32 and the leapfrog scheme (eq. WaveSchemeA, first step
// eq. implicitFirstStep with alpha = 0) is advanced in its increment form
//   D^{n+1/2} = D^{n-1/2} + kappa_n (c^2 Delta_h W^n - F^n),   W^{n+1} = W^n + D^{n+1/2},
// with D^{-1/2} = 0, kappa_0 = dt^2/2 and kappa_n = dt^2 otherwise.  In exact
// arithmetic this is the same recurrence as W^{n+1} = 2W^n - W^{n-1} + ...; in
// FP32 it keeps the velocity D exactly where the two-level form would round it,
// so a rounding of W^{n+1} stays a position error instead of turning into a
// velocity error that grows over the N_t steps.  The Laplacian is taken as sums
// of neighbour differences, (W_e - W) + (W_w - W), which are small and nearly
// exact for smooth fields.
//
// The filter sums q_m = sum_n w_{n,m} W^n (eq. pDefQ) are accumulated in FP32
// with Kahan's compensated summation: a pair (s_m, c_m) per point and frequency,
// q_m = s_m - c_m.  The filter solve V = B^{-1} q (eq. waveHoltzMatrixIteration)
// and everything after it are FP64.
//
// Four kernels advance the scheme:
//  * k_tb2d32: 2D, T steps per launch on overlapped tiles whose points, halo included, live
//    in the registers of one CTA for all T steps;
//  * k_ring2d32: the same on smaller tiles in shared memory, for grids of few tiles;
//  * k_tb3d32: the same in 3D with T = 2 or 4;
//  * k_step32 / k_last32: one step per launch, 2D or 3D, second- or fourth-order L_h.
// All are dependent launches (launch_dependent): one step on 33^3, N_f = 2, took 4.3 us, now 2.6.
// (k_step32 releases the next one at its end, for the reason that k_step does.)
// All perform the same FP32 operations per point in the same order, so their
// results are bit-identical.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "kernels.h"

namespace mfwh {

// The four host launchers of one frequency count, collected so that the
// translation units wave32_p1.cu .. wave32_p8.cu can each instantiate two counts.
struct W32Ops {
  void (*init)(const Geom&, const double*, float*, float*, float*, const float*, cudaStream_t);
  void (*step)(const Geom&, const float*, const float*, float*, float*, const float*, float*,
               float*, const Step32Host&, cudaStream_t);
  void (*last)(const Geom&, const float*, const float*, const float*, const float*, const float*,
               double*, const double*, const Step32Host&, const StepHost&, cudaStream_t);
  void (*tb)(const Geom&, const float*, const float*, float*, float*, const float*, float*, float*,
             double*, const double*, const TB32Host&, cudaStream_t);
};

namespace {

// Epilogue V^{k+1} = C q + E V^k (E != 0 only for the explicit filter).
template <int NF>
struct Last32Binv {
  double binv[NF * NF];      // C
  double emat[NF * NF];      // E
  const double* vprev;       // V^k
  int has_e;
};

template <int NF>
struct Init32Args {
  float w0[NF];
};

template <int NF>
struct Step32Args {
  Coef32 lo, hi;
  float fc[NF];     // kappa_n cos(omega~_m t^n)
  float wq[NF];     // w_{n+1,m}
  int forced;
  int group;        // sums: 0 Kahan, else partial over several steps, 1 the first, 2 the last, 3 both
  float* part;      // [NF][points] partial sums
};

__device__ __forceinline__ bool interior2(int64_t gx, int64_t gy, const Geom& g) {
  return gx > 0 && gx < g.nx && gy > 0 && gy < g.ny;
}

__device__ __forceinline__ void kahan_add(float& s, float& c, float w, float x) {
  const float y = fmaf(w, x, -c);
  const float t = s + y;
  c = (t - s) - y;
  s = t;
}

// Fold a partial sum x into the Kahan pair (s, c).
__device__ __forceinline__ void kahan_fold(float& s, float& c, float x) {
  const float y = x - c;
  const float t = s + y;
  c = (t - s) - y;
  s = t;
}

// kappa c^2 Delta_h W at a point whose neighbour sums of differences are dxx, dyy, dzz, minus
// the forcing (f is laid out like the wave levels, q the point's index there); same order in
// every kernel.
template <int NF, int DIM>
__device__ __forceinline__ float increment(const Coef32& L, float dxx, float dyy, float dzz,
                                           const float* fc, const float* __restrict__ f,
                                           int64_t q, int64_t wpoints, int forced) {
  float inc = L.Ay * dyy;
  if (DIM == 3) inc = fmaf(L.Az, dzz, inc);
  inc = fmaf(L.Ax, dxx, inc);
  if (forced) {
#pragma unroll
    for (int m = 0; m < NF; ++m) inc = fmaf(-fc[m], f[m * wpoints + q], inc);
  }
  return inc;
}

// ---- one step per launch (2D and 3D) -------------------------------------------

constexpr int kBX = 32, kBY = 8;

template <int DIM>
__device__ __forceinline__ bool index_of(const Geom& g, int64_t& i, int64_t& j, int64_t& k,
                                         int64_t& p, bool& interior) {
  i = (int64_t)blockIdx.x * kBX + threadIdx.x;
  j = (int64_t)blockIdx.y * kBY + threadIdx.y;
  k = DIM == 3 ? (int64_t)blockIdx.z : 0;
  const bool inside = i <= g.nx && j <= g.ny;
  p = k * g.sz + j * g.sy + i;
  interior = inside && i > 0 && i < g.nx && j > 0 && j < g.ny &&
             (DIM == 2 || (k > 0 && k < g.nz));
  return inside;
}

// Fourth-order combination 16 d1 - d2 along one axis at index idx of n cells, from the
// first-neighbour difference sum d1 and the second neighbours (ghost values beyond the
// boundary are minus the centre value, so their difference is -2w).
__device__ __forceinline__ float comb4(const float* W, int64_t p, int64_t s, int64_t idx,
                                       int64_t n, float w, float d1) {
  const float dm = idx == 1 ? -2.0f * w : W[p - 2 * s] - w;
  const float dp = idx == n - 1 ? -2.0f * w : W[p + 2 * s] - w;
  return fmaf(16.0f, d1, -(dm + dp));
}

// Index of grid point (i, j, k) in the wave-level arrays W and D (padded rows in 2D).
__device__ __forceinline__ int64_t wpos(const Geom& g, int64_t i, int64_t j, int64_t k) {
  return k * g.szw + j * g.syw + i;
}

template <int NF, int DIM, int ORDER>
__device__ __forceinline__ void step_point(const float* W, const float* D,
                                           const float* __restrict__ f, const Step32Args<NF>& a,
                                           const Geom& g, int64_t i, int64_t j, int64_t k,
                                           float& wn, float& dn) {
  const int64_t li = g.layer_axis == 0 ? i : (g.layer_axis == 1 ? j : k);
  const Coef32& L = li >= g.layer_split ? a.hi : a.lo;
  const int64_t q = wpos(g, i, j, k);
  const float w = W[q];
  float dxx = (W[q - 1] - w) + (W[q + 1] - w);
  float dyy = (W[q - g.syw] - w) + (W[q + g.syw] - w);
  float dzz = DIM == 3 ? (W[q - g.szw] - w) + (W[q + g.szw] - w) : 0.0f;
  if (ORDER == 4) {
    dxx = comb4(W, q, 1, i, g.nx, w, dxx);
    dyy = comb4(W, q, g.syw, j, g.ny, w, dyy);
    if (DIM == 3) dzz = comb4(W, q, g.szw, k, g.nz, w, dzz);
  }
  const float inc = increment<NF, DIM>(L, dxx, dyy, dzz, a.fc, f, q, g.wpoints, a.forced);
  dn = (D ? D[q] : 0.0f) + inc;
  wn = w + dn;
}

// The term of one step added to the pair (s, c), or (a.group) to the partial sum of the steps of one
// launch of the blocked kernels, which the last of them folds into the pair: the same operations as
// theirs.  Returns whether the pair has changed; a partial sum that goes on is in t.
template <int NF>
__device__ __forceinline__ bool add_term(float& s, float& c, float& t, const Step32Args<NF>& a,
                                         int m, int64_t o, float wn) {
  if (a.group == 0) {
    kahan_add(s, c, a.wq[m], wn);
    return true;
  }
  t = fmaf(a.wq[m], wn, (a.group & 1) ? 0.0f : a.part[o]);
  if (!(a.group & 2)) return false;
  kahan_fold(s, c, t);
  return true;
}

// W_out = W + D', D' = D + increment (D_out may alias D_in; W_out must not alias W_in); sums
// updated in place.
// GROUP: partial sums (a.group not 0).
template <int NF, int DIM, int ORDER, bool GROUP>
__global__ void __launch_bounds__(kBX * kBY)
k_step32(const float* W, const float* D_in, float* __restrict__ W_out, float* D_out,
         const float* __restrict__ f, float* __restrict__ qs, float* __restrict__ qc,
         const Step32Args<NF> a, const Geom g) {
  pdl_wait();
  int64_t i, j, k, p;
  bool interior;
  index_of<DIM>(g, i, j, k, p, interior);
  if (!interior) return;
  float wn, dn;
  step_point<NF, DIM, ORDER>(W, D_in, f, a, g, i, j, k, wn, dn);
  W_out[wpos(g, i, j, k)] = wn;
  D_out[wpos(g, i, j, k)] = dn;
#pragma unroll
  for (int m = 0; m < NF; ++m) {
    const int64_t o = m * g.points + p;
    if constexpr (GROUP) {
      float s = 0.0f, c = 0.0f, t = 0.0f;
      if (a.group & 2) {
        s = qs[o];
        c = qc[o];
      }
      if (add_term(s, c, t, a, m, o, wn)) {
        qs[o] = s;
        qc[o] = c;
      } else {
        a.part[o] = t;
      }
    } else {
      float s = qs[o], c = qc[o];
      kahan_add(s, c, a.wq[m], wn);
      qs[o] = s;
      qc[o] = c;
    }
  }
  pdl_release();
}

template <int NF>
__device__ __forceinline__ void filter_solve_out(const float* s, const float* c,
                                                 const Last32Binv<NF>& b, int subtract,
                                                 const double* vsub, double* vout,
                                                 int64_t p, int64_t points, bool interior) {
  double qd[NF], vk[NF];
#pragma unroll
  for (int m = 0; m < NF; ++m) {
    qd[m] = (double)s[m] - (double)c[m];
    vk[m] = (b.has_e && interior) ? b.vprev[m * points + p] : 0.0;
  }
#pragma unroll
  for (int m = 0; m < NF; ++m) {
    double acc = 0.0;
#pragma unroll
    for (int j = 0; j < NF; ++j) acc = fma(b.binv[m * NF + j], qd[j], acc);
    if (b.has_e) {
#pragma unroll
      for (int j = 0; j < NF; ++j) acc = fma(b.emat[m * NF + j], vk[j], acc);
    }
    double val = 0.0;
    if (interior) val = subtract ? vsub[m * points + p] - acc : acc;
    vout[m * points + p] = val;
  }
}

template <int NF, int DIM, int ORDER>
__global__ void __launch_bounds__(kBX * kBY)
k_last32(const float* W, const float* D, const float* __restrict__ f,
         const float* qs, const float* qc, double* vout,
         const double* vsub, const Step32Args<NF> a, const Last32Binv<NF> b, int subtract,
         const Geom g) {
  pdl_begin();
  int64_t i, j, k, p;
  bool interior;
  if (!index_of<DIM>(g, i, j, k, p, interior)) return;
  float s[NF], c[NF];
#pragma unroll
  for (int m = 0; m < NF; ++m) s[m] = c[m] = 0.0f;
  if (interior) {
    float wn, dn;
    step_point<NF, DIM, ORDER>(W, D, f, a, g, i, j, k, wn, dn);
#pragma unroll
    for (int m = 0; m < NF; ++m) {
      s[m] = qs[m * g.points + p];
      c[m] = qc[m * g.points + p];
      float t;
      add_term(s[m], c[m], t, a, m, m * g.points + p, wn);   // (a last step ends its group)
    }
  }
  filter_solve_out<NF>(s, c, b, subtract, vsub, vout, p, g.points, interior);
}

// ---- temporally blocked 2D kernel ----------------------------------------------
//
// One CTA per SM (16 warps) holds an extended tile of 128 x 64 points (fewer rows where the grid
// would leave SMs idle: rt_warps) in registers, W and D of 4 x 4 points per thread: lane l has
// columns 4l .. 4l + 3, warp w rows 4w .. 4w + 3.  Every step updates all of them (the outermost
// ring of valid values shrinks by one point a step, so after T steps the (128 - 2T) x (64 - 2T)
// points in the middle are exact), except that a warp rests
// once no later step reads its rows.  Left and right neighbours come from the thread itself or by
// one shuffle per row and side, vertical neighbours from the thread itself or, above and below
// its four rows, from the edge rows that the warps exchange through shared memory (double
// buffered: one barrier per step).  A step of a point is 8 FP32 operations (each neighbour
// difference is formed once and serves both of its points: W_w - W at a point is exactly minus
// W_e - W at its left neighbour) plus about 1.5 instructions of exchange, with no index
// arithmetic and no per-point tests away from the boundary.  (The form it replaces, 32 x 32 tiles
// with the halo ring in shared memory and a flat index over it, issued 169 instructions per
// point-step at N_f = 5, this one 58: 30.1 against 19.2 ms for a map on 2049^2, N_f = 5, depth 16,
// 1717 steps.)
//
// The filter sums are not touched while stepping.  Each step stores the owned points' new values
// in shared memory (T x 4 bytes per owned point: 192 KB of the 227 KB, which sets the tile);
// after the last step every thread takes owned points one by one, reads their T values back and
// updates all N_f sums in registers, in step order, with the weights as constant operands.
//   ACC = 0: Kahan update of (s_m, c_m) at every step.
//   ACC = 1: plain FP32 partial sums over the steps of one launch, folded into the Kahan
//            pair once per launch (compensated across launches; the partial of at most T
//            terms carries a rounding error far below that of the FP32 wave levels).
constexpr int kRtWarps = 16, kRtThreads = 32 * kRtWarps;
constexpr int kRtEX = 128, kRtEY = 64;    // extended tile

template <int NF, int T>
struct RT32Args {
  Coef32 reg_lo, reg_hi, first_lo, first_hi;
  int n0, steps, forced, last, subtract;
  int warps;          // that step: the tile has 4 warps rows (k_tb2d32)
  float wq[T * NF];   // w_{n+1,m} of step s: [s * NF + m]
  float fc[T * NF];   // kappa_n cos(omega~_m t^n)
};

template <int T>
constexpr size_t rt32_smem_bytes() {
  return sizeof(float) * ((size_t)T * (kRtEX - 2 * T) * (kRtEY - 2 * T) +
                          (size_t)2 * kRtWarps * 2 * kRtEX);
}

// FULL: all kRtWarps warps step (with their number at run time the loop over the sums is 4 to 20 %
// slower above 6 frequencies: 769^2, N_f = 16, depth 16, partial sums, 82 us a launch and 91).
template <int NF, int T, int ACC, bool FULL>
__global__ void __launch_bounds__(kRtThreads, 1)
k_tb2d32(const float* W_in, const float* D_in,
         float* __restrict__ W_out, float* __restrict__ D_out, const float* __restrict__ f,
         float* __restrict__ qs, float* __restrict__ qc, double* vout, const double* vsub,
         const __grid_constant__ RT32Args<NF, T> a, const __grid_constant__ Last32Binv<NF> b,
         const Geom g) {
  pdl_begin();
  constexpr int VX = kRtEX - 2 * T, VYM = kRtEY - 2 * T;   // owned columns, rows at most
  static_assert(T % 4 == 0 && VX > 0 && VYM > 0, "owned points are whole 4 x 4 blocks");
  const int warps = FULL ? kRtWarps : a.warps;             // that step
  const int VY = 4 * warps - 2 * T;                        // owned rows
  extern __shared__ __align__(16) float sm32[];
  float* hist = sm32;                       // [T][VYM][VX] owned values step by step
  float* edge = sm32 + T * VX * VYM;        // [2][warp][top, bottom][128] edge rows
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t x0 = (int64_t)blockIdx.x * VX - T, y0 = (int64_t)blockIdx.y * VY - T;
  const int lx = 4 * lane, ly = 4 * warp;
  const int64_t gx = x0 + lx, gy = y0 + ly;   // this thread's first point
  const bool owner = lx >= T && lx < T + VX && ly >= T && ly < T + VY;
  const bool lay_x = g.layer_axis == 0;
  // the thread's points: interior (bit 4k + c of in_mask), upper layer (of hi_mask)
  unsigned in_mask = 0, hi_mask = 0;
  float w[4][4], d[4][4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int64_t y = gy + k;
    const bool row = warp < warps && y >= 0 && y <= g.ny;
    const int64_t base = y * g.syw + gx;
    if (row && gx >= 0 && gx + 3 <= g.nx) {
      const float4 v = *reinterpret_cast<const float4*>(W_in + base);
      w[k][0] = v.x; w[k][1] = v.y; w[k][2] = v.z; w[k][3] = v.w;
      float4 u = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (D_in != nullptr) u = *reinterpret_cast<const float4*>(D_in + base);
      d[k][0] = u.x; d[k][1] = u.y; d[k][2] = u.z; d[k][3] = u.w;
    } else {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const bool in = row && gx + c >= 0 && gx + c <= g.nx;
        w[k][c] = in ? W_in[base + c] : 0.0f;
        d[k][c] = (in && D_in != nullptr) ? D_in[base + c] : 0.0f;
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int64_t x = gx + c;
      if (x > 0 && x < g.nx && y > 0 && y < g.ny) in_mask |= 1u << (4 * k + c);
      if ((lay_x ? x : y) >= g.layer_split) hi_mask |= 1u << (4 * k + c);
    }
  }
  // Ask L2 for the sums that the end of the launch updates (an owner's rows of 4 points).
  if (owner) {
    for (int e = 0; e < 2 * NF; ++e) {
      const float* base = (e & 1 ? qc : qs) + (int64_t)(e >> 1) * g.points;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if ((in_mask >> (4 * k) & 1u) && (lane & 3) == 0)   // one request per 64 bytes
          asm volatile("prefetch.global.L2 [%0];" ::"l"(base + (gy + k) * g.sy + gx));
    }
  }
  auto edge_row = [&](int buf, int wp, int which) {
    return reinterpret_cast<float4*>(edge + ((buf * kRtWarps + wp) * 2 + which) * kRtEX) + lane;
  };
  auto put_edges = [&](int buf) {
    *edge_row(buf, warp, 0) = make_float4(w[0][0], w[0][1], w[0][2], w[0][3]);
    *edge_row(buf, warp, 1) = make_float4(w[3][0], w[3][1], w[3][2], w[3][3]);
  };
  // One step of the thread's points from the edge rows of buffer buf.  PLAIN: every point is
  // interior with one c^2 (a whole warp's); the values are the same.
  auto step_points = [&](int s, int buf, auto plain_c, auto forced_c) {
    constexpr bool PLAIN = decltype(plain_c)::value, FORCED = decltype(forced_c)::value;
    const bool first = a.n0 + s == 0;
    const Coef32 lo = first ? a.first_lo : a.reg_lo;
    const Coef32 hi = first ? a.first_hi : a.reg_hi;
    const Coef32 one = (hi_mask & 1) ? hi : lo;
    // the outermost rows have no neighbour warp: their values are never read
    const float4 u4 = *edge_row(buf, warp > 0 ? warp - 1 : 0, 1);
    const float4 b4 = *edge_row(buf, warp < kRtWarps - 1 ? warp + 1 : warp, 0);
    const float up[4] = {u4.x, u4.y, u4.z, u4.w}, below[4] = {b4.x, b4.y, b4.z, b4.w};
    // W - W_above of the current row; row k + 1's is taken before row k is overwritten
    float dv[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) dv[c] = w[0][c] - up[c];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float left = __shfl_up_sync(0xffffffffu, w[k][3], 1);
      const float right = __shfl_down_sync(0xffffffffu, w[k][0], 1);
      float dx[5];   // W - W_left of columns 0 .. 4
      dx[0] = w[k][0] - left;
#pragma unroll
      for (int c = 1; c < 4; ++c) dx[c] = w[k][c] - w[k][c - 1];
      dx[4] = right - w[k][3];
      float inc[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float wc = w[k][c];
        const float dn = (k < 3 ? w[k < 3 ? k + 1 : 3][c] : below[c]) - wc;
        const float dxx = dx[c + 1] - dx[c];   // (W_w - W) + (W_e - W)
        const float dyy = dn - dv[c];
        dv[c] = dn;
        const bool upper = hi_mask >> (4 * k + c) & 1u;
        const float Ax = PLAIN ? one.Ax : (upper ? hi.Ax : lo.Ax);
        const float Ay = PLAIN ? one.Ay : (upper ? hi.Ay : lo.Ay);
        inc[c] = Ay * dyy;
        inc[c] = fmaf(Ax, dxx, inc[c]);
      }
      if constexpr (FORCED) {
        if (in_mask >> (4 * k) & 15u) {   // rows of f are padded like those of W
          const float* fp = f + (gy + k) * g.syw + gx;
#pragma unroll 4
          for (int m = 0; m < NF; ++m) {
            const float4 v = *reinterpret_cast<const float4*>(fp + m * g.wpoints);
            const float fc = a.fc[s * NF + m];
            inc[0] = fmaf(-fc, v.x, inc[0]);
            inc[1] = fmaf(-fc, v.y, inc[1]);
            inc[2] = fmaf(-fc, v.z, inc[2]);
            inc[3] = fmaf(-fc, v.w, inc[3]);
          }
        }
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float dnew = d[k][c] + inc[c];
        const float wnew = w[k][c] + dnew;
        const bool in = PLAIN || (in_mask >> (4 * k + c) & 1u);
        d[k][c] = in ? dnew : 0.0f;   // boundary and outside points keep W = 0
        w[k][c] = in ? wnew : 0.0f;
      }
    }
  };
  const bool plain = __all_sync(0xffffffffu, in_mask == 0xFFFFu) &&
                     (__all_sync(0xffffffffu, hi_mask == 0u) ||
                      __all_sync(0xffffffffu, hi_mask == 0xFFFFu));
  put_edges(0);
  __syncthreads();
  for (int s = 0; s < a.steps; ++s) {
    const int r = a.steps - 1 - s;   // later steps read the owned points grown by r
    if (ly + 3 >= T - r && ly < T + VY + r) {
      if (a.forced)
        step_points(s, s & 1, std::false_type{}, std::true_type{});
      else if (plain)
        step_points(s, s & 1, std::true_type{}, std::false_type{});
      else
        step_points(s, s & 1, std::false_type{}, std::false_type{});
      put_edges((s + 1) & 1);
      if (owner) {
        float* h = hist + (size_t)s * VX * VYM + (ly - T) * VX + lx - T;
#pragma unroll
        for (int k = 0; k < 4; ++k)
          *reinterpret_cast<float4*>(h + k * VX) =
              make_float4(w[k][0], w[k][1], w[k][2], w[k][3]);
      }
    }
    __syncthreads();
  }
  if (owner && !a.last) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (gy + k > g.ny || gx >= g.syw) continue;
      const int64_t base = (gy + k) * g.syw + gx;
      *reinterpret_cast<float4*>(W_out + base) = make_float4(w[k][0], w[k][1], w[k][2], w[k][3]);
      *reinterpret_cast<float4*>(D_out + base) = make_float4(d[k][0], d[k][1], d[k][2], d[k][3]);
    }
  }
  // The filter sums of the owned points.
  for (int i = tid; i < VX * VY; i += kRtThreads) {
    const int ry = i / VX, rx = i - ry * VX;
    const int64_t x = x0 + T + rx, y = y0 + T + ry;
    const bool in = x > 0 && x < g.nx && y > 0 && y < g.ny;
    if (!in && !(a.last && x <= g.nx && y <= g.ny)) continue;
    const int64_t p = y * g.sy + x;
    float ks[NF], kc[NF];
#pragma unroll
    for (int m = 0; m < NF; ++m) {
      ks[m] = in ? qs[m * g.points + p] : 0.0f;
      kc[m] = in ? qc[m * g.points + p] : 0.0f;
    }
    if (in) {
      float part[ACC == 1 ? NF : 1];
      if constexpr (ACC == 1) {
#pragma unroll
        for (int m = 0; m < NF; ++m) part[m] = 0.0f;
      }
      auto add = [&](int s, float v) {
#pragma unroll
        for (int m = 0; m < NF; ++m) {
          if constexpr (ACC == 1)
            part[m] = fmaf(a.wq[s * NF + m], v, part[m]);
          else
            kahan_add(ks[m], kc[m], a.wq[s * NF + m], v);
        }
      };
      if (a.steps == T) {
#pragma unroll
        for (int s = 0; s < T; ++s) add(s, hist[s * VX * VYM + i]);
      } else {
#pragma unroll 1
        for (int s = 0; s < a.steps; ++s) add(s, hist[s * VX * VYM + i]);
      }
      if constexpr (ACC == 1) {
#pragma unroll
        for (int m = 0; m < NF; ++m) kahan_fold(ks[m], kc[m], part[m]);
      }
    }
    if (!a.last) {
#pragma unroll
      for (int m = 0; m < NF; ++m) {
        qs[m * g.points + p] = ks[m];
        qc[m * g.points + p] = kc[m];
      }
    } else {
      filter_solve_out<NF>(ks, kc, b, a.subtract, vsub, vout, p, g.points, in);
    }
  }
}

// ---- temporally blocked 2D kernel for grids of few tiles ------------------------------
//
// Where a grid has fewer tiles than the device has SMs, k_tb2d32 leaves a launch to a few CTAs, and
// what it does for a tile's many points after and (forced) during the steps is a long chain of L2
// latencies.  This kernel has tiles of 32 x 16 points (32 x 32 up to 4 frequencies), 512 threads: the
// tile plus a halo of T points in shared memory, a thread's one or two points and their sums in
// registers, the ring of the halo that later steps still read spread evenly over all threads.  It
// stages nothing for the sums and has all of a point's f in flight at once, but issues about three
// times the instructions per point-step, so larger grids are slower (ring_faster).  Per point the
// operations are those of k_tb2d32 in the same order.  us per launch of 16 steps with Kahan sums, in
// k_tb2d32 with 64 rows a tile, with the rows that rt_warps picks, and here: 129^2, N_f = 8,
// homogeneous 42, 20, 18, forced 67, 46, 25; 257^2, N_f = 16, homogeneous 65, 32, 26, forced 121, 85,
// 48.  (513^2, N_f = 6, homogeneous 25 there and 39 here.)
constexpr int kRingX = 32, kRingRows = 16, kRingThreads = kRingX * kRingRows;
constexpr int kRingNF = 4;   // frequencies from which it is used (tb32_launch)
__host__ __device__ constexpr int ring_k(int nf) { return nf <= 4 ? 2 : 1; }   // rows of a thread

struct RingArgs {
  Coef32 reg_lo, reg_hi, first_lo, first_hi;
  int n0, steps, forced, last, subtract;
};

template <int NF, int T>
constexpr size_t ring_smem_bytes() {
  return sizeof(float) *
         (3 * (kRingX + 2 * T) * (kRingRows * ring_k(NF) + 2 * T) + 2 * T * NF + 2 * T);
}

template <int NF, int T, int ACC>
__global__ void __launch_bounds__(kRingThreads, ACC == 0 || NF > 8 ? 1 : 2)
k_ring2d32(const float* W_in, const float* D_in,
           float* __restrict__ W_out, float* __restrict__ D_out, const float* __restrict__ f,
           float* __restrict__ qs, float* __restrict__ qc, double* vout, const double* vsub,
           const float* __restrict__ wq_table, const float* __restrict__ fc_table,
           const __grid_constant__ RingArgs a, const __grid_constant__ Last32Binv<NF> b,
           const Geom g) {
  pdl_wait();
  constexpr int K = ring_k(NF), BX = kRingX, BY = kRingRows * K;
  constexpr int EX = BX + 2 * T, EY = BY + 2 * T, E = EX * EY;
  extern __shared__ __align__(16) float sm32[];
  float* Wc = sm32;          // W^n on the extended tile
  float* Wn = sm32 + E;      // W^{n+1}
  float* Dv = sm32 + 2 * E;  // D on the halo (the tile's own is in registers)
  float* s_wq = sm32 + 3 * E;   // [T][NF] w_{n+1,m} and kappa_n cos(omega~_m t^n) of step s
  float* s_fc = s_wq + T * NF;
  unsigned* s_div = reinterpret_cast<unsigned*>(s_fc + T * NF);   // [T][2] divisors of radius r
  const int tid = threadIdx.x, tx = tid % BX, ty = tid / BX;
  const int64_t x0 = (int64_t)blockIdx.x * BX - T, y0 = (int64_t)blockIdx.y * BY - T;
  auto local = [](int64_t v) { return v < -1 ? -1 : (v > 128 ? 128 : (int)v); };
  // local bounds of the interior and of the grid; first local index of the upper layer
  const int ilx = local(1 - x0), ihx = local(g.nx - 1 - x0);
  const int ily = local(1 - y0), ihy = local(g.ny - 1 - y0);
  const bool lay_x = g.layer_axis == 0;
  const int thr = local(g.layer_split - (lay_x ? x0 : y0));
  // points outside the grid are 0, and so is the padding of its rows
  for (int e = tid; e < E / 4; e += kRingThreads) {
    const int ly = e / (EX / 4), lx = 4 * (e % (EX / 4));
    const int64_t x = x0 + lx, y = y0 + ly;
    float4 w = make_float4(0.0f, 0.0f, 0.0f, 0.0f), d = w;
    if (x >= 0 && x < g.syw && y >= 0 && y <= g.ny) {
      w = *reinterpret_cast<const float4*>(W_in + y * g.syw + x);
      if (D_in != nullptr) d = *reinterpret_cast<const float4*>(D_in + y * g.syw + x);
    }
    reinterpret_cast<float4*>(Wc)[e] = w;
    reinterpret_cast<float4*>(Wn)[e] = w;   // (boundary values of the next level)
    reinterpret_cast<float4*>(Dv)[e] = d;
  }
  for (int e = tid; e < a.steps * NF; e += kRingThreads) {
    s_wq[e] = wq_table[(int64_t)(a.n0 + 1) * NF + e];
    if (a.forced) s_fc[e] = fc_table[(int64_t)a.n0 * NF + e];
  }
  // e / d = umulhi(e, 2^32 / d rounded up), exact for e < 2^16 and 2 <= d < 2^7
  if (tid < T) {
    s_div[2 * tid] = 0xFFFFFFFFu / (unsigned)(BX + 2 * tid) + 1u;
    s_div[2 * tid + 1] = tid > 0 ? 0xFFFFFFFFu / (unsigned)(2 * tid) + 1u : 0u;
  }
  // every point that is updated is interior, with one c^2
  const bool simple = ilx <= 1 && ihx >= EX - 2 && ily <= 1 && ihy >= EY - 2 &&
                      (thr <= 0 || thr >= (lay_x ? EX : EY));
  const int lxo = T + tx, lyo = T + ty * K;   // this thread's first point
  const int64_t p0 = (y0 + lyo) * g.sy + x0 + lxo, f0 = (y0 + lyo) * g.syw + x0 + lxo;
  bool own[K], up[K];
  float wr[K], dr[K], ks[K][NF], kc[K][NF], part[K][NF];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    own[k] = lxo >= ilx && lxo <= ihx && lyo + k >= ily && lyo + k <= ihy;
    up[k] = (lay_x ? lxo : lyo + k) >= thr;
#pragma unroll
    for (int m = 0; m < NF; ++m) {
      part[k][m] = 0.0f;
      const int64_t o = m * g.points + p0 + k * g.sy;
      if (ACC == 0) {
        ks[k][m] = own[k] ? qs[o] : 0.0f;
        kc[k][m] = own[k] ? qc[o] : 0.0f;
      } else if (own[k] && (tid & 7) == 0) {   // read at the end of the launch
        asm volatile("prefetch.global.L2 [%0];" ::"l"(qs + o));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(qc + o));
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) {
    wr[k] = Wc[(lyo + k) * EX + lxo];
    dr[k] = Dv[(lyo + k) * EX + lxo];
  }
  // PLAIN: homogeneous launches of such CTAs; the values are the same.
  auto run_steps = [&](auto plain_c) {
    constexpr bool PLAIN = decltype(plain_c)::value;
    const int forced = PLAIN ? 0 : a.forced;
    for (int s = 0; s < a.steps; ++s) {
      const int r = a.steps - 1 - s;   // later steps read the tile grown by r
      const bool first = a.n0 + s == 0;
      const Coef32 lo = first ? a.first_lo : a.reg_lo, hi = first ? a.first_hi : a.reg_hi;
      const Coef32 one = thr <= 0 ? hi : lo;
      const float* fc = s_fc + s * NF;
      constexpr int R = ACC == 0 && NF > 12 ? NF : 1;   // (in registers where that spares loads)
      float wr_q[R];
#pragma unroll
      for (int m = 0; m < R; ++m) wr_q[m] = s_wq[s * NF + m];
      auto wq = [&](int m) { return R > 1 ? wr_q[R > 1 ? m : 0] : s_wq[s * NF + m]; };
      {
        const float above = Wc[(lyo - 1) * EX + lxo], below = Wc[(lyo + K) * EX + lxo];
        float wnew[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
          const float w = wr[k];
          wnew[k] = w;
          if (!PLAIN && !own[k]) continue;   // boundary and outside points keep W = 0
          const int l = (lyo + k) * EX + lxo;
          const float wu = k == 0 ? above : wr[k > 0 ? k - 1 : 0];
          const float wd = k == K - 1 ? below : wr[k < K - 1 ? k + 1 : k];
          const Coef32 L = PLAIN ? one : (up[k] ? hi : lo);
          const float inc =
              increment<NF, 2>(L, (Wc[l - 1] - w) + (Wc[l + 1] - w), (wu - w) + (wd - w), 0.0f, fc,
                               f, f0 + k * g.syw, g.wpoints, forced);
          dr[k] = dr[k] + inc;
          wnew[k] = w + dr[k];
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
          wr[k] = wnew[k];
          Wn[(lyo + k) * EX + lxo] = wnew[k];
          if (!PLAIN && !own[k]) continue;
#pragma unroll
          for (int m = 0; m < NF; ++m) {
            if (ACC == 0)
              kahan_add(ks[k][m], kc[k][m], wq(m), wnew[k]);
            else
              part[k][m] = fmaf(wq(m), wnew[k], part[k][m]);
          }
        }
      }
      // The ring of radius r around the tile: first the 2 r rows of BX + 2 r points above and
      // below it, then the BY rows of 2 r points at its sides.
      const int RW = BX + 2 * r, top = 2 * r * RW, ring = top + 2 * r * BY;
      const unsigned m_rw = s_div[2 * r], m_2r = s_div[2 * r + 1];
      auto ring_pass = [&](auto simple_c) {
        constexpr bool SIMPLE = decltype(simple_c)::value;
        for (int e = tid; e < ring; e += kRingThreads) {
          int lx, ly;
          if (e < top) {
            const int row = (int)__umulhi((unsigned)e, m_rw);
            lx = T - r + (e - row * RW);
            ly = row < r ? T - r + row : T + BY + row - r;
          } else {
            const int row = (int)__umulhi((unsigned)(e - top), m_2r), col = e - top - row * 2 * r;
            ly = T + row;
            lx = col < r ? T - r + col : T + BX + col - r;
          }
          if (!SIMPLE && (lx < ilx || lx > ihx || ly < ily || ly > ihy)) continue;
          const int l = ly * EX + lx;
          const float w = Wc[l];
          const Coef32 L = SIMPLE ? one : ((lay_x ? lx : ly) >= thr ? hi : lo);
          const float inc = increment<NF, 2>(L, (Wc[l - 1] - w) + (Wc[l + 1] - w),
                                             (Wc[l - EX] - w) + (Wc[l + EX] - w), 0.0f, fc, f,
                                             (y0 + ly) * g.syw + x0 + lx, g.wpoints, forced);
          const float dn = Dv[l] + inc;
          Dv[l] = dn;
          Wn[l] = w + dn;
        }
      };
      if (PLAIN || simple)
        ring_pass(std::true_type{});
      else
        ring_pass(std::false_type{});
      __syncthreads();
      float* t = Wc;
      Wc = Wn;
      Wn = t;
    }
  };
  if (simple && !a.forced)
    run_steps(std::true_type{});
  else
    run_steps(std::false_type{});
  pdl_release();
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int64_t p = p0 + k * g.sy;
    if (ACC == 1 && own[k]) {
#pragma unroll
      for (int m = 0; m < NF; ++m) {
        ks[k][m] = qs[m * g.points + p];
        kc[k][m] = qc[m * g.points + p];
        kahan_fold(ks[k][m], kc[k][m], part[k][m]);
      }
    }
    if (!a.last) {
      if (!own[k]) continue;
      W_out[f0 + k * g.syw] = wr[k];
      D_out[f0 + k * g.syw] = dr[k];
#pragma unroll
      for (int m = 0; m < NF; ++m) {
        qs[m * g.points + p] = ks[k][m];
        qc[m * g.points + p] = kc[k][m];
      }
    } else if (x0 + lxo <= g.nx && y0 + lyo + k <= g.ny) {
      if (!own[k]) {
#pragma unroll
        for (int m = 0; m < NF; ++m) ks[k][m] = kc[k][m] = 0.0f;
      }
      filter_solve_out<NF>(ks[k], kc[k], b, a.subtract, vsub, vout, p, g.points, own[k]);
    }
  }
}

// ---- init and conversion ---------------------------------------------------------

template <int NF, int DIM>
__global__ void __launch_bounds__(kBX * kBY)
k_init32(const double* __restrict__ v, float* __restrict__ W0, float* __restrict__ qs,
         float* __restrict__ qc, const Init32Args<NF> a, const Geom g) {
  int64_t i, j, k, p;
  bool interior;
  if (!index_of<DIM>(g, i, j, k, p, interior)) return;
  double w = 0.0;
  if (interior && v != nullptr) {
#pragma unroll
    for (int m = 0; m < NF; ++m) w += v[m * g.points + p];
  }
  const float wf = (float)w;
  W0[wpos(g, i, j, k)] = wf;
#pragma unroll
  for (int m = 0; m < NF; ++m) {
    qs[m * g.points + p] = a.w0[m] * wf;
    qc[m * g.points + p] = 0.0f;
  }
}

// ---- temporally blocked 3D kernel ------------------------------------------------
// The 2D kernel's scheme in 3D: one CTA per SM (16 warps) holds an extended tile of 64 x 16 x 20
// points in registers, warp w the row y = w, lane l its columns 2l, 2l + 1 of all 20 planes, and
// steps all of it T times (T = 2 or 4; planes and rows that no later step reads rest), after
// which the (64 - 2T) x (16 - 2T) x (20 - 2T) points in the middle are exact.  Neighbours along z
// are in the thread, along x in the thread or one shuffle away; along y they come from a copy of
// the whole tile in shared memory, rewritten every step (two barriers a step).  As in 2D the new
// values of the owned points are kept in shared memory and all filter updates made after the last
// step, with the weights as constant operands.  Per point the operations are those of
// step_point<NF, 3, 2> in the same order, so with ACC = 0 every depth is bit-identical to one step
// per launch.
//
// HBM bounds it: 16 + 16 N_f bytes per owned point and launch, and the halo of W and D.  257^3,
// N_f = 4, two layers, depth 4 (one map of 885 steps): 235 ms for the form it replaces (a flat tile
// in shared memory, 61 % issue, 13 % DRAM), 141 ms for this one.
constexpr int kR3X = 64, kR3Y = 16, kR3Z = 20, kR3Threads = 32 * kR3Y;

template <int NF, int T>
struct R3Args {
  Coef32 reg_lo, reg_hi, first_lo, first_hi;
  int n0, steps, forced, last, subtract;
  float wq[T * NF];   // w_{n+1,m} of step s: [s * NF + m]
  float fc[T * NF];   // kappa_n cos(omega~_m t^n)
};

template <int T>
constexpr size_t r3_smem_bytes() {
  return sizeof(float) * ((size_t)kR3X * kR3Y * kR3Z +
                          (size_t)T * (kR3X - 2 * T) * (kR3Y - 2 * T) * (kR3Z - 2 * T));
}

template <int NF, int T, int ACC>
__global__ void __launch_bounds__(kR3Threads, 1)
k_tb3d32(const float* W_in, const float* D_in,
         float* __restrict__ W_out, float* __restrict__ D_out, const float* __restrict__ f,
         float* __restrict__ qs, float* __restrict__ qc, double* vout, const double* vsub,
         const __grid_constant__ R3Args<NF, T> a, const __grid_constant__ Last32Binv<NF> b,
         const Geom g) {
  pdl_begin();
  constexpr int VX = kR3X - 2 * T, VY = kR3Y - 2 * T, VZ = kR3Z - 2 * T;   // owned points
  constexpr int VXY = VX * VY, V = VXY * VZ;
  extern __shared__ __align__(16) float sm3[];
  float* tile = sm3;                          // [z][y][x] the level being read
  float* hist = sm3 + kR3X * kR3Y * kR3Z;     // [T][VZ][VY][VX] owned values step by step
  const int tid = threadIdx.x, lane = tid & 31, ly = tid >> 5, lx = 2 * lane;
  const int64_t x0 = (int64_t)blockIdx.x * VX - T, y0 = (int64_t)blockIdx.y * VY - T,
                z0 = (int64_t)blockIdx.z * VZ - T;
  // local bounds (32-bit): interior columns, rows and planes, planes of the grid
  auto local = [](int64_t v) { return v < -1 ? -1 : (v > 64 ? 64 : (int)v); };
  const int ilx = local(1 - x0), ihx = local(g.nx - 1 - x0);
  const int ily = local(1 - y0), ihy = local(g.ny - 1 - y0);
  const int ilz = local(1 - z0), ihz = local(g.nz - 1 - z0);
  const bool in_y = ly >= ily && ly <= ihy;
  const bool in0 = in_y && lx >= ilx && lx <= ihx, in1 = in_y && lx + 1 >= ilx && lx + 1 <= ihx;
  // c^2 layer: local index along the layer axis from which hi holds
  const int thr = local(g.layer_split - (g.layer_axis == 0 ? x0 : (g.layer_axis == 1 ? y0 : z0)));
  const bool owner_xy = lx >= T && lx < T + VX && ly >= T && ly < T + VY;
  const int64_t gbase = z0 * g.szw + (y0 + ly) * g.syw + x0 + lx;

  float w[kR3Z][2], d[kR3Z][2];
  {
    // x0 + lx is even and rows are padded: both columns lie in a row of the arrays or none
    const bool col = y0 + ly >= 0 && y0 + ly <= g.ny && x0 + lx >= 0 && x0 + lx < g.syw;
#pragma unroll
    for (int k = 0; k < kR3Z; ++k) {
      float2 v = make_float2(0.0f, 0.0f), u = v;
      if (col && k >= ilz && k <= ihz) {   // outside the interior W = 0
        v = *reinterpret_cast<const float2*>(W_in + gbase + k * g.szw);
        if (D_in != nullptr) u = *reinterpret_cast<const float2*>(D_in + gbase + k * g.szw);
      }
      w[k][0] = in0 ? v.x : 0.0f;
      w[k][1] = in1 ? v.y : 0.0f;
      d[k][0] = in0 ? u.x : 0.0f;
      d[k][1] = in1 ? u.y : 0.0f;
    }
  }
  // Ask L2 for the sums that the end of the launch updates.
  if (owner_xy && (lane & 7) == T / 2) {
    const int64_t p = (z0 + T) * g.sz + (y0 + ly) * g.sy + x0 + lx;
    for (int e = 0; e < 2 * NF; ++e) {
      const float* base = (e & 1 ? qc : qs) + (int64_t)(e >> 1) * g.points;
      for (int k = 0; k < VZ; ++k)
        if (in0 && k + T >= ilz && k + T <= ihz)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(base + p + k * g.sz));
    }
  }
  // PLAIN: all points of the CTA are interior with one c^2, no forcing; the values are the same.
  auto run_steps = [&](auto plain_c) {
    constexpr bool PLAIN = decltype(plain_c)::value;
    float* mine = tile + ly * kR3X + lx;
    for (int s = 0; s < a.steps; ++s) {
      const int r = a.steps - 1 - s;   // later steps read the owned points grown by r
      const bool first = a.n0 + s == 0;
      const Coef32 lo = first ? a.first_lo : a.reg_lo, hi = first ? a.first_hi : a.reg_hi;
      const Coef32 one = thr <= 0 ? hi : lo;
      const bool upper_y = g.layer_axis == 1 && ly >= thr;
      const bool upper0 = upper_y || (g.layer_axis == 0 && lx >= thr);
      const bool upper1 = upper_y || (g.layer_axis == 0 && lx + 1 >= thr);
      // rows read at this step: those updated and one beyond
      if (ly >= T - r - 1 && ly <= T + VY + r) {
#pragma unroll
        for (int k = 0; k < kR3Z; ++k)
          *reinterpret_cast<float2*>(mine + k * (kR3X * kR3Y)) = make_float2(w[k][0], w[k][1]);
      }
      __syncthreads();
      if (ly >= T - r && ly < T + VY + r) {
        float dz0 = 0.0f, dz1 = 0.0f;   // W - W_below of the current plane
#pragma unroll
        for (int k = 0; k < kR3Z; ++k) {
          const float w0 = w[k][0], w1 = w[k][1];
          float dn0 = 0.0f, dn1 = 0.0f;
          if (k + 1 < kR3Z) {
            dn0 = w[k + 1 < kR3Z ? k + 1 : k][0] - w0;
            dn1 = w[k + 1 < kR3Z ? k + 1 : k][1] - w1;
          }
          if (k >= T - r && k < T + VZ + r) {
            const float left = __shfl_up_sync(0xffffffffu, w1, 1);
            const float right = __shfl_down_sync(0xffffffffu, w0, 1);
            const float2 ym = *reinterpret_cast<const float2*>(mine + k * (kR3X * kR3Y) - kR3X);
            const float2 yp = *reinterpret_cast<const float2*>(mine + k * (kR3X * kR3Y) + kR3X);
            const float dx0 = w0 - left, dx1 = w1 - w0, dx2 = right - w1;
            const float dxx0 = dx1 - dx0, dxx1 = dx2 - dx1;
            const float dyy0 = (ym.x - w0) + (yp.x - w0), dyy1 = (ym.y - w1) + (yp.y - w1);
            const float dzz0 = dn0 - dz0, dzz1 = dn1 - dz1;
            const bool uz = !PLAIN && g.layer_axis == 2 && k >= thr;
            const Coef32 L0 = PLAIN ? one : ((upper0 || uz) ? hi : lo);
            const Coef32 L1 = PLAIN ? one : ((upper1 || uz) ? hi : lo);
            float i0 = L0.Ay * dyy0, i1 = L1.Ay * dyy1;
            i0 = fmaf(L0.Az, dzz0, i0);
            i1 = fmaf(L1.Az, dzz1, i1);
            i0 = fmaf(L0.Ax, dxx0, i0);
            i1 = fmaf(L1.Ax, dxx1, i1);
            if (!PLAIN && a.forced && (in0 || in1) && k >= ilz && k <= ihz) {
              const float* fp = f + gbase + k * g.szw;   // rows of f are padded like those of W
#pragma unroll 4
              for (int m = 0; m < NF; ++m) {
                const float2 v = *reinterpret_cast<const float2*>(fp + m * g.wpoints);
                i0 = fmaf(-a.fc[s * NF + m], v.x, i0);
                i1 = fmaf(-a.fc[s * NF + m], v.y, i1);
              }
            }
            float d0 = d[k][0] + i0, d1 = d[k][1] + i1;
            float n0 = w0 + d0, n1 = w1 + d1;
            if (!PLAIN) {   // boundary and outside points keep W = 0
              const bool iz = k >= ilz && k <= ihz;
              if (!(in0 && iz)) d0 = n0 = 0.0f;
              if (!(in1 && iz)) d1 = n1 = 0.0f;
            }
            d[k][0] = d0;
            d[k][1] = d1;
            w[k][0] = n0;
            w[k][1] = n1;
          }
          dz0 = dn0;
          dz1 = dn1;
        }
        if (owner_xy) {
          float* h = hist + (size_t)s * V + (ly - T) * VX + lx - T;
#pragma unroll
          for (int k = T; k < T + VZ; ++k)
            *reinterpret_cast<float2*>(h + (k - T) * VXY) = make_float2(w[k][0], w[k][1]);
        }
      }
      __syncthreads();
    }
  };
  const bool simple = !a.forced && ilx <= 0 && ihx >= kR3X - 1 && ily <= 0 && ihy >= kR3Y - 1 &&
                      ilz <= 0 && ihz >= kR3Z - 1 &&
                      (thr <= 0 || thr >= (g.layer_axis == 0 ? kR3X : (g.layer_axis == 1 ? kR3Y : kR3Z)));
  if (simple)
    run_steps(std::true_type{});
  else
    run_steps(std::false_type{});
  if (owner_xy && !a.last && y0 + ly <= g.ny && x0 + lx < g.syw) {
#pragma unroll
    for (int k = T; k < T + VZ; ++k) {
      if (z0 + k > g.nz) continue;
      *reinterpret_cast<float2*>(W_out + gbase + k * g.szw) = make_float2(w[k][0], w[k][1]);
      *reinterpret_cast<float2*>(D_out + gbase + k * g.szw) = make_float2(d[k][0], d[k][1]);
    }
  }
  // The filter sums of the owned points.
#pragma unroll 2
  for (int i = tid; i < V; i += kR3Threads) {
    const int rz = i / VXY, rest = i - rz * VXY, ry = rest / VX, rx = rest - ry * VX;
    const int64_t x = x0 + T + rx, y = y0 + T + ry, z = z0 + T + rz;
    const bool in = x > 0 && x < g.nx && y > 0 && y < g.ny && z > 0 && z < g.nz;
    if (!in && !(a.last && x <= g.nx && y <= g.ny && z <= g.nz)) continue;
    const int64_t p = z * g.sz + y * g.sy + x;
    float ks[NF], kc[NF];
#pragma unroll
    for (int m = 0; m < NF; ++m) {
      ks[m] = in ? qs[m * g.points + p] : 0.0f;
      kc[m] = in ? qc[m * g.points + p] : 0.0f;
    }
    if (in) {
      float part[ACC == 1 ? NF : 1];
      if constexpr (ACC == 1) {
#pragma unroll
        for (int m = 0; m < NF; ++m) part[m] = 0.0f;
      }
      auto add = [&](int s, float v) {
#pragma unroll
        for (int m = 0; m < NF; ++m) {
          if constexpr (ACC == 1)
            part[m] = fmaf(a.wq[s * NF + m], v, part[m]);
          else
            kahan_add(ks[m], kc[m], a.wq[s * NF + m], v);
        }
      };
      if (a.steps == T) {
#pragma unroll
        for (int s = 0; s < T; ++s) add(s, hist[s * V + i]);
      } else {
#pragma unroll 1
        for (int s = 0; s < a.steps; ++s) add(s, hist[s * V + i]);
      }
      if constexpr (ACC == 1) {
#pragma unroll
        for (int m = 0; m < NF; ++m) kahan_fold(ks[m], kc[m], part[m]);
      }
    }
    if (!a.last) {
#pragma unroll
      for (int m = 0; m < NF; ++m) {
        qs[m * g.points + p] = ks[m];
        qc[m * g.points + p] = kc[m];
      }
    } else {
      filter_solve_out<NF>(ks, kc, b, a.subtract, vsub, vout, p, g.points, in);
    }
  }
}

// ---- host launchers --------------------------------------------------------------

template <int NF>
Step32Args<NF> step_args(const Step32Host& h) {
  Step32Args<NF> a;
  a.lo = h.lo;
  a.hi = h.hi;
  for (int m = 0; m < NF; ++m) {
    a.fc[m] = h.fc[m];
    a.wq[m] = h.wq[m];
  }
  a.forced = h.forced;
  a.group = h.group;
  a.part = h.part;
  return a;
}

template <int NF>
Last32Binv<NF> binv_args(const double* binv, const double* emat, int has_e,
                         const double* vprev) {
  Last32Binv<NF> b;
  for (int m = 0; m < NF; ++m)
    for (int j = 0; j < NF; ++j) {
      b.binv[m * NF + j] = binv[m * MFWH_MAX_NF + j];
      b.emat[m * NF + j] = emat[m * MFWH_MAX_NF + j];
    }
  b.has_e = has_e && vprev != nullptr;
  b.vprev = vprev;
  return b;
}

dim3 grid_of(const Geom& g) {
  return dim3((unsigned)((g.nx + kBX) / kBX), (unsigned)((g.ny + kBY) / kBY),
              (unsigned)(g.dim == 3 ? g.nz + 1 : 1));
}

template <int NF>
void step32_nf(const Geom& g, const float* W, const float* D_in, float* W_out, float* D_out,
               const float* f, float* qs, float* qc, const Step32Host& h, cudaStream_t st) {
  const Step32Args<NF> a = step_args<NF>(h);
  const dim3 grid = grid_of(g), blk(kBX, kBY);
  if (g.order == 4) {
    if (g.dim == 3)
      launch_dependent(k_step32<NF, 3, 4, false>, grid, blk, 0, st, W, D_in, W_out, D_out, f, qs, qc, a, g);
    else
      launch_dependent(k_step32<NF, 2, 4, false>, grid, blk, 0, st, W, D_in, W_out, D_out, f, qs, qc, a, g);
  } else if (g.dim == 3) {
    if (h.group)
      launch_dependent(k_step32<NF, 3, 2, true>, grid, blk, 0, st, W, D_in, W_out, D_out, f, qs, qc, a, g);
    else
      launch_dependent(k_step32<NF, 3, 2, false>, grid, blk, 0, st, W, D_in, W_out, D_out, f, qs, qc, a, g);
  } else {
    launch_dependent(k_step32<NF, 2, 2, false>, grid, blk, 0, st, W, D_in, W_out, D_out, f, qs, qc, a, g);
  }
}

template <int NF>
void last32_nf(const Geom& g, const float* W, const float* D, const float* f, const float* qs,
               const float* qc, double* vout, const double* vsub, const Step32Host& h,
               const StepHost& epi, cudaStream_t st) {
  const Step32Args<NF> a = step_args<NF>(h);
  const Last32Binv<NF> b = binv_args<NF>(epi.binv, epi.emat, epi.has_e, epi.vprev);
  const int sub = vsub != nullptr;
  const dim3 grid = grid_of(g), blk(kBX, kBY);
  if (g.order == 4) {
    if (g.dim == 3)
      launch_dependent(k_last32<NF, 3, 4>, grid, blk, 0, st, W, D, f, qs, qc, vout, vsub, a, b, sub, g);
    else
      launch_dependent(k_last32<NF, 2, 4>, grid, blk, 0, st, W, D, f, qs, qc, vout, vsub, a, b, sub, g);
  } else if (g.dim == 3) {
    launch_dependent(k_last32<NF, 3, 2>, grid, blk, 0, st, W, D, f, qs, qc, vout, vsub, a, b, sub, g);
  } else {
    launch_dependent(k_last32<NF, 2, 2>, grid, blk, 0, st, W, D, f, qs, qc, vout, vsub, a, b, sub, g);
  }
}

template <int NF>
void init32_nf(const Geom& g, const double* v, float* W0, float* qs, float* qc, const float* w0,
               cudaStream_t st) {
  Init32Args<NF> a;
  for (int m = 0; m < NF; ++m) a.w0[m] = w0[m];
  if (g.dim == 3)
    k_init32<NF, 3><<<grid_of(g), dim3(kBX, kBY), 0, st>>>(v, W0, qs, qc, a, g);
  else
    k_init32<NF, 2><<<grid_of(g), dim3(kBX, kBY), 0, st>>>(v, W0, qs, qc, a, g);
}

// Step warps of k_tb2d32: a launch takes about as many rounds as the grid has tiles per SM, of a time
// that grows with the tile's rows (step warps and, more with more frequencies, sums of the rows
// owned).  Lower tiles have to promise 5 % (7 % at depth 8 above 12 frequencies, 10 % at depth 16,
// where the promise of a grid of just over a round of tiles is not kept: 1501 x 301, N_f = 4, forced,
// 60.8 us a launch with 160 tiles of 64 rows, 67.9 with 208 of 56).  Problems of a batch share the
// SMs: with each one's tiles for the whole device, whose halos are more work in all, six of 257^2 to
// 1025^2 took 65.0 ms for a map and four products, and take 61.8 with tiles as for one SM.
inline int rt_warps(const Geom& g, int nf, int T, int sms) {
  const int64_t tx = (g.nx + kRtEX - 2 * T) / (kRtEX - 2 * T);
  const double part = T == 16 ? 0.90 : (T == 8 && nf > 12 ? 0.93 : 0.95);
  int best = kRtWarps;
  double cost = 0.0;
  for (int w = kRtWarps; w > T / 2; --w) {
    const int vy = 4 * w - 2 * T;
    const int64_t t = tx * ((g.ny + vy) / vy);
    const double r = 0.5 * ((double)((t + sms - 1) / sms) + std::max(1.0, (double)t / sms));
    const double c = r * (2.0 + w + 0.15 * nf * (w - T / 2)) *
                     (T >= 8 && w < kRtWarps && nf > 6 ? 1.0 + 0.01 * (nf - 6) : 1.0);   // (FULL)
    if (w == kRtWarps || c < part * cost) {
      best = w;
      cost = c;
    }
  }
  return best;
}

// Whether k_ring2d32 is the faster one: up to a number of 32 x 32 tiles per SM (of 152: 257^2 0.53,
// 385^2 1.1, 449^2 1.5) that grows with the frequencies, more so forced and for shallow launches.
// Measured on 16 grids of 65^2 to 1501^2, N_f 1 to 16, depths 4, 8, 16.
inline bool ring_faster(const Geom& g, int nf, int T, bool kahan, int forced, int sms) {
  const double r = (double)((g.nx + 32) / 32 * ((g.ny + 32) / 32)) / sms;
  const double up_to = nf >= 14 ? 1.5 : 1.25;
  if (T == 16) return forced ? r <= 1.0 && (nf >= 5 || kahan) : r <= 0.55 && nf >= (kahan ? 5 : 12);
  if (T == 8)
    return forced ? r <= (nf >= 5 || kahan ? up_to : 0.55) : nf >= 5 && r <= (nf >= 14 ? 1.5 : 0.55);
  return nf >= 5 || kahan ? r <= up_to : forced && r <= 0.55;
}

template <int NF, int T, int ACC>
void tb32_launch(const Geom& g, const float* W_in, const float* D_in, float* W_out, float* D_out,
                 const float* f, float* qs, float* qc, double* vout, const double* vsub,
                 const TB32Host& h, cudaStream_t st) {
  constexpr size_t smem = rt32_smem_bytes<T>();
  static bool configured[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    cudaFuncSetAttribute(k_tb2d32<NF, T, ACC, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)smem);
    if constexpr (T >= 8)
      cudaFuncSetAttribute(k_tb2d32<NF, T, ACC, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)smem);
    if constexpr (NF >= kRingNF)
      cudaFuncSetAttribute(k_ring2d32<NF, T, ACC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)ring_smem_bytes<NF, T>());
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  const Last32Binv<NF> b = binv_args<NF>(h.binv, h.emat, h.has_e, h.vprev);
  if constexpr (NF >= kRingNF) {
    constexpr int BY = kRingRows * ring_k(NF);
    const dim3 grid((unsigned)((g.nx + kRingX) / kRingX), (unsigned)((g.ny + BY) / BY));
    if (ring_faster(g, NF, T, ACC == 0, h.forced, h.sms)) {
      const RingArgs r{h.reg_lo, h.reg_hi, h.first_lo, h.first_hi, h.n0, h.steps, h.forced, h.last,
                       vsub != nullptr};
      launch_dependent(k_ring2d32<NF, T, ACC>, grid, dim3(kRingThreads), ring_smem_bytes<NF, T>(), st,
                       W_in, D_in, W_out, D_out, f, qs, qc, vout, vsub, h.wq, h.fc, r, b, g);
      return;
    }
  }
  RT32Args<NF, T> a;
  a.reg_lo = h.reg_lo;
  a.reg_hi = h.reg_hi;
  a.first_lo = h.first_lo;
  a.first_hi = h.first_hi;
  a.n0 = h.n0;
  a.steps = h.steps;
  a.forced = h.forced;
  a.last = h.last;
  a.subtract = vsub != nullptr;
  a.warps = rt_warps(g, NF, T, h.sms);
  for (int s = 0; s < T; ++s)
    for (int m = 0; m < NF; ++m) {
      a.wq[s * NF + m] = s < h.steps ? h.wq_host[(size_t)(h.n0 + s + 1) * NF + m] : 0.0f;
      a.fc[s * NF + m] = s < h.steps && h.forced ? h.fc_host[(size_t)(h.n0 + s) * NF + m] : 0.0f;
    }
  constexpr int VX = kRtEX - 2 * T;
  const int VY = 4 * a.warps - 2 * T;
  const dim3 grid((unsigned)((g.nx + VX) / VX), (unsigned)((g.ny + VY) / VY));
  auto* fn = k_tb2d32<NF, T, ACC, false>;
  if constexpr (T >= 8)
    if (a.warps == kRtWarps) fn = k_tb2d32<NF, T, ACC, true>;
  launch_dependent(fn, grid, dim3(kRtThreads), smem, st, W_in, D_in, W_out, D_out, f, qs, qc, vout,
                   vsub, a, b, g);
}

template <int NF, int T>
void tb32_acc(const Geom& g, const float* W_in, const float* D_in, float* W_out, float* D_out,
              const float* f, float* qs, float* qc, double* vout, const double* vsub,
              const TB32Host& h, cudaStream_t st) {
  if (h.acc == 1)
    tb32_launch<NF, T, 1>(g, W_in, D_in, W_out, D_out, f, qs, qc, vout, vsub, h, st);
  else
    tb32_launch<NF, T, 0>(g, W_in, D_in, W_out, D_out, f, qs, qc, vout, vsub, h, st);
}

template <int NF>
void tb32_nf(const Geom& g, const float* W_in, const float* D_in, float* W_out, float* D_out,
             const float* f, float* qs, float* qc, double* vout, const double* vsub,
             const TB32Host& h, cudaStream_t st) {
  if (h.depth <= 4)
    tb32_acc<NF, 4>(g, W_in, D_in, W_out, D_out, f, qs, qc, vout, vsub, h, st);
  else if (h.depth <= 8)
    tb32_acc<NF, 8>(g, W_in, D_in, W_out, D_out, f, qs, qc, vout, vsub, h, st);
  else
    tb32_acc<NF, 16>(g, W_in, D_in, W_out, D_out, f, qs, qc, vout, vsub, h, st);
}

template <int NF, int T, int ACC>
void tb3d32_launch(const Geom& g, const float* W_in, const float* D_in, float* W_out,
                   float* D_out, const float* f, float* qs, float* qc, double* vout,
                   const double* vsub, const TB32Host& h, cudaStream_t st) {
  constexpr size_t smem = r3_smem_bytes<T>();
  static bool configured[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    cudaFuncSetAttribute(k_tb3d32<NF, T, ACC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)smem);
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  R3Args<NF, T> a;
  a.reg_lo = h.reg_lo;
  a.reg_hi = h.reg_hi;
  a.first_lo = h.first_lo;
  a.first_hi = h.first_hi;
  a.n0 = h.n0;
  a.steps = h.steps;
  a.forced = h.forced;
  a.last = h.last;
  a.subtract = vsub != nullptr;
  for (int s = 0; s < T; ++s)
    for (int m = 0; m < NF; ++m) {
      a.wq[s * NF + m] = s < h.steps ? h.wq_host[(size_t)(h.n0 + s + 1) * NF + m] : 0.0f;
      a.fc[s * NF + m] = s < h.steps && h.forced ? h.fc_host[(size_t)(h.n0 + s) * NF + m] : 0.0f;
    }
  const Last32Binv<NF> b = binv_args<NF>(h.binv, h.emat, h.has_e, h.vprev);
  constexpr int VX = kR3X - 2 * T, VY = kR3Y - 2 * T, VZ = kR3Z - 2 * T;
  const dim3 grid((unsigned)((g.nx + VX) / VX), (unsigned)((g.ny + VY) / VY),
                  (unsigned)((g.nz + VZ) / VZ));
  launch_dependent(k_tb3d32<NF, T, ACC>, grid, dim3(kR3Threads), smem, st, W_in, D_in, W_out, D_out, f, qs, qc, vout,
                                                       vsub, a, b, g);
}

// Depth 2 or 4 (a launch of at most T steps; the halo is T points).
template <int NF>
void tb3d32_nf(const Geom& g, const float* W_in, const float* D_in, float* W_out, float* D_out,
               const float* f, float* qs, float* qc, double* vout, const double* vsub,
               const TB32Host& h, cudaStream_t st) {
  if (h.depth <= 2) {
    if (h.acc == 1)
      tb3d32_launch<NF, 2, 1>(g, W_in, D_in, W_out, D_out, f, qs, qc, vout, vsub, h, st);
    else
      tb3d32_launch<NF, 2, 0>(g, W_in, D_in, W_out, D_out, f, qs, qc, vout, vsub, h, st);
  } else {
    if (h.acc == 1)
      tb3d32_launch<NF, 4, 1>(g, W_in, D_in, W_out, D_out, f, qs, qc, vout, vsub, h, st);
    else
      tb3d32_launch<NF, 4, 0>(g, W_in, D_in, W_out, D_out, f, qs, qc, vout, vsub, h, st);
  }
}

template <int NF>
W32Ops make_w32_ops() {
  return W32Ops{init32_nf<NF>, step32_nf<NF>, last32_nf<NF>, tb32_nf<NF>};
}

using Tb3dFn = void (*)(const Geom&, const float*, const float*, float*, float*, const float*,
                        float*, float*, double*, const double*, const TB32Host&, cudaStream_t);

}  // namespace

// Defined in wave32_p1.cu .. wave32_p8.cu for nf in 1-2, 3-4, ..., 15-16.
W32Ops w32_ops_p1(int nf);
W32Ops w32_ops_p2(int nf);
W32Ops w32_ops_p3(int nf);
W32Ops w32_ops_p4(int nf);
W32Ops w32_ops_p5(int nf);
W32Ops w32_ops_p6(int nf);
W32Ops w32_ops_p7(int nf);
W32Ops w32_ops_p8(int nf);
// The 3D blocked launcher for nf, from the translation unit that instantiates nf.
Tb3dFn w32_tb3_p1(int nf);
Tb3dFn w32_tb3_p2(int nf);
Tb3dFn w32_tb3_p3(int nf);
Tb3dFn w32_tb3_p4(int nf);
Tb3dFn w32_tb3_p5(int nf);
Tb3dFn w32_tb3_p6(int nf);
Tb3dFn w32_tb3_p7(int nf);
Tb3dFn w32_tb3_p8(int nf);

}  // namespace mfwh
