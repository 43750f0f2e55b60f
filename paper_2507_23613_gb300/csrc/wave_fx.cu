// Start of a fixed-point wave solve (wave_fx_kernels.cuh): the forcing's unit, the first quantum,
// W^0 and the first filter terms; the forcing of a launch's steps; dispatch of the step launches on the frequency count.
#include <cuda_runtime.h>

#include "wave_fx_kernels.cuh"

namespace mfwh {
namespace {

// Largest key of the block (warps of 32 threads in x) into *out; keys are bits of non-negative
// doubles, which order like the values (NaN above infinity).
__device__ __forceinline__ void max_key(unsigned long long mx, unsigned long long* out) {
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long t = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = t > mx ? t : mx;
  }
  if (threadIdx.x == 0 && mx > 0) atomicMax(out, mx);
}

__device__ __forceinline__ unsigned long long abs_key(double v) {
  return (unsigned long long)__double_as_longlong(v) & ~(1ull << 63);
}

// W^0 = sum_m v_m on the interior points (0 on the boundary and in the padding) as doubles in W,
// and the largest |W^0|.
__global__ void __launch_bounds__(256)
k_fx_sum(const double* __restrict__ v, int nf, int64_t* __restrict__ W, const Geom g,
         unsigned long long* __restrict__ wmax) {
  unsigned long long mx = 0;
  const int64_t x = (int64_t)blockIdx.x * 32 + threadIdx.x;
  for (int64_t y = (int64_t)blockIdx.y * 8 + threadIdx.y; y <= g.ny; y += (int64_t)gridDim.y * 8) {
    if (x >= g.syw || !MFWH_IDX(g.fault, y * g.syw + x, g.wpoints)) continue;
    double w = 0.0;
    if (v != nullptr && x > 0 && x < g.nx && y > 0 && y < g.ny) {
      const int64_t p = y * g.sy + x;
#pragma unroll 4
      for (int m = 0; m < nf; ++m) w += v[m * g.points + p];
    }
    W[y * g.syw + x] = __double_as_longlong(w);
    const unsigned long long b = abs_key(w);
    mx = b > mx ? b : mx;
  }
  max_key(mx, wmax);
}

// max |f_m| over the interior points, one layer of blocks per frequency.
__global__ void __launch_bounds__(256)
k_fx_fmax(const double* __restrict__ f, const Geom g, unsigned long long* __restrict__ fmax) {
  const double* fm = f + blockIdx.z * g.points;
  unsigned long long mx = 0;
  const int64_t x = 1 + (int64_t)blockIdx.x * 32 + threadIdx.x;
  for (int64_t y = 1 + (int64_t)blockIdx.y * 8 + threadIdx.y; y < g.ny; y += (int64_t)gridDim.y * 8) {
    if (x >= g.nx || !MFWH_IDX(g.fault, y * g.sy + x, g.points)) continue;
    const unsigned long long b = abs_key(fm[y * g.sy + x]);
    mx = b > mx ? b : mx;
  }
  max_key(mx, fmax + blockIdx.z);
}

// The unit of the forcing's integers (the largest |f| has 58 bits) and sum_m max |f_m|.
__global__ void k_fx_funit(const unsigned long long* fmax, int nf, FxForcing* out) {
  double mx = 0.0, sum = 0.0;
  for (int m = 0; m < nf; ++m) {
    const double v = __longlong_as_double((int64_t)fmax[m]);
    sum += v;
    mx = v > mx || !(v == v) ? v : mx;
  }
  int ex = 0;
  if (mx > 0.0 && mx < 1e300) frexp(mx, &ex);   // mx < 2^ex
  out->fe = ex - 58;
  out->fsum = sum;
}

// The forcing of a launch's steps in its quanta, F_s = sum_m fc[s][m] f_m: f / 2^fe (58 bits) and the
// coefficients / 2^ce (59 bits) as two digits each, their high digits' products summed exactly and
// the mixed ones in FP32 (2^-24 of terms that are 2^-28 of the largest), rounded once.  In the step
// kernel this sum would be made twice per point (halo) and its terms read from L2 in every step: at
// 1025^2, N_f = 8, a forced launch of 8 steps took 288 us that way, 182 us with three integer
// products per term here, and 160 us now (an unforced one takes 76).  Bound by instruction issue:
// per point and f_m the conversion and 8 steps' product and two FMAs.
struct FxForceArgs {
  float gw, gd;
  int steps, nf, wsum, ce;
  int gh[8 * MFWH_MAX_NF];                              // high digits, [m * 8 + s]
  float ghf[8 * MFWH_MAX_NF], glf[8 * MFWH_MAX_NF];     // the digits / 2^32 in FP32
};
// STEPS: of a launch.
template <int STEPS>
__global__ void __launch_bounds__(128, 4)
k_fx_force(const double* __restrict__ f, int64_t* __restrict__ force,
           const __grid_constant__ FxForceArgs a, const FxScale* scale,
           const FxState* state, const Geom g) {
  pdl_wait();
  const FxScale sc = *scale;
  if (sc.mode) return;
  // the sum of high products is in units of 2^(fe + ce + 64)
  const int sh = sc.fe + a.ce + 64 - fx_quantum(*state, sc, a.gw, a.gd, a.wsum, STEPS == 4 ? 4 : 2).e;
  const int64_t x = 1 + (int64_t)blockIdx.x * 32 + threadIdx.x;
  if (x >= g.nx) return;
  // two rows per thread
  for (int64_t y = 1 + (int64_t)blockIdx.y * 8 + threadIdx.y; y < g.ny; y += (int64_t)gridDim.y * 8) {
    const int64_t p = y * g.sy + x, o = y * g.syw + x;
    if (!MFWH_IDX(g.fault, p, g.points) || !MFWH_IDX(g.fault, o, g.wpoints)) continue;
    const bool two = y + 4 < g.ny && MFWH_IDX(g.fault, p + 4 * g.sy, g.points) &&
                     MFWH_IDX(g.fault, o + 4 * g.syw, g.wpoints);
    const int64_t p2 = two ? p + 4 * g.sy : p;
    int64_t S[2][STEPS];
    float r[2][STEPS];
#pragma unroll
    for (int s = 0; s < STEPS; ++s) {
      S[0][s] = S[1][s] = 0;
      r[0][s] = r[1][s] = 0.0f;
    }
    constexpr int MG = 4;   // frequencies at a time: their loads are in flight together
    for (int m0 = 0; m0 < a.nf; m0 += MG) {
      double v[2][MG];
#pragma unroll
      for (int j = 0; j < MG; ++j) {
        const bool is = m0 + j < a.nf;
        v[0][j] = is ? f[(m0 + j) * g.points + p] : 0.0;
        v[1][j] = is ? f[(m0 + j) * g.points + p2] : 0.0;
      }
#pragma unroll
      for (int j = 0; j < MG; ++j) {
        if (m0 + j >= a.nf) break;
        int hi[2];
        float hf[2], lf[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          int lo;
          fx_digits(fx_from_bits((uint64_t)__double_as_longlong(v[k][j]), sc.fe), hi[k], lo);
          hf[k] = (float)hi[k];
          lf[k] = (float)lo;
        }
#pragma unroll
        for (int s = 0; s < STEPS; ++s) {
          const int i = (m0 + j) * 8 + s;
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            S[k][s] += (int64_t)a.gh[i] * hi[k];
            r[k][s] = fmaf(a.glf[i], hf[k], fmaf(a.ghf[i], lf[k], r[k][s]));
          }
        }
      }
    }
    // |r| <= 16 (2^26 2^-1 + 2^31 2^-5) < 2^31
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int s = 0; s < STEPS; ++s)
        if (s < a.steps && (k == 0 || two))
          force[s * g.wpoints + o + k * 4 * g.syw] =
              fx_rescale(S[k][s] + __float2int_rn(r[k][s]), sh);
  }
  pdl_release();
}

// The first quantum, which puts max |W^0| and the forcing's part of the first levels below 2^58;
// mode 1 for values that are not finite or too near the ends of the double range.  Resets wmax for
// the next wave solve.
__global__ void k_fx_scale(unsigned long long* wmax, const FxForcing* forcing, double gf_dt2, int wsum,
                           FxScale* out, FxState* state) {
  pdl_begin();
  auto usable = [](double v) { return v == 0.0 || (v > 1e-250 && v < 1e250); };
  const double w = __longlong_as_double((int64_t)*wmax);
  const double fs = gf_dt2 > 0.0 ? gf_dt2 * forcing->fsum : 0.0;
  FxScale sc;
  sc.fe = forcing->fe;
  sc.mode = usable(w) && usable(fs) && (gf_dt2 == 0.0 || usable(forcing->fsum)) ? 0 : 1;
  sc.fm = 0.0f;
  sc.fx = 0;
  int ex = 58;
  if (sc.mode == 0) {
    if (fs > 0.0) sc.fm = __double2float_ru(frexp(fs, &sc.fx));
    if (fs > w)
      ex = sc.fx;
    else if (w > 0.0)
      frexp(w, &ex);   // w < 2^ex
  }
  *out = sc;
  state[0].e = ex - 58;
  state[0].eq = ex + wsum - 62;
  // w in quanta, rounded up
  state[0].wmax = sc.mode == 0 && w > 0.0 ? (unsigned long long)ldexp(w, 58 - ex) + 1 : 0ull;
  state[0].dmax = 0;
  state[1].wmax = state[1].dmax = 0;
  state[2].wmax = state[2].dmax = 0;
  *wmax = 0;
}

struct FxInit {
  double w0[MFWH_MAX_NF];
  int wexp[MFWH_MAX_NF];
};

// W^0 in quanta and q_m = w_{0,m} W^0.
__global__ void __launch_bounds__(256)
k_fx_init(int64_t* W, int64_t* q, int nf, const FxInit a, const FxScale* scale,
          const FxState* state, const Geom g, int64_t tiles_x, int vy) {
  pdl_begin();
  const int64_t x = (int64_t)blockIdx.x * 32 + threadIdx.x;
  const int64_t y = (int64_t)blockIdx.y * 8 + threadIdx.y;
  const int64_t i = y * g.syw + x;
  if (x >= g.syw || y > g.ny || !MFWH_IDX(g.fault, i, g.wpoints)) return;
  const double w = __longlong_as_double(W[i]);
  if (!scale->mode) W[i] = fx_from_bits((uint64_t)__double_as_longlong(w), state->e);
  if (x >= tiles_x * kFxTileX) return;
  const int64_t o = (y / vy * tiles_x + x / kFxTileX) * nf * kFxTile + y % vy * kFxTileX +
                    x % kFxTileX;
  if (!MFWH_IDX(g.fault, o + (nf - 1) * kFxTile, (g.ny + vy) / vy * tiles_x * nf * kFxTile)) return;
  int64_t* qp = q + o;
  for (int m = 0; m < nf; ++m) {
    const double t = a.w0[m] * w;
    qp[m * kFxTile] = scale->mode ? __double_as_longlong(t)
                                      : fx_from_bits((uint64_t)__double_as_longlong(t),
                                                     state->eq - a.wexp[m]);
  }
}

FxFn fx_fn(int nf) {
  if (nf <= 3) return fx_fn_p1(nf);
  if (nf <= 6) return fx_fn_p2(nf);
  if (nf <= 8) return fx_fn_p3(nf);
  if (nf <= 11) return fx_fn_p4(nf);
  if (nf <= 14) return fx_fn_p5(nf);
  return fx_fn_p6(nf);
}

}  // namespace

// A launch takes about ceil(tiles / SMs) + 0.7 times the time of a tile (0.7: the sums of the last
// one), which is that of its rows, 4 per step warp, and a fixed part worth about 3 warps.  Measured
// per launch of 8 steps, N_f = 8: 65^2 10.4 us with 5 warps, 19.6 with 12; 257^2 13.4 with 7, 14.1
// with 8; 513^2 31.8, 26.4, 28.7, 33.6 with 8, 9, 10, 12; 1025^2 81.4 with 11, 75.7 with 12.
int fx_warps(int64_t nx, int64_t ny, int sms) {
  int best = kFxStep;
  double cost = 0.0;
  for (int w = kFxStep; w > 4; --w) {
    const int64_t t = fx_tiles(nx, ny, w);
    const double c = ((double)((t + sms - 1) / sms) + 0.7) * (w + 3.0);
    if (w == kFxStep || c < cost) {
      best = w;
      cost = c;
    }
  }
  return best;
}

void launch_fx_forcing(int nf, const Geom& g, const double* f, unsigned long long* fmax,
                       FxForcing* unit, cudaStream_t st) {
  cudaMemsetAsync(fmax, 0, sizeof(unsigned long long) * nf, st);
  const unsigned bx = (unsigned)((g.syw + 31) / 32), by = (unsigned)((g.ny + 1 + 7) / 8);
  const unsigned cap = bx < 128 ? 512 / bx + 1 : 4;
  k_fx_fmax<<<dim3(bx, by < cap ? by : cap, (unsigned)nf), dim3(32, 8), 0, st>>>(f, g, fmax);
  k_fx_funit<<<1, 1, 0, st>>>(fmax, nf, unit);
}

void launch_fx_init(int nf, const Geom& g, const double* v, int64_t* W, int64_t* q,
                    const double* w0, const int* wexp, int wsum, int warps,
                    double gf_dt2, unsigned long long* wmax, const FxForcing* forcing, FxScale* scale,
                    FxState* state, cudaStream_t st) {
  FxInit a;
  for (int m = 0; m < nf; ++m) {
    a.w0[m] = w0[m];
    a.wexp[m] = wexp[m];
  }
  const unsigned bx = (unsigned)((g.syw + 31) / 32), by = (unsigned)((g.ny + 1 + 7) / 8);
  const unsigned cap = bx < 512 ? 2048 / bx + 1 : 4;   // blocks of the reduction: a few per SM
  k_fx_sum<<<dim3(bx, by < cap ? by : cap), dim3(32, 8), 0, st>>>(v, nf, W, g, wmax);
  launch_dependent(k_fx_scale, dim3(1), dim3(1), 0, st, wmax, forcing, gf_dt2, wsum, scale, state);
  launch_dependent(k_fx_init, dim3(bx, by), dim3(32, 8), 0, st, W, q, nf, a, scale, state, g,
                   (g.nx + kFxTileX) / kFxTileX, 4 * warps - 16);
}

void launch_fx2d(int nf, const Geom& g, const FxArrays& in, const FxArrays& out, int64_t* q,
                 double* vout, const double* vsub, const FxHost& h, cudaStream_t st) {
  if (h.forced) {
    FxForceArgs a;
    a.gw = fx_up(h.gw);
    a.gd = fx_up(h.gd);
    a.wsum = h.wsum;
    a.steps = h.steps;
    a.nf = nf;
    int ex;
    std::frexp(h.dt2, &ex);   // the coefficients are at most dt^2 < 2^ex
    a.ce = ex - 59;
    for (int m = 0; m < nf; ++m)
      for (int s = 0; s < 8; ++s) {
        const double fc = s < h.steps ? fx_forcing_coef(h, h.n0 + s, nf, m) : 0.0;
        int lo;
        fx_digits((int64_t)std::llrint(std::ldexp(fc, -a.ce)), a.gh[m * 8 + s], lo);
        a.ghf[m * 8 + s] = std::ldexp((float)a.gh[m * 8 + s], -32);
        a.glf[m * 8 + s] = std::ldexp((float)lo, -32);
      }
    const unsigned bx = (unsigned)((g.nx + 30) / 32), by = (unsigned)((g.ny + 6) / 8);
    const unsigned held = 4u * (unsigned)h.sms;   // blocks that the SMs hold
    const unsigned cap = bx < held ? held / bx : 1;
    auto* fn = g.order == 4 ? k_fx_force<4> : k_fx_force<8>;
    const dim3 grid(bx, by < cap ? by : cap);
    const FxState* state = h.state + h.n0 / fx_launch_steps(g.order) % 3;
    // A dependent launch saves 2 us; of more blocks than a few SMs hold, those that come early fill
    // the SMs that k_fx2d leaves idle and take longer there (401^2, N_f = 16: 9.4 ms against 8.1 a map).
    if (grid.x * grid.y < (unsigned)h.sms)
      launch_dependent(fn, grid, dim3(32, 4), 0, st, h.f, h.force, a, h.scale, state, g);
    else
      fn<<<grid, dim3(32, 4), 0, st>>>(h.f, h.force, a, h.scale, state, g);
  }
  fx_fn(nf)(g, in, out, q, vout, vsub, h, st);
}

}  // namespace mfwh
