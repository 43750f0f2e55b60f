// Warm-start predictor for MFWH: a small convolutional network that maps a forcing f_m and
// its frequency omega_m to an initial iterate V_m^0 for GMRES (the learned warm start; the
// paper itself starts from zero).  L layers of 3 x 3 "same" convolutions (zero padding) with
// bias, ReLU after every layer but the last, images [B][C][H][W].
//
// Arithmetic: activations and weights in BF16, products accumulated in FP32 on the
// 5th-generation tensor cores (tcgen05.mma with the accumulator in tensor memory, operands in
// shared memory: an implicit GEMM whose rows are 128 consecutive pixels of the batch and whose
// reduction runs over (input channel, tap)), for the forward convolutions and the input
// gradients; gradients, master weights and the Adam state in FP32.  The weight gradient, a
// reduction over every pixel of the batch, runs on the FP32 CUDA cores.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <random>
#include <string>
#include <type_traits>
#include <vector>

#include "internal.h"
#include "kernels.h"
#include "mfwh.h"

namespace mfwh {
namespace {

__host__ __device__ inline int round_up(int x, int m) { return (x + m - 1) / m * m; }

// ---- 3 x 3 convolution as an implicit GEMM on the 5th-generation tensor cores ----------
// D[p][n] = sum_k A[p][k] B[n][k] with p a pixel, n an output channel and k the position of
// (input channel ci, tap = dy * 3 + dx) in the order of conv_kidx below: A[p][k] =
// in[ci][y + dy - 1][x + dx - 1] (zero outside the image), B[n][k] = Wk[n][k].
//
// Layout.  The network's own images are channel-innermost, [B][H][W][Cp] with the channels
// padded with zeros to Cp = 8, 16 or 32 (chan_pad), so that the 8 channels of one tap of one
// pixel, a core-matrix row of A, are 16 consecutive bytes.  A persistent CTA of 128 threads
// walks over tiles of 128 consecutive pixels (M = 128, all output channels N = 16 or 32).
// Thread t copies pixel t's taps straight into the canonical K-major layout without swizzle by
// cp.async (16 bytes each, zeros outside the image): 8 x 16-byte core matrices, the 16 row
// groups of a k-chunk 128 bytes apart (the descriptor's stride byte offset), successive k-chunks
// 16 * 128 bytes apart (its leading byte offset).  B (all of K, loaded once per CTA) likewise
// with N / 8 row groups.  One thread issues the tile's MMAs (tcgen05.mma, kind::f16, BF16
// operands, FP32 accumulator in tensor memory), channel groups outermost, and commits them to an
// mbarrier (bounded wait); the next tile's copies are issued before the epilogue, in which every
// warp reads its 32 rows of the accumulator (tcgen05.ld) and applies bias and ReLU, or, for the
// input gradient, the ReLU mask of the layer below, and writes FP32 and BF16 in one pass.
//
// What bounds it: the L2-to-shared copies (576 bytes per pixel of a 32-channel layer, most of them
// L1 hits) and their latency; two CTAs per SM (92 KB each) cover each other's waits.  The K order
// and the MMA shape are those of the planar form it replaces, so the outputs are bit-identical.
// One training step of 48 images of 129^2, 5 layers of 32 channels, with a prediction on 12 images:
// 34.7 ms with planar images (rows staged and transposed in shared memory per tile, the weight
// gradient by one CTA per channel pair), 2.85 ms in this form.
constexpr int kConvM = 128;              // pixels per CTA (accumulator lanes)
constexpr int kConvTmemCols = 32;        // tensor-memory columns allocated per CTA (N <= 32)
constexpr int kConvMaxKp = 288;          // 32 input channels x 9 taps

// K order.  The input channels are taken in groups of GC = 8 (at most 8 channels) or 16;
// within a group k = tap * GC + c (c the channel within the group, tap = dy * 3 +
// dx), padded to a multiple of 16 (9 x 8 = 72 -> 80; 9 x 16 = 144).  So each 8-value k-chunk is
// one tap of 8 consecutive channels.
__host__ __device__ constexpr int conv_group(int cin) { return cin <= 8 ? 8 : 16; }
__host__ __device__ constexpr int conv_pass_k(int gc) { return (9 * gc + 15) / 16 * 16; }
// Padded K of a convolution with cin input channels, and the position of (ci, tap) in it.
__host__ __device__ constexpr int conv_kp(int cin) {
  return (cin + conv_group(cin) - 1) / conv_group(cin) * conv_pass_k(conv_group(cin));
}
__host__ __device__ constexpr int conv_kidx(int cin, int ci, int tap) {
  return ci / conv_group(cin) * conv_pass_k(conv_group(cin)) + tap * conv_group(cin) +
         ci % conv_group(cin);
}

// Channels of an image in memory: a whole number of groups.
__host__ __device__ constexpr int chan_pad(int c) {
  return (c + conv_group(c) - 1) / conv_group(c) * conv_group(c);
}

// Dynamic shared memory of k_conv_tc: A and B of all of K.
__host__ __device__ constexpr size_t conv_smem_bytes(int nt, int kp) {
  return (size_t)kp / 8 * (kConvM / 8) * 128 + (size_t)kp / 8 * (nt / 8) * 128;
}

// Asynchronous 16-byte copy global -> shared; src_bytes = 0 writes zeros and reads nothing.
__device__ __forceinline__ void copy16_async(uint32_t dst, const void* src, int src_bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
               "r"(src_bytes)
               : "memory");
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor (tcgen05): start address, leading byte offset (between core
// matrices along K), stride byte offset (between 8-row groups), all >> 4; descriptor version 1
// (bit 46); no swizzle (layout type 0 in bits 61-63).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), BF16 A and B (bits 7-9
// and 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 in bits 17-22, M >> 4 in bits 24-28.
__host__ __device__ constexpr uint32_t conv_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(kConvM >> 4) << 24);
}

// Bounded wait for phase `parity` of an mbarrier; false when the bound ran out.
__device__ __forceinline__ bool conv_mbar_wait(uint32_t bar, uint32_t parity, int limit) {
  for (int it = 0; it < limit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// in: [B][H][W][Cp]; out_bf: [B][H][W][Cop] BF16 (Cop = chan_pad(Cout) <= NT), out_f:
// [B][H][W][Fp] FP32 (Fp = 1 for one output channel, else Cop); mask (BF16, as out_bf): outputs
// are zeroed where it is not positive.
template <int NT, int GC>
__global__ void __launch_bounds__(kConvM)
k_conv_tc(const __nv_bfloat16* __restrict__ in, const __nv_bfloat16* __restrict__ Wk,
          const float* __restrict__ bias, int Cp, int Cout, int Kp, int Np, int64_t total, int H,
          int W, int relu, const __nv_bfloat16* __restrict__ mask,
          __nv_bfloat16* __restrict__ out_bf, float* __restrict__ out_f, int Cop, int Fp,
          int* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char conv_smem[];
  __shared__ __align__(8) uint64_t mma_bar;
  __shared__ uint32_t tmem_base;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int nk = Kp / 8;                                  // k-chunks of 8 (Kp = conv_kp(Cin))
  constexpr int kPassChunks = conv_pass_k(GC) / 8;        // 18 (GC = 16) or 10 (GC = 8)
  constexpr int kGroups = GC / 8;                         // k-chunks per tap
  constexpr uint32_t kSbo = 128;                          // 8-row groups 128 bytes apart
  constexpr uint32_t kLboA = (kConvM / 8) * 128;          // 2048 bytes per k-chunk of A
  constexpr uint32_t kLboB = (NT / 8) * 128;              // bytes per k-chunk of B
  const uint32_t sA = smem_u32(conv_smem);                // kConvM x Kp BF16
  unsigned char* sBp = conv_smem + (size_t)nk * kLboA;    // NT x Kp BF16
  const uint32_t sB = smem_u32(sBp);
  const int64_t plane = (int64_t)H * W;
  const int64_t tiles = (total + kConvM - 1) / kConvM;
  const uint32_t bar = smem_u32(&mma_bar);

  if (warp == 0) {   // tensor memory for the accumulator (whole warp, aligned)
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_base)),
                 "r"(kConvTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // Copies of a tile's rows of A: this thread's pixel, one 16-byte chunk per tap and 8 channels.
  const uint32_t arow = sA + (tid >> 3) * kSbo + (tid & 7) * 16;
  auto load_tile = [&](int64_t tile) {
    const int64_t pix = tile * kConvM + tid;
    const bool valid = pix < total;
    const int64_t rem = valid ? pix % plane : 0;
    const int y = (int)(rem / W), x = (int)(rem - (int64_t)y * W);
    const __nv_bfloat16* src = in + (valid ? pix : 0) * Cp;
    uint32_t dst = arow;
    for (int c0 = 0; c0 < nk; c0 += kPassChunks) {
#pragma unroll
      for (int kc = 0; kc < kPassChunks; ++kc) {
        const int tap = kc / kGroups, g = kc - tap * kGroups;
        const int dy = tap / 3 - 1, dx = tap % 3 - 1;
        const bool is = tap < 9 && valid && y + dy >= 0 && y + dy < H && x + dx >= 0 && x + dx < W;
        copy16_async(dst, is ? src + ((int64_t)dy * W + dx) * Cp + 8 * g : in, is ? 16 : 0);
        dst += kLboA;
      }
      src += GC;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  int64_t tile = blockIdx.x;
  load_tile(tile);   // the grid has at most one CTA per tile
  // B: NT rows of the weights (rows Np .. NT - 1 zero), 16 bytes per (row, k-chunk)
  for (int e = tid; e < NT * nk; e += kConvM) {
    const int n = e / nk, kc = e - n * nk;
    uint4 row = make_uint4(0u, 0u, 0u, 0u);
    if (n < Np) row = *reinterpret_cast<const uint4*>(Wk + (size_t)n * Kp + kc * 8);
    *reinterpret_cast<uint4*>(sBp + (size_t)kc * kLboB + (n >> 3) * kSbo + (n & 7) * 16) = row;
  }

  bool ok = true;
  uint32_t parity = 0;
  for (; tile < tiles; tile += gridDim.x, parity ^= 1) {
    // this tile's A has arrived; make the operands visible to the tensor core's asynchronous
    // proxy, then issue
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t taddr = tmem_base;
    if (tid == 0) {
      constexpr uint32_t idesc = conv_idesc(NT);
      for (int ks = 0; ks < nk / 2; ++ks) {
        const uint64_t ad = smem_desc(sA + ks * 2 * kLboA, kLboA, kSbo);
        const uint64_t bd = smem_desc(sB + ks * 2 * kLboB, kLboB, kSbo);
        const uint32_t acc = ks > 0 ? 1u : 0u;
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(taddr),
            "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
            : "memory");
      }
      asm volatile(
          "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
              bar)
          : "memory");
    }
    ok = conv_mbar_wait(bar, parity, 1 << 22);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (__syncthreads_or(!ok)) {
      ok = false;
      break;
    }
    // A is free again: the next tile's copies run under this tile's epilogue
    if (tile + gridDim.x < tiles) load_tile(tile + gridDim.x);
    // accumulator row tid (lanes 32 warp .. 32 warp + 31), NT columns
    float accv[NT];
    const uint32_t lane_addr = taddr + ((uint32_t)(warp * 32) << 16);
    uint32_t r[NT];
    if constexpr (NT == 16) {
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
          "%14,%15}, [%16];"
          : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
            "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
            "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
          : "r"(lane_addr));
    } else {
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
          "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
          : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
            "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
            "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
            "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
            "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
            "=r"(r[31])
          : "r"(lane_addr));
    }
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    const int64_t pix = tile * kConvM + tid;
    if (pix < total) {
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        float v = __uint_as_float(r[n]) + ((bias && n < Cout) ? bias[n] : 0.0f);
        accv[n] = relu ? fmaxf(v, 0.0f) : v;
      }
#pragma unroll
      for (int n0 = 0; n0 < NT; n0 += 8) {   // 8 channels at a time (columns past Cout are 0)
        if (n0 >= Cop) break;
        if (mask) {
          const uint4 mk = *reinterpret_cast<const uint4*>(mask + pix * Cop + n0);
          const uint32_t mw[4] = {mk.x, mk.y, mk.z, mk.w};
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float av = __uint_as_float((j & 1) ? mw[j >> 1] & 0xFFFF0000u : mw[j >> 1] << 16);
            if (!(av > 0.0f)) accv[n0 + j] = 0.0f;
          }
        }
        if (out_f) {
          if (Fp == 1) {
            if (n0 == 0) out_f[pix] = accv[0];
          } else {
#pragma unroll
            for (int j = 0; j < 8; j += 4)
              *reinterpret_cast<float4*>(out_f + pix * Fp + n0 + j) = make_float4(
                  accv[n0 + j], accv[n0 + j + 1], accv[n0 + j + 2], accv[n0 + j + 3]);
          }
        }
        if (out_bf) {
          uint32_t pk[4];
#pragma unroll
          for (int j = 0; j < 8; j += 2) {
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(accv[n0 + j], accv[n0 + j + 1]);
            pk[j >> 1] = *reinterpret_cast<const uint32_t*>(&h2);
          }
          *reinterpret_cast<uint4*>(out_bf + pix * Cop + n0) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
        }
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");   // the next MMAs come after
  }
  if (!ok) {
    // The MMAs did not complete within the bound: report it, give their commit one more bounded
    // wait, release the tensor memory and stop.
    if (tid == 0) atomicExch(err, 1);
    conv_mbar_wait(bar, parity, 1 << 22);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                 "r"(kConvTmemCols)
                 : "memory");
  }
}

// ---- weight and bias gradients -------------------------------------------------------------
// gw[co][ci][tap] = sum_{b,y,x} g[b][y][x][co] in[b][y + dy - 1][x + dx - 1][ci] and gb[co] =
// sum g[b][y][x][co], products and sums in FP32 on the CUDA cores (g is FP32, so a BF16
// tensor-core product would round it; 2 * 9 * Cin * Cout flops per pixel).
//
// A persistent CTA of 8 warps walks over strips of the images (up to kWgX columns by kWgRows
// rows of one image, fewer where the images make fewer strips than CTAs: one row after the other,
// each behind a barrier, a strip of 16 rows takes 16 us however few columns it has; FULL: kWgRows,
// known at compile time).  The rows it needs are in shared memory: four rows of `in` (the three of
// the window and the one being copied) and two of g, copied a row ahead by cp.async.  A warp
// takes CO output channels and one part of the strip's columns, a lane one input channel (Cp < 32:
// 32 / Cp lanes share a channel and split the columns again).  The lane keeps its CO x 9 sums and
// the 3 x 3 window of `in` in registers: one step along x loads 3 values of `in` and CO of g (as
// broadcast 16-byte loads) for 9 CO multiply-adds, so the FP32 pipe bounds it.  Every warp writes
// its sums to its own slot and k_wgrad_sum adds the slots in order, so the result does not depend
// on the schedule.
constexpr int kWgX = 64, kWgRows = 16, kWgWarps = 8;

// Column parts of a strip = slots per CTA: warps per group of output channels.
__host__ __device__ constexpr int wgrad_parts(int cout) {
  return cout <= 8 ? kWgWarps : (cout <= 16 ? kWgWarps / 2 : kWgWarps / 4);
}

template <int CO, bool FULL>
__global__ void __launch_bounds__(32 * kWgWarps, 2)
k_wgrad(const __nv_bfloat16* __restrict__ in, const float* __restrict__ g, int Cp, int Cin,
        int Cout, int Gp, int B, int H, int W, int xc, int chunks, int rows_arg, int segs,
        float* __restrict__ part) {
  const int rows = FULL ? kWgRows : rows_arg;
  extern __shared__ __align__(16) unsigned char wg_smem[];
  const int inrow = (xc + 2) * Cp;                                   // BF16 values of a row
  __nv_bfloat16* s_in = reinterpret_cast<__nv_bfloat16*>(wg_smem);   // [4][xc + 2][Cp]
  float* s_g = reinterpret_cast<float*>(wg_smem + (size_t)4 * inrow * 2);   // [2][xc][Gp]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int parts = wgrad_parts(Cout), subs = 32 / Cp;
  const int cg = warp / parts, pg = warp - cg * parts, co0 = cg * CO;
  const int ci = lane & (Cp - 1), sub = lane / Cp;
  const bool active = co0 < Cout;
  float acc[CO][9];
#pragma unroll
  for (int c = 0; c < CO; ++c)
#pragma unroll
    for (int t = 0; t < 9; ++t) acc[c][t] = 0.0f;
  float accb = 0.0f;
  const int64_t items = (int64_t)B * chunks * segs;
  for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
    const int seg = (int)(it % segs), ch = (int)(it / segs % chunks), b = (int)(it / segs / chunks);
    const int x0 = ch * xc, xn = W - x0 < xc ? W - x0 : xc;
    const int y0 = seg * rows, yn = H - y0 < rows ? H - y0 : rows;
    // copy row y of `in` (columns x0 - 1 .. x0 + xn, zeros outside the image) into slot y & 3
    auto copy_in = [&](int y) {
      const int per = Cp / 8, n = (xn + 2) * per;
      const bool row = y >= 0 && y < H;
      const __nv_bfloat16* src = in + ((int64_t)b * H + (row ? y : 0)) * W * Cp;
      const uint32_t dst = smem_u32(s_in + (size_t)(y & 3) * inrow);
      for (int e = tid; e < n; e += 32 * kWgWarps) {
        const int c = e / per, x = x0 - 1 + c;
        const bool is = row && x >= 0 && x < W;
        copy16_async(dst + e * 16, is ? src + (int64_t)(x0 - 1) * Cp + e * 8 : in, is ? 16 : 0);
      }
    };
    auto copy_g = [&](int y) {   // row y of g into slot y & 1
      const float* src = g + (((int64_t)b * H + y) * W + x0) * Gp;
      float* dst = s_g + (size_t)(y & 1) * xc * Gp;
      if constexpr (CO == 1) {
        for (int e = tid; e < xn; e += 32 * kWgWarps) dst[e] = src[e];
      } else {
        for (int e = tid; e < xn * Gp / 4; e += 32 * kWgWarps)
          copy16_async(smem_u32(dst + e * 4), src + e * 4, 16);
      }
    };
    __syncthreads();   // the previous strip's rows have been read
    copy_in(y0 - 1);
    copy_in(y0);
    copy_in(y0 + 1);
    copy_g(y0);
    asm volatile("cp.async.commit_group;" ::: "memory");
    // the warp's columns, and the lane's among them
    const int w0 = pg * xn / parts, w1 = (pg + 1) * xn / parts;
    const int xs = w0 + sub * (w1 - w0) / subs, xe = w0 + (sub + 1) * (w1 - w0) / subs;
    for (int y = y0; y < y0 + yn; ++y) {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();
      if (y + 1 < y0 + yn) {
        copy_in(y + 2);
        copy_g(y + 1);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      if (!active) continue;
      const float* gr = s_g + (size_t)(y & 1) * xc * Gp + co0;
      const __nv_bfloat16* r[3];
      float wnd[3][3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        r[d] = s_in + (size_t)((y - 1 + d) & 3) * inrow + ci;
        wnd[d][1] = xs < xe ? __bfloat162float(r[d][xs * Cp]) : 0.0f;
        wnd[d][2] = xs < xe ? __bfloat162float(r[d][(xs + 1) * Cp]) : 0.0f;
      }
      for (int x = xs; x < xe; ++x) {
        float gv[CO];
        if constexpr (CO == 8) {
          const float4 g0 = *reinterpret_cast<const float4*>(gr + x * Gp);
          const float4 g1 = *reinterpret_cast<const float4*>(gr + x * Gp + 4);
          gv[0] = g0.x; gv[1] = g0.y; gv[2] = g0.z; gv[3] = g0.w;
          gv[4] = g1.x; gv[5] = g1.y; gv[6] = g1.z; gv[7] = g1.w;
        } else {
          gv[0] = gr[x * Gp];
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          wnd[d][0] = wnd[d][1];
          wnd[d][1] = wnd[d][2];
          wnd[d][2] = __bfloat162float(r[d][(x + 2) * Cp]);
        }
#pragma unroll
        for (int c = 0; c < CO; ++c)
#pragma unroll
          for (int t = 0; t < 9; ++t) acc[c][t] = fmaf(gv[c], wnd[t / 3][t % 3], acc[c][t]);
      }
      // the bias: lane (i, c) adds channel co0 + c of the warp's columns w0 + i, w0 + i + 32/CO ..
      for (int x = w0 + lane / CO; x < w1; x += 32 / CO) accb += gr[x * Gp + lane % CO];
    }
  }
  if (!active) return;
  // the warp's slot: [Cout][Cin][9], then the Cout bias sums
  const int E = Cout * Cin * 9 + Cout;
  float* slot = part + ((int64_t)blockIdx.x * parts + pg) * E;
#pragma unroll
  for (int c = 0; c < CO; ++c)
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      float v = acc[c][t];
      for (int o = Cp; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane < Cin && co0 + c < Cout) slot[((co0 + c) * Cin + ci) * 9 + t] = v;
    }
  for (int o = CO; o < 32; o <<= 1) accb += __shfl_xor_sync(0xffffffffu, accb, o);
  if (lane < CO && co0 + lane < Cout) slot[Cout * Cin * 9 + co0 + lane] = accb;
}

// out[e] = (add: out[e] +) the sum over the slots of part[slot][e]: 8 interleaved partial sums per
// output.
__global__ void __launch_bounds__(256)
k_wgrad_sum(const float* __restrict__ part, int slots, int E, int add, float* __restrict__ out) {
  const int e = blockIdx.x * 32 + (threadIdx.x & 31), s0 = threadIdx.x >> 5;
  float v = 0.0f;
  if (e < E)
    for (int s = s0; s < slots; s += 8) v += part[(int64_t)s * E + e];
  __shared__ float red[8][32];
  red[s0][threadIdx.x & 31] = v;
  __syncthreads();
  if (s0 == 0 && e < E) {
#pragma unroll
    for (int i = 1; i < 8; ++i) v += red[i][threadIdx.x];
    out[e] = add ? out[e] + v : v;
  }
}

// Planar FP32 images [B][C][plane] to channel-innermost BF16 [B][plane][Cp] (zeros past C).
__global__ void k_to_images(const float* __restrict__ x, __nv_bfloat16* __restrict__ y, int C,
                            int Cp, int64_t plane, int64_t pixels) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < pixels;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = i / plane, r = i - b * plane;
    for (int c0 = 0; c0 < Cp; c0 += 8) {
      uint32_t pk[4];
#pragma unroll
      for (int j = 0; j < 8; j += 2) {
        const float lo = c0 + j < C ? x[(b * C + c0 + j) * plane + r] : 0.0f;
        const float hi = c0 + j + 1 < C ? x[(b * C + c0 + j + 1) * plane + r] : 0.0f;
        const __nv_bfloat162 h2 = __floats2bfloat162_rn(lo, hi);
        pk[j >> 1] = *reinterpret_cast<const uint32_t*>(&h2);
      }
      *reinterpret_cast<uint4*>(y + i * Cp + c0) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
    }
  }
}

// Sum of the mask's values (one block, FP64) and 1 / max(1, sum * batch), the mean's factor.
__global__ void __launch_bounds__(1024)
k_mask_sum(const float* __restrict__ mask, int64_t n, int B, float* __restrict__ inv) {
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) s += mask[i];
  __shared__ double red[32];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int w = 0; w < 32; ++w) v += red[w];
    v *= B;
    *inv = (float)(1.0 / (v > 1.0 ? v : 1.0));
  }
}

// Masked mean squared error: g = 2 (y - t) m / count (FP32, and BF16 images of 8 channels, 7 of
// them 0), partial sums of (y - t)^2 m per block (add: on those of the images before).
__global__ void __launch_bounds__(256)
k_mse(const float* __restrict__ y, const float* __restrict__ t, const float* __restrict__ mask,
      int64_t plane, int64_t n, const float* __restrict__ inv_count, float* __restrict__ g,
      __nv_bfloat16* __restrict__ gbf, int add, float* __restrict__ part) {
  const float inv = *inv_count;
  float s = 0.0f;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float d = (y[i] - t[i]) * mask[i % plane];
    const float gi = 2.0f * d * inv;
    g[i] = gi;
    *reinterpret_cast<uint4*>(gbf + i * 8) =
        make_uint4(__bfloat16_as_ushort(__float2bfloat16(gi)), 0u, 0u, 0u);
    s = fmaf(d, d, s);
  }
  __shared__ float red[8];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float v = 0.0f;
    for (int w = 0; w < 8; ++w) v += red[w];
    part[blockIdx.x] = add ? part[blockIdx.x] + v : v;
  }
}

// Adam (bias-corrected moments) on the FP32 master parameters.
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int64_t n, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// BF16 GEMM layouts of one layer's weights w[co][ci][3][3] in the K order of conv_kidx: forward
// Wk[co][kidx(ci, tap)] and, for the input gradient, the flipped transpose
// Wt[ci][kidx(co, 8 - tap)].
__global__ void k_pack(const float* __restrict__ w, int Cin, int Cout, int Kp, int Kpt,
                       __nv_bfloat16* __restrict__ Wk, __nv_bfloat16* __restrict__ Wt) {
  const int n = Cout * Cin * 9;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int tap = i % 9, ci = (i / 9) % Cin, co = i / (9 * Cin);
    const __nv_bfloat16 v = __float2bfloat16(w[i]);
    Wk[(size_t)co * Kp + conv_kidx(Cin, ci, tap)] = v;
    Wt[(size_t)ci * Kpt + conv_kidx(Cout, co, 8 - tap)] = v;
  }
}

// ---- features and targets of the warm start (2D grids, H = ny + 1 rows, W = nx + 1) ----
// For frequency m: input channels x[m][0] = f_m / max|f_m| and x[m][1] = omega_m / omega_scale;
// target t[m] = V_m / max|V_m| (the shape of the solution); the prediction is that shape with
// 0 on the boundary, its amplitude fitted afterwards to the Helmholtz residual.

__global__ void k_ws_scale(const double* __restrict__ f, int64_t P, double* __restrict__ scale) {
  const int m = blockIdx.x;
  double mx = 0.0;
  for (int64_t i = threadIdx.x; i < P; i += blockDim.x) mx = fmax(mx, fabs(f[m * P + i]));
  __shared__ double red[8];
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int w = 0; w < 8; ++w) v = fmax(v, red[w]);
    scale[m] = v > 0.0 ? v : 1.0;
  }
}

struct WsFreq {
  double omega[MFWH_MAX_NF];
};

__global__ void k_ws_features(const double* __restrict__ f, const double* __restrict__ v,
                              const double* __restrict__ fscale, const double* __restrict__ vscale,
                              const WsFreq fr, int nf, int64_t P, double omega_scale,
                              float* __restrict__ x, float* __restrict__ t) {
  const int64_t n = (int64_t)nf * P;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int m = (int)(e / P);
    const int64_t i = e - (int64_t)m * P;
    x[((int64_t)m * 2) * P + i] = (float)(f[e] / fscale[m]);
    x[((int64_t)m * 2 + 1) * P + i] = (float)(fr.omega[m] / omega_scale);
    if (t) t[e] = (float)(v[e] / vscale[m]);
  }
}

__global__ void k_ws_output(const float* __restrict__ y, int nf, int H, int W,
                            double* __restrict__ v) {
  const int64_t P = (int64_t)H * W, n = (int64_t)nf * P;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e % P;
    const int xx = (int)(i % W), yy = (int)(i / W);
    const bool interior = xx > 0 && xx < W - 1 && yy > 0 && yy < H - 1;
    v[e] = interior ? (double)y[e] : 0.0;
  }
}

mfwh_status cnn_fail(mfwh_status st, const std::string& m) {
  set_error(m);
  return st;
}

}  // namespace
}  // namespace mfwh

using namespace mfwh;

struct mfwh_cnn_s {
  int layers = 0, channels = 0, in_channels = 0;
  cudaStream_t stream = nullptr;
  std::vector<int> cin, cout;          // per layer
  std::vector<int64_t> woff, boff;     // offsets of w and b in the flat parameter vector
  int64_t nparams = 0;
  float* p = nullptr;                  // FP32 master parameters
  float* grad = nullptr;               // gradients (same layout)
  float* m = nullptr;
  float* v = nullptr;
  int step = 0;
  std::vector<__nv_bfloat16*> Wk, Wt;  // BF16 GEMM layouts per layer
  std::vector<int> Kp, Kpt, Np, Npt;
  // activation workspace, sized for cap elements per channel plane times the batch
  int64_t cap = 0;                     // B * H * W the workspace holds
  int64_t refused = 0;                 // the smallest one that did not fit (0: none so far)
  std::vector<__nv_bfloat16*> act;     // inputs of each layer (BF16), [B][H][W][chan_pad(C)]
  float* y = nullptr;                  // network output [B][1][H][W]
  float* g0 = nullptr;                 // gradients of a layer's output, [B][H][W][chan_pad(C)]
  float* g1 = nullptr;                 //   (the last layer's: [B][H][W])
  __nv_bfloat16* gbf0 = nullptr;       // the same in BF16 (always padded)
  __nv_bfloat16* gbf1 = nullptr;
  float* wpart = nullptr;              // weight-gradient slots
  int sms = 0;                         // SMs of the device
  float* part = nullptr;               // loss partial sums, then the mean's factor
  float* part_h = nullptr;             // pinned
  int* err = nullptr;                  // device flag: a convolution's MMA wait ran out
};

namespace {

constexpr int kLossBlocks = 256;

#define CKC(call)                                                                  \
  do {                                                                             \
    cudaError_t e_ = (call);                                                       \
    if (e_ != cudaSuccess)                                                         \
      return cnn_fail(MFWH_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

void free_ws(mfwh_cnn_t c) {
  for (auto& a : c->act)
    if (a) cudaFree(a);
  for (float* b : {c->y, c->g0, c->g1})
    if (b) cudaFree(b);
  if (c->gbf0) cudaFree(c->gbf0);
  if (c->gbf1) cudaFree(c->gbf1);
  c->y = c->g0 = c->g1 = nullptr;
  c->gbf0 = c->gbf1 = nullptr;
  c->act.assign(c->layers, nullptr);
  c->cap = 0;
}

cudaError_t alloc_ws(mfwh_cnn_t c, int64_t bhw) {
  cudaError_t e = cudaSuccess;
  auto take = [&](auto** p, int64_t n) {
    void* v = nullptr;
    if (e == cudaSuccess) e = device_alloc(&v, sizeof(**p) * n);
    if (e == cudaSuccess) *p = static_cast<std::remove_reference_t<decltype(*p)>>(v);
  };
  const int gc = chan_pad(c->channels);
  for (int l = 0; l < c->layers; ++l) take(&c->act[l], bhw * chan_pad(c->cin[l]));
  take(&c->y, bhw);
  take(&c->g0, bhw * gc);
  take(&c->g1, bhw * gc);
  take(&c->gbf0, bhw * gc);
  take(&c->gbf1, bhw * gc);
  return e;
}

// Workspace for a batch of B images of hw pixels, or, where memory ends, for as many of them at a
// time as fit (the padded channels take up to 8 times the memory of the images' own): *images.
mfwh_status ensure_ws(mfwh_cnn_t c, int B, int64_t hw, int* images) {
  int n = B;
  if (c->refused > 0 && n * hw >= c->refused && c->cap >= hw) n = (int)(c->cap / hw);
  while (n * hw > c->cap) {
    free_ws(c);
    const cudaError_t e = alloc_ws(c, n * hw);
    if (e == cudaSuccess) {
      c->cap = n * hw;
      break;
    }
    free_ws(c);
    if (e != cudaErrorMemoryAllocation || n == 1)
      return cnn_fail(e == cudaErrorMemoryAllocation ? MFWH_ERR_NOMEM : MFWH_ERR_CUDA,
                      std::string("cnn workspace: ") + cudaGetErrorString(e));
    (void)cudaGetLastError();
    c->refused = c->refused > 0 ? std::min(c->refused, n * hw) : n * hw;
    n = (n + 1) / 2;
  }
  *images = std::min(n, B);
  return MFWH_OK;
}

// One convolution of channel-innermost images: cin -> cout channels; mask, out_bf, out_f as in
// k_conv_tc.  Two persistent CTAs per SM, or one per tile when there are fewer tiles.
void conv(mfwh_cnn_t c, const __nv_bfloat16* in, const __nv_bfloat16* Wk, const float* bias,
          int cin, int cout, int Kp, int Np, int B, int H, int W, int relu,
          const __nv_bfloat16* mask, __nv_bfloat16* out_bf, float* out_f) {
  const int64_t total = (int64_t)B * H * W;
  const unsigned blocks =
      (unsigned)std::min<int64_t>((total + kConvM - 1) / kConvM, (int64_t)2 * c->sms);
  auto launch = [&](auto kernel, int nt) {
    kernel<<<blocks, kConvM, conv_smem_bytes(nt, Kp), c->stream>>>(
        in, Wk, bias, chan_pad(cin), cout, Kp, Np, total, H, W, relu, mask, out_bf, out_f,
        chan_pad(cout), cout == 1 ? 1 : chan_pad(cout), c->err);
  };
  const bool g8 = conv_group(cin) == 8;
  if (chan_pad(cout) <= 16)
    g8 ? launch(k_conv_tc<16, 8>, 16) : launch(k_conv_tc<16, 16>, 16);
  else
    g8 ? launch(k_conv_tc<32, 8>, 32) : launch(k_conv_tc<32, 16>, 32);
}

// Weight and bias gradients of layer l from the gradient g of its output, into c->grad (w and b
// of a layer are adjacent in the flat parameter vector); add: added to those of the images before.
void wgrad(mfwh_cnn_t c, int l, const float* g, int B, int H, int W, int add) {
  const int cin = c->cin[l], cout = c->cout[l], cp = chan_pad(cin);
  const int gp = cout == 1 ? 1 : chan_pad(cout);
  const int chunks = (W + kWgX - 1) / kWgX, xc = (W + chunks - 1) / chunks;   // even strips
  const int64_t want = ((int64_t)B * chunks * H + 2 * c->sms - 1) / (2 * c->sms);
  const int rows = (int)std::min<int64_t>(kWgRows, std::max<int64_t>(2, want));
  const int segs = (H + rows - 1) / rows;
  const int blocks =
      (int)std::min<int64_t>((int64_t)B * chunks * segs, (int64_t)2 * c->sms);
  const size_t smem = (size_t)4 * (xc + 2) * cp * 2 + (size_t)2 * xc * gp * 4;
  const int E = cout * cin * 9 + cout;
  const bool full = rows == kWgRows;
  auto* fn = cout == 1 ? (full ? k_wgrad<1, true> : k_wgrad<1, false>)
                       : (full ? k_wgrad<8, true> : k_wgrad<8, false>);
  fn<<<blocks, 32 * kWgWarps, smem, c->stream>>>(c->act[l], g, cp, cin, cout, gp, B, H, W, xc, chunks,
                                                 rows, segs, c->wpart);
  k_wgrad_sum<<<(E + 31) / 32, 256, 0, c->stream>>>(c->wpart, blocks * wgrad_parts(cout), E,
                                                    add, c->grad + c->woff[l]);
}

// The convolution kernels' shared-memory limit, once per device.
mfwh_status conv_configure() {
  static bool done[64] = {};
  int dev = 0;
  CKC(cudaGetDevice(&dev));
  if (dev >= 0 && dev < 64 && done[dev]) return MFWH_OK;
  CKC(cudaFuncSetAttribute(k_conv_tc<16, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)conv_smem_bytes(16, conv_kp(8))));
  CKC(cudaFuncSetAttribute(k_conv_tc<16, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)conv_smem_bytes(16, kConvMaxKp)));
  CKC(cudaFuncSetAttribute(k_conv_tc<32, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)conv_smem_bytes(32, conv_kp(8))));
  CKC(cudaFuncSetAttribute(k_conv_tc<32, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)conv_smem_bytes(32, kConvMaxKp)));
  if (dev >= 0 && dev < 64) done[dev] = true;
  return MFWH_OK;
}

// A convolution's bounded MMA wait ran out since the last check: report it and clear the flag.
mfwh_status check_err(mfwh_cnn_t c) {
  int flag = 0;
  CKC(cudaMemcpyAsync(&flag, c->err, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  CKC(cudaStreamSynchronize(c->stream));
  if (!flag) return MFWH_OK;
  CKC(cudaMemsetAsync(c->err, 0, sizeof(int), c->stream));
  return cnn_fail(MFWH_ERR_TIMEOUT, "cnn: a convolution's tensor-core wait timed out");
}

mfwh_status pack_all(mfwh_cnn_t c) {
  for (int l = 0; l < c->layers; ++l) {   // (the padding was zeroed at creation)
    k_pack<<<32, 256, 0, c->stream>>>(c->p + c->woff[l], c->cin[l], c->cout[l], c->Kp[l],
                                      c->Kpt[l], c->Wk[l], c->Wt[l]);
  }
  CKC(cudaGetLastError());
  return MFWH_OK;
}

// The network on planar images x (as many as the workspace holds at most); its output (one
// channel) to y.
mfwh_status forward_impl(mfwh_cnn_t c, const float* x, int B, int H, int W, float* y) {
  const int64_t bhw = (int64_t)B * H * W;
  k_to_images<<<8 * c->sms, 256, 0, c->stream>>>(x, c->act[0], c->in_channels,
                                                 chan_pad(c->in_channels), (int64_t)H * W, bhw);
  for (int l = 0; l < c->layers; ++l) {
    const bool last = l + 1 == c->layers;
    conv(c, c->act[l], c->Wk[l], c->p + c->boff[l], c->cin[l], c->cout[l], c->Kp[l], c->Np[l], B,
         H, W, last ? 0 : 1, nullptr, last ? nullptr : c->act[l + 1], last ? y : nullptr);
  }
  CKC(cudaGetLastError());
  return MFWH_OK;
}

}  // namespace

extern "C" {

mfwh_status mfwh_cnn_create(int layers, int channels, int in_channels, uint64_t seed,
                            void* stream, mfwh_cnn_t* out) {
  if (!out || layers < 2 || layers > 16 || channels < 1 || channels > 32 || in_channels < 1 ||
      in_channels > 32)
    return cnn_fail(MFWH_ERR_INVALID_ARG, "cnn: 2..16 layers, 1..32 channels and inputs");
  *out = nullptr;
  auto* c = new (std::nothrow) mfwh_cnn_s();
  if (!c) return cnn_fail(MFWH_ERR_NOMEM, "host allocation failed");
  c->layers = layers;
  c->channels = channels;
  c->in_channels = in_channels;
  c->stream = static_cast<cudaStream_t>(stream);
  for (int l = 0; l < layers; ++l) {
    const int ci = l == 0 ? in_channels : channels, co = l + 1 == layers ? 1 : channels;
    c->cin.push_back(ci);
    c->cout.push_back(co);
    c->woff.push_back(c->nparams);
    c->nparams += (int64_t)co * ci * 9;
    c->boff.push_back(c->nparams);
    c->nparams += co;
    c->Kp.push_back(conv_kp(ci));
    c->Np.push_back(round_up(co, 8));
    c->Kpt.push_back(conv_kp(co));
    c->Npt.push_back(round_up(ci, 8));
  }
  // He-normal weights (std sqrt(2 / (9 Cin))), zero biases, from a seeded host generator
  std::vector<float> h(c->nparams, 0.0f);
  std::mt19937_64 rng(seed);
  for (int l = 0; l < layers; ++l) {
    std::normal_distribution<double> nd(0.0, std::sqrt(2.0 / (9.0 * c->cin[l])));
    for (int64_t i = 0; i < (int64_t)c->cout[l] * c->cin[l] * 9; ++i)
      h[c->woff[l] + i] = (float)nd(rng);
  }
  auto fail_free = [&](mfwh_status s) {
    mfwh_cnn_destroy(c);
    return s;
  };
  for (float** b : {&c->p, &c->grad, &c->m, &c->v})
    if (cudaMalloc(b, sizeof(float) * c->nparams) != cudaSuccess)
      return fail_free(cnn_fail(MFWH_ERR_NOMEM, "cnn: parameter allocation failed"));
  c->Wk.assign(layers, nullptr);
  c->Wt.assign(layers, nullptr);
  for (int l = 0; l < layers; ++l)
    if (cudaMalloc(&c->Wk[l], sizeof(__nv_bfloat16) * c->Np[l] * c->Kp[l]) != cudaSuccess ||
        cudaMalloc(&c->Wt[l], sizeof(__nv_bfloat16) * c->Npt[l] * c->Kpt[l]) != cudaSuccess)
      return fail_free(cnn_fail(MFWH_ERR_NOMEM, "cnn: weight allocation failed"));
  if (cudaMalloc(&c->part, sizeof(float) * (kLossBlocks + 1)) != cudaSuccess ||
      cudaMallocHost(&c->part_h, sizeof(float) * (kLossBlocks + 1)) != cudaSuccess ||
      cudaMalloc(&c->err, sizeof(int)) != cudaSuccess)
    return fail_free(cnn_fail(MFWH_ERR_NOMEM, "cnn: allocation failed"));
  if (cudaMemsetAsync(c->err, 0, sizeof(int), c->stream) != cudaSuccess)
    return fail_free(cnn_fail(MFWH_ERR_CUDA, "cnn: initialisation failed"));
  if (conv_configure() != MFWH_OK) return fail_free(MFWH_ERR_CUDA);
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return fail_free(cnn_fail(MFWH_ERR_CUDA, "cnn: device query failed"));
  // weight-gradient slots: at most two CTAs per SM, wgrad_parts slots each
  int64_t slots = 0;
  for (int l = 0; l < layers; ++l)
    slots = std::max(slots, (int64_t)wgrad_parts(c->cout[l]) *
                                (c->cout[l] * c->cin[l] * 9 + c->cout[l]));
  if (cudaMalloc(&c->wpart, sizeof(float) * slots * 2 * c->sms) != cudaSuccess)
    return fail_free(cnn_fail(MFWH_ERR_NOMEM, "cnn: workspace allocation failed"));
  for (int l = 0; l < layers; ++l)   // the weights' padding stays 0
    if (cudaMemsetAsync(c->Wk[l], 0, sizeof(__nv_bfloat16) * c->Np[l] * c->Kp[l], c->stream) !=
            cudaSuccess ||
        cudaMemsetAsync(c->Wt[l], 0, sizeof(__nv_bfloat16) * c->Npt[l] * c->Kpt[l], c->stream) !=
            cudaSuccess)
      return fail_free(cnn_fail(MFWH_ERR_CUDA, "cnn: initialisation failed"));
  if (cudaMemcpyAsync(c->p, h.data(), sizeof(float) * c->nparams, cudaMemcpyHostToDevice,
                      c->stream) != cudaSuccess ||
      cudaMemsetAsync(c->m, 0, sizeof(float) * c->nparams, c->stream) != cudaSuccess ||
      cudaMemsetAsync(c->v, 0, sizeof(float) * c->nparams, c->stream) != cudaSuccess ||
      cudaMemsetAsync(c->grad, 0, sizeof(float) * c->nparams, c->stream) != cudaSuccess)
    return fail_free(cnn_fail(MFWH_ERR_CUDA, "cnn: initialisation failed"));
  mfwh_status st = pack_all(c);
  if (st == MFWH_OK && cudaStreamSynchronize(c->stream) != cudaSuccess) st = MFWH_ERR_CUDA;
  if (st != MFWH_OK) return fail_free(st);
  *out = c;
  return MFWH_OK;
}

int64_t mfwh_cnn_param_count(mfwh_cnn_t c) { return c ? c->nparams : 0; }

mfwh_status mfwh_cnn_set_params(mfwh_cnn_t c, const float* host, int64_t count) {
  if (!c || !host || count != c->nparams)
    return cnn_fail(MFWH_ERR_INVALID_ARG, "cnn: parameter count mismatch");
  CKC(cudaMemcpyAsync(c->p, host, sizeof(float) * count, cudaMemcpyHostToDevice, c->stream));
  CKC(cudaMemsetAsync(c->m, 0, sizeof(float) * count, c->stream));
  CKC(cudaMemsetAsync(c->v, 0, sizeof(float) * count, c->stream));
  c->step = 0;
  mfwh_status st = pack_all(c);
  if (st != MFWH_OK) return st;
  CKC(cudaStreamSynchronize(c->stream));
  return MFWH_OK;
}

mfwh_status mfwh_cnn_get_params(mfwh_cnn_t c, float* host, float* grads_host, int64_t count) {
  if (!c || !host || count != c->nparams)
    return cnn_fail(MFWH_ERR_INVALID_ARG, "cnn: parameter count mismatch");
  CKC(cudaMemcpyAsync(host, c->p, sizeof(float) * count, cudaMemcpyDeviceToHost, c->stream));
  if (grads_host)
    CKC(cudaMemcpyAsync(grads_host, c->grad, sizeof(float) * count, cudaMemcpyDeviceToHost,
                        c->stream));
  CKC(cudaStreamSynchronize(c->stream));
  return check_err(c);
}

mfwh_status mfwh_cnn_forward(mfwh_cnn_t c, const float* x, int B, int H, int W, float* y) {
  if (!c || !x || !y || B < 1 || H < 1 || W < 1)
    return cnn_fail(MFWH_ERR_INVALID_ARG, "cnn: bad forward arguments");
  const int64_t hw = (int64_t)H * W;
  int images = 0;
  mfwh_status st = ensure_ws(c, B, hw, &images);
  for (int b = 0; b < B && st == MFWH_OK; b += images)
    st = forward_impl(c, x + b * hw * c->in_channels, std::min(images, B - b), H, W, y + b * hw);
  return st;
}

mfwh_status mfwh_cnn_train_step(mfwh_cnn_t c, const float* x, const float* target,
                                const float* mask, int B, int H, int W, float lr, float* loss) {
  if (!c || !x || !target || !mask || B < 1 || H < 1 || W < 1 || !(lr > 0.0f))
    return cnn_fail(MFWH_ERR_INVALID_ARG, "cnn: bad training arguments");
  const int64_t hw = (int64_t)H * W;
  int images = 0;
  mfwh_status st = ensure_ws(c, B, hw, &images);
  if (st != MFWH_OK) return st;
  float* inv = c->part + kLossBlocks;
  k_mask_sum<<<1, 1024, 0, c->stream>>>(mask, hw, B, inv);
  for (int b = 0; b < B; b += images) {
    const int n = std::min(images, B - b);
    st = forward_impl(c, x + b * hw * c->in_channels, n, H, W, c->y);
    if (st != MFWH_OK) return st;
    float* g = c->g0;
    float* gnext = c->g1;
    __nv_bfloat16* gb = c->gbf0;
    __nv_bfloat16* gbnext = c->gbf1;
    k_mse<<<kLossBlocks, 256, 0, c->stream>>>(c->y, target + b * hw, mask, hw, n * hw, inv, g, gb,
                                              b > 0, c->part);
    for (int l = c->layers - 1; l >= 0; --l) {
      wgrad(c, l, g, n, H, W, b > 0);
      if (l > 0) {   // the input gradient, through the ReLU of the layer below
        conv(c, gb, c->Wt[l], nullptr, c->cout[l], c->cin[l], c->Kpt[l], c->Npt[l], n, H, W, 0,
             c->act[l], gbnext, gnext);
        std::swap(g, gnext);
        std::swap(gb, gbnext);
      }
    }
  }
  c->step++;
  const float b1 = 0.9f, b2 = 0.999f;
  k_adam<<<256, 256, 0, c->stream>>>(c->p, c->grad, c->m, c->v, c->nparams, lr, b1, b2, 1e-8f,
                                     1.0f - std::pow(b1, (float)c->step),
                                     1.0f - std::pow(b2, (float)c->step));
  st = pack_all(c);
  if (st != MFWH_OK) return st;
  CKC(cudaMemcpyAsync(c->part_h, c->part, sizeof(float) * (kLossBlocks + 1),
                      cudaMemcpyDeviceToHost, c->stream));
  CKC(cudaStreamSynchronize(c->stream));
  double s = 0.0;
  for (int i = 0; i < kLossBlocks; ++i) s += c->part_h[i];
  if (loss) *loss = (float)(s * c->part_h[kLossBlocks]);
  return check_err(c);
}

void mfwh_cnn_destroy(mfwh_cnn_t c) {
  if (!c) return;
  cudaStreamSynchronize(c->stream);
  free_ws(c);
  for (float* b : {c->p, c->grad, c->m, c->v, c->part, c->wpart})
    if (b) cudaFree(b);
  for (auto* w : c->Wk)
    if (w) cudaFree(w);
  for (auto* w : c->Wt)
    if (w) cudaFree(w);
  for (auto* a : c->act)
    if (a) cudaFree(a);
  if (c->part_h) cudaFreeHost(c->part_h);
  if (c->err) cudaFree(c->err);
  delete c;
}

}  // extern "C"

namespace mfwh {

// Training pairs of one solved 2D problem (device arrays; see the feature definition above).
// scale: device scratch of 2 nf doubles.
mfwh_status cnn_ws_data(const double* f, const double* v, const double* omega, int nf, int H,
                        int W, double omega_scale, float* x, float* t, double* scale,
                        cudaStream_t st) {
  WsFreq fr{};
  for (int m = 0; m < nf; ++m) fr.omega[m] = omega[m];
  const int64_t P = (int64_t)H * W;
  k_ws_scale<<<nf, 256, 0, st>>>(f, P, scale);
  if (v) k_ws_scale<<<nf, 256, 0, st>>>(v, P, scale + nf);
  k_ws_features<<<256, 256, 0, st>>>(f, v, scale, scale + nf, fr, nf, P, omega_scale, x, t);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? MFWH_OK : cnn_fail(MFWH_ERR_CUDA, cudaGetErrorString(e));
}

// The network's solution shape for every frequency of a 2D problem (0 on the boundary).
mfwh_status cnn_ws_predict(mfwh_cnn_t c, const double* f, const double* omega, int nf, int H,
                           int W, double omega_scale, double* v, cudaStream_t st) {
  if (c->in_channels != 2) return cnn_fail(MFWH_ERR_INVALID_ARG, "warm start needs 2 inputs");
  const int64_t P = (int64_t)H * W;
  float* x = nullptr;
  float* y = nullptr;
  double* scale = nullptr;
  mfwh_status res = MFWH_OK;
  if (cudaMalloc(&x, sizeof(float) * 2 * nf * P) != cudaSuccess ||
      cudaMalloc(&y, sizeof(float) * nf * P) != cudaSuccess ||
      cudaMalloc(&scale, sizeof(double) * 2 * nf) != cudaSuccess) {
    res = cnn_fail(MFWH_ERR_NOMEM, "warm start: allocation failed");
  } else {
    res = cnn_ws_data(f, nullptr, omega, nf, H, W, omega_scale, x, nullptr, scale, st);
    cudaStream_t keep = c->stream;
    c->stream = st;
    if (res == MFWH_OK) res = mfwh_cnn_forward(c, x, nf, H, W, y);
    c->stream = keep;
    if (res == MFWH_OK) {
      k_ws_output<<<256, 256, 0, st>>>(y, nf, H, W, v);
      if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess)
        res = cnn_fail(MFWH_ERR_CUDA, "warm start: output kernel failed");
    }
    if (res == MFWH_OK) {
      c->stream = st;
      res = check_err(c);
      c->stream = keep;
    }
  }
  cudaStreamSynchronize(st);
  if (x) cudaFree(x);
  if (y) cudaFree(y);
  if (scale) cudaFree(scale);
  return res;
}

}  // namespace mfwh
