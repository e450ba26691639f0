// Learned right preconditioner: a small convolutional U-Net, trained and
// evaluated with this library's own kernels.  The paper preconditions its
// Krylov solve with FFT and diffusion solvers (Section 4.4); here a network
// maps (sigma_t, sigma_s, b) to the smooth part of (I - K)^{-1} b, and FGMRES
// (vie_solve_gmres with a preconditioner set) absorbs that it is nonlinear.
//
// Network (L levels, C channels; tensors FP32 NCHW, weights [Co][Ci][k][k]):
//   encoder l = 0..L-1: a_l = relu(conv3(x_l)), e_l = relu(conv3(a_l)),
//                       x_0 = input (3 channels), x_l = avgpool2(e_{l-1});
//   decoder l = L-2..0: c_l = [upsample2(d_{l+1}), e_l], b_l = relu(conv3(c_l)),
//                       d_l = relu(conv3(b_l)), d_{L-1} = e_{L-1};
//   output  o = conv1(d_0).
// e_l (l < L-1) is written straight into the second half of c_l's channels.
// Training minimises mean((o - t)^2) with Adam; inference can use a BF16 copy
// of the weights (FP32 accumulation either way).
#include <cuda.h>
#include <cuda_bf16.h>
#include <math.h>
#include <stdio.h>

#include <algorithm>
#include <type_traits>
#include <string>
#include <vector>

#include "tcgen05.cuh"
#include "vie_internal.cuh"

namespace vie {

namespace {

constexpr int TX = 32;            // output tile width of the 3x3 convolution kernels
constexpr int CIB = 8;            // input channels staged per step
constexpr int COB = 32;           // output channels per CTA of the weight-gradient kernel

// ------------------------------------------------------------ kernels

// 3x3 convolution, zero padding 1, + bias (+ relu).  A CTA computes a TX x TY
// pixel tile for COBC output channels; thread (tx, ty), ty in 0..7, owns the
// pixels (x0 + tx, y0 + ty + 8 k), k < TY / 8, for all COBC outputs.  Every
// output sums its input channels and taps in the same order whatever TY and
// COBC are, so the tile shape changes no result bit.
template <bool RELU, typename WT, int TY, int COBC>
__global__ void __launch_bounds__(256) k_conv3(const float *__restrict__ in, long in_bs, int Ci,
                                               const WT *__restrict__ w, const float *__restrict__ bias,
                                               float *__restrict__ out, long out_bs, int Co, int H,
                                               int W, int co_blocks) {
  static_assert(TY % 8 == 0 && COBC % 4 == 0, "tile shape");
  constexpr int PY = TY / 8;
  __shared__ float in_s[CIB][TY + 2][TX + 2];
  __shared__ __align__(16) float w_s[CIB][9][COBC];
  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;  // ty in 0..7
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
  const int b = blockIdx.z / co_blocks, cb = blockIdx.z % co_blocks;
  const int co0 = cb * COBC;
  float acc[PY][COBC];
#pragma unroll
  for (int k = 0; k < PY; ++k)
#pragma unroll
    for (int c = 0; c < COBC; ++c) acc[k][c] = 0.f;
  const float *inb = in + b * in_bs;
  const long plane = (long)H * W;
  // Each step stages CIB input channels: the padded pixel tile through
  // asynchronous 4-byte copies (zero-filled outside the image), the weights
  // through registers, all loads in flight together.  Flat index i of a
  // staging array is its shared-memory offset.
  constexpr int IN_N = CIB * (TY + 2) * (TX + 2);
  constexpr int W_N = CIB * 9 * COBC, W_K = (W_N + 255) / 256;
  const unsigned in_s0 = (unsigned)__cvta_generic_to_shared(&in_s[0][0][0]);
  for (int ci0 = 0; ci0 < Ci; ci0 += CIB) {
    __syncthreads();
    for (int i = threadIdx.x; i < IN_N; i += 256) {
      const int c = i / ((TY + 2) * (TX + 2)), r = i % ((TY + 2) * (TX + 2));
      const int gy = y0 - 1 + r / (TX + 2), gx = x0 - 1 + r % (TX + 2);
      const bool ok = ci0 + c < Ci && gy >= 0 && gy < H && gx >= 0 && gx < W;
      const float *src = ok ? inb + (ci0 + c) * plane + (long)gy * W + gx : inb;
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(in_s0 + 4u * i), "l"(src),
                   "r"(ok ? 4 : 0)
                   : "memory");
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    float pwt[W_K];
#pragma unroll
    for (int k = 0; k < W_K; ++k) {
      const int i = threadIdx.x + 256 * k;
      const int c = i / (9 * COBC), r = i % (9 * COBC);
      const int tap = r / COBC, co = r % COBC;
      pwt[k] = i < W_N && ci0 + c < Ci && co0 + co < Co
                   ? (float)w[((long)(co0 + co) * Ci + ci0 + c) * 9 + tap]
                   : 0.f;
    }
#pragma unroll
    for (int k = 0; k < W_K; ++k)
      if (threadIdx.x + 256 * k < W_N) (&w_s[0][0][0])[threadIdx.x + 256 * k] = pwt[k];
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
#pragma unroll 1
    for (int c = 0; c < CIB; ++c) {
#pragma unroll
      for (int tap = 0; tap < 9; ++tap) {
        const int dy = tap / 3, dx = tap % 3;
        float v[PY];
#pragma unroll
        for (int k = 0; k < PY; ++k) v[k] = in_s[c][ty + 8 * k + dy][tx + dx];
        const float4 *wr = reinterpret_cast<const float4 *>(&w_s[c][tap][0]);
#pragma unroll
        for (int q = 0; q < COBC / 4; ++q) {
          const float4 wv = wr[q];
#pragma unroll
          for (int k = 0; k < PY; ++k) {
            acc[k][4 * q + 0] = fmaf(v[k], wv.x, acc[k][4 * q + 0]);
            acc[k][4 * q + 1] = fmaf(v[k], wv.y, acc[k][4 * q + 1]);
            acc[k][4 * q + 2] = fmaf(v[k], wv.z, acc[k][4 * q + 2]);
            acc[k][4 * q + 3] = fmaf(v[k], wv.w, acc[k][4 * q + 3]);
          }
        }
      }
    }
  }
  const int x = x0 + tx;
  float *ob = out + b * out_bs;
#pragma unroll
  for (int c = 0; c < COBC; ++c) {
    const int co = co0 + c;
    if (co >= Co || x >= W) continue;
    const float bv = bias ? bias[co] : 0.f;
#pragma unroll
    for (int k = 0; k < PY; ++k) {
      const int yk = y0 + ty + 8 * k;
      float vk = acc[k][c] + bv;
      if (RELU) vk = fmaxf(vk, 0.f);
      if (yk < H) ob[co * plane + (long)yk * W + x] = vk;
    }
  }
}

// Tensor-core convolution tiles: 128 TMEM lanes (pixels) per tile.
constexpr int kTcM = 128;

// The BF16 convolution as an implicit GEMM fed by the tensor memory
// accelerator.  The input is first rounded to BF16 and laid out NHWC with its
// channels padded to S slices of 32 (k_to_nhwc_bf16).  A tile is 128 TMEM
// lanes = R rows x Wb pixels of one image (Wb = min(W, 128), R = 128 / Wb);
// for each tap (dy, dx) and channel slice the A operand is the input shifted
// by the tap: one TMA box (32 channels, Wb, R, 1) at (slice, x0 + dx - 1,
// y0 + dy - 1, image), whose out-of-image part the TMA fills with zeros --
// exactly the zero padding of the convolution.  Its rows are 64 bytes (32
// BF16 along K), written with the 64-byte swizzle that the MMA's K-major
// descriptor reads.  The B operand of the same step is the weights' [Co][32]
// block of that tap and slice (packed by k_pack_tc_weights).
//
// Images of at most 64 pixels a row, BF16 (NP = 1): the flat form.  One box of
// W + 2 pixels times the tile's rows and two more lies in shared memory as the
// zero-padded image at pitch P = W + 2; a tile is 128 consecutive positions
// y P + x of it (those with x >= W are dropped), and the input of tap (dy, dx)
// is the same rows dy P + dx further on, so one box serves all 9 taps of a
// slice.  A box per tap (9 times the loads, 63 bytes a clock and SM: the L2
// path's limit) took 31 us per 32-channel layer of 64 images at 64^2 and 54 for 64
// channels, this 24 and 34; in
// split precision the products bound it, and the boxes of all parts would not
// fit.  The order of the products is the same.
//
// Two CTAs per SM (half of its shared memory each) take tiles blockIdx.x,
// blockIdx.x + G, ... in a warp-specialised pipeline: the weights are loaded once; warp 4 streams the A
// boxes of its tiles into a ring of nst stages (a tile of one image row
// takes, per slice, its 3 input rows once as boxes of Wb + 2 pixels, and the
// MMAs read the 3 taps of a row at 64-byte offsets into them: a third of the
// TMA rows; other tiles take one box per tap and slice); warp 5 issues two
// tcgen05.mma (M = 128, N = Co, K = 16) per tap into one of kAcc tensor-
// memory accumulators (FP32), committing each stage back to the producer and
// each finished tile to the epilogue; warps 0-3 read their 32 lanes of a
// finished accumulator, hand it back, add the bias (and relu) and write FP32
// NCHW, while the next tiles' loads and products run.  Waits are bounded (wl;
// the first operand wait takes wl.first).  On expiry the CTA stops issuing,
// writes NaN for the tiles it has not finished, sets *err, waits (bounded by
// wl.limit) for the loads and products it issued and frees its tensor memory.
constexpr int kTmaSlice = 32;   // channels per K slice (64 bytes of BF16)
constexpr int kAcc = 4;         // tensor-memory accumulators (Co <= 32 columns each)
constexpr int kConvThreads = 192;

// one ring stage: a tap box of 128 pixels, or a halo box of Wb + 2 (Wb = 128)
// rounded up to 1024 bytes
// (flat form, fr box rows: every position a tap of the tile reaches)
__host__ __device__ inline int conv_stage_bytes(int Wb, int fr = 0) {
  if (fr > 0) {
    const int rows = fr * (Wb + 2), reach = kTcM + 3 * (Wb + 2) + 2;
    return ((rows > reach ? rows : reach) * 64 + 1023) & ~1023;
  }
  return Wb == kTcM ? 9216 : kTcM * 64;
}
// box rows of the flat form: the most image rows 128 positions touch, and two; 0: another form
inline int conv_flat_rows(int H, int W, int np) {
  if (np != 1 || W > kTcM / 2 || H < 2) return 0;
  const int P = W + 2;
  return std::min((kTcM - 1 + P - 1) / P + 1, H) + 2;
}
// ring stages of a CTA with `budget` bytes of shared memory
// (np = 2: split precision, operands in two parts)
int conv_stages(int S, int Co, int Wb, size_t budget, int np, int fr) {
  const size_t b = (size_t)np * 9 * S * Co * 64, fixed = 1024 + b + 1024;
  if (budget <= fixed) return 0;
  return (int)std::min<size_t>(32, (budget - fixed) / ((size_t)np * conv_stage_bytes(Wb, fr)));
}
size_t conv_tma_smem(int S, int Co, int Wb, int nst, int np, int fr) {
  return 1024 + (size_t)np * 9 * S * Co * 64 + (size_t)nst * np * conv_stage_bytes(Wb, fr) + 8 * (2 * nst + 2 * kAcc + 2) +
         16;
}

// The split-precision operands of training: v = p0 + p1 [+ p2], p0 = bf16(v),
// each later part the BF16 rounding of what the earlier ones leave (exact in
// FP32): 16 significant bits for two parts, 24 (all of FP32's) for three.
__device__ __forceinline__ void split_parts(float v, int np, __nv_bfloat16 (&part)[3]) {
  float r = v;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    part[q] = __float2bfloat16_rn(q < np ? r : 0.f);
    r -= __bfloat162float(part[q]);
  }
}

// 8 consecutive channels as NP BF16 parts, one 16-byte store each at element o
template <int NP>
__device__ __forceinline__ void store_parts(const float *v, __nv_bfloat16 *__restrict__ out0,
                                            __nv_bfloat16 *__restrict__ out1, __nv_bfloat16 *__restrict__ out2,
                                            long o) {
  unsigned w[3][4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    __nv_bfloat16 p0[3], p1[3];
    split_parts(v[2 * e], NP, p0);
    split_parts(v[2 * e + 1], NP, p1);
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      const __nv_bfloat162 h2 = __halves2bfloat162(p0[q], p1[q]);
      w[q][e] = *reinterpret_cast<const unsigned *>(&h2);
    }
  }
  *reinterpret_cast<uint4 *>(out0 + o) = make_uint4(w[0][0], w[0][1], w[0][2], w[0][3]);
  if (NP > 1) *reinterpret_cast<uint4 *>(out1 + o) = make_uint4(w[1][0], w[1][1], w[1][2], w[1][3]);
  if (NP > 2) *reinterpret_cast<uint4 *>(out2 + o) = make_uint4(w[2][0], w[2][1], w[2][2], w[2][3]);
}

// NP > 1: the FP32 convolutions of training in split precision: input and
// weights each as NP BF16 parts (v = p0 + p1 [+ p2], each part the BF16
// rounding of what the earlier ones leave; map_x1 / map_w1, map_x2 / map_w2
// the later parts), every tap the products of parts i, j with i + j < NP
// into the FP32 accumulator (the terms left out are below 2^-8 NP of the
// kept ones: 2^-16 for two parts, 2^-24 for three); a stage holds the parts'
// boxes one after the other.  A product of 128 pixels takes about 65 cycles to
// read its operand however few columns it has, so two parts (the input
// gradients) take p0 against both weight parts at once, in 64 columns whose
// halves the epilogue adds (16 images at 128^2, 13 layers: 222 us with a product
// per pair of parts, 206 so).  Three parts keep one accumulator: the
// training loss keeps its bits.  Inputs of at most 16 channels skip the second
// half of their slice, all zeros.
template <bool RELU, int NP>
__global__ void __launch_bounds__(kConvThreads, 2)
    k_conv3_tma(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w,
                const __grid_constant__ CUtensorMap map_x1, const __grid_constant__ CUtensorMap map_w1,
                const __grid_constant__ CUtensorMap map_x2, const __grid_constant__ CUtensorMap map_w2,
                const float *__restrict__ bias, float *__restrict__ out, long out_bs, int Co, int H, int W, int S,
                int Wb, int R, int fr, int kks, int tiles_x, int tiles, int nst, WaitLimits wl, int *err,
                __nv_bfloat16 *__restrict__ out_h, __nv_bfloat16 *__restrict__ out_h1,
                __nv_bfloat16 *__restrict__ out_h2, long oh_bs, int oh_cp, int oh_c0,
                const void *__restrict__ head_w, const float *__restrict__ head_b, float *__restrict__ head_o) {
  using namespace tc;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char *smem = (unsigned char *)(((size_t)smem_raw + 1023) & ~(size_t)1023);
  // halo: tiles of one image row take, per slice, the 3 input rows once
  // (Wb + 2 pixels each) and the 3 taps of a row as 64-byte offsets into
  // that box; other tiles take one box per tap and slice
  const bool halo = R == 1, flat = NP == 1 && fr > 0;
  const int P = W + 2;  // (flat)
  const int steps = flat ? S : (halo ? 3 : 9) * S, taps_step = halo ? 3 : 1;
  const int tiles_img = flat ? (H * P + kTcM - 1) / kTcM : tiles_x * ((H + R - 1) / R);
  const int a_part = conv_stage_bytes(Wb, fr), a_bytes = NP * a_part, b_bytes = Co * 64;
  // weights: block k's parts one part apart, two parts side by side
  constexpr int kCols = NP == 2 ? 64 : 32;  // columns of an accumulator
  const size_t b_part = NP == 2 ? (size_t)b_bytes : (size_t)9 * S * b_bytes;
  const int b_step = NP == 2 ? 2 * b_bytes : b_bytes;
  unsigned char *Bs = smem;
  unsigned char *As = smem + (size_t)NP * 9 * S * b_bytes;
  unsigned long long *full = (unsigned long long *)(As + (size_t)nst * a_bytes);
  unsigned long long *empty = full + nst, *tfull = empty + nst, *tempty = tfull + kAcc;
  unsigned long long *wbar = tempty + kAcc, *done = wbar + 1;
  unsigned *tmem_slot = (unsigned *)(done + 1);
  volatile int *abort_flag = (volatile int *)(tmem_slot + 1);
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  const int G = gridDim.x;
  if (tid == 0) {
    for (int i = 0; i < nst; ++i) {
      mbar_init(su32(full + i), 1);
      mbar_init(su32(empty + i), 1);
    }
    for (int i = 0; i < kAcc; ++i) {
      mbar_init(su32(tfull + i), 1);
      mbar_init(su32(tempty + i), 4);  // one arrival per epilogue warp
    }
    mbar_init(su32(wbar), 1);
    mbar_init(su32(done), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 5) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)),
                 "r"(kAcc * kCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem = *tmem_slot;
  const unsigned box_bytes = (unsigned)(kTmaSlice * 2 * (flat ? P * fr : halo ? Wb + 2 : Wb * R));
  int issued_loads = 0;
  if (warp == 4 && lane == 0) {
    // TMA producer: the weights once, then every step's shifted input box
    mbar_arrive_expect_tx(su32(wbar), (unsigned)(NP * 9 * S * b_bytes));
    for (int k = 0; k < 9 * S; ++k) {
      tma_load_2d(su32(Bs + (size_t)k * b_step), &map_w, su32(wbar), 0, k * Co);
      if (NP > 1) tma_load_2d(su32(Bs + b_part + (size_t)k * b_step), &map_w1, su32(wbar), 0, k * Co);
      if (NP > 2) tma_load_2d(su32(Bs + 2 * b_part + (size_t)k * b_step), &map_w2, su32(wbar), 0, k * Co);
    }
    int g = 0;
    bool go = true;
    for (int t = blockIdx.x; t < tiles && go; t += G) {
      const int img = t / tiles_img, r = t - img * tiles_img;
      int x0 = (r % tiles_x) * Wb, y0 = (r / tiles_x) * R;
      for (int k = 0; k < steps; ++k, ++g) {
        const int st = g % nst, use = g / nst;
        if (use > 0 && !mbar_wait(su32(empty + st), (use - 1) & 1, abort_flag, wl.limit)) {
          atomicExch(err, 1);
          *abort_flag = 1;
          go = false;
          break;
        }
        // step k: slice sl of input row dy (halo) or of tap (dy, dx)
        // (flat: slice k of the tile's rows and their neighbours)
        const int q = flat ? 0 : k / S, sl = k - q * S;
        const int dy = halo ? q : q / 3, dx = halo ? 0 : q % 3;
        if (flat) {
          x0 = 0;
          y0 = r * kTcM / P;
        }
        mbar_arrive_expect_tx(su32(full + st), NP * box_bytes);
        tma_load_4d(su32(As + (size_t)st * a_bytes), &map_x, su32(full + st), sl * kTmaSlice, x0 + dx - 1,
                    y0 + dy - 1, img);
        if (NP > 1)
          tma_load_4d(su32(As + (size_t)st * a_bytes + a_part), &map_x1, su32(full + st), sl * kTmaSlice,
                      x0 + dx - 1, y0 + dy - 1, img);
        if (NP > 2)
          tma_load_4d(su32(As + (size_t)st * a_bytes + 2 * a_part), &map_x2, su32(full + st), sl * kTmaSlice,
                      x0 + dx - 1, y0 + dy - 1, img);
        ++issued_loads;
      }
    }
  } else if (warp == 5 && elect_one()) {
    // MMA issuer: one elected lane (about 65 cycles per product; 90 behind `lane == 0`)
    const unsigned idesc = idesc_bf16(kTcM, Co);
    bool go = mbar_wait(su32(wbar), 0, abort_flag, wl.first);
    int g = 0, j = 0;
    for (int t = blockIdx.x; t < tiles && go; t += G, ++j) {
      const int b = j % kAcc;
      if (j >= kAcc && !mbar_wait(su32(tempty + b), (j / kAcc - 1) & 1, abort_flag, wl.limit)) {
        go = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const unsigned d = tmem + (unsigned)(b * kCols);
      if (flat) {
        // every slice of the tile (at most nst), then tap by tap in the other forms' order
        for (int sl = 0; sl < S && go; ++sl)
          go = mbar_wait(su32(full + (g + sl) % nst), ((g + sl) / nst) & 1, abort_flag,
                         g + sl == 0 ? wl.first : wl.limit);
        if (!go) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int v0 = (t % tiles_img) * kTcM, s0 = v0 - v0 / P * P;  // the tile's first position in the box
        for (int tap = 0; tap < 9; ++tap) {
          const unsigned row = 64u * (unsigned)(s0 + tap / 3 * P + tap % 3);
          for (int sl = 0; sl < S; ++sl) {
            const unsigned long long ad = smem_desc_sw64(su32(As + (size_t)((g + sl) % nst) * a_bytes) + row);
            const unsigned long long bd = smem_desc_sw64(su32(Bs + (size_t)(tap * S + sl) * b_step));
#pragma unroll
            for (int kk = 0; kk < 2; ++kk)
              if (kk < kks)
                mma_bf16(d, ad + (unsigned)(kk * 2), bd + (unsigned)(kk * 2), idesc,
                         (tap > 0 || sl > 0 || kk > 0) ? 1u : 0u);
          }
        }
        for (int sl = 0; sl < S; ++sl, ++g) mma_commit(su32(empty + g % nst));
        mma_commit(su32(tfull + b));
        continue;
      }
      for (int k = 0; k < steps; ++k, ++g) {
        const int st = g % nst;
        if (!mbar_wait(su32(full + st), (g / nst) & 1, abort_flag, g == 0 ? wl.first : wl.limit)) {
          go = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int q = k / S, sl = k - q * S;
        for (int e = 0; e < taps_step; ++e) {
          // tap (dy, dx): its weights, and its input rows e pixels into a halo box
          const int tap = halo ? 3 * q + e : q;
          // (descriptors by addition to the start address field, in 16-byte units)
          const unsigned long long ad = smem_desc_sw64(su32(As + (size_t)st * a_bytes) + 64u * (unsigned)e);
          const unsigned long long bd = smem_desc_sw64(su32(Bs + (size_t)(tap * S + sl) * b_step));
#pragma unroll
          for (int kk = 0; kk < 2; ++kk) {
            if (kk >= kks) break;
            if constexpr (NP == 2) {
              mma_bf16(d, ad + (unsigned)(kk * 2), bd + (unsigned)(kk * 2), idesc_bf16(kTcM, kCols),
                       (k > 0 || e > 0 || kk > 0) ? 1u : 0u);
              mma_bf16(d, ad + (unsigned)((a_part >> 4) + kk * 2), bd + (unsigned)(kk * 2), idesc, 1u);
              continue;
            }
            // parts i of the input and j of the weights, i + j < NP
#pragma unroll
            for (int i = 0; i < NP; ++i)
#pragma unroll
              for (int j = 0; i + j < NP; ++j)
                mma_bf16(d, ad + (unsigned)(i * (a_part >> 4) + kk * 2),
                         bd + (unsigned)(j * (int)(b_part >> 4) + kk * 2), idesc,
                         (k > 0 || e > 0 || kk > 0 || i > 0 || j > 0) ? 1u : 0u);
          }
        }
        mma_commit(su32(empty + st));  // the stage is free once these products finish
      }
      if (!go) break;
      mma_commit(su32(tfull + b));     // the tile's accumulator is complete
    }
    if (!go) {
      atomicExch(err, 1);
      *abort_flag = 1;
    }
    mma_commit(su32(done));            // every product this thread issued
  } else if (warp < 4) {
    // epilogue: warp w reads TMEM lanes 32 w .. 32 w + 31
    const int i = warp * 32 + lane;  // this thread's lane: pixel (x0 + i % Wb, y0 + i / Wb) of the tile
    const long plane = (long)H * W;
    float bv[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) bv[c] = bias && c < Co ? bias[c] : 0.f;
    float hv[32];  // the head's weights
#pragma unroll
    for (int c = 0; c < 32; ++c) {
      hv[c] = 0.f;
      if (head_o && c < Co)
        hv[c] = NP == 1 ? (float)static_cast<const __nv_bfloat16 *>(head_w)[c] : static_cast<const float *>(head_w)[c];
    }
    int j = 0;
    for (int t = blockIdx.x; t < tiles; t += G, ++j) {
      const int b = j % kAcc;
      const int img = t / tiles_img, r = t - img * tiles_img;
      int px = (r % tiles_x) * Wb + i % Wb, py = (r / tiles_x) * R + i / Wb;
      if (flat) {
        py = (r * kTcM + i) / P;
        px = r * kTcM + i - py * P;
      }
      const bool pvalid = (flat || i < Wb * R) && px < W && py < H;
      bool ok = *abort_flag == 0 && mbar_wait(su32(tfull + b), (j / kAcc) & 1, abort_flag, wl.limit);
      ok = __all_sync(0xffffffffu, ok);  // tcgen05.ld is warp-collective
      float v[32];
      if (ok) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const unsigned ta = tmem + ((unsigned)(warp * 32) << 16) + (unsigned)(b * kCols);
        tmem_ld16(ta, v);
        if (Co > 16) tmem_ld16(ta + 16, v + 16);
        if constexpr (NP == 2) {
          float v1[32];
          tmem_ld16(ta + 32, v1);
          tmem_ld16(ta + 48, v1 + 16);
#pragma unroll
          for (int c = 0; c < 32; ++c) v[c] += v1[c];
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(su32(tempty + b));  // the accumulator may be overwritten
      } else if (lane == 0) {
        atomicExch(err, 1);
        *abort_flag = 1;
      }
      float *ob = out + img * out_bs + (long)py * W + px;
#pragma unroll
      for (int c = 0; c < 32; ++c) {
        float x = ok ? v[c] + bv[c] : __int_as_float(0x7fc00000);
        if (RELU && ok) x = fmaxf(x, 0.f);
        v[c] = x;
        if (c < Co && pvalid) ob[(long)c * plane] = x;
      }
      if (out_h && pvalid) {
        // the same values in BF16 (NP = 3: in three parts) for the next
        // convolution's NHWC input: channels oh_c0 .. oh_c0 + Co of this pixel,
        // 16 bytes at a time
        const long ho = img * oh_bs + ((long)py * W + px) * oh_cp + oh_c0;
#pragma unroll
        for (int g8 = 0; g8 < 4; ++g8) {
          if (8 * g8 >= Co) break;
          store_parts<NP == 3 ? 3 : 1>(v + 8 * g8, out_h, out_h1, out_h2, ho + 8 * g8);
        }
      }
      if (head_o && pvalid) {
        // the 1x1 head on this pixel's channels, k_head's sum in its order
        float s = __ldg(head_b);
#pragma unroll
        for (int c = 0; c < 32; ++c) {
          if (c >= Co) break;
          s = fmaf(hv[c], v[c], s);
        }
        head_o[img * plane + (long)py * W + px] = s;
      }
    }
  }
  __syncwarp();
  // everything issued has landed before shared and tensor memory are released
  // (bounded by the full limit): the producer waits for the weights and for
  // the last load into each stage, the issuer for its last commit
  if (warp == 4 && lane == 0) {
    const long long t0 = clock64();
    while (!mbar_test(su32(wbar), 0) && clock64() - t0 < wl.limit) {
    }
    for (int s = 0; s < nst && s < issued_loads; ++s) {
      const int use = (issued_loads - 1 - s) / nst;
      while (!mbar_test(su32(full + s), use & 1) && clock64() - t0 < wl.limit) {
      }
    }
  }
  if (warp == 5 && lane == 0) {
    const long long t0 = clock64();
    while (!mbar_test(su32(done), 0) && clock64() - t0 < wl.limit) {
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 5) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kAcc * kCols) : "memory");
  }
}

// in: FP32 [B][Ci][plane] (image stride in_bs) -> BF16 [B][plane][Cp], rounded
// to nearest even, channels Ci..Cp-1 zero.  One thread per (image, pixel):
// a warp reads 32 consecutive pixels of a channel plane at a time and writes
// its pixels' Cp channels as 16-byte groups.
__global__ void k_to_nhwc_bf16(const float *__restrict__ in, long in_bs, int Ci, long plane, int Cp, int B,
                               __nv_bfloat16 *__restrict__ out) {
  const long total = (long)B * plane;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
    const long b = t / plane, p = t - b * plane;
    const float *src = in + b * in_bs + p;
    uint4 *dst = reinterpret_cast<uint4 *>(out + t * Cp);
    for (int gq = 0; gq < Cp / 8; ++gq) {
      unsigned w[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int c = gq * 8 + 2 * e;
        const float lo = c < Ci ? src[(long)c * plane] : 0.f, hi = c + 1 < Ci ? src[(long)(c + 1) * plane] : 0.f;
        const __nv_bfloat162 q = __floats2bfloat162_rn(lo, hi);
        w[e] = *reinterpret_cast<const unsigned *>(&q);
      }
      dst[gq] = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

// Weights of one 3x3 convolution, FP32 [Co][Ci][9] -> BF16 [9 S][Co][32]:
// block k = tap S + slice holds w[co][slice 32 + c][tap] (zero past Ci).
__global__ void k_pack_tc_weights(const float *__restrict__ w, int Co, int Ci, int S,
                                  __nv_bfloat16 *__restrict__ out) {
  const long total = (long)9 * S * Co * kTmaSlice;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
    const int c = (int)(t % kTmaSlice);
    const long r = t / kTmaSlice;
    const int co = (int)(r % Co);
    const int k = (int)(r / Co);
    const int tap = k / S, ci = (k - tap * S) * kTmaSlice + c;
    out[t] = __float2bfloat16_rn(ci < Ci ? w[((long)co * Ci + ci) * 9 + tap] : 0.f);
  }
}

// Input: FP32 [B][Ci][plane] -> NP BF16 parts [B][plane][Cp] (out0, out1,
// out2), one thread per (image, pixel) as in k_to_nhwc_bf16.
template <int NP>
__global__ void k_to_nhwc_split(const float *__restrict__ in, long in_bs, int Ci, long plane, int Cp, int B,
                                __nv_bfloat16 *__restrict__ out0, __nv_bfloat16 *__restrict__ out1,
                                __nv_bfloat16 *__restrict__ out2) {
  const long total = (long)B * plane;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
    const long b = t / plane, p = t - b * plane;
    const float *src = in + b * in_bs + p;
    for (int gq = 0; gq < Cp / 8; ++gq) {
      float v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = gq * 8 + e < Ci ? src[(long)(gq * 8 + e) * plane] : 0.f;
      store_parts<NP>(v, out0, out1, out2, t * Cp + 8 * gq);
    }
  }
}

// The gradient of a 32-channel convolution's output, masked by its ReLU
// (a > 0), as three BF16 parts [B][plane][32], and the bias gradient's block
// sums part[block][32].  A thread takes 8 of the channels of one pixel, and
// `steps` pixels 64 apart in turn (up to 8; small levels have too few pixels).
// Where the gradient comes from (FROM): g itself (kFromG); the 1x1 head, w_c times
// the output's gradient g (kFromHead, g one plane); 2x2 upsampling, the sum over
// the 4 pixels of the finer g (kFromUp); g plus a quarter of the pooled level's
// gradient g2 (kFromPool).  (As kernels of their own these three passed the
// gradient through memory once more, 65 us of 16 images' step at 128^2.)
enum GradFrom { kFromG = 0, kFromHead = 1, kFromUp = 2, kFromPool = 3 };
int split_steps(long total) { return (int)std::max(1L, std::min(8L, total / (64 * 512))); }
int split_blocks(long total) { return (int)((total + 64 * split_steps(total) - 1) / (64 * split_steps(total))); }
template <int FROM>
__global__ void __launch_bounds__(256) k_mask_split(const float *__restrict__ g, long g_bs,
                                                    const float *__restrict__ g2, long g2_bs,
                                                    const float *__restrict__ a, long a_bs, int W, long plane, int B,
                                                    __nv_bfloat16 *__restrict__ out0,
                                                    __nv_bfloat16 *__restrict__ out1,
                                                    __nv_bfloat16 *__restrict__ out2, float *__restrict__ part, int steps) {
  __shared__ float red[32][65];
  const int px = threadIdx.x & 63, gq = threadIdx.x >> 6;
  float sum[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) sum[e] = 0.f;
  const long total = (long)B * plane;
#pragma unroll 2
  for (int k = 0; k < steps; ++k) {
    const long t = ((long)blockIdx.x * steps + k) * 64 + px;
    if (t >= total) break;
    const long b = t / plane, p = t - b * plane;
    const float *ap = a + b * a_bs + p + 8 * gq * plane;
    float v[8];
    if constexpr (FROM == kFromHead) {
      const float go = g[b * g_bs + p];
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = g2[8 * gq + e] * go;
    } else if constexpr (FROM == kFromUp) {
      const int y = (int)p / W, x = (int)p - y * W;
      const float *gp = g + b * g_bs + 32 * gq * plane + 4L * y * W + 2 * x;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float2 r0 = *reinterpret_cast<const float2 *>(gp + 4 * e * plane);
        const float2 r1 = *reinterpret_cast<const float2 *>(gp + 4 * e * plane + 2 * W);
        v[e] = r0.x + r0.y + r1.x + r1.y;
      }
    } else {
      const float *gp = g + b * g_bs + p + 8 * gq * plane;
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = gp[e * plane];
      if constexpr (FROM == kFromPool) {
        const int y = (int)p / W, x = (int)p - y * W;
        const float *cp = g2 + b * g2_bs + 2 * gq * plane + (long)(y / 2) * (W / 2) + x / 2;
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] += 0.25f * cp[e * (plane / 4)];
      }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      v[e] = ap[e * plane] > 0.f ? v[e] : 0.f;
      sum[e] += v[e];
    }
    store_parts<3>(v, out0, out1, out2, t * 32 + 8 * gq);
  }
#pragma unroll
  for (int e = 0; e < 8; ++e) red[8 * gq + e][px] = sum[e];
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int c = 4 * warp + q;
    float s = red[c][lane] + red[c][lane + 32];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) part[blockIdx.x * 32 + c] = s;
  }
}

// The split weights of a training step's convolutions in one launch (as one
// per layer, with the flips of the adjoints: 43 launches, 89 us and as much in
// the gaps between them).  A job packs 32 output channels co0 .. of one
// convolution from the FP32 parameters [co][ci][9], as np BF16 parts in
// k_pack_tc_weights's block order [9 S][32][32], one after the other at out; the
// adjoint of a layer with zero padding (flip) is the convolution from its
// outputs to its inputs with the flipped taps.
struct PackJob {
  long w_off, out;
  int Ci, Co, S, co0, np, flip;  // of the convolution packed (the adjoint's own when flip)
};
constexpr int kPackJobs = 32;
struct PackJobs {
  PackJob job[kPackJobs];
};
__global__ void k_pack_split_weights(const __grid_constant__ PackJobs jobs, const float *__restrict__ p,
                                     __nv_bfloat16 *__restrict__ out) {
  const PackJob &j = jobs.job[blockIdx.y];
  const int total = 9 * j.S * 32 * kTmaSlice;
  const float *w = p + j.w_off;
  __nv_bfloat16 *o = out + j.out;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    const int c = t % kTmaSlice, r = t / kTmaSlice, co = j.co0 + r % 32, k = r / 32;
    const int tap = k / j.S, ci = (k - tap * j.S) * kTmaSlice + c;
    float v = 0.f;
    if (ci < j.Ci && co < j.Co) v = j.flip ? w[(ci * j.Co + co) * 9 + 8 - tap] : w[(co * j.Ci + ci) * 9 + tap];
    __nv_bfloat16 part[3];
    split_parts(v, j.np, part);
    for (int q = 0; q < j.np; ++q) o[(long)q * total + t] = part[q];
  }
}

// Gradient of a 3x3 convolution's weights and bias over one 32 x 8 pixel tile
// of images b0 .. b1 and 8 input channels; thread (co, ci) keeps its 9 taps
// over those images and adds them into dw with atomics once.  A 3 x 3 window
// of the input slides along x in registers.
constexpr int WY = 8;
__global__ void __launch_bounds__(256, 3) k_conv3_dw(const float *__restrict__ x, long x_bs, int Ci,
                                                  const float *__restrict__ gy, long g_bs, int Co,
                                                  int H, int W, float *__restrict__ dw,
                                                  float *__restrict__ db, int ci_blocks,
                                                  int co_blocks, int B, int b_splits) {
  __shared__ float g_s[COB][WY * TX + 1];
  __shared__ float x_s[CIB][WY + 2][TX + 2];
  const int co_l = threadIdx.x % 32, ci_l = threadIdx.x / 32;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * WY;
  int z = blockIdx.z;
  const int cib = z % ci_blocks;
  z /= ci_blocks;
  const int cob = z % co_blocks;
  const int bs = z / co_blocks;
  const int ci0 = cib * CIB, co0 = cob * COB;
  const long plane = (long)H * W;
  float acc[9];
#pragma unroll
  for (int t = 0; t < 9; ++t) acc[t] = 0.f;
  float bsum = 0.f;
  const int b_lo = (int)((long)B * bs / b_splits), b_hi = (int)((long)B * (bs + 1) / b_splits);
  for (int b = b_lo; b < b_hi; ++b) {
  if (b > b_lo) __syncthreads();  // the previous image's tiles are consumed
  for (int i = threadIdx.x; i < COB * WY * TX; i += 256) {
    const int c = i / (WY * TX), p = i % (WY * TX);
    const int yy = p / TX, xx = p % TX;
    const int gyy = y0 + yy, gxx = x0 + xx;
    float v = 0.f;
    if (co0 + c < Co && gyy < H && gxx < W) v = gy[b * g_bs + (co0 + c) * plane + (long)gyy * W + gxx];
    g_s[c][p] = v;
  }
  for (int i = threadIdx.x; i < CIB * (WY + 2) * (TX + 2); i += 256) {
    const int c = i / ((WY + 2) * (TX + 2)), r = i % ((WY + 2) * (TX + 2));
    const int yy = r / (TX + 2), xx = r % (TX + 2);
    const int gyy = y0 - 1 + yy, gxx = x0 - 1 + xx;
    float v = 0.f;
    if (ci0 + c < Ci && gyy >= 0 && gyy < H && gxx >= 0 && gxx < W)
      v = x[b * x_bs + (ci0 + c) * plane + (long)gyy * W + gxx];
    x_s[c][yy][xx] = v;
  }
  __syncthreads();
  for (int yy = 0; yy < WY; ++yy) {
    float win[3][3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      win[r][0] = x_s[ci_l][yy + r][0];
      win[r][1] = x_s[ci_l][yy + r][1];
    }
    // unrolled by four along the row: the window's shift is register
    // renaming within each group
#pragma unroll 4
    for (int xx = 0; xx < TX; ++xx) {
#pragma unroll
      for (int r = 0; r < 3; ++r) win[r][2] = x_s[ci_l][yy + r][xx + 2];
      const float g = g_s[co_l][yy * TX + xx];
#pragma unroll
      for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) acc[r * 3 + c] = fmaf(g, win[r][c], acc[r * 3 + c]);
      if (ci_l == 0) bsum += g;  // the bias gradient: warp 0 alone adds it
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        win[r][0] = win[r][1];
        win[r][1] = win[r][2];
      }
    }
  }
  }
  const int co = co0 + co_l, ci = ci0 + ci_l;
  if (co < Co && ci < Ci) {
#pragma unroll
    for (int t = 0; t < 9; ++t) atomicAdd(&dw[((long)co * Ci + ci) * 9 + t], acc[t]);
  }
  if (db && cib == 0 && ci_l == 0 && co < Co) atomicAdd(&db[co], bsum);
}

// Weight gradient of a 3x3 convolution with 32 outputs on the tensor cores:
//   dw[co][ci][ky][kx] = sum over pixels of g[co][p] x[ci][p + (ky - 1, kx - 1)],
// a contraction over pixels.  The operands are the split-precision NHWC copies
// the other convolutions use (three BF16 parts, the six products of parts i,
// j with i + j < 3), read MN-major: a row of shared memory is one pixel's 32
// channels, so that a shift by one pixel is a shift by one 64-byte row.  One
// tcgen05.mma takes 16 pixels of a row and has M = 128 = 4 shifts kx (the
// fourth is not used) x 32 input channels: the four blocks of 32 lie 64 bytes
// apart in the same input row (the descriptor's leading offset).  N is the 32
// output channels of as many parts of the gradient as part i of the input
// meets: 96, 64 and 32 columns for i = 0, 1, 2, three instructions for the six
// products, since an instruction of M = 128 takes about 64 cycles to read its
// operand however narrow N is.
//
// A CTA takes one slice of 32 input channels (blockIdx.y) and a run of image
// rows (segments of at most 128 pixels).  Warp 4 streams the rows by TMA (an
// input row of Wp + 2 pixels serves three output rows; zero fill outside the
// image is the convolution's padding and pads Wp to a multiple of 16), warp 5
// issues the products of one row and one ky into one of kDwAcc accumulators of
// 96 columns, warps 0-2 add the finished ones to FP32 sums in registers.  The
// accumulation of tcgen05 truncates, so chains are short (a row) and each column
// block has products of one size, parts i + j = 0, 1 and 2: the large ones are
// not truncated again for every small one (against FP64 6e-8 to 9e-8 relative at
// 128^2 and 136^2; with all parts of the input against the same columns 3.5e-7,
// the CUDA-core form 1.8e-7).  The CTAs' sums are added by k_dw_reduce, in order.
// What bounds it is the operand traffic of the products.  The CUDA-core form
// (k_conv3_dw, other widths) took 95 us per layer of 16 images at 128^2 on
// average; this takes 30 us (50 us for a 32 -> 32 layer at 128^2).
// Waits are bounded as in k_conv3_tma; on expiry the CTA's sums are NaN.
constexpr int kDwParts = 3;
constexpr int kDwAcc = 5;  // accumulators of 32 kDwParts tensor-memory columns
__host__ __device__ inline int dw_x_bytes(int Wp) { return ((Wp + 3) * 64 + 1023) / 1024 * 1024; }
__host__ __device__ inline int dw_g_bytes(int Wp) { return (Wp * 64 + 1023) / 1024 * 1024; }
// ring slots of input and gradient rows
__host__ __device__ inline int dw_x_slots(int Wp) { return Wp > 64 ? 5 : 8; }
__host__ __device__ inline int dw_g_slots(int Wp) { return Wp > 64 ? 3 : 6; }
inline size_t dw_smem(int Wp) {
  const int nx = dw_x_slots(Wp), ng = dw_g_slots(Wp);
  return 1024 + (size_t)kDwParts * (nx * dw_x_bytes(Wp) + ng * dw_g_bytes(Wp)) +
         8 * (2 * nx + 2 * ng + 2 * kDwAcc + 1) + 16;
}

struct DwMaps {
  CUtensorMap x[kDwParts], g[kDwParts];
};

__global__ void __launch_bounds__(kConvThreads, 1)
    k_conv3_dw_tc(const __grid_constant__ DwMaps maps, int H, int W, int B, int Wp, int segs,
                  float *__restrict__ part, WaitLimits wl, int *err) {
  using namespace tc;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char *smem = (unsigned char *)(((size_t)smem_raw + 1023) & ~(size_t)1023);
  const int nx = dw_x_slots(Wp), ng = dw_g_slots(Wp);
  const int xp = dw_x_bytes(Wp), gp = dw_g_bytes(Wp);
  unsigned char *Xs = smem, *Gs = smem + (size_t)kDwParts * nx * xp;
  unsigned long long *xfull = (unsigned long long *)(Gs + (size_t)kDwParts * ng * gp);
  unsigned long long *xempty = xfull + nx, *gfull = xempty + nx, *gempty = gfull + ng;
  unsigned long long *tfull = gempty + ng, *tempty = tfull + kDwAcc, *done = tempty + kDwAcc;
  unsigned *tmem_slot = (unsigned *)(done + 1);
  volatile int *abort_flag = (volatile int *)(tmem_slot + 1);
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  if (tid == 0) {
    for (int i = 0; i < nx; ++i) {
      mbar_init(su32(xfull + i), 1);
      mbar_init(su32(xempty + i), 1);
    }
    for (int i = 0; i < ng; ++i) {
      mbar_init(su32(gfull + i), 1);
      mbar_init(su32(gempty + i), 1);
    }
    for (int i = 0; i < kDwAcc; ++i) {
      mbar_init(su32(tfull + i), 1);
      mbar_init(su32(tempty + i), 3);  // one arrival per adding warp
    }
    mbar_init(su32(done), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 5) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem = *tmem_slot;
  // this CTA's rows q: row q % H of column q / H (an image's segment)
  const long rows = (long)B * segs * H;
  const int q0 = (int)(rows * blockIdx.x / gridDim.x), q1 = (int)(rows * (blockIdx.x + 1) / gridDim.x);
  int xs = 0, gs = 0;  // rows loaded so far (warp 4)
  if (warp == 4 && lane == 0) {
    bool go = true;
    auto load_x = [&](int col, int y) {
      const int st = xs % nx, use = xs / nx;
      if (!go || (use > 0 && !mbar_wait(su32(xempty + st), (use - 1) & 1, abort_flag, wl.limit))) {
        go = false;
        return;
      }
      mbar_arrive_expect_tx(su32(xfull + st), (unsigned)(kDwParts * (Wp + 2) * 64));
#pragma unroll
      for (int i = 0; i < kDwParts; ++i)
        tma_load_4d(su32(Xs + (size_t)(st * kDwParts + i) * xp), &maps.x[i], su32(xfull + st),
                    (int)blockIdx.y * kTmaSlice, col % segs * kTcM - 1, y, col / segs);
      ++xs;
    };
    for (int q = q0; q < q1 && go; ++q) {
      const int col = q / H, y = q % H;
      if (q == q0 || y == 0) {
        load_x(col, y - 1);
        load_x(col, y);
      }
      load_x(col, y + 1);
      const int st = gs % ng, use = gs / ng;
      if (!go || (use > 0 && !mbar_wait(su32(gempty + st), (use - 1) & 1, abort_flag, wl.limit))) {
        go = false;
        break;
      }
      mbar_arrive_expect_tx(su32(gfull + st), (unsigned)(kDwParts * Wp * 64));
#pragma unroll
      for (int i = 0; i < kDwParts; ++i)
        tma_load_4d(su32(Gs + (size_t)(st * kDwParts + i) * gp), &maps.g[i], su32(gfull + st), 0, col % segs * kTcM, y,
                    col / segs);
      ++gs;
    }
    if (!go) {
      atomicExch(err, 1);
      *abort_flag = 1;
    }
  } else if (warp == 5 && elect_one()) {
    bool go = true;
    int xb = 0, xw = 0;  // first input row of the current output row, rows waited for
    for (int q = q0; q < q1 && go; ++q) {
      const int i = q - q0, y = q % H;
      for (; xw <= xb + 2 && go; ++xw)
        go = mbar_wait(su32(xfull + xw % nx), (xw / nx) & 1, abort_flag, xw == 0 ? wl.first : wl.limit);
      go = go && mbar_wait(su32(gfull + i % ng), (i / ng) & 1, abort_flag, wl.limit);
      for (int ky = 0; ky < 3 && go; ++ky) {
        const int item = 3 * i + ky, st = item % kDwAcc;
        if (item >= kDwAcc && !mbar_wait(su32(tempty + st), (item / kDwAcc - 1) & 1, abort_flag, wl.limit)) {
          go = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // descriptors by addition to the start address field (in 16-byte
        // units: shared memory ends below its 14 bits)
        unsigned long long xd = smem_desc_sw64_mn(su32(Xs + (size_t)((xb + ky) % nx) * kDwParts * xp), 64);
        unsigned long long gd = smem_desc_sw64_mn(su32(Gs + (size_t)(i % ng) * kDwParts * gp), (unsigned)gp);
        const unsigned d = tmem + (unsigned)(st * 32 * kDwParts);
        for (int s = 0; s < Wp / 16; ++s, xd += 1024 >> 4, gd += 1024 >> 4)
#pragma unroll
          for (int a = 0; a < kDwParts; ++a)
            mma_bf16(d + 32u * (unsigned)a, xd + (unsigned)(a * (xp >> 4)), gd,
                     idesc_bf16(kTcM, 32 * (kDwParts - a), true), a > 0 || s > 0 ? 1u : 0u);
        mma_commit(su32(tfull + st));
      }
      if (!go) break;
      mma_commit(su32(gempty + i % ng));
      mma_commit(su32(xempty + xb % nx));
      if (y == H - 1 || q == q1 - 1) {
        // the run of rows ends here: its last two input rows are free as well
        mma_commit(su32(xempty + (xb + 1) % nx));
        mma_commit(su32(xempty + (xb + 2) % nx));
        xb += 3;
      } else {
        ++xb;
      }
    }
    if (!go) {
      atomicExch(err, 1);
      *abort_flag = 1;
    }
    mma_commit(su32(done));  // every product this thread issued
  } else if (warp < 3) {
    // warp kx, lane ci: the sums of the 32 outputs for each ky
    float acc[3][32];
#pragma unroll
    for (int ky = 0; ky < 3; ++ky)
#pragma unroll
      for (int c = 0; c < 32; ++c) acc[ky][c] = 0.f;
    bool ok = true;
    for (int i = 0; i < q1 - q0 && ok; ++i) {
#pragma unroll
      for (int ky = 0; ky < 3; ++ky) {
        const int item = 3 * i + ky, st = item % kDwAcc;
        ok = ok && *abort_flag == 0 && mbar_wait(su32(tfull + st), (item / kDwAcc) & 1, abort_flag, wl.limit);
        ok = __all_sync(0xffffffffu, ok);  // tcgen05.ld is warp-collective
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float v[kDwParts][16];
#pragma unroll
          for (int b = 0; b < kDwParts; ++b)
            tmem_ld16(tmem + ((unsigned)(warp * 32) << 16) + (unsigned)((st * kDwParts + b) * 32 + h * 16), v[b]);
#pragma unroll
          for (int c = 0; c < 16; ++c) acc[ky][16 * h + c] += v[0][c] + (v[1][c] + v[2][c]);
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(su32(tempty + st));
      }
    }
    if (!ok && lane == 0) {
      atomicExch(err, 1);
      *abort_flag = 1;
    }
    float4 *out = reinterpret_cast<float4 *>(part + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * 9 * 1024);
#pragma unroll
    for (int ky = 0; ky < 3; ++ky)
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const float nan = __int_as_float(0x7fc00000);
        out[(size_t)((ky * 3 + warp) * 32 + lane) * 8 + c] =
            ok ? make_float4(acc[ky][4 * c], acc[ky][4 * c + 1], acc[ky][4 * c + 2], acc[ky][4 * c + 3])
               : make_float4(nan, nan, nan, nan);
      }
  }
  __syncwarp();
  // everything issued has landed before shared and tensor memory are released
  if (warp == 4 && lane == 0) {
    const long long t0 = clock64();
    for (int s = 0; s < nx && s < xs; ++s)
      while (!mbar_test(su32(xfull + s), ((xs - 1 - s) / nx) & 1) && clock64() - t0 < wl.limit) {
      }
    for (int s = 0; s < ng && s < gs; ++s)
      while (!mbar_test(su32(gfull + s), ((gs - 1 - s) / ng) & 1) && clock64() - t0 < wl.limit) {
      }
  }
  if (warp == 5 && lane == 0) {
    const long long t0 = clock64();
    while (!mbar_test(su32(done), 0) && clock64() - t0 < wl.limit) {
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 5) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

// dw[co][ci][tap] += the sum of the CTAs' partials [slice][cta][tap][32 ci][32
// co] and db[co] += that of part_b[block][32], in a fixed order: block (tap,
// ci) of each slice, and a last one for db; 8 runs of the partials side by
// side, at most 64 terms at a time in FP32, joined in FP64.
// (One launch for all layers, blockIdx.y the layer.)
struct DwJob {
  long part, part_b;  // the layer's sums in dw_part and db_part
  long w_off, b_off;
  int ctas, S, Ci, blocks;
};
constexpr int kDwJobs = 32;
struct DwJobs {
  DwJob job[kDwJobs];
};
__global__ void __launch_bounds__(256) k_dw_reduce(const __grid_constant__ DwJobs jobs,
                                                   const float *__restrict__ parts,
                                                   const float *__restrict__ parts_b, float *__restrict__ g) {
  __shared__ double red[8][32];
  const DwJob &jb = jobs.job[blockIdx.y];
  const int last = jb.S * 9 * 32;
  if ((int)blockIdx.x > last) return;
  const int ctas = jb.ctas, Ci = jb.Ci;
  const float *part = parts + jb.part;
  float *dw = g + jb.w_off, *db = g + jb.b_off;
  const int co = threadIdx.x & 31, run = threadIdx.x >> 5;
  const bool bias = (int)blockIdx.x == last;
  const int slice = blockIdx.x / (9 * 32), r = blockIdx.x % (9 * 32), tap = r / 32, ci = slice * 32 + r % 32;
  const float *p = bias ? parts_b + jb.part_b : part + ((size_t)slice * ctas * 9 * 32 + r) * 32;
  const size_t step = bias ? 32 : (size_t)9 * 1024;
  const int n = bias ? jb.blocks : ctas;
  double s = 0.0;
  for (int c = run; c < n;) {
    const int end = min(n, c + 512);
    float f = 0.f;
#pragma unroll 8
    for (; c < end; c += 8) f += p[c * step + co];
    s += f;
  }
  red[run][co] = s;
  __syncthreads();
  if (run > 0 || (!bias && ci >= Ci)) return;
  for (int q = 1; q < 8; ++q) s += red[q][co];
  if (bias)
    db[co] += (float)s;
  else
    dw[((long)co * Ci + ci) * 9 + tap] += (float)s;
}

// wt[ci][co][8 - tap] = w[co][ci][tap]: the adjoint of a 3x3 convolution with
// zero padding is the convolution with the flipped, transposed kernel.
__global__ void k_flip(const float *__restrict__ w, int Co, int Ci, float *__restrict__ wt) {
  const long total = (long)Co * Ci * 9;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
    const long co = i / (Ci * 9), r = i % (Ci * 9), ci = r / 9, tap = r % 9;
    wt[(ci * Co + co) * 9 + (8 - tap)] = w[i];
  }
}

// 1x1 convolution to one channel: o = sum_c w_c d_c + b
template <typename WT>
__global__ void k_head(const float *__restrict__ d, long d_bs, int C, const WT *__restrict__ w,
                       const float *__restrict__ bias, float *__restrict__ o, long plane, int B) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < (long)B * plane; i += (long)gridDim.x * blockDim.x) {
    const long b = i / plane, p = i % plane;
    float s = bias[0];
    for (int c = 0; c < C; ++c) s = fmaf((float)w[c], d[b * d_bs + c * plane + p], s);
    o[i] = s;
  }
}

// head backward: dd_c = w_c go (written), dw_c += sum go d_c, db += sum go
__global__ void k_head_bwd_data(const float *__restrict__ go, int C, const float *__restrict__ w,
                                float *__restrict__ dd, long dd_bs, long plane, int B) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < (long)B * plane * C; i += (long)gridDim.x * blockDim.x) {
    const long b = i / (plane * C), r = i % (plane * C), c = r / plane, p = r % plane;
    dd[b * dd_bs + c * plane + p] = w[c] * go[b * plane + p];
  }
}

// Gradient of the 1x1 head's weights and bias in two passes, deterministic:
// block (c, k) sums channel c's products (c == C: the bias) over the k-th of
// gridDim.y slices of the B planes into part[c][k]; k_head_bwd_w_finish adds
// each channel's slices in order.
__global__ void k_head_bwd_w(const float *__restrict__ go, const float *__restrict__ d, long d_bs, int C,
                             long plane, int B, double *__restrict__ part) {
  __shared__ double red[256];
  const int c = blockIdx.x, k = blockIdx.y, K = gridDim.y;
  const long total = (long)B * plane, i0 = total * k / K, i1 = total * (k + 1) / K;
  double s = 0.0;
  long b = (i0 + threadIdx.x) / plane, p = i0 + threadIdx.x - b * plane;
  const float *dc = d + c * plane;
  // 64 terms at a time in FP32, the rest in FP64: the rounding does not grow with the image
  for (long i = i0 + threadIdx.x; i < i1;) {
    const long end = min(i1, i + 64L * blockDim.x);
    float f = 0.f;
#pragma unroll 4
    for (; i < end; i += blockDim.x, p += blockDim.x) {
      for (; p >= plane; p -= plane) ++b;  // (no division per term)
      f += go[i] * (c < C ? dc[b * d_bs + p] : 1.f);
    }
    s += f;
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[c * K + k] = red[0];
}

__global__ void k_head_bwd_w_finish(const double *__restrict__ part, int C, int K, float *__restrict__ dw,
                                    float *__restrict__ db) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c > C) return;
  double s = 0.0;
  for (int k = 0; k < K; ++k) s += part[c * K + k];
  if (c < C)
    dw[c] += (float)s;
  else
    db[0] += (float)s;
}

// The 2x2 pooling and upsampling kernels take one thread per coarse pixel of
// one plane (blockIdx.y = b C + c): 32-bit pixel arithmetic, the fine pixels
// of a row pair as float2.  H, W: the fine size (even).
__device__ __forceinline__ bool coarse_pixel(int H, int W, int C, int &b, int &c, int &y, int &x, int &q) {
  const int Wo = W / 2;
  q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= (H / 2) * Wo) return false;
  b = blockIdx.y / C;
  c = blockIdx.y - b * C;
  y = q / Wo;
  x = q - y * Wo;
  return true;
}
dim3 coarse_grid(int H, int W, int C, int B) { return dim3((unsigned)(((H / 2) * (W / 2) + 255) / 256), (unsigned)(B * C)); }

__global__ void k_avgpool(const float *__restrict__ in, long in_bs, float *__restrict__ out, long out_bs,
                          int C, int H, int W, int B) {
  int b, c, y, x, q;
  if (!coarse_pixel(H, W, C, b, c, y, x, q)) return;
  const float *p = in + b * in_bs + (long)c * H * W + (long)(2 * y) * W + 2 * x;
  const float2 r0 = *reinterpret_cast<const float2 *>(p), r1 = *reinterpret_cast<const float2 *>(p + W);
  out[b * out_bs + (long)c * (H / 2) * (W / 2) + q] = 0.25f * (r0.x + r0.y + r1.x + r1.y);
}

// The pooled planes in FP32 and as the next convolution's NHWC input in NP BF16
// parts (Cp channels, those past C zero): a thread takes 8 channels (blockIdx.y)
// of one coarse pixel of one image.  H, W: the fine size.
template <int NP>
__global__ void k_avgpool_nhwc(const float *__restrict__ in, long in_bs, float *__restrict__ out, long out_bs, int C,
                               int H, int W, int B, __nv_bfloat16 *__restrict__ out0,
                               __nv_bfloat16 *__restrict__ out1, __nv_bfloat16 *__restrict__ out2, int Cp) {
  const int Wo = W / 2, per = (H / 2) * Wo, c0 = 8 * blockIdx.y;
  const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (t >= (long)B * per) return;
  const int b = (int)(t / per), q = (int)(t - (long)b * per), y = q / Wo, x = q - y * Wo;
  float v[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) v[e] = 0.f;
  if (c0 < C) {
    const float *p = in + b * in_bs + ((long)c0 * H + 2 * y) * W + 2 * x;
    float2 r0[8], r1[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      r0[e] = *reinterpret_cast<const float2 *>(p + (long)e * H * W);
      r1[e] = *reinterpret_cast<const float2 *>(p + (long)e * H * W + W);
    }
    float *o = out + b * out_bs + (long)c0 * per + q;
#pragma unroll
    for (int e = 0; e < 8; ++e) o[(long)e * per] = v[e] = 0.25f * (r0[e].x + r0[e].y + r1[e].x + r1[e].y);
  }
  store_parts<NP>(v, out0, out1, out2, t * Cp + c0);
}

// grad of avgpool: g_in (+)= g_out / 4 on each 2x2 block
__global__ void k_avgpool_bwd(const float *__restrict__ go, long go_bs, float *__restrict__ gi, long gi_bs,
                              int C, int H, int W, int B, int accumulate) {
  int b, c, y, x, q;
  if (!coarse_pixel(H, W, C, b, c, y, x, q)) return;
  const float v = 0.25f * go[b * go_bs + (long)c * (H / 2) * (W / 2) + q];
  float2 *d0 = reinterpret_cast<float2 *>(gi + b * gi_bs + (long)c * H * W + (long)(2 * y) * W + 2 * x);
  float2 *d1 = reinterpret_cast<float2 *>(reinterpret_cast<float *>(d0) + W);
  if (accumulate) {
    const float2 a0 = *d0, a1 = *d1;
    *d0 = make_float2(a0.x + v, a0.y + v);
    *d1 = make_float2(a1.x + v, a1.y + v);
  } else {
    *d0 = make_float2(v, v);
    *d1 = make_float2(v, v);
  }
}

__global__ void k_upsample(const float *__restrict__ in, long in_bs, float *__restrict__ out, long out_bs,
                           int C, int H, int W, int B) {  // H, W: output size
  int b, c, y, x, q;
  if (!coarse_pixel(H, W, C, b, c, y, x, q)) return;
  const float v = in[b * in_bs + (long)c * (H / 2) * (W / 2) + q];
  float *o = out + b * out_bs + (long)c * H * W + (long)(2 * y) * W + 2 * x;
  *reinterpret_cast<float2 *>(o) = make_float2(v, v);
  *reinterpret_cast<float2 *>(o + W) = make_float2(v, v);
}

__global__ void k_upsample_bwd(const float *__restrict__ go, long go_bs, float *__restrict__ gi, long gi_bs,
                               int C, int H, int W, int B) {  // H, W: upsampled size
  int b, c, y, x, q;
  if (!coarse_pixel(H, W, C, b, c, y, x, q)) return;
  const float *p = go + b * go_bs + (long)c * H * W + (long)(2 * y) * W + 2 * x;
  const float2 r0 = *reinterpret_cast<const float2 *>(p), r1 = *reinterpret_cast<const float2 *>(p + W);
  gi[b * gi_bs + (long)c * (H / 2) * (W / 2) + q] = r0.x + r0.y + r1.x + r1.y;
}

// The decoder's upsampled half straight into its NHWC concatenation in NP BF16 parts:
// coarse FP32 planes (image stride in_bs) -> channels 0 .. C (C a multiple of
// 8) of the 4 fine pixels of each coarse pixel, pixels o_cp channels apart.
// One thread per (image, coarse pixel, group of 8 channels), the groups
// fastest, so a warp's stores cover whole 16-byte runs of each fine pixel.
// H, W: the fine size.
template <int NP>
__global__ void k_upsample_nhwc(const float *__restrict__ in, long in_bs, int C, int H, int W, int B,
                                __nv_bfloat16 *__restrict__ out0, __nv_bfloat16 *__restrict__ out1,
                                __nv_bfloat16 *__restrict__ out2, long o_bs, int o_cp) {
  const int Wc = W / 2, G8 = C / 8;
  const long per = (long)(H / 2) * Wc;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < (long)B * per * G8;
       t += (long)gridDim.x * blockDim.x) {
    const long pq = t / G8;
    const int g8 = (int)(t - pq * G8);
    const long b = pq / per;
    const int q = (int)(pq - b * per), y = q / Wc, x = q - y * Wc;
    const float *src = in + b * in_bs + (long)(8 * g8) * per + q;
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = src[(long)e * per];
    const long o = b * o_bs + ((long)(2 * y) * W + 2 * x) * o_cp + 8 * g8;
    store_parts<NP>(v, out0, out1, out2, o);
    store_parts<NP>(v, out0, out1, out2, o + o_cp);
    store_parts<NP>(v, out0, out1, out2, o + (long)W * o_cp);
    store_parts<NP>(v, out0, out1, out2, o + (long)(W + 1) * o_cp);
  }
}

// g *= (a > 0): relu backward through a stored activation
__global__ void k_relu_mask(float *__restrict__ g, long g_bs, const float *__restrict__ a, long a_bs,
                            long per, int B) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < (long)B * per; i += (long)gridDim.x * blockDim.x) {
    const long b = i / per, r = i % per;
    if (!(a[b * a_bs + r] > 0.f)) g[b * g_bs + r] = 0.f;
  }
}

// loss = mean(w_b (o - t)^2) (block partials in double), go = 2 w_b (o - t) / n;
// w_b = sample weight of image b (1 without weights), plane pixels per image
__global__ void k_mse(const float *__restrict__ o, const float *__restrict__ t, long n, long plane,
                      const float *__restrict__ wts, float *__restrict__ go, double *__restrict__ part) {
  __shared__ double red[256];
  double s = 0.0;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const float d = o[i] - t[i];
    const float wb = wts ? wts[i / plane] : 1.f;
    s += (double)wb * d * d;
    go[i] = 2.f * wb * d / (float)n;
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int k = 128; k > 0; k >>= 1) {
    if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

__global__ void k_adam(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, __nv_bfloat16 *__restrict__ pb, long n, float lr,
                       float b1, float b2, float eps, float c1, float c2) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
    pb[i] = __float2bfloat16_rn(pi);
  }
}

__global__ void k_to_bf16(const float *__restrict__ p, __nv_bfloat16 *__restrict__ pb, long n) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    pb[i] = __float2bfloat16_rn(p[i]);
}

// Preconditioner input [1][3][n][n]: (sigma_t / s_ref, sigma_s / s_ref, v / rms(v))
__global__ void k_net_input(const double *__restrict__ st, const double *__restrict__ ss,
                            const double *__restrict__ v, const double *__restrict__ vnorm2, long N,
                            float inv_ref, float *__restrict__ x) {
  const double rms = sqrt(*vnorm2 / (double)N);
  const double inv = rms > 0.0 ? 1.0 / rms : 0.0;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x) {
    x[i] = (float)st[i] * inv_ref;
    x[N + i] = (float)ss[i] * inv_ref;
    x[2 * N + i] = (float)(v[i] * inv);
  }
}

// z = base + rms(v) o (base: v itself, or another preconditioner's z_0 = M_0 v)
__global__ void k_net_output(const double *__restrict__ base, const double *__restrict__ vnorm2,
                             const float *__restrict__ o, long N, double *__restrict__ z) {
  const double rms = sqrt(*vnorm2 / (double)N);
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x)
    z[i] = base[i] + rms * (double)o[i];
}

int gridn(long n) { return (int)std::max(1L, std::min((n + 255) / 256, 8192L)); }

// The same for R vectors at once (blockIdx.y = r): v_r at v + r ldv, ||v_r||^2
// at scal[8 r + slot], input image r at x + 3 r N, z_r at z + r ldz.
__global__ void k_net_input_b(const double *__restrict__ st, const double *__restrict__ ss,
                              const double *__restrict__ v, long ldv, const double *__restrict__ scal, int slot,
                              long N, float inv_ref, float *__restrict__ x) {
  const int r = blockIdx.y;
  const double rms = sqrt(scal[8 * r + slot] / (double)N);
  const double inv = rms > 0.0 ? 1.0 / rms : 0.0;
  const double *vr = v + (long)r * ldv;
  float *xr = x + 3L * r * N;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x) {
    xr[i] = (float)st[i] * inv_ref;
    xr[N + i] = (float)ss[i] * inv_ref;
    xr[2 * N + i] = (float)(vr[i] * inv);
  }
}

__global__ void k_net_output_b(const double *__restrict__ base, long ldb, const double *__restrict__ scal, int slot,
                               const float *__restrict__ o, long N, double *__restrict__ z, long ldz) {
  const int r = blockIdx.y;
  const double rms = sqrt(scal[8 * r + slot] / (double)N);
  const double *br = base + (long)r * ldb;
  const float *orr = o + (long)r * N;
  double *zr = z + (long)r * ldz;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x)
    zr[i] = br[i] + rms * (double)orr[i];
}

}  // namespace

// ------------------------------------------------------------ network host

struct ConvLayer {
  int co, ci, k;
  long w_off, b_off;  // into the flat parameter array
  long tc_off;        // 3x3 layers: their packed BF16 weights [9 S][co][32] in UnetImpl::ptc
};

// A cached TMA descriptor (encoding one costs host time on every launch).
struct MapEntry {
  const void *base;
  unsigned long long key[4];
  CUtensorMap map;
};

struct UnetImpl {
  int L = 4, C = 32, device = 0;
  std::vector<ConvLayer> layers;
  long nparams = 0;
  float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr, *wt = nullptr;
  __nv_bfloat16 *pb = nullptr;
  long step = 0;
  // activations for (B, n)
  int B = 0, n = 0;
  std::vector<float *> xin, a, cat, bl, dl, ebot;  // per level
  std::vector<float *> gx, ga, gcat, gbl, gdl, gebot;
  float *o = nullptr, *go = nullptr;
  double *part = nullptr, *h_part = nullptr;
  float *xin0_owned = nullptr;
  int *dev_err = nullptr;  // set by a tensor-core convolution whose bounded wait gave up
  // BF16 tensor-core forward: packed weights (rebuilt when the parameters
  // change), the NHWC BF16 copy of the current convolution's input, cached maps
  __nv_bfloat16 *ptc = nullptr;
  long ptc_elems = 0;
  bool ptc_dirty = true;
  __nv_bfloat16 *nhwc = nullptr;
  // BF16 NHWC inputs written by the convolutions themselves: hx, a level's
  // second convolution's input (C channels padded to slices); hcat[l], the
  // decoder's concatenation at level l (the upsampled half, then the skip)
  __nv_bfloat16 *hx = nullptr;
  std::vector<__nv_bfloat16 *> hcat;
  int train_tc = 0;  // operand parts of the training convolutions on the tensor cores (0: CUDA cores)
  // training buffers for the current (B, n), by form.  Tensor cores (dw_ready):
  // the split inputs of every convolution, kept by the forward for the weight
  // gradients, the split gradient of the current output, the partial sums.  CUDA
  // cores (core_ready): the FP32 gradient planes gdl and gebot, and the later
  // parts of a converted input.
  bool dw_ready = false, core_ready = false;
  std::vector<__nv_bfloat16 *> xsplit;  // 3 per layer
  __nv_bfloat16 *gsplit[3] = {nullptr, nullptr, nullptr};
  float *dw_part = nullptr, *db_part = nullptr;
  std::vector<DwJob> dw_jobs;  // per layer
  __nv_bfloat16 *nhwc_lo = nullptr, *nhwc_p2 = nullptr;
  // the split weights of every convolution of a training step and of its
  // adjoint: packed by the jobs, layer i's at wsp + wsp_f[i] and wsp + wsp_b[i]
  // (-1: on the CUDA cores)
  __nv_bfloat16 *wsp = nullptr;
  std::vector<PackJob> pack_jobs;
  long wsp_elems = 0;
  std::vector<long> wsp_f, wsp_b;
  std::vector<MapEntry> maps;
};

namespace {

void free_dw(UnetImpl *u) {
  for (__nv_bfloat16 *q : u->xsplit)
    if (q) vie_free(q);
  u->xsplit.clear();
  for (__nv_bfloat16 *&q : u->gsplit) {
    if (q) vie_free(q);
    q = nullptr;
  }
  if (u->dw_part) vie_free(u->dw_part);
  if (u->db_part) vie_free(u->db_part);
  u->dw_part = u->db_part = nullptr;
  u->dw_ready = false;
}

void free_acts(UnetImpl *u) {
  auto fr = [](std::vector<float *> &vv) {
    for (float *&q : vv)
      if (q) vie_free(q);
    vv.clear();
  };
  fr(u->xin); fr(u->a); fr(u->cat); fr(u->bl); fr(u->dl); fr(u->ebot);
  fr(u->gx); fr(u->ga); fr(u->gcat); fr(u->gbl); fr(u->gdl); fr(u->gebot);
  if (u->o) vie_free(u->o);
  if (u->go) vie_free(u->go);
  if (u->part) vie_free(u->part);
  if (u->h_part) vie_free_host(u->h_part);
  if (u->nhwc) vie_free(u->nhwc);
  u->nhwc = nullptr;
  if (u->hx) vie_free(u->hx);
  u->hx = nullptr;
  for (__nv_bfloat16 **q : {&u->nhwc_lo, &u->nhwc_p2, &u->wsp}) {
    if (*q) vie_free(*q);
    *q = nullptr;
  }
  for (__nv_bfloat16 *q : u->hcat)
    if (q) vie_free(q);
  u->hcat.clear();
  free_dw(u);
  u->core_ready = false;
  u->maps.clear();
  u->o = u->go = nullptr;
  u->part = nullptr;
  u->h_part = nullptr;
  u->B = u->n = 0;
}

// FP32 convolutions that training takes to the tensor cores in split precision
bool conv_split_ok(int Ci, int Co) { return Ci <= 2 * kTmaSlice && Co % 32 == 0 && Co <= 64; }

vie_status ensure_acts(UnetImpl *u, int B, int n, cudaStream_t st) {
  if (u->B >= B && u->n == n) return VIE_OK;
  free_acts(u);
  const int L = u->L, C = u->C;
  auto al = [](float **q, long count) -> vie_status {
    VIE_CUDA(vie_malloc((void **)q, sizeof(float) * std::max(1L, count)));
    return VIE_OK;
  };
  u->xin.assign(L, nullptr); u->a.assign(L, nullptr); u->cat.assign(L, nullptr);
  u->bl.assign(L, nullptr); u->dl.assign(L, nullptr); u->ebot.assign(1, nullptr);
  u->gx.assign(L, nullptr); u->ga.assign(L, nullptr); u->gcat.assign(L, nullptr);
  u->gbl.assign(L, nullptr); u->gdl.assign(L, nullptr); u->gebot.assign(1, nullptr);
  vie_status s;
  for (int l = 0; l < L; ++l) {
    const long hw = (long)(n >> l) * (n >> l);
    const int cin = l == 0 ? 3 : C;
    if ((s = al(&u->xin[l], (long)B * cin * hw)) != VIE_OK) return s;
    if ((s = al(&u->a[l], (long)B * C * hw)) != VIE_OK) return s;
    if ((s = al(&u->gx[l], (long)B * cin * hw)) != VIE_OK) return s;
    if ((s = al(&u->ga[l], (long)B * C * hw)) != VIE_OK) return s;
    if (l < L - 1) {
      if ((s = al(&u->cat[l], (long)B * 2 * C * hw)) != VIE_OK) return s;
      if ((s = al(&u->bl[l], (long)B * C * hw)) != VIE_OK) return s;
      if ((s = al(&u->dl[l], (long)B * C * hw)) != VIE_OK) return s;
      if ((s = al(&u->gcat[l], (long)B * 2 * C * hw)) != VIE_OK) return s;
      if ((s = al(&u->gbl[l], (long)B * C * hw)) != VIE_OK) return s;
    }
  }
  const long hwb = (long)(n >> (L - 1)) * (n >> (L - 1));
  if ((s = al(&u->ebot[0], (long)B * C * hwb)) != VIE_OK) return s;
  if ((s = al(&u->o, (long)B * n * n)) != VIE_OK) return s;
  if ((s = al(&u->go, (long)B * n * n)) != VIE_OK) return s;
  VIE_CUDA(vie_malloc((void **)&u->part, sizeof(double) * 1024));
  VIE_CUDA(vie_malloc_host((void **)&u->h_part, sizeof(double) * 1024));
  // the widest convolution input: 2 C channels (a decoder's concatenation), padded to slices
  VIE_CUDA(vie_malloc((void **)&u->nhwc,
                      sizeof(__nv_bfloat16) * (size_t)B * n * n * (size_t)(((2 * C + 31) / 32) * 32)));
  {
    // split weights: three parts for the forward convolutions, two for the adjoints
    const auto jobs = [u](const ConvLayer &c, bool flip) -> long {
      const int Ci = flip ? c.co : c.ci, Co = flip ? c.ci : c.co, np = flip ? 2 : 3;
      if (c.k != 3 || !conv_split_ok(Ci, Co)) return -1;
      const long at = u->wsp_elems;
      const int S = (Ci + kTmaSlice - 1) / kTmaSlice;
      for (int co0 = 0; co0 < Co; co0 += 32) {
        u->pack_jobs.push_back({c.w_off, u->wsp_elems, Ci, Co, S, co0, np, flip});
        u->wsp_elems += (long)np * 9 * S * 32 * kTmaSlice;
      }
      return at;
    };
    u->pack_jobs.clear();
    u->wsp_f.clear();
    u->wsp_b.clear();
    u->wsp_elems = 0;
    for (const ConvLayer &c : u->layers) {
      u->wsp_f.push_back(jobs(c, false));
      u->wsp_b.push_back(jobs(c, true));
    }
    VIE_CUDA(vie_malloc((void **)&u->wsp, sizeof(__nv_bfloat16) * (size_t)std::max(1L, u->wsp_elems)));
  }
  // the hand-off buffers, zeroed once: their padding channels are never written
  const size_t cp1 = (size_t)((C + 31) / 32) * 32, cp2 = (size_t)((2 * C + 31) / 32) * 32;
  VIE_CUDA(vie_malloc((void **)&u->hx, sizeof(__nv_bfloat16) * (size_t)B * n * n * cp1));
  VIE_CUDA(cudaMemsetAsync(u->hx, 0, sizeof(__nv_bfloat16) * (size_t)B * n * n * cp1, st));
  u->hcat.assign(L, nullptr);
  for (int l = 0; l < L - 1; ++l) {
    const size_t bytes = sizeof(__nv_bfloat16) * (size_t)B * (n >> l) * (n >> l) * cp2;
    VIE_CUDA(vie_malloc((void **)&u->hcat[l], bytes));
    VIE_CUDA(cudaMemsetAsync(u->hcat[l], 0, bytes, st));
  }
  u->B = B;
  u->n = n;
  return VIE_OK;
}

template <bool RELU, typename WT, int TY, int COBC>
void launch_conv3(const float *in, long in_bs, int Ci, const WT *w, const float *bias, float *out, long out_bs,
                  int Co, int H, int W, int B, cudaStream_t st) {
  const int cob = (Co + COBC - 1) / COBC;
  dim3 grid((W + TX - 1) / TX, (H + TY - 1) / TY, B * cob);
  k_conv3<RELU, WT, TY, COBC><<<grid, 256, 0, st>>>(in, in_bs, Ci, w, bias, out, out_bs, Co, H, W, cob);
}

// Tile shapes by decreasing work per thread: (TY, COBC) = (16, 32), (16, 16),
// (8, 16), (8, 8).  The first whose grid covers two CTAs per SM is taken, the
// smallest otherwise: the coarse U-Net levels have too few pixels to fill the
// GPU with 64 outputs per thread.
template <bool RELU, typename WT>
void conv3_shape(const float *in, long in_bs, int Ci, const WT *w, const float *bias, float *out, long out_bs,
                 int Co, int H, int W, int B, cudaStream_t st) {
  const long tx = (W + TX - 1) / TX;
  auto ctas = [&](int ty, int cobc) { return tx * ((H + ty - 1) / ty) * B * ((Co + cobc - 1) / cobc); };
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const long want = 2L * (sms > 0 ? sms : 1);
  if (ctas(16, 32) >= want)
    launch_conv3<RELU, WT, 16, 32>(in, in_bs, Ci, w, bias, out, out_bs, Co, H, W, B, st);
  else if (ctas(16, 16) >= want)
    launch_conv3<RELU, WT, 16, 16>(in, in_bs, Ci, w, bias, out, out_bs, Co, H, W, B, st);
  else if (ctas(8, 16) >= want)
    launch_conv3<RELU, WT, 8, 16>(in, in_bs, Ci, w, bias, out, out_bs, Co, H, W, B, st);
  else
    launch_conv3<RELU, WT, 8, 8>(in, in_bs, Ci, w, bias, out, out_bs, Co, H, W, B, st);
}

// the tensor map for (base, key), encoded on first use and copied out by
// value (the cache may grow, and move its entries, on a later call)
vie_status cached_map(UnetImpl *u, const void *base, const unsigned long long (&key)[4], int rank,
                      const unsigned long long *dims, const unsigned long long *strides, const unsigned *box,
                      CUtensorMap *out) {
  for (const MapEntry &e : u->maps)
    if (e.base == base && e.key[0] == key[0] && e.key[1] == key[1] && e.key[2] == key[2] && e.key[3] == key[3]) {
      *out = e.map;
      return VIE_OK;
    }
  MapEntry e{base, {key[0], key[1], key[2], key[3]}, CUtensorMap{}};
  VIE_TRY(encode_bf16_map(&e.map, rank, base, dims, strides, box, 64));
  if (u->maps.size() >= 256) u->maps.clear();
  u->maps.push_back(e);
  *out = e.map;
  return VIE_OK;
}

// the BF16 convolutions the tensor-core kernel takes
bool conv_on_tensor_cores(const void *wtc, int Ci, int Co, const float *bias) {
  return wtc && Co % 16 == 0 && Co >= 16 && Co <= 32 && Ci <= 2 * kTmaSlice && bias;
}

// The BF16 3x3 convolution on the tensor cores (k_conv3_tma): input to BF16
// NHWC, then the implicit GEMM.  wtc: the layer's packed weights.
// Fused NHWC hand-off between convolutions (all optional): in_h, the input
// already in BF16 NHWC with S 32-channel slices (else `in` is converted);
// out_h, a second output in BF16 NHWC at channel oh_c0 of pixels oh_cp
// channels apart (image stride oh_bs elements).
struct NhwcIo {
  const __nv_bfloat16 *in_h = nullptr;
  __nv_bfloat16 *out_h[3] = {nullptr, nullptr, nullptr};  // (parts past the first: split precision)
  long oh_bs = 0;
  int oh_cp = 0, oh_c0 = 0;
  bool wrote = false;  // set when out_h was written
  __nv_bfloat16 *const *split = nullptr;  // split-precision convolutions: where the input's parts are kept
  bool split_ready = false;               // they are there already (else they are written from the FP32 input)
  // the 1x1 head on the (at most 32) output channels: weights (BF16, or FP32 in
  // split precision), bias, result; head_done set when it was computed
  const void *head_w = nullptr;
  const float *head_b = nullptr;
  float *head_o = nullptr;
  bool head_done = false;
};

// the input's tensor map: NHWC BF16 at src, S slices; tiles of one row load
// halo boxes of Wb + 2 pixels (the kernel's halo mode)
// (fr > 0: the flat form's boxes of W + 2 pixels and fr rows)
vie_status conv_input_map(UnetImpl *u, const __nv_bfloat16 *src, int S, int H, int W, int B, int fr,
                          CUtensorMap *mx) {
  const int Cp = S * kTmaSlice, Wb = std::min(W, kTcM), R = fr > 0 ? fr : std::min(kTcM / Wb, H);
  const unsigned bw = R == 1 || fr > 0 ? (unsigned)Wb + 2 : (unsigned)Wb;
  const unsigned long long key[4] = {(unsigned long long)Cp | ((unsigned long long)bw << 32),
                                     (unsigned long long)W | ((unsigned long long)R << 32), (unsigned long long)H,
                                     (unsigned long long)B};
  const unsigned long long dims[4] = {(unsigned long long)Cp, (unsigned long long)W, (unsigned long long)H,
                                      (unsigned long long)B};
  const unsigned long long strides[3] = {2ull * Cp, 2ull * Cp * W, 2ull * Cp * W * H};
  const unsigned box[4] = {(unsigned)kTmaSlice, bw, (unsigned)R, 1u};
  return cached_map(u, src, key, 4, dims, strides, box, mx);
}

// packed weights [9 S][Co][32] at wtc
vie_status conv_weight_map(UnetImpl *u, const __nv_bfloat16 *wtc, int S, int Co, CUtensorMap *mw) {
  const unsigned long long key[4] = {(unsigned long long)S, (unsigned long long)Co, 0ull, 1ull};
  const unsigned long long dims[2] = {(unsigned long long)kTmaSlice, 9ull * S * Co};
  const unsigned long long strides[1] = {2ull * kTmaSlice};
  const unsigned box[2] = {(unsigned)kTmaSlice, (unsigned)Co};
  return cached_map(u, wtc, key, 2, dims, strides, box, mw);
}

// Launch k_conv3_tma with np operand parts (maps mx[p], mw[p]; np > 1: the
// split-precision form).
vie_status launch_conv_tma(UnetImpl *u, const CUtensorMap *mx, const CUtensorMap *mw, int np, const float *bias,
                           float *out, long out_bs, int Co, int H, int W, int Ci, int B, bool relu, cudaStream_t st,
                           NhwcIo *io) {
  const int S = (Ci + kTmaSlice - 1) / kTmaSlice;
  const int Wb = std::min(W, kTcM), R = std::min(kTcM / Wb, H);
  const int fr = conv_flat_rows(H, W, np);
  const int tiles_x = (W + Wb - 1) / Wb, tiles_y = (H + R - 1) / R;
  int dev = 0;
  VIE_CUDA(cudaGetDevice(&dev));
  DevProps prop;
  VIE_TRY(get_dev_props(dev, &prop));
  // two CTAs per SM (two epilogues and issuers in flight), each with half of
  // the SM's shared memory less the per-CTA reserve, where three stages fit;
  // else one with all of it.  Measured with 64 images at 128^2: one CTA per
  // SM 1.69 ms per forward, two 1.25, three 1.42, four 1.45.  (The occupancy
  // query reports one CTA per SM for this kernel at any shared-memory size;
  // two run side by side all the same, and a grid they could not share would
  // only run in two waves, each CTA taking every G-th tile.)
  const size_t optin = (size_t)prop.sharedMemPerBlockOptin;
  int per_sm = 2, nst = conv_stages(S, Co, Wb, (optin + 1024) / 2 - 1024, np, fr);
  if (nst < 3) {
    per_sm = 1;
    nst = conv_stages(S, Co, Wb, optin, np, fr);
  }
  if (nst < 2 || (fr > 0 && nst < S)) {
    set_error("BF16 convolution: not enough shared memory for two stages");
    return VIE_ERR_UNSUPPORTED;
  }
  const size_t smem = conv_tma_smem(S, Co, Wb, nst, np, fr);
  const void *k = np == 3   ? (relu ? (const void *)k_conv3_tma<true, 3> : (const void *)k_conv3_tma<false, 3>)
                  : np == 2 ? (relu ? (const void *)k_conv3_tma<true, 2> : (const void *)k_conv3_tma<false, 2>)
                            : (relu ? (const void *)k_conv3_tma<true, 1> : (const void *)k_conv3_tma<false, 1>);
  VIE_TRY(raise_smem_limit(k, smem));
  // all of the SM's unified memory as shared memory, so that two CTAs fit
  VIE_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
  WaitLimits wl = wait_limits(dev);
  // per_sm CTAs per SM, each taking every G-th tile
  int tiles = (fr > 0 ? (H * (W + 2) + kTcM - 1) / kTcM : tiles_x * tiles_y) * B;
  const int grid = std::min(tiles, per_sm * prop.multiProcessorCount);
  __nv_bfloat16 *oh = io ? io->out_h[0] : nullptr, *oh1 = io ? io->out_h[1] : nullptr,
                *oh2 = io ? io->out_h[2] : nullptr;
  long oh_bs = io ? io->oh_bs : 0;
  int oh_cp = io ? io->oh_cp : 0, oh_c0 = io ? io->oh_c0 : 0;
  const void *hw = io ? io->head_w : nullptr;
  const float *hb = io ? io->head_b : nullptr;
  float *ho = io ? io->head_o : nullptr;
  int nst_i = nst, S_i = S, Co_i = Co, H_i = H, W_i = W, Wb_i = Wb, R_i = R, fr_i = fr, tx_i = tiles_x;
  int kks = Ci <= 16 ? 1 : 2;  // 16-channel halves of a slice that are not all padding
  int *err = u->dev_err;
  // maps of the parts past np: copies of part 0 (not read)
  const CUtensorMap *x1 = np > 1 ? mx + 1 : mx, *w1 = np > 1 ? mw + 1 : mw;
  const CUtensorMap *x2 = np > 2 ? mx + 2 : mx, *w2 = np > 2 ? mw + 2 : mw;
  void *args[] = {(void *)mx, (void *)mw, (void *)x1, (void *)w1, (void *)x2, (void *)w2, (void *)&bias, (void *)&out,
                  (void *)&out_bs, (void *)&Co_i, (void *)&H_i, (void *)&W_i, (void *)&S_i, (void *)&Wb_i,
                  (void *)&R_i, (void *)&fr_i, (void *)&kks, (void *)&tx_i, (void *)&tiles, (void *)&nst_i, (void *)&wl, (void *)&err,
                  (void *)&oh, (void *)&oh1, (void *)&oh2, (void *)&oh_bs, (void *)&oh_cp, (void *)&oh_c0,
                  (void *)&hw, (void *)&hb, (void *)&ho};
  VIE_CUDA(cudaLaunchKernel(k, dim3((unsigned)grid), dim3(kConvThreads), args, smem, st));
  if (io) {
    io->wrote = oh != nullptr;
    io->head_done = ho != nullptr;
  }
  VIE_CHECK_LAUNCH("k_conv3_tma");
  return VIE_OK;
}

vie_status conv3_tma(UnetImpl *u, const float *in, long in_bs, int Ci, const __nv_bfloat16 *wtc, const float *bias,
                     float *out, long out_bs, int Co, int H, int W, int B, bool relu, cudaStream_t st, NhwcIo *io) {
  const int S = (Ci + kTmaSlice - 1) / kTmaSlice, Cp = S * kTmaSlice;
  const long plane = (long)H * W;
  const __nv_bfloat16 *src = io && io->in_h ? io->in_h : u->nhwc;
  if (!io || !io->in_h) {
    k_to_nhwc_bf16<<<gridn((long)B * plane), 256, 0, st>>>(in, in_bs, Ci, plane, Cp, B, u->nhwc);
    VIE_CHECK_LAUNCH("k_to_nhwc_bf16");
  }
  CUtensorMap mx, mw;
  VIE_TRY(conv_input_map(u, src, S, H, W, B, conv_flat_rows(H, W, 1), &mx));
  VIE_TRY(conv_weight_map(u, wtc, S, Co, &mw));
  return launch_conv_tma(u, &mx, &mw, 1, bias, out, out_bs, Co, H, W, Ci, B, relu, st, io);
}

// The FP32 convolution of training on the tensor cores in split precision: the
// input in np BF16 NHWC parts (xin), the weights packed per block of 32 output
// channels (wsp: np parts of every block), one launch per block.
vie_status conv3_split_run(UnetImpl *u, __nv_bfloat16 *const *xin, int Ci, const __nv_bfloat16 *wsp,
                           const float *bias, float *out, long out_bs, int Co, int H, int W, int B, bool relu, int np,
                           cudaStream_t st, NhwcIo *io = nullptr) {
  const int S = (Ci + kTmaSlice - 1) / kTmaSlice;
  const long plane = (long)H * W, part = 9L * S * 32 * kTmaSlice;
  CUtensorMap mx[3], mw[3];
  for (int q = 0; q < np; ++q) VIE_TRY(conv_input_map(u, xin[q], S, H, W, B, 0, &mx[q]));
  for (int co0 = 0; co0 < Co; co0 += 32, wsp += np * part) {
    for (int q = 0; q < np; ++q) VIE_TRY(conv_weight_map(u, wsp + q * part, S, 32, &mw[q]));
    VIE_TRY(launch_conv_tma(u, mx, mw, np, bias ? bias + co0 : nullptr, out + co0 * plane, out_bs, 32, H, W, Ci, B,
                            relu, st, io));
  }
  return VIE_OK;
}

vie_status conv3_split(UnetImpl *u, const float *in, long in_bs, int Ci, const __nv_bfloat16 *wsp, const float *bias,
                       float *out, long out_bs, int Co, int H, int W, int B, bool relu, int np, cudaStream_t st,
                       NhwcIo *io) {
  const int S = (Ci + kTmaSlice - 1) / kTmaSlice, Cp = S * kTmaSlice;
  const long plane = (long)H * W;
  __nv_bfloat16 *own[3] = {u->nhwc, u->nhwc_lo, u->nhwc_p2};
  __nv_bfloat16 *const *xin = io && io->split ? io->split : own;
  if (!(io && io->split && io->split_ready)) {
    if (np == 3)
      k_to_nhwc_split<3><<<gridn((long)B * plane), 256, 0, st>>>(in, in_bs, Ci, plane, Cp, B, xin[0], xin[1], xin[2]);
    else
      k_to_nhwc_split<2><<<gridn((long)B * plane), 256, 0, st>>>(in, in_bs, Ci, plane, Cp, B, xin[0], xin[1], xin[2]);
    VIE_CHECK_LAUNCH("k_to_nhwc_split");
  }
  return conv3_split_run(u, xin, Ci, wsp, bias, out, out_bs, Co, H, W, B, relu, np, st, io);
}

// every split weight of a training step
vie_status pack_split_weights(UnetImpl *u, cudaStream_t st) {
  for (size_t i = 0; i < u->pack_jobs.size(); i += kPackJobs) {
    const size_t cnt = std::min<size_t>(kPackJobs, u->pack_jobs.size() - i);
    PackJobs jobs{};
    std::copy_n(u->pack_jobs.begin() + i, cnt, jobs.job);
    k_pack_split_weights<<<dim3(18, (unsigned)cnt), 256, 0, st>>>(jobs, u->p, u->wsp);
    VIE_CHECK_LAUNCH("k_pack_split_weights");
  }
  return VIE_OK;
}

// wtc: the packed weights (BF16), or the split ones (FP32 in training; nullptr: CUDA cores)
// io (tensor-core path only; ignored, with io->wrote false, on the CUDA cores)
template <typename WT>
vie_status conv3(UnetImpl *u, const float *in, long in_bs, int Ci, const WT *w, const __nv_bfloat16 *wtc,
                 const float *bias, float *out, long out_bs, int Co, int H, int W, int B, bool relu,
                 cudaStream_t st, NhwcIo *io = nullptr) {
  if (io) io->wrote = io->head_done = false;
  if (io && Co > 32) io->head_o = nullptr;  // (more than one launch's channels)
  if constexpr (std::is_same<WT, __nv_bfloat16>::value) {
    if (conv_on_tensor_cores(wtc, Ci, Co, bias))
      return conv3_tma(u, in, in_bs, Ci, wtc, bias, out, out_bs, Co, H, W, B, relu, st, io);
  } else {
    if (u->train_tc > 1 && wtc)
      return conv3_split(u, in, in_bs, Ci, wtc, bias, out, out_bs, Co, H, W, B, relu, u->train_tc, st, io);
  }
  if (relu)
    conv3_shape<true, WT>(in, in_bs, Ci, w, bias, out, out_bs, Co, H, W, B, st);
  else
    conv3_shape<false, WT>(in, in_bs, Ci, w, bias, out, out_bs, Co, H, W, B, st);
  VIE_CHECK_LAUNCH("k_conv3");
  return VIE_OK;
}

// Forward through the network; weights FP32 (pw) or BF16 (pbw).
// the packed BF16 weights of every 3x3 layer, from the FP32 parameters
vie_status pack_tc_weights(UnetImpl *u, cudaStream_t st) {
  if (!u->ptc_dirty) return VIE_OK;
  for (const ConvLayer &c : u->layers) {
    if (c.k != 3) continue;
    const int S = (c.ci + kTmaSlice - 1) / kTmaSlice;
    k_pack_tc_weights<<<gridn(9L * S * c.co * kTmaSlice), 256, 0, st>>>(u->p + c.w_off, c.co, c.ci, S,
                                                                       u->ptc + c.tc_off);
    VIE_CHECK_LAUNCH("k_pack_tc_weights");
  }
  u->ptc_dirty = false;
  return VIE_OK;
}

template <typename WT>
vie_status forward(UnetImpl *u, const WT *pw, const float *x, int B, int n, cudaStream_t st) {
  const int L = u->L, C = u->C;
  vie_status s;
  int li = 0;
  const bool tc = std::is_same<WT, __nv_bfloat16>::value;
  if (tc && (s = pack_tc_weights(u, st)) != VIE_OK) return s;
  // training with kept split inputs: they are written by the layers before
  const bool split = !tc && u->train_tc == 3 && u->dw_ready;
  auto wtc = [&](const ConvLayer &c) -> const __nv_bfloat16 * {
    if (tc) return u->ptc + c.tc_off;
    const long at = u->train_tc == 3 ? u->wsp_f[&c - u->layers.data()] : -1;
    return at >= 0 ? u->wsp + at : nullptr;
  };
  const float *xl = x;
  long xl_bs = 3L * n * n;
  // NHWC hand-off (tensor cores): each convolution also writes the next one's
  // input, the encoder's second convolution its skip into the decoder's
  // concatenation, and pooling and upsampling theirs
  const int cp1 = ((C + 31) / 32) * 32, cp2 = ((2 * C + 31) / 32) * 32;
  const bool handoff = split || (tc && C % 8 == 0);
  // a layer's kept split input (3 parts)
  auto kept = [&](const ConvLayer &c) { return split ? &u->xsplit[3 * (&c - u->layers.data())] : nullptr; };
  // where a layer's input is handed over: its kept parts, else h
  auto hand = [&](NhwcIo &io, const ConvLayer &next, __nv_bfloat16 *h, long bs, int cp, int c0) {
    if (!handoff) return;
    for (int q = 0; q < (split ? 3 : 1); ++q) io.out_h[q] = split ? kept(next)[q] : h;
    io.oh_bs = bs;
    io.oh_cp = cp;
    io.oh_c0 = c0;
  };
  auto take = [&](NhwcIo &io, const ConvLayer &c, bool there, const __nv_bfloat16 *h) {
    io.split = kept(c);
    io.split_ready = split && there;
    io.in_h = tc && there ? h : nullptr;
  };
  // the last convolution takes the 1x1 head along (as a pass of its own 40 us
  // of a forward of 64 images at 128^2)
  const ConvLayer &hd = u->layers.back();
  bool head_done = false;
  auto head = [&](NhwcIo &io) {
    io.head_w = pw + hd.w_off;
    io.head_b = u->p + hd.b_off;
    io.head_o = u->o;
  };
  std::vector<char> skip_h(L, 0);
  bool pooled = false;  // the level's input was handed over by the pooling
  for (int l = 0; l < L; ++l) {
    const int H = n >> l;
    const long hw = (long)H * H;
    const ConvLayer &c1 = u->layers[li++], &c2 = u->layers[li++];
    NhwcIo io1, io2;
    take(io1, c1, pooled, u->nhwc);
    hand(io1, c2, u->hx, hw * cp1, cp1, 0);
    if ((s = conv3(u, xl, xl_bs, c1.ci, pw + c1.w_off, wtc(c1), u->p + c1.b_off, u->a[l], (long)C * hw, C, H,
                   H, B, true, st, &io1)) != VIE_OK)
      return s;
    float *e = l < L - 1 ? u->cat[l] + (long)C * hw : u->ebot[0];
    const long e_bs = l < L - 1 ? 2L * C * hw : (long)C * hw;
    take(io2, c2, io1.wrote, u->hx);
    if (l < L - 1) hand(io2, u->layers[2 * L + 2 * (L - 2 - l)], u->hcat[l], hw * cp2, cp2, C);
    if (L == 1) head(io2);
    if ((s = conv3(u, u->a[l], (long)C * hw, C, pw + c2.w_off, wtc(c2), u->p + c2.b_off, e, e_bs, C, H, H, B,
                   true, st, &io2)) != VIE_OK)
      return s;
    head_done = io2.head_done;
    skip_h[l] = io2.wrote;
    if (l < L - 1) {
      const ConvLayer &next = u->layers[li];
      xl = u->xin[l + 1];
      xl_bs = (long)C * hw / 4;
      const dim3 grid((unsigned)((B * hw / 4 + 255) / 256), (unsigned)(cp1 / 8));
      pooled = handoff && (split || conv_on_tensor_cores(wtc(next), next.ci, next.co, u->p + next.b_off));
      if (!pooled)
        k_avgpool<<<coarse_grid(H, H, C, B), 256, 0, st>>>(e, e_bs, u->xin[l + 1], xl_bs, C, H, H, B);
      else if (split)
        k_avgpool_nhwc<3><<<grid, 256, 0, st>>>(e, e_bs, u->xin[l + 1], xl_bs, C, H, H, B, kept(next)[0],
                                                kept(next)[1], kept(next)[2], cp1);
      else
        k_avgpool_nhwc<1><<<grid, 256, 0, st>>>(e, e_bs, u->xin[l + 1], xl_bs, C, H, H, B, u->nhwc, nullptr, nullptr,
                                                cp1);
      VIE_CHECK_LAUNCH("k_avgpool");
    }
  }
  const float *d = u->ebot[0];
  long d_bs = (long)C * (n >> (L - 1)) * (n >> (L - 1));
  for (int l = L - 2; l >= 0; --l) {
    const int H = n >> l;
    const long hw = (long)H * H;
    const ConvLayer &c1 = u->layers[li++], &c2 = u->layers[li++];
    NhwcIo io1, io2;
    const bool up_h = skip_h[l] && (split || conv_on_tensor_cores(wtc(c1), c1.ci, c1.co, u->p + c1.b_off));
    if (up_h) {
      // the upsampled half beside the skip the encoder wrote; the FP32
      // concatenation's first half is not written (vie_unet_layer_io rebuilds it)
      const long per = hw / 4;
      const int grid = gridn((long)B * per * (C / 8));
      if (split)
        k_upsample_nhwc<3><<<grid, 256, 0, st>>>(d, d_bs, C, H, H, B, kept(c1)[0], kept(c1)[1], kept(c1)[2],
                                                 hw * cp2, cp2);
      else
        k_upsample_nhwc<1><<<grid, 256, 0, st>>>(d, d_bs, C, H, H, B, u->hcat[l], nullptr, nullptr, hw * cp2, cp2);
      VIE_CHECK_LAUNCH("k_upsample_nhwc");
    } else {
      k_upsample<<<coarse_grid(H, H, C, B), 256, 0, st>>>(d, d_bs, u->cat[l], 2L * C * hw, C, H, H, B);
      VIE_CHECK_LAUNCH("k_upsample");
    }
    take(io1, c1, up_h, u->hcat[l]);
    hand(io1, c2, u->hx, hw * cp1, cp1, 0);
    if ((s = conv3(u, u->cat[l], 2L * C * hw, 2 * C, pw + c1.w_off, wtc(c1), u->p + c1.b_off, u->bl[l],
                   (long)C * hw, C, H, H, B, true, st, &io1)) != VIE_OK)
      return s;
    take(io2, c2, io1.wrote, u->hx);
    if (l == 0) head(io2);
    if ((s = conv3(u, u->bl[l], (long)C * hw, C, pw + c2.w_off, wtc(c2), u->p + c2.b_off, u->dl[l],
                   (long)C * hw, C, H, H, B, true, st, &io2)) != VIE_OK)
      return s;
    head_done = io2.head_done;
    d = u->dl[l];
    d_bs = (long)C * hw;
  }
  if (head_done) return VIE_OK;
  k_head<WT><<<gridn((long)B * n * n), 256, 0, st>>>(d, d_bs, C, pw + hd.w_off, u->p + hd.b_off, u->o,
                                                     (long)n * n, B);
  VIE_CHECK_LAUNCH("k_head");
  return VIE_OK;
}

// the weight gradients of training take the tensor cores (k_conv3_dw_tc)
bool dw_on_tensor_cores(const UnetImpl *u) { return u->C == 32; }

// buffers of the tensor-core weight gradients for the current (B, n)
vie_status alloc_dw(UnetImpl *u) {
  DevProps prop;
  VIE_TRY(get_dev_props(u->device, &prop));
  u->xsplit.assign(3 * u->layers.size(), nullptr);
  for (size_t i = 0; i < u->layers.size(); ++i) {
    const ConvLayer &c = u->layers[i];
    if (c.k != 3) continue;
    const int l = (int)i < 2 * u->L ? (int)i / 2 : u->L - 2 - ((int)i - 2 * u->L) / 2;
    const size_t px = (size_t)u->B * (u->n >> l) * (u->n >> l), Cp = (size_t)(c.ci + 31) / 32 * 32;
    for (int q = 0; q < 3; ++q) VIE_CUDA(vie_malloc((void **)&u->xsplit[3 * i + q], sizeof(__nv_bfloat16) * px * Cp));
  }
  const size_t px = (size_t)u->B * u->n * u->n;
  for (__nv_bfloat16 *&q : u->gsplit) VIE_CUDA(vie_malloc((void **)&q, sizeof(__nv_bfloat16) * px * 32));
  // every layer's partial sums (added up by one launch at the end)
  long part = 0, part_b = 0;
  u->dw_jobs.assign(u->layers.size(), DwJob{});
  for (size_t i = 0; i < u->layers.size(); ++i) {
    const ConvLayer &c = u->layers[i];
    if (c.k != 3) continue;
    const int l = (int)i < 2 * u->L ? (int)i / 2 : u->L - 2 - ((int)i - 2 * u->L) / 2;
    const long lpx = (long)u->B * (u->n >> l) * (u->n >> l);
    u->dw_jobs[i] = {part, part_b, c.w_off, c.b_off, 0, (c.ci + 31) / 32, c.ci, 0};
    part += (long)prop.multiProcessorCount * 9 * 1024;
    part_b += 32 * (lpx / 64 < 1024 ? lpx / 64 + 1 : std::max(1024L, lpx / 512 + 1));
  }
  VIE_CUDA(vie_malloc((void **)&u->dw_part, sizeof(float) * (size_t)part));
  VIE_CUDA(vie_malloc((void **)&u->db_part, sizeof(float) * (size_t)part_b));
  u->dw_ready = true;
  return VIE_OK;
}

// buffers of the training step on the CUDA cores
vie_status alloc_core(UnetImpl *u) {
  const size_t B = (size_t)u->B, C = (size_t)u->C, n = (size_t)u->n;
  for (int l = 0; l < u->L; ++l) {
    const size_t hw = (n >> l) * (n >> l);
    VIE_CUDA(vie_malloc((void **)(l < u->L - 1 ? &u->gdl[l] : &u->gebot[0]), sizeof(float) * B * C * hw));
  }
  const size_t bytes = sizeof(__nv_bfloat16) * B * n * n * ((2 * C + 31) / 32 * 32);
  VIE_CUDA(vie_malloc((void **)&u->nhwc_lo, bytes));
  if (u->C == 32) VIE_CUDA(vie_malloc((void **)&u->nhwc_p2, bytes));  // (its forward has three parts)
  u->core_ready = true;
  return VIE_OK;
}

// The tensor-core form keeps every layer's split input (with four levels 1 KB a pixel of
// the batch more than the other form needs); where that does not fit, 32 channels
// train on the CUDA cores as the other widths do.
vie_status ensure_train(UnetImpl *u) {
  if (u->dw_ready || u->core_ready) return VIE_OK;
  vie_status s = VIE_ERR_OOM;
  if (dw_on_tensor_cores(u)) {
    if ((s = alloc_dw(u)) == VIE_OK) return VIE_OK;
    free_dw(u);
  }
  if (s == VIE_ERR_OOM) s = alloc_core(u);
  if (s != VIE_OK) free_acts(u);  // what was allocated goes with the activations
  return s;
}

// tensor map of NHWC rows: boxes of 32 channels x `bw` pixels of one row
vie_status conv_row_map(UnetImpl *u, const __nv_bfloat16 *src, int Cp, int H, int W, int B, int bw, CUtensorMap *m) {
  const unsigned long long key[4] = {(unsigned long long)Cp | ((unsigned long long)bw << 32), (unsigned long long)W,
                                     (unsigned long long)H, (unsigned long long)B | (1ull << 40)};
  const unsigned long long dims[4] = {(unsigned long long)Cp, (unsigned long long)W, (unsigned long long)H,
                                      (unsigned long long)B};
  const unsigned long long strides[3] = {2ull * Cp, 2ull * Cp * W, 2ull * Cp * W * H};
  const unsigned box[4] = {(unsigned)kTmaSlice, (unsigned)bw, 1u, 1u};
  return cached_map(u, src, key, 4, dims, strides, box, m);
}

// The backward pass of one 3x3 convolution with ReLU (output `act`) on the
// tensor cores: gout is masked by act > 0 and split once, for the weight
// gradient (three parts), the bias gradient's sums and the input gradient (the
// first two parts).
struct GradIn {
  int from = kFromG;  // GradFrom
  const float *g = nullptr, *g2 = nullptr;
  long bs = 0, bs2 = 0;
};
vie_status conv3_backward_tc(UnetImpl *u, const ConvLayer &c, const GradIn &go, const float *act, long a_bs,
                             float *gin, long gin_bs, int H, int B, cudaStream_t st) {
  const long hw = (long)H * H;
  const int blocks = split_blocks(B * hw), steps = split_steps(B * hw);
  DwJob &job = u->dw_jobs[&c - u->layers.data()];
  const auto mask = [&](auto k) {
    k<<<blocks, 256, 0, st>>>(go.g, go.bs, go.g2, go.bs2, act, a_bs, H, hw, B, u->gsplit[0], u->gsplit[1],
                              u->gsplit[2], u->db_part + job.part_b, steps);
  };
  if (go.from == kFromHead)
    mask(k_mask_split<kFromHead>);
  else if (go.from == kFromUp)
    mask(k_mask_split<kFromUp>);
  else if (go.from == kFromPool)
    mask(k_mask_split<kFromPool>);
  else
    mask(k_mask_split<kFromG>);
  VIE_CHECK_LAUNCH("k_mask_split");
  DevProps prop;
  VIE_TRY(get_dev_props(u->device, &prop));
  const int S = (c.ci + kTmaSlice - 1) / kTmaSlice, Wp = std::min(kTcM, (H + 15) / 16 * 16);
  const int segs = (H + kTcM - 1) / kTcM;
  const int ctas = (int)std::max(1L, std::min((long)prop.multiProcessorCount / S, (long)B * segs * H));
  DwMaps maps;
  const size_t layer = &c - u->layers.data();
  for (int q = 0; q < kDwParts; ++q) {
    VIE_TRY(conv_row_map(u, u->xsplit[3 * layer + q], S * kTmaSlice, H, H, B, Wp + 2, &maps.x[q]));
    VIE_TRY(conv_row_map(u, u->gsplit[q], 32, H, H, B, Wp, &maps.g[q]));
  }
  const size_t smem = dw_smem(Wp);
  VIE_TRY(raise_smem_limit((const void *)k_conv3_dw_tc, smem));
  k_conv3_dw_tc<<<dim3((unsigned)ctas, (unsigned)S), kConvThreads, smem, st>>>(
      maps, H, H, B, Wp, segs, u->dw_part + job.part, wait_limits(u->device), u->dev_err);
  VIE_CHECK_LAUNCH("k_conv3_dw_tc");
  job.ctas = ctas;
  job.blocks = blocks;
  if (gin)
    VIE_TRY(conv3_split_run(u, u->gsplit, c.co, u->wsp + u->wsp_b[layer], nullptr, gin, gin_bs, c.ci, H, H, B, false, 2,
                            st));
  return VIE_OK;
}

// u->g += the partial sums that conv3_backward_tc left for every layer
vie_status dw_reduce(UnetImpl *u, cudaStream_t st) {
  DwJobs jobs{};
  int cnt = 0, blocks = 0;
  for (size_t i = 0; i < u->layers.size(); ++i) {
    if (u->layers[i].k == 3) {
      blocks = std::max(blocks, u->dw_jobs[i].S * 9 * 32 + 1);
      jobs.job[cnt++] = u->dw_jobs[i];
    }
    if (cnt > 0 && (cnt == kDwJobs || i + 1 == u->layers.size())) {
      k_dw_reduce<<<dim3((unsigned)blocks, (unsigned)cnt), 256, 0, st>>>(jobs, u->dw_part, u->db_part, u->g);
      VIE_CHECK_LAUNCH("k_dw_reduce");
      cnt = 0;
    }
  }
  return VIE_OK;
}

// dw/db of a 3x3 convolution and, if gin, the input gradient (adjoint conv).
vie_status conv3_backward(UnetImpl *u, const ConvLayer &c, const float *in, long in_bs, const float *gout,
                          long g_bs, float *gin, long gin_bs, int H, int B, cudaStream_t st) {
  const int cib = (c.ci + CIB - 1) / CIB, cob = (c.co + COB - 1) / COB;
  // images per CTA: about four CTAs per SM in all, each adding its sums once
  const long per_split = (long)((H + TX - 1) / TX) * ((H + WY - 1) / WY) * cob * cib;
  int sms = 0, dev = 0;
  VIE_CUDA(cudaGetDevice(&dev));
  DevProps prop;
  VIE_TRY(get_dev_props(dev, &prop));
  sms = prop.multiProcessorCount;
  const int splits = (int)std::max(1L, std::min<long>(B, (4L * sms + per_split - 1) / per_split));
  dim3 grid((H + TX - 1) / TX, (H + WY - 1) / WY, splits * cob * cib);
  k_conv3_dw<<<grid, 256, 0, st>>>(in, in_bs, c.ci, gout, g_bs, c.co, H, H, u->g + c.w_off, u->g + c.b_off,
                                  cib, cob, B, splits);
  VIE_CHECK_LAUNCH("k_conv3_dw");
  if (gin) {
    const long at = u->wsp_b[&c - u->layers.data()];
    if (at < 0) {
      k_flip<<<gridn((long)c.co * c.ci * 9), 256, 0, st>>>(u->p + c.w_off, c.co, c.ci, u->wt);
      VIE_CHECK_LAUNCH("k_flip");
    }
    vie_status s = conv3<float>(u, gout, g_bs, c.co, u->wt, at < 0 ? nullptr : u->wsp + at, nullptr, gin, gin_bs,
                                c.ci, H, H, B, false, st);
    if (s != VIE_OK) return s;
  }
  return VIE_OK;
}

vie_status relu_mask(float *g, long g_bs, const float *a, long a_bs, long per, int B, cudaStream_t st) {
  k_relu_mask<<<gridn((long)B * per), 256, 0, st>>>(g, g_bs, a, a_bs, per, B);
  VIE_CHECK_LAUNCH("k_relu_mask");
  return VIE_OK;
}

// Backward pass from go (d loss / d o); gradients accumulate into u->g.
vie_status backward(UnetImpl *u, const float *x, int B, int n, cudaStream_t st) {
  const int L = u->L, C = u->C;
  vie_status s;
  // one convolution's backward pass; gout is masked by its ReLU's output act
  // first (on the tensor cores that pass also takes the step that gout would
  // come from, where `from` is given)
  auto back = [&](const ConvLayer &c, const float *in, long in_bs, float *gout, long g_bs, const float *act,
                  long a_bs, float *gin, long gin_bs, int H, const GradIn *from = nullptr) -> vie_status {
    if (u->dw_ready) {
      GradIn go;
      go.g = gout;
      go.bs = g_bs;
      return conv3_backward_tc(u, c, from ? *from : go, act, a_bs, gin, gin_bs, H, B, st);
    }
    VIE_TRY(relu_mask(gout, g_bs, act, a_bs, (long)C * H * H, B, st));
    return conv3_backward(u, c, in, in_bs, gout, g_bs, gin, gin_bs, H, B, st);
  };
  int li = (int)u->layers.size() - 1;
  const ConvLayer &hd = u->layers[li];
  const float *d = L > 1 ? u->dl[0] : u->ebot[0];
  float *gd = L > 1 ? u->gdl[0] : u->gebot[0];
  const long plane0 = (long)n * n;
  {
    // (C + 1) x K blocks, K slices of the pixels (the partials fit u->part's 1024 doubles)
    const int K = std::max(1, std::min(1024 / (C + 1), (int)std::min(64L, (long)B * plane0 / 4096 + 1)));
    k_head_bwd_w<<<dim3((unsigned)(C + 1), (unsigned)K), 256, 0, st>>>(u->go, d, (long)C * plane0, C, plane0, B,
                                                                      u->part);
    VIE_CHECK_LAUNCH("k_head_bwd_w");
    k_head_bwd_w_finish<<<1, ((C + 1 + 31) / 32) * 32, 0, st>>>(u->part, C, K, u->g + hd.w_off, u->g + hd.b_off);
    VIE_CHECK_LAUNCH("k_head_bwd_w_finish");
  }
  // where the next convolution's output gradient comes from (tensor cores)
  GradIn from;
  from.from = kFromHead;
  from.g = u->go;
  from.bs = plane0;
  from.g2 = u->p + hd.w_off;
  if (!u->dw_ready) {
    k_head_bwd_data<<<gridn((long)B * C * plane0), 256, 0, st>>>(u->go, C, u->p + hd.w_off, gd, (long)C * plane0,
                                                                  plane0, B);
    VIE_CHECK_LAUNCH("k_head_bwd_data");
  }
  --li;
  // decoder, l = 0 .. L-2 (reverse of the forward order)
  for (int l = 0; l <= L - 2; ++l) {
    const int H = n >> l;
    const long hw = (long)H * H;
    const ConvLayer &c2 = u->layers[li--];
    const ConvLayer &c1 = u->layers[li--];
    if ((s = back(c2, u->bl[l], (long)C * hw, u->gdl[l], (long)C * hw, u->dl[l], (long)C * hw, u->gbl[l],
                  (long)C * hw, H, &from)) != VIE_OK)
      return s;
    if ((s = back(c1, u->cat[l], 2L * C * hw, u->gbl[l], (long)C * hw, u->bl[l], (long)C * hw, u->gcat[l],
                  2L * C * hw, H)) != VIE_OK)
      return s;
    // upsample part of the concat -> gradient of d_{l+1}
    float *gnext = (l + 1 <= L - 2) ? u->gdl[l + 1] : u->gebot[0];
    from = GradIn{kFromUp, u->gcat[l], nullptr, 2L * C * hw, 0};
    if (!u->dw_ready) {
      k_upsample_bwd<<<coarse_grid(H, H, C, B), 256, 0, st>>>(u->gcat[l], 2L * C * hw, gnext, (long)C * hw / 4,
                                                                   C, H, H, B);
      VIE_CHECK_LAUNCH("k_upsample_bwd");
    }
  }
  // encoder, l = L-1 .. 0; grad of e_l: concat slice (l < L-1) + pool path
  for (int l = L - 1; l >= 0; --l) {
    const int H = n >> l;
    const long hw = (long)H * H;
    const ConvLayer &c1 = u->layers[2 * l], &c2 = u->layers[2 * l + 1];
    float *ge;
    long ge_bs;
    const float *e;
    long e_bs;
    if (l < L - 1) {
      ge = u->gcat[l] + (long)C * hw;
      ge_bs = 2L * C * hw;
      e = u->cat[l] + (long)C * hw;
      e_bs = 2L * C * hw;
      // + pool path from level l+1's input gradient
      from = GradIn{kFromPool, ge, u->gx[l + 1], ge_bs, (long)C * hw / 4};
      if (!u->dw_ready) {
        k_avgpool_bwd<<<coarse_grid(H, H, C, B), 256, 0, st>>>(u->gx[l + 1], (long)C * hw / 4, ge, ge_bs, C, H, H,
                                                                B, 1);
        VIE_CHECK_LAUNCH("k_avgpool_bwd");
      }
    } else {
      ge = u->gebot[0];
      ge_bs = (long)C * hw;
      e = u->ebot[0];
      e_bs = (long)C * hw;
    }
    if ((s = back(c2, u->a[l], (long)C * hw, ge, ge_bs, e, e_bs, u->ga[l], (long)C * hw, H, &from)) != VIE_OK)
      return s;
    const float *xl = l == 0 ? x : u->xin[l];
    const long xl_bs = l == 0 ? 3L * hw : (long)C * hw;
    if ((s = back(c1, xl, xl_bs, u->ga[l], (long)C * hw, u->a[l], (long)C * hw, l > 0 ? u->gx[l] : nullptr,
                  (long)C * hw, H)) != VIE_OK)
      return s;
  }
  return u->dw_ready ? dw_reduce(u, st) : VIE_OK;
}

vie_status loss_grad(UnetImpl *u, const float *x, const float *t, const float *wts, int B, int n, double *loss,
                     cudaStream_t st) {
  vie_status s;
  if ((s = ensure_acts(u, B, n, st)) != VIE_OK || (s = ensure_train(u)) != VIE_OK) return s;
  if ((s = pack_split_weights(u, st)) != VIE_OK) return s;
  // the training convolutions on the tensor cores in split precision: the
  // forward in three parts (24 bits an operand, FP32's own; the tensor cores'
  // accumulation truncates, about 1e-5 of the loss: in two parts its
  // ~1e-5 relative error flipped the ReLU masks of pre-activations near zero,
  // each flip moving a gradient entry by a whole term, 3.6e-3 relative
  // against the FP64 reference, 1e-4 allowed), the input gradients in two
  struct TrainTc {
    UnetImpl *u;
    TrainTc(UnetImpl *q, int np) : u(q) { u->train_tc = np; }
    ~TrainTc() { u->train_tc = 0; }
  };
  {
    TrainTc tc3(u, 3);
    if ((s = forward<float>(u, u->p, x, B, n, st)) != VIE_OK) return s;
  }
  const long cnt = (long)B * n * n;
  const int blocks = 512;
  k_mse<<<blocks, 256, 0, st>>>(u->o, t, cnt, (long)n * n, wts, u->go, u->part);
  VIE_CHECK_LAUNCH("k_mse");
  // the loss partials leave u->part before the backward pass reuses it
  VIE_CUDA(cudaMemcpyAsync(u->h_part, u->part, sizeof(double) * blocks, cudaMemcpyDeviceToHost, st));
  VIE_CUDA(cudaMemsetAsync(u->g, 0, sizeof(float) * u->nparams, st));
  {
    TrainTc tc2(u, 2);
    if ((s = backward(u, x, B, n, st)) != VIE_OK) return s;
  }
  // a tensor-core kernel that gave up on a wait left NaN in the gradients
  int *e = reinterpret_cast<int *>(u->h_part + blocks);
  VIE_CUDA(cudaMemcpyAsync(e, u->dev_err, sizeof(int), cudaMemcpyDeviceToHost, st));
  VIE_CUDA(cudaStreamSynchronize(st));
  if (*e != 0) return unet_take_error(u, st);
  double sum = 0.0;
  for (int i = 0; i < blocks; ++i) sum += u->h_part[i];
  *loss = sum / (double)cnt;
  return VIE_OK;
}

}  // namespace

// ---- used by the FGMRES driver (vie_api.cu)
vie_status unet_precondition(UnetImpl *u, const double *sigma_t, const double *sigma_s, double inv_ref,
                             const double *v, const double *vnorm2, int n, float *xbuf, const double *base,
                             double *z, cudaStream_t st) {
  vie_status s;
  if ((s = ensure_acts(u, 1, n, st)) != VIE_OK) return s;
  const long N = (long)n * n;
  k_net_input<<<gridn(N), 256, 0, st>>>(sigma_t, sigma_s, v, vnorm2, N, (float)inv_ref, xbuf);
  VIE_CHECK_LAUNCH("k_net_input");
  if ((s = forward<__nv_bfloat16>(u, u->pb, xbuf, 1, n, st)) != VIE_OK) return s;
  k_net_output<<<gridn(N), 256, 0, st>>>(base ? base : v, vnorm2, u->o, N, z);
  VIE_CHECK_LAUNCH("k_net_output");
  return VIE_OK;
}

// R preconditioner applications in one forward pass of R images (the batched
// FGMRES driver): z_r = base_r + rms(v_r) Net(sigma_t / s_ref, sigma_s / s_ref,
// v_r / rms(v_r)), BF16 weights; base_r = v_r, or (base non-null) another
// preconditioner's result that the network corrects.
vie_status unet_precondition_batch(UnetImpl *u, const double *sigma_t, const double *sigma_s, double inv_ref,
                                   const double *v, long ldv, const double *scal, int slot, int R, int n,
                                   float *xbuf, const double *base, long ldb, double *z, long ldz, cudaStream_t st) {
  vie_status s;
  if ((s = ensure_acts(u, R, n, st)) != VIE_OK) return s;
  const long N = (long)n * n;
  const dim3 grid((unsigned)std::max(1L, std::min((N + 255) / 256, 1024L)), (unsigned)R);
  k_net_input_b<<<grid, 256, 0, st>>>(sigma_t, sigma_s, v, ldv, scal, slot, N, (float)inv_ref, xbuf);
  VIE_CHECK_LAUNCH("k_net_input_b");
  if ((s = forward<__nv_bfloat16>(u, u->pb, xbuf, R, n, st)) != VIE_OK) return s;
  k_net_output_b<<<grid, 256, 0, st>>>(base ? base : v, base ? ldb : ldv, scal, slot, u->o, N, z, ldz);
  VIE_CHECK_LAUNCH("k_net_output_b");
  return VIE_OK;
}

// VIE_ERR_TIMEOUT (and the word cleared) if a tensor-core convolution of this
// network gave up on a bounded wait since the last check; synchronises `st`.
vie_status unet_take_error(UnetImpl *u, cudaStream_t st) {
  int e = 0;
  VIE_CUDA(cudaMemcpyAsync(&e, u->dev_err, sizeof(int), cudaMemcpyDeviceToHost, st));
  VIE_CUDA(cudaStreamSynchronize(st));
  if (e == 0) return VIE_OK;
  VIE_CUDA(cudaMemsetAsync(u->dev_err, 0, sizeof(int), st));
  set_error("a tensor-core convolution gave up on a bounded device wait (its output is NaN)");
  return VIE_ERR_TIMEOUT;
}

int *unet_error_word(UnetImpl *u) { return u->dev_err; }

}  // namespace vie

using namespace vie;

struct vie_unet {
  UnetImpl impl;
};

namespace vie {
UnetImpl *unet_impl(vie_unet *u) { return &u->impl; }
int unet_levels(vie_unet *u) { return u->impl.L; }
}  // namespace vie

extern "C" {

vie_status vie_unet_create(vie_unet **out, int levels, int channels, unsigned long long seed, int device) {
  if (!out || levels < 1 || levels > 6 || channels < 1 || channels > 32) {
    set_error("vie_unet_create: 1 <= levels <= 6, 1 <= channels <= 32");
    return VIE_ERR_INVALID_ARG;
  }
  *out = nullptr;
  int prev = -1;
  cudaGetDevice(&prev);
  VIE_CUDA(cudaSetDevice(device));
  vie_unet *u = new vie_unet();
  UnetImpl &U = u->impl;
  U.L = levels;
  U.C = channels;
  U.device = device;
  long off = 0;
  long tc = 0;  // packed BF16 weights of the 3x3 layers
  auto add = [&](int co, int ci, int k) {
    ConvLayer c{co, ci, k, off, off + (long)co * ci * k * k, tc};
    off = c.b_off + co;
    if (k == 3) tc += 9L * ((ci + kTmaSlice - 1) / kTmaSlice) * co * kTmaSlice;
    U.layers.push_back(c);
  };
  for (int l = 0; l < levels; ++l) {
    add(channels, l == 0 ? 3 : channels, 3);
    add(channels, channels, 3);
  }
  for (int l = levels - 2; l >= 0; --l) {
    add(channels, 2 * channels, 3);
    add(channels, channels, 3);
  }
  add(1, channels, 1);
  U.nparams = off;
  U.ptc_elems = tc;
  long max_w = 0;
  for (auto &c : U.layers) max_w = std::max(max_w, (long)c.co * c.ci * c.k * c.k);
  // He initialisation from SplitMix64 + Box-Muller, biases zero
  std::vector<float> h(off, 0.f);
  unsigned long long state = seed;
  auto next = [&]() {
    state += 0x9E3779B97F4A7C15ull;
    unsigned long long z = state;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return ((z >> 11) + 0.5) * (1.0 / 9007199254740992.0);
  };
  for (auto &c : U.layers) {
    const double std = sqrt(2.0 / (c.ci * c.k * c.k));
    for (long i = 0; i < (long)c.co * c.ci * c.k * c.k; ++i) {
      const double u1 = next(), u2 = next();
      h[c.w_off + i] = (float)(std * sqrt(-2.0 * log(u1)) * cos(2.0 * kPi * u2));
    }
  }
  vie_status s = VIE_OK;
  cudaError_t e = cudaSuccess;
  for (float **q : {&U.p, &U.g, &U.m, &U.v})
    if (e == cudaSuccess) e = vie_malloc((void **)q, sizeof(float) * off);
  if (e == cudaSuccess) e = vie_malloc((void **)&U.wt, sizeof(float) * max_w);
  if (e == cudaSuccess) e = vie_malloc((void **)&U.pb, sizeof(__nv_bfloat16) * off);
  if (e == cudaSuccess) e = vie_malloc((void **)&U.dev_err, sizeof(int));
  if (e == cudaSuccess) e = vie_malloc((void **)&U.ptc, sizeof(__nv_bfloat16) * std::max(1L, U.ptc_elems));
  if (e == cudaSuccess) e = cudaMemset(U.dev_err, 0, sizeof(int));
  if (e == cudaSuccess) e = cudaMemcpy(U.p, h.data(), sizeof(float) * off, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(U.m, 0, sizeof(float) * off);
  if (e == cudaSuccess) e = cudaMemset(U.v, 0, sizeof(float) * off);
  if (e != cudaSuccess) s = cuda_fail(e, "vie_unet_create");
  if (s == VIE_OK) {
    k_to_bf16<<<gridn(off), 256>>>(U.p, U.pb, off);
    e = cudaDeviceSynchronize();
    if (e != cudaSuccess) s = cuda_fail(e, "vie_unet_create");
  }
  if (prev >= 0) cudaSetDevice(prev);
  if (s != VIE_OK) {
    for (void *q : {(void *)U.p, (void *)U.g, (void *)U.m, (void *)U.v, (void *)U.wt, (void *)U.pb,
                    (void *)U.dev_err, (void *)U.ptc})
      if (q) vie_free(q);
    delete u;
    return s;
  }
  *out = u;
  return VIE_OK;
}

vie_status vie_unet_destroy(vie_unet *u) {
  if (!u) return VIE_OK;
  cudaSetDevice(u->impl.device);
  cudaDeviceSynchronize();
  free_acts(&u->impl);
  for (void *q : {(void *)u->impl.p, (void *)u->impl.g, (void *)u->impl.m, (void *)u->impl.v,
                  (void *)u->impl.wt, (void *)u->impl.pb, (void *)u->impl.dev_err, (void *)u->impl.ptc})
    if (q) vie_free(q);
  delete u;
  return VIE_OK;
}

vie_status vie_unet_num_params(vie_unet *u, long long *n) {
  if (!u || !n) return VIE_ERR_INVALID_ARG;
  *n = u->impl.nparams;
  return VIE_OK;
}

vie_status vie_unet_get_params(vie_unet *u, float *host) {
  if (!u || !host) return VIE_ERR_INVALID_ARG;
  VIE_CUDA(cudaSetDevice(u->impl.device));
  VIE_CUDA(cudaMemcpy(host, u->impl.p, sizeof(float) * u->impl.nparams, cudaMemcpyDeviceToHost));
  return VIE_OK;
}

vie_status vie_unet_set_params(vie_unet *u, const float *host) {
  if (!u || !host) return VIE_ERR_INVALID_ARG;
  VIE_CUDA(cudaSetDevice(u->impl.device));
  VIE_CUDA(cudaMemcpy(u->impl.p, host, sizeof(float) * u->impl.nparams, cudaMemcpyHostToDevice));
  u->impl.ptc_dirty = true;
  k_to_bf16<<<gridn(u->impl.nparams), 256>>>(u->impl.p, u->impl.pb, u->impl.nparams);
  VIE_CHECK_LAUNCH("k_to_bf16");
  VIE_CUDA(cudaDeviceSynchronize());
  return VIE_OK;
}

vie_status vie_unet_forward(vie_unet *u, const float *x, float *o, int B, int n, int use_bf16, void *stream) {
  if (!u || !x || !o || B < 1 || n < 1 || (n % (1 << (u->impl.L - 1))) != 0) {
    set_error("vie_unet_forward: n must be divisible by 2^(levels-1)");
    return VIE_ERR_INVALID_ARG;
  }
  VIE_CUDA(cudaSetDevice(u->impl.device));
  cudaStream_t st = (cudaStream_t)stream;
  vie_status s = ensure_acts(&u->impl, B, n, st);
  if (s != VIE_OK) return s;
  s = use_bf16 ? forward<__nv_bfloat16>(&u->impl, u->impl.pb, x, B, n, st)
               : forward<float>(&u->impl, u->impl.p, x, B, n, st);
  if (s != VIE_OK) return s;
  VIE_CUDA(cudaMemcpyAsync(o, u->impl.o, sizeof(float) * (long)B * n * n, cudaMemcpyDeviceToDevice, st));
  // the tensor-core convolutions report a bounded wait that gave up here
  if (use_bf16) return unet_take_error(&u->impl, st);
  return VIE_OK;
}

vie_status vie_unet_layer_io(vie_unet *u, int layer, float *in, float *out, void *stream) {
  if (!u || !out || layer < 0 || layer >= (int)u->impl.layers.size() || u->impl.B < 1) {
    set_error("vie_unet_layer_io: no forward yet, or layer out of range");
    return VIE_ERR_INVALID_ARG;
  }
  UnetImpl &U = u->impl;
  VIE_CUDA(cudaSetDevice(U.device));
  cudaStream_t st = (cudaStream_t)stream;
  const int L = U.L, C = U.C, B = U.B, n = U.n;
  const ConvLayer &c = U.layers[layer];
  // where the most recent forward keeps this layer's input and output
  const float *src_in = nullptr, *src_out = nullptr;
  long in_bs = 0, out_bs = 0;
  int H = n;
  if (layer < 2 * L) {  // encoder level l: a_l = conv(x_l), e_l = conv(a_l)
    const int l = layer / 2;
    H = n >> l;
    const long hw = (long)H * H;
    if (layer % 2 == 0) {
      src_in = l == 0 ? nullptr : U.xin[l];
      in_bs = (long)c.ci * hw;
      src_out = U.a[l];
      out_bs = (long)C * hw;
    } else {
      src_in = U.a[l];
      in_bs = (long)C * hw;
      src_out = l < L - 1 ? U.cat[l] + (long)C * hw : U.ebot[0];
      out_bs = l < L - 1 ? 2L * C * hw : (long)C * hw;
    }
  } else if (layer < 2 * L + 2 * (L - 1)) {  // decoder, deepest level first
    const int k = layer - 2 * L, l = L - 2 - k / 2;
    H = n >> l;
    const long hw = (long)H * H;
    if (k % 2 == 0) {
      src_in = U.cat[l];
      in_bs = 2L * C * hw;
      src_out = U.bl[l];
      if (in) {
        // the BF16 forward hands the upsampled half to the convolution in
        // BF16 only: rebuild its FP32 copy from the level below
        const float *d = l == L - 2 ? U.ebot[0] : U.dl[l + 1];
        k_upsample<<<coarse_grid(H, H, C, B), 256, 0, st>>>(d, (long)C * hw / 4, U.cat[l], 2L * C * hw, C, H, H, B);
        VIE_CHECK_LAUNCH("k_upsample");
      }
    } else {
      src_in = U.bl[l];
      in_bs = (long)C * hw;
      src_out = U.dl[l];
    }
    out_bs = (long)C * hw;
  } else {  // head
    const long hw = (long)n * n;
    src_in = L > 1 ? U.dl[0] : U.ebot[0];
    in_bs = (long)C * hw;
    src_out = U.o;
    out_bs = hw;
  }
  const long hw = (long)H * H;
  if (in && src_in)
    VIE_CUDA(cudaMemcpy2DAsync(in, sizeof(float) * c.ci * hw, src_in, sizeof(float) * in_bs, sizeof(float) * c.ci * hw,
                               B, cudaMemcpyDefault, st));
  VIE_CUDA(cudaMemcpy2DAsync(out, sizeof(float) * c.co * hw, src_out, sizeof(float) * out_bs,
                             sizeof(float) * c.co * hw, B, cudaMemcpyDefault, st));
  VIE_CUDA(cudaStreamSynchronize(st));
  return VIE_OK;
}

vie_status vie_unet_loss_grad(vie_unet *u, const float *x, const float *t, int B, int n, float *grads_host,
                              double *loss, void *stream) {
  if (!u || !x || !t || !loss || B < 1 || (n % (1 << (u->impl.L - 1))) != 0) {
    set_error("vie_unet_loss_grad: bad arguments");
    return VIE_ERR_INVALID_ARG;
  }
  VIE_CUDA(cudaSetDevice(u->impl.device));
  cudaStream_t st = (cudaStream_t)stream;
  vie_status s = loss_grad(&u->impl, x, t, nullptr, B, n, loss, st);
  if (s != VIE_OK) return s;
  if (grads_host)
    VIE_CUDA(cudaMemcpy(grads_host, u->impl.g, sizeof(float) * u->impl.nparams, cudaMemcpyDeviceToHost));
  return VIE_OK;
}

vie_status vie_unet_train_step(vie_unet *u, const float *x, const float *t, const float *weights, int B,
                               int n, float lr, double *loss, void *stream) {
  if (!u || !x || !t || !loss || B < 1 || (n % (1 << (u->impl.L - 1))) != 0 || !(lr > 0.f)) {
    set_error("vie_unet_train_step: bad arguments");
    return VIE_ERR_INVALID_ARG;
  }
  VIE_CUDA(cudaSetDevice(u->impl.device));
  cudaStream_t st = (cudaStream_t)stream;
  UnetImpl &U = u->impl;
  vie_status s = loss_grad(&U, x, t, weights, B, n, loss, st);
  if (s != VIE_OK) return s;
  U.step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)U.step), c2 = 1.f - powf(b2, (float)U.step);
  k_adam<<<gridn(U.nparams), 256, 0, st>>>(U.p, U.g, U.m, U.v, U.pb, U.nparams, lr, b1, b2, 1e-8f, c1, c2);
  VIE_CHECK_LAUNCH("k_adam");
  U.ptc_dirty = true;
  return VIE_OK;
}

// File layout: int32 header {"UNET", version, levels, channels}, int64
// parameter count np, np FP32 parameters; version 2 adds the Adam state
// (int64 step, np FP32 first moments, np FP32 second moments) so that
// training can resume where it stopped.  Version 1 files (parameters only)
// still load, with the optimizer state reset.
vie_status vie_unet_save(vie_unet *u, const char *path) {
  if (!u || !path) return VIE_ERR_INVALID_ARG;
  UnetImpl &U = u->impl;
  const long np = U.nparams;
  std::vector<float> h(np), hm(np), hv(np);
  vie_status s = vie_unet_get_params(u, h.data());
  if (s != VIE_OK) return s;
  VIE_CUDA(cudaMemcpy(hm.data(), U.m, sizeof(float) * np, cudaMemcpyDeviceToHost));
  VIE_CUDA(cudaMemcpy(hv.data(), U.v, sizeof(float) * np, cudaMemcpyDeviceToHost));
  FILE *f = fopen(path, "wb");
  if (!f) {
    set_error(std::string("vie_unet_save: cannot open ") + path);
    return VIE_ERR_INVALID_ARG;
  }
  const int hdr[4] = {0x54454e55 /* "UNET" */, 2, U.L, U.C};
  const long long n64 = np, step = U.step;
  bool ok = fwrite(hdr, sizeof hdr, 1, f) == 1 && fwrite(&n64, sizeof n64, 1, f) == 1 &&
            fwrite(h.data(), sizeof(float), h.size(), f) == h.size() && fwrite(&step, sizeof step, 1, f) == 1 &&
            fwrite(hm.data(), sizeof(float), hm.size(), f) == hm.size() &&
            fwrite(hv.data(), sizeof(float), hv.size(), f) == hv.size();
  ok = (fclose(f) == 0) && ok;
  if (!ok) {
    set_error("vie_unet_save: write failed");
    return VIE_ERR_INVALID_ARG;
  }
  return VIE_OK;
}

vie_status vie_unet_load(vie_unet *u, const char *path) {
  if (!u || !path) return VIE_ERR_INVALID_ARG;
  UnetImpl &U = u->impl;
  FILE *f = fopen(path, "rb");
  if (!f) {
    set_error(std::string("vie_unet_load: cannot open ") + path);
    return VIE_ERR_INVALID_ARG;
  }
  int hdr[4];
  long long np = 0, step = 0;
  std::vector<float> h(U.nparams), hm(U.nparams, 0.f), hv(U.nparams, 0.f);
  bool ok = fread(hdr, sizeof hdr, 1, f) == 1 && fread(&np, sizeof np, 1, f) == 1 && hdr[0] == 0x54454e55 &&
            (hdr[1] == 1 || hdr[1] == 2) && hdr[2] == U.L && hdr[3] == U.C && np == U.nparams &&
            fread(h.data(), sizeof(float), h.size(), f) == h.size();
  if (ok && hdr[1] == 2)
    ok = fread(&step, sizeof step, 1, f) == 1 && step >= 0 &&
         fread(hm.data(), sizeof(float), hm.size(), f) == hm.size() &&
         fread(hv.data(), sizeof(float), hv.size(), f) == hv.size();
  fclose(f);
  if (!ok) {
    set_error("vie_unet_load: file does not match this network");
    return VIE_ERR_INVALID_ARG;
  }
  vie_status s = vie_unet_set_params(u, h.data());
  if (s != VIE_OK) return s;
  VIE_CUDA(cudaMemcpy(U.m, hm.data(), sizeof(float) * U.nparams, cudaMemcpyHostToDevice));
  VIE_CUDA(cudaMemcpy(U.v, hv.data(), sizeof(float) * U.nparams, cudaMemcpyHostToDevice));
  U.step = (long)step;
  return VIE_OK;
}

vie_status vie_unet_train_state(vie_unet *u, long long *step) {
  if (!u || !step) return VIE_ERR_INVALID_ARG;
  *step = u->impl.step;
  return VIE_OK;
}

}  // extern "C"
