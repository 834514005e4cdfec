// cnn.cu -- the learned initial guess: a 4-layer 3x3 convolutional network
// mapping per-cell (log c, f_1, f_2) to a per-cell guess (u_1 on the west
// face, u_2 on the south face, p), trained on solves of the method itself.
//
// Channels 3 -> 32 -> 32 -> 32 -> 3, zero padding, ReLU after the first three
// layers.  Weights and activations are stored in BF16, every product is
// accumulated in FP32; the optimizer (Adam) keeps FP32 master weights.
// Inputs, targets and outputs are planes with the x index fastest; weights
// [out][in][3][3].
#include "../../include/mgdarcy.h"
#include "async.cuh"
#include "ops.h"

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

namespace mgd {
namespace {

constexpr int NL = 4;
constexpr int CH[NL + 1] = {3, 32, 32, 32, 3};
constexpr int TILE = 16;   // output pixels per block side

inline unsigned cdiv(int64_t a, int64_t b) { return (unsigned)((a + b - 1) / b); }

__device__ __forceinline__ float bf(const __nv_bfloat16 v) { return __bfloat162float(v); }

// 32-channel tensors (pre-activations, BF16; backward signals, FP32) hold the
// channels of a pixel together: 64 or 128 contiguous bytes, moved 16 at a time.
// With planes per channel every block gathered its tile by 2- and 4-byte loads with
// two divisions each, which took three quarters of the time (for 16 images of 128^2:
// 32 -> 32 forward 49 -> 19 us, input gradient 80 -> 33, weight gradient 170 -> 33).  The network's
// input, target and output keep their planes.
constexpr int MT_HALO = TILE + 2;   // 18 x 18 input pixels per 16 x 16 output tile

// Output channel of row r of the 32-row weight tables: the accumulator columns that
// lane q of the four sharing a pixel holds become channels 4 q .. 4 q + 3 and 16 + 4 q ..,
// so that the four write whole 32-byte sectors.
__host__ __device__ constexpr int row_channel(int r) {
  return (r >> 4) * 16 + ((r & 7) >> 1) * 4 + ((r >> 3) & 1) * 2 + (r & 1);
}

// v where the pre-activation z is positive
__device__ __forceinline__ float4 relu_mask(const float4 v, const uint2 z) {
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&z);
  return make_float4(bf(h[0].x) <= 0.f ? 0.f : v.x, bf(h[0].y) <= 0.f ? 0.f : v.y, bf(h[1].x) <= 0.f ? 0.f : v.z,
                     bf(h[1].y) <= 0.f ? 0.f : v.w);
}
__device__ __forceinline__ uint2 to_bf16x4(const float4 v) {
  uint2 s;
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&s);
  h[0] = __floats2bfloat162_rn(v.x, v.y);
  h[1] = __floats2bfloat162_rn(v.z, v.w);
  return s;
}

// acc += a b on both halves (one instruction, each half rounded as fmaf)
__device__ __forceinline__ void fma2(float2& acc, const float2 a, const float2 b) {
  asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmov.b64 z, {%0, %1};\n\t"
      "fma.rn.f32x2 z, x, y, z;\n\tmov.b64 {%0, %1}, z;\n\t}"
      : "+f"(acc.x), "+f"(acc.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
}

// 3 x 3 convolution from 3 planes (FP32) to 32 channels in FP32 on the CUDA cores:
// the first layer (DGRAD false: y = conv + bias, BF16) and the input gradient of the
// last one (DGRAD true: flipped kernel, times the ReLU mask of zin, FP32).  A thread
// holds eight channels of eight pixels of a row: a window of ten values and six
// 16-byte weight reads serve 192 FMAs (two an instruction), so that shared memory keeps up with
// the FMA units (18 and 22 us for 16 images of 128^2; a pixel or two with all 32
// channels: 23 and 30, bound by the weight reads).  w: [27 = channel, tap][32].
constexpr int C3_PITCH = 20;
template <bool DGRAD>
__global__ void __launch_bounds__(128) k_conv3(const float* x, const float* w,
                                              const float* bias, const __nv_bfloat16* zin, int n,
                                              __nv_bfloat16* y, float* gx) {
  __shared__ __align__(16) float sx[3][MT_HALO][C3_PITCH];
  __shared__ __align__(16) float sw[27 * 32];
  pdl_wait();
  pdl_launch_dependents();
  const int b = blockIdx.z, tx0 = blockIdx.x * TILE, ty0 = blockIdx.y * TILE, tid = threadIdx.x;
  const float* xb = x + (int64_t)b * 3 * n * n;
  for (int q = tid; q < 3 * MT_HALO * MT_HALO; q += 128) {
    const int c = q / (MT_HALO * MT_HALO), r = q - c * MT_HALO * MT_HALO, ry = r / MT_HALO, rx = r - ry * MT_HALO;
    const int yy = ty0 + ry - 1, xx = tx0 + rx - 1;
    sx[c][ry][rx] = (yy >= 0 && yy < n && xx >= 0 && xx < n) ? xb[(int64_t)c * n * n + (int64_t)yy * n + xx] : 0.f;
  }
  for (int q = tid; q < 27 * 8; q += 128)
    reinterpret_cast<float4*>(sw)[q] = reinterpret_cast<const float4*>(w)[q];
  __syncthreads();
  const int c0 = (tid & 3) * 4, py = tid >> 3, px = ((tid >> 2) & 1) * 8;   // channels c0 .. c0 + 3 and c0 + 16 ..
  float2 acc[8][4];   // pixel, channel pair
#pragma unroll
  for (int o = 0; o < 4; ++o) {
    const float2 v = DGRAD ? make_float2(0.f, 0.f) : make_float2(bias[c0 + (o >> 1) * 16 + 2 * (o & 1)], bias[c0 + (o >> 1) * 16 + 2 * (o & 1) + 1]);
#pragma unroll
    for (int p = 0; p < 8; ++p) acc[p][o] = v;
  }
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int dy = 0; dy < 3; ++dy) {
      const float* row = &sx[c][py + dy][px];
      const float4 f0 = *reinterpret_cast<const float4*>(row), f1 = *reinterpret_cast<const float4*>(row + 4);
      const float2 f2 = *reinterpret_cast<const float2*>(row + 8);
      const float wnd[10] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w, f2.x, f2.y};
#pragma unroll
      for (int dx = 0; dx < 3; ++dx) {
        const float4* wr = reinterpret_cast<const float4*>(sw + (c * 9 + dy * 3 + dx) * 32 + c0);
        const float4 w0 = wr[0], w1 = wr[4];
        const float2 wp[4] = {{w0.x, w0.y}, {w0.z, w0.w}, {w1.x, w1.y}, {w1.z, w1.w}};
#pragma unroll
        for (int p = 0; p < 8; ++p)
#pragma unroll
          for (int o = 0; o < 4; ++o) fma2(acc[p][o], wp[o], make_float2(wnd[p + dx], wnd[p + dx]));
      }
    }
  const int oy = ty0 + py;
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    const int ox = tx0 + px + p;
    if (ox >= n || oy >= n) continue;
    const int64_t at = (((int64_t)b * n + oy) * n + ox) * 32 + c0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float4 v = make_float4(acc[p][2 * h].x, acc[p][2 * h].y, acc[p][2 * h + 1].x, acc[p][2 * h + 1].y);
      if constexpr (DGRAD)
        *reinterpret_cast<float4*>(gx + at + 16 * h) = relu_mask(v, *reinterpret_cast<const uint2*>(zin + at + 16 * h));
      else
        *reinterpret_cast<uint2*>(y + at + 16 * h) = to_bf16x4(v);
    }
  }
}

// Weight and bias gradients of the layers with a 3-channel side, FP32 on the CUDA
// cores: sums over all pixels of v[channel] s[plane][pixel + offset], v a 32-channel
// tensor (layer 0: its backward signal; layer 3: its input with ReLU, V3 true), s the
// three planes (layer 0: the input; layer 3: the output's gradient, whose offsets are
// the flipped taps).  Lane = channel, 27 sums in registers; the windows of a plane row
// serve eight pixels of two rows (three shared-memory reads for up to 48 FMAs).  Blocks take tiles in
// turn and keep their sums, so a block writes once: partial[block][27 x 32, bias].
// 93 -> 19 us per layer for 16 images of 128^2 (FMA units: 6).
constexpr int W3_PITCH = 20, W3_M = 28 * 32;
template <bool V3>
__global__ void __launch_bounds__(256, 3) k_wgrad3(const void* v_, const float* s, int n, int tx,
                                               int tiles, float* partial) {
  __shared__ __align__(16) float ss[3][MT_HALO][W3_PITCH];
  __shared__ float red[8][28][32];
  pdl_wait();
  pdl_launch_dependents();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float acc[27], bias[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int q = 0; q < 27; ++q) acc[q] = 0.f;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int b = tile / (tx * tx), r0 = tile - b * tx * tx, ty0 = r0 / tx * TILE, tx0 = (r0 % tx) * TILE;
    __syncthreads();   // the tile before has been read
    const float* sb = s + (int64_t)b * 3 * n * n;
    for (int q = tid; q < 3 * MT_HALO * MT_HALO; q += 256) {
      const int c = q / (MT_HALO * MT_HALO), r = q - c * MT_HALO * MT_HALO, ry = r / MT_HALO, rx = r - ry * MT_HALO;
      const int yy = ty0 + ry - 1, xx = tx0 + rx - 1;
      ss[c][ry][rx] = (yy >= 0 && yy < n && xx >= 0 && xx < n) ? sb[(int64_t)c * n * n + (int64_t)yy * n + xx] : 0.f;
    }
    __syncthreads();
    const int oy = ty0 + 2 * warp;   // rows oy and oy + 1
    const int64_t at = (((int64_t)b * n + oy) * n + tx0) * 32 + lane;
#pragma unroll 1
    for (int g = 0; g < TILE; g += 8) {
      float v[2][8];
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int p = 0; p < 8; ++p) {
          const bool in = oy + m < n && tx0 + g + p < n;
          const int64_t q = at + ((int64_t)m * n + g + p) * 32;
          if constexpr (V3) v[m][p] = in ? fmaxf(bf(reinterpret_cast<const __nv_bfloat16*>(v_)[q]), 0.f) : 0.f;
          else v[m][p] = in ? reinterpret_cast<const float*>(v_)[q] : 0.f;
        }
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int r = 0; r < 4; ++r) {   // plane rows of the windows of the two rows
          const float* row = &ss[c][2 * warp + r][g];
          const float4 f0 = *reinterpret_cast<const float4*>(row), f1 = *reinterpret_cast<const float4*>(row + 4);
          const float2 f2 = *reinterpret_cast<const float2*>(row + 8);
          const float wnd[10] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w, f2.x, f2.y};
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            const int dy = r - m;
            if (dy < 0 || dy > 2) continue;
#pragma unroll
            for (int dx = 0; dx < 3; ++dx)
#pragma unroll
              for (int p = 0; p < 8; ++p) acc[c * 9 + dy * 3 + dx] += v[m][p] * wnd[p + dx];
          }
        }
      if constexpr (!V3)
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
          for (int p = 0; p < 8; ++p) bias[0] += v[m][p];
    }
    if constexpr (V3)   // outside the image the planes read zero
#pragma unroll
      for (int c = 0; c < 3; ++c) bias[c] += ss[c][1 + tid / TILE][1 + tid % TILE];
  }
#pragma unroll
  for (int q = 0; q < 27; ++q) red[warp][q][lane] = acc[q];
  if constexpr (V3) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float a = bias[c];
#pragma unroll
      for (int sh = 16; sh > 0; sh >>= 1) a += __shfl_xor_sync(0xffffffffu, a, sh);
      if (lane == 0) red[warp][27][c] = a;
    }
  } else red[warp][27][lane] = bias[0];
  __syncthreads();
  for (int q = tid; q < W3_M; q += 256) {   // (the last layer's biases are three: the rest of the row stays unused)
    if (V3 && q >= 27 * 32 + 3) break;
    float a = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) a += red[w][q >> 5][q & 31];
    partial[(int64_t)blockIdx.x * W3_M + q] = a;
  }
}

// --- tensor-core convolutions ------------------------------------------------
// The 32-channel layers are contractions over K = 9 taps x 32 channels per
// output pixel: implicit GEMMs on the tensor cores (mma.sync m16n8k16, BF16
// operands, FP32 accumulation).  An FP32 operand (the backward signal) enters
// as two BF16 parts, hi = bf16(v) and lo = bf16(v - hi), each multiplied and
// accumulated in FP32, so that it keeps 16 significant bits.
constexpr int MT_CP = 40;                  // channel pitch of a pixel in shared memory (80 bytes: eight rows
                                           // of an ldmatrix fall into different banks)
constexpr int MT_KP = 9 * 32 + 8;          // weight row pitch (K = 288 plus padding)
constexpr int MT_WARPS = 8;                // warp w computes output rows 2w, 2w + 1 of the tile

__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// four 8 x 8 matrices of 16-bit values; lane l gives the address of row l % 8 of matrix l / 8
template <bool TRANS>
__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], const __nv_bfloat16* p) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  if constexpr (TRANS)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}

__device__ __forceinline__ uint4 relu8(uint4 v) {   // ReLU of a BF16 value is exact
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&v);
  const __nv_bfloat162 z = __floats2bfloat162_rn(0.f, 0.f);
#pragma unroll
  for (int e = 0; e < 4; ++e) h[e] = __hmax2(h[e], z);
  return v;
}

// hi and lo parts of four values
__device__ __forceinline__ void split4(const float4 v, uint2& hi, uint2& lo) {
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&hi);
  __nv_bfloat162* l = reinterpret_cast<__nv_bfloat162*>(&lo);
  h[0] = __floats2bfloat162_rn(v.x, v.y);
  h[1] = __floats2bfloat162_rn(v.z, v.w);
  l[0] = __floats2bfloat162_rn(v.x - bf(h[0].x), v.y - bf(h[0].y));
  l[1] = __floats2bfloat162_rn(v.z - bf(h[1].x), v.w - bf(h[1].y));
}

// The tile with a one-pixel halo (zero outside the image) of a BF16 tensor, ReLU
// applied, into xs [18][18][MT_CP].
template <int NTHREADS>
__device__ __forceinline__ void load_act_tile(const __nv_bfloat16* x, int b, int ty0, int tx0, int n,
                                              __nv_bfloat16* xs) {
  constexpr int CNT = MT_HALO * MT_HALO * 4, IT = (CNT + NTHREADS - 1) / NTHREADS;
  uint4 v[IT];
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int q = threadIdx.x + it * NTHREADS, p = q >> 2, ry = p / MT_HALO, rx = p - ry * MT_HALO;
    const int yy = ty0 + ry - 1, xx = tx0 + rx - 1;
    v[it] = make_uint4(0, 0, 0, 0);
    if (q < CNT && yy >= 0 && yy < n && xx >= 0 && xx < n)
      v[it] = reinterpret_cast<const uint4*>(x + (((int64_t)b * n + yy) * n + xx) * 32)[q & 3];
  }
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int q = threadIdx.x + it * NTHREADS;
    if (q < CNT) *reinterpret_cast<uint4*>(xs + (q >> 2) * MT_CP + (q & 3) * 8) = relu8(v[it]);
  }
}

// Shared memory of k_conv_mma: NPART input parts [18][18][MT_CP] then the
// weights [NOUTP][MT_KP], all BF16.
template <int NPART, int NOUTP>
constexpr size_t conv_mma_smem() {
  return sizeof(__nv_bfloat16) * ((size_t)NPART * MT_HALO * MT_HALO * MT_CP + (size_t)NOUTP * MT_KP);
}

// One 3x3 convolution from 32 input channels to NOUT output channels as an
// implicit GEMM per 16 x 16 output tile: M = 256 pixels, N = NOUT (padded to
// NOUTP, a multiple of 8), K = 288 ordered (tap, channel).
//  forward (DGRAD false): in = the BF16 pre-activation of the previous layer,
//    ReLU applied on load; NOUT = 32: y = conv + bias in BF16; NOUT = 3 (the last
//    layer): yf = conv + bias, FP32 planes;
//  input gradient (DGRAD true): in = the FP32 gradient of the layer output
//    (two BF16 parts), the flipped kernel with input and output channels
//    swapped; yf = result times the ReLU mask of zin (the pre-activation that
//    fed this layer), FP32.
// w: the layer's table [NOUTP][288] (rows in row_channel order for 32 channels).
template <int NOUT, bool DGRAD>
__global__ void __launch_bounds__(MT_WARPS * 32) k_conv_mma(const void* in_, const __nv_bfloat16* w,
                                                          const float* bias,
                                                          const __nv_bfloat16* zin, int n,
                                                          __nv_bfloat16* y, float* yf) {
  constexpr int NPART = DGRAD ? 2 : 1;
  constexpr int NOUTP = (NOUT + 7) / 8 * 8;
  constexpr int NT = NOUTP / 8;
  constexpr int NTHREADS = MT_WARPS * 32, PART = MT_HALO * MT_HALO * MT_CP;
  extern __shared__ __align__(16) unsigned char smraw[];
  __nv_bfloat16* xs = reinterpret_cast<__nv_bfloat16*>(smraw);   // [NPART][18][18][MT_CP]
  __nv_bfloat16* ws = xs + NPART * PART;                         // [NOUTP][MT_KP]
  const int b = blockIdx.z, tx0 = blockIdx.x * TILE, ty0 = blockIdx.y * TILE;
  const int tid = threadIdx.x;
  pdl_wait();
  pdl_launch_dependents();
  for (int q = tid; q < NOUTP * 36; q += NTHREADS) {   // 36 chunks of 16 bytes a row
    const int r = q / 36, k = q - r * 36;
    *reinterpret_cast<uint4*>(ws + r * MT_KP + k * 8) = reinterpret_cast<const uint4*>(w)[q];
  }
  if constexpr (DGRAD) {
    constexpr int CNT = MT_HALO * MT_HALO * 8, HALF = 6;
#pragma unroll
    for (int q0 = 0; q0 < CNT; q0 += HALF * NTHREADS) {
      float4 v[HALF];
#pragma unroll
      for (int it = 0; it < HALF; ++it) {
        const int q = q0 + tid + it * NTHREADS, p = q >> 3, ry = p / MT_HALO, rx = p - ry * MT_HALO;
        const int yy = ty0 + ry - 1, xx = tx0 + rx - 1;
        v[it] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (q < CNT && yy >= 0 && yy < n && xx >= 0 && xx < n)
          v[it] = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(in_) +
                                                  (((int64_t)b * n + yy) * n + xx) * 32)[q & 7];
      }
#pragma unroll
      for (int it = 0; it < HALF; ++it) {
        const int q = q0 + tid + it * NTHREADS;
        if (q >= CNT) continue;
        uint2 hi, lo;
        split4(v[it], hi, lo);
        __nv_bfloat16* dst = xs + (q >> 3) * MT_CP + (q & 7) * 4;
        *reinterpret_cast<uint2*>(dst) = hi;
        *reinterpret_cast<uint2*>(dst + PART) = lo;
      }
    }
  } else {
    load_act_tile<NTHREADS>(reinterpret_cast<const __nv_bfloat16*>(in_), b, ty0, tx0, n, xs);
  }
  __syncthreads();
  const int warp = tid >> 5, lane = tid & 31, g = lane >> 2, tq = lane & 3;
  float acc[2][NT][4];
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[m][j][i] = 0.f;
  const __nv_bfloat16* xa = xs + (2 * warp * MT_HALO + (lane & 15)) * MT_CP + (lane >> 4) * 8;
  // two n-tiles a load; with one n-tile (NOUT = 3) the upper matrices repeat it
  const __nv_bfloat16* wb = ws + ((NT > 1 ? (lane >> 4) * 8 : 0) + (lane & 7)) * MT_KP + ((lane >> 3) & 1) * 8;
#pragma unroll 2
  for (int kt = 0; kt < 18; ++kt) {
    const int t = kt >> 1, c0 = (kt & 1) * 16, dy = t / 3, dx = t - 3 * dy;
    uint32_t bfr[(NT + 1) / 2][4];
#pragma unroll
    for (int j = 0; j < (NT + 1) / 2; ++j) ldmatrix4<false>(bfr[j], wb + j * 16 * MT_KP + kt * 16);
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int part = 0; part < NPART; ++part) {
        uint32_t a[4];
        ldmatrix4<false>(a, xa + part * PART + ((m + dy) * MT_HALO + dx) * MT_CP + c0);
#pragma unroll
        for (int j = 0; j < NT; ++j) mma_16816(acc[m][j], a, bfr[j >> 1] + (j & 1) * 2);
      }
  }
#pragma unroll
  for (int m = 0; m < 2; ++m) {
    const int oy = ty0 + 2 * warp + m;
    if constexpr (NOUT == 32) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {   // pixels g and g + 8
        const int ox = tx0 + g + 8 * h;
        if (ox >= n || oy >= n) continue;
        const int64_t at = (((int64_t)b * n + oy) * n + ox) * 32 + 4 * tq;
#pragma unroll
        for (int k = 0; k < 2; ++k) {   // channels 4 tq .. 4 tq + 3, and 16 further
          float4 v = make_float4(acc[m][2 * k][2 * h], acc[m][2 * k][2 * h + 1], acc[m][2 * k + 1][2 * h], acc[m][2 * k + 1][2 * h + 1]);
          if constexpr (DGRAD) {
            *reinterpret_cast<float4*>(yf + at + 16 * k) = relu_mask(v, *reinterpret_cast<const uint2*>(zin + at + 16 * k));
          } else {
            const float* bs = bias + 4 * tq + 16 * k;
            v.x += bs[0], v.y += bs[1], v.z += bs[2], v.w += bs[3];
            *reinterpret_cast<uint2*>(y + at + 16 * k) = to_bf16x4(v);
          }
        }
      }
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int o = 2 * tq + (i & 1), ox = tx0 + g + (i >= 2 ? 8 : 0);
        if (o < NOUT && ox < n && oy < n)
          yf[(((int64_t)b * NOUT + o) * n + oy) * n + ox] = acc[m][0][i] + bias[o];
      }
    }
  }
}

// Weight and bias gradients of a 32 -> 32 layer as a GEMM on the tensor cores:
// C[o][tap * 32 + c] = sum over the pixels of gz[o][p] act(x)[c][p + tap offset],
// M = 32, N = 288, K = 256 pixels per tile (one k-step per tile row).  gz (FP32)
// enters as two BF16 parts; the activations are BF16 values with the ReLU applied,
// exact.  One warp per tap; both operands lie pixel by pixel, so their fragments come
// from transposing ldmatrix loads and a tap is an offset (no shifted copies).  Blocks
// take tiles in turn and keep their sums in the accumulators: three blocks per SM
// write one partial each instead of one per tile (38 MB for 16 images of 128^2).
// partial[block][(o, tap, c), bias].
constexpr int WG_THREADS = 9 * 32;
constexpr int WG_M = 32 * 32 * 9 + 32;
constexpr size_t wgrad_mma_smem() {
  return sizeof(__nv_bfloat16) * ((size_t)2 * TILE * TILE * MT_CP + (size_t)MT_HALO * MT_HALO * MT_CP);
}

__global__ void __launch_bounds__(WG_THREADS, 3) k_wgrad_mma(const float* gz, const __nv_bfloat16* x,
                                                         int n, int tx, int tiles, float* partial) {
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int GPART = TILE * TILE * MT_CP;
  __nv_bfloat16* gs = reinterpret_cast<__nv_bfloat16*>(smraw);   // [2][256 pixels][MT_CP]
  __nv_bfloat16* xs = gs + 2 * GPART;                            // [18][18][MT_CP]
  const int tid = threadIdx.x, tap = tid >> 5, lane = tid & 31, g = lane >> 2, tq = lane & 3;
  float acc[2][4][4];
  float4 bsum = make_float4(0.f, 0.f, 0.f, 0.f);   // of the channels 4 (tid % 8) ..
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[m][j][i] = 0.f;
  const __nv_bfloat16* ga = gs + ((lane >> 4) * 8 + (lane & 7)) * MT_CP + ((lane >> 3) & 1) * 8;
  const __nv_bfloat16* xb = xs + ((tap / 3) * MT_HALO + tap % 3 + ((lane >> 3) & 1) * 8 + (lane & 7)) * MT_CP + (lane >> 4) * 8;
  pdl_wait();
  pdl_launch_dependents();
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int b = tile / (tx * tx), r0 = tile - b * tx * tx, ty0 = r0 / tx * TILE, tx0 = (r0 % tx) * TILE;
    if (tile != (int)blockIdx.x) __syncthreads();   // the tile before has been read
    constexpr int CNT = TILE * TILE * 8, HALF = 4;
#pragma unroll
    for (int q0 = 0; q0 < CNT; q0 += HALF * WG_THREADS) {
      float4 v[HALF];
#pragma unroll
      for (int it = 0; it < HALF; ++it) {
        const int q = q0 + tid + it * WG_THREADS, p = q >> 3, yy = ty0 + p / TILE, xx = tx0 + p % TILE;
        v[it] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (q < CNT && yy < n && xx < n)
          v[it] = reinterpret_cast<const float4*>(gz + (((int64_t)b * n + yy) * n + xx) * 32)[q & 7];
      }
#pragma unroll
      for (int it = 0; it < HALF; ++it) {
        const int q = q0 + tid + it * WG_THREADS;
        if (q >= CNT) continue;
        uint2 hi, lo;
        split4(v[it], hi, lo);
        __nv_bfloat16* dst = gs + (q >> 3) * MT_CP + (q & 7) * 4;
        *reinterpret_cast<uint2*>(dst) = hi;
        *reinterpret_cast<uint2*>(dst + GPART) = lo;
        bsum.x += v[it].x, bsum.y += v[it].y, bsum.z += v[it].z, bsum.w += v[it].w;
      }
    }
    load_act_tile<WG_THREADS>(x, b, ty0, tx0, n, xs);
    __syncthreads();
#pragma unroll 2
    for (int kt = 0; kt < TILE; ++kt) {   // pixel row kt of the tile
      uint32_t bfr[2][4];
#pragma unroll
      for (int j = 0; j < 2; ++j) ldmatrix4<true>(bfr[j], xb + kt * MT_HALO * MT_CP + j * 16);
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int part = 0; part < 2; ++part) {
          uint32_t a[4];
          ldmatrix4<true>(a, ga + part * GPART + kt * TILE * MT_CP + m * 16);
#pragma unroll
          for (int j = 0; j < 4; ++j) mma_16816(acc[m][j], a, bfr[j >> 1] + (j & 1) * 2);
        }
    }
  }
  float* pb = partial + (int64_t)blockIdx.x * WG_M;
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        *reinterpret_cast<float2*>(pb + ((m * 16 + g + 8 * h) * 9 + tap) * 32 + j * 8 + 2 * tq) =
            make_float2(acc[m][j][2 * h], acc[m][j][2 * h + 1]);
  __syncthreads();
  float* red = reinterpret_cast<float*>(smraw);   // [thread][4]
  reinterpret_cast<float4*>(red)[tid] = bsum;
  __syncthreads();
  if (tid < 32) {
    float a = 0.f;
    for (int q = tid >> 2; q < WG_THREADS; q += 8) a += red[4 * q + (tid & 3)];
    pb[32 * 32 * 9 + tid] = a;
  }
}

// Sums of the weight-gradient partials of all layers, in a fixed order, into the
// layers' [out][in][3][3] gradients, and the loss (last block, FP64).  A block takes 32
// entries; eight lanes read them 16 bytes each, 32 groups of lanes share the partials
// (one thread per entry reading all partials one after the other took 65 us a layer,
// eight groups with 4-byte reads 34 us for all layers; now 12).
struct GradSums {
  const float* part[NL];
  int nblk[NL], m[NL], pitch[NL], first[NL + 1];   // partials, entries, partial size, first block of each layer
  int64_t out[NL];                      // offset of the layer's weights, then its biases
};
__global__ void __launch_bounds__(256) k_sum_gradients(const __grid_constant__ GradSums S, const float* lpart,
                                                      int nl, double count, float* grad,
                                                      float* loss) {
  __shared__ __align__(16) float red[32][32];
  const int tid = threadIdx.x;
  pdl_wait();
  if ((int)blockIdx.x == S.first[NL]) {
    __shared__ double dred[256];
    double s = 0.0;
#pragma unroll 4
    for (int i = tid; i < nl; i += 256) s += lpart[i];
    dred[tid] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
      if (tid < o) dred[tid] += dred[tid + o];
      __syncthreads();
    }
    if (tid == 0) *loss = (float)(dred[0] / count);
    return;
  }
  int l = 0;
  while ((int)blockIdx.x >= S.first[l + 1]) ++l;
  const int q0 = ((int)blockIdx.x - S.first[l]) * 32, w = tid >> 3, nblk = S.nblk[l], pitch = S.pitch[l];
  const float* p = S.part[l] + q0 + 4 * (tid & 7);
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
  for (int b = w; b < nblk; b += 32) {
    const float4 v = *reinterpret_cast<const float4*>(p + (int64_t)b * pitch);
    a.x += v.x, a.y += v.y, a.z += v.z, a.w += v.w;
  }
  *reinterpret_cast<float4*>(&red[w][4 * (tid & 7)]) = a;
  __syncthreads();
  const int q = q0 + tid;
  if (tid >= 32 || q >= S.m[l]) return;
  float s = 0.f;
#pragma unroll
  for (int k = 0; k < 32; ++k) s += red[k][tid];
  int at = q;   // biases follow the weights
  if (l == 0 && q < 864) at = (q & 31) * 27 + (q >> 5);                                 // (plane, offset), channel
  if (l == 3 && q < 864) at = ((q >> 5) / 9 * 32 + (q & 31)) * 9 + 8 - (q >> 5) % 9;    // flipped
  if ((l == 1 || l == 2) && q < 9216) at = (q / 288 * 32 + (q & 31)) * 9 + (q % 288 >> 5);
  grad[S.out[l] + at] = s;
}

// loss partial sums and dL/dy = 2 (y - t) / count for the mean squared error
__global__ void k_mse(const float* y, const float* t, int64_t count, float* g,
                      float* lpart) {
  __shared__ float red[32];
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  float d = 0.f;
  pdl_wait();
  pdl_launch_dependents();
  if (i < count) {
    d = y[i] - t[i];
    g[i] = 2.f * d / (float)count;
  }
  float s = d * d;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float a = 0.f;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) a += red[q];
    lpart[blockIdx.x] = a;
  }
}

__global__ void k_adam(float* __restrict__ w, float* __restrict__ m, float* __restrict__ v, const float* __restrict__ g,
                       int64_t count, float lr, float b1, float b2, float c1, float c2, float eps) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// The layers' weights in BF16, in the orders the kernels read: for the 3-channel sides
// (as FP32 numbers) c3f = layer 0 [in, tap][out], c3b = layer 3 flipped [out, tap][in];
// for the tensor cores mf[l] = [row][tap, in] and mb[l] = the flipped kernel [row][tap, out],
// rows in row_channel order (layer 3: out, padded to 8).  One launch per change of
// the weights; the convolutions copy their table in 16-byte pieces.
struct WeightTables {
  float *c3f, *c3b;
  __nv_bfloat16 *mf[NL], *mb[NL];
};
__global__ void k_weight_tables(const float* __restrict__ w, int64_t o0, int64_t o1, int64_t o2, int64_t o3, WeightTables T) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  auto rnd = [](float v) { return __bfloat162float(__float2bfloat16(v)); };
  if (i < 864) {
    T.c3f[i] = rnd(w[o0 + (i & 31) * 27 + (i >> 5)]);
    const int o = (i >> 5) / 9, t = (i >> 5) % 9;
    T.c3b[i] = rnd(w[o3 + (o * 32 + (i & 31)) * 9 + 8 - t]);
  }
  if (i >= 9216) return;
  const int r = i / 288, t = i % 288 >> 5, c = i & 31, o = row_channel(r);
  T.mf[1][i] = __float2bfloat16(w[o1 + (o * 32 + c) * 9 + t]);
  T.mf[2][i] = __float2bfloat16(w[o2 + (o * 32 + c) * 9 + t]);
  T.mb[1][i] = __float2bfloat16(w[o1 + (c * 32 + o) * 9 + 8 - t]);
  T.mb[2][i] = __float2bfloat16(w[o2 + (c * 32 + o) * 9 + 8 - t]);
  if (r < 8) T.mf[3][i] = __float2bfloat16(r < 3 ? w[o3 + (r * 32 + c) * 9 + t] : 0.f);
}

// network input features from the problem data: (log c, f_1, f_2), normalised
__global__ void k_features(const double* __restrict__ c, const double* __restrict__ f, int64_t cells,
                           const float* __restrict__ norm, float* __restrict__ in) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= cells) return;
  in[i] = ((float)log(c[i]) - norm[0]) / norm[3];
  in[cells + i] = ((float)f[i] - norm[1]) / norm[4];
  in[2 * cells + i] = ((float)f[cells + i] - norm[2]) / norm[5];
}

// RT_0 on n x n cells: per-cell (u_1 west face, u_2 south face, p) <-> dofs.
__global__ void k_fields_to_dofs(const float* __restrict__ out, const float* __restrict__ norm, int n,
                                 double* __restrict__ x) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nux = (int64_t)(n + 1) * n, cells = (int64_t)n * n;
  if (i >= 2 * nux + cells) return;
  if (i < nux) {   // u_x at (ix, iy), ix in [0, n]
    const int ix = (int)(i % (n + 1)), iy = (int)(i / (n + 1));
    x[i] = (ix == 0 || ix == n) ? 0.0 : (double)(out[(int64_t)iy * n + ix] * norm[9] + norm[6]);
  } else if (i < 2 * nux) {   // u_y at (ix, iy), iy in [0, n]
    const int64_t r = i - nux;
    const int ix = (int)(r % n), iy = (int)(r / n);
    x[i] = (iy == 0 || iy == n) ? 0.0 : (double)(out[cells + (int64_t)iy * n + ix] * norm[10] + norm[7]);
  } else {
    const int64_t r = i - 2 * nux;
    x[i] = (double)(out[2 * cells + r] * norm[11] + norm[8]);
  }
}

__global__ void k_dofs_to_fields(const double* __restrict__ x, const float* __restrict__ norm, int n,
                                 float* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nux = (int64_t)(n + 1) * n, cells = (int64_t)n * n;
  if (i >= cells) return;
  const int ix = (int)(i % n), iy = (int)(i / n);
  out[i] = ((float)x[(int64_t)iy * (n + 1) + ix] - norm[6]) / norm[9];
  out[cells + i] = ((float)x[nux + (int64_t)iy * n + ix] - norm[7]) / norm[10];
  out[2 * cells + i] = ((float)x[2 * nux + i] - norm[8]) / norm[11];
}

}  // namespace
}  // namespace mgd

using namespace mgd;

struct mg_cnn {
  int n = 0, max_batch = 0;
  cudaStream_t stream = nullptr;
  int64_t nparam = 0;
  int64_t woff[NL], boff[NL];
  float* master = nullptr;   // FP32 weights and biases, all layers
  float* m = nullptr;
  float* v = nullptr;
  float* grad = nullptr;     // gradients, then the loss
  float* host = nullptr;     // pinned copy of them
  WeightTables wt = {};           // BF16 weights
  __nv_bfloat16* z[NL - 1] = {};  // pre-activations of the 32-channel layers, channels of a pixel together
  float* gbuf[2] = {nullptr, nullptr};
  float* outf = nullptr;          // FP32 output of the last layer
  float* partial[NL] = {};        // weight-gradient partials of each layer
  int wg_blocks[NL] = {};         // at most this many
  float* lpart = nullptr;
  float* norm = nullptr;          // 12 floats: input mean[3], std[3], output mean[3], std[3]
  float* feat = nullptr;          // features of one problem for mg_cnn_guess
  int step = 0;
  std::vector<void*> allocs;
  ~mg_cnn() {
    for (void* p : allocs) cudaFree(p);
    if (host) cudaFreeHost(host);
  }
  template <typename T>
  cudaError_t alloc(T** p, size_t count) {
    void* q = nullptr;
    cudaError_t e = cudaMalloc(&q, count * sizeof(T));
    if (e == cudaSuccess) {
      allocs.push_back(q);
      *p = (T*)q;
    }
    return e;
  }
};

namespace {

// Whether the CUDA runtime reports p as device (or managed) memory.
bool on_device(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

mg_status not_on_device() { return set_last_error(MG_ERR_INVALID_ARG, "device pointers required"); }

mg_status cnn_cuda(cudaError_t e, const char* what) {
  if (e == cudaSuccess) return MG_OK;
  return set_last_error(e == cudaErrorMemoryAllocation ? MG_ERR_OOM : MG_ERR_CUDA,
                        std::string(what) + ": " + cudaGetErrorString(e));
}

// Launches of a pass follow one another (launch_pdl).
template <typename... KArgs, typename... Args>
void chain(const mg_cnn* N, dim3 grid, int threads, size_t smem, void (*kernel)(KArgs...), Args... args) {
  launch_pdl(kernel, grid, threads, smem, N->stream, args...);
}

// 3-plane convolution to 32 channels on the CUDA cores (k_conv3).
template <bool DGRAD>
void conv3(const mg_cnn* N, const float* x, const float* w, const float* bias, const __nv_bfloat16* zin, int batch,
           __nv_bfloat16* y, float* gx) {
  const dim3 grid(cdiv(N->n, TILE), cdiv(N->n, TILE), batch);
  chain(N, grid, 128, 0, k_conv3<DGRAD>, x, w, bias, zin, N->n, y, gx);
}

// 32-input-channel convolution on the tensor cores (k_conv_mma).
template <int NOUT, bool DGRAD>
void conv_mma(const mg_cnn* N, const void* in, const __nv_bfloat16* w, const float* bias, const __nv_bfloat16* zin,
              int batch, __nv_bfloat16* y, float* yf) {
  constexpr size_t smem = conv_mma_smem<DGRAD ? 2 : 1, (NOUT + 7) / 8 * 8>();
  static std::atomic<unsigned long long> attr{0};
  once_per_device(attr, [] {
    cudaFuncSetAttribute(k_conv_mma<NOUT, DGRAD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  });
  const dim3 grid(cdiv(N->n, TILE), cdiv(N->n, TILE), batch);
  chain(N, grid, MT_WARPS * 32, smem, k_conv_mma<NOUT, DGRAD>, in, w, bias, zin, N->n, y, yf);
}

// Blocks of layer l's weight gradient: the tiles, at most what the device holds at once.
int64_t tiles_of(const mg_cnn* N, int batch) { return (int64_t)cdiv(N->n, TILE) * cdiv(N->n, TILE) * batch; }
int wgrad_blocks(const mg_cnn* N, int l, int batch) { return (int)std::min<int64_t>(tiles_of(N, batch), N->wg_blocks[l]); }

constexpr int partial_pitch(int l) { return l == 0 || l == 3 ? W3_M : WG_M; }

// weight and bias gradients of a 32 -> 32 layer on the tensor cores
void wgrad_mma(const mg_cnn* N, int l, const float* gz, const __nv_bfloat16* x, int batch) {
  constexpr size_t smem = wgrad_mma_smem();
  static std::atomic<unsigned long long> attr{0};
  once_per_device(attr, [] {
    cudaFuncSetAttribute(k_wgrad_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  });
  chain(N, wgrad_blocks(N, l, batch), WG_THREADS, smem, k_wgrad_mma, gz, x, N->n, (int)cdiv(N->n, TILE),
        (int)tiles_of(N, batch), N->partial[l]);
}

// forward of the whole network on `batch` inputs (FP32, B x 3 x n x n): the
// first layer (3 input channels, K = 27) on the CUDA cores, the three layers
// with 32 input channels on the tensor cores
void forward(mg_cnn* N, const float* in, int batch) {
  conv3<false>(N, in, N->wt.c3f, N->master + N->boff[0], nullptr, batch, N->z[0], nullptr);
  conv_mma<32, false>(N, N->z[0], N->wt.mf[1], N->master + N->boff[1], nullptr, batch, N->z[1], nullptr);
  conv_mma<32, false>(N, N->z[1], N->wt.mf[2], N->master + N->boff[2], nullptr, batch, N->z[2], nullptr);
  conv_mma<3, false>(N, N->z[2], N->wt.mf[3], N->master + N->boff[3], nullptr, batch, nullptr, N->outf);
}

// gradients of the mean squared error into N->grad; returns the loss, and the
// gradients if grads_host is given
mg_status backward(mg_cnn* N, const float* in, const float* target, int batch, float* loss, float* grads_host) {
  const int64_t cnt = (int64_t)batch * 3 * N->n * N->n;
  const int tx = (int)cdiv(N->n, TILE), tiles = (int)tiles_of(N, batch);
  float* g3 = N->gbuf[0];
  chain(N, cdiv(cnt, 256), 256, 0, k_mse, N->outf, target, cnt, g3, N->lpart);
  // layer 3 (32 -> 3), input z[2] through ReLU
  chain(N, wgrad_blocks(N, 3, batch), 256, 0, k_wgrad3<true>, N->z[2], g3, N->n, tx, tiles, N->partial[3]);
  conv3<true>(N, g3, N->wt.c3b, nullptr, N->z[2], batch, nullptr, N->gbuf[1]);
  wgrad_mma(N, 2, N->gbuf[1], N->z[1], batch);
  conv_mma<32, true>(N, N->gbuf[1], N->wt.mb[2], nullptr, N->z[1], batch, nullptr, N->gbuf[0]);
  wgrad_mma(N, 1, N->gbuf[0], N->z[0], batch);
  conv_mma<32, true>(N, N->gbuf[0], N->wt.mb[1], nullptr, N->z[0], batch, nullptr, N->gbuf[1]);
  chain(N, wgrad_blocks(N, 0, batch), 256, 0, k_wgrad3<false>, N->gbuf[1], in, N->n, tx, tiles, N->partial[0]);
  GradSums S;
  S.first[0] = 0;
  for (int l = 0; l < NL; ++l) {
    S.part[l] = N->partial[l];
    S.nblk[l] = wgrad_blocks(N, l, batch);
    S.m[l] = CH[l + 1] * CH[l] * 9 + CH[l + 1];
    S.pitch[l] = partial_pitch(l);
    S.first[l + 1] = S.first[l] + (int)cdiv(S.m[l], 32);
    S.out[l] = N->woff[l];
  }
  chain(N, S.first[NL] + 1, 256, 0, k_sum_gradients, S, N->lpart, (int)cdiv(cnt, 256), (double)cnt, N->grad,
        N->grad + N->nparam);
  const int64_t from = grads_host ? 0 : N->nparam;   // the loss lies behind the gradients
  mg_status st = cnn_cuda(cudaMemcpyAsync(N->host + from, N->grad + from, (N->nparam + 1 - from) * sizeof(float),
                                          cudaMemcpyDeviceToHost, N->stream), "loss");
  if (st != MG_OK) return st;
  st = cnn_cuda(cudaStreamSynchronize(N->stream), "backward");
  if (st != MG_OK) return st;
  if (loss) *loss = N->host[N->nparam];
  if (grads_host) std::memcpy(grads_host, N->host, N->nparam * sizeof(float));
  return MG_OK;
}

void refresh_bf16(mg_cnn* N) {
  k_weight_tables<<<cdiv(9216, 256), 256, 0, N->stream>>>(N->master, N->woff[0], N->woff[1], N->woff[2], N->woff[3], N->wt);
}

uint64_t splitmix(uint64_t& s) {
  uint64_t z = (s += 0x9e3779b97f4a7c15ull);
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

}  // namespace

extern "C" {

mg_status mg_cnn_create(int n, int max_batch, uint64_t seed, void* cuda_stream, mg_cnn** out) {
  if (!out || n < 1 || max_batch < 1) return set_last_error(MG_ERR_INVALID_ARG, "bad network arguments");
  *out = nullptr;
  mg_cnn* N = new mg_cnn();
  N->n = n;
  N->max_batch = max_batch;
  N->stream = (cudaStream_t)cuda_stream;
  int64_t off = 0;
  for (int l = 0; l < NL; ++l) {
    N->woff[l] = off;
    off += (int64_t)CH[l + 1] * CH[l] * 9;
    N->boff[l] = off;
    off += CH[l + 1];
  }
  N->nparam = off;
  const int64_t act = (int64_t)max_batch * 32 * n * n;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (sms < 1) sms = 152;
  cudaError_t e = cudaSuccess;
  auto A = [&](cudaError_t r) {
    if (e == cudaSuccess) e = r;
  };
  A(N->alloc(&N->master, off));
  A(N->alloc(&N->m, off));
  A(N->alloc(&N->v, off));
  A(N->alloc(&N->grad, off + 1));
  A(cudaMallocHost((void**)&N->host, (off + 1) * sizeof(float)));
  A(N->alloc(&N->wt.c3f, 864));
  A(N->alloc(&N->wt.c3b, 864));
  for (int l = 1; l < NL; ++l) A(N->alloc(&N->wt.mf[l], l == 3 ? 8 * 288 : 9216));
  for (int l = 1; l < NL - 1; ++l) A(N->alloc(&N->wt.mb[l], 9216));
  for (int l = 0; l < NL - 1; ++l) A(N->alloc(&N->z[l], (size_t)act));
  A(N->alloc(&N->gbuf[0], act));
  A(N->alloc(&N->gbuf[1], act));
  A(N->alloc(&N->outf, (size_t)max_batch * 3 * n * n));
  for (int l = 0; l < NL; ++l) {
    N->wg_blocks[l] = 3 * sms;   // what 67 KB of shared memory leave room for (32 -> 32)
    A(N->alloc(&N->partial[l], (size_t)wgrad_blocks(N, l, max_batch) * partial_pitch(l)));
  }
  A(N->alloc(&N->lpart, cdiv((int64_t)max_batch * 3 * n * n, 256)));
  A(N->alloc(&N->norm, 12));
  A(N->alloc(&N->feat, (size_t)3 * n * n));
  if (e != cudaSuccess) {
    delete N;
    return cnn_cuda(e, "mg_cnn_create");
  }
  // He-normal weights (Box-Muller on a splitmix64 stream), zero biases
  std::vector<float> h(off, 0.f);
  uint64_t s = seed;
  for (int l = 0; l < NL; ++l) {
    const double sd = std::sqrt(2.0 / (9.0 * CH[l]));
    for (int64_t i = N->woff[l]; i < N->boff[l]; ++i) {
      const double u1 = ((splitmix(s) >> 11) + 0.5) * (1.0 / 9007199254740992.0);
      const double u2 = ((splitmix(s) >> 11) + 0.5) * (1.0 / 9007199254740992.0);
      h[i] = (float)(sd * std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2));
    }
  }
  const float nrm[12] = {0, 0, 0, 1, 1, 1, 0, 0, 0, 1, 1, 1};
  cudaMemcpy(N->master, h.data(), off * sizeof(float), cudaMemcpyHostToDevice);
  cudaMemcpy(N->norm, nrm, sizeof(nrm), cudaMemcpyHostToDevice);
  cudaMemset(N->m, 0, off * sizeof(float));
  cudaMemset(N->v, 0, off * sizeof(float));
  refresh_bf16(N);
  mg_status st = cnn_cuda(cudaStreamSynchronize(N->stream), "mg_cnn_create");
  if (st != MG_OK) {
    delete N;
    return st;
  }
  *out = N;
  return MG_OK;
}

void mg_cnn_destroy(mg_cnn* N) { delete N; }

int64_t mg_cnn_param_count(const mg_cnn* N) { return N ? N->nparam : 0; }

mg_status mg_cnn_get_params(mg_cnn* N, float* host) {
  if (!N || !host) return set_last_error(MG_ERR_INVALID_ARG, "null argument");
  return cnn_cuda(cudaMemcpy(host, N->master, N->nparam * sizeof(float), cudaMemcpyDeviceToHost), "get params");
}

mg_status mg_cnn_set_params(mg_cnn* N, const float* host) {
  if (!N || !host) return set_last_error(MG_ERR_INVALID_ARG, "null argument");
  mg_status st = cnn_cuda(cudaMemcpy(N->master, host, N->nparam * sizeof(float), cudaMemcpyHostToDevice), "set params");
  if (st != MG_OK) return st;
  refresh_bf16(N);
  return cnn_cuda(cudaStreamSynchronize(N->stream), "set params");
}

mg_status mg_cnn_set_normalisation(mg_cnn* N, const float* host12) {
  if (!N || !host12) return set_last_error(MG_ERR_INVALID_ARG, "null argument");
  return cnn_cuda(cudaMemcpy(N->norm, host12, 12 * sizeof(float), cudaMemcpyHostToDevice), "normalisation");
}

mg_status mg_cnn_forward(mg_cnn* N, const float* in, int batch, float* out) {
  if (!N || !in || !out || batch < 1 || batch > N->max_batch) return set_last_error(MG_ERR_INVALID_ARG, "bad arguments");
  if (!on_device(in) || !on_device(out)) return not_on_device();
  forward(N, in, batch);
  return cnn_cuda(cudaMemcpyAsync(out, N->outf, (size_t)batch * 3 * N->n * N->n * sizeof(float),
                                  cudaMemcpyDeviceToDevice, N->stream), "forward");
}

mg_status mg_cnn_gradients(mg_cnn* N, const float* in, const float* target, int batch, float* loss, float* grads_host) {
  if (!N || !in || !target || batch < 1 || batch > N->max_batch)
    return set_last_error(MG_ERR_INVALID_ARG, "bad arguments");
  if (!on_device(in) || !on_device(target)) return not_on_device();
  forward(N, in, batch);
  return backward(N, in, target, batch, loss, grads_host);
}

mg_status mg_cnn_train_step(mg_cnn* N, const float* in, const float* target, int batch, float lr, float* loss) {
  if (!N || !in || !target || batch < 1 || batch > N->max_batch || !(lr > 0.f))
    return set_last_error(MG_ERR_INVALID_ARG, "bad arguments");
  if (!on_device(in) || !on_device(target)) return not_on_device();
  forward(N, in, batch);
  mg_status st = backward(N, in, target, batch, loss, nullptr);
  if (st != MG_OK) return st;
  ++N->step;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - std::pow(b1, (float)N->step), c2 = 1.f - std::pow(b2, (float)N->step);
  k_adam<<<cdiv(N->nparam, 256), 256, 0, N->stream>>>(N->master, N->m, N->v, N->grad, N->nparam, lr, b1, b2, c1, c2,
                                                     1e-8f);
  refresh_bf16(N);
  return cnn_cuda(cudaGetLastError(), "train step");
}

mg_status mg_cnn_features(mg_cnn* N, const double* c, const double* f, float* in) {
  if (!N || !c || !f || !in) return set_last_error(MG_ERR_INVALID_ARG, "null argument");
  if (!on_device(c) || !on_device(f) || !on_device(in)) return not_on_device();
  const int64_t cells = (int64_t)N->n * N->n;
  k_features<<<cdiv(cells, 256), 256, 0, N->stream>>>(c, f, cells, N->norm, in);
  return cnn_cuda(cudaGetLastError(), "features");
}

mg_status mg_cnn_targets(mg_cnn* N, const double* x, float* target) {
  if (!N || !x || !target) return set_last_error(MG_ERR_INVALID_ARG, "null argument");
  if (!on_device(x) || !on_device(target)) return not_on_device();
  const int64_t cells = (int64_t)N->n * N->n;
  k_dofs_to_fields<<<cdiv(cells, 256), 256, 0, N->stream>>>(x, N->norm, N->n, target);
  return cnn_cuda(cudaGetLastError(), "targets");
}

mg_status mg_cnn_guess(mg_cnn* N, const double* c, const double* f, double* x0) {
  if (!N || !c || !f || !x0) return set_last_error(MG_ERR_INVALID_ARG, "null argument");
  if (!on_device(c) || !on_device(f) || !on_device(x0)) return not_on_device();
  const int64_t cells = (int64_t)N->n * N->n;
  k_features<<<cdiv(cells, 256), 256, 0, N->stream>>>(c, f, cells, N->norm, N->feat);
  forward(N, N->feat, 1);
  const int64_t ndof = 2 * (int64_t)(N->n + 1) * N->n + cells;
  k_fields_to_dofs<<<cdiv(ndof, 256), 256, 0, N->stream>>>(N->outf, N->norm, N->n, x0);
  return cnn_cuda(cudaGetLastError(), "guess");
}

}  // extern "C"
