// wsnet.cu -- the learned warm start: a small convolutional network that
// predicts the initial guess x0 of a variable-coefficient diffusion solve
// from the log-coefficient field g and the right-hand side b, trained on
// solutions the library's own solver produced.  Not in the paper: it extends
// the method, and plain zero-start CG stays the reference it is judged by.
//
// Network: six 3x3 convolutions with dilations d_l and zero padding,
// channels 2 -> 32 -> 32 -> 32 -> 32 -> 32 -> 1, ReLU between layers.
// Input (B, 2, H, W) = [g, b / rms(b)]; output (B, 1, H, W) =
// x / (rms(b) * out_scale).  Activations are NCHW.
//
// Training (FP32, deterministic): forward, mean-squared-error loss, backward
// (data gradients as a forward convolution with flipped, transposed weights;
// weight gradients as per-block partial sums reduced in a fixed order), Adam.
// Inference: weights, biases and activations in BF16, products formed in FP32
// (exact for BF16 operands) and summed in FP32; the four 32 -> 32 layers run
// on the tensor cores (tcgen05.mma, accumulator in tensor memory).
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <memory>
#include <vector>

#include "gk_device.cuh"
#include "gk_internal.h"

namespace gk {
namespace {

constexpr int kLayers = 6;
constexpr int kCh[kLayers + 1] = {2, 32, 32, 32, 32, 32, 1};
constexpr int kConvThreads = 256;

__device__ __forceinline__ float to_f(float v) { return v; }
template <typename T>
__device__ __forceinline__ T from_f(float v);
template <>
__device__ __forceinline__ float from_f<float>(float v) { return v; }

enum ConvMode { CONV_LINEAR = 0, CONV_RELU = 1, CONV_MASK = 2 };

// y[b, o, p] = epilogue(sum_{c, ky, kx} w[o, c, ky, kx] x[b, c, p + d (ky-1, kx-1)])
// One thread per output pixel computes all COUT channels; the weights sit in
// shared memory as [c * 9 + tap][o] (o padded to a multiple of 4) and are
// read as float4 broadcasts.  Sum order: c, then ky, then kx, then + bias.
// CONV_MASK (data gradient): no bias, result * (mask[b, o, p] > 0).
template <int CIN, int COUT, int MODE, typename TI, typename TW, typename TO>
__global__ void __launch_bounds__(kConvThreads) conv_fwd_kernel(const TI* __restrict__ x, const TW* __restrict__ w,
                                                                const TW* __restrict__ bias, int H, int W, int dil,
                                                                TO* __restrict__ y, const float* __restrict__ mask) {
  constexpr int CO4 = (COUT + 3) / 4 * 4;
  __shared__ __align__(16) float ws[CIN * 9 * CO4];
  __shared__ float bs[CO4];
  for (int idx = threadIdx.x; idx < CIN * 9 * CO4; idx += blockDim.x) {
    const int ct = idx / CO4, o = idx - ct * CO4;
    ws[idx] = o < COUT ? to_f(w[o * CIN * 9 + ct]) : 0.0f;
  }
  for (int o = threadIdx.x; o < CO4; o += blockDim.x) bs[o] = (MODE != CONV_MASK && o < COUT) ? to_f(bias[o]) : 0.0f;
  __syncthreads();
  const int HW = H * W;
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= HW) return;
  const int b = blockIdx.y;
  const int i = p / W, j = p - (p / W) * W;
  float acc[CO4];
#pragma unroll
  for (int o = 0; o < CO4; ++o) acc[o] = 0.0f;
  const TI* xb = x + static_cast<int64_t>(b) * CIN * HW;
  for (int c = 0; c < CIN; ++c) {
    const TI* xc = xb + static_cast<int64_t>(c) * HW;
#pragma unroll
    for (int ky = 0; ky < 3; ++ky) {
      const int ii = i + dil * (ky - 1);
      const bool rok = ii >= 0 && ii < H;
#pragma unroll
      for (int kx = 0; kx < 3; ++kx) {
        const int jj = j + dil * (kx - 1);
        const float v = (rok && jj >= 0 && jj < W) ? to_f(xc[ii * W + jj]) : 0.0f;
        const float4* wr = reinterpret_cast<const float4*>(ws + (c * 9 + ky * 3 + kx) * CO4);
#pragma unroll
        for (int q = 0; q < CO4 / 4; ++q) {
          const float4 wv = wr[q];
          acc[4 * q] = fmaf(wv.x, v, acc[4 * q]);
          acc[4 * q + 1] = fmaf(wv.y, v, acc[4 * q + 1]);
          acc[4 * q + 2] = fmaf(wv.z, v, acc[4 * q + 2]);
          acc[4 * q + 3] = fmaf(wv.w, v, acc[4 * q + 3]);
        }
      }
    }
  }
  const int64_t ob = static_cast<int64_t>(b) * COUT * HW + p;
#pragma unroll
  for (int o = 0; o < COUT; ++o) {
    float r = acc[o];
    if (MODE == CONV_MASK) {
      r = mask[ob + static_cast<int64_t>(o) * HW] > 0.0f ? r : 0.0f;
    } else {
      r += bs[o];
      if (MODE == CONV_RELU) r = fmaxf(r, 0.0f);
    }
    y[ob + static_cast<int64_t>(o) * HW] = from_f<TO>(r);
  }
}

// Two FP32 multiply-adds in one instruction, each rounded as fmaf.
__device__ __forceinline__ void fma2(unsigned long long& acc, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long dup2(float v) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

// The 32 -> 32 layers' convolution (forward and data gradient), as
// conv_fwd_kernel sums it, bit for bit.  The FP32 pipe bounds it: 9,216
// multiply-adds per pixel.  A 16-byte broadcast of shared memory holds its
// pipe for 2 cycles and conv_fwd_kernel needs 8 per input value, which is
// twice the time of the 32 multiply-adds; here a thread takes four pixels, so
// each weight read serves four, and the multiply-adds go two output channels
// to an instruction (the same rate, half the issue slots).  The four pixels
// are d rows apart in one column, so they share input rows: 18 values per
// input channel instead of 36, the next channel's loaded while this one's
// are used.
// Persistent blocks stage the weights once.  Measured (16 images of 256^2):
// 440 - 460 us a layer against 700.
constexpr int kC32Threads = 128;
constexpr int kC32Ppt = 4;  // pixels per thread: rows y, y + d, y + 2 d, y + 3 d of one column
// Columns per tile, and the (row class, four rows) units of a column.
__host__ __device__ constexpr int c32_width(int W) { return W > 64 ? 128 : W > 32 ? 64 : 32; }
__host__ __device__ constexpr int c32_units(int H, int dil) {
  return dil * (((H + dil - 1) / dil + kC32Ppt - 1) / kC32Ppt);
}
constexpr size_t kC32Smem = sizeof(float) * (32 * 9 * 32 + 32);

template <int MODE>
__global__ void __launch_bounds__(kC32Threads, 2) conv32_kernel(const float* __restrict__ x,
                                                                const float* __restrict__ w,
                                                                const float* __restrict__ bias, int B, int H, int W,
                                                                int dil, float* __restrict__ y,
                                                                const float* __restrict__ mask) {
  extern __shared__ __align__(16) float c32[];  // [c * 9 + tap][o], then the bias
  float* const bs = c32 + 32 * 9 * 32;
  const int t = threadIdx.x;
  for (int i = t; i < 32 * 9 * 32; i += kC32Threads) {
    const int o = i / 288, ct = i - o * 288;  // coalesced reads
    c32[ct * 32 + o] = w[i];
  }
  if (t < 32) bs[t] = MODE != CONV_MASK ? bias[t] : 0.0f;
  __syncthreads();
  const int HW = H * W;
  const int tw = c32_width(W), groups = kC32Threads / tw;
  const int tiles_x = (W + tw - 1) / tw;
  const int units = c32_units(H, dil), tiles_u = (units + groups - 1) / groups;
  for (int item = blockIdx.x; item < tiles_x * tiles_u * B; item += gridDim.x) {
    const int b = item / (tiles_x * tiles_u), r0 = item - b * (tiles_x * tiles_u);
    const int ut = r0 / tiles_x, xt = r0 - ut * tiles_x;
    const int unit = ut * groups + t / tw, j = xt * tw + t % tw;
    const int y0 = unit % dil + kC32Ppt * dil * (unit / dil);  // the thread's first row
    const bool mine = unit < units && j < W;
    // which of the 6 x 3 inputs of the thread's pixels lie inside the image
    unsigned int ok = 0u;
#pragma unroll
    for (int e = 0; e < 18; ++e) {
      const int ii = y0 + dil * (e / 3 - 1), jj = j + dil * (e % 3 - 1);
      if (mine && ii >= 0 && ii < H && jj >= 0 && jj < W) ok |= 1u << e;
    }
    const int64_t at0 = static_cast<int64_t>(y0) * W + j;
    const float* xc = x + static_cast<int64_t>(b) * 32 * HW;
    float v[kC32Ppt + 2][3];
    auto load = [&](const float* src, float (&dst)[kC32Ppt + 2][3]) {
#pragma unroll
      for (int e = 0; e < 18; ++e) {
        dst[e / 3][e % 3] = 0.0f;
        if ((ok >> e) & 1u) dst[e / 3][e % 3] = __ldg(src + at0 + dil * ((e / 3 - 1) * W + e % 3 - 1));
      }
    };
    unsigned long long acc[kC32Ppt][16];
#pragma unroll
    for (int u = 0; u < kC32Ppt; ++u)
#pragma unroll
      for (int q = 0; q < 16; ++q) acc[u][q] = 0ull;
    load(xc, v);
#pragma unroll 1
    for (int c = 0; c < 32; ++c) {
      float nv[kC32Ppt + 2][3];
      xc += HW;
      if (c < 31) load(xc, nv);
#pragma unroll
      for (int tap = 0; tap < 9; ++tap) {
        const ulonglong2* wr = reinterpret_cast<const ulonglong2*>(c32 + (c * 9 + tap) * 32);
        unsigned long long a[kC32Ppt];
#pragma unroll
        for (int u = 0; u < kC32Ppt; ++u) a[u] = dup2(v[u + tap / 3][tap % 3]);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const ulonglong2 wv = wr[q];
#pragma unroll
          for (int u = 0; u < kC32Ppt; ++u) {
            fma2(acc[u][2 * q], wv.x, a[u]);
            fma2(acc[u][2 * q + 1], wv.y, a[u]);
          }
        }
      }
#pragma unroll
      for (int e = 0; e < 18; ++e) v[e / 3][e % 3] = nv[e / 3][e % 3];
    }
#pragma unroll
    for (int u = 0; u < kC32Ppt; ++u) {
      if (!mine || y0 + u * dil >= H) continue;
      const int64_t ob = static_cast<int64_t>(b) * 32 * HW + at0 + static_cast<int64_t>(u * dil) * W;
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const float2 r2 = unpack2(acc[u][q]);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int64_t at = ob + static_cast<int64_t>(2 * q + e) * HW;
          float r = e ? r2.y : r2.x;
          if (MODE == CONV_MASK) {
            r = mask[at] > 0.0f ? r : 0.0f;
          } else {
            r += bs[2 * q + e];
            if (MODE == CONV_RELU) r = fmaxf(r, 0.0f);
          }
          y[at] = r;
        }
      }
    }
  }
}

// Asynchronous global -> shared copy of 4 bytes (cp.async, through L1); the
// bytes past src_bytes are zero-filled, and with src_bytes 0 nothing is read
// from src.
__device__ __forceinline__ void cp_async4(void* dst, const void* src, uint32_t src_bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(src_bytes)
               : "memory");
}

// Waits for all of this thread's cp.async copies.
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Weight gradients, dw[o, c, tap] = sum_p dy[o, p] x[c, p + d tap], and bias
// gradients sum_p dy[o, p], as partial sums: each block writes one slot of
// COUT * CIN * 9 + COUT floats in the parameter layout, and
// wgrad_chunk_kernel and wgrad_final_kernel add the slots in a fixed order.
//
// wgrad32_kernel (32 -> 32), bound by the FP32 pipe (9,216 multiply-adds per
// pixel).  A work item is a strip of image rows y0, y0 + d, ... of one image
// and one column segment; a thread owns 8 output channels x 1 input channel
// x 9 taps for half of the segment's columns, so a column costs it 11 reads
// of shared memory (two of 16 bytes) for 72 multiply-adds.  Consecutive rows of a strip share two of their
// three input rows: a ring of four staged rows, filled by asynchronous copies
// one row ahead, reads each input row once.  (One thread per 4 output
// channels, 13 reads for 36 multiply-adds and all three input rows staged
// again for every row took 1,600 us a layer on 16 images of 256^2; this form
// 555, and 740 at dilation 64.)
constexpr int kW32Threads = 256;
constexpr int kW32Dy = 36;  // floats per staged column of dy: 32, padded so that the transposing copies spread over the banks
constexpr int kW32Stride = 32 * 32 * 9 + 32;

// Columns per segment: narrower at wide dilations, whose staged rows are
// mostly halo, so that two blocks fit an SM.
__host__ __device__ constexpr int w32_seg(int dil) { return dil > 32 ? 32 : 64; }
__host__ __device__ constexpr int w32_xs(int dil) { return (w32_seg(dil) + 2 * dil) | 1; }  // floats per staged row of x: odd
__host__ __device__ constexpr size_t w32_smem(int dil) {
  const size_t stage = 4 * 32 * static_cast<size_t>(w32_xs(dil)) + 2 * static_cast<size_t>(w32_seg(dil)) * kW32Dy;
  return sizeof(float) * (stage > kW32Stride ? stage : kW32Stride);
}

// A thread's sums go to the block's slot after this many products, so that
// no sum is longer than before the slots (kWgradRows * W was 1,024).
constexpr int kW32Run = 512;

// Rows per strip: at most 16, and few enough that every resident block gets
// about six items (a strip stages two rows more than it multiplies).
int w32_rows(int B, int H, int W, int dil) {
  const int64_t columns = static_cast<int64_t>(B) * ((W + w32_seg(dil) - 1) / w32_seg(dil));
  const int64_t want = 6 * 2 * static_cast<int64_t>(sm_count());
  const int64_t rows = std::max<int64_t>(1, std::min<int64_t>(16, columns * H / want));
  return static_cast<int>(std::min<int64_t>(rows, (H + dil - 1) / dil));
}
int64_t w32_items(int B, int H, int W, int dil) {
  const int rows = w32_rows(B, H, W, dil), per_class = (H + dil - 1) / dil;
  return static_cast<int64_t>(B) * ((W + w32_seg(dil) - 1) / w32_seg(dil)) * dil * ((per_class + rows - 1) / rows);
}

__global__ void __launch_bounds__(kW32Threads, 2) wgrad32_kernel(const float* __restrict__ x,
                                                                 const float* __restrict__ dy, int B, int H, int W,
                                                                 int dil, int rows, float* __restrict__ partials) {
  extern __shared__ __align__(16) float w32[];
  const int seg = w32_seg(dil), XS = w32_xs(dil);
  float* const dys = w32;                          // [2][seg][kW32Dy]
  float* const xs = w32 + 2 * seg * kW32Dy;        // [4][32][XS], column x0 + j at j + dil
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int co0 = 8 * (lane & 3), ci = (lane >> 2) + 8 * (warp & 3), half = warp >> 2;
  const int warp_u = __shfl_sync(0xffffffffu, warp & 3, 0);  // uniform: 0 sums the bias gradient
  const int HW = H * W;
  const int tiles_x = (W + seg - 1) / seg;
  const int per_class = (H + dil - 1) / dil, chunks = (per_class + rows - 1) / rows;
  const int n_items = B * tiles_x * dil * chunks;
  float acc[9][8], dacc[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    dacc[k] = 0.0f;
#pragma unroll
    for (int tap = 0; tap < 9; ++tap) acc[tap][k] = 0.0f;
  }
  int run = 0;         // products in each of the thread's sums
  bool stored = false;  // the block's slot holds earlier sums
  float* const out = partials + static_cast<int64_t>(blockIdx.x) * kW32Stride;
  for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
    int rest = item;
    const int ch = rest % chunks;
    rest /= chunks;
    const int cls = rest % dil;
    rest /= dil;
    const int xt = rest % tiles_x;
    const int b = rest / tiles_x;
    const int x0 = xt * seg, y0 = cls + ch * rows * dil;
    const int nrow = y0 < H ? min(rows, (H - 1 - y0) / dil + 1) : 0;
    const float* xb = x + static_cast<int64_t>(b) * 32 * HW;
    const float* db = dy + static_cast<int64_t>(b) * 32 * HW;
    const int xw = seg + 2 * dil;
    // input row yy (zeros outside the image) into ring slot q: a warp takes
    // a channel at a time
    auto stage_x = [&](int yy, int q) {
      for (int c = warp; c < 32; c += kW32Threads / 32) {
        float* dst = xs + (q * 32 + c) * XS;
        const float* src = xb + static_cast<int64_t>(c) * HW + static_cast<int64_t>(yy) * W;
        for (int j = lane; j < xw; j += 32) {
          const int xx = x0 - dil + j;
          const bool in = yy >= 0 && yy < H && xx >= 0 && xx < W;
          cp_async4(dst + j, in ? src + xx : x, in ? 4u : 0u);
        }
      }
    };
    // output-gradient row yy, transposed: 8 columns x 4 channels per warp
    // and copy, which read whole sectors and write 32 different banks
    auto stage_dy = [&](int yy, int q) {
      float* dst = dys + q * seg * kW32Dy;
      for (int e = warp; e < seg; e += kW32Threads / 32) {  // seg / 8 column groups x 8 channel groups
        const int j = (e >> 3) * 8 + (lane >> 2), c = (e & 7) * 4 + (lane & 3);
        const bool in = x0 + j < W;
        cp_async4(dst + j * kW32Dy + c, in ? db + static_cast<int64_t>(c) * HW + static_cast<int64_t>(yy) * W + x0 + j : dy,
                  in ? 4u : 0u);
      }
    };
    __syncthreads();  // the previous item's rows (and sums) have been read
    if (nrow > 0) {
      stage_x(y0 - dil, 0);
      stage_x(y0, 1);
      stage_x(y0 + dil, 2);
      stage_dy(y0, 0);
    }
    for (int k = 0; k < nrow; ++k) {
      cp_async_wait_all();
      __syncthreads();
      if (k + 1 < nrow) {  // the slots of input row k - 2 and of dy row k - 1: every warp is past them
        stage_x(y0 + (k + 2) * dil, (k + 3) & 3);
        stage_dy(y0 + (k + 1) * dil, (k + 1) & 1);
      }
      const float* dr = dys + (k & 1) * seg * kW32Dy + co0;
      const float* xr[3];
#pragma unroll
      for (int ky = 0; ky < 3; ++ky) xr[ky] = xs + (((k + ky) & 3) * 32 + ci) * XS;
      const int j0 = half * (seg / 2);
#pragma unroll 2
      for (int j = j0; j < j0 + seg / 2; ++j) {
        const float4 d0 = *reinterpret_cast<const float4*>(dr + j * kW32Dy);
        const float4 d1 = *reinterpret_cast<const float4*>(dr + j * kW32Dy + 4);
        const float d[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
#pragma unroll
        for (int ky = 0; ky < 3; ++ky)
#pragma unroll
          for (int kx = 0; kx < 3; ++kx) {
            const float v = xr[ky][j + dil * kx];
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[ky * 3 + kx][k] = fmaf(d[k], v, acc[ky * 3 + kx][k]);
          }
        if (warp_u == 0) {
#pragma unroll
          for (int k = 0; k < 8; ++k) dacc[k] += d[k];
        }
      }
    }
    run += nrow * (seg / 2);
    if (run < kW32Run && item + static_cast<int>(gridDim.x) < n_items) continue;
    // the halves' sums meet in the staging area, then go to the block's slot
    __syncthreads();
#pragma unroll
    for (int h = 1; h >= 0; --h) {
      if (half == h) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
#pragma unroll
          for (int tap = 0; tap < 9; ++tap) {
            const int e = ((co0 + k) * 32 + ci) * 9 + tap;
            w32[e] = h ? acc[tap][k] : w32[e] + acc[tap][k];
            acc[tap][k] = 0.0f;
          }
          if (ci == 0) {
            const int e = 32 * 32 * 9 + co0 + k;
            w32[e] = h ? dacc[k] : w32[e] + dacc[k];
          }
          dacc[k] = 0.0f;
        }
      }
      __syncthreads();
    }
    for (int e = t; e < kW32Stride; e += kW32Threads) out[e] = stored ? out[e] + w32[e] : w32[e];
    stored = true;
    run = 0;
  }
}

// wgrad_thin_kernel: the layers with a thin side (2 -> 32 and 32 -> 1), bound
// by reading the 32-channel tensor (dy, or x) once.  A lane takes a column, a
// warp 4 of the 32 channels.  For the 2 -> 32 layer the wide tensor is dy and
// the thin one x, read at p + d tap; for the 32 -> 1 layer the wide one is x,
// and x[q] meets dy at q - d tap.  A block takes kThinRows rows y0, y0 + d,
// ..., so that a row adds 3 thin values per channel to the 6 kept from the
// rows before; the next row's values are loaded while this one's are used.
// At the end the lanes are added by a butterfly.  (16 images of 256^2:
// 116 and 83 us, against 217 and 337 with both tensors staged in
// shared memory, one thread per channel pair; reading all 9 thin values of
// every pixel took 181 and 143.)
constexpr int kThinRows = 8;

// Blocks per image: (row class, kThinRows rows) units.
__host__ __device__ constexpr int thin_units(int H, int dil) {
  return dil * (((H + dil - 1) / dil + kThinRows - 1) / kThinRows);
}

template <int CIN, int COUT>
__global__ void __launch_bounds__(256, 2) wgrad_thin_kernel(const float* __restrict__ x,
                                                            const float* __restrict__ dy, int H, int W, int dil,
                                                            float* __restrict__ partials) {
  static_assert((CIN == 32) != (COUT == 32), "one wide side");
  constexpr bool kWideOut = COUT == 32;
  constexpr int T = kWideOut ? CIN : COUT;  // thin channels
  constexpr int STRIDE = COUT * CIN * 9 + COUT;
  const int lane = threadIdx.x & 31;
  const int warp = warp_uniform(threadIdx.x >> 5);
  const int b = blockIdx.y, unit = blockIdx.x;
  const int y0 = unit % dil + kThinRows * dil * (unit / dil);
  const int nrow = y0 < H ? min(kThinRows, (H - 1 - y0) / dil + 1) : 0;
  const int HW = H * W;
  const float* wide = (kWideOut ? dy : x) + (static_cast<int64_t>(b) * 32 + 4 * warp) * HW;
  const float* thin = (kWideOut ? x : dy) + static_cast<int64_t>(b) * T * HW;
  float acc[4][T][9], sum[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    sum[k] = 0.0f;
#pragma unroll
    for (int c = 0; c < T; ++c)
#pragma unroll
      for (int tap = 0; tap < 9; ++tap) acc[k][c][tap] = 0.0f;
  }
  for (int x0 = 0; x0 < W; x0 += 32) {
    const int xx = x0 + lane;
    auto load_thin = [&](int m, float (&dst)[T][3]) {  // row m of the unit, columns xx - d, xx, xx + d
      const int ii = y0 + m * dil;
#pragma unroll
      for (int c = 0; c < T; ++c)
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          const int jj = xx + dil * (e - 1);
          dst[c][e] = 0.0f;
          if (ii >= 0 && ii < H && jj >= 0 && jj < W)
            dst[c][e] = __ldg(thin + static_cast<int64_t>(c) * HW + static_cast<int64_t>(ii) * W + jj);
        }
    };
    auto load_wide = [&](int m, float (&dst)[4]) {
      const int ii = y0 + m * dil;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        dst[k] = 0.0f;
        if (m < nrow && xx < W)
          dst[k] = __ldg(wide + static_cast<int64_t>(k) * HW + static_cast<int64_t>(ii) * W + xx);
      }
    };
    float v[3][T][3], nv[T][3], a[4], na[4];  // v: thin rows m - 1, m, m + 1
    load_thin(-1, v[1]);
    load_thin(0, v[2]);
    load_thin(1, nv);
    load_wide(0, na);
#pragma unroll 1
    for (int m = 0; m < nrow; ++m) {
#pragma unroll
      for (int c = 0; c < T; ++c)
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          v[0][c][e] = v[1][c][e];
          v[1][c][e] = v[2][c][e];
          v[2][c][e] = nv[c][e];
        }
#pragma unroll
      for (int k = 0; k < 4; ++k) a[k] = na[k];
      load_thin(m + 2, nv);
      load_wide(m + 1, na);
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int c = 0; c < T; ++c)
#pragma unroll
          for (int tap = 0; tap < 9; ++tap) {
            const int e = kWideOut ? tap : 8 - tap;
            acc[k][c][tap] = fmaf(a[k], v[e / 3][c][e % 3], acc[k][c][tap]);
          }
      if (kWideOut) {
#pragma unroll
        for (int k = 0; k < 4; ++k) sum[k] += a[k];
      } else if (xx < W) {
        sum[0] += v[1][0][1];  // dy itself
      }
    }
  }
  float* out = partials + (static_cast<int64_t>(blockIdx.y) * gridDim.x + blockIdx.x) * STRIDE;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int w = 4 * warp + k;  // the wide channel
#pragma unroll
    for (int c = 0; c < T; ++c)
#pragma unroll
      for (int tap = 0; tap < 9; ++tap) {
        float r[1] = {acc[k][c][tap]};
        warp_sum<1, float>(r);
        if (lane == 0) out[(kWideOut ? w * CIN + c : w) * 9 + tap] = r[0];
      }
    if (kWideOut || (warp == 0 && k == 0)) {
      float r[1] = {sum[k]};
      warp_sum<1, float>(r);
      if (lane == 0) out[COUT * CIN * 9 + (kWideOut ? w : 0)] = r[0];
    }
  }
}

// Slot sums in two fixed-order passes: chunk[ch][e] = sum of the slots
// [ch * per, (ch + 1) * per) in order; grads[e] = sum of the chunks in order.
constexpr int kReduceChunks = 32;

__global__ void wgrad_chunk_kernel(const float* __restrict__ partials, int64_t nslots, int stride, int64_t per,
                                   float* __restrict__ chunk) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const int ch = blockIdx.y;
  if (e >= stride) return;
  float sum = 0.0f;
  const int64_t s1 = min(nslots, (ch + 1) * per);
  for (int64_t sl = ch * per; sl < s1; ++sl) sum += partials[sl * stride + e];
  chunk[static_cast<int64_t>(ch) * stride + e] = sum;
}

__global__ void wgrad_final_kernel(const float* __restrict__ chunk, int nch, int stride, float* __restrict__ grads) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= stride) return;
  float sum = 0.0f;
  for (int ch = 0; ch < nch; ++ch) sum += chunk[static_cast<int64_t>(ch) * stride + e];
  grads[e] = sum;
}

// Flipped, transposed weights of one layer for its data gradient:
// wf[c, o, ky, kx] = w[o, c, 2 - ky, 2 - kx].
__global__ void flip_kernel(const float* __restrict__ w, int cin, int cout, float* __restrict__ wf) {
  const int n = cin * cout * 9;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += gridDim.x * blockDim.x) {
    const int tp = idx % 9, oc = idx / 9;
    const int c = oc / cout, o = oc - c * cout;  // idx indexes wf as [c][o][tap]
    wf[idx] = w[(o * cin + c) * 9 + (8 - tp)];
  }
}

// Mean squared error: dout = 2 (out - t) / N; per-block partial sums of
// (out - t)^2 (fixed order), the last block adds them in order into *loss.
__global__ void __launch_bounds__(256) mse_kernel(const float* __restrict__ out, const float* __restrict__ tgt,
                                                  int64_t n, float* __restrict__ dout, float* partials,
                                                  unsigned int* counter, float* loss) {
  __shared__ float scratch[kRedScratch];
  float sq = 0.0f;
  const float sc = 2.0f / static_cast<float>(n);
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const float d = out[i] - tgt[i];
    dout[i] = sc * d;
    sq = fmaf(d, d, sq);
  }
  float v[1] = {sq}, tot[1];
  if (grid_sum<1, float>(v, partials, counter, scratch, tot) && threadIdx.x == 0) *loss = tot[0] / static_cast<float>(n);
}

// Energy-norm loss L = (1 / N) sum_p e_p (A e)_p, e = out - target, with A
// the 5-point variable-coefficient operator of the sample (cell coefficients
// exp(g), g = input channel 0; faces the harmonic mean of the two cells, a
// boundary face the cell's own coefficient).  dout = 2 A e / N (A is
// symmetric).  Per-block partial sums of e.(A e), reduced like mse_kernel.
__device__ __forceinline__ float face(float ca, float cb) { return 2.0f * ca * cb / (ca + cb); }

__global__ void __launch_bounds__(256) energy_kernel(const float* __restrict__ out, const float* __restrict__ tgt,
                                                     const float* __restrict__ feat, int B, int H, int W,
                                                     float* __restrict__ dout, float* partials,
                                                     unsigned int* counter, float* loss) {
  __shared__ float scratch[kRedScratch];
  const int64_t HW = static_cast<int64_t>(H) * W, n = B * HW;
  const float sc = 2.0f / static_cast<float>(n);
  float acc = 0.0f;
  for (int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; q < n;
       q += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t b = q / HW, p = q - b * HW;
    const int i = static_cast<int>(p / W), j = static_cast<int>(p - (p / W) * W);
    const float* g = feat + b * 2 * HW;  // channel 0 of sample b
    const float* e0 = out + b * HW;
    const float* t0 = tgt + b * HW;
    const float c = expf(g[p]);
    const float e = e0[p] - t0[p];
    float diag = 0.0f, off = 0.0f;
    const int di[4] = {-1, 0, 0, 1}, dj[4] = {0, -1, 1, 0};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int ii = i + di[k], jj = j + dj[k];
      if (ii >= 0 && ii < H && jj >= 0 && jj < W) {
        const int64_t pn = static_cast<int64_t>(ii) * W + jj;
        const float f = face(c, expf(g[pn]));
        diag += f;
        off = fmaf(f, e0[pn] - t0[pn], off);
      } else {
        diag += c;
      }
    }
    const float ae = fmaf(diag, e, -off);
    dout[q] = sc * ae;
    acc = fmaf(e, ae, acc);
  }
  float v[1] = {acc}, tot[1];
  if (grid_sum<1, float>(v, partials, counter, scratch, tot) && threadIdx.x == 0) *loss = tot[0] / static_cast<float>(n);
}

// Adam (Kingma and Ba, 2015), step t >= 1.
__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, int64_t n, float lr, float b1, float b2, float eps, float c1,
                            float c2) {
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

__global__ void to_bf16_kernel(const float* __restrict__ in, __nv_bfloat16* __restrict__ out, int64_t n) {
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    out[i] = __float2bfloat16_rn(in[i]);
}

// rms of b (fixed-order reduction): the last block stores it.
__global__ void __launch_bounds__(256) rms_kernel(const double* __restrict__ b, int64_t n, double* partials,
                                                  unsigned int* counter, double* rms) {
  __shared__ double scratch[kRedScratch];
  double s = 0.0;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    s = fma(b[i], b[i], s);
  double v[1] = {s}, tot[1];
  if (grid_sum<1, double>(v, partials, counter, scratch, tot) && threadIdx.x == 0) {
    const double r = sqrt(tot[0] / static_cast<double>(n));
    *rms = r > 0.0 ? r : 1.0;
  }
}

// Network input [g, b / rms(b)] in FP32 and, when x is given, the target
// x / (rms(b) * out_scale).
__global__ void features_kernel(const double* __restrict__ g, const double* __restrict__ b,
                                const double* __restrict__ x, const double* __restrict__ rms, double out_scale,
                                int64_t n, float* __restrict__ feat, float* __restrict__ tgt) {
  const double inv = 1.0 / *rms;
  const double tinv = 1.0 / (*rms * out_scale);
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    feat[i] = static_cast<float>(g[i]);
    feat[n + i] = static_cast<float>(b[i] * inv);
    if (x) tgt[i] = static_cast<float>(x[i] * tinv);
  }
}

// x0 = y * rms(b) * out_scale in FP64.
__global__ void scale_out_kernel(const float* __restrict__ y, const double* __restrict__ rms, double out_scale,
                                 int64_t n, double* __restrict__ x0) {
  const double sc = *rms * out_scale;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    x0[i] = static_cast<double>(y[i]) * sc;
}

// Galerkin scaling of the prediction: (x0.b, x0.A x0) -> x0 *= alpha with
// alpha = (x0.b) / (x0.A x0) (the multiple of x0 closest to the solution in
// the A-norm, so never farther than x = 0 for SPD A).  Sums first (last
// block stores alpha), the scaling in a second launch.
__global__ void __launch_bounds__(256) galerkin_sums_kernel(const double* __restrict__ x0,
                                                            const double* __restrict__ b,
                                                            const double* __restrict__ ax0, int64_t n,
                                                            double* partials, unsigned int* counter,
                                                            double* alpha) {
  __shared__ double scratch[kRedScratch];
  double s0 = 0.0, s1 = 0.0;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    s0 = fma(x0[i], b[i], s0);
    s1 = fma(x0[i], ax0[i], s1);
  }
  double v[2] = {s0, s1}, tot[2];
  if (grid_sum<2, double>(v, partials, counter, scratch, tot) && threadIdx.x == 0)
    *alpha = (tot[1] > 0.0 && isfinite(tot[0] / tot[1])) ? tot[0] / tot[1] : 0.0;
}

__global__ void scale_kernel(double* __restrict__ x0, const double* __restrict__ alpha, int64_t n) {
  const double a = *alpha;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    x0[i] *= a;
}

// ---------------------------------------------------------------------------
// BF16 inference on the tensor cores.  Activations between the layers are
// BF16 in four planes of 8 channels per image row (tc_act).  The 32 -> 32
// layers run as an implicit GEMM on tcgen05: a tile is 128 consecutive
// pixels of one image row (M = 128), N = 32 output channels, K = 9 taps x 32
// input channels, issued as 18 MMAs of K = 16 (BF16 operands, FP32
// accumulator in tensor memory).  A block works down a strip of rows with a
// ring of staged input rows, each from x0 - d to x0 + 127 + d (zeros outside
// the image): bulk copies fill it, and the three taps kx of a row are the
// same staged window read from slot kx d on, so the MMA's A operand is the
// window with a start address shifted by kx d rows.  Operands are K-major
// without swizzling: a core matrix is 8 rows x 16 bytes (8 channels); rows of
// a matrix are 16 bytes apart and its 8-channel chunks LBO bytes apart.  The
// first layer (2 input channels, K = 18 padded to 32) runs on the tensor
// cores too, from the FP32 input (conv_first_tc_kernel); the last (1 output
// channel) is folded into the layer before it as nine FP32 planes of
// per-tap products, which conv_last_sum_kernel adds up.
// ---------------------------------------------------------------------------

constexpr int kTcThreads = 192;                 // 4 epilogue warps (one TMEM lane quarter each), an MMA warp, a copy warp
constexpr int kTcFirstThreads = 128;
constexpr int kTcTile = 128;                    // pixels per tile (MMA M)
constexpr int kTcStripMax = 16;                 // output rows per work item (a strip), at most
constexpr int kTcMaxDil = 64;                   // largest dilation (gk_wsnet_create checks it)
constexpr uint32_t kTcChunkB = 32 * 16;         // bytes between 8-channel chunks of a tap's weights
constexpr int kTcPacked = 9 * 4 * 32 * 8;       // packed BF16 weights of one 32 -> 32 layer
constexpr int kTcMidLayers = kLayers - 2;

// Activations between layers: per image row, four planes (8-channel chunks)
// of W pixels x 16 bytes, so that a window of a row is four contiguous runs
// for the bulk copies and a warp's epilogue stores are contiguous.
__device__ __forceinline__ int64_t tc_act(int64_t row, int chunk, int W, int px) {  // in 16-byte units
  return (row * 4 + chunk) * W + px;
}

// Shared memory of a block: this header, then the ring of kTcRing staged
// input rows, [row slot][chunk][pixel slot][8 channels], 128 + 2 dil pixel
// slots per chunk.
constexpr int kTcRing = 5;
struct TcSmem {
  __nv_bfloat16 b[kTcPacked];           // [tap][chunk][out][8 channels]
  float bias[32];
  uint64_t full[kTcRing];               // a slot's row has landed
  uint64_t free_[kTcRing];              // the last MMAs that read a slot have completed
  uint64_t done[2];                     // an accumulator's MMAs have completed
  uint64_t empty[2];                    // an accumulator has been read by the four epilogue warps
  uint32_t tmem;
  int zero_x0[kTcRing];                 // the column range a slot's zeros outside the image were written for
};
constexpr size_t kTcAOffset = (sizeof(TcSmem) + 127) / 128 * 128;
__host__ __device__ constexpr size_t tc_ring_bytes(int dil) { return kTcRing * 4 * static_cast<size_t>(kTcTile + 2 * dil) * 16; }
constexpr size_t tc_smem_bytes(int dil) { return kTcAOffset + tc_ring_bytes(dil); }
// ... and the folded last layer's weights after the ring (conv_tc_kernel<true>)
constexpr size_t kTcLastBytes = 9 * 32 * sizeof(float);

// Instruction descriptor of tcgen05.mma kind::f16: FP32 accumulator (bits
// 4-5 = 1), A and B BF16 (bits 7-9, 10-12 = 1), both K-major (bits 15, 16 =
// 0), N / 8 in bits 17-22, M / 16 in bits 24-28.
constexpr uint32_t kTcIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((32u >> 3) << 17) | ((128u >> 4) << 24);

// Shared-memory matrix descriptor: start address / 16 (bits 0-13), leading
// (K-direction) byte offset / 16 (bits 16-29), stride (M/N-direction) byte
// offset / 16 (bits 32-45), the fixed version bits 46-48 = 0b001, no
// swizzle (bits 61-63 = 0).
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return static_cast<uint64_t>((addr & 0x3FFFFu) >> 4) | (static_cast<uint64_t>(lbo >> 4) << 16) |
         (static_cast<uint64_t>(sbo >> 4) << 32) | (1ull << 46);
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tc_mma(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(ad), "l"(bd), "r"(kTcIdesc), "r"(accumulate)
      : "memory");
}

// The same with the descriptors' low words (address and leading offset; the
// high word is the same for every operand here), so that a step between the
// operands of one row is one 32-bit addition.
__device__ __forceinline__ uint32_t tc_desc_lo(uint32_t addr, uint32_t lbo) {
  return ((addr & 0x3FFFFu) >> 4) | ((lbo >> 4) << 16);
}
__device__ __forceinline__ void tc_mma_lo(uint32_t tmem, uint32_t a, uint32_t b, uint32_t accumulate) {
  constexpr uint32_t kHi = (128u >> 4) | (1u << 14);  // stride 128 bytes, version bits
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 da, db;\n setp.ne.b32 p, %5, 0;\n mov.b64 da, {%1, %3};\n"
      " mov.b64 db, {%2, %3};\n tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n}\n" ::"r"(tmem),
      "r"(a), "r"(b), "r"(kHi), "r"(kTcIdesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

// 32 consecutive FP32 columns of the warp's 32 TMEM lanes (lane = pixel).
__device__ __forceinline__ void tc_load32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  const uint32_t l = __bfloat16_as_ushort(__float2bfloat16_rn(lo));
  const uint32_t h = __bfloat16_as_ushort(__float2bfloat16_rn(hi));
  return l | (h << 16);
}

// A pixel's 32 channels: bias, ReLU, BF16, to the four planes of its row.
__device__ __forceinline__ void tc_store_row(const float (&v)[32], const float* bias, uint4* dst, int W) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    float o[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) o[e] = fmaxf(v[c * 8 + e] + bias[c * 8 + e], 0.0f);
    dst[static_cast<int64_t>(c) * W] =
        make_uint4(pack_bf16x2(o[0], o[1]), pack_bf16x2(o[2], o[3]), pack_bf16x2(o[4], o[5]), pack_bf16x2(o[6], o[7]));
  }
}

// One 32 -> 32 layer with ReLU: x, y BF16 in the layout of tc_act; wp the
// packed weights [tap][chunk][out][8]; bias BF16.  Persistent over strips;
// err gets kErrTimeout if a wait gives up.
//
// A work item is a strip: the output rows y0, y0 + dil, ..., of one image and
// one 128-pixel column range (at most `strip` of them).  Output row y_k reads
// input rows y_k - dil, y_k and y_k + dil, so consecutive rows of a strip
// share two of their three input rows.  What bounds a row is the chain of its
// steps (copy, MMAs, read-back, stores), so they run side by side: a copy
// warp fills a ring of staged rows (four bulk copies each), one thread of
// another warp issues a row's 18 MMAs into one of two accumulators, and the
// four epilogue warps read the other back and store.  The staged rows of all
// strips form one sequence (row s in slot s % kTcRing), so the copies run
// ahead across strips.
// (Copies by the block's threads, 16 bytes per instruction and 64 apart, and
// one accumulator: 186, 186 and 201 us a layer on 64 images of 256^2 at
// dilations 4, 16 and 64, 231 for the last; this form 109, 107, 143 and 158;
// the layers' compulsory bytes take 80 and 63.  What is left is shared memory:
// the MMAs read each staged row nine times, about 580 cycles a row.  Rings of
// 4 and 6 rows: 719 and 751 us a batch against 676.)
//
// LAST: this is the network's last 32 -> 32 layer and the 32 -> 1 layer
// after it is folded into its epilogue: since that layer has one output
// channel, its output is y(p) = b + sum over taps of t_tap(p + offset_tap)
// with t_tap(q) = sum over channels of w[tap][c] h(q)[c]; the epilogue
// rounds h to BF16 (the value the unfused form stores) and writes the nine
// t_tap(q) as FP32 planes T[tap][pixel] to y, and conv_last_sum_kernel adds
// them up.  The 64-byte activation is then never written nor read back.
template <bool LAST>
__global__ void __launch_bounds__(kTcThreads) conv_tc_kernel(const __nv_bfloat16* __restrict__ x,
                                                             const __nv_bfloat16* __restrict__ wp,
                                                             const __nv_bfloat16* __restrict__ bias, int B, int H,
                                                             int W, int dil, int strip,
                                                             const __nv_bfloat16* __restrict__ w_last,
                                                             __nv_bfloat16* __restrict__ y, int* err) {
  extern __shared__ __align__(1024) unsigned char tc_raw[];
  TcSmem& S = *reinterpret_cast<TcSmem*>(tc_raw);
  const int t = threadIdx.x, lane = t & 31;
  const int warp = warp_uniform(t >> 5);
  for (int i = t; i < kTcPacked / 8; i += kTcThreads)
    reinterpret_cast<uint4*>(S.b)[i] = __ldg(reinterpret_cast<const uint4*>(wp) + i);
  if (t < 32) S.bias[t] = __bfloat162float(bias[t]);
  // LAST: the 32 -> 1 layer's weights [tap][channel], after the ring
  float* const w_last_s = reinterpret_cast<float*>(tc_raw + kTcAOffset + tc_ring_bytes(dil));
  if (LAST)
    for (int i = t; i < 9 * 32; i += kTcThreads) w_last_s[i] = __bfloat162float(w_last[(i & 31) * 9 + (i >> 5)]);
  if (t == 0) {
    for (int q = 0; q < kTcRing; ++q) {
      mbar_init(&S.full[q], 1);
      mbar_init(&S.free_[q], 1);
      S.zero_x0[q] = -1;
    }
    for (int q = 0; q < 2; ++q) {
      mbar_init(&S.done[q], 1);
      mbar_init(&S.empty[q], 4);
    }
    fence_mbar_init();
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 64;" ::"r"(smem_u32(&S.tmem))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the weights -> tensor core reads
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = S.tmem;
  const int nslot = kTcTile + 2 * dil;              // pixel slots of a staged row
  const uint32_t chunk_a = static_cast<uint32_t>(nslot) * 16;  // bytes between its 8-channel chunks
  uint4* const ring = reinterpret_cast<uint4*>(tc_raw + kTcAOffset);
  const int tiles_x = (W + kTcTile - 1) / kTcTile;
  const int per_class = (H + dil - 1) / dil;             // rows of the fullest residue class
  const int chunks = (per_class + strip - 1) / strip;
  const int n_strips = B * tiles_x * dil * chunks;
  // item -> its image's first row, first column, first output row, rows
  auto item_of = [&](int item, int64_t& row0, int& x0, int& y0) {
    int rest = item;
    const int ch = rest % chunks;
    rest /= chunks;
    const int cls = rest % dil;
    rest /= dil;
    x0 = (rest % tiles_x) * kTcTile;
    row0 = static_cast<int64_t>(rest / tiles_x) * H;
    y0 = cls + ch * strip * dil;
    return y0 < H ? min(strip, (H - 1 - y0) / dil + 1) : 0;
  };
  uint32_t g = 0;  // output rows so far: row g uses accumulator g % 2
  if (warp == 5) {
    // ---- copies: input rows y0 - dil, y0, ..., y0 + nrow dil of every strip
    uint32_t st = 0;  // staged rows so far: row st in slot st % kTcRing
    bool ok = true;
    for (int item = blockIdx.x; item < n_strips && ok; item += gridDim.x) {
      int64_t row0;
      int x0, y0;
      const int nrow = item_of(item, row0, x0, y0);
      const int lo = max(0, dil - x0), hi = min(nslot, W - x0 + dil);  // slots inside the image
      const uint32_t bytes = static_cast<uint32_t>(hi - lo) * 16;
      for (int i = 0; nrow > 0 && i < nrow + 2; ++i, ++st) {
        const uint32_t q = st % kTcRing;
        if (st >= kTcRing) {
          ok = __all_sync(0xffffffffu, mbar_wait(&S.free_[q], (st / kTcRing - 1) & 1, err));
          if (!ok) break;
        }
        uint4* const dst = ring + q * 4 * nslot;
        if (S.zero_x0[q] != x0) {  // columns outside the image are zero, whichever row the slot holds
          for (int c = 0; c < 4; ++c) {
            for (int sl = lane; sl < lo; sl += 32) dst[c * nslot + sl] = make_uint4(0u, 0u, 0u, 0u);
            for (int sl = hi + lane; sl < nslot; sl += 32) dst[c * nslot + sl] = make_uint4(0u, 0u, 0u, 0u);
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // before the MMAs' reads
          __syncwarp();
          if (lane == 0) S.zero_x0[q] = x0;
          __syncwarp();
        }
        if (lane == 0) {
          const int yy = y0 + (i - 1) * dil;
          if (yy >= 0 && yy < H) {
            mbar_arrive_expect_tx(&S.full[q], 4 * bytes);
            const uint4* src = reinterpret_cast<const uint4*>(x) + tc_act(row0 + yy, 0, W, x0 - dil + lo);
#pragma unroll
            for (int c = 0; c < 4; ++c)
              bulk_g2s(dst + c * nslot + lo, src + static_cast<int64_t>(c) * W, bytes, &S.full[q]);
          } else {
            mbar_arrive(&S.full[q]);  // a row outside the image is left out of the sums
          }
        }
      }
    }
    // no copy of this block is in flight at exit (they have all been waited
    // for unless a wait gave up: bounded)
    if (lane == 0)
      for (uint32_t u = st > kTcRing ? st - kTcRing : 0; u < st; ++u)
        mbar_wait(&S.full[u % kTcRing], (u / kTcRing) & 1, err);
  } else if (warp == 4) {
    // ---- MMAs, issued by one thread
    if (lane == 0) {
      const uint32_t a0 = tc_desc_lo(smem_u32(ring), chunk_a), b0 = tc_desc_lo(smem_u32(S.b), kTcChunkB);
      const uint32_t step_h = 2 * nslot, step_slot = 4 * nslot;  // in 16-byte units
      uint32_t st = 0;  // the strip's first staged row
      bool ok = true;
      for (int item = blockIdx.x; item < n_strips && ok; item += gridDim.x) {
        int64_t row0;
        int x0, y0;
        const int nrow = item_of(item, row0, x0, y0);
        if (nrow == 0) continue;
        auto landed = [&](uint32_t u) { return mbar_wait(&S.full[u % kTcRing], (u / kTcRing) & 1, err); };
        ok = landed(st) && landed(st + 1);
        for (int k = 0; k < nrow && ok; ++k) {
          if (!(ok = landed(st + k + 2))) break;
          if (g >= 2 && !(ok = mbar_wait(&S.empty[g & 1], ((g >> 1) - 1) & 1, err))) break;
          tc_fence_after();
          const uint32_t d = tmem + 32 * (g & 1);
          uint32_t acc = 0;
#pragma unroll
          for (int ky = 0; ky < 3; ++ky) {
            const int yy = y0 + (k - 1 + ky) * dil;
            if (yy < 0 || yy >= H) continue;
            const uint32_t a_row = a0 + ((st + k + ky) % kTcRing) * step_slot;
#pragma unroll
            for (int kx = 0; kx < 3; ++kx)
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                tc_mma_lo(d, a_row + kx * dil + h * step_h, b0 + ((ky * 3 + kx) * 4 + 2 * h) * (kTcChunkB / 16), acc);
                acc = 1;
              }
          }
          tc_commit(&S.done[g & 1]);
          tc_commit(&S.free_[(st + k) % kTcRing]);
          if (k == nrow - 1) {
            tc_commit(&S.free_[(st + k + 1) % kTcRing]);
            tc_commit(&S.free_[(st + k + 2) % kTcRing]);
          }
          ++g;
        }
        st += nrow + 2;
      }
      // the last MMAs have completed before the tensor memory is released
      if (g > 0) mbar_wait(&S.done[(g - 1) & 1], ((g - 1) >> 1) & 1, err);
    }
  } else {
    // ---- epilogue: warp w reads TMEM lanes 32 w .. 32 w + 31 (lane = pixel) ----
    const int64_t n_pix = static_cast<int64_t>(B) * H * W;  // LAST: the T planes' stride
    bool ok = true;
    for (int item = blockIdx.x; item < n_strips && ok; item += gridDim.x) {
      int64_t row0;
      int x0, y0;
      const int nrow = item_of(item, row0, x0, y0);
      const int px = x0 + warp * 32 + lane;
      // reads row g's accumulator into v and gives it back
      auto read = [&](float (&v)[32]) {
        if (!__all_sync(0xffffffffu, mbar_wait(&S.done[g & 1], (g >> 1) & 1, err))) return false;
        tc_fence_after();
        tc_load32(tmem + (static_cast<uint32_t>(warp * 32) << 16) + 32 * (g & 1), v);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.empty[g & 1]);
        ++g;
        return true;
      };
      if (LAST) {
        // two rows at a time: a read of the tap weights (72 of 16 bytes) serves
        // two pixels, since the shared memory is what the MMAs' operands, the
        // copies and these reads compete for
        auto relu = [&](float (&v)[32]) {
#pragma unroll
          for (int c = 0; c < 32; ++c) v[c] = __bfloat162float(__float2bfloat16_rn(fmaxf(v[c] + S.bias[c], 0.0f)));
        };
        for (int k = 0; k < nrow && ok; k += 2) {
          float h0[32], h1[32];
          const bool two = k + 1 < nrow;
          if (!(ok = read(h0))) break;
          relu(h0);
          if (two) {
            if (!(ok = read(h1))) break;
            relu(h1);
          } else {
#pragma unroll
            for (int c = 0; c < 32; ++c) h1[c] = 0.0f;
          }
          float* T = reinterpret_cast<float*>(y) + (row0 + y0 + k * dil) * W + px;
          const int64_t down = static_cast<int64_t>(dil) * W;
#pragma unroll
          for (int tap = 0; tap < 9; ++tap) {
            float t0 = 0.0f, t1 = 0.0f;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              const float4 w = reinterpret_cast<const float4*>(w_last_s)[tap * 8 + c];
              t0 = fmaf(w.x, h0[4 * c], t0);
              t1 = fmaf(w.x, h1[4 * c], t1);
              t0 = fmaf(w.y, h0[4 * c + 1], t0);
              t1 = fmaf(w.y, h1[4 * c + 1], t1);
              t0 = fmaf(w.z, h0[4 * c + 2], t0);
              t1 = fmaf(w.z, h1[4 * c + 2], t1);
              t0 = fmaf(w.w, h0[4 * c + 3], t0);
              t1 = fmaf(w.w, h1[4 * c + 3], t1);
            }
            if (px < W) {
              T[tap * n_pix] = t0;
              if (two) T[tap * n_pix + down] = t1;
            }
          }
        }
      } else {
        for (int k = 0; k < nrow; ++k) {
          float v[32];
          if (!(ok = read(v))) break;
          if (px < W) tc_store_row(v, S.bias, reinterpret_cast<uint4*>(y) + tc_act(row0 + y0 + k * dil, 0, W, px), W);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 64;" ::"r"(tmem) : "memory");
  }
}

// The first layer (2 -> 32, ReLU) on the tensor cores: an implicit GEMM
// with K = 2 channels x 9 taps = 18, padded with zeros to 32 (two MMAs of
// K = 16).  A tile is 128 pixels of one image row (M = 128), one per thread:
// the thread's 18 inputs, read in FP32 and rounded to BF16, go into the A
// tile, K-major without swizzle like conv_tc_kernel's operands (8-value
// chunks 128 x 16 bytes apart); the block packs the 32 x 18 weights the same
// way once ([chunk][out][8], zero-padded); the epilogue is conv_tc_kernel's.
// A block walks strips of rows y0, y0 + dil, ...: a thread reads 6 new inputs
// per row and keeps the other 12, the A tile and the accumulator are double,
// and a row's read-back and stores overlap the next row's MMAs.  (All 18
// inputs of every pixel, one tile at a time, from a BF16 copy of the input
// made by another pass: 119 + 10 us on 64 images of 256^2; this form 78.)
constexpr int kTcFirstChunkA = kTcTile * 16;  // bytes between the A tile's 8-value chunks

struct TcFirstSmem {
  __nv_bfloat16 a[2][4 * kTcTile * 8];  // [chunk][pixel][8 values of k]
  __nv_bfloat16 b[4 * 32 * 8];          // [chunk][out][8 values of k]
  float bias[32];
  uint64_t done[2];
  uint32_t tmem;
};

__global__ void __launch_bounds__(kTcFirstThreads) conv_first_tc_kernel(const float* __restrict__ x,
                                                                        const __nv_bfloat16* __restrict__ w,
                                                                        const __nv_bfloat16* __restrict__ bias,
                                                                        int B, int H, int W, int dil, int strip,
                                                                        __nv_bfloat16* __restrict__ y, int* err) {
  __shared__ __align__(1024) TcFirstSmem S;
  const int t = threadIdx.x;
  const int warp = warp_uniform(t >> 5);
  // weights [chunk j][out n][e] = w[n][8 j + e] (k = channel * 9 + tap), zero past k = 17
  for (int i = t; i < 4 * 32 * 8; i += kTcFirstThreads) {
    const int e = i & 7, n = (i >> 3) & 31, j = i >> 8;
    const int k = 8 * j + e;
    S.b[i] = k < 18 ? w[n * 18 + k] : __float2bfloat16_rn(0.0f);
  }
  if (t < 32) S.bias[t] = __bfloat162float(bias[t]);
#pragma unroll
  for (int q = 0; q < 2; ++q)  // k = 24 .. 31 stay zero
    reinterpret_cast<uint4*>(S.a[q])[3 * kTcTile + t] = make_uint4(0u, 0u, 0u, 0u);
  if (t == 0) {
    mbar_init(&S.done[0], 1);
    mbar_init(&S.done[1], 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 64;" ::"r"(smem_u32(&S.tmem))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = S.tmem;
  const int tiles_x = (W + kTcTile - 1) / kTcTile;
  const int per_class = (H + dil - 1) / dil, chunks = (per_class + strip - 1) / strip;
  const int n_strips = B * tiles_x * dil * chunks;
  const int64_t HW = static_cast<int64_t>(H) * W;
  uint32_t g = 0;  // rows so far: row g uses buffers g % 2
  int64_t out_row = -1;  // the row whose accumulator has not been read back
  int out_px = 0;
  bool ok = true;
  // reads row g - 1's accumulator back and stores its pixels
  auto finish = [&]() {
    if (out_row < 0) return true;
    if (!__syncthreads_and(mbar_wait(&S.done[(g - 1) & 1], ((g - 1) >> 1) & 1, err))) return false;
    tc_fence_after();
    float acc[32];
    tc_load32(tmem + (static_cast<uint32_t>(warp * 32) << 16) + 32 * ((g - 1) & 1), acc);
    if (out_px < W) tc_store_row(acc, S.bias, reinterpret_cast<uint4*>(y) + tc_act(out_row, 0, W, out_px), W);
    out_row = -1;
    return true;
  };
  for (int item = blockIdx.x; item < n_strips && ok; item += gridDim.x) {
    int rest = item;
    const int ch = rest % chunks;
    rest /= chunks;
    const int cls = rest % dil;
    rest /= dil;
    const int px = (rest % tiles_x) * kTcTile + t;
    const int b = rest / tiles_x;
    const int y0 = cls + ch * strip * dil;
    const int nrow = y0 < H ? min(strip, (H - 1 - y0) / dil + 1) : 0;
    const float* xb = x + static_cast<int64_t>(b) * 2 * HW;
    // inputs of three rows: in[channel][row][kx]
    float in[2][3][3];
    auto load = [&](int m, float (&dst)[2][3]) {  // row m of the strip
      const int ii = y0 + m * dil;
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int kx = 0; kx < 3; ++kx) {
          const int jj = px + dil * (kx - 1);
          dst[c][kx] = 0.0f;
          if (px < W && ii >= 0 && ii < H && jj >= 0 && jj < W)
            dst[c][kx] = __ldg(xb + c * HW + static_cast<int64_t>(ii) * W + jj);
        }
    };
    float r0[2][3], r1[2][3], next[2][3];
    load(-1, r0);
    load(0, r1);
    load(1, next);
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int kx = 0; kx < 3; ++kx) {
        in[c][0][kx] = 0.0f;
        in[c][1][kx] = r0[c][kx];
        in[c][2][kx] = r1[c][kx];
      }
    for (int k = 0; k < nrow; ++k) {
      const int q = g & 1;  // free: row g - 2 was read back before row g - 1 was issued
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int kx = 0; kx < 3; ++kx) {
          in[c][0][kx] = in[c][1][kx];
          in[c][1][kx] = in[c][2][kx];
          in[c][2][kx] = next[c][kx];
        }
      load(k + 2, next);
      float v[24];
#pragma unroll
      for (int e = 0; e < 24; ++e) v[e] = e < 18 ? in[e / 9][(e % 9) / 3][e % 3] : 0.0f;
#pragma unroll
      for (int j = 0; j < 3; ++j)
        reinterpret_cast<uint4*>(S.a[q])[j * kTcTile + t] =
            make_uint4(pack_bf16x2(v[8 * j], v[8 * j + 1]), pack_bf16x2(v[8 * j + 2], v[8 * j + 3]),
                       pack_bf16x2(v[8 * j + 4], v[8 * j + 5]), pack_bf16x2(v[8 * j + 6], v[8 * j + 7]));
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic writes -> tensor core reads
      tc_fence_before();
      __syncthreads();
      if (t == 0) {
        tc_fence_after();
        const uint32_t a_base = smem_u32(S.a[q]), b_base = smem_u32(S.b);
#pragma unroll
        for (int h = 0; h < 2; ++h)
          tc_mma(tmem + 32 * q, tc_desc(a_base + 2 * h * kTcFirstChunkA, kTcFirstChunkA, 128),
                 tc_desc(b_base + 2 * h * kTcChunkB, kTcChunkB, 128), h);
        tc_commit(&S.done[q]);
      }
      if (!(ok = finish())) {
        ++g;  // this row's MMAs are waited for below
        break;
      }
      out_row = static_cast<int64_t>(b) * H + y0 + k * dil;
      out_px = px;
      ++g;
    }
  }
  if (ok) finish();
  // the last MMAs have completed before their tensor memory is released
  // (after a wait that gave up: bounded)
  if (g > 0) mbar_wait(&S.done[(g - 1) & 1], ((g - 1) >> 1) & 1, err);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 64;" ::"r"(tmem) : "memory");
  }
}

// Packs the 32 -> 32 layers' FP32 weights (out, in, 3, 3) into the MMA's B
// layout [tap][chunk][out][8 channels], rounded to BF16.
__global__ void pack_tc_kernel(const float* __restrict__ p, int64_t off0, int64_t stride,
                               __nv_bfloat16* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= kTcMidLayers * kTcPacked) return;
  const int l = i / kTcPacked, r = i - l * kTcPacked;
  const int e = r & 7, o = (r >> 3) & 31, kc = (r >> 8) & 3, tap = r >> 10;
  const int c = kc * 8 + e;
  out[i] = __float2bfloat16_rn(p[off0 + l * stride + (o * 32 + c) * 9 + tap]);
}

// The last layer (32 -> 1, linear), second half: y(p) = b + sum over the
// nine taps of T[tap][p + offset_tap] (zero outside the image), the planes
// the last 32 -> 32 layer's epilogue wrote (conv_tc_kernel<true>); taps in
// (ky, kx) order.  y FP32 (B, 1, H, W).
// A thread sums four pixels, so that 36 loads are in flight.
constexpr int kLastPix = 4;

__global__ void __launch_bounds__(256) conv_last_sum_kernel(const float* __restrict__ T,
                                                            const __nv_bfloat16* __restrict__ bias, int B, int H,
                                                            int W, int dil, float* __restrict__ y) {
  const int HW = H * W;
  const int b = blockIdx.y;
  const int64_t n_pix = static_cast<int64_t>(B) * HW;
  const float* Tb = T + static_cast<int64_t>(b) * HW;
  const float b0 = __bfloat162float(bias[0]);
  float t[kLastPix][9];
#pragma unroll
  for (int u = 0; u < kLastPix; ++u) {
    const int p = (blockIdx.x * kLastPix + u) * 256 + threadIdx.x;
    const int i = p / W, j = p - i * W;
#pragma unroll
    for (int tap = 0; tap < 9; ++tap) {
      const int ii = i + dil * (tap / 3 - 1), jj = j + dil * (tap % 3 - 1);
      t[u][tap] = 0.0f;
      if (p < HW && ii >= 0 && ii < H && jj >= 0 && jj < W) t[u][tap] = __ldg(Tb + tap * n_pix + ii * W + jj);
    }
  }
#pragma unroll
  for (int u = 0; u < kLastPix; ++u) {
    const int p = (blockIdx.x * kLastPix + u) * 256 + threadIdx.x;
    float acc = b0;
#pragma unroll
    for (int tap = 0; tap < 9; ++tap) acc += t[u][tap];
    if (p < HW) y[static_cast<int64_t>(b) * HW + p] = acc;
  }
}

int ew_grid(int64_t n) {
  return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 8 * sm_count())));
}

}  // namespace

struct WsNet {
  int device = 0;
  int H = 0, W = 0, Bmax = 0;
  int dil[kLayers] = {};
  int64_t off_w[kLayers] = {}, off_b[kLayers] = {};
  int64_t nparams = 0;
  int step = 0;
  int loss_kind = 0;  // 0 mean squared error, 1 energy norm
  int64_t device_bytes = 0;
  float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;  // flat FP32 master, gradient, Adam moments
  float* wflip = nullptr;                                          // flipped weights (same offsets)
  __nv_bfloat16* pbf = nullptr;                                    // BF16 copy for inference
  bool bf_stale = true;
  float* act[kLayers + 1] = {};  // act[0] unused (the caller's input); act[l + 1] = layer l output
  float* dbuf[2] = {};           // data-gradient ping-pong
  __nv_bfloat16* hbf[2] = {};    // inference: ping-pong activations (layout of tc_act)
  __nv_bfloat16* wtc = nullptr;  // the 32 -> 32 layers' weights in the tensor-core layout
  int* err = nullptr;            // device-side wait that gave up (kErrTimeout)
  int tc_smem_sm = 0, tc_reserved = 0;  // shared memory per SM and reserved per block
  float* partials = nullptr;
  int64_t partial_floats = 0;
  float* chunk = nullptr;  // kReduceChunks x the largest stride
  float* red = nullptr;
  unsigned int* counter = nullptr;
  double* dred = nullptr;
  unsigned int* dcounter = nullptr;
  double* scal = nullptr;  // [0] rms(b), [1] alpha
  float* feat = nullptr;   // one problem's input (2 H W) and output (H W)
  double* ax = nullptr;    // A x0 (warm start with projection)
  int64_t ax_n = 0;
};

namespace {

void wsnet_release(WsNet* N) {
  if (!N) return;
  const int prev = current_device();
  cudaSetDevice(N->device);
  void* ptrs[] = {N->p,      N->g,      N->m,        N->v,     N->wflip,   N->pbf,  N->dbuf[0],
                  N->dbuf[1], N->hbf[0], N->hbf[1], N->partials, N->chunk, N->red,
                  N->counter, N->dred,   N->dcounter, N->scal,  N->feat,     N->ax,      N->wtc, N->err};
  for (void* q : ptrs) dfree(q);
  for (int l = 1; l <= kLayers; ++l) dfree(N->act[l]);
  cudaSetDevice(prev);
  delete N;
}

struct WsDeleter {
  void operator()(WsNet* n) const { wsnet_release(n); }
};

template <int CIN, int COUT, int MODE, typename TI, typename TW, typename TO>
int launch_conv(const TI* x, const TW* w, const TW* bias, int B, int H, int W, int dil, TO* y, const float* mask,
                cudaStream_t s) {
  const dim3 grid((H * W + kConvThreads - 1) / kConvThreads, B);
  conv_fwd_kernel<CIN, COUT, MODE, TI, TW, TO><<<grid, kConvThreads, 0, s>>>(x, w, bias, H, W, dil, y, mask);
  GK_TRY_CUDA(cudaGetLastError());
  return GK_OK;
}

template <int MODE>
int launch_conv32(const float* x, const float* w, const float* bias, int B, int H, int W, int dil, float* y,
                  const float* mask, cudaStream_t s) {
  const int tw = c32_width(W), groups = kC32Threads / tw;
  const int64_t items =
      static_cast<int64_t>(B) * ((W + tw - 1) / tw) * ((c32_units(H, dil) + groups - 1) / groups);
  const int grid = static_cast<int>(std::min<int64_t>(items, 2 * static_cast<int64_t>(sm_count())));
  conv32_kernel<MODE><<<grid, kC32Threads, kC32Smem, s>>>(x, w, bias, B, H, W, dil, y, mask);
  GK_TRY_CUDA(cudaGetLastError());
  return GK_OK;
}

int forward_layer(int l, const float* x, const float* w, const float* bias, int B, int H, int W, int dil, float* y,
                  cudaStream_t s) {
  if (l == 0) return launch_conv<2, 32, CONV_RELU>(x, w, bias, B, H, W, dil, y, nullptr, s);
  if (l < kLayers - 1) return launch_conv32<CONV_RELU>(x, w, bias, B, H, W, dil, y, nullptr, s);
  return launch_conv<32, 1, CONV_LINEAR>(x, w, bias, B, H, W, dil, y, nullptr, s);
}

// The documented limit on the width: one row of a layer's two tensors, three
// input rows with their halo, would fit a block's shared memory.  (No kernel
// stages whole rows any more.)
size_t width_limit_bytes(int cin, int cout, int W, int dil) {
  const int co_t = cout >= 4 ? 4 : 1;
  const size_t xsplit = kConvThreads / (cin * (cout / co_t));
  const size_t staging = static_cast<size_t>(cout) * (W | 1) + 3 * static_cast<size_t>(cin) * ((W + 2 * dil) | 1);
  const size_t classes = xsplit * (static_cast<size_t>(cout) * cin * 9 + cout);
  return sizeof(float) * std::max(staging, classes);
}

// Slots of a layer's weight-gradient partials for a batch of B.
int64_t wgrad_slots(int cin, int cout, int B, int H, int W, int dil) {
  if (cin == 32 && cout == 32) return std::min<int64_t>(w32_items(B, H, W, dil), 2 * sm_count());
  return static_cast<int64_t>(B) * thin_units(H, dil);
}

template <int CIN, int COUT>
int launch_wgrad(const WsNet& N, const float* x, const float* dy, int B, int dil, float* grads, cudaStream_t s) {
  constexpr int STRIDE = COUT * CIN * 9 + COUT;
  const int64_t nslots = wgrad_slots(CIN, COUT, B, N.H, N.W, dil);
  if (nslots * STRIDE > N.partial_floats) return set_error(GK_ERR_UNSUPPORTED, "wsnet: gradient scratch too small");
  if constexpr (CIN == 32 && COUT == 32) {
    wgrad32_kernel<<<static_cast<int>(nslots), kW32Threads, w32_smem(dil), s>>>(
        x, dy, B, N.H, N.W, dil, w32_rows(B, N.H, N.W, dil), N.partials);
  } else {
    wgrad_thin_kernel<CIN, COUT>
        <<<dim3(thin_units(N.H, dil), B), 256, 0, s>>>(x, dy, N.H, N.W, dil, N.partials);
  }
  GK_TRY_CUDA(cudaGetLastError());
  const int nch = static_cast<int>(std::min<int64_t>(kReduceChunks, nslots));
  const int64_t per = (nslots + nch - 1) / nch;
  wgrad_chunk_kernel<<<dim3((STRIDE + 255) / 256, nch), 256, 0, s>>>(N.partials, nslots, STRIDE, per, N.chunk);
  GK_TRY_CUDA(cudaGetLastError());
  wgrad_final_kernel<<<(STRIDE + 255) / 256, 256, 0, s>>>(N.chunk, nch, STRIDE, grads);
  GK_TRY_CUDA(cudaGetLastError());
  return GK_OK;
}

int check_batch(const WsNet* N, int32_t B) {
  if (!N) return set_error(GK_ERR_ARG, "wsnet: NULL handle");
  if (B < 1 || B > N->Bmax) return set_error(GK_ERR_DIM, "wsnet: batch %d outside 1..%d", B, N->Bmax);
  return GK_OK;
}

// FP32 forward of a batch into N.act[1..6].
int forward_f32(WsNet& N, int B, const float* x, cudaStream_t s) {
  const float* in = x;
  for (int l = 0; l < kLayers; ++l) {
    GK_TRY(forward_layer(l, in, N.p + N.off_w[l], N.p + N.off_b[l], B, N.H, N.W, N.dil[l], N.act[l + 1], s));
    in = N.act[l + 1];
  }
  return GK_OK;
}

// Loss (into N.red[0], device) and gradients (into N.g) of a batch.
int gradients(WsNet& N, int B, const float* x, const float* target, cudaStream_t s) {
  GK_TRY(forward_f32(N, B, x, s));
  const int64_t nout = static_cast<int64_t>(B) * N.H * N.W;
  float* dout = N.dbuf[0];
  if (N.loss_kind == 1)
    energy_kernel<<<ew_grid(nout), 256, 0, s>>>(N.act[kLayers], target, x, B, N.H, N.W, dout, N.red + 2, N.counter,
                                                N.red);
  else
    mse_kernel<<<ew_grid(nout), 256, 0, s>>>(N.act[kLayers], target, nout, dout, N.red + 2, N.counter, N.red);
  GK_TRY_CUDA(cudaGetLastError());
  for (int l = 0; l < kLayers; ++l) {
    flip_kernel<<<ew_grid(kCh[l] * kCh[l + 1] * 9), 256, 0, s>>>(N.p + N.off_w[l], kCh[l], kCh[l + 1],
                                                                  N.wflip + N.off_w[l]);
    GK_TRY_CUDA(cudaGetLastError());
  }
  const float* gcur = dout;
  int pp = 0;
  for (int l = kLayers - 1; l >= 0; --l) {
    const float* xin = l == 0 ? x : N.act[l];
    float* gw = N.g + N.off_w[l];  // the bias gradient follows the weights
    if (l == 0) GK_TRY((launch_wgrad<2, 32>(N, xin, gcur, B, N.dil[l], gw, s)));
    else if (l < kLayers - 1) GK_TRY((launch_wgrad<32, 32>(N, xin, gcur, B, N.dil[l], gw, s)));
    else GK_TRY((launch_wgrad<32, 1>(N, xin, gcur, B, N.dil[l], gw, s)));
    if (l == 0) break;
    float* gnext = N.dbuf[1 - pp];
    // data gradient of layer l, masked by the ReLU of layer l - 1 (its output act[l])
    if (l == kLayers - 1)
      GK_TRY((launch_conv<1, 32, CONV_MASK, float, float, float>(gcur, N.wflip + N.off_w[l], nullptr, B, N.H, N.W,
                                                                 N.dil[l], gnext, N.act[l], s)));
    else
      GK_TRY(launch_conv32<CONV_MASK>(gcur, N.wflip + N.off_w[l], nullptr, B, N.H, N.W, N.dil[l], gnext, N.act[l],
                                      s));
    gcur = gnext;
    pp = 1 - pp;
  }
  return GK_OK;
}

int infer_bf16(WsNet& N, int B, const float* x, float* y, cudaStream_t s) {
  if (N.bf_stale) {
    to_bf16_kernel<<<ew_grid(N.nparams), 256, 0, s>>>(N.p, N.pbf, N.nparams);
    GK_TRY_CUDA(cudaGetLastError());
    pack_tc_kernel<<<(kTcMidLayers * kTcPacked + 255) / 256, 256, 0, s>>>(N.p, N.off_w[1], N.off_w[2] - N.off_w[1],
                                                                          N.wtc);
    GK_TRY_CUDA(cudaGetLastError());
    N.bf_stale = false;
  }
  const dim3 pg((N.H * N.W + 256 * kLastPix - 1) / (256 * kLastPix), B);
  const int64_t tiles = static_cast<int64_t>(B) * N.H * ((N.W + kTcTile - 1) / kTcTile);
  // strips as long as the work still gives every resident CTA about four of
  // them (a batch of one image runs single rows, each reading its three input
  // rows; large batches reuse rows along strips of up to 16), then evened out
  // over the rows of a residue class
  auto strip_for = [&](int grid, int dil) {
    const int target = static_cast<int>(
        std::max<int64_t>(1, std::min<int64_t>(kTcStripMax, tiles / (4 * static_cast<int64_t>(grid)))));
    const int per_class = (N.H + dil - 1) / dil;
    const int n_chunks = (per_class + target - 1) / target;
    return (per_class + n_chunks - 1) / n_chunks;
  };
  // 8 resident blocks per SM: 64 of the 512 tensor-memory columns each
  const int grid1 = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(tiles, 8 * sm_count())));
  conv_first_tc_kernel<<<grid1, kTcFirstThreads, 0, s>>>(x, N.pbf + N.off_w[0], N.pbf + N.off_b[0], B, N.H, N.W,
                                                         N.dil[0], strip_for(grid1, N.dil[0]), N.hbf[0], N.err);
  GK_TRY_CUDA(cudaGetLastError());
  const __nv_bfloat16* in = N.hbf[0];
  for (int l = 1; l < kLayers - 1; ++l) {
    __nv_bfloat16* out = N.hbf[l & 1];
    // resident blocks per SM: shared memory is the limit (registers, warps
    // and the 512 tensor-memory columns allow 8 blocks of 64 columns), and
    // it depends on the dilation through the staged rows' width
    const size_t smem = tc_smem_bytes(N.dil[l]) + (l == kLayers - 2 ? kTcLastBytes : 0);
    int per_sm = std::max(1, std::min(8, static_cast<int>(static_cast<size_t>(N.tc_smem_sm) / (smem + N.tc_reserved))));
    // small batches keep three blocks per SM (the count the widest rows
    // allow): more blocks would shorten every block's strips, and each strip
    // stages two rows more than it computes
    if (tiles < 16 * 3 * static_cast<int64_t>(sm_count())) per_sm = std::min(per_sm, 3);
    const int grid = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(tiles, int64_t(per_sm) * sm_count())));
    const int strip = strip_for(grid, N.dil[l]);
    // the last 32 -> 32 layer also folds in the 32 -> 1 layer: it writes the
    // nine tap planes (36 bytes per pixel, within the 64 of the buffer)
    if (l == kLayers - 2)
      conv_tc_kernel<true><<<grid, kTcThreads, smem, s>>>(in, N.wtc + (l - 1) * kTcPacked, N.pbf + N.off_b[l], B,
                                                          N.H, N.W, N.dil[l], strip, N.pbf + N.off_w[kLayers - 1],
                                                          out, N.err);
    else
      conv_tc_kernel<false><<<grid, kTcThreads, smem, s>>>(in, N.wtc + (l - 1) * kTcPacked, N.pbf + N.off_b[l], B,
                                                           N.H, N.W, N.dil[l], strip, nullptr, out, N.err);
    GK_TRY_CUDA(cudaGetLastError());
    in = out;
  }
  conv_last_sum_kernel<<<pg, 256, 0, s>>>(reinterpret_cast<const float*>(in), N.pbf + N.off_b[kLayers - 1], B, N.H,
                                          N.W, N.dil[kLayers - 1], y);
  GK_TRY_CUDA(cudaGetLastError());
  return GK_OK;
}

}  // namespace
}  // namespace gk

using namespace gk;

extern "C" int gk_wsnet_create(int32_t H, int32_t W, int32_t batch_max, const int32_t* dilations, gk_wsnet* out) {
  if (!out || !dilations) return set_error(GK_ERR_ARG, "gk_wsnet_create: NULL argument");
  *out = nullptr;
  if (H < 1 || W < 1 || batch_max < 1 || static_cast<int64_t>(H) * W > (1 << 26))
    return set_error(GK_ERR_DIM, "gk_wsnet_create: H %d, W %d, batch %d", H, W, batch_max);
  std::unique_ptr<WsNet, WsDeleter> hold(new WsNet);
  WsNet* N = hold.get();
  N->device = current_device();
  N->H = H;
  N->W = W;
  N->Bmax = batch_max;
  int64_t off = 0;
  for (int l = 0; l < kLayers; ++l) {
    N->dil[l] = dilations[l];
    if (dilations[l] < 1 || dilations[l] > kTcMaxDil)
      return set_error(GK_ERR_ARG, "gk_wsnet_create: dilation %d outside 1..64", dilations[l]);
    N->off_w[l] = off;
    off += static_cast<int64_t>(kCh[l]) * kCh[l + 1] * 9;
    N->off_b[l] = off;
    off += kCh[l + 1];
  }
  N->nparams = off;
  int smem_max = 0;
  GK_TRY_CUDA(cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, N->device));
  for (int l = 0; l < kLayers; ++l)
    if (width_limit_bytes(kCh[l], kCh[l + 1], W, N->dil[l]) > static_cast<size_t>(smem_max))
      return set_error(GK_ERR_UNSUPPORTED, "gk_wsnet_create: width %d with dilation %d exceeds the limit",
                       W, N->dil[l]);
  int64_t* by = &N->device_bytes;
  const size_t np = static_cast<size_t>(off);
  for (float** q : {&N->p, &N->g, &N->m, &N->v, &N->wflip}) GK_TRY(dalloc_n(q, np, by));
  GK_TRY(dalloc_n(&N->pbf, np, by));
  const size_t img = static_cast<size_t>(H) * W;
  const size_t big = static_cast<size_t>(batch_max) * 32 * img;
  for (int l = 1; l <= kLayers; ++l)
    GK_TRY(dalloc_n(&N->act[l], l < kLayers ? big : static_cast<size_t>(batch_max) * img, by));
  for (float** q : {&N->dbuf[0], &N->dbuf[1]}) GK_TRY(dalloc_n(q, big, by));
  for (__nv_bfloat16** q : {&N->hbf[0], &N->hbf[1]}) GK_TRY(dalloc_n(q, big, by));
  GK_TRY(dalloc_n(&N->wtc, static_cast<size_t>(kTcMidLayers) * kTcPacked, by));
  GK_TRY(dalloc_n(&N->err, 1, by));
  GK_TRY_CUDA(cudaMemset(N->err, 0, sizeof(int)));
  GK_TRY(set_smem(wgrad32_kernel, std::max(w32_smem(kTcMaxDil), w32_smem(32))));
  GK_TRY(set_smem(conv32_kernel<CONV_RELU>, kC32Smem));
  GK_TRY(set_smem(conv32_kernel<CONV_MASK>, kC32Smem));
  GK_TRY(set_smem(conv_tc_kernel<false>, tc_smem_bytes(kTcMaxDil)));
  GK_TRY(set_smem(conv_tc_kernel<true>, tc_smem_bytes(kTcMaxDil) + kTcLastBytes));
  // the grid of each layer is sized from its shared-memory footprint (the
  // occupancy query has been seen to report 1 for this kernel where 3 fit)
  GK_TRY_CUDA(cudaDeviceGetAttribute(&N->tc_smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, N->device));
  GK_TRY_CUDA(cudaDeviceGetAttribute(&N->tc_reserved, cudaDevAttrReservedSharedMemoryPerBlock, N->device));
  // weight-gradient slots: the most any layer and batch needs
  int64_t pf = 0;
  for (int l = 0; l < kLayers; ++l)
    for (int B = 1; B <= batch_max; ++B)
      pf = std::max(pf, wgrad_slots(kCh[l], kCh[l + 1], B, H, W, N->dil[l]) *
                            (static_cast<int64_t>(kCh[l]) * kCh[l + 1] * 9 + kCh[l + 1]));
  N->partial_floats = pf;
  GK_TRY(dalloc_n(&N->partials, static_cast<size_t>(pf), by));
  GK_TRY(dalloc_n(&N->chunk, static_cast<size_t>(kReduceChunks) * kW32Stride, by));
  const int rg = 8 * sm_count() + 8;
  GK_TRY(dalloc_n(&N->red, static_cast<size_t>(rg + 4), by));
  GK_TRY(dalloc_n(&N->counter, 1, by));
  GK_TRY(dalloc_n(&N->dred, static_cast<size_t>(2 * rg + 4), by));
  GK_TRY(dalloc_n(&N->dcounter, 1, by));
  GK_TRY(dalloc_n(&N->scal, 4, by));
  GK_TRY(dalloc_n(&N->feat, 3 * img, by));
  GK_TRY_CUDA(cudaMemset(N->counter, 0, sizeof(unsigned int)));
  GK_TRY_CUDA(cudaMemset(N->dcounter, 0, sizeof(unsigned int)));
  GK_TRY_CUDA(cudaMemset(N->m, 0, np * sizeof(float)));
  GK_TRY_CUDA(cudaMemset(N->v, 0, np * sizeof(float)));
  GK_TRY_CUDA(cudaMemset(N->p, 0, np * sizeof(float)));
  GK_TRY_CUDA(cudaDeviceSynchronize());
  *out = reinterpret_cast<gk_wsnet>(hold.release());
  return GK_OK;
}

extern "C" int gk_wsnet_num_params(gk_wsnet h, int64_t* n) {
  WsNet* N = reinterpret_cast<WsNet*>(h);
  if (!N || !n) return set_error(GK_ERR_ARG, "gk_wsnet_num_params: NULL argument");
  *n = N->nparams;
  return GK_OK;
}

extern "C" int gk_wsnet_set_params(gk_wsnet h, const float* params, void* stream) {
  WsNet* N = reinterpret_cast<WsNet*>(h);
  if (!N || !params) return set_error(GK_ERR_ARG, "gk_wsnet_set_params: NULL argument");
  DeviceGuard dg(N->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  GK_TRY_CUDA(cudaMemcpyAsync(N->p, params, sizeof(float) * N->nparams, cudaMemcpyDefault, s));
  GK_TRY_CUDA(cudaMemsetAsync(N->m, 0, sizeof(float) * N->nparams, s));
  GK_TRY_CUDA(cudaMemsetAsync(N->v, 0, sizeof(float) * N->nparams, s));
  GK_TRY_CUDA(cudaStreamSynchronize(s));
  N->step = 0;
  N->bf_stale = true;
  return GK_OK;
}

extern "C" int gk_wsnet_set_loss(gk_wsnet h, int32_t kind) {
  WsNet* N = reinterpret_cast<WsNet*>(h);
  if (!N) return set_error(GK_ERR_ARG, "gk_wsnet_set_loss: NULL handle");
  if (kind != 0 && kind != 1) return set_error(GK_ERR_ARG, "gk_wsnet_set_loss: kind %d (0 or 1)", kind);
  N->loss_kind = kind;
  return GK_OK;
}

extern "C" int gk_wsnet_get_params(gk_wsnet h, float* params, void* stream) {
  WsNet* N = reinterpret_cast<WsNet*>(h);
  if (!N || !params) return set_error(GK_ERR_ARG, "gk_wsnet_get_params: NULL argument");
  DeviceGuard dg(N->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  GK_TRY_CUDA(cudaMemcpyAsync(params, N->p, sizeof(float) * N->nparams, cudaMemcpyDefault, s));
  GK_TRY_CUDA(cudaStreamSynchronize(s));
  return GK_OK;
}

extern "C" int gk_wsnet_forward(gk_wsnet h, int32_t B, const float* x, float* y, void* stream) {
  WsNet* N = reinterpret_cast<WsNet*>(h);
  GK_TRY(check_batch(N, B));
  if (!x || !y) return set_error(GK_ERR_ARG, "gk_wsnet_forward: NULL argument");
  DeviceGuard dg(N->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  GK_TRY(forward_f32(*N, B, x, s));
  GK_TRY_CUDA(cudaMemcpyAsync(y, N->act[kLayers], sizeof(float) * B * N->H * N->W, cudaMemcpyDeviceToDevice, s));
  return GK_OK;
}

extern "C" int gk_wsnet_gradients(gk_wsnet h, int32_t B, const float* x, const float* target, float* loss,
                                  float* grads, void* stream) {
  WsNet* N = reinterpret_cast<WsNet*>(h);
  GK_TRY(check_batch(N, B));
  if (!x || !target) return set_error(GK_ERR_ARG, "gk_wsnet_gradients: NULL argument");
  DeviceGuard dg(N->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  GK_TRY(gradients(*N, B, x, target, s));
  if (grads) GK_TRY_CUDA(cudaMemcpyAsync(grads, N->g, sizeof(float) * N->nparams, cudaMemcpyDefault, s));
  if (loss) GK_TRY_CUDA(cudaMemcpyAsync(loss, N->red, sizeof(float), cudaMemcpyDefault, s));
  GK_TRY_CUDA(cudaStreamSynchronize(s));
  return GK_OK;
}

extern "C" int gk_wsnet_train_step(gk_wsnet h, int32_t B, const float* x, const float* target, float lr,
                                   float* loss, void* stream) {
  WsNet* N = reinterpret_cast<WsNet*>(h);
  GK_TRY(check_batch(N, B));
  if (!x || !target) return set_error(GK_ERR_ARG, "gk_wsnet_train_step: NULL argument");
  if (!(lr > 0.0f)) return set_error(GK_ERR_ARG, "gk_wsnet_train_step: learning rate %g", lr);
  DeviceGuard dg(N->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  GK_TRY(gradients(*N, B, x, target, s));
  N->step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.0f - powf(b1, static_cast<float>(N->step)), c2 = 1.0f - powf(b2, static_cast<float>(N->step));
  adam_kernel<<<ew_grid(N->nparams), 256, 0, s>>>(N->p, N->g, N->m, N->v, N->nparams, lr, b1, b2, 1e-8f, c1, c2);
  GK_TRY_CUDA(cudaGetLastError());
  N->bf_stale = true;
  if (loss) GK_TRY_CUDA(cudaMemcpyAsync(loss, N->red, sizeof(float), cudaMemcpyDefault, s));
  return GK_OK;
}

extern "C" int gk_wsnet_infer_bf16(gk_wsnet h, int32_t B, const float* x, float* y, void* stream) {
  WsNet* N = reinterpret_cast<WsNet*>(h);
  GK_TRY(check_batch(N, B));
  if (!x || !y) return set_error(GK_ERR_ARG, "gk_wsnet_infer_bf16: NULL argument");
  DeviceGuard dg(N->device);
  return infer_bf16(*N, B, x, y, static_cast<cudaStream_t>(stream));
}

extern "C" int gk_wsnet_check(gk_wsnet h, void* stream) {
  WsNet* N = reinterpret_cast<WsNet*>(h);
  if (!N) return set_error(GK_ERR_ARG, "gk_wsnet_check: NULL handle");
  DeviceGuard dg(N->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int e = 0;
  GK_TRY_CUDA(cudaMemcpyAsync(&e, N->err, sizeof(int), cudaMemcpyDeviceToHost, s));
  GK_TRY_CUDA(cudaStreamSynchronize(s));
  if (e != 0) {
    GK_TRY_CUDA(cudaMemsetAsync(N->err, 0, sizeof(int), s));
    GK_TRY_CUDA(cudaStreamSynchronize(s));
    return set_error(GK_ERR_TIMEOUT, "gk_wsnet_check: a tensor-core completion wait gave up");
  }
  return GK_OK;
}

extern "C" int gk_wsnet_features(gk_wsnet h, const double* g, const double* b, const double* x, double out_scale,
                                 float* feat, float* target, void* stream) {
  WsNet* N = reinterpret_cast<WsNet*>(h);
  if (!N || !g || !b || !feat || (x && !target)) return set_error(GK_ERR_ARG, "gk_wsnet_features: NULL argument");
  if (!(out_scale > 0.0)) return set_error(GK_ERR_ARG, "gk_wsnet_features: out_scale must be positive");
  DeviceGuard dg(N->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int64_t n = static_cast<int64_t>(N->H) * N->W;
  rms_kernel<<<ew_grid(n), 256, 0, s>>>(b, n, N->dred + 4, N->dcounter, N->scal);
  GK_TRY_CUDA(cudaGetLastError());
  features_kernel<<<ew_grid(n), 256, 0, s>>>(g, b, x, N->scal, out_scale, n, feat, target);
  GK_TRY_CUDA(cudaGetLastError());
  return GK_OK;
}

extern "C" int gk_wsnet_warm_start(gk_wsnet h, gk_matrix A, const double* g, const double* b, double out_scale,
                                   double* x0, void* stream) {
  WsNet* N = reinterpret_cast<WsNet*>(h);
  if (!N || !g || !b || !x0) return set_error(GK_ERR_ARG, "gk_wsnet_warm_start: NULL argument");
  if (!(out_scale > 0.0)) return set_error(GK_ERR_ARG, "gk_wsnet_warm_start: out_scale must be positive");
  DeviceGuard dg(N->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int64_t n = static_cast<int64_t>(N->H) * N->W;
  Matrix* M = A ? as_matrix(A) : nullptr;
  if (M && (M->n_rows != n || M->n_cols != n))
    return set_error(GK_ERR_DIM, "gk_wsnet_warm_start: matrix is %lld x %lld, the grid has %lld points",
                     (long long)M->n_rows, (long long)M->n_cols, (long long)n);
  rms_kernel<<<ew_grid(n), 256, 0, s>>>(b, n, N->dred + 4, N->dcounter, N->scal);
  GK_TRY_CUDA(cudaGetLastError());
  features_kernel<<<ew_grid(n), 256, 0, s>>>(g, b, nullptr, N->scal, out_scale, n, N->feat, nullptr);
  GK_TRY_CUDA(cudaGetLastError());
  float* y = N->feat + 2 * n;
  GK_TRY(infer_bf16(*N, 1, N->feat, y, s));
  scale_out_kernel<<<ew_grid(n), 256, 0, s>>>(y, N->scal, out_scale, n, x0);
  GK_TRY_CUDA(cudaGetLastError());
  if (M) {
    if (N->ax_n < n) {
      dfree(N->ax);
      N->ax = nullptr;
      GK_TRY(dalloc_n(&N->ax, static_cast<size_t>(n), &N->device_bytes));
      N->ax_n = n;
    }
    Epi e;
    e.mode = EPI_COPY;
    e.y = N->ax;
    e.err = M->err;
    GK_TRY(spmv_launch(*M, x0, e, s));
    galerkin_sums_kernel<<<ew_grid(n), 256, 0, s>>>(x0, b, N->ax, n, N->dred + 4, N->dcounter, N->scal + 1);
    GK_TRY_CUDA(cudaGetLastError());
    scale_kernel<<<ew_grid(n), 256, 0, s>>>(x0, N->scal + 1, n);
    GK_TRY_CUDA(cudaGetLastError());
  }
  return GK_OK;
}

extern "C" int gk_wsnet_destroy(gk_wsnet h) {
  if (!h) return set_error(GK_ERR_ARG, "gk_wsnet_destroy: NULL handle");
  wsnet_release(reinterpret_cast<WsNet*>(h));
  return GK_OK;
}
