// The convolutional SNN's layout kernels (Tab. I CSNN: 5x5 convolutions and
// 2x2 max pooling), for channel-last bf16 activations [M, H, W, C] with
// M = T*B.  A convolution runs as a tensor-core GEMM over patch rows:
//   im2col   cols[(m, oy, ox), (ky, kx, c)] = X[m, oy+ky, ox+kx, c]
//            (columns past KH*KW*Cin up to Kpad are zero), so the layer's
//            input current is cols * W^T with W [Cout, KH, KW, Cin];
//   col2im   dX[m, y, x, c] = sum over the (ky, kx) with a valid output
//            pixel (y-ky, x-kx) of dcols[(m, y-ky, x-kx), (ky, kx, c)],
//            added in (ky, kx) order in fp32 (deterministic);
//   max pool 2x2 windows, stride 2; the first maximum in window order
//            (row major) is kept and its position recorded, and the
//            backward routes the gradient there (every input element
//            belongs to one window, so no two threads write one element).
// With a channel count that is a multiple of 8 every kernel moves 8
// channels (16 bytes) per thread; otherwise one element per thread.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <climits>
#include <cstdint>

#include "scan_host.cuh"
#include "snn.h"

namespace snn {
namespace {

constexpr int kThreads = 256;

// Eight consecutive columns of one patch row per thread (one 16-byte store).
template <typename Ix>
__global__ void __launch_bounds__(kThreads) im2col_kernel(const __nv_bfloat16* __restrict__ X,
                                                          __nv_bfloat16* __restrict__ cols,
                                                          Ix rows, int H, int W, int Cin,
                                                          int KH, int KW, int Kpad) {
  grid_dep_wait();
  const int Ho = H - KH + 1, Wo = W - KW + 1;
  const int K = KH * KW * Cin;
  const int vec_per_row = Kpad / 8;
  const Ix i = (Ix)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= rows * vec_per_row) return;
  const Ix r = i / vec_per_row;
  const int k0 = (int)(i - r * vec_per_row) * 8;
  const Ix m = r / (Ho * Wo);
  const int p = (int)(r - m * (Ho * Wo));
  const int oy = p / Wo, ox = p - oy * Wo;
  const __nv_bfloat16* xm = X + m * H * W * Cin;
  __align__(16) __nv_bfloat16 v[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int k = k0 + j;
    __nv_bfloat16 e = __float2bfloat16_rn(0.0f);
    if (k < K) {
      const int ky = k / (KW * Cin);
      const int rem = k - ky * KW * Cin;
      const int kx = rem / Cin, c = rem - kx * Cin;
      e = xm[((oy + ky) * W + (ox + kx)) * Cin + c];
    }
    v[j] = e;
  }
  *reinterpret_cast<uint4*>(cols + r * Kpad + k0) = *reinterpret_cast<const uint4*>(v);
}

template <typename Ix>
__global__ void __launch_bounds__(kThreads) col2im_kernel(const __nv_bfloat16* __restrict__ dcols,
                                                          __nv_bfloat16* __restrict__ dX,
                                                          Ix total, int H, int W, int Cin,
                                                          int KH, int KW, int Kpad) {
  grid_dep_wait();
  const int Ho = H - KH + 1, Wo = W - KW + 1;
  const Ix i = (Ix)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  const int c = (int)(i % Cin);
  const Ix q = i / Cin;
  const int x = (int)(q % W);
  const Ix q2 = q / W;
  const int y = (int)(q2 % H);
  const Ix m = q2 / H;
  float s = 0.0f;
  for (int ky = 0; ky < KH; ++ky) {
    const int oy = y - ky;
    if (oy < 0 || oy >= Ho) continue;
    for (int kx = 0; kx < KW; ++kx) {
      const int ox = x - kx;
      if (ox < 0 || ox >= Wo) continue;
      const Ix r = (m * Ho + oy) * Wo + ox;
      s += __bfloat162float(dcols[r * Kpad + (ky * KW + kx) * Cin + c]);
    }
  }
  dX[i] = __float2bfloat16_rn(s);
}

template <typename Ix>
__global__ void __launch_bounds__(kThreads) maxpool_fwd_kernel(const __nv_bfloat16* __restrict__ X,
                                                               __nv_bfloat16* __restrict__ Y,
                                                               uint8_t* __restrict__ idx,
                                                               Ix total, int H, int W,
                                                               int C) {
  grid_dep_wait();
  const Ix i = (Ix)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  const int Hp = H / 2, Wp = W / 2;
  const int c = (int)(i % C);
  const Ix q = i / C;
  const int px = (int)(q % Wp);
  const Ix q2 = q / Wp;
  const int py = (int)(q2 % Hp);
  const Ix m = q2 / Hp;
  const __nv_bfloat16* base = X + ((m * H + 2 * py) * W + 2 * px) * C + c;
  const Ix off[4] = {0, (Ix)C, (Ix)W * C, (Ix)W * C + C};
  float best = __bfloat162float(base[0]);
  int arg = 0;
#pragma unroll
  for (int j = 1; j < 4; ++j) {
    const float v = __bfloat162float(base[off[j]]);
    if (v > best) {  // strict: the first maximum is kept
      best = v;
      arg = j;
    }
  }
  Y[i] = __float2bfloat16_rn(best);
  idx[i] = (uint8_t)arg;
}

template <typename Ix>
__global__ void __launch_bounds__(kThreads) maxpool_bwd_kernel(const __nv_bfloat16* __restrict__ dY,
                                                               const uint8_t* __restrict__ idx,
                                                               __nv_bfloat16* __restrict__ dX,
                                                               Ix total, int H, int W,
                                                               int C) {
  grid_dep_wait();
  const Ix i = (Ix)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  const int Hp = H / 2, Wp = W / 2;
  const int c = (int)(i % C);
  const Ix q = i / C;
  const int x = (int)(q % W);
  const Ix q2 = q / W;
  const int y = (int)(q2 % H);
  const Ix m = q2 / H;
  const Ix o = ((m * Hp + y / 2) * Wp + x / 2) * C + c;
  const int pos = (y & 1) * 2 + (x & 1);
  dX[i] = idx[o] == pos ? dY[o] : __float2bfloat16_rn(0.0f);
}

// ---- 8 channels per thread (C % 8 == 0, 16-byte aligned tensors) --------

union Pack8 {
  uint4 u;
  __nv_bfloat16 h[8];
};

// Thread i copies column group j = i % (Kpad/8) of patch row i / (Kpad/8):
// the 8 channels of one tap (groups past K are zero).
template <typename Ix>
__global__ void __launch_bounds__(kThreads) im2col_vec8_kernel(const uint4* __restrict__ X,
                                                               uint4* __restrict__ cols,
                                                               Ix rows, int H, int W, int Cin,
                                                               int KH, int KW, int Kpad) {
  grid_dep_wait();
  const int Ho = H - KH + 1, Wo = W - KW + 1;
  const int G = Cin / 8;  // channel groups per tap
  const int vpr = Kpad / 8;
  const Ix i = (Ix)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= rows * vpr) return;
  const Ix r = i / vpr;
  const int j = (int)(i - r * vpr);
  uint4 v = make_uint4(0u, 0u, 0u, 0u);
  if (j < KH * KW * G) {
    const Ix m = r / (Ho * Wo);
    const int p = (int)(r - m * (Ho * Wo));
    const int oy = p / Wo, ox = p - oy * Wo;
    const int tap = j / G, g = j - tap * G;
    const int ky = tap / KW, kx = tap - ky * KW;
    v = X[((m * H + oy + ky) * W + ox + kx) * G + g];
  }
  cols[i] = v;
}

// As im2col_vec8_kernel for any number of patch rows whose column groups fit
// a table: a block writes a run of consecutive patch rows (about
// kIm2colBlockVecs vectors), and both halves of a vector's source address,
// the patch row's first pixel and the column group's tap, come from
// shared-memory tables that the block fills once.  The row and group of a
// thread's next vector follow from the last one's by an addition, so a
// vector costs no division: with three per vector the kernel was bound by
// issue slots (42 us for the 164 MB of the CSNN's second layer at M = 3200,
// 64 rows of 400 columns; 24 us at 6.8 TB/s), now 31 us.
constexpr int kIm2colMaxGroups = 4096;  // column groups (Kpad / 8) the table holds
constexpr int kIm2colBlockVecs = 4096;
constexpr int kIm2colMaxRows = 1024;
constexpr int kIm2colPer = 4;  // vectors a thread loads before it stores them

template <typename Ix>
__global__ void __launch_bounds__(kThreads) im2col_rows_kernel(const uint4* __restrict__ X,
                                                               uint4* __restrict__ cols, Ix rows,
                                                               int H, int W, int Cin, int KH, int KW,
                                                               int Kpad, int block_rows) {
  extern __shared__ __align__(16) unsigned char sm[];
  const int Ho = H - KH + 1, Wo = W - KW + 1;
  const int G = Cin / 8, vpr = Kpad / 8;
  Ix* row0 = reinterpret_cast<Ix*>(sm);                   // first pixel of row r (16-byte units)
  int* toff = reinterpret_cast<int*>(row0 + block_rows);  // offset of group j's tap, or -1
  const Ix r_lo = (Ix)blockIdx.x * block_rows;
  const int nr = (int)min((Ix)block_rows, rows - r_lo);
  for (int j = threadIdx.x; j < vpr; j += kThreads) {
    int t = -1;
    if (j < KH * KW * G) {
      const int tap = j / G, g = j - tap * G;
      const int ky = tap / KW, kx = tap - ky * KW;
      t = (ky * W + kx) * G + g;
    }
    toff[j] = t;
  }
  for (int r = threadIdx.x; r < nr; r += kThreads) {
    const Ix m = (r_lo + r) / (Ho * Wo);
    const int p = (int)(r_lo + r - m * (Ho * Wo));
    const int oy = p / Wo, ox = p - oy * Wo;
    row0[r] = ((m * H + oy) * W + ox) * G;
  }
  __syncthreads();
  grid_dep_wait();
  const int dr = kThreads / vpr, dj = kThreads - dr * vpr;
  int r = threadIdx.x / vpr, j = threadIdx.x - r * vpr;
  uint4* out = cols + r_lo * vpr;
  const int n = nr * vpr;
  for (int i = threadIdx.x; i < n; i += kIm2colPer * kThreads) {
    uint4 v[kIm2colPer];
#pragma unroll
    for (int u = 0; u < kIm2colPer; ++u) {
      v[u] = make_uint4(0u, 0u, 0u, 0u);
      if (r < nr) {
        const int t = toff[j];
        if (t >= 0) v[u] = __ldg(X + row0[r] + t);
      }
      r += dr;
      j += dj;
      if (j >= vpr) {
        j -= vpr;
        ++r;
      }
    }
#pragma unroll
    for (int u = 0; u < kIm2colPer; ++u)
      if (i + u * kThreads < n) out[i + u * kThreads] = v[u];
  }
}

// Thread i sums the 8 channels of group i % G of pixel i / G over the taps
// that read it, in (ky, kx) order.
template <typename Ix, int KH_ = 0, int KW_ = 0>
__global__ void __launch_bounds__(kThreads) col2im_vec8_kernel(const uint4* __restrict__ dcols,
                                                               uint4* __restrict__ dX,
                                                               Ix total, int H, int W, int Cin,
                                                               int KH, int KW, int Kpad) {
  grid_dep_wait();
  const int Ho = H - KH + 1, Wo = W - KW + 1;
  const int G = Cin / 8, vpr = Kpad / 8;
  const Ix i = (Ix)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  const Ix q = i / G;
  const int g = (int)(i - q * G);
  const int x = (int)(q % W);
  const Ix q2 = q / W;
  const int y = (int)(q2 % H);
  const Ix m = q2 / H;
  float s[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) s[e] = 0.0f;
  if constexpr (KH_ > 0) {
    // fixed taps: one filter row's KW_ loads issued before its adds, which
    // still run in (ky, kx) order
#pragma unroll 1
    for (int ky = 0; ky < KH_; ++ky) {
      const int oy = y - ky;
      if (oy < 0 || oy >= Ho) continue;
      Pack8 v[KW_];
#pragma unroll
      for (int kx = 0; kx < KW_; ++kx) {
        const int ox = x - kx;
        v[kx].u = (ox >= 0 && ox < Wo) ? dcols[((m * Ho + oy) * Wo + ox) * vpr + (ky * KW_ + kx) * G + g]
                                       : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int kx = 0; kx < KW_; ++kx) {
        const int ox = x - kx;
        if (ox >= 0 && ox < Wo) {
#pragma unroll
          for (int e = 0; e < 8; ++e) s[e] += __bfloat162float(v[kx].h[e]);
        }
      }
    }
  } else {
    for (int ky = 0; ky < KH; ++ky) {
      const int oy = y - ky;
      if (oy < 0 || oy >= Ho) continue;
      for (int kx = 0; kx < KW; ++kx) {
        const int ox = x - kx;
        if (ox < 0 || ox >= Wo) continue;
        const Ix r = (m * Ho + oy) * Wo + ox;
        Pack8 v;
        v.u = dcols[r * vpr + (ky * KW + kx) * G + g];
#pragma unroll
        for (int e = 0; e < 8; ++e) s[e] += __bfloat162float(v.h[e]);
      }
    }
  }
  Pack8 o;
#pragma unroll
  for (int e = 0; e < 8; ++e) o.h[e] = __float2bfloat16_rn(s[e]);
  dX[i] = o.u;
}

// As col2im_vec8_kernel with an image's patch rows staged whole in shared
// memory: its 25 (or 9) taps of 32 bytes per pixel are scattered over rows
// 2*Kpad bytes apart, which as direct loads kept 16 sectors per request in
// flight; staged, the rows stream in contiguously (cp.async) and the gather
// reads shared memory without conflicts.  Four blocks share an SM, so the
// copies of three are in flight while one sums (two blocks with two stages
// each were slower: their copies waited for their own sums).  Images are
// taken from the last to the first: the product that wrote dcols has just
// written the last ones, which are still in L2.  35 us for the CSNN's second
// layer (164 MB; 24 us at 6.8 TB/s) with direct loads, now 30 us.
// The sums keep the (ky, kx) order, so both kernels give the same bits.
constexpr int kCol2imThreads = 288;  // one (pixel, 8 channels) each of a 12 x 12 x 16 map
constexpr int kCol2imPerSm = 4;
constexpr int kCol2imMaxStage = 56 * 1024;  // four blocks fit an SM

__device__ __forceinline__ void col2im_cp16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// (low, high) bf16 of a word as floats
__device__ __forceinline__ float2 bf2_floats(uint32_t w) {
  return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}

template <int KH, int KW>
__global__ void __launch_bounds__(kCol2imThreads, kCol2imPerSm) col2im_staged_kernel(
    const uint4* __restrict__ dcols, uint4* __restrict__ dX, int64_t M, int H, int W, int Cin,
    int Kpad) {
  extern __shared__ __align__(16) unsigned char sm[];
  const int Ho = H - KH + 1, Wo = W - KW + 1;
  const int G = Cin / 8, vpr = Kpad / 8;
  const int vecs = Ho * Wo * vpr, outs = H * W * G;
  const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(sm));
  const uint4* d = reinterpret_cast<const uint4*>(sm);
  grid_dep_wait();
  for (int64_t m = M - 1 - blockIdx.x; m >= 0; m -= gridDim.x) {
    const uint4* src = dcols + m * vecs;
    for (int v = threadIdx.x; v < vecs; v += kCol2imThreads) col2im_cp16(base + (uint32_t)v * 16u, src + v);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();  // the image has landed for every thread
    for (int o = threadIdx.x; o < outs; o += kCol2imThreads) {
      const int q = o / G, g = o - q * G;
      const int y = q / W, x = q - y * W;
      float2 s[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) s[e] = make_float2(0.0f, 0.0f);
      const uint4* dg = d + (y * Wo + x) * vpr + g;  // the tap (ky, kx) is at pixel (y - ky, x - kx)
#pragma unroll
      for (int ky = 0; ky < KH; ++ky) {
        const bool in_y = (unsigned)(y - ky) < (unsigned)Ho;
#pragma unroll
        for (int kx = 0; kx < KW; ++kx) {
          if (in_y && (unsigned)(x - kx) < (unsigned)Wo) {
            const uint4 v = dg[(ky * KW + kx) * G - (ky * Wo + kx) * vpr];
            s[0] = __fadd2_rn(s[0], bf2_floats(v.x));
            s[1] = __fadd2_rn(s[1], bf2_floats(v.y));
            s[2] = __fadd2_rn(s[2], bf2_floats(v.z));
            s[3] = __fadd2_rn(s[3], bf2_floats(v.w));
          }
        }
      }
      uint4 r;
      uint32_t* rw = reinterpret_cast<uint32_t*>(&r);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(s[e].x, s[e].y);
        rw[e] = *reinterpret_cast<const uint32_t*>(&h);
      }
      dX[m * outs + o] = r;
    }
    __syncthreads();  // the stage is free for the next image
  }
}

template <int KH, int KW>
cudaError_t launch_col2im_staged(const void* dcols, void* dX, int64_t M, int H, int W, int Cin, int Kpad,
                                 size_t smem, cudaStream_t st) {
  const void* k = (const void*)col2im_staged_kernel<KH, KW>;
  cudaError_t e = ensure_smem(k, smem);
  DeviceInfo d;
  if (e == cudaSuccess) e = device_info(&d);
  if (e != cudaSuccess) return e;
  const int64_t slots = kCol2imPerSm * (int64_t)d.sms;
  return launch_pdl(col2im_staged_kernel<KH, KW>, dim3((unsigned)(M < slots ? M : slots)),
                    dim3(kCol2imThreads), smem, st, static_cast<const uint4*>(dcols),
                    static_cast<uint4*>(dX), M, H, W, Cin, Kpad);
}

// Thread i pools the 8 channels of group i % G of output pixel i / G.
template <typename Ix>
__global__ void __launch_bounds__(kThreads) maxpool_fwd_vec8_kernel(const uint4* __restrict__ X,
                                                                    uint4* __restrict__ Y,
                                                                    uint2* __restrict__ idx,
                                                                    Ix total, int H, int W,
                                                                    int C) {
  grid_dep_wait();
  const Ix i = (Ix)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  const int G = C / 8, Hp = H / 2, Wp = W / 2;
  const Ix q = i / G;
  const int g = (int)(i - q * G);
  const int px = (int)(q % Wp);
  const Ix q2 = q / Wp;
  const int py = (int)(q2 % Hp);
  const Ix m = q2 / Hp;
  const Ix base = ((m * H + 2 * py) * W + 2 * px) * G + g;
  Pack8 w[4];
  w[0].u = X[base];
  w[1].u = X[base + G];
  w[2].u = X[base + (Ix)W * G];
  w[3].u = X[base + (Ix)W * G + G];
  Pack8 best = w[0];
  uint8_t arg[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
  for (int j = 1; j < 4; ++j) {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (__bfloat162float(w[j].h[e]) > __bfloat162float(best.h[e])) {  // first maximum kept
        best.h[e] = w[j].h[e];
        arg[e] = (uint8_t)j;
      }
    }
  }
  Y[i] = best.u;
  uint2 a;
  a.x = (uint32_t)arg[0] | ((uint32_t)arg[1] << 8) | ((uint32_t)arg[2] << 16) | ((uint32_t)arg[3] << 24);
  a.y = (uint32_t)arg[4] | ((uint32_t)arg[5] << 8) | ((uint32_t)arg[6] << 16) | ((uint32_t)arg[7] << 24);
  idx[i] = a;
}

// Thread i routes the 8 channels of group i % G of output pixel i / G back
// to its window, writing all four positions (zero where not the maximum).
template <typename Ix>
__global__ void __launch_bounds__(kThreads) maxpool_bwd_vec8_kernel(const uint4* __restrict__ dY,
                                                                    const uint2* __restrict__ idx,
                                                                    uint4* __restrict__ dX,
                                                                    Ix total, int H, int W,
                                                                    int C) {
  grid_dep_wait();
  const Ix i = (Ix)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  const int G = C / 8, Hp = H / 2, Wp = W / 2;
  const Ix q = i / G;
  const int g = (int)(i - q * G);
  const int px = (int)(q % Wp);
  const Ix q2 = q / Wp;
  const int py = (int)(q2 % Hp);
  const Ix m = q2 / Hp;
  Pack8 d;
  d.u = dY[i];
  const uint2 a = idx[i];
  const __nv_bfloat16 zero = __float2bfloat16_rn(0.0f);
  Pack8 o[4];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const int pos = (int)(((e < 4 ? a.x : a.y) >> (8 * (e & 3))) & 0xFFu);
#pragma unroll
    for (int j = 0; j < 4; ++j) o[j].h[e] = pos == j ? d.h[e] : zero;
  }
  const Ix base = ((m * H + 2 * py) * W + 2 * px) * G + g;
  dX[base] = o[0].u;
  dX[base + G] = o[1].u;
  dX[base + (Ix)W * G] = o[2].u;
  dX[base + (Ix)W * G + G] = o[3].u;
}

bool aligned(const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

unsigned blocks_for(int64_t n) { return (unsigned)((n + kThreads - 1) / kThreads); }

}  // namespace
}  // namespace snn

using namespace snn;

extern "C" snn_status_t snn_im2col_nhwc(int64_t M, int64_t H, int64_t W, int64_t Cin, int64_t KH,
                                        int64_t KW, int64_t Kpad, const void* X, void* cols,
                                        snn_stream_t stream) {
  if (M < 0 || KH < 1 || KW < 1 || H < KH || W < KW || Cin < 1) return SNN_ERR_INVALID_ARG;
  if (H * W * Cin > INT_MAX / 2 || Kpad > INT_MAX / 2) return SNN_ERR_INVALID_ARG;
  if (Kpad < KH * KW * Cin || Kpad % 8 != 0) return SNN_ERR_INVALID_ARG;
  if (M == 0) return SNN_OK;
  if (!X || !cols) return SNN_ERR_INVALID_ARG;
  if (!aligned(cols, 16) || !aligned(X, 2)) return SNN_ERR_ALIGNMENT;
  const int64_t rows = M * (H - KH + 1) * (W - KW + 1);
  const int64_t n = rows * (Kpad / 8);
  if (n / kThreads >= INT_MAX) return SNN_ERR_INVALID_ARG;
  const bool i32 = rows * Kpad < INT_MAX && M * H * W * Cin < INT_MAX;  // 32-bit index math
  if (Cin % 8 == 0 && aligned(X, 16) && Kpad / 8 <= kIm2colMaxGroups) {
    const int64_t vpr = Kpad / 8;
    int64_t br = kIm2colBlockVecs / vpr;  // rows per block
    br = br < 16 ? 16 : br > kIm2colMaxRows ? kIm2colMaxRows : br;
    const unsigned nb = (unsigned)((rows + br - 1) / br);
    const size_t smem = (size_t)br * (i32 ? 4 : 8) + (size_t)vpr * 4;  // at most 24 KB
    const cudaError_t e =
        i32 ? launch_pdl(im2col_rows_kernel<int>, dim3(nb), dim3(kThreads), smem,
                         reinterpret_cast<cudaStream_t>(stream), static_cast<const uint4*>(X),
                         static_cast<uint4*>(cols), rows, (int)H, (int)W, (int)Cin, (int)KH,
                         (int)KW, (int)Kpad, (int)br)
            : launch_pdl(im2col_rows_kernel<int64_t>, dim3(nb), dim3(kThreads), smem,
                         reinterpret_cast<cudaStream_t>(stream), static_cast<const uint4*>(X),
                         static_cast<uint4*>(cols), rows, (int)H, (int)W, (int)Cin, (int)KH,
                         (int)KW, (int)Kpad, (int)br);
    return e == cudaSuccess ? SNN_OK : SNN_ERR_CUDA;
  }
  if (Cin % 8 == 0 && aligned(X, 16)) {
    const cudaError_t e = i32 ? launch_pdl(im2col_vec8_kernel<int>, dim3(blocks_for(n)), dim3(kThreads), 0,
                                     reinterpret_cast<cudaStream_t>(stream),
                                     static_cast<const uint4*>(X), static_cast<uint4*>(cols), rows,
                                     (int)H, (int)W, (int)Cin, (int)KH, (int)KW, (int)Kpad)
                                   : launch_pdl(im2col_vec8_kernel<int64_t>, dim3(blocks_for(n)), dim3(kThreads), 0,
                                     reinterpret_cast<cudaStream_t>(stream),
                                     static_cast<const uint4*>(X), static_cast<uint4*>(cols), rows,
                                     (int)H, (int)W, (int)Cin, (int)KH, (int)KW, (int)Kpad);
    return e == cudaSuccess ? SNN_OK : SNN_ERR_CUDA;
  }
  const cudaError_t e = i32 ? launch_pdl(im2col_kernel<int>, dim3(blocks_for(n)), dim3(kThreads), 0,
                                   reinterpret_cast<cudaStream_t>(stream),
                                   static_cast<const __nv_bfloat16*>(X),
                                   static_cast<__nv_bfloat16*>(cols), rows, (int)H, (int)W, (int)Cin,
                                   (int)KH, (int)KW, (int)Kpad)
                                   : launch_pdl(im2col_kernel<int64_t>, dim3(blocks_for(n)), dim3(kThreads), 0,
                                   reinterpret_cast<cudaStream_t>(stream),
                                   static_cast<const __nv_bfloat16*>(X),
                                   static_cast<__nv_bfloat16*>(cols), rows, (int)H, (int)W, (int)Cin,
                                   (int)KH, (int)KW, (int)Kpad);
  return e == cudaSuccess ? SNN_OK : SNN_ERR_CUDA;
}

extern "C" snn_status_t snn_col2im_nhwc(int64_t M, int64_t H, int64_t W, int64_t Cin, int64_t KH,
                                        int64_t KW, int64_t Kpad, const void* dcols, void* dX,
                                        snn_stream_t stream) {
  if (M < 0 || KH < 1 || KW < 1 || H < KH || W < KW || Cin < 1) return SNN_ERR_INVALID_ARG;
  if (H * W * Cin > INT_MAX / 2 || Kpad > INT_MAX / 2) return SNN_ERR_INVALID_ARG;
  if (Kpad < KH * KW * Cin) return SNN_ERR_INVALID_ARG;
  if (M == 0) return SNN_OK;
  if (!dcols || !dX) return SNN_ERR_INVALID_ARG;
  if (!aligned(dcols, 2) || !aligned(dX, 2)) return SNN_ERR_ALIGNMENT;
  const int64_t n = M * H * W * Cin;
  if (n / kThreads >= INT_MAX) return SNN_ERR_INVALID_ARG;
  const bool i32 = M * (H - KH + 1) * (W - KW + 1) * Kpad < INT_MAX && n < INT_MAX;
  if (Cin % 8 == 0 && Kpad % 8 == 0 && aligned(dcols, 16) && aligned(dX, 16)) {
    cudaError_t e;
    const int64_t stage = (H - KH + 1) * (W - KW + 1) * Kpad * 2;  // bytes of an image's patch rows
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (KH == 5 && KW == 5 && stage <= kCol2imMaxStage)
      e = launch_col2im_staged<5, 5>(dcols, dX, M, (int)H, (int)W, (int)Cin, (int)Kpad, stage, st);
    else if (KH == 3 && KW == 3 && stage <= kCol2imMaxStage)
      e = launch_col2im_staged<3, 3>(dcols, dX, M, (int)H, (int)W, (int)Cin, (int)Kpad, stage, st);
    else if (KH == 5 && KW == 5 && i32)
      e = launch_pdl(col2im_vec8_kernel<int, 5, 5>, dim3(blocks_for(n / 8)), dim3(kThreads), 0,
                     reinterpret_cast<cudaStream_t>(stream), static_cast<const uint4*>(dcols),
                     static_cast<uint4*>(dX), n / 8, (int)H, (int)W, (int)Cin, (int)KH, (int)KW,
                     (int)Kpad);
    else
      e = i32 ? launch_pdl(col2im_vec8_kernel<int>, dim3(blocks_for(n / 8)), dim3(kThreads), 0,
                                     reinterpret_cast<cudaStream_t>(stream),
                                     static_cast<const uint4*>(dcols), static_cast<uint4*>(dX),
                                     n / 8, (int)H, (int)W, (int)Cin, (int)KH, (int)KW, (int)Kpad)
                                   : launch_pdl(col2im_vec8_kernel<int64_t>, dim3(blocks_for(n / 8)), dim3(kThreads), 0,
                                     reinterpret_cast<cudaStream_t>(stream),
                                     static_cast<const uint4*>(dcols), static_cast<uint4*>(dX),
                                     n / 8, (int)H, (int)W, (int)Cin, (int)KH, (int)KW, (int)Kpad);
    return e == cudaSuccess ? SNN_OK : SNN_ERR_CUDA;
  }
  const cudaError_t e = i32 ? launch_pdl(col2im_kernel<int>, dim3(blocks_for(n)), dim3(kThreads), 0,
                                   reinterpret_cast<cudaStream_t>(stream),
                                   static_cast<const __nv_bfloat16*>(dcols),
                                   static_cast<__nv_bfloat16*>(dX), n, (int)H, (int)W, (int)Cin,
                                   (int)KH, (int)KW, (int)Kpad)
                                   : launch_pdl(col2im_kernel<int64_t>, dim3(blocks_for(n)), dim3(kThreads), 0,
                                   reinterpret_cast<cudaStream_t>(stream),
                                   static_cast<const __nv_bfloat16*>(dcols),
                                   static_cast<__nv_bfloat16*>(dX), n, (int)H, (int)W, (int)Cin,
                                   (int)KH, (int)KW, (int)Kpad);
  return e == cudaSuccess ? SNN_OK : SNN_ERR_CUDA;
}

extern "C" snn_status_t snn_maxpool2_fwd_nhwc(int64_t M, int64_t H, int64_t W, int64_t C,
                                              const void* X, void* Y, uint8_t* idx,
                                              snn_stream_t stream) {
  if (M < 0 || H < 2 || W < 2 || C < 1 || H % 2 || W % 2) return SNN_ERR_INVALID_ARG;
  if (H * W * C > INT_MAX / 2) return SNN_ERR_INVALID_ARG;
  if (M == 0) return SNN_OK;
  if (!X || !Y || !idx) return SNN_ERR_INVALID_ARG;
  if (!aligned(X, 2) || !aligned(Y, 2)) return SNN_ERR_ALIGNMENT;
  const int64_t n = M * (H / 2) * (W / 2) * C;
  if (n / kThreads >= INT_MAX) return SNN_ERR_INVALID_ARG;
  const bool i32 = M * H * W * C < INT_MAX;
  if (C % 8 == 0 && aligned(X, 16) && aligned(Y, 16) && aligned(idx, 8)) {
    const cudaError_t e = i32 ? launch_pdl(maxpool_fwd_vec8_kernel<int>, dim3(blocks_for(n / 8)),
                                     dim3(kThreads), 0, reinterpret_cast<cudaStream_t>(stream),
                                     static_cast<const uint4*>(X), static_cast<uint4*>(Y),
                                     reinterpret_cast<uint2*>(idx), n / 8, (int)H, (int)W, (int)C)
                                   : launch_pdl(maxpool_fwd_vec8_kernel<int64_t>, dim3(blocks_for(n / 8)),
                                     dim3(kThreads), 0, reinterpret_cast<cudaStream_t>(stream),
                                     static_cast<const uint4*>(X), static_cast<uint4*>(Y),
                                     reinterpret_cast<uint2*>(idx), n / 8, (int)H, (int)W, (int)C);
    return e == cudaSuccess ? SNN_OK : SNN_ERR_CUDA;
  }
  const cudaError_t e = i32 ? launch_pdl(maxpool_fwd_kernel<int>, dim3(blocks_for(n)), dim3(kThreads), 0,
                                   reinterpret_cast<cudaStream_t>(stream),
                                   static_cast<const __nv_bfloat16*>(X),
                                   static_cast<__nv_bfloat16*>(Y), idx, n, (int)H, (int)W, (int)C)
                                   : launch_pdl(maxpool_fwd_kernel<int64_t>, dim3(blocks_for(n)), dim3(kThreads), 0,
                                   reinterpret_cast<cudaStream_t>(stream),
                                   static_cast<const __nv_bfloat16*>(X),
                                   static_cast<__nv_bfloat16*>(Y), idx, n, (int)H, (int)W, (int)C);
  return e == cudaSuccess ? SNN_OK : SNN_ERR_CUDA;
}

extern "C" snn_status_t snn_maxpool2_bwd_nhwc(int64_t M, int64_t H, int64_t W, int64_t C,
                                              const void* dY, const uint8_t* idx, void* dX,
                                              snn_stream_t stream) {
  if (M < 0 || H < 2 || W < 2 || C < 1 || H % 2 || W % 2) return SNN_ERR_INVALID_ARG;
  if (H * W * C > INT_MAX / 2) return SNN_ERR_INVALID_ARG;
  if (M == 0) return SNN_OK;
  if (!dY || !idx || !dX) return SNN_ERR_INVALID_ARG;
  if (!aligned(dY, 2) || !aligned(dX, 2)) return SNN_ERR_ALIGNMENT;
  const int64_t n = M * H * W * C;
  if (n / kThreads >= INT_MAX) return SNN_ERR_INVALID_ARG;
  const bool i32 = n < INT_MAX;
  if (C % 8 == 0 && aligned(dY, 16) && aligned(dX, 16) && aligned(idx, 8)) {
    const int64_t np = n / 32;  // output pixels x channel groups
    const cudaError_t e = i32 ? launch_pdl(maxpool_bwd_vec8_kernel<int>, dim3(blocks_for(np)),
                                     dim3(kThreads), 0, reinterpret_cast<cudaStream_t>(stream),
                                     static_cast<const uint4*>(dY),
                                     reinterpret_cast<const uint2*>(idx), static_cast<uint4*>(dX),
                                     np, (int)H, (int)W, (int)C)
                                   : launch_pdl(maxpool_bwd_vec8_kernel<int64_t>, dim3(blocks_for(np)),
                                     dim3(kThreads), 0, reinterpret_cast<cudaStream_t>(stream),
                                     static_cast<const uint4*>(dY),
                                     reinterpret_cast<const uint2*>(idx), static_cast<uint4*>(dX),
                                     np, (int)H, (int)W, (int)C);
    return e == cudaSuccess ? SNN_OK : SNN_ERR_CUDA;
  }
  const cudaError_t e = i32 ? launch_pdl(maxpool_bwd_kernel<int>, dim3(blocks_for(n)), dim3(kThreads), 0,
                                   reinterpret_cast<cudaStream_t>(stream),
                                   static_cast<const __nv_bfloat16*>(dY), idx,
                                   static_cast<__nv_bfloat16*>(dX), n, (int)H, (int)W, (int)C)
                                   : launch_pdl(maxpool_bwd_kernel<int64_t>, dim3(blocks_for(n)), dim3(kThreads), 0,
                                   reinterpret_cast<cudaStream_t>(stream),
                                   static_cast<const __nv_bfloat16*>(dY), idx,
                                   static_cast<__nv_bfloat16*>(dX), n, (int)H, (int)W, (int)C);
  return e == cudaSuccess ? SNN_OK : SNN_ERR_CUDA;
}
