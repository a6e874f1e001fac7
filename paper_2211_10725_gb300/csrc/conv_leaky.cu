// First-layer convolution fused with its Leaky scan and 2x2 max pooling
// (the CSNN's 5x5 filters over a 1-channel map, Tab. I; Eqs. 3-4): the
// fp32 currents never reach HBM, and the pooled map is formed from the
// spikes while they are in registers.
//
// What bounds it: issue slots and the stores (2 + 2 bytes per neuron-step of spk and mem,
// the bits and the pooled map).  As three kernels the currents made a 4 + 4
// byte round trip and the spikes were read back for pooling.  At T = 25,
// B = 128, 28x28 -> [24, 24, 16] (146 MB written: 21 us at 6.8 TB/s) the
// three kernels took 48 + 45 + 12 us one at a time from a cold cache, this
// one 30 us (58% of issue slots); with the weight gradient's product (see
// conv_small.cu) the CSNN's training step went from 510 to 406 us.
//
// Mapping: a warp owns 8 pooled pixels (2x2 windows) for all T steps.  Per
// step their currents are one product on the tensor cores,
//   I[16 pixel pairs, 2 x 16 channels] = patches[16, K] * B[K, 32]
// (mma m16n8k16): row r is the horizontal pixel pair of window r's upper
// output row, row r + 8 of its lower one; the columns are the left pixel's
// channels and the right pixel's.  K runs over the filter rows with KS + 1
// slots each, the window of the pair: the left pixel's filter sits in slots
// 0 .. KS-1 of B, the right one's in slots 1 .. KS, so that an A register
// (two neighbouring slots) is one aligned word of the staged image for every
// thread.  A first version with one pixel per row had to load two words and
// permute them for every odd pixel, and issued 270 instructions per 16
// pixels a step (46 us); this one 320 per 32.
// The tensor core truncates its sums, so a patch's two products start from
// zero and are added in rounded fp32.  Error of a current over its summed
// magnitudes, rms in units of 2^-24, uniform pixels: 0.119 so, 0.145 with the
// first sum handed to the second product, 0.136 with fp32 multiply-adds
// (normal pixels 0.129, 0.149, 0.132); 30.2 us at T = 25, B = 128.
// The 9 taps of a 3x3 filter are fp32 multiply-adds in filter order, the
// separate convolution's bits: as one product their error was 0.076 against
// 0.066, and a product for each filter row with compensated sums between them
// took 59 us where this takes 38.9 (three kernels 88).
// A tcgen05 tile (M = 128, 64-deep swizzled K blocks) would need the patch
// rows built in shared memory, which is the traffic this avoids; the product
// is 8 mma per 32 pixels and not what bounds the kernel.
//
// The accumulator layout gives a thread the same lanes at every step, so
// the membrane state stays in registers and no step needs a barrier.  The
// order of B's columns is chosen so that a thread holds 8 neighbouring
// channels of one pixel and the four threads of a pair its 64 contiguous
// bytes (16-byte stores, 512 contiguous bytes per warp), one byte of the
// spike bits, and, with its neighbour's byte, the whole pooling window.
//
// A slot outside a pixel's own window meets a zero in B; so that an infinity
// or NaN there stays outside, a block whose staged pixels hold one (tested
// once per 8 steps) masks those slots in A instead.
//
// A block is 2 warps: its few image rows (not the whole image) are staged 8
// steps at a time with cp.async (through registers for an X that starts off a
// 16-byte boundary), double-buffered, two barriers per 8 steps.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <climits>
#include <cstdint>
#include <type_traits>

#include "scan_host.cuh"
#include "scan_kernels.cuh"
#include "snn.h"

namespace snn {
namespace {

constexpr int kClWarps = 2;
constexpr int kClThreads = 32 * kClWarps;
constexpr int kClSteps = 8;   // time steps staged per buffer
constexpr int kClCout = 16;   // output channels

struct ConvLeakyArgs {
  int T, H, W, Ho, Wo, ldw;
  int64_t B, L;  // lanes per step: B * Ho * Wo * Cout
  int beta_ch, thr_ch;  // 1: one value per channel, 0: scalar
  const __nv_bfloat16* X;
  const __nv_bfloat16* Wt;
  const float* beta;
  const float* thr;
  __nv_bfloat16* spk;
  __nv_bfloat16* mem;
  unsigned char* bits;
  int64_t bits_row;
  __nv_bfloat16* pool;  // [T*B, Ho/2, Wo/2, Cout] or null
  unsigned char* idx;   // likewise (both or neither)
  int slice;            // bytes of one step's staged rows (a multiple of 16)
  int x_aligned;        // X starts on a 16-byte boundary (then every image does)
};

__device__ __forceinline__ void cl_cp16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// A product from zero: a tensor core truncates its sums, so the two k-steps
// of a patch are added in rounded fp32 instead of the first being handed to
// the second.
__device__ __forceinline__ void mma_bf16_zero(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%10, %10, %10, %10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "f"(0.0f));
}

// fwd_pair with the reset-to-zero state kept as (1 - z)*u (exact: u or a
// zero of its sign), so that z need not outlive the step.
template <int RESET>
__device__ __forceinline__ float2 leaky_pair(float2 beta, float2 negthr, float2 in, float2& u, float2& z) {
  if (RESET == RESET_ZERO) {
    const float2 un = add2_rn(mul_rn_pair(beta, u), in);
    z = fire2(un, negthr);
    u = mul2_rn(make_float2(1.0f - z.x, 1.0f - z.y), un);
    return un;
  }
  float2 none = f2(0.0f);
  fwd_pair<false, RESET>(0, beta, negthr, none, in, u, z, none);
  return u;
}

// One byte per bit of the low four.
__device__ __forceinline__ uint32_t spread4(uint32_t x) { return ((x & 15u) * 0x00204081u) & 0x01010101u; }

// KS: filter size (3 or 5).
template <int KS, int RESET>
__global__ void __launch_bounds__(kClThreads, 8) conv_leaky_kernel(const ConvLeakyArgs a) {
  constexpr int PR = (KS + 1) / 2;          // words per filter row
  constexpr int PAIRS = KS * PR;            // words per patch: 15 (5x5), 6 (3x3)
  constexpr bool MMA = KS == 5;
  constexpr int KSTEPS = MMA ? (PAIRS + 7) / 8 : 0;  // k16 steps
  extern __shared__ __align__(16) unsigned char sm[];
  const int lid = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lid >> 2, q = lid & 3;
  const int Wp = a.Wo >> 1, Pp = (a.Ho >> 1) * Wp;  // pooled pixels
  const int parts = (Pp + 8 * kClWarps - 1) / (8 * kClWarps);
  const int64_t b = blockIdx.x / parts;
  const int p_lo = (int)(blockIdx.x - b * parts) * 8 * kClWarps;  // the block's first window
  const int pw = p_lo + 8 * warp + g;
  const bool on = pw < Pp;                                  // this thread's window exists
  const int pc = on ? pw : Pp - 1;                          // one past the map repeats the last
  const int py = pc / Wp, px = pc - py * Wp;
  // staged rows: from the first row of the block's first window, from the
  // 16-byte boundary below
  const int e_lo = (2 * (p_lo / Wp) * a.W) & ~7;            // first staged element of an image
  const int img = a.H * a.W;
  grid_dep_wait();

  // B fragments.  Column 8*nb + c belongs to thread c / 2 of the quad, as its
  // value v = 2*nb + (c & 1): pixel (c / 2) & 1 of the pair, channel 8*(c /
  // 4) + v
  uint32_t wb[MMA ? KSTEPS : 1][4][2];
  {
    const int ch8 = 8 * (g >> 2), right = (g >> 1) & 1;
    const unsigned short* w = reinterpret_cast<const unsigned short*>(a.Wt);
#pragma unroll
    for (int ks = 0; ks < KSTEPS; ++ks)
#pragma unroll
      for (int nb = 0; nb < 4; ++nb)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int pi = ks * 8 + q + 4 * h, ky = pi / PR, s = 2 * (pi % PR) - right;
          const unsigned short* wr = w + (int64_t)(ch8 + 2 * nb + (g & 1)) * a.ldw + ky * KS;
          uint32_t v = 0;
          if (pi < PAIRS) {
            if (s >= 0 && s < KS) v = wr[s];
            if (s + 1 < KS) v |= (uint32_t)wr[s + 1] << 16;
          }
          wb[ks][nb][h] = v;
        }
  }
  // byte offset of the thread's A words from the pair's first pixel
  uint32_t aoff[MMA ? KSTEPS : 1][2];
#pragma unroll
  for (int ks = 0; ks < KSTEPS; ++ks)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int pi = ks * 8 + q + 4 * h, ky = pi / PR, s = 2 * (pi % PR);
      aoff[ks][h] = pi < PAIRS ? 2u * (uint32_t)(ky * a.W + s) : 0u;
    }
  // 3x3: the filters as fp32 [tap][channel] behind the staged rows
  const uint32_t w_addr = smem_u32(sm) + (uint32_t)(2 * kClSteps * a.slice);
  if constexpr (!MMA) {
    float* wsm = reinterpret_cast<float*>(sm + 2 * kClSteps * a.slice);
    for (int e = threadIdx.x; e < KS * KS * kClCout; e += kClThreads)
      wsm[e] = __bfloat162float(a.Wt[(int64_t)(e % kClCout) * a.ldw + e / kClCout]);
  }
  const int right = q & 1, ch0 = 8 * (q >> 1);  // this thread's pixel of the pair, first channel
  float2 beta[4], negthr[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int ch = ch0 + 2 * j;
    beta[j] = a.beta_ch ? make_float2(a.beta[ch], a.beta[ch + 1]) : f2(a.beta[0]);
    negthr[j] = a.thr_ch ? make_float2(-a.thr[ch], -a.thr[ch + 1]) : f2(-a.thr[0]);
  }
  float2 u[2][4], z[2][4];
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int j = 0; j < 4; ++j) u[r][j] = z[r][j] = f2(0.0f);

  const uint32_t sbase = smem_u32(sm);
  const int vecs = a.slice >> 4;  // 16-byte pieces of a step
  auto stage = [&](int t0, int buf) {
    const int n = min(kClSteps, a.T - t0);
    const __nv_bfloat16* src = a.X + ((int64_t)t0 * a.B + b) * img + e_lo;
    for (int v = threadIdx.x; v < n * vecs; v += kClThreads) {
      const int s = v / vecs, c = v - s * vecs;
      if (e_lo + 8 * c >= img) continue;  // the last rows' slice may reach past the image
      const uint32_t at = (uint32_t)((buf * kClSteps + s) * a.slice + 16 * c);
      const __nv_bfloat16* x = src + (int64_t)s * a.B * img + 8 * c;
      if (a.x_aligned) {
        cl_cp16(sbase + at, x);
      } else {  // a view off the 16-byte boundary: element by element, through registers
        const unsigned short* e = reinterpret_cast<const unsigned short*>(x);
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) w[k] = (uint32_t)e[2 * k] | ((uint32_t)e[2 * k + 1] << 16);
        *reinterpret_cast<uint4*>(sm + at) = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const uint32_t pix_addr = 2u * (uint32_t)(2 * py * a.W + 2 * px - e_lo);
  const uint32_t row_b = 2u * (uint32_t)a.W;            // bytes of an image row
  // the thread's lanes: 8 channels of one pixel of the upper row; the lower
  // row's are `below` elements on
  const int64_t pix = b * (a.Ho * a.Wo) + (int64_t)(2 * py) * a.Wo + 2 * px + right;
  __nv_bfloat16* spk = a.spk + pix * kClCout + ch0;
  __nv_bfloat16* mem = a.mem + pix * kClCout + ch0;
  unsigned char* bits = a.bits ? a.bits + pix * 2 + (q >> 1) : nullptr;
  const int below = a.Wo * kClCout;
  int64_t po = (b * Pp + pc) * kClCout + ch0;           // of the pooled pixel's channels
  const int64_t pool_step = a.B * Pp * kClCout;

  // one time step from the staged rows at p0; MASK: slots outside the
  // pixel's window are cleared from A (else they only meet zeros in B)
  auto step = [&](uint32_t p0, auto mask) {
    float2 cur[2][4];  // currents of the upper and lower pixel, 4 pairs of channels
    if constexpr (!MMA) {
      float x[KS + 1][KS];  // this pixel's windows of both rows
#pragma unroll
      for (int y = 0; y <= KS; ++y) {
        uint32_t w0, w1;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w0) : "r"(p0 + y * row_b));
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w1) : "r"(p0 + y * row_b + 4));
        const uint32_t w = __funnelshift_r(w0, w1, 16 * right);
        x[y][0] = __uint_as_float(w << 16);
        x[y][1] = __uint_as_float(w & 0xffff0000u);
        x[y][2] = __uint_as_float(right ? w1 & 0xffff0000u : w1 << 16);
      }
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j) cur[r][j] = f2(0.0f);
#pragma unroll
      for (int k = 0; k < KS * KS; ++k) {
        float2 w[4];
#pragma unroll
        for (int j = 0; j < 4; j += 2)
          asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                       : "=f"(w[j].x), "=f"(w[j].y), "=f"(w[j + 1].x), "=f"(w[j + 1].y)
                       : "r"(w_addr + 4u * (uint32_t)(k * kClCout + ch0 + 2 * j)));
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
          for (int j = 0; j < 4; ++j) cur[r][j] = fma2(f2(x[r + k / KS][k % KS]), w[j], cur[r][j]);
      }
    } else {
      constexpr bool MASK = decltype(mask)::value;
      uint32_t av[KSTEPS][4];
#pragma unroll
      for (int ks = 0; ks < KSTEPS; ++ks)
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int r = 0; r < 2; ++r)  // a0: (upper row, h 0), a1: (lower, 0), a2: (upper, 1), ...
            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(av[ks][2 * h + r]) : "r"(p0 + aoff[ks][h] + r * row_b));
#pragma unroll
      for (int nb = 0; nb < 4; ++nb) {
        float d[KSTEPS][4];
#pragma unroll
        for (int ks = 0; ks < KSTEPS; ++ks) {
          if (!MASK) {
            mma_bf16_zero(d[ks], av[ks], wb[ks][nb]);
          } else {
            // left pixels' columns without slot KS, right pixels' without slot
            // 0: two products, each kept by the threads of its pixel
            uint32_t al[4], ar[4];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int pi = ks * 8 + q + 4 * h, wi = pi % PR;
              const uint32_t ml = pi >= PAIRS ? 0u : wi == PR - 1 ? 0x0000ffffu : 0xffffffffu;
              const uint32_t mr = pi >= PAIRS ? 0u : wi == 0 ? 0xffff0000u : 0xffffffffu;
#pragma unroll
              for (int r = 0; r < 2; ++r) {
                al[2 * h + r] = av[ks][2 * h + r] & ml;
                ar[2 * h + r] = av[ks][2 * h + r] & mr;
              }
            }
            float r[4];
            mma_bf16_zero(d[ks], al, wb[ks][nb]);
            mma_bf16_zero(r, ar, wb[ks][nb]);
#pragma unroll
            for (int k = 0; k < 4; ++k) d[ks][k] = right ? r[k] : d[ks][k];
          }
        }
#pragma unroll
        for (int r = 0; r < 2; ++r)
          cur[r][nb] = add2(make_float2(d[0][2 * r], d[0][2 * r + 1]), make_float2(d[1][2 * r], d[1][2 * r + 1]));
      }
    }
    uint32_t zb[2];  // the 8 channels' spikes, upper and lower pixel
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      uint32_t zw[4], uw[4], acc = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 un = leaky_pair<RESET>(beta[j], negthr[j], cur[r][j], u[r][j], z[r][j]);
        uw[j] = Elem<__nv_bfloat16>::from2(un.x, un.y);
        zw[j] = Elem<__nv_bfloat16>::from2(z[r][j].x, z[r][j].y);
        acc |= (zw[j] & 0x00800080u) >> (7 - 2 * j);  // 1.0 is 0x3F80: bit 7 of each half
      }
      zb[r] = (acc | (acc >> 15)) & 0xffu;
      if (on) {
        *reinterpret_cast<uint4*>(spk + r * below) = make_uint4(zw[0], zw[1], zw[2], zw[3]);
        *reinterpret_cast<uint4*>(mem + r * below) = make_uint4(uw[0], uw[1], uw[2], uw[3]);
        if (bits) bits[r * 2 * a.Wo] = (unsigned char)zb[r];
      }
    }
    if (a.pool) {
      // window order: (y, x), (y, x+1), (y+1, x), (y+1, x+1); the first
      // spike is the maximum, position 0 when there is none.  The left
      // pixel's thread writes the values, the right one's the positions.
      const uint32_t mine = zb[0] | (zb[1] << 8);
      const uint32_t other = __shfl_xor_sync(0xffffffffu, mine, 1);
      const uint32_t l = right ? other : mine, rt = right ? mine : other;
      if (on) {
        const uint32_t top = l | rt;  // bits 0-7: any of the upper pixels
        if (!right) {
          const uint32_t any = top | (top >> 8);
          uint32_t y[4];
#pragma unroll
          for (int j = 0; j < 4; ++j)
            y[j] = (((any >> (2 * j)) & 1u) | ((any << (15 - 2 * j)) & 0x00010000u)) * 0x3F80u;
          *reinterpret_cast<uint4*>(a.pool + po) = make_uint4(y[0], y[1], y[2], y[3]);
        } else {
          const uint32_t hi = ~top & (top >> 8);                                // position 2 or 3
          const uint32_t lo = (~l & rt) | (hi & ~(l >> 8));                     // position 1 or 3
          *reinterpret_cast<uint2*>(a.idx + po) =
              make_uint2(spread4(lo) | (spread4(hi) << 1), spread4(lo >> 4) | (spread4(hi >> 4) << 1));
        }
      }
    }
    spk += a.L;
    mem += a.L;
    if (bits) bits += a.bits_row;
    po += pool_step;
  };

  stage(0, 0);
  for (int t0 = 0, buf = 0; t0 < a.T; t0 += kClSteps, buf ^= 1) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // these steps have landed; the other buffer is no longer read
    if (t0 + kClSteps < a.T) stage(t0 + kClSteps, buf ^ 1);
    const int n = min(kClSteps, a.T - t0);
    const uint32_t p0 = sbase + (uint32_t)(buf * kClSteps * a.slice) + pix_addr;
    if constexpr (!MMA) {  // a pixel's window alone: nothing to mask
      for (int s = 0; s < n; ++s) step(p0 + (uint32_t)(s * a.slice), std::false_type());
      continue;
    }
    // an infinity or NaN among the staged pixels (elements of the slice past
    // the image were never written and are skipped): an exponent of all ones
    // plus one unit of it sets the half's top bit
    const int in_img = min(vecs, (img - e_lo) >> 3);
    uint32_t odd = 0;
    for (int v = threadIdx.x; v < n * vecs; v += kClThreads) {
      const uint4 x = *reinterpret_cast<const uint4*>(sm + buf * kClSteps * a.slice + 16 * v);
      if (v % vecs < in_img) {
        constexpr uint32_t e = 0x7f807f80u, one = 0x00800080u;
        odd |= ((x.x & e) + one) | ((x.y & e) + one) | ((x.z & e) + one) | ((x.w & e) + one);
      }
    }
    if (!__syncthreads_or(odd & 0x80008000u)) {
      for (int s = 0; s < n; ++s) step(p0 + (uint32_t)(s * a.slice), std::false_type());
    } else {
      for (int s = 0; s < n; ++s) step(p0 + (uint32_t)(s * a.slice), std::true_type());
    }
  }
}

template <int KS, int RESET>
cudaError_t launch_conv_leaky_reset(const ConvLeakyArgs& a, unsigned grid, size_t smem, cudaStream_t st) {
  const auto kernel = conv_leaky_kernel<KS, RESET>;
  if (smem > 48 * 1024) {
    const cudaError_t e = ensure_smem((const void*)kernel, smem);
    if (e != cudaSuccess) return e;
  }
  return launch_pdl(kernel, dim3(grid), dim3(kClThreads), smem, st, a);
}

template <int KS>
cudaError_t launch_conv_leaky(const ConvLeakyArgs& a, int reset, unsigned grid, size_t smem,
                              cudaStream_t st) {
  switch (reset) {
    case RESET_SUBTRACT: return launch_conv_leaky_reset<KS, RESET_SUBTRACT>(a, grid, smem, st);
    case RESET_ZERO: return launch_conv_leaky_reset<KS, RESET_ZERO>(a, grid, smem, st);
    default: return launch_conv_leaky_reset<KS, RESET_NONE>(a, grid, smem, st);
  }
}

bool cl_al16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace
}  // namespace snn

using namespace snn;

extern "C" snn_status_t snn_conv2d_small_leaky_fwd_nhwc(
    const snn_scan_desc* d, int64_t H, int64_t W, int64_t Cin, int64_t Cout, int64_t KH, int64_t KW,
    int64_t ldw, const void* X, const void* Wt, const float* beta, const float* thr, void* spk,
    void* mem, float* ckpt, void* pool, uint8_t* idx, snn_stream_t stream) {
  if (!d || Cin < 1 || KH < 1 || KW < 1 || H < KH || W < KW || Cout < 1) return SNN_ERR_INVALID_ARG;
  if (d->T < 1 || d->B < 1 || d->reserved0 != 0 || d->reserved1 != 0) return SNN_ERR_INVALID_ARG;
  if (d->reset < SNN_RESET_SUBTRACT || d->reset > SNN_RESET_NONE) return SNN_ERR_INVALID_ARG;
  if (ldw < KH * KW * Cin || !pool != !idx) return SNN_ERR_INVALID_ARG;
  if (H > 32768 || W > 32768) return SNN_ERR_INVALID_ARG;
  const int64_t Ho = H - KH + 1, Wo = W - KW + 1;
  if (d->N != Ho * Wo * Cout) return SNN_ERR_INVALID_ARG;
  if (d->io_dtype != SNN_BF16 || d->save != SNN_SAVE_MEM) return SNN_ERR_UNSUPPORTED;
  // two output rows and an even row of pixels per group; whole 16-byte
  // pieces per image, so that every image starts on such a boundary
  if (Cin != 1 || KH != KW || (KH != 3 && KH != 5) || Cout != kClCout || Ho % 2 != 0 ||
      Wo % 2 != 0 || (H * W) % 8 != 0 || H * W > 8192)
    return SNN_ERR_UNSUPPORTED;
  if (d->T > INT_MAX / 2 || d->B > INT_MAX / 64 || d->T * d->B * d->N > ((int64_t)1 << 46))
    return SNN_ERR_INVALID_ARG;
  auto mode = [&](int32_t m, int* ch) {
    *ch = m == SNN_P_PER_CHANNEL;
    return m == SNN_P_SCALAR || (m == SNN_P_PER_CHANNEL && d->C == Cout && d->HW == 1);
  };
  ConvLeakyArgs a{};
  if (!mode(d->beta_mode, &a.beta_ch) || !mode(d->thr_mode, &a.thr_ch)) return SNN_ERR_UNSUPPORTED;
  if (!X || !Wt || !beta || !thr || !spk || !mem) return SNN_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(X) & 1u) || !cl_al16(spk) || !cl_al16(mem) || (ckpt && !cl_al16(ckpt)) ||
      (pool && (!cl_al16(pool) || !cl_al16(idx))) || (reinterpret_cast<uintptr_t>(Wt) & 1u))
    return SNN_ERR_ALIGNMENT;
  a.T = (int)d->T;
  a.H = (int)H;
  a.W = (int)W;
  a.Ho = (int)Ho;
  a.Wo = (int)Wo;
  a.ldw = (int)ldw;
  a.B = d->B;
  a.L = d->B * d->N;
  a.X = static_cast<const __nv_bfloat16*>(X);
  a.Wt = static_cast<const __nv_bfloat16*>(Wt);
  a.beta = beta;
  a.thr = thr;
  a.spk = static_cast<__nv_bfloat16*>(spk);
  a.mem = static_cast<__nv_bfloat16*>(mem);
  a.bits = reinterpret_cast<unsigned char*>(ckpt);
  a.bits_row = ((d->B * d->N + 7) / 8 + 15) / 16 * 16;
  a.pool = static_cast<__nv_bfloat16*>(pool);
  a.idx = idx;
  a.x_aligned = cl_al16(X);
  const int64_t Wp = Wo / 2, Pp = (Ho / 2) * Wp;
  const int64_t parts = (Pp + 8 * kClWarps - 1) / (8 * kClWarps);
  // image rows a block can touch: its consecutive windows span at most
  // (8*kClWarps - 1 + Wp - 1) / Wp + 1 rows of windows
  int64_t rows = 2 * ((8 * kClWarps + Wp - 2) / Wp + 1) + KH - 1;
  if (rows > H) rows = H;
  a.slice = (int)(((rows * W + 8) * 2 + 15) / 16 * 16);  // + 8 elements for the start's round-down
  size_t smem = (size_t)2 * kClSteps * a.slice;
  if (smem > 48 * 1024 || d->B * parts > INT_MAX) return SNN_ERR_UNSUPPORTED;
  if (KH == 3) smem += (size_t)(KH * KW * Cout) * sizeof(float);  // and the filters
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const unsigned grid = (unsigned)(d->B * parts);
  cudaError_t e;
  if (KH == 5) e = launch_conv_leaky<5>(a, d->reset, grid, smem, st);
  else e = launch_conv_leaky<3>(a, d->reset, grid, smem, st);
  return e == cudaSuccess ? SNN_OK : SNN_ERR_CUDA;
}
