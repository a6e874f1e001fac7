// Templated launchers for the scan kernels; each .cu file instantiates one
// family so the library compiles in parallel.
#pragma once

#include <type_traits>

#include "scan_host.cuh"

namespace snn {

// dtype pairs (input, io) whose staged backward gets loops specialised on
// the reset mode and surrogate; other pairs use the run-time-mode loop.
template <typename TI, typename TO>
constexpr bool kSpecialise =
    (std::is_same<TI, float>::value && std::is_same<TO, float>::value) ||
    (std::is_same<TI, __nv_bfloat16>::value && std::is_same<TO, __nv_bfloat16>::value) ||
    (std::is_same<TI, float>::value && std::is_same<TO, __nv_bfloat16>::value);

// Few lanes for the GPU: with 8 lanes a thread, an SM would hold fewer than
// about 8 warps.
inline bool few_lanes(int64_t L) {
  DeviceInfo d;
  return device_info(&d) == cudaSuccess && L < 2048 * (int64_t)d.sms;
}

// Lanes of the plain kernels from which other warps hide a load (see there).
inline bool many_lanes(int64_t L) {
  DeviceInfo d;
  return device_info(&d) == cudaSuccess && L >= kPlainManyLanes * (int64_t)d.sms;
}

template <bool SYN, typename TI, typename TO, int RESET, bool REC, int VL, bool CK>
cudaError_t fwd_staged_ck(ScanArgs a, cudaStream_t st, bool* launched) {
  const void* k = (const void*)scan_fwd_staged<SYN, TI, TO, RESET, REC, VL, CK>;
  StagedPlan p;
  // a stage holds kFwdRows steps of the strip's input row; one CTA per SM
  // where it fits (the longer rows stream faster), two for short sequences
  // (T <= 64: a CTA's few stages fill and drain while the SM's other CTA
  // computes; measured 2-4% faster at T = 25, 0.5% slower at T = 500)
  if (!plan_staged(k, a.L, ceil_div(a.T, kFwdRows), kFwdRows * (int)sizeof(TI), 0, VL, &p, 0, 0,
                   a.T <= 64 ? 2 : 1))
    return cudaSuccess;
  a.lanes_per_cta = p.lanes_per_cta;
  a.stages = p.stages;
  a.stage_bytes = p.stage_bytes;
  *launched = true;
  return launch_pdl(scan_fwd_staged<SYN, TI, TO, RESET, REC, VL, CK>, dim3((unsigned)p.grid),
                    dim3(p.threads), p.smem, st, a);
}

template <bool SYN, typename TI, typename TO, int RESET, bool REC, int VL>
cudaError_t fwd_staged_vl(ScanArgs a, cudaStream_t st, bool* launched) {
  return a.ckpt ? fwd_staged_ck<SYN, TI, TO, RESET, REC, VL, true>(a, st, launched)
                : fwd_staged_ck<SYN, TI, TO, RESET, REC, VL, false>(a, st, launched);
}

// 4 lanes a thread instead of 8 (Leaky) with few lanes, which then make more
// warps (T = 64, 128 x 1000 lanes in bf16: 9.4 us against 12.9; T = 100, 64 x
// 4096: 20% faster), and for short sequences of fp32 currents (T = 25, 128 x
// 6912 lanes: 43.9 us against 55.2).  Longer ones are better with 8 (T = 500,
// 64 x 8192 lanes, store mode: 9% faster), and so are many lanes of short half
// sequences (T = 10, 6.7 M lanes, recompute: 60.8 us against 68.8).  CTAs that
// walk several strips with one ring were up to a fifth faster around 0.5 M
// lanes (T = 25, fp32 recompute: 16.5 us against 20.1) but slower for many
// (T = 1, 67 M lanes in bf16: 636 us against 291; T = 25, 128 x 6912 Synaptic
// lanes: 64.5 against 58.8), so a CTA takes one.
template <bool SYN, typename TI, typename TO, int RESET, bool REC = false>
cudaError_t fwd_staged(ScanArgs a, cudaStream_t st, bool* launched) {
  if constexpr (!SYN)
    if (few_lanes(a.L) || (a.T <= 64 && sizeof(TI) == 4))
      return fwd_staged_vl<SYN, TI, TO, RESET, REC, 4>(a, st, launched);
  return fwd_staged_vl<SYN, TI, TO, RESET, REC, kLanes<SYN>>(a, st, launched);
}

template <bool SYN, typename TI, typename TO, int RESET, int REC>
cudaError_t fwd_plain(ScanArgs a, cudaStream_t st) {
  return launch_pdl(scan_fwd_plain<SYN, TI, TO, RESET, REC>, dim3((unsigned)ceil_div(a.L, 128)), dim3(128),
                    0, st, a);
}

template <bool SYN, typename TI, typename TO>
cudaError_t fwd_t(ScanArgs a, bool staged, cudaStream_t st) {
  if (staged && a.L > 0) {
    bool launched = false;
    cudaError_t e;
    if (!SYN && a.rec) e = fwd_staged<false, TI, TO, RESET_SUBTRACT, true>(a, st, &launched);
    else if (a.reset == RESET_SUBTRACT) e = fwd_staged<SYN, TI, TO, RESET_SUBTRACT>(a, st, &launched);
    else if (a.reset == RESET_ZERO) e = fwd_staged<SYN, TI, TO, RESET_ZERO>(a, st, &launched);
    else e = fwd_staged<SYN, TI, TO, -1>(a, st, &launched);
    if (launched || e != cudaSuccess) return e;
  }
  if (a.L == 0) return cudaSuccess;
  if constexpr (!SYN)
    if (a.rec) return fwd_plain<SYN, TI, TO, RESET_SUBTRACT, 1>(a, st);
  if (a.reset == RESET_SUBTRACT) return fwd_plain<SYN, TI, TO, RESET_SUBTRACT, 0>(a, st);
  if (a.reset == RESET_ZERO) return fwd_plain<SYN, TI, TO, RESET_ZERO, 0>(a, st);
  return fwd_plain<SYN, TI, TO, RESET_NONE, 0>(a, st);
}

template <bool SYN, bool RECOMP, typename TI, typename TO, int RESET, int SG, int KC, bool REC,
          int VL>
cudaError_t bwd_staged_vl(ScanArgs a, cudaStream_t st, bool* launched) {
  const void* k = (const void*)scan_bwd_staged<SYN, RECOMP, TI, TO, RESET, SG, KC, REC, VL>;
  int per_lane, seg, fixed;
  int64_t items;
  if (RECOMP) {
    const int fwd_item = (int)sizeof(TI);
    const int bwd_item = (int)sizeof(TO) * (a.gm ? 2 : 1);
    per_lane = fwd_item > bwd_item ? fwd_item : bwd_item;
    seg = kLanes<SYN> * 4 * a.K * (SYN ? 2 : 1);
    fixed = 2 * 4 * (SYN ? 2 : 1);  // two checkpoint slots
    items = 2 * a.T;
  } else {
    const int n = 2 + (sizeof(TO) != 4 ? 1 : 0) + ((SYN && a.part_alpha) ? 1 : 0) + (a.gm ? 1 : 0);
    per_lane = kBwdRows * n * (int)sizeof(TO);
    seg = 0;
    fixed = 0;
    items = ceil_div(a.T, kBwdRows);
  }
  StagedPlan p;
  // Short store-mode sequences may have a ring of two items (8 steps): asking
  // for three made their strips narrower than the lanes of one wave, and the
  // second wave cost more than the third item gives (us, T = 13, per-neuron
  // parameters: 262,144 fp32 Synaptic lanes 18.8 -> 15.0, 524,288 fp32 Leaky
  // lanes 22.7 -> 20.1; 4 M bf16 Leaky lanes 78 -> 82)
  const int ring = !RECOMP && a.T <= 64 ? 2 : 3;
  if (!plan_staged(k, a.L, items, per_lane, seg, VL, &p, fixed, KC, 2, part_align(a), ring)) return cudaSuccess;
  choose_parts(a, p, VL);
  a.lanes_per_cta = p.lanes_per_cta;
  a.stages = p.stages;
  a.stage_bytes = p.stage_bytes;
  *launched = true;
  return launch_pdl(scan_bwd_staged<SYN, RECOMP, TI, TO, RESET, SG, KC, REC, VL>,
                    dim3((unsigned)p.grid), dim3(p.threads), p.smem, st, a);
}

// The staged backward with its lanes per thread: 4 for the Leaky neuron's
// store mode on sequences of at most 64 steps or with few lanes, else kLanes.
template <bool SYN, bool RECOMP, typename TI, typename TO, int RESET, int SG, int KC = 0,
          bool REC = false>
cudaError_t bwd_staged(ScanArgs a, cudaStream_t st, bool* launched) {
  if constexpr (!SYN && !RECOMP) {
    if (a.T <= 64 || few_lanes(a.L))
      return bwd_staged_vl<SYN, RECOMP, TI, TO, RESET, SG, KC, REC, 4>(a, st, launched);
  }
  return bwd_staged_vl<SYN, RECOMP, TI, TO, RESET, SG, KC, REC, kLanes<SYN>>(a, st, launched);
}

template <bool SYN, bool RECOMP, typename TI, typename TO, int RESET, int SG, int REC, int AHEAD>
cudaError_t bwd_plain_ahead(ScanArgs a, cudaStream_t st) {
  const int threads = 128;
  const size_t smem = RECOMP ? (size_t)a.K * threads * 4 * (SYN ? 2 : 1) : 0;
  const auto kernel = scan_bwd_plain<SYN, RECOMP, TI, TO, RESET, SG, REC, AHEAD>;
  const cudaError_t e = ensure_smem((const void*)kernel, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kernel, dim3((unsigned)ceil_div(a.L, threads)), dim3(threads), smem, st, a);
}

template <bool SYN, bool RECOMP, typename TI, typename TO, int RESET, int SG, int REC>
cudaError_t bwd_plain(ScanArgs a, cudaStream_t st) {
  constexpr int few = RECOMP ? kPlainAheadSeg : kPlainAhead;
  constexpr int many = RECOMP ? kPlainAheadSegMany : kPlainAheadMany;
  return many_lanes(a.L) ? bwd_plain_ahead<SYN, RECOMP, TI, TO, RESET, SG, REC, many>(a, st)
                         : bwd_plain_ahead<SYN, RECOMP, TI, TO, RESET, SG, REC, few>(a, st);
}

template <bool SYN, bool RECOMP, typename TI, typename TO>
cudaError_t bwd_t(ScanArgs a, bool staged, cudaStream_t st) {
  if (staged && a.L > 0) {
    bool launched = false;
    cudaError_t e = cudaSuccess;
    bool done = false;
    if (!SYN && a.rec) {  // recurrent Leaky neuron: reset by subtraction (Eq. 7)
      if constexpr (kSpecialise<TI, TO>) {
        if (a.sg == SG_ATAN)
          e = bwd_staged<false, RECOMP, TI, TO, RESET_SUBTRACT, SG_ATAN, 0, true>(a, st, &launched);
        else
          e = bwd_staged<false, RECOMP, TI, TO, RESET_SUBTRACT, SG_FAST_SIGMOID, 0, true>(a, st,
                                                                                      &launched);
      } else {
        e = bwd_staged<false, RECOMP, TI, TO, RESET_SUBTRACT, -1, 0, true>(a, st, &launched);
      }
      done = true;
    } else if constexpr (kSpecialise<TI, TO>) {
      done = true;
      const int key = (a.reset == RESET_NONE ? 9 : a.reset * 2 + a.sg);
      // the recompute variant with the default checkpoint interval K = 8
      // also has a fully unrolled segment body (ring of exactly 8 stages)
      const bool k8 = RECOMP && a.K == 8;
      switch (key) {
        case 0:
          if (k8) e = bwd_staged<SYN, RECOMP, TI, TO, RESET_SUBTRACT, SG_FAST_SIGMOID, 8>(a, st, &launched);
          if (!launched && e == cudaSuccess)
            e = bwd_staged<SYN, RECOMP, TI, TO, RESET_SUBTRACT, SG_FAST_SIGMOID>(a, st, &launched);
          break;
        case 1:
          if (k8) e = bwd_staged<SYN, RECOMP, TI, TO, RESET_SUBTRACT, SG_ATAN, 8>(a, st, &launched);
          if (!launched && e == cudaSuccess)
            e = bwd_staged<SYN, RECOMP, TI, TO, RESET_SUBTRACT, SG_ATAN>(a, st, &launched);
          break;
        case 2: e = bwd_staged<SYN, RECOMP, TI, TO, RESET_ZERO, SG_FAST_SIGMOID>(a, st, &launched); break;
        case 3: e = bwd_staged<SYN, RECOMP, TI, TO, RESET_ZERO, SG_ATAN>(a, st, &launched); break;
        default: done = false;
      }
    }
    if (!done) e = bwd_staged<SYN, RECOMP, TI, TO, -1, -1>(a, st, &launched);
    if (launched || e != cudaSuccess) return e;
  }
  if (a.L == 0) return cudaSuccess;
  // the modes of a ragged layer: a warp has a scheduler nearly to itself, so
  // every instruction of a step shows; run-time modes only for the mixed
  // input and storage types and for no reset
  if constexpr (std::is_same<TI, TO>::value) {
    const bool atan = a.sg == SG_ATAN;
    if constexpr (!SYN)
      if (a.rec)
        return atan ? bwd_plain<SYN, RECOMP, TI, TO, RESET_SUBTRACT, SG_ATAN, 1>(a, st)
                    : bwd_plain<SYN, RECOMP, TI, TO, RESET_SUBTRACT, SG_FAST_SIGMOID, 1>(a, st);
    if (a.reset == RESET_SUBTRACT)
      return atan ? bwd_plain<SYN, RECOMP, TI, TO, RESET_SUBTRACT, SG_ATAN, 0>(a, st)
                  : bwd_plain<SYN, RECOMP, TI, TO, RESET_SUBTRACT, SG_FAST_SIGMOID, 0>(a, st);
    if (a.reset == RESET_ZERO)
      return atan ? bwd_plain<SYN, RECOMP, TI, TO, RESET_ZERO, SG_ATAN, 0>(a, st)
                  : bwd_plain<SYN, RECOMP, TI, TO, RESET_ZERO, SG_FAST_SIGMOID, 0>(a, st);
  }
  return bwd_plain<SYN, RECOMP, TI, TO, -1, -1, -1>(a, st);
}

// dtype codes (snn_dtype_t): 0 f32, 1 bf16, 2 f16.  Instantiated pairs
// (in, io): (f32,f32) (bf16,bf16) (f16,f16) (f32,bf16) (f32,f16).
#define SNN_DTYPE_DISPATCH(IN_DT, IO_DT, CALL)                                   \
  do {                                                                           \
    if ((IN_DT) == 0 && (IO_DT) == 0) { using TI = float; using TO = float; CALL; } \
    if ((IN_DT) == 1 && (IO_DT) == 1) { using TI = __nv_bfloat16; using TO = __nv_bfloat16; CALL; } \
    if ((IN_DT) == 2 && (IO_DT) == 2) { using TI = __half; using TO = __half; CALL; } \
    if ((IN_DT) == 0 && (IO_DT) == 1) { using TI = float; using TO = __nv_bfloat16; CALL; } \
    if ((IN_DT) == 0 && (IO_DT) == 2) { using TI = float; using TO = __half; CALL; } \
    return cudaErrorNotSupported;                                                \
  } while (0)

}  // namespace snn
