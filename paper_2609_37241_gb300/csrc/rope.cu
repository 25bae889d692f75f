// rope.cu -- RoPE on q/k with KV-cache append, optionally after per-head q/k RMSNorm.
//
// Work unit: one head-row (token t, head hh) of D elements; per token there are
// NH = Hq + 2*Hkv of them (q heads, k heads, v heads). The vector kernels give a warp an item
// of consecutive head-rows of one token (RopeGeom, rope_pair_rows in device_common.cuh): D / 16
// lanes per head-row, each lane holding both halves of its rotated pairs, so that a rotation
// needs no exchange between lanes and a token's angles are computed once per lane and item.
// Four entries, by the call's size (rope_plan): one head-row per lane group, for heads of 64 also in
// larger blocks, two where it pays, and for calls of many tokens three, staged in shared memory by
// cp.async.bulk (rope_bulk_kernel). Other head sizes that are multiples of 16 take rope_any_kernel,
// the same with lanes left over; the generic kernel gives each head-row one warp and scalar
// accesses (any alignment, any even D). All compute (cos, sin) of pos * theta^(-2i/D) in the kernel
// from the version's double-float frequency table [D/2], which the host splits from fp64 at
// registration.
//
// Bound: HBM at prefill sizes, launch and memory latency at decode sizes. Before, a lane held
// one vector of a head-row and exchanged its partner by eight shuffles, and each of the two
// lanes of a pair computed the pair's sines and cosines: issue-bound (72 % SM throughput by
// ncu at 3333 tokens with q/k norm, 0.45 of the 6.8 TB/s copy rate). Llama head counts
// (32 + 8 + 8 of D 128), device time per call, before -> now, with q/k norm / without:
//   30 tokens    3.36 -> 2.06 / 2.95 -> 1.91 us      500 tokens    7.66 -> 4.67 / 6.86 -> 4.20 us
//   120 tokens   3.58 -> 3.01 / 3.18 -> 2.77 us     3333 tokens   26.5 -> 15.1 / 20.8 -> 13.7 us
//   250 tokens   5.13 -> 3.22 / 4.48 -> 3.04 us     8192 tokens   51.7 -> 33.3 / 41.8 -> 30.9 us
// (8192 tokens without the norm: 0.91-0.96 of the copy rate.)
#include "device_common.cuh"

namespace trident {

// One head-row per lane group (small entry) or two (mid), by the call's one-row items per SM. Up
// to three the call is one memory round trip, and a second row only lengthens it; on long calls
// two rows halve the warps that fetch the same frequency and weight lines (60 tokens of 32 + 8 + 8
// heads, D 128, with q/k norm 2.33 us against 2.62, 500 tokens 4.67 / 5.51). In between the lines are
// measured, not derived: launches of the same call back to back go in steps of about 0.8 us, one more
// where a grid no longer starts within the one before it, and each form steps at sizes of its own.
// Heads of 128 and 256, with q/k norm: two rows from 4.5 to 6 items per SM (75 tokens of 32 + 8 + 8 2.40 /
// 2.66) and from 27 (400 tokens 4.36 / 4.59), one row elsewhere: 45 tokens 2.25 -> 2.05 us, 90 3.32 -> 2.73,
// 140 3.39 -> 2.62, 225 3.66 -> 3.33, 28 + 4 + 4 heads at 150 3.77 -> 2.89. Without the norm one row from 10.5
// to 12 and from 13 to 15 items: 28 head-rows (20 + 4 + 4) at 240 / 257 tokens 2.87 / 2.87 -> 2.33 / 2.35, 180
// tokens of 48 2.87 -> 2.47, D 256 at 130 2.87 -> 2.46; between those, 28 head-rows at 264 tokens (12.2) 2.84 /
// 3.31, and outside, 105 tokens of 48 (8.3) 2.04 / 2.80, 320 (25) 3.55 / 4.08. (As one of a layer's four
// single-op launches two rows win there too, mean per launch 144 / 176 tokens of 32 + 8 + 8 2.37 / 2.56 us, one
// row 2.77 / 2.99.)
// Heads of 64, half the bytes per item, by the blocks of two-row items, and one row in larger blocks
// beyond them: without the norm two rows up to 2.28 blocks per SM (230 / 240 tokens of 32 + 8 + 8 2.06 / 2.85),
// then one in 64 threads up to 8 items (400 of 16 + 4 + 4 2.20 / 2.72), in 128 from 10.9 to 12 (300 of 32 + 8 + 8
// 2.26, in 256 2.68, two rows 2.91) and in 256 up to 24 (250 / 320 / 400 of 32 + 8 + 8 2.42 / 2.59 / 2.32 against
// 2.87 / 2.87 / 2.83); with it two rows from 4.5 items to 1.72 blocks per SM (150 of 32 + 8 + 8 2.38 / 2.88; 260
// of 16 + 4 + 4 2.31 / 2.76, 280 3.19 / 2.79), then one in 128 threads up to one wave of them, 32 items (300 of
// 32 + 8 + 8 2.95, in 64 threads 3.08, two rows 3.29).
constexpr int kRopeThreads = 64;     // block of the small and mid entries (128: the same within 3 %)
constexpr int kRopeMaxThreads = 256;
struct RopeChoice { bool two; int32_t threads; };
static RopeChoice rope_choice(int64_t one, int64_t two, int32_t D, bool qk, int64_t sms) {  // items with one and two rows
  const int64_t n = 2 * one;  // in half items
  if (n <= 6 * sms) return {false, 64};
  if (D > 64) {
    const bool small = qk ? n <= 54 * sms && !(n > 9 * sms && n <= 12 * sms)
                          : (n > 21 * sms && n <= 24 * sms) || (n > 26 * sms && n <= 30 * sms);
    return {!small, 64};
  }
  const int64_t blocks = (two + 1) / 2;
  if (qk) {
    if (n <= 9 * sms) return {false, 64};
    if (100 * blocks <= 172 * sms || one > 32 * sms) return {true, 64};
    return {false, 128};
  }
  if (100 * blocks <= 228 * sms || one > 24 * sms) return {true, 64};
  if (one <= 8 * sms) return {false, 64};
  return {false, 10 * one > 109 * sms && one <= 12 * sms ? 128 : 256};
}
// Calls of at least this many tokens and bulk items take the bulk-copy entry: 640 tokens (2560
// items) with q/k norm 5.06 us against 5.80 with two register-held rows per group, 2048 tokens
// 10.5 / 8.9 (with / without the norm) against 12.3 / 10.5, 8192 33.3 / 30.9 against 38.0 / 32.8.
// With fewer items, the same tokens of few heads, a warp's serial copy, rotate and store is the
// call: 8 + 2 + 2 heads at 700 / 1600 tokens 4.53 / 5.22 against 2.85 (one row) / 4.61.
constexpr int32_t kRopeBulkTokens = 512;
constexpr int64_t kRopeBulkItems = 2304;

// Before the launch wait: the lane's frequencies (the version's table is written only at
// registration; with p.freq_late the previous kernel writes it, and they are read after), and with
// p.prefetch the L2 prefetch of the item's row lines and position.
// NT: the largest block; blocks of more than 64 threads at most four per SM of 256 (more resident ones
// take the SM from the launch before: 300 tokens of 32 + 8 + 8 heads of D 64 2.26 us, without the limit 2.66).
template <int DT, int D, bool QKNORM, int R, int NT>
__global__ void __launch_bounds__(NT, NT == kRopeThreads ? 0 : 4) rope_pair_kernel(const RopeParams p) {
  pdl_trigger();
  int64_t t;
  int first, end;
  const int64_t item = (int64_t)blockIdx.x * ((NT == kRopeThreads ? NT : blockDim.x) / 32) + threadIdx.x / 32;
  const bool live = rope_item(p, item, &t, &first, &end);
  float4 fq[4];
  if (!p.freq_late) rope_pair_freqs(p.inv_freq, (threadIdx.x & 31) % RopeGeom<D>::LPG, fq);
  if (p.prefetch && live) rope_item_prefetch<D, R>(p, t, first, end);
  pdl_wait();
  if (p.freq_late) rope_pair_freqs_late(p.inv_freq, (threadIdx.x & 31) % RopeGeom<D>::LPG, fq);
  if (live) rope_pair_rows<DT, D, QKNORM, R, true>(p, t, first, end, fq);
}

// Calls of many tokens: a warp's item is three head-rows per lane group (3 KB), staged in the
// warp's own shared memory by bulk copies (cp.async.bulk: an item's q, k and v rows are each
// contiguous, so one to three copies) on the warp's own mbarrier; meanwhile the lanes compute
// the token's angles, once per item. No block barrier: each warp waits for its own copies,
// rotates its rows out of shared memory and stores them. Staged rows take no registers, so 24
// warps of 3 KB are in flight per SM. Other shapes measured at 3333 tokens (q/k norm): this one
// 15.1 us; 6 rows per group 15.4; 12 rows 17.8-18.3; 8 blocks per SM (spills) 16.4; three
// register-held rows 17.0; the former two tokens per block behind a block barrier 26.5.
//
// The wait is bounded (bp.first_wait_polls try_wait polls, kBulkWaitPolls by default): a warp
// whose copies have not landed by then sets TRIDENT_DEVERR_TIMEOUT, waits (again bounded) for
// them and returns without writing.
constexpr int kRopeBulkRows = 3;      // head-rows per lane group
constexpr int kRopeBulkThreads = 128;

template <int DT, int D, bool QKNORM>
__global__ void __launch_bounds__(kRopeBulkThreads, 6) rope_bulk_kernel(const RopeBulkParams bp) {
  const RopeParams& p = bp.rp;
  constexpr int LPG = RopeGeom<D>::LPG, GW = RopeGeom<D>::GW, RB = D * 2;
  __shared__ __align__(128) char s_rows[kRopeBulkThreads / 32][kRopeBulkRows * GW * RB];
  __shared__ __align__(8) unsigned long long s_bar[kRopeBulkThreads / 32];
  const int w = threadIdx.x / 32, lane = (threadIdx.x & 31) % LPG;
  const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&s_bar[w]);
  if ((threadIdx.x & 31) == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();  // the barrier is initialised before any lane waits on it
  pdl_trigger();
  int64_t t;
  int first, end;
  const bool live = rope_item(p, (int64_t)blockIdx.x * (kRopeBulkThreads / 32) + w, &t, &first, &end);
  pdl_wait();
  if (!live) return;
  if ((threadIdx.x & 31) == 0) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                 :: "r"(bar), "r"((uint32_t)((end - first) * RB)) : "memory");
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(s_rows[w]);
    int h = first;
    const int upto[3] = {min(end, p.Hq), min(end, p.Hq + p.Hkv), end};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (h < upto[k]) {
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     :: "r"(dst + (uint32_t)((h - first) * RB)), "l"(rope_row_src<D>(p, t, h)),
                        "r"((uint32_t)((upto[k] - h) * RB)), "r"(bar) : "memory");
        h = upto[k];
      }
    }
  }
  const int32_t pos = __ldg(p.pos + t);
  const bool pos_ok = pos >= 0 && (int64_t)pos < p.S;
  RopeAngles an;
  {
    float4 fq[4];
    rope_pair_freqs_late(p.inv_freq, lane, fq);
    rope_angles(pos_ok ? pos : 0, fq, &an);
  }
  auto landed = [&](uint32_t polls) -> bool {
    uint32_t done = 0;
    for (uint32_t it = 0; it < polls && !done; ++it)
      asm volatile("{ .reg .pred q; mbarrier.try_wait.parity.shared::cta.b64 q, [%1], 0; selp.u32 %0, 1, 0, q; }"
                   : "=r"(done) : "r"(bar) : "memory");
    return done != 0;
  };
  const bool ok = landed(bp.first_wait_polls);
  if (__any_sync(0xffffffffu, !ok)) {  // one decision for the whole warp
    if ((threadIdx.x & 31) == 0) atomicOr(p.err, kErrTimeout);
    if (!ok) landed(kBulkWaitPolls);  // a second bounded wait for the copies before the warp exits
    return;
  }
  if (!pos_ok) {
    if ((threadIdx.x & 31) == 0) atomicOr(p.err, kErrPos);
    return;
  }
  RopeGamma g;
  int kind = 0;
  const int hh0 = first + (threadIdx.x & 31) / LPG;
#pragma unroll
  for (int j = 0; j < kRopeBulkRows; ++j) {
    const int hh = hh0 + j * GW;
    if (hh >= end) break;
    const char* row = s_rows[w] + (hh - first) * RB + lane * 16;
    rope_pair_finish<DT, D, QKNORM, true>(p, t, hh, lane, pos, ld16(row), ld16(row + D), an, &g, &kind);
  }
}

// Head sizes without a kernel of their own, and versions that promise no alignment, when a call's
// tensors are 16-byte aligned and D is a multiple of 16 of at most 256: the pair layout with LPG
// lanes per head-row, D / 16 of them holding part of it.
template <int DT, int LPG, bool QKNORM, int R>
__global__ void __launch_bounds__(kRopeThreads) rope_any_kernel(const RopeParams p) {
  pdl_prologue();
  constexpr int GW = 32 / LPG;
  const int D = p.D, l = (threadIdx.x & 31) % LPG, lane = min(l, D / 16 - 1);
  const bool on = l == lane;
  int64_t t;
  int first, end;
  if (!rope_item(p, (int64_t)blockIdx.x * (kRopeThreads / 32) + threadIdx.x / 32, &t, &first, &end)) return;
  const int hh0 = first + (threadIdx.x & 31) / LPG;
  uint4 lo[R], hi[R];
#pragma unroll
  for (int j = 0; j < R; ++j) {  // groups past the item's end load its last row and drop it
    const char* src = rope_row_src(p, t, min(hh0 + j * GW, end - 1), D) + lane * 16;
    lo[j] = ld16(src);
    hi[j] = ld16(src + D);
  }
  const int32_t pos = __ldg(p.pos + t);
  if (pos < 0 || (int64_t)pos >= p.S) {
    if ((threadIdx.x & 31) == 0) atomicOr(p.err, kErrPos);
    return;
  }
  float4 fq[4];
  rope_pair_freqs(p.inv_freq, lane, fq);
  RopeAngles an;
  rope_angles(pos, fq, &an);
#pragma unroll
  for (int j = 0; j < R; ++j) {
    const int hh = hh0 + j * GW;
    if (hh >= end) break;
    char* dst = rope_row_dst(p, t, hh, pos, D) + lane * 16;
    if (hh >= p.Hq + p.Hkv) {  // bit copy into the cache
      if (on) {
        st16(dst, lo[j]);
        st16(dst + D, hi[j]);
      }
      continue;
    }
    F2 A[4], B[4];
    rope_unpack<DT>(lo[j], hi[j], A, B);
    if (QKNORM) {
      RopeGamma g;
      rope_pair_gamma(hh < p.Hq ? p.gamma_q : p.gamma_k, lane, D, &g);
      rope_scale(rope_inv_rms<LPG>(p, A, B, on), g, A, B);
    }
    if (on) rope_rotate<DT>(dst, D, an, A, B);
  }
}

template <int DT, bool QKNORM>
__global__ void __launch_bounds__(kThreads) rope_generic_kernel(const RopeParams p) {
  pdl_prologue();
  const int lane = threadIdx.x & 31;
  const int64_t total = p.T * p.NH;
  const int64_t nwarps = (int64_t)gridDim.x * (kThreads / 32);
  const int half = p.D / 2;
  for (int64_t unit = ((int64_t)blockIdx.x * kThreads + threadIdx.x) / 32; unit < total;
       unit += nwarps) {
    const int64_t t = unit / p.NH;
    const int hh = (int)(unit - t * p.NH);
    const int32_t pos = p.pos[t];
    if (pos < 0 || (int64_t)pos >= p.S) {
      if (lane == 0) atomicOr(p.err, kErrPos);
      continue;
    }
    if (hh >= p.Hq + p.Hkv) {
      const int h = hh - p.Hq - p.Hkv;
      const int64_t so = t * p.v_rs + (int64_t)h * p.D;
      const int64_t dst = ((int64_t)h * p.S + pos) * p.D;
      const uint16_t* vs = reinterpret_cast<const uint16_t*>(p.v);  // bit copy (2-byte types)
      uint16_t* vd = reinterpret_cast<uint16_t*>(p.v_cache);
      for (int j = lane; j < p.D; j += 32) vd[dst + j] = vs[so + j];
      continue;
    }
    const bool is_q = hh < p.Hq;
    const int h = is_q ? hh : hh - p.Hq;
    const void* src = is_q ? (const void*)p.q : p.k;
    const int64_t so = t * (is_q ? p.q_rs : p.k_rs) + (int64_t)h * p.D;
    const float* gam = is_q ? p.gamma_q : p.gamma_k;
    float inv = 1.f;
    if (QKNORM) {
      float ss = 0.f;
      for (int j = lane; j < p.D; j += 32) {
        const float v = load_elem<DT>(src, so + j);
        ss = fmaf(v, v, ss);
      }
      inv = rsqrtf(warp_sum(ss) * p.inv_D + p.eps);
    }
    for (int i = lane; i < half; i += 32) {
      float lo = load_elem<DT>(src, so + i), hi = load_elem<DT>(src, so + i + half);
      if (QKNORM) {
        lo = lo * inv * gam[i];
        hi = hi * inv * gam[i + half];
      }
      const float2 f = p.inv_freq[i];
      float sn, cs;
      rope_sincos((float)pos, f.x, f.y, &sn, &cs);
      const float ylo = fmaf(lo, cs, -hi * sn);
      const float yhi = fmaf(hi, cs, lo * sn);
      if (is_q) {
        store_elem<DT>(p.q, so + i, ylo);
        store_elem<DT>(p.q, so + i + half, yhi);
      } else {
        const int64_t dst = ((int64_t)h * p.S + pos) * p.D;
        store_elem<DT>(p.k_cache, dst + i, ylo);
        store_elem<DT>(p.k_cache, dst + i + half, yhi);
      }
    }
  }
}

static int rope_any_lanes(int32_t D) {  // 0: no such kernel
  if (D < 32 || D > 256 || D % 16 != 0) return 0;
  return D <= 64 ? 4 : D <= 128 ? 8 : 16;
}

void rope_plans(int64_t NH, int32_t D, RopePlans* out) {
  if (const int lanes = rope_any_lanes(D)) {
    out->any[0] = rope_split(NH, 32 / lanes, 1);
    out->any[1] = rope_split(NH, 32 / lanes, 3);
  }
  if (D != 64 && D != 128 && D != 256) return;
  out->split[ROPE_SMALL] = out->split[ROPE_BLOCKS] = rope_split(NH, 512 / D, 1);
  out->split[ROPE_MID] = rope_split(NH, 512 / D, 2);
  out->split[ROPE_BULK] = rope_split(NH, 512 / D, kRopeBulkRows);
}

RopeEntry rope_plan(const RopePlans& plans, RopeParams* p, int32_t* threads, int64_t* blocks, int32_t sms) {
  RopeEntry e = ROPE_BULK;
  *threads = kRopeBulkThreads;
  if (p->T < kRopeBulkTokens || p->T * plans.split[ROPE_BULK].ipt < kRopeBulkItems) {
    const RopeChoice c = rope_choice(p->T * plans.split[ROPE_SMALL].ipt, p->T * plans.split[ROPE_MID].ipt, p->D,
                                     p->gamma_q != nullptr, sms);
    e = c.two ? ROPE_MID : c.threads > kRopeThreads ? ROPE_BLOCKS : ROPE_SMALL;
    *threads = c.threads;
  }
  const RopeSplit& r = plans.split[e];
  p->ipt = r.ipt;
  p->rpi = r.rpi;
  p->ipt_magic = r.magic;
  p->ipt_shift = r.shift;
  *blocks = (p->T * r.ipt + *threads / 32 - 1) / (*threads / 32);
  return e;
}

// The rope_any_kernel entry of a call of a version without an aligned kernel, or -1: one row per
// lane group below about three items per SM, three from there. D 96, 32 + 8 + 8 heads, against
// the generic kernel, with q/k norm / without: 20 tokens 3.50 -> 2.31 / 2.44 -> 2.01 us, 3000
// tokens 55.7 -> 14.6 / 41.4 -> 10.9; D 160, 16 + 8 + 8 heads with the norm 40.5 -> 18.5.
int rope_any_plan(const RopePlans& plans, RopeParams* p, int32_t* threads, int64_t* blocks, int32_t sms) {
  if (plans.any[0].ipt == 0) return -1;
  const uintptr_t ptrs = (uintptr_t)p->q | (uintptr_t)p->k | (uintptr_t)p->v | (uintptr_t)p->k_cache |
                         (uintptr_t)p->v_cache | (uintptr_t)p->gamma_q | (uintptr_t)p->gamma_k;
  if (ptrs % 16 != 0 || (p->T > 1 && (p->q_rs % 8 != 0 || p->k_rs % 8 != 0 || p->v_rs % 8 != 0))) return -1;
  const int e = p->T * plans.any[0].ipt > 3 * (int64_t)sms ? 1 : 0;
  const RopeSplit& r = plans.any[e];
  p->ipt = r.ipt;
  p->rpi = r.rpi;
  p->ipt_magic = r.magic;
  p->ipt_shift = r.shift;
  *threads = kRopeThreads;
  *blocks = (p->T * r.ipt + kRopeThreads / 32 - 1) / (kRopeThreads / 32);
  return e;
}

template <int DT, bool QK>
static void pick_any(int32_t D, KernelEntry* out) {
  const int lanes = rope_any_lanes(D);
  if (lanes == 4) {
    out->any_fn[0] = (const void*)rope_any_kernel<DT, 4, QK, 1>;
    out->any_fn[1] = (const void*)rope_any_kernel<DT, 4, QK, 3>;
  } else if (lanes == 8) {
    out->any_fn[0] = (const void*)rope_any_kernel<DT, 8, QK, 1>;
    out->any_fn[1] = (const void*)rope_any_kernel<DT, 8, QK, 3>;
  } else if (lanes == 16) {
    out->any_fn[0] = (const void*)rope_any_kernel<DT, 16, QK, 1>;
    out->any_fn[1] = (const void*)rope_any_kernel<DT, 16, QK, 3>;
  }
}

template <int DT, bool QK, int D>
static void pick_d(KernelEntry* out) {
  out->fn = (const void*)rope_pair_kernel<DT, D, QK, 1, kRopeThreads>;
  if constexpr (D == 64) out->fn_blocks = (const void*)rope_pair_kernel<DT, D, QK, 1, kRopeMaxThreads>;
  out->fn_mid = (const void*)rope_pair_kernel<DT, D, QK, 2, kRopeThreads>;
  out->fn_large = (const void*)rope_bulk_kernel<DT, D, QK>;
}

template <int DT, bool QK>
static void pick_vec(int32_t D, KernelEntry* out) {
  if (D == 64) pick_d<DT, QK, 64>(out);
  else if (D == 128) pick_d<DT, QK, 128>(out);
  else if (D == 256) pick_d<DT, QK, 256>(out);
}

bool rope_kernel(int32_t dtype, int32_t variant, int32_t D, bool qknorm, KernelEntry* out,
                 const char** why) {
  if (dtype != DT_BF16 && dtype != DT_FP16) { *why = "RoPE supports bf16 and fp16"; return false; }
  if (D < 2 || D % 2 != 0) { *why = "head size D must be even"; return false; }
  if (variant == 1) {  // GENERIC
    out->kind = KK_ROPE_WARP;
    if (dtype == DT_BF16) qknorm ? pick_any<DT_BF16, true>(D, out) : pick_any<DT_BF16, false>(D, out);
    else qknorm ? pick_any<DT_FP16, true>(D, out) : pick_any<DT_FP16, false>(D, out);
    out->vec = 1;
    if (dtype == DT_BF16) out->fn = qknorm ? (const void*)rope_generic_kernel<DT_BF16, true>
                                           : (const void*)rope_generic_kernel<DT_BF16, false>;
    else out->fn = qknorm ? (const void*)rope_generic_kernel<DT_FP16, true>
                          : (const void*)rope_generic_kernel<DT_FP16, false>;
    return true;
  }
  out->kind = KK_ROPE_PAIR;
  out->vec = 8;
  out->fn = nullptr;
  if (dtype == DT_BF16) qknorm ? pick_vec<DT_BF16, true>(D, out) : pick_vec<DT_BF16, false>(D, out);
  else qknorm ? pick_vec<DT_FP16, true>(D, out) : pick_vec<DT_FP16, false>(D, out);
  if (!out->fn) { *why = "vector RoPE supports D in {64, 128, 256}"; return false; }
  return true;
}

}  // namespace trident
