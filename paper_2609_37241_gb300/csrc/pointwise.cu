// pointwise.cu -- elementwise operators: silu, add, neg, masked_fill, and SwiGLU
// (out = silu(g) * u, silu(g) = g / (1 + exp(-g))).
//
// FlagGems-style operators of the paper's kernel benchmark (§4.1), where silu and masked_fill
// show its largest per-call gains (§4.2), and the gated activation of an LLM's MLP. Pure
// streams, a few bytes and at most one exp per element: HBM is the bound at size, launch
// latency below. Three kernels, by the call's layout (pointwise_plan):
//   flat     dense tensors with a common offset from a 16-byte boundary are one long row of
//            T * W elements, whatever W is: 16-byte vectors between a scalar head and tail
//   rows     other 16-byte aligned rows (views): a flat index over all rows' vectors, the row
//            found by a multiplication
//   generic  anything else: a flat grid-stride loop with scalar accesses
// Before, a block took a tile of one row (512 vectors), so a row of another width left threads
// idle or blocks nearly empty, and odd widths or offsets took the generic kernel, which divided
// 64-bit indices per element. Device time per call, before -> now: silu 16384 x 1000 bf16
// 18.3 -> 10.1 us (6.5 TB/s), add 300000 x 96 fp16 165 -> 25.1, masked_fill 256 x 50257 bf16
// 57.0 -> 10.8, swiglu halves of 20000 x 1088 29.4 -> 20.0, swiglu 567 x 9735 22.7 -> 5.0, one row
// of 14336 1.47 -> 1.19; swiglu 4096 x 14336 halves (7.06 TB/s) 49.9 -> 49.8.
#include "device_common.cuh"
#include "measure.h"

namespace trident {

template <int DT, int OP>
__device__ __forceinline__ float pw_apply(float a, float b, uint8_t m, float scalar) {
  if (OP == PW_SWIGLU) return silu_mul<DT>(a, b);
  if (OP == PW_SILU) return silu_mul<DT>(a, 1.0f);
  if (OP == PW_ADD) return a + b;
  if (OP == PW_NEG) return -a;
  return m ? scalar : a;  // PW_MASKED_FILL
}
__host__ __device__ constexpr bool pw_binary(int op) { return op == PW_ADD || op == PW_SWIGLU; }

// One 16-byte vector of y. MASKED_FILL keeps unmasked elements bit for bit (NaN payloads too).
template <int DT, int OP>
__device__ __forceinline__ uint4 pw_vector(const uint4& av, const uint4& bv, const uint8_t* m, float scalar) {
  constexpr int VE = Act<DT>::VE;
  float af[VE], bf[VE], of[VE];
  unpack<DT>(av, af);
  if (pw_binary(OP)) unpack<DT>(bv, bf);
#pragma unroll
  for (int e = 0; e < VE; ++e)
    of[e] = pw_apply<DT, OP>(af[e], pw_binary(OP) ? bf[e] : 0.f, OP == PW_MASKED_FILL ? m[e] : (uint8_t)0, scalar);
  uint4 out = pack<DT>(of);
  if (OP == PW_MASKED_FILL) {
    uint16_t* o16 = reinterpret_cast<uint16_t*>(&out);
    const uint16_t* a16 = reinterpret_cast<const uint16_t*>(&av);
    uint32_t* o32 = reinterpret_cast<uint32_t*>(&out);
    const uint32_t* a32 = reinterpret_cast<const uint32_t*>(&av);
#pragma unroll
    for (int e = 0; e < VE; ++e) {
      if (!m[e]) {
        if (Act<DT>::BYTES == 2) o16[e] = a16[e];
        else o32[e] = a32[e];
      }
    }
  }
  return out;
}

// The VE mask bytes of one vector.
template <int VE>
__device__ __forceinline__ void pw_mask(const uint8_t* m, int32_t vec, uint8_t* out) {
  if (vec) {
    if (VE == 8) {
      const uint2 w = __ldg(reinterpret_cast<const uint2*>(m));
      memcpy(out, &w, 8);
    } else {
      const uint32_t w = __ldg(reinterpret_cast<const uint32_t*>(m));
      memcpy(out, &w, 4);
    }
  } else {
#pragma unroll
    for (int e = 0; e < VE; ++e) out[e] = __ldg(m + e);
  }
}

// One element, by its index in each tensor.
template <int DT, int OP>
__device__ __forceinline__ void pw_element(const PointwiseParams& p, int64_t ai, int64_t bi, int64_t mi, int64_t yi) {
  if (OP == PW_MASKED_FILL && !p.mask[mi]) {  // bit copy of x
    if (Act<DT>::BYTES == 2)
      reinterpret_cast<uint16_t*>(p.y)[yi] = reinterpret_cast<const uint16_t*>(p.a)[ai];
    else
      reinterpret_cast<uint32_t*>(p.y)[yi] = reinterpret_cast<const uint32_t*>(p.a)[ai];
    return;
  }
  const float a = load_elem<DT>(p.a, ai);
  const float b = pw_binary(OP) ? load_elem<DT>(p.b, bi) : 0.f;
  store_elem<DT>(p.y, yi, pw_apply<DT, OP>(a, b, (uint8_t)1, p.scalar));
}

// UNROLL vectors per thread, a block's vectors contiguous, every load issued before the first
// use.
template <int DT, int OP, int UNROLL, bool ROWS>
__global__ void __launch_bounds__(kThreads) pointwise_vec_kernel(const PointwiseParams p) {
  pdl_trigger();
  constexpr int VE = Act<DT>::VE;
  constexpr int EB = Act<DT>::BYTES;
  const int64_t u0 = (int64_t)blockIdx.x * (UNROLL * kThreads) + threadIdx.x;
  // element index of vector u in a tensor with row stride rs
  int64_t row[UNROLL], col[UNROLL];
#pragma unroll
  for (int k = 0; k < UNROLL; ++k) {
    const int64_t u = u0 + k * kThreads;
    if (!ROWS) {
      row[k] = 0;
      col[k] = p.peel + u * VE;
    } else {
      row[k] = p.units <= 0x7fffffffll ? (int64_t)fast_div((uint32_t)u, p.magic, p.shift) : u / p.row_vecs;
      col[k] = (u - row[k] * p.row_vecs) * VE;
    }
  }
  auto at = [&](const void* base, int k, int64_t rs) {
    return reinterpret_cast<const char*>(base) + (ROWS ? row[k] * rs + col[k] : col[k]) * EB;
  };
  if (p.prefetch && (threadIdx.x & 7) == 0) {  // the block's lines (prefetch_l2)
#pragma unroll
    for (int k = 0; k < UNROLL; ++k) {
      if (u0 + k * kThreads < p.units) {
        prefetch_l2(at(p.a, k, p.a_rs));
        if (pw_binary(OP)) prefetch_l2(at(p.b, k, p.b_rs));
      }
    }
  }
  pdl_wait();
  uint4 av[UNROLL], bv[UNROLL];
  uint8_t mv[UNROLL][VE];
#pragma unroll
  for (int k = 0; k < UNROLL; ++k) {
    if (u0 + k * kThreads < p.units) {
      av[k] = ldg16(at(p.a, k, p.a_rs));
      if (pw_binary(OP)) bv[k] = ldg16(at(p.b, k, p.b_rs));
      if (OP == PW_MASKED_FILL) pw_mask<VE>(p.mask + (ROWS ? row[k] * p.m_rs + col[k] : col[k]), p.mask_vec, mv[k]);
    }
  }
#pragma unroll
  for (int k = 0; k < UNROLL; ++k)
    if (u0 + k * kThreads < p.units)
      st16(const_cast<char*>(at(p.y, k, p.y_rs)), pw_vector<DT, OP>(av[k], bv[k], mv[k], p.scalar));
  if (!ROWS && blockIdx.x == gridDim.x - 1) {  // head and tail elements (fewer than a vector each)
    const int i = threadIdx.x;
    if (i < p.peel + p.tail) {
      const int64_t e = i < p.peel ? i : i + p.units * VE;
      pw_element<DT, OP>(p, e, e, e, e);
    }
  }
}

template <int DT, int OP>
__global__ void __launch_bounds__(kThreads) pointwise_generic_kernel(const PointwiseParams p) {
  pdl_prologue();
  const int64_t total = p.T * p.W;
  const int64_t stride = (int64_t)gridDim.x * kThreads;
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < total; i += stride) {
    const int64_t row = total <= 0x7fffffffll ? (int64_t)fast_div((uint32_t)i, p.magic, p.shift) : i / p.W;
    const int64_t col = i - row * p.W;
    pw_element<DT, OP>(p, row * p.a_rs + col, row * p.b_rs + col, row * p.m_rs + col, row * p.y_rs + col);
  }
}

// Two vectors per thread for one-input operators only (pointwise_plan).
template <int DT, int OP>
static void pick(KernelEntry* out) {
  constexpr int U = pw_binary(OP) ? 1 : 2;
  out->pw_fn[PW_FLAT] = (const void*)pointwise_vec_kernel<DT, OP, 1, false>;
  out->pw_fn[PW_FLAT2] = (const void*)pointwise_vec_kernel<DT, OP, U, false>;
  out->pw_fn[PW_ROWS] = (const void*)pointwise_vec_kernel<DT, OP, 1, true>;
  out->pw_fn[PW_ROWS2] = (const void*)pointwise_vec_kernel<DT, OP, U, true>;
  out->pw_fn[PW_GENERIC] = (const void*)pointwise_generic_kernel<DT, OP>;
}

template <int OP>
static void pick(int32_t dtype, KernelEntry* out) {
  if (dtype == DT_BF16) pick<DT_BF16, OP>(out);
  else if (dtype == DT_FP16) pick<DT_FP16, OP>(out);
  else pick<DT_FP32, OP>(out);
}

// One vector per thread, two for one-input operators of more than one and a half waves of
// threads (2048 per SM). With one vector a thread's life is one round trip and the grid has the
// most blocks to hand out, which is faster at every size with two inputs (same-box device times,
// 1 / 2 / 4 vectors per thread: swiglu 64 x 14336 2.65 / 3.78 / 3.88 us, 4096 x 14336 50.0 / 50.6 /
// 50.3, 4096 x 28672 96.9 / 102.0 / 98.9) and for small one-input calls (silu 1024 x 1024
// 2.00 / 2.40 / 3.51); with a single 16-byte load per thread a large one has too few bytes in
// flight (silu 4096 / 8192 / 16384 x 1000 2.84 / 5.66 / 11.6 against 2.87 / 4.20 / 10.1 with two).
// Cache hints (evict-first stores, no L1 allocation) changed nothing or lost 1-4 %.
int pointwise_plan(PointwiseParams* p, int32_t op, int32_t eb, int64_t* blocks, int32_t sms) {
  const int64_t ve = 16 / eb, n = p->T * p->W;
  const bool binary = pw_binary(op), masked = op == PW_MASKED_FILL;
  const uintptr_t off = (uintptr_t)p->a & 15;
  const bool together = ((uintptr_t)p->y & 15) == off && (!binary || ((uintptr_t)p->b & 15) == off);
  const bool dense = p->T <= 1 || (p->a_rs == p->W && p->y_rs == p->W && (!binary || p->b_rs == p->W) &&
                                   (!masked || p->m_rs == p->W));
  const bool rows16 = together && off == 0 && p->W % ve == 0 && p->a_rs % ve == 0 && p->y_rs % ve == 0 &&
                      (!binary || p->b_rs % ve == 0);
  p->peel = p->tail = 0;
  p->magic = 0;
  p->shift = 0;
  p->row_vecs = 0;
  bool rows = false;
  if (dense && together) {
    const int64_t peel = off ? (16 - (int64_t)off) / eb : 0;
    p->peel = (int32_t)(peel < n ? peel : n);
    p->units = (n - p->peel) / ve;
    p->tail = (int32_t)(n - p->peel - p->units * ve);
    p->mask_vec = ((uintptr_t)p->mask + (uintptr_t)p->peel) % (uintptr_t)ve == 0;
  } else if (rows16) {
    rows = true;
    p->row_vecs = p->W / ve;
    p->units = p->T * p->row_vecs;
    if (p->units <= 0x7fffffffll) div_magic((uint32_t)p->row_vecs, &p->magic, &p->shift);
    p->mask_vec = (uintptr_t)p->mask % (uintptr_t)ve == 0 && p->m_rs % ve == 0;
  } else {
    if (n <= 0x7fffffffll) div_magic((uint32_t)p->W, &p->magic, &p->shift);
    p->units = 0;
    p->mask_vec = 0;
    *blocks = (n + kThreads - 1) / kThreads;
    if (*blocks > (int64_t)sms * 64) *blocks = (int64_t)sms * 64;
    return PW_GENERIC;
  }
  const bool two = !binary && p->units > 3 * (int64_t)sms * 2048 / 2;
  const int64_t per = (two ? 2 : 1) * kThreads;
  *blocks = (p->units + per - 1) / per;
  return rows ? (two ? PW_ROWS2 : PW_ROWS) : (two ? PW_FLAT2 : PW_FLAT);
}

// Latency-floor probe (trident_launch_floor): a kernel that does nothing but take part in
// programmatic dependent launch like every kernel of the library.
__global__ void empty_kernel() {
  pdl_trigger();
  pdl_wait();
}

const void* empty_kernel_entry() { return (const void*)empty_kernel; }

// Copy-floor probe (trident_copy_floor), see CopyFloorParams. With prefetch, a block's read
// lines go to L2 between the launch trigger and the wait, as the layer chain's blocks do.
__global__ void __launch_bounds__(kThreads) copy_floor_kernel(const CopyFloorParams p) {
  pdl_trigger();
  const int64_t g = gridDim.x;
  const int64_t rpb = (p.nr + g - 1) / g, wpb = (p.nw + g - 1) / g;
  const int64_t r0 = (int64_t)blockIdx.x * rpb, w0 = (int64_t)blockIdx.x * wpb;
  const uint4* src = static_cast<const uint4*>(p.src);
  uint4* dst = static_cast<uint4*>(p.dst);
  if (p.prefetch) {
    for (int64_t i = (int64_t)threadIdx.x * 8; i < rpb; i += (int64_t)kThreads * 8)
      if (r0 + i < p.nr) prefetch_l2(src + r0 + i);
  }
  pdl_wait();
  uint4 acc = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 4
  for (int64_t i = threadIdx.x; i < rpb; i += kThreads) {
    if (r0 + i < p.nr) {
      const uint4 v = ldg16(src + r0 + i);
      acc.x ^= v.x; acc.y ^= v.y; acc.z ^= v.z; acc.w ^= v.w;
    }
  }
  for (int64_t j = threadIdx.x; j < wpb; j += kThreads)
    if (w0 + j < p.nw) st16(dst + w0 + j, acc);
}

const void* copy_floor_entry() { return (const void*)copy_floor_kernel; }

bool pointwise_kernel(int32_t op, int32_t dtype, int32_t variant, int64_t W, KernelEntry* out,
                      const char** why) {
  if (dtype != DT_BF16 && dtype != DT_FP16 && dtype != DT_FP32) { *why = "dtype"; return false; }
  if (W < 1) { *why = "row width must be >= 1"; return false; }
  const int eb = dtype == DT_FP32 ? 4 : 2;
  if (variant != 1 && (W * eb) % 16 != 0) {
    *why = "the vector variant needs row width * elem_size % 16 == 0";
    return false;
  }
  out->kind = KK_POINTWISE;
  out->vec = 16 / eb;
  switch (op) {
    case PW_SWIGLU: pick<PW_SWIGLU>(dtype, out); break;
    case PW_SILU: pick<PW_SILU>(dtype, out); break;
    case PW_ADD: pick<PW_ADD>(dtype, out); break;
    case PW_NEG: pick<PW_NEG>(dtype, out); break;
    case PW_MASKED_FILL: pick<PW_MASKED_FILL>(dtype, out); break;
    default: *why = "unknown pointwise op"; return false;
  }
  out->fn = out->pw_fn[PW_GENERIC];
  return true;
}

}  // namespace trident
