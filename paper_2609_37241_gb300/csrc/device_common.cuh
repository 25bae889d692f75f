// device_common.cuh -- device-side building blocks shared by the kernels of this library.
//
// Every kernel is memory bound (a few flops per byte), so the building blocks are about
// moving bytes: 16-byte vector loads and stores per thread, fp32 math in registers,
// warp-shuffle reductions. Each kernel starts with the programmatic-dependent-launch
// pair (trigger, then wait) so that, when launched with programmatic stream
// serialisation, the next kernel's launch overlaps this one while every global memory
// access still waits for the previous kernel to finish; between the two, small grids
// prefetch their first lines into L2 (prefetch_l2).
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include "internal.h"

namespace trident {

constexpr uint32_t kErrPos = 0x1u;  // TRIDENT_DEVERR_POS
constexpr uint32_t kErrTimeout = 0x2u;  // TRIDENT_DEVERR_TIMEOUT

__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_prologue() {
  pdl_trigger();
  pdl_wait();
}

// L2 prefetch of one line. Kernels issue prefetches of the lines they read first between
// pdl_trigger and pdl_wait, while the previous kernel of the stream may still run: a
// prefetch changes no value that a later load returns (the loads come after the wait), it
// only lets the DRAM fetch overlap the previous kernel's tail and the launch handoff. The
// host enables it (params.prefetch) for grids of at most 256 threads per SM (a layer chain's: one
// block) launched with programmatic stream serialisation: a grid that fills the GPU becomes resident only as the
// previous kernel's blocks retire, and its prefetches then compete with that kernel.
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.L2 [%0];" :: "l"(p)); }

template <int DT> struct Act;
template <> struct Act<DT_BF16> { static constexpr int VE = 8; static constexpr int BYTES = 2; };
template <> struct Act<DT_FP16> { static constexpr int VE = 8; static constexpr int BYTES = 2; };
template <> struct Act<DT_FP32> { static constexpr int VE = 4; static constexpr int BYTES = 4; };

// ---------------------------------------------------------------- 16-byte vectors
__device__ __forceinline__ uint4 ldg16(const void* p) { return __ldg(reinterpret_cast<const uint4*>(p)); }
__device__ __forceinline__ uint4 ld16(const void* p) { return *reinterpret_cast<const uint4*>(p); }
__device__ __forceinline__ void st16(void* p, uint4 v) { *reinterpret_cast<uint4*>(p) = v; }
__device__ __forceinline__ float4 ldg_f4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }

template <int DT> __device__ __forceinline__ void unpack(const uint4& v, float* f);
template <> __device__ __forceinline__ void unpack<DT_BF16>(const uint4& v, float* f) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    f[2 * i] = __uint_as_float(w[i] << 16);
    f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
  }
}
template <> __device__ __forceinline__ void unpack<DT_FP16>(const uint4& v, float* f) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    __half2 h;
    memcpy(&h, &w[i], 4);
    float2 ff = __half22float2(h);
    f[2 * i] = ff.x;
    f[2 * i + 1] = ff.y;
  }
}
template <> __device__ __forceinline__ void unpack<DT_FP32>(const uint4& v, float* f) {
  f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y);
  f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
}

template <int DT> __device__ __forceinline__ uint4 pack(const float* f);
template <> __device__ __forceinline__ uint4 pack<DT_BF16>(const float* f) {
  uint32_t w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    __nv_bfloat162 b = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
    memcpy(&w[i], &b, 4);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}
template <> __device__ __forceinline__ uint4 pack<DT_FP16>(const float* f) {
  uint32_t w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    __half2 h = __floats2half2_rn(f[2 * i], f[2 * i + 1]);
    memcpy(&w[i], &h, 4);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}
template <> __device__ __forceinline__ uint4 pack<DT_FP32>(const float* f) {
  return make_uint4(__float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]),
                    __float_as_uint(f[3]));
}

// ---------------------------------------------------------------- scalar elements
template <int DT> __device__ __forceinline__ float load_elem(const void* p, int64_t i);
template <> __device__ __forceinline__ float load_elem<DT_BF16>(const void* p, int64_t i) {
  return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p)[i]);
}
template <> __device__ __forceinline__ float load_elem<DT_FP16>(const void* p, int64_t i) {
  return __half2float(reinterpret_cast<const __half*>(p)[i]);
}
template <> __device__ __forceinline__ float load_elem<DT_FP32>(const void* p, int64_t i) {
  return reinterpret_cast<const float*>(p)[i];
}
template <int DT> __device__ __forceinline__ void store_elem(void* p, int64_t i, float v);
template <> __device__ __forceinline__ void store_elem<DT_BF16>(void* p, int64_t i, float v) {
  reinterpret_cast<__nv_bfloat16*>(p)[i] = __float2bfloat16_rn(v);
}
template <> __device__ __forceinline__ void store_elem<DT_FP16>(void* p, int64_t i, float v) {
  reinterpret_cast<__half*>(p)[i] = __float2half_rn(v);
}
template <> __device__ __forceinline__ void store_elem<DT_FP32>(void* p, int64_t i, float v) {
  reinterpret_cast<float*>(p)[i] = v;
}
// Rounds v to the activation type and back (the value a store would hold).
template <int DT> __device__ __forceinline__ float round_act(float v);
template <> __device__ __forceinline__ float round_act<DT_BF16>(float v) {
  return __bfloat162float(__float2bfloat16_rn(v));
}
template <> __device__ __forceinline__ float round_act<DT_FP16>(float v) {
  return __half2float(__float2half_rn(v));
}
template <> __device__ __forceinline__ float round_act<DT_FP32>(float v) { return v; }

__device__ __forceinline__ const char* row_ptr(const void* base, int64_t row, int64_t rs, int eb) {
  return reinterpret_cast<const char*>(base) + row * rs * eb;
}
__device__ __forceinline__ char* row_ptr(void* base, int64_t row, int64_t rs, int eb) {
  return reinterpret_cast<char*>(base) + row * rs * eb;
}

// ---------------------------------------------------------------- reductions
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum over the block; every thread gets the same total (same summation order).
// `red` holds kThreads/32 floats and must not be reused until after a barrier.
__device__ __forceinline__ float block_sum(float v, float* red) {
  constexpr int NW = kThreads / 32;
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float t = 0.f;
#pragma unroll
  for (int i = 0; i < NW; ++i) t += red[i];
  return t;
}

// ---------------------------------------------------------------- RoPE angles
// sin and cos of the angle pos * f, with f = fhi + flo (a double-float split of
// theta^(-2i/D) made in fp64 on the host). The product is kept as ah + al (al holds the
// exact rounding error of pos * fhi, from one fma, plus pos * flo); ah is reduced modulo
// 2 pi with the Cody-Waite method (Cody and Waite, "Software Manual for the Elementary
// Functions", 1980) using 2 pi = A + B + C, A with 12 significant bits so that k * A is
// exact for k < 4096, i.e. angles up to about 25700 rad; the reduced angle, within about
// [-pi, pi], goes to the hardware sine/cosine (absolute error about 2^-21).
constexpr float kInv2Pi = 0.159154936671257019f;     // 1 / (2 pi), rounded to fp32
constexpr float k2PiA = 6.283203125f;                // 2 pi to 12 significant bits (3217/512)
constexpr float k2PiB = -1.78178197529632598e-05f;   // fp32(2 pi - A)
constexpr float k2PiC = -6.60559822986128669e-13f;   // fp32(2 pi - A - B)

__device__ __forceinline__ void rope_sincos(float pos, float fhi, float flo, float* s, float* c) {
  const float ah = pos * fhi;
  const float al = fmaf(pos, fhi, -ah) + pos * flo;
  const float k = rintf(ah * kInv2Pi);
  float r = fmaf(-k, k2PiA, ah);
  r = fmaf(-k, k2PiB, r);
  r = fmaf(-k, k2PiC, r);
  __sincosf(r + al, s, c);
}

// ---------------------------------------------------------------- division
// n / d for a 32-bit n and a divisor d known per launch, from the host's round-up multiplier
// m and shift l for d (div_magic; Granlund and Montgomery, "Division by invariant integers
// using multiplication", 1994): (h + ((n - h) >> 1)) >> (l - 1) with h = umulhi(n, m), exact
// for every 32-bit n; l = 0 stands for d = 1. A division by a runtime divisor is otherwise a
// long instruction sequence (64-bit: several times longer).
__device__ __forceinline__ uint32_t fast_div(uint32_t n, uint32_t m, int32_t l) {
  if (l == 0) return n;
  const uint32_t h = __umulhi(n, m);
  return (h + ((n - h) >> 1)) >> (l - 1);
}

// ---------------------------------------------------------------- packed fp32 pairs
// Two fp32 values in one 64-bit register pair; sm_100's f32x2 instructions do both lanes'
// multiply (or fused multiply-add) in one issue, each rounded as the scalar instruction rounds.
struct F2 { unsigned long long v; };
__device__ __forceinline__ F2 f2_pack(float a, float b) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2_unpack(F2 x, float* a, float* b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(*a), "=f"(*b) : "l"(x.v));
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}

// ---------------------------------------------------------------- RoPE, both halves per lane
// A head-row of D elements by D / 16 lanes: lane l owns elements [8l, 8l + 8) and their
// rotate-half partners [D/2 + 8l, D/2 + 8l + 8), so a rotation needs no other lane (with one
// vector per lane it took eight shuffles per vector, and the two lanes of a pair computed the
// same eight sines and cosines). A warp holds GW = 512 / D lane groups and works on one item:
// rpi consecutive head-rows of one token (RopeParams.ipt items per token), group g taking the
// rows g, g + GW, ... of it; the lane's angles are computed once per item.
template <int D>
struct RopeGeom {
  static constexpr int LPG = D / 16;     // lanes per head-row
  static constexpr int GW = 32 / LPG;    // head-rows per warp at a time
  static_assert(LPG >= 2 && LPG <= 32 && (LPG & (LPG - 1)) == 0, "head size");
};

// The item of warp `item` of the grid: its token and head-rows [*first, *end); false past the
// grid's last item.
__device__ __forceinline__ bool rope_item(const RopeParams& p, int64_t item, int64_t* t, int* first, int* end) {
  if (item >= p.T * p.ipt) return false;
  const uint32_t tok = fast_div((uint32_t)item, p.ipt_magic, p.ipt_shift);
  *t = tok;
  *first = (int)((uint32_t)item - tok * (uint32_t)p.ipt) * p.rpi;
  *end = min(p.NH, *first + p.rpi);
  return true;
}

// Source of head-row hh of token t (its lane-0 vector).
__device__ __forceinline__ const char* rope_row_src(const RopeParams& p, int64_t t, int hh, int D) {
  const int RB = D * 2;
  return hh < p.Hq ? row_ptr(p.q, t, p.q_rs, 2) + (int64_t)hh * RB
       : hh < p.Hq + p.Hkv ? row_ptr(p.k, t, p.k_rs, 2) + (int64_t)(hh - p.Hq) * RB
                           : row_ptr(p.v, t, p.v_rs, 2) + (int64_t)(hh - p.Hq - p.Hkv) * RB;
}
template <int D>
__device__ __forceinline__ const char* rope_row_src(const RopeParams& p, int64_t t, int hh) {
  return rope_row_src(p, t, hh, D);
}

// Sines and cosines of a lane's eight pairs for position pos; fq holds the lane's frequencies.
struct RopeAngles { F2 sn[4], ns[4], cs[4]; };  // ns = -sn
__device__ __forceinline__ void rope_angles(int32_t pos, const float4* fq, RopeAngles* a) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float s0, c0, s1, c1;
    rope_sincos((float)pos, fq[q].x, fq[q].y, &s0, &c0);
    rope_sincos((float)pos, fq[q].z, fq[q].w, &s1, &c1);
    a->sn[q] = f2_pack(s0, s1);
    a->ns[q] = f2_pack(-s0, -s1);
    a->cs[q] = f2_pack(c0, c1);
  }
}
__device__ __forceinline__ void rope_pair_freqs(const float2* inv_freq, int lane, float4* fq) {
#pragma unroll
  for (int q = 0; q < 4; ++q) fq[q] = ldg_f4(reinterpret_cast<const float*>(inv_freq) + 16 * lane + 4 * q);
}
// The same from a table that the previous kernel of the stream may have written, called after
// pdl_wait: that kernel may have written it while this grid was already resident, so the loads are
// plain, coherent ones (__ldg is defined only for what nothing writes during the kernel), which
// pdl_wait's memory clobber keeps behind it.
__device__ __forceinline__ void rope_pair_freqs_late(const float2* inv_freq, int lane, float4* fq) {
#pragma unroll
  for (int q = 0; q < 4; ++q)
    fq[q] = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(inv_freq) + 16 * lane + 4 * q);
}

// A lane's q- or k-norm weights (kind 1: q, 2: k), for its low and high halves.
struct RopeGamma { F2 lo[4], hi[4]; };
__device__ __forceinline__ void rope_pair_gamma(const float* gamma, int lane, int D, RopeGamma* g) {
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const float4 a = ldg_f4(gamma + lane * 8 + 4 * q), b = ldg_f4(gamma + D / 2 + lane * 8 + 4 * q);
    g->lo[2 * q] = f2_pack(a.x, a.y);
    g->lo[2 * q + 1] = f2_pack(a.z, a.w);
    g->hi[2 * q] = f2_pack(b.x, b.y);
    g->hi[2 * q + 1] = f2_pack(b.z, b.w);
  }
}

template <int DT>
__device__ __forceinline__ void rope_unpack(const uint4& lo, const uint4& hi, F2* A, F2* B) {
  float a[8], b[8];
  unpack<DT>(lo, a);
  unpack<DT>(hi, b);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    A[q] = f2_pack(a[2 * q], a[2 * q + 1]);
    B[q] = f2_pack(b[2 * q], b[2 * q + 1]);
  }
}

// 1 / rms of a head-row held by the lane group (LPG lanes; on: the lane holds part of it), in
// both halves of a pair.
template <int LPG>
__device__ __forceinline__ F2 rope_inv_rms(const RopeParams& p, const F2* A, const F2* B, bool on = true) {
  F2 s2 = f2_mul(A[0], A[0]);
#pragma unroll
  for (int q = 1; q < 4; ++q) s2 = f2_fma(A[q], A[q], s2);
#pragma unroll
  for (int q = 0; q < 4; ++q) s2 = f2_fma(B[q], B[q], s2);
  float s0, s1;
  f2_unpack(s2, &s0, &s1);
  float ss = on ? s0 + s1 : 0.f;
  const unsigned mask =
      LPG == 32 ? 0xffffffffu : (((1u << LPG) - 1u) << ((threadIdx.x & 31) & ~(LPG - 1)));
#pragma unroll
  for (int o = LPG / 2; o > 0; o >>= 1) ss += __shfl_xor_sync(mask, ss, o, LPG);
  const float inv = rsqrtf(ss * p.inv_D + p.eps);
  return f2_pack(inv, inv);
}
__device__ __forceinline__ void rope_scale(F2 inv, const RopeGamma& g, F2* A, F2* B) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    A[q] = f2_mul(f2_mul(A[q], inv), g.lo[q]);
    B[q] = f2_mul(f2_mul(B[q], inv), g.hi[q]);
  }
}

// Where head-row hh of token t goes (its lane-0 vector).
__device__ __forceinline__ char* rope_row_dst(const RopeParams& p, int64_t t, int hh, int32_t pos, int D) {
  const int RB = D * 2;
  if (hh < p.Hq) return row_ptr(p.q, t, p.q_rs, 2) + (int64_t)hh * RB;
  const bool is_v = hh >= p.Hq + p.Hkv;
  return reinterpret_cast<char*>(is_v ? p.v_cache : p.k_cache) +
         ((int64_t)(hh - p.Hq - (is_v ? p.Hkv : 0)) * p.S + pos) * RB;
}

// Rotates a lane's pairs and stores them at dst (the lane's low vector; D bytes on, the high one).
template <int DT>
__device__ __forceinline__ void rope_rotate(char* dst, int D, const RopeAngles& an, const F2* A, const F2* B) {
  float a[8], b[8];
  // low half: x_i c - x_{i+D/2} s;  high half: x_{i+D/2} c + x_i s
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    f2_unpack(f2_fma(A[q], an.cs[q], f2_mul(B[q], an.ns[q])), &a[2 * q], &a[2 * q + 1]);
    f2_unpack(f2_fma(B[q], an.cs[q], f2_mul(A[q], an.sn[q])), &b[2 * q], &b[2 * q + 1]);
  }
  st16(dst, pack<DT>(a));
  st16(dst + D, pack<DT>(b));
}

// Finishes head-row hh of token t from its two vectors: [q/k norm,] rotation, store (v: copy).
// KEEP: *g holds a kind's weights (*kind; 0: none yet) from row to row, as rows of an item
// mostly share them; otherwise each row loads its own (fewer registers).
template <int DT, int D, bool QKNORM, bool KEEP>
__device__ __forceinline__ void rope_pair_finish(const RopeParams& p, int64_t t, int hh, int lane, int32_t pos,
                                                 const uint4& lo, const uint4& hi, const RopeAngles& an,
                                                 RopeGamma* g, int* kind) {
  char* dst = rope_row_dst(p, t, hh, pos, D) + lane * 16;
  if (hh >= p.Hq + p.Hkv) {  // bit copy into the cache
    st16(dst, lo);
    st16(dst + D, hi);
    return;
  }
  F2 A[4], B[4];
  rope_unpack<DT>(lo, hi, A, B);
  constexpr int LPG = RopeGeom<D>::LPG;
  if (QKNORM) {
    const bool is_q = hh < p.Hq;
    const F2 inv = rope_inv_rms<LPG>(p, A, B);
    if (KEEP) {
      const int want = is_q ? 1 : 2;
      if (*kind != want) {
        rope_pair_gamma(is_q ? p.gamma_q : p.gamma_k, lane, D, g);
        *kind = want;
      }
      rope_scale(inv, *g, A, B);
    } else {
      RopeGamma own;
      rope_pair_gamma(is_q ? p.gamma_q : p.gamma_k, lane, D, &own);
      rope_scale(inv, own, A, B);
    }
  }
  rope_rotate<DT>(dst, D, an, A, B);
}

// L2 prefetch of an item's row lines (at most R rows per lane group) and position.
template <int D, int R>
__device__ __forceinline__ void rope_item_prefetch(const RopeParams& p, int64_t t, int first, int end) {
  constexpr int LPG = RopeGeom<D>::LPG, GW = RopeGeom<D>::GW;
  const int lane = (threadIdx.x & 31) % LPG, g = (threadIdx.x & 31) / LPG;
  if (lane % 8 != 0) return;
#pragma unroll
  for (int j = 0; j < R; ++j) {
    if (first + g + j * GW < end) {
      const char* src = rope_row_src<D>(p, t, first + g + j * GW) + lane * 16;
      prefetch_l2(src);
      prefetch_l2(src + D);
    }
  }
  if ((threadIdx.x & 31) == 0) prefetch_l2(p.pos + t);
}

// One item's rows [first, end) of token t, at most R per lane group: every load the rows need
// is issued first, without a branch (with one per row the loads followed one another). fq: the
// lane's frequencies.
template <int DT, int D, bool QKNORM, int R, bool KEEP>
__device__ __forceinline__ void rope_pair_rows(const RopeParams& p, int64_t t, int first, int end, const float4* fq) {
  constexpr int LPG = RopeGeom<D>::LPG, GW = RopeGeom<D>::GW;
  const int lane = (threadIdx.x & 31) % LPG;
  const int hh0 = first + (threadIdx.x & 31) / LPG;
  uint4 lo[R], hi[R];
#pragma unroll
  for (int j = 0; j < R; ++j) {  // groups past the item's end load its last row and drop it
    const char* src = rope_row_src<D>(p, t, min(hh0 + j * GW, end - 1)) + lane * 16;
    lo[j] = ld16(src);
    hi[j] = ld16(src + D);
  }
  const int32_t pos = __ldg(p.pos + t);
  RopeGamma g;
  int kind = 0;
  if (QKNORM && (KEEP || R == 1) && hh0 < end && hh0 < p.Hq + p.Hkv) {  // v rows need none
    kind = hh0 < p.Hq ? 1 : 2;
    rope_pair_gamma(kind == 1 ? p.gamma_q : p.gamma_k, lane, D, &g);
  }
  if (pos < 0 || (int64_t)pos >= p.S) {  // uniform over the warp: one token per item
    if ((threadIdx.x & 31) == 0) atomicOr(p.err, kErrPos);
    return;
  }
  RopeAngles an;
  if (QKNORM && R == 1) {  // the norm first: its weights' registers are free before the angles'
    if (hh0 >= end) return;
    F2 A[4], B[4];
    if (hh0 >= p.Hq + p.Hkv) {  // bit copy into the cache
      char* dst = rope_row_dst(p, t, hh0, pos, D) + lane * 16;
      st16(dst, lo[0]);
      st16(dst + D, hi[0]);
      return;
    }
    rope_unpack<DT>(lo[0], hi[0], A, B);
    rope_scale(rope_inv_rms<LPG>(p, A, B), g, A, B);
    rope_angles(pos, fq, &an);
    rope_rotate<DT>(rope_row_dst(p, t, hh0, pos, D) + lane * 16, D, an, A, B);
    return;
  }
  rope_angles(pos, fq, &an);
#pragma unroll
  for (int j = 0; j < R; ++j)
    if (hh0 + j * GW < end)
      rope_pair_finish<DT, D, QKNORM, KEEP>(p, t, hh0 + j * GW, lane, pos, lo[j], hi[j], an, &g, &kind);
}

// ---------------------------------------------------------------- SwiGLU tile
template <int DT> __device__ __forceinline__ float silu_mul(float g, float u);
// bf16/fp16 outputs: fast exp and divide (relative error ~1e-6, far below the output ulp;
// for g below about -87 the result is -0, the limit of g * sigmoid(g)).
template <> __device__ __forceinline__ float silu_mul<DT_BF16>(float g, float u) {
  return __fdividef(g, 1.0f + __expf(-g)) * u;
}
template <> __device__ __forceinline__ float silu_mul<DT_FP16>(float g, float u) {
  return __fdividef(g, 1.0f + __expf(-g)) * u;
}
// fp32 outputs: full-precision exp and IEEE division.
template <> __device__ __forceinline__ float silu_mul<DT_FP32>(float g, float u) {
  return g / (1.0f + expf(-g)) * u;
}

// L2 prefetch of the gate and up lines of one SwiGLU tile (threads on a line boundary).
template <int DT, int UNROLL, int NT>
__device__ __forceinline__ void swiglu_prefetch(const SwigluParams& p, int64_t row, int64_t v0,
                                                int tid) {
  constexpr int VE = Act<DT>::VE;
  constexpr int EB = Act<DT>::BYTES;
  if ((tid & 7) != 0 || row >= p.T) return;
  const int64_t nvec = p.I / VE;
  const uint4* g = reinterpret_cast<const uint4*>(row_ptr(p.g, row, p.g_rs, EB));
  const uint4* u = reinterpret_cast<const uint4*>(row_ptr(p.u, row, p.u_rs, EB));
#pragma unroll
  for (int k = 0; k < UNROLL; ++k) {
    const int64_t vi = v0 + (int64_t)k * NT + tid;
    if (vi < nvec) {
      prefetch_l2(g + vi);
      prefetch_l2(u + vi);
    }
  }
}

// One tile of UNROLL * NT vectors of one row, starting at vector index v0. Its loads stand
// in no branch (each behind its own, the compiler finishes one pair before it issues the next):
// threads past the row's end (not FULL) load its last vector and drop it.
template <int DT, int UNROLL, int NT, bool FULL>
__device__ __forceinline__ void swiglu_tile_body(const SwigluParams& p, int64_t row, int64_t v0, int tid) {
  constexpr int VE = Act<DT>::VE;
  constexpr int EB = Act<DT>::BYTES;
  const int64_t nvec = p.I / VE;
  const uint4* g = reinterpret_cast<const uint4*>(row_ptr(p.g, row, p.g_rs, EB));
  const uint4* u = reinterpret_cast<const uint4*>(row_ptr(p.u, row, p.u_rs, EB));
  uint4* o = reinterpret_cast<uint4*>(row_ptr(p.out, row, p.o_rs, EB));
  uint4 gv[UNROLL], uv[UNROLL];
#pragma unroll
  for (int k = 0; k < UNROLL; ++k) {
    const int64_t vk = v0 + (int64_t)k * NT + tid, vi = FULL ? vk : min(vk, nvec - 1);
    gv[k] = ldg16(g + vi);
    uv[k] = ldg16(u + vi);
  }
#pragma unroll
  for (int k = 0; k < UNROLL; ++k) {
    const int64_t vi = v0 + (int64_t)k * NT + tid;
    if (FULL || vi < nvec) {
      float gf[VE], uf[VE], of[VE];
      unpack<DT>(gv[k], gf);
      unpack<DT>(uv[k], uf);
#pragma unroll
      for (int e = 0; e < VE; ++e) of[e] = silu_mul<DT>(gf[e], uf[e]);
      st16(o + vi, pack<DT>(of));
    }
  }
}

// A row's last tile: the narrowest power-of-two width that holds what is left of the row (an
// I of 22016 leaves 192 of 512 vectors: 128 tokens at H 8192 10.4 us at the full width,
// 8.5 us so; taking it in two parts instead cost a second round trip, 206 -> 209 us at 8192
// tokens of I 14336). The width depends on the block alone.
template <int DT, int UNROLL, int NT>
__device__ __forceinline__ void swiglu_tile(const SwigluParams& p, int64_t row, int64_t v0, int tid) {
  const int64_t left = p.I / Act<DT>::VE - v0;
  if (left >= UNROLL * NT) {
    swiglu_tile_body<DT, UNROLL, NT, true>(p, row, v0, tid);
    return;
  }
  if constexpr (UNROLL > 1) {
    if (left <= UNROLL / 2 * NT) {
      swiglu_tile<DT, UNROLL / 2, NT>(p, row, v0, tid);
      return;
    }
  }
  if (left > 0) swiglu_tile_body<DT, UNROLL, NT, false>(p, row, v0, tid);
}

}  // namespace trident
