// norm.cu -- RMSNorm, with or without a fused residual add (sm_103a).
//
//   RMSNORM      y = round(x * rsqrt(mean(x^2) + eps) * gamma)
//   ADD_RMSNORM  s = x + r (fp32);  r_out = round(s);  y = round(s * rsqrt(mean(s^2) + eps) * gamma)
//
// rms_norm is the paper's running example (Fig. 1, §2.3; its motivation experiment uses
// x (1024, 128)); the residual add fused in front of it is how decoder layers call it. All
// kernels but the last two read a row once and write it once:
//   norm_rows_kernel   rows of at most 128 vectors: LPR lanes per row, reduced by shuffles alone
//   norm_rows_edge_kernel  long calls of such rows at any element offset that all tensors share
//                      (odd widths, shifted bases): a warp per row, the vectors between a scalar
//                      head and tail
//   norm_block_kernel  longer rows, one block per row, one barrier; one or two vectors per thread,
//                      four or eight in long fp32 calls. EDGE: at any common element offset
//   norm_bulk_kernel   long calls of such rows in 16 bits: the row staged by bulk copies
//   norm_row_kernel    some calls of 256, 512 and 1024 vectors in 16 bits: blocks of 256 threads
//   norm_loop_kernel   16-byte rows of more than 2048 vectors (two passes)
//   norm_generic_kernel  anything else (scalar accesses)
//
// Bound: HBM for long calls; below about a thousand rows the launch and one row's dependent
// phases (load, reduce, scale, store). Before, only power-of-two widths kept their row in
// registers, in blocks of 256 threads; other widths read it twice, in a loop, and odd widths went
// element by element. Device time per call, before -> now:
//   add 1 x 4096 bf16      1.48 -> 1.03 us     rms 131072 x 128 bf16    15.6 -> 12.1 us
//   add 24 x 5120 bf16     2.72 -> 1.35        rms 30000 x 192 bf16     32.0 -> 5.1
//   add 64 x 8192 bf16     3.11 -> 1.83        rms 2050 x 3000 fp32     10.9 -> 8.7
//   add 256 x 4096 bf16    3.17 -> 1.95        rms 4096 x 4096 bf16     12.9 -> 11.7
//   add 3001 x 5120 bf16   23.7 -> 19.6        rms 16384 x 5120 bf16    59.5 -> 50.7
//   add 4096 x 8192 bf16   40.4 -> 40.1        rms 2000 x 16384 fp16    36.1 -> 23.7
//   add 4096 x 12288 bf16  65.1 -> 59.4        add 3000 x 2585 bf16     21.3 -> 12.5
//   add 20000 x 576 bf16   34.9 -> 19.4        rms 1 x 4096 bf16        1.39 -> 1.11
// The long residual rows run at the 6.8 TB/s copy rate (4096 x 8192: 6.7, 4096 x 12288: 6.8).
#include "device_common.cuh"

namespace trident {
// Calls of more rows than a number of waves of norm_block_kernel's blocks (norm_block_sm rows per SM
// and wave) take the entry of long calls: two waves with one vector per thread, one with two. Within
// them the short-lived blocks win, beyond them rows kept in fewer registers per SM do. In 16 bits that
// entry is norm_bulk_kernel, block / bulk either side of the line: residual 560 x 6144 6.0 / 6.4, 620
// 7.8 / 6.6; 850 x 5120 6.7 / 7.7, 1000 9.1 / 8.6; 600 x 8192 7.7 / 8.6, 680 10.0 / 9.3; 152 x 12288
// 4.1 / 4.6, 228 6.8 / 6.1; without it 600 x 6144 4.0 / 4.4, 680 5.4 / 4.7; 1200 x 4096 4.6 / 4.7, 1400
// 5.7 / 5.4. In fp32 without the residual it is norm_block_kernel with four vectors per thread, eight
// from more than 1280 vectors (us, block / this / bulk copies): 600 x 4096 4.5 / 4.8 / 5.2, 1000 8.0 /
// 6.5 / 6.9; 1400 x 2048 5.3 / 4.8 / 5.2; 500 x 8192 7.8 / 6.7 / 8.3, 1200 15.2 / 12.9 / 15.8; with it
// nothing beats the block (500 x 8192 11.5 against 13.4 with bulk copies, 1000 x 6144 16.0 / 17.0).
// Rows of up to 256 vectors without the residual hold out four waves (3000 x 2048 bf16 5.5 / 6.0, 7000
// 10.9 / 10.5); shorter ones in 16 bits any number (7000 x 1536 8.7 / 10.2).
static float norm_block_sm(int threads, int vpt, int ve) {
  return vpt == 2 && ve == 8 ? 1.f : (float)(2048 / threads);  // two 16-bit vectors per thread: 64 registers
}
// norm_row_kernel's ranges, in rows per SM: where its blocks still fit one wave (or two fit better
// than norm_block_kernel's). Block or bulk / this: residual 1400 x 2048 5.36 / 5.20; 640 x 4096 5.16 /
// 4.88, 760 5.66 / 5.52, 850 5.94 / 5.96; 620 x 8192 8.79 / 8.24, 850 10.75 / 10.50, 1000 11.9 / 12.0;
// without it 700 x 4096 3.10 / 2.96, 760 3.40 / 3.22, 680 2.94 / 2.94. Residual calls of 512 vectors
// beyond two waves take it too: 1600 / 3001 / 6000 rows 9.25 / 15.6 / 29.1 us against 9.49 / 15.8 /
// 29.6 with bulk copies.
struct NormRange { float lo, hi; };
static NormRange norm_row_range(bool res, int vpt) {
  if (!res) return vpt == 2 ? NormRange{4.5f, 5.25f} : NormRange{0.f, 0.f};
  return vpt == 1 ? NormRange{8.f, 12.f} : vpt == 2 ? NormRange{4.f, 5.25f} : NormRange{4.f, 6.f};
}
// Two rows per lane group of norm_rows_kernel (no residual, one vector per lane) from this many
// vectors of x per SM: half the threads have twice the loads in flight (16384 x 128 3.26 -> 2.90 us,
// 131072 x 128 15.3 -> 12.1; 8192 x 64, below the line, 1.98 / 2.16).
constexpr float kNormRows2Vecs = 1024.f;
// EDGE rows of 33 to 128 vectors take a block per row below this many rows, a warp per row (two or
// four vectors per lane, one after the other) from there, where the rate at which blocks start
// bounds the block per row; with the residual and more than 64 vectors always a block. Warp / block
// per row: 832 bf16 at 24 / 600 / 2400 / 5000 rows 2.59 / 1.65, 4.34 / 3.20, 5.02 / 4.51, 6.13 /
// 6.98 us; 333 at 2400 / 5000 4.11 / 4.08, 3.30 / 5.29; the residual on 1000 fp16 at 3 / 5000 /
// 30000 2.74 / 1.59, 12.4 / 8.1, 51.8 / 38.0. Up to 32 vectors a warp is enough: 101 at 24 / 2400
// rows 1.50 / 1.59, 2.88 / 3.45.
constexpr int64_t kNormEdgeRows = 3072;
// fp32 EDGE rows of more than 512 vectors take two vectors per thread from this many rows (more
// rows resident): 4000 x 3001 25.4 -> 20.6 us, with the residual 34.8 -> 30.7; 8559 x 2222 35.7 ->
// 29.6; at 300 rows 2.31 / 2.76. (16 bits: 3000 x 3999 12.5 / 13.7.) Up to 768 vectors without the residual
// from half as many: 1200 x 2222 5.55 / 4.57, 800 x 2222 4.20 / 4.89.
constexpr int64_t kNormEdgeWideRows = 2048;
// (Both on 152 SMs; norm_plan scales them.) EDGE rows of more than 1024 vectors without the residual:
// two vectors per thread leave one block per SM, which long calls do not hide. In fp32 eight per thread
// from one row per SM, six where two blocks fit (us, two / eight): 304 x 6001 5.5 / 4.8, 1200 17.8 / 13.9, 5000
// 67.7 / 47.9 (scalar accesses 61.0); 800 x 5001 8.9 / 8.6, 3000 26.4 / 23.5. In 16 bits from two rows per SM
// four up to 1280 vectors, eight up to 1536, as many as still give whole blocks an SM to share: 600 /
// 9000 x 9501 10.1 / 142 -> 8.4 / 99.5 (scalar 108), x 11201 11.6 / 156 -> 11.0 / 120 (127); 9001, where two
// blocks of two fit, 7.9 / 95 against 8.4 / 96. Above 1536 scalar accesses from 25 rows per SM: 4500 / 9000
// x 12478 85.2 / 166 -> 79.3 / 140, 3000 57.5 / 60.4 (four per thread 176 at 9000).
constexpr int kNormEdgeSms = 152;
constexpr int64_t kNormEdgeNever = (int64_t)1 << 40;

// Calls of few rows, in rows per SM. Rows of 33 to 128 vectors: norm_block_kernel, a vector per thread,
// instead of two or four per lane one after the other (warp / block, us): 64 x 1024 bf16 1.87 / 1.19, 2200
// 3.20 / 3.00, 3000 3.62 / 3.85; 1300 x 512 2.60 / 1.98, 2200 2.67 / 3.02; 1300 x 320 2.05 / 1.93, 1700
// 2.06 / 2.25; residual 64 x 1024 2.06 / 1.11, 2200 4.43 / 3.40, 4331 in fp16 4.73 / 5.42; 1300 x 320 2.25 / 2.10,
// 2200 2.65 / 3.22. Rows of 2048 vectors: eight per thread of 256 instead of two per thread of 1024, whose
// one block per SM waits longest on itself: 64 / 152 x 16384 bf16 2.63 / 3.63 -> 2.34 / 3.13, residual 3.91
// / 4.91 -> 3.42 / 4.17; fp32 only below half a row per SM (64 x 8192 3.04 -> 2.53, 100 3.40 / 3.97), with
// the residual only above 0.4 (40 x 8192 3.74 / 4.07, 100 4.75 -> 4.29).
static NormRange norm_few_range(bool res, int ve, int64_t nvec) {
  if (nvec == kNormBlockVecs) return ve == 8 ? NormRange{0.f, 1.f} : res ? NormRange{0.4f, 1.f} : NormRange{0.f, 0.5f};
  if (nvec > 32 && nvec <= 64) return {0.f, 9.f};
  if (nvec > 64 && nvec <= 128) return {0.f, res ? 16.f : 14.f};
  return {0.f, 0.f};
}
// EDGE rows in 16 bits, a block per row: from lo to hi threads per SM the loads stand in no branch
// (EDGE 2). With fewer, the branches' round trips hide in the launch; with more, the loads they save
// count. Branches / none, at an odd offset: 600 x 333 2.05 / 2.87 us, 900 3.67 / 2.93; 300 x 1001 2.42 /
// 3.29, 450 3.94 / 3.37, 900 4.08 / 3.34, 2000 4.56 / 4.67; 300 x 1537 3.81 / 3.42, 1333 4.26 / 4.42;
// residual 450 x 333 1.94 / 2.86, 1333 3.59 / 2.97; 600 x 1001 3.60 / 3.40, 900 3.19 / 3.82. With two
// vectors per thread never (80 x 12478 3.50 / 3.68). In fp32, with half the weights per vector, the branches are faster (600 x 1001 2.06 / 2.48).
static NormRange norm_edge_range(bool res) { return res ? NormRange{200.f, 570.f} : NormRange{300.f, 1280.f}; }

template <int DT>
__device__ __forceinline__ void load_gamma(const float* g, float* out) {
#pragma unroll
  for (int q = 0; q < Act<DT>::VE / 4; ++q) {
    const float4 v = ldg_f4(g + 4 * q);
    out[4 * q] = v.x; out[4 * q + 1] = v.y; out[4 * q + 2] = v.z; out[4 * q + 3] = v.w;
  }
}

// The weights of a vector whose first element is i, not a multiple of 4 (its offset from one, the
// same for the whole block): the aligned float4s around them, shifted, where those lie within
// the H weights and gamma itself is aligned; by element otherwise. By element everywhere, every
// weight load of a warp touched 32 sectors for 128 bytes. FLAT: without the branch that only a row's
// last vectors take: the last float4's weights one by one (past the row's end: the last weight, not
// used).
template <int DT, bool FLAT>
__device__ __forceinline__ void load_gamma_at(const float* gamma, int i, int H, float* out) {
  constexpr int VE = Act<DT>::VE;
  const int sh = i & 3, b = i - sh;
  if ((reinterpret_cast<uintptr_t>(gamma) & 15) == 0 && (FLAT || b + VE + 4 <= H)) {
    float t[VE + 4];
#pragma unroll
    for (int q = 0; q < VE / 4 + (FLAT ? 0 : 1); ++q) {
      const float4 v = ldg_f4(gamma + b + 4 * q);
      t[4 * q] = v.x; t[4 * q + 1] = v.y; t[4 * q + 2] = v.z; t[4 * q + 3] = v.w;
    }
    if (FLAT) {
#pragma unroll
      for (int j = 0; j < 3; ++j) t[VE + j] = __ldg(gamma + min(b + VE + j, H - 1));
    }
#pragma unroll
    for (int e = 0; e < VE; ++e) out[e] = sh < 2 ? (sh == 0 ? t[e] : t[e + 1]) : (sh == 2 ? t[e + 2] : t[e + 3]);
  } else {
#pragma unroll
    for (int e = 0; e < VE; ++e) out[e] = __ldg(gamma + i + e);
  }
}

// LPR lanes per row, VPT vectors per lane (VPT > 1 only with 32 lanes); lane l owns the
// vectors l + LPR * v. FULL: the lanes' vectors are exactly the row's. R rows per lane group at
// a time, their loads issued together. The grid covers every row, so the loop runs once.
template <int DT, bool RES, int LPR, int VPT, bool FULL, int R>
__global__ void __launch_bounds__(kThreads) norm_rows_kernel(const NormParams p) {
  pdl_trigger();
  constexpr int VE = Act<DT>::VE;
  constexpr int EB = Act<DT>::BYTES;
  constexpr int RPB = kThreads / LPR;
  const int lane = threadIdx.x % LPR;
  const unsigned mask =
      (LPR == 32) ? 0xffffffffu : (((1u << LPR) - 1u) << ((threadIdx.x & 31) & ~(LPR - 1)));
  const int64_t row0 = (int64_t)blockIdx.x * (RPB * R) + threadIdx.x / LPR;
  if (p.prefetch && (lane & 7) == 0) {  // the first row's lines (prefetch_l2)
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
      const int vi = lane + LPR * v;
      if (row0 < p.T && vi < p.nvec) {
        prefetch_l2(row_ptr(p.x, row0, p.x_rs, EB) + vi * 16);
        if (RES) prefetch_l2(row_ptr(p.r, row0, p.r_rs, EB) + vi * 16);
      }
    }
  }
  pdl_wait();
  for (int64_t base = row0; base < p.T; base += (int64_t)gridDim.x * (RPB * R)) {
    uint4 xv[R][VPT], rv[R][VPT];
    float g[VPT][VE];
#pragma unroll
    for (int k = 0; k < R; ++k) {
      const int64_t row = R == 1 ? base : min(base + k * RPB, p.T - 1);
#pragma unroll
      for (int v = 0; v < VPT; ++v) {
        const int vi = lane + LPR * v;
        if (FULL || vi < p.nvec) {
          xv[k][v] = ldg16(row_ptr(p.x, row, p.x_rs, EB) + vi * 16);
          if (RES) rv[k][v] = ldg16(row_ptr(p.r, row, p.r_rs, EB) + vi * 16);
          if (k == 0) load_gamma<DT>(p.gamma + vi * VE, g[v]);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < R; ++k) {
      const int64_t row = base + k * RPB;
      const bool on = R == 1 || row < p.T;
      float s[VPT][VE], ss = 0.f;
#pragma unroll
      for (int v = 0; v < VPT; ++v) {
        const int vi = lane + LPR * v;
        if (FULL || vi < p.nvec) {
          unpack<DT>(xv[k][v], s[v]);
          if (RES) {
            float rf[VE];
            unpack<DT>(rv[k][v], rf);
#pragma unroll
            for (int e = 0; e < VE; ++e) s[v][e] += rf[e];
            if (on) st16(row_ptr(p.r_out, row, p.ro_rs, EB) + vi * 16, pack<DT>(s[v]));
          }
#pragma unroll
          for (int e = 0; e < VE; ++e) ss = fmaf(s[v][e], s[v][e], ss);
        }
      }
#pragma unroll
      for (int o = LPR / 2; o > 0; o >>= 1) ss += __shfl_xor_sync(mask, ss, o, LPR);
      const float inv = rsqrtf(ss * p.inv_H + p.eps);
#pragma unroll
      for (int v = 0; v < VPT; ++v) {
        const int vi = lane + LPR * v;
        if (FULL || vi < p.nvec) {
#pragma unroll
          for (int e = 0; e < VE; ++e) s[v][e] = s[v][e] * inv * g[v][e];
          if (on) st16(row_ptr(p.y, row, p.y_rs, EB) + vi * 16, pack<DT>(s[v]));
        }
      }
    }
  }
}

// Sum over a block of any number of whole warps; every thread gets the same total. Up to 16
// warps by reading every warp's sum, beyond by a second round of shuffles.
__device__ __forceinline__ float norm_block_sum(float v, float* red) {
  const int nw = blockDim.x >> 5;
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  if (threadIdx.x < 32 && (int)threadIdx.x >= nw) red[threadIdx.x] = 0.f;
  __syncthreads();
  if (nw <= 16) {
    const float4* r4 = reinterpret_cast<const float4*>(red);
    const float4 a = r4[0], b = r4[1], c = r4[2], d = r4[3];
    return ((a.x + a.y) + (a.z + a.w)) + ((b.x + b.y) + (b.z + b.w)) +
           (((c.x + c.y) + (c.z + c.w)) + ((d.x + d.y) + (d.z + d.w)));
  }
  return warp_sum(red[threadIdx.x & 31]);
}

// Thread `tid` owns the row's vectors tid + blockDim.x * v, v < VPT. One vector per thread where
// the row allows it: at call sizes where latency counts, more threads with less each are faster
// (24 x 5120 1.35 us against 1.8 with two and 2.1 with four). Threads past the row's end load its
// last vector and drop it: with the loads behind a branch the compiler finished them before
// leaving it (256 x 4096 3.3 us). FULL: no such threads. EDGE: the row's tensors
// start at one common offset from a 16-byte boundary; the first peel and last tail elements
// (fewer than a vector each) go to threads of their own, and gamma is read by load_gamma_at. EDGE 2:
// every load without a branch (norm_edge_range).
template <int DT, bool RES, int VPT, int EDGE, bool FULL>
__global__ void __launch_bounds__(VPT >= 8 ? 256 : VPT >= 4 ? 512 : 1024) norm_block_kernel(const NormParams p) {
  pdl_trigger();
  __shared__ __align__(16) float red[32];
  constexpr int VE = Act<DT>::VE;
  constexpr int EB = Act<DT>::BYTES;
  const int tid = threadIdx.x;
  const int64_t row = blockIdx.x;
  const char* xr = row_ptr(p.x, row, p.x_rs, EB);
  const char* rr = RES ? row_ptr(p.r, row, p.r_rs, EB) : nullptr;
  int nvec = p.nvec, peel = 0, edge = -1;  // edge: this thread's scalar element
  if (EDGE) {
    peel = (int)((16 - (reinterpret_cast<uintptr_t>(xr) & 15)) & 15) / EB;
    if (peel > p.H) peel = (int)p.H;
    nvec = (int)(p.H - peel) / VE;
    const int tail = (int)p.H - peel - nvec * VE;
    if (tid < peel) edge = tid;
    else if (tid < peel + tail) edge = nvec * VE + tid;
    xr += peel * EB;
    if (RES) rr += peel * EB;
  }
  if (p.prefetch && (tid & 7) == 0) {  // the row's lines (prefetch_l2)
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
      const int vi = tid + (int)blockDim.x * v;
      if (vi < nvec) {
        prefetch_l2(xr + (int64_t)vi * 16);
        if (RES) prefetch_l2(rr + (int64_t)vi * 16);
      }
    }
  }
  pdl_wait();
  uint4 xv[VPT], rv[VPT];
  float g[VPT][VE], s[VPT][VE], es = 0.f, eg = 0.f;
#pragma unroll
  for (int v = 0; v < VPT; ++v) {
    const int vi = FULL ? tid + (int)blockDim.x * v : min(tid + (int)blockDim.x * v, nvec - 1);
    xv[v] = ldg16(xr + (int64_t)vi * 16);
    if (RES) rv[v] = ldg16(rr + (int64_t)vi * 16);
    if (EDGE) {
      load_gamma_at<DT, EDGE == 2>(p.gamma, peel + vi * VE, (int)p.H, g[v]);
    } else {
      load_gamma<DT>(p.gamma + (int64_t)vi * VE, g[v]);
    }
  }
  if (EDGE == 2 || (EDGE && edge >= 0)) {  // 2: threads without an edge element load the first and drop it
    const int ec = EDGE == 2 ? max(edge, 0) : edge;
    es = load_elem<DT>(p.x, row * p.x_rs + ec);
    if (RES) es += load_elem<DT>(p.r, row * p.r_rs + ec);
    eg = __ldg(p.gamma + ec);
    if (EDGE == 2 && edge < 0) es = 0.f;
  }
  char* ro = RES ? row_ptr(p.r_out, row, p.ro_rs, EB) + peel * EB : nullptr;
  float ss = EDGE ? es * es : 0.f;
#pragma unroll
  for (int v = 0; v < VPT; ++v) {
    const int vi = tid + (int)blockDim.x * v;
    float sv[VE], sq = 0.f;
    unpack<DT>(xv[v], sv);
    if (RES) {
      float rf[VE];
      unpack<DT>(rv[v], rf);
#pragma unroll
      for (int e = 0; e < VE; ++e) s[v][e] = sv[e] = sv[e] + rf[e];
      if (FULL || vi < nvec) st16(ro + (int64_t)vi * 16, pack<DT>(sv));
    }
#pragma unroll
    for (int e = 0; e < VE; ++e) sq = fmaf(sv[e], sv[e], sq);
    ss += FULL || vi < nvec ? sq : 0.f;
  }
  if (EDGE && RES && edge >= 0) store_elem<DT>(p.r_out, row * p.ro_rs + edge, es);
  const float inv = rsqrtf(norm_block_sum(ss, red) * p.inv_H + p.eps);
  char* yr = row_ptr(p.y, row, p.y_rs, EB) + peel * EB;
#pragma unroll
  for (int v = 0; v < VPT; ++v) {
    const int vi = tid + (int)blockDim.x * v;
    if (!RES) unpack<DT>(xv[v], s[v]);
#pragma unroll
    for (int e = 0; e < VE; ++e) s[v][e] = s[v][e] * inv * g[v][e];
    if (FULL || vi < nvec) st16(yr + (int64_t)vi * 16, pack<DT>(s[v]));
  }
  if (EDGE && edge >= 0) store_elem<DT>(p.y, row * p.y_rs + edge, es * inv * eg);
}

// Long calls of EDGE rows of at most 128 vectors: a warp per row, eight rows per block, VPT vectors per lane;
// a block per row (of one warp) was bound by the rate at which blocks start (20000 x 101 20.4 us).
template <int DT, bool RES, int VPT>
__global__ void __launch_bounds__(kThreads) norm_rows_edge_kernel(const NormParams p) {
  pdl_prologue();
  constexpr int VE = Act<DT>::VE;
  constexpr int EB = Act<DT>::BYTES;
  const int lane = threadIdx.x & 31, H = (int)p.H;
  const int64_t row = (int64_t)blockIdx.x * (kThreads / 32) + threadIdx.x / 32;
  if (row >= p.T) return;
  const char* xr = row_ptr(p.x, row, p.x_rs, EB);
  const int peel = (int)((16 - (reinterpret_cast<uintptr_t>(xr) & 15)) & 15) / EB;
  const int nvec = (H - peel) / VE, tail = H - peel - nvec * VE;
  const int edge = lane < peel ? lane : (lane < peel + tail ? nvec * VE + lane : -1);
  xr += peel * EB;
  const char* rr = RES ? row_ptr(p.r, row, p.r_rs, EB) + peel * EB : nullptr;
  uint4 xv[VPT], rv[VPT];
  float g[VPT][VE], s[VPT][VE], es = 0.f, eg = 0.f, ss = 0.f;
#pragma unroll
  for (int v = 0; v < VPT; ++v) {  // lanes past the row's end load its last vector and drop it
    const int vi = min(lane + 32 * v, nvec - 1);
    xv[v] = ldg16(xr + vi * 16);
    if (RES) rv[v] = ldg16(rr + vi * 16);
    load_gamma_at<DT, false>(p.gamma, peel + vi * VE, H, g[v]);
  }
  if (edge >= 0) {
    es = load_elem<DT>(p.x, row * p.x_rs + edge);
    if (RES) es += load_elem<DT>(p.r, row * p.r_rs + edge);
    eg = __ldg(p.gamma + edge);
    ss = es * es;
    if (RES) store_elem<DT>(p.r_out, row * p.ro_rs + edge, es);
  }
  char* ro = RES ? row_ptr(p.r_out, row, p.ro_rs, EB) + peel * EB : nullptr;
#pragma unroll
  for (int v = 0; v < VPT; ++v) {
    const int vi = lane + 32 * v;
    float sq = 0.f;
    unpack<DT>(xv[v], s[v]);
    if (RES) {
      float rf[VE];
      unpack<DT>(rv[v], rf);
#pragma unroll
      for (int e = 0; e < VE; ++e) s[v][e] += rf[e];
      if (vi < nvec) st16(ro + vi * 16, pack<DT>(s[v]));
    }
#pragma unroll
    for (int e = 0; e < VE; ++e) sq = fmaf(s[v][e], s[v][e], sq);
    ss += vi < nvec ? sq : 0.f;
  }
  const float inv = rsqrtf(warp_sum(ss) * p.inv_H + p.eps);
  char* yr = row_ptr(p.y, row, p.y_rs, EB) + peel * EB;
#pragma unroll
  for (int v = 0; v < VPT; ++v) {
    const int vi = lane + 32 * v;
#pragma unroll
    for (int e = 0; e < VE; ++e) s[v][e] = s[v][e] * inv * g[v][e];
    if (vi < nvec) st16(yr + vi * 16, pack<DT>(s[v]));
  }
  if (edge >= 0) store_elem<DT>(p.y, row * p.y_rs + edge, es * inv * eg);
}

// Long calls: the row's x (and r) are staged in shared memory by bulk copies (cp.async.bulk,
// completion counted on an mbarrier) issued by one thread, while every thread loads its gamma
// vectors; s = x + r is formed from shared memory twice (the same fp32 addition both times). With
// the rows out of the registers more of them are in flight per SM. Two vectors per thread with a
// residual (40 registers), four without, where the fewer threads leave room for more blocks
// (16384 x 5120 50.7 us against 52-61 with two). gamma loaded after the reduction instead cost
// 2-3 us per call. The wait is bounded: if it runs out, the block sets TRIDENT_DEVERR_TIMEOUT,
// waits again (bounded) for its copies and returns without writing.
// NT, MB: at most NT threads, at least MB blocks per SM. Without the residual and its bound, 64 registers
// left two blocks of 272 to 384 threads (rows of 1025 to 1536 vectors): 7000 x 10752 57.8 us, 49.4 with three,
// the two-pass kernel before 52.5; wider rows, two blocks of up to 512 either way, take eight vectors per
// thread of 256: 7000 x 12544 64.6 -> 59.3 (61.1), 4000 x 16384 44.4 -> 40.3.
template <int DT, bool RES, int VPT, bool FULL, int NT, int MB>
__global__ void __launch_bounds__(NT, MB) norm_bulk_kernel(const NormParams p) {
  constexpr int VE = Act<DT>::VE;
  constexpr int EB = Act<DT>::BYTES;
  extern __shared__ __align__(128) uint4 s_rows[];
  __shared__ __align__(8) unsigned long long bar;
  __shared__ __align__(16) float red[32];
  const int tid = threadIdx.x, nt = blockDim.x, nvec = p.nvec;
  const int64_t row = blockIdx.x;
  const uint32_t bar_a = (uint32_t)__cvta_generic_to_shared(&bar);
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(bar_a) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  pdl_trigger();
  pdl_wait();
  if (tid == 0) {
    const uint32_t rb = (uint32_t)nvec * 16;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                 :: "r"(bar_a), "r"((RES ? 2 : 1) * rb) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"((uint32_t)__cvta_generic_to_shared(s_rows)), "l"(row_ptr(p.x, row, p.x_rs, EB)),
                    "r"(rb), "r"(bar_a) : "memory");
    if (RES)
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                   :: "r"((uint32_t)__cvta_generic_to_shared(s_rows + nvec)), "l"(row_ptr(p.r, row, p.r_rs, EB)),
                      "r"(rb), "r"(bar_a) : "memory");
  }
  float g[VPT][VE];
#pragma unroll
  for (int v = 0; v < VPT; ++v) load_gamma<DT>(p.gamma + (int64_t)(FULL ? tid + nt * v : min(tid + nt * v, nvec - 1)) * VE, g[v]);
  __syncthreads();  // the barrier is initialised before anyone waits on it
  auto landed = [&](uint32_t polls) -> bool {
    uint32_t done = 0;
    for (uint32_t it = 0; it < polls && !done; ++it)
      asm volatile("{ .reg .pred q; mbarrier.try_wait.parity.shared::cta.b64 q, [%1], 0; selp.u32 %0, 1, 0, q; }"
                   : "=r"(done) : "r"(bar_a) : "memory");
    return done != 0;
  };
  const bool ok = landed(p.first_wait_polls);
  if (__syncthreads_or(!ok)) {  // one decision for the whole block
    if (tid == 0 && p.err) atomicOr(p.err, kErrTimeout);
    if (!ok) landed(kBulkWaitPolls);  // a second bounded wait for the copies before the block exits
    return;
  }
  char* ro = RES ? row_ptr(p.r_out, row, p.ro_rs, EB) : nullptr;
  float ss = 0.f;
#pragma unroll
  for (int v = 0; v < VPT; ++v) {
    const int vi = tid + nt * v, vc = FULL ? vi : min(vi, nvec - 1);
    float sv[VE], sq = 0.f;
    unpack<DT>(s_rows[vc], sv);
    if (RES) {
      float rf[VE];
      unpack<DT>(s_rows[nvec + vc], rf);
#pragma unroll
      for (int e = 0; e < VE; ++e) sv[e] += rf[e];
      if (FULL || vi < nvec) st16(ro + (int64_t)vi * 16, pack<DT>(sv));
    }
#pragma unroll
    for (int e = 0; e < VE; ++e) sq = fmaf(sv[e], sv[e], sq);
    ss += FULL || vi < nvec ? sq : 0.f;
  }
  const float inv = rsqrtf(norm_block_sum(ss, red) * p.inv_H + p.eps);
  char* yr = row_ptr(p.y, row, p.y_rs, EB);
#pragma unroll
  for (int v = 0; v < VPT; ++v) {
    const int vi = tid + nt * v, vc = FULL ? vi : min(vi, nvec - 1);
    float sv[VE];
    unpack<DT>(s_rows[vc], sv);
    if (RES) {
      float rf[VE];
      unpack<DT>(s_rows[nvec + vc], rf);
#pragma unroll
      for (int e = 0; e < VE; ++e) sv[e] += rf[e];
    }
#pragma unroll
    for (int e = 0; e < VE; ++e) sv[e] = sv[e] * inv * g[v][e];
    if (FULL || vi < nvec) st16(yr + (int64_t)vi * 16, pack<DT>(sv));
  }
}

// Rows of exactly VPT vectors per thread of 256, in 16 bits: fewer and longer-lived blocks than
// norm_block_kernel's, which fit one wave up to a third more rows (norm_row_range). A block has one
// row, so the loop runs once; it holds the weights' loads in front of the reduction, behind which
// ptxas otherwise moves them, a second round trip (residual 700 x 8192 9.2 us, without it 11.1).
template <int DT, bool RES, int VPT>
__global__ void __launch_bounds__(kThreads) norm_row_kernel(const NormParams p) {
  pdl_trigger();
  __shared__ float red[kThreads / 32];
  constexpr int EB = Act<DT>::BYTES;
  constexpr int VE = Act<DT>::VE;
  const int tid = threadIdx.x;
  pdl_wait();
  for (int64_t row = blockIdx.x; row < p.T; row += gridDim.x) {
    const uint4* xp = reinterpret_cast<const uint4*>(row_ptr(p.x, row, p.x_rs, EB));
    const uint4* rp = RES ? reinterpret_cast<const uint4*>(row_ptr(p.r, row, p.r_rs, EB)) : nullptr;
    uint4 xv[VPT], rv[VPT];
    float g[VPT][VE], s[VPT][VE];
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
      const int64_t vi = (int64_t)v * kThreads + tid;
      xv[v] = ldg16(xp + vi);
      if (RES) rv[v] = ldg16(rp + vi);
      load_gamma<DT>(p.gamma + vi * VE, g[v]);
    }
    uint4* rop = RES ? reinterpret_cast<uint4*>(row_ptr(p.r_out, row, p.ro_rs, EB)) : nullptr;
    float ss = 0.f;
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
      unpack<DT>(xv[v], s[v]);
      if (RES) {
        float rf[VE];
        unpack<DT>(rv[v], rf);
#pragma unroll
        for (int e = 0; e < VE; ++e) s[v][e] += rf[e];
      }
#pragma unroll
      for (int e = 0; e < VE; ++e) ss = fmaf(s[v][e], s[v][e], ss);
      if (RES) st16(rop + (int64_t)v * kThreads + tid, pack<DT>(s[v]));
    }
    const float inv = rsqrtf(block_sum(ss, red) * p.inv_H + p.eps);
    uint4* yp = reinterpret_cast<uint4*>(row_ptr(p.y, row, p.y_rs, EB));
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
      float y[VE];
      if (!RES) unpack<DT>(xv[v], s[v]);
#pragma unroll
      for (int e = 0; e < VE; ++e) y[e] = s[v][e] * inv * g[v][e];
      st16(yp + (int64_t)v * kThreads + tid, pack<DT>(y));
    }
    __syncthreads();  // before the next row's sums
  }
}

// Two passes: the first only reduces, the second recomputes s and writes, so that in-place
// calls (r_out = r, y = x) never read a value they already overwrote.
template <int DT, bool RES>
__global__ void __launch_bounds__(kThreads) norm_loop_kernel(const NormParams p) {
  pdl_prologue();
  __shared__ __align__(16) float red[32];
  constexpr int EB = Act<DT>::BYTES;
  constexpr int VE = Act<DT>::VE;
  const int tid = threadIdx.x;
  const int64_t row = blockIdx.x, nvec = p.H / VE;
  const uint4* x = reinterpret_cast<const uint4*>(row_ptr(p.x, row, p.x_rs, EB));
  const uint4* r = RES ? reinterpret_cast<const uint4*>(row_ptr(p.r, row, p.r_rs, EB)) : nullptr;
  float ss = 0.f;
  for (int64_t vi = tid; vi < nvec; vi += kThreads) {
    float xf[VE], rf[VE];
    unpack<DT>(ld16(x + vi), xf);
    if (RES) unpack<DT>(ld16(r + vi), rf);
#pragma unroll
    for (int e = 0; e < VE; ++e) {
      const float s = RES ? xf[e] + rf[e] : xf[e];
      ss = fmaf(s, s, ss);
    }
  }
  const float inv = rsqrtf(norm_block_sum(ss, red) * p.inv_H + p.eps);
  uint4* y = reinterpret_cast<uint4*>(row_ptr(p.y, row, p.y_rs, EB));
  uint4* ro = RES ? reinterpret_cast<uint4*>(row_ptr(p.r_out, row, p.ro_rs, EB)) : nullptr;
  for (int64_t vi = tid; vi < nvec; vi += kThreads) {
    float xf[VE], rf[VE], g[VE];
    unpack<DT>(ld16(x + vi), xf);
    if (RES) {
      unpack<DT>(ld16(r + vi), rf);
#pragma unroll
      for (int e = 0; e < VE; ++e) xf[e] += rf[e];
      st16(ro + vi, pack<DT>(xf));
    }
    load_gamma<DT>(p.gamma + vi * VE, g);
#pragma unroll
    for (int e = 0; e < VE; ++e) xf[e] = xf[e] * inv * g[e];
    st16(y + vi, pack<DT>(xf));
  }
}

// The loop goes on only past 2^31 - 1 rows, the grid's limit.
template <int DT, bool RES>
__global__ void __launch_bounds__(kThreads) norm_generic_kernel(const NormParams p) {
  pdl_prologue();
  __shared__ __align__(16) float red[32];
  const int tid = threadIdx.x;
  for (int64_t row = blockIdx.x; row < p.T; row += gridDim.x) {
    const int64_t xo = row * p.x_rs, ro = row * p.r_rs;
    float ss = 0.f;
    for (int64_t j = tid; j < p.H; j += kThreads) {
      const float s = RES ? load_elem<DT>(p.x, xo + j) + load_elem<DT>(p.r, ro + j) : load_elem<DT>(p.x, xo + j);
      ss = fmaf(s, s, ss);
    }
    const float inv = rsqrtf(norm_block_sum(ss, red) * p.inv_H + p.eps);
    for (int64_t j = tid; j < p.H; j += kThreads) {
      const float s = RES ? load_elem<DT>(p.x, xo + j) + load_elem<DT>(p.r, ro + j) : load_elem<DT>(p.x, xo + j);
      if (RES) store_elem<DT>(p.r_out, row * p.ro_rs + j, s);
      store_elem<DT>(p.y, row * p.y_rs + j, s * inv * p.gamma[j]);
    }
    __syncthreads();  // `red` is reused by the next row
  }
}

constexpr int kNormRowsVecs = 128;    // rows of at most this many vectors: norm_rows_kernel, but in calls of few rows

// Threads of a block for a row of nvec vectors at vpt per thread.
static int norm_threads(int64_t nvec, int vpt) { return (int)(((nvec + vpt - 1) / vpt + 31) / 32 * 32); }

template <int DT, bool RES, int LPR, int VPT>
static void pick_rows(int64_t nvec, KernelEntry* out) {
  const bool full = nvec == LPR * VPT;
  out->rows = kThreads / LPR;
  out->nm_fn[NM_VEC] = full ? (const void*)norm_rows_kernel<DT, RES, LPR, VPT, true, 1>
                            : (const void*)norm_rows_kernel<DT, RES, LPR, VPT, false, 1>;
  if constexpr (!RES && VPT == 1) {
    out->nm_fn[NM_LARGE] = full ? (const void*)norm_rows_kernel<DT, RES, LPR, VPT, true, 2>
                                : (const void*)norm_rows_kernel<DT, RES, LPR, VPT, false, 2>;
    out->large_per = kThreads / LPR * 2;
    out->large_sm = kNormRows2Vecs / (float)nvec;
  }
}

template <int DT, bool RES>
static const void* norm_bulk(int64_t nvec, int vpt, bool full) {
  if constexpr (RES) {
    if (vpt == 2) return full ? (const void*)norm_bulk_kernel<DT, RES, 2, true, 512, 3>
                              : (const void*)norm_bulk_kernel<DT, RES, 2, false, 512, 3>;
    return full ? (const void*)norm_bulk_kernel<DT, RES, 4, true, 512, 2>
                : (const void*)norm_bulk_kernel<DT, RES, 4, false, 512, 2>;
  } else {
    if (nvec <= 1024) return full ? (const void*)norm_bulk_kernel<DT, RES, 4, true, 512, 1>
                                  : (const void*)norm_bulk_kernel<DT, RES, 4, false, 512, 1>;
    if (vpt == 4) return full ? (const void*)norm_bulk_kernel<DT, RES, 4, true, 384, 3>
                              : (const void*)norm_bulk_kernel<DT, RES, 4, false, 384, 3>;
    return full ? (const void*)norm_bulk_kernel<DT, RES, 8, true, 256, 3>
                : (const void*)norm_bulk_kernel<DT, RES, 8, false, 256, 3>;
  }
}

template <int DT, bool RES>
static void pick(int64_t H, KernelEntry* out) {
  constexpr int VE = Act<DT>::VE;
  const int64_t nvec = H / VE;
  for (int k = 0; k < kNormEntries; ++k) {
    out->nm_fn[k] = nullptr;
    out->nm_threads[k] = kThreads;
  }
  out->nm_fn[NM_GENERIC] = (const void*)norm_generic_kernel<DT, RES>;
  out->rows = out->large_per = 1;
  out->large_sm = out->mid_lo = out->mid_hi = out->few_lo = out->few_hi = out->edge_lo = out->edge_hi = 0.f;
  out->large_smem = 0;
  const int vpt = nvec <= 1024 ? 1 : 2;
  const int threads = norm_threads(nvec, vpt);
  const NormRange few = norm_few_range(RES, VE, nvec);
  if (H % VE == 0 && few.hi > 0.f) {
    const int fv = nvec <= kNormRowsVecs ? 1 : 8;
    const int ft = norm_threads(nvec, fv);
    out->few_lo = few.lo;
    out->few_hi = few.hi;
    out->nm_threads[NM_FEW] = ft;
    out->nm_fn[NM_FEW] = fv == 8 ? (const void*)norm_block_kernel<DT, RES, 8, 0, true>
                         : ft == nvec ? (const void*)norm_block_kernel<DT, RES, 1, 0, true>
                                      : (const void*)norm_block_kernel<DT, RES, 1, 0, false>;
  }
  // rows that begin anywhere hold nvec or nvec - 1 whole vectors, and at least one
  out->edge_rows = 1;
  out->edge_many = kNormEdgeNever;
  if (nvec >= 2 && nvec <= kNormBlockVecs) {
    out->nm_threads[NM_EDGE] = threads;
    if constexpr (VE == 8) {
      if (vpt == 1) {
        const NormRange r = norm_edge_range(RES);
        out->edge_lo = r.lo / (float)threads;
        out->edge_hi = r.hi / (float)threads;
        out->nm_threads[NM_EDGE_FLAT] = threads;
        out->nm_fn[NM_EDGE_FLAT] = (const void*)norm_block_kernel<DT, RES, 1, 2, false>;
      }
    }
    out->nm_fn[NM_EDGE] = vpt == 1 ? (const void*)norm_block_kernel<DT, RES, 1, 1, false>
                                   : (const void*)norm_block_kernel<DT, RES, 2, 1, false>;
    if (nvec <= 64 || (!RES && nvec <= kNormRowsVecs)) {
      out->edge_rows = kThreads / 32;
      out->edge_many = nvec <= 32 ? 0 : kNormEdgeRows;
      if (nvec <= 32) out->nm_fn[NM_EDGE_MANY] = (const void*)norm_rows_edge_kernel<DT, RES, 1>;
      else if (nvec <= 64) out->nm_fn[NM_EDGE_MANY] = (const void*)norm_rows_edge_kernel<DT, RES, 2>;
      else if constexpr (!RES) out->nm_fn[NM_EDGE_MANY] = (const void*)norm_rows_edge_kernel<DT, RES, 4>;
    } else if (VE == 4 && vpt == 1 && nvec > 512) {
      out->edge_many = RES || nvec > 768 ? kNormEdgeWideRows : kNormEdgeWideRows / 2;
      out->nm_threads[NM_EDGE_MANY] = norm_threads(nvec, 2);
      out->nm_fn[NM_EDGE_MANY] = (const void*)norm_block_kernel<DT, RES, 2, 1, false>;
    } else if constexpr (!RES) {
      const int ev = nvec <= (VE == 8 ? 1152 : 1024) ? 0 : VE == 8 && nvec <= 1280 ? 4 : VE == 8 && nvec > 1536 ? 1 : 8;
      if (ev == 1) {
        out->edge_many = (threads <= 832 ? 25 : 40) * kNormEdgeSms;
        out->nm_fn[NM_EDGE_MANY] = out->nm_fn[NM_GENERIC];
      } else if (ev) {
        out->edge_many = (VE == 8 ? 2 : threads <= 640 ? 6 : 1) * kNormEdgeSms + 1;
        out->nm_threads[NM_EDGE_MANY] = norm_threads(nvec, ev);
        out->nm_fn[NM_EDGE_MANY] = ev == 4 ? (const void*)norm_block_kernel<DT, RES, 4, 1, false>
                                           : (const void*)norm_block_kernel<DT, RES, 8, 1, false>;
      }
    }
  }
  if (H % VE != 0) return;
  if (nvec <= kNormRowsVecs) {
    if (nvec > 64) pick_rows<DT, RES, 32, 4>(nvec, out);
    else if (nvec > 32) pick_rows<DT, RES, 32, 2>(nvec, out);
    else if (nvec > 16) pick_rows<DT, RES, 32, 1>(nvec, out);
    else if (nvec > 8) pick_rows<DT, RES, 16, 1>(nvec, out);
    else if (nvec > 4) pick_rows<DT, RES, 8, 1>(nvec, out);
    else if (nvec > 2) pick_rows<DT, RES, 4, 1>(nvec, out);
    else if (nvec > 1) pick_rows<DT, RES, 2, 1>(nvec, out);
    else pick_rows<DT, RES, 1, 1>(nvec, out);
  } else if (nvec <= kNormBlockVecs) {
    const bool full = threads * vpt == nvec;
    out->nm_threads[NM_VEC] = threads;
    out->nm_fn[NM_VEC] = vpt == 1 ? (full ? (const void*)norm_block_kernel<DT, RES, 1, 0, true>
                                          : (const void*)norm_block_kernel<DT, RES, 1, 0, false>)
                                  : (full ? (const void*)norm_block_kernel<DT, RES, 2, 0, true>
                                          : (const void*)norm_block_kernel<DT, RES, 2, 0, false>);
    const float wave = norm_block_sm(threads, vpt, VE);
    out->large_sm = vpt == 2 ? wave : (!RES && nvec <= 256 ? 4 : 2) * wave;
    if constexpr (VE == 8) {
      if (RES || nvec >= 256) {
        const int bv = RES ? (nvec <= 1024 ? 2 : 4) : nvec <= 1536 ? 4 : 8;
        const int bt = norm_threads(nvec, bv);
        const bool bfull = bt * bv == nvec;
        out->nm_threads[NM_LARGE] = bt;
        out->nm_fn[NM_LARGE] = norm_bulk<DT, RES>(nvec, bv, bfull);
        out->large_smem = (int32_t)(nvec * 16 * (RES ? 2 : 1));
      }
      const int rv = nvec % kThreads == 0 ? (int)(nvec / kThreads) : 0;
      if (RES && rv == 1) out->nm_fn[NM_MID] = (const void*)norm_row_kernel<DT, RES, 1>;
      if (RES && rv == 4) out->nm_fn[NM_MID] = (const void*)norm_row_kernel<DT, RES, 4>;
      if (rv == 2) out->nm_fn[NM_MID] = (const void*)norm_row_kernel<DT, RES, 2>;
      if (out->nm_fn[NM_MID]) {
        const NormRange r = norm_row_range(RES, rv);
        out->mid_lo = r.lo;
        out->mid_hi = r.hi;
      }
      if (RES && rv == 2) {
        out->nm_threads[NM_LARGE] = kThreads;
        out->nm_fn[NM_LARGE] = out->nm_fn[NM_MID];
        out->large_smem = 0;
      }
    } else if constexpr (!RES) {
      const int bv = nvec <= 1280 ? 4 : 8;
      const int bt = norm_threads(nvec, bv);
      const bool bfull = bt * bv == nvec;
      out->nm_threads[NM_LARGE] = bt;
      out->nm_fn[NM_LARGE] = bv == 4 ? (bfull ? (const void*)norm_block_kernel<DT, RES, 4, 0, true>
                                              : (const void*)norm_block_kernel<DT, RES, 4, 0, false>)
                                     : (bfull ? (const void*)norm_block_kernel<DT, RES, 8, 0, true>
                                              : (const void*)norm_block_kernel<DT, RES, 8, 0, false>);
    }
  } else {
    out->nm_fn[NM_VEC] = (const void*)norm_loop_kernel<DT, RES>;
  }
}

bool norm_kernel(bool res, int32_t dtype, int32_t variant, int64_t H, KernelEntry* out, const char** why) {
  if (dtype != DT_BF16 && dtype != DT_FP16 && dtype != DT_FP32) { *why = "dtype"; return false; }
  if (H < 1) { *why = "H must be >= 1"; return false; }
  const int eb = dtype == DT_FP32 ? 4 : 2;
  if (variant != 1 && (H * eb) % 16 != 0) { *why = "the vector norms need H * elem_size % 16 == 0"; return false; }
  out->kind = KK_NORM;
  out->vec = 16 / eb;
  if (dtype == DT_BF16) res ? pick<DT_BF16, true>(H, out) : pick<DT_BF16, false>(H, out);
  else if (dtype == DT_FP16) res ? pick<DT_FP16, true>(H, out) : pick<DT_FP16, false>(H, out);
  else res ? pick<DT_FP32, true>(H, out) : pick<DT_FP32, false>(H, out);
  out->fn = out->nm_fn[NM_GENERIC];
  return true;
}

NormEntry norm_plan(const KernelEntry& ke, NormParams* p, bool res, int32_t eb, int32_t* threads, int64_t* blocks,
                    int32_t* smem, int32_t sms) {
  const uintptr_t off = (uintptr_t)p->x & 15;
  const int64_t ve = 16 / eb, rs = p->x_rs % ve;
  // all rows of all tensors share their offsets from 16-byte boundaries
  const bool together = ((uintptr_t)p->y & 15) == off &&
                        (!res || (((uintptr_t)p->r & 15) == off && ((uintptr_t)p->r_out & 15) == off)) &&
                        (p->T <= 1 || (p->y_rs % ve == rs && (!res || (p->r_rs % ve == rs && p->ro_rs % ve == rs))));
  const bool aligned = together && off == 0 && (p->T <= 1 || rs == 0) && ((uintptr_t)p->gamma & 15) == 0;
  p->nvec = (int32_t)(p->H / ve < INT32_MAX ? p->H / ve : INT32_MAX);  // the loop kernel counts its own
  NormEntry e = NM_GENERIC;
  const float rows_sm = (float)p->T / (float)sms;
  if (aligned && ke.nm_fn[NM_VEC])
    e = ke.nm_fn[NM_FEW] && rows_sm > ke.few_lo && rows_sm <= ke.few_hi ? NM_FEW
        : ke.nm_fn[NM_MID] && rows_sm > ke.mid_lo && rows_sm <= ke.mid_hi ? NM_MID
        : ke.nm_fn[NM_LARGE] && rows_sm > ke.large_sm ? NM_LARGE : NM_VEC;
  else if (together && ke.nm_fn[NM_EDGE] && p->T <= INT32_MAX)
    e = p->T >= ke.edge_many * sms / kNormEdgeSms ? NM_EDGE_MANY
        : ke.nm_fn[NM_EDGE_FLAT] && rows_sm > ke.edge_lo && rows_sm <= ke.edge_hi ? NM_EDGE_FLAT : NM_EDGE;
  *threads = ke.nm_threads[e];
  *smem = e == NM_LARGE ? ke.large_smem : 0;
  const int64_t per = e == NM_VEC ? ke.rows : e == NM_LARGE ? ke.large_per : e == NM_EDGE_MANY ? ke.edge_rows : 1;
  *blocks = (p->T + per - 1) / per;
  return e;
}

}  // namespace trident
