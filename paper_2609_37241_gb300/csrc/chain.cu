// chain.cu -- one decoder layer's non-GEMM chain in a single launch.
//
//   add+RMSNorm(h, r0) -> x1, r1;  [q/k RMSNorm +] RoPE(q, k) + KV append;
//   add+RMSNorm(attn_out, r1) -> x2, r2;  SwiGLU(g, u) -> o
//
// The only data dependency inside the chain is r1 feeding the second norm, and it is
// row-local: the block that produces row t of r1 keeps it in registers and runs the
// second norm of row t itself. So no grid-wide barrier is needed; the launch is a
// horizontal fusion where blocks take different roles:
//   norm     two add+RMSNorm steps, one or two blocks per token (the longest per-block
//            work)
//   RoPE     RoPE/KV head-rows, a warp item per warp (RopeGeom), or per few warps of a block on
//            small grids: one head-row per lane group, or up to three of one token on grids
//            several waves long
//   SwiGLU   tiles of one row each, twice as wide on grids of many waves
// Grids are role-major ([norms | RoPE | SwiGLU], so the longest blocks start first), the
// smallest ones token-major (chain_block_tok), so that consecutive blocks mix roles. Under
// programmatic dependent launch, role-major grids that fit the resident slots with their
// own norm blocks run the LATE entry, whose short blocks trigger the next launch only at
// their exit (the next grid is then placed one norm block per SM). One launch replaces
// four, which is what matters at decode sizes, where each step moves well under a
// microsecond of HBM traffic. chain_step_kernel runs several independent calls' grids in
// one launch.
#include "device_common.cuh"

namespace trident {

// Norm role: part `part` (< SPLIT) of token `row`'s two add+RMSNorm steps.
template <int DT, int NT, int VPT, int SPLIT>
__device__ __forceinline__ void chain_norm(const ChainParams& c, const int64_t row, const int part) {
  constexpr int EB = Act<DT>::BYTES;
  constexpr int VE = Act<DT>::VE;
  const int tid = threadIdx.x;
  {
    // Both norms of one token. The second residual sum s2 = attn_out + round(s1) is
    // elementwise, so both sums of squares are formed before any reduction and reduced
    // together: one barrier. With a_split = 2 two CTAs share a token: each reads the whole
    // row (the sums need it) but loads only its half of both gamma vectors and writes only
    // its half of the four outputs, so no SM carries the token's full 56 KB. s1 and s2 are
    // recomputed from the packed inputs after the reduction rather than kept in registers.
    __shared__ float2 red[NT / 32];
    constexpr int PP = VPT / SPLIT;  // vectors per thread this CTA writes
    static_assert(VPT % SPLIT == 0, "split");
    const NormParams& n1 = c.n1;
    const NormParams& n2 = c.n2;
    uint4 hv[VPT], rv[VPT], av[VPT];
    float ga[PP][VE], gm[PP][VE];
    const uint4* hp = reinterpret_cast<const uint4*>(row_ptr(n1.x, row, n1.x_rs, EB));
    const uint4* rp = reinterpret_cast<const uint4*>(row_ptr(n1.r, row, n1.r_rs, EB));
    const uint4* ap = reinterpret_cast<const uint4*>(row_ptr(n2.x, row, n2.x_rs, EB));
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
      const int64_t vi = (int64_t)v * NT + tid;
      hv[v] = ldg16(hp + vi);
      rv[v] = ldg16(rp + vi);
      av[v] = ldg16(ap + vi);
      if (v / PP == part) {
#pragma unroll
        for (int q = 0; q < VE / 4; ++q) {
          const float4 g1 = ldg_f4(n1.gamma + vi * VE + 4 * q);
          const float4 g2 = ldg_f4(n2.gamma + vi * VE + 4 * q);
          float* a = ga[v % PP];
          float* m = gm[v % PP];
          a[4 * q] = g1.x; a[4 * q + 1] = g1.y; a[4 * q + 2] = g1.z; a[4 * q + 3] = g1.w;
          m[4 * q] = g2.x; m[4 * q + 1] = g2.y; m[4 * q + 2] = g2.z; m[4 * q + 3] = g2.w;
        }
      }
    }
    uint4* r1p = reinterpret_cast<uint4*>(row_ptr(n1.r_out, row, n1.ro_rs, EB));
    uint4* r2p = reinterpret_cast<uint4*>(row_ptr(n2.r_out, row, n2.ro_rs, EB));
    float ss1 = 0.f, ss2 = 0.f;
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
      const int64_t vi = (int64_t)v * NT + tid;
      float hf[VE], rf[VE], af[VE], s1[VE], s2[VE];
      unpack<DT>(hv[v], hf);
      unpack<DT>(rv[v], rf);
      unpack<DT>(av[v], af);
#pragma unroll
      for (int e = 0; e < VE; ++e) {
        s1[e] = hf[e] + rf[e];
        ss1 = fmaf(s1[e], s1[e], ss1);
      }
      const uint4 r1 = pack<DT>(s1);
      float r1f[VE];
      unpack<DT>(r1, r1f);
#pragma unroll
      for (int e = 0; e < VE; ++e) {
        s2[e] = af[e] + r1f[e];
        ss2 = fmaf(s2[e], s2[e], ss2);
      }
      if (v / PP == part) {
        st16(r1p + vi, r1);              // r1, then r2: in place (r2 = r1) keeps r2
        st16(r2p + vi, pack<DT>(s2));
      }
    }
    float2 sums = make_float2(ss1, ss2);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      sums.x += __shfl_xor_sync(0xffffffffu, sums.x, o);
      sums.y += __shfl_xor_sync(0xffffffffu, sums.y, o);
    }
    if ((tid & 31) == 0) red[tid >> 5] = sums;
    __syncthreads();
    float2 tot = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < NT / 32; ++i) {
      tot.x += red[i].x;
      tot.y += red[i].y;
    }
    const float inv1 = rsqrtf(tot.x * n1.inv_H + n1.eps);
    const float inv2 = rsqrtf(tot.y * n2.inv_H + n2.eps);
    uint4* x1p = reinterpret_cast<uint4*>(row_ptr(n1.y, row, n1.y_rs, EB));
    uint4* x2p = reinterpret_cast<uint4*>(row_ptr(n2.y, row, n2.y_rs, EB));
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
      if (v / PP != part) continue;
      const int64_t vi = (int64_t)v * NT + tid;
      float hf[VE], rf[VE], af[VE], s1[VE], y1[VE], y2[VE];
      unpack<DT>(hv[v], hf);
      unpack<DT>(rv[v], rf);
      unpack<DT>(av[v], af);
#pragma unroll
      for (int e = 0; e < VE; ++e) s1[e] = hf[e] + rf[e];
      float r1f[VE];
      unpack<DT>(pack<DT>(s1), r1f);
#pragma unroll
      for (int e = 0; e < VE; ++e) {
        y1[e] = s1[e] * inv1 * ga[v % PP][e];
        y2[e] = (af[e] + r1f[e]) * inv2 * gm[v % PP][e];
      }
      st16(x1p + vi, pack<DT>(y1));
      st16(x2p + vi, pack<DT>(y2));
    }
  }
}

// RoPE role: RoPE block rb (< nB), i.e. the warp items [ipb rb, ipb (rb + 1)) of the call (RopeGeom),
// ipb = rope_ipb; fq holds the lane's frequencies. Items of at most one head-row per lane group, or of
// kChainRopeRows on grids several waves long (rope_k), which only the one-CTA-per-token entries
// (ROWS) carry, so the others keep their registers.
template <int DT, int D, bool QKNORM, bool ROWS>
__device__ __forceinline__ void chain_rope_rows(const ChainParams& c, int64_t t, int first, int end, const float4* fq) {
  if (ROWS && c.rope_k > 1) rope_pair_rows<DT, D, QKNORM, kChainRopeRows, false>(c.rope, t, first, end, fq);
  else rope_pair_rows<DT, D, QKNORM, 1, false>(c.rope, t, first, end, fq);
}
template <int DT, int NT, int D, bool QKNORM, bool ROWS>
__device__ __forceinline__ void chain_rope(const ChainParams& c, const int64_t rb, const float4* fq) {
  int64_t t;
  int first, end;
  const int w = threadIdx.x / 32;
  if (w < c.rope_ipb && rope_item(c.rope, rb * c.rope_ipb + w, &t, &first, &end))
    chain_rope_rows<DT, D, QKNORM, ROWS>(c, t, first, end, fq);
}
// The item of this warp in RoPE block `part` of token t (token-major grids).
template <int NT>
__device__ __forceinline__ bool chain_tok_item(const ChainParams& c, int part, int* first, int* end) {
  const int w = (int)threadIdx.x / 32, item = part * c.rope_ipb + w;
  *first = item * c.rope.rpi;
  *end = min(c.rope.NH, *first + c.rope.rpi);
  return w < c.rope_ipb && item < c.rope.ipt;
}

// Before the PDL wait: the RoPE lane frequencies of a RoPE block (other roles load none).
template <int DT, int D>
__device__ __forceinline__ void chain_rope_freqs(const ChainParams& c, const bool is_rope, float4* fq) {
  if (is_rope) rope_pair_freqs(c.rope.inv_freq, (threadIdx.x & 31) % RopeGeom<D>::LPG, fq);
}

// SwiGLU role: column tile `col_tile` of row `row`, SWU x NT 16-byte vectors of g and of u
// (kChainTileVecs or kChainWideTileVecs in all for one call's grid, kChainStepTileVecs for a step's).
template <int DT, int NT, int SWU>
__device__ __forceinline__ void chain_swiglu(const ChainParams& c, const int64_t row, const int64_t col_tile) {
  swiglu_tile<DT, SWU, NT>(c.sw, row, col_tile * SWU * NT, threadIdx.x);
}

// Row of SwiGLU tile `tile`. A single call's kernel divides by the host's multiplier
// (fast_div: the 64-token layer step 3.32 -> 3.29 us); the whole-step kernel (STEP), which
// reads its call's parameters at a block-varying index, keeps the division (the multiplier
// measured 3-5 % slower there).
template <bool STEP>
__device__ __forceinline__ int64_t swiglu_tile_row(const ChainParams& c, const int64_t tile) {
  if (STEP) return tile / c.sw_tiles_per_row;
  return fast_div((uint32_t)tile, c.sw_magic, c.sw_shift);
}

// Block b of one call's role-major grid (b < nA + nB + nC): [norms | RoPE | SwiGLU].
template <int DT, int NT, int VPT, int SPLIT, int D, bool QKNORM, int SWU, bool STEP>
__device__ __forceinline__ void chain_block(const ChainParams& c, const int b, const float4* fq) {
  if (b < c.nA) {
    const int64_t row = b / SPLIT;
    chain_norm<DT, NT, VPT, SPLIT>(c, row, b - (int)row * SPLIT);
  } else if (b < c.nA + c.nB) {
    chain_rope<DT, NT, D, QKNORM, SPLIT == 1>(c, b - c.nA, fq);
  } else {
    const int64_t tile = b - c.nA - c.nB;
    if (tile >= c.sw_tiles) return;
    const int64_t row = swiglu_tile_row<STEP>(c, tile);
    chain_swiglu<DT, NT, SWU>(c, row, tile - row * c.sw_tiles_per_row);
  }
}

// Token-major grid (SPLIT + rope_per_tok + sw_tiles_per_row, T): block (q, t) is token t's
// q-th block -- its norm parts, then its RoPE blocks, then its SwiGLU tiles. Blocks are
// dispatched x first, so consecutive blocks belong to one token and any few of them carry a
// mix of roles: under programmatic launch the blocks of a grid land on SMs as the previous
// kernel's blocks retire, several consecutive blocks on one SM, and a role-major order can
// give one SM four norm blocks (160 KB) while another gets 24 KB. Both indices come from
// special registers, so no remapped index stays live in a register through the body.
template <int DT, int NT, int VPT, int SPLIT, int D, bool QKNORM>
__device__ __forceinline__ void chain_block_tok(const ChainParams& c, const float4* fq) {
  const int q = blockIdx.x;
  if (q < SPLIT) {
    chain_norm<DT, NT, VPT, SPLIT>(c, blockIdx.y, q);
  } else if (q < SPLIT + c.rope_per_tok) {
    int first, end;
    if (chain_tok_item<NT>(c, q - SPLIT, &first, &end))
      chain_rope_rows<DT, D, QKNORM, false>(c, blockIdx.y, first, end, fq);
  } else {
    chain_swiglu<DT, NT, kChainTileVecs / NT>(c, blockIdx.y, q - SPLIT - c.rope_per_tok);
  }
}

// L2 prefetch of the lines a block reads first -- the norm rows, the RoPE head-rows and
// positions, the SwiGLU tile -- one prefetch per 128-byte line, between the launch trigger
// and the PDL wait (see prefetch_l2).
// A token's SPLIT norm blocks share its rows' lines: part p prefetches vectors v = p mod SPLIT.
template <int DT, int NT, int VPT, int SPLIT>
__device__ __forceinline__ void norm_prefetch(const ChainParams& c, const int64_t row, const int part) {
  constexpr int EB = Act<DT>::BYTES;
  constexpr int VE = Act<DT>::VE;
  const int tid = threadIdx.x;
  if ((tid & 3) != 0) return;  // a line is 8 threads' 16-byte row vectors, 4 threads' gamma floats
  const uint4* hp = reinterpret_cast<const uint4*>(row_ptr(c.n1.x, row, c.n1.x_rs, EB));
  const uint4* rp = reinterpret_cast<const uint4*>(row_ptr(c.n1.r, row, c.n1.r_rs, EB));
  const uint4* ap = reinterpret_cast<const uint4*>(row_ptr(c.n2.x, row, c.n2.x_rs, EB));
#pragma unroll
  for (int v = 0; v < VPT; ++v) {
    if (v % SPLIT != part) continue;
    const int64_t vi = (int64_t)v * NT + tid;
    if ((tid & 7) == 0) {
      prefetch_l2(hp + vi);
      prefetch_l2(rp + vi);
      prefetch_l2(ap + vi);
    }
    prefetch_l2(c.n1.gamma + vi * VE);  // this part's half of both norms' weights
    prefetch_l2(c.n2.gamma + vi * VE);
  }
}

// The token's RoPE head-rows (its q, k and v rows), prefetched by its norm blocks: part p of
// SPLIT takes head-rows [p * ceil(NH / SPLIT), ...), one thread per 128-byte line.
template <int DT, int SPLIT, int D>
__device__ __forceinline__ void norm_rope_prefetch(const ChainParams& c, const int64_t row, const int part) {
  constexpr int LINES = (D * Act<DT>::BYTES + 127) / 128;  // 128-byte lines per head-row
  const int per = (c.rope.NH + SPLIT - 1) / SPLIT;
  const int k = threadIdx.x / LINES;
  if (k >= per || part * per + k >= c.rope.NH) return;
  prefetch_l2(rope_row_src<D>(c.rope, row, part * per + k) + (threadIdx.x % LINES) * 128);
  if (threadIdx.x == 0) prefetch_l2(c.rope.pos + row);
}

// prefetch == 1: every block its own first lines; prefetch == 2: only the norm blocks, which
// take their token's rows and its RoPE head-rows (the other roles' own prefetches, issued by
// hundreds of blocks while the previous kernel finishes, measured slower).
template <int DT, int NT, int VPT, int SPLIT, int D, int SWU, bool STEP>
__device__ __forceinline__ void chain_prefetch(const ChainParams& c, const int b) {
  const int tid = threadIdx.x;
  if (b < c.nA) {
    norm_prefetch<DT, NT, VPT, SPLIT>(c, b / SPLIT, b % SPLIT);
    if (c.prefetch == 2) norm_rope_prefetch<DT, SPLIT, D>(c, b / SPLIT, b % SPLIT);
  } else if (c.prefetch == 2) {
    return;
  } else if (b < c.nA + c.nB) {
    if (c.rope_k != 1) return;  // several head-rows per lane group: grids too long to prefetch
    int64_t t;
    int first, end;
    if (tid / 32 < c.rope_ipb &&
        rope_item(c.rope, (int64_t)(b - c.nA) * c.rope_ipb + tid / 32, &t, &first, &end))
      rope_item_prefetch<D, 1>(c.rope, t, first, end);
  } else {
    const int64_t tile = b - c.nA - c.nB;
    if (tile >= c.sw_tiles) return;
    const int64_t row = swiglu_tile_row<STEP>(c, tile);
    swiglu_prefetch<DT, SWU, NT>(c.sw, row, (tile - row * c.sw_tiles_per_row) * SWU * NT, tid);
  }
}

template <int DT, int NT, int VPT, int SPLIT, int D>
__device__ __forceinline__ void chain_prefetch_tok(const ChainParams& c) {
  const int tid = threadIdx.x, q = blockIdx.x;
  if (q < SPLIT) {
    norm_prefetch<DT, NT, VPT, SPLIT>(c, blockIdx.y, q);
  } else if (q < SPLIT + c.rope_per_tok) {
    int first, end;
    if (chain_tok_item<NT>(c, q - SPLIT, &first, &end)) rope_item_prefetch<D, 1>(c.rope, blockIdx.y, first, end);
  } else {
    swiglu_prefetch<DT, kChainTileVecs / NT, NT>(
        c.sw, blockIdx.y, (int64_t)(q - SPLIT - c.rope_per_tok) * kChainTileVecs, tid);
  }
}

// 1024 resident threads per SM (64 registers): the 64-token grid at H 4096 (480 blocks of 256
// threads) then fits one wave on 152 SMs; one register more would cost a quarter of them.
// LATE (role-major grids only): only the norm blocks trigger the next launch at their start,
// the RoPE and SwiGLU blocks at their exit. The next launch then starts once this grid's
// short blocks are gone, and its blocks are placed while several slots per SM are free, one
// norm block per SM, instead of filling each slot the moment it frees (up to four norm
// blocks on one SM). The trigger is otherwise the kernel's first instruction: even one
// parameter read ahead of it measured 0.05 us slower per launch.
template <int DT, int NT, int VPT, int SPLIT, int D, bool QKNORM, bool LATE, int SWU>
__global__ void __launch_bounds__(NT, 1024 / NT)
    chain_kernel(const __grid_constant__ ChainParams c) {
  if (!LATE || (int)blockIdx.x < c.nA) pdl_trigger();
  float4 fq[4];
  if (!LATE && SWU == kChainTileVecs / NT && c.tok_grid) {
    if (c.prefetch) chain_prefetch_tok<DT, NT, VPT, SPLIT, D>(c);
    chain_rope_freqs<DT, D>(c, (int)blockIdx.x >= SPLIT && (int)blockIdx.x < SPLIT + c.rope_per_tok, fq);
    pdl_wait();
    chain_block_tok<DT, NT, VPT, SPLIT, D, QKNORM>(c, fq);
  } else {
    // A role-major grid fills the GPU: its RoPE blocks become resident only as the previous
    // kernel's blocks retire, and their frequency loads measured faster after the wait.
    const int b = blockIdx.x;
    if (c.prefetch) chain_prefetch<DT, NT, VPT, SPLIT, D, SWU, false>(c, b);
    pdl_wait();
    chain_rope_freqs<DT, D>(c, b >= c.nA && b < c.nA + c.nB, fq);
    chain_block<DT, NT, VPT, SPLIT, D, QKNORM, SWU, false>(c, b, fq);
  }
}

// Several independent calls in one launch: a block finds its call by binary search over
// the first-block table (uniform across the block, so the parameter reads broadcast).
// ROLE (one-CTA-per-token steps of one to two waves): role-major block order over the whole
// step -- every call's norm blocks, then every call's RoPE blocks, then every call's SwiGLU
// tiles -- so that the longer blocks fill the first wave (a separate entry: the call-major
// kernel measured about 1 % slower with this branch in it).
template <int DT, int NT, int VPT, int SPLIT, int D, bool QKNORM, bool ROLE>
__global__ void __launch_bounds__(NT, 1024 / NT)
    chain_step_kernel(const __grid_constant__ ChainStepParams p) {
  pdl_trigger();
  const int b = blockIdx.x;
  int lo = 0, hi = p.n - 1;
  if constexpr (ROLE) {
    const int r = b < p.role_first[1][0] ? 0 : (b < p.role_first[2][0] ? 1 : 2);
    const int32_t* f = p.role_first[r];
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (b >= f[mid]) lo = mid;
      else hi = mid - 1;
    }
    const ChainParams& c = p.c[lo];
    const int bl = b - f[lo] + (r == 0 ? 0 : (r == 1 ? c.nA : c.nA + c.nB));
    float4 fq[4];
    chain_rope_freqs<DT, D>(c, r == 1, fq);
    pdl_wait();
    chain_block<DT, NT, VPT, SPLIT, D, QKNORM, kChainStepTileVecs / NT, true>(c, bl, fq);
  } else {
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (b >= p.first[mid]) lo = mid;
      else hi = mid - 1;
    }
    const ChainParams& c = p.c[lo];
    const int bl = b - p.first[lo];
    if (c.prefetch) chain_prefetch<DT, NT, VPT, SPLIT, D, kChainStepTileVecs / NT, true>(c, bl);
    float4 fq[4];
    chain_rope_freqs<DT, D>(c, bl >= c.nA && bl < c.nA + c.nB, fq);
    pdl_wait();
    chain_block<DT, NT, VPT, SPLIT, D, QKNORM, kChainStepTileVecs / NT, true>(c, bl, fq);
  }
}

// Up to three head-rows per RoPE lane group on grids several waves long: a grid whose
// one-CTA-per-token form with one head-row per lane group (`one` blocks) exceeds the resident
// slots. There blocks queue for slots and a RoPE block that moves three rows for the same fixed
// costs pays; within one wave a block's own latency is the step. Same-box device times of the
// role as it was (a lane per 16-byte vector, partners exchanged by shuffles, loads behind a
// branch per row), as it is with two rows and with three: Llama layers of 128 / 256 / 1024 / 8192
// tokens 5.16 / 8.88 / 29.4 / 221.8, 5.02 / 8.45 / 27.7 / 210.9, 4.99 / 8.30 / 27.1 / 205.4 us
// (8192 tokens: 6.7 TB/s, 0.99 of the 6.8 TB/s copy rate); 36 layers with q/k norm in one launch
// at 8 / 32 / 128 tokens 10.7 / 33.7 / 124.8, 10.0 / 31.0 / 116.7, 9.4 / 30.3 / 110.7 us. 80 tokens
// 5.11 / 3.65, which now fit one wave.
// With q/k norm, whose rows are the longer, only from one and a quarter waves: 110 / 116 / 122
// tokens 4.57 / 5.15 / 5.24 us with three rows, 4.28 / 4.88 / 4.82 with one; 128 tokens 5.36 / 4.95.
int32_t chain_rope_k(int64_t one, int64_t wave, bool qk) {
  return one > (qk ? wave + wave / 4 : wave) ? kChainRopeRows : 1;
}

ChainPlan chain_plan(int64_t T, int64_t I, const RopeSplit* rope, int32_t threads, int32_t vec, int64_t wave, int32_t sms,
                     bool inplace, bool qk, bool pdl) {
  const int32_t warps = threads / 32;
  const bool big = threads > kThreads;  // blocks of 512 threads (H 8192)
  auto tiles = [&](int64_t width) { return T * ((I + width * vec - 1) / (width * vec)); };
  auto items = [&](int k, int64_t ipb) { return (T * rope[k].ipt + ipb - 1) / ipb; };
  int64_t nC = tiles(kChainTileVecs);
  const int64_t one = T + items(0, warps) + nC;  // one norm CTA per token, one head-row per lane group
  ChainPlan pl{};
  // Two CTAs per token for the norms -- so no SM carries a whole token's norm traffic -- while the
  // grid still fits in one wave, and unless an output is written over an input the partner CTA still
  // reads (in-place calls keep one CTA per token).
  pl.split = !inplace && T + one <= wave ? 2 : 1;
  pl.rope_k = pl.split == 1 ? chain_rope_k(one, wave, qk) : 1;
  bool early = false;  // no late trigger
  // Wider SwiGLU tiles on grids of more than four waves: same-box probe, one Llama layer at 1024 /
  // 4096 tokens 34.2 / 122.8 -> 31.3 / 112.6 us; at 256 tokens (3.4 waves) 9.81 -> 9.75 us, at 128
  // tokens (1.7 waves) 4.72 -> 5.11 us.
  pl.wide = pl.split == 1 && one > 4 * wave;
  // With blocks of 512 threads, where a tile is one or two vectors per thread, beyond one wave: with one
  // head-row per lane group where the wider tiles let the grid fit one wave (44 tokens of I 28672 5.26
  // -> 4.40 us), with q/k norm up to 1.7 waves (50 / 62 / 80 tokens 5.27 / 5.53 / 6.25 -> 4.71 / 5.11 /
  // 5.96 us; three rows 6.10 / 5.59 / 5.97, which at 100 tokens take 6.66, one row 7.01); three rows
  // beyond that (without the norm 66 / 80 / 128 tokens 5.23 / 6.02 / 8.80 -> 5.03 / 5.58 / 7.78). (With
  // 256 threads, 100 and 110 tokens at H 4096, 4.14 / 4.35 -> 4.46 / 4.74.) Past one wave the late
  // trigger loses (50 tokens with q/k norm 4.71 / 4.59, 54 4.85 / 4.98, 62 5.11 / 5.38).
  if (pl.split == 1 && !pl.wide && big && one > wave) {
    const int64_t rest = T + tiles(kChainWideTileVecs);
    const int64_t w1 = rest + items(0, warps);
    pl.wide = true;
    pl.rope_k = w1 <= wave || (qk && 10 * w1 <= 17 * wave) ? 1 : kChainRopeRows;
    early = rest + items(pl.rope_k > 1, warps) > wave;
  }
  if (pl.wide) nC = tiles(kChainWideTileVecs);
  const int64_t nA = T * pl.split;
  const int k = pl.rope_k > 1;
  pl.ipb = warps;
  // Few blocks: a RoPE block takes four or eight items (a quarter or half of its warps) while the grid
  // still leaves an SM to every block, or with blocks of 256 threads a quarter of the SMs idle; a warp's
  // angles are issue-bound, and the warps of fewer items per SM finish sooner. With q/k norm, where a
  // lane's norm is added to its angles, and two norm CTAs per token up to 1.6 blocks per SM, or in blocks of 512 threads eight items up to two if the late trigger below still applies (without
  // the norm 18 tokens 1.86 / 1.91). H 8192 at 2 / 4 / 10 tokens with q/k norm 2.42 / 2.44 / 2.78 -> 2.22 /
  // 2.24 / 2.56 us, 16 / 18 / 20 2.67 / 2.70 / 2.70 -> 2.52 / 2.55 / 2.58 (28 of I 22016, too many for the
  // late trigger, 2.84 / 3.58); H 4096 at 10 tokens 1.85 -> 1.82, with q/k norm 17 / 24 / 30 2.00 / 2.04 /
  // 2.18 -> 1.91 / 1.99 / 2.14, 32 2.18 / 2.26.
  for (int32_t ipb = 4; ipb < warps; ipb *= 2) {
    const int64_t blocks = nA + items(k, ipb) + nC;
    const bool more = qk && pl.split == 2 &&
                      (big ? ipb == 8 && blocks <= 2 * (int64_t)sms && blocks + nA <= wave + wave / 8
                           : 5 * blocks <= 8 * (int64_t)sms);
    if (blocks <= (big ? sms : sms * 3 / 4) || more) {
      pl.ipb = ipb;
      break;
    }
  }
  pl.blocks = nA + items(k, pl.ipb) + nC;
  // Under PDL, a role-major grid of more than a quarter block per SM whose blocks, with
  // its own norm blocks, fit the resident slots give or take an eighth of them launches a
  // late entry (fn_late, fn_inplace_late): its RoPE and SwiGLU blocks trigger the next launch
  // at their exit, so the next grid is placed whole while this one's norm blocks finish, one
  // norm block per SM instead of up to four. Same-box A/B of Llama layer steps against the
  // grids below: 6 tokens 2.22 -> 2.12 us, 16 tokens 2.58 -> 2.29, 32 tokens 2.98 -> 2.57, 56
  // tokens 3.31 -> 3.19; with one norm CTA per token 90 tokens 5.10 -> 3.80, 100 tokens 5.24 ->
  // 4.08, H 8192 at 37 tokens 4.86 -> 3.70. Equal at 2 and 4 tokens and at 1 token 1.5-2 %
  // slower (nothing to place, and the next launch starts later), hence the lower bound; a few
  // dozen blocks placed late cost less than stacked norm blocks, but with 96 blocks placed
  // late the probe measured 3.51 -> 3.69 us, hence the upper bound; with one norm CTA per
  // token, whose grids hold half the norm blocks, a quarter of the slots (H 8192 56 tokens 4.92 ->
  // 4.18 us, 110 tokens with q/k norm 4.57 -> 4.32).
  // Otherwise a token-major grid (chain_block_tok) for grids of at most two blocks per SM
  // with one head-row per RoPE lane group: consecutive blocks then mix roles, so the blocks
  // that land together on one SM are not all norm blocks (measured against role-major grids
  // without the late trigger: 16 tokens 3.55 -> 2.85 us per layer step, 1 token 2.20 -> 2.04
  // us). Larger grids are role-major, which starts the longest (norm) blocks first.
  const int64_t q = threads / kThreads;  // the bounds below count blocks of 256 threads
  pl.late = pdl && !early && 4 * q * pl.blocks > sms && pl.blocks + nA <= wave + (pl.split == 1 ? 2 : 1) * wave / 8;
  pl.tok = !pl.late && pl.rope_k == 1 && T >= 1 && T <= 65535 && !pl.wide && q * pl.blocks <= 2 * (int64_t)sms;
  return pl;
}

template <int DT, bool QK, int NT, int VPT>
static void pick(KernelEntry* out) {
  constexpr int U = kChainTileVecs / NT;
  out->threads = NT;
  out->fn = (const void*)chain_kernel<DT, NT, VPT, 2, 128, QK, false, U>;
  out->fn_late = (const void*)chain_kernel<DT, NT, VPT, 2, 128, QK, true, U>;
  out->fn_inplace = (const void*)chain_kernel<DT, NT, VPT, 1, 128, QK, false, U>;
  out->fn_inplace_late = (const void*)chain_kernel<DT, NT, VPT, 1, 128, QK, true, U>;
  out->fn_wide = (const void*)chain_kernel<DT, NT, VPT, 1, 128, QK, false, kChainWideTileVecs / NT>;
  out->fn_wide_late = (const void*)chain_kernel<DT, NT, VPT, 1, 128, QK, true, kChainWideTileVecs / NT>;
  out->fn_step = (const void*)chain_step_kernel<DT, NT, VPT, 2, 128, QK, false>;
  out->fn_step_inplace = (const void*)chain_step_kernel<DT, NT, VPT, 1, 128, QK, false>;
  out->fn_step_role = (const void*)chain_step_kernel<DT, NT, VPT, 1, 128, QK, true>;
}

// H 4096: 256 threads, two vectors each. H 8192: 512 threads, two vectors each, instead of four
// for 256 threads: at 64 registers 1024 threads fit an SM instead of 512 (28 tokens 4.70 -> 2.90
// us, 200 tokens 12.5 -> 10.7, 3000 tokens of I 22016 167 -> 137 us; with four vectors and the
// other changes of these kernels 3.43 us and 152). H 4096 with 512 threads of one vector lost
// (64 tokens 3.21 / 3.76 us, 8192 tokens 205.7 / 222): twice the slots per SwiGLU tile.
template <int DT, bool QK>
static void pick(int64_t H, KernelEntry* out) {
  if (H == 4096) pick<DT, QK, 256, 2>(out);
  else if (H == 8192) pick<DT, QK, 512, 2>(out);
}

bool chain_kernel(int32_t dtype, int64_t H, int32_t D, bool qknorm, KernelEntry* out,
                  const char** why) {
  if (dtype != DT_BF16 && dtype != DT_FP16) { *why = "layer chain supports bf16 and fp16"; return false; }
  if (D != 128) { *why = "layer chain supports D = 128"; return false; }
  out->kind = KK_CHAIN;
  out->vec = 8;
  // fn: two blocks per token for the norms; fn_inplace: one block per token (calls whose outputs
  // overwrite inputs, and grids too large for one wave); fn_late, fn_inplace_late: the same with
  // the late launch trigger; fn_wide: fn_inplace with wider SwiGLU tiles (grids of many waves);
  // fn_step*: the same for several calls per launch (fn_step_role: role-major order)
  out->fn = nullptr;
  if (dtype == DT_BF16) qknorm ? pick<DT_BF16, true>(H, out) : pick<DT_BF16, false>(H, out);
  else qknorm ? pick<DT_FP16, true>(H, out) : pick<DT_FP16, false>(H, out);
  if (!out->fn) { *why = "layer chain supports H in {4096, 8192}"; return false; }
  return true;
}

}  // namespace trident
