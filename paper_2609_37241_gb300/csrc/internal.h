// internal.h -- interface between the SCM host core (scm.cpp) and the kernels (*.cu).
//
// Each kernel takes one parameter struct by value. The host core packs it on the hit
// path (argument preparation, §3.2 and §3.5 of the paper: graph operands are rebuilt
// only after every guard passed) and launches the kernel entry that was resolved when
// the version was registered (§3.3).
#pragma once
#include <stdint.h>

namespace trident {

// Activation element types (values equal trident_dtype).
enum : int32_t { DT_BF16 = 1, DT_FP16 = 2, DT_FP32 = 3 };

constexpr int kThreads = 256;  // block size of the kernels that do not say otherwise

// RMSNorm over T rows of H elements, with a residual add or without (r, r_out unused). Row
// strides in elements.
struct NormParams {
  const void* x;
  const void* r;
  const float* gamma;
  void* y;
  void* r_out;
  int64_t T, H;
  int64_t x_rs, r_rs, y_rs, ro_rs;
  float eps, inv_H;
  int32_t prefetch;  // 1: prefetch this block's first lines into L2 before the PDL wait
  int32_t nvec;      // whole 16-byte vectors per row (H / VE)
  uint32_t first_wait_polls;  // bulk-copy kernel: polls of its first wait for the copies
                              // (kBulkWaitPolls; 0 under TRIDENT_OPT_TEST_WAIT_TIMEOUT)
  uint32_t* err;     // device status word (the bulk-copy kernel reports a timed-out wait)
};

// Bound of every mbarrier wait of the bulk-copy kernel (try_wait polls, each itself bounded
// by the hardware's suspend time).
constexpr uint32_t kBulkWaitPolls = 1u << 20;

// Elementwise operators over T rows of W elements (a: x, the first addend or the gate; b: the
// second addend or up; mask: u8 for MASKED_FILL). Row strides in elements. The vector kernels
// run over `units` 16-byte vectors of y:
//   flat  dense tensors that all start at the same offset from a 16-byte boundary, taken as
//         one row of T * W elements: `peel` elements before the first boundary, units vectors,
//         `tail` elements after them
//   rows  16-byte aligned rows of `row_vecs` vectors (units = T * row_vecs); the row of a
//         vector by fast_div where units < 2^31
enum PointwiseOp : int32_t { PW_SWIGLU = 4, PW_SILU = 8, PW_ADD = 9, PW_NEG = 10, PW_MASKED_FILL = 11 };
struct PointwiseParams {
  const void* a;
  const void* b;
  const uint8_t* mask;
  void* y;
  int64_t T, W;
  int64_t a_rs, b_rs, m_rs, y_rs;
  float scalar;
  int32_t prefetch;
  int64_t units, row_vecs;
  int32_t peel, tail;
  int32_t mask_vec;   // masks can be read a vector's elements at a time (aligned)
  uint32_t magic;     // division by row_vecs (rows kernel) or by W (generic kernel)
  int32_t shift;
};

// RoPE on q/k (optionally after per-head RMSNorm) plus KV-cache append.
// q/k/v rows: token stride *_rs, head stride D, element stride 1. Caches dense [Hkv][S][D].
// inv_freq: [D/2] pairs (hi, lo), theta^(-2i/D) = hi + lo, split from fp64 on the host.
struct RopeParams {
  void* q;
  const void* k;
  const void* v;
  const int32_t* pos;
  void* k_cache;
  void* v_cache;
  const float* gamma_q;
  const float* gamma_k;
  const float2* inv_freq;
  uint32_t* err;
  int64_t T, S;
  int64_t q_rs, k_rs, v_rs;
  int32_t Hq, Hkv, D, NH;  // NH = Hq + 2 Hkv head-rows per token
  float eps, inv_D;
  int32_t prefetch;
  int32_t freq_late;   // 1: inv_freq is written by the previous kernel of the stream: read it after the wait
  int32_t ipt, rpi;    // warp items per token, head-rows per item (RopeSplit)
  uint32_t ipt_magic;  // item / ipt by fast_div
  int32_t ipt_shift;
};

// RoPE with each warp's rows staged by bulk copies (rope_bulk_kernel, calls of many tokens).
struct RopeBulkParams {
  RopeParams rp;
  uint32_t first_wait_polls;  // polls of the wait for the copies (kBulkWaitPolls; 0 under
                              // TRIDENT_OPT_TEST_WAIT_TIMEOUT)
};

// out = silu(g) * u over T rows of I elements (the layer chain's role).
struct SwigluParams {
  const void* g;
  const void* u;
  void* out;
  int64_t T, I;
  int64_t g_rs, u_rs, o_rs;
  int32_t prefetch;
};

// One decoder layer's chain in one launch. Blocks [0, nA) run the two add+RMSNorm steps
// of one token each, [nA, nA+nB) the RoPE/KV head-rows, the rest SwiGLU tiles.
struct ChainParams {
  NormParams n1;   // h, r0 -> x1, r1
  NormParams n2;   // attn_out, (r1 from registers) -> x2, r2; n2.r is unused
  RopeParams rope;
  SwigluParams sw;
  int32_t nA, nB, nC, sw_tiles_per_row;
  int32_t a_split;   // CTAs per token for the norms (2, or 1 for in-place calls)
  int32_t prefetch;  // before the PDL wait, into L2: 1 every block's first input lines,
                     // 2 only the norm blocks' rows, 0 none
  int32_t tok_grid;  // 1: grid (a_split + rope_per_tok + sw_tiles_per_row, T), token-major
  int32_t rope_per_tok;  // RoPE blocks per token (token-major grid: nB = T * rope_per_tok)
  int32_t rope_k;    // head-rows per RoPE lane group at most: 1, or kChainRopeRows on grids several
                     // waves long
  int32_t rope_ipb;  // RoPE warp items per block: a warp each, fewer on grids that leave SMs idle
  uint32_t sw_magic;  // tile / sw_tiles_per_row by fast_div
  int32_t sw_shift;
  int64_t sw_tiles;  // T * sw_tiles_per_row (valid SwiGLU tiles)
};

// Several independent layer-chain calls in one launch (a decoder step's chains). Call i
// owns blocks [first[i], first[i+1]); inside its range a block plays the same role as in
// the single-call kernel. The struct is passed as the kernel parameter (about 25 KB, under
// the 32 KB parameter limit), so no device buffer is written before the launch.
constexpr int kStepMax = 48;
// SwiGLU tile width of the layer chain's blocks, in 16-byte vectors of g and of u: one call's
// grid keeps tiles small (more blocks for small token counts); a whole step's grid, several waves
// long, does better with fewer, larger tiles (measured on 36 Qwen3 layers: 8 tokens 11.7 -> 11.4
// us, 32 tokens 39.1 -> 37.2 us, 128 tokens 155 -> 150 us; the same change on single calls made
// them slower, 64 tokens 3.56 -> 4.09 us). A single call's grid of many waves (one CTA per token)
// takes the wider tiles too: blocks queue for slots there, and a tile that moves twice the bytes
// for the same fixed costs pays.
constexpr int kChainRopeRows = 3;
// RoPE items per block of small whole-step grids (blocks of 256 and of 512 threads).
constexpr int kChainStepItems = 3;
constexpr int kChainStepItemsWide = 4;
constexpr int kChainTileVecs = 512;
constexpr int kChainStepTileVecs = 1024;
constexpr int kChainWideTileVecs = 1024;
struct ChainStepParams {
  int32_t n;
  int32_t first[kStepMax + 1];  // call-major: call i owns blocks [first[i], first[i+1])
  int32_t role_first[3][kStepMax + 1];  // role-major: call i's norm / RoPE / SwiGLU blocks
                                        // start at role_first[r][i]; [r][n] ends role r
  ChainParams c[kStepMax];
};

// Elementwise entries (pointwise_plan): flat and rows kernels with one or two vectors per
// thread, and the generic kernel.
enum PointwiseEntry : int32_t { PW_FLAT, PW_FLAT2, PW_ROWS, PW_ROWS2, PW_GENERIC, kPwEntries };
// Picks the entry of a call (index into pw_fn) from its packed params, fills their vector
// fields and sets the grid. eb: element size.
int pointwise_plan(PointwiseParams* p, int32_t op, int32_t eb, int64_t* blocks, int32_t sms);

// Norm entries (norm_plan): 16-byte aligned rows, rows at any common offset (few or many rows),
// scalar accesses, the entry of long aligned calls (bulk copies, more vectors per thread, or two
// rows at a time for short rows), those of few rows and of some in between (norm_row_kernel), and rows
// at other offsets with the loads out of branches.
constexpr int kNormBlockVecs = 2048;  // norm_block_kernel, norm_bulk_kernel: vectors of a row at most
enum NormEntry : int32_t { NM_VEC, NM_EDGE, NM_EDGE_MANY, NM_GENERIC, NM_LARGE, NM_FEW, NM_MID,
                           NM_EDGE_FLAT, kNormEntries };

// Kernel entry (host stub address) plus its launch shape rule.
struct KernelEntry {
  const void* fn = nullptr;
  const void* fn_inplace = nullptr;  // chain only: the entry for calls that write in place
  const void* fn_late = nullptr;     // chain only: fn with the late launch trigger (LATE)
  const void* fn_inplace_late = nullptr;  // chain only: fn_inplace with the late launch trigger
  const void* fn_wide = nullptr;     // chain only: fn_inplace with kChainWideTileVecs tiles
  const void* fn_wide_late = nullptr;  // chain only: fn_wide with the late launch trigger
  const void* fn_step_role = nullptr;  // chain only: fn_step_inplace, role-major block order
  const void* fn_step = nullptr;          // chain only: several calls per launch (ChainStepParams)
  const void* fn_step_inplace = nullptr;  // ... one block per token for the norms
  const void* fn_large = nullptr;  // RoPE: the bulk-copy entry (rope_plan chooses)
  const void* any_fn[2] = {};      // RoPE versions of the generic kind: rope_any_kernel (or NULL)
  const void* fn_mid = nullptr;    // RoPE: two head-rows per lane group
  const void* fn_blocks = nullptr;  // RoPE, D 64: fn for blocks of 128 or 256 threads
  const void* pw_fn[kPwEntries] = {};  // elementwise, by PointwiseEntry
  float large_sm = 0;      // norms: calls of more rows per SM take the NM_LARGE entry
  float few_lo = 0, few_hi = 0;  // ... of rows per SM in (few_lo, few_hi] the NM_FEW entry
  float mid_lo = 0, mid_hi = 0;  // ... and of rows per SM in (mid_lo, mid_hi] the NM_MID entry
  float edge_lo = 0, edge_hi = 0;  // the same for rows at other offsets and the NM_EDGE_FLAT entry
  int32_t large_per = 1;   // ... that entry's rows per block
  int32_t large_smem = 0;  // ... and its dynamic shared memory (rows staged by bulk copies)
  int32_t kind = 0;      // which grid rule the host applies (KernelKind)
  int32_t vec = 0;       // elements per vector (VE)
  int32_t threads = 0;   // chain: block size
  const void* nm_fn[kNormEntries] = {};  // norms, by NormEntry (NULL: none for this H)
  int32_t nm_threads[kNormEntries] = {};
  int32_t rows = 1;      // norms: rows per block of the NM_VEC entry
  int32_t edge_rows = 1;  // ... and of the NM_EDGE_MANY entry,
  int64_t edge_many = 0;  // which calls of at least this many rows take (on 152 SMs)
};

enum KernelKind : int32_t {
  KK_NORM = 1,          // entry, block size and grid by norm_plan
  KK_ROPE_PAIR = 2,     // vector: grid by rope_plan
  KK_ROPE_WARP = 3,     // generic: one warp per head-row
  KK_POINTWISE = 4,     // flat, rows or generic entry by the call's layout (pw_fn)
  KK_CHAIN = 6
};

// Lookup of compiled kernels. Return false (with a reason) if no kernel fits.
bool norm_kernel(bool res, int32_t dtype, int32_t variant, int64_t H, KernelEntry* out, const char** why);
bool pointwise_kernel(int32_t op, int32_t dtype, int32_t variant, int64_t W, KernelEntry* out,
                      const char** why);
bool rope_kernel(int32_t dtype, int32_t variant, int32_t D, bool qknorm, KernelEntry* out,
                 const char** why);
bool chain_kernel(int32_t dtype, int64_t H, int32_t D, bool qknorm, KernelEntry* out,
                  const char** why);
// The entry a call takes from its packed params (sets p->nvec), its block size and grid.
NormEntry norm_plan(const KernelEntry& ke, NormParams* p, bool res, int32_t eb, int32_t* threads, int64_t* blocks,
                    int32_t* smem, int32_t sms);
// Round-up multiplier and shift for dividing 32-bit unsigned integers by d (1 <= d < 2^31):
// l = ceil(log2 d), m = floor(2^32 (2^l - d) / d) + 1; the kernels take the quotient as
// (h + ((n - h) >> 1)) >> (l - 1) with h = umulhi(n, m) (fast_div; Granlund and Montgomery,
// 1994), and l = 0 (d = 1) as n itself. d = 0 (no divisor: callers reject such calls first)
// stays defined.
inline void div_magic(uint32_t d, uint32_t* m, int32_t* l) {
  *m = 0;
  *l = 0;
  if (d == 0) return;
  int32_t s = 0;
  while ((1ull << s) < d) ++s;
  *m = (uint32_t)(((1ull << 32) * ((1ull << s) - d)) / d + 1);
  *l = s;
}

// How a token's NH head-rows are split into warp items of at most `max_rows` rows per lane
// group (gw groups per warp), as evenly as the groups allow.
struct RopeSplit {
  int32_t ipt, rpi;  // items per token, head-rows per item
  uint32_t magic;    // item / ipt by fast_div
  int32_t shift;
};
inline RopeSplit rope_split(int64_t NH, int64_t gw, int32_t max_rows) {
  RopeSplit r{};
  const int64_t quads = (NH + gw - 1) / gw, ipt = (quads + max_rows - 1) / max_rows;
  if (ipt < 1) return r;
  const int64_t rpi = (quads + ipt - 1) / ipt * gw;
  r.rpi = (int32_t)rpi;
  r.ipt = (int32_t)((NH + rpi - 1) / rpi);  // no item without rows
  div_magic((uint32_t)r.ipt, &r.magic, &r.shift);
  return r;
}

// A single chain call's launch: norm CTAs per token, RoPE head-rows per lane group at most and items
// per block, SwiGLU tile width, launch trigger and block order. rope: the call's item splits with one
// and with kChainRopeRows rows; wave: blocks resident at once.
struct ChainPlan {
  int32_t split, rope_k, ipb;
  bool wide, late, tok;
  int64_t blocks;  // role-major grid
};
ChainPlan chain_plan(int64_t T, int64_t I, const RopeSplit* rope, int32_t threads, int32_t vec, int64_t wave, int32_t sms,
                     bool inplace, bool qk, bool pdl);
int32_t chain_rope_k(int64_t one, int64_t wave, bool qk);
const void* empty_kernel_entry();  // the latency-floor probe's kernel (does nothing)

// Validation, guard-equivalent checks (sizes, layouts, 16-byte alignment, overlap) and
// parameter packing of a ROPE_KV / QKNORM_ROPE_KV argument tuple without an SCM. Leaves
// p->inv_freq and p->err NULL. Returns a trident_status (message in trident_scm_last_error).
int32_t prepare_rope_args(const void* trident_args_ptr, RopeParams* p, int32_t* dtype,
                          bool* qknorm);

// Sets the thread-local last-error message and returns `status`.
int32_t internal_fail(int32_t status, const char* msg);

// Which vector RoPE entry a call of T tokens takes, and its launch shape. The splits depend
// only on the version's head counts and head size (rope_plans, at registration).
enum RopeEntry : int32_t { ROPE_SMALL = 0, ROPE_MID = 1, ROPE_BULK = 2, ROPE_BLOCKS = 3, kRopeEntries };
struct RopePlans {
  RopeSplit split[kRopeEntries];  // by RopeEntry
  RopeSplit any[2];    // rope_any_kernel with one and with three rows per lane group (ipt 0: none)
};
void rope_plans(int64_t NH, int32_t D, RopePlans* out);
RopeEntry rope_plan(const RopePlans& plans, RopeParams* p, int32_t* threads, int64_t* blocks, int32_t sms);
int rope_any_plan(const RopePlans& plans, RopeParams* p, int32_t* threads, int64_t* blocks, int32_t sms);

}  // namespace trident
