// plan_probe.cpp -- prints the kernel entry that a call's dispatch rule chooses, one line per input
// line, without a GPU: it is linked with the library's own objects and calls the rules that the host
// core calls. Lines (152 SMs):
//   norm RES DTYPE H T OFF RS    RES 0/1, rows at element offset OFF of a 16-byte boundary, row stride RS
//   chain QK H HQ HKV I T INPLACE PDL    norm CTAs per token, SwiGLU tiles, launch trigger, block order;
//                                        head-rows per RoPE lane group and items per RoPE block
//   rope ANY QK HQ HKV D T       ANY 1: a version of any alignment; QK 1: with q/k norm
#include <cinttypes>
#include <cstdio>
#include <cstring>

#include <cuda_runtime.h>

#include "internal.h"

using namespace trident;

constexpr int32_t kSms = 152;

static void norm_line(const char* s) {
  int res, dtype;
  int64_t H, T, off, rs;
  if (std::sscanf(s, "%d %d %" SCNd64 " %" SCNd64 " %" SCNd64 " %" SCNd64, &res, &dtype, &H, &T, &off, &rs) != 6) return;
  const int eb = dtype == DT_FP32 ? 4 : 2;
  KernelEntry ke;
  const char* why = "";
  if (!norm_kernel(res != 0, dtype, (H * eb) % 16 != 0 ? 1 : 0, H, &ke, &why)) {
    std::printf("error %s\n", why);
    return;
  }
  NormParams p;
  std::memset(&p, 0, sizeof p);
  const uintptr_t at = 4096 + (uintptr_t)(off * eb);
  p.x = reinterpret_cast<const void*>(at);
  p.r = res ? p.x : nullptr;
  p.y = reinterpret_cast<void*>(at);
  p.r_out = res ? p.y : nullptr;
  p.gamma = reinterpret_cast<const float*>((uintptr_t)4096);
  p.T = T;
  p.H = H;
  p.x_rs = p.r_rs = p.y_rs = p.ro_rs = rs;
  int32_t threads = 0, smem = 0;
  int64_t blocks = 0;
  const NormEntry e = norm_plan(ke, &p, res != 0, eb, &threads, &blocks, &smem, kSms);
  static const char* const names[kNormEntries] = {"vec", "edge", "edge_many", "generic", "large", "few", "mid", "edge_flat"};
  std::printf("%s%s\n", names[e], e == NM_LARGE ? (smem ? "_bulk" : ke.large_per > 1 ? "_rows2" : "_regs") : "");
}

static void rope_line(const char* s) {
  int qk, Hq, Hkv, D, any;
  int64_t T;
  if (std::sscanf(s, "%d %d %d %d %d %" SCNd64, &any, &qk, &Hq, &Hkv, &D, &T) != 6) return;
  KernelEntry ke;
  const char* why = "";
  if (!rope_kernel(DT_BF16, any ? 1 : 2, D, qk != 0, &ke, &why)) {
    std::printf("error %s\n", why);
    return;
  }
  RopeParams p;
  std::memset(&p, 0, sizeof p);
  p.gamma_q = p.gamma_k = qk ? reinterpret_cast<const float*>((uintptr_t)4096) : nullptr;
  p.T = T;
  p.Hq = Hq;
  p.Hkv = Hkv;
  p.D = D;
  p.NH = Hq + 2 * Hkv;
  p.q_rs = p.k_rs = p.v_rs = (int64_t)p.NH * D;
  RopePlans plans{};
  rope_plans(p.NH, D, &plans);
  int32_t threads = 0;
  int64_t blocks = 0;
  if (any) {
    const int e = rope_any_plan(plans, &p, &threads, &blocks, kSms);
    std::printf("%s\n", e < 0 ? "generic" : e == 0 ? "any1" : "any3");
    return;
  }
  const RopeEntry e = rope_plan(plans, &p, &threads, &blocks, kSms);
  std::printf("%s_%d\n", e == ROPE_MID ? "two" : e == ROPE_BULK ? "bulk" : "one", threads);
}

static void chain_line(const char* s) {
  int qk, Hq, Hkv, inplace, pdl;
  int64_t H, I, T;
  if (std::sscanf(s, "%d %" SCNd64 " %d %d %" SCNd64 " %" SCNd64 " %d %d", &qk, &H, &Hq, &Hkv, &I, &T, &inplace, &pdl) != 8)
    return;
  KernelEntry ke;
  const char* why = "";
  if (!chain_kernel(DT_BF16, H, 128, qk != 0, &ke, &why)) {
    std::printf("error %s\n", why);
    return;
  }
  const RopeSplit split[2] = {rope_split(Hq + 2 * Hkv, 4, 1), rope_split(Hq + 2 * Hkv, 4, kChainRopeRows)};
  const int64_t wave = (int64_t)kSms * (1024 / ke.threads);  // the kernels' launch bounds
  const ChainPlan p = chain_plan(T, I, split, ke.threads, ke.vec, wave, kSms, inplace != 0, qk != 0, pdl != 0);
  std::printf("%s%s%s rows%d ipb%d\n", p.split == 2 ? "two" : p.wide ? "wide" : "one", p.late ? "_late" : "",
              p.tok ? "_tok" : "", p.rope_k, p.ipb);
}

int main() {
  char line[256];
  while (std::fgets(line, sizeof line, stdin)) {
    if (std::strncmp(line, "norm ", 5) == 0) norm_line(line + 5);
    else if (std::strncmp(line, "rope ", 5) == 0) rope_line(line + 5);
    else if (std::strncmp(line, "chain ", 6) == 0) chain_line(line + 6);
    else std::printf("error unknown line\n");
  }
  return 0;
}
