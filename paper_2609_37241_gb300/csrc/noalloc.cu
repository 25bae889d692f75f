// noalloc.cu -- RoPE + KV-cache append that allocates nothing.
//
// The SCM path keeps two pieces of scratch memory in device allocations it makes itself:
// the frequency table of a RoPE version (cudaMalloc at registration) and the device
// status word (cudaMalloc at creation). Some callers cannot allocate device memory at
// all: a serving engine that has handed every byte of HBM to its own pool, or code running
// where a cudaMalloc would synchronise the device and stall other streams. For them,
// trident_rope_kv_noalloc runs the same vector RoPE/KV kernel with its scratch in a
// file-scope static device array of fixed size, so no call allocates anything (no
// cudaMalloc, no cudaFree, no allocating library routine).
//
// Scratch layout (kScratchBytes = 256 + 1024 bytes, held by every GPU that loads the
// library until the process exits): bytes [0, 4) the status word, bytes [256, end) the
// frequency table, (hi, lo) fp32 pairs of theta^(-2i/D) for i < D/2, at most kMaxPairs =
// 128 pairs (D <= 256). Every call first launches one small kernel on the caller's stream
// that clears the status word and rewrites the table for its own (theta, D), then the
// RoPE kernel. The host keeps no record of what the array holds, so nothing on the host
// can disagree with the device: whatever ran on the stream before, and whether or not an
// earlier launch failed, the RoPE kernel reads the table its own call wrote. It is launched
// with programmatic serialisation, so that its launch overlaps the preparing kernel, and reads
// its frequencies only after griddepcontrol.wait (RopeParams.freq_late), when that kernel has
// finished, by coherent loads (rope_pair_freqs_late); the preparing kernel itself starts after
// everything before it on the stream.
#include <cuda_runtime.h>

#include <cmath>
#include <mutex>

#include "device_common.cuh"
#include "trident_scm.h"

namespace trident {
namespace {

constexpr size_t kTableOffset = 256;
constexpr int64_t kMaxPairs = 128;
constexpr size_t kScratchBytes = kTableOffset + size_t(kMaxPairs) * sizeof(float2);
constexpr int kMaxDevices = 64;

static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

struct DeviceScratch {
  std::once_flag once;
  cudaError_t setup_error = cudaSuccess;
  unsigned char* addr = nullptr;  // device address of g_scratch on this device
  int sms = 0;                    // its multiprocessors
};
DeviceScratch g_dev[kMaxDevices];

// theta^(-2 * 2^b / D) for b < 7, in fp64: the factors of every f_i = theta^(-2i/D), i < 128.
struct FreqPowers { double p[7]; };

// Prepares the scratch for one call: clears the status word and writes the frequency
// table f_i = theta^(-2i/D) in fp64, stored as (fp32(f), fp32(f - hi)), for i < D/2: the product of
// the powers at the bits of i. At most seven factors, each off by at most 2^-52 (pow), and six
// roundings of 2^-53: 20 * 2^-53 in all, below the 2^-48 that the pair keeps. (One pow per thread
// instead, in the kernel, was 7 us of every call: fp64 runs at a small fraction of fp32's rate.)
__global__ void prepare_scratch(uint32_t* status, float2* tab, int32_t D, const FreqPowers pw) {
  pdl_trigger();
  const int i = threadIdx.x;
  if (i == 0) *status = 0u;
  if (i < D / 2) {
    double f = 1.0;
#pragma unroll
    for (int b = 0; b < 7; ++b)
      if (i >> b & 1) f *= pw.p[b];
    const float hi = (float)f;
    tab[i] = make_float2(hi, (float)(f - (double)hi));
  }
}

}  // namespace
}  // namespace trident

using namespace trident;

extern "C" __attribute__((visibility("default"))) int32_t trident_rope_kv_noalloc(
    const trident_args* args, void* stream, uint32_t* out_status) {
  RopeParams p;
  int32_t dtype = 0;
  bool qknorm = false;
  int32_t st = prepare_rope_args(args, &p, &dtype, &qknorm);
  if (st != TRIDENT_OK) return st;
  const int dev = args->t[0].device;
  if (dev >= kMaxDevices) return internal_fail(TRIDENT_ERR_INVALID, "device ordinal too large");
  int cur = -1;
  if (cudaGetDevice(&cur) != cudaSuccess || cur != dev)
    return internal_fail(TRIDENT_ERR_INVALID, "the tensors' device must be the current device");
  if (p.D / 2 > kMaxPairs)
    return internal_fail(TRIDENT_ERR_INVALID,
                         "D/2 exceeds the static scratch maximum of 128 frequency pairs (D <= 256)");
  KernelEntry ke;
  const char* why = "";
  if (!rope_kernel(dtype, TRIDENT_VARIANT_VECTOR, p.D, qknorm, &ke, &why))
    return internal_fail(TRIDENT_ERR_INVALID, why);

  // one-time set-up on this device: the device address of the static array, the SM count
  DeviceScratch& ds = g_dev[dev];
  std::call_once(ds.once, [&] {
    void* a = nullptr;
    ds.setup_error = cudaGetSymbolAddress(&a, g_scratch);
    ds.addr = static_cast<unsigned char*>(a);
    if (ds.setup_error == cudaSuccess)
      ds.setup_error = cudaDeviceGetAttribute(&ds.sms, cudaDevAttrMultiProcessorCount, dev);
  });
  if (ds.setup_error != cudaSuccess || !ds.addr)
    return internal_fail(TRIDENT_ERR_CUDA, "set-up of the scratch array failed");

  cudaStream_t s = static_cast<cudaStream_t>(stream);
  uint32_t* status = reinterpret_cast<uint32_t*>(ds.addr);
  float2* table = reinterpret_cast<float2*>(ds.addr + kTableOffset);
  FreqPowers pw;
  for (int b = 0; b < 7; ++b) pw.p[b] = std::pow(args->rope_theta, -2.0 * (double)(1 << b) / (double)p.D);
  // Every failure is read from the failing call itself and taken out of the thread's last error:
  // an error that some earlier call left there is not this call's.
  auto failed = [](cudaError_t e) {
    if (e == cudaSuccess) return false;
    (void)cudaGetLastError();
    return true;
  };
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(1);
  cfg.blockDim = dim3((unsigned)kMaxPairs);
  cfg.stream = s;
  if (failed(cudaLaunchKernelEx(&cfg, prepare_scratch, status, table, p.D, pw)))
    return internal_fail(TRIDENT_ERR_CUDA, "scratch preparation launch failed");
  p.inv_freq = table;
  p.freq_late = 1;
  p.err = status;
  RopeBulkParams bp;
  RopePlans plans;
  int32_t threads = 0;
  int64_t blocks = 0;
  rope_plans(p.NH, p.D, &plans);
  const RopeEntry entry = rope_plan(plans, &p, &threads, &blocks, ds.sms);
  bp.rp = p;
  bp.first_wait_polls = kBulkWaitPolls;
  const void* const fns[kRopeEntries] = {ke.fn, ke.fn_mid, ke.fn_large, ke.fn_blocks};  // by RopeEntry
  const void* fn = fns[entry];
  void* kargs[1] = {entry == ROPE_BULK ? (void*)&bp : (void*)&p};
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3((unsigned)(blocks < 0x7fffffff ? blocks : 0x7fffffff));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  if (failed(cudaLaunchKernelExC(&cfg, fn, kargs))) return internal_fail(TRIDENT_ERR_CUDA, "RoPE launch failed");
  if (out_status && failed(cudaMemcpyAsync(out_status, status, sizeof(uint32_t), cudaMemcpyDeviceToHost, s)))
    return internal_fail(TRIDENT_ERR_CUDA, "status copy failed");
  return TRIDENT_OK;
}
