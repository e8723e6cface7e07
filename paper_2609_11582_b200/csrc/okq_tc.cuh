// Building blocks of the kernels that feed tcgen05.mma from TMA copies: descriptors, bounded waits on mbarriers, the tensor-map
// encoder.
#pragma once
#include <cuda.h>   // CUtensorMap and the type of cuTensorMapEncodeTiled only; the entry point is fetched at run time

#include "okq_common.cuh"

namespace okq {

namespace {

constexpr long long WAIT_LIMIT_CLOCKS = 4000000000ll;   // about two seconds of SM clocks

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ bool elect_one() {
  uint32_t pred = 0;
  asm volatile("{\n\t.reg .b32 rx;\n\t.reg .pred px;\n\telect.sync rx|px, 0xffffffff;\n\tselp.u32 %0, 1, 0, px;\n\t}\n" : "=r"(pred));
  return pred != 0;
}

// shared-memory matrix descriptor of a TMA-written tile: K-major, 128-byte swizzle (rows of 64 fp16 = 128
// bytes, 8-row groups 1024 bytes apart; the leading-dimension field is not used by this layout)
__device__ __forceinline__ uint64_t make_desc_sw128(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3fff) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) |
         ((uint64_t)2 << 61);
}

// Bounded wait of a whole warp for one phase of an mbarrier (each try may suspend the thread for a short,
// system-chosen time).  Gives up after about two seconds, or as soon as another role has given up; giving
// up raises the abort flag.
template <class SM>
__device__ __forceinline__ bool mbar_wait(SM& sm, unsigned long long* bar, uint32_t parity) {
  const uint32_t mbar = smem_u32(bar);
  bool done = false;
  const long long t0 = clock64();
  while (!done) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
                 : "=r"(ok) : "r"(mbar), "r"(parity) : "memory");
    done = ok != 0;
    if (!done && (sm.abort || clock64() - t0 > sm.limit)) break;
  }
  if (!done) sm.abort = 1;
  return __all_sync(0xffffffffu, done);   // called by whole warps: one answer per warp
}
// After a timeout: wait, again with a limit and whatever the abort flag says, for a phase that this warp's own
// asynchronous work (bulk copies, tensor-core products) will complete.  Returns false if it did not.
__device__ __forceinline__ bool mbar_drain(unsigned long long* bar, uint32_t parity) {
  const uint32_t mbar = smem_u32(bar);
  bool done = false;
  const long long t0 = clock64();
  while (!done && clock64() - t0 < WAIT_LIMIT_CLOCKS / 8) {   // a quarter of a second, whatever the caller's limit
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
                 : "=r"(ok) : "r"(mbar), "r"(parity) : "memory");
    done = ok != 0;
  }
  return __all_sync(0xffffffffu, done);
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}

using EncodeTiledFn = decltype(&cuTensorMapEncodeTiled);

// cuTensorMapEncodeTiled, looked up through the runtime (no link against the driver library)
EncodeTiledFn encode_tiled() {
  static EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  return fn;
}

}  // namespace

}  // namespace okq
