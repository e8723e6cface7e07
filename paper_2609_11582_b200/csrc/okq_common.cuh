// Host-side helpers: argument checks and CUDA error capture.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/okq.h"
#include "okq_layout.cuh"

namespace okq {

void set_last_cuda_error(int e);
int sm_count();   // SMs of the current device (cached per thread)

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// shape checks shared by every entry point; `need_ptrs` also checks the buffers
okq_status check_cache(const okq_cache* c, bool need_ptrs);

inline CacheView make_view(const okq_cache* c) {
  CacheView v;
  v.n_layers = c->n_layers; v.batch = c->batch; v.n_kv_heads = c->n_kv_heads; v.n_q_heads = c->n_q_heads;
  v.capacity = c->capacity;
  v.fmt = c->meta_format;
  v.sched = c->schedule;
  v.records = static_cast<unsigned char*>(c->records);
  v.modality = c->modality;
  v.k_tail = static_cast<__half*>(c->k_tail);
  v.v_tail = static_cast<__half*>(c->v_tail);
  v.seq_len = c->seq_len;
  v.status = c->status;
  return v;
}

// Function attributes (dynamic shared memory size) are per device: `mask` remembers, per calling thread and
// call site, the devices on which they have been set.  Returns true when the current device still needs them.
inline bool attr_needed(unsigned long long& mask, int& dev_out) {
  int dev = 0;
  cudaGetDevice(&dev);
  dev_out = dev;
  return dev < 0 || dev >= 64 || !((mask >> dev) & 1ull);
}
inline void attr_done(unsigned long long& mask, int dev) {
  if (dev >= 0 && dev < 64) mask |= 1ull << dev;
}

// Launch that may overlap the end of the kernel before it in the stream: its blocks are placed and set up as soon as that
// kernel has let go (depend_wait below) or is through.  Every kernel launched this way calls depend_wait before it touches
// global memory: it returns once the kernel before has completed and its writes are visible, whatever that kernel was.
template <class... P, class... A>
inline cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, int cluster, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = cluster; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
#ifdef __CUDACC__
__device__ __forceinline__ void depend_wait() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");   // the next kernel may be placed; it waits for this one's end
}
#endif

inline okq_status launch_status() {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_last_cuda_error((int)e);
    return OKQ_ERR_CUDA;
  }
  return OKQ_OK;
}

}  // namespace okq
