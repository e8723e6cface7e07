// What a bulk call stores besides the packed windows: the raw tokens behind them (token t in slot t mod slots of the
// schedule), the sequence lengths and, for the value call, the modality bytes.  Shared by the key and value quantisers:
// it used to be a launch of its own behind each of them (3 us per call).
#pragma once
#include "okq_layout.cuh"

namespace okq {

// thread `id` of `count` working on (layer, sequence b, head h)
__device__ __forceinline__ void bulk_tail_rows(const CacheView& cv, int layer, int b, int h, const __half* src, long long sb,
                                               long long sh, long long st, int n_tokens, bool is_value, int id, int count) {
  const int n_packed = is_value ? cv.v_packed(n_tokens) : cv.k_packed(n_tokens);
  __half* dst = is_value ? cv.v_tail + cv.v_tail_off(layer, b, h) : cv.k_tail + cv.k_tail_off(layer, b, h);
  for (int idx = id; idx < (n_tokens - n_packed) * (D / 8); idx += count) {
    const int t = n_packed + idx / (D / 8), c8 = idx % (D / 8);
    const int slot = is_value ? cv.v_slot(t) : cv.k_slot(t);
    reinterpret_cast<uint4*>(dst + slot * D)[c8] =
        *reinterpret_cast<const uint4*>(src + b * sb + h * sh + (long long)t * st + c8 * 8);
  }
  if (h == 0 && id == 0) cv.seq_len[layer * cv.batch + b] = n_tokens;
}

// thread `id` of `count` working on sequence b: ids beyond the three modalities count as text
__device__ __forceinline__ void bulk_modality(const CacheView& cv, int b, const unsigned char* modality, int n_tokens, int id, int count) {
  const unsigned char* src = modality + (size_t)b * n_tokens;
  unsigned char* dst = cv.modality + (size_t)b * cv.capacity;
  auto one = [](unsigned m) { return (unsigned char)(m > 2 ? 0 : m); };
  if (((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 3) == 0) {   // four bytes at a time
    for (int i = id; i < n_tokens / 4; i += count) {
      const uchar4 m = reinterpret_cast<const uchar4*>(src)[i];
      reinterpret_cast<uchar4*>(dst)[i] = make_uchar4(one(m.x), one(m.y), one(m.z), one(m.w));
    }
    for (int i = (n_tokens & ~3) + id; i < n_tokens; i += count) dst[i] = one(src[i]);
  } else {
    for (int i = id; i < n_tokens; i += count) dst[i] = one(src[i]);
  }
}

}  // namespace okq
