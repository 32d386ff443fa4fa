// 16-byte loads at any alignment: the two aligned chunks that hold the bytes
// are loaded and shifted together in registers (tvc_ragged.cu says when this
// pays).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace tvcg {

struct Chunks {
  uint4 a, b;
};

// The aligned chunks that hold bytes [ad, ad + bytes), 1 <= bytes <= 16.
// KEEP: ordinary loads instead of evict-first ones (the callers say why).
template <bool KEEP = false>
__device__ __forceinline__ void ld_chunks(uint64_t ad, int bytes, Chunks& c) {
  const uint4* p = reinterpret_cast<const uint4*>(ad & ~(uint64_t)15);
  c.a = KEEP ? __ldg(p) : __ldcs(p);
  c.b = make_uint4(0u, 0u, 0u, 0u);
  if ((int)(ad & 15) + bytes > 16) c.b = KEEP ? __ldg(p + 1) : __ldcs(p + 1);
}

// The 16 bytes that start k = ad & 15 bytes into the chunks (ES: element
// size, k a multiple of it).
template <int ES>
__device__ __forceinline__ uint4 cut(const Chunks& c, uint32_t k) {
  uint32_t w0 = c.a.x, w1 = c.a.y, w2 = c.a.z, w3 = c.a.w, w4 = c.b.x, w5 = c.b.y, w6 = c.b.z;
  const uint32_t w7 = c.b.w;
  if (k & 8) {
    w0 = w2;
    w1 = w3;
    w2 = w4;
    w3 = w5;
    w4 = w6;
    w5 = w7;
  }
  if (k & 4) {
    w0 = w1;
    w1 = w2;
    w2 = w3;
    w3 = w4;
    w4 = w5;
  }
  if constexpr (ES < 4) {
    const uint32_t s = (k & 3) * 8;
    w0 = __funnelshift_r(w0, w1, s);
    w1 = __funnelshift_r(w1, w2, s);
    w2 = __funnelshift_r(w2, w3, s);
    w3 = __funnelshift_r(w3, w4, s);
  }
  return make_uint4(w0, w1, w2, w3);
}

}  // namespace tvcg
