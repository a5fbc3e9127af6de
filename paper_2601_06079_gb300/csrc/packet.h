// 16-byte packets that carry their own arrival: two 64-bit words, each a value's
// 32 bits under the tag of the exchange (k_onchip2d.cu, k_newton2d.cu).  A word is
// one memory operation, so a reader that finds the tag has the value with it; the
// two words need no order, as each has a tag of its own.  No fence and no flag
// lie on the path of what a packet carries.
#pragma once

#include <cuda_runtime.h>

namespace pf {

struct alignas(16) Packet {
  unsigned long long a, b;
};

__device__ __forceinline__ unsigned long long tagged(unsigned value, unsigned tag) {
  unsigned long long w;
  asm("mov.b64 %0, {%1, %2};" : "=l"(w) : "r"(value), "r"(tag));
  return w;
}
__device__ __forceinline__ unsigned value_of(unsigned long long w) {
  unsigned v;
  asm("{ .reg .b32 t; mov.b64 {%0, t}, %1; }" : "=r"(v) : "l"(w));
  return v;
}
__device__ __forceinline__ unsigned tag_of(unsigned long long w) {
  unsigned t;
  asm("{ .reg .b32 v; mov.b64 {v, %0}, %1; }" : "=r"(t) : "l"(w));
  return t;
}

__device__ __forceinline__ void publish(Packet* p, unsigned a, unsigned b, unsigned tag) {
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(tagged(a, tag)),
               "l"(tagged(b, tag))
               : "memory");
}
__device__ __forceinline__ Packet look(const Packet* p) {
  Packet q;
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];"
               : "=l"(q.a), "=l"(q.b)
               : "l"(p)
               : "memory");
  return q;
}
__device__ __forceinline__ bool arrived(const Packet& q, unsigned tag) {
  return tag_of(q.a) == tag && tag_of(q.b) == tag;
}

}  // namespace pf
