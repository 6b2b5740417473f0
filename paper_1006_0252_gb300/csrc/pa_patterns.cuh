// pa_patterns.cuh -- the neighbour patterns of many sites as byte offsets into
// tables of 64 entries, and the compare of a uniform with such an entry
// (threshold-table kernels of the cubic lattices and of general boxes).
#pragma once
#include "pa_device.cuh"

namespace pa {

// Patterns of the sites at bits b = 8 j + r of the words x[0..5]: byte j of
// f[r], x_d at bit d + 2 of the byte (four times the pattern: a byte offset in
// the site's entries).  Pairs of words are first merged into fields of two
// bits (sites of even and of odd b), then fields of the three pairs into bytes.
struct Patterns {
  uint32_t f[8];
  __device__ __forceinline__ explicit Patterns(const uint32_t (&x)[6]) {
    uint32_t e[3], o[3];  // fields i of a byte: sites r = 2 i and 2 i + 1
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      e[d] = (x[2 * d] & 0x55555555u) | ((x[2 * d + 1] << 1) & 0xAAAAAAAAu);
      o[d] = ((x[2 * d] >> 1) & 0x55555555u) | (x[2 * d + 1] & 0xAAAAAAAAu);
    }
    bytes(e, 0);
    bytes(o, 1);
  }
  __device__ __forceinline__ void bytes(const uint32_t (&p)[3], int r) {
    const uint32_t lo = (p[0] & 0x33333333u) | ((p[1] << 2) & 0xCCCCCCCCu);  // fields 0 and 2 of both pairs
    const uint32_t hi = ((p[0] >> 2) & 0x33333333u) | (p[1] & 0xCCCCCCCCu);  // fields 1 and 3
    f[r + 0] = ((lo << 2) & 0x3C3C3C3Cu) | ((p[2] << 6) & 0xC0C0C0C0u);
    f[r + 2] = ((hi << 2) & 0x3C3C3C3Cu) | ((p[2] << 4) & 0xC0C0C0C0u);
    f[r + 4] = ((lo >> 2) & 0x3C3C3C3Cu) | ((p[2] << 2) & 0xC0C0C0C0u);
    f[r + 6] = ((hi >> 2) & 0x3C3C3C3Cu) | (p[2] & 0xC0C0C0C0u);
  }
};

template <int OFF>
__device__ __forceinline__ uint32_t load_shared(uint32_t addr) {
  uint32_t t;
  asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(t) : "r"(addr), "n"(OFF));
  return t;
}

// 2 ge + [u + entry carries].  Both additions run at the full integer rate,
// where a compare into a predicate and a select would each take a half-rate
// slot.  With the entry 2^32 - t the bit is [u >= t].
__device__ __forceinline__ uint32_t shift_in_carry(uint32_t ge, uint32_t u, uint32_t entry) {
  uint32_t r;
  asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %1, %2;\n\taddc.u32 %0, %3, %3;\n\t}"
      : "=r"(r)
      : "r"(u), "r"(entry), "r"(ge));
  return r;
}

}  // namespace pa
