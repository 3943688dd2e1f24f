// What the two split-operand kernels share: the exact three-term split of fp32 into bf16 and the
// magnitudes at which it holds.
//
// fp32 on the tensor cores.  x = h + m + l with h = bf16(x), m = bf16(x - h), l = bf16(x - h - m): three
// significands of 8 bits hold all 24 of x, so of a product x u the six partial products down to
// 2^-16 (hh, hm, mh, mm, hl, lh) leave out less than the rounding of one fp32 operation.  bf16
// products are exact in fp32, but the tensor cores TRUNCATE each addition to an accumulator (measured:
// -6.6e-9 of the value per MMA, a bias of 8.5e-7 after 128 of them where a chain of FMAs errs by
// 1e-7).  Both kernels therefore keep the chains short: the small products have an accumulator of
// their own, and the projection moves the leading one to registers (fp32 additions) every 64 columns.
//
// The split needs room below and above x: rows whose largest magnitude is under kSplitTiny (the low
// terms would leave the range of bf16) or at or over kSplitHuge (h, or a partial sum of it, would
// overflow; infinities and NaN too) are flagged and computed with plain fp32 FMAs instead.
#pragma once

#include "codec_umma.cuh"
#include "generic_kernels.cuh"

namespace ssn {

constexpr uint32_t kSplitHugeBits = 0x7B800000u;   // 2^120
constexpr uint32_t kSplitTinyBits = 0x17800000u;   // 2^-80

__device__ __forceinline__ uint32_t magnitude_bits(float v) { return __float_as_uint(v) & 0x7FFFFFFFu; }
__device__ __forceinline__ bool split_unsafe(uint32_t largest_bits) {
  return largest_bits >= kSplitHugeBits || (largest_bits != 0 && largest_bits < kSplitTinyBits);
}

// Parts h, m, l (NP = 3) or h alone (NP = 1) of the pair (v0, v1), v0 in the low half.
template <int NP>
__device__ __forceinline__ void split_pair(float v0, float v1, uint32_t (&p)[NP]) {
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    p[i] = pack_bf16(v0, v1);
    if (i + 1 < NP) {
      v0 -= __uint_as_float(p[i] << 16);
      v1 -= __uint_as_float(p[i] & 0xFFFF0000u);
    }
  }
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
__device__ __forceinline__ void st_shared_b32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.b32 [%0], %1;\n" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void st_shared_v2(uint32_t addr, uint32_t a, uint32_t b) {
  asm volatile("st.shared.v2.b32 [%0], {%1,%2};\n" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};\n" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// Two neighbouring elements as stored, zeros past `valid` of them; `vec`: the pair may be read at once.
template <typename T> struct Pair { uint32_t w[sizeof(T) / 2]; };
template <typename T>
__device__ __forceinline__ Pair<T> load_pair(const T *p, int valid, bool vec) {
  Pair<T> v;
  if constexpr (sizeof(T) == 4) {
    if (vec && valid > 1) {
      const uint2 x = __ldg(reinterpret_cast<const uint2 *>(p));
      v.w[0] = x.x;
      v.w[1] = x.y;
    } else {
      v.w[0] = valid > 0 ? __float_as_uint(p[0]) : 0u;
      v.w[1] = valid > 1 ? __float_as_uint(p[1]) : 0u;
    }
  } else {
    if (vec && valid > 1) {
      v.w[0] = __ldg(reinterpret_cast<const uint32_t *>(p));
    } else {
      v.w[0] = valid > 0 ? __bfloat16_as_ushort(p[0]) : 0u;
      if (valid > 1) v.w[0] |= (uint32_t)__bfloat16_as_ushort(p[1]) << 16;
    }
  }
  return v;
}
template <typename T>
__device__ __forceinline__ uint32_t pair_magnitude(const Pair<T> &v) {   // of the larger one, as fp32 bits
  if constexpr (sizeof(T) == 4) return max(v.w[0] & 0x7FFFFFFFu, v.w[1] & 0x7FFFFFFFu);
  else return max(v.w[0] & 0x7FFF0000u, (v.w[0] << 16) & 0x7FFF0000u);
}
// Its bf16 parts: three of an fp32 pair (or NP = 1), itself for a bf16 pair.
template <typename T, int NP>
__device__ __forceinline__ void split_pair(const Pair<T> &v, uint32_t (&p)[NP]) {
  if constexpr (sizeof(T) == 4) {
    split_pair<NP>(__uint_as_float(v.w[0]), __uint_as_float(v.w[1]), p);
  } else {
    static_assert(NP == 1, "a bf16 value is its own only part");
    p[0] = v.w[0];
  }
}
inline bool pairs_aligned(const void *p, int64_t ld, int esz) {
  return (reinterpret_cast<uintptr_t>(p) & (2 * esz - 1)) == 0 && (ld & 1) == 0;
}

}  // namespace ssn
