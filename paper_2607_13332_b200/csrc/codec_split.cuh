// What the two split-operand kernels share: the exact three-term split of fp32 into bf16 and the
// magnitudes at which it holds.
//
// fp32 on the tensor cores.  x = h + m + l with h = bf16(x), m = bf16(x - h), l = bf16(x - h - m): three
// significands of 8 bits hold all 24 of x, so of a product x u the six partial products down to
// 2^-16 (hh, hm, mh, mm, hl, lh) leave out less than the rounding of one fp32 operation.  bf16
// products are exact in fp32, but the tensor cores TRUNCATE each addition to an accumulator (measured:
// -6.6e-9 of the value per MMA, a bias of 8.5e-7 after 128 of them where a chain of FMAs errs by
// 1e-7).  Both kernels therefore keep the chains short: the small products have accumulators of
// their own, and the projection moves the leading ones to registers every 64 or 128 columns and adds them up with
// compensation, so that its results are no further from 64-bit sums than those of plain FMAs.
//
// The split needs room: the products of the low parts must not fall below the range of fp32 (2^-126), nor sums of the
// leading ones rise above it.  A row whose largest magnitude is below kSplitTinyRow, or a row or column of an fp32
// U below kSplitTinyU, is computed with plain sums instead, and so is what overflows: the expansion looks for magnitudes
// from kSplitHugeRow and kSplitHugeU on (infinities too), the projection, whose sums are long, for
// sums that are not finite.
#pragma once

#include "codec_umma.cuh"
#include "generic_kernels.cuh"

namespace ssn {

constexpr float kSplitTinyRow = 0x1p-70f, kSplitTinyU = 0x1p-40f, kSplitHugeRow = 0x1p80f, kSplitHugeU = 0x1p40f;

// Two fp32 operations in one instruction.
__device__ __forceinline__ void sub2(float &a0, float &a1, float b0, float b1) {
  asm("{\n.reg .b64 a, b;\nmov.b64 a, {%0, %1};\nmov.b64 b, {%2, %3};\nsub.rn.f32x2 a, a, b;\nmov.b64 {%0, %1}, a;\n}\n"
      : "+f"(a0), "+f"(a1) : "f"(b0), "f"(b1));
}
__device__ __forceinline__ void add2(float &a0, float &a1, float b0, float b1) {
  asm("{\n.reg .b64 a, b;\nmov.b64 a, {%0, %1};\nmov.b64 b, {%2, %3};\nadd.rn.f32x2 a, a, b;\nmov.b64 {%0, %1}, a;\n}\n"
      : "+f"(a0), "+f"(a1) : "f"(b0), "f"(b1));
}

// Parts h, m, l (NP = 3) or h alone (NP = 1) of the pair (v0, v1), v0 in the low half.
template <int NP>
__device__ __forceinline__ void split_pair(float v0, float v1, uint32_t (&p)[NP]) {
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    p[i] = pack_bf16(v0, v1);
    if (i + 1 < NP) sub2(v0, v1, __uint_as_float(p[i] << 16), __uint_as_float(p[i] & 0xFFFF0000u));
  }
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%8], {%0,%1,%2,%3,%4,%5,%6,%7};\n"
               :: "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(taddr) : "memory");
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

__device__ __forceinline__ uint4 ld_shared_v4(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}

// Loads that are predicated, not branched around.
__device__ __forceinline__ uint32_t load_global_b32_if(const void *p, bool ok) {
  uint32_t v;
  asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %2, 0;\nmov.b32 %0, 0;\n@p ld.global.nc.b32 %0, [%1];\n}\n"
               : "=&r"(v) : "l"(p), "r"((int)ok));
  return v;
}
__device__ __forceinline__ uint32_t load_global_b16_if(const void *p, bool ok) {
  uint16_t v;
  asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %2, 0;\nmov.b16 %0, 0;\n@p ld.global.nc.b16 %0, [%1];\n}\n"
               : "=&h"(v) : "l"(p), "r"((int)ok));
  return v;
}
__device__ __forceinline__ uint2 load_global_v2(const void *p) {
  uint2 v;
  asm volatile("ld.global.nc.v2.b32 {%0,%1}, [%2];\n" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ uint32_t load_global_b32(const void *p) {
  uint32_t v;
  asm volatile("ld.global.nc.b32 %0, [%1];\n" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ uint32_t load_global_b16(const void *p) {
  uint16_t v;
  asm volatile("ld.global.nc.b16 %0, [%1];\n" : "=h"(v) : "l"(p));
  return v;
}

__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];\n" ::"l"(p)); }

// Two neighbouring elements as loaded.  A bf16 pair has one word per element until joined() puts them
// into w[0] (w[1] = 0: read at once).
template <typename T> struct Pair { uint32_t w[2]; };
// The pairs at at(0) .. at(N - 1): `valid` says how many of a pair's elements exist (the same for all; the
// others read as 0, and none at all leaves v as it is), `vec` whether a pair may be read at once.  One branch
// for all of them: with one per pair the loads and what follows them were serialised.
template <int N, typename T, typename At>
__device__ __forceinline__ void load_pairs(Pair<T> (&v)[N], At at, int valid, bool vec) {
  if (valid > 1 && vec) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      if constexpr (sizeof(T) == 4) {
        const uint2 x = load_global_v2(at(i));
        v[i].w[0] = x.x;
        v[i].w[1] = x.y;
      } else {
        v[i].w[0] = load_global_b32(at(i));
        v[i].w[1] = 0;
      }
    }
  } else if (valid > 1) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const T *p = at(i);
      v[i].w[0] = sizeof(T) == 4 ? load_global_b32(p) : load_global_b16(p);
      v[i].w[1] = sizeof(T) == 4 ? load_global_b32(p + 1) : load_global_b16(p + 1);
    }
  } else if (valid > 0) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      v[i].w[0] = sizeof(T) == 4 ? load_global_b32(at(i)) : load_global_b16(at(i));
      v[i].w[1] = 0;
    }
  }
}
// The pair as used: two fp32 words, or both bf16 values in w[0].
template <typename T>
__device__ __forceinline__ Pair<T> joined(Pair<T> v) {
  if constexpr (sizeof(T) == 2) {
    v.w[0] |= v.w[1] << 16;
    v.w[1] = 0;
  }
  return v;
}
template <typename T>
__device__ __forceinline__ float pair_magnitude(const Pair<T> &v) {   // of the larger one
  if constexpr (sizeof(T) == 4) return fmaxf(fabsf(__uint_as_float(v.w[0])), fabsf(__uint_as_float(v.w[1])));
  else return fmaxf(fabsf(__uint_as_float(v.w[0] << 16)), fabsf(__uint_as_float(v.w[0] & 0xFFFF0000u)));
}
template <typename T>
__device__ __forceinline__ void pair_maxima(const Pair<T> &v, float (&m)[2]) {   // of either one, into running maxima
  m[0] = fmaxf(m[0], fabsf(__uint_as_float(sizeof(T) == 4 ? v.w[0] : v.w[0] << 16)));
  m[1] = fmaxf(m[1], fabsf(__uint_as_float(sizeof(T) == 4 ? v.w[1] : v.w[0] & 0xFFFF0000u)));
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

// 16 bytes of a row from column c on, element by element (zeros past column d and for a missing row).
template <typename T>
__device__ __forceinline__ uint4 load_row_piece(const T *row, int c, int d) {
  uint32_t w[4];
  const bool ok = row != nullptr;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if constexpr (sizeof(T) == 4)
      w[i] = load_global_b32_if(row + c + i, ok && c + i < d);
    else
      w[i] = load_global_b16_if(row + c + 2 * i, ok && c + 2 * i < d) | load_global_b16_if(row + c + 2 * i + 1, ok && c + 2 * i + 1 < d) << 16;
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}
// The same with an asynchronous copy to shared memory; `ok` = false writes zeros.
__device__ __forceinline__ void cp_async16_if(uint32_t dst, const void *src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}

template <typename T> __device__ __forceinline__ void widen_piece(const uint4 &raw, float *f);
template <> __device__ __forceinline__ void widen_piece<float>(const uint4 &raw, float *f) {
  f[0] = __uint_as_float(raw.x); f[1] = __uint_as_float(raw.y);
  f[2] = __uint_as_float(raw.z); f[3] = __uint_as_float(raw.w);
}
template <> __device__ __forceinline__ void widen_piece<__nv_bfloat16>(const uint4 &raw, float *f) {
  const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    f[2 * i] = __uint_as_float(w[i] << 16);
    f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
  }
}

}  // namespace ssn
