// Split-operand tcgen05 projection of the SSN codec:
//     Z = (X [+ R] [- E[ids]] [- P[pos]]) U
// for fp32 storage, and for the bf16 calls whose operands the TMA projection cannot fetch: leading
// dimensions or addresses off the 16-byte grid, positions per token, a residual addend beside row tables.
//
// Threads load the rows straight into registers (any alignment, any row per token), form the residual
// in fp32 as the general kernel does, split it into bf16 parts (codec_split.cuh) and write them as
// swizzled operand tiles; the basis is split the same way, stage by stage.  With bf16 rows and no
// subtraction one part is exact, and bf16 bases have one part.
//
// Sixteen warps (128 registers a thread), all in the same roles, one 64-column stage per step:
//   - the residuals of the stage are formed from the rows in flight, and the rows of the next one are
//     requested (16 values per thread and operand: what covers the HBM latency);
//   - one thread issues the MMAs of the stage before: Ah x (Uh|Um|Ul), Am x (Uh|Um), Al x Uh, the parts of U
//     side by side on N so that three instructions per K step cover the six products (rank above
//     64: five instructions, (Uh|Um) being 256 columns wide);
//   - the finished accumulator of the stage two back is added to the fp32 sums in registers (see
//     codec_split.cuh on why the chains are this short); warp w reads TMEM lanes 32 (w % 4) .. +31 and a
//     quarter of the columns;
//   - the residuals and the slice of U are split and written to the stage.
// Waiting for the accumulator of step s - 2 before writing step s is also what makes two stages of
// shared memory enough, with no barrier for a free stage or a free accumulator.
//
// A CTA takes whole tiles of 128 tokens; when there are fewer tiles than SMs, a cluster of 2, 4 or 8
// CTAs shares one tile, each contracting a slice of d, and the partial sums meet through distributed
// shared memory, every CTA finishing its share of the rows.
#pragma once

#include "codec_split.cuh"

namespace ssn {

struct SplitProjectArgs {
  const void *src, *src2, *U;
  void *zout;
  int64_t lds, lds2, ldu, ldzout, n;
  int32_t d, k;
  int32_t wire, wire_ids;      // fp32 words out, word k of a row = the token id
  int32_t has_e, has_p;
  int32_t vec_rows;            // every row operand may be read 16 bytes at a time
  int32_t vec_u, vec_out;      // two coordinates of U may be read, four coordinates stored at a time
  ShiftTables shift;
};

constexpr int kSplitProjectWarps = 16;
constexpr int kSplitProjectThreads = 32 * kSplitProjectWarps;
constexpr int kSplitCols = 64;                        // columns of d per stage
constexpr int kSplitPartBytes = kUmmaTile * 128;      // one bf16 part of a [128 x 64] operand

template <typename T, int KN, int NSLOT>
struct SplitProjectConfig {
  static_assert(KN == 32 || KN == 64 || KN == 128, "coordinates, rounded up");
  static constexpr bool kF32 = sizeof(T) == 4;
  static constexpr int kNX = kF32 || NSLOT > 0 ? 3 : 1;    // parts of the residual
  static constexpr int kNU = kF32 ? 3 : 1;                 // parts of U
  static constexpr int kStack = kNU == 3 ? (KN <= 64 ? 3 : 2) : 1;   // parts of U under one Ah product
  static constexpr int kDCols = kNX == 1 ? KN : (kStack == 3 ? 3 : 2) * KN;
  static constexpr int kDStride = kDCols <= 32 ? 32 : (kDCols <= 64 ? 64 : (kDCols <= 128 ? 128 : 256));
  static constexpr int kTmemCols = 2 * kDStride;
  static constexpr int kABytes = kNX * kSplitPartBytes;
  static constexpr int kBGroups = (kNU * KN + 63) / 64;     // 64-coordinate groups of all parts
  static constexpr int kGroupBytes = kSplitCols * 128;
  static constexpr int kStageBytes = kABytes + kBGroups * kGroupBytes;
  static constexpr int kSumPitch = KN + 4;                  // floats per row of the exchanged sums
  // two stages, or the exchanged sums in their place
  static constexpr int kRingBytes = 2 * kStageBytes > kUmmaTile * kSumPitch * 4 ? 2 * kStageBytes : kUmmaTile * kSumPitch * 4;
  static constexpr int kBars = 4;
  static constexpr int kSmemBytes = 1024 + kRingBytes + kBars * 8 + 16;   // barriers, TMEM address, unsafe-value flags
  static_assert(kSmemBytes <= 227 * 1024, "no room for two stages");
  static constexpr int kCtasPerSm = kNX == 1 && KN <= 64 ? 2 : 1;   // one part and few sums: two CTAs hide each other's waits
  static constexpr int kPairs = KN / 16;                    // pairs of U per thread and stage
  static constexpr int kSums = KN / 4;                      // coordinates of one row per thread
  static constexpr int kVecs = kF32 ? 4 : 2;                // 16-byte pieces per thread, operand and stage
  static constexpr int kVecElems = kF32 ? 4 : 8;
};

// 16 bytes of a row from column c on (zeros past column d and for a missing row).
template <typename T>
__device__ __forceinline__ uint4 load_row_piece(const T *row, int c, int d, bool vec) {
  constexpr int E = 16 / (int)sizeof(T);
  uint4 raw = make_uint4(0, 0, 0, 0);
  if (row == nullptr || c >= d) return raw;
  if (vec) return __ldg(reinterpret_cast<const uint4 *>(row + c));   // vec: d is a multiple of E
  T e[E];
#pragma unroll
  for (int i = 0; i < E; ++i) e[i] = c + i < d ? row[c + i] : from_f32<T>(0.f);
  memcpy(&raw, e, 16);
  return raw;
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

template <typename T>
__device__ __forceinline__ void store_coords4(const SplitProjectArgs &a, int64_t t, int j, const float (&v)[4]) {
  if (j >= a.k) return;
  if (a.wire || sizeof(T) == 4) {
    float *z = static_cast<float *>(a.zout) + t * a.ldzout + j;
    if (a.vec_out && j + 4 <= a.k) {
      *reinterpret_cast<float4 *>(z) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (j + e < a.k) z[e] = v[e];
    }
  } else {
    __nv_bfloat16 *z = static_cast<__nv_bfloat16 *>(a.zout) + t * a.ldzout + j;
    if (a.vec_out && j + 4 <= a.k) {
      *reinterpret_cast<uint2 *>(z) = make_uint2(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]));
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (j + e < a.k) z[e] = __float2bfloat16_rn(v[e]);
    }
  }
}

// Rows [row0, row0 + rows) of a tile again with plain FMAs, those whose residual the split does not hold
// (all of them with `all`): one warp per row, lane = coordinate.
template <typename T>
__device__ __noinline__ void project_unsafe_rows(const SplitProjectArgs &a, int64_t tile, int row0, int rows, bool all) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const T *U = static_cast<const T *>(a.U);
  for (int rr = row0 + warp; rr < row0 + rows; rr += kSplitProjectWarps) {
    const int64_t t = tile * kUmmaTile + rr;
    if (t >= a.n) return;
    const T *x = static_cast<const T *>(a.src) + t * a.lds;
    const T *x2 = a.src2 != nullptr ? static_cast<const T *>(a.src2) + t * a.lds2 : nullptr;
    const int64_t er = a.has_e ? embedding_row(a.shift, t) : -1, pr = a.has_p ? position_row(a.shift, t) : -1;
    const T *e = er >= 0 ? static_cast<const T *>(a.shift.E) + er * a.shift.lde : nullptr;
    const T *p = pr >= 0 ? static_cast<const T *>(a.shift.P) + pr * a.shift.ldp : nullptr;
    auto residual = [&](int i) {
      float r = to_f32(x[i]);
      if (x2 != nullptr) r += to_f32(x2[i]);
      if (e != nullptr) r -= to_f32(e[i]);
      if (p != nullptr) r -= to_f32(p[i]);
      return r;
    };
    uint32_t m = 0;
    for (int i = lane; i < a.d; i += 32) m = max(m, magnitude_bits(residual(i)));
    m = __reduce_max_sync(0xffffffffu, m);
    if (!all && !split_unsafe(m)) continue;
    for (int j = lane; j < a.k; j += 32) {
      float acc = 0.f;
      for (int i = 0; i < a.d; ++i) acc = fmaf(residual(i), to_f32(U[(int64_t)i * a.ldu + j]), acc);
      if (a.wire || sizeof(T) == 4)
        static_cast<float *>(a.zout)[t * a.ldzout + j] = acc;
      else
        static_cast<__nv_bfloat16 *>(a.zout)[t * a.ldzout + j] = __float2bfloat16_rn(acc);
    }
  }
}

template <typename T, int KN, int NSLOT>
__global__ void __launch_bounds__(kSplitProjectThreads, (SplitProjectConfig<T, KN, NSLOT>::kCtasPerSm))
codec_split_project_kernel(const SplitProjectArgs a) {
  using Cfg = SplitProjectConfig<T, KN, NSLOT>;
  constexpr int NX = Cfg::kNX, NU = Cfg::kNU;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  uint32_t cluster_size, cta_rank;
  asm volatile("mov.u32 %0, %%cluster_nctaid.x;\n" : "=r"(cluster_size));
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(cta_rank));
  const int64_t ntiles = (a.n + kUmmaTile - 1) / kUmmaTile;
  const int64_t groups = gridDim.x / cluster_size, group = blockIdx.x / cluster_size;
  const int nst = (a.d + kSplitCols - 1) / kSplitCols;
  const int st_lo = (int)((int64_t)nst * cta_rank / cluster_size);
  const int nloc = (int)((int64_t)nst * (cta_rank + 1) / cluster_size) - st_lo;   // >= 1: cluster_size <= nst
  const int my_tiles = (int)((ntiles - group + groups - 1) / groups);             // 1 with clusters
  const int steps = my_tiles * nloc;

  const uint32_t smem_u = smem_u32(smem_raw), smem0 = (smem_u + 1023u) & ~1023u;
  const uint32_t bars = smem0 + Cfg::kRingBytes;
  auto full_bar = [&](int s) { return bars + s * 8; };
  auto acc_full_bar = [&](int b) { return bars + (2 + b) * 8; };
  unsigned char *tail = smem_raw + (bars - smem_u) + Cfg::kBars * 8;
  volatile uint32_t *tmem_slot_ptr = reinterpret_cast<volatile uint32_t *>(tail);
  // bit 0: some row may hold values its split does not; bit 1: U does
  uint32_t *unsafe = reinterpret_cast<uint32_t *>(tail + 4);

  if (tid == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(full_bar(s), kSplitProjectWarps);
      mbar_init(acc_full_bar(s), 1);
    }
    *unsafe = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tail)),
                 "r"(Cfg::kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem_base = *tmem_slot_ptr;
  // set-up done; nothing in global memory is touched before the kernel in front has completed
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  bool dead = false;
  auto timed_out = [&]() {
    dead = true;
    if (a.shift.dev_status) atomicOr(a.shift.dev_status, SSN_DEV_TIMEOUT);
  };

  float sum[Cfg::kSums];
#pragma unroll
  for (int i = 0; i < Cfg::kSums; ++i) sum[i] = 0.f;
  const int quarter = warp & 3, part = warp >> 2;     // TMEM lanes and columns of this warp's sums
  const int sum_row = quarter * 32 + lane, sum_col = part * Cfg::kSums;

  // Four lanes per row; the order of a warp's eight rows makes the swizzled stores conflict-free
  // (8-byte stores per half warp, 16-byte ones per quarter).
  const int idx = lane >> 2, q = lane & 3;
  const int row = warp * 8 + (Cfg::kF32 ? ((idx & 3) << 1 | idx >> 2) : ((idx & 1) << 2 | idx >> 1));
  const bool vec = a.vec_rows != 0;
  const T *U = static_cast<const T *>(a.U);
  const T *ptr[1 + NSLOT];                 // this thread's row: X, then R, E, P as far as present
  uint4 in[1 + NSLOT][Cfg::kVecs];
  Pair<T> ureg[Cfg::kPairs];
  const bool has_r = NSLOT > 0 && a.src2 != nullptr;

  auto row_pointers = [&](int64_t tile) {
    const int64_t t = tile * kUmmaTile + row;
    const bool live = t < a.n;
    ptr[0] = live ? static_cast<const T *>(a.src) + t * a.lds : nullptr;
    if (NSLOT > 0) {
      int s = 1;
      const T *r = nullptr, *e = nullptr, *p = nullptr;
      if (live) {
        if (has_r) r = static_cast<const T *>(a.src2) + t * a.lds2;
        const int64_t er = a.has_e ? embedding_row(a.shift, t) : -1, pr = a.has_p ? position_row(a.shift, t) : -1;
        if (er >= 0) e = static_cast<const T *>(a.shift.E) + er * a.shift.lde;
        if (pr >= 0) p = static_cast<const T *>(a.shift.P) + pr * a.shift.ldp;
      }
      // slots in the order R, E, P; with constant indexes so that the array stays in registers
      const T *list[3] = {r, e, p};
      const bool present[3] = {has_r, a.has_e != 0, a.has_p != 0};
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (!present[c]) continue;
#pragma unroll
        for (int i = 1; i <= NSLOT; ++i)
          if (i == s) ptr[i] = list[c];
        ++s;
      }
    }
  };
  auto issue = [&](int st) {               // rows and slice of U of a stage into registers
    const int c0 = (st_lo + st) * kSplitCols;
#pragma unroll
    for (int i = 0; i < Cfg::kPairs; ++i) {
      const int p = tid + i * kSplitProjectThreads, kk = p / (KN / 2), j = 2 * (p % (KN / 2));
      ureg[i] = load_pair<T>(U + (int64_t)(c0 + kk) * a.ldu + j, c0 + kk < a.d ? a.k - j : 0, a.vec_u != 0);
    }
#pragma unroll
    for (int o = 0; o < 1 + NSLOT; ++o)
#pragma unroll
      for (int i = 0; i < Cfg::kVecs; ++i)
        in[o][i] = load_row_piece<T>(ptr[o], c0 + (4 * i + q) * Cfg::kVecElems, a.d, vec);
  };
  auto issue_mma = [&](int step) {         // one thread
    const int buf = step & 1;
    if (!dead && !mbar_wait(full_bar(buf), (uint32_t)((step >> 1) & 1))) timed_out();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    // A: K-major rows of 128 bytes, 8-row groups 1024 bytes apart, one part after the other.  B: MN-major,
    // 64-coordinate groups kGroupBytes apart, 8-row groups 1024 bytes apart.
    constexpr uint32_t id1 = umma_idesc(KN, false), id2 = umma_idesc(Cfg::kStack >= 2 ? 2 * KN : KN, false),
                       id3 = umma_idesc(Cfg::kStack == 3 ? 3 * KN : KN, false);
    const uint32_t base = smem0 + (uint32_t)buf * Cfg::kStageBytes;
    const uint32_t D = tmem_base + (uint32_t)buf * Cfg::kDStride;
    const uint64_t ad = umma_desc(base, 16, 1024, 2), bd = umma_desc(base + Cfg::kABytes, Cfg::kGroupBytes, 1024, 2);
    constexpr uint32_t kPart = kSplitPartBytes >> 4;                             // next part of A
    constexpr uint32_t kBPart = (uint32_t)(KN / 64) * (Cfg::kGroupBytes >> 4);   // next part of B (KN = 128 only)
#pragma unroll
    for (int j = 0; j < kSplitCols / 16; ++j) {
      const uint64_t A = ad + j * 2, B = bd + j * 128;   // 32 bytes of an A row; 16 rows of B
      const uint32_t more = j > 0 ? 1u : 0u;
      if (NX == 1) {
        umma_bf16(D, A, B, id1, more);
      } else if (NU == 1) {
        umma_bf16(D, A, B, id1, more);
        umma_bf16(D + KN, A + kPart, B, id1, more);
        umma_bf16(D + KN, A + 2 * kPart, B, id1, 1u);
      } else if (Cfg::kStack == 3) {
        umma_bf16(D, A, B, id3, more);
        umma_bf16(D + KN, A + kPart, B, id2, 1u);
        umma_bf16(D + 2 * KN, A + 2 * kPart, B, id1, 1u);
      } else {
        umma_bf16(D, A, B, id2, more);
        umma_bf16(D + KN, A + kPart, B, id1, 1u);
        umma_bf16(D + KN, A + kPart, B + kBPart, id1, 1u);
        umma_bf16(D + KN, A + 2 * kPart, B, id1, 1u);
        umma_bf16(D + KN, A, B + 2 * kBPart, id1, 1u);
      }
    }
    umma_commit(acc_full_bar(buf));
  };

  int ld_tile = 0, ld_st = 0;              // the step whose rows are in flight
  row_pointers(group);
  issue(0);
  int fin_tile = 0, fin_st = 0;            // the step whose accumulator is being added
  uint32_t u_max = 0, row_max = 0;
  for (int step = 0; step < steps + 2; ++step) {
    const bool writing = step < steps;
    float r[NX == 3 ? 16 : 1];             // the residuals of the step, or its rows as they are
    uint4 raw[NX == 3 ? 1 : Cfg::kVecs];
    Pair<T> u[Cfg::kPairs];
    if (writing) {
#pragma unroll
      for (int i = 0; i < Cfg::kPairs; ++i) u[i] = ureg[i];
      if constexpr (NX == 1) {
#pragma unroll
        for (int i = 0; i < Cfg::kVecs; ++i) raw[i] = in[0][i];
      } else {
        constexpr int E = Cfg::kVecElems;
#pragma unroll
        for (int i = 0; i < Cfg::kVecs; ++i) {
          widen_piece<T>(in[0][i], r + E * i);
#pragma unroll
          for (int o = 1; o <= NSLOT; ++o) {
            float w[E];
            widen_piece<T>(in[o][i], w);
            const bool plus = o == 1 && has_r;
#pragma unroll
            for (int e = 0; e < E; ++e) r[E * i + e] = plus ? r[E * i + e] + w[e] : r[E * i + e] - w[e];
          }
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) row_max = max(row_max, magnitude_bits(r[i]));
#pragma unroll
        for (int i = 0; i < Cfg::kPairs; ++i) u_max = max(u_max, pair_magnitude<T>(u[i]));
      }
      if (step + 1 < steps) {
        if (++ld_st == nloc) {
          ld_st = 0;
          ++ld_tile;
          row_pointers(group + ld_tile * groups);
          // this thread's part of the row: a row can be unsafe only if one of its parts is
          if (NX == 3 && split_unsafe(row_max)) atomicOr(unsafe, 1u);
          row_max = 0;
        }
        issue(ld_st);
      }
    }
    if (warp == 0 && step >= 1 && step <= steps) {
      if (lane == 0) issue_mma(step - 1);
      __syncwarp();
    }
    if (step >= 2) {
      // -------- the accumulator of two steps back into the sums
      const int s2 = step - 2, buf = s2 & 1;
      if (!dead && !mbar_wait(acc_full_bar(buf), (uint32_t)((s2 >> 1) & 1))) timed_out();
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      if (sum_col < a.k) {
        const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)buf * Cfg::kDStride + sum_col;
#pragma unroll
        for (int c = 0; c < Cfg::kSums; c += 8) {
          uint32_t v0[8], v1[8], v2[8];
          tmem_ld8(taddr + c, v0);
          if (NX > 1) tmem_ld8(taddr + KN + c, v1);
          if (Cfg::kStack == 3) tmem_ld8(taddr + 2 * KN + c, v2);
          asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            float v = __uint_as_float(v0[e]);
            if (Cfg::kStack == 3)
              v += __uint_as_float(v1[e]) + __uint_as_float(v2[e]);
            else if (NX > 1)
              v += __uint_as_float(v1[e]);
            sum[c + e] += v;
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      if (++fin_st == nloc) {              // a tile is complete
        fin_st = 0;
        const int64_t t = (group + (int64_t)fin_tile * groups) * kUmmaTile + sum_row;
        ++fin_tile;
        if (cluster_size == 1) {
          if (t < a.n) {
#pragma unroll
            for (int c = 0; c < Cfg::kSums; c += 4)
              store_coords4<T>(a, t, sum_col + c, {sum[c], sum[c + 1], sum[c + 2], sum[c + 3]});
            if (a.wire_ids && part == 0) static_cast<int32_t *>(a.zout)[t * a.ldzout + a.k] = a.shift.ids[t];
          }
#pragma unroll
          for (int i = 0; i < Cfg::kSums; ++i) sum[i] = 0.f;
        }
      }
    }
    if (writing) {
      // -------- residuals and basis into the stage
      const uint32_t base = smem0 + (uint32_t)(step & 1) * Cfg::kStageBytes;
      const uint32_t arow = base + row * 128;
      if constexpr (NX == 1) {             // columns 32 i + 8 q .. +7
#pragma unroll
        for (int i = 0; i < Cfg::kVecs; ++i)
          st_shared_v4(arow + (((4 * i + q) ^ (row & 7)) << 4), raw[i].x, raw[i].y, raw[i].z, raw[i].w);
      } else if constexpr (Cfg::kF32) {    // columns 16 i + 4 q .. +3
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          uint32_t lo[3], hi[3];
          split_pair<3>(r[4 * i], r[4 * i + 1], lo);
          split_pair<3>(r[4 * i + 2], r[4 * i + 3], hi);
          const uint32_t addr = arow + (((2 * i + (q >> 1)) ^ (row & 7)) << 4) + (q & 1) * 8;
#pragma unroll
          for (int p = 0; p < 3; ++p) st_shared_v2(addr + p * kSplitPartBytes, lo[p], hi[p]);
        }
      } else {                             // columns 32 i + 8 q .. +7
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          uint32_t w[4][3];
#pragma unroll
          for (int e = 0; e < 4; ++e) split_pair<3>(r[8 * i + 2 * e], r[8 * i + 2 * e + 1], w[e]);
          const uint32_t addr = arow + (((4 * i + q) ^ (row & 7)) << 4);
#pragma unroll
          for (int p = 0; p < 3; ++p) st_shared_v4(addr + p * kSplitPartBytes, w[0][p], w[1][p], w[2][p], w[3][p]);
        }
      }
      const uint32_t bbase = base + Cfg::kABytes;
#pragma unroll
      for (int i = 0; i < Cfg::kPairs; ++i) {
        const int p = tid + i * kSplitProjectThreads, kk = p / (KN / 2), j = 2 * (p % (KN / 2));
        uint32_t up[NU];
        split_pair<T, NU>(u[i], up);
#pragma unroll
        for (int s = 0; s < NU; ++s) {
          const int n = s * KN + j;
          st_shared_b32(bbase + (n >> 6) * Cfg::kGroupBytes + kk * 128 + ((((n & 63) >> 3) ^ (kk & 7)) << 4) + (n & 7) * 2,
                        up[s]);
        }
      }
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(full_bar(step & 1));
    }
  }
  if (NX == 3) {
    if (split_unsafe(row_max)) atomicOr(unsafe, 1u);
    if (u_max >= kSplitHugeBits) atomicOr(unsafe, 2u);
  }

  if (cluster_size > 1) {
    // Every accumulator has been read, so every stage is consumed and the ring can carry the sums.
    __syncthreads();
    const uint32_t dst = smem0 + (uint32_t)(sum_row * Cfg::kSumPitch + sum_col) * 4;
#pragma unroll
    for (int c = 0; c < Cfg::kSums; c += 4)
      st_shared_v4(dst + c * 4, __float_as_uint(sum[c]), __float_as_uint(sum[c + 1]), __float_as_uint(sum[c + 2]),
                   __float_as_uint(sum[c + 3]));
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    const int rows = kUmmaTile / (int)cluster_size, row0 = rows * (int)cta_rank;
    auto peer = [](uint32_t addr, uint32_t rank) {
      uint32_t r;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(addr), "r"(rank));
      return r;
    };
    for (int i = tid; i < rows * (KN / 4); i += kSplitProjectThreads) {
      const int rr = row0 + i / (KN / 4), j = 4 * (i % (KN / 4));
      const int64_t t = group * kUmmaTile + rr;
      if (t >= a.n || j >= a.k) continue;
      float v[4] = {0.f, 0.f, 0.f, 0.f};
      for (uint32_t rk = 0; rk < cluster_size; ++rk) {
        float w0, w1, w2, w3;
        asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];\n"
                     : "=f"(w0), "=f"(w1), "=f"(w2), "=f"(w3)
                     : "r"(peer(smem0 + (uint32_t)(rr * Cfg::kSumPitch + j) * 4, rk)));
        v[0] += w0; v[1] += w1; v[2] += w2; v[3] += w3;
      }
      store_coords4<T>(a, t, j, v);
      if (a.wire_ids && j == 0) static_cast<int32_t *>(a.zout)[t * a.ldzout + a.k] = a.shift.ids[t];
    }
    uint32_t bad = 0;
    if (NX == 3) {
      for (uint32_t rk = 0; rk < cluster_size; ++rk) {
        uint32_t f;
        asm volatile("ld.shared::cluster.u32 %0, [%1];\n" : "=r"(f) : "r"(peer(smem_u32(unsafe), rk)));
        bad |= f;
      }
    }
    // nobody leaves while its sums can still be read
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    if (NX == 3 && bad != 0) project_unsafe_rows<T>(a, group, row0, rows, (bad & 2) != 0);
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"(Cfg::kTmemCols)
                 : "memory");
  }
  if (NX == 3 && cluster_size == 1) {      // the rows stored above are complete behind the barrier
    const uint32_t bad = *unsafe;
    if (bad != 0)
      for (int i = 0; i < my_tiles; ++i) project_unsafe_rows<T>(a, group + i * groups, 0, kUmmaTile, (bad & 2) != 0);
  }
}

}  // namespace ssn
