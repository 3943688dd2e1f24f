// tcgen05 / TMA projection of bf16 rows as they are, for the calls that keep the sums of the split kernels
// (codec_split_project.cuh) or whose basis TMA cannot fetch:
//     Z = X U        fp32 words or bf16 rows out, any leading dimension of U and Z
//
// Products of bf16 values are exact, so one part of either operand is all there is, and no thread need touch a row:
//
//   warp 0           producer: the X tile of a stage (128 tokens x 64 columns) by TMA.
//   warps 3, 12-14   basis: 64 rows of U per stage, a stage per warp in turn (see BasisPairs).
//   warps 1, 2       one thread each issues the MMAs of every other stage, the four K steps into four accumulators: each
//                    is written by one MMA, so that nothing is truncated twice (see SplitProjectConfig on what that costs).
//   warps 4-11       sums: of every stage, the four accumulators and the compensated running sum of 32 (or 16)
//                    coordinates of a row per thread, all in registers.  The issuers take turns with two or four sets of accumulators.
//
// What bounds it: no unit by itself.  A stage of 12288 x 5120, rank 51 takes a CTA 0.76 us; the stream alone would take 35 us in all
// (96 CTAs, one tile each), its four MMAs take about 0.2 us, and without the additions, or without the loads of the basis,
// the call takes 59.8 us instead of 63.6.  What is left is the hand-over: from the commit of a stage to the release of its
// accumulators a sum warp reads them in eight rounds of two loads, and two sets of accumulators are in turn.
// In the split kernel the warps that add also copied rows and basis through registers, and a tile was spread over four CTAs
// in three waves.  us, split -> this kernel: 12288 x 5120, rank 51 103 -> 63.6; 40000 x 1536, rank 27 85 -> 41.5; 700 x 1024, rank 19
// 10.7 -> 9.1 (fp32 words out).  Issuers that wait for their own stages only: 12288 x 5120, rank 32 45.9 -> 36.2.
//
// CAREFUL (see kSplitCarefulCols) adds the four accumulators one by one, with compensation: the same sums as the split kernel's.
// 20000 x 320, rank 32: 4.1e-8 from 64-bit sums instead of 5.3e-8, 13.0 us instead of 12.0 (the split kernel 21).
//
// Clusters and halves as in the split kernel.  Every wait is bounded; one that runs out sets SSN_DEV_TIMEOUT and the
// kernel still runs to its end.
#pragma once

#include <type_traits>

#include "codec_split_project.cuh"

namespace ssn {

constexpr int kPlainThreads = 480, kPlainSumWarps = 8, kPlainBasisWarps = 4;

template <int KN>
struct PlainProjectConfig {
  static_assert(KN == 32 || KN == 64, "coordinates, rounded up");
  static constexpr int kXBytes = kUmmaTile * 128, kUBytes = kUmmaCols * 128, kStageBytes = kXBytes + kUBytes;
  static constexpr int kStagesN = 8;
  static constexpr int kAccs = kUmmaCols / 16;                // one accumulator per K step of a stage
  static constexpr int kAccCols = kAccs * KN, kBufs = 512 / kAccCols, kTmemCols = 512;
  static_assert(kAccs == 4, "the sums add up four accumulators per stage");
  static constexpr int kSums = KN / 2;                        // coordinates of one row per thread
  static constexpr int kRingBytes = kStagesN * kStageBytes;
  static_assert(kRingBytes >= 2 * kUmmaTile * (KN + 4) * 4, "the exchanged sums take the place of the ring");
  static constexpr int kBars = 2 * kStagesN + 2 * kBufs;
  static constexpr int kSmemBytes = 1024 + kRingBytes + kBars * 8 + 16;
  static_assert(kSmemBytes <= 227 * 1024, "the ring does not fit in shared memory");
  // A parity tells only the current phase of a barrier from the one before it, so whoever waits has to see every phase.  Stage i
  // belongs to issuer i % 2 and basis warp i % 4; with these numbers a slot, or a set of accumulators, keeps its owners, and
  // an owner waits for each of its phases in turn.
  static_assert(kStagesN % kPlainBasisWarps == 0 && kStagesN % 2 == 0 && kBufs % 2 == 0, "a wait would span two phases");
};

// 64 rows of a bf16 U, at any address and pitch, as a swizzled MN-major operand: one warp, a 4-byte word per lane and row,
// KN / 2 lanes to a row, all rows in flight at a time (one wait for memory per stage).  A row that starts between two words takes
// the second half of each word and the first half of the next lane's.  ODD0, ODD1: whether the even and the odd rows do;
// fixed, so that a row is a load, at most a shuffle and a permutation, a mask and a store (decided row by row, and half
// the rows at a time: 85 us instead of 67 at the sizes above).
template <int KN, bool ODD0, bool ODD1>
struct BasisPairs {
  static constexpr int kLanes = KN / 2, kRows = kUmmaCols * kLanes / 32;   // rows per lane
  const __nv_bfloat16 *U, *u_begin, *u_end;   // this lane's first column; the matrix
  int64_t ldu;
  int d, rank, lane, pair, row0;
  uint32_t mask, w[kRows], last[2];
  // Two rows of an access are 4 apart, so that their swizzled pieces lie in different banks.
  static __device__ __forceinline__ constexpr int row_of(int i) { return KN == 64 ? i : (i >> 2) * 8 + (i & 3); }
  static __device__ __forceinline__ constexpr int odd(int i) { return (i & 1) != 0 ? ODD1 : ODD0; }   // row0 is even
  __device__ __forceinline__ BasisPairs(const SplitProjectArgs &a, const SplitSchedule &s, int lane_) {
    lane = lane_;
    pair = lane % kLanes;
    row0 = lane / kLanes * 4;
    rank = s.rank();
    const int valid = rank - 2 * pair;           // coordinates from this pair on
    mask = valid > 1 ? 0xFFFFFFFFu : (valid == 1 ? 0xFFFFu : 0u);
    u_begin = static_cast<const __nv_bfloat16 *>(a.U);
    u_end = u_begin + (int64_t)(a.d - 1) * a.ldu + a.k;
    // lanes past the last coordinate read the word behind it (which the lane before may need) or one of the row's
    U = u_begin + s.j_lo() + 2 * min(pair, rank / 2);
    ldu = a.ldu;
    d = a.d;
  }
  // the rows of the stage whose first one is c0
  __device__ __forceinline__ void load(int c0) {
    const __nv_bfloat16 *up = U + (int64_t)(c0 + row0) * ldu;
    if (c0 > 0 && c0 + kUmmaCols < d) {
#pragma unroll
      for (int i = 0; i < kRows; ++i) w[i] = load_global_b32(up + row_of(i) * ldu - odd(i));
    } else {   // a word may begin before the matrix or end behind it: half by half
#pragma unroll
      for (int i = 0; i < kRows; ++i) {
        const __nv_bfloat16 *p = up + row_of(i) * ldu - odd(i);
        const bool in = c0 + row0 + row_of(i) < d;
        w[i] = load_global_b16_if(p, in && p >= u_begin && p < u_end);
        w[i] |= load_global_b16_if(p + 1, in && p + 1 >= u_begin && p + 1 < u_end) << 16;
      }
    }
    // the last coordinate of a full row that starts between words has no next lane: lane i fetches those of rows i and
    // i + 32 (or of the two rows of access i)
    if ((ODD0 || ODD1) && rank == KN) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int row = c0 + (KN == 64 ? lane + 32 * h : row_of(lane) + 4 * h);
        last[h] = load_global_b16_if(U + (int64_t)row * ldu + (KN - 1 - 2 * pair), row < d);
      }
    }
  }
  __device__ __forceinline__ void store(uint32_t base) const {
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      uint32_t v = w[i];
      if (odd(i)) {
        uint32_t next = __shfl_down_sync(0xffffffffu, v, 1);
        if (rank == KN) {
          const uint32_t l0 = __shfl_sync(0xffffffffu, KN == 64 ? last[i / 32] : last[0], i % 32);
          const uint32_t l1 = KN == 64 ? l0 : __shfl_sync(0xffffffffu, last[1], i % 32);
          if (pair == kLanes - 1) next = lane < kLanes ? l0 : l1;
        }
        v = __byte_perm(v, next, 0x5432);
      }
      const int r = row_of(i);                   // row0 does not touch the bits that the swizzle of row r takes, but bit 2
      st_shared_b32(base + (row0 + r) * 128 + (((pair >> 2) ^ ((r & 7) + row0)) << 4) + (pair & 3) * 4, v & mask);
    }
  }
};

template <int KN, bool CAREFUL>
__global__ void __launch_bounds__(kPlainThreads, 1)
codec_plain_project_kernel(const SplitProjectArgs a, const __grid_constant__ CUtensorMap x_map) {
  using Cfg = PlainProjectConfig<KN>;
  using T = __nv_bfloat16;
  constexpr int S = Cfg::kStagesN;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

  const SplitSchedule s(a, kUmmaCols);
  const int steps = s.my_tiles * s.nloc;

  const uint32_t smem0 = (smem_u32(smem_raw) + 1023u) & ~1023u, bars = smem0 + Cfg::kRingBytes;
  auto full_bar = [&](int i) { return bars + i * 8; };
  auto empty_bar = [&](int i) { return bars + (S + i) * 8; };
  auto acc_full_bar = [&](int b) { return bars + (2 * S + b) * 8; };
  auto acc_empty_bar = [&](int b) { return bars + (2 * S + Cfg::kBufs + b) * 8; };
  const uint32_t tmem_slot = bars + Cfg::kBars * 8;
  volatile uint32_t *tmem_slot_ptr = reinterpret_cast<volatile uint32_t *>(smem_raw + (tmem_slot - smem_u32(smem_raw)));

  if (threadIdx.x == 0) {
    for (int i = 0; i < S; ++i) {
      mbar_init(full_bar(i), 2);        // the producer and the stage's basis warp
      mbar_init(empty_bar(i), 1);
    }
    for (int b = 0; b < Cfg::kBufs; ++b) {
      mbar_init(acc_full_bar(b), 1);
      mbar_init(acc_empty_bar(b), kPlainSumWarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(tmem_slot),
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

  if (warp == 0) {
    // ------------------------------------------------------------------------- producer
    const uint64_t stream_in = l2_policy_evict_first();
    int slot = 0;
    uint32_t parity = 1;
    for (int it = 0; it < s.my_tiles; ++it) {
      const int tok0 = (int)(s.tile(it) * kUmmaTile);
      for (int st = 0; st < s.nloc; ++st) {
        if (!dead && !mbar_wait(empty_bar(slot), parity)) timed_out();
        if (lane == 0) {
          mbar_expect_tx(full_bar(slot), Cfg::kXBytes);
          tma_load_2d_hint(smem0 + (uint32_t)slot * Cfg::kStageBytes, &x_map, full_bar(slot), (s.st_lo + st) * kUmmaCols, tok0,
                           stream_in);
        }
        __syncwarp();
        if (++slot == S) {
          slot = 0;
          parity ^= 1u;
        }
      }
    }
  } else if (warp == 1 || warp == 2) {
    // ------------------------------------------------------------------------- MMA issuers
    if (lane == 0) {
      constexpr uint32_t idesc = umma_idesc(KN, false);
      const uint64_t adesc0 = umma_desc(0, 16, 1024, 2), bdesc0 = umma_desc(0, Cfg::kUBytes, 1024, 2);
      int slot = warp - 1, buf = warp - 1;
      uint32_t parity = 0, acc_parity = 1;
      for (int step = warp - 1; step < steps; step += 2) {
        if (!dead && !mbar_wait(full_bar(slot), parity)) timed_out();
        if (!dead && !mbar_wait(acc_empty_bar(buf), acc_parity)) timed_out();
        const uint32_t acc = tmem_base + (uint32_t)buf * Cfg::kAccCols;
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const uint32_t base = smem0 + (uint32_t)slot * Cfg::kStageBytes;
        const uint64_t ad = adesc0 + umma_desc_addr(base), bd = bdesc0 + umma_desc_addr(base + Cfg::kXBytes);
#pragma unroll
        for (int j = 0; j < Cfg::kAccs; ++j) umma_bf16(acc + (uint32_t)j * KN, ad + j * 2, bd + j * 128, idesc, 0u);
        umma_commit(empty_bar(slot));
        umma_commit(acc_full_bar(buf));
        slot += 2;
        if (slot >= S) {
          slot -= S;
          parity ^= 1u;
        }
        buf += 2;
        if (buf >= Cfg::kBufs) {
          buf -= Cfg::kBufs;
          acc_parity ^= 1u;
        }
      }
    }
    __syncwarp();
  } else if (warp == 3 || warp >= 12) {
    // ------------------------------------------------------------------------- basis
    auto run = [&](auto odd0, auto odd1) {
      BasisPairs<KN, decltype(odd0)::value, decltype(odd1)::value> u(a, s, lane);
      int slot = warp == 3 ? 0 : warp - 11, st = slot;
      uint32_t parity = 1;
      for (int step = slot; step < steps; step += kPlainBasisWarps) {
        while (st >= s.nloc) st -= s.nloc;
        u.load((s.st_lo + st) * kUmmaCols);
        if (!dead && !mbar_wait(empty_bar(slot), parity)) timed_out();
        u.store(smem0 + (uint32_t)slot * Cfg::kStageBytes + Cfg::kXBytes);
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(full_bar(slot));
        st += kPlainBasisWarps;
        slot += kPlainBasisWarps;
        if (slot >= S) {
          slot -= S;
          parity ^= 1u;
        }
      }
    };
    const bool odd0 = (reinterpret_cast<uintptr_t>(a.U) & 2) != 0, odd1 = odd0 != ((a.ldu & 1) != 0);   // j_lo() is even
    if (odd0) {
      if (odd1) run(std::true_type{}, std::true_type{});
      else run(std::true_type{}, std::false_type{});
    } else {
      if (odd1) run(std::false_type{}, std::true_type{});
      else run(std::false_type{}, std::false_type{});
    }
  } else {
    // ------------------------------------------------------------------------- sums
    const int quarter = warp & 3, row = quarter * 32 + lane, col0 = (warp - 4) / 4 * Cfg::kSums;
    const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + col0;
    float sum[Cfg::kSums], comp[Cfg::kSums];
    int buf = 0;
    uint32_t acc_parity = 0;
    for (int it = 0; it < s.my_tiles; ++it) {
#pragma unroll
      for (int i = 0; i < Cfg::kSums; ++i) sum[i] = comp[i] = 0.f;
      for (int st = 0; st < s.nloc; ++st) {
        if (!dead && !mbar_wait(acc_full_bar(buf), acc_parity)) timed_out();
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        // eight coordinates of two accumulators at a time; the next ones are on their way while these are added up
        uint32_t v[2][2][8];
        auto fetch = [&](int h) {
#pragma unroll
          for (int q = 0; q < 2; ++q)
            tmem_ld8(taddr + (uint32_t)(buf * Cfg::kAccCols + (2 * (h & 1) + q) * KN + h / 2 * 8), v[h & 1][q]);
        };
        fetch(0);
        float x[8];
#pragma unroll
        for (int h = 0; h < Cfg::kSums / 4; ++h) {
          asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
          if (h + 1 < Cfg::kSums / 4) fetch(h + 1);
          const int i = h / 2 * 8;
#pragma unroll
          for (int e = 0; e < 8; e += 2) {
            if constexpr (CAREFUL) {
#pragma unroll
              for (int q = 0; q < 2; ++q)
                add_compensated2(sum[i + e], sum[i + e + 1], comp[i + e], comp[i + e + 1], __uint_as_float(v[h & 1][q][e]),
                                 __uint_as_float(v[h & 1][q][e + 1]));
              continue;
            }
            float y0 = __uint_as_float(v[h & 1][0][e]), y1 = __uint_as_float(v[h & 1][0][e + 1]);
            add2(y0, y1, __uint_as_float(v[h & 1][1][e]), __uint_as_float(v[h & 1][1][e + 1]));
            if ((h & 1) == 0) {
              x[e] = y0, x[e + 1] = y1;
            } else {
              add2(x[e], x[e + 1], y0, y1);
              add_compensated2(sum[i + e], sum[i + e + 1], comp[i + e], comp[i + e + 1], x[e], x[e + 1]);
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty_bar(buf));
        if (++buf == Cfg::kBufs) {
          buf = 0;
          acc_parity ^= 1u;
        }
      }
      if (s.cluster_size == 1) {
        const int64_t t = s.tile(it) * kUmmaTile + row;
        if (t < a.n) {
          uint32_t bad = 0;
#pragma unroll
          for (int i = 0; i < Cfg::kSums; i += 4) {
            const float v[4] = {sum[i], sum[i + 1], sum[i + 2], sum[i + 3]};
            store_coords4<T>(a, t, s.j_lo() + col0 + i, s.j_end(), v);
            if (!sums_stand(v, nullptr)) bad |= 1u << (i / 4);
          }
          if (bad != 0) {
#pragma unroll 1
            for (int i = 0; i < Cfg::kSums / 4 && col0 + 4 * i < s.rank(); ++i)
              if (bad >> i & 1) store_plain_coords4<T>(a, t, s.j_lo() + col0 + 4 * i, s.j_end());
          }
          if (a.wire_ids && col0 == 0 && !s.lower()) static_cast<int32_t *>(a.zout)[t * a.ldzout + a.k] = a.shift.ids[t];
        }
      }
    }
    if (s.cluster_size > 1) {   // the last accumulators are complete, so every stage is consumed: the ring carries the sums
      const uint32_t dst = smem0 + (uint32_t)(row * (KN + 4) + col0) * 4;
#pragma unroll
      for (int c = 0; c < Cfg::kSums; c += 4) {
        st_shared_v4(dst + c * 4, __float_as_uint(sum[c]), __float_as_uint(sum[c + 1]), __float_as_uint(sum[c + 2]),
                     __float_as_uint(sum[c + 3]));
        if (!CAREFUL && s.cluster_size <= kFewSlices)
          st_shared_v4(dst + kUmmaTile * (KN + 4) * 4 + c * 4, __float_as_uint(comp[c]), __float_as_uint(comp[c + 1]),
                       __float_as_uint(comp[c + 2]), __float_as_uint(comp[c + 3]));
      }
    }
  }

  if (s.cluster_size > 1) finish_slices<T, KN, kPlainThreads, false, !CAREFUL>(a, s, smem0, 0, 0);
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"(Cfg::kTmemCols) : "memory");
  }
}

}  // namespace ssn
