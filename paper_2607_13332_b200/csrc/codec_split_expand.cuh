// Split-operand tcgen05 expansion of the SSN codec:
//     Xhat = Z U^T [+ E[ids]] [+ P[pos]]
// for fp32 storage, for fp32 wire rows, and for the bf16 calls the TMA expansion does not take: leading
// dimensions or addresses off the 16-byte grid, positions per token or of any sequence length.
//
// A unit is 128 tokens x 128 output columns; the units are dealt to the CTAs in contiguous ranges.
//
//   warps 0-7    epilogue, two warps per 32 rows: TMEM lane = row; 128 bytes of every row at a time (a piece),
//                half of it per warp, the E and P pieces added from shared memory, the sum written in place and
//                handed to a TMA store (or, off the 16-byte grid, stored by the warps themselves).  Plain stores
//                of the whole output blocked the load pipe for everyone else (8192 x 2048 fp32: E and P rows
//                76 -> 45 us with TMA stores and gathered rows, no tables 35 -> 31 us).  Both warps take every piece, so each follows the phases of
//                every stage of the ring.
//   warps 8-11   gather the E and P rows with cp.async into a ring of such pieces (E, then P), 32 rows each; a
//                quarter of a stage is handed over at a time.
//   warps 12-19  operands: Z once per tile and 128 rows of U per unit, loaded pair by pair of elements, split
//                into bf16 parts (codec_split.cuh) and written as swizzled K-major tiles of 64 coordinates; a
//                ring of such U tiles runs ahead of the MMAs.
//   warp 20      one thread issues the MMAs (M = 128, N = 128): the leading product into one accumulator,
//                the small ones (hm, mh, mm, hl, lh) into a second, two sets of both.  A warp of its own, since
//                every MMA blocks its thread for about 80 clocks.
//
// Coordinates past k are zeroed once (above rank 64, where a stage of U serves both groups of 64, with every tile
// of U), rows past n or d repeat the last one and are never stored.
#pragma once

#include <type_traits>

#include "codec_split.cuh"
#include "codec_umma_roundtrip.cuh"

namespace ssn {

struct SplitExpandArgs {
  const void *zin, *U;
  void *dst;
  int64_t ldzin, ldu, lddst, n;
  int32_t d, k;
  int32_t has_e, has_p;
  int32_t vec_z, vec_u;        // two coordinates of Z / U may be read at a time
  int32_t vec_rows;            // E and P rows may be read 16 bytes at a time and g_zero_row holds a row
  int32_t tma_out;             // the output is stored through the tensor map
  ShiftTables shift;
};

constexpr int kSplitEpilogueWarps = 8, kSplitGatherWarps = 4, kSplitOperandWarps = 8;
constexpr int kSplitOperandWarp0 = kSplitEpilogueWarps + kSplitGatherWarps, kSplitMmaWarp = kSplitOperandWarp0 + kSplitOperandWarps;
constexpr int kSplitExpandThreads = 32 * (kSplitMmaWarp + 1);
constexpr int kSplitTileBytes = kUmmaTile * 128;     // one part of [128 rows x 64 coordinates]; one piece of 128 rows

// TZ: type of the coordinates (float for fp32 storage and wire rows), T: storage type, KG: groups of 64 coordinates
template <typename T, typename TZ, int KG, int NSLOT>
struct SplitExpandConfig {
  static constexpr int kNZ = sizeof(TZ) == 4 ? 3 : 1, kNU = sizeof(T) == 4 ? 3 : 1;
  static constexpr int kZBytes = kNZ * KG * kSplitTileBytes;
  static constexpr int kZBufs = kNZ == 1 ? 2 : 1;
  static constexpr int kUStageBytes = kNU * kSplitTileBytes;
  static constexpr int kUStages = kNU == 3 ? 2 : 3;
  static constexpr bool kLow = kNZ > 1 || kNU > 1;          // a second accumulator for the small products
  static constexpr int kDCols = (kLow ? 2 : 1) * kChunkCols;
  static constexpr int kTmemCols = 2 * kDCols;
  static constexpr int kPieceCols = 128 / (int)sizeof(T), kPieces = kChunkCols / kPieceCols;
  static constexpr int kOperandBytes = kZBufs * kZBytes + kUStages * kUStageBytes;
  static constexpr int kRoom = 227 * 1024 - 1024 - 2048 - kOperandBytes;
  // the ring of pieces: gathered rows that become output, or output alone
  static constexpr int kFit = kRoom / kSplitTileBytes;
  static constexpr int kRing = NSLOT == 0 ? (kFit < 4 ? kFit : 4) : (kFit < 10 ? kFit : 10);
  static_assert(kRing >= 2, "no room for the output");
  // a stage goes back when the next store is under way, unless the ring is too short to wait for that
  static constexpr bool kHold = NSLOT == 0 ? kRing > 2 : kRing >= 4 * NSLOT;
  static constexpr int kOutBytes = kRing * kSplitTileBytes;
  static constexpr int kBars = 4 + 2 * kUStages + 4 + 8 * kRing;
  static constexpr int kUnsafeSlots = 8;                    // units whose U values may be flagged at a time
  static constexpr int kTailBytes = kBars * 8 + 16 + kUnsafeSlots * kSplitOperandWarps + 4 * kUmmaTile;
  static constexpr int kSmemBytes = 1024 + kOperandBytes + kOutBytes + kTailBytes;
  static_assert(kSmemBytes <= 227 * 1024, "the operands do not fit in shared memory");
};

// What a row's largest magnitude (by fmaxf, which skips NaN: a NaN stays one through its leading part) says about its
// split, ordered so that the larger class of two halves is that of the whole row.
__device__ __forceinline__ unsigned char magnitude_class(float largest) {
  return largest == 0.f ? 0 : (largest < kSplitTinyRow ? 1 : (largest < kSplitHugeRow ? 2 : 3));
}

template <typename T, typename TZ, int KG, int NSLOT>
__global__ void __launch_bounds__(kSplitExpandThreads, 1) codec_split_expand_kernel(const SplitExpandArgs a, const __grid_constant__ CUtensorMap out_map) {
  using Cfg = SplitExpandConfig<T, TZ, KG, NSLOT>;
  constexpr int NZ = Cfg::kNZ, NU = Cfg::kNU, SU = Cfg::kUStages, SE = Cfg::kRing;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nchunks = (a.d + kChunkCols - 1) / kChunkCols;
  const int64_t ntiles = (a.n + kUmmaTile - 1) / kUmmaTile;

  const uint32_t smem_u = smem_u32(smem_raw), smem0 = (smem_u + 1023u) & ~1023u;
  const uint32_t z_base = smem0, u_ring = z_base + Cfg::kZBufs * Cfg::kZBytes, out_base = smem0 + Cfg::kOperandBytes;
  const uint32_t bars = out_base + Cfg::kOutBytes;
  auto z_full_bar = [&](int b) { return bars + b * 8; };
  auto z_empty_bar = [&](int b) { return bars + (2 + b) * 8; };
  auto u_full_bar = [&](int s) { return bars + (4 + s) * 8; };
  auto u_empty_bar = [&](int s) { return bars + (4 + SU + s) * 8; };
  auto d_full_bar = [&](int b) { return bars + (4 + 2 * SU + b) * 8; };
  auto d_empty_bar = [&](int b) { return bars + (4 + 2 * SU + 2 + b) * 8; };
  auto e_full_bar = [&](int s, int q) { return bars + (4 + 2 * SU + 4 + 4 * s + q) * 8; };
  auto e_empty_bar = [&](int s, int q) { return bars + (4 + 2 * SU + 4 + 4 * SE + 4 * s + q) * 8; };
  unsigned char *tail = smem_raw + (bars - smem_u) + Cfg::kBars * 8;
  volatile uint32_t *tmem_slot_ptr = reinterpret_cast<volatile uint32_t *>(tail);
  // [unit % kUnsafeSlots][operand warp]: U of the unit holds values its split does not
  volatile unsigned char *unit_flags = tail + 16;
  // [tile & 3][row]: magnitude class of the row of Z
  volatile unsigned char *row_class = unit_flags + Cfg::kUnsafeSlots * kSplitOperandWarps;

  if (a.k % 16 != 0) {   // the coordinates a K step reads past k
    for (uint32_t i = tid; i < Cfg::kOperandBytes / 16; i += kSplitExpandThreads) st_shared_v4(smem0 + i * 16, 0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  }
  if (tid == 0) {
    for (int b = 0; b < 2; ++b) {
      mbar_init(z_full_bar(b), kSplitOperandWarps);
      mbar_init(z_empty_bar(b), 1);
      mbar_init(d_full_bar(b), 1);
      mbar_init(d_empty_bar(b), kSplitEpilogueWarps);
    }
    for (int s = 0; s < SE; ++s)
      for (int q = 0; q < 4; ++q) {
        mbar_init(e_full_bar(s, q), 32);
        mbar_init(e_empty_bar(s, q), 1);
      }
    for (int s = 0; s < SU; ++s) {
      mbar_init(u_full_bar(s), kSplitOperandWarps);
      mbar_init(u_empty_bar(s), 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == kSplitMmaWarp) {
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
  const int64_t units = ntiles * nchunks;
  const int64_t u_lo = (units * blockIdx.x) / gridDim.x, u_hi = (units * (blockIdx.x + 1)) / gridDim.x;
  const T *U = static_cast<const T *>(a.U);
  // first unit of this CTA, and how many: the roles walk (tile, chunk) without dividing
  const int count_units = (int)(u_hi - u_lo);
  const int64_t tile_lo = u_lo / nchunks;
  const int chunk_lo = (int)(u_lo - tile_lo * nchunks);

  if (warp >= kSplitOperandWarp0 && warp < kSplitMmaWarp) {
    // ------------------------------------------------------------------------- operands
    // Lane = pair of coordinates (32, or 16 or 8 lanes per row where the rank leaves the others without
    // work), so the loads are coalesced and the swizzled stores hit all banks once.  The rows of a lane are
    // 8 or more apart, so its place in the swizzled rows never changes.
    const int ow = warp - kSplitOperandWarp0;
    const int lpr_log = KG == 2 || a.k > 32 ? 5 : (a.k > 16 ? 4 : 3), rpw = 32 >> lpr_log;
    const int row0 = ow * rpw + (lane >> lpr_log), pair = lane & ((1 << lpr_log) - 1);
    const int nit = kUmmaTile / (kSplitOperandWarps * rpw), row_step = kSplitOperandWarps * rpw;
    const uint32_t off0 = row0 * 128 + (((pair >> 2) ^ (row0 & 7)) << 4) + (pair & 3) * 4;
    const int ksteps16 = (a.k + 15) & ~15;   // coordinates that the MMAs read
    // rows first .. first + 127 of a matrix (the last one repeated), coordinates 64 kg ..: parts into smem
    auto move_tile = [&](auto np, auto batch, const auto *M, int64_t ld, int64_t first, int64_t rows, int kg, bool vec_m,
                         uint32_t base, uint32_t part_bytes, int class_slot, auto wait_free) {
      constexpr int NP = decltype(np)::value, B = decltype(batch)::value;   // B: rows in flight per lane
      using E = std::remove_const_t<std::remove_pointer_t<decltype(M)>>;
      const int j = kg * 64 + 2 * pair, valid = a.k - j;
      float largest = 0.f;
      bool tiny = false;                                 // a row of U that its split does not hold
      const bool inside = first + kUmmaTile <= rows;
      const E *col = M + (first + row0) * ld + j;        // read only where `inside`
      const int64_t step = (int64_t)row_step * ld;
#pragma unroll 1
      for (int b = 0; b < nit; b += B) {
        Pair<E> v[B];
        if (inside) {
          load_pairs<B, E>(v, [&](int i) { return col + i * step; }, valid, vec_m);
          col += B * step;
        } else {
          load_pairs<B, E>(v, [&](int i) { return M + min(first + row0 + (int64_t)(b + i) * row_step, rows - 1) * ld + j; }, valid, vec_m);
        }
        if (b == 0) wait_free();
        if (NZ == 3 && class_slot >= 0) {                // a row of Z: its lanes agree on its class
#pragma unroll
          for (int i = 0; i < B; ++i) {
            float m = valid > 0 ? pair_magnitude<E>(joined<E>(v[i])) : 0.f;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1)
              if (off < (1 << lpr_log)) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
            if (pair == 0) {
              volatile unsigned char *c = row_class + class_slot * kUmmaTile + row0 + (b + i) * row_step;
              const unsigned char cls = magnitude_class(m);
              *c = kg == 0 ? cls : max(cls, (unsigned char)*c);
            }
          }
        }
        if (NP == 3 && class_slot < 0) {
          float m[B];
          bool some = false;
#pragma unroll
          for (int i = 0; i < B; ++i) {
            m[i] = valid > 0 ? pair_magnitude<E>(joined<E>(v[i])) : 0.f;
            some = some || (m[i] != 0.f && m[i] < kSplitTinyU);
          }
          if (__any_sync(0xffffffffu, some)) {           // hardly ever: look at whole rows
#pragma unroll
            for (int i = 0; i < B; ++i) {
#pragma unroll
              for (int off = 16; off > 0; off >>= 1)
                if (off < (1 << lpr_log)) m[i] = fmaxf(m[i], __shfl_xor_sync(0xffffffffu, m[i], off));
              tiny = tiny || (m[i] != 0.f && m[i] < kSplitTinyU);
            }
          }
        }
        if (valid > 0) {
          const uint32_t dst = base + off0 + (uint32_t)b * row_step * 128;
#pragma unroll
          for (int i = 0; i < B; ++i) {
            const Pair<E> w = joined<E>(v[i]);
            if (Cfg::kLow) largest = fmaxf(largest, pair_magnitude<E>(w));
            uint32_t p[NP];
            split_pair<E, NP>(w, p);
#pragma unroll
            for (int s = 0; s < NP; ++s) st_shared_b32(dst + (uint32_t)i * row_step * 128 + s * part_bytes, p[s]);
          }
        } else if (KG == 2 && class_slot < 0 && j < ksteps16) {
          // A stage of U that held the first 64 coordinates of another chunk now holds the second: what the last
          // K step reads past k must be zero again, since 0 (of Z) times a stale infinity is no 0.
          const uint32_t dst = base + off0 + (uint32_t)b * row_step * 128;
#pragma unroll
          for (int i = 0; i < B; ++i)
#pragma unroll
            for (int s = 0; s < NP; ++s) st_shared_b32(dst + (uint32_t)i * row_step * 128 + s * part_bytes, 0);
        }
      }
      return tiny || largest >= kSplitHugeU;             // U only
    };
    using Eight = std::integral_constant<int, 8>;
    using Four = std::integral_constant<int, 4>;
    int64_t tile = tile_lo;
    int chunk = chunk_lo, tcount = 0, slot = 0;
    uint32_t parity = 1;
    for (int unit = 0; unit < count_units; ++unit) {
      if (unit == 0 || chunk == 0) {
        const int zb = tcount % Cfg::kZBufs;
        const uint32_t z_parity = (uint32_t)(((tcount / Cfg::kZBufs) & 1) ^ 1);
        for (int kg = 0; kg < KG; ++kg) {
          auto z_tile = [&](auto batch) {
            move_tile(std::integral_constant<int, NZ>{}, batch, static_cast<const TZ *>(a.zin), a.ldzin, tile * kUmmaTile, a.n, kg,
                      a.vec_z != 0, z_base + zb * Cfg::kZBytes + kg * kSplitTileBytes, KG * kSplitTileBytes, tcount & 3, [&]() {
                        if (kg == 0 && !dead && !mbar_wait(z_empty_bar(zb), z_parity)) timed_out();
                      });
          };
          if (nit >= 8) z_tile(Eight{});
          else z_tile(Four{});
        }
        ++tcount;
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(z_full_bar(zb));
      }
      const int col0 = chunk * kChunkCols;
      bool flagged = false;
      for (int kg = 0; kg < KG; ++kg) {
        auto u_tile = [&](auto batch) {
          return move_tile(std::integral_constant<int, NU>{}, batch, U, a.ldu, (int64_t)col0, (int64_t)a.d, kg, a.vec_u != 0,
                           u_ring + (uint32_t)slot * Cfg::kUStageBytes, kSplitTileBytes, -1, [&]() {
                             if (!dead && !mbar_wait(u_empty_bar(slot), parity)) timed_out();
                           });
        };
        const bool bad = nit >= 8 ? u_tile(Eight{}) : u_tile(Four{});
        if (Cfg::kLow) {   // the slot's readers were eight units ago, and the ring holds fewer
          flagged = flagged || __any_sync(0xffffffffu, bad);
          if (lane == 0) unit_flags[(unit % Cfg::kUnsafeSlots) * kSplitOperandWarps + ow] = flagged ? 1 : 0;
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(u_full_bar(slot));
        if (++slot == SU) {
          slot = 0;
          parity ^= 1u;
        }
      }
      if (++chunk == nchunks) {
        chunk = 0;
        ++tile;
      }
    }
  } else if (warp == kSplitMmaWarp) {
    // ------------------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      constexpr uint32_t idesc = umma_idesc_kk(kChunkCols);
      constexpr uint32_t kZPart = (uint32_t)(KG * kSplitTileBytes) >> 4, kUPart = (uint32_t)kSplitTileBytes >> 4;
      const uint64_t kdesc = umma_desc(0, 16, 1024, 2);
      int chunk = chunk_lo, tcount = -1, slot = 0;
      uint32_t parity = 0;
      for (int unit = 0; unit < count_units; ++unit) {
        if (unit == 0 || chunk == 0) {
          ++tcount;
          if (!dead && !mbar_wait(z_full_bar(tcount % Cfg::kZBufs), (uint32_t)((tcount / Cfg::kZBufs) & 1))) timed_out();
        }
        const int zb = tcount % Cfg::kZBufs, db = unit & 1;
        if (!dead && !mbar_wait(d_empty_bar(db), (uint32_t)(((unit >> 1) & 1) ^ 1))) timed_out();
        const uint32_t hi = tmem_base + (uint32_t)db * Cfg::kDCols, lo = hi + kChunkCols;
#pragma unroll
        for (int kg = 0; kg < KG; ++kg) {
          if (!dead && !mbar_wait(u_full_bar(slot), parity)) timed_out();
          asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
          const uint64_t zd = kdesc + umma_desc_addr(z_base + zb * Cfg::kZBytes + kg * kSplitTileBytes);
          const uint64_t ud = kdesc + umma_desc_addr(u_ring + (uint32_t)slot * Cfg::kUStageBytes);
          const int ksteps = (min(a.k - kg * 64, 64) + 15) / 16;
          for (int j = 0; j < ksteps; ++j) {
            const uint64_t z = zd + j * 2, u = ud + j * 2;
            const uint32_t more = kg > 0 || j > 0 ? 1u : 0u;
            umma_bf16(hi, z, u, idesc, more);
            if (NZ == 3) {
              umma_bf16(lo, z + kZPart, u, idesc, more);
              umma_bf16(lo, z + 2 * kZPart, u, idesc, 1u);
            }
            if (NU == 3) {
              umma_bf16(lo, z, u + kUPart, idesc, NZ == 3 ? 1u : more);
              umma_bf16(lo, z, u + 2 * kUPart, idesc, 1u);
            }
            if (NZ == 3 && NU == 3) umma_bf16(lo, z + kZPart, u + kUPart, idesc, 1u);
          }
          umma_commit(u_empty_bar(slot));
          if (++slot == SU) {
            slot = 0;
            parity ^= 1u;
          }
        }
        umma_commit(d_full_bar(db));
        if (++chunk == nchunks) chunk = 0;
        if (unit + 1 == count_units || chunk == 0) umma_commit(z_empty_bar(zb));
      }
    }
    __syncwarp();
  } else if (warp >= kSplitEpilogueWarps) {
    // ------------------------------------------------------------------------- row gather (E, P)
    // 8 lanes copy 128 bytes of one row; the stage's quarter is full when every thread's copies have landed.
    if (NSLOT > 0) {
      const int gw = warp - kSplitEpilogueWarps, piece = lane & 7, sub = lane >> 3;   // rows 32 gw .. +31
      constexpr int kUnitElems = 16 / (int)sizeof(T);
      const bool vec = a.vec_rows != 0;
      const T *E = a.has_e ? static_cast<const T *>(a.shift.E) : nullptr, *P = a.has_p ? static_cast<const T *>(a.shift.P) : nullptr;
      const T *src[NSLOT > 0 ? NSLOT : 1][8];
      uint32_t dst[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int r = gw * 32 + i * 4 + sub;
        dst[i] = r * 128 + ((piece ^ (r & 7)) << 4);
      }
      int64_t tile = tile_lo;
      int chunk = chunk_lo, slot = 0;
      uint32_t parity = 1;
      for (int unit = 0; unit < count_units; ++unit) {
        if (unit == 0 || chunk == 0) {
          const T *none = vec ? reinterpret_cast<const T *>(g_zero_row) : nullptr;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int64_t t = tile * kUmmaTile + gw * 32 + i * 4 + sub;
            const int64_t er = t < a.n && E != nullptr ? embedding_row(a.shift, t) : -1;
            const int64_t pr = t < a.n && P != nullptr ? position_row(a.shift, t) : -1;
            const T *erow = er >= 0 ? E + er * a.shift.lde : none, *prow = pr >= 0 ? P + pr * a.shift.ldp : none;
            src[0][i] = NSLOT == 2 || E != nullptr ? erow : prow;
            if (NSLOT == 2) src[NSLOT - 1][i] = prow;
          }
        }
        // the lines of the next unit into L2: the ring alone does not hold enough in flight for HBM latency
        if (vec && piece < Cfg::kPieces && (chunk + 1) * kChunkCols + piece * Cfg::kPieceCols < a.d) {
#pragma unroll
          for (int o = 0; o < NSLOT; ++o)
#pragma unroll
            for (int i = 0; i < 8; ++i) prefetch_l2(src[o][i] + (chunk + 1) * kChunkCols + piece * Cfg::kPieceCols);
        }
#pragma unroll 1
        for (int g = 0; g < Cfg::kPieces; ++g) {
          const int c = chunk * kChunkCols + g * Cfg::kPieceCols + piece * kUnitElems;
          const bool ok = c < a.d;
#pragma unroll
          for (int o = 0; o < NSLOT; ++o) {
            if (!dead && !mbar_wait(e_empty_bar(slot, gw), parity)) timed_out();
            const uint32_t base = out_base + (uint32_t)slot * kSplitTileBytes;
            if (vec) {
#pragma unroll
              for (int i = 0; i < 8; ++i) cp_async16_if(base + dst[i], src[o][i] + (ok ? c : 0), ok);
              asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];\n" ::"r"(e_full_bar(slot, gw)) : "memory");
            } else {
#pragma unroll 1
              for (int i = 0; i < 8; ++i) {
                const T *row = nullptr;
                uint32_t to = 0;
#pragma unroll
                for (int h = 0; h < 8; ++h)
                  if (h == i) {
                    row = src[o][h];
                    to = dst[h];
                  }
                const uint4 v = load_row_piece<T>(row, c, a.d);
                st_shared_v4(base + to, v.x, v.y, v.z, v.w);
              }
              mbar_arrive(e_full_bar(slot, gw));
            }
            if (++slot == SE) {
              slot = 0;
              parity ^= 1u;
            }
          }
        }
        if (++chunk == nchunks) {
          chunk = 0;
          ++tile;
        }
      }
      cp_async_commit();
      cp_async_wait<0>();
    }
  } else {
    // ------------------------------------------------------------------------- epilogue
    const int quarter = warp & 3, half = warp >> 2;        // TMEM lanes 32 quarter .. +31; half of every piece
    constexpr int kHalfCols = Cfg::kPieceCols / 2, kUnitElems = 16 / (int)sizeof(T);
    const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16);
    const uint64_t stream_out = l2_policy_evict_first();   // the output is written once and not read here
    auto meet = [&]() { asm volatile("bar.sync %0, 64;\n" ::"r"(1 + quarter) : "memory"); };   // the quarter's two warps
    int64_t tile = tile_lo;
    int chunk = chunk_lo, tcount = 0, slot = 0;
    uint32_t parity = 0;
    int held = -1;                                         // stage whose store may still be reading it
    for (int unit = 0; unit < count_units; ++unit) {
      const int db = unit & 1, col0 = chunk * kChunkCols;
      const int64_t row0 = tile * kUmmaTile + quarter * 32, t = row0 + lane;
      if (!dead && !mbar_wait(d_full_bar(db), (uint32_t)((unit >> 1) & 1))) timed_out();
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      bool bad = false;                                    // this row by plain FMAs
      if (Cfg::kLow) {
        const unsigned char cls = NZ == 3 ? row_class[(tcount & 3) * kUmmaTile + quarter * 32 + lane] : 2;
        bad = t < a.n && (cls == 1 || cls == 3 ||
                          reinterpret_cast<volatile unsigned long long *>(tail + 16)[unit % Cfg::kUnsafeSlots] != 0);
      }
#pragma unroll 1
      for (int g = 0; g < Cfg::kPieces; ++g) {
        // the piece's stage: full of E or P rows, or (no tables) free; and the P stage behind an E stage
        const int eslot = slot;
        if (NSLOT > 0) {
          if (!dead && !mbar_wait(e_full_bar(slot, quarter), parity)) timed_out();
        } else {
          if (!dead && !mbar_wait(e_empty_bar(slot, quarter), parity ^ 1u)) timed_out();
        }
        if (++slot == SE) {
          slot = 0;
          parity ^= 1u;
        }
        const int pslot = slot;
        if (NSLOT == 2) {
          if (!dead && !mbar_wait(e_full_bar(slot, quarter), parity)) timed_out();
          if (++slot == SE) {
            slot = 0;
            parity ^= 1u;
          }
        }
        const uint32_t out = out_base + (uint32_t)eslot * kSplitTileBytes + (uint32_t)quarter * 4096;   // 32 rows x 128 bytes
        const uint32_t orow = out + lane * 128;
        const uint32_t prow = out_base + (uint32_t)pslot * kSplitTileBytes + (uint32_t)quarter * 4096 + lane * 128;
        const int pcol = g * Cfg::kPieceCols + half * kHalfCols;   // this warp's columns of the unit
#pragma unroll
        for (int h = 0; h < kHalfCols / 16; ++h) {         // 16 columns at a time
          const uint32_t taddr = lane_addr + (uint32_t)db * Cfg::kDCols + pcol + h * 16;
          uint32_t v[16];
          tmem_ld16(taddr, v);
          if (Cfg::kLow) {
            uint32_t w[16];
            tmem_ld16(taddr + kChunkCols, w);
            asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
            for (int e = 0; e < 16; ++e) v[e] = __float_as_uint(__uint_as_float(v[e]) + __uint_as_float(w[e]));
          } else {
            asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
          }
          if (Cfg::kLow && bad) {
            const TZ *z = static_cast<const TZ *>(a.zin) + t * a.ldzin;
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              const int c = col0 + pcol + h * 16 + e;
              if (c >= a.d) continue;
              float acc = 0.f;
#pragma unroll 1
              for (int j = 0; j < a.k; ++j) acc = fmaf(to_f32(z[j]), to_f32(U[(int64_t)c * a.ldu + j]), acc);
              v[e] = __float_as_uint(acc);
            }
          }
#pragma unroll
          for (int c = 0; c < 16 / kUnitElems; ++c) {      // 16 bytes of the row
            const uint32_t off = (((half * 4 + h * (16 / kUnitElems) + c) ^ (lane & 7)) << 4);
            float f[kUnitElems];
#pragma unroll
            for (int e = 0; e < kUnitElems; ++e) f[e] = __uint_as_float(v[c * kUnitElems + e]);
            if (NSLOT > 0) {
              float e0[kUnitElems];
              widen_piece<T>(ld_shared_v4(orow + off), e0);
#pragma unroll
              for (int e = 0; e < kUnitElems; ++e) f[e] += e0[e];
            }
            if (NSLOT == 2) {
              float p0[kUnitElems];
              widen_piece<T>(ld_shared_v4(prow + off), p0);
#pragma unroll
              for (int e = 0; e < kUnitElems; ++e) f[e] += p0[e];
            }
            if constexpr (sizeof(T) == 4)
              st_shared_v4(orow + off, __float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]), __float_as_uint(f[3]));
            else
              st_shared_v4(orow + off, pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]), pack_bf16(f[4], f[5]), pack_bf16(f[6], f[7]));
          }
        }
        if (g == Cfg::kPieces - 1) {                       // the accumulator has been read
          asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(d_empty_bar(db));
        }
        const int col = col0 + g * Cfg::kPieceCols;
        if (a.tma_out) {
          asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
          meet();
          if (half == 0 && lane == 0) {
            if (NSLOT == 2) mbar_arrive(e_empty_bar(pslot, quarter));
            if (row0 < a.n && col < a.d) tma_store_2d_hint(&out_map, out, col, (int)row0, stream_out);
            bulk_commit();
            // hand back the stage of the store before this one, and this one's too where the ring is short
            if (Cfg::kHold) {
              bulk_wait_read<1>();
              if (held >= 0) mbar_arrive(e_empty_bar(held, quarter));
              held = eslot;
            } else {
              bulk_wait_read<0>();
              mbar_arrive(e_empty_bar(eslot, quarter));
            }
          }
        } else {
          // any alignment: row by row, 128 bytes of it by one of the two warps
          meet();
#pragma unroll 1
          for (int r = half; r < 32; r += 2) {
            if (row0 + r >= a.n) break;
            uint32_t w;
            asm volatile("ld.shared.b32 %0, [%1];\n"
                         : "=r"(w) : "r"(out + r * 128 + (((lane >> 2) ^ (r & 7)) << 4) + (lane & 3) * 4) : "memory");
            T *o = static_cast<T *>(a.dst) + (row0 + r) * a.lddst;
            if constexpr (sizeof(T) == 4) {
              if (col + lane < a.d) o[col + lane] = __uint_as_float(w);
            } else {
              const int c = col + 2 * lane;
              if (c < a.d) o[c] = __ushort_as_bfloat16((unsigned short)w);
              if (c + 1 < a.d) o[c + 1] = __ushort_as_bfloat16((unsigned short)(w >> 16));
            }
          }
          meet();
          if (half == 0 && lane == 0) {
            mbar_arrive(e_empty_bar(eslot, quarter));
            if (NSLOT == 2) mbar_arrive(e_empty_bar(pslot, quarter));
          }
        }
      }
      if (++chunk == nchunks) {
        chunk = 0;
        ++tile;
        ++tcount;
      }
    }
    if (half == 0 && lane == 0) bulk_wait<0>();
  }

  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == kSplitMmaWarp) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"(Cfg::kTmemCols)
                 : "memory");
  }
}

}  // namespace ssn
