// Split-operand tcgen05 expansion of the SSN codec:
//     Xhat = Z U^T [+ E[ids]] [+ P[pos]]
// for fp32 storage, for fp32 wire rows, and for the bf16 calls the TMA expansion does not take: leading
// dimensions or addresses off the 16-byte grid, positions per token or of any sequence length.
//
// A unit is 128 tokens x 128 output columns; the units are dealt to the CTAs in contiguous ranges.
//
//   warps 0-15   output: TMEM -> a staging tile in shared memory (half a unit, 64 columns, at a time)
//                -> rows again, 16 lanes per row, so that the E and P rows are read and the output is
//                written in whole sectors whatever their alignment; the row pieces of the next
//                half are in flight while this one is staged, and their lines two units on are
//                requested into L2 (the loads in registers alone do not cover HBM latency).
//   warps 16-23  operands: Z once per tile and 128 rows of U per unit, loaded pair by pair of elements, split
//                into bf16 parts (codec_split.cuh) and written as swizzled K-major tiles of 64 coordinates; a
//                ring of such U tiles runs ahead of the MMAs.  One warp per scheduler could not keep up
//                with the splitting.
//   warp 24      one thread issues the MMAs (M = 128, N = 128): the leading product into one accumulator,
//                the small ones (hm, mh, mm, hl, lh) into a second, two sets of both.  A warp of its own, since
//                every MMA blocks its thread for about 80 clocks.
//
// Coordinates past k are zeroed once, rows past n or d repeat the last one and are never stored.
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
  int32_t vec_out;             // four elements of the output and of the E and P rows may be moved at a time
  ShiftTables shift;
};

constexpr int kSplitOutWarps = 16, kSplitOperandWarps = 8;
constexpr int kSplitOutThreads = 32 * kSplitOutWarps;
constexpr int kSplitExpandThreads = 32 * (kSplitOutWarps + kSplitOperandWarps + 1);
constexpr int kSplitTileBytes = kUmmaTile * 128;     // one part of [128 rows x 64 coordinates]
constexpr int kSplitHalf = 64;                       // output columns staged at a time

// TZ: type of the coordinates (float for fp32 storage and wire rows), T: storage type, KG: groups of 64 coordinates
template <typename T, typename TZ, int KG, int NSLOT>
struct SplitExpandConfig {
  static constexpr int kNZ = sizeof(TZ) == 4 ? 3 : 1, kNU = sizeof(T) == 4 ? 3 : 1;
  static constexpr int kZBytes = kNZ * KG * kSplitTileBytes;
  static constexpr int kZBufs = kNZ == 1 ? 2 : 1;
  static constexpr int kUStageBytes = kNU * kSplitTileBytes;
  static constexpr int kUStages = kNU == 3 ? 2 : 3;
  static constexpr int kHalfBytes = kUmmaTile * kSplitHalf * 4;
  static constexpr int kStagings = kNU == 3 && KG == 2 ? 1 : 2;
  static constexpr bool kLow = kNZ > 1 || kNU > 1;          // a second accumulator for the small products
  static constexpr int kDCols = (kLow ? 2 : 1) * kChunkCols;
  static constexpr int kTmemCols = 2 * kDCols;
  static constexpr int kOperandBytes = kZBufs * kZBytes + kUStages * kUStageBytes;
  static constexpr int kBars = 4 + 2 * kUStages + 4;
  static constexpr int kUnsafeSlots = 8;                    // units whose U values may be flagged at a time
  static constexpr int kTailBytes = kBars * 8 + 16 + kUnsafeSlots * kSplitOperandWarps;
  static constexpr int kSmemBytes = 1024 + kOperandBytes + kStagings * kHalfBytes + kTailBytes;
  static_assert(kSmemBytes <= 227 * 1024, "the operands do not fit in shared memory");
};

// Four elements of a row from column c on (zeros past column d and for a missing row), as stored.
template <typename T> struct RowPiece4 { uint32_t w[sizeof(T)]; };
template <typename T>
__device__ __forceinline__ RowPiece4<T> load_row4(const T *row, int c, int d, bool vec) {
  RowPiece4<T> f;
  const bool ok = row != nullptr;
  if constexpr (sizeof(T) == 4) {
    if (vec) {   // d is a multiple of 4 then
      const uint4 v = load_global_v4_if(row + c, ok && c < d);
      f.w[0] = v.x; f.w[1] = v.y; f.w[2] = v.z; f.w[3] = v.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) f.w[e] = load_global_b32_if(row + c + e, ok && c + e < d);
    }
  } else {
    if (vec) {
      const uint2 v = load_global_v2_if(row + c, ok && c < d);
      f.w[0] = v.x; f.w[1] = v.y;
    } else {
#pragma unroll
      for (int e = 0; e < 2; ++e)
        f.w[e] = load_global_b16_if(row + c + 2 * e, ok && c + 2 * e < d) |
                 load_global_b16_if(row + c + 2 * e + 1, ok && c + 2 * e + 1 < d) << 16;
    }
  }
  return f;
}
template <typename T>
__device__ __forceinline__ float piece_element(const RowPiece4<T> &f, int e) {
  if constexpr (sizeof(T) == 4) return __uint_as_float(f.w[e]);
  else return __uint_as_float(e & 1 ? f.w[e >> 1] & 0xFFFF0000u : f.w[e >> 1] << 16);
}

template <typename T, typename TZ, int KG, int NSLOT>
__global__ void __launch_bounds__(kSplitExpandThreads, 1) codec_split_expand_kernel(const SplitExpandArgs a) {
  using Cfg = SplitExpandConfig<T, TZ, KG, NSLOT>;
  constexpr int NZ = Cfg::kNZ, NU = Cfg::kNU, SU = Cfg::kUStages;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nchunks = (a.d + kChunkCols - 1) / kChunkCols;
  const int64_t ntiles = (a.n + kUmmaTile - 1) / kUmmaTile;

  const uint32_t smem_u = smem_u32(smem_raw), smem0 = (smem_u + 1023u) & ~1023u;
  const uint32_t z_base = smem0, u_ring = z_base + Cfg::kZBufs * Cfg::kZBytes, staging = smem0 + Cfg::kOperandBytes;
  const uint32_t bars = staging + Cfg::kStagings * Cfg::kHalfBytes;
  auto z_full_bar = [&](int b) { return bars + b * 8; };
  auto z_empty_bar = [&](int b) { return bars + (2 + b) * 8; };
  auto u_full_bar = [&](int s) { return bars + (4 + s) * 8; };
  auto u_empty_bar = [&](int s) { return bars + (4 + SU + s) * 8; };
  auto d_full_bar = [&](int b) { return bars + (4 + 2 * SU + b) * 8; };
  auto d_empty_bar = [&](int b) { return bars + (4 + 2 * SU + 2 + b) * 8; };
  unsigned char *tail = smem_raw + (bars - smem_u) + Cfg::kBars * 8;
  volatile uint32_t *tmem_slot_ptr = reinterpret_cast<volatile uint32_t *>(tail);
  // [unit % kUnsafeSlots][operand warp]: U of the unit holds values its split does not
  volatile unsigned char *unit_flags = tail + 16;

  if (a.k % 16 != 0) {   // the coordinates a K step reads past k
    for (uint32_t i = tid; i < Cfg::kOperandBytes / 16; i += kSplitExpandThreads) st_shared_v4(smem0 + i * 16, 0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  }
  if (tid == 0) {
    for (int b = 0; b < 2; ++b) {
      mbar_init(z_full_bar(b), kSplitOperandWarps);
      mbar_init(z_empty_bar(b), 1);
      mbar_init(d_full_bar(b), 1);
      mbar_init(d_empty_bar(b), kSplitOutWarps);
    }
    for (int s = 0; s < SU; ++s) {
      mbar_init(u_full_bar(s), kSplitOperandWarps);
      mbar_init(u_empty_bar(s), 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == kSplitOutWarps + kSplitOperandWarps) {
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

  if (warp >= kSplitOutWarps && warp < kSplitOutWarps + kSplitOperandWarps) {
    // ------------------------------------------------------------------------- operands
    // Lane = pair of coordinates (32, or 16 or 8 lanes per row where the rank leaves the others without
    // work), so the loads are coalesced and the swizzled stores hit all banks once.  The rows of a lane are
    // 8 or more apart, so its place in the swizzled rows never changes.
    const int ow = warp - kSplitOutWarps;
    const int lpr_log = KG == 2 || a.k > 32 ? 5 : (a.k > 16 ? 4 : 3), rpw = 32 >> lpr_log;
    const int row0 = ow * rpw + (lane >> lpr_log), pair = lane & ((1 << lpr_log) - 1);
    const int nit = kUmmaTile / (kSplitOperandWarps * rpw), row_step = kSplitOperandWarps * rpw;
    const uint32_t off0 = row0 * 128 + (((pair >> 2) ^ (row0 & 7)) << 4) + (pair & 3) * 4;
    // rows first .. first + 127 of a matrix (the last one repeated), coordinates 64 kg ..: parts into smem
    auto move_tile = [&](auto np, auto batch, const auto *M, int64_t ld, int64_t first, int64_t rows, int kg, bool vec_m,
                         uint32_t base, uint32_t part_bytes, auto wait_free) {
      constexpr int NP = decltype(np)::value, B = decltype(batch)::value;   // B: rows in flight per lane
      using E = std::remove_const_t<std::remove_pointer_t<decltype(M)>>;
      const int j = kg * 64 + 2 * pair, valid = a.k - j;
      float largest = 0.f;
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
        }
      }
      return largest;
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
                      a.vec_z != 0, z_base + zb * Cfg::kZBytes + kg * kSplitTileBytes, KG * kSplitTileBytes, [&]() {
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
      bool huge = false;
      for (int kg = 0; kg < KG; ++kg) {
        auto u_tile = [&](auto batch) {
          return move_tile(std::integral_constant<int, NU>{}, batch, U, a.ldu, (int64_t)col0, (int64_t)a.d, kg, a.vec_u != 0,
                           u_ring + (uint32_t)slot * Cfg::kUStageBytes, kSplitTileBytes, [&]() {
                             if (!dead && !mbar_wait(u_empty_bar(slot), parity)) timed_out();
                           });
        };
        const float largest = nit >= 8 ? u_tile(Eight{}) : u_tile(Four{});
        if (Cfg::kLow) {   // the slot's readers were eight units ago, and the ring holds fewer
          huge = huge || __any_sync(0xffffffffu, largest >= kSplitHuge);
          if (lane == 0) unit_flags[(unit % Cfg::kUnsafeSlots) * kSplitOperandWarps + ow] = huge ? 1 : 0;
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
  } else if (warp == kSplitOutWarps + kSplitOperandWarps) {
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
  } else {
    // ------------------------------------------------------------------------- output
    const int quarter = warp & 3, cpart = warp >> 2;       // TMEM lanes; 16 of the 64 columns of a half
    const int trow = quarter * 32 + lane;                  // row this thread stages
    const int sub = lane >> 4, c4 = (lane & 15) * 4;       // rows 2 i + sub of the warp's eight, columns c4 .. +3
    const bool vec = a.vec_out != 0;
    int64_t tile = tile_lo;
    int chunk = chunk_lo;
    int32_t er = -1, pr = -1;                              // lanes 0-7: table rows of the warp's rows
    uint32_t unsafe_rows = 0;
    int live_rows = 0;                                     // of the warp's eight, those before row n
    T *out0 = nullptr;                                     // column c4 of row `sub` of the warp's eight
    RowPiece4<T> in[NSLOT > 0 ? NSLOT : 1][4];
    const T *E = a.has_e ? static_cast<const T *>(a.shift.E) : nullptr, *P = a.has_p ? static_cast<const T *>(a.shift.P) : nullptr;
    auto row_of = [&](bool want_e, int i) -> const T * {   // E or P row of the warp's row i
      const int32_t r = __shfl_sync(0xffffffffu, want_e ? er : pr, i);
      return r < 0 ? nullptr : (want_e ? E + (int64_t)r * a.shift.lde : P + (int64_t)r * a.shift.ldp);
    };
    auto issue = [&](int col) {                            // E and P pieces of the warp's rows
#pragma unroll
      for (int i = 0; i < (NSLOT > 0 ? 4 : 0); ++i) {
        in[0][i] = load_row4<T>(row_of(NSLOT == 2 || a.has_e, 2 * i + sub), col + c4, a.d, vec);
        if (NSLOT == 2) in[NSLOT - 1][i] = load_row4<T>(row_of(false, 2 * i + sub), col + c4, a.d, vec);
      }
    };
    auto prefetch = [&](int col) {                         // the lines of 128 columns of the warp's rows
      constexpr int kLines = kChunkCols * (int)sizeof(T) / 128, kLineElems = 128 / (int)sizeof(T);
      if (NSLOT == 0 || col >= a.d) return;
      const int r = lane / kLines, c = col + (lane % kLines) * kLineElems;   // bf16: the upper lanes have no row
#pragma unroll
      for (int o = 0; o < NSLOT; ++o) {
        const T *row = row_of(NSLOT == 2 ? o == 0 : a.has_e != 0, r & 7);
        if (r < 8 && row != nullptr && c < a.d) prefetch_l2(row + c);
      }
    };
    auto enter_tile = [&](int64_t ut) {
      const int64_t t0 = ut * kUmmaTile + warp * 8, t = t0 + lane;
      live_rows = (int)max((int64_t)0, min((int64_t)8, a.n - t0));
      out0 = static_cast<T *>(a.dst) + (t0 + sub) * a.lddst + c4;
      er = pr = -1;
      if (NSLOT > 0 && lane < live_rows) {
        if (a.has_e) er = (int32_t)embedding_row(a.shift, t);
        if (a.has_p) pr = (int32_t)position_row(a.shift, t);
      }
      if (NZ == 3) {                                       // rows whose split does not hold
        unsafe_rows = 0;
        for (int r = 0; r < live_rows; ++r) {
          const TZ *z = static_cast<const TZ *>(a.zin) + (t0 + r) * a.ldzin;
          float m = 0.f;
          for (int j = lane; j < a.k; j += 32) m = fmaxf(m, fabsf(to_f32(z[j])));
          m = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m)));   // floats >= 0 order like their bits
          if (split_unsafe(m)) unsafe_rows |= 1u << r;
        }
      }
    };
    if (count_units > 0) {
      enter_tile(tile);
      issue(chunk * kChunkCols);
      prefetch((chunk + 1) * kChunkCols);
    }
    for (int unit = 0; unit < count_units; ++unit) {
      const int col0 = chunk * kChunkCols, db = unit & 1;
      if (!dead && !mbar_wait(d_full_bar(db), (uint32_t)((unit >> 1) & 1))) timed_out();
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      uint32_t bad = 0;
      if (Cfg::kLow) {
        bad = unsafe_rows;
        if (reinterpret_cast<volatile unsigned long long *>(tail + 16)[unit % Cfg::kUnsafeSlots] != 0) bad = 0xFFu;
      }
      prefetch(col0 + 2 * kChunkCols);
#pragma unroll
      for (int g = 0; g < kChunkCols / kSplitHalf; ++g) {
        uint32_t v[2][8];
        const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)db * Cfg::kDCols + g * kSplitHalf + cpart * 16;
        tmem_ld8(taddr, v[0]);
        tmem_ld8(taddr + 8, v[1]);
        if (Cfg::kLow) {
          uint32_t w[2][8];
          tmem_ld8(taddr + kChunkCols, w[0]);
          tmem_ld8(taddr + kChunkCols + 8, w[1]);
          asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int e = 0; e < 8; ++e) v[h][e] = __float_as_uint(__uint_as_float(v[h][e]) + __uint_as_float(w[h][e]));
        } else {
          asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
        }
        if (g == kChunkCols / kSplitHalf - 1) {
          asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(d_empty_bar(db));
        }
        // staging row: 64 floats, 16-byte units XORed with the row so that neither side conflicts
        const uint32_t stage = staging + (Cfg::kStagings == 2 ? g : 0) * Cfg::kHalfBytes;
        if (Cfg::kStagings == 1) asm volatile("bar.sync 1, %0;\n" ::"n"(kSplitOutThreads) : "memory");   // read by everyone
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const uint32_t *w = &v[h >> 1][(h & 1) * 4];
          st_shared_v4(stage + trow * 256 + (((cpart * 4 + h) ^ (trow & 15)) << 4), w[0], w[1], w[2], w[3]);
        }
        asm volatile("bar.sync 1, %0;\n" ::"n"(kSplitOutThreads) : "memory");
        float o[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = warp * 8 + 2 * i + sub;
          const uint4 w = ld_shared_v4(stage + r * 256 + (((lane & 15) ^ (r & 15)) << 4));
          o[i][0] = __uint_as_float(w.x); o[i][1] = __uint_as_float(w.y);
          o[i][2] = __uint_as_float(w.z); o[i][3] = __uint_as_float(w.w);
        }
        const int col = col0 + g * kSplitHalf;
        if (Cfg::kLow && bad != 0) {                       // plain FMAs for the flagged rows
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if (!(bad >> (2 * i + sub) & 1) || 2 * i + sub >= live_rows) continue;
            const TZ *z = static_cast<const TZ *>(a.zin) + (tile * kUmmaTile + warp * 8 + 2 * i + sub) * a.ldzin;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int c = col + c4 + e;
              if (c >= a.d) continue;
              float acc = 0.f;
#pragma unroll 1
              for (int j = 0; j < a.k; ++j) acc = fmaf(to_f32(z[j]), to_f32(U[(int64_t)c * a.ldu + j]), acc);
              o[i][e] = acc;
            }
          }
        }
        if (NSLOT > 0) {
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              o[i][e] += piece_element<T>(in[0][i], e);
              if (NSLOT == 2) o[i][e] += piece_element<T>(in[NSLOT - 1][i], e);
            }
        }
        T *out = out0 + col;
        const int live = live_rows, cols = a.d - (col + c4);
        if (g == 0) {
          issue(col + kSplitHalf);
        } else {
          if (++chunk == nchunks) {
            chunk = 0;
            ++tile;
            if (unit + 1 < count_units) {
              enter_tile(tile);
              prefetch(kChunkCols);
            }
          }
          if (unit + 1 < count_units) issue(chunk * kChunkCols);
        }
        if (vec && live == 8) {                            // d is a multiple of 4
          if (cols > 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              if constexpr (sizeof(T) == 4)
                *reinterpret_cast<float4 *>(out + 2 * i * a.lddst) = make_float4(o[i][0], o[i][1], o[i][2], o[i][3]);
              else
                *reinterpret_cast<uint2 *>(out + 2 * i * a.lddst) = make_uint2(pack_bf16(o[i][0], o[i][1]), pack_bf16(o[i][2], o[i][3]));
            }
          }
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if (2 * i + sub >= live) continue;
#pragma unroll
            for (int e = 0; e < 4; ++e)
              if (e < cols) out[2 * i * a.lddst + e] = from_f32<T>(o[i][e]);
          }
        }
      }
    }
  }

  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == kSplitOutWarps + kSplitOperandWarps) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"(Cfg::kTmemCols)
                 : "memory");
  }
}

}  // namespace ssn
