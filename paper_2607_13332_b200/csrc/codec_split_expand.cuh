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
//                half are in flight while this one is staged.
//   warps 16-19  operands: Z once per tile and 128 rows of U per unit, loaded element pair by element
//                pair, split into bf16 parts (codec_split.cuh) and written as swizzled K-major tiles of 64
//                coordinates; a ring of such U tiles runs ahead of the MMAs.
//   warp 20      one thread issues the MMAs (M = 128, N = 128): the leading product into one accumulator,
//                the small ones (hm, mh, mm, hl, lh) into a second, two sets of both.
#pragma once

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

constexpr int kSplitOutWarps = 16, kSplitOperandWarps = 4;   // 21 warps: 80 registers a thread
constexpr int kSplitOutThreads = 32 * kSplitOutWarps;
constexpr int kSplitExpandThreads = 32 * (kSplitOutWarps + kSplitOperandWarps + 1);
constexpr int kSplitTileBytes = kUmmaTile * 128;     // one part of [128 rows x 64 coordinates]
constexpr int kSplitHalf = 64;                       // output columns staged at a time

// TZ: type of the coordinates (float for fp32 storage and wire rows), T: storage type, KG: groups of 64 coordinates
template <typename T, typename TZ, int KG, int NSLOT>
struct SplitExpandConfig {
  static constexpr int kNZ = sizeof(TZ) == 4 ? 3 : 1, kNU = sizeof(T) == 4 ? 3 : 1;
  static constexpr int kZBytes = kNZ * KG * kSplitTileBytes;
  static constexpr int kUStageBytes = kNU * kSplitTileBytes;
  static constexpr int kUStages = kNU == 3 ? 2 : 3;
  static constexpr int kHalfBytes = kUmmaTile * kSplitHalf * 4;
  static constexpr int kStagings = kNU == 3 && KG == 2 ? 1 : 2;
  static constexpr bool kLow = kNZ > 1 || kNU > 1;          // a second accumulator for the small products
  static constexpr int kDCols = (kLow ? 2 : 1) * kChunkCols;
  static constexpr int kTmemCols = 2 * kDCols;
  static constexpr int kBars = 2 + 2 * kUStages + 4;
  static constexpr int kUnsafeSlots = 8;                    // units whose U values may be flagged at a time
  static constexpr int kTailBytes = kBars * 8 + 16 + kUnsafeSlots * 4;
  static constexpr int kSmemBytes = 1024 + kZBytes + kUStages * kUStageBytes + kStagings * kHalfBytes + kTailBytes;
  static_assert(kSmemBytes <= 227 * 1024, "the operands do not fit in shared memory");
};

// Four elements of a row from column c on (zeros past column d and for a missing row), as stored.
template <typename T> struct RowPiece4 { uint32_t w[sizeof(T)]; };
template <typename T>
__device__ __forceinline__ RowPiece4<T> load_row4(const T *row, int c, int d, bool vec) {
  RowPiece4<T> f;
#pragma unroll
  for (int i = 0; i < (int)sizeof(T); ++i) f.w[i] = 0;
  if (row == nullptr || c >= d) return f;
  if (vec) {   // d is a multiple of 4 then
    if constexpr (sizeof(T) == 4) {
      const uint4 v = __ldg(reinterpret_cast<const uint4 *>(row + c));
      f.w[0] = v.x; f.w[1] = v.y; f.w[2] = v.z; f.w[3] = v.w;
    } else {
      const uint2 v = __ldg(reinterpret_cast<const uint2 *>(row + c));
      f.w[0] = v.x; f.w[1] = v.y;
    }
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (c + e >= d) continue;
      if constexpr (sizeof(T) == 4)
        f.w[e] = __float_as_uint(row[c + e]);
      else
        f.w[e >> 1] |= (uint32_t)__bfloat16_as_ushort(row[c + e]) << (16 * (e & 1));
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
  const uint32_t z_base = smem0, u_ring = z_base + Cfg::kZBytes, staging = u_ring + SU * Cfg::kUStageBytes;
  const uint32_t bars = staging + Cfg::kStagings * Cfg::kHalfBytes;
  const uint32_t z_full_bar = bars, z_empty_bar = bars + 8;
  auto u_full_bar = [&](int s) { return bars + (2 + s) * 8; };
  auto u_empty_bar = [&](int s) { return bars + (2 + SU + s) * 8; };
  auto d_full_bar = [&](int b) { return bars + (2 + 2 * SU + b) * 8; };
  auto d_empty_bar = [&](int b) { return bars + (2 + 2 * SU + 2 + b) * 8; };
  unsigned char *tail = smem_raw + (bars - smem_u) + Cfg::kBars * 8;
  volatile uint32_t *tmem_slot_ptr = reinterpret_cast<volatile uint32_t *>(tail);
  // [unit % kUnsafeSlots][operand warp]: U of the unit holds values its split does not
  volatile unsigned char *unit_flags = tail + 16;

  if (tid == 0) {
    mbar_init(z_full_bar, kSplitOperandWarps);
    mbar_init(z_empty_bar, 1);
    for (int s = 0; s < SU; ++s) {
      mbar_init(u_full_bar(s), kSplitOperandWarps);
      mbar_init(u_empty_bar(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(d_full_bar(b), 1);
      mbar_init(d_empty_bar(b), kSplitOutWarps);
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

  if (warp >= kSplitOutWarps && warp < kSplitOutWarps + kSplitOperandWarps) {
    // ------------------------------------------------------------------------- operands
    // A warp takes every fourth row of a tile, 16 rows in flight; lane = pair of coordinates, so the
    // loads are coalesced and the swizzled stores of a row hit all banks once.
    const int ow = warp - kSplitOutWarps;
    constexpr int R = 16, kBatches = kUmmaTile / (R * kSplitOperandWarps);
    int64_t tile = -1;
    int slot = 0;
    uint32_t parity = 1, z_parity = 1;
    for (int64_t unit = u_lo; unit < u_hi; ++unit) {
      const int64_t ut = unit / nchunks;
      const int col0 = (int)(unit - ut * nchunks) * kChunkCols;
      if (ut != tile) {
        tile = ut;
        const TZ *Z = static_cast<const TZ *>(a.zin);
#pragma unroll 1
        for (int kb = 0; kb < KG * kBatches; ++kb) {
          const int kg = kb / kBatches, r0 = (kb % kBatches) * R * kSplitOperandWarps + ow, j = kg * 64 + 2 * lane;
          Pair<TZ> z[R];
#pragma unroll
          for (int i = 0; i < R; ++i) {
            const int64_t t = tile * kUmmaTile + r0 + i * kSplitOperandWarps;
            z[i] = load_pair<TZ>(Z + t * a.ldzin + j, t < a.n ? a.k - j : 0, a.vec_z != 0);
          }
          if (kb == 0) {
            if (!dead && !mbar_wait(z_empty_bar, z_parity)) timed_out();
            z_parity ^= 1u;
          }
#pragma unroll
          for (int i = 0; i < R; ++i) {
            const int r = r0 + i * kSplitOperandWarps;
            uint32_t p[NZ];
            split_pair<TZ, NZ>(z[i], p);
            const uint32_t addr = z_base + kg * kSplitTileBytes + r * 128 + (((lane >> 2) ^ (r & 7)) << 4) + (lane & 3) * 4;
#pragma unroll
            for (int s = 0; s < NZ; ++s) st_shared_b32(addr + s * KG * kSplitTileBytes, p[s]);
          }
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(z_full_bar);
      }
#pragma unroll 1
      for (int kg = 0; kg < KG; ++kg) {
        const int j = kg * 64 + 2 * lane;
        const uint32_t base = u_ring + (uint32_t)slot * Cfg::kUStageBytes;
        uint32_t u_max = 0;
#pragma unroll 1
        for (int b = 0; b < kBatches; ++b) {
          const int r0 = b * R * kSplitOperandWarps + ow;
          Pair<T> u[R];
#pragma unroll
          for (int i = 0; i < R; ++i) {
            const int c = col0 + r0 + i * kSplitOperandWarps;
            u[i] = load_pair<T>(U + (int64_t)c * a.ldu + j, c < a.d ? a.k - j : 0, a.vec_u != 0);
          }
          if (b == 0 && !dead && !mbar_wait(u_empty_bar(slot), parity)) timed_out();
#pragma unroll
          for (int i = 0; i < R; ++i) {
            const int r = r0 + i * kSplitOperandWarps;
            uint32_t p[NU];
            split_pair<T, NU>(u[i], p);
            if (Cfg::kLow) u_max = max(u_max, pair_magnitude<T>(u[i]));
            const uint32_t addr = base + r * 128 + (((lane >> 2) ^ (r & 7)) << 4) + (lane & 3) * 4;
#pragma unroll
            for (int s = 0; s < NU; ++s) st_shared_b32(addr + s * kSplitTileBytes, p[s]);
          }
        }
        if (Cfg::kLow) {   // the flag of this unit: the last reader of its slot was eight units ago
          const bool huge = __any_sync(0xffffffffu, u_max >= kSplitHugeBits);
          volatile unsigned char *flag = unit_flags + (int)((unit - u_lo) % Cfg::kUnsafeSlots) * kSplitOperandWarps + ow;
          if (lane == 0 && (kg == 0 || huge)) *flag = huge ? 1 : 0;
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(u_full_bar(slot));
        if (++slot == SU) {
          slot = 0;
          parity ^= 1u;
        }
      }
    }
  } else if (warp == kSplitOutWarps + kSplitOperandWarps) {
    // ------------------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      constexpr uint32_t idesc = umma_idesc_kk(kChunkCols);
      const uint64_t kdesc = umma_desc(0, 16, 1024, 2);
      int64_t tile = -1, count = 0;
      int slot = 0;
      uint32_t parity = 0, z_parity = 0;
      for (int64_t unit = u_lo; unit < u_hi; ++unit, ++count) {
        const int64_t ut = unit / nchunks;
        if (ut != tile) {
          tile = ut;
          if (!dead && !mbar_wait(z_full_bar, z_parity)) timed_out();
          z_parity ^= 1u;
        }
        const int db = (int)(count & 1);
        if (!dead && !mbar_wait(d_empty_bar(db), (uint32_t)(((count >> 1) & 1) ^ 1))) timed_out();
        const uint32_t hi = tmem_base + (uint32_t)db * Cfg::kDCols, lo = hi + kChunkCols;
#pragma unroll
        for (int kg = 0; kg < KG; ++kg) {
          if (!dead && !mbar_wait(u_full_bar(slot), parity)) timed_out();
          asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
          const uint64_t zd = kdesc + umma_desc_addr(z_base + kg * kSplitTileBytes);
          const uint64_t ud = kdesc + umma_desc_addr(u_ring + (uint32_t)slot * Cfg::kUStageBytes);
          constexpr uint32_t kZPart = (uint32_t)(KG * kSplitTileBytes) >> 4, kUPart = (uint32_t)kSplitTileBytes >> 4;
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
        if (unit + 1 == u_hi || (unit + 1) / nchunks != tile) umma_commit(z_empty_bar);
      }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------------------- output
    const int quarter = warp & 3, cpart = warp >> 2;       // TMEM lanes; 16 of the 64 columns of a half
    const int trow = quarter * 32 + lane;                  // row this thread stages
    const int sub = lane >> 4, c4 = (lane & 15) * 4;       // rows 2 i + sub of the warp's eight, columns c4 .. +3
    const bool vec = a.vec_out != 0;
    int64_t tile = -1, count = 0;
    int32_t er = -1, pr = -1;                              // lanes 0-7: table rows of the warp's rows
    uint32_t unsafe_rows = 0;
    RowPiece4<T> in[NSLOT > 0 ? NSLOT : 1][4];
    auto issue = [&](int col) {                            // E and P pieces of the warp's rows
#pragma unroll
      for (int i = 0; i < (NSLOT > 0 ? 4 : 0); ++i) {
        const int32_t e = __shfl_sync(0xffffffffu, er, 2 * i + sub), p = __shfl_sync(0xffffffffu, pr, 2 * i + sub);
        const T *erow = e >= 0 ? static_cast<const T *>(a.shift.E) + (int64_t)e * a.shift.lde : nullptr;
        const T *prow = p >= 0 ? static_cast<const T *>(a.shift.P) + (int64_t)p * a.shift.ldp : nullptr;
        if (NSLOT == 2) {
          in[0][i] = load_row4<T>(erow, col + c4, a.d, vec);
          in[NSLOT - 1][i] = load_row4<T>(prow, col + c4, a.d, vec);
        } else {
          in[0][i] = load_row4<T>(a.has_e ? erow : prow, col + c4, a.d, vec);
        }
      }
    };
    auto enter_tile = [&](int64_t ut) {
      const int64_t t = ut * kUmmaTile + warp * 8 + lane;
      er = pr = -1;
      if (NSLOT > 0 && lane < 8 && t < a.n) {
        if (a.has_e) er = (int32_t)embedding_row(a.shift, t);
        if (a.has_p) pr = (int32_t)position_row(a.shift, t);
      }
      if (NZ == 3) {                                       // rows whose split does not hold
        unsafe_rows = 0;
        for (int r = 0; r < 8; ++r) {
          const int64_t tr = ut * kUmmaTile + warp * 8 + r;
          uint32_t m = 0;
          if (tr < a.n) {
            const TZ *z = static_cast<const TZ *>(a.zin) + tr * a.ldzin;
            for (int j = lane; j < a.k; j += 32) m = max(m, magnitude_bits(to_f32(z[j])));
          }
          m = __reduce_max_sync(0xffffffffu, m);
          if (split_unsafe(m)) unsafe_rows |= 1u << r;
        }
      }
    };
    if (u_lo < u_hi) {
      tile = u_lo / nchunks;
      enter_tile(tile);
      issue((int)(u_lo - tile * nchunks) * kChunkCols);
    }
    for (int64_t unit = u_lo; unit < u_hi; ++unit, ++count) {
      const int col0 = (int)(unit - tile * nchunks) * kChunkCols;
      const int db = (int)(count & 1);
      if (!dead && !mbar_wait(d_full_bar(db), (uint32_t)((count >> 1) & 1))) timed_out();
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      uint32_t bad = 0;
      if (Cfg::kLow) {
        bad = unsafe_rows;
        if (reinterpret_cast<volatile uint32_t *>(tail + 16)[(int)(count % Cfg::kUnsafeSlots)] != 0) bad = 0xFFu;
      }
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
          asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];\n"
                       : "=f"(o[i][0]), "=f"(o[i][1]), "=f"(o[i][2]), "=f"(o[i][3])
                       : "r"(stage + r * 256 + (((lane & 15) ^ (r & 15)) << 4)));
        }
        const int col = col0 + g * kSplitHalf;
        if (Cfg::kLow && bad != 0) {                       // plain FMAs for the flagged rows
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int64_t t = tile * kUmmaTile + warp * 8 + 2 * i + sub;
            if (!(bad >> (2 * i + sub) & 1) || t >= a.n) continue;
            const TZ *z = static_cast<const TZ *>(a.zin) + t * a.ldzin;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int c = col + c4 + e;
              if (c >= a.d) continue;
              float acc = 0.f;
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
        const int64_t out_tile = tile;
        if (g == 0) {
          issue(col + kSplitHalf);
        } else if (unit + 1 < u_hi) {
          const int64_t ut = (unit + 1) / nchunks;
          if (ut != tile) {
            tile = ut;
            enter_tile(tile);
          }
          issue((int)(unit + 1 - tile * nchunks) * kChunkCols);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int64_t t = out_tile * kUmmaTile + warp * 8 + 2 * i + sub;
          const int c = col + c4;
          if (t >= a.n || c >= a.d) continue;
          T *out = static_cast<T *>(a.dst) + t * a.lddst + c;
          if (vec) {
            if (sizeof(T) == 4)
              *reinterpret_cast<float4 *>(out) = make_float4(o[i][0], o[i][1], o[i][2], o[i][3]);
            else
              *reinterpret_cast<uint2 *>(out) = make_uint2(pack_bf16(o[i][0], o[i][1]), pack_bf16(o[i][2], o[i][3]));
          } else {
#pragma unroll
            for (int e = 0; e < 4; ++e)
              if (c + e < a.d) out[e] = from_f32<T>(o[i][e]);
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
