// Split-operand tcgen05 projection of the SSN codec:
//     Z = (X [+ R] [- E[ids]] [- P[pos]]) U
// for fp32 storage, and for the bf16 calls whose operands the TMA projection cannot fetch: leading
// dimensions or addresses off the 16-byte grid, positions per token, a residual addend beside row tables.
//
// cp.async brings the rows in, 16 bytes at a time and any row per token, several steps ahead (what is in
// flight is bounded by shared memory, not by registers); the residual is formed in fp32 as the general
// kernel does, split into bf16 parts (codec_split.cuh) and written as swizzled operand tiles; the basis is split
// the same way, step by step.  With bf16 rows and no subtraction one part is exact, and bf16 bases have
// one part.  A step is 128 bytes of every row: 32 columns of fp32, 64 of bf16.
//
//   warps 0-15  every thread reads back the pieces it copied itself (no barrier), writes their parts and its
//               share of U to the step's operand stage, and requests the rows of the step RD - 1 ahead.
//               Every 64 columns a finished accumulator is added to fp32 sums in registers (see
//               codec_split.cuh on why the chains are this short): warp w reads TMEM lanes 32 (w % 4) .. +31
//               and a quarter of the columns.
//   warp 16     one thread issues the MMAs: Ah x (Uh|Um|Ul), Am x (Uh|Um), Al x Uh, the parts of U side by
//               side on N so that three instructions per K step cover the six products (rank above 64:
//               five instructions, (Uh|Um) being 256 columns wide).  It is a warp of its own because each
//               of these instructions blocks its thread for about 100 clocks.
//
// A CTA takes whole tiles of 128 tokens, or a cluster of 2 to 8 CTAs shares one tile where that fills the
// SMs better: each contracts a slice of d, and the partial sums meet through distributed shared memory, every
// CTA finishing its share of the rows.
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
  int32_t vec_rows;            // every row operand may be read 16 bytes at a time and g_zero_row holds a row
  int32_t vec_u, vec_out;      // two coordinates of U may be read, four coordinates stored at a time
  ShiftTables shift;
};

constexpr int kSplitRowWarps = 16, kSplitRowThreads = 32 * kSplitRowWarps;
constexpr int kSplitProjectThreads = kSplitRowThreads + 32;
constexpr int kSplitRawBytes = kUmmaTile * 128;       // one operand's rows of one step

template <typename T, int KN, int NSLOT>
struct SplitProjectConfig {
  static_assert(KN == 32 || KN == 64 || KN == 128, "coordinates, rounded up");
  static constexpr bool kF32 = sizeof(T) == 4;
  static constexpr int kNX = kF32 || NSLOT > 0 ? 3 : 1;    // parts of the residual
  static constexpr int kNU = kF32 ? 3 : 1;                 // parts of U
  static constexpr int kStack = kNU == 3 ? (KN <= 64 ? 3 : 2) : 1;   // parts of U under one Ah product
  // KN-wide accumulators of a chain, all of them summed in fp32 where it ends.  fp32: hi and low products, side by
  // side.  bf16 bases leave room to deal the K steps of the leading product to several: gradients
  // of 4096 columns, rank 51, one accumulator 1.6e-7 from 64-bit sums, four 9.2e-8, plain FMAs 9.5e-8.
  static constexpr int kHiAccs = kNU == 3 ? 1 : (kNX == 1 ? (KN <= 64 ? 4 : 2) : (KN <= 64 ? 2 : 1));
  static constexpr int kAccs = kNU == 3 ? kStack : kHiAccs + (kNX == 3 ? 1 : 0);
  static constexpr int kDCols = kAccs * KN;
  static constexpr int kDStride = kDCols <= 32 ? 32 : (kDCols <= 64 ? 64 : (kDCols <= 128 ? 128 : 256));
  static constexpr int kTmemCols = 2 * kDStride;
  static constexpr int kCols = kF32 ? 32 : 64;              // columns of d per step
  static constexpr int kPartBytes = kUmmaTile * kCols * 2;  // one bf16 part of a [128 x kCols] operand
  static constexpr int kRowBytes = kCols * 2;               // its rows, swizzled within 64 or 128 bytes
  static constexpr int kABytes = kNX * kPartBytes;
  static constexpr int kBGroups = (kNU * KN + 63) / 64;     // 64-coordinate groups of all parts
  static constexpr int kGroupBytes = kCols * 128;
  static constexpr int kStageBytes = kABytes + kBGroups * kGroupBytes;
  static constexpr int kRawStepBytes = (1 + NSLOT) * kSplitRawBytes;
  static constexpr int kSumPitch = KN + 4;                  // floats per row of the exchanged sums
  static constexpr int kSumBytes = kUmmaTile * kSumPitch * 4;
  // barriers, TMEM address, largest magnitude per column of U, and of four tiles: rows the split does not hold
  static constexpr int kBars = 8;
  static constexpr int kTailBytes = kBars * 8 + 16 + 4 * KN + 4 * kUmmaTile;
  static constexpr int kRoom = 227 * 1024 - 1024 - 1152;
  static_assert(kTailBytes <= 1152, "the tail");
  // two operand stages unless that leaves no two steps of rows (bf16, three more operands)
  static constexpr int kStages = kRoom - 2 * kStageBytes >= 2 * kRawStepBytes ? 2 : 1;
  static constexpr int kFit = (kRoom - kStages * kStageBytes) / kRawStepBytes;
  static constexpr int kRaw = kFit < 6 ? kFit : 6;          // steps of rows in flight or being read
  static_assert(kRaw >= 2, "no room for two steps of rows");
  static constexpr int kRingBytes = kStages * kStageBytes + kRaw * kRawStepBytes;
  static_assert(kRingBytes >= kSumBytes, "the exchanged sums take the place of the rings");
  static constexpr int kSmemBytes = 1024 + kRingBytes + kTailBytes;
  static constexpr int kChain = 64 / kCols;                 // steps per accumulator
  static constexpr int kPairs = kCols * KN / 2 / kSplitRowThreads;   // pairs of U per thread and step
  static constexpr int kSums = KN / 4;                      // coordinates of one row per thread
  static constexpr int kVecElems = kF32 ? 4 : 8;            // of a 16-byte piece; a thread has two per operand and step
};

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

// Whether four finished sums stand: finite, and from columns of U that the split holds (largest magnitudes as bits;
// zero columns are fine).
__device__ __forceinline__ bool sums_stand(const float (&v)[4], const uint32_t *largest) {
  bool ok = true;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    ok = ok && fabsf(v[c]) < __int_as_float(0x7f800000);
    if (largest != nullptr) ok = ok && (largest[c] == 0 || largest[c] >= __float_as_uint(kSplitTinyU));
  }
  return ok;
}

// Coordinates j .. j + 3 of token t again, as plain sums in 64 bits: for rows or columns of U that the split does not
// hold, and for sums that left the range of fp32 on the way.
template <typename T>
__device__ __noinline__ void store_plain_coords4(const SplitProjectArgs &a, int64_t t, int j) {
  const T *U = static_cast<const T *>(a.U), *x = static_cast<const T *>(a.src) + t * a.lds;
  const T *x2 = a.src2 != nullptr ? static_cast<const T *>(a.src2) + t * a.lds2 : nullptr;
  const int64_t er = a.has_e ? embedding_row(a.shift, t) : -1, pr = a.has_p ? position_row(a.shift, t) : -1;
  const T *e = er >= 0 ? static_cast<const T *>(a.shift.E) + er * a.shift.lde : nullptr;
  const T *p = pr >= 0 ? static_cast<const T *>(a.shift.P) + pr * a.shift.ldp : nullptr;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
  for (int i = 0; i < a.d; ++i) {
    float r = to_f32(x[i]);
    if (x2 != nullptr) r += to_f32(x2[i]);
    if (e != nullptr) r -= to_f32(e[i]);
    if (p != nullptr) r -= to_f32(p[i]);
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (j + c < a.k) acc[c] = fma((double)r, (double)to_f32(U[(int64_t)i * a.ldu + j + c]), acc[c]);
  }
  store_coords4<T>(a, t, j, {(float)acc[0], (float)acc[1], (float)acc[2], (float)acc[3]});
}

template <typename T, int KN, int NSLOT>
__global__ void __launch_bounds__(kSplitProjectThreads, 1) codec_split_project_kernel(const SplitProjectArgs a) {
  using Cfg = SplitProjectConfig<T, KN, NSLOT>;
  constexpr int NX = Cfg::kNX, NU = Cfg::kNU, S = Cfg::kStages, RD = Cfg::kRaw, G = Cfg::kChain;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  uint32_t cluster_size, cta_rank;
  asm volatile("mov.u32 %0, %%cluster_nctaid.x;\n" : "=r"(cluster_size));
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(cta_rank));
  const int64_t ntiles = (a.n + kUmmaTile - 1) / kUmmaTile;
  const int64_t groups = gridDim.x / cluster_size, group = blockIdx.x / cluster_size;
  const int nst = (a.d + Cfg::kCols - 1) / Cfg::kCols;
  const int st_lo = (int)((int64_t)nst * cta_rank / cluster_size);
  const int nloc = (int)((int64_t)nst * (cta_rank + 1) / cluster_size) - st_lo;   // >= 1: cluster_size <= nst
  const int my_tiles = (int)((ntiles - group + groups - 1) / groups);             // 1 with clusters
  const int steps = my_tiles * nloc;

  const uint32_t smem_u = smem_u32(smem_raw), smem0 = (smem_u + 1023u) & ~1023u;
  const uint32_t raw0 = smem0 + S * Cfg::kStageBytes, bars = smem0 + Cfg::kRingBytes;
  auto full_bar = [&](int s) { return bars + s * 8; };
  auto empty_bar = [&](int s) { return bars + (2 + s) * 8; };
  auto acc_full_bar = [&](int b) { return bars + (4 + b) * 8; };
  auto acc_empty_bar = [&](int b) { return bars + (6 + b) * 8; };
  unsigned char *tail = smem_raw + (bars - smem_u) + Cfg::kBars * 8;
  volatile uint32_t *tmem_slot_ptr = reinterpret_cast<volatile uint32_t *>(tail);
  uint32_t *u_largest = reinterpret_cast<uint32_t *>(tail + 16);       // [coordinate], as bits
  volatile unsigned char *row_flags = tail + 16 + 4 * KN;              // [tile & 3][row]

  if (tid == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(full_bar(s), kSplitRowWarps);
      mbar_init(empty_bar(s), 1);
      mbar_init(acc_full_bar(s), 1);
      mbar_init(acc_empty_bar(s), kSplitRowWarps);
    }
    for (int j = 0; j < KN; ++j) u_largest[j] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == kSplitRowWarps) {
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

  if (warp == kSplitRowWarps) {
    // ------------------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      // A: K-major rows of kRowBytes, 8-row groups 8 kRowBytes apart, one part after the other.  B: MN-major,
      // 64-coordinate groups kGroupBytes apart, 8-row groups 1024 bytes apart.
      constexpr uint32_t kLayoutA = Cfg::kF32 ? 4 : 2;       // 64- or 128-byte swizzle
      constexpr uint32_t id1 = umma_idesc(KN, false), id2 = umma_idesc(Cfg::kStack >= 2 ? 2 * KN : KN, false),
                         id3 = umma_idesc(Cfg::kStack == 3 ? 3 * KN : KN, false);
      constexpr uint32_t kPart = Cfg::kPartBytes >> 4;                             // next part of A
      constexpr uint32_t kBPart = (uint32_t)(KN / 64) * (Cfg::kGroupBytes >> 4);   // next part of B (KN = 128 only)
      int slot = 0, st = 0, in_chain = 0, chain = 0;
      uint32_t parity = 0;
      for (int step = 0; step < steps; ++step) {
        const int buf = chain & 1;
        if (in_chain == 0 && !dead && !mbar_wait(acc_empty_bar(buf), (uint32_t)(((chain >> 1) & 1) ^ 1))) timed_out();
        if (!dead && !mbar_wait(full_bar(slot), parity)) timed_out();
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const uint32_t base = smem0 + (uint32_t)slot * Cfg::kStageBytes;
        const uint32_t D = tmem_base + (uint32_t)buf * Cfg::kDStride;
        const uint64_t ad = umma_desc(base, 16, 8 * Cfg::kRowBytes, kLayoutA);
        const uint64_t bd = umma_desc(base + Cfg::kABytes, Cfg::kGroupBytes, 1024, 2);
#pragma unroll
        for (int j = 0; j < Cfg::kCols / 16; ++j) {
          const uint64_t A = ad + j * 2, B = bd + j * 128;   // 32 bytes of an A row; 16 rows of B
          const uint32_t more = in_chain > 0 || j > 0 ? 1u : 0u;
          if (NU == 1) {                       // a bf16 chain is one step
            umma_bf16(D + (j % Cfg::kHiAccs) * KN, A, B, id1, j >= Cfg::kHiAccs ? 1u : 0u);
            if (NX == 3) {
              umma_bf16(D + Cfg::kHiAccs * KN, A + kPart, B, id1, more);
              umma_bf16(D + Cfg::kHiAccs * KN, A + 2 * kPart, B, id1, 1u);
            }
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
        umma_commit(empty_bar(slot));
        if (++st == nloc) st = 0;
        if (++in_chain == G || st == 0) {    // chains never reach into the next tile
          umma_commit(acc_full_bar(buf));
          in_chain = 0;
          ++chain;
        }
        if (++slot == S) {
          slot = 0;
          parity ^= 1u;
        }
      }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------------------- rows, basis, sums
    // Two 16-byte pieces per operand and step: rows tid / 8 and tid / 8 + 64, piece tid % 8.
    const int row = tid >> 3, unit = tid & 7;
    const bool vec = a.vec_rows != 0;
    // the pairs of U this thread moves: rows u_row, u_row + kURows, ... of the step (8 divides kURows)
    constexpr int kURows = 2 * kSplitRowThreads / KN;
    const int u_row = tid / (KN / 2), u_col = 2 * (tid % (KN / 2)), u_valid = max(a.k - u_col, 0);
    const int64_t u_step = kURows * a.ldu;
    const bool vec_u = a.vec_u != 0;
    const T *U = static_cast<const T *>(a.U);
    const T *ptr[1 + NSLOT][2];              // this thread's rows: X, then R, E, P as far as present
    Pair<T> ureg[Cfg::kPairs];
    const bool has_r = NSLOT > 0 && a.src2 != nullptr;

    auto row_pointers = [&](int64_t tile) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int64_t t = min(tile * kUmmaTile + row + 64 * h, a.n - 1);   // past the end: the last row again, never stored
        ptr[0][h] = static_cast<const T *>(a.src) + t * a.lds;
        if (NSLOT > 0) {
          int s = 1;
          const T *none = vec ? reinterpret_cast<const T *>(g_zero_row) : nullptr;   // an id or position outside its table
          const T *r = has_r ? static_cast<const T *>(a.src2) + t * a.lds2 : none, *e = none, *p = none;
          const int64_t er = a.has_e ? embedding_row(a.shift, t) : -1, pr = a.has_p ? position_row(a.shift, t) : -1;
          if (er >= 0) e = static_cast<const T *>(a.shift.E) + er * a.shift.lde;
          if (pr >= 0) p = static_cast<const T *>(a.shift.P) + pr * a.shift.ldp;
          // slots in the order R, E, P; with constant indexes so that the array stays in registers
          const T *list[3] = {r, e, p};
          const bool present[3] = {has_r, a.has_e != 0, a.has_p != 0};
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            if (!present[c]) continue;
#pragma unroll
            for (int i = 1; i <= NSLOT; ++i)
              if (i == s) ptr[i][h] = list[c];
            ++s;
          }
        }
      }
    };
    const uint32_t raw_off = (uint32_t)tid * 16;             // + 8192: the second piece
    auto issue_rows = [&](int st, int rslot) {
      const int c = (st_lo + st) * Cfg::kCols + unit * Cfg::kVecElems;
      const uint32_t dst = raw0 + (uint32_t)rslot * Cfg::kRawStepBytes + raw_off;
      if (vec) {
        const bool ok = c < a.d;                             // d is a multiple of the piece
#pragma unroll
        for (int o = 0; o < 1 + NSLOT; ++o)
#pragma unroll
          for (int h = 0; h < 2; ++h) cp_async16_if(dst + o * kSplitRawBytes + h * 8192, ptr[o][h] + (ok ? c : 0), ok);
      } else {
#pragma unroll
        for (int o = 0; o < 1 + NSLOT; ++o)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const uint4 v = load_row_piece<T>(ptr[o][h], c, a.d);
            st_shared_v4(dst + o * kSplitRawBytes + h * 8192, v.x, v.y, v.z, v.w);
          }
      }
    };
    auto issue_u = [&](int st) {
      const int c0 = (st_lo + st) * Cfg::kCols;
      const T *up = U + (int64_t)(c0 + u_row) * a.ldu + u_col;
      if (c0 + Cfg::kCols <= a.d) {          // whole step; a pair past column k stays the zero it is
        load_pairs<Cfg::kPairs, T>(ureg, [&](int i) { return up + i * u_step; }, u_valid, vec_u);
      } else {
#pragma unroll
        for (int i = 0; i < Cfg::kPairs; ++i) {
          const bool in = c0 + u_row + i * kURows < a.d;
          if constexpr (Cfg::kF32) {
            ureg[i].w[0] = load_global_b32_if(up + i * u_step, in && u_valid > 0);
            ureg[i].w[1] = load_global_b32_if(up + i * u_step + 1, in && u_valid > 1);
          } else {
            ureg[i].w[0] = load_global_b16_if(up + i * u_step, in && u_valid > 0);
            ureg[i].w[1] = load_global_b16_if(up + i * u_step + 1, in && u_valid > 1);
          }
        }
      }
    };
    int chain = 0, fin_tile = 0;             // accumulators written so far, tiles finished
    // adds accumulator c to the sums; `last`: it completes a tile
    auto take_chain = [&](int c, bool last) {
      const int buf = c & 1;
      if (!dead && !mbar_wait(acc_full_bar(buf), (uint32_t)((c >> 1) & 1))) timed_out();
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      if (sum_col < a.k) {
        const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)buf * Cfg::kDStride + sum_col;
#pragma unroll
        for (int i = 0; i < Cfg::kSums; i += 8) {
          uint32_t v[Cfg::kAccs][8];
#pragma unroll
          for (int c2 = 0; c2 < Cfg::kAccs; ++c2) tmem_ld8(taddr + c2 * KN + i, v[c2]);
          asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
          for (int e = 0; e < 8; e += 2) {
            // from the last on: the low products come last
            float w0 = __uint_as_float(v[Cfg::kAccs - 1][e]), w1 = __uint_as_float(v[Cfg::kAccs - 1][e + 1]);
#pragma unroll
            for (int c2 = Cfg::kAccs - 2; c2 >= 0; --c2) add2(w0, w1, __uint_as_float(v[c2][e]), __uint_as_float(v[c2][e + 1]));
            add2(sum[i + e], sum[i + e + 1], w0, w1);
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty_bar(buf));
      if (last) {
        const int64_t t = (group + (int64_t)fin_tile * groups) * kUmmaTile + sum_row;
        if (cluster_size == 1) {
          if (t < a.n) {
            uint32_t bad = NX == 3 && row_flags[(fin_tile & 3) * kUmmaTile + sum_row] != 0 ? ~0u : 0u;
#pragma unroll
            for (int i = 0; i < Cfg::kSums; i += 4) {
              const float v[4] = {sum[i], sum[i + 1], sum[i + 2], sum[i + 3]};
              store_coords4<T>(a, t, sum_col + i, v);
              if (NX == 3 && !sums_stand(v, NU == 3 ? u_largest + sum_col + i : nullptr)) bad |= 1u << (i / 4);
            }
            if (bad != 0) {
#pragma unroll 1
              for (int i = 0; i < Cfg::kSums / 4 && sum_col + 4 * i < a.k; ++i)
                if (bad >> i & 1) store_plain_coords4<T>(a, t, sum_col + 4 * i);
            }
            if (a.wire_ids && part == 0) static_cast<int32_t *>(a.zout)[t * a.ldzout + a.k] = a.shift.ids[t];
          }
#pragma unroll
          for (int i = 0; i < Cfg::kSums; ++i) sum[i] = 0.f;
        }
        ++fin_tile;
      }
    };

    int ld_tile = 0, ld_st = 0, ld_slot = 0;
    auto advance_rows = [&](bool more) {     // requests one more step (or commits an empty group)
      if (more) {
        if (ld_st == 0) row_pointers(group + (int64_t)ld_tile * groups);
        issue_rows(ld_st, ld_slot);
        if (++ld_st == nloc) {
          ld_st = 0;
          ++ld_tile;
        }
        if (++ld_slot == RD) ld_slot = 0;
      }
      cp_async_commit();
    };
#pragma unroll
    for (int i = 0; i < Cfg::kPairs; ++i) ureg[i].w[0] = ureg[i].w[1] = 0;
    issue_u(0);
    for (int i = 0; i < RD - 1; ++i) advance_rows(i < steps);

    int slot = 0, rslot = 0, st = 0, in_chain = 0;
    uint32_t parity = 1;
    int tile = 0;                            // of this CTA, being filled
    bool prev_last = false;
    float u_max[2] = {0.f, 0.f}, row_max[2] = {0.f, 0.f};
    const uint32_t a_off = Cfg::kF32 ? row * 64 + (((unit >> 1) ^ ((row >> 1) & 3)) << 4) + (unit & 1) * 8
                                     : row * 128 + ((unit ^ (row & 7)) << 4);   // + 64 rows: the second piece
    for (int step = 0; step < steps; ++step) {
      cp_async_wait<RD - 2>();
      const int next_st = st + 1 == nloc ? 0 : st + 1;
      uint4 x[2], w[NSLOT > 0 ? NSLOT : 1][2];
      const uint32_t src = raw0 + (uint32_t)rslot * Cfg::kRawStepBytes + raw_off;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        x[h] = ld_shared_v4(src + h * 8192);
#pragma unroll
        for (int o = 0; o < NSLOT; ++o) w[o][h] = ld_shared_v4(src + (o + 1) * kSplitRawBytes + h * 8192);
      }
      if (!dead && !mbar_wait(empty_bar(slot), parity)) timed_out();
      const uint32_t base = smem0 + (uint32_t)slot * Cfg::kStageBytes;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t addr = base + a_off + h * 64 * Cfg::kRowBytes;
        if constexpr (NX == 1) {
          st_shared_v4(addr, x[h].x, x[h].y, x[h].z, x[h].w);
        } else {
          constexpr int E = Cfg::kVecElems;
          float r[E];
          widen_piece<T>(x[h], r);
#pragma unroll
          for (int o = 0; o < NSLOT; ++o) {
            float v[E];
            widen_piece<T>(w[o][h], v);
            const bool plus = o == 0 && has_r;
#pragma unroll
            for (int e = 0; e < E; e += 2) {
              if (plus) add2(r[e], r[e + 1], v[e], v[e + 1]);
              else sub2(r[e], r[e + 1], v[e], v[e + 1]);
            }
          }
#pragma unroll
          for (int e = 0; e < E; ++e) row_max[h] = fmaxf(row_max[h], fabsf(r[e]));
          uint32_t p[E / 2][3];
#pragma unroll
          for (int e = 0; e < E / 2; ++e) split_pair<3>(r[2 * e], r[2 * e + 1], p[e]);
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            if constexpr (Cfg::kF32) st_shared_v2(addr + i * Cfg::kPartBytes, p[0][i], p[1][i]);
            else st_shared_v4(addr + i * Cfg::kPartBytes, p[0][i], p[1][i], p[2][i], p[3][i]);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < Cfg::kPairs; ++i) {
        const Pair<T> u = joined<T>(ureg[i]);
        if (NU == 3) pair_maxima<T>(u, u_max);
        uint32_t up[NU];
        split_pair<T, NU>(u, up);
#pragma unroll
        for (int s = 0; s < NU; ++s) {
          const int n = s * KN + u_col;
          st_shared_b32(base + Cfg::kABytes + (n >> 6) * Cfg::kGroupBytes + (u_row + i * kURows) * 128 +
                            ((((n & 63) >> 3) ^ (u_row & 7)) << 4) + (n & 7) * 2, up[s]);
        }
      }
      if (NX == 3 && next_st == 0) {
        // the tile's rows, and U, are complete: the eight threads of a row agree on its largest magnitude
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
          for (int off = 4; off > 0; off >>= 1) row_max[h] = fmaxf(row_max[h], __shfl_xor_sync(0xffffffffu, row_max[h], off));
          if (unit == 0) row_flags[(tile & 3) * kUmmaTile + row + 64 * h] = row_max[h] != 0.f && row_max[h] < kSplitTinyRow ? 1 : 0;
          row_max[h] = 0.f;
        }
        if (NU == 3 && tile == 0) {
          atomicMax(u_largest + u_col, __float_as_uint(u_max[0]));
          atomicMax(u_largest + u_col + 1, __float_as_uint(u_max[1]));
        }
      }
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(full_bar(slot));
      if (step + 1 < steps) issue_u(next_st);
      advance_rows(step + RD - 1 < steps);   // into the slot read in the step before
      if (++slot == S) {
        slot = 0;
        parity ^= 1u;
      }
      if (++rslot == RD) rslot = 0;
      st = next_st;
      if (st == 0) ++tile;
      if (++in_chain == G || st == 0) {      // the accumulator before the one just filled
        if (chain > 0) take_chain(chain - 1, prev_last);
        prev_last = st == 0;
        in_chain = 0;
        ++chain;
      }
    }
    take_chain(chain - 1, true);
    cp_async_wait<0>();
  }

  if (cluster_size > 1) {
    // Every accumulator has been read, so every stage is consumed and the rings can carry the sums.
    __syncthreads();
    if (warp < kSplitRowWarps) {
      const uint32_t dst = smem0 + (uint32_t)(sum_row * Cfg::kSumPitch + sum_col) * 4;
#pragma unroll
      for (int c = 0; c < Cfg::kSums; c += 4)
        st_shared_v4(dst + c * 4, __float_as_uint(sum[c]), __float_as_uint(sum[c + 1]), __float_as_uint(sum[c + 2]),
                     __float_as_uint(sum[c + 3]));
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    const int row0 = (int)(kUmmaTile * cta_rank / cluster_size), rows = (int)(kUmmaTile * (cta_rank + 1) / cluster_size) - row0;
    auto peer = [](uint32_t addr, uint32_t rank) {
      uint32_t r;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(addr), "r"(rank));
      return r;
    };
    const uint32_t row_flags_addr = smem_u32(const_cast<unsigned char *>(row_flags));   // of tile 0, the only one
    for (int i = tid; i < rows * (KN / 4); i += kSplitProjectThreads) {
      const int rr = row0 + i / (KN / 4), j = 4 * (i % (KN / 4));
      const int64_t t = group * kUmmaTile + rr;
      if (t >= a.n || j >= a.k) continue;
      float v[4] = {0.f, 0.f, 0.f, 0.f};
      uint32_t largest[4] = {0, 0, 0, 0}, bad_row = 0;
      for (uint32_t rk = 0; rk < cluster_size; ++rk) {
        float w0, w1, w2, w3;
        asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];\n"
                     : "=f"(w0), "=f"(w1), "=f"(w2), "=f"(w3)
                     : "r"(peer(smem0 + (uint32_t)(rr * Cfg::kSumPitch + j) * 4, rk)));
        v[0] += w0; v[1] += w1; v[2] += w2; v[3] += w3;
        if (NX == 3) {
          uint32_t m0, m1, m2, m3, f;
          asm volatile("ld.shared::cluster.v4.u32 {%0,%1,%2,%3}, [%4];\n"
                       : "=r"(m0), "=r"(m1), "=r"(m2), "=r"(m3) : "r"(peer(smem_u32(u_largest + j), rk)));
          largest[0] = max(largest[0], m0); largest[1] = max(largest[1], m1);
          largest[2] = max(largest[2], m2); largest[3] = max(largest[3], m3);
          asm volatile("ld.shared::cluster.u8 %0, [%1];\n" : "=r"(f) : "r"(peer(row_flags_addr + rr, rk)));
          bad_row |= f;
        }
      }
      store_coords4<T>(a, t, j, v);
      if (NX == 3 && (bad_row != 0 || !sums_stand(v, NU == 3 ? largest : nullptr))) store_plain_coords4<T>(a, t, j);
      if (a.wire_ids && j == 0) static_cast<int32_t *>(a.zout)[t * a.ldzout + a.k] = a.shift.ids[t];
    }
    // nobody leaves while its sums can still be read
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == kSplitRowWarps) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"(Cfg::kTmemCols)
                 : "memory");
  }
}

}  // namespace ssn
