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
//               At the end of a chain of 64 or 128 columns its accumulators are added to compensated fp32 sums in
//               registers (see SplitProjectConfig on the lengths): warp w reads TMEM lanes 32 (w % 4) .. +31 and a
//               quarter of the columns.
//   warp 16     one thread issues the MMAs: Ah x Uh into the leading accumulators; Ah x (Um|Ul), Am x (Uh|Um) and
//               Al x Uh into the small ones, the parts of U side by side on N.  A warp of its own, because each of
//               these instructions blocks its thread for about 100 clocks; above rank 32 warp 17 takes half of them.
//
// A CTA takes whole tiles of 128 tokens, or a cluster of 2 to 8 CTAs shares one tile where that fills the
// SMs better: each contracts a slice of d, and the partial sums meet through distributed shared memory, every
// CTA finishing its share of the rows.  Ranks above 64 are two halves on CTAs side by side: accumulators, sums and
// their compensation for 128 coordinates do not fit a thread's registers (8192 x 2048 fp32, rank 100, E rows: one
// CTA for all 136 us, halves 84).
#pragma once

#include "codec_split.cuh"

namespace ssn {

struct SplitProjectArgs {
  const void *src, *src2, *U;
  void *zout;
  int64_t lds, lds2, ldu, ldzout, n;
  int32_t d, k;
  int32_t halves, k_half;      // ranks above 64: two halves, each CTA computes k_half coordinates or the rest; else one of k
  int32_t wire, wire_ids;      // fp32 words out, word k of a row = the token id
  int32_t has_e, has_p;
  int32_t vec_rows;            // every row operand may be read 16 bytes at a time and g_zero_row holds a row
  int32_t vec_u, vec_out;      // two coordinates of U may be read, four coordinates stored at a time
  ShiftTables shift;
};

constexpr int kSplitRowWarps = 16, kSplitRowThreads = 32 * kSplitRowWarps;
constexpr int kSplitRawBytes = kUmmaTile * 128;       // one operand's rows of one step

// Slices of d of fewer columns take the CAREFUL kernel: over so few terms plain FMAs are at their best (products of
// bf16 values add up exactly at first), and the additions among a chain's accumulators show.  Gradients of 128
// columns in bf16, error against 64-bit sums: 5.1e-8, careful 4.7e-8, FMAs 4.8e-8.
constexpr int kSplitCarefulCols = 256, kSplitCarefulColsPlain = 384;   // bf16 rows as they are

template <typename T, int KN, int NSLOT, bool CAREFUL>
struct SplitProjectConfig {
  static_assert(KN == 32 || KN == 64, "coordinates, rounded up");
  static constexpr bool kF32 = sizeof(T) == 4;
  static constexpr int kNX = kF32 || NSLOT > 0 ? 3 : 1;    // parts of the residual
  static constexpr int kNU = kF32 ? 3 : 1;                 // parts of U
  // Columns of d per chain and its accumulators, each KN columns of tensor memory, added up in fp32 where the chain
  // ends: kHi for the leading products, which take turns with the K steps, and kLow for the small ones.  An
  // accumulator is truncated with every MMA that is added to it.  Coordinates of 256 to 1024 columns, error against
  // 64-bit sums, rank 8: four K steps in one accumulator 8.2e-8, in four 3.8e-8, plain FMAs 4.2e-8 (4.8e-8 at rank
  // 33, 5.5e-8 at 100: there two K steps per accumulator are near enough, 4.5e-8 and 4.8e-8).  KN columns more hold
  // the compensation of the sums over chains.  What is left decides whether there are two sets, so that a chain is
  // summed while the next is written.
  // CAREFUL (see kSplitCarefulCols) adds the accumulators one by one, with compensation.
  static constexpr bool kOneStage = !kF32 && NSLOT == 3;   // see kStages: there a second set pays more than long chains
  static constexpr int kChainCols = KN == 32 || kOneStage || kNX == 1 || CAREFUL ? 64 : 128;
  static constexpr int kHi = KN == 32 || CAREFUL ? 4 : (kOneStage ? 2 : (kNX == 1 ? 3 : 4));
  static constexpr int kLow = kNX == 1 ? 0 : (kF32 ? 2 : 1);
  static constexpr int kDCols = (kHi + kLow) * KN;
  static constexpr int kBufs = 2 * kDCols + KN <= 512 ? 2 : 1;
  static constexpr int kCompCol = kBufs * kDCols;
  static constexpr int kTmemCols = kCompCol + KN <= 256 ? 256 : 512;
  static_assert(kCompCol + KN <= 512, "tensor memory");
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
  // MMA-issuing warps.  Two where the instructions of one thread, about 100 clocks each, would take longer than the
  // rows: one issues the leading products, the other the small ones (or they share the accumulators out).
  static constexpr int kIssuers = KN == 64 ? 2 : 1;
  static constexpr int kThreads = kSplitRowThreads + 32 * kIssuers;
  static constexpr int kRoom = 227 * 1024 - 1024 - 896;
  static_assert(kTailBytes <= 896, "the tail");
  // two operand stages unless that leaves no two steps of rows (bf16, three more operands)
  static constexpr int kStages = kRoom - 2 * kStageBytes >= 2 * kRawStepBytes ? 2 : 1;
  static_assert(kStages == 2 || kOneStage, "chosen above without these sizes");
  static constexpr int kFit = (kRoom - kStages * kStageBytes) / kRawStepBytes;
  static constexpr int kRaw = kFit < 6 ? kFit : 6;          // steps of rows in flight or being read
  static_assert(kRaw >= 2, "no room for two steps of rows");
  static constexpr int kRingBytes = kStages * kStageBytes + kRaw * kRawStepBytes;
  static_assert(kRingBytes >= kSumBytes, "the exchanged sums take the place of the rings");
  static constexpr int kSmemBytes = 1024 + kRingBytes + kTailBytes;
  static constexpr int kChain = kChainCols / kCols;         // steps per chain
  static constexpr int kPairs = kCols * KN / 2 / kSplitRowThreads;   // pairs of U per thread and step
  static constexpr int kSums = KN / 4;                      // coordinates of one row per thread
  // Place of part s of U on N.  Rank up to 32: m, l, h, so that the pair m | l and h alone both start a group.
  __host__ __device__ static constexpr int b_part(int s) { return kF32 && KN == 32 ? (s + 2) % 3 : s; }
  static constexpr int kVecElems = kF32 ? 4 : 8;            // of a 16-byte piece; a thread has two per operand and step
};

template <typename T>
__device__ __forceinline__ void store_coords4(const SplitProjectArgs &a, int64_t t, int j, int j_end, const float (&v)[4]) {
  if (j >= j_end) return;
  if (a.wire || sizeof(T) == 4) {
    float *z = static_cast<float *>(a.zout) + t * a.ldzout + j;
    if (a.vec_out && j + 4 <= j_end) {
      *reinterpret_cast<float4 *>(z) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (j + e < j_end) z[e] = v[e];
    }
  } else {
    __nv_bfloat16 *z = static_cast<__nv_bfloat16 *>(a.zout) + t * a.ldzout + j;
    if (a.vec_out && j + 4 <= j_end) {
      *reinterpret_cast<uint2 *>(z) = make_uint2(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]));
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (j + e < j_end) z[e] = __float2bfloat16_rn(v[e]);
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

// Coordinates j .. j + 3 (below j_end) of token t again, as plain sums in 64 bits: for rows or columns of U that the split does not
// hold, and for sums that left the range of fp32 on the way.
template <typename T>
__device__ __noinline__ void store_plain_coords4(const SplitProjectArgs &a, int64_t t, int j, int j_end) {
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
      if (j + c < j_end) acc[c] = fma((double)r, (double)to_f32(U[(int64_t)i * a.ldu + j + c]), acc[c]);
  }
  store_coords4<T>(a, t, j, j_end, {(float)acc[0], (float)acc[1], (float)acc[2], (float)acc[3]});
}

// Clusters of few CTAs pass on the compensations as well: the rounding of a slice's sum shows where the slices are few.  Rows
// of the subspace, error against 64-bit sums without and with: 20000 x 4096 in three slices 3.4e-8, 3.2e-8; 3000 x 5120,
// rank 99 in two 3.8e-8, 3.0e-8.  Eight slices err by 3.1e-8 without.  It takes 1 us (3000 x 2048, rank 51 in four 17.2 -> 18.2).
constexpr uint32_t kFewSlices = 4;

// What a CTA of a launch with a.halves halves computes: its tiles, columns of d and coordinates.
struct SplitSchedule {
  uint32_t cluster_size, cta_rank;
  int64_t groups, group;       // CTAs (clusters) side by side, and this one
  bool upper;
  int st_lo, nloc, my_tiles;   // steps of d; one tile with clusters
  const SplitProjectArgs &a;
  __device__ __forceinline__ SplitSchedule(const SplitProjectArgs &args, int cols) : a(args) {
    asm volatile("mov.u32 %0, %%cluster_nctaid.x;\n" : "=r"(cluster_size));
    asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(cta_rank));
    const int64_t ntiles = (a.n + kUmmaTile - 1) / kUmmaTile;
    // the two halves of a tile's coordinates run side by side, so that its rows come from HBM once
    groups = gridDim.x / cluster_size / a.halves;
    group = blockIdx.x / cluster_size / a.halves;
    upper = a.halves > 1 && (blockIdx.x / cluster_size & 1) != 0;
    const int nst = (a.d + cols - 1) / cols;
    st_lo = (int)((int64_t)nst * cta_rank / cluster_size);
    nloc = (int)((int64_t)nst * (cta_rank + 1) / cluster_size) - st_lo;   // >= 1: cluster_size <= nst
    my_tiles = (int)((ntiles - group + groups - 1) / groups);
  }
  __device__ __forceinline__ int64_t tile(int i) const { return group + (int64_t)i * groups; }
  __device__ __forceinline__ bool lower() const { return a.halves > 1 && !upper; }   // coordinates j_lo() to j_end()
  __device__ __forceinline__ int j_lo() const { return upper ? a.k_half : 0; }
  __device__ __forceinline__ int j_end() const { return lower() ? a.k_half : a.k; }
  __device__ __forceinline__ int rank() const { return j_end() - j_lo(); }
};

// s += x with compensation c, two sums at a time.
__device__ __forceinline__ void add_compensated2(float &s0, float &s1, float &c0, float &c1, float x0, float x1) {
  sub2(x0, x1, c0, c1);
  float t0 = s0, t1 = s1;
  add2(t0, t1, x0, x1);
  c0 = t0, c1 = t1;
  sub2(c0, c1, s0, s1);
  sub2(c0, c1, x0, x1);
  s0 = t0, s1 = t1;
}

// The CTAs of a cluster have left their sums [128][KN + 4] at smem0; each adds up, and stores, its share of the rows.
// FLAGS: beside them lie the largest magnitudes per column of U and, per row, whether the split does not hold it.
// COMP: in clusters of up to kFewSlices, behind them lie the compensations of the sums, [128][KN + 4] too.
template <typename T, int KN, int THREADS, bool FLAGS, bool COMP>
__device__ __forceinline__ void finish_slices(const SplitProjectArgs &a, const SplitSchedule &s, uint32_t smem0, uint32_t u_largest_addr,
                                              uint32_t row_flags_addr) {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
  const int row0 = (int)(kUmmaTile * s.cta_rank / s.cluster_size), rows = (int)(kUmmaTile * (s.cta_rank + 1) / s.cluster_size) - row0;
  auto peer = [](uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
  };
  for (int i = threadIdx.x; i < rows * (KN / 4); i += THREADS) {
    const int rr = row0 + i / (KN / 4), j = 4 * (i % (KN / 4));
    const int64_t t = s.group * kUmmaTile + rr;
    if (t >= a.n || j >= s.rank()) continue;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    uint32_t largest[4] = {0, 0, 0, 0}, bad_row = 0;
    auto slice = [&](int row, uint32_t rk, float (&w)[4]) {
      asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];\n"
                   : "=f"(w[0]), "=f"(w[1]), "=f"(w[2]), "=f"(w[3])
                   : "r"(peer(smem0 + (uint32_t)(row * (KN + 4) + j) * 4, rk)));
    };
    if (COMP && s.cluster_size <= kFewSlices) {
      // sums and compensations, all on their way at a time, the rounding of each addition kept with the latter
      float w[kFewSlices][4], c[kFewSlices][4], rest[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (uint32_t rk = 0; rk < kFewSlices; ++rk)
        if (rk < s.cluster_size) {
          slice(rr, rk, w[rk]);
          slice(kUmmaTile + rr, rk, c[rk]);
        }
#pragma unroll
      for (uint32_t rk = 0; rk < kFewSlices; ++rk)
        if (rk < s.cluster_size) {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float t = v[e] + w[rk][e], b = t - v[e];
            rest[e] += ((v[e] - (t - b)) + (w[rk][e] - b)) - c[rk][e];
            v[e] = t;
          }
        }
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] += rest[e];
    } else {
      // up to eight slices of the sum in 64 bits: in fp32 their additions alone would err by 4e-8
      double z[4] = {0.0, 0.0, 0.0, 0.0};
      for (uint32_t rk = 0; rk < s.cluster_size; ++rk) {
        float w[4];
        slice(rr, rk, w);
        z[0] += w[0]; z[1] += w[1]; z[2] += w[2]; z[3] += w[3];
        if (FLAGS) {
          uint32_t m0, m1, m2, m3, f;
          asm volatile("ld.shared::cluster.v4.u32 {%0,%1,%2,%3}, [%4];\n"
                       : "=r"(m0), "=r"(m1), "=r"(m2), "=r"(m3) : "r"(peer(u_largest_addr + j * 4, rk)));
          largest[0] = max(largest[0], m0); largest[1] = max(largest[1], m1);
          largest[2] = max(largest[2], m2); largest[3] = max(largest[3], m3);
          asm volatile("ld.shared::cluster.u8 %0, [%1];\n" : "=r"(f) : "r"(peer(row_flags_addr + rr, rk)));
          bad_row |= f;
        }
      }
      v[0] = (float)z[0]; v[1] = (float)z[1]; v[2] = (float)z[2]; v[3] = (float)z[3];
    }
    store_coords4<T>(a, t, s.j_lo() + j, s.j_end(), v);
    if (bad_row != 0 || !sums_stand(v, FLAGS && sizeof(T) == 4 ? largest : nullptr)) store_plain_coords4<T>(a, t, s.j_lo() + j, s.j_end());
    if (a.wire_ids && j == 0 && !s.lower()) static_cast<int32_t *>(a.zout)[t * a.ldzout + a.k] = a.shift.ids[t];
  }
  // nobody leaves while its sums can still be read
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

template <typename T, int KN, int NSLOT, bool CAREFUL>
__global__ void __launch_bounds__((SplitProjectConfig<T, KN, NSLOT, CAREFUL>::kThreads), 1) codec_split_project_kernel(const SplitProjectArgs a) {
  using Cfg = SplitProjectConfig<T, KN, NSLOT, CAREFUL>;
  constexpr int NX = Cfg::kNX, NU = Cfg::kNU, S = Cfg::kStages, RD = Cfg::kRaw, G = Cfg::kChain, NB = Cfg::kBufs;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  const SplitSchedule sched(a, Cfg::kCols);
  const int st_lo = sched.st_lo, nloc = sched.nloc;
  const int steps = sched.my_tiles * nloc;

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
      mbar_init(empty_bar(s), Cfg::kIssuers);
      mbar_init(acc_full_bar(s), Cfg::kIssuers);
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

  if (warp >= kSplitRowWarps) {
    // ------------------------------------------------------------------------- MMA issuers
    if (lane == 0) {
      // A: K-major rows of kRowBytes, 8-row groups 8 kRowBytes apart, one part after the other.  B: MN-major,
      // 64-coordinate groups kGroupBytes apart, 8-row groups 1024 bytes apart.
      constexpr uint32_t kLayoutA = Cfg::kF32 ? 4 : 2;       // 64- or 128-byte swizzle
      constexpr uint32_t id1 = umma_idesc(KN, false), id2 = umma_idesc(2 * KN, false);
      constexpr uint32_t kPart = Cfg::kPartBytes >> 4;                             // next part of A
      // where the parts of B start (see b_part)
      constexpr uint32_t kGroup = Cfg::kGroupBytes >> 4;
      constexpr uint32_t kBh = KN == 32 && NU == 3 ? kGroup : 0, kBm = KN == 32 ? 0 : kGroup;
      const bool first = warp == kSplitRowWarps, lead = first || Cfg::kIssuers == 1, small = !first || Cfg::kIssuers == 1;
      int slot = 0, st = 0, in_chain = 0, chain = 0;
      uint32_t parity = 0;
      for (int step = 0; step < steps; ++step) {
        const int buf = chain % NB;
        if (in_chain == 0 && !dead && !mbar_wait(acc_empty_bar(buf), (uint32_t)(((chain / NB) & 1) ^ 1))) timed_out();
        if (!dead && !mbar_wait(full_bar(slot), parity)) timed_out();
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const uint32_t base = smem0 + (uint32_t)slot * Cfg::kStageBytes;
        const uint32_t D = tmem_base + (uint32_t)buf * Cfg::kDCols, L0 = D + Cfg::kHi * KN, L1 = L0 + KN;
        const uint64_t ad = umma_desc(base, 16, 8 * Cfg::kRowBytes, kLayoutA);
        const uint64_t bd = umma_desc(base + Cfg::kABytes, Cfg::kGroupBytes, 1024, 2);
#pragma unroll
        for (int j = 0; j < Cfg::kCols / 16; ++j) {
          const uint64_t A = ad + j * 2, B = bd + j * 128;   // 32 bytes of an A row; 16 rows of B
          const int ks = in_chain * (Cfg::kCols / 16) + j;   // K step of the chain
          const uint32_t more = ks > 0 ? 1u : 0u;
          // an accumulator belongs to one thread: its MMAs keep their order
          if (NX == 1 && (Cfg::kHi % 2 != 0 ? ks % Cfg::kHi != 0 : j % 2 != 0) ? small : lead)
            umma_bf16(D + (uint32_t)(ks % Cfg::kHi) * KN, A, B + kBh, id1, ks >= Cfg::kHi ? 1u : 0u);
          if (NX == 1 || !small) continue;
          if (NU == 1) {
            umma_bf16(L0, A + kPart, B, id1, more);
            umma_bf16(L0, A + 2 * kPart, B, id1, 1u);
          } else {
            umma_bf16(L0, A, B + kBm, id2, more);            // m and l side by side
            if (KN == 64) {
              umma_bf16(L0, A + kPart, B, id2, 1u);          // h and m
            } else {
              umma_bf16(L0, A + kPart, B + kBh, id1, 1u);
              umma_bf16(L1, A + kPart, B + kBm, id1, 1u);
            }
            umma_bf16(L1, A + 2 * kPart, B + kBh, id1, 1u);
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
    const int u_row = tid / (KN / 2), u_col = 2 * (tid % (KN / 2)), u_valid = max(sched.rank() - u_col, 0);
    const int64_t u_step = kURows * a.ldu;
    const bool vec_u = a.vec_u != 0;
    const T *U = static_cast<const T *>(a.U) + sched.j_lo();
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
    int chain = 0, fin_tile = 0;             // chains complete so far, tiles finished
    bool fresh = true;                       // the next chain is a tile's first
    // Adds chain c, of `chain_steps` steps, to the sums, with compensation: over 4096 columns of coherent rows 64 plain
    // additions err by 1.2e-7, these by 3e-8.  `last`: it completes a tile.
    auto take_chain = [&](int c, int chain_steps, bool last) {
      const int buf = c % NB;
      const int written = chain_steps * (Cfg::kCols / 16);   // leading accumulators that the chain has written
      if (!dead && !mbar_wait(acc_full_bar(buf), (uint32_t)((c / NB) & 1))) timed_out();
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      if (sum_col < a.k_half) {
        const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16) + sum_col;
        const uint32_t taddr = lane_addr + (uint32_t)buf * Cfg::kDCols, caddr = lane_addr + Cfg::kCompCol;
        asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");   // the compensation of the chain before
        constexpr int H0 = Cfg::kHi / 2, H1 = Cfg::kHi - H0;
#pragma unroll
        for (int i = 0; i < Cfg::kSums; i += 8) {
          if constexpr (CAREFUL) {
            uint32_t comp[8], v[8];
            tmem_ld8(caddr + i, comp);
#pragma unroll
            for (int q = 0; q < Cfg::kHi + Cfg::kLow; ++q) {
              if (q >= written && q < Cfg::kHi) continue;
              tmem_ld8(taddr + q * KN + i, v);
              asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
              for (int e = 0; e < 8; e += 2) {
                float c0 = q == 0 && fresh ? 0.f : __uint_as_float(comp[e]), c1 = q == 0 && fresh ? 0.f : __uint_as_float(comp[e + 1]);
                add_compensated2(sum[i + e], sum[i + e + 1], c0, c1, __uint_as_float(v[e]), __uint_as_float(v[e + 1]));
                comp[e] = __float_as_uint(c0), comp[e + 1] = __float_as_uint(c1);
              }
            }
            tmem_st8(caddr + i, comp);
          } else {
            // One half of the leading sums, then the other with the small ones: additions at half the sum's size.
            float h[2][8];
            uint32_t v[H1][8], w[Cfg::kLow + 1][8];
#pragma unroll
            for (int part2 = 0; part2 < 2; ++part2) {
#pragma unroll
              for (int q = 0; q < (part2 == 0 ? H0 : H1); ++q) {
                if (part2 * H0 + q < Cfg::kCols / 16 || part2 * H0 + q < written) {
                  tmem_ld8(taddr + (part2 * H0 + q) * KN + i, v[q]);
                } else {
#pragma unroll
                  for (int e = 0; e < 8; ++e) v[q][e] = 0;
                }
              }
              if (part2 == 1) {
#pragma unroll
                for (int q = 0; q < Cfg::kLow; ++q) tmem_ld8(taddr + (Cfg::kHi + q) * KN + i, w[q]);
                tmem_ld8(caddr + i, w[Cfg::kLow]);
              }
              asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
              for (int e = 0; e < 8; e += 2) {
                float x0 = __uint_as_float(v[0][e]), x1 = __uint_as_float(v[0][e + 1]);
#pragma unroll
                for (int q = 1; q < (part2 == 0 ? H0 : H1); ++q) add2(x0, x1, __uint_as_float(v[q][e]), __uint_as_float(v[q][e + 1]));
                h[part2][e] = x0, h[part2][e + 1] = x1;
              }
            }
            uint32_t comp[8];
#pragma unroll
            for (int e = 0; e < 8; e += 2) {
              float *const h0 = h[0], *const g = h[1];
              if (Cfg::kLow > 0) {
                float l0 = __uint_as_float(w[0][e]), l1 = __uint_as_float(w[0][e + 1]);
                if (Cfg::kLow > 1) add2(l0, l1, __uint_as_float(w[Cfg::kLow - 1][e]), __uint_as_float(w[Cfg::kLow - 1][e + 1]));
                add2(g[e], g[e + 1], l0, l1);
              }
              add2(h0[e], h0[e + 1], g[e], g[e + 1]);
              float c0 = fresh ? 0.f : __uint_as_float(w[Cfg::kLow][e]), c1 = fresh ? 0.f : __uint_as_float(w[Cfg::kLow][e + 1]);
              add_compensated2(sum[i + e], sum[i + e + 1], c0, c1, h0[e], h0[e + 1]);
              comp[e] = __float_as_uint(c0), comp[e + 1] = __float_as_uint(c1);
            }
            tmem_st8(caddr + i, comp);
          }
        }
      }
      fresh = last;
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty_bar(buf));
      if (last) {
        const int64_t t = sched.tile(fin_tile) * kUmmaTile + sum_row;
        if (sched.cluster_size == 1) {
          if (t < a.n) {
            uint32_t bad = NX == 3 && row_flags[(fin_tile & 3) * kUmmaTile + sum_row] != 0 ? ~0u : 0u;
#pragma unroll
            for (int i = 0; i < Cfg::kSums; i += 4) {
              const float v[4] = {sum[i], sum[i + 1], sum[i + 2], sum[i + 3]};
              store_coords4<T>(a, t, sched.j_lo() + sum_col + i, sched.j_end(), v);
              if (!sums_stand(v, NU == 3 ? u_largest + sum_col + i : nullptr)) bad |= 1u << (i / 4);
            }
            if (bad != 0) {
#pragma unroll 1
              for (int i = 0; i < Cfg::kSums / 4 && sum_col + 4 * i < sched.rank(); ++i)
                if (bad >> i & 1) store_plain_coords4<T>(a, t, sched.j_lo() + sum_col + 4 * i, sched.j_end());
            }
            if (a.wire_ids && part == 0 && !sched.lower()) static_cast<int32_t *>(a.zout)[t * a.ldzout + a.k] = a.shift.ids[t];
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
        if (ld_st == 0) row_pointers(sched.tile(ld_tile));
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
    int prev_steps = 0;
    float u_max[2] = {0.f, 0.f}, row_max[2] = {0.f, 0.f};
    const uint32_t a_off = Cfg::kF32 ? row * 64 + (((unit >> 1) ^ ((row >> 1) & 3)) << 4) + (unit & 1) * 8
                                     : row * 128 + ((unit ^ (row & 7)) << 4);   // + 64 rows: the second piece
    for (int step = 0; step < steps; ++step) {
      cp_async_wait<RD - 2>();
      // Into the slot read in the step before: at once where the next step is the only one ahead (bf16, three operands or
      // more: 152 -> 141 us for X, R and E rows of 12288 x 5120), else after this step's work (fp32 E and P: 53 against 55).
      if (RD == 2) advance_rows(step + RD - 1 < steps);
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
          const int n = Cfg::b_part(s) * KN + u_col;
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
      if (RD > 2) advance_rows(step + RD - 1 < steps);
      if (++slot == S) {
        slot = 0;
        parity ^= 1u;
      }
      if (++rslot == RD) rslot = 0;
      st = next_st;
      if (st == 0) ++tile;
      // With two sets the chain before the one just filled; with one the chain before this one, as soon as this
      // one's first step is filled, because its MMAs wait for it.
      if (NB == 1 && in_chain == 0 && chain > 0) take_chain(chain - 1, prev_steps, prev_last);
      if (++in_chain == G || st == 0) {
        if (NB == 2 && chain > 0) take_chain(chain - 1, prev_steps, prev_last);
        prev_last = st == 0;
        prev_steps = in_chain;
        in_chain = 0;
        ++chain;
      }
    }
    take_chain(chain - 1, prev_steps, true);
    cp_async_wait<0>();
    asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");   // before tensor memory is given back
  }

  if (sched.cluster_size > 1) {
    // Every accumulator has been read, so every stage is consumed and the rings can carry the sums.
    __syncthreads();
    if (warp < kSplitRowWarps) {
      const uint32_t dst = smem0 + (uint32_t)(sum_row * Cfg::kSumPitch + sum_col) * 4;
#pragma unroll
      for (int c = 0; c < Cfg::kSums; c += 4)
        st_shared_v4(dst + c * 4, __float_as_uint(sum[c]), __float_as_uint(sum[c + 1]), __float_as_uint(sum[c + 2]),
                     __float_as_uint(sum[c + 3]));
    }
    finish_slices<T, KN, Cfg::kThreads, NX == 3, false>(a, sched, smem0, smem_u32(u_largest), smem_u32(const_cast<unsigned char *>(row_flags)));
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
