// tcgen05 / TMA contraction over TOKENS (bf16 in, fp32 out, sm_100a), k <= 128:
//     G [m x k] = H^T C = sum_t H[t, :]^T C[t, :]          H: [n x m], C: [n x k]
// the weight-factor gradient of the reparameterized SSN (Eq. reparam and the chain rule quoted
// with it: dL/dZw = (dL/dW) U_k = H^T (dY U_k); C = dY U_k comes from the projection kernel).
//
// A work unit is a block of 128 columns of H (the M of the MMA) over a range of tokens (the K):
// per stage of 64 tokens the block arrives as an MN-major A operand (two TMA boxes of 64 tokens x
// 64 columns, as stored) and the 64 rows of C as an MN-major B operand (as stored); four
// tcgen05.mma (M=128, N=k rounded up to 16, K=16) accumulate in TMEM.
//
// One CTA per SM takes an equal, contiguous range of all (column block, stage) pairs, so it streams without a
// pause and ends with the others.  At the end of a block, and after kTokensChain stages of one, the fp32 partial
// sums are added to the (zeroed) output with red.global, from one of two accumulators while the next stages
// go on in the other.  A block summed at once is stored.  (As a grid of one CTA per block and token range, ten
// waves of 20 stages for 14336 columns: 170 us with the projection in front of it, 16384 tokens, rank 40; like
// this 131 us.  CTAs that walk the blocks in step, so that together they read whole rows of H: 142 us.)
//
//   warp 0  producer     warp 1  MMA issuer, owns the TMEM allocation     warps 2-5  epilogue
// Every wait is bounded; a wait that runs out sets the status word (when given) and the kernel
// still runs to its end.
#pragma once

#include "codec_umma.cuh"

namespace ssn {

constexpr int kTokensThreads = 192;
// Stages summed in one accumulator before its sums leave it: the tensor cores truncate every addition, so
// that a chain of 80 MMAs is biased by 5e-7 and one over a CTA's whole range would be by 5e-6.
constexpr int kTokensChain = 20;

struct TokensArgs {
  float *out;        // [m x k] fp32, leading dimension ldout; zeroed by the caller unless every CTA has whole blocks
  int64_t ldout;
  int64_t n;         // tokens
  int32_t m, k;
  int32_t vec;       // rows of out take 16 bytes at a time
  int32_t *dev_status;
};

struct UmmaTokensMaps {
  CUtensorMap h;             // H: boxes of 64 token rows x 64 columns
  CUtensorMap c, c_wide;     // C: boxes of 64 token rows x 64 coordinates (c_wide: see UmmaMaps)
};

// Four neighbouring sums.  The lanes of a warp hold rows, so that every access is a sector per lane: one for four
// sums instead of one each.
__device__ __forceinline__ void store_or_add4(float *p, uint32_t a, uint32_t b, uint32_t c, uint32_t d, bool store) {
  if (store)
    asm volatile("st.global.v4.b32 [%0], {%1,%2,%3,%4};\n" ::"l"(p), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
  else
    asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1,%2,%3,%4};\n"
                 ::"l"(p), "f"(__uint_as_float(a)), "f"(__uint_as_float(b)), "f"(__uint_as_float(c)), "f"(__uint_as_float(d)) : "memory");
}

template <int NTP>
struct UmmaTokensConfig {
  static_assert(NTP % 2 == 0 && NTP >= 2 && NTP <= 16, "N = 8*NTP must be a multiple of 16 up to 128");
  static constexpr int kN = NTP * 8;
  static constexpr int kKG = kN <= 64 ? 1 : 2;
  static constexpr int kABytes = 2 * kUmmaCols * 128;           // 64 tokens x 128 columns, two 64-column groups
  static constexpr int kBGroupBytes = kUmmaCols * 128;          // 64 tokens x 64 coordinates
  static constexpr int kStageBytes = kABytes + kKG * kBGroupBytes;
  static constexpr int kMaxSmem = 227 * 1024;
  static constexpr int kFit = (kMaxSmem - 1024 - 512) / kStageBytes;
  static constexpr int kStagesN = kFit < 8 ? kFit : 8;
  static constexpr int kAccCols = kN <= 32 ? 32 : (kN <= 64 ? 64 : 128);
  static constexpr int kTmemCols = 2 * kAccCols;
  static constexpr int kSmemBytes = 1024 + kStagesN * kStageBytes + (2 * kStagesN + 4) * 8 + 16;
};

template <int NTP>
__global__ void __launch_bounds__(kTokensThreads, 1)
codec_umma_tokens_kernel(const TokensArgs a, const __grid_constant__ UmmaTokensMaps maps) {
  using Cfg = UmmaTokensConfig<NTP>;
  constexpr int S = Cfg::kStagesN;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

  const int64_t nstage_all = (a.n + kUmmaCols - 1) / kUmmaCols;
  const int64_t units = nstage_all * ((a.m + kUmmaTile - 1) / kUmmaTile);
  const int64_t u_lo = (units * blockIdx.x) / gridDim.x, u_hi = (units * (blockIdx.x + 1)) / gridDim.x;
  // the chains of this CTA in order: (block, first stage, end stage)
  int64_t at = u_lo;
  auto next_segment = [&](int &blk, int64_t &st_lo, int64_t &st_hi) {
    if (at >= u_hi) return false;
    blk = (int)(at / nstage_all);
    st_lo = at - blk * nstage_all;
    st_hi = st_lo + min(min(u_hi - at, nstage_all - st_lo), (int64_t)kTokensChain);
    at += st_hi - st_lo;
    return true;
  };

  const uint32_t smem0 = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t bars = smem0 + S * Cfg::kStageBytes;
  auto full_bar = [&](int s) { return bars + s * 8; };
  auto empty_bar = [&](int s) { return bars + (S + s) * 8; };
  auto acc_full_bar = [&](int b) { return bars + (2 * S + b) * 8; };
  auto acc_empty_bar = [&](int b) { return bars + (2 * S + 2 + b) * 8; };
  const uint32_t tmem_slot = bars + (2 * S + 4) * 8;
  volatile uint32_t *tmem_slot_ptr =
      reinterpret_cast<volatile uint32_t *>(smem_raw + (tmem_slot - smem_u32(smem_raw)));

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(acc_full_bar(b), 1);
      mbar_init(acc_empty_bar(b), 4);
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
  int blk;
  int64_t st_lo, st_hi;
  bool dead = false;
  auto timed_out = [&]() {
    dead = true;
    if (a.dev_status) atomicOr(a.dev_status, SSN_DEV_TIMEOUT);
  };

  if (warp == 0) {
    // ------------------------------------------------------------------------- producer
    const uint64_t stream_in = l2_policy_evict_first();   // H is read once; C comes back for every column block
    int slot = 0;
    uint32_t parity = 1;
    while (next_segment(blk, st_lo, st_hi)) {
      const int col0 = blk * kUmmaTile;
      for (int64_t st = st_lo; st < st_hi; ++st) {
        if (!dead && !mbar_wait(empty_bar(slot), parity)) timed_out();
        const uint32_t base = smem0 + (uint32_t)slot * Cfg::kStageBytes;
        if (lane == 0) {
          const int tok0 = (int)(st * kUmmaCols);
          mbar_expect_tx(full_bar(slot), Cfg::kStageBytes);
          tma_load_2d_hint(base, &maps.h, full_bar(slot), col0, tok0, stream_in);
          tma_load_2d_hint(base + Cfg::kABytes / 2, &maps.h, full_bar(slot), col0 + 64, tok0, stream_in);
          // the last box of C would read past its buffer through the wide map
#pragma unroll
          for (int g = 0; g < Cfg::kKG; ++g)
            tma_load_2d(base + Cfg::kABytes + g * Cfg::kBGroupBytes, st == nstage_all - 1 ? &maps.c : &maps.c_wide,
                        full_bar(slot), g * 64, tok0);
        }
        __syncwarp();
        if (++slot == S) {
          slot = 0;
          parity ^= 1u;
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      // both operands MN-major (bits 15 and 16)
      constexpr uint32_t idesc = umma_idesc(Cfg::kN, false) | (1u << 15);
      const uint64_t adesc0 = umma_desc(0, Cfg::kABytes / 2, 1024, 2);       // two 64-column groups 8 KB apart
      const uint64_t bdesc0 = umma_desc(0, Cfg::kBGroupBytes, 1024, 2);
      int slot = 0, seg = 0;
      uint32_t parity = 0;
      for (; next_segment(blk, st_lo, st_hi); ++seg) {
        const int buf = seg & 1;
        const uint32_t acc = tmem_base + (uint32_t)buf * Cfg::kAccCols;
        if (!dead && !mbar_wait(acc_empty_bar(buf), (uint32_t)(((seg >> 1) & 1) ^ 1))) timed_out();
        for (int64_t st = st_lo; st < st_hi; ++st) {
          if (!dead && !mbar_wait(full_bar(slot), parity)) timed_out();
          asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
          const uint32_t base = smem0 + (uint32_t)slot * Cfg::kStageBytes;
          const uint64_t ad = adesc0 + umma_desc_addr(base), bd = bdesc0 + umma_desc_addr(base + Cfg::kABytes);
#pragma unroll
          for (int j = 0; j < kUmmaCols / 16; ++j)   // a K step: 16 token rows = 2048 bytes of either tile
            umma_bf16(acc, ad + j * 128, bd + j * 128, idesc, (st > st_lo || j > 0) ? 1u : 0u);
          umma_commit(empty_bar(slot));
          if (st == st_hi - 1) umma_commit(acc_full_bar(buf));
          if (++slot == S) {
            slot = 0;
            parity ^= 1u;
          }
        }
      }
    }
  } else {
    // ------------------------------------------------------------------------- epilogue
    const int quarter = warp & 3;   // TMEM lanes 32*quarter .. +31: columns col0 + 32*quarter + lane of H
    for (int seg = 0; next_segment(blk, st_lo, st_hi); ++seg) {
      const int buf = seg & 1;
      if (!dead && !mbar_wait(acc_full_bar(buf), (uint32_t)((seg >> 1) & 1))) timed_out();
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      const bool whole = st_lo == 0 && st_hi == nstage_all;
      const int row = blk * kUmmaTile + quarter * 32 + lane;          // row of the output = column of H
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)buf * Cfg::kAccCols;
#pragma unroll
      for (int q = 0; q < Cfg::kN / 16; ++q) {
        uint32_t v[16];
        tmem_ld16(taddr + q * 16, v);
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
        if (row < a.m) {
          float *orow = a.out + (int64_t)row * a.ldout;
#pragma unroll
          for (int i = 0; i < 16; i += 4) {
            const int col = q * 16 + i;
            if (a.vec) {
              if (col < a.k) store_or_add4(orow + col, v[i], v[i + 1], v[i + 2], v[i + 3], whole);
            } else {
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                if (col + e < a.k) {
                  if (whole) orow[col + e] = __uint_as_float(v[i + e]);
                  else atomicAdd(orow + col + e, __uint_as_float(v[i + e]));
                }
              }
            }
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty_bar(buf));
    }
  }

  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base),
                 "r"(Cfg::kTmemCols) : "memory");
  }
}

}  // namespace ssn
