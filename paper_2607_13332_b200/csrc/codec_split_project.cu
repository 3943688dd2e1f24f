// Launchers of the split-operand projection kernel (codec_split_project.cuh) and of its form for bf16 rows as they are
// (codec_plain_project.cuh).
#include "codec_split_project.cuh"

#include <algorithm>

#include "codec_mma_launch.h"
#include "codec_plain_project.cuh"
#include "codec_split.h"
#include "codec_tensor_maps.h"

namespace ssn {
namespace {

// CTAs per tile: the c whose waves of tiles, each 1 / c of a tile's time plus a fixed cost, end first.  The fixed
// cost of a wave (set-up, first loads, exchange of the sums) is about that of kWaveStages stages of 64 columns.
// Large batches keep whole tiles, which one persistent CTA runs back to back.  43 tiles of 64 stages: two CTAs per
// tile 110 us, three 80 us.
constexpr int kWaveStages = 5;
// clusters of 1 .. 8 CTAs of one per SM that a B200's 148 SMs run at once (cudaOccupancyMaxActiveClusters)
constexpr int kClustersAtOnce[8] = {148, 74, 45, 33, 26, 22, 15, 15};
int cluster_of(int64_t ntiles, int nst, int sms) {
  int best = 1;
  double best_cost = (double)((ntiles + sms - 1) / sms) * nst + kWaveStages;
  for (int c = 2; c <= 8 && c <= nst; ++c) {
    const int at_once = kClustersAtOnce[c - 1] * sms / 148;
    if (at_once < 1) break;
    const double cost = (double)((ntiles + at_once - 1) / at_once) * ((double)((nst + c - 1) / c) + kWaveStages);
    if (cost < 0.97 * best_cost) {
      best = c;
      best_cost = cost;
    }
  }
  return best;
}

int64_t units_of(const SplitProjectArgs &a) { return (a.n + kUmmaTile - 1) / kUmmaTile * a.halves; }   // tiles, or halves of them

// Launches either kernel with clusters of c, or with single CTAs on a device that cannot co-schedule them.
template <typename Kernel, typename... Args>
cudaError_t launch_slices(Kernel kernel, int threads, int smem, int variant, const SplitProjectArgs &a, int c, int sms,
                          cudaStream_t stream, Args... args) {
  const int64_t units = units_of(a);
  // whole tiles: as many CTAs for either half
  const int64_t single = units < sms ? units : (sms > 1 ? sms - sms % a.halves : a.halves), grid = c > 1 ? units * c : single;
  cudaError_t e = launch_dependent(kernel, (unsigned)grid, threads, smem, stream, c, a, args...);
  if (e != cudaSuccess && c > 1) {
    cudaGetLastError();
    e = launch_dependent(kernel, (unsigned)single, threads, smem, stream, 1, a, args...);
  }
  note_kernel(SSN_KERNEL_SPLIT_PROJECT, variant | (a.has_e ? SSN_KVAR_E : 0) | (a.has_p ? SSN_KVAR_P : 0) |
                                            (a.halves > 1 ? SSN_KVAR_WIDE : 0) | (c > 1 ? SSN_KVAR_ALT : 0));
  return e;
}

template <typename T, int KN, int NSLOT, bool CAREFUL>
cudaError_t launch_one(const SplitProjectArgs &a, int c, int sms, cudaStream_t stream) {
  using Cfg = SplitProjectConfig<T, KN, NSLOT, CAREFUL>;
  auto kernel = codec_split_project_kernel<T, KN, NSLOT, CAREFUL>;
  static std::atomic<uint64_t> configured{0};
  const cudaError_t e = allow_dynamic_smem(kernel, Cfg::kSmemBytes, configured);
  if (e != cudaSuccess) return e;
  return launch_slices(kernel, Cfg::kThreads, Cfg::kSmemBytes, 0, a, c, sms, stream);
}

// The plain kernel's CTAs per tile, by a rough cost that orders the choices: a stage takes a CTA kPlainStageNs, or the time of
// the 16 KB that every CTA at work takes from HBM, whichever is longer; a wave of clusters kPlainWaveNs besides.  Single CTAs are
// persistent.  us with 1, 2, 3, ... CTAs, the chosen number in brackets: 100 x 2048, rank 27 19.1 14.2 12.2 11.6 10.7 [10.7] 10.6 10.5;
// 3000 x 4096, rank 27 31.7 20.9 16.7 [15.4] 14.3 24.3; 9000 x 4096, rank 51 53.7 [36.1] 52.1 66.9; 5000 x 4096, rank 51 53.0 33.1 [27.3]
// 45.3; 12288 x 5120, rank 51 [63.5] 76.2 84.2; 20000 x 2048, rank 51 [59.8] 68.4 75.0; it errs at 20000 x 4096, rank 27 58.7 62.1 [66.4].
constexpr double kPlainStageNs = 260, kPlainHbmNs = 2.65, kPlainWaveNs = 4000;
int plain_cluster_of(const SplitProjectArgs &a, int nst, int sms) {
  const int64_t units = units_of(a);
  auto stage_ns = [&](int64_t ctas) { return std::max(kPlainStageNs, kPlainHbmNs * (double)ctas / a.halves); };
  int best = 1;
  double best_ns = kPlainWaveNs + (double)((units + sms - 1) / sms) * nst * stage_ns(units < sms ? units : sms);
  for (int c = 2; c <= 8 && c <= nst; ++c) {
    const int64_t at_once = kClustersAtOnce[c - 1] * sms / 148;
    if (at_once < 1) break;
    const double ns = (double)((units + at_once - 1) / at_once) *
                      (kPlainWaveNs + (double)((nst + c - 1) / c) * stage_ns((units < at_once ? units : at_once) * c));
    if (ns < 0.97 * best_ns) {
      best = c;
      best_ns = ns;
    }
  }
  return best;
}

template <int KN, bool CAREFUL>
cudaError_t launch_plain(const SplitProjectArgs &a, const CUtensorMap &x, int c, int sms, cudaStream_t stream) {
  auto kernel = codec_plain_project_kernel<KN, CAREFUL>;
  constexpr int smem = PlainProjectConfig<KN>::kSmemBytes;
  static std::atomic<uint64_t> configured{0};
  const cudaError_t e = allow_dynamic_smem(kernel, smem, configured);
  if (e != cudaSuccess) return e;
  return launch_slices(kernel, kPlainThreads, smem, SSN_KVAR_PLAIN, a, c, sms, stream, x);
}

cudaError_t launch_plain_rank(const SplitProjectArgs &a, const CUtensorMap &x, int sms, cudaStream_t s) {
  const int nst = (a.d + kUmmaCols - 1) / kUmmaCols, c = plain_cluster_of(a, nst, sms);
  const bool careful = (nst + c - 1) / c * kUmmaCols < kSplitCarefulColsPlain;
  if (a.k <= 32) return careful ? launch_plain<32, true>(a, x, c, sms, s) : launch_plain<32, false>(a, x, c, sms, s);
  return careful ? launch_plain<64, true>(a, x, c, sms, s) : launch_plain<64, false>(a, x, c, sms, s);
}

template <typename T, int NSLOT>
cudaError_t launch_rank(const SplitProjectArgs &a, int sms, cudaStream_t s) {
  const int nst = (a.d + 63) / 64, c = cluster_of(units_of(a), nst, sms);
  constexpr int careful = sizeof(T) == 2 && NSLOT == 0 ? kSplitCarefulColsPlain : kSplitCarefulCols;
  if ((nst + c - 1) / c * 64 < careful) return launch_one<T, 64, NSLOT, true>(a, c, sms, s);
  if (a.k <= 32) return launch_one<T, 32, NSLOT, false>(a, c, sms, s);
  return launch_one<T, 64, NSLOT, false>(a, c, sms, s);
}

template <typename T>
cudaError_t launch_slots(const SplitProjectArgs &a, int slots, int sms, cudaStream_t s) {
  if (slots == 0) return launch_rank<T, 0>(a, sms, s);
  if (slots == 1) return launch_rank<T, 1>(a, sms, s);
  if (slots == 2) return launch_rank<T, 2>(a, sms, s);
  return launch_rank<T, 3>(a, sms, s);
}

// Where the plain kernel is the faster one, us, split -> plain.  One stage is too little for its set-up, and above rank 32 the
// first and last rows of the basis, fetched half a word at a time, cost it 3 us that wide rows, or many, have to earn.
//   rank 27: 16000 x 64 9.5 -> 10.2 (rank 8 7.5 -> 8.3, 20000 rows 9.1 -> 8.8), 40000 x 64 15.4 -> 14.8, 100 x 72 9.1 -> 8.9, 9000 x 128 9.8 -> 10.1, 20000 x 128 15.2 -> 12.2,
//            3000 x 256 9.1 -> 9.4, 6000 x 256 11.3 -> 10.1, 100 x 640 10.5 -> 9.5, 9000 x 4096 41 -> 23; rank 32, the most of one
//            group, 1500 x 256 9.0 -> 9.6
//   rank 51: 9000 x 1024 20.4 -> 21.5, 16000 x 1024 31.9 -> 27.3, 100 x 2048 14.7 -> 14.9, 3000 x 2048 18.7 -> 18.9, 5000 x 2048
//            23.9 -> 20.8, 1500 x 2304 16.9 -> 15.2, 100 x 4096 18.4 -> 17.0; rank 64 loses up to 2 us more
//   rank 99: 2048 x 2048 19.2 -> 22.2, 3000 x 2048 29.9 -> 26.5, 2048 x 3072 24.6 -> 24.6, 1500 x 4096 26.2 -> 23.8
bool plain_pays(const SplitProjectArgs &a) {
  const double size = (double)a.n * a.d;
  if (a.k <= 32) return a.d > kUmmaCols || a.n >= 20000;
  if (a.d >= 2048 && (a.k <= 64 || size >= 6e6)) return true;
  return a.d >= 1024 && size >= 16000. * 1024;
}

bool rows16(const void *p, int64_t ld, int esz) {
  return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && (ld * esz) % 16 == 0;
}

}  // namespace

cudaError_t launch_codec_split_project(const TokenArgs &a, int32_t dtype, int sm_count, cudaStream_t stream) {
  if (a.src == nullptr || a.zout == nullptr || a.dst != nullptr || a.rowsumsq != nullptr || a.k > kSplitMaxRank ||
      a.U2 != nullptr || a.n > 0x7fffffffLL || sm_count < 1)
    return cudaErrorNotSupported;
  const int esz = dtype == SSN_F32 ? 4 : 2;
  SplitProjectArgs p{};
  p.src = a.src;
  p.src2 = a.src2;
  p.U = a.U;
  p.zout = a.zout;
  p.lds = a.lds;
  p.lds2 = a.lds2;
  p.ldu = a.ldu;
  p.ldzout = a.ldzout;
  p.n = a.n;
  p.d = a.d;
  p.k = a.k;
  p.halves = a.k > 64 ? 2 : 1;
  p.k_half = a.k > 64 ? (a.k + 31) / 32 * 16 : a.k;
  p.wire = a.wire;
  p.wire_ids = a.wire_ids;
  p.shift = a.shift;
  p.has_e = a.sub_shift && a.shift.E != nullptr;
  p.has_p = a.sub_shift && a.shift.P != nullptr;
  p.vec_rows = (int64_t)a.d * esz % 16 == 0 && (int64_t)a.d * esz <= kZeroRowBytes && rows16(a.src, a.lds, esz) &&
               (a.src2 == nullptr || rows16(a.src2, a.lds2, esz)) &&
               (!p.has_e || rows16(a.shift.E, a.shift.lde, esz)) && (!p.has_p || rows16(a.shift.P, a.shift.ldp, esz));
  p.vec_u = pairs_aligned(a.U, a.ldu, esz);
  // four coordinates are 16 bytes of words or 8 bytes of bf16
  p.vec_out = (a.ldzout & 3) == 0 && (reinterpret_cast<uintptr_t>(a.zout) & (a.wire || dtype == SSN_F32 ? 15 : 7)) == 0;
  const int slots = (a.src2 != nullptr) + p.has_e + p.has_p;
  if (dtype == SSN_BF16 && slots == 0 && rows16(a.src, a.lds, esz) && plain_pays(p)) {   // rows that TMA can fetch, and nothing to add
    CUtensorMap x;
    if (make_sw128_map(&x, a.src, a.n, a.d, a.lds, kUmmaTile))
      return launch_plain_rank(p, x, sm_count, stream);
  }
  return dtype == SSN_F32 ? launch_slots<float>(p, slots, sm_count, stream)
                          : launch_slots<__nv_bfloat16>(p, slots, sm_count, stream);
}

}  // namespace ssn
