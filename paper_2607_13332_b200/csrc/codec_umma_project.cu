// Launcher of the tcgen05 projection kernel (see codec_umma.cuh).
#include "codec_umma.cuh"
#include "codec_tensor_maps.h"
#include "codec_mma_launch.h"

namespace ssn {
namespace {

template <int NTP, bool HAS_E, int PMODE>
cudaError_t launch_umma_one(const MmaArgs &a, const UmmaMaps &maps, int sm_count, cudaStream_t stream) {
  auto kernel = codec_umma_project_kernel<NTP, HAS_E, PMODE>;
  constexpr int smem = UmmaProjectConfig<NTP, HAS_E, PMODE>::kSmemBytes;
  static std::atomic<uint64_t> configured{0};   // per instantiation, one bit per device
  {
    cudaError_t e = allow_dynamic_smem(kernel, smem, configured);
    if (e != cudaSuccess) return e;
  }
  note_kernel(SSN_KERNEL_UMMA_PROJECT, (HAS_E ? SSN_KVAR_E : 0) | (PMODE != kPNone ? SSN_KVAR_P : 0) |
                                           (NTP > 8 ? SSN_KVAR_WIDE : 0) | (a.pshare ? SSN_KVAR_ALT : 0));
  return launch_tile_pairs(kernel, UmmaProjectConfig<NTP, HAS_E, PMODE>::kThreads, smem, a, maps, sm_count, stream);
}

template <int NTP>
cudaError_t launch_umma_ntp(const MmaArgs &a, bool has_e, int pmode, const UmmaMaps &maps, int sm_count, cudaStream_t s) {
  if (pmode == kPGather)
    return has_e ? launch_umma_one<NTP, true, kPGather>(a, maps, sm_count, s)
                 : launch_umma_one<NTP, false, kPGather>(a, maps, sm_count, s);
  if (pmode == kPTma)
    return has_e ? launch_umma_one<NTP, true, kPTma>(a, maps, sm_count, s)
                 : launch_umma_one<NTP, false, kPTma>(a, maps, sm_count, s);
  return has_e ? launch_umma_one<NTP, true, kPNone>(a, maps, sm_count, s)
               : launch_umma_one<NTP, false, kPNone>(a, maps, sm_count, s);
}

}  // namespace

// Projection on tcgen05.  Returns cudaErrorNotSupported when the call should take the mma.sync
// kernel instead: small batches, k > 128, d not a multiple of 64, no tensor map.
cudaError_t launch_codec_umma_project(const MmaArgs &a, bool shift, int sm_count, cudaStream_t stream) {
  if ((a.zout == nullptr) == (a.zout32 == nullptr) || a.dst != nullptr || a.src == nullptr)
    return cudaErrorNotSupported;
  if (a.d % kUmmaCols != 0 || a.k > 128 || a.n < 4 * kUmmaTile || a.n > 0x7fffffffLL)
    return cudaErrorNotSupported;
  // a term with a prepared table is subtracted in the epilogue and needs no operand
  const bool has_e = shift && a.shift.E != nullptr && a.shift.EU == nullptr;
  const bool has_p = shift && a.shift.P != nullptr && a.shift.PU == nullptr;
  // positions given per token, wrapping inside a 128-token tile or past the table: the P rows are gathered
  const bool consecutive = a.shift.pos == nullptr && a.shift.seq_len % kUmmaTile == 0 && a.shift.seq_len <= a.shift.max_pos;
  const int pmode = !has_p ? kPNone : (consecutive ? kPTma : kPGather);
  if (pmode == kPGather) {
    // Wire rows stay on the split kernel, whose short chains keep their fp32 accuracy.
    if (a.zout32 != nullptr) return cudaErrorNotSupported;
    // Measured against the mma.sync kernels, E and P rows, us (theirs -> this one): up to 16 tokens per SM they
    // win at every width (rank 40: 2155 x 512 6.9 -> 11.3, 2155 x 2048 13.0 -> 16.7), above it this one does
    // (10007 x 256 22 -> 11, 10007 x 2048 51 -> 23) except on narrow rows in large batches (40000 x 256
    // 17.5 -> 22); ranks above 64 from 512 columns on (2155 x 512 13.8 -> 13.3, 2155 x 2048 45 -> 18.5).
    // Up to 32 tokens per SM small ranks keep theirs too (4096 tokens: rank 8, 512 columns 6.8 -> 11.0, 4096 columns
    // 20.6 -> 24.3; rank 16 7.7 -> 10.3, 19.6 -> 21.6; rank 40, 256 columns 8.4 -> 10.3, 2048 columns 17.1 -> 16.5).
    const bool narrow = a.d < 512;
    if (a.n <= 32 * (int64_t)sm_count && a.k <= 64 && (a.k <= 16 || narrow || (a.k <= 32 && a.d <= 1024))) return cudaErrorNotSupported;
    if (a.k > 64 ? narrow : a.n <= 16 * (int64_t)sm_count || (narrow && a.n > 128 * (int64_t)sm_count))
      return cudaErrorNotSupported;
  }
  const int ntp = 2 * ((a.k + 15) / 16);
  MmaArgs b = a;
  if (!shift) b.shift.EU = b.shift.PU = nullptr;
  // whole sequences of 128-position blocks: tiles of one block share their positional product
  b.pshare = has_e && pmode == kPTma && a.k <= 64 && a.n % a.shift.seq_len == 0 ? 1 : 0;
  UmmaMaps maps;
  if (!make_sw128_map(&maps.x, a.src, a.n, a.d, a.lds, kUmmaTile)) return cudaErrorNotSupported;
  if (!make_sw128_map(&maps.u, a.U, a.d, a.k, a.ldu, kUmmaCols)) return cudaErrorNotSupported;
  if (!make_sw128_map(&maps.u_wide, a.U, a.d, a.k <= 64 ? 64 : 128, a.ldu, kUmmaCols))
    return cudaErrorNotSupported;
  maps.p = maps.x;
  maps.x2 = maps.x;
  if (a.src2 != nullptr) {   // a second addend: only the launches without row operands take it
    if (has_e || has_p) return cudaErrorNotSupported;
    if (!make_sw128_map(&maps.x2, a.src2, a.n, a.d, a.lds2, kUmmaTile)) return cudaErrorNotSupported;
  }
  if (pmode == kPTma && !make_sw128_map(&maps.p, a.shift.P, a.shift.max_pos, a.d, a.shift.ldp, kUmmaTile))
    return cudaErrorNotSupported;
  if (ntp <= 2) return launch_umma_ntp<2>(b, has_e, pmode, maps, sm_count, stream);
  if (ntp <= 4) return launch_umma_ntp<4>(b, has_e, pmode, maps, sm_count, stream);
  if (ntp <= 6) return launch_umma_ntp<6>(b, has_e, pmode, maps, sm_count, stream);
  if (ntp <= 8) return launch_umma_ntp<8>(b, has_e, pmode, maps, sm_count, stream);
  if (ntp <= 12) return launch_umma_ntp<12>(b, has_e, pmode, maps, sm_count, stream);
  return launch_umma_ntp<16>(b, has_e, pmode, maps, sm_count, stream);
}

}  // namespace ssn
