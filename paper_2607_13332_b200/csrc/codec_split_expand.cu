// Launcher of the split-operand expansion kernel (see codec_split_expand.cuh).
#include "codec_split_expand.cuh"

#include "codec_mma_launch.h"
#include "codec_split.h"
#include "codec_tensor_maps.h"

namespace ssn {
namespace {

template <typename T, typename TZ, int KG, int NSLOT>
cudaError_t launch_one(const SplitExpandArgs &a, const CUtensorMap &out, int sms, cudaStream_t stream) {
  auto kernel = codec_split_expand_kernel<T, TZ, KG, NSLOT>;
  constexpr int smem = SplitExpandConfig<T, TZ, KG, NSLOT>::kSmemBytes;
  static std::atomic<uint64_t> configured{0};
  cudaError_t e = allow_dynamic_smem(kernel, smem, configured);
  if (e != cudaSuccess) return e;
  const int64_t units = ((a.n + kUmmaTile - 1) / kUmmaTile) * ((a.d + kChunkCols - 1) / kChunkCols);
  e = launch_dependent(kernel, (unsigned)(units < sms ? units : sms), kSplitExpandThreads, smem, stream, 1, a, out);
  note_kernel(SSN_KERNEL_SPLIT_EXPAND, (a.has_e ? SSN_KVAR_E : 0) | (a.has_p ? SSN_KVAR_P : 0) | (KG == 2 ? SSN_KVAR_WIDE : 0) |
                                           (sizeof(TZ) == 4 && sizeof(T) == 2 ? SSN_KVAR_ALT : 0));
  return e;
}

template <typename T, typename TZ>
cudaError_t launch_all(const SplitExpandArgs &a, const CUtensorMap &out, int sms, cudaStream_t s) {
  const int slots = a.has_e + a.has_p;
  if (a.k <= 64) {
    if (slots == 0) return launch_one<T, TZ, 1, 0>(a, out, sms, s);
    if (slots == 1) return launch_one<T, TZ, 1, 1>(a, out, sms, s);
    return launch_one<T, TZ, 1, 2>(a, out, sms, s);
  }
  if (slots == 0) return launch_one<T, TZ, 2, 0>(a, out, sms, s);
  if (slots == 1) return launch_one<T, TZ, 2, 1>(a, out, sms, s);
  return launch_one<T, TZ, 2, 2>(a, out, sms, s);
}

bool rows16(const void *p, int64_t ld, int esz) {
  return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && ld * esz % 16 == 0;
}

}  // namespace

cudaError_t launch_codec_split_expand(const TokenArgs &a, int32_t dtype, int sm_count, cudaStream_t stream) {
  if (a.src != nullptr || a.zin == nullptr || a.dst == nullptr || a.rowsumsq != nullptr || a.k > kSplitMaxRank ||
      a.U2 != nullptr || a.n > 0x7fffffffLL || sm_count < 1)
    return cudaErrorNotSupported;
  const int esz = dtype == SSN_F32 ? 4 : 2;
  SplitExpandArgs p{};
  p.zin = a.zin;
  p.U = a.U;
  p.dst = a.dst;
  p.ldzin = a.ldzin;
  p.ldu = a.ldu;
  p.lddst = a.lddst;
  p.n = a.n;
  p.d = a.d;
  p.k = a.k;
  p.shift = a.shift;
  p.has_e = a.add_shift && a.shift.E != nullptr;
  p.has_p = a.add_shift && a.shift.P != nullptr;
  p.vec_z = pairs_aligned(a.zin, a.ldzin, a.wire ? 4 : esz);
  p.vec_u = pairs_aligned(a.U, a.ldu, esz);
  p.vec_rows = (int64_t)a.d * esz % 16 == 0 && (int64_t)a.d * esz <= kZeroRowBytes &&
               (!p.has_e || rows16(a.shift.E, a.shift.lde, esz)) && (!p.has_p || rows16(a.shift.P, a.shift.ldp, esz));
  // 32 rows x 128 bytes; a store clips whole 16 bytes at the end of a row
  CUtensorMap out{};
  p.tma_out = (int64_t)a.d * esz % 16 == 0 && rows16(a.dst, a.lddst, esz) &&
              (dtype == SSN_F32 ? make_sw128_map_f32(&out, a.dst, a.n, a.d, a.lddst, 32) : make_sw128_map(&out, a.dst, a.n, a.d, a.lddst, 32));
  if (dtype == SSN_F32) return launch_all<float, float>(p, out, sm_count, stream);
  if (a.wire) return launch_all<__nv_bfloat16, float>(p, out, sm_count, stream);
  return launch_all<__nv_bfloat16, __nv_bfloat16>(p, out, sm_count, stream);
}

}  // namespace ssn
