// rpca_wide.cu -- host side of the wide / complex path: kernel tables.
#include <cuda_runtime.h>

#include <algorithm>

#include "rpca_internal.h"
#include "rpca_wide.cuh"

namespace rpca {

template <int TP, int RP, bool CPLX>
WideKernels make_wide() {
  WideKernels k;
  k.pass[PM_INIT] = (void*)pass_tile_kernel<TP, RP, PM_INIT, CPLX>;
  k.pass[PM_FUSED] = (void*)pass_tile_kernel<TP, RP, PM_FUSED, CPLX>;
  k.pass[PM_UPDATE] = (void*)pass_tile_kernel<TP, RP, PM_UPDATE, CPLX>;
  k.pass[PM_GRAM] = (void*)pass_tile_kernel<TP, RP, PM_GRAM, CPLX>;
  k.tile = RP;
  k.per_sm = tile_blocks_per_sm(TP, CPLX);
  k.pass_threads = kWideThreads;
  k.eig = (void*)eig_wide_kernel;
  k.eig_threads = kEigWThreads;
  k.eig_ctas = kEigWRanks;
  for (int i = 0; i < 4; ++i) {
    k.pass_tc[i] = nullptr;
    k.pass_tc_smem[i] = 0;
  }
  k.pass_tc_threads = kWtcThreads;
  // the tiled tensor-core pass: real windows of 33..128 frames, complex ones
  // of up to 64 frames (128 real columns; 16 frames and fewer padded to 64)
  constexpr int TPW = wtc_tp(TP);
  if constexpr ((CPLX || TP >= 64) && TPW <= 128) {
    k.pass_tc[RPCA_PREC_TF32X3] = (void*)pass_wtc_kernel<TPW, false, CPLX>;
    k.pass_tc_smem[RPCA_PREC_TF32X3] = WtcShape<TPW, false>::SMEM;
    k.pass_tc[RPCA_PREC_BF16X3] = (void*)pass_wtc_kernel<TPW, true, CPLX>;
    k.pass_tc_smem[RPCA_PREC_BF16X3] = WtcShape<TPW, true>::SMEM;
  }
  return k;
}

size_t wide_eig_scr_bytes(int T) { return T <= kMaxT ? 1 : eig_scr_bytes(T); }

size_t wide_tc_img_bytes(int T, int precision) {
  const int TP = wtc_tp(T);
  if (TP > 128) return 0;
  if (precision == RPCA_PREC_TF32X3) return wtc_img_bytes(TP, false);
  if (precision == RPCA_PREC_BF16X3) return wtc_img_bytes(TP, true);
  return 0;
}

void wide_launch_shape(int T, bool cplx, int64_t m, int sms, int* tile, int* per_sm) {
  *tile = tile_rp(T, cplx, m, sms);
  *per_sm = tile_blocks_per_sm(tile_tp(T, cplx), cplx);
}

bool wide_kernels(int T, bool cplx, bool force, int64_t m, int sms, WideKernels* out) {
  if (T > kMaxTW || T < 1) return false;
  if (!cplx && T <= kMaxT && !force) return false;
  if (cplx && (T & 1)) return false;
  const int RP = tile_rp(T, cplx, m, sms);
  switch (tile_tp(T, cplx)) {
    case 32: *out = cplx ? make_wide<32, 128, true>() : make_wide<32, 128, false>(); break;
    case 64: *out = cplx ? make_wide<64, 128, true>() : RP == 64 ? make_wide<64, 64, false>() : make_wide<64, 128, false>(); break;
    case 96: *out = cplx ? make_wide<96, 128, true>() : RP == 64 ? make_wide<96, 64, false>() : make_wide<96, 128, false>(); break;
    case 128: *out = cplx ? make_wide<128, 128, true>() : RP == 64 ? make_wide<128, 64, false>() : make_wide<128, 128, false>(); break;
    case 160: *out = make_wide<160, 64, false>(); break;
    case 192: *out = cplx ? make_wide<192, 64, true>() : make_wide<192, 64, false>(); break;
    case 224: *out = make_wide<224, 64, false>(); break;
    default: *out = make_wide<256, 64, true>(); break;
  }
  out->pass_smem = tile_pass_smem(T, RP, cplx);
  // The kernels are shared by plans of other frame counts, which may have been made before and launch with their own
  // size: the limits are those of the largest one, whatever this plan needs.
  const int pass_max = (int)tile_pass_smem(std::min(tile_tp(T, cplx), kMaxTW), RP, cplx);
  size_t eig_max;
  if (T <= kMaxT) {
    out->eig = (void*)eig_small_kernel;
    out->eig_threads = kEigThreads;
    out->eig_ctas = 1;
    out->eig_smem = eig_max = sizeof(Eig64Smem);
  } else {
    // the sweeps' columns, or one rank's operands of a product, as far as they fit
    const size_t ops = 2 * sizeof(float) * (size_t)T * (eig_ld(T) + (eig_ld(T) / 4 + kEigWRanks - 1) / kEigWRanks * 4);
    static_assert(eig_wide_smem(kMaxTW) <= kEigWMaxSmem, "the sweeps of the longest columns fit");
    out->eig_smem = std::max(eig_wide_smem(T), std::min(ops, kEigWMaxSmem));
    eig_max = kEigWMaxSmem;
  }
  if (cudaFuncSetAttribute(out->eig, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)eig_max) != cudaSuccess) return false;
  for (int i = 0; i < 4; ++i)
    if (cudaFuncSetAttribute(out->pass[i], cudaFuncAttributeMaxDynamicSharedMemorySize, pass_max) != cudaSuccess)
      return false;
  for (int i = 0; i < 4; ++i)
    if (out->pass_tc[i] && cudaFuncSetAttribute(out->pass_tc[i], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                (int)out->pass_tc_smem[i]) != cudaSuccess)
      return false;
  return true;
}

}  // namespace rpca
