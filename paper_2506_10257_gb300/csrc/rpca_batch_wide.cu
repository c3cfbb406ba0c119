// rpca_batch_wide.cu -- the batched persistent kernel for batches that hold a
// wide (T > 32) or complex window: every window of such a batch runs the tiled
// pass and eigen-step bodies (rpca_wide.cuh) under the same lane schedule,
// publication counters and bounded waits as the narrow batch kernel
// (rpca_batch.cuh).  Kept in its own translation unit so it compiles in
// parallel with the rest of the library.
#include <cuda_runtime.h>

#include "rpca_kernels.cuh"
#include "rpca_internal.h"
#include "rpca_wide.cuh"

namespace rpca {
#include "rpca_batch.cuh"

// The tiled bodies are called, not inlined, into the one kernel that serves
// every column count: each compiles once, which keeps the build short.
template <int TP, int RP, int MODE, bool CPLX>
__device__ __noinline__ bool wide_pass_call(Bufs b, int lc, int nc, float* f) {
  return pass_tile_body<TP, RP, MODE, CPLX>(b, lc, nc, f);
}
__device__ __noinline__ void wide_eig_call(Bufs b, int flags, float* f, int eig_floats) {
  eig_wide_body<8>(b, flags, 0, 0, f, eig_floats, 0, 1);
}

// The tiled steps of a window by its padded columns (TB of the descriptor).
template <bool CPLX>
struct WideDisp {
  template <int TP>
  static __device__ bool run(Bufs b, bool init, int lc, int nc, float* f) {
    constexpr int RP = TP > 128 ? 64 : 128;
    return init ? wide_pass_call<TP, RP, PM_INIT, CPLX>(b, lc, nc, f) : wide_pass_call<TP, RP, PM_FUSED, CPLX>(b, lc, nc, f);
  }
  static __device__ bool pass(WinDesc& wd, bool init, int lc, int nc, unsigned char* dsm) {
    float* f = reinterpret_cast<float*>(dsm);
    switch (wd.TB) {
      case 32: return run<32>(wd.b, init, lc, nc, f);
      case 64: return run<64>(wd.b, init, lc, nc, f);
      case 96: return run<96>(wd.b, init, lc, nc, f);
      case 128: return run<128>(wd.b, init, lc, nc, f);
      case 192: return run<192>(wd.b, init, lc, nc, f);
      default: break;
    }
    if constexpr (CPLX) {
      if (wd.TB == 256) return run<256>(wd.b, init, lc, nc, f);
    } else {
      if (wd.TB == 160) return run<160>(wd.b, init, lc, nc, f);
      if (wd.TB == 224) return run<224>(wd.b, init, lc, nc, f);
    }
    return false;
  }
  static __device__ void eig(WinDesc& wd, int flags, unsigned char* dsm, int eig_floats) {
    // (up to 32 columns: the narrow step, as in plans; a batch of four 8-frame complex
    // 100 x 100 windows takes 2.1 ms, 4.2 with the wide one)
    if (wd.b.T <= kMaxT)
      eig64_body<false>(wd.b, flags, 0, 0, dsm);
    else
      wide_eig_call(wd.b, flags, reinterpret_cast<float*>(dsm), eig_floats);
  }
};

// Batches holding a wide or complex window: every window runs the tiled
// bodies (TB of a window: its padded columns), 16 warps a CTA.
template <bool CPLX>
__global__ void __launch_bounds__(kWideThreads, 1) batch_kernel_wide(BatchDesc* bd) {
  extern __shared__ __align__(16) unsigned char batch_dsm[];
  const int nl = bd->nlanes;
  int l = 0;
  while (l + 1 < nl && (int)blockIdx.x >= bd->lane[l + 1].cta0) ++l;
  const LaneDesc ld = bd->lane[l];
  const int lc = (int)blockIdx.x - ld.cta0;
  if (lc < 0 || lc >= ld.ncta) return;
  const unsigned long long limit = bd->spin_limit;
  const int eig_floats = bd->eig_floats;
  run_lane<WideDisp<CPLX>>(bd, ld, lc, batch_dsm, limit, &bd->stop, eig_floats, lane_is_paired(bd->paired, ld));
}

void* batch_wide_kernel_fn(bool cplx) {
  return cplx ? (void*)batch_kernel_wide<true> : (void*)batch_kernel_wide<false>;
}

}  // namespace rpca
