// rpca_wide.cuh -- the iteration for windows of many frames (kMaxT < T <= kMaxTW) and for
// complex windows: device bodies and kernels (host side in rpca_wide.cu).
//
// Same algebra as the register-resident path (see rpca_device.cuh): per
// iteration one fused pass over the pixels (Eq. 4-6 through the Gram of Z, the
// residual of Sec. II-A, and the rotated Gram of the next Z) and one
// eigen-step (rpca_eig_wide.cuh).  With T up to 224 a pixel row no longer fits in
// one thread's registers, so the pass works on tiles of RP pixels:
//   1. X, S, Y of the tile are read (16 bytes a load) and Z = X - S + Y/mu goes to
//      shared memory, frame-major;
//   2. Q = Z Wbar, 4 pixels x CPT columns per thread;
//   3. the Eq. 5-6 update of the thread's 4 pixels and CPT frames, with S and Y
//      read again (L2 holds them since step 1), S' and Y' written and Z' put in
//      Z's place;
//   4. U = Z' V, in the same registers, then pixel-major over Z';
//   5. the partial Gram U^T U in registers across the CTA's tiles: 4 x 4 blocks
//      of the upper triangle, the tile's pixels split over as many groups of
//      threads as the blocks leave room for.
// Complex windows repeat steps 4 and 5 for the rows of i Z'.
// Up to 128 columns Wbar and V stay in shared memory; above, they stream through
// it kWKC rows at a time, the next rows arriving while the current ones are used.
// The tile holds Z alone (not S and Y too, as it once did), which leaves room for
// 128-pixel tiles and 16 warps; windows with fewer such tiles than SMs take
// 64-pixel tiles.  What bounds the pass is the FP32 pipe: per k a thread loads one
// 16-byte group of Z (four in a warp) and CPT values of Wbar or V (eight groups in a
// warp, each a conflict-free 16-byte load) for 4 CPT multiply-adds.
// Measured, with the tile that held S and Y -> now: 262144 x 50 248 -> 192 us (FMA pipe
// 33 % busy, most stalls on shared memory), 87880 x 132 760 -> 430 us, complex
// 65536 x 50 331 -> 261 us.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include "rpca_kernels.cuh"

namespace rpca {

constexpr int kWideThreads = 512;
constexpr int kWKC = 16;          // rows of Wbar / V per streamed step (more than 128 columns)
constexpr int kWideLd = 4;        // frame rows a warp loads before their shared-memory stores: the compiler cannot
                                  // tell those stores from the loads after them

// Shared-memory position of pixel pp of frame row t in the frame-major tile: rows
// of RP pixels, the pixel index XOR-ed with 4 * ((t / 4) % 8) so that the Eq. 5-6
// update, whose threads walk down the columns of a tile 4 rows apart, spreads over
// eight banks instead of one; groups of 4 pixels stay contiguous.
template <int RP>
__device__ __forceinline__ int tile_at(int t, int pp) { return t * RP + (pp ^ (((t >> 2) & 7) << 2)); }

template <int TP, int RP, bool CPLX>
struct TileShape {
  static constexpr int PG = RP / 4;                       // pixel groups of 4
  static constexpr int CG = kWideThreads / PG;            // column groups
  static constexpr int CPT = TP / CG;                     // columns per thread
  static constexpr bool RES = TP <= 128;                  // Wbar and V resident
  static constexpr bool SEP = CPLX && !RES;               // U beside Z (its two row sets come one after the other)
  static constexpr int NB = TP < kMaxTW ? TP / 4 : kMaxTW / 4;
  static constexpr int NBLK = NB * (NB + 1) / 2;
  static constexpr int BPT = (NBLK + kWideThreads - 1) / kWideThreads;
  static_assert(RP % 32 == 0 && TP % CG == 0 && (CPT % 2 == 0 || !CPLX), "tile shape");
};

// Padded columns: a multiple of 32, of 64 for complex windows beyond 128 (an even
// number of columns a thread at 64-pixel tiles).
__host__ __device__ constexpr int tile_tp(int T, bool cplx) {
  const int TP = (T + 31) / 32 * 32;
  return cplx && TP > 128 ? (T + 63) / 64 * 64 : TP;
}
// Dynamic shared memory of the tiled pass for T real columns.
__host__ __device__ constexpr size_t tile_pass_smem(int T, int RP, bool cplx) {
  const size_t T4 = (T + 3) / 4 * 4, TP = tile_tp(T, cplx);
  const size_t u = (size_t)RP * (T4 + 4), scratch = (size_t)kWideThreads * 16;  // U over Z; the Gram groups' sums
  const size_t zu = u > scratch ? u : scratch;
  return sizeof(float) * (TP <= 128 ? 2 * T * TP + zu : 2 * kWKC * TP + zu + (cplx ? u : 0));
}
// Pixels per tile: 128, or 64 beyond 128 columns and (plans of real windows) where
// 128 would leave SMs without a tile.
__host__ __device__ constexpr int tile_rp(int T, bool cplx, int64_t m, int sms) {
  return tile_tp(T, cplx) > 128 || (!cplx && T > 32 && m < (int64_t)128 * sms) ? 64 : 128;
}

// First column of a thread's j-th column pair or group: whole groups of 4 columns
// lie 4 CG apart (conflict-free 16-byte loads), what is left follows in pairs or
// single columns.
template <int TP, int RP, bool CPLX>
__device__ __forceinline__ int tile_col(int cg, int j) {
  using TS = TileShape<TP, RP, CPLX>;
  constexpr int C4 = TS::CPT / 4 * 4, R = TS::CPT - C4;
  if (j < C4) return (j / 4) * 4 * TS::CG + 4 * cg + (j & 3);
  const int r = j - C4;
  if constexpr (R == 2) return C4 * TS::CG + 2 * cg + r;
  if constexpr (R == 3) return r < 2 ? C4 * TS::CG + 2 * cg + r : (C4 + 2) * TS::CG + cg;
  return C4 * TS::CG + cg + r;
}

// acc[i][j] += sum over rows k0 <= k < k1 of z(k)[i] * M(k, col(j)), in increasing k
// (zrow(k, r): row k + r)
template <int TP, int RP, bool CPLX, typename ZF>
__device__ __forceinline__ void tile_times(float (&acc)[4][TileShape<TP, RP, CPLX>::CPT], const float* sM, int k0, int k1,
                                           int cg, ZF zrow) {
  using TS = TileShape<TP, RP, CPLX>;
  constexpr int CPT = TS::CPT, C4 = CPT / 4 * 4, R = CPT - C4, H = CPT / 2;
  constexpr bool ODD = R == 1 || R == 3;
  uint64_t a2[4][H ? H : 1];
  float a1[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int h = 0; h < H; ++h) a2[i][h] = f2_pack(acc[i][2 * h], acc[i][2 * h + 1]);
    a1[i] = ODD ? acc[i][CPT - 1] : 0.f;
  }
  auto step = [&](int k, const float4 z) {
    const uint64_t zz[4] = {f2_pack(z.x, z.x), f2_pack(z.y, z.y), f2_pack(z.z, z.z), f2_pack(z.w, z.w)};
    const float* row = sM + (k - (TS::RES ? 0 : k0)) * TP;
#pragma unroll
    for (int g = 0; g < C4 / 4; ++g) {
      const float4 v = *reinterpret_cast<const float4*>(row + 4 * g * TS::CG + 4 * cg);
      const uint64_t w0 = f2_pack(v.x, v.y), w1 = f2_pack(v.z, v.w);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        a2[i][2 * g] = f2_fma(zz[i], w0, a2[i][2 * g]);
        a2[i][2 * g + 1] = f2_fma(zz[i], w1, a2[i][2 * g + 1]);
      }
    }
    if constexpr (R >= 2) {
      const float2 v = *reinterpret_cast<const float2*>(row + C4 * TS::CG + 2 * cg);
      const uint64_t w0 = f2_pack(v.x, v.y);
#pragma unroll
      for (int i = 0; i < 4; ++i) a2[i][C4 / 2] = f2_fma(zz[i], w0, a2[i][C4 / 2]);
    }
    if constexpr (ODD) {
      const float v = row[(C4 + (R == 3 ? 2 : 0)) * TS::CG + cg];
      a1[0] = fmaf(z.x, v, a1[0]);
      a1[1] = fmaf(z.y, v, a1[1]);
      a1[2] = fmaf(z.z, v, a1[2]);
      a1[3] = fmaf(z.w, v, a1[3]);
    }
  };
  // rows four at a time (k0 is a multiple of four: they share one swizzle)
  int k = k0;
  for (; k + 4 <= k1; k += 4) {
    float4 z[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) z[r] = zrow(k, r);
#pragma unroll
    for (int r = 0; r < 4; ++r) step(k + r, z[r]);
  }
  for (; k < k1; ++k) step(k, zrow(k & ~3, k & 3));
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int h = 0; h < H; ++h) {
      const float2 v = f2_unpack(a2[i][h]);
      acc[i][2 * h] = v.x;
      acc[i][2 * h + 1] = v.y;
    }
    if (ODD) acc[i][CPT - 1] = a1[i];
  }
}

// Rows [k0, k0 + kWKC) of a T x T row-major matrix into sM[kWKC][TP] by
// asynchronous copies (columns beyond T keep whatever is there; rows beyond T are
// not used).
template <int TP>
__device__ __forceinline__ void stream_rows(float* sM, const float* M, int k0, int T) {
  const int n = min(kWKC, T - k0) * T;
  for (int i = threadIdx.x; i < n; i += kWideThreads) {
    const int r = i / T, c = i - r * T;
    cp_async4(&sM[r * TP + c], M + (size_t)k0 * T + i);
  }
  cp_async_commit();
}

// acc = z M over all k; M resident at res, or streamed through the two buffers
template <int TP, int RP, bool CPLX, typename ZF>
__device__ __forceinline__ void contract(float (&acc)[4][TileShape<TP, RP, CPLX>::CPT], const float* res, float* buf0,
                                         float* buf1, const float* M, int T, int cg, ZF zrow) {
  using TS = TileShape<TP, RP, CPLX>;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < TS::CPT; ++j) acc[i][j] = 0.f;
  if constexpr (TS::RES) {
    tile_times<TP, RP, CPLX>(acc, res, 0, T, cg, zrow);
  } else {
    stream_rows<TP>(buf0, M, 0, T);
    for (int k0 = 0, par = 0; k0 < T; k0 += kWKC, par ^= 1) {
      cp_async_wait<0>();
      __syncthreads();  // these rows are here, and the other buffer's last readers are done
      if (k0 + kWKC < T) stream_rows<TP>(par ? buf0 : buf1, M, k0 + kWKC, T);
      tile_times<TP, RP, CPLX>(acc, par ? buf1 : buf0, k0, min(k0 + kWKC, T), cg, zrow);
    }
    __syncthreads();
  }
}

// Rows of U in the standard basis (initial pass): the thread's pixels and columns of Z itself
template <int TP, int RP, bool CPLX, typename ZF>
__device__ __forceinline__ void take_rows(float (&out)[4][TileShape<TP, RP, CPLX>::CPT], int T, int cg, ZF zrow) {
#pragma unroll
  for (int j = 0; j < TileShape<TP, RP, CPLX>::CPT; ++j) {
    const int t = tile_col<TP, RP, CPLX>(cg, j);
    const float4 v = t < T ? zrow(t & ~3, t & 3) : make_float4(0.f, 0.f, 0.f, 0.f);
    out[0][j] = v.x;
    out[1][j] = v.y;
    out[2][j] = v.z;
    out[3][j] = v.w;
  }
}

// 4 consecutive floats of frame row `row` from pixel p: one load where `vec`
// (16-byte aligned and inside the window), else guarded ones.
__device__ __forceinline__ float4 load4(const float* row, int64_t p, int64_t m, bool vec) {
  if (vec) return *reinterpret_cast<const float4*>(row + p);
  return make_float4(p < m ? row[p] : 0.f, p + 1 < m ? row[p + 1] : 0.f, p + 2 < m ? row[p + 2] : 0.f,
                     p + 3 < m ? row[p + 3] : 0.f);
}
__device__ __forceinline__ void store4(float* row, int64_t p, int64_t m, bool vec, const float (&v)[4]) {
  if (vec) {
    *reinterpret_cast<float4*>(row + p) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (p + i < m) row[p + i] = v[i];
  }
}
// (re, im) of 4 consecutive pixels of a complex frame row
__device__ __forceinline__ void load4c(const float2* row, int64_t p, int64_t m, bool vec, float4& re, float4& im) {
  if (vec) {
    const float4 a = *reinterpret_cast<const float4*>(row + p), b = *reinterpret_cast<const float4*>(row + p + 2);
    re = make_float4(a.x, a.z, b.x, b.z);
    im = make_float4(a.y, a.w, b.y, b.w);
  } else {
    float2 v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = p + i < m ? row[p + i] : make_float2(0.f, 0.f);
    re = make_float4(v[0].x, v[1].x, v[2].x, v[3].x);
    im = make_float4(v[0].y, v[1].y, v[2].y, v[3].y);
  }
}
__device__ __forceinline__ void store4c(float2* row, int64_t p, int64_t m, bool vec, const float (&re)[4],
                                        const float (&im)[4]) {
  if (vec) {
    *reinterpret_cast<float4*>(row + p) = make_float4(re[0], im[0], re[1], im[1]);
    *reinterpret_cast<float4*>(row + p + 2) = make_float4(re[2], im[2], re[3], im[3]);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (p + i < m) row[p + i] = make_float2(re[i], im[i]);
  }
}

// CPLX: complex windows as their interleaved real embedding (column 2t = Re,
// 2t + 1 = Im of frame t; T = 2 x frames).  The Hermitian Gram Z^H Z is the
// real Gram of the 2m rows a = [Re z, Im z] and b = a P = [-Im z, Re z] (the
// row of i z) per pixel, so the pass adds both rows of every pixel to the
// Gram; the shrink of Eq. 5 acts on the magnitude of each complex entry.
template <int TP, int RP, int MODE, bool CPLX>
__device__ bool pass_tile_body(Bufs b, int lc, int nc, float* smem) {
  using TS = TileShape<TP, RP, CPLX>;
  constexpr int CPT = TS::CPT;
  constexpr bool kGram = (MODE != PM_UPDATE);
  __shared__ double sRed[2][kWideThreads / 32];
  __shared__ double sScal[2 * kMaxGroups];
  __shared__ int sLast;

  const Ctrl* ctrl = b.ctrl;
  if (solve_done_uniform(ctrl)) return false;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  constexpr int NW = kWideThreads / 32;
  // a warp holds 4 pixel groups x 8 column groups
  const int pg = (w % (TS::PG / 4)) * 4 + (lane >> 3), cg = (w / (TS::PG / 4)) * 8 + (lane & 7);
  const int p0 = 4 * pg;
  if (tid == 0) atomicMin(&b.red->t_start, gtimer());
  const int T = b.T, T4 = (T + 3) / 4 * 4, UP = T4 + 4;
  const int64_t m = b.m;
  const float* X = b.job->X;
  float* S = b.job->S;
  float *Y0 = b.job->Y0, *Y1 = b.job->Y1;
  const int kc = __ldcg(&ctrl->k);
  const bool first = (kc == 0) && !__ldcg(&ctrl->warm);
  const float f_mu = __ldcg(&ctrl->f_mu), inv_mu = __ldcg(&ctrl->f_inv_mu), gamma = __ldcg(&ctrl->f_gamma);
  const float inv_mu_nxt = __ldcg(&ctrl->f_inv_mu_nxt);
  const float* Yin = (kc & 1) ? Y1 : Y0;
  float* Yout = (kc & 1) ? Y0 : Y1;
  const bool read_sy = MODE != PM_INIT && !first;
  // whole groups of 4 pixels are 16-byte aligned in every frame row
  const bool aligned = CPLX ? m % 2 == 0 : m % 4 == 0;

  float* sW = smem;                                            // [T][TP], or two streamed buffers [kWKC][TP]
  float* sV = sW + (TS::RES ? T * TP : kWKC * TP);
  float* sZ = sV + (TS::RES ? T * TP : kWKC * TP);             // [T][RP] swizzled; then U [RP][UP]
  float* sU = TS::SEP ? sZ + (size_t)RP * UP : sZ;
  if (TS::RES && MODE != PM_INIT) {
    for (int i = tid; i < T * TP; i += kWideThreads) {
      const int r = i / TP, c = i % TP;
      const bool in = c < T;
      sW[i] = in ? __ldcg(&b.Ww[r * T + c]) : 0.f;
      sV[i] = in ? __ldcg(&b.Vw[r * T + c]) : 0.f;
    }
  } else if (!TS::RES) {
    // (columns beyond T of the streamed buffers: read, never used)
    for (int i = tid; i < 2 * kWKC * TP; i += kWideThreads) sW[i] = 0.f;
  }

  // Gram blocks of this thread: block index within the T-frame triangle and pixel
  // group (blocks beyond the threads go to the first group's second round)
  const int nb = T4 / 4, nblk = nb * (nb + 1) / 2;
  const int ngrp = nblk <= kWideThreads ? kWideThreads / nblk : 1;
  const int grp = nblk <= kWideThreads ? tid / nblk : 0;
  int gbi[TS::BPT], gbj[TS::BPT];
  float gacc[TS::BPT][16];
#pragma unroll
  for (int u = 0; u < TS::BPT; ++u) {
    const int blk = nblk <= kWideThreads ? (u == 0 && grp < ngrp ? tid - grp * nblk : nblk) : tid + u * kWideThreads;
    gbi[u] = gbj[u] = -1;
    if (kGram && blk < nblk) tri_coords(blk, nb, gbi[u], gbj[u]);
#pragma unroll
    for (int i = 0; i < 16; ++i) gacc[u][i] = 0.f;
  }
  auto gram_add = [&]() {
#pragma unroll
    for (int u = 0; u < TS::BPT; ++u) {
      if (gbi[u] < 0) continue;
      const float* pa = sU + 4 * gbi[u];
      const float* pc = sU + 4 * gbj[u];
      uint64_t g2[8];  // g2[2i + h] = (gacc[4i + 2h], gacc[4i + 2h + 1])
#pragma unroll
      for (int i = 0; i < 8; ++i) g2[i] = f2_pack(gacc[u][2 * i], gacc[u][2 * i + 1]);
#pragma unroll 2
      for (int pp = grp; pp < RP; pp += ngrp) {
        const float4 a = *reinterpret_cast<const float4*>(pa + pp * UP);
        const float4 c = *reinterpret_cast<const float4*>(pc + pp * UP);
        const float av[4] = {a.x, a.y, a.z, a.w};
        const uint64_t c01 = f2_pack(c.x, c.y), c23 = f2_pack(c.z, c.w);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint64_t ai = f2_pack(av[i], av[i]);
          g2[2 * i] = f2_fma(ai, c01, g2[2 * i]);
          g2[2 * i + 1] = f2_fma(ai, c23, g2[2 * i + 1]);
        }
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float2 v = f2_unpack(g2[i]);
        gacc[u][2 * i] = v.x;
        gacc[u][2 * i + 1] = v.y;
      }
    }
  };
  float e2 = 0.f, l1 = 0.f;

  const int64_t ntiles = (m + RP - 1) / RP;
  for (int64_t tile = lc; tile < ntiles; tile += nc) {
    const int64_t pb = tile * RP;
    const bool whole = aligned && pb + RP <= m;
    __syncthreads();  // the previous tile's U (and the resident matrices) are consumed / ready
    // ---- 1. stage: a warp takes frame rows, a lane 4 pixels ----
    constexpr int LPR = RP / 4;                // lanes per frame row (32, or 16: two rows a warp)
    constexpr int RPW = 32 / LPR;
    const int pl = 4 * (lane % LPR);
    const int nrow = CPLX ? T / 2 : T;
    for (int r0 = w * RPW + lane / LPR; r0 < nrow; r0 += NW * RPW * kWideLd) {
      float4 xr[kWideLd], sr[kWideLd], yr[kWideLd], xi[kWideLd], si[kWideLd], yi[kWideLd];
#pragma unroll
      for (int u = 0; u < kWideLd; ++u) {
        const int t = min(r0 + u * NW * RPW, nrow - 1);
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        sr[u] = yr[u] = si[u] = yi[u] = zero;
        if constexpr (CPLX) {
          load4c(reinterpret_cast<const float2*>(X) + (int64_t)t * m, pb + pl, m, whole, xr[u], xi[u]);
          if (read_sy) {
            load4c(reinterpret_cast<const float2*>(S) + (int64_t)t * m, pb + pl, m, whole, sr[u], si[u]);
            load4c(reinterpret_cast<const float2*>(Yin) + (int64_t)t * m, pb + pl, m, whole, yr[u], yi[u]);
          }
        } else {
          xr[u] = load4(X + (int64_t)t * m, pb + pl, m, whole);
          if (read_sy) {
            sr[u] = load4(S + (int64_t)t * m, pb + pl, m, whole);
            yr[u] = load4(Yin + (int64_t)t * m, pb + pl, m, whole);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < kWideLd; ++u) {
        const int t = r0 + u * NW * RPW;
        if (t >= nrow) break;
        auto zf = [&](const float4& x, const float4& s, const float4& y) {
          return make_float4(form_z(x.x, s.x, y.x, inv_mu), form_z(x.y, s.y, y.y, inv_mu),
                             form_z(x.z, s.z, y.z, inv_mu), form_z(x.w, s.w, y.w, inv_mu));
        };
        if constexpr (CPLX) {
          const float4 zr = MODE == PM_INIT ? xr[u] : zf(xr[u], sr[u], yr[u]);
          const float4 zi = MODE == PM_INIT ? xi[u] : zf(xi[u], si[u], yi[u]);
          *reinterpret_cast<float4*>(&sZ[tile_at<RP>(2 * t, pl)]) = zr;
          *reinterpret_cast<float4*>(&sZ[tile_at<RP>(2 * t + 1, pl)]) = zi;
          if (MODE == PM_INIT) {
            const float a2[4] = {fmaf(zr.x, zr.x, zi.x * zi.x), fmaf(zr.y, zr.y, zi.y * zi.y),
                                 fmaf(zr.z, zr.z, zi.z * zi.z), fmaf(zr.w, zr.w, zi.w * zi.w)};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              e2 += a2[i];
              l1 += sqrtf(a2[i]);
            }
          }
        } else {
          const float4 z = MODE == PM_INIT ? xr[u] : zf(xr[u], sr[u], yr[u]);
          *reinterpret_cast<float4*>(&sZ[tile_at<RP>(t, pl)]) = z;
          if (MODE == PM_INIT) {
            e2 = fmaf(z.x, z.x, fmaf(z.y, z.y, fmaf(z.z, z.z, fmaf(z.w, z.w, e2))));
            l1 += (fabsf(z.x) + fabsf(z.y)) + (fabsf(z.z) + fabsf(z.w));
          }
        }
      }
    }
    __syncthreads();
    // the next tile's rows on their way to L2
    if (tile + nc < ntiles) {
      const int64_t nx = (tile + nc) * RP * (CPLX ? 2 : 1);
      constexpr int LINES = RP * (CPLX ? 2 : 1) / 32;
      const int64_t row = m * (CPLX ? 2 : 1);
      for (int i = tid; i < nrow * LINES; i += kWideThreads) {
        const int64_t c = nx + 32 * (i % LINES);
        if (c >= row) continue;
        const int64_t off = (int64_t)(i / LINES) * row + c;
        prefetch_l2(X + off);
        if (read_sy) {
          prefetch_l2(S + off);
          prefetch_l2(Yin + off);
        }
      }
    }
    // row k + r of the thread's pixels, k a multiple of four and r < 4
    auto zrow = [&](int k, int r) { return *reinterpret_cast<const float4*>(&sZ[tile_at<RP>(k, p0) + r * RP]); };
    auto zat = [&](int t) { return zrow(t & ~3, t & 3); };
    auto zrow_i = [&](int k, int r) {  // rows of i Z (complex): (-Im, Re) per frame
      const float4 v = zrow(k, r ^ 1);
      return (r & 1) ? v : make_float4(-v.x, -v.y, -v.z, -v.w);
    };
    float u[4][CPT], ui[CPLX ? 4 : 1][CPT];
    if (MODE == PM_INIT) {
      take_rows<TP, RP, CPLX>(u, T, cg, zrow);
      if constexpr (CPLX && !TS::SEP) take_rows<TP, RP, CPLX>(ui, T, cg, zrow_i);
    } else {
      if (MODE != PM_GRAM) {
        // ---- 2. Q = Z Wbar ----
        float q[4][CPT];
        contract<TP, RP, CPLX>(q, sW, sW, sV, b.Ww, T, cg, zrow);
        __syncthreads();  // every thread has read Z before Z' replaces it
        // ---- 3. Eq. 5-6 for 4 pixels x CPT columns: the S, Y loads of up to four
        //      columns, then their S', Y' stores ----
        const bool vec = whole;
        const int64_t p = pb + p0;
        if constexpr (CPLX) {
          constexpr int G = CPT >= 4 ? 4 : 2;
#pragma unroll
          for (int j0 = 0; j0 < CPT; j0 += G) {
            float4 sr[G / 2], si[G / 2], yr[G / 2], yi[G / 2];
#pragma unroll
            for (int g = 0; g < G / 2; ++g) {
              if (j0 + 2 * g >= CPT) continue;
              const int64_t f = min(tile_col<TP, RP, CPLX>(cg, j0 + 2 * g), T - 2) >> 1;
              sr[g] = si[g] = yr[g] = yi[g] = make_float4(0.f, 0.f, 0.f, 0.f);
              if (read_sy) {
                load4c(reinterpret_cast<const float2*>(S) + f * m, p, m, vec, sr[g], si[g]);
                load4c(reinterpret_cast<const float2*>(Yin) + f * m, p, m, vec, yr[g], yi[g]);
              }
            }
#pragma unroll
            for (int g = 0; g < G / 2; ++g) {
              if (j0 + 2 * g >= CPT) continue;
              const int j = j0 + 2 * g, t = tile_col<TP, RP, CPLX>(cg, j);
              if (t >= T) continue;
              const float4 zr = zat(t), zi = zat(t + 1);
              const float zrv[4] = {zr.x, zr.y, zr.z, zr.w}, ziv[4] = {zi.x, zi.y, zi.z, zi.w};
              const float srv[4] = {sr[g].x, sr[g].y, sr[g].z, sr[g].w}, siv[4] = {si[g].x, si[g].y, si[g].z, si[g].w};
              const float yrv[4] = {yr[g].x, yr[g].y, yr[g].z, yr[g].w}, yiv[4] = {yi[g].x, yi[g].y, yi[g].z, yi[g].w};
              float snr[4], sni[4], ynr[4], yni[4], znr[4], zni[4];
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const float dr = yrv[i] * inv_mu, di = yiv[i] * inv_mu;
                const float rr = srv[i] + q[i][j], ri = siv[i] + q[i][j + 1];
                const float mag = sqrtf(fmaf(rr, rr, ri * ri));
                const float f = (mag > gamma) ? gamma / mag : 1.f;   // clip to the disc of radius gamma
                const float cr = rr * f, ci = ri * f;
                snr[i] = rr - cr;                                    // Eq. 5 (magnitude shrink)
                sni[i] = ri - ci;
                ynr[i] = f_mu * cr;                                  // Eq. 6
                yni[i] = f_mu * ci;
                const float er = cr - dr, ei = ci - di;
                const bool in = vec || p + i < m;
                if (in) e2 = fmaf(er, er, fmaf(ei, ei, e2));
                znr[i] = in ? ((zrv[i] - dr) - q[i][j]) + cr + ynr[i] * inv_mu_nxt : 0.f;
                zni[i] = in ? ((ziv[i] - di) - q[i][j + 1]) + ci + yni[i] * inv_mu_nxt : 0.f;
              }
              const int64_t f = t >> 1;
              store4c(reinterpret_cast<float2*>(S) + f * m, p, m, vec, snr, sni);
              store4c(reinterpret_cast<float2*>(Yout) + f * m, p, m, vec, ynr, yni);
              *reinterpret_cast<float4*>(&sZ[tile_at<RP>(t, p0)]) = make_float4(znr[0], znr[1], znr[2], znr[3]);
              *reinterpret_cast<float4*>(&sZ[tile_at<RP>(t + 1, p0)]) = make_float4(zni[0], zni[1], zni[2], zni[3]);
            }
          }
        } else {
          constexpr int G = 4;
#pragma unroll
          for (int j0 = 0; j0 < CPT; j0 += G) {
            float4 sg[G], yg[G];
#pragma unroll
            for (int g = 0; g < G; ++g) {
              if (j0 + g >= CPT) continue;
              const int64_t t = min(tile_col<TP, RP, CPLX>(cg, j0 + g), T - 1);
              sg[g] = yg[g] = make_float4(0.f, 0.f, 0.f, 0.f);
              if (read_sy) {
                sg[g] = load4(S + t * m, p, m, vec);
                yg[g] = load4(Yin + t * m, p, m, vec);
              }
            }
#pragma unroll
            for (int g = 0; g < G; ++g) {
              if (j0 + g >= CPT) continue;
              const int j = j0 + g, t = tile_col<TP, RP, CPLX>(cg, j);
              if (t >= T) continue;
              const float4 z4 = zat(t);
              const float zv[4] = {z4.x, z4.y, z4.z, z4.w}, sv[4] = {sg[g].x, sg[g].y, sg[g].z, sg[g].w};
              const float yv[4] = {yg[g].x, yg[g].y, yg[g].z, yg[g].w};
              float sn[4], yn[4], zn[4];
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const float d = yv[i] * inv_mu;
                const float r = sv[i] + q[i][j];                   // X - L + Y/mu
                const float c = fminf(fmaxf(r, -gamma), gamma);    // clip to +-lambda/mu
                sn[i] = r - c;                                     // Eq. 5
                yn[i] = f_mu * c;                                  // Eq. 6
                const float e = c - d;                             // X - L - S'
                const bool in = vec || p + i < m;
                if (in) e2 = fmaf(e, e, e2);
                // Z' = X - S' + Y'/mu' with X = Z + S - Y/mu and S' = S + Q - clip
                zn[i] = in ? ((zv[i] - d) - q[i][j]) + c + yn[i] * inv_mu_nxt : 0.f;
              }
              store4(S + (int64_t)t * m, p, m, vec, sn);
              store4(Yout + (int64_t)t * m, p, m, vec, yn);
              *reinterpret_cast<float4*>(&sZ[tile_at<RP>(t, p0)]) = make_float4(zn[0], zn[1], zn[2], zn[3]);
            }
          }
        }
        __syncthreads();  // Z' complete
      }
      if (kGram) {
        // ---- 4. U = Z' V (complex: and (i Z') V) ----
        contract<TP, RP, CPLX>(u, sV, sW, sV, b.Vw, T, cg, zrow);
        if constexpr (CPLX && !TS::SEP) contract<TP, RP, CPLX>(ui, sV, sW, sV, b.Vw, T, cg, zrow_i);
      }
    }
    if (kGram) {
      auto put_rows = [&](float (&v)[4][CPT]) {
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
          const int t = tile_col<TP, RP, CPLX>(cg, j);
          if (t < T4) {
#pragma unroll
            for (int i = 0; i < 4; ++i) sU[(p0 + i) * UP + t] = t < T ? v[i][j] : 0.f;
          }
        }
      };
      __syncthreads();  // every thread is done with Z'
      put_rows(u);
      __syncthreads();
      gram_add();  // ---- 5. ----
      if constexpr (CPLX) {
        if constexpr (TS::SEP) {
          if (MODE == PM_INIT)
            take_rows<TP, RP, CPLX>(ui, T, cg, zrow_i);
          else
            contract<TP, RP, CPLX>(ui, sV, sW, sV, b.Vw, T, cg, zrow_i);
        }
        __syncthreads();
        put_rows(ui);
        __syncthreads();
        gram_add();
      }
    }
  }

  // ---- CTA partials: the groups' blocks added in group order ----
  const int TT = T * T;
  if (kGram) {
    __syncthreads();
    if (nblk <= kWideThreads) {
      float* red = sZ;  // [ngrp][nblk][16]
      if (gbi[0] >= 0) {
#pragma unroll
        for (int i = 0; i < 16; ++i) red[(size_t)tid * 16 + i] = gacc[0][i];
      }
      __syncthreads();
      for (int e = tid; e < nblk * 16; e += kWideThreads) {
        float s = 0.f;
        for (int g = 0; g < ngrp; ++g) s += red[(size_t)g * nblk * 16 + e];
        int bi, bj;
        tri_coords(e / 16, nb, bi, bj);
        const int a = 4 * bi + (e % 16) / 4, c = 4 * bj + e % 4;
        if (a < T && c < T && a <= c) {
          b.gram_part[(int64_t)lc * TT + a * T + c] = s;
          b.gram_part[(int64_t)lc * TT + c * T + a] = s;
        }
      }
    } else {
#pragma unroll
      for (int uu = 0; uu < TS::BPT; ++uu) {
        if (gbi[uu] < 0) continue;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int a = 4 * gbi[uu] + i / 4, c = 4 * gbj[uu] + i % 4;
          if (a < T && c < T && a <= c) {
            b.gram_part[(int64_t)lc * TT + a * T + c] = gacc[uu][i];
            b.gram_part[(int64_t)lc * TT + c * T + a] = gacc[uu][i];
          }
        }
      }
    }
  }
  {
    const double v0 = warp_sum_d((double)e2), v1 = warp_sum_d((double)l1);
    if (lane == 0) {
      sRed[0][w] = v0;
      sRed[1][w] = v1;
    }
    __syncthreads();
    if (tid == 0) {
      double s0 = 0, s1 = 0;
      for (int i = 0; i < NW; ++i) {
        s0 += sRed[0][i];
        s1 += sRed[1][i];
      }
      b.scal_part[2 * lc] = s0;
      b.scal_part[2 * lc + 1] = s1;
    }
  }
  return cross_cta_reduce<4>(b, kGram, sScal, &sLast, lc, nc);
}

// CTAs per SM: 16 warps of 128 registers a thread (two CTAs of 64 registers spill).
__host__ __device__ constexpr int tile_blocks_per_sm(int, bool) { return 1; }

template <int TP, int RP, int MODE, bool CPLX>
__global__ void __launch_bounds__(kWideThreads, tile_blocks_per_sm(TP, CPLX)) pass_tile_kernel(Bufs b) {
  extern __shared__ __align__(16) float tile_smem[];
  pass_tile_body<TP, RP, MODE, CPLX>(b, blockIdx.x, gridDim.x, tile_smem);
}

#include "rpca_wide_tc.cuh"

// The B operand images of the tiled tensor-core pass (b.wtc), written by the
// eigen-step once Ww and Vw are final.
__device__ __forceinline__ void wtc_images(const Bufs& b, const float* v, int sn, int sk, int rank, int nr) {
  const int TP = wtc_tp(b.T);
  if (b.wtc == 1) {
    if (TP == 64) wtc_write_images<64, false>(b, v, sn, sk, rank, nr);
    else if (TP == 96) wtc_write_images<96, false>(b, v, sn, sk, rank, nr);
    else if (TP == 128) wtc_write_images<128, false>(b, v, sn, sk, rank, nr);
  } else if (b.wtc == 2) {
    if (TP == 64) wtc_write_images<64, true>(b, v, sn, sk, rank, nr);
    else if (TP == 96) wtc_write_images<96, true>(b, v, sn, sk, rank, nr);
    else if (TP == 128) wtc_write_images<128, true>(b, v, sn, sk, rank, nr);
  }
}

#include "rpca_eig_wide.cuh"

// The eigen-step of a plan of at most kMaxT real columns on the tiled path: the
// narrow one on one CTA, then the operand images.  The cluster's products and
// barriers cost more there than the whole narrow step: measured, a 4-frame
// complex 64 x 64 window 1.43 -> 0.75 ms a solve.
static __global__ void __launch_bounds__(kEigThreads) eig_small_kernel(Bufs b, int flags, cudaGraphConditionalHandle h,
                                                                       int use_cond, int) {
  extern __shared__ __align__(16) unsigned char eigs_smem[];
  if (eig64_body<true>(b, flags, h, use_cond, eigs_smem) && b.wtc) {
    __syncthreads();  // Ww and Vw written
    wtc_images(b, b.Vw, 1, b.T, 0, 1);
  }
}

}  // namespace rpca
