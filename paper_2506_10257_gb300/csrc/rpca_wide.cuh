// rpca_wide.cuh -- the iteration for windows of many frames (kMaxT < T <= kMaxTW) and for
// complex windows: device bodies and kernels (host side in rpca_wide.cu).
//
// Same algebra as the register-resident path (see rpca_device.cuh): per
// iteration one fused pass over the pixels (Eq. 4-6 through the Gram of Z, the
// residual of Sec. II-A, and the rotated Gram of the next Z) and one
// eigen-step on one CTA.  With T up to 224 a pixel row no longer fits in one
// thread's registers, so the pass works on tiles of 32 pixels x TP frames
// (TP = T rounded up to a multiple of 32) staged in shared memory:
//   1. X, S, Y of the tile -> shared memory, frame-major [t][p] (coalesced);
//   2. Q = Z Wbar (Z = X - S + Y/mu formed on the fly), Wbar streamed through
//      shared memory 32 rows at a time; lane = pixel, warp = 1/8 of the
//      columns, so every Wbar read is a warp-wide broadcast;
//   3. the Eq. 5-6 update of the lane's pixel for the warp's frames, S' and
//      Y' written straight to HBM (coalesced), Z' kept in shared memory;
//   4. U = Z' V (the next Gram's basis), written pixel-major;
//   5. the partial Gram U^T U accumulated in registers across the CTA's tiles
//      (4 x 4 blocks of the upper triangle spread over the CTA's threads).
// The CTA partials go through the same two-level reduction as the narrow path.
//
// The eigen-step is in rpca_eig_wide.cuh.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include "rpca_kernels.cuh"

namespace rpca {

constexpr int kWP = 32;           // pixels per tile (one per lane)
// Frame rows per warp whose loads the tiled passes' staging issues together:
// the compiler cannot tell the staging's shared-memory stores from the global
// loads that follow them, so a load placed after a store waits for the store's
// operand, i.e. for the previous load.
constexpr int kResLd = 4;
constexpr int kWKC = 32;          // rows of Wbar / V staged per step
constexpr int kWideThreads = 256;

template <int CW>
struct WideShape {
  static constexpr int TP = 8 * CW;               // padded frames (8 warps x CW columns)
  static constexpr int UP = TP + 4;               // row stride of the pixel-major U
  static constexpr int NB = TP / 4;               // 4-frame blocks
  static constexpr int NBLK = NB * (NB + 1) / 2;  // upper-triangle 4 x 4 blocks of the Gram
  static constexpr int BPT = (NBLK + kWideThreads - 1) / kWideThreads;  // blocks per thread
  static constexpr size_t smem = sizeof(float) * (3 * (size_t)TP * kWP + (size_t)kWKC * TP);
  static_assert(CW % 4 == 0, "columns per warp must be a multiple of 4");
  static_assert((size_t)kWP * UP <= 2 * (size_t)TP * kWP, "U must fit in the S and Y tiles");
};

// Dynamic shared memory of the tiled pass with CW columns per warp.
__host__ __device__ constexpr size_t wide_pass_smem_bytes(int CW) {
  return sizeof(float) * (3 * (size_t)(8 * CW) * kWP + (size_t)kWKC * (8 * CW));
}

// Stages rows [k0, k0 + kWKC) of a T x T row-major matrix into sM[kWKC][TP]
// (zero outside T x T).
template <int TP>
__device__ __forceinline__ void stage_rows(float* sM, const float* M, int k0, int T) {
  for (int i = threadIdx.x; i < kWKC * TP; i += kWideThreads) {
    const int r = i / TP, c = i % TP;
    const int k = k0 + r;
    sM[i] = (k < T && c < T) ? __ldcg(&M[(size_t)k * T + c]) : 0.f;
  }
}

// acc[j] = sum_t z(t) * M[t][w*CW + j], z(t) from zfun(t), M streamed from
// global, in increasing t; column pairs share one paired FMA (fma.rn.f32x2).
template <int CW, typename ZF>
__device__ __forceinline__ void tile_times(float (&acc)[CW], float* sM, const float* M, int T, int w, ZF zfun) {
  constexpr int TP = WideShape<CW>::TP;
  uint64_t a2[CW / 2];  // a2[h] = (acc[2h], acc[2h + 1])
#pragma unroll
  for (int h = 0; h < CW / 2; ++h) a2[h] = 0;  // (+0.f, +0.f)
  for (int k0 = 0; k0 < T; k0 += kWKC) {
    __syncthreads();
    stage_rows<TP>(sM, M, k0, T);
    __syncthreads();
    const int kn = min(kWKC, T - k0);
    for (int kk = 0; kk < kn; ++kk) {
      const float z = zfun(k0 + kk);
      const uint64_t zz = f2_pack(z, z);
      const float4* row = reinterpret_cast<const float4*>(&sM[kk * TP + w * CW]);
#pragma unroll
      for (int j4 = 0; j4 < CW / 4; ++j4) {
        const float4 v = row[j4];
        a2[2 * j4] = f2_fma(zz, f2_pack(v.x, v.y), a2[2 * j4]);
        a2[2 * j4 + 1] = f2_fma(zz, f2_pack(v.z, v.w), a2[2 * j4 + 1]);
      }
    }
  }
#pragma unroll
  for (int h = 0; h < CW / 2; ++h) {
    const float2 v = f2_unpack(a2[h]);
    acc[2 * h] = v.x;
    acc[2 * h + 1] = v.y;
  }
}

// CPLX: complex windows as their interleaved real embedding (column 2t = Re,
// 2t + 1 = Im of frame t; T = 2 x frames).  The Hermitian Gram Z^H Z is the
// real Gram of the 2m rows a = [Re z, Im z] and b = a P = [-Im z, Re z] (the
// row of i z) per pixel, so the pass adds both rows of every pixel to the
// Gram; the shrink of Eq. 5 acts on the magnitude of each complex entry.
template <int CW, int MODE, bool CPLX>
__device__ bool pass_wide_body(Bufs b, int lc, int nc, float* wide_smem) {
  using WS = WideShape<CW>;
  constexpr int TP = WS::TP;
  constexpr int UP = CPLX ? TP : WS::UP;       // U row stride (complex: 64 rows over the S, Y tiles)
  constexpr int NROWS = CPLX ? 2 * kWP : kWP;  // Gram rows per tile
  constexpr bool kGram = (MODE != PM_UPDATE);
  float* sX = wide_smem;               // [TP][kWP]
  float* sS = sX + TP * kWP;           // [TP][kWP]
  float* sY = sS + TP * kWP;           // [TP][kWP]
  float* sM = sY + TP * kWP;           // [kWKC][TP]
  float* sU = sS;                      // [NROWS][UP], over the S and Y tiles once they are used
  __shared__ double sRed[2][kWideThreads / 32];
  __shared__ double sScal[2 * kMaxGroups];
  __shared__ int sLast;

  const Ctrl* ctrl = b.ctrl;
  if (solve_done_uniform(ctrl)) return false;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (tid == 0) atomicMin(&b.red->t_start, gtimer());
  const int T = b.T;
  const int64_t m = b.m;
  const Job job = *b.job;
  const int kc = __ldcg(&ctrl->k);
  const bool first = (kc == 0) && !__ldcg(&ctrl->warm);
  const float f_mu = __ldcg(&ctrl->f_mu), inv_mu = __ldcg(&ctrl->f_inv_mu), gamma = __ldcg(&ctrl->f_gamma);
  const float inv_mu_nxt = __ldcg(&ctrl->f_inv_mu_nxt);
  const float* Yin = (kc & 1) ? job.Y1 : job.Y0;
  float* Yout = (kc & 1) ? job.Y0 : job.Y1;

  // Gram blocks owned by this thread
  int gbi[WS::BPT], gbj[WS::BPT];
  float gacc[WS::BPT][16];
#pragma unroll
  for (int u = 0; u < WS::BPT; ++u) {
    const int blk = tid + u * kWideThreads;
    gbi[u] = gbj[u] = -1;
    if (blk < WS::NBLK) blk_coords(blk, WS::NB, gbi[u], gbj[u]);
#pragma unroll
    for (int i = 0; i < 16; ++i) gacc[u][i] = 0.f;
  }
  float e2 = 0.f, l1 = 0.f;

  const int64_t ntiles = (m + kWP - 1) / kWP;
  for (int64_t tile = lc; tile < ntiles; tile += nc) {
    const int64_t p = tile * kWP + lane;
    const bool valid = p < m;
    __syncthreads();  // the previous tile's U is consumed
    // ---- 1. stage the tile (frame-major); the loads of kResLd frame rows
    //      per warp are issued before their shared-memory stores ----
    if constexpr (CPLX) {
      const float2* X2 = reinterpret_cast<const float2*>(job.X);
      const float2* S2 = reinterpret_cast<const float2*>(job.S);
      const float2* Y2 = reinterpret_cast<const float2*>(Yin);
      constexpr int G = kResLd / 2;
      static_assert((TP / 2) % (8 * G) == 0, "whole groups of frame rows");
      for (int f0 = w; f0 < TP / 2; f0 += 8 * G) {
        float2 xg[G], sg[G], yg[G];
#pragma unroll
        for (int i = 0; i < G; ++i) {
          const int f = f0 + 8 * i;
          const bool in = valid && 2 * f < T;
          const int64_t gi = in ? (int64_t)f * m + p : 0;
          xg[i] = in ? X2[gi] : make_float2(0.f, 0.f);
          sg[i] = (MODE != PM_INIT && in && !first) ? S2[gi] : make_float2(0.f, 0.f);
          yg[i] = (MODE != PM_INIT && in && !first) ? Y2[gi] : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < G; ++i) {
          const int f = f0 + 8 * i;
          const float2 x = xg[i];
          sX[(2 * f) * kWP + lane] = x.x;
          sX[(2 * f + 1) * kWP + lane] = x.y;
          if (MODE == PM_INIT) {
            const float a2 = fmaf(x.x, x.x, x.y * x.y);
            e2 += a2;
            l1 += sqrtf(a2);
          } else {
            sS[(2 * f) * kWP + lane] = sg[i].x;
            sS[(2 * f + 1) * kWP + lane] = sg[i].y;
            sY[(2 * f) * kWP + lane] = yg[i].x;
            sY[(2 * f + 1) * kWP + lane] = yg[i].y;
          }
        }
      }
    } else {
      constexpr int G = kResLd;
      static_assert(TP % (8 * G) == 0, "whole groups of frame rows");
      for (int t0 = w; t0 < TP; t0 += 8 * G) {
        float xg[G], sg[G], yg[G];
#pragma unroll
        for (int i = 0; i < G; ++i) {
          const int t = t0 + 8 * i;
          const bool in = valid && t < T;
          const int64_t gi = in ? (int64_t)t * m + p : 0;
          xg[i] = in ? job.X[gi] : 0.f;
          sg[i] = (MODE != PM_INIT && in && !first) ? job.S[gi] : 0.f;
          yg[i] = (MODE != PM_INIT && in && !first) ? Yin[gi] : 0.f;
        }
#pragma unroll
        for (int i = 0; i < G; ++i) {
          const int t = t0 + 8 * i;
          const float x = xg[i];
          sX[t * kWP + lane] = x;
          if (MODE == PM_INIT) {
            e2 = fmaf(x, x, e2);
            l1 += fabsf(x);
          } else {
            sS[t * kWP + lane] = sg[i];
            sY[t * kWP + lane] = yg[i];
          }
        }
      }
    }
    __syncthreads();
    if (MODE == PM_INIT) {
      // U = X (standard basis), pixel-major; complex: also the rows of i X
      for (int i = tid; i < TP * kWP; i += kWideThreads) {
        const int t = i / kWP, pp = i % kWP;
        sU[pp * UP + t] = sX[t * kWP + pp];
        if (CPLX) sU[(kWP + pp) * UP + t] = (t & 1) ? sX[(t - 1) * kWP + pp] : -sX[(t + 1) * kWP + pp];
      }
    } else {
      if (MODE != PM_GRAM) {
        // ---- 2. Q = Z Wbar ----
        float q[CW];
        tile_times<CW>(q, sM, b.Ww, T, w, [&](int t) {
          return form_z(sX[t * kWP + lane], sS[t * kWP + lane], sY[t * kWP + lane], inv_mu);
        });
        __syncthreads();  // every warp has read the whole tile before Z' overwrites X
        // ---- 3. Eq. 5-6 for (lane's pixel, warp's frames) ----
        if constexpr (CPLX) {
          float2* S2 = reinterpret_cast<float2*>(job.S);
          float2* Yo2 = reinterpret_cast<float2*>(Yout);
#pragma unroll
          for (int j = 0; j < CW; j += 2) {
            const int t = w * CW + j;   // even: (Re, Im) of frame t / 2
            if (t < T) {
              const float xr = sX[t * kWP + lane], xi = sX[(t + 1) * kWP + lane];
              const float sr = sS[t * kWP + lane], si = sS[(t + 1) * kWP + lane];
              const float yr = sY[t * kWP + lane], yi = sY[(t + 1) * kWP + lane];
              const float rr = sr + q[j], ri = si + q[j + 1];
              const float mag = sqrtf(fmaf(rr, rr, ri * ri));
              const float f = (mag > gamma) ? gamma / mag : 1.f;   // clip to the disc of radius gamma
              const float cr = rr * f, ci = ri * f;
              const float snr = rr - cr, sni = ri - ci;           // Eq. 5 (magnitude shrink)
              const float ynr = f_mu * cr, yni = f_mu * ci;       // Eq. 6
              const float er = cr - yr * inv_mu, ei = ci - yi * inv_mu;
              e2 = fmaf(er, er, fmaf(ei, ei, e2));
              if (valid) {
                S2[(int64_t)(t >> 1) * m + p] = make_float2(snr, sni);
                Yo2[(int64_t)(t >> 1) * m + p] = make_float2(ynr, yni);
              }
              sX[t * kWP + lane] = valid ? form_z(xr, snr, ynr, inv_mu_nxt) : 0.f;
              sX[(t + 1) * kWP + lane] = valid ? form_z(xi, sni, yni, inv_mu_nxt) : 0.f;
            }
          }
        } else {
#pragma unroll
          for (int j = 0; j < CW; ++j) {
            const int t = w * CW + j;
            if (t < T) {
              const float x = sX[t * kWP + lane], s = sS[t * kWP + lane], y = sY[t * kWP + lane];
              const float r = s + q[j];
              const float c = fminf(fmaxf(r, -gamma), gamma);
              const float sn = r - c;
              const float yn = f_mu * c;
              const float e = c - y * inv_mu;
              e2 = fmaf(e, e, e2);
              if (valid) {
                job.S[(int64_t)t * m + p] = sn;
                Yout[(int64_t)t * m + p] = yn;
              }
              // Z' of the next iteration replaces X in the tile (only this thread reads it)
              sX[t * kWP + lane] = valid ? form_z(x, sn, yn, inv_mu_nxt) : 0.f;
            }
          }
        }
      } else {
        // Z of the current iterate in place of X
        for (int t = w; t < T; t += 8)
          sX[t * kWP + lane] = form_z(sX[t * kWP + lane], sS[t * kWP + lane], sY[t * kWP + lane], inv_mu);
      }
      if (kGram) {
        // ---- 4. U = Z' V, pixel-major over the dead S, Y tiles ----
        float u[CW];
        tile_times<CW>(u, sM, b.Vw, T, w, [&](int t) { return sX[t * kWP + lane]; });
        __syncthreads();  // every warp is done reading S, Y (aliased by U)
        float4* dst = reinterpret_cast<float4*>(&sU[lane * UP + w * CW]);
#pragma unroll
        for (int j4 = 0; j4 < CW / 4; ++j4) dst[j4] = make_float4(u[4 * j4], u[4 * j4 + 1], u[4 * j4 + 2], u[4 * j4 + 3]);
        if constexpr (CPLX) {
          // rows of i Z': (-Im, Re) per frame, in the same basis
          tile_times<CW>(u, sM, b.Vw, T, w, [&](int t) {
            return (t & 1) ? sX[(t - 1) * kWP + lane] : -sX[(t + 1) * kWP + lane];
          });
          float4* dstb = reinterpret_cast<float4*>(&sU[(kWP + lane) * UP + w * CW]);
#pragma unroll
          for (int j4 = 0; j4 < CW / 4; ++j4)
            dstb[j4] = make_float4(u[4 * j4], u[4 * j4 + 1], u[4 * j4 + 2], u[4 * j4 + 3]);
        }
      }
    }
    if (kGram) {
      __syncthreads();
      // ---- 5. partial Gram U^T U (upper 4 x 4 blocks) ----
#pragma unroll
      for (int uu = 0; uu < WS::BPT; ++uu) {
        if (gbi[uu] < 0) continue;
        const int bi = gbi[uu], bj = gbj[uu];
        uint64_t g2[8];  // g2[2i + h] = (gacc[4i + 2h], gacc[4i + 2h + 1])
#pragma unroll
        for (int i = 0; i < 8; ++i) g2[i] = f2_pack(gacc[uu][2 * i], gacc[uu][2 * i + 1]);
        for (int pp = 0; pp < NROWS; ++pp) {
          const float4 a = *reinterpret_cast<const float4*>(&sU[pp * UP + 4 * bi]);
          const float4 c = *reinterpret_cast<const float4*>(&sU[pp * UP + 4 * bj]);
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
          gacc[uu][2 * i] = v.x;
          gacc[uu][2 * i + 1] = v.y;
        }
      }
    }
  }

  // ---- CTA partials ----
  const int TT = T * T;
  if (kGram) {
#pragma unroll
    for (int uu = 0; uu < WS::BPT; ++uu) {
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
  {
    const double v0 = warp_sum_d((double)e2), v1 = warp_sum_d((double)l1);
    if (lane == 0) {
      sRed[0][w] = v0;
      sRed[1][w] = v1;
    }
    __syncthreads();
    if (tid == 0) {
      double s0 = 0, s1 = 0;
      for (int i = 0; i < kWideThreads / 32; ++i) {
        s0 += sRed[0][i];
        s1 += sRed[1][i];
      }
      b.scal_part[2 * lc] = s0;
      b.scal_part[2 * lc + 1] = s1;
    }
  }
  return cross_cta_reduce<4>(b, kGram, sScal, &sLast, lc, nc);
}

template <int CW, int MODE, bool CPLX>
__global__ void __launch_bounds__(kWideThreads, 1) pass_wide_kernel(Bufs b) {
  extern __shared__ __align__(16) float wide_smem[];
  pass_wide_body<CW, MODE, CPLX>(b, blockIdx.x, gridDim.x, wide_smem);
}

// ---------------------------------------------------------------------------
// Tiled pass with Wbar and V resident in shared memory (TP <= 128 columns).
// Tiles of 64 pixels; thread (tx, ty) of a 16 x 16 grid owns 4 pixels x TP/16
// columns of both contractions (register-blocked: per k one 16-byte load of
// Z and TP/16 values of Wbar or V feed 4 TP/16 FMAs).  The tile holds Z (in
// place of X), S and Y/mu; Z' = Z - Y/mu - Q + clip(R) + Y'/mu' needs no X.
// ---------------------------------------------------------------------------
constexpr int kRP = 64;   // pixels per tile

// Shared-memory position of pixel pp of frame row t in the frame-major tiles
// (Z, S, Y/mu): rows of 64 pixels, the pixel index XOR-ed with 4 * ((t / 4) % 8)
// so that the Eq. 5-6 update, whose threads walk down the columns of a tile 4
// rows apart, spreads over eight banks instead of one; groups of 4 pixels stay
// contiguous and 16-byte aligned for the contractions' vector loads.
__device__ __forceinline__ int res_at(int t, int pp) { return t * kRP + (pp ^ (((t >> 2) & 7) << 2)); }

template <int TP, bool CPLX>
struct ResShape {
  static constexpr int CPT = TP / 16;                     // columns per thread
  static constexpr int NR = CPLX ? 2 * kRP : kRP;         // Gram rows per tile
  static constexpr int UP = CPLX ? TP : TP + 4;           // U row stride
  static constexpr int NB = TP / 4;
  static constexpr int NBLK = NB * (NB + 1) / 2;
  static constexpr int BPT = (NBLK + kWideThreads - 1) / kWideThreads;
  static constexpr size_t floats = 2 * (size_t)TP * TP + 3 * (size_t)TP * kRP;
  static constexpr size_t smem = sizeof(float) * floats;
  static_assert(TP % 32 == 0 && TP <= 128, "resident tiles need TP in {32, 64, 96, 128}");
  static_assert((size_t)NR * UP <= 2 * (size_t)TP * kRP, "U must fit over the S and Y/mu tiles");
};

__host__ __device__ constexpr size_t res_pass_smem_bytes(int TP) {
  return sizeof(float) * (2 * (size_t)TP * TP + 3 * (size_t)TP * kRP);
}

// acc[i][j] = sum_k zrow(k)[i] * M[k][c0 + j], 4 pixels i, CPT columns j, in
// increasing k; column pairs (j, j + 1) share one paired FMA (fma.rn.f32x2)
template <int TP, typename ZF>
__device__ __forceinline__ void res_times(float (&acc)[4][TP / 16], const float* sM, int T, int c0, ZF zrow) {
  constexpr int CPT = TP / 16;
  uint64_t a2[4][CPT / 2];  // a2[i][h] = (acc[i][2h], acc[i][2h + 1])
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int h = 0; h < CPT / 2; ++h) a2[i][h] = 0;  // (+0.f, +0.f)
  for (int k = 0; k < T; ++k) {
    const float4 z = zrow(k);
    const float2* wr = reinterpret_cast<const float2*>(&sM[k * TP + c0]);
    const uint64_t zz[4] = {f2_pack(z.x, z.x), f2_pack(z.y, z.y), f2_pack(z.z, z.z), f2_pack(z.w, z.w)};
#pragma unroll
    for (int h = 0; h < CPT / 2; ++h) {
      const float2 v = wr[h];
      const uint64_t w2 = f2_pack(v.x, v.y);
#pragma unroll
      for (int i = 0; i < 4; ++i) a2[i][h] = f2_fma(zz[i], w2, a2[i][h]);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int h = 0; h < CPT / 2; ++h) {
      const float2 v = f2_unpack(a2[i][h]);
      acc[i][2 * h] = v.x;
      acc[i][2 * h + 1] = v.y;
    }
}

template <int TP, int MODE, bool CPLX>
__device__ bool pass_res_body(Bufs b, int lc, int nc, float* smem) {
  using RS = ResShape<TP, CPLX>;
  constexpr int CPT = RS::CPT;
  constexpr int UP = RS::UP;
  constexpr bool kGram = (MODE != PM_UPDATE);
  float* sW = smem;                    // Wbar [TP][TP]
  float* sV = sW + TP * TP;            // V [TP][TP]
  float* sZ = sV + TP * TP;            // [TP][kRP]: X, then Z, then Z'
  float* sS = sZ + TP * kRP;           // [TP][kRP]
  float* sD = sS + TP * kRP;           // [TP][kRP]: Y / mu
  float* sU = sS;                      // [NR][UP], over S and Y/mu once they are used
  __shared__ double sRed[2][kWideThreads / 32];
  __shared__ double sScal[2 * kMaxGroups];
  __shared__ int sLast;

  const Ctrl* ctrl = b.ctrl;
  if (solve_done_uniform(ctrl)) return false;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int tx = tid & 15, ty = tid >> 4;     // column group, pixel group
  const int c0 = tx * CPT, p0 = 4 * ty;
  if (tid == 0) atomicMin(&b.red->t_start, gtimer());
  const int T = b.T;
  const int64_t m = b.m;
  const Job job = *b.job;
  const int kc = __ldcg(&ctrl->k);
  const bool first = (kc == 0) && !__ldcg(&ctrl->warm);
  const float f_mu = __ldcg(&ctrl->f_mu), inv_mu = __ldcg(&ctrl->f_inv_mu), gamma = __ldcg(&ctrl->f_gamma);
  const float inv_mu_nxt = __ldcg(&ctrl->f_inv_mu_nxt);
  const float* Yin = (kc & 1) ? job.Y1 : job.Y0;
  float* Yout = (kc & 1) ? job.Y0 : job.Y1;

  // Wbar and V resident for the whole pass (zero outside T x T)
  if (MODE != PM_INIT) {
    for (int i = tid; i < TP * TP; i += kWideThreads) {
      const int r = i / TP, c = i % TP;
      const bool in = r < T && c < T;
      sW[i] = in ? __ldcg(&b.Ww[r * T + c]) : 0.f;
      sV[i] = in ? __ldcg(&b.Vw[r * T + c]) : 0.f;
    }
  }

  int gbi[RS::BPT], gbj[RS::BPT];
  float gacc[RS::BPT][16];
#pragma unroll
  for (int u = 0; u < RS::BPT; ++u) {
    const int blk = tid + u * kWideThreads;
    gbi[u] = gbj[u] = -1;
    if (blk < RS::NBLK) blk_coords(blk, RS::NB, gbi[u], gbj[u]);
#pragma unroll
    for (int i = 0; i < 16; ++i) gacc[u][i] = 0.f;
  }
  float e2 = 0.f, l1 = 0.f;

  const int64_t ntiles = (m + kRP - 1) / kRP;
  for (int64_t tile = lc; tile < ntiles; tile += nc) {
    const int64_t pb = tile * kRP;
    __syncthreads();  // the previous tile (and the resident matrices) are ready / consumed
    // ---- 1. stage: warp w takes frames w, w + 8, ...; lane l pixels l, l + 32;
    //      the loads of kResLd frame rows per warp are issued before their
    //      shared-memory stores ----
    if constexpr (CPLX) {
      const float2* X2 = reinterpret_cast<const float2*>(job.X);
      const float2* S2 = reinterpret_cast<const float2*>(job.S);
      const float2* Y2 = reinterpret_cast<const float2*>(Yin);
      constexpr int G = kResLd / 2;   // TP / 2 is a multiple of 16
      for (int f0 = w; f0 < TP / 2; f0 += 8 * G) {
        float2 xg[G][2], sg[G][2], yg[G][2];
#pragma unroll
        for (int i = 0; i < G; ++i)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int f = f0 + 8 * i, pp = lane + 32 * h;
            const bool in = (pb + pp < m) && 2 * f < T;
            const int64_t gi = in ? (int64_t)f * m + pb + pp : 0;
            xg[i][h] = in ? X2[gi] : make_float2(0.f, 0.f);
            sg[i][h] = (MODE != PM_INIT && in && !first) ? S2[gi] : make_float2(0.f, 0.f);
            yg[i][h] = (MODE != PM_INIT && in && !first) ? Y2[gi] : make_float2(0.f, 0.f);
          }
#pragma unroll
        for (int i = 0; i < G; ++i)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int f = f0 + 8 * i, pp = lane + 32 * h;
            const float2 x = xg[i][h];
            if (MODE == PM_INIT) {
              sZ[res_at(2 * f, pp)] = x.x;
              sZ[res_at(2 * f + 1, pp)] = x.y;
              const float a2 = fmaf(x.x, x.x, x.y * x.y);
              e2 += a2;
              l1 += sqrtf(a2);
            } else {
              const float2 sv = sg[i][h], yv = yg[i][h];
              sZ[res_at(2 * f, pp)] = form_z(x.x, sv.x, yv.x, inv_mu);
              sZ[res_at(2 * f + 1, pp)] = form_z(x.y, sv.y, yv.y, inv_mu);
              sS[res_at(2 * f, pp)] = sv.x;
              sS[res_at(2 * f + 1, pp)] = sv.y;
              sD[res_at(2 * f, pp)] = yv.x * inv_mu;
              sD[res_at(2 * f + 1, pp)] = yv.y * inv_mu;
            }
          }
      }
    } else {
      constexpr int G = kResLd;       // TP is a multiple of 32
      for (int t0 = w; t0 < TP; t0 += 8 * G) {
        float xg[G][2], sg[G][2], yg[G][2];
#pragma unroll
        for (int i = 0; i < G; ++i)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int t = t0 + 8 * i, pp = lane + 32 * h;
            const bool in = (pb + pp < m) && t < T;
            const int64_t gi = in ? (int64_t)t * m + pb + pp : 0;
            xg[i][h] = in ? job.X[gi] : 0.f;
            sg[i][h] = (MODE != PM_INIT && in && !first) ? job.S[gi] : 0.f;
            yg[i][h] = (MODE != PM_INIT && in && !first) ? Yin[gi] : 0.f;
          }
#pragma unroll
        for (int i = 0; i < G; ++i)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int t = t0 + 8 * i, pp = lane + 32 * h;
            const float x = xg[i][h];
            if (MODE == PM_INIT) {
              sZ[res_at(t, pp)] = x;
              e2 = fmaf(x, x, e2);
              l1 += fabsf(x);
            } else {
              const float sv = sg[i][h], yv = yg[i][h];
              sZ[res_at(t, pp)] = form_z(x, sv, yv, inv_mu);
              sS[res_at(t, pp)] = sv;
              sD[res_at(t, pp)] = yv * inv_mu;
            }
          }
      }
    }
    __syncthreads();
    auto zrow = [&](int k) { return *reinterpret_cast<const float4*>(&sZ[res_at(k, p0)]); };
    auto zrow_i = [&](int k) {  // rows of i Z (complex): (-Im, Re) per frame
      const float4 v = (k & 1) ? *reinterpret_cast<const float4*>(&sZ[res_at(k - 1, p0)])
                               : *reinterpret_cast<const float4*>(&sZ[res_at(k + 1, p0)]);
      return (k & 1) ? v : make_float4(-v.x, -v.y, -v.z, -v.w);
    };
    if (MODE == PM_INIT) {
      // U = X (standard basis), pixel-major; complex: also the rows of i X
      for (int i = tid; i < TP * kRP; i += kWideThreads) {
        const int t = i / kRP, pp = i % kRP;
        sU[pp * UP + t] = sZ[res_at(t, pp)];
        if (CPLX) sU[(kRP + pp) * UP + t] = (t & 1) ? sZ[res_at(t - 1, pp)] : -sZ[res_at(t + 1, pp)];
      }
    } else {
      if (MODE != PM_GRAM) {
        // ---- 2. Q = Z Wbar ----
        float q[4][CPT];
        res_times<TP>(q, sW, T, c0, zrow);
        __syncthreads();  // every thread has read Z before Z' replaces it
        // ---- 3. Eq. 5-6 for (4 pixels, CPT columns) ----
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int pp = p0 + i;
          const bool valid = pb + pp < m;
          if constexpr (CPLX) {
            float2* S2 = reinterpret_cast<float2*>(job.S);
            float2* Yo2 = reinterpret_cast<float2*>(Yout);
#pragma unroll
            for (int j = 0; j < CPT; j += 2) {
              const int t = c0 + j;
              if (t < T) {
                const float zr = sZ[res_at(t, pp)], zi = sZ[res_at(t + 1, pp)];
                const float sr = sS[res_at(t, pp)], si = sS[res_at(t + 1, pp)];
                const float dr = sD[res_at(t, pp)], di = sD[res_at(t + 1, pp)];
                const float rr = sr + q[i][j], ri = si + q[i][j + 1];
                const float mag = sqrtf(fmaf(rr, rr, ri * ri));
                const float f = (mag > gamma) ? gamma / mag : 1.f;
                const float cr = rr * f, ci = ri * f;
                const float ynr = f_mu * cr, yni = f_mu * ci;
                const float er = cr - dr, ei = ci - di;
                e2 = fmaf(er, er, fmaf(ei, ei, e2));
                if (valid) {
                  S2[(int64_t)(t >> 1) * m + pb + pp] = make_float2(rr - cr, ri - ci);
                  Yo2[(int64_t)(t >> 1) * m + pb + pp] = make_float2(ynr, yni);
                }
                sZ[res_at(t, pp)] = valid ? ((zr - dr) - q[i][j]) + cr + ynr * inv_mu_nxt : 0.f;
                sZ[res_at(t + 1, pp)] = valid ? ((zi - di) - q[i][j + 1]) + ci + yni * inv_mu_nxt : 0.f;
              }
            }
          } else {
#pragma unroll
            for (int j = 0; j < CPT; ++j) {
              const int t = c0 + j;
              if (t < T) {
                const float z = sZ[res_at(t, pp)], sv = sS[res_at(t, pp)], d = sD[res_at(t, pp)];
                const float r = sv + q[i][j];                      // X - L + Y/mu
                const float c = fminf(fmaxf(r, -gamma), gamma);    // clip to +-lambda/mu
                const float yn = f_mu * c;                         // Eq. 6
                const float e = c - d;                             // X - L - S'
                e2 = fmaf(e, e, e2);
                if (valid) {
                  job.S[(int64_t)t * m + pb + pp] = r - c;         // Eq. 5
                  Yout[(int64_t)t * m + pb + pp] = yn;
                }
                // Z' = X - S' + Y'/mu' with X = Z + S - Y/mu and S' = S + Q - clip
                sZ[res_at(t, pp)] = valid ? ((z - d) - q[i][j]) + c + yn * inv_mu_nxt : 0.f;
              }
            }
          }
        }
        __syncthreads();  // Z' complete; S, Y/mu are free for U
      }
      if (kGram) {
        // ---- 4. U = Z' V (complex: and (i Z') V), pixel-major ----
        float u[4][CPT];
        res_times<TP>(u, sV, T, c0, zrow);
        if (MODE == PM_GRAM) __syncthreads();  // (no update phase: S, Y/mu read up to here)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < CPT; ++j) sU[(p0 + i) * UP + c0 + j] = u[i][j];
        if constexpr (CPLX) {
          res_times<TP>(u, sV, T, c0, zrow_i);
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < CPT; ++j) sU[(kRP + p0 + i) * UP + c0 + j] = u[i][j];
        }
      }
    }
    if (kGram) {
      __syncthreads();
      // ---- 5. partial Gram U^T U (upper 4 x 4 blocks) ----
#pragma unroll
      for (int uu = 0; uu < RS::BPT; ++uu) {
        if (gbi[uu] < 0) continue;
        const int bi = gbi[uu], bj = gbj[uu];
        uint64_t g2[8];  // g2[2i + h] = (gacc[4i + 2h], gacc[4i + 2h + 1])
#pragma unroll
        for (int i = 0; i < 8; ++i) g2[i] = f2_pack(gacc[uu][2 * i], gacc[uu][2 * i + 1]);
        for (int pp = 0; pp < RS::NR; ++pp) {
          const float4 a = *reinterpret_cast<const float4*>(&sU[pp * UP + 4 * bi]);
          const float4 c = *reinterpret_cast<const float4*>(&sU[pp * UP + 4 * bj]);
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
          gacc[uu][2 * i] = v.x;
          gacc[uu][2 * i + 1] = v.y;
        }
      }
    }
  }

  // ---- CTA partials ----
  const int TT = T * T;
  if (kGram) {
#pragma unroll
    for (int uu = 0; uu < RS::BPT; ++uu) {
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
  {
    const double v0 = warp_sum_d((double)e2), v1 = warp_sum_d((double)l1);
    if (lane == 0) {
      sRed[0][w] = v0;
      sRed[1][w] = v1;
    }
    __syncthreads();
    if (tid == 0) {
      double s0 = 0, s1 = 0;
      for (int i = 0; i < kWideThreads / 32; ++i) {
        s0 += sRed[0][i];
        s1 += sRed[1][i];
      }
      b.scal_part[2 * lc] = s0;
      b.scal_part[2 * lc + 1] = s1;
    }
  }
  return cross_cta_reduce<4>(b, kGram, sScal, &sLast, lc, nc);
}

// CTAs per SM: two below 64 columns (128 registers a thread), else one.
__host__ __device__ constexpr int res_blocks_per_sm(int TP) { return TP <= 64 ? 2 : 1; }

template <int TP, int MODE, bool CPLX>
__global__ void __launch_bounds__(kWideThreads, res_blocks_per_sm(TP)) pass_res_kernel(Bufs b) {
  extern __shared__ __align__(16) float res_smem[];
  pass_res_body<TP, MODE, CPLX>(b, blockIdx.x, gridDim.x, res_smem);
}

#include "rpca_wide_tc.cuh"

// The B operand images of the tiled tensor-core pass (b.wtc), written by the
// eigen-step once Ww and Vw are final.
__device__ __forceinline__ void wtc_images(const Bufs& b) {
  const int TP = wtc_tp(b.T);
  if (b.wtc == 1) {
    if (TP == 64) wtc_write_images<64, false>(b);
    else if (TP == 96) wtc_write_images<96, false>(b);
    else if (TP == 128) wtc_write_images<128, false>(b);
  } else if (b.wtc == 2) {
    if (TP == 64) wtc_write_images<64, true>(b);
    else if (TP == 96) wtc_write_images<96, true>(b);
    else if (TP == 128) wtc_write_images<128, true>(b);
  }
}

#include "rpca_eig_wide.cuh"

}  // namespace rpca
