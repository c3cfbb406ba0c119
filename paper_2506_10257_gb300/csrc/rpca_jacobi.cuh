// rpca_jacobi.cuh -- the symmetric eigensolver inside every eigen-step: FP32
// one-sided block Jacobi on a Cholesky factor, on one CTA (included inside
// namespace rpca by rpca_kernels.cuh).
//
// The eigen-steps decompose the rotated Gram G (T x T, positive semidefinite,
// nearly diagonal after the first iteration).  With G = L L^T, one-sided
// (Hestenes) rotations make the columns of L Q orthogonal; then L Q = U S, and
// the normalised columns U are the eigenvectors of G, so no product of rotations
// has to be accumulated (Veselic and Hari, "A note on a one-sided Jacobi
// algorithm", 1989).  Only U is taken from here: it may carry the FP32 rounding
// of all rotations, because the callers recompute U^T G U from G itself and
// correct for what is left off its diagonal to first order.
//
// Layout.  Columns are stored one after the other (column stride LD floats) and
// come in blocks of four.  A warp takes a pair of blocks (I, J) into registers:
// lane octet o holds column o of I and one column of J, eight lanes per column,
// rows 2 l8 + 16 k.  A column pair's inner product is then three shuffles, its
// rotation is formed by the octet itself and applied to registers, and the
// columns of J move on to the next octet; after four such steps all 16 pairs of
// the two blocks have been rotated and the blocks go back to shared memory.  One
// CTA barrier per block round (the circle method over the blocks), a quarter of
// the rounds that pairwise ordering needs.  What bounds a step is the chain
// inner product - three shuffles - square root - rotation.
#pragma once

#include "rpca_eig_rule.cuh"

// Row pairs (float2) a lane holds per column: the frame count rounded up to a
// multiple of 16 rows, in the sizes below.
__host__ __device__ constexpr int jac_r2(int T) {
  return T <= 16 ? 1 : T <= 32 ? 2 : T <= 48 ? 3 : T <= 64 ? 4 : T <= 80 ? 5 : T <= 96 ? 6 : T <= 112 ? 7
       : T <= 128 ? 8 : T <= 144 ? 9 : T <= 160 ? 10 : T <= 192 ? 12 : 14;
}
// Column stride: an odd multiple of 16 floats, so that the two columns a
// half-warp reads lie in different halves of the banks (224 rows keep their
// length: the next stride would not fit in shared memory beside the rest).
__host__ __device__ constexpr int jac_ld(int T) {
  const int rows = 16 * jac_r2(T);
  return (rows / 16) % 2 == 1 || rows > 208 ? rows : rows + 16;
}
// Blocks of four columns, rounded up to an even number.
__host__ __device__ constexpr int jac_blocks(int T) { return ((T + 3) / 4 + 1) / 2 * 2; }
__host__ __device__ constexpr size_t jac_floats(int T) { return (size_t)4 * jac_blocks(T) * jac_ld(T); }

constexpr float kJacTol = 1e-6f;    // a pair of smaller cosine is left alone
constexpr float kJacFar = 0.1f;     // weight of the cosine of two short columns in the stopping rule
constexpr float kJacFloor = 1e-6f;  // smallest pivot of the factorisation relative to the diagonal entry

// Upper-triangle block (A, C), A <= C < K, of linear index idx in row order
// (row A holds K - A blocks): closed form with one correction step.
__device__ __forceinline__ void tri_coords(int idx, int K, int& A, int& C) {
  const float k2 = 2.f * K + 1.f;
  int a = (int)floorf(0.5f * (k2 - sqrtf(fmaxf(k2 * k2 - 8.f * (float)idx, 0.f))));
  a = max(0, min(a, K - 1));
  while (a > 0 && a * K - a * (a - 1) / 2 > idx) --a;
  while (a + 1 < K && (a + 1) * K - (a + 1) * a / 2 <= idx) ++a;
  A = a;
  C = a + (idx - (a * K - a * (a - 1) / 2));
}

__device__ __forceinline__ float oct_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v;
}

template <int R2>
__device__ __forceinline__ float oct_dot(const uint64_t (&a)[R2], const uint64_t (&b)[R2]) {
  uint64_t s0 = f2_mul(a[0], b[0]), s1 = 0;
#pragma unroll
  for (int k = 1; k < R2; ++k) {
    if (k & 1)
      s1 = f2_fma(a[k], b[k], s1);
    else
      s0 = f2_fma(a[k], b[k], s0);
  }
  const float2 h = f2_unpack(f2_add(s0, s1));
  return oct_sum(h.x + h.y);
}

// 1 / sqrt(x), the SM's approximation (x a normal number)
__device__ __forceinline__ float rsqrt_fast(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// The rotation (c, s) that makes columns p, q of squared lengths app, aqq and
// inner product d orthogonal, the identity when their cosine is at most kJacTol;
// t = s / c.  With dd = aqq - app and r = 1 / sqrt(dd^2 + 4 d^2), cos 2 theta =
// |dd| r, so c^2 = (1 + |dd| r) / 2 and s = sign(dd) d r / c: two reciprocal
// square roots in a row where the tangent's formula has three steps of that
// length.  Two columns so short that dd^2 + 4 d^2 underflows are left alone too (the
// formula would not be a rotation).  Returns the cosine.
__device__ __forceinline__ float jac_rotation(float app, float aqq, float d, float& c, float& s, float& t) {
  const float cosv = fabsf(d) * (rsqrt_fast(fmaxf(app, 1e-37f)) * rsqrt_fast(fmaxf(aqq, 1e-37f)));
  const float dd = aqq - app, d2 = d + d;
  const float q = fmaf(dd, dd, d2 * d2), r = rsqrt_fast(fmaxf(q, 1e-37f));
  const bool act = cosv > kJacTol && cosv < 1.5f && q >= 1e-37f;  // (a zero column's cosine is zero; not a number is left alone)
  const float c2 = fmaf(0.5f * fabsf(dd), r, 0.5f);
  const float ic = rsqrt_fast(fmaxf(c2, 0.5f));
  c = act ? c2 * ic : 1.f;
  s = act ? copysignf(ic, dd) * (d * r) : 0.f;
  t = s * ic;
  return act ? cosv : 0.f;
}

// The pairs inside a block: octet o holds the block's column o; the columns of
// octets o and o ^ (x / 8) rotate against each other, each octet updating its own.
template <int R2>
__device__ __forceinline__ void jac_within(uint64_t (&a)[R2], float& na, int x, float t2, float& mx) {
  const unsigned full = 0xffffffffu;
  uint64_t o[R2];
#pragma unroll
  for (int k = 0; k < R2; ++k) o[k] = __shfl_xor_sync(full, a[k], x);
  const float no = __shfl_xor_sync(full, na, x);
  const float d = oct_dot<R2>(a, o);
  const bool lower = ((threadIdx.x & 31) & x) < ((threadIdx.x & 31 ^ x) & x);
  float c, s, t;
  const float cosv = jac_rotation(lower ? na : no, lower ? no : na, d, c, s, t);
  mx = fmaxf(mx, fmaxf(na, no) > t2 ? cosv : kJacFar * cosv);
  const float sg = lower ? -s : s;  // p' = c p - s q, q' = s p + c q
  const uint64_t c2 = f2_pack(c, c), s2 = f2_pack(sg, sg);
#pragma unroll
  for (int k = 0; k < R2; ++k) a[k] = f2_fma(s2, o[k], f2_mul(c2, a[k]));
  na = lower ? fmaf(-t, d, na) : fmaf(t, d, na);
}

// Rotates the columns of W (nb blocks) until no pair whose longer column has a
// squared length above t2 was seen with a cosine above `stop` in a whole sweep
// (what such a sweep leaves is quadratically smaller), and none of two shorter
// columns above stop / kJacFar (they must stay a basis), or for max_sweeps sweeps.
// nrm: 4 nb floats; smax: two words, zero on entry.  All threads of the CTA call
// it (after a barrier) and get the number of sweeps; smax is read after its last
// barrier, so the caller resets it after one of its own.
template <int R2>
static __device__ __noinline__ int jac_sweeps(float* W, int LD, int nb, float* nrm, unsigned* smax, float stop, float t2,
                                              int max_sweeps) {
  __builtin_assume(__isShared(W));
  __builtin_assume(__isShared(nrm));
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int o = lane >> 3, l8 = lane & 7;
  int sweep = 0;
  while (sweep < max_sweeps) {
    float mx = 0.f;
    for (int r = 0; r < nb - 1; ++r) {
      for (int task = warp; task < nb / 2; task += nwarps) {
        int bi, bj;
        rr_pair(r, task, nb, bi, bj);
        uint64_t* pa = reinterpret_cast<uint64_t*>(W + (4 * bi + o) * LD + 2 * l8);
        uint64_t* pb = reinterpret_cast<uint64_t*>(W + (4 * bj + o) * LD + 2 * l8);
        uint64_t a[R2], b[R2];
#pragma unroll
        for (int k = 0; k < R2; ++k) {
          a[k] = pa[8 * k];
          b[k] = pb[8 * k];
        }
        float na, nbv;
        if (r == 0) {  // once a sweep: exact lengths, and the pairs inside the blocks
          na = oct_dot<R2>(a, a);
          nbv = oct_dot<R2>(b, b);
#pragma unroll 1
          for (int x = 8; x <= 24; x += 8) {
            jac_within<R2>(a, na, x, t2, mx);
            jac_within<R2>(b, nbv, x, t2, mx);
          }
        } else {
          na = nrm[4 * bi + o];
          nbv = nrm[4 * bj + o];
        }
#pragma unroll 1
        for (int st = 0; st < 4; ++st) {
          const float d = oct_dot<R2>(a, b);
          float c, s, t;
          const float cosv = jac_rotation(na, nbv, d, c, s, t);
          mx = fmaxf(mx, fmaxf(na, nbv) > t2 ? cosv : kJacFar * cosv);
          const uint64_t c2 = f2_pack(c, c), s2 = f2_pack(s, s), n2 = f2_pack(-s, -s);
#pragma unroll
          for (int k = 0; k < R2; ++k) {
            const uint64_t p = a[k], q = b[k];
            a[k] = f2_fma(n2, q, f2_mul(c2, p));
            b[k] = f2_fma(s2, p, f2_mul(c2, q));
          }
          na = fmaf(-t, d, na);
          nbv = fmaf(t, d, nbv);
          // (after the fourth step every octet has its first column of J again)
#pragma unroll
          for (int k = 0; k < R2; ++k) b[k] = __shfl_sync(full, b[k], (lane + 8) & 31);
          nbv = __shfl_sync(full, nbv, (lane + 8) & 31);
        }
#pragma unroll
        for (int k = 0; k < R2; ++k) {
          pa[8 * k] = a[k];
          pb[8 * k] = b[k];
        }
        if (l8 == 0) {
          nrm[4 * bi + o] = na;
          nrm[4 * bj + o] = nbv;
        }
      }
      __syncthreads();
    }
    if (threadIdx.x == 0) smax[(sweep + 1) & 1] = 0u;  // (its last readers passed the barriers above)
    const unsigned m = __reduce_max_sync(full, __float_as_uint(mx));
    if (lane == 0) atomicMax(&smax[sweep & 1], m);
    __syncthreads();
    const float seen = __uint_as_float(smax[sweep & 1]);
    ++sweep;
    if (!(seen > stop)) break;
  }
  return sweep;
}

// The panels of four columns in rows 32 UB .. 32 UB + 31, and what they change
// beyond; rows 32 u + lane, u in [UB, RU), so the row groups above are left out at
// compile time.  v: warp 0's current panel (set by the caller for column 0).
template <int RU, int UB>
__device__ __forceinline__ void jac_chol_rows(float* W, int LD, int T, const float* diag, float* piv, float (&v)[4][RU]) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
#pragma unroll 1
  for (int j0 = 32 * UB; j0 < min(32 * UB + 32, T); j0 += 4) {
    const int l0 = j0 - 32 * UB;  // lane of the panel's first row
    if (warp == 0) {
      // factor the panel in registers
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const bool in = j0 + c < T;
        const float raw = __shfl_sync(full, v[c][UB], l0 + c), floor = in ? fmaxf(kJacFloor * diag[j0 + c], 1e-30f) : 1.f;
        const float pv = fmaxf(raw, floor);
        if (!(raw > floor)) {
#pragma unroll
          for (int u = UB; u < RU; ++u) v[c][u] = 0.f;
        }
        if (lane == l0 + c) v[c][UB] = pv;
        if (lane < l0 + c) v[c][UB] = 0.f;
        if (lane == 0 && in) piv[j0 + c] = pv;
        const float rd = __fdividef(1.f, pv);
#pragma unroll
        for (int e = c + 1; e < 4; ++e) {
          const float f = __shfl_sync(full, v[c][UB], l0 + e) * rd;
#pragma unroll
          for (int u = UB; u < RU; ++u) v[e][u] = fmaf(-f, v[c][u], v[e][u]);
        }
      }
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int u = UB; u < RU; ++u)
          if (j0 + c < T && 32 * u + lane < T) W[(j0 + c) * LD + 32 * u + lane] = v[c][u];
    }
    __syncthreads();
    if (j0 + 4 >= T) break;
    // the columns after the panel: warp 0 takes the next panel and keeps it, the
    // others the rest (their updates are done by the next barrier)
    float rd[4], w[4][RU];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      rd[c] = __fdividef(1.f, piv[j0 + c]);
#pragma unroll
      for (int u = UB; u < RU; ++u) w[c][u] = warp == 0 ? v[c][u] : 32 * u + lane < T ? W[(j0 + c) * LD + 32 * u + lane] : 0.f;
    }
    if (warp == 0) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int k = j0 + 4 + e;
        float f[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) f[c] = k < T ? -rd[c] * W[(j0 + c) * LD + k] : 0.f;
#pragma unroll
        for (int u = UB; u < RU; ++u) {
          float x = k < T && 32 * u + lane < T ? W[k * LD + 32 * u + lane] : 0.f;
#pragma unroll
          for (int c = 0; c < 4; ++c) x = fmaf(f[c], w[c][u], x);
          v[e][u] = x;
        }
      }
    } else {
      for (int k = j0 + 8 + warp - 1; k < T; k += nwarps - 1) {
        float f[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) f[c] = -rd[c] * W[(j0 + c) * LD + k];
#pragma unroll
        for (int u = UB; u < RU; ++u) {
          const int i = 32 * u + lane;
          if (i >= k && i < T) {
            float x = W[k * LD + i];
#pragma unroll
            for (int c = 0; c < 4; ++c) x = fmaf(f[c], w[c][u], x);
            W[k * LD + i] = x;
          }
        }
      }
    }
    __syncthreads();
  }
}
template <int RU, int UB = 0>
__device__ __forceinline__ void jac_chol_all(float* W, int LD, int T, const float* diag, float* piv, float (&v)[4][RU]) {
  if constexpr (UB < RU) {
    jac_chol_rows<RU, UB>(W, LD, T, diag, piv, v);
    jac_chol_all<RU, UB + 1>(W, LD, T, diag, piv, v);
  }
}

// Cholesky factor of the matrix whose lower triangle is in W (column j at
// W + j LD, entry i at + i; zero elsewhere, and zero beyond T), in place, four
// columns at a time: warp 0 factors a panel in registers (lane = row), then all
// warps update the columns after it, warp 0 those of the next panel.  A pivot
// below kJacFloor times its diagonal entry diag[j] (a numerically dependent
// column, or one of a block that rounding left indefinite) is raised to that and
// the rest of its column dropped, so that the columns stay independent and
// bounded.  piv: T floats of scratch.  RU: rows / 32 rounded up.  At least two
// warps; all threads call it after a barrier; it ends with one.
template <int RU>
static __device__ __noinline__ void jac_cholesky(float* W, int LD, int T, const float* diag, float* piv) {
  __builtin_assume(__isShared(W));
  __builtin_assume(__isShared(diag));
  __builtin_assume(__isShared(piv));
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  float v[4][RU];
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int u = 0; u < RU; ++u) v[c][u] = warp == 0 && c < T && 32 * u + lane < T ? W[c * LD + 32 * u + lane] : 0.f;
  jac_chol_all<RU>(W, LD, T, diag, piv, v);
  __syncthreads();
  for (int j = warp; j < T; j += nwarps) {
    const float r = rsqrtf(piv[j]);
    for (int i = j + lane; i < T; i += 32) W[j * LD + i] *= r;
  }
  __syncthreads();
}

// Even e with 2^e about the largest of the warp's values (0 if none is positive
// and finite): scaling a Gram by 2^-e and its singular values by 2^(-e/2) is exact.
__device__ __forceinline__ int even_exponent(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
  if (!(x > 0.f) || !(x <= 3.4e38f)) return 0;
  const int e = (int)(__float_as_uint(x) >> 23) - 127;
  const int ev = e + (e & 1);
  return max(-120, min(120, ev));
}
__device__ __forceinline__ float exp2i(int e) { return __uint_as_float((unsigned)(e + 127) << 23); }

// First-order change of g = min(1, tau / sigma) of the symmetric matrix
// V diag(sigma^2) V^T per unit of its (p, q) entry: the divided difference
// (g_p - g_q) / (sigma_p^2 - sigma_q^2) (Daleckii and Krein), written without
// cancellation; sp >= sq.  Equal arguments give the derivative.
__device__ __forceinline__ float g_divided_difference(float sp, float sq, float tau) {
  if (!(sp > tau)) return 0.f;
  if (sq > tau) return -tau / (sp * sq * (sp + sq));
  return -((sp - tau) / (sp - sq)) / (sp * (sp + sq));
}
