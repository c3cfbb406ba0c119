// rpca_eig64.cuh -- the narrow eigen-step (T <= 32): from the reduced Gram of
// the rotated Z to Wbar and the next basis, to well beyond FP32 (included inside
// namespace rpca by rpca_kernels.cuh).  One CTA of kEigThreads threads, or the
// threads of a batch's CTA.  Windows of the tiled path with at most 32 real
// columns (complex ones of up to 16 frames, short ones in a batch with long
// ones) take it too (b.wide says where G, V and Wbar lie).
//
// GB300 runs FP64 at about 1/64 of its FP32 rate, so FP64 Jacobi sweeps bound
// this step (262144 x 20: 105 us, of which 83 us sweeps; x 29: 310 us).  Here the
// sweeps run in FP32 (rpca_jacobi.cuh) and only propose the eigenvectors U; what
// the iteration uses is then formed from the Gram G and the basis V by products
// whose sums are carried as two-float (hi, lo) pairs (Dot2 of Ogita, Rump and
// Oishi, "Accurate sum and dot product", 2005: about 2^-46 of the terms) on the
// FP32 pipe:
//   Vn = V U,  Omega = Vn^T Vn - I,  H = G U,  Gp = U^T H   (= Vn^T (Z^T Z) Vn)
// Omega is what U and the FP32-rounded V lack in orthonormality.  The larger
// eigenvalue's vector keeps its direction: P = Vn (I - C), C_pq = Omega_pq for the
// larger p, Omega_pp / 2 on the diagonal, so to first order
//   P^T (Z^T Z) P = diag(d) + E,  d_p = Gp_pp (1 - Omega_pp),
//                                 E_pq = Gp_pq - max(d_p, d_q) Omega_pq.
// Wbar = f(Z^T Z) with f(sigma^2) = min(1, tau / sigma) is then
//   I - P (diag(1 - g) - F o E) P^T,  F the divided differences of f
// (g_divided_difference), right to first order in E and Omega; only the vectors
// with sigma > tau enter it, so the others need not be separated from one another
// and the sweeps stop once what is neglected is about the result's FP32 rounding,
// the kink of f at tau included (rpca_eig_rule.cuh).  A step that finds more left
// runs another round of sweeps on diag(d) + E.  sigma, the sigma > tau decision, g and mu are FP64.  Measured on
// the windows above: 26 us (load 3, factor and sweeps 13, products and decisions 10)
// and 38 to 40 us, at 0.84 to 0.95 of the errors of L and S against 64 bits (means of
// 12 seeds: 1.0e-7 and 2.2e-7).
#pragma once

constexpr int kEigThreads = 256;   // threads of the eigen-step CTA
constexpr int kEigPasses = 8;      // rounds of sweeps one eigen-step may take
constexpr float kEigStop = 3e-3f;  // largest cosine a sweep may meet and be the last
constexpr float kEigInitStop = 1e-5f;  // ... of the first eigen-step, whose largest eigenvalue sets mu
constexpr float kEigNear = 0.25f;       // a sweep's cosines count where the longer column's sigma^2 / tau^2 is above this

struct Eig64Smem {
  static constexpr int LD = kMaxT + 1;
  static constexpr int N = kMaxT * LD;
  float W[jac_floats(kMaxT)];         // columns of the Cholesky factor, then of L Q
  float Gh[N], Gl[N];                 // G (scaled), columns and rows in descending order of the diagonal
  float Vh[N], Vl[N];                 // the basis, columns in that order; then P
  float U[N];
  float Nh[N], Nl[N];                 // Vn; then K = P (diag(1 - g) - F o E)
  float Hh[N], Hl[N];                 // H
  float Om[N], E[N], C[N], B[N];
  double d[kMaxT];
  float sig[kMaxT], gh[kMaxT], gl[kMaxT] /* 1 - g */, diag[kMaxT], piv[kMaxT], nrm[kMaxT];
  int perm[kMaxT], keep[kMaxT];
  unsigned smax[2], lift;
};

// Dot2: (s, c) += a b, with the rounding errors of the product and of the sum in c.
__device__ __forceinline__ void dot2(float& s, float& c, float a, float b) {
  const float p = __fmul_rn(a, b);
  const float e = fmaf(a, b, -p);
  const float t = __fadd_rn(s, p);
  const float z = __fsub_rn(t, s);
  c = __fadd_rn(c, __fadd_rn(__fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z)), e));
  s = t;
}
// (h, l) = s + c, normalised
__device__ __forceinline__ void fast_two_sum(float s, float c, float& h, float& l) {
  h = __fadd_rn(s, c);
  l = __fsub_rn(c, __fsub_rn(h, s));
}

// Returns whether the solve goes on (Wbar and V are written).  COND: whether the kernel
// may drive a graph's loop; without, it holds no code that does (ncu does not profile
// kernel nodes that could).
template <bool COND>
static __device__ __noinline__ bool eig64_body(Bufs b, int flags, cudaGraphConditionalHandle h, int use_cond,
                                               unsigned char* dsm) {
  Eig64Smem& S = *reinterpret_cast<Eig64Smem*>(dsm);
  constexpr int LD = Eig64Smem::LD;
  __shared__ EigCtl sCtl;
  __shared__ double sTau;

  Ctrl* ctrl = b.ctrl;
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nwarps = nthr >> 5;
  if constexpr (!COND) use_cond = 0;
  const int T = b.T, TT = T * T;
  const int JL = jac_ld(T), nb = jac_blocks(T);
  const unsigned long long t0 = gtimer();
  const bool init = (flags & EF_INIT) != 0;
  float* Vg = b.wide ? b.Vw : b.eig->V32;
  float* Wg = b.wide ? b.Ww : b.eig->Wbar;
  const double* Gg = b.wide ? b.Gw : b.red->G;
  const int ldg = b.wide ? T : kMaxT;

  // T x T arrays: row = warp, warp + 8, ..., column = lane.  Upper triangles: entries
  // (ep, eq) of this thread (at most ceil(528 / 256) = 3).
  const int NE = T * (T + 1) / 2;
  int ep[3], eq[3];
#pragma unroll
  for (int u = 0; u < 3; ++u) {
    int e = tid + u * nthr, p = 0;
    const bool in = e < NE;
    if (in) tri_coords(e, T, p, e);
    ep[u] = in ? p : -1;
    eq[u] = e;
  }

  // the basis (its loads overlap the control part's)
  float v0[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = warp + u * nwarps;
    v0[u] = init ? (r == lane ? 1.f : 0.f) : (r < T && lane < T) ? __ldcg(&Vg[r * ldg + lane]) : 0.f;
  }
  const bool go = eig_control(b, flags, h, use_cond, &sCtl, [&](int i0, int n) {
    if (b.finalize) {
      for (int i = i0; i < TT; i += n) {
        const int r = i / T, c = i % T;
        const double x = __ldcg(&Gg[r * ldg + c]);
        const float xh = (float)x;
        S.Hh[r * LD + c] = xh;
        S.Hl[r * LD + c] = (float)(x - (double)xh);
      }
    } else {
      sum_rows(b.group_part, 0, __ldcg(&b.red->ngroups_last), TT, [&](int e, float gh, float gl) {
        S.Hh[e / T * LD + e % T] = gh;
        S.Hl[e / T * LD + e % T] = gl;
      }, i0, n);
    }
  });
  if (!go) {
    if (tid == nthr - 1) eig_control_tail(b, &sCtl);
    return false;
  }

  // ---- the Gram scaled by a power of four to about 1; the basis ----
  const int pw = even_exponent(T <= 32 && lane < T ? S.Hh[lane * LD + lane] : 0.f);
  const float scale = exp2i(-pw), rootf = exp2i(-pw / 2);
  __syncthreads();
  static_assert(kEigThreads / 32 * 4 >= kMaxT, "four rows a warp");
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = warp + u * nwarps;
    if (r >= T || lane >= T) break;
    S.Hh[r * LD + lane] *= scale;
    S.Hl[r * LD + lane] *= scale;
    S.Nh[r * LD + lane] = v0[u];
    S.Nl[r * LD + lane] = 0.f;
  }
  if (tid < 2) S.smax[tid] = 0u;
  if (tid == 0) S.lift = 0u;
  if (tid == 0) sTau = sCtl.tau;
  const double root = (double)rootf;
  __syncthreads();
  const unsigned long long t1 = gtimer();
  unsigned long long t2 = t1, t3 = t1;
  int sweeps = 0, pass = 0, more = 0;
  const double mu_prev = init ? __ldcg(&ctrl->mu_cur) : 0.0;  // (of the plan's previous solve)
  for (;; ++pass) {
    // ---- descending order of the diagonal; Cholesky factor; one-sided Jacobi ----
    // (every warp works the order out and writes the same values)
    const float dl = lane < T ? S.Hh[lane * LD + lane] : 0.f;
    int pos = 0;
#pragma unroll 4
    for (int j = 0; j < T; ++j) {
      const float dj = S.Hh[j * LD + j];
      pos += (int)(dj > dl) | ((int)(dj == dl) & (int)(j < lane));
    }
    if (lane < T) S.perm[pos] = lane;
    __syncwarp();
    auto perm = [&](int i) { return min((unsigned)S.perm[i < T ? i : 0], (unsigned)(T - 1)); };  // (in range for any values)
    const int pl = perm(lane);
    // a further round's matrix may be indefinite: shifted by at least twice its most
    // negative eigenvalue it has a factor, and the same eigenvectors
    const float lift = 2.f * __uint_as_float(S.lift);
    for (int c = warp; c < 4 * nb; c += nwarps) {
      const int pc = perm(c);
      if (lane < 16 * jac_r2(T))
        S.W[c * JL + lane] = (lane < T && c <= lane) ? S.Hh[pl * LD + pc] + (c == lane ? lift : 0.f) : 0.f;
      if (c < T && lane < T) {
        const float gh = S.Hh[pc * LD + pl];
        S.Gh[c * LD + lane] = gh;
        S.Gl[c * LD + lane] = S.Hl[pc * LD + pl];
        S.Vh[c * LD + lane] = S.Nh[c * LD + pl];
        S.Vl[c * LD + lane] = S.Nl[c * LD + pl];
        if (c == lane) S.diag[c] = gh + lift;
      }
    }
    __syncthreads();
    jac_cholesky<1>(S.W, JL, T, S.diag, S.piv);
    // the pairs that Wbar depends on: those with a singular value near or above tau
    // (the first step wants them all: its tau comes from its eigenvalues)
    const float taus = (float)(sTau * root);
    const float lim = init ? 0.f : fminf(kEigNear * taus * taus, 0.5f * S.diag[0]);
    const float stop = init ? kEigInitStop : kEigStop;
    const int cap = (init || (flags & EF_FULL)) ? 16 : 8;
    sweeps += jac_r2(T) == 1 ? jac_sweeps<1>(S.W, JL, nb, S.nrm, S.smax, stop, lim, cap)
                             : jac_sweeps<2>(S.W, JL, nb, S.nrm, S.smax, stop, lim, cap);
    for (int c = warp; c < T; c += nwarps) {
      const float x = lane < T ? S.W[c * JL + lane] : 0.f;
      float n = x * x;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
      if (lane < T) S.U[lane * LD + c] = n > 0.f ? x * rsqrtf(n) : (lane == c ? 1.f : 0.f);
    }
    __syncthreads();
    if (tid < 2) S.smax[tid] = 0u;  // (every warp has left the sweeps)
    if (tid == 0) S.lift = 0u;
    t2 = gtimer();
    // ---- Vn = V U, H = G U ----
#pragma unroll 1
    for (int r = warp; r < T; r += nwarps) {
      if (lane >= T) break;
      const int c = lane;
      float s = 0.f, e = 0.f, hs = 0.f, he = 0.f;
#pragma unroll 2
      for (int k = 0; k < T; ++k) {
        const float u = S.U[k * LD + c];
        dot2(s, e, S.Vh[r * LD + k], u);
        e = fmaf(S.Vl[r * LD + k], u, e);
        dot2(hs, he, S.Gh[r * LD + k], u);
        he = fmaf(S.Gl[r * LD + k], u, he);
      }
      fast_two_sum(s, e, S.Nh[r * LD + c], S.Nl[r * LD + c]);
      fast_two_sum(hs, he, S.Hh[r * LD + c], S.Hl[r * LD + c]);
    }
    __syncthreads();
    // ---- Omega = Vn^T Vn - I, Gp = U^T H (upper triangles; Gp stays in registers) ----
    float gph[3], gpl[3];
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      if (u * kEigThreads >= NE) break;
      const int p = ep[u], q = eq[u];
      if (p < 0) continue;
      float s = p == q ? -1.f : 0.f, e = 0.f, gs = 0.f, ge = 0.f;
#pragma unroll 2
      for (int k = 0; k < T; ++k) {
        const float ph = S.Nh[k * LD + p], qh = S.Nh[k * LD + q];
        dot2(s, e, ph, qh);
        e = fmaf(ph, S.Nl[k * LD + q], fmaf(S.Nl[k * LD + p], qh, e));
        const float up = S.U[k * LD + p];
        dot2(gs, ge, up, S.Hh[k * LD + q]);
        ge = fmaf(up, S.Hl[k * LD + q], ge);
      }
      S.Om[p * LD + q] = __fadd_rn(s, e);
      fast_two_sum(gs, ge, gph[u], gpl[u]);
      if (p == q) {
        const double gp = (double)gph[u] + (double)gpl[u];
        S.d[p] = gp - gp * (double)S.Om[p * LD + p];
      }
    }
    __syncthreads();
    // ---- FP64 decisions: mu (first call), tau, sigma > tau, g ----
    if (init && tid == 0) {
      double lmax = 0.0;
      for (int a = 0; a < T; ++a) lmax = fmax(lmax, S.d[a]);
      init_mu(b, lmax / (double)scale, mu_prev);
      sTau = ctrl->inv_cur;
    }
    if (init) __syncthreads();
    if (tid < T) {
      const double tau = sTau * root;
      // 1 / sigma by one third-order (Halley) step from its FP32 value: a few FP64
      // operations where a square root and a division would take tens
      const double dv = S.d[tid];
      const bool pos = dv > 1e-36;  // (scaled by the largest: below that it is rounding)
      const double y0 = pos ? (double)rsqrtf((float)dv) : 0.0;
      const double er = fma(-dv * y0, y0, 1.0);
      const double y = fma(y0 * er, fma(er, 0.375, 0.5), y0);
      const double sg = pos ? dv * y : 0.0;
      const int keep = sg > tau;
      const double g1 = keep ? fma(-tau, y, 1.0) : 0.0;
      S.keep[tid] = keep;
      S.sig[tid] = (float)sg;
      S.gh[tid] = (float)g1;
      S.gl[tid] = (float)(g1 - (double)(float)g1);
    }
    __syncthreads();
    // ---- E, C and -F o E ----
    const float tauf = (float)(sTau * root);
    more = 0;
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      const int p = ep[u], q = eq[u];
      if (p < 0) continue;
      const float om = S.Om[p * LD + q];
      if (p == q) {
        S.C[p * LD + p] = 0.5f * om;
        S.E[p * LD + p] = 0.f;
        S.B[p * LD + p] = 0.f;
        continue;
      }
      const bool pbig = S.d[p] >= S.d[q];
      const float dm = (float)(pbig ? S.d[p] : S.d[q]);
      const float sp = fmaxf(S.sig[p], S.sig[q]), sq = fminf(S.sig[p], S.sig[q]);
      const float ev = fmaf(-dm, om, gph[u]) + gpl[u];
      S.C[p * LD + q] = pbig ? om : 0.f;
      S.C[q * LD + p] = pbig ? 0.f : om;
      S.E[p * LD + q] = ev;
      S.E[q * LD + p] = ev;
      const float bv = -g_divided_difference(sp, sq, tauf) * ev;
      S.B[p * LD + q] = bv;
      S.B[q * LD + p] = bv;
    }
    __syncthreads();
    // ---- P = Vn (I - C); whether E is small enough (rpca_eig_rule.cuh) ----
#pragma unroll 1
    for (int r = warp; r < T; r += nwarps) {
      const int c = lane < T ? lane : 0;
      float s = 0.f;
#pragma unroll 4
      for (int k = 0; k < T; ++k) s = fmaf(S.Nh[r * LD + k], S.C[k * LD + c], s);
      const float sr = S.sig[r], sc = S.sig[c], ev = fabsf(S.E[r * LD + c]);
      const float hi = fmaxf(sr, sc), lo = fminf(sr, sc), om = fabsf(S.Om[min(r, c) * LD + max(r, c)]);
      const int kept = S.keep[r] + S.keep[c];
      const bool pair = lane < T && r != c;
      if (pair && kept && eig_pair_off(ev, om, hi, lo, kept)) more = 1;
      auto row_off = [&](float shift) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) shift += __shfl_xor_sync(0xffffffffu, shift, o);
        return eig_row_off(S.keep[r], sr, shift, tauf);
      };
      // (a bound without divisions first: few rows lie near tau)
      if (row_off(pair && kept != 1 ? eig_pair_most(ev, om, hi) : 0.f) &&
          row_off(pair && kept != 1 ? eig_pair_shift(ev, om, hi, lo) : 0.f))
        more = 1;
      if (lane < T) fast_two_sum(S.Nh[r * LD + c], S.Nl[r * LD + c] - s, S.Vh[r * LD + c], S.Vl[r * LD + c]);
    }
    more = __syncthreads_or(more);
    if (!more || pass + 1 == kEigPasses) break;
    // another round on diag(d) + E in the basis P; how far below zero its eigenvalues may
    // lie (the row bound of the stopping rule)
#pragma unroll 1
    for (int r = warp; r < T; r += nwarps) {
      const int c = lane < T ? lane : 0;
      const float dr = (float)S.d[r], dc = (float)S.d[c];
      float below = lane >= T ? 0.f : r == c ? -dr : eig_shift(fabsf(S.E[r * LD + c]), fabsf(dr - dc));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) below += __shfl_xor_sync(0xffffffffu, below, o);
      if (lane == 0 && below > 0.f) atomicMax(&S.lift, __float_as_uint(below));
      if (lane >= T) continue;
      const double x = r == c ? S.d[r] : (double)S.E[r * LD + c];
      const float xh = (float)x;
      S.Hh[r * LD + c] = xh;
      S.Hl[r * LD + c] = (float)(x - (double)xh);
      S.Nh[r * LD + c] = S.Vh[r * LD + c];
      S.Nl[r * LD + c] = S.Vl[r * LD + c];
    }
    __syncthreads();
  }
  t3 = gtimer();
  // ---- K = P (diag(1 - g) - F o E), then Wbar = I - K P^T (upper triangle, mirrored) ----
  if (tid == nthr - 1) eig_control_tail(b, &sCtl);
#pragma unroll 1
  for (int r = warp; r < T; r += nwarps) {
    if (lane >= T) break;
    const int c = lane;
    float s = 0.f;
#pragma unroll 4
    for (int k = 0; k < T; ++k) s = fmaf(S.Vh[r * LD + k], S.B[k * LD + c], s);
    const float ph = S.Vh[r * LD + c], gh = S.gh[c];
    const float p = __fmul_rn(ph, gh);
    const float e = fmaf(ph, gh, -p) + fmaf(ph, S.gl[c], S.Vl[r * LD + c] * gh);
    fast_two_sum(p, e + s, S.Nh[r * LD + c], S.Nl[r * LD + c]);
    Vg[r * ldg + c] = ph;  // (normalised: the pair rounded to FP32)
  }
  const int rank = __syncthreads_count(tid < T && S.keep[tid]);
#pragma unroll
  for (int u = 0; u < 3; ++u) {
    const int p = ep[u], q = eq[u];
    if (p < 0) continue;
    float s = p == q ? -1.f : 0.f, e = 0.f;
#pragma unroll 2
    for (int k = 0; k < T; ++k) {
      const float kh = S.Nh[p * LD + k], ph = S.Vh[q * LD + k];
      dot2(s, e, kh, ph);
      e = fmaf(kh, S.Vl[q * LD + k], fmaf(S.Nl[p * LD + k], ph, e));
    }
    const float w = -(s + e);
    Wg[p * ldg + q] = w;
    Wg[q * ldg + p] = w;
  }
  if (tid < T) (b.wide ? b.evw : b.eig->evals)[tid] = S.d[tid] / (double)scale;
  if (tid == 0) {
    ctrl->rank = rank;
    ctrl->sweeps = sweeps;
    ctrl->total_sweeps += sweeps;
    const unsigned long long t4 = gtimer();
    ctrl->eig_ns += t4 - t0;
    ctrl->eig_cnt += 1;
    ctrl->eig_phase_ns[0] += t1 - t0;
    ctrl->eig_phase_ns[1] += t2 - t1;
    ctrl->eig_phase_ns[2] += t3 - t2;
    ctrl->eig_phase_ns[3] += t4 - t3;
    ctrl->eig_rounds += sweeps * (nb - 1);
    ctrl->eig_further += pass;
    ctrl->eig_unfinished += more ? 1 : 0;
    set_cond(h, use_cond, 1u);
  }
  return true;
}

static __global__ void __launch_bounds__(kEigThreads) eig64_kernel(Bufs b, int flags, cudaGraphConditionalHandle h,
                                                                   int use_cond) {
  extern __shared__ __align__(16) unsigned char eig64_smem_raw[];
  eig64_body<true>(b, flags, h, use_cond, eig64_smem_raw);
}
