// rpca_eig_wide.cuh -- the eigen-step of wide and complex windows (up to kMaxTW
// real columns), included inside namespace rpca by rpca_wide.cuh.
//
// The algebra is that of the narrow step (rpca_eig64.cuh): FP32 one-sided Jacobi
// proposes the eigenvectors U of the rotated Gram G, and Vn = V U, Omega, H = G U,
// Gp = U^T H, P and Wbar = I - P (diag(1 - g) - F o E) P^T follow from G and V
// themselves.  What Wbar multiplies has components up to 1e4 times as large as the
// smallest it has to get right, so Vn, Omega, P and K P^T carry errors well below
// FP32's rounding: their operands, of unit columns, are split as a = ah + al with
// ah a multiple of 2^-11, so that sums of ah bh are exact in FP32 and ah bl + al b
// adds the rest to about 2^-34 (the splitting of Ozaki, Ogita, Oishi and Rump,
// "Error-free transformations of matrix multiplication", 2012; three FMAs a term
// where a compensated sum takes eleven operations), and Vn, P and K are kept as
// (hi, lo) pairs.  H and Gp, whose errors scale with the entries they belong to, are
// plain FP32 in the form G U = G + G D, D = U - I, but for the first step: its Gram is
// not rotated, every entry holds the largest eigenvalue's share, and G, H and Gp are
// (hi, lo) pairs there (Dot2, as in the narrow step).  With all of them in plain FP32
// the error of L on 64 x 64 x 100 pixels and frames is five times as large.
// The sigma > tau decision, g and mu are FP64.
//
// A step is one thread-block cluster of nr CTAs (one CTA in the batched form):
// rank 0 factors and sweeps with the matrix in its shared memory; the Gram's
// cross-CTA sums and the five T x T x T products are spread over the ranks by
// rows, with every T x T operand in the workspace (L2) and a cluster barrier
// between products.  Bound by the factor and the sweeps on rank 0's SM, which wait
// at its barriers.  Measured with 8 ranks, against cyclic Jacobi on the Gram itself:
// 50 frames 294 -> 124 us (factor and sweeps 50, products 50), 100 frames
// 1106 -> 273 us (168, 66), 132 frames 2313 -> 512 to 550 us (366 to 410, 96).  One CTA,
// beside the other lanes of a batch, takes 238 us at 63 frames and 437 us at 93.
#pragma once

// Matrices of the step's scratch, each eig_ld(T)^2 floats.
enum EigScr { ES_G = 0, ES_GS, ES_VT, ES_D, ES_VN, ES_VNL, ES_VNT, ES_VNTL, ES_H, ES_OM,
              ES_GP, ES_C, ES_B, ES_E, ES_PT, ES_PTL, ES_KT, ES_KTL, ES_COUNT };
__host__ __device__ constexpr int eig_ld(int T) { return (T + 7) / 8 * 8; }
__host__ __device__ constexpr size_t eig_scr_bytes(int T) {
  return sizeof(float) * ES_COUNT * (size_t)eig_ld(T) * eig_ld(T) + sizeof(int) * (kMaxTW + 16);
}

constexpr int kEigWThreads = 512;   // 128 registers a thread: the longest columns of a sweep fit
static_assert(1 + kEigPasses <= 15, "the flags of a step");
constexpr int kEigWRanks = 8;       // CTAs of a plan's eigen-step
constexpr float kEigWStop = 1e-3f;   // largest cosine of a last sweep: 3e-3, as in the narrow step, left one step in
                                    // four of 132 frames short, and a second round costs more than the extra sweeps
constexpr float kEigNoise = 2e-6f;  // FP32 rounding of E relative to the larger eigenvalue (not worth another pass)

// Dynamic shared memory of a step: the columns of the Jacobi sweeps; the products
// stage their operands in the same space.
__host__ __device__ constexpr size_t eig_wide_smem(int T) {
  return sizeof(float) * (jac_floats(T) > 32 * (size_t)eig_ld(T) ? jac_floats(T) : 32 * (size_t)eig_ld(T));
}

// ... of a plan's step, beside what EigWideSh and the control part hold statically.
constexpr size_t kEigWMaxSmem = 216 * 1024;

struct EigWideSh {
  double d[kMaxTW], mu_prev;
  float sig[kMaxTW], g1[kMaxTW], g1l[kMaxTW], diag[kMaxTW], piv[kMaxTW], nrm[kMaxTW];
  int perm[kMaxTW], keep[kMaxTW];
  unsigned smax[2], lift;
  EigCtl ctl;
};

// Barrier over the step's CTAs, ordering their global writes.
__device__ __forceinline__ void eig_sync(int nr) {
  if (nr > 1) {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  } else {
    __syncthreads();
  }
}

// a rounded to a multiple of 2^-11 (|a| < 2^11)
__device__ __forceinline__ float split_hi(float a) { return __fsub_rn(__fadd_rn(a, 6144.f), 6144.f); }

// Copies rows k < K of `quads` float4 each, at src(k, q) in global memory, to
// dst(k, q, value), four loads under way per thread before their stores.
template <typename Src, typename Dst>
__device__ __forceinline__ void stage_quads(int K, int quads, Src src, Dst dst) {
  const int n = K * quads, step = blockDim.x;
  for (int i0 = threadIdx.x; i0 < n; i0 += 4 * step) {
    float4 v[4];
    int k[4], q[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = min(i0 + u * step, n - 1);
      k[u] = i / quads;
      q[u] = i - k[u] * quads;
      v[u] = src(k[u], q[u]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i0 + u * step < n) dst(k[u], q[u], v[u]);
  }
}

// acc(i, j) = sum_k A(k, i) B(k, j) for the RT-row tiles of this rank (tile rows
// rank, rank + nr, ...), k < K, in increasing k; rowa(k) and rowb(k) give the
// global rows (16-byte aligned, ld floats of room), and with SPLIT rowal(k) and
// rowbl(k) those of the operands' low parts (null: none).  out(i0, j0, acc, rest)
// takes a tile; the sum is acc, and acc + rest with SPLIT.  upper: tiles wholly
// below the diagonal are left out.  Operands are staged in shared memory (smf
// floats) for all k, and for all rows and columns of the rank when that fits.
template <int RT, bool SPLIT, typename RA, typename RAL, typename RB, typename RBL, typename Out>
__device__ __forceinline__ void eig_product(int K, int ld, bool upper, int rank, int nr, float* sm, int smf, RA rowa,
                                            RAL rowal, RB rowb, RBL rowbl, Out out) {
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int nt = ld / RT;                                  // tile rows (ld is a multiple of 8)
  const int own = nt > rank ? (nt - rank + nr - 1) / nr : 0;
  const int per_k = smf / K / (SPLIT ? 2 : 1);             // values of room per k
  int jc = ld, ic = own;
  if (ld + own * RT > per_k) {
    jc = max(4, min(ld, per_k / 2) / 4 * 4);
    ic = max(1, min(own, (per_k - jc) / RT));
  }
  for (int t0 = 0; t0 < own; t0 += ic) {
    const int nti = min(ic, own - t0), wa = nti * RT;
    float* sa = sm;
    float* sal = sm + K * wa;
    float* sb = SPLIT ? sal + K * wa : sal;
    auto put = [&](float* hi, float* lo, float4 v, float4 l) {
      if constexpr (SPLIT) {
        const float4 vh = make_float4(split_hi(v.x), split_hi(v.y), split_hi(v.z), split_hi(v.w));
        *reinterpret_cast<float4*>(hi) = vh;
        *reinterpret_cast<float4*>(lo) =
            make_float4((v.x - vh.x) + l.x, (v.y - vh.y) + l.y, (v.z - vh.z) + l.z, (v.w - vh.w) + l.w);
      } else {
        *reinterpret_cast<float4*>(hi) = v;
      }
    };
    auto low = [&](const float* row, int at) {
      return row ? __ldcg(reinterpret_cast<const float4*>(row + at)) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    for (int j0 = 0; j0 < ld; j0 += jc) {
      const int nj = min(jc, ld - j0);
      float* sbl = sb + K * nj;
      __syncthreads();  // (the staging space is free)
      auto cola = [&](int q) { return (rank + (t0 + 4 * q / RT) * nr) * RT + 4 * q % RT; };
      if (j0 == 0)
        stage_quads(K, wa / 4, [&](int k, int q) { return __ldcg(reinterpret_cast<const float4*>(rowa(k) + cola(q))); },
                    [&](int k, int q, float4 v) {
                      const float4 l = SPLIT ? low(rowal(k), cola(q)) : v;
                      put(&sa[k * wa + 4 * q], &sal[k * wa + 4 * q], v, l);
                    });
      stage_quads(K, nj / 4, [&](int k, int q) { return __ldcg(reinterpret_cast<const float4*>(rowb(k) + j0 + 4 * q)); },
                  [&](int k, int q, float4 v) {
                    const float4 l = SPLIT ? low(rowbl(k), j0 + 4 * q) : v;
                    put(&sb[k * nj + 4 * q], &sbl[k * nj + 4 * q], v, l);
                  });
      __syncthreads();
      const int ntj = nj / 4;
      for (int t = tid; t < nti * ntj; t += nthr) {
        const int ti = t / ntj, tj = t % ntj;
        const int i0 = (rank + (t0 + ti) * nr) * RT, jj = j0 + 4 * tj;
        if (upper && jj + 3 < i0) continue;
        uint64_t a2[RT][2], r2[RT][2];
#pragma unroll
        for (int i = 0; i < RT; ++i) a2[i][0] = a2[i][1] = r2[i][0] = r2[i][1] = 0;
        const float* pa = sa + ti * RT;
        const float* pal = sal + ti * RT;
        const float* pb = sb + 4 * tj;
        const float* pbl = sbl + 4 * tj;
#pragma unroll 2
        for (int k = 0; k < K; ++k) {
          const float4 v = *reinterpret_cast<const float4*>(pb + k * nj);
          const uint64_t v0 = f2_pack(v.x, v.y), v1 = f2_pack(v.z, v.w);
          uint64_t l0 = 0, l1 = 0, f0 = 0, f1 = 0;
          if constexpr (SPLIT) {
            const float4 l = *reinterpret_cast<const float4*>(pbl + k * nj);
            l0 = f2_pack(l.x, l.y);
            l1 = f2_pack(l.z, l.w);
            f0 = f2_add(v0, l0);
            f1 = f2_add(v1, l1);
          }
#pragma unroll
          for (int h = 0; h < RT / 4; ++h) {
            const float4 u = *reinterpret_cast<const float4*>(pa + k * wa + 4 * h);
            const float uv[4] = {u.x, u.y, u.z, u.w};
            float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
            if constexpr (SPLIT) w = *reinterpret_cast<const float4*>(pal + k * wa + 4 * h);
            const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const uint64_t uu = f2_pack(uv[i], uv[i]);
              a2[4 * h + i][0] = f2_fma(uu, v0, a2[4 * h + i][0]);
              a2[4 * h + i][1] = f2_fma(uu, v1, a2[4 * h + i][1]);
              if constexpr (SPLIT) {
                const uint64_t ww = f2_pack(wv[i], wv[i]);
                r2[4 * h + i][0] = f2_fma(uu, l0, f2_fma(ww, f0, r2[4 * h + i][0]));
                r2[4 * h + i][1] = f2_fma(uu, l1, f2_fma(ww, f1, r2[4 * h + i][1]));
              }
            }
          }
        }
        float acc[RT][4], rest[RT][4];
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const float2 x = f2_unpack(a2[i][j]), y = f2_unpack(r2[i][j]);
            acc[i][2 * j] = x.x;
            acc[i][2 * j + 1] = x.y;
            rest[i][2 * j] = y.x;
            rest[i][2 * j + 1] = y.y;
          }
        out(i0, jj, acc, rest);
      }
    }
  }
  __syncthreads();
}

// out = c + a^T b in two-float arithmetic for this rank's share of the T x T entries, four
// rows a thread, of (hi, lo) pairs (a null low part: single floats), k increasing; upper:
// only the entries with i <= j, mirrored.  Operands come from L2.  Run once a solve, and
// not inlined, so that the body's own loops keep their place (132 columns, eight ranks: 0.2 ms
// of a 30 ms solve).
static __device__ __noinline__ void eig_product_dd(int T, int ld, bool upper, int rank, int nr, const float* a,
                                                   const float* al, const float* b, const float* bl, const float* c,
                                                   const float* cl, float* out, float* outl) {
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int g = rank * (int)blockDim.x + (int)threadIdx.x; g < (T + 3) / 4 * T; g += nr * (int)blockDim.x) {
    const int i0 = g / T * 4, j = g % T;
    if (upper && j < i0) continue;
    float s[4], r[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      s[u] = __ldcg(&c[(i0 + u) * ld + j]);
      r[u] = __ldcg(&cl[(i0 + u) * ld + j]);
    }
#pragma unroll 4
    for (int k = 0; k < T; ++k) {
      const float4 x = __ldcg(reinterpret_cast<const float4*>(a + k * ld + i0));
      const float4 xl = al ? __ldcg(reinterpret_cast<const float4*>(al + k * ld + i0)) : zero;
      const float y = __ldcg(&b[k * ld + j]), yl = bl ? __ldcg(&bl[k * ld + j]) : 0.f;
      const float xv[4] = {x.x, x.y, x.z, x.w}, xw[4] = {xl.x, xl.y, xl.z, xl.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        dot2(s[u], r[u], xv[u], y);
        r[u] = fmaf(xv[u], yl, fmaf(xw[u], y, r[u]));
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = i0 + u;
      if (i >= T || (upper && i > j)) continue;
      float hi, lo;
      fast_two_sum(s[u], r[u], hi, lo);
      out[i * ld + j] = hi;
      outl[i * ld + j] = lo;
      if (upper) {
        out[j * ld + i] = hi;
        outl[j * ld + i] = lo;
      }
    }
  }
}

// Sweeps for the window's column length.
static __device__ __noinline__ int eig_wide_factor(float* W, int T, EigWideSh& S, float stop, float lim, int cap) {
  const int LD = jac_ld(T), nb = jac_blocks(T), r2 = jac_r2(T);
  if (r2 <= 2) jac_cholesky<1>(W, LD, T, S.diag, S.piv);
  else if (r2 <= 4) jac_cholesky<2>(W, LD, T, S.diag, S.piv);
  else if (r2 <= 8) jac_cholesky<4>(W, LD, T, S.diag, S.piv);
  else if (r2 <= 10) jac_cholesky<5>(W, LD, T, S.diag, S.piv);
  else jac_cholesky<7>(W, LD, T, S.diag, S.piv);
  switch (r2) {
#define RPCA_JAC(R) \
  case R: return jac_sweeps<R>(W, LD, nb, S.nrm, S.smax, stop, lim, cap);
    RPCA_JAC(1) RPCA_JAC(2) RPCA_JAC(3) RPCA_JAC(4) RPCA_JAC(5) RPCA_JAC(6) RPCA_JAC(7) RPCA_JAC(8) RPCA_JAC(9)
    RPCA_JAC(10) RPCA_JAC(12)
#undef RPCA_JAC
    default: return jac_sweeps<14>(W, LD, nb, S.nrm, S.smax, stop, lim, cap);
  }
}

// The step on CTA `rank` of nr; sm holds smf floats (at least eig_wide_smem(T)
// bytes) of shared memory.  RT: rows of a product's tile.
template <int RT>
static __device__ void eig_wide_body(Bufs b, int flags, cudaGraphConditionalHandle h, int use_cond, float* sm, int smf,
                                     int rank, int nr) {
  __shared__ EigWideSh S;
  Ctrl* ctrl = b.ctrl;
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nwarps = nthr >> 5;
  const int T = b.T, TT = T * T, ld = eig_ld(T);
  const size_t msz = (size_t)ld * ld;
  auto M = [&](int i) { return b.eig_scr + i * msz; };
  int* iscr = reinterpret_cast<int*>(b.eig_scr + ES_COUNT * msz);  // perm[kMaxTW], then flags
  int* gflag = iscr + kMaxTW;  // [0] go on, [1 + pass] another pass wanted, [15] scale exponent
  const bool init = (flags & EF_INIT) != 0;
  const unsigned long long t0 = gtimer();

  // ---- the Gram, this rank's share of the sums over the CTAs of the pass ----
  // (the first step's low parts lie where later matrices of the step go)
  float* G = M(ES_G);
  enum { ES_GL = ES_B, ES_GSL = ES_C, ES_HL = ES_KT, ES_GPL = ES_KTL };
  auto put_gram = [&](int e, float gh, float gl) {
    float hi, lo;
    fast_two_sum(gh, gl, hi, lo);
    G[e / T * ld + e % T] = hi;
    if (init) M(ES_GL)[e / T * ld + e % T] = lo;
  };
  auto gram = [&](int i, int n) {
    const int e0 = (int)((int64_t)TT * rank / nr), e1 = (int)((int64_t)TT * (rank + 1) / nr);
    if (b.finalize) {
      for (int e = e0 + i; e < e1; e += n) {
        const double g = __ldcg(&b.Gw[e]);
        put_gram(e, (float)g, (float)(g - (double)(float)g));
      }
    } else if (__ldcg(&b.red->gram_last)) {
      sum_rows<4, 8>(b.group_part, 0, __ldcg(&b.red->ngroups_last), TT, put_gram, i, n, e0, e1);
    }
  };
  bool go;
  if (rank == 0) {
    go = eig_control(b, flags, h, use_cond, &S.ctl, gram);
    if (tid == 0) {
      gflag[0] = go;
      for (int i = 1; i <= kEigPasses; ++i) gflag[i] = 0;
    }
    if (tid == nthr - 1) eig_control_tail(b, &S.ctl);
  } else {
    gram(tid, nthr);
  }
  eig_sync(nr);
  if (rank != 0) go = __ldcg(&gflag[0]) != 0;
  if (!go) return;
  const unsigned long long t1 = gtimer();
  unsigned long long t2 = t1, t3 = t1;
  const float* src = G;            // this pass's Gram
  const float* vt = M(ES_VT);      // the basis, transposed
  float scale = 1.f, rootf = 1.f;
  int sweeps = 0, pass = 0;
  double tau = init ? 0.0 : __ldcg(&ctrl->inv_cur);
  if (init && tid == 0) S.mu_prev = __ldcg(&ctrl->mu_cur);  // (of the plan's previous solve; read by this thread)
  float tauf = 0.f;
  for (;; ++pass) {
    if (rank == 0) {
      // ---- descending order of the diagonal, scaling, factor, sweeps ----
      for (int i = tid; i < T; i += nthr) {
        S.diag[i] = __ldcg(&src[i * ld + i]);
        S.perm[i] = i;
      }
      if (tid < 2) S.smax[tid] = 0u;
      if (tid == 0) S.lift = 0u;
      __syncthreads();
      if (pass > 0) {
        // a further round's matrix may be indefinite: shifted by at least twice its most
        // negative eigenvalue (the row bound of the stopping rule) it has a factor, and the
        // same eigenvectors
        for (int p = warp; p < T; p += nwarps) {
          float below = 0.f;
          for (int q = lane; q < T; q += 32)
            below += q == p ? -S.diag[p] : eig_shift(fabsf(__ldcg(&src[p * ld + q])), fabsf(S.diag[p] - S.diag[q]));
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) below += __shfl_xor_sync(0xffffffffu, below, o);
          if (lane == 0 && below > 0.f) atomicMax(&S.lift, __float_as_uint(below));
        }
      } else {
        float mx = 0.f;
        for (int i = lane; i < T; i += 32) mx = fmaxf(mx, S.diag[i]);
        const int pw = even_exponent(mx);
        scale = exp2i(-pw);
        rootf = exp2i(-pw / 2);
        if (tid == 0) gflag[15] = pw;
      }
      int pos = 0;
      if (tid < T) {
        const float di = S.diag[tid];
#pragma unroll 4
        for (int j = 0; j < T; ++j) {
          const float dj = S.diag[j];
          pos += (int)(dj > di) | ((int)(dj == di) & (int)(j < tid));
        }
      }
      __syncthreads();
      if (tid < T) S.perm[pos] = tid;  // (in range whatever the values are)
      __syncthreads();
      const float sc = pass == 0 ? scale : 1.f, lift = 2.f * __uint_as_float(S.lift);
      const int LD = jac_ld(T), rows = 16 * jac_r2(T);
      for (int c = warp; c < 4 * jac_blocks(T); c += nwarps) {
        const int pc = c < T ? S.perm[c] : 0;
        for (int r = lane; r < rows; r += 32) {
          float v = 0.f;
          if (c < T && r < T) {
            v = __ldcg(&src[pc * ld + S.perm[r]]) * sc;
            M(ES_GS)[c * ld + r] = v;
            if (init && pass == 0) M(ES_GSL)[c * ld + r] = __ldcg(&M(ES_GL)[pc * ld + S.perm[r]]) * sc;
          }
          sm[c * LD + r] = c < r ? v : c == r && r < T ? v + lift : 0.f;
        }
      }
      float dg = 0.f;
      if (tid < T) dg = S.diag[S.perm[tid]] * sc + lift;
      __syncthreads();
      if (tid < T) {
        S.diag[tid] = dg;
        iscr[tid] = S.perm[tid];
      }
      if (init && pass == 0)
        for (int i = tid; i < TT; i += nthr) M(ES_VT)[i / T * ld + i % T] = i / T == i % T ? 1.f : 0.f;
      __syncthreads();
      const float taus = (float)(tau * (double)rootf);
      const float lim = init ? 0.f : fminf(kEigNear * taus * taus, 0.5f * S.diag[0]);
      sweeps += eig_wide_factor(sm, T, S, init ? kEigInitStop : kEigWStop, lim,
                                (init || (flags & EF_FULL)) ? 16 : 8);
      // D = U - I from the normalised columns
      for (int c = warp; c < T; c += nwarps) {
        float n = 0.f;
        for (int r = lane; r < T; r += 32) n = fmaf(sm[c * LD + r], sm[c * LD + r], n);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
        if (lane == 0) S.piv[c] = n > 0.f ? 1.f / sqrtf(n) : 0.f;
      }
      __syncthreads();
      for (int r = warp; r < T; r += nwarps)
        for (int c = lane; c < T; c += 32) {
          const float u = S.piv[c] > 0.f ? sm[c * LD + r] * S.piv[c] : (r == c ? 1.f : 0.f);
          M(ES_D)[r * ld + c] = r == c ? u - 1.f : u;
        }
    }
    eig_sync(nr);
    if (rank != 0) {
      for (int i = tid; i < T; i += nthr) S.perm[i] = __ldcg(&iscr[i]);
      if (pass == 0) {
        const int pw = __ldcg(&gflag[15]);
        scale = exp2i(-pw);
        rootf = exp2i(-pw / 2);
      }
      __syncthreads();
    }
    t2 = gtimer();
    // ---- Vn = V + V D, H = G + G D ----
    auto row = [&](int m) { return [=](int k) { return b.eig_scr + m * msz + (size_t)k * ld; }; };
    auto none = [](int) { return (const float*)nullptr; };
    const float* vtl = pass ? M(ES_PTL) : nullptr;  // (the basis of a further pass is P)
    eig_product<RT, true>(
        T, ld, false, rank, nr, sm, smf, [&](int k) { return vt + S.perm[k] * ld; },
        [&](int k) { return vtl ? vtl + S.perm[k] * ld : nullptr; }, row(ES_D), none,
        [&](int i0, int j0, float (&acc)[RT][4], float (&rest)[RT][4]) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (j0 + j >= T) break;
            const int pj = S.perm[j0 + j] * ld;
#pragma unroll
            for (int i = 0; i < RT; ++i) {
              // V + acc + rest as a (hi, lo) pair (Knuth's TwoSum)
              const float v = __ldcg(&vt[pj + i0 + i]), x = acc[i][j];
              const float s = __fadd_rn(v, x), z = __fsub_rn(s, v);
              const float e = __fadd_rn(__fsub_rn(v, __fsub_rn(s, z)), __fsub_rn(x, z));
              float hi, lo;
              fast_two_sum(s, e + rest[i][j] + (vtl ? __ldcg(&vtl[pj + i0 + i]) : 0.f), hi, lo);
              M(ES_VN)[(i0 + i) * ld + j0 + j] = hi;
              M(ES_VNL)[(i0 + i) * ld + j0 + j] = lo;
              M(ES_VNT)[(j0 + j) * ld + i0 + i] = hi;
              M(ES_VNTL)[(j0 + j) * ld + i0 + i] = lo;
            }
          }
        });
    if (init && pass == 0)
      eig_product_dd(T, ld, false, rank, nr, M(ES_GS), M(ES_GSL), M(ES_D), nullptr, M(ES_GS), M(ES_GSL), M(ES_H), M(ES_HL));
    else
      eig_product<RT, false>(T, ld, false, rank, nr, sm, smf, row(ES_GS), none, row(ES_D), none,
                             [&](int i0, int j0, float (&acc)[RT][4], float (&)[RT][4]) {
#pragma unroll
                               for (int i = 0; i < RT; ++i) {
                                 const float4 g = __ldcg(reinterpret_cast<const float4*>(M(ES_GS) + (i0 + i) * ld + j0));
                                 *reinterpret_cast<float4*>(M(ES_H) + (i0 + i) * ld + j0) =
                                     make_float4(g.x + acc[i][0], g.y + acc[i][1], g.z + acc[i][2], g.w + acc[i][3]);
                               }
                             });
    eig_sync(nr);
    // ---- Omega = Vn^T Vn - I, Gp = U^T H = H + D^T H (upper triangles, mirrored) ----
    eig_product<RT, true>(T, ld, true, rank, nr, sm, smf, row(ES_VN), row(ES_VNL), row(ES_VN), row(ES_VNL),
                          [&](int i0, int j0, float (&acc)[RT][4], float (&rest)[RT][4]) {
#pragma unroll
                            for (int i = 0; i < RT; ++i)
#pragma unroll
                              for (int j = 0; j < 4; ++j) {
                                const int p = i0 + i, q = j0 + j;
                                if (p > q) continue;
                                const float v = (p == q ? acc[i][j] - 1.f : acc[i][j]) + rest[i][j];
                                M(ES_OM)[p * ld + q] = v;
                                M(ES_OM)[q * ld + p] = v;
                              }
                          });
    if (init && pass == 0)
      eig_product_dd(T, ld, true, rank, nr, M(ES_D), nullptr, M(ES_H), M(ES_HL), M(ES_H), M(ES_HL), M(ES_GP), M(ES_GPL));
    else
      eig_product<RT, false>(T, ld, true, rank, nr, sm, smf, row(ES_D), none, row(ES_H), none,
                             [&](int i0, int j0, float (&acc)[RT][4], float (&)[RT][4]) {
#pragma unroll
                               for (int i = 0; i < RT; ++i)
#pragma unroll
                                 for (int j = 0; j < 4; ++j) {
                                   const int p = i0 + i, q = j0 + j;
                                   if (p > q) continue;
                                   const float v = __ldcg(&M(ES_H)[p * ld + q]) + acc[i][j];
                                   M(ES_GP)[p * ld + q] = v;
                                   M(ES_GP)[q * ld + p] = v;
                                 }
                             });
    eig_sync(nr);
    // ---- FP64 decisions (every rank makes the same ones) ----
    for (int i = tid; i < T; i += nthr) {
      const double gp = (double)__ldcg(&M(ES_GP)[i * ld + i]) + (init && pass == 0 ? (double)__ldcg(&M(ES_GPL)[i * ld + i]) : 0.0);
      S.d[i] = gp - gp * (double)__ldcg(&M(ES_OM)[i * ld + i]);
    }
    __syncthreads();
    if (init) {
      if (rank == 0 && tid == 0) {
        double lmax = 0.0;
        for (int a = 0; a < T; ++a) lmax = fmax(lmax, S.d[a]);
        init_mu(b, lmax / (double)scale, S.mu_prev);
      }
      eig_sync(nr);
      tau = __ldcg(&ctrl->inv_cur);
    }
    const double taus = tau * (double)rootf;
    tauf = (float)taus;
    for (int i = tid; i < T; i += nthr) {
      const double dv = S.d[i];
      const bool pos = dv > 1e-36;
      const double y0 = pos ? (double)rsqrtf((float)dv) : 0.0;  // 1 / sigma: one Halley step from FP32
      const double er = fma(-dv * y0, y0, 1.0);
      const double y = fma(y0 * er, fma(er, 0.375, 0.5), y0);
      const double sg = pos ? dv * y : 0.0;
      const int keep = sg > taus;
      S.keep[i] = keep;
      S.sig[i] = (float)sg;
      const double g1 = keep ? fma(-taus, y, 1.0) : 0.0;
      S.g1[i] = (float)g1;
      S.g1l[i] = (float)(g1 - (double)(float)g1);
    }
    __syncthreads();
    // ---- C, -F o E, E, and whether E (beyond its FP32 rounding) and Omega are small enough ----
    const float noise = init ? 0.f : kEigNoise;
    int more = 0;
    for (int p = rank + nr * warp; p < T; p += nr * nwarps) {
      float most = 0.f;
      const float sp = S.sig[p], dp = (float)S.d[p];
      const int kp = S.keep[p];
      for (int q = lane; q < T; q += 32) {
        const float om = __ldcg(&M(ES_OM)[p * ld + q]);
        if (q == p) {
          M(ES_C)[p * ld + p] = 0.5f * om;
          M(ES_B)[p * ld + p] = 0.f;
          M(ES_E)[p * ld + p] = dp;
          continue;
        }
        const float sq = S.sig[q], dq = (float)S.d[q];
        const bool pbig = S.d[p] > S.d[q] || (S.d[p] == S.d[q] && p < q);
        const float hi = fmaxf(sp, sq), lo = fminf(sp, sq), dm = pbig ? dp : dq;
        const float ev = fmaf(-dm, om, __ldcg(&M(ES_GP)[p * ld + q])) + (init && pass == 0 ? __ldcg(&M(ES_GPL)[p * ld + q]) : 0.f);
        M(ES_C)[p * ld + q] = pbig ? om : 0.f;
        M(ES_B)[p * ld + q] = -g_divided_difference(hi, lo, tauf) * ev;
        M(ES_E)[p * ld + q] = ev;
        const float e = fmaxf(fabsf(ev) - noise * dm, 0.f);
        const int kept = kp + S.keep[q];
        if (kept && eig_pair_off(e, fabsf(om), hi, lo, kept)) more = 1;
        if (kept != 1) most += eig_pair_most(e, fabsf(om), hi);
      }
      auto row_off = [&](float shift) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) shift += __shfl_xor_sync(0xffffffffu, shift, o);
        return eig_row_off(kp, sp, shift, tauf);
      };
      if (row_off(most)) {  // (a bound without divisions: few rows lie near tau)
        float shift = 0.f;
        for (int q = lane; q < T; q += 32) {
          if (q == p || S.keep[q] != kp) continue;
          const float sq = S.sig[q], dm = fmaxf(dp, (float)S.d[q]);
          const float e = fmaxf(fabsf(M(ES_E)[p * ld + q]) - noise * dm, 0.f);  // (this lane's own store)
          shift += eig_pair_shift(e, fabsf(__ldcg(&M(ES_OM)[p * ld + q])), fmaxf(sp, sq), fminf(sp, sq));
        }
        if (row_off(shift)) more = 1;
      }
    }
    more = __syncthreads_or(more);
    if (more && tid == 0) atomicOr(&gflag[1 + pass], 1);
    eig_sync(nr);
    const bool last = pass + 1 == kEigPasses || __ldcg(&gflag[1 + pass]) == 0;
    // ---- P = Vn - Vn C ----
    eig_product<RT, false>(T, ld, false, rank, nr, sm, smf, row(ES_VNT), none, row(ES_C), none,
                           [&](int i0, int j0, float (&acc)[RT][4], float (&)[RT][4]) {
#pragma unroll
                             for (int j = 0; j < 4; ++j) {
                               if (j0 + j >= T) break;
#pragma unroll
                               for (int i = 0; i < RT; ++i) {
                                 const size_t at = (size_t)(j0 + j) * ld + i0 + i;
                                 float hi, lo;
                                 fast_two_sum(__ldcg(&M(ES_VNT)[at]), __ldcg(&M(ES_VNTL)[at]) - acc[i][j], hi, lo);
                                 M(ES_PT)[at] = hi;
                                 M(ES_PTL)[at] = lo;
                                 if (last) {
                                   M(ES_VT)[at] = hi;
                                   if (i0 + i < T) b.Vw[(i0 + i) * T + j0 + j] = hi;
                                 }
                               }
                             }
                           });
    if (last) break;
    src = M(ES_E);
    vt = M(ES_PT);
    eig_sync(nr);
  }
  t3 = gtimer();
  // ---- K = P (diag(1 - g) - F o E), Wbar = I - K P^T (upper triangle, mirrored) ----
  auto row = [&](int m) { return [=](int k) { return b.eig_scr + m * msz + (size_t)k * ld; }; };
  auto none = [](int) { return (const float*)nullptr; };
  eig_product<RT, false>(T, ld, false, rank, nr, sm, smf, row(ES_PT), none, row(ES_B), none,
                         [&](int i0, int j0, float (&acc)[RT][4], float (&)[RT][4]) {
#pragma unroll
                           for (int j = 0; j < 4; ++j) {
                             if (j0 + j >= T) break;
                             const float g = S.g1[j0 + j], gl = S.g1l[j0 + j];
#pragma unroll
                             for (int i = 0; i < RT; ++i) {
                               const size_t at = (size_t)(j0 + j) * ld + i0 + i;
                               const float ph = __ldcg(&M(ES_PT)[at]), p = __fmul_rn(ph, g);
                               const float e = fmaf(ph, g, -p) + fmaf(ph, gl, __ldcg(&M(ES_PTL)[at]) * g);
                               // (acc may exceed p where 1 - g is zero: TwoSum)
                               const float x = acc[i][j], s = __fadd_rn(p, x), z = __fsub_rn(s, p);
                               const float r = __fadd_rn(__fsub_rn(p, __fsub_rn(s, z)), __fsub_rn(x, z));
                               M(ES_KT)[at] = s;
                               M(ES_KTL)[at] = r + e;
                             }
                           }
                         });
  eig_sync(nr);
  eig_product<RT, true>(T, ld, true, rank, nr, sm, smf, row(ES_KT), row(ES_KTL), row(ES_PT), row(ES_PTL),
                        [&](int i0, int j0, float (&acc)[RT][4], float (&rest)[RT][4]) {
#pragma unroll
                          for (int i = 0; i < RT; ++i)
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                              const int a = i0 + i, c = j0 + j;
                              if (a > c || c >= T) continue;
                              const float v = (a == c ? 1.f - acc[i][j] : -acc[i][j]) - rest[i][j];
                              b.Ww[a * T + c] = v;
                              b.Ww[c * T + a] = v;
                            }
                        });
  int kept = 0;
  for (int i = tid; i < T; i += nthr) kept += S.keep[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) kept += __shfl_xor_sync(0xffffffffu, kept, o);
  __syncthreads();
  if (lane == 0) S.perm[warp] = kept;
  if (b.wtc) {
    eig_sync(nr);  // Ww and Vw written by every rank
    wtc_images(b, M(ES_VT), ld, 1, rank, nr);
  } else {
    __syncthreads();
  }
  if (rank == 0) {
    for (int i = tid; i < T; i += nthr) b.evw[i] = S.d[i] / (double)scale;
    if (tid == 0) {
      int rk = 0;
      for (int w = 0; w < nwarps; ++w) rk += S.perm[w];
      ctrl->rank = rk;
      ctrl->sweeps = sweeps;
      ctrl->total_sweeps += sweeps;
      const unsigned long long t4 = gtimer();
      ctrl->eig_ns += t4 - t0;
      ctrl->eig_cnt += 1;
      ctrl->eig_phase_ns[0] += t1 - t0;
      ctrl->eig_phase_ns[1] += t2 - t1;
      ctrl->eig_phase_ns[2] += t3 - t2;
      ctrl->eig_phase_ns[3] += t4 - t3;
      ctrl->eig_rounds += sweeps * (jac_blocks(T) - 1);
      ctrl->eig_further += pass;
      ctrl->eig_unfinished += __ldcg(&gflag[1 + pass]);
      set_cond(h, use_cond, 1u);
    }
  }
}

static __global__ void __cluster_dims__(kEigWRanks, 1, 1) __launch_bounds__(kEigWThreads, 1)
    eig_wide_kernel(Bufs b, int flags, cudaGraphConditionalHandle h, int use_cond, int smf) {
  extern __shared__ __align__(16) float eigw_smem[];
  eig_wide_body<4>(b, flags, h, use_cond, eigw_smem, smf, (int)blockIdx.x, kEigWRanks);
}
