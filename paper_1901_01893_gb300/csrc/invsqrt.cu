// IRLS weights W_l = (G_l + eps I)^(-1/2) (the nuclear-norm majoriser of Eq. 10) without an
// eigen-decomposition.
//
// With A = (G + eps I)/c, c >= the largest eigenvalue, the best quadrature of the Cauchy integral
// for the square root on [eps/c, 1] (N. Hale, N. Higham, L. Trefethen, "Computing A^alpha, log(A)
// and related matrix functions by contour integrals", SIAM J. Numer. Anal. 46, 2008, method 3)
// gives W = c^(-1/2) sum_j a_j (A + b_j I)^(-1) with a_j, b_j > 0: 7 terms for c/eps = 100, 13 for
// 1.6e5, error below IS_TOL.  Every term is one Hermitian positive definite inverse by Cholesky,
// and the terms of all matrices are independent: one CTA (C <= 192; a cluster of four above)
// each.  A Jacobi sweep of a 144 x 144 matrix is 143 dependent rounds on two SMs, 3 to 13 sweeps
// per outer iteration; a term is nine dependent block steps and the chip works on every term.
// Measured, the weight step of an outer iteration (mean over a solve; before: Jacobi): two 144 x 144
// matrices 2.14 -> 0.10 ms, 52 of them 2.4 -> 0.44 ms (0.46 with the probe below), four 288 x 288 12.8 -> 0.57 ms.
//
// Accuracy: the terms add without cancellation, and a Cholesky inverse in FP32 is that of a matrix
// off by FP32 rounding, as G itself is once it is held in FP32.  Against the 64-bit weight, on the
// Grams of the 128 x 128 workload over its 20 outer iterations (relative Frobenius error, and of
// G^(1/2) W G^(1/2), what acts on the data): 4e-7 .. 1.8e-4 and 3e-7 .. 4e-6; the Jacobi
// eigensolver 8e-6 .. 1.4e-4 and 1.3e-6 .. 7e-6; W of G rounded to FP32 1.5e-7 .. 7e-5 and 1e-8 ..
// 8e-7.  At eps 1e-5 of the largest eigenvalue (c/eps near 2^20), solves of six geometries, C = 32 .. 288, two
// outer iterations, are 5.8e-7 .. 6.1e-6 from the oracle, with the Jacobi eigensolver 5.8e-7 .. 1.5e-5, and eps_1
// is within 3.4e-7 of its 64-bit value (Jacobi: 1.4e-6).  (A Newton-Schulz iteration for A^(-1/2), which needs GEMMs only, was five times worse
// on the data; a Gauss-Jordan sweep in place of Cholesky a hundred times worse on W.)
//
// eps_1 = eps0_rel times the largest eigenvalue: G is squared IS_SQ times (normalised by its
// trace), S = G^(2^IS_SQ), and tr(G S)/tr(S) is a mean of G's eigenvalues weighted with their
// 2^IS_SQ-th powers (the worst two-eigenvalue gap leaves 0.28 / 2^IS_SQ = 4e-6 of it).
//
// A matrix with c/eps above 2^IS_MAXQ (the start much smaller than the iterates, so that eps is
// near G's FP32 rounding) is left to the eigensolver: is_flag is set and the Jacobi kernels, which
// otherwise return at once, take it.  So is one whose elimination met a pivot below half its shift: every
// pivot of a positive semidefinite G plus the shift is at least the shift, so the rounding of G or of the
// elimination has then made it indefinite.  The eigensolver's weights clamp negative eigenvalues at 0; here they
// stay what they are, which only the reduced-precision Gram makes matter: its three products leave out the
// square of what a value loses to its first BF16 piece, up to 1.4e-5 of the largest eigenvalue.  There one more
// elimination, of G + IS_PROBE eps I, says whether an eigenvalue lies below -IS_PROBE eps (it moves W by 3 %).
#include <math.h>

#include "common.cuh"
#include "jacobi.cuh"

#define IS_TOL 2e-7   // largest relative error of the quadrature
#define IS_SQ 16      // squarings for the largest eigenvalue
#define IS_PROBE 0.0625f
#define RB 16         // block edge of the inverse

// acc.x += a.x * b.x, acc.y += a.y * b.y in one instruction
__device__ __forceinline__ void ffma2(float2& acc, float2 a, float2 b) {
  unsigned long long d = *reinterpret_cast<unsigned long long*>(&acc);
  asm("fma.rn.f32x2 %0, %1, %2, %0;"
      : "+l"(d)
      : "l"(*reinterpret_cast<unsigned long long*>(&a)), "l"(*reinterpret_cast<unsigned long long*>(&b)));
  acc = *reinterpret_cast<float2*>(&d);
}

// G in FP32, scaled by the power of two that brings its largest diagonal entry into [1, 2), and each row's
// sum of |g| and of |g|^2: one warp per row.  (G has the square of the data's scale and is squared again from here
// on: unscaled, data of 2^-45 or 2^30 times unit size left FP32's range.  A power of two changes no bits.)
__global__ void __launch_bounds__(256) k_is_cvt(const double2* __restrict__ G, float2* __restrict__ G32,
                                                float2* __restrict__ rows, IsParam* __restrict__ prm, int C) {
  const int l = blockIdx.y, row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= C) return;
  const size_t off = ((size_t)l * C + row) * C;
  constexpr int NV = (SMSM_MAX_C + 31) / 32;
  double2 g[NV];  // the row's loads and the diagonal's in flight together
#pragma unroll
  for (int k = 0; k < NV; ++k)
    if (lane + 32 * k < C) g[k] = G[off + lane + 32 * k];
  int e = -1023;  // largest exponent of the diagonal (-1023: all zero, 1024: not finite)
  for (int j = lane; j < C; j += 32)
    e = max(e, ((__double2hiint(G[((size_t)l * C + j) * C + j].x) >> 20) & 0x7ff) - 1023);
  for (int o = 16; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
  e = e == -1023 || e == 1024 ? 0 : min(max(e, -126), 126);
  const float scale = __int_as_float((127 - e) << 23);
  if (row == 0 && lane == 0) prm[l].scale = scale;
  float s1 = 0.f, s2 = 0.f;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    if (lane + 32 * k >= C) break;
    const float2 v = cmk((float)g[k].x * scale, (float)g[k].y * scale);
    G32[off + lane + 32 * k] = v;
    const float q = fmaf(v.x, v.x, v.y * v.y);
    s1 += sqrtf(q);
    s2 += q;
  }
  for (int o = 16; o > 0; o >>= 1) {
    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    s2 += __shfl_xor_sync(0xffffffffu, s2, o);
  }
  if (lane == 0) rows[(size_t)l * C + row] = cmk(s1, s2);
}

// The squaring X X / tr(X)^2 of a Hermitian X, C x C, FP32 (0 for X = 0: an empty slice).  A CTA computes a (16 R)^2 tile, a
// thread R x R entries 16 apart, K in chunks fetched to registers one chunk ahead.  The left operand
// is staged as (re, re, im, im), so that a complex multiply-add is two packed FMAs on loaded
// registers: re x (b) and im x (b), summed apart and combined at the end.  R = 3 (48 x 48 tiles) when
// the tiles fill the chip, R = 1 for a few matrices, where a CTA's serial K loop sets the time.
template <int R>
__global__ void __launch_bounds__(256, R == 1 ? 5 : 3) k_is_square(const float2* __restrict__ X, float2* __restrict__ out, int C) {
  constexpr int T = 16 * R;
  constexpr int KT = R == 1 ? 48 : 16;
  constexpr int NE = (T * KT + 255) / 256;
  __shared__ __align__(16) float4 As[2][KT][T + 1];
  __shared__ __align__(16) float2 Bs[2][KT][T];
  __shared__ float red[8];
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int m0 = blockIdx.y * T, n0 = blockIdx.x * T;
  const size_t off = (size_t)blockIdx.z * C * C;
  const float2* Xl = X + off;
  float2 a[NE], b[NE];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int i = 0; i < NE; ++i) {
      const int e = tid + 256 * i, j = e % T, k = k0 + e / T;
      a[i] = b[i] = cmk(0.f, 0.f);
      if (e < T * KT && k < C) {
        if (m0 + j < C) a[i] = conjf2(Xl[(size_t)k * C + m0 + j]);  // X[m][k]
        if (n0 + j < C) b[i] = Xl[(size_t)k * C + n0 + j];
      }
    }
  };
  auto stage = [&](int s) {
#pragma unroll
    for (int i = 0; i < NE; ++i) {
      const int e = tid + 256 * i;
      if (e < T * KT) {
        As[s][e / T][e % T] = make_float4(a[i].x, a[i].x, a[i].y, a[i].y);
        Bs[s][e / T][e % T] = b[i];
      }
    }
  };
  fetch(0);
  float t = 0.f;  // tr(X), the same in every CTA of the matrix
  for (int j = tid; j < C; j += 256) t += Xl[(size_t)j * C + j].x;
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if ((tid & 31) == 0) red[tid >> 5] = t;
  float2 ar[R][R], ai[R][R];
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int j = 0; j < R; ++j) ar[i][j] = ai[i][j] = cmk(0.f, 0.f);
  stage(0);
  __syncthreads();
  t = 0.f;
#pragma unroll
  for (int k = 0; k < 8; ++k) t += red[k];
  const float sc = t > 0.f ? 1.f / t : 0.f;  // (a NaN in X stays one)
  int s = 0;
  for (int k0 = 0; k0 < C; k0 += KT, s ^= 1) {
    const bool more = k0 + KT < C;
    if (more) fetch(k0 + KT);
#pragma unroll 8
    for (int k = 0; k < KT; ++k) {
      float4 av[R];
      float2 bv[R];
#pragma unroll
      for (int i = 0; i < R; ++i) av[i] = As[s][k][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < R; ++j) bv[j] = Bs[s][k][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) {
          ffma2(ar[i][j], cmk(av[i].x, av[i].y), bv[j]);
          ffma2(ai[i][j], cmk(av[i].z, av[i].w), bv[j]);
        }
    }
    if (more) stage(s ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int m = m0 + ty + 16 * i, n = n0 + tx + 16 * j;
      if (m < C && n < C)
        out[off + (size_t)m * C + n] =
            cmk((ar[i][j].x - ai[i][j].y) * sc * sc, (ar[i][j].y + ai[i][j].x) * sc * sc);
    }
}

// largest eigenvalue of each (scaled) G: tr(G S) / tr(S), S = the normalised 2^IS_SQ-th power; 0 for G = 0
__global__ void __launch_bounds__(1024) k_is_lmax(const float2* __restrict__ G32, const float2* __restrict__ S,
                                                  float* __restrict__ lmax, int C) {
  __shared__ double num[32], den[32];
  const int l = blockIdx.x, tid = threadIdx.x;
  const size_t off = (size_t)l * C * C;
  float n = 0.f, d = 0.f;
  for (int e = tid; e < C * C; e += 1024) {
    const float2 g = G32[off + e], s = S[off + e];
    n = fmaf(g.x, s.x, fmaf(g.y, s.y, n));
  }
  for (int j = tid; j < C; j += 1024) d += S[off + (size_t)j * C + j].x;
  double dn = n, dd = d;
  for (int o = 16; o > 0; o >>= 1) {
    dn += __shfl_xor_sync(0xffffffffu, dn, o);
    dd += __shfl_xor_sync(0xffffffffu, dd, o);
  }
  if ((tid & 31) == 0) {
    num[tid >> 5] = dn;
    den[tid >> 5] = dd;
  }
  __syncthreads();
  if (tid == 0) {
    dn = dd = 0.0;
    for (int k = 0; k < 32; ++k) {
      dn += num[k];
      dd += den[k];
    }
    lmax[l] = dd == 0.0 ? 0.f : (float)(dn / dd);
  }
}

// One CTA per direction: the eps schedule (as k_eps), every slice's scale c and the quadrature for
// its c/eps (row q of the table serves [2^-q, 1]).
__global__ void __launch_bounds__(256) k_is_sched(const float2* __restrict__ rows, const float* __restrict__ lmax,
                                                  SolverState* st, DevReport* rep, IsParam* __restrict__ prm,
                                                  int* __restrict__ flag, const IsRow* __restrict__ tab, int L, int C,
                                                  int outer, double eps0_rel, double eta, double eps_min_rel) {
  __shared__ double eps_s;
  const int d = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    SolverState* sd = st + d;
    if (outer == 0) {
      double m = 0.0;
      for (int l = 0; l < L; ++l) {
        const double v = (double)lmax[d * L + l] * (double)__frcp_rn(prm[d * L + l].scale);  // (exact: a power of two)
        m = v > m || v != v ? v : m;  // a NaN stays one
      }
      sd->eps0 = eps0_rel * m;
      sd->eps = sd->eps0;
      sd->eps_min = eps_min_rel * sd->eps0;
    } else {
      sd->eps = fmax(sd->eps / eta, sd->eps_min);
    }
    eps_s = sd->eps;
  }
  __syncthreads();
  for (int l = warp; l < L; l += 8) {  // a warp per slice
    const size_t off = (size_t)(d * L + l) * C;
    float m = 0.f, q = 0.f;
    for (int j = lane; j < C; j += 32) {
      const float2 v = rows[off + j];
      m = fmaxf(m, v.x);
      q += v.y;
    }
    for (int o = 16; o > 0; o >>= 1) {
      m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      q += __shfl_xor_sync(0xffffffffu, q, o);
    }
    if (lane == 0) {
      // c bounds the largest eigenvalue of the scaled G: row sums or the Frobenius norm (a little above,
      // for rounding); with eps > 0 an empty slice has c = eps and weight I/sqrt(eps).  Whatever c
      // rounds to, the shift and the final scale are of the same one.
      IsParam p = prm[d * L + l];
      const double eps = eps_s * p.scale;
      const float c = (float)(1.0001 * ((double)fminf(m, sqrtf(q)) + eps));
      p.inv_c = 1.f / c;
      p.shift = (float)(eps * p.inv_c);
      p.wscale = sqrtf(p.inv_c * p.scale);  // (the product is exact)
      p.q = 0;
      p.n = 0;
      const float cond = c / (float)eps;
      if (q >= 0.f && c >= 1e-30f && cond <= (float)(1 << IS_MAXQ)) {  // false for NaN too
        int k = 0;
        while ((float)(1 << k) < cond) ++k;
        p.q = k;
        p.n = tab[k].n;
      }
      const int had = outer > 0 ? flag[d * L + l] & IS_EIG : 0;  // the eigenvectors before this are there
      flag[d * L + l] = p.n > 0 ? 0 : (had ? IS_EIG | IS_WARM : IS_EIG);
      prm[d * L + l] = p;
    }
  }
  if (d == 0 && tid == 0 && outer < SMSM_MAX_OUTER) {  // the report follows direction 0
    rep->eps[outer] = eps_s;
    rep->sweeps[outer] = 0;  // raised by the eigensolver where it takes a matrix
  }
}

// One term a (A + b I)^(-1) of one matrix, in 16 x 16 blocks of the lower triangle held in
// registers.  Block step k eliminates row block k of the Hermitian R (R = A + b I at first), B = its
// 16 rows (blocks j <= k from row k, blocks i > k as the conjugate of column k):
//   D = L_kk^(-1) of the pivot block,  Q = D B with the pivot block's columns replaced by D itself,
//   row and column k of R cleared, then R_ij += s_i Q_i^H Q_j,  s_i = -1 for i > k, +1 for i <= k.
// For j > k this is the Cholesky update of the trailing matrix; rows i > k collect the right-hand side
// of the forward substitution in their columns j <= k, so that Q_j, j <= k, is row k of L^(-1); and
// rows i <= k collect the inverse, the sum of Q_i^H Q_j over those rows.  All blocks are updated in
// every step, nb (nb+1)/2 block products in each of nb steps: C^3/2 complex multiply-adds.
// FMA-bound in the update (32 FMAs per 3 shared loads of 16 bytes); what is serial is the pivot block
// (one warp, 16 dependent columns), about a fifth of a step at C = 144.
// Warp w of CTA r holds blocks (r NW + w) + s CL NW.  With CL = 4 the row block is written into the
// shared memory of all four CTAs (two buffers: the step after may already be written while a
// neighbour reads this one), one cluster barrier per step.
#define RAT_NW 16
__host__ __device__ inline size_t rat_smem(int nb, int cl) {
  return (size_t)((cl > 1 ? 2 : 1) + 1) * RB * (RB * nb + 2) * sizeof(float2) + RB * (RB + 1) * sizeof(float2);
}

__device__ __forceinline__ void rat_block(int b, int& i, int& j) {  // b = i (i + 1)/2 + j
  i = (int)((sqrtf(8.f * b + 1.f) - 1.f) * 0.5f);
  while (i * (i + 1) / 2 > b) --i;
  while ((i + 1) * (i + 2) / 2 <= b) ++i;
  j = b - i * (i + 1) / 2;
}

// The warm start of a matrix left to the eigensolver, by the CTAs its terms and their sum would have had (own
// launches would cost every solve their latency): T = G V here, from the eigenvectors of the outer
// iteration before, V^H T (two-CTA solver) or T itself (cluster solver) in k_is_sum.
__device__ __noinline__ void is_gv(const float2* __restrict__ G32, const float2* __restrict__ V, float2* __restrict__ T,
                                   float inv_scale, int C, int share, int shares) {
  for (int e = share * blockDim.x + threadIdx.x; e < C * C; e += shares * blockDim.x) {
    const int a = e / C, b = e - a * C;
    float2 t = cmk(0.f, 0.f);
    for (int k = 0; k < C; ++k) cfma(t, G32[(size_t)a * C + k], V[(size_t)k * C + b]);
    T[e] = cscale(t, inv_scale);
  }
}

template <int SLOTS, int CL>
__global__ void __launch_bounds__(32 * RAT_NW, 1)
    k_is_term(const float2* __restrict__ G32, const IsParam* __restrict__ prm, const IsRow* __restrict__ tab,
              float2* __restrict__ part, int* __restrict__ flag, const float2* __restrict__ V, int C, int nb, int l0,
              int probes) {
  extern __shared__ __align__(16) float2 rsm[];
  const int task = blockIdx.x / CL, l = l0 + task / IS_MAXN, term = task % IS_MAXN;
  const IsParam pm = prm[l];
  const bool probe = probes && pm.n > 0 && term == pm.n;
  if (term >= pm.n && !probe) {  // every CTA of a cluster alike
    if (pm.n == 0 && (flag[l] & IS_WARM))
      is_gv(G32 + (size_t)l * C * C, V + (size_t)l * C * C,
            part + (size_t)(l - l0) * IS_MAXN * (nb * (nb + 1) / 2) * (RB * RB), __frcp_rn(pm.scale), C,
            blockIdx.x % (IS_MAXN * CL), IS_MAXN * CL);
    return;
  }
  const int ld = RB * nb + 2;
  float2* Bf = rsm;                                   // [1 or 2][RB][ld]
  float2* Q = rsm + (CL > 1 ? 2 : 1) * RB * ld;       // [RB][ld]
  float2* D = Q + RB * ld;                            // [RB][RB + 1]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = CL > 1 ? (int)cl_rank() : 0;
  const int r0 = (lane >> 3) * 4, c0 = (lane & 7) * 2;
  const int nblk = nb * (nb + 1) / 2;
  const float shift = probe ? IS_PROBE * pm.shift : pm.shift + tab[pm.q].b[term];
  const float most = probe ? 3e38f : rsqrtf(0.5f * shift);  // of 1/sqrt(pivot)
  const float2* Gl = G32 + (size_t)l * C * C;
  float2 R[SLOTS][4][2];
  int bi[SLOTS], bj[SLOTS];
#pragma unroll
  for (int s = 0; s < SLOTS; ++s) {
    const int b = rank * RAT_NW + warp + s * CL * RAT_NW;
    bi[s] = -1;
    bj[s] = 0;
    if (b < nblk) rat_block(b, bi[s], bj[s]);
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const int row = bi[s] * RB + r0 + u, col = bj[s] * RB + c0 + v;
        float2 g = cmk(0.f, 0.f);
        if (bi[s] >= 0) {
          if (row < C && col < C) {
            g = cscale(Gl[(size_t)row * C + col], pm.inv_c);
            if (row == col) g = cmk(g.x + shift, 0.f);
          } else if (row == col) {
            g.x = 1.f;  // padding: the unit matrix
          }
        }
        R[s][u][v] = g;
      }
  }
  bool bad = false;  // (warp 1) a pivot was not what a positive definite matrix has
  if (CL > 1) cl_sync();  // every CTA runs before any writes into another's shared memory
  for (int k = 0; k < nb; ++k) {
    float2* Bk = Bf + (CL > 1 ? (k & 1) * RB * ld : 0);
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      const int i = bi[s], j = bj[s];
      if (i == k || (j == k && i >= 0)) {  // row k as it is, column k conjugated
        const bool rowk = i == k;
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            float2* dst = rowk ? Bk + (r0 + u) * ld + j * RB + c0 + v : Bk + (c0 + v) * ld + i * RB + r0 + u;
            const float2 val = rowk ? R[s][u][v] : conjf2(R[s][u][v]);
            if (CL > 1) {
#pragma unroll
              for (int t = 0; t < CL; ++t) cl_st_v2(cl_map(dst, (uint32_t)t), val);
            } else {
              *dst = val;
            }
            R[s][u][v] = cmk(0.f, 0.f);
          }
      }
    }
    if (CL > 1)
      cl_sync();
    else
      __syncthreads();
    if (warp == 0) {
      // lanes 0-15: the columns of the pivot block; 16-31: those of the unit matrix.  Elimination
      // without square roots, then D's rows scaled by 1/sqrt(pivot).
      float2 v[RB];
#pragma unroll
      for (int i = 0; i < RB; ++i)
        v[i] = lane < RB ? Bk[i * ld + k * RB + lane] : cmk(i == lane - RB ? 1.f : 0.f, 0.f);
      float sp[RB];
#pragma unroll
      for (int c = 0; c < RB; ++c) {
        const float p = __shfl_sync(0xffffffffu, v[c].x, c);
        const float rp = __frcp_rn(p);
        sp[c] = __frsqrt_rn(p);
#pragma unroll
        for (int i = c + 1; i < RB; ++i) {
          const float2 m = cmk(__shfl_sync(0xffffffffu, v[i].x, c) * rp, __shfl_sync(0xffffffffu, v[i].y, c) * rp);
          v[i].x = fmaf(-m.x, v[c].x, fmaf(m.y, v[c].y, v[i].x));
          v[i].y = fmaf(-m.x, v[c].y, fmaf(-m.y, v[c].x, v[i].y));
        }
      }
      if (lane >= RB) {
#pragma unroll
        for (int i = 0; i < RB; ++i) D[i * (RB + 1) + lane - RB] = cscale(v[i], sp[i]);
      }
    }
    __syncthreads();
    // D's diagonal: 1/sqrt(pivot), a NaN where it is negative (looked at here, off the pivot block's chain)
    if (warp == 1 && lane < RB && k * RB + lane < C) bad |= !(D[lane * (RB + 2)].x <= most);
    for (int e = tid; e < RB * nb * 4; e += 32 * RAT_NW) {
      const int rg = e / (RB * nb), col = e - rg * RB * nb;  // four rows of one column
      float2 q[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) q[u] = cmk(0.f, 0.f);
      if (col / RB == k) {
#pragma unroll
        for (int u = 0; u < 4; ++u) q[u] = D[(rg * 4 + u) * (RB + 1) + col - k * RB];
      } else {
        for (int kk = 0; kk < rg * 4 + 4; ++kk) {
          const float2 b = Bk[kk * ld + col];
#pragma unroll
          for (int u = 0; u < 4; ++u) cfma(q[u], D[(rg * 4 + u) * (RB + 1) + kk], b);
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) Q[(rg * 4 + u) * ld + col] = q[u];
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      if (bi[s] < 0 || (probe && bj[s] <= k)) continue;  // (the probe needs the trailing matrix only)
      const float2* qi = Q + bi[s] * RB + r0;
      const float2* qj = Q + bj[s] * RB + c0;
      float2 t[4][2];
#pragma unroll
      for (int u = 0; u < 4; ++u) t[u][0] = t[u][1] = cmk(0.f, 0.f);
#pragma unroll 4
      for (int kk = 0; kk < RB; ++kk) {
        const float4 a0 = *reinterpret_cast<const float4*>(qi + kk * ld);
        const float4 a1 = *reinterpret_cast<const float4*>(qi + kk * ld + 2);
        const float4 b = *reinterpret_cast<const float4*>(qj + kk * ld);
        const float2 a[4] = {cmk(a0.x, a0.y), cmk(a0.z, a0.w), cmk(a1.x, a1.y), cmk(a1.z, a1.w)};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          cfmacj(t[u][0], a[u], cmk(b.x, b.y));
          cfmacj(t[u][1], a[u], cmk(b.z, b.w));
        }
      }
      const float sg = bi[s] > k ? -1.f : 1.f;
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 2; ++v)
          R[s][u][v] = cmk(fmaf(sg, t[u][v].x, R[s][u][v].x), fmaf(sg, t[u][v].y, R[s][u][v].y));
    }
  }
  if (bad) atomicOr(flag + l, 1);
  if (probe) return;
  const float w = tab[pm.q].a[term];
  float2* out = part + ((size_t)(l - l0) * IS_MAXN + term) * nblk * (RB * RB);
#pragma unroll
  for (int s = 0; s < SLOTS; ++s) {
    if (bi[s] < 0) continue;
    const int b = rank * RAT_NW + warp + s * CL * RAT_NW;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      *reinterpret_cast<float4*>(out + (size_t)b * RB * RB + (r0 + u) * RB + c0) =
          make_float4(w * R[s][u][0].x, w * R[s][u][0].y, w * R[s][u][1].x, w * R[s][u][1].y);
  }
}

// W = c^(-1/2) times the sum of the terms (fixed order); the upper triangle mirrors the lower
// (for a matrix left to the eigensolver: its warm start's matrix into Gw, see is_gv)
__global__ void __launch_bounds__(RB* RB) k_is_sum(const float2* __restrict__ part, float2* __restrict__ W,
                                                   const IsParam* __restrict__ prm, const int* __restrict__ flag,
                                                   const float2* __restrict__ V, float2* __restrict__ Gw, int one_sided,
                                                   int C, int nblk, int l0) {
  __shared__ float2 t[RB][RB + 1];
  const int l = l0 + blockIdx.y, b = blockIdx.x, tid = threadIdx.x, r = tid / RB, c = tid % RB;
  const int n = prm[l].n;
  int i, j;
  rat_block(b, i, j);
  if (n == 0) {
    if (!(flag[l] & IS_WARM)) return;
    const float2* T = part + (size_t)blockIdx.y * IS_MAXN * nblk * (RB * RB);
    const float2* Vl = V + (size_t)l * C * C;
    float2* out = Gw + (size_t)l * C * C;
    const int a = i * RB + r, bb = j * RB + c;  // of the lower triangle's blocks
    if (a >= C || bb >= C) return;
    if (one_sided) {
      out[(size_t)a * C + bb] = T[(size_t)a * C + bb];
      out[(size_t)bb * C + a] = T[(size_t)bb * C + a];
    } else if (bb <= a) {  // the eigensolver takes the mean of an entry and its mirror's conjugate
      float2 s = cmk(0.f, 0.f);
      for (int k = 0; k < C; ++k) cfmacj(s, Vl[(size_t)k * C + a], T[(size_t)k * C + bb]);
      out[(size_t)a * C + bb] = s;
      out[(size_t)bb * C + a] = conjf2(s);
    }
    return;
  }
  float2 s = cmk(0.f, 0.f);
  const float2* p = part + ((size_t)blockIdx.y * IS_MAXN * nblk + b) * (RB * RB) + tid;
  for (int k = 0; k < n; ++k) s = cadd(s, p[(size_t)k * nblk * (RB * RB)]);
  t[r][c] = cscale(s, prm[l].wscale);
  __syncthreads();
  float2* Wl = W + (size_t)l * C * C;
  const int row = i * RB + r, col = j * RB + c;
  if (row < C && col < C) {
    float2 v = t[r][c];
    if (i == j) v = r > c ? v : (r == c ? cmk(v.x, 0.f) : conjf2(t[c][r]));
    Wl[(size_t)row * C + col] = v;
  }
  const int mrow = j * RB + r, mcol = i * RB + c;
  if (i != j && mrow < C && mcol < C) Wl[(size_t)mrow * C + mcol] = conjf2(t[c][r]);
}

// Quadrature nodes and weights for [2^-q, 1], q = 0 .. IS_MAXQ: b_j = m tan^2, a_j = (2 K' sqrt(m) /
// (pi n)) dn/cn^2 with m = 2^-q and sn, cn, dn of (j - 1/2) K'/n at parameter 1 - m; the least n whose
// error is within IS_TOL.  Elliptic functions by the arithmetic-geometric mean (descending Landen).
static void elliptic(double u, double m1, double* sn, double* cn, double* dn) {  // parameter 1 - m1
  double a[32], c[32];
  a[0] = 1.0;
  c[0] = sqrt(1.0 - m1);
  double b = sqrt(m1);
  int n = 0;
  while (fabs(c[n]) > 1e-17 * a[n] && n < 30) {
    a[n + 1] = 0.5 * (a[n] + b);
    c[n + 1] = 0.5 * (a[n] - b);
    b = sqrt(a[n] * b);
    ++n;
  }
  double phi = ldexp(a[n] * u, n);
  for (; n > 0; --n) phi = 0.5 * (phi + asin(c[n] / a[n] * sin(phi)));
  *sn = sin(phi);
  *cn = cos(phi);
  *dn = sqrt(*cn * *cn + m1 * *sn * *sn);
}

static std::vector<IsRow> make_table() {
  std::vector<IsRow> tab(IS_MAXQ + 1);
  for (int q = 0; q <= IS_MAXQ; ++q) {
    const double m = ldexp(1.0, -q);
    double x = 1.0, y = sqrt(m);
    for (int k = 0; k < 40; ++k) {
      const double t = 0.5 * (x + y);
      y = sqrt(x * y);
      x = t;
    }
    const double K = M_PI / (2.0 * x);
    for (int n = 2; n < IS_MAXN; ++n) {  // (one slot is the probe's)
      double a[IS_MAXN], b[IS_MAXN], worst = 0.0;
      for (int j = 0; j < n; ++j) {
        double sn, cn, dn;
        elliptic((j + 0.5) * K / n, m, &sn, &cn, &dn);
        b[j] = m * (sn / cn) * (sn / cn);
        a[j] = 2.0 * K * sqrt(m) / (M_PI * n) * dn / (cn * cn);
      }
      for (int k = 0; k <= 400; ++k) {
        const double v = pow(m, k / 400.0);
        double f = 0.0;
        for (int j = 0; j < n; ++j) f += a[j] / (v + b[j]);
        worst = fmax(worst, fabs(f * sqrt(v) - 1.0));
      }
      tab[q].n = n;
      for (int j = 0; j < n; ++j) {
        tab[q].a[j] = (float)a[j];
        tab[q].b[j] = (float)b[j];
      }
      if (worst <= IS_TOL) break;
    }
  }
  return tab;
}

// the same for every plan: made once per process
const std::vector<IsRow>& invsqrt_table() {
  static const std::vector<IsRow> tab = make_table();
  return tab;
}

// This route serves IRLS weights at the solver's own eigen-step settings; a caller who sets a
// rotation threshold, a sweep cap or a cold start, or asks for the cluster eigensolver or the generic
// kernels, gets the eigensolver.  eps may fall to eps0_rel eps_min_rel (1e-4 by default) of the first
// largest eigenvalue and the scale c reaches some ten times that eigenvalue (19 on the 128 x 128
// workload), so below 1e-5 most matrices would pass 2^IS_MAXQ.
bool invsqrt_applies(const smsm_plan_s* P, const smsm_params* prm) {
  return prm->mode == SMSM_MODE_IRLS && !(P->flags & (SMSM_FLAG_CLUSTER_EIG | SMSM_FLAG_GENERIC_KERNELS)) &&
         !prm->eig_cold && prm->eig_tol == 0.f && (prm->max_sweeps <= 0 || prm->max_sweeps >= SMSM_MAX_SWEEPS) &&
         prm->eps0_rel * prm->eps_min_rel >= 1e-5;
}

static int rat_nb(int C) { return (C + RB - 1) / RB; }

size_t invsqrt_per(const smsm_plan_s* P) {  // complex values of one matrix's terms
  const size_t nb = rat_nb(P->C);
  return (size_t)IS_MAXN * (nb * (nb + 1) / 2) * RB * RB;
}

typedef void (*TermFn)(const float2*, const IsParam*, const IsRow*, float2*, int*, const float2*, int, int, int, int);

// Slots = blocks per warp.  One CTA's 16 warps hold up to 5 blocks each (C <= 192), 16 of a lane's 128 registers
// each (four or five blocks spill 100 and 600 bytes); above, four CTAs hold the 105 (C = 208+) to 210 (C = 320)
// blocks with 2 to 4 each.
// Two matrices or fewer leave most SMs idle: four CTAs per term then, too (the same blocks, the same sums), where a
// warp has several blocks to give away (two matrices: C = 144 89 -> 62 us; C = 100 53 -> 62, left alone).
static TermFn term_fn(int C, int LD, int* cl) {
  const int nb = rat_nb(C), nblk = nb * (nb + 1) / 2;
  *cl = nb > 12 || (LD <= 2 && nb > 8) ? 4 : 1;
  if (*cl == 1) {
    switch ((nblk + RAT_NW - 1) / RAT_NW) {
      case 1: return k_is_term<1, 1>;
      case 2: return k_is_term<2, 1>;
      case 3: return k_is_term<3, 1>;
      case 4: return k_is_term<4, 1>;
      default: return k_is_term<5, 1>;
    }
  }
  switch ((nblk + 4 * RAT_NW - 1) / (4 * RAT_NW)) {
    case 1: return k_is_term<1, 4>;
    case 2: return k_is_term<2, 4>;
    case 3: return k_is_term<3, 4>;
    default: return k_is_term<4, 4>;
  }
}

smsm_status invsqrt_init_attrs(const smsm_plan_s* P) {
  cudaError_t e = cudaSuccess;
  for (int LD : {1, P->LD}) {  // a lane's sub-batch may be smaller than the plan
    int cl;
    TermFn fn = term_fn(P->C, LD, &cl);
    // per kernel, not per plan: the most any C of the instance uses
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)rat_smem(cl > 1 ? rat_nb(SMSM_MAX_C) : 12, cl));
  }
  if (e != cudaSuccess) {
    smsm_set_error("inverse square root: %s", cudaGetErrorString(e));
    return SMSM_ERR_CUDA;
  }
  return SMSM_OK;
}

// V: where the eigenvectors of matrices left to the eigensolver in the outer iteration before are
smsm_status launch_invsqrt(const smsm_plan_s* P, const double2* G, const float2* V, int outer, const smsm_params* prm,
                           cudaStream_t s, Timer* T) {
  const int C = P->C, LD = P->LD, nb = rat_nb(C), nblk = nb * (nb + 1) / 2;
  if (T) T->begin(SMSM_STAGE_EIG);
  float2 *A = P->Gw, *Za = P->V, *Zb = P->Gw2;
  k_is_cvt<<<dim3((C + 7) / 8, LD), 256, 0, s>>>(G, A, P->is_rows, P->is_prm, C);
  SMSM_LAUNCH_CHECK("k_is_cvt");
  if (outer == 0) {
    const float2* X = A;
    const int n3 = (C + 47) / 48, n1 = (C + 15) / 16;
    for (int k = 0; k < IS_SQ; ++k) {
      float2* Y = (k & 1) ? Zb : Za;
      if (n3 * n3 * LD >= 152)
        k_is_square<3><<<dim3(n3, n3, LD), 256, 0, s>>>(X, Y, C);
      else
        k_is_square<1><<<dim3(n1, n1, LD), 256, 0, s>>>(X, Y, C);
      SMSM_LAUNCH_CHECK("k_is_square");
      X = Y;
    }
    k_is_lmax<<<LD, 1024, 0, s>>>(A, X, P->is_lmax, C);
    SMSM_LAUNCH_CHECK("k_is_lmax");
  }
  k_is_sched<<<P->D, 256, 0, s>>>(P->is_rows, P->is_lmax, P->st, P->rep, P->is_prm, P->is_flag, P->is_tab, P->L, C,
                                  outer, prm->eps0_rel, prm->eta, prm->eps_min_rel);
  SMSM_LAUNCH_CHECK("k_is_sched");
  int cl;
  TermFn fn = term_fn(C, LD, &cl);
  const int chunk = scratch_cap(P);
  for (int l0 = 0; l0 < LD; l0 += chunk) {
    const int n = LD - l0 < chunk ? LD - l0 : chunk;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(n * IS_MAXN * cl));
    cfg.blockDim = dim3(32 * RAT_NW);
    cfg.dynamicSmemBytes = rat_smem(nb, cl);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cl;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    SMSM_CUDA_TRY(cudaLaunchKernelEx(&cfg, fn, (const float2*)A, (const IsParam*)P->is_prm, (const IsRow*)P->is_tab,
                                     P->scratch, P->is_flag, V, C, nb, l0,
                                     (int)(P->precision == SMSM_PRECISION_BF16_SPLIT)));
    k_is_sum<<<dim3(nblk, n), RB * RB, 0, s>>>(P->scratch, P->Wf, P->is_prm, P->is_flag, V, P->Gw, P->eig_cluster, C,
                                                nblk, l0);
    SMSM_LAUNCH_CHECK("k_is_sum");
  }
  if (T) T->end(SMSM_STAGE_EIG);
  return SMSM_OK;
}
