// Shared-memory batched FFT (mixed radix 2/3/4, Stockham autosort).
//
// Each pass with radix R over a length-n transform reads element j + r*n/R,
// applies the twiddle w^(r*k*n/(s*R)) (k = j mod s, s = product of the
// earlier radices, w = exp(-2 pi i/n)), does an R-point DFT, and writes
// element (j/s)*s*R + k + r*s of the other buffer.  After all passes the
// result is in natural order; no bit reversal is needed.  The twiddle table
// holds exp(-2 pi i k/n), k < n, computed on the host in FP64.
#pragma once
#include "common.cuh"

// (-1)^n as a float
__device__ __forceinline__ float sgn_par(int n) { return (n & 1) ? -1.f : 1.f; }

template <bool INV>
__device__ __forceinline__ float2 tw_get(const float2* tw, int idx) {
  float2 w = tw[idx];
  return INV ? conjf2(w) : w;
}

template <bool INV>
__device__ __forceinline__ void dft2(float2* v) {
  float2 a = v[0], b = v[1];
  v[0] = cadd(a, b);
  v[1] = csub(a, b);
}

template <bool INV>
__device__ __forceinline__ void dft4(float2* v) {
  // forward: X1 = a0 - i a1 - a2 + i a3 ; inverse swaps the sign of i
  float2 s02 = cadd(v[0], v[2]), d02 = csub(v[0], v[2]);
  float2 s13 = cadd(v[1], v[3]), d13 = csub(v[1], v[3]);
  // -i * d13 = (d13.y, -d13.x)
  float2 rot = INV ? cmk(-d13.y, d13.x) : cmk(d13.y, -d13.x);
  v[0] = cadd(s02, s13);
  v[2] = csub(s02, s13);
  v[1] = cadd(d02, rot);
  v[3] = csub(d02, rot);
}

// 8-point DFT in registers, natural order in and out: two 4-point DFTs of the even and odd
// elements, the odd ones turned by w8^k (w8 = exp(-+ 2 pi i / 8)), then one radix-2 step
template <bool INV>
__device__ __forceinline__ void dft8(float2* v) {
  const float h = 0.707106781186547524f;  // sqrt(1/2)
  float2 e[4] = {v[0], v[2], v[4], v[6]};
  float2 o[4] = {v[1], v[3], v[5], v[7]};
  dft4<INV>(e);
  dft4<INV>(o);
  // forward: w8 = h (1 - i), w8^2 = -i, w8^3 = h (-1 - i); inverse: their conjugates
  const float2 o1 = INV ? cmk(h * (o[1].x - o[1].y), h * (o[1].x + o[1].y))
                        : cmk(h * (o[1].x + o[1].y), h * (o[1].y - o[1].x));
  const float2 o2 = INV ? cmk(-o[2].y, o[2].x) : cmk(o[2].y, -o[2].x);
  const float2 o3 = INV ? cmk(-h * (o[3].x + o[3].y), h * (o[3].x - o[3].y))
                        : cmk(h * (o[3].y - o[3].x), -h * (o[3].x + o[3].y));
  v[0] = cadd(e[0], o[0]);
  v[4] = csub(e[0], o[0]);
  v[1] = cadd(e[1], o1);
  v[5] = csub(e[1], o1);
  v[2] = cadd(e[2], o2);
  v[6] = csub(e[2], o2);
  v[3] = cadd(e[3], o3);
  v[7] = csub(e[3], o3);
}

template <bool INV>
__device__ __forceinline__ void dft3(float2* v) {
  // X1 = a0 - t1/2 -+ i (sqrt3/2) t2, X2 = a0 - t1/2 +- i (sqrt3/2) t2, t1 = a1+a2, t2 = a1-a2
  const float h3 = 0.866025403784438647f;
  float2 t1 = cadd(v[1], v[2]), t2 = csub(v[1], v[2]);
  float2 m = cmk(v[0].x - 0.5f * t1.x, v[0].y - 0.5f * t1.y);
  // -i * h3 * t2 = (h3 t2.y, -h3 t2.x)
  float2 j = INV ? cmk(-h3 * t2.y, h3 * t2.x) : cmk(h3 * t2.y, -h3 * t2.x);
  v[0] = cadd(v[0], t1);
  v[1] = cadd(m, j);
  v[2] = csub(m, j);
}

// exp(-2 pi i m / R) for the products m met in a two-step DFT of length R
template <int R>
__device__ __forceinline__ constexpr float rf_cos(int m) {
  constexpr float c16[10] = {1.f, 0.92387953251128674f, 0.70710678118654752f, 0.38268343236508977f, 0.f,
                             -0.38268343236508977f, -0.70710678118654752f, -0.92387953251128674f, -1.f,
                             -0.92387953251128674f};
  constexpr float c12[7] = {1.f, 0.86602540378443865f, 0.5f, 0.f, -0.5f, -0.86602540378443865f, -1.f};
  constexpr float c9[5] = {1.f, 0.76604444311897804f, 0.17364817766693035f, -0.5f, -0.93969262078590838f};
  constexpr float c6[3] = {1.f, 0.5f, -0.5f};
  return R == 16 ? c16[m] : (R == 12 ? c12[m] : (R == 9 ? c9[m] : c6[m]));
}
template <int R>
__device__ __forceinline__ constexpr float rf_sin(int m) {
  constexpr float s16[10] = {0.f, 0.38268343236508977f, 0.70710678118654752f, 0.92387953251128674f, 1.f,
                             0.92387953251128674f, 0.70710678118654752f, 0.38268343236508977f, 0.f,
                             -0.38268343236508977f};
  constexpr float s12[7] = {0.f, 0.5f, 0.86602540378443865f, 1.f, 0.86602540378443865f, 0.5f, 0.f};
  constexpr float s9[5] = {0.f, 0.64278760968653933f, 0.98480775301220806f, 0.86602540378443865f,
                           0.34202014332566873f};
  constexpr float s6[3] = {0.f, 0.86602540378443865f, 0.86602540378443865f};
  return R == 16 ? s16[m] : (R == 12 ? s12[m] : (R == 9 ? s9[m] : s6[m]));
}

template <int R, bool INV>
__device__ __forceinline__ void rf_dft(float2* v) {
  if constexpr (R == 2) {
    dft2<INV>(v);
  } else if constexpr (R == 3) {
    dft3<INV>(v);
  } else if constexpr (R == 4) {
    dft4<INV>(v);
  } else if constexpr (R == 8) {
    dft8<INV>(v);
  } else {  // A B points: n = B n1 + n2, X[k1 + A k2]
    constexpr int A = R == 16 ? 4 : (R == 12 ? 4 : 3), B = R / A;
    float2 t[A][B];
#pragma unroll
    for (int n2 = 0; n2 < B; ++n2) {
      float2 u[A];
#pragma unroll
      for (int n1 = 0; n1 < A; ++n1) u[n1] = v[B * n1 + n2];
      rf_dft<A, INV>(u);
#pragma unroll
      for (int k1 = 0; k1 < A; ++k1) {
        const int m = n2 * k1;
        if (m == 0)
          t[k1][n2] = u[k1];
        else
          t[k1][n2] = cmul(u[k1], cmk(rf_cos<R>(m), INV ? rf_sin<R>(m) : -rf_sin<R>(m)));
      }
    }
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) {
      rf_dft<B, INV>(t[k1]);
#pragma unroll
      for (int k2 = 0; k2 < B; ++k2) v[k1 + A * k2] = t[k1][k2];
    }
  }
}

// One radix-R pass (R in {2, 3, 4, 8}) of the Stockham FFT described above, with
// the transform length N, R and the product S of the earlier radices fixed at
// compile time (so every index division is by a constant); then the next pass.
// Radices are taken in the order 8, ..., 8, 4, 2, 3, ..., 3: fewer passes through
// shared memory than the runtime descriptor's 4, ..., 4, 2, 3, ..., 3 (used only for
// the lengths without a fixed chain).
template <bool INV, int N, int S>
__device__ __forceinline__ float2* fft_fixed_from(float2* src, float2* dst, int nbatch, int bstride,
                                                  const float2* tw) {
  if constexpr (S == N) {
    return src;
  } else {
    constexpr int REM = N / S;
    constexpr int R = (REM % 8 == 0) ? 8 : ((REM % 4 == 0) ? 4 : ((REM % 2 == 0) ? 2 : 3));
    constexpr int nR = N / R;
    constexpr int tstep = N / (S * R);
    const int ntask = nbatch * nR;
    for (int t = threadIdx.x; t < ntask; t += blockDim.x) {
      const int bb = t / nR;
      const int j = t - bb * nR;
      const float2* Sp = src + bb * bstride;
      float2* Dp = dst + bb * bstride;
      const int k = j % S;
      const int base = (j - k) * R + k;
      float2 v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = Sp[j + r * nR];
      if (S > 1 && k) {
#pragma unroll
        for (int r = 1; r < R; ++r) v[r] = cmul(v[r], tw_get<INV>(tw, r * k * tstep));
      }
      if constexpr (R == 8)
        dft8<INV>(v);
      else if constexpr (R == 4)
        dft4<INV>(v);
      else if constexpr (R == 2)
        dft2<INV>(v);
      else
        dft3<INV>(v);
#pragma unroll
      for (int r = 0; r < R; ++r) Dp[base + r * S] = v[r];
    }
    __syncthreads();
    return fft_fixed_from<INV, N, S * R>(dst, src, nbatch, bstride, tw);
  }
}

// Batched FFT of `nbatch` transforms of length d.n; transform b starts at
// a + b*bstride (and b + b*bstride for the ping-pong buffer).  All threads
// of the block take part; the routine ends with __syncthreads() after every
// pass and returns the buffer that holds the result.  Unnormalised.  The
// common lengths run a compile-time pass chain.
template <bool INV>
__device__ float2* fft_smem(float2* a, float2* b, int nbatch, int bstride, const FftDesc& d,
                            const float2* tw) {
  switch (d.n) {
    case 64: return fft_fixed_from<INV, 64, 1>(a, b, nbatch, bstride, tw);
    case 96: return fft_fixed_from<INV, 96, 1>(a, b, nbatch, bstride, tw);
    case 128: return fft_fixed_from<INV, 128, 1>(a, b, nbatch, bstride, tw);
    case 192: return fft_fixed_from<INV, 192, 1>(a, b, nbatch, bstride, tw);
    case 256: return fft_fixed_from<INV, 256, 1>(a, b, nbatch, bstride, tw);
    default: break;
  }
  const int n = d.n;
  int s = 1;
  float2* src = a;
  float2* dst = b;
  for (int ps = 0; ps < d.np; ++ps) {
    const unsigned rc = (d.code >> (2 * ps)) & 3u;
    const int R = rc == 2u ? 4 : (rc == 1u ? 3 : 2);
    const int nR = n / R;
    const int tstep = n / (s * R);
    const int ntask = nbatch * nR;
    for (int t = threadIdx.x; t < ntask; t += blockDim.x) {
      const int bb = t / nR;
      const int j = t - bb * nR;
      const float2* S = src + bb * bstride;
      float2* D = dst + bb * bstride;
      const int k = j % s;
      const int base = (j - k) * R + k;
      float2 v[4];
      if (R == 4) {
#pragma unroll
        for (int r = 0; r < 4; ++r) v[r] = S[j + r * nR];
        if (k) {
#pragma unroll
          for (int r = 1; r < 4; ++r) v[r] = cmul(v[r], tw_get<INV>(tw, r * k * tstep));
        }
        dft4<INV>(v);
#pragma unroll
        for (int r = 0; r < 4; ++r) D[base + r * s] = v[r];
      } else if (R == 2) {
        v[0] = S[j];
        v[1] = S[j + nR];
        if (k) v[1] = cmul(v[1], tw_get<INV>(tw, k * tstep));
        dft2<INV>(v);
        D[base] = v[0];
        D[base + s] = v[1];
      } else {  // R == 3
#pragma unroll
        for (int r = 0; r < 3; ++r) v[r] = S[j + r * nR];
        if (k) {
          v[1] = cmul(v[1], tw_get<INV>(tw, k * tstep));
          v[2] = cmul(v[2], tw_get<INV>(tw, 2 * k * tstep));
        }
        dft3<INV>(v);
#pragma unroll
        for (int r = 0; r < 3; ++r) D[base + r * s] = v[r];
      }
    }
    __syncthreads();
    float2* t = src;
    src = dst;
    dst = t;
    s *= R;
  }
  return src;
}

// fft_smem as an out-of-line call: kernels instantiated many times over other
// template parameters share one copy of every pass chain
template <bool INV>
__device__ __noinline__ float2* fft_smem_call(float2* a, float2* b, int nbatch, int bstride, const FftDesc& d,
                                              const float2* tw) {
  return fft_smem<INV>(a, b, nbatch, bstride, d, tw);
}


// Centred unitary transforms of `nb` lines of N = R1 R2 points by two register DFTs and one exchange (see rowfft.cu):
// src [nb][N] -> z [nb][lines2_ld] -> out(line, k, value), every value once.  Threads of the whole block; src may be
// overwritten by `out` (it is read before the barrier between the steps only).  No barrier at the end.
template <bool INV, int R1, int R2, class Out>
__device__ __forceinline__ void fft_lines2(const float2* src, float2* z, int nb, const float2* tw, float sN, Out out) {
  constexpr int N = R1 * R2, Q = R2 | 1, LD = R1 * Q;
  for (int t = threadIdx.x; t < nb * R2; t += blockDim.x) {
    const int b = t / R2, j = t - b * R2;
    float2 v[R1];
#pragma unroll
    for (int r = 0; r < R1; ++r) {
      v[r] = src[b * N + j + R2 * r];
      if ((R2 * r) & 1) v[r] = cmk(-v[r].x, -v[r].y);
    }
    rf_dft<R1, INV>(v);
    const float sj = sgn_par(j);
    z[b * LD + j] = cscale(v[0], sj);
#pragma unroll
    for (int k = 1; k < R1; ++k) {
      const float2 w = tw_get<INV>(tw, j * k);
      z[b * LD + k * Q + j] = cmul(v[k], cmk(sj * w.x, sj * w.y));
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < nb * R1; t += blockDim.x) {
    const int b = t / R1, k1 = t - b * R1;
    float2 v[R2];
#pragma unroll
    for (int j = 0; j < R2; ++j) v[j] = z[b * LD + k1 * Q + j];
    rf_dft<R2, INV>(v);
    const float sc = sN * sgn_par(k1);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) out(b, k1 + R1 * k2, cscale(v[k2], ((R1 * k2) & 1) ? -sc : sc));
  }
}

// line pitch of z for the lengths that fft_lines2 serves (0: none)
__host__ __device__ inline int lines2_ld(int N) {
  switch (N) {
    case 48: return 8 * 7;
    case 64: return 8 * 9;
    case 72: return 8 * 9;
    case 96: return 12 * 9;
    case 108: return 12 * 9;
    case 128: return 16 * 9;
    case 144: return 12 * 13;
    case 192: return 16 * 13;
    case 256: return 16 * 17;
    default: return 0;
  }
}
#define FFT_LINES2_SWITCH(N, CALL) \
  switch (N) {                     \
    case 48: CALL(8, 6); break;    \
    case 64: CALL(8, 8); break;    \
    case 72: CALL(8, 9); break;    \
    case 96: CALL(12, 8); break;   \
    case 108: CALL(12, 9); break;  \
    case 128: CALL(16, 8); break;  \
    case 144: CALL(12, 12); break; \
    case 192: CALL(16, 12); break; \
    default: CALL(16, 16); break;  \
  }
// in shared memory, [nb][N] -> [nb][N] (in place allowed)
template <bool INV>
__device__ __noinline__ void fft_lines2_smem(const float2* src, float2* z, float2* dst, int nb, int N, const float2* tw,
                                             float sN) {
#define FFT_L2(R1, R2) \
  fft_lines2<INV, R1, R2>(src, z, nb, tw, sN, [&](int b, int k, float2 v) { dst[b * (R1 * R2) + k] = v; })
  FFT_LINES2_SWITCH(N, FFT_L2)
#undef FFT_L2
}
// to global lines dst + b stride
template <bool INV>
__device__ __noinline__ void fft_lines2_global(const float2* src, float2* z, float2* dst, size_t stride, int nb, int N,
                                               const float2* tw, float sN) {
#define FFT_L2(R1, R2) \
  fft_lines2<INV, R1, R2>(src, z, nb, tw, sN, [&](int b, int k, float2 v) { dst[b * stride + k] = v; })
  FFT_LINES2_SWITCH(N, FFT_L2)
#undef FFT_L2
}
