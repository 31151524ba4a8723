// Row FFTs (x transforms with the transpose fused in) of the lengths N = R1 R2 that two register DFTs cover.
//
// The transforms of operators.cu's k_rowfft_*, here with one exchange through shared memory instead of one per
// radix pass plus staging: a thread loads the R1 points j + R2 r of a row straight from global memory, transforms
// and twiddles them; after one barrier another thread takes the R2 values of one k1 and its R2 results k1 + R1 k2
// go straight to global memory:
//   X[k1 + R1 k2] = sum_j w_R2^(j k2) w_N^(j k1) sum_r w_R1^(r k1) x[j + R2 r].
// The side that is transposed is the one whose threads run along the CTA's 16 rows (128-byte segments), the other
// one's run along j or k1.  HBM-bound in the limit.
// Measured (k_rowfft_* before): 48 images of 256 x 256 25 -> 12 us (50 MB), 3328 x 32 data lines of 128 72 -> 36 us,
// 24 images of 256 x 256 15 -> 8 us, 8 images of 128 x 128 5.7 -> 4.3 us.
#include "common.cuh"
#include "fft.cuh"

enum { RF_OUT = 0, RF_IN = 1, RF_CGP = 2 };

// RF_OUT: in[b][rows][N] -> out[b][N][rows];  RF_IN: in[b][N][rows] -> out[b][rows][N], band > 0 as in
// launch_rowfft_in_T;  RF_CGP: RF_OUT of p after p = r + beta p (in place), beta from the partial sums as in
// k_rowfft_out_T_cgp.
template <int R1, int R2, int TY, bool INV, int MODE>
__global__ void __launch_bounds__(256) k_rowfft2(const float2* __restrict__ in, float2* __restrict__ out, int rows,
                                                 const float2* __restrict__ tw, float sN, int band,
                                                 float2* __restrict__ p, const double* __restrict__ rr_new,
                                                 const double* __restrict__ rr_old, int nrr, int B) {
  constexpr int N = R1 * R2, Q = R2 | 1, LD = (R1 * Q) | 1;
  __shared__ float2 z[TY * LD];
  __shared__ float beta_s;
  const int tid = threadIdx.x, b = blockIdx.y, r0 = blockIdx.x * TY;
  float beta = 0.f;
  if (MODE == RF_CGP) {
    if (tid < 32) {  // one warp: lane-strided sums, then a fixed butterfly
      const size_t poff = (size_t)(b / B) * SMSM_PART_MAX;
      double sn = 0.0, so = 0.0;
      for (int k = tid; k < nrr; k += 32) {
        sn += rr_new[poff + k];
        so += rr_old[poff + k];
      }
      for (int o = 16; o > 0; o >>= 1) {
        sn += __shfl_xor_sync(0xffffffffu, sn, o);
        so += __shfl_xor_sync(0xffffffffu, so, o);
      }
      const double q = so > 0.0 ? sn / so : 0.0;
      if (tid == 0) beta_s = isfinite(q) ? (float)q : 0.f;
    }
    __syncthreads();
    beta = beta_s;
  }
  constexpr int T1 = TY * R2;
#pragma unroll
  for (int t0 = 0; t0 < T1; t0 += 256) {
    const int t = t0 + tid;
    const int row = MODE == RF_IN ? t % TY : t / R2, j = MODE == RF_IN ? t / TY : t % R2;
    if ((T1 % 256 == 0 || t < T1) && r0 + row < rows) {
      float2 v[R1];
      if (MODE == RF_IN) {
        const float2* src = in + (size_t)b * N * rows + r0 + row;
#pragma unroll
        for (int r = 0; r < R1; ++r) v[r] = __ldg(src + (size_t)(j + R2 * r) * rows);
      } else {
        const size_t o = ((size_t)b * rows + r0 + row) * N + j;
#pragma unroll
        for (int r = 0; r < R1; ++r) v[r] = __ldg(in + o + R2 * r);
        if (MODE == RF_CGP) {
          float2 pv[R1];
#pragma unroll
          for (int r = 0; r < R1; ++r) pv[r] = p[o + R2 * r];
#pragma unroll
          for (int r = 0; r < R1; ++r) {
            v[r] = cmk(fmaf(beta, pv[r].x, v[r].x), fmaf(beta, pv[r].y, v[r].y));
            p[o + R2 * r] = v[r];
          }
        }
      }
      // centring: (-1)^(j + R2 r)
#pragma unroll
      for (int r = 1; r < R1; ++r)
        if ((R2 * r) & 1) v[r] = cmk(-v[r].x, -v[r].y);
      rf_dft<R1, INV>(v);
      const float sj = sgn_par(j);
      z[row * LD + j] = cscale(v[0], sj);
#pragma unroll
      for (int k = 1; k < R1; ++k) {
        const float2 w = __ldg(tw + j * k);
        z[row * LD + k * Q + j] = cmul(v[k], cmk(sj * w.x, INV ? -sj * w.y : sj * w.y));
      }
    }
  }
  __syncthreads();
  constexpr int T2 = TY * R1;
#pragma unroll
  for (int t0 = 0; t0 < T2; t0 += 256) {
    const int t = t0 + tid;
    const int row = MODE == RF_IN ? t / R1 : t % TY, k1 = MODE == RF_IN ? t % R1 : t / TY;
    if ((T2 % 256 == 0 || t < T2) && r0 + row < rows) {
      float2 v[R2];
#pragma unroll
      for (int j = 0; j < R2; ++j) v[j] = z[row * LD + k1 * Q + j];
      rf_dft<R2, INV>(v);
      const float sc = sN * sgn_par(k1);
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) {
        const int k = k1 + R1 * k2;
        float2 u = cscale(v[k2], ((R1 * k2) & 1) ? -sc : sc);
        if (MODE == RF_IN) {
          float2* o = out + ((size_t)b * rows + r0 + row) * N + k;
          if (band && (r0 + row < band || r0 + row >= rows - band || k < band || k >= N - band)) u = cadd(u, *o);
          *o = u;
        } else {
          out[((size_t)b * N + k) * rows + r0 + row] = u;
        }
      }
    }
  }
}

typedef void (*RfFn)(const float2*, float2*, int, const float2*, float, int, float2*, const double*, const double*, int,
                     int);
template <int R1, int R2, int TY>
static RfFn rf_fn(int mode, int inverse) {
  if (mode == RF_CGP) return k_rowfft2<R1, R2, TY, true, RF_CGP>;
  if (mode == RF_OUT) return inverse ? k_rowfft2<R1, R2, TY, true, RF_OUT> : k_rowfft2<R1, R2, TY, false, RF_OUT>;
  return inverse ? k_rowfft2<R1, R2, TY, true, RF_IN> : k_rowfft2<R1, R2, TY, false, RF_IN>;
}

// SMSM_ERR_ARG: a length without such a kernel, or the generic kernels are asked for
smsm_status launch_rowfft2(const smsm_plan_s* P, int mode, const float2* in, float2* out, int nb, int rows, int inverse,
                           int band, float2* p, const double* rr_new, const double* rr_old, int nrr, cudaStream_t s) {
  if (P->flags & SMSM_FLAG_GENERIC_KERNELS) return SMSM_ERR_ARG;
  const bool few = rows <= 8;  // (data lines of a short shot: half the CTA's rows would be missing)
  RfFn fn;
#define RF_N(R1, R2)                                                            \
  case R1 * R2:                                                                 \
    fn = few ? rf_fn<R1, R2, 8>(mode, inverse) : rf_fn<R1, R2, 16>(mode, inverse); \
    break;
  switch (P->N) {
    RF_N(8, 6)
    RF_N(8, 8)
    RF_N(8, 9)
    RF_N(12, 8)
    RF_N(12, 9)
    RF_N(16, 8)
    RF_N(12, 12)
    RF_N(16, 12)
    RF_N(16, 16)
    default: return SMSM_ERR_ARG;
  }
#undef RF_N
  const int ty = few ? 8 : 16;
  fn<<<dim3((rows + ty - 1) / ty, nb), 256, 0, s>>>(in, out, rows, P->twN, P->sN, band, p, rr_new, rr_old, nrr,
                                                    P->L * P->Ns);
  SMSM_LAUNCH_CHECK("k_rowfft2");
  return SMSM_OK;
}
