// IRLS + CG solve of the SMS-MUSSELS cost (Eq. 10), entirely on the device.
//
// Outer iteration k: Gram of the current x -> Jacobi eigen-decomposition ->
// W_k -> filters (periodic multipliers + border-class filters) -> J steps of
// textbook CG on (A^H A + lambda P_W) x = A^H y from the current x.  All CG
// scalars are reduced in FP64 from per-CTA partials in a fixed order, so
// every CTA computes the same alpha/beta and runs are bit-reproducible; no
// scalar ever goes back to the host, which lets the whole solve be captured
// as one CUDA graph (replayed by later calls with the same parameters).
#include <math.h>
#include <string.h>

#include <mutex>
#include <vector>

#include "common.cuh"

void solver_free_timing(smsm_plan_s* P) {
  TimingPool* tp = (TimingPool*)P->tpool;
  if (!tp) return;
  for (cudaEvent_t e : tp->ev) cudaEventDestroy(e);
  delete tp;
  P->tpool = nullptr;
}

#define VEC_THREADS 256

// CTAs per direction of the CG vector kernels (chosen once per plan from the whole batch,
// so a sub-batch view splits its reductions the same way)
int vec_blocks(const smsm_plan_s* P) {
  if (P->nvb > 0) return P->nvb;
  const size_t n2 = (size_t)P->L * P->Ns * P->N * P->N / 2;  // float4 = two complex
  size_t b = (n2 + VEC_THREADS - 1) / VEC_THREADS;
  size_t cap = (size_t)(4 * 152 + P->D - 1) / P->D;
  if (cap < 8) cap = 8;
  if (b > cap) b = cap;
  return (int)b;
}

// Scratch of the Gram and the weight step (which follow one another in a lane), per matrix.  Launches take
// at most scratch_cap matrices, 96 MB; the buffer has room for every matrix of the plan or, when
// that is more, one launch's room per lane.
static size_t scratch_per(const smsm_plan_s* P) {
  const size_t a = invsqrt_per(P), b = gram_lag_per(P);
  return a > b ? a : b;
}
int scratch_cap(const smsm_plan_s* P) {
  const size_t n = (size_t)96 * 1024 * 1024 / (scratch_per(P) * sizeof(float2));
  return n < 1 ? 1 : (int)(n < 4096 ? n : 4096);
}
size_t scratch_count(const smsm_plan_s* P) {
  const size_t cap = scratch_cap(P);
  return scratch_per(P) * ((size_t)P->LD <= cap ? (size_t)P->LD : cap * SMSM_MAX_LANES);
}
static size_t scratch_offset(const smsm_plan_s* P, int d0, int lane) {
  const size_t cap = scratch_cap(P);
  return scratch_per(P) * ((size_t)P->LD <= cap ? (size_t)d0 * P->L : cap * lane);
}

// Sum of partial arrays a[0..na) + b[0..nb) in a fixed order; every thread
// returns the same value.  `red` is VEC_THREADS doubles of shared memory.
__device__ double sum_parts(const double* __restrict__ a, int na, const double* __restrict__ b, int nb, double* red) {
  double s = 0.0;
  for (int k = threadIdx.x; k < na; k += blockDim.x) s += a[k];
  for (int k = threadIdx.x; k < nb; k += blockDim.x) s += b[k];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  double r = red[0];
  __syncthreads();
  return r;
}

// The same fixed-order sums by one warp (lane-strided, then a butterfly), both
// results broadcast to the CTA through shared memory: one barrier instead of a tree.
__device__ void warp_sums(const double* __restrict__ a, int na, const double* __restrict__ b, int nb,
                          const double* __restrict__ c, int nc, double* out2) {
  if (threadIdx.x < 32) {
    double s0 = 0.0, s1 = 0.0;
    for (int k = threadIdx.x; k < na; k += 32) s0 += a[k];
    for (int k = threadIdx.x; k < nb; k += 32) s0 += b[k];
    for (int k = threadIdx.x; k < nc; k += 32) s1 += c[k];
    for (int o = 16; o > 0; o >>= 1) {
      s0 += __shfl_xor_sync(0xffffffffu, s0, o);
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    }
    if (threadIdx.x == 0) {
      out2[0] = s0;
      out2[1] = s1;
    }
  }
  __syncthreads();
}

__device__ void block_partial(double v, double* red, double* out) {
  red[threadIdx.x] = v;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[blockIdx.x] = red[0];
}

// squared norm of a float4, accumulated in FP32: a thread sums only a few dozen of
// them before its partial goes on in FP64 (FP64 arithmetic is scarce on this part)
__device__ __forceinline__ float norm2_4(float4 v, float acc) {
  return fmaf(v.w, v.w, fmaf(v.z, v.z, fmaf(v.y, v.y, fmaf(v.x, v.x, acc))));
}

// Vectors are [D][n4] float4 (direction d = blockIdx.y); partial arrays are
// [D][SMSM_PART_MAX]; every direction has its own CG scalars.
#define DIR_OFFSETS(n4)                          \
  const size_t d_ = blockIdx.y;                 \
  const size_t off_ = d_ * (n4);                \
  const size_t poff_ = d_ * SMSM_PART_MAX;

// r = b - q; p = r; partial ||r||^2
__global__ void __launch_bounds__(VEC_THREADS) k_cg_init(const float4* __restrict__ b, const float4* __restrict__ q,
                                                         float4* __restrict__ r, float4* __restrict__ p, size_t n4,
                                                         double* __restrict__ part_rr) {
  __shared__ double red[VEC_THREADS];
  DIR_OFFSETS(n4)
  b += off_;
  q += off_;
  r += off_;
  p += off_;
  float s = 0.f;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n4; e += (size_t)gridDim.x * blockDim.x) {
    float4 bv = b[e], qv = q[e];
    float4 rv = make_float4(bv.x - qv.x, bv.y - qv.y, bv.z - qv.z, bv.w - qv.w);
    r[e] = rv;
    p[e] = rv;
    s = norm2_4(rv, s);
  }
  block_partial((double)s, red, part_rr + poff_);
}

// alpha = <r,r>/<p,q>; x += alpha p; r -= alpha q; partial ||r||^2
__global__ void __launch_bounds__(VEC_THREADS) k_cg_update(float4* __restrict__ x, float4* __restrict__ r,
                                                           const float4* __restrict__ p, const float4* __restrict__ q,
                                                           size_t n4, const double* __restrict__ pq_col, int ncol,
                                                           const double* __restrict__ pq_band, int nband,
                                                           const double* __restrict__ rr_in, int nrr,
                                                           double* __restrict__ rr_out, SolverState* st) {
  __shared__ double red[VEC_THREADS];
  DIR_OFFSETS(n4)
  x += off_;
  r += off_;
  p += off_;
  q += off_;
  warp_sums(pq_col + poff_, ncol, pq_band + poff_, nband, rr_in + poff_, nrr, red);
  const double pq = red[0], rr = red[1];
  __syncthreads();  // red is reused by the partial below
  double alpha = rr / pq;
  if (!(pq > 0.0) || !isfinite(alpha)) {
    if (blockIdx.x == 0 && threadIdx.x == 0 && st[d_].status == 0)
      st[d_].status = isfinite(pq) ? SMSM_ERR_NOT_PD : SMSM_ERR_DIVERGED;
    alpha = 0.0;
  }
  const float a = (float)alpha;
  float s = 0.f;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n4; e += (size_t)gridDim.x * blockDim.x) {
    float4 xv = x[e], rv = r[e];
    const float4 pv = p[e], qv = q[e];
    xv.x = fmaf(a, pv.x, xv.x);
    xv.y = fmaf(a, pv.y, xv.y);
    xv.z = fmaf(a, pv.z, xv.z);
    xv.w = fmaf(a, pv.w, xv.w);
    rv.x = fmaf(-a, qv.x, rv.x);
    rv.y = fmaf(-a, qv.y, rv.y);
    rv.z = fmaf(-a, qv.z, rv.z);
    rv.w = fmaf(-a, qv.w, rv.w);
    x[e] = xv;
    r[e] = rv;
    s = norm2_4(rv, s);
  }
  block_partial((double)s, red, rr_out + poff_);
}

// beta = rr_new/rr_old; p = r + beta p
__global__ void __launch_bounds__(VEC_THREADS) k_cg_pupdate(const float4* __restrict__ r, float4* __restrict__ p,
                                                            size_t n4, const double* __restrict__ rr_new,
                                                            const double* __restrict__ rr_old, int nrr) {
  __shared__ double red[VEC_THREADS];
  DIR_OFFSETS(n4)
  r += off_;
  p += off_;
  const double rn = sum_parts(rr_new + poff_, nrr, nullptr, 0, red);
  const double ro = sum_parts(rr_old + poff_, nrr, nullptr, 0, red);
  double beta = ro > 0.0 ? rn / ro : 0.0;
  if (!isfinite(beta)) beta = 0.0;
  const float bta = (float)beta;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n4; e += (size_t)gridDim.x * blockDim.x) {
    const float4 rv = r[e];
    float4 pv = p[e];
    pv.x = fmaf(bta, pv.x, rv.x);
    pv.y = fmaf(bta, pv.y, rv.y);
    pv.z = fmaf(bta, pv.z, rv.z);
    pv.w = fmaf(bta, pv.w, rv.w);
    p[e] = pv;
  }
}

// partials of Re<a, b> (FP32 per thread, FP64 per CTA), [D][SMSM_PART_MAX]
__global__ void __launch_bounds__(VEC_THREADS) k_vdot_part(const float4* __restrict__ a, const float4* __restrict__ b,
                                                           size_t n4, double* __restrict__ part) {
  __shared__ double red[VEC_THREADS];
  DIR_OFFSETS(n4)
  a += off_;
  b += off_;
  float s = 0.f;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n4; e += (size_t)gridDim.x * blockDim.x) {
    const float4 u = a[e], v = b[e];
    s = fmaf(u.x, v.x, fmaf(u.y, v.y, fmaf(u.z, v.z, fmaf(u.w, v.w, s))));
  }
  block_partial((double)s, red, part + poff_);
}

__global__ void k_fill_one(float2* __restrict__ v, size_t n) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x)
    v[e] = cmk(1.f, 0.f);
}

// which = 0: record ||r||^2 of direction 0 at the start of outer iteration `outer`; 1: at its end
__global__ void k_record(DevReport* rep, int outer, int which, const double* __restrict__ rr, int nrr) {
  __shared__ double red[VEC_THREADS];
  const double a = sum_parts(rr, nrr, nullptr, 0, red);
  if (threadIdx.x == 0 && outer < SMSM_MAX_OUTER) {
    if (which == 0)
      rep->rr_start[outer] = a;
    else
      rep->rr_end[outer] = a;
  }
}

__global__ void k_reset_state(SolverState* st, int D) {
  for (int d = threadIdx.x; d < D; d += blockDim.x) {
    st[d].status = 0;
    st[d].eps = 0.0;
    st[d].eps0 = 0.0;
    st[d].eps_min = 0.0;
  }
}

// q = (A^H A + lambda P_W) v.  With with_dots, the per-CTA partials of
// Re<v, q> go to part_pq_col (column stage, image domain, Parseval) and
// part_pq_band (border correction).
// With pupd (CG steps after the first), v is first updated in place as
// v = r + beta v, beta from the rr partial banks (fused into the x-transform).
struct PUpdate {
  const float2* r;
  const double *rr_new, *rr_old;
  int nrr;
};

static smsm_status normal_pen_timed(smsm_plan_s* P, const float2* v, float2* q, float lambda, int with_dots,
                                    cudaStream_t s, Timer* T, const PUpdate* pupd = nullptr) {
  const int B = P->L * P->Ns;
  smsm_status st;
  if (T) T->begin(SMSM_STAGE_ROWFFT_INV);
  if (pupd) {
    if ((st = launch_rowfft_out_T_cgp(P, const_cast<float2*>(v), pupd->r, P->hA, P->D * B, pupd->rr_new,
                                      pupd->rr_old, pupd->nrr, s)))
      return st;
  } else if ((st = launch_rowfft_out_T(P, v, P->hA, P->D * B, P->N, 1, s))) {
    return st;
  }
  if (T) T->end(SMSM_STAGE_ROWFFT_INV);
  // The border band needs v only: while the solve is captured it is a branch of its own beside the column
  // stage, and the x transform that follows both adds its result to the band's pixels of q.  (Timed
  // solves keep one stream, so that a bracket holds its stage alone.)
  const bool fork = T && !T->mask && lambda != 0.f;
  cudaStream_t bs = fork ? P->band_s[P->lane] : s;
  if (lambda != 0.f) {
    if (fork) {
      SMSM_CUDA_TRY(cudaEventRecord(P->band_ev[2 * P->lane], s));
      SMSM_CUDA_TRY(cudaStreamWaitEvent(bs, P->band_ev[2 * P->lane], 0));
    }
    if (T) T->begin(SMSM_STAGE_BAND);
    if ((st = launch_band(P, v, q, lambda, with_dots ? P->part_pq_band : nullptr, 0, bs))) return st;
    if (T) T->end(SMSM_STAGE_BAND);
    if (fork) SMSM_CUDA_TRY(cudaEventRecord(P->band_ev[2 * P->lane + 1], bs));
  } else if (with_dots) {
    SMSM_CUDA_TRY(cudaMemsetAsync(P->part_pq_band, 0, sizeof(double) * SMSM_PART_MAX * P->D, s));
  }
  if (T) T->begin(SMSM_STAGE_COLUMN);
  if ((st = launch_col(P, COL_NORMAL, 0, P->hA, P->hB, nullptr, lambda != 0.f ? P->multT : nullptr, lambda,
                       with_dots ? P->part_pq_col : nullptr, s)))
    return st;
  if (T) T->end(SMSM_STAGE_COLUMN);
  if (T) T->begin(SMSM_STAGE_ROWFFT_FWD);
  if (fork) SMSM_CUDA_TRY(cudaStreamWaitEvent(s, P->band_ev[2 * P->lane + 1], 0));
  if ((st = launch_rowfft_in_T(P, P->hB, q, P->D * B, P->N, 0, s, lambda != 0.f ? band_width(P) : 0))) return st;
  if (T) T->end(SMSM_STAGE_ROWFFT_FWD);
  return SMSM_OK;
}

smsm_status apply_normal_pen(smsm_plan_s* P, const float2* v, float2* q, float lambda, int with_dots,
                             cudaStream_t s) {
  return normal_pen_timed(P, v, q, lambda, with_dots, s, nullptr);
}

// The plan restricted to directions [d0, d0 + nd): same geometry, tables and
// coil data; every per-direction buffer offset to the sub-batch; its own report
// record and CG scalar banks.  Used to solve sub-batches as concurrent lanes.
static smsm_plan_s lane_view(const smsm_plan_s* P, int d0, int nd, int lane) {
  smsm_plan_s v = *P;
  const size_t L = P->L, Ns = P->Ns, NN = (size_t)P->N * P->N, C = P->C, Cp = P->Cp, R2 = P->R2;
  const size_t B = L * Ns, dd = (size_t)d0;
  v.D = nd;
  v.LD = nd * P->L;
  const size_t vec = dd * B * NN;
  v.hA += vec;
  v.hB += vec;
  v.phaseT += vec;
  v.xs += vec;
  v.bv += vec;
  v.rv += vec;
  v.pv += vec;
  v.qv += vec;
  const size_t yv = dd * Ns * P->Nc * P->M * P->N;
  v.yh += yv;
  v.ybuf += yv;
  const size_t cc = dd * L * C * C;
  v.G64 += cc;
  v.V += cc;
  v.Wf += cc;
  v.Gw += cc;
  v.Gw2 += cc;
  v.is_rows += dd * L * C;
  v.is_lmax += dd * L;
  v.is_prm += dd * L;
  v.is_flag += dd * L;
  v.scratch += scratch_offset(P, d0, lane);
  v.Gpart += cc * P->gram_nkx;
  v.eig += dd * L * Cp;
  v.sweeps += dd * L;
  v.wper += dd * L * Ns * Ns * R2 * R2;
  v.wcls += dd * L * R2 * R2 * Ns * Ns * R2 * R2;
  v.multT += dd * L * mult_planes(Ns) * NN;
  v.part_pq_col += dd * SMSM_PART_MAX;
  v.part_pq_band += dd * SMSM_PART_MAX;
  v.part_rr += 2 * dd * SMSM_PART_MAX;
  v.st += dd;
  v.rep = P->rep + lane;
  v.lane = lane;
  if (P->Rpart) {
    const size_t R2C = 2 * (size_t)gram_tc_cp(P);
    v.Rpart += dd * L * P->gram_tc_nG * R2C * R2C;
  }
  return v;
}

// b = A^H y and the starting point
static smsm_status enqueue_prologue(smsm_plan_s* P, const smsm_params* prm, cudaStream_t s, Timer* T) {
  smsm_status st;
  const int B = P->L * P->Ns;
  const int D = P->D;
  k_reset_state<<<1, 128, 0, s>>>(P->st, D);
  SMSM_LAUNCH_CHECK("k_reset_state");
  T->begin(SMSM_STAGE_ADJOINT);
  if ((st = launch_rowfft_out_T(P, P->ybuf, P->yh, D * P->Ns * P->Nc, P->M, 1, s))) return st;
  if ((st = launch_col(P, COL_ADJ, 0, P->yh, P->hB, nullptr, nullptr, 0.f, nullptr, s))) return st;
  if ((st = launch_rowfft_in_T(P, P->hB, P->bv, D * B, P->N, 0, s))) return st;
  T->end(SMSM_STAGE_ADJOINT);
  if (!prm->warm)
    SMSM_CUDA_TRY(cudaMemcpyAsync(P->xs, P->bv, sizeof(float2) * (size_t)D * B * P->N * P->N,
                                  cudaMemcpyDeviceToDevice, s));
  return SMSM_OK;
}

// Outer iteration k: Gram, eigen step and weights (after `eig_wait` when given;
// `eig_done` recorded after them when given), filters, J CG steps.
static smsm_status enqueue_outer(smsm_plan_s* P, const smsm_params* prm, int k, cudaStream_t s, Timer* T,
                                 cudaEvent_t eig_wait, cudaEvent_t eig_done) {
  smsm_status st;
  const int B = P->L * P->Ns;
  const int D = P->D;
  const size_t n4 = (size_t)B * P->N * P->N / 2;  // float4 per direction
  const int nvb = vec_blocks(P);
  const int nbb = band_blocks(P);
  const float lam = (float)prm->lambda;
  double* rr0 = P->part_rr;
  double* rr1 = P->part_rr + (size_t)SMSM_PART_MAX * D;
  const dim3 vg(nvb, D);
  T->begin(SMSM_STAGE_GRAM);
  if ((st = gram_lag_supported(P) ? launch_gram_lag(P, P->xs, P->G64, s) : launch_gram(P, P->xs, P->G64, s)))
    return st;
  T->end(SMSM_STAGE_GRAM);
  if (eig_wait) SMSM_CUDA_TRY(cudaStreamWaitEvent(s, eig_wait, 0));
  if ((st = launch_eig_weights(P, P->G64, k, prm, s, T))) return st;
  if (eig_done) SMSM_CUDA_TRY(cudaEventRecord(eig_done, s));
  T->begin(SMSM_STAGE_FILTERS);
  if ((st = launch_filters(P, P->Wf, s))) return st;
  T->end(SMSM_STAGE_FILTERS);
  if ((st = normal_pen_timed(P, P->xs, P->qv, lam, 0, s, T))) return st;
  T->begin(SMSM_STAGE_CG);
  k_cg_init<<<vg, VEC_THREADS, 0, s>>>((const float4*)P->bv, (const float4*)P->qv, (float4*)P->rv, (float4*)P->pv,
                                        n4, rr0);
  SMSM_LAUNCH_CHECK("k_cg_init");
  T->end(SMSM_STAGE_CG);
  // the report's sums go to the lane's side stream, which the next band step joins again before rr0 is rewritten
  const bool side = !T->mask && lam != 0.f && prm->cg_iters > 0;
  cudaStream_t rs = side ? P->band_s[P->lane] : s;
  auto fork = [&]() -> cudaError_t {
    if (!side) return cudaSuccess;
    cudaError_t e = cudaEventRecord(P->band_ev[2 * P->lane], s);
    return e == cudaSuccess ? cudaStreamWaitEvent(rs, P->band_ev[2 * P->lane], 0) : e;
  };
  SMSM_CUDA_TRY(fork());
  k_record<<<1, VEC_THREADS, 0, rs>>>(P->rep, k, 0, rr0, nvb);
  SMSM_LAUNCH_CHECK("k_record");
  for (int j = 0; j < prm->cg_iters; ++j) {
    double* rin = (j & 1) ? rr1 : rr0;
    double* rout = (j & 1) ? rr0 : rr1;
    // step j > 0 first completes step j-1: p = r + beta p, beta = rr(rin) / rr(rout) (the
    // rout bank still holds the previous <r,r> until this step's update overwrites it)
    const PUpdate pu{P->rv, rin, rout, nvb};
    if ((st = normal_pen_timed(P, P->pv, P->qv, lam, 1, s, T, j ? &pu : nullptr))) return st;
    T->begin(SMSM_STAGE_CG);
    k_cg_update<<<vg, VEC_THREADS, 0, s>>>((float4*)P->xs, (float4*)P->rv, (const float4*)P->pv,
                                            (const float4*)P->qv, n4, P->part_pq_col, P->N, P->part_pq_band,
                                            lam != 0.f ? nbb : 0, rin, nvb, rout, P->st);
    SMSM_LAUNCH_CHECK("k_cg_update");
    T->end(SMSM_STAGE_CG);
  }
  double* rend = (prm->cg_iters & 1) ? rr1 : rr0;  // bank of the last write
  SMSM_CUDA_TRY(fork());
  k_record<<<1, VEC_THREADS, 0, rs>>>(P->rep, k, 1, rend, nvb);
  SMSM_LAUNCH_CHECK("k_record");
  if (side && k + 1 == prm->outer_iters) {  // nothing joins it any more
    SMSM_CUDA_TRY(cudaEventRecord(P->band_ev[2 * P->lane + 1], rs));
    SMSM_CUDA_TRY(cudaStreamWaitEvent(s, P->band_ev[2 * P->lane + 1], 0));
  }
  return SMSM_OK;
}

// lanes actually used for these parameters
static int solve_lanes(const smsm_plan_s* P, const smsm_params* prm) {
  int n = prm->lanes > 0 ? prm->lanes : (P->tuned_lanes > 0 ? P->tuned_lanes : (P->D >= 9 ? 3 : (P->D >= 4 ? 2 : 1)));
  if (n > SMSM_MAX_LANES) n = SMSM_MAX_LANES;
  if (n > P->D) n = P->D;
  return n < 1 ? 1 : n;
}

// The whole solve on stream s (being captured).  Stage timing brackets the
// launches of lane 0 (its own stream).  With several lanes, lane k solves
// directions [k D / n, (k+1) D / n) on its own stream, and lane k's first weight
// step waits for lane k-1's: the lanes start out of phase, so that one lane's
// latency-bound kernels (the eigensolvers above all, where they run: a few CTAs)
// are beside the other lanes' full-GPU ones.  Without an eigen-decomposition the lanes matter little: the
// autotuner's shortened solve of 26 directions of 128 x 128 takes 23.6, 23.5 and 23.3 ms with one, two and three.
// (Forcing the eigen steps to alternate for the whole solve measured slower with three or more lanes: it
// serialises them.)
static smsm_status enqueue_solve(smsm_plan_s* P, const smsm_params* prm, cudaStream_t s) {
  smsm_status st;
  if (prm->timing && !P->tpool) P->tpool = new TimingPool();
  if (P->tpool) ((TimingPool*)P->tpool)->used = 0;
  Timer T{(TimingPool*)P->tpool, prm->timing, s};
  Timer T0{nullptr, 0, s};
  const int nl = solve_lanes(P, prm);
  if (nl == 1) {
    if ((st = enqueue_prologue(P, prm, s, &T))) return st;
    for (int k = 0; k < prm->outer_iters; ++k)
      if ((st = enqueue_outer(P, prm, k, s, &T, nullptr, nullptr))) return st;
  } else {
    smsm_plan_s view[SMSM_MAX_LANES];
    cudaStream_t ls[SMSM_MAX_LANES];
    cudaEvent_t fork = P->lane_ev[0];
    cudaEvent_t* join = P->lane_ev + 1;                   // [nl]
    cudaEvent_t* eigd = P->lane_ev + 1 + SMSM_MAX_LANES;  // [nl]
    SMSM_CUDA_TRY(cudaEventRecord(fork, s));
    for (int k = 0; k < nl; ++k) {
      const int d0 = (int)((long)k * P->D / nl), d1 = (int)((long)(k + 1) * P->D / nl);
      view[k] = lane_view(P, d0, d1 - d0, k);
      ls[k] = k == 0 ? s : P->lane_s[k];
      if (k) SMSM_CUDA_TRY(cudaStreamWaitEvent(ls[k], fork, 0));
      if ((st = enqueue_prologue(&view[k], prm, ls[k], k ? &T0 : &T))) return st;
    }
    for (int j = 0; j < prm->outer_iters; ++j)
      for (int k = 0; k < nl; ++k) {
        cudaEvent_t wait = (k && j == 0) ? eigd[k - 1] : nullptr;
        if ((st = enqueue_outer(&view[k], prm, j, ls[k], k ? &T0 : &T, wait, eigd[k]))) return st;
      }
    for (int k = 1; k < nl; ++k) {
      SMSM_CUDA_TRY(cudaEventRecord(join[k], ls[k]));
      SMSM_CUDA_TRY(cudaStreamWaitEvent(s, join[k], 0));
    }
  }
  if (T.err != cudaSuccess) {
    smsm_set_error("timing events: %s", cudaGetErrorString(T.err));
    return SMSM_ERR_CUDA;
  }
  return SMSM_OK;
}

static bool same_params(const smsm_params* a, const smsm_params* b) { return memcmp(a, b, sizeof(*a)) == 0; }

// Capture (once per parameter set) and instantiate the plan's solve graph.
void solver_drop_graph(smsm_plan_s* P) {
  if (!P->has_graph) return;
  cudaGraphExecDestroy(P->gexec);
  cudaGraphDestroy(P->graph);
  P->has_graph = 0;
  ++P->graph_gen;
}

static smsm_status ensure_graph(smsm_plan_s* P, const smsm_params* prm) {
  if (!P->has_graph || !same_params(&P->gparams, prm)) {
    solver_drop_graph(P);
    cudaGraph_t g;
    SMSM_CUDA_TRY(cudaStreamBeginCapture(P->cap_stream, cudaStreamCaptureModeThreadLocal));
    smsm_status st = enqueue_solve(P, prm, P->cap_stream);
    cudaError_t ce = cudaStreamEndCapture(P->cap_stream, &g);
    if (st) return st;
    if (ce != cudaSuccess) {
      smsm_set_error("stream capture of the solve failed: %s", cudaGetErrorString(ce));
      return SMSM_ERR_CUDA;
    }
    size_t nn = 0;
    cudaGraphGetNodes(g, nullptr, &nn);
    std::vector<cudaGraphNode_t> nodes(nn);
    if (nn) cudaGraphGetNodes(g, nodes.data(), &nn);
    int nk = 0;
    for (size_t i = 0; i < nn; ++i) {
      cudaGraphNodeType t;
      if (cudaGraphNodeGetType(nodes[i], &t) == cudaSuccess && t == cudaGraphNodeTypeKernel) ++nk;
    }
    P->graph_kernels = nk;
    ce = cudaGraphInstantiate(&P->gexec, g, 0);
    if (ce != cudaSuccess) {
      cudaGraphDestroy(g);
      smsm_set_error("graph instantiation failed: %s", cudaGetErrorString(ce));
      return SMSM_ERR_CUDA;
    }
    P->graph = g;  // kept: the group launch embeds it as a child graph
    P->gparams = *prm;
    P->has_graph = 1;
  }
  return SMSM_OK;
}

// The solve of y into x on stream s: inputs in, graph replay, result out.
static smsm_status enqueue_run(smsm_plan_s* P, const void* y, void* x, const smsm_params* prm, cudaStream_t s) {
  const size_t nx = (size_t)P->D * P->L * P->Ns * P->N * P->N;
  const size_t ny = (size_t)P->D * P->Ns * P->Nc * P->M * P->N;
  SMSM_CUDA_TRY(cudaMemcpyAsync(P->ybuf, y, sizeof(float2) * ny, cudaMemcpyDeviceToDevice, s));
  if (prm->warm) SMSM_CUDA_TRY(cudaMemcpyAsync(P->xs, x, sizeof(float2) * nx, cudaMemcpyDeviceToDevice, s));
  SMSM_CUDA_TRY(cudaEventRecord(P->ev0, s));
  SMSM_CUDA_TRY(cudaGraphLaunch(P->gexec, s));
  SMSM_CUDA_TRY(cudaEventRecord(P->ev1, s));
  SMSM_CUDA_TRY(cudaMemcpyAsync(x, P->xs, sizeof(float2) * nx, cudaMemcpyDeviceToDevice, s));
  return SMSM_OK;
}

// Fill *report after the solve enqueued on s (synchronises s).
static smsm_status fill_report(smsm_plan_s* P, const smsm_params* prm, smsm_report* report, cudaStream_t s) {
  DevReport hr;
  std::vector<SolverState> hs(P->D);
  SMSM_CUDA_TRY(cudaMemcpyAsync(&hr, P->rep, sizeof(hr), cudaMemcpyDeviceToHost, s));
  SMSM_CUDA_TRY(cudaMemcpyAsync(hs.data(), P->st, sizeof(SolverState) * P->D, cudaMemcpyDeviceToHost, s));
  SMSM_CUDA_TRY(cudaStreamSynchronize(s));
  memset(report, 0, sizeof(*report));
  for (int d = 0; d < P->D && !report->status; ++d) report->status = hs[d].status;
  int flag = 0;
  SMSM_CUDA_TRY(cudaMemcpy(&flag, P->devflag, sizeof(int), cudaMemcpyDeviceToHost));
  if (!report->status && flag) report->status = flag;
  report->outer_done = prm->outer_iters;
  const int K = prm->outer_iters < SMSM_MAX_OUTER ? prm->outer_iters : SMSM_MAX_OUTER;
  for (int k = 0; k < K; ++k) {
    report->eps[k] = hr.eps[k];
    report->rr_start[k] = hr.rr_start[k];
    report->rr_end[k] = hr.rr_end[k];
    report->sweeps[k] = hr.sweeps[k];
  }
  float ms = 0.f;
  SMSM_CUDA_TRY(cudaEventElapsedTime(&ms, P->ev0, P->ev1));
  report->elapsed_ms = ms;
  report->lanes = solve_lanes(P, prm);
  report->lane0_batch = P->D / report->lanes;
  report->graph_kernels = P->graph_kernels;
  TimingPool* tp = (TimingPool*)P->tpool;
  if (tp && prm->timing) {
    for (size_t k = 0; k < tp->used; ++k) {
      float t = 0.f;
      SMSM_CUDA_TRY(cudaEventElapsedTime(&t, tp->ev[2 * k], tp->ev[2 * k + 1]));
      report->stage_ms[tp->stage[k]] += t;
      report->stage_launches[tp->stage[k]] += 1;
    }
  }
  return SMSM_OK;
}

smsm_status solver_reconstruct(smsm_plan_s* P, const void* y, void* x, const smsm_params* prm,
                               smsm_report* report, cudaStream_t s) {
  smsm_status st;
  if ((st = ensure_graph(P, prm))) return st;
  if ((st = enqueue_run(P, y, x, prm, s))) return st;
  return report ? fill_report(P, prm, report, s) : SMSM_OK;
}

// Independent slice groups, possibly of different geometry (one plan each), solved
// concurrently: every plan's graph runs on the plan's own stream, forked from s and
// joined back into it, so the kernels of small and large groups share the GPU.
// One graph for a whole call of smsm_reconstruct_groups: per group the copy of y in
// (and of the warm start), the group's captured solve as a child graph bracketed by its
// timing events, and the copy of x out; the groups are independent branches, so a single
// graph launch runs every group concurrently.  Instantiated graphs are kept for the
// most recent lists of plans (same captured solves); a call with other y or x buffers
// only re-points the copy nodes.  A plan's destruction drops the graphs holding it.
struct GroupExec {
  std::vector<smsm_plan_s*> plans;
  std::vector<unsigned> gens;
  std::vector<const void*> ys;
  std::vector<void*> xs;
  std::vector<cudaGraphNode_t> in_y, in_x, out;  // copy nodes of each group (in_x: warm start only)
  int warm;
  cudaGraph_t graph;
  cudaGraphExec_t exec;
};
static std::mutex g_group_mu;
static std::vector<GroupExec> g_groups;
#define GROUP_CACHE 8

static void free_group(GroupExec& ge) {
  if (ge.exec) cudaGraphExecDestroy(ge.exec);
  if (ge.graph) cudaGraphDestroy(ge.graph);
}

void solver_forget_plan(smsm_plan_s* P) {
  std::lock_guard<std::mutex> lock(g_group_mu);
  for (size_t i = 0; i < g_groups.size();) {
    bool has = false;
    for (smsm_plan_s* q : g_groups[i].plans) has = has || q == P;
    if (has) {
      free_group(g_groups[i]);
      g_groups.erase(g_groups.begin() + i);
    } else {
      ++i;
    }
  }
}

static size_t group_nx(const smsm_plan_s* P) { return sizeof(float2) * P->D * P->L * P->Ns * P->N * P->N; }
static size_t group_ny(const smsm_plan_s* P) { return sizeof(float2) * P->D * P->Ns * P->Nc * P->M * P->N; }

static cudaError_t build_group_exec(GroupExec& ge) {
  cudaError_t e = cudaGraphCreate(&ge.graph, 0);
  if (e != cudaSuccess) return e;
  const size_t n = ge.plans.size();
  ge.in_y.assign(n, nullptr);
  ge.in_x.assign(n, nullptr);
  ge.out.assign(n, nullptr);
  for (size_t k = 0; k < n && e == cudaSuccess; ++k) {
    smsm_plan_s* P = ge.plans[k];
    cudaGraphNode_t in[2], e0, child, e1;
    int nin = 1;
    e = cudaGraphAddMemcpyNode1D(&in[0], ge.graph, nullptr, 0, P->ybuf, ge.ys[k], group_ny(P),
                                 cudaMemcpyDeviceToDevice);
    ge.in_y[k] = in[0];
    if (e == cudaSuccess && ge.warm) {
      e = cudaGraphAddMemcpyNode1D(&in[1], ge.graph, nullptr, 0, P->xs, ge.xs[k], group_nx(P),
                                   cudaMemcpyDeviceToDevice);
      ge.in_x[k] = in[1];
      nin = 2;
    }
    if (e == cudaSuccess) e = cudaGraphAddEventRecordNode(&e0, ge.graph, in, nin, P->ev0);
    if (e == cudaSuccess) e = cudaGraphAddChildGraphNode(&child, ge.graph, &e0, 1, P->graph);
    if (e == cudaSuccess) e = cudaGraphAddEventRecordNode(&e1, ge.graph, &child, 1, P->ev1);
    if (e == cudaSuccess)
      e = cudaGraphAddMemcpyNode1D(&ge.out[k], ge.graph, &e1, 1, ge.xs[k], P->xs, group_nx(P),
                                   cudaMemcpyDeviceToDevice);
  }
  if (e == cudaSuccess) e = cudaGraphInstantiate(&ge.exec, ge.graph, 0);
  return e;
}

// point the copy nodes of an instantiated group graph at this call's buffers
static cudaError_t repoint_group(GroupExec& ge, const void* const* ys, void* const* xs) {
  cudaError_t e = cudaSuccess;
  for (size_t k = 0; k < ge.plans.size() && e == cudaSuccess; ++k) {
    smsm_plan_s* P = ge.plans[k];
    if (ge.ys[k] != ys[k]) {
      e = cudaGraphExecMemcpyNodeSetParams1D(ge.exec, ge.in_y[k], P->ybuf, ys[k], group_ny(P),
                                             cudaMemcpyDeviceToDevice);
      if (e == cudaSuccess) ge.ys[k] = ys[k];
    }
    if (e == cudaSuccess && ge.xs[k] != xs[k]) {
      if (ge.warm)
        e = cudaGraphExecMemcpyNodeSetParams1D(ge.exec, ge.in_x[k], P->xs, xs[k], group_nx(P),
                                               cudaMemcpyDeviceToDevice);
      if (e == cudaSuccess)
        e = cudaGraphExecMemcpyNodeSetParams1D(ge.exec, ge.out[k], xs[k], P->xs, group_nx(P),
                                               cudaMemcpyDeviceToDevice);
      if (e == cudaSuccess) ge.xs[k] = xs[k];
    }
  }
  return e;
}

// the instantiated group graph of this call (built on first use) or nullptr when it cannot
// be built (the call then falls back to one graph launch per group on forked streams); the
// caller holds g_group_mu until it has launched it, so no other call can evict it meanwhile
static cudaGraphExec_t group_exec(int n, smsm_plan_s* const* plans, const void* const* ys, void* const* xs,
                                  int warm) {
  for (size_t i = 0; i < g_groups.size(); ++i) {
    GroupExec& ge = g_groups[i];
    if ((int)ge.plans.size() != n || ge.warm != warm) continue;
    bool same = true;
    for (int k = 0; k < n && same; ++k) same = ge.plans[k] == plans[k] && ge.gens[k] == plans[k]->graph_gen;
    if (!same) continue;
    if (repoint_group(ge, ys, xs) == cudaSuccess) return ge.exec;
    cudaGetLastError();
    free_group(ge);
    g_groups.erase(g_groups.begin() + i);
    break;
  }
  GroupExec ge;
  ge.plans.assign(plans, plans + n);
  for (int k = 0; k < n; ++k) ge.gens.push_back(plans[k]->graph_gen);
  ge.ys.assign(ys, ys + n);
  ge.xs.assign(xs, xs + n);
  ge.warm = warm;
  ge.graph = nullptr;
  ge.exec = nullptr;
  if (build_group_exec(ge) != cudaSuccess) {
    cudaGetLastError();
    free_group(ge);
    return nullptr;
  }
  if (g_groups.size() >= GROUP_CACHE) {
    free_group(g_groups.front());
    g_groups.erase(g_groups.begin());
  }
  g_groups.push_back(ge);
  return ge.exec;
}

smsm_status solver_reconstruct_groups(int n, smsm_plan_s* const* plans, const void* const* ys, void* const* xs,
                                      const smsm_params* prm, smsm_report* reports, cudaStream_t s) {
  smsm_status st;
  for (int k = 0; k < n; ++k)
    if ((st = ensure_graph(plans[k], prm))) return st;
  // timed solves carry their own event records: those stay on the per-group path
  bool launched = false;
  if (!prm->timing) {
    std::lock_guard<std::mutex> lock(g_group_mu);
    cudaGraphExec_t ex = group_exec(n, plans, ys, xs, prm->warm ? 1 : 0);
    if (ex) {
      SMSM_CUDA_TRY(cudaGraphLaunch(ex, s));
      launched = true;
    }
  }
  if (launched) {
    if (reports)
      for (int k = 0; k < n; ++k)
        if ((st = fill_report(plans[k], prm, &reports[k], s))) return st;
    return SMSM_OK;
  }
  cudaEvent_t fork = plans[0]->lane_ev[0];
  SMSM_CUDA_TRY(cudaEventRecord(fork, s));
  for (int k = 0; k < n; ++k) {
    smsm_plan_s* P = plans[k];
    SMSM_CUDA_TRY(cudaStreamWaitEvent(P->cap_stream, fork, 0));
    if ((st = enqueue_run(P, ys[k], xs[k], prm, P->cap_stream))) return st;
    SMSM_CUDA_TRY(cudaEventRecord(P->lane_ev[1], P->cap_stream));
    SMSM_CUDA_TRY(cudaStreamWaitEvent(s, P->lane_ev[1], 0));
  }
  if (reports)
    for (int k = 0; k < n; ++k)
      if ((st = fill_report(plans[k], prm, &reports[k], s))) return st;
  return SMSM_OK;
}

// SMS-SENSE (the comparison reconstruction of the paper's figures): one k-space per
// slice shared by the shots (Eq. 4 with the given image-domain phase, or unit phase:
// no phase correction), slices unfolded by least squares -- J CG steps on
// A^H A x = A^H y from x = 0.  A^H A is the forward column stage followed by the
// adjoint one (the data-side x transforms of A and A^H cancel, so they are skipped).
smsm_status solver_sense(smsm_plan_s* P, const void* y, const void* phase, void* x, int J, smsm_report* report,
                         cudaStream_t s) {
  smsm_status st;
  const int L = P->L, Ns = P->Ns, N = P->N, D = P->D;
  const size_t NN = (size_t)N * N;
  const size_t nx = (size_t)D * L * NN;  // shared k-space per slice
  const size_t ny = (size_t)D * Ns * P->Nc * P->M * N;
  const size_t n4 = (size_t)L * NN / 2;
  const int nvb = vec_blocks(P);
  const dim3 vg(nvb, D);
  double* rr0 = P->part_rr;
  double* rr1 = P->part_rr + (size_t)SMSM_PART_MAX * D;
  SMSM_CUDA_TRY(cudaMemcpyAsync(P->ybuf, y, sizeof(float2) * ny, cudaMemcpyDeviceToDevice, s));
  if (phase) {
    if ((st = launch_transpose((const float2*)phase, P->phaseT, D * L * Ns, N, N, s))) return st;
  } else {
    k_fill_one<<<256, 256, 0, s>>>(P->phaseT, (size_t)D * L * Ns * NN);
    SMSM_LAUNCH_CHECK("k_fill_one");
  }
  k_reset_state<<<1, 128, 0, s>>>(P->st, D);
  SMSM_LAUNCH_CHECK("k_reset_state");
  // b = A^H y
  if ((st = launch_rowfft_out_T(P, P->ybuf, P->yh, D * Ns * P->Nc, P->M, 1, s))) return st;
  if ((st = launch_col(P, COL_ADJ, 1, P->yh, P->hB, P->phaseT, nullptr, 0.f, nullptr, s))) return st;
  if ((st = launch_rowfft_in_T(P, P->hB, P->bv, D * L, N, 0, s))) return st;
  SMSM_CUDA_TRY(cudaMemsetAsync(P->xs, 0, sizeof(float2) * nx, s));
  SMSM_CUDA_TRY(cudaMemsetAsync(P->qv, 0, sizeof(float2) * nx, s));
  k_cg_init<<<vg, VEC_THREADS, 0, s>>>((const float4*)P->bv, (const float4*)P->qv, (float4*)P->rv, (float4*)P->pv,
                                        n4, rr0);
  SMSM_LAUNCH_CHECK("k_cg_init");
  for (int j = 0; j < J; ++j) {
    double* rin = (j & 1) ? rr1 : rr0;
    double* rout = (j & 1) ? rr0 : rr1;
    if ((st = launch_rowfft_out_T(P, P->pv, P->hA, D * L, N, 1, s))) return st;
    if ((st = launch_col(P, COL_FWD, 1, P->hA, P->yh, P->phaseT, nullptr, 0.f, nullptr, s))) return st;
    if ((st = launch_col(P, COL_ADJ, 1, P->yh, P->hB, P->phaseT, nullptr, 0.f, nullptr, s))) return st;
    if ((st = launch_rowfft_in_T(P, P->hB, P->qv, D * L, N, 0, s))) return st;
    k_vdot_part<<<vg, VEC_THREADS, 0, s>>>((const float4*)P->pv, (const float4*)P->qv, n4, P->part_pq_col);
    SMSM_LAUNCH_CHECK("k_vdot_part");
    k_cg_update<<<vg, VEC_THREADS, 0, s>>>((float4*)P->xs, (float4*)P->rv, (const float4*)P->pv,
                                            (const float4*)P->qv, n4, P->part_pq_col, nvb, P->part_pq_band, 0, rin,
                                            nvb, rout, P->st);
    SMSM_LAUNCH_CHECK("k_cg_update");
    k_cg_pupdate<<<vg, VEC_THREADS, 0, s>>>((const float4*)P->rv, (float4*)P->pv, n4, rout, rin, nvb);
    SMSM_LAUNCH_CHECK("k_cg_pupdate");
  }
  SMSM_CUDA_TRY(cudaMemcpyAsync(x, P->xs, sizeof(float2) * nx, cudaMemcpyDeviceToDevice, s));
  if (report) {
    std::vector<SolverState> hs(P->D);
    int flag = 0;  // raised by the column stage where a wait for its copies ran out
    SMSM_CUDA_TRY(cudaMemcpyAsync(hs.data(), P->st, sizeof(SolverState) * P->D, cudaMemcpyDeviceToHost, s));
    SMSM_CUDA_TRY(cudaMemcpyAsync(&flag, P->devflag, sizeof(int), cudaMemcpyDeviceToHost, s));
    SMSM_CUDA_TRY(cudaStreamSynchronize(s));
    memset(report, 0, sizeof(*report));
    for (int d = 0; d < P->D && !report->status; ++d) report->status = hs[d].status;
    if (!report->status && flag) report->status = flag;
    report->lanes = 1;
    report->lane0_batch = P->D;
  }
  return SMSM_OK;
}

// ---------------------------------------------------------------------------
// Autotuner: the split-K block count of the tensor-core Gram and the number of
// concurrent lanes, timed on the plan's own data (y), chosen for the shortest
// device time and remembered per shape for every later plan of that shape in
// the process.
// ---------------------------------------------------------------------------
#include <map>
#include <mutex>
#include <tuple>

typedef std::tuple<int, int, int, int, int, int, int, int, int, int> TuneKey;
static std::mutex g_tune_mu;
static std::map<TuneKey, std::pair<int, int>> g_tune;

static TuneKey tune_key(const smsm_plan_s* P) {
  return TuneKey(P->L, P->Ns, P->Nc, P->N, P->r, P->D, P->precision, P->periodic, P->flags, P->Ldiv);
}

int tune_cache_lookup(const smsm_plan_s* P, int* nG, int* lanes) {
  std::lock_guard<std::mutex> lock(g_tune_mu);
  auto it = g_tune.find(tune_key(P));
  if (it == g_tune.end()) return 0;
  *nG = it->second.first;
  *lanes = it->second.second;
  return 1;
}

smsm_status solver_autotune(smsm_plan_s* P, const void* y, const smsm_params* prm, smsm_tune_report* out,
                            cudaStream_t s) {
  smsm_tune_report rep;
  memset(&rep, 0, sizeof(rep));
  cudaEvent_t e0, e1;
  SMSM_CUDA_TRY(cudaEventCreate(&e0));
  SMSM_CUDA_TRY(cudaEventCreate(&e1));
  smsm_status st = SMSM_OK;
  float ms = 0.f;
  // 1. the Gram's split-K blocks, on the starting point A^H y (FP32 VALID solves take the lagged Gram: there they
  // serve smsm_hankel_gram)
  if (P->gram_tc) {
    const size_t ny = (size_t)P->D * P->Ns * P->Nc * P->M * P->N;
    cudaError_t ce = cudaMemcpyAsync(P->ybuf, y, sizeof(float2) * ny, cudaMemcpyDeviceToDevice, s);
    if (ce != cudaSuccess) st = SMSM_ERR_CUDA;
    if (!st) st = launch_rowfft_out_T(P, P->ybuf, P->yh, P->D * P->Ns * P->Nc, P->M, 1, s);
    if (!st) st = launch_col(P, COL_ADJ, 0, P->yh, P->hB, nullptr, nullptr, 0.f, nullptr, s);
    if (!st) st = launch_rowfft_in_T(P, P->hB, P->xs, P->D * P->L * P->Ns, P->N, 0, s);
    int cand[8];
    const int nc = gram_tc_nG_candidates(P, cand, 8);
    const int keep = P->gram_tc_nG;
    float best = 1e30f;
    int bestn = keep;
    for (int k = 0; k < nc && !st && k < 8; ++k) {
      if (cand[k] > P->gram_nG_max) continue;
      P->gram_tc_nG = cand[k];
      if ((st = launch_gram(P, P->xs, P->G64, s))) break;  // warm-up
      SMSM_CUDA_TRY(cudaEventRecord(e0, s));
      for (int rep3 = 0; rep3 < 3 && !st; ++rep3) st = launch_gram(P, P->xs, P->G64, s);
      SMSM_CUDA_TRY(cudaEventRecord(e1, s));
      SMSM_CUDA_TRY(cudaEventSynchronize(e1));
      SMSM_CUDA_TRY(cudaEventElapsedTime(&ms, e0, e1));
      ms /= 3.f;
      rep.gram_candidates[rep.n_gram] = cand[k];
      rep.gram_ms[rep.n_gram] = ms;
      ++rep.n_gram;
      if (ms < best) {
        best = ms;
        bestn = cand[k];
      }
    }
    P->gram_tc_nG = st ? keep : bestn;
    rep.gram_nG = P->gram_tc_nG;
  }
  // 2. the lanes, on a shortened solve of the same data: six outer iterations (or K), so
  // that the first weight step -- which the lanes start one after another -- weighs as
  // little in the timing as in a full solve (with the eigensolvers, two iterations picked one lane
  // where three were 9 % faster at K = 20)
  if (!st) {
    smsm_params q = *prm;
    q.outer_iters = prm->outer_iters < 6 ? prm->outer_iters : 6;
    q.timing = 0;
    q.warm = 0;
    float best = 1e30f;
    int bestl = 1;
    const int maxl = P->D < SMSM_MAX_LANES ? P->D : SMSM_MAX_LANES;
    for (int l = 1; l <= maxl && !st; ++l) {
      q.lanes = l;
      if ((st = solver_reconstruct(P, y, P->hA, &q, nullptr, s))) break;  // capture + warm-up
      SMSM_CUDA_TRY(cudaEventRecord(e0, s));
      if (!st) st = solver_reconstruct(P, y, P->hA, &q, nullptr, s);
      SMSM_CUDA_TRY(cudaEventRecord(e1, s));
      SMSM_CUDA_TRY(cudaEventSynchronize(e1));
      SMSM_CUDA_TRY(cudaEventElapsedTime(&ms, e0, e1));
      rep.lane_ms[l - 1] = ms;
      if (ms < best) {
        best = ms;
        bestl = l;
      }
    }
    if (!st) {
      P->tuned_lanes = bestl;
      rep.lanes = bestl;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  solver_drop_graph(P);  // the next solve captures with the chosen configuration
  if (st) return st;
  {
    std::lock_guard<std::mutex> lock(g_tune_mu);
    g_tune[tune_key(P)] = std::make_pair(P->gram_tc ? P->gram_tc_nG : 0, P->tuned_lanes);
  }
  if (out) *out = rep;
  return SMSM_OK;
}
