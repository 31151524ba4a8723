// The FP32 solve's Hankel Gram from lagged products (Eqs. 8-9, VALID patches).
//
//   G[(i,p),(j,q)] = sum over n in p + [0, V)^2 of conj(x_i[n]) x_j[n + d],   d = q - p,  V = N - r + 1:
// only the window of the sum depends on p, so all (r - |dy|)(r - |dx|) entries of one lag d share
// their products except on the frame of r - 1 pixels along the image's edges.  The products are formed
// once per (i, j, d), (2r-1)^2 Ns^2 / 2 per pixel instead of the direct C^2 / 2 (C = Ns r^2: ten times
// fewer at r = 6), on FP32 FMAs at every product's full precision.
//
// k_lag: a warp takes one task -- shot i, lag row dy >= 0, NJ shots j -- for 32 image rows, a lane per
// row.  It sweeps along x with the 2r-1 lags dx as accumulators and x_j's 2r-1 neighbours in a rotating
// register window (unrolled over one turn of the window, so nothing is moved): 1 + NJ shared loads per
// NJ (2r-1) complex multiply-adds, FMA-bound.  Columns fall into the left edge (r-1), the core and
// the right edge; the sums over the edges are running ones, one flush per edge column:
//   slot px < r-1: columns px .. r-2;  slot r-1: the core;  slot r-1+px: columns V .. V+px-1,
// so that the window of p along x is slots px, r-1 and r-1+px.  A flush sums over the lanes that hold
// core rows (a halving butterfly) and stores the edge rows' values each on its own.  The core is summed
// in blocks of 2r-1 pixels added to a total, which keeps the FP32 sums' rounding near 5e-8 of
// sqrt(G_ii G_jj), as far as the tensor-core Gram's.
// k_lag_sum: every entry of G from its row tiles and the r-1 edge rows of its window, with
// compensated sums in a fixed order; the lower triangle is the conjugate of the upper.
// Measured per Gram (before: three-piece BF16 split on the tensor cores, C > 144: direct FMA):
// two 128 x 128 slices of 4 shots, r = 6: 330 -> 64 us; six 256 x 256: 740 -> 150 us; four 192 x 192 of 8
// shots: 1750 -> 300 us.  (Tiles copied with plain loads between two barriers: 160, 220 and 506 us.)
#include "common.cuh"

#define LAG_MAXW 8  // warps per CTA at most

__host__ __device__ constexpr int lag_k(int R) { return (32 + 2 * R - 2) / (2 * R - 1); }  // window turns per tile
__host__ __device__ constexpr int lag_xt(int R) { return (2 * R - 1) * lag_k(R); }         // columns per tile
__host__ __device__ constexpr int lag_pitch(int R) { return (lag_xt(R) + 2 * (R - 1)) | 1; }  // odd: lanes a row apart

// sum of v[0..n) over the warp, values dealt out as it goes: afterwards this lane holds the sums
// idx .. idx + cnt - 1 in v[0..cnt) (idx = 0, cnt = n at the start)
template <int n, int h>
__device__ __forceinline__ void lag_halve(float* v, int lane, int& idx, int& cnt) {
  if constexpr (h >= 1) {
    constexpr int n2 = (n + 1) / 2;
    const bool up = lane & h;
#pragma unroll
    for (int k = 0; k < n2; ++k) {
      const float hi = k + n2 < n ? v[k + n2] : 0.f;
      const float got = __shfl_xor_sync(0xffffffffu, up ? v[k] : hi, h);
      v[k] = (up ? hi : v[k]) + got;
    }
    if (up) idx += n2;
    cnt = up ? max(cnt - n2, 0) : min(cnt, n2);
    lag_halve<n2, h / 2>(v, lane, idx, cnt);
  }
}
__host__ __device__ constexpr int lag_left(int n) {  // values per lane after five halvings
  for (int k = 0; k < 5; ++k) n = (n + 1) / 2;
  return n;
}

template <int R, int NJ>
__global__ void __launch_bounds__(32 * LAG_MAXW) k_lag(const float2* __restrict__ x, float2* __restrict__ part, int Ns,
                                                       int N, int ntask, int l0, int nbuf) {
  constexpr int R2 = 2 * R - 1, E = R - 1, K = lag_k(R), XT = lag_xt(R), LP = lag_pitch(R), W = XT + 2 * E;
  constexpr int ROWS = 32 + E, NV = NJ * R2;
  extern __shared__ float2 lsm[];  // [nbuf][Ns][ROWS][LP]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int task = blockIdx.x * (blockDim.x >> 5) + warp;
  const bool live = task < ntask;
  const int njg = (Ns + NJ - 1) / NJ;
  const int dy = live ? task % R : 0, jg = live ? (task / R) % njg : 0, i = live ? task / (R * njg) : 0;
  const int V = N - R + 1, y0 = blockIdx.y * 32, row = y0 + lane;
  const int edge = row < E ? row : (row >= V ? E + row - V : -1);  // edge row index (rows from N on: idle lanes)
  const bool core = edge < 0;
  const int nty = gridDim.y;
  const float2* xl = x + (size_t)(l0 + blockIdx.z) * Ns * N * N;
  float2* tl = part + ((size_t)blockIdx.z * ntask + (live ? task : 0)) * (nty + 2 * E) * R2 * NV;
  // the tiles along x: the left edge, the core's, the right edge; columns [xs - E, xs + XT + E) of rows
  // y0 .. y0 + 31 + E of every shot, zero outside the image, a warp per row, by asynchronous copies.
  // With two buffers a tile is on its way while the one before is summed.
  const int ncore = (V - E + XT - 1) / XT, ntile = ncore + (E > 0 ? 2 : 0), tile_elems = Ns * ROWS * LP;
  auto tile_xs = [&](int t) { return E == 0 ? t * XT : (t == 0 ? 0 : (t == ntile - 1 ? V : E + (t - 1) * XT)); };
  auto issue = [&](int t) {
    const int xs = tile_xs(t);
    float2* dst = lsm + (t % nbuf) * tile_elems;
    for (int rr = warp; rr < Ns * ROWS; rr += blockDim.x >> 5) {
      const int s = rr / ROWS, gy = y0 + rr - s * ROWS;
      const float2* src = xl + ((size_t)s * N + (gy < N ? gy : 0)) * N;
#pragma unroll
      for (int c0 = 0; c0 < W; c0 += 32) {
        const int c = c0 + lane, gx = xs - E + c;
        if (c < W) cp_async8_zero(dst + rr * LP + c, gx >= 0 && gx < N ? src + gx : src, gy < N && gx >= 0 && gx < N);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const float2* pa;
  const float2* pb[NJ];
  // tile t is in shared memory and, with two buffers, tile t + 1 on its way
  auto arrive = [&](int t) {
    if (nbuf == 1) {
      if (t) {
        __syncthreads();  // tile t - 1 is no longer read
        issue(t);
      }
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();  // tile t has landed for everyone, and tile t - 1's buffer is free
      if (t + 1 < ntile) issue(t + 1);
    }
    const float2* base = lsm + (t % nbuf) * tile_elems;
    pa = base + (i * ROWS + lane) * LP + E;
#pragma unroll
    for (int jj = 0; jj < NJ; ++jj) {
      const int j = min(jg * NJ + jj, Ns - 1);
      pb[jj] = base + (j * ROWS + lane + dy) * LP;  // neighbour dx of column c: pb[c + E + dx]
    }
  };
  issue(0);
  int tile = 0;
  float2 acc[NJ][R2];
  auto clear = [&](float2(&a)[NJ][R2]) {
#pragma unroll
    for (int jj = 0; jj < NJ; ++jj)
#pragma unroll
      for (int d = 0; d < R2; ++d) a[jj][d] = cmk(0.f, 0.f);
  };
  auto flush = [&](int f) {
    if (!live) return;
    float v[2 * NV];
    if (!core && row < N) {
      float2* o = tl + ((size_t)(nty + edge) * R2 + f) * NV;
#pragma unroll
      for (int jj = 0; jj < NJ; ++jj)
#pragma unroll
        for (int d = 0; d < R2; ++d) o[jj * R2 + d] = acc[jj][d];
    }
#pragma unroll
    for (int jj = 0; jj < NJ; ++jj)
#pragma unroll
      for (int d = 0; d < R2; ++d) {
        v[2 * (jj * R2 + d)] = core ? acc[jj][d].x : 0.f;
        v[2 * (jj * R2 + d) + 1] = core ? acc[jj][d].y : 0.f;
      }
    int idx = 0, cnt = 2 * NV;
    lag_halve<2 * NV, 16>(v, lane, idx, cnt);
    float* o = reinterpret_cast<float*>(tl + ((size_t)blockIdx.y * R2 + f) * NV);
#pragma unroll
    for (int k = 0; k < lag_left(2 * NV); ++k)
      if (k < cnt) o[idx + k] = v[k];
  };
  auto one = [&](int c) {  // the products of tile column c
    const float2 a = pa[c];
#pragma unroll
    for (int jj = 0; jj < NJ; ++jj)
#pragma unroll
      for (int d = 0; d < R2; ++d) cfmacj(acc[jj][d], a, pb[jj][c + d]);
  };
  if (E > 0) {  // left edge: columns E-1 .. 0, each flushed on top of those before
    arrive(tile++);
    clear(acc);
    for (int e = E - 1; e >= 0; --e) {
      one(e);
      flush(e);
    }
  }
  clear(acc);
  for (int xs = E; xs < V; xs += XT) {
    arrive(tile++);
    float2 w[NJ][R2];
#pragma unroll
    for (int jj = 0; jj < NJ; ++jj)
#pragma unroll
      for (int t = 0; t + 1 < R2; ++t) w[jj][t] = pb[jj][t];
    for (int kb = 0; kb < K; ++kb) {
      if (xs + kb * R2 >= V) break;
      float2 blk[NJ][R2];
      clear(blk);
#pragma unroll
      for (int u = 0; u < R2; ++u) {
        const int c = kb * R2 + u;
        float2 a = pa[c];
        if (xs + c >= V) a = cmk(0.f, 0.f);
#pragma unroll
        for (int jj = 0; jj < NJ; ++jj) {
          w[jj][(u + R2 - 1) % R2] = pb[jj][c + 2 * E];
#pragma unroll
          for (int d = 0; d < R2; ++d) cfmacj(blk[jj][d], a, w[jj][(u + d) % R2]);
        }
      }
#pragma unroll
      for (int jj = 0; jj < NJ; ++jj)
#pragma unroll
        for (int d = 0; d < R2; ++d) acc[jj][d] = cadd(acc[jj][d], blk[jj][d]);
    }
  }
  flush(E);
  if (E > 0) {  // right edge: columns V .. N-1
    arrive(tile);
    clear(acc);
    for (int e = 0; e < E; ++e) {
      one(e);
      flush(E + 1 + e);
    }
  }
}

// One warp per (matrix, task, p_y, p_x), lanes over the NJ (2r-1) lags of the task.
__global__ void __launch_bounds__(256) k_lag_sum(const float2* __restrict__ part, double2* __restrict__ G, int Ns, int r,
                                                 int C, int nj, int ntask, int nty, int l0) {
  const int R2 = 2 * r - 1, E = r - 1, NV = nj * R2, rr = r * r;
  const int lane = threadIdx.x & 31;
  const int item = blockIdx.x * 8 + (threadIdx.x >> 5);  // task * r * r + py * r + px
  if (item >= ntask * rr) return;
  const int px = item % r, py = (item / r) % r, task = item / rr;
  const int njg = (Ns + nj - 1) / nj;
  const int dy = task % r, jg = (task / r) % njg, i = task / (r * njg);
  if (py + dy >= r) return;
  const float2* t = part + ((size_t)blockIdx.y * ntask + task) * (nty + 2 * E) * R2 * NV;
  double2* Gl = G + (size_t)(l0 + blockIdx.y) * C * C;
  for (int k = lane; k < NV; k += 32) {
    const int jj = k / R2, dx = k - jj * R2 - E, j = jg * nj + jj;
    const int qx = px + dx;
    if (j >= Ns || qx < 0 || qx >= r) continue;
    if (dy == 0 && (j < i || (j == i && dx < 0))) continue;  // the conjugate entry writes this one
    float sx = 0.f, sy = 0.f, cx = 0.f, cy = 0.f;
    auto row = [&](int slot) {  // the window along x of one row tile or edge row
      const float2* o = t + (size_t)slot * R2 * NV + k;
      float2 v = o[(size_t)E * NV];
      add2(sx, cx, v.x);
      add2(sy, cy, v.y);
      if (px < E) {
        v = o[(size_t)px * NV];
        add2(sx, cx, v.x);
        add2(sy, cy, v.y);
      }
      if (px > 0) {
        v = o[(size_t)(E + px) * NV];
        add2(sx, cx, v.x);
        add2(sy, cy, v.y);
      }
    };
    for (int ty = 0; ty < nty; ++ty) row(ty);
    for (int e = py; e < E; ++e) row(nty + e);      // rows py .. r-2
    for (int e = 0; e < py; ++e) row(nty + E + e);  // rows V .. V+py-1
    const int a = i * rr + py * r + px, b = j * rr + (py + dy) * r + qx;
    const double re = (double)sx + (double)cx, im = a == b ? 0.0 : (double)sy + (double)cy;
    Gl[(size_t)a * C + b] = make_double2(re, im);
    if (a != b) Gl[(size_t)b * C + a] = make_double2(re, -im);
  }
}

typedef void (*LagFn)(const float2*, float2*, int, int, int, int, int);

// two shots per task up to r = 8 (their sums, block sums and windows fit the registers)
static int lag_nj(int r, int Ns) { return r <= 8 && Ns > 1 ? 2 : 1; }
static int lag_ntask(const smsm_plan_s* P) {
  const int nj = lag_nj(P->r, P->Ns);
  return P->Ns * P->r * ((P->Ns + nj - 1) / nj);
}
static int lag_nty(const smsm_plan_s* P) { return (P->N + 31) / 32; }
static size_t lag_smem(const smsm_plan_s* P) {
  return (size_t)P->Ns * (32 + P->r - 1) * lag_pitch(P->r) * sizeof(float2);
}

size_t gram_lag_per(const smsm_plan_s* P) {  // complex values of one matrix's partial sums
  if (!gram_lag_supported(P)) return 0;
  return (size_t)lag_ntask(P) * (lag_nty(P) + 2 * (P->r - 1)) * P->R2 * lag_nj(P->r, P->Ns) * P->R2;
}

// VALID patches in the FP32 form.  The reduced-precision form asks for BF16 products, PERIODIC patches need no
// windows and wrap around, the generic kernels are asked for.
int gram_lag_supported(const smsm_plan_s* P) {
  return !P->periodic && P->precision == SMSM_PRECISION_FP32 && !(P->flags & SMSM_FLAG_GENERIC_KERNELS);
}

static LagFn lag_fn(int r, int nj) {
  switch (2 * r + nj) {
    case 3: return k_lag<1, 1>;
    case 4: return k_lag<1, 2>;
    case 5: return k_lag<2, 1>;
    case 6: return k_lag<2, 2>;
    case 7: return k_lag<3, 1>;
    case 8: return k_lag<3, 2>;
    case 9: return k_lag<4, 1>;
    case 10: return k_lag<4, 2>;
    case 11: return k_lag<5, 1>;
    case 12: return k_lag<5, 2>;
    case 13: return k_lag<6, 1>;
    case 14: return k_lag<6, 2>;
    case 15: return k_lag<7, 1>;
    case 16: return k_lag<7, 2>;
    case 17: return k_lag<8, 1>;
    case 18: return k_lag<8, 2>;
    case 19: return k_lag<9, 1>;
    case 21: return k_lag<10, 1>;
    case 23: return k_lag<11, 1>;
    default: return k_lag<12, 1>;
  }
}

smsm_status gram_lag_init_attrs(const smsm_plan_s* P) {
  if (!gram_lag_supported(P)) return SMSM_OK;
  // per kernel, not per plan: the most shots
  cudaError_t e = cudaFuncSetAttribute(lag_fn(P->r, lag_nj(P->r, P->Ns)), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       200 * 1024);
  if (e != cudaSuccess || lag_smem(P) > 200 * 1024) {
    smsm_set_error("lagged Gram needs %zu bytes of shared memory: %s", lag_smem(P), cudaGetErrorString(e));
    return SMSM_ERR_ARG;
  }
  return SMSM_OK;
}

smsm_status launch_gram_lag(const smsm_plan_s* P, const float2* x, double2* G, cudaStream_t s) {
  const int nj = lag_nj(P->r, P->Ns), ntask = lag_ntask(P), nty = lag_nty(P);
  const LagFn fn = lag_fn(P->r, nj);
  const int chunk = scratch_cap(P);
  for (int l0 = 0; l0 < P->LD; l0 += chunk) {
    const int n = P->LD - l0 < chunk ? P->LD - l0 : chunk;
    // warps per CTA: they share the staged tile; fewer while that puts CTAs on idle SMs
    int w = LAG_MAXW;
    while (w > 2 && (long)((ntask + w - 1) / w) * nty * n < 152) w /= 2;
    // two tile buffers where they fit beside a second CTA's
    const int nbuf = 2 * lag_smem(P) <= 110 * 1024 ? 2 : 1;
    fn<<<dim3((ntask + w - 1) / w, nty, n), 32 * w, nbuf * lag_smem(P), s>>>(x, P->scratch, P->Ns, P->N, ntask, l0,
                                                                              nbuf);
    SMSM_LAUNCH_CHECK("k_lag");
    k_lag_sum<<<dim3((ntask * P->r * P->r + 7) / 8, n), 256, 0, s>>>(P->scratch, G, P->Ns, P->r, P->C, nj, ntask, nty,
                                                                      l0);
    SMSM_LAUNCH_CHECK("k_lag_sum");
  }
  return SMSM_OK;
}
