// Column stage of A and A^H, a warp per set of transforms.
//
// The mathematics of k_col (operators.cu), per image column x: y transform of the slice-shot lines, then for every
// coil the product with its map, the M-point transform of the folded line (M = N/Ns, the shot mask), the
// CAIPI phase and slice sum (Fig. 1; Eqs. 1-3), or the adjoint chain.  What bounds it is the coil loop,
// Nc L Ns transforms of M points per column and some 8 Ns multiply-adds per transformed point; k_col
// took four to five block barriers per coil and every pass through shared memory.  Here a warp transforms CPW
// coils at once (CPW M = 256 points: eight per lane) on its own: the first pass gets its points straight
// from the folded products in registers, the last one hands them on in registers, and the exchanges between
// go through the warp's own buffer with warp barriers only.
//  * forward: a warp takes (shot i, CPW coils) and walks over the slices: the slice sum stays in the
//    registers of the last pass.  The shot's twiddle is in the image lines beforehand.
//  * adjoint: a warp takes (slice l, shot i) and walks over the coils: the coil sum of its pixels stays in
//    registers (NSM pixels per point), is summed over the warp's CPW coils at the end and gets the shot's
//    conjugate twiddle.
// The coil maps (and the adjoint's data lines) of the next CPW coils are on their way into a second stage by
// bulk copies meanwhile: with loads straight from global memory the warps waited for them three
// quarters of the time.  Instruction issue (27 to 34 %) and shared-memory latency bound it now.
// Tried for the per-coil A^H A as well (forward and adjoint alternating through a buffer of data lines): 252 us
// per 256 x 256 column stage of two directions against k_col_fast's 221, not kept.
// A short set of 128 points for 3 or more shots halves what an adjoint lane accumulates: two CTAs of 12 warps
// per SM instead of one (248 -> 205 us in the second figure).
// Measured (k_col before): A, 256 x 256, 3 slices, 4 shots, 32 coils, 2 directions 273 -> 119 us; A^H, 128 x 128, 2
// slices, 4 shots, 32 coils, 26 directions 571 -> 205 us; 192 x 192, 3 slices, 2 shots, 16 coils, 4 directions
// with phase: A 126 -> 58 us, A^H 84 -> 62 us; A, 64 x 64, 2 slices, 4 shots, 8 coils 40 -> 10 us.
#include "common.cuh"
#include "fft.cuh"
#include "umma.cuh"

template <int M>
__host__ __device__ constexpr int cw_radix(int s) {  // radix of the pass after the radices of product s
  const int rem = M / s;
  if (M == 8) return s == 1 ? 4 : 2;  // a short last pass: what an adjoint lane accumulates
  return rem % 8 == 0 ? 8 : (rem % 4 == 0 ? 4 : (rem % 2 == 0 ? 2 : 3));
}
template <int M>
__host__ __device__ constexpr int cw_last() {  // radix of the last pass
  int s = 1;
  while (s * cw_radix<M>(s) < M) s *= cw_radix<M>(s);
  return cw_radix<M>(s);
}
__host__ __device__ constexpr int cw_cpw(int M, int elems) { return elems / M > 0 ? elems / M : 1; }
// buffer index of point e of a line: one slot of padding per eight points, so that the strided stores of a
// radix-8 pass fall into distinct banks
__host__ __device__ constexpr int cw_at(int e) { return e + (e >> 3); }
__host__ __device__ constexpr int cw_ld(int M) { return cw_at(M) + 1; }

template <int R, bool INV>
__device__ __forceinline__ void cw_dft(float2* v) {
  if constexpr (R == 8)
    dft8<INV>(v);
  else if constexpr (R == 4)
    dft4<INV>(v);
  else if constexpr (R == 2)
    dft2<INV>(v);
  else
    dft3<INV>(v);
}

// index step of r in cw_at(base + r * step), a multiple of eight apart (0: not one)
__host__ __device__ constexpr int cw_step(int step) { return step % 8 == 0 ? step + step / 8 : 0; }

// The passes after product S of the M-point transforms of the warp's CPW lines, in place in buf (a pass holds its
// points in registers between its loads and its stores) -> sink(round, line, j, v): points j + r M/R, r < R, of
// the result.
template <bool INV, int M, int CPW, int S, class Sink>
__device__ __forceinline__ void cw_rest(float2* buf, const float2* tw, int lane, Sink sink) {
  constexpr int R = cw_radix<M>(S), nR = M / R, LD = cw_ld(M), ROUNDS = (CPW * nR + 31) / 32;
  constexpr bool last = S * R == M;
  float2 v[ROUNDS][R];
#pragma unroll
  for (int rd = 0; rd < ROUNDS; ++rd) {
    const int t = lane + 32 * rd;
    if (t < CPW * nR) {
      const int cs = t / nR, j = t - cs * nR;
      const float2* src = buf + cs * LD;
      if constexpr (cw_step(nR) > 0) {
        src += cw_at(j);
#pragma unroll
        for (int r = 0; r < R; ++r) v[rd][r] = src[r * cw_step(nR)];
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r) v[rd][r] = src[cw_at(j + r * nR)];
      }
    }
  }
  if constexpr (!last) __syncwarp();
#pragma unroll
  for (int rd = 0; rd < ROUNDS; ++rd) {
    const int t = lane + 32 * rd;
    if (t < CPW * nR) {
      const int cs = t / nR, j = t - cs * nR, k = j % S;
#pragma unroll
      for (int r = 1; r < R; ++r) v[rd][r] = cmul(v[rd][r], tw_get<INV>(tw, r * k * (M / (S * R))));
      cw_dft<R, INV>(v[rd]);
      if constexpr (last) {
        sink(rd, cs, j, v[rd]);
      } else {
        float2* dst = buf + cs * LD;
        if constexpr (cw_step(S) > 0) {
          dst += cw_at((j - k) * R + k);
#pragma unroll
          for (int r = 0; r < R; ++r) dst[r * cw_step(S)] = v[rd][r];
        } else {
#pragma unroll
          for (int r = 0; r < R; ++r) dst[cw_at((j - k) * R + k + r * S)] = v[rd][r];
        }
      }
    }
  }
  if constexpr (!last) {
    __syncwarp();
    cw_rest<INV, M, CPW, S * R>(buf, tw, lane, sink);
  }
}

// M-point transforms of CPW lines: source(line, j, v) fills points j + r M/R of the first pass
template <bool INV, int M, int CPW, class Source, class Sink>
__device__ __forceinline__ void cw_fft(float2* buf, const float2* tw, int lane, Source source, Sink sink) {
  constexpr int R = cw_radix<M>(1), nR = M / R, LD = cw_ld(M), ROUNDS = (CPW * nR + 31) / 32;
#pragma unroll
  for (int rd = 0; rd < ROUNDS; ++rd) {
    const int t = lane + 32 * rd;
    if (t < CPW * nR) {
      const int cs = t / nR, j = t - cs * nR;
      float2 v[R];
      source(cs, j, v);
      cw_dft<R, INV>(v);
      float2* dst = buf + cs * LD + cw_at(j * R);
      if constexpr (8 % R == 0) {  // eight consecutive points have no padding between
#pragma unroll
        for (int r = 0; r < R; ++r) dst[r] = v[r];
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r) buf[cs * LD + cw_at(j * R + r)] = v[r];
      }
    }
  }
  __syncwarp();
  cw_rest<INV, M, CPW, R>(buf, tw, lane, sink);
  __syncwarp();  // the buffer may be written again
}

struct CwShared {
  float2 *img, *tmp;            // [B][N] lines (tmp shares its place with a stage)
  float2 *twN, *twM, *cp;       // tables: [N], [M], [L][Ns][M]
  const float2* ts;             // [Ns][N] shot twiddles (global)
  float2* buf;                  // this warp's transform buffer
  float2* stage[2];             // staged coils: maps [L][CG][lds], data [Ns][CG][ldd] (adjoint)
  int lds, ldd, cg;             // pitches of a staged map and data line, coils per stage
};

template <int M, int ELEMS>
__host__ __device__ constexpr int cw_buf() { return (cw_cpw(M, ELEMS) * cw_ld(M) + 1) & ~1; }
// padding of a staged line that a pass of radix R reads: the lines of a warp's coils then start in the banks
// after one another's
__host__ __device__ constexpr int cw_pad(int M, int R) { return (M / R + 1) & ~1; }

__host__ __device__ inline int cw_even(int n) { return (n + 1) & ~1; }  // 16-byte alignment of what follows

// Coils [t cg, t cg + cg) into stage t & 1: one bulk copy per line, by thread 0
__device__ __forceinline__ void cw_issue(const ColArgs& a, const CwShared& s, uint64_t* bar, const float2* data, int t,
                                         int x) {
  const int c0 = t * s.cg, n = min(s.cg, a.Nc - c0), N = a.N, M = a.M;
  float2* st = s.stage[t & 1];
  const uint32_t row = (uint32_t)(N * sizeof(float2)), drow = (uint32_t)(M * sizeof(float2));
  mbar_arrive_expect_tx(&bar[t & 1], (uint32_t)(a.L * n) * row + (data ? (uint32_t)(a.Ns * n) * drow : 0u));
  for (int l = 0; l < a.L; ++l)
    for (int c = 0; c < n; ++c)
      tma_bulk_g2s(st + (l * s.cg + c) * s.lds, a.sensT + ((size_t)(l * a.Nc + c0 + c) * N + x) * N, row, &bar[t & 1]);
  if (data) {
    float2* dy = st + a.L * s.cg * s.lds;
    for (int i = 0; i < a.Ns; ++i)
      for (int c = 0; c < n; ++c)
        tma_bulk_g2s(dy + (i * s.cg + c) * s.ldd, data + ((size_t)(i * a.Nc + c0 + c) * N + x) * M, drow, &bar[t & 1]);
  }
}

#define CW_MAXITER (1L << 22)
__device__ __forceinline__ bool cw_wait(uint64_t* bar, uint32_t parity) {  // bounded
  for (long it = 0; it < CW_MAXITER; ++it) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.b32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// Stage t has landed for every thread and stage t - 1 is no longer read: thread 0 sends for stage t + 1.
// False (for every thread alike) when the bounded wait ran out; the copies in flight have then been waited for.
__device__ __forceinline__ bool cw_arrive(const ColArgs& a, const CwShared& s, uint64_t* bar, const float2* data, int t,
                                          int nst, int x) {
  if (!__syncthreads_and(cw_wait(&bar[t & 1], (uint32_t)((t >> 1) & 1)))) {
    if (threadIdx.x == 0) {
      atomicExch(a.errflag, SMSM_ERR_TIMEOUT);
      cw_wait(&bar[t & 1], (uint32_t)((t >> 1) & 1));
      if (t == 0 && nst > 1) cw_wait(&bar[1], 0);
    }
    return false;
  }
  if (threadIdx.x == 0 && t > 0 && t + 1 < nst) cw_issue(a, s, bar, data, t + 1, x);
  return true;
}

// contribution of slice l to shot i's data lines of the CPW staged coils from k0 on: sink(round, coil, j, v) with v =
// the transform of the folded products, points j + r M/RL
template <int M, int CPW, class Sink>
__device__ __forceinline__ void cw_fold_fft(const ColArgs& a, const CwShared& s, const float2* st, const float2* line,
                                            int l, int k0, int n, int lane, Sink sink) {
  cw_fft<false, M, CPW>(
      s.buf, s.twM, lane,
      [&](int cs, int j, float2* v) {
        constexpr int R = cw_radix<M>(1), nR = M / R;
        const float2* srow = st + (l * s.cg + min(k0 + cs, n - 1)) * s.lds + j;
        const float2* q = line + j;
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = cmk(0.f, 0.f);
#pragma unroll 2
        for (int t = 0; t < a.Ns; ++t, srow += M, q += M)
#pragma unroll
          for (int r = 0; r < R; ++r) cfma(v[r], srow[r * nR], q[r * nR]);
      },
      sink);
}

// pixels of (l, i) of the CPW staged coils from k0 on added to acc; in(coil, m) is the data (conjugate CAIPI phase
// applied here)
template <int M, int CPW, int NSM, class In>
__device__ __forceinline__ void cw_adjoint(const ColArgs& a, const CwShared& s, const float2* st, int l, int i, int k0,
                                           int n, int lane,
                                           float2 (&acc)[NSM][(CPW * (M / cw_last<M>()) + 31) / 32][cw_last<M>()],
                                           In in) {
  constexpr int RL = cw_last<M>(), NL = M / RL;
  const float2* cp = s.cp + (l * a.Ns + i) * M;
  cw_fft<true, M, CPW>(
      s.buf, s.twM, lane,
      [&](int cs, int j, float2* v) {
        constexpr int R = cw_radix<M>(1), nR = M / R;
        const bool live = k0 + cs < n;
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = live ? cmulcj(cp[j + r * nR], in(k0 + cs, j + r * nR)) : cmk(0.f, 0.f);
      },
      [&](int rd, int cs, int j, const float2* v) {
        const float2* srow = st + (l * s.cg + min(k0 + cs, n - 1)) * s.lds + j;
#pragma unroll
        for (int t = 0; t < NSM; ++t)
          if (t < a.Ns) {
#pragma unroll
            for (int r = 0; r < RL; ++r) cfmacj(acc[t][rd][r], srow[t * M + r * NL], v[r]);
          }
      });
}

// acc summed over the warp's coils, times the shot's conjugate twiddle: line (l, i) of dst (added with add)
template <int M, int CPW, int NSM>
__device__ __forceinline__ void cw_collect(const ColArgs& a, const CwShared& s, int l, int i, int lane,
                                           float2 (&acc)[NSM][(CPW * (M / cw_last<M>()) + 31) / 32][cw_last<M>()],
                                           float2* dst, bool add) {
  constexpr int RL = cw_last<M>(), NL = M / RL, ROUNDS = (CPW * NL + 31) / 32;
  constexpr bool POW2 = (M & (M - 1)) == 0 && NL <= 32;
  float2* d = dst + (l * a.Ns + i) * a.N;
  const float2* ts = s.ts + i * a.N;
  if constexpr (POW2) {
    // NL divides 32: lanes NL, 2 NL, ... apart and further rounds hold other coils' same pixels
#pragma unroll
    for (int t = 0; t < NSM; ++t)
      if (t < a.Ns) {
#pragma unroll
        for (int r = 0; r < RL; ++r) {
          float2 v = acc[t][0][r];
#pragma unroll
          for (int rd = 1; rd < ROUNDS; ++rd) v = cadd(v, acc[t][rd][r]);
#pragma unroll
          for (int o = NL; o < 32; o <<= 1) {
            v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
            v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
          }
          if (lane < NL) {
            const int y = lane + r * NL + t * M;
            const float2 u = cmulcj(__ldg(ts + y), v);
            d[y] = add ? cadd(d[y], u) : u;
          }
        }
      }
  } else {
    for (int c = 0; c < CPW; ++c) {  // one coil of the set after the other
#pragma unroll
      for (int rd = 0; rd < ROUNDS; ++rd) {
        const int t0 = lane + 32 * rd, cs = t0 / NL, j = t0 - cs * NL;
        if (t0 < CPW * NL && cs == c) {
#pragma unroll
          for (int t = 0; t < NSM; ++t)
            if (t < a.Ns) {
#pragma unroll
              for (int r = 0; r < RL; ++r) {
                const int y = j + r * NL + t * M;
                const float2 u = cmulcj(__ldg(ts + y), acc[t][rd][r]);
                d[y] = (c || add) ? cadd(d[y], u) : u;
              }
            }
        }
      }
      __syncwarp();
    }
  }
}

// lines in the hybrid layout -> s.img
__device__ __forceinline__ void cw_lines_in(const ColArgs& a, const CwShared& s, const float2* in, int lines, int stride,
                                            int x) {
  const int N = a.N;
  const size_t NN = (size_t)N * N;
  for (int e = threadIdx.x; e < lines * N; e += blockDim.x) {
    const int b = e / N, ky = e - b * N;
    s.img[b * stride + ky] = cscale(in[(size_t)b * NN + (size_t)x * N + ky], sgn_par(ky));
  }
  __syncthreads();
}

// Shared-memory layout, the same function on host and device: everything in complex values, every part 16-byte
// aligned.  The lines' second buffer takes stage 1's place.
enum { CW_FWD = 0, CW_ADJ = 1 };
template <int M, int ELEMS>
__host__ __device__ inline size_t cw_plan(int mode, int L, int Ns, int N, int nw, int cg, CwShared* s, float2* sm,
                                          int warp) {
  const int B = L * Ns, lines = cw_even(B * N);
  const int lds = N + cw_pad(M, mode == CW_FWD ? cw_radix<M>(1) : cw_last<M>()), ldd = M + cw_pad(M, cw_radix<M>(1));
  int stage = cw_even(L * cg * lds + (mode == CW_ADJ ? Ns * cg * ldd : 0));
  const int second = lines > stage ? lines : stage;
  size_t o = 0;
  const size_t o_img = o;
  o += lines;
  const size_t o_st0 = o;
  o += stage;
  const size_t o_st1 = o;
  o += second;
  const size_t o_buf = o;
  o += (size_t)nw * cw_buf<M, ELEMS>();
  const size_t o_twN = o;
  o += cw_even(N);
  const size_t o_twM = o;
  o += cw_even(M);
  const size_t o_cp = o;
  o += cw_even(B * M);
  if (s) {
    s->img = sm + o_img;
    s->tmp = sm + o_st1;
    s->stage[0] = sm + o_st0;
    s->stage[1] = sm + o_st1;
    s->buf = sm + o_buf + (size_t)warp * cw_buf<M, ELEMS>();
    s->twN = sm + o_twN;
    s->twM = sm + o_twM;
    s->cp = sm + o_cp;
    s->lds = lds;
    s->ldd = ldd;
    s->cg = cg;
  }
  return o * sizeof(float2);
}

template <int M, int ELEMS>
__device__ __forceinline__ CwShared cw_begin(const ColArgs& a, int mode, float2* sm, int cg, uint64_t* bar) {
  CwShared s;
  cw_plan<M, ELEMS>(mode, a.L, a.Ns, a.N, blockDim.x >> 5, cg, &s, sm, threadIdx.x >> 5);
  s.ts = a.tw_shot;
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  for (int e = threadIdx.x; e < a.N; e += blockDim.x) s.twN[e] = a.twN[e];
  for (int e = threadIdx.x; e < M; e += blockDim.x) s.twM[e] = a.twM[e];
  for (int e = threadIdx.x; e < a.L * a.Ns * M; e += blockDim.x) s.cp[e] = a.cph[e];
  __syncthreads();
  return s;
}

#define CW_THREADS 512

// A: data lines of every shot and coil of one image column; warp = (shot, CPW coils of the stage)
template <int M, bool PHASE>
__global__ void __launch_bounds__(256) k_colw_fwd(ColArgs a, int cg) {
  constexpr int ELEMS = 256, CPW = cw_cpw(M, ELEMS);
  constexpr int RL = cw_last<M>(), NL = M / RL, ROUNDS = (CPW * NL + 31) / 32;
  extern __shared__ __align__(16) float2 sm[];
  __shared__ __align__(8) uint64_t bar[2];
  const int L = a.L, Ns = a.Ns, N = a.N, B = L * Ns, x = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const size_t NN = (size_t)N * N, d = blockIdx.y;
  const CwShared s = cw_begin<M, ELEMS>(a, CW_FWD, sm, cg, bar);
  const int nst = (a.Nc + cg - 1) / cg;
  if (threadIdx.x == 0) cw_issue(a, s, bar, nullptr, 0, x);
  const int Bin = PHASE ? L : B, stride = PHASE ? Ns * N : N;
  cw_lines_in(a, s, a.in + d * Bin * NN, Bin, stride, x);
  float2* R = fft_smem_call<true>(s.img, s.tmp, Bin, stride, a.fN, s.twN);
  if (PHASE) {
    const float2* ph = a.phaseT + d * B * NN + (size_t)x * N;
    for (int e = threadIdx.x; e < L * N; e += blockDim.x) {
      const int l = e / N, y = e - l * N;
      const float2 v = cscale(R[l * stride + y], a.sN * sgn_par(y));
      for (int i = Ns - 1; i >= 0; --i)
        s.img[(l * Ns + i) * N + y] = cmul(cmul(v, ph[(size_t)(l * Ns + i) * NN + y]), __ldg(s.ts + i * N + y));
    }
  } else {
    for (int e = threadIdx.x; e < B * N; e += blockDim.x) {
      const int b = e / N, y = e - b * N;
      s.img[e] = cmul(cscale(R[e], a.sN * sgn_par(y)), __ldg(s.ts + (b % Ns) * N + y));
    }
  }
  fence_async_smem();  // stage 1 takes the place of the lines' second buffer
  __syncthreads();
  if (threadIdx.x == 0 && nst > 1) cw_issue(a, s, bar, nullptr, 1, x);
  float2* out = a.out + d * (size_t)Ns * a.Nc * N * M;
  const int i = warp % Ns, k0 = warp / Ns * CPW;
  for (int t = 0; t < nst; ++t) {
    if (!cw_arrive(a, s, bar, nullptr, t, nst, x)) return;
    const int c0 = t * cg, n = min(cg, a.Nc - c0);
    if (k0 >= n) continue;  // (a whole warp; the barrier is met at the top)
    float2 Y[ROUNDS][RL];
#pragma unroll
    for (int rd = 0; rd < ROUNDS; ++rd)
#pragma unroll
      for (int r = 0; r < RL; ++r) Y[rd][r] = cmk(0.f, 0.f);
    for (int l = 0; l < L; ++l) {
      const float2* cp = s.cp + (l * Ns + i) * M;
      cw_fold_fft<M, CPW>(a, s, s.stage[t & 1], s.img + (l * Ns + i) * N, l, k0, n, lane,
                          [&](int rd, int cs, int j, const float2* v) {
#pragma unroll
                            for (int r = 0; r < RL; ++r) cfma(Y[rd][r], cp[j + r * NL], v[r]);
                          });
    }
#pragma unroll
    for (int rd = 0; rd < ROUNDS; ++rd) {
      const int q = lane + 32 * rd, cs = q / NL, j = q - cs * NL;
      if (q < CPW * NL && k0 + cs < n) {
        float2* o = out + ((size_t)(i * a.Nc + c0 + k0 + cs) * N + x) * M + j;
#pragma unroll
        for (int r = 0; r < RL; ++r) o[r * NL] = Y[rd][r];
      }
    }
  }
}

// A^H: slice-shot lines of one image column (summed over the shots with the conjugate phase); warp = (slice, shot)
template <int M, int NSM, bool PHASE>
__global__ void __launch_bounds__(NSM <= 4 ? 384 : CW_THREADS, NSM <= 4 ? 2 : 1) k_colw_adj(ColArgs a, int cg) {
  constexpr int ELEMS = NSM > 2 ? 128 : 256, CPW = cw_cpw(M, ELEMS);
  constexpr int RL = cw_last<M>(), ROUNDS = (CPW * (M / RL) + 31) / 32;
  extern __shared__ __align__(16) float2 sm[];
  __shared__ __align__(8) uint64_t bar[2];
  const int L = a.L, Ns = a.Ns, N = a.N, B = L * Ns, x = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const size_t NN = (size_t)N * N, d = blockIdx.y;
  const CwShared s = cw_begin<M, ELEMS>(a, CW_ADJ, sm, cg, bar);
  const float2* in = a.in + d * (size_t)Ns * a.Nc * N * M;
  const int nst = (a.Nc + cg - 1) / cg;
  if (threadIdx.x == 0) {
    cw_issue(a, s, bar, in, 0, x);
    if (nst > 1) cw_issue(a, s, bar, in, 1, x);
  }
  const int l = warp / Ns, i = warp - l * Ns;
  const bool mine = warp < B;
  float2 acc[NSM][ROUNDS][RL];
#pragma unroll
  for (int t = 0; t < NSM; ++t)
#pragma unroll
    for (int rd = 0; rd < ROUNDS; ++rd)
#pragma unroll
      for (int r = 0; r < RL; ++r) acc[t][rd][r] = cmk(0.f, 0.f);
  for (int t = 0; t < nst; ++t) {
    if (!cw_arrive(a, s, bar, in, t, nst, x)) return;
    const int n = min(cg, a.Nc - t * cg);
    const float2* dy = s.stage[t & 1] + L * cg * s.lds + i * cg * s.ldd;
    if (mine)
      for (int k0 = 0; k0 < n; k0 += CPW)
        cw_adjoint<M, CPW, NSM>(a, s, s.stage[t & 1], l, i, k0, n, lane, acc,
                                [&](int c, int m) { return dy[c * s.ldd + m]; });
  }
  if (mine) cw_collect<M, CPW, NSM>(a, s, l, i, lane, acc, s.img, false);
  __syncthreads();
  int Bout = B, ostride = N;
  if (PHASE) {
    const float2* ph = a.phaseT + d * B * NN + (size_t)x * N;
    for (int e = threadIdx.x; e < L * N; e += blockDim.x) {
      const int ls = e / N, y = e - ls * N;
      float2 v = cmk(0.f, 0.f);
      for (int k = 0; k < Ns; ++k) cfmacj(v, ph[(size_t)(ls * Ns + k) * NN + y], s.img[(ls * Ns + k) * N + y]);
      s.img[ls * Ns * N + y] = v;
    }
    Bout = L;
    ostride = Ns * N;
    __syncthreads();
  }
  for (int e = threadIdx.x; e < Bout * N; e += blockDim.x) {
    const int b = e / N, y = e - b * N;
    s.img[b * ostride + y] = cscale(s.img[b * ostride + y], sgn_par(y));
  }
  __syncthreads();
  const float2* R = fft_smem_call<false>(s.img, s.tmp, Bout, ostride, a.fN, s.twN);
  float2* out = a.out + d * Bout * NN;
  for (int e = threadIdx.x; e < Bout * N; e += blockDim.x) {
    const int b = e / N, ky = e - b * N;
    out[(size_t)b * NN + (size_t)x * N + ky] = cscale(R[b * ostride + ky], a.sN * sgn_par(ky));
  }
}

typedef void (*CwFn)(ColArgs, int);
typedef size_t (*CwPlan)(int, int, int, int, int, int, CwShared*, float2*, int);
struct CwEntry {
  int M, nsm;  // nsm 0: any number of shots
  CwFn plain, phase;
  CwPlan plan;  // shared-memory bytes
  int cpw;
};
#define CW_F(M) {M, 0, k_colw_fwd<M, false>, k_colw_fwd<M, true>, cw_plan<M, 256>, cw_cpw(M, 256)}
#define CW_E(NS) (NS > 2 ? 128 : 256)
#define CW_A(M, NS) \
  {M, NS, k_colw_adj<M, NS, false>, k_colw_adj<M, NS, true>, cw_plan<M, CW_E(NS)>, cw_cpw(M, CW_E(NS))}
static const CwEntry kFwd[] = {CW_F(8),  CW_F(12), CW_F(16), CW_F(18),  CW_F(24),  CW_F(32),  CW_F(36), CW_F(48),
                               CW_F(54), CW_F(64), CW_F(72), CW_F(96), CW_F(108), CW_F(128), CW_F(144), CW_F(192),
                               CW_F(256)};
static const CwEntry kAdj[] = {
    CW_A(8, 4),   CW_A(8, 8),   CW_A(12, 4),  CW_A(12, 8), CW_A(16, 4),  CW_A(16, 8),  CW_A(18, 4),  CW_A(18, 8),
    CW_A(24, 2),  CW_A(24, 4),  CW_A(24, 8),  CW_A(32, 2), CW_A(32, 4),  CW_A(32, 8),  CW_A(36, 2),  CW_A(36, 4),
    CW_A(36, 8),  CW_A(48, 2),  CW_A(48, 4),  CW_A(54, 2), CW_A(54, 4),  CW_A(64, 2),  CW_A(64, 4),  CW_A(72, 2),
    CW_A(72, 4),  CW_A(96, 2),  CW_A(96, 4),  CW_A(108, 2), CW_A(128, 2), CW_A(128, 4), CW_A(144, 2), CW_A(192, 2),
    CW_A(256, 2)};
template <int K>
static const CwEntry* cw_find(const CwEntry (&t)[K], int M, int Ns) {
  for (const CwEntry& e : t)  // the table lists the shot limits of a length in ascending order
    if (e.M == M && (e.nsm == 0 || e.nsm >= Ns)) return &e;
  return nullptr;
}

smsm_status colwarp_init_attrs() {
  cudaError_t err = cudaSuccess;
  auto set = [&](CwFn f) {
    if (f && err == cudaSuccess) err = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  };
  for (const CwEntry& e : kFwd) set(e.plain), set(e.phase);
  for (const CwEntry& e : kAdj) set(e.plain), set(e.phase);
  if (err != cudaSuccess) {
    smsm_set_error("cudaFuncSetAttribute (column stage): %s", cudaGetErrorString(err));
    return SMSM_ERR_CUDA;
  }
  return SMSM_OK;
}

// SMSM_ERR_ARG: no kernel for this geometry (the caller takes the generic one)
smsm_status launch_col_warp(const smsm_plan_s* P, int mode, int with_phase, const ColArgs& a, cudaStream_t s) {
  const int B = P->L * P->Ns;
  const CwEntry* e = mode == COL_FWD ? cw_find(kFwd, P->M, P->Ns)
                     : mode == COL_ADJ ? cw_find(kAdj, P->M, P->Ns)
                                       : nullptr;
  if (!e) return SMSM_ERR_ARG;
  if (mode != COL_FWD && B > (e->nsm <= 4 ? 12 : CW_THREADS / 32)) return SMSM_ERR_ARG;  // the kernels' launch bounds
  int nw = B, cg = e->cpw;
  if (mode == COL_FWD) {
    // coil sets per stage: at least four warps, no more sets than coils
    int g = (4 + P->Ns - 1) / P->Ns;
    const int most = (P->Nc + e->cpw - 1) / e->cpw;
    if (g > most) g = most;
    nw = g * P->Ns;
    cg = g * e->cpw;
  }
  if (mode == COL_ADJ && e->nsm > 2) cg = 2 * e->cpw;
  if (cg > P->Nc) cg = P->Nc;  // (staged coils; a set's further lanes repeat the last one)
  if (mode == COL_ADJ && nw < 4) nw = 4;  // idle in the coil loop, busy in the transforms of the lines
  const size_t sm = e->plan(mode == COL_FWD ? CW_FWD : CW_ADJ, P->L, P->Ns, P->N, nw, cg,
                            nullptr, nullptr, 0);
  if (sm > 200 * 1024) return SMSM_ERR_ARG;
  (with_phase ? e->phase : e->plain)<<<dim3(P->N, P->D), 32 * nw, sm, s>>>(a, cg);
  SMSM_LAUNCH_CHECK("k_colw");
  return SMSM_OK;
}
