// Learned warm start: a small complex CNN trained on the GPU by these kernels.
//
// The paper has no learned component.  This network seeds the IRLS solve of
// Eq. 10: from the aliased, zero-filled image of every (slice, shot),
// a = F^-1(A^H y), it predicts a starting image x0 = a + f(a), whose k-space
// F x0 is the solve's first iterate and so also its first Gram and annihilating
// filters (Eq. 9).  f is six complex 3x3 convolutions (B -> width -> ... -> B,
// B = L*Ns) with CReLU (ReLU on the real and on the imaginary part) between them.
//
// Arithmetic: weights are held as FP32 master copies and used rounded to BF16
// (every product takes a BF16 weight); activations, products and accumulation
// are FP32.  Convolution (cross-correlation, zero padding):
//     z[o, p] = b[o] + sum_c sum_k W[o, c, k] h[c, p + k - 1].
// Gradients of the real loss are carried as G = dL/dRe + i dL/dIm:
//     dW[o, c, k] = sum_p G[o, p] conj(h[c, p + k - 1]),  db[o] = sum_p G[o, p],
//     dh[c, q]   = sum_o sum_k conj(W[o, c, k]) G[o, q - k + 1]
// -- the last is again a convolution of G, with the weights conjugated,
// transposed and their 3x3 taps reversed, so one kernel serves both.
// Loss of one sample: ||x0 - t||^2 / ||t||^2; a batch averages its samples.
// Optimiser: Adam on the master weights.  Every reduction (loss, weight
// gradients over the pixels) runs in a fixed order, so training is
// bit-reproducible.
#include <cuda_bf16.h>
#include <math.h>
#include <string.h>

#include <vector>

#include "common.cuh"
#include "umma.cuh"

#define WG_OCB 32   // weight gradient: output channels per CTA
#define WG_ICB 32   // weight gradient: input channels per CTA
#define WG_TY 8     // weight gradient pixel tile: 8 rows x 16 columns
#define WG_TX 16
#define WG_CP 181   // staged channel pitch (float2) of the weight-gradient input tile
#define WG_SPLIT 64 // pixel splits of the weight gradient (partials reduced in a fixed order)

struct smsm_cnn_s {
  int B, width, layers, H, W, maxn;
  int dev;
  std::vector<int> cin, cout;      // per layer
  std::vector<size_t> woff, boff;  // complex offsets of W_k and b_k in the parameter vector
  size_t count;                    // complex parameters
  float2 *master, *wbf, *grad, *m1, *m2;  // [count]
  float2* wt;                      // transposed-conjugated-reversed weights, largest layer
  std::vector<float2*> z;          // pre-activations per layer [maxn][cout][H][W]
  float2 *gA, *gB;                 // gradient ping-pong [maxn][width][H][W]
  float2* wpart;                   // weight-gradient partials [WG_SPLIT][max Cout*Cin*9 + Cout]
  __nv_bfloat16* wB;               // weights of one layer in the convolution's order
  int* devflag;                    // raised when a bounded wait of a convolution ran out
  double* lpart;                   // per-sample [2] sums (||x0 - t||^2, ||t||^2)
  int step;                        // Adam step
  size_t bytes;
};

__device__ __forceinline__ float2 crelu2(float2 v) { return cmk(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f)); }

__device__ __forceinline__ float bf16r(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

// ---------------------------------------------------------------------------
// Convolution: out[n][o] = bias[o] + sum_c sum_k Wp[o][c][k] g(in[n][c])(p + k - 1)
//   g = CReLU when in_relu, identity otherwise; then + resid[n][o] when given, and
//   each component zeroed where that component of mask[n][o] is not > 0 when given.
// On the tensor cores (tcgen05, BF16 operands, FP32 accumulation in TMEM).  The weights are BF16 values; an
// FP32 activation is split exactly into three BF16 pieces, so every product is exact and what is rounded is the
// accumulation, as in an FP32 FMA loop.  Every MMA rounds its accumulator once, so the leading piece's products
// are dealt out to three accumulators by tap row (24 roundings each for 64 channels) and the two small
// pieces' (2^-8 and 2^-16 of them) to a fourth, all added in the epilogue: with one accumulator for the
// leading products the learned start of two 256 x 256 groups was 2.9e-6 from its 64-bit value, with three 7.8e-7 ..
// 9.3e-7 over seeds and sizes at 64 channels, 2.9e-7 .. 4e-7 at 16 to 40 (FP32 FMAs: 7.5e-7 .. 1.06e-6 and 3.3e-7 ..
// 6.5e-7).  An infinite weight (a diverged network) gives NaN: its products with the small pieces have both signs.
//
// Implicit GEMM without copies: the image is cut into column strips of TW pixels, padded to P = TW + 2 columns, and
// a strip is read as one line of pixels; a CTA takes 128 consecutive ones and stages them with
// P + 1 more on both sides.  A staged K slab is 8 BF16 values (re and im of four channels) of every pixel, pixel
// after pixel, 16 bytes each: the no-swizzle K-major layout with its 8-row groups back to back.  A tap (ky, kx)
// is the same slab from ky P + kx pixels further on, so the nine taps are nine start addresses of
// the A descriptor.  Pixels in the padding columns give values nobody stores.
//   * eight producer warps load the next 8 channels, apply CReLU, split and stage them (two stages);
//   * one thread brings the 8 channels' weights of all taps (k_cnn_wprep's order: one bulk copy);
//   * one thread issues 9 taps x 3 pieces of 128 x NT x 16 MMAs;
//   * the producer warps write the outputs from TMEM at the end.
// N = NT columns: the real parts of up to 64 output channels, then the imaginary ones.  Waits are bounded; on a
// timeout the network's error flag is raised.
// Measured (before: FP32 FMAs, a 16 x 16 pixel tile x 32 channels per CTA), two 256 x 256 images: 12 -> 64 channels
// 160 -> 60 us, 64 -> 64 770 -> 120 us, 64 -> 12 438 -> 139 us; the learned start of both groups (6 layers, width 64)
// 3.73 -> 0.74 ms.
// ---------------------------------------------------------------------------
#define CV_TL 128                 // pixels of a strip per CTA (one M = 128 block)
#define CV_MAXP 66                // strip pitch at most
#define CV_SR (CV_TL + 2 * CV_MAXP + 2)  // staged pixels at most
#define CV_PROD 256
#define CV_THREADS (CV_PROD + 64)
#define CV_MAXITER (1L << 22)

struct ConvShape {
  int Cin, Cout, H, W, in_relu;
  int TW, P, nstrip, ntl;  // strip width and pitch, strips per image, CTAs per strip
  int NT, nchunk;          // MMA columns, chunks of 8 input channels
};

// weights in the order the MMAs take them: [block of 64 outputs][chunk][tap][slab][NT][8] BF16; column n of a block
// is Re (n < NT/2) or Im of output n mod NT/2; slab values are (re, im) of four channels
__global__ void __launch_bounds__(256) k_cnn_wprep(const float2* __restrict__ Wp, __nv_bfloat16* __restrict__ dst,
                                                   ConvShape g, int nblk) {
  const int half = g.NT / 2, total = nblk * g.nchunk * 9 * 2 * g.NT;
  for (int e = blockIdx.x * 256 + threadIdx.x; e < total; e += gridDim.x * 256) {
    int t = e;
    const int n = t % g.NT;
    t /= g.NT;
    const int slab = t & 1;
    t >>= 1;
    const int tap = t % 9;
    t /= 9;
    const int ch = t % g.nchunk, nb = t / g.nchunk;
    const int o = nb * 64 + n % half, im = n / half;
    __align__(16) __nv_bfloat16 v[8];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = ch * 8 + slab * 4 + q;
      float2 w = cmk(0.f, 0.f);
      if (o < g.Cout && n % half < 64 && c < g.Cin) w = Wp[((size_t)o * g.Cin + c) * 9 + tap];
      v[2 * q] = __float2bfloat16_rn(im ? w.y : w.x);
      v[2 * q + 1] = __float2bfloat16_rn(im ? w.x : -w.y);
    }
    reinterpret_cast<uint4*>(dst)[e] = *reinterpret_cast<const uint4*>(v);
  }
}

__device__ __forceinline__ bool cv_wait(uint64_t* mbar, uint32_t parity, volatile int* abort_flag) {
  for (long it = 0; it < CV_MAXITER; ++it) {
    if (mbar_wait(mbar, parity, 1)) return true;
    if ((it & 255) == 255 && *abort_flag) return false;
  }
  *abort_flag = 1;
  return false;
}

// Two floats in BF16 (lo in the low half).  The first two pieces saturate: a finite value above the largest BF16 one
// leaves a remainder that the other pieces hold, and an infinite one goes to the third piece, where inf - inf would
// make a remainder a NaN.
__device__ __forceinline__ uint32_t cv_pack_sat(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}
__device__ __forceinline__ uint32_t cv_pack(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}

__host__ __device__ inline uint32_t cv_a_bytes(const ConvShape& g) {  // one piece of one stage
  return 2u * (uint32_t)(CV_TL + 2 * g.P + 2) * 16u;
}
__host__ __device__ inline uint32_t cv_b_bytes(const ConvShape& g) { return 9u * 2u * (uint32_t)g.NT * 16u; }

__global__ void __launch_bounds__(CV_THREADS, 1)
    k_cnn_conv(const float2* __restrict__ in, const __nv_bfloat16* __restrict__ wB, const float2* __restrict__ bias,
               const float2* __restrict__ resid, const float2* __restrict__ mask, float2* __restrict__ out,
               ConvShape g, int* __restrict__ errflag) {
  extern __shared__ __align__(128) unsigned char csm[];  // [2 stages][3 pieces of A, B]
  __shared__ uint32_t tmem_base;
  __shared__ __align__(8) uint64_t afull[2], bfull[2], empty[2], fin;
  __shared__ volatile int s_abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int strip = blockIdx.x / g.ntl, t0 = (blockIdx.x - strip * g.ntl) * CV_TL;
  const int nb = blockIdx.y, n = blockIdx.z;
  const int SR = CV_TL + 2 * g.P + 2;
  const uint32_t ab = cv_a_bytes(g), bb = cv_b_bytes(g), stage = 3 * ab + bb;
  const size_t HW = (size_t)g.H * g.W;
  int cols = 32;
  while (cols < 4 * g.NT) cols <<= 1;
  if (warp == 0) tmem_alloc(&tmem_base, cols);
  if (tid == 0) {
    for (int k = 0; k < 2; ++k) {
      mbar_init(&afull[k], CV_PROD);
      mbar_init(&bfull[k], 1);
      mbar_init(&empty[k], 1);
    }
    mbar_init(&fin, 1);
    asm volatile("fence.mbarrier_init.release.cluster;");
    s_abort = 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;

  if (tid < CV_PROD) {
    // ---------------- producers ----------------
    constexpr int NI = (2 * CV_SR + CV_PROD - 1) / CV_PROD;
    int off[NI];       // pixel of the image, or -1 (zero)
    uint32_t dst[NI];  // byte in a piece
    int slab[NI];
#pragma unroll
    for (int k = 0; k < NI; ++k) {
      const int e = tid + CV_PROD * k;
      slab[k] = e >= SR;
      const int m = e - slab[k] * SR;  // staged pixel
      off[k] = -1;
      dst[k] = 0xffffffffu;
      if (e < 2 * SR) {
        dst[k] = (uint32_t)(slab[k] * SR + m) * 16u;
        const int q = t0 + m - g.P - 1 + 2 * g.P;  // two rows up: never negative
        const int y = q / g.P - 2, xq = q - (y + 2) * g.P, x = strip * g.TW + xq - 1;
        if (y >= 0 && y < g.H && x >= 0 && x < g.W) off[k] = y * g.W + x;
      }
    }
    const float2* inn = in + (size_t)n * g.Cin * HW;
    for (int it = 0; it < g.nchunk; ++it) {
      const int s = it & 1;
      float2 v[NI][4];
#pragma unroll
      for (int k = 0; k < NI; ++k)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int c = it * 8 + slab[k] * 4 + q;
          v[k][q] = cmk(0.f, 0.f);
          if (off[k] >= 0 && c < g.Cin) v[k][q] = __ldg(inn + (size_t)c * HW + off[k]);
        }
      if (it >= 2 && !cv_wait(&empty[s], (uint32_t)((it / 2 - 1) & 1), &s_abort)) break;
      unsigned char* st = csm + s * stage;
#pragma unroll
      for (int k = 0; k < NI; ++k) {
        if (dst[k] == 0xffffffffu) continue;
        float f[8];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 u = g.in_relu ? crelu2(v[k][q]) : v[k][q];
          f[2 * q] = u.x;
          f[2 * q + 1] = u.y;
        }
#pragma unroll
        for (int piece = 0; piece < 3; ++piece) {
          uint32_t h[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            h[q] = piece < 2 ? cv_pack_sat(f[2 * q], f[2 * q + 1]) : cv_pack(f[2 * q], f[2 * q + 1]);
            f[2 * q] -= __uint_as_float(h[q] << 16);  // exact: the remainder of a round-to-nearest
            f[2 * q + 1] -= __uint_as_float(h[q] & 0xffff0000u);
          }
          *reinterpret_cast<uint4*>(st + piece * ab + dst[k]) = make_uint4(h[0], h[1], h[2], h[3]);
        }
      }
      fence_async_smem();
      mbar_arrive(&afull[s]);
    }
    // ---------------- epilogue: warp w takes TMEM lanes 32 (w mod 4) .. and every second 16 channels ----------------
    if (__all_sync(0xffffffffu, cv_wait(&fin, 0, &s_abort)) && !s_abort) {
      tc_fence_after();
      const int half = g.NT / 2;
      const int q = t0 + 32 * (warp & 3) + lane;
      const int y = q / g.P, xq = q - y * g.P, x = strip * g.TW + xq - 1;
      const bool live = y < g.H && xq >= 1 && xq <= g.TW && x < g.W;
      const uint32_t base = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
      const size_t pix = (size_t)y * g.W + x;
      for (int o0 = 16 * (warp >> 2); o0 < half; o0 += 32) {
        float re[16], im[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) re[k] = im[k] = 0.f;
#pragma unroll
        for (int acc = 3; acc >= 0; --acc) {  // the small products first
          __syncwarp();  // the TMEM loads are .sync.aligned
          uint32_t d[16];
          tmem_ld16(base + acc * g.NT + o0, d);
#pragma unroll
          for (int k = 0; k < 16; ++k) re[k] += __uint_as_float(d[k]);
          tmem_ld16(base + acc * g.NT + half + o0, d);
#pragma unroll
          for (int k = 0; k < 16; ++k) im[k] += __uint_as_float(d[k]);
        }
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const int oc = nb * 64 + o0 + k;
          if (live && oc < g.Cout) {
            float2 w = cmk(re[k], im[k]);
            if (bias) w = cadd(w, bias[oc]);
            const size_t o = ((size_t)n * g.Cout + oc) * HW + pix;
            if (resid) w = cadd(w, resid[o]);
            if (mask) {
              const float2 mk = mask[o];
              w = cmk(mk.x > 0.f ? w.x : 0.f, mk.y > 0.f ? w.y : 0.f);
            }
            out[o] = w;
          }
        }
      }
      tc_fence_before();
    }
  } else if (tid == CV_PROD) {
    // ---------------- MMA issue ----------------
    const uint32_t idesc = umma_idesc(1u, 128, g.NT), lboA = (uint32_t)SR * 16u, lboB = (uint32_t)g.NT * 16u;
    for (int it = 0; it < g.nchunk; ++it) {
      const int s = it & 1;
      const uint32_t ph = (uint32_t)((it / 2) & 1);
      if (!cv_wait(&afull[s], ph, &s_abort) || !cv_wait(&bfull[s], ph, &s_abort)) break;
      tc_fence_after();
      const uint32_t a0 = smem_u32(csm + s * stage), b0 = a0 + 3 * ab;
      for (int tap = 0; tap < 9; ++tap) {
        const uint64_t bd = umma_desc(b0 + (uint32_t)tap * 2 * lboB, lboB, 128);
        const uint32_t shift = (uint32_t)((tap / 3) * g.P + tap % 3) * 16u;  // staged pixel 0 is P + 1 before the first
        const uint32_t ar = a0 + shift;
        umma_bf16(tmem + (tap / 3) * g.NT, umma_desc(ar, lboA, 128), bd, idesc, (it || tap % 3) ? 1u : 0u);
        umma_bf16(tmem + 3 * g.NT, umma_desc(ar + ab, lboA, 128), bd, idesc, (it || tap) ? 1u : 0u);
        umma_bf16(tmem + 3 * g.NT, umma_desc(ar + 2 * ab, lboA, 128), bd, idesc, 1u);
      }
      umma_commit(&empty[s]);
    }
    umma_commit(&fin);  // every MMA issued above has finished before TMEM and the stages are released
    mbar_wait(&fin, 0, CV_MAXITER);
  } else if (tid == CV_PROD + 32) {
    // ---------------- weights ----------------
    const unsigned char* src = reinterpret_cast<const unsigned char*>(wB) + (size_t)nb * g.nchunk * bb;
    int sent = 0;
    for (int it = 0; it < g.nchunk; ++it, ++sent) {
      const int s = it & 1;
      if (it >= 2 && !cv_wait(&empty[s], (uint32_t)((it / 2 - 1) & 1), &s_abort)) break;
      mbar_arrive_expect_tx(&bfull[s], bb);
      tma_bulk_g2s(csm + s * stage + 3 * ab, src + (size_t)it * bb, bb, &bfull[s]);
    }
    // copies still in flight land before the shared memory is released
    for (int it = sent > 2 ? sent - 2 : 0; it < sent; ++it) mbar_wait(&bfull[it & 1], (uint32_t)((it / 2) & 1), CV_MAXITER);
  }
  __syncthreads();
  if (s_abort && tid == 0) atomicExch(errflag, SMSM_ERR_TIMEOUT);
  if (warp == 0) tmem_dealloc(tmem, cols);
}

// ---------------------------------------------------------------------------
// Weight gradient: part[s][o][c][k] = sum over split s's pixels of G[n][o][p] conj(h[n][c][p+k-1]),
// part[s][Cout*Cin*9 + o] = sum G[n][o][p] (bias), h = CReLU(in) when in_relu.
// CTA = (32 output channels, 32 input channels, split s); thread = 4 output channels x
// 1 input channel x 9 taps.  Pixel tiles (8 x 16) of all samples are dealt to the splits
// in order; a thread slides a 3 x 3 window of h along each tile row.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_cnn_wgrad(const float2* __restrict__ G, const float2* __restrict__ in,
                                                   float2* __restrict__ part, int n, int Cin, int Cout, int H, int W,
                                                   int in_relu) {
  extern __shared__ __align__(16) float2 wsm[];
  float2* sG = wsm;                                 // [WG_OCB][WG_TY][WG_TX]
  float2* sH = wsm + WG_OCB * WG_TY * WG_TX;        // [WG_ICB][WG_CP] (10 x 18 used)
  const int o0 = blockIdx.x * WG_OCB, c0 = blockIdx.y * WG_ICB, sp = blockIdx.z;
  const int tid = threadIdx.x, og = tid >> 5, cl = tid & 31;
  const int tilesx = (W + WG_TX - 1) / WG_TX, tilesy = (H + WG_TY - 1) / WG_TY;
  const long ntile = (long)n * tilesx * tilesy;
  const long t0 = ntile * sp / WG_SPLIT, t1 = ntile * (sp + 1) / WG_SPLIT;
  const size_t HW = (size_t)H * W;
  float2 acc[4][9];
  float2 bacc[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    bacc[a] = cmk(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 9; ++k) acc[a][k] = cmk(0.f, 0.f);
  }
  for (long t = t0; t < t1; ++t) {
    const int s = (int)(t / (tilesx * tilesy)), r = (int)(t - (long)s * tilesx * tilesy);
    const int ty0 = (r / tilesx) * WG_TY, tx0 = (r % tilesx) * WG_TX;
    for (int e = tid; e < WG_OCB * WG_TY * WG_TX; e += 256) {
      const int o = e / (WG_TY * WG_TX), rem = e - o * WG_TY * WG_TX;
      const int yy = rem / WG_TX, xx = rem - yy * WG_TX;
      const int gy = ty0 + yy, gx = tx0 + xx;
      float2 v = cmk(0.f, 0.f);
      if (o0 + o < Cout && gy < H && gx < W) v = G[((size_t)s * Cout + o0 + o) * HW + (size_t)gy * W + gx];
      sG[e] = v;
    }
    for (int e = tid; e < WG_ICB * (WG_TY + 2) * (WG_TX + 2); e += 256) {
      const int c = e / ((WG_TY + 2) * (WG_TX + 2)), rem = e - c * (WG_TY + 2) * (WG_TX + 2);
      const int yy = rem / (WG_TX + 2), xx = rem - yy * (WG_TX + 2);
      const int gy = ty0 + yy - 1, gx = tx0 + xx - 1;
      float2 v = cmk(0.f, 0.f);
      if (c0 + c < Cin && gy >= 0 && gy < H && gx >= 0 && gx < W) {
        v = in[((size_t)s * Cin + c0 + c) * HW + (size_t)gy * W + gx];
        if (in_relu) v = crelu2(v);
      }
      sH[c * WG_CP + yy * (WG_TX + 2) + xx] = v;
    }
    __syncthreads();
    const float2* hc = sH + cl * WG_CP;
    for (int yy = 0; yy < WG_TY; ++yy) {
      float2 win[3][3];  // h at rows yy..yy+2, columns xx..xx+2 of the staged tile
#pragma unroll
      for (int ky = 0; ky < 3; ++ky) {
        win[ky][1] = hc[(yy + ky) * (WG_TX + 2) + 0];
        win[ky][2] = hc[(yy + ky) * (WG_TX + 2) + 1];
      }
#pragma unroll 4
      for (int xx = 0; xx < WG_TX; ++xx) {
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) {
          win[ky][0] = win[ky][1];
          win[ky][1] = win[ky][2];
          win[ky][2] = hc[(yy + ky) * (WG_TX + 2) + xx + 2];
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const float2 g = sG[((og * 4 + a) * WG_TY + yy) * WG_TX + xx];
          bacc[a] = cadd(bacc[a], g);
#pragma unroll
          for (int ky = 0; ky < 3; ++ky)
#pragma unroll
            for (int kx = 0; kx < 3; ++kx) cfmacj(acc[a][ky * 3 + kx], win[ky][kx], g);
        }
      }
    }
    __syncthreads();
  }
  const size_t stride = (size_t)Cout * Cin * 9 + Cout;
  float2* ps = part + (size_t)sp * stride;
  const int c = c0 + cl;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int o = o0 + og * 4 + a;
    if (o >= Cout) continue;
    if (c < Cin)
#pragma unroll
      for (int k = 0; k < 9; ++k) ps[((size_t)o * Cin + c) * 9 + k] = acc[a][k];
    if (blockIdx.y == 0 && cl == 0) ps[(size_t)Cout * Cin * 9 + o] = bacc[a];
  }
}

// grad[i] = scale * sum_s part[s][i] in a fixed order
__global__ void k_cnn_wgrad_reduce(const float2* __restrict__ part, float2* __restrict__ grad, size_t count,
                                   float scale) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x) {
    double re = 0.0, im = 0.0;
    for (int s = 0; s < WG_SPLIT; ++s) {
      const float2 v = part[(size_t)s * count + i];
      re += v.x;
      im += v.y;
    }
    grad[i] = cmk((float)(re * scale), (float)(im * scale));
  }
}

// wt[c][o][k] = conj(W[o][c][8 - k]): the convolution whose output is dh
__global__ void k_cnn_wt(const float2* __restrict__ Wk, float2* __restrict__ wt, int Cin, int Cout) {
  const int total = Cout * Cin * 9;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const int k = e % 9, o = (e / 9) % Cout, c = e / (9 * Cout);
    wt[e] = conjf2(Wk[((size_t)o * Cin + c) * 9 + (8 - k)]);
  }
}

// per-sample sums ||x0 - t||^2 and ||t||^2 (one CTA per sample, fixed order)
__global__ void __launch_bounds__(256) k_cnn_loss_sums(const float2* __restrict__ x0, const float2* __restrict__ t,
                                                       size_t per, double* __restrict__ sums) {
  __shared__ double r0[256], r1[256];
  const float2* a = x0 + (size_t)blockIdx.x * per;
  const float2* b = t + (size_t)blockIdx.x * per;
  double s0 = 0.0, s1 = 0.0;
  for (size_t e = threadIdx.x; e < per; e += 256) {
    const float2 u = a[e], v = b[e];
    const float dx = u.x - v.x, dy = u.y - v.y;
    s0 += (double)(dx * dx + dy * dy);
    s1 += (double)(v.x * v.x + v.y * v.y);
  }
  r0[threadIdx.x] = s0;
  r1[threadIdx.x] = s1;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      r0[threadIdx.x] += r0[threadIdx.x + o];
      r1[threadIdx.x] += r1[threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    sums[2 * blockIdx.x] = r0[0];
    sums[2 * blockIdx.x + 1] = r1[0];
  }
}

// G = 2 (x0 - t) / ||t||^2 of each sample (the gradient of its loss)
__global__ void k_cnn_loss_grad(const float2* __restrict__ x0, const float2* __restrict__ t, size_t per,
                                const double* __restrict__ sums, float2* __restrict__ G) {
  const size_t total = per * gridDim.y;
  const int n = blockIdx.y;
  const float sc = (float)(2.0 / sums[2 * n + 1]);
  (void)total;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < per; e += (size_t)gridDim.x * blockDim.x) {
    const size_t i = (size_t)n * per + e;
    const float2 u = x0[i], v = t[i];
    G[i] = cmk(sc * (u.x - v.x), sc * (u.y - v.y));
  }
}

// Adam on the FP32 master weights; the BF16-rounded copy is what the convolutions use
__global__ void k_cnn_adam(float2* __restrict__ master, float2* __restrict__ wbf, const float2* __restrict__ grad,
                           float2* __restrict__ m1, float2* __restrict__ m2, size_t count, float lr, float c1,
                           float c2) {
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x) {
    const float2 g = grad[i];
    float2 m = m1[i], v = m2[i], w = master[i];
    m = cmk(b1 * m.x + (1.f - b1) * g.x, b1 * m.y + (1.f - b1) * g.y);
    v = cmk(b2 * v.x + (1.f - b2) * g.x * g.x, b2 * v.y + (1.f - b2) * g.y * g.y);
    w.x -= lr * (m.x / c1) / (sqrtf(v.x / c2) + eps);
    w.y -= lr * (m.y / c1) / (sqrtf(v.y / c2) + eps);
    m1[i] = m;
    m2[i] = v;
    master[i] = w;
    wbf[i] = cmk(bf16r(w.x), bf16r(w.y));
  }
}

__global__ void k_cnn_round(const float2* __restrict__ master, float2* __restrict__ wbf, size_t count) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x) {
    const float2 w = master[i];
    wbf[i] = cmk(bf16r(w.x), bf16r(w.y));
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static size_t wgrad_smem() { return (size_t)(WG_OCB * WG_TY * WG_TX + WG_ICB * WG_CP) * sizeof(float2); }

static ConvShape conv_shape(int Cin, int Cout, int H, int W, int in_relu) {
  ConvShape g;
  g.Cin = Cin;
  g.Cout = Cout;
  g.H = H;
  g.W = W;
  g.in_relu = in_relu;
  g.nstrip = (W + CV_MAXP - 3) / (CV_MAXP - 2);  // strips of at most 64 columns, all alike
  g.TW = (W + g.nstrip - 1) / g.nstrip;
  g.P = g.TW + 2;
  g.ntl = (int)(((long)H * g.P + CV_TL - 1) / CV_TL);
  g.NT = 32 * (((Cout < 64 ? Cout : 64) + 15) / 16);
  g.nchunk = (Cin + 7) / 8;
  return g;
}

static size_t conv_weight_elems(int Cin, int Cout) {  // BF16 values of k_cnn_wprep's output
  const ConvShape g = conv_shape(Cin, Cout, 1, 1, 0);
  return (size_t)((Cout + 63) / 64) * g.nchunk * 9 * 2 * g.NT * 8;
}

static smsm_status conv(const smsm_cnn_s* c, const float2* in, const float2* Wp, const float2* bias,
                        const float2* resid, const float2* mask, float2* out, int n, int Cin, int Cout, int in_relu,
                        int* errflag, cudaStream_t s) {
  const ConvShape g = conv_shape(Cin, Cout, c->H, c->W, in_relu);
  const int nblk = (Cout + 63) / 64;
  k_cnn_wprep<<<(nblk * g.nchunk * 9 * 2 * g.NT + 255) / 256, 256, 0, s>>>(Wp, c->wB, g, nblk);
  SMSM_LAUNCH_CHECK("k_cnn_wprep");
  const size_t sm = 2 * ((size_t)3 * cv_a_bytes(g) + cv_b_bytes(g));
  k_cnn_conv<<<dim3(g.nstrip * g.ntl, nblk, n), CV_THREADS, sm, s>>>(in, c->wB, bias, resid, mask, out, g, errflag);
  SMSM_LAUNCH_CHECK("k_cnn_conv");
  return SMSM_OK;
}

static void cnn_free(smsm_cnn_s* c) {
  if (!c) return;
  void* ptrs[] = {c->master, c->wbf, c->grad, c->m1, c->m2, c->wt, c->gA, c->gB, c->wpart, c->lpart, c->wB, c->devflag};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  for (float2* p : c->z)
    if (p) cudaFree(p);
  delete c;
}

template <typename T>
static smsm_status calloc_dev(smsm_cnn_s* c, T** p, size_t count) {
  const size_t bytes = count * sizeof(T) > 0 ? count * sizeof(T) : 16;
  cudaError_t e = cudaMalloc((void**)p, bytes);
  if (e != cudaSuccess) {
    *p = nullptr;
    smsm_set_error("smsm_cnn_create: cudaMalloc of %zu bytes failed: %s", bytes, cudaGetErrorString(e));
    return SMSM_ERR_NOMEM;
  }
  c->bytes += bytes;
  e = cudaMemset(*p, 0, bytes);
  if (e != cudaSuccess) {
    smsm_set_error("smsm_cnn_create: %s", cudaGetErrorString(e));
    return SMSM_ERR_CUDA;
  }
  return SMSM_OK;
}

extern "C" smsm_status smsm_cnn_create(smsm_cnn_t* out, int channels, int width, int layers, int height, int wdt,
                                       int max_batch) {
  if (!out) {
    smsm_set_error("smsm_cnn_create: out is NULL");
    return SMSM_ERR_ARG;
  }
  *out = nullptr;
  if (channels < 1 || channels > 256 || width < 1 || width > 256 || layers < 1 || layers > 32 || height < 1 ||
      wdt < 1 || height > 4096 || wdt > 4096 || max_batch < 1 || max_batch > 4096) {
    smsm_set_error("smsm_cnn_create: need channels, width in [1, 256], layers in [1, 32], image sides in "
                   "[1, 4096], max_batch in [1, 4096]");
    return SMSM_ERR_ARG;
  }
  smsm_cnn_s* c = new smsm_cnn_s();
  c->B = channels;
  c->width = width;
  c->layers = layers;
  c->H = height;
  c->W = wdt;
  c->maxn = max_batch;
  cudaGetDevice(&c->dev);
  size_t off = 0, maxw = 0;
  for (int k = 0; k < layers; ++k) {
    const int ci = k == 0 ? channels : width, co = k + 1 == layers ? channels : width;
    c->cin.push_back(ci);
    c->cout.push_back(co);
    c->woff.push_back(off);
    off += (size_t)co * ci * 9;
    c->boff.push_back(off);
    off += co;
    maxw = maxw > (size_t)co * ci * 9 + co ? maxw : (size_t)co * ci * 9 + co;
  }
  c->count = off;
  const size_t HW = (size_t)height * wdt;
  const int wmax = width > channels ? width : channels;
  smsm_status st = SMSM_OK;
  if (!st) st = calloc_dev(c, &c->master, off);
  if (!st) st = calloc_dev(c, &c->wbf, off);
  if (!st) st = calloc_dev(c, &c->grad, off);
  if (!st) st = calloc_dev(c, &c->m1, off);
  if (!st) st = calloc_dev(c, &c->m2, off);
  if (!st) st = calloc_dev(c, &c->wt, maxw);
  c->z.assign(layers, nullptr);
  for (int k = 0; k < layers && !st; ++k) st = calloc_dev(c, &c->z[k], (size_t)max_batch * c->cout[k] * HW);
  if (!st) st = calloc_dev(c, &c->gA, (size_t)max_batch * wmax * HW);
  if (!st) st = calloc_dev(c, &c->gB, (size_t)max_batch * wmax * HW);
  if (!st) st = calloc_dev(c, &c->wpart, (size_t)WG_SPLIT * maxw);
  if (!st) st = calloc_dev(c, &c->lpart, (size_t)2 * max_batch);
  size_t wmaxB = 0;
  for (int k = 0; k < layers; ++k) {  // both ways: the data gradient's convolution has them exchanged
    const size_t f = conv_weight_elems(c->cin[k], c->cout[k]), r = conv_weight_elems(c->cout[k], c->cin[k]);
    wmaxB = wmaxB > f ? wmaxB : f;
    wmaxB = wmaxB > r ? wmaxB : r;
  }
  if (!st) st = calloc_dev(c, &c->wB, wmaxB);
  if (!st) st = calloc_dev(c, &c->devflag, (size_t)1);
  if (!st) {
    cudaError_t e = cudaFuncSetAttribute(k_cnn_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wgrad_smem());
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_cnn_conv, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               2 * (3 * 2 * CV_SR * 16 + 9 * 2 * 128 * 16));
    if (e != cudaSuccess) {
      smsm_set_error("smsm_cnn_create: %s", cudaGetErrorString(e));
      st = SMSM_ERR_CUDA;
    }
  }
  if (st) {
    cnn_free(c);
    return st;
  }
  *out = c;
  return SMSM_OK;
}

smsm_status cnn_shape(const smsm_cnn_s* c, int* B, int* H, int* W, int* maxn) {
  *B = c->B;
  *H = c->H;
  *W = c->W;
  *maxn = c->maxn;
  return SMSM_OK;
}

extern "C" smsm_status smsm_cnn_destroy(smsm_cnn_t cnn) {
  cnn_free(cnn);
  return SMSM_OK;
}

extern "C" size_t smsm_cnn_param_count(smsm_cnn_t cnn) { return cnn ? cnn->count : 0; }

static smsm_status check_cnn(smsm_cnn_t cnn, const char* fn, int n) {
  if (!cnn) {
    smsm_set_error("%s: cnn is NULL", fn);
    return SMSM_ERR_ARG;
  }
  if (n < 0 || n > cnn->maxn) {
    smsm_set_error("%s: batch %d outside [0, %d]", fn, n, cnn->maxn);
    return SMSM_ERR_ARG;
  }
  int dev = -1;
  cudaGetDevice(&dev);
  if (dev != cnn->dev) {
    smsm_set_error("%s: the network lives on device %d, the current device is %d", fn, cnn->dev, dev);
    return SMSM_ERR_ARG;
  }
  return SMSM_OK;
}

static bool al16(const void* p) { return p && ((uintptr_t)p & 15u) == 0; }

extern "C" smsm_status smsm_cnn_set_params(smsm_cnn_t cnn, const void* params, void* stream) {
  smsm_status st;
  if ((st = check_cnn(cnn, "smsm_cnn_set_params", 0))) return st;
  if (!al16(params)) {
    smsm_set_error("smsm_cnn_set_params: params must be a 16-byte aligned device pointer");
    return SMSM_ERR_ARG;
  }
  cudaStream_t s = (cudaStream_t)stream;
  SMSM_CUDA_TRY(cudaMemcpyAsync(cnn->master, params, cnn->count * sizeof(float2), cudaMemcpyDeviceToDevice, s));
  SMSM_CUDA_TRY(cudaMemsetAsync(cnn->m1, 0, cnn->count * sizeof(float2), s));
  SMSM_CUDA_TRY(cudaMemsetAsync(cnn->m2, 0, cnn->count * sizeof(float2), s));
  cnn->step = 0;
  k_cnn_round<<<256, 256, 0, s>>>(cnn->master, cnn->wbf, cnn->count);
  SMSM_LAUNCH_CHECK("k_cnn_round");
  return SMSM_OK;
}

extern "C" smsm_status smsm_cnn_get_params(smsm_cnn_t cnn, void* params, void* stream) {
  smsm_status st;
  if ((st = check_cnn(cnn, "smsm_cnn_get_params", 0))) return st;
  if (!al16(params)) {
    smsm_set_error("smsm_cnn_get_params: params must be a 16-byte aligned device pointer");
    return SMSM_ERR_ARG;
  }
  SMSM_CUDA_TRY(cudaMemcpyAsync(params, cnn->master, cnn->count * sizeof(float2), cudaMemcpyDeviceToDevice,
                                (cudaStream_t)stream));
  return SMSM_OK;
}

// forward through every layer, keeping the pre-activations in z; x0 = a + z_last
static smsm_status cnn_forward(smsm_cnn_s* c, const float2* a, float2* x0, int n, int* errflag, cudaStream_t s) {
  smsm_status st;
  const float2* h = a;
  for (int k = 0; k < c->layers; ++k) {
    const bool last = k + 1 == c->layers;
    float2* o = last ? x0 : c->z[k];
    if ((st = conv(c, h, c->wbf + c->woff[k], c->wbf + c->boff[k], last ? a : nullptr, nullptr, o, n, c->cin[k],
                   c->cout[k], k > 0, errflag, s)))
      return st;
    h = c->z[k];
  }
  return SMSM_OK;
}

// a wait that runs out raises errflag: the network's own, or the plan's in smsm_learned_start
smsm_status cnn_forward_checked(smsm_cnn_s* cnn, const void* a, void* x0, int n, int* errflag, cudaStream_t s) {
  smsm_status st;
  if ((st = check_cnn(cnn, "smsm_cnn_forward", n))) return st;
  if (!al16(a) || !al16(x0) || a == x0) {
    smsm_set_error("smsm_cnn_forward: a and x0 must be distinct 16-byte aligned device pointers");
    return SMSM_ERR_ARG;
  }
  if (n == 0) return SMSM_OK;
  return cnn_forward(cnn, (const float2*)a, (float2*)x0, n, errflag ? errflag : cnn->devflag, s);
}

extern "C" smsm_status smsm_cnn_forward(smsm_cnn_t cnn, const void* a, void* x0, int n, void* stream) {
  return cnn_forward_checked(cnn, a, x0, n, nullptr, (cudaStream_t)stream);
}

// the device error flag, cleared once it is reported; synchronises s
static smsm_status cnn_status(smsm_cnn_s* c, cudaStream_t s) {
  int flag = 0;
  SMSM_CUDA_TRY(cudaMemcpyAsync(&flag, c->devflag, sizeof(int), cudaMemcpyDeviceToHost, s));
  SMSM_CUDA_TRY(cudaStreamSynchronize(s));
  if (!flag) return SMSM_OK;
  SMSM_CUDA_TRY(cudaMemsetAsync(c->devflag, 0, sizeof(int), s));
  smsm_set_error("a convolution gave up a bounded wait (device status %d)", flag);
  return (smsm_status)flag;
}

extern "C" smsm_status smsm_cnn_device_status(smsm_cnn_t cnn, void* stream) {
  smsm_status st;
  if ((st = check_cnn(cnn, "smsm_cnn_device_status", 0))) return st;
  return cnn_status(cnn, (cudaStream_t)stream);
}

// Not part of the interface: raises the flag as a kernel whose wait ran out does, for tests of what callers hear.
extern "C" smsm_status smsm_cnn_raise_for_test(smsm_cnn_t cnn, int status) {
  if (!cnn) return SMSM_ERR_ARG;
  SMSM_CUDA_TRY(cudaMemcpy(cnn->devflag, &status, sizeof(int), cudaMemcpyHostToDevice));
  return SMSM_OK;
}

// loss (mean over the batch) and its gradients into cnn->grad; x0 lands in z[last]
static smsm_status cnn_backward(smsm_cnn_s* c, const float2* a, const float2* t, int n, double* loss,
                                cudaStream_t s) {
  smsm_status st;
  const int Lk = c->layers;
  const size_t HW = (size_t)c->H * c->W, per = (size_t)c->B * HW;
  float2* x0 = c->z[Lk - 1];
  if ((st = cnn_forward(c, a, x0, n, c->devflag, s))) return st;
  k_cnn_loss_sums<<<n, 256, 0, s>>>(x0, t, per, c->lpart);
  SMSM_LAUNCH_CHECK("k_cnn_loss_sums");
  float2* G = c->gA;
  float2* Gn = c->gB;
  k_cnn_loss_grad<<<dim3(64, n), 256, 0, s>>>(x0, t, per, c->lpart, G);
  SMSM_LAUNCH_CHECK("k_cnn_loss_grad");
  for (int k = Lk - 1; k >= 0; --k) {
    const int ci = c->cin[k], co = c->cout[k];
    const float2* h = k == 0 ? a : c->z[k - 1];
    dim3 gw((co + WG_OCB - 1) / WG_OCB, (ci + WG_ICB - 1) / WG_ICB, WG_SPLIT);
    k_cnn_wgrad<<<gw, 256, wgrad_smem(), s>>>(G, h, c->wpart, n, ci, co, c->H, c->W, k > 0);
    SMSM_LAUNCH_CHECK("k_cnn_wgrad");
    const size_t cnt = (size_t)co * ci * 9 + co;  // W_k and b_k are contiguous
    k_cnn_wgrad_reduce<<<(int)((cnt + 255) / 256), 256, 0, s>>>(c->wpart, c->grad + c->woff[k], cnt, 1.f / n);
    SMSM_LAUNCH_CHECK("k_cnn_wgrad_reduce");
    if (k > 0) {
      k_cnn_wt<<<(int)(((size_t)co * ci * 9 + 255) / 256), 256, 0, s>>>(c->wbf + c->woff[k], c->wt, ci, co);
      SMSM_LAUNCH_CHECK("k_cnn_wt");
      // dh_{k} = conv(G, wt); times the CReLU mask of z_{k-1}: the gradient of z_{k-1}
      if ((st = conv(c, G, c->wt, nullptr, nullptr, c->z[k - 1], Gn, n, co, ci, 0, c->devflag, s))) return st;
      float2* tmp = G;
      G = Gn;
      Gn = tmp;
    }
  }
  if (loss) {
    std::vector<double> h(2 * (size_t)n);
    SMSM_CUDA_TRY(cudaMemcpyAsync(h.data(), c->lpart, h.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
    if ((st = cnn_status(c, s))) return st;
    double L = 0.0;
    for (int i = 0; i < n; ++i) L += h[2 * i] / h[2 * i + 1];
    *loss = L / n;
  }
  return SMSM_OK;
}

static smsm_status check_train_args(smsm_cnn_t cnn, const char* fn, const void* a, const void* t, int n) {
  smsm_status st;
  if ((st = check_cnn(cnn, fn, n))) return st;
  if (n < 1 || !al16(a) || !al16(t)) {
    smsm_set_error("%s: need n >= 1 and 16-byte aligned device pointers a, t", fn);
    return SMSM_ERR_ARG;
  }
  return SMSM_OK;
}

extern "C" smsm_status smsm_cnn_gradients(smsm_cnn_t cnn, const void* a, const void* t, int n, void* grad,
                                          double* loss, void* stream) {
  smsm_status st;
  if ((st = check_train_args(cnn, "smsm_cnn_gradients", a, t, n))) return st;
  if (!al16(grad)) {
    smsm_set_error("smsm_cnn_gradients: grad must be a 16-byte aligned device pointer");
    return SMSM_ERR_ARG;
  }
  cudaStream_t s = (cudaStream_t)stream;
  if ((st = cnn_backward(cnn, (const float2*)a, (const float2*)t, n, loss, s))) return st;
  SMSM_CUDA_TRY(cudaMemcpyAsync(grad, cnn->grad, cnn->count * sizeof(float2), cudaMemcpyDeviceToDevice, s));
  return SMSM_OK;
}

extern "C" smsm_status smsm_cnn_train_step(smsm_cnn_t cnn, const void* a, const void* t, int n, float lr,
                                           double* loss, void* stream) {
  smsm_status st;
  if ((st = check_train_args(cnn, "smsm_cnn_train_step", a, t, n))) return st;
  if (!(lr > 0.f)) {
    smsm_set_error("smsm_cnn_train_step: learning rate must be > 0");
    return SMSM_ERR_ARG;
  }
  cudaStream_t s = (cudaStream_t)stream;
  if ((st = cnn_backward(cnn, (const float2*)a, (const float2*)t, n, loss, s))) return st;
  cnn->step += 1;
  const float c1 = 1.f - powf(0.9f, (float)cnn->step), c2 = 1.f - powf(0.999f, (float)cnn->step);
  k_cnn_adam<<<512, 256, 0, s>>>(cnn->master, cnn->wbf, cnn->grad, cnn->m1, cnn->m2, cnn->count, lr, c1, c2);
  SMSM_LAUNCH_CHECK("k_cnn_adam");
  return SMSM_OK;
}
