// Training of the per-site noise-scale network (learned extension, not in the
// paper): forward/backward in FP32 over sampled per-site inputs, the correlator
// loss in its Gram form, deterministic gradient reduction, and Adam.
//
// Loss (runs r, included wave vectors k, hydrodynamic pairs p):
//   L = 1/(R P K) sum_r sum_{k,p} | D_rp(k) + sum_c (m_rc - 1) G^c_rp(k) |^2,
//   D = S^plain - delta_p,  m_rc = mean_b s_c(x_rb)^2,
// which expands per run into d0 + 2 g.(m-1) + (m-1)^T H (m-1) with
//   d0 = sum |D|^2,  g_c = Re sum D^* G^c,  H_cc' = Re sum G^c* G^c'.
// flb_mlp_gram computes (d0, g, H) once; every training step then needs only
// the network.  Weight vector layout: W1 (32x3), W2 (32x32), W3 (6x32), b1, b2, b3.
#include <algorithm>
#include <cstring>

#include "fft_common.cuh"

namespace flb {

constexpr int kH = kMlpHidden, kO = kMlpOut;
constexpr int kOffW1 = 0, kOffW2 = kOffW1 + kH * 3, kOffW3 = kOffW2 + kH * kH;
constexpr int kOffB1 = kOffW3 + kO * kH, kOffB2 = kOffB1 + kH, kOffB3 = kOffB2 + kH;
constexpr int kNParams = kOffB3 + kO;                       // 1382
constexpr int kGram = 1 + kO + kO * kO;                     // d0, g[6], H[6][6]
constexpr int kPairs = 6;
constexpr int kTrainBlock = 256;

// (d0, g, H) per run.  Splain: [R][P][K] complex, G: [R][C][P][K] complex (re, im).
// One block per run; fixed-order block reduction.
__global__ void k_mlp_gram(const double* __restrict__ Sp, const double* __restrict__ G, int P, int K,
                           double* __restrict__ out) {
  const int r = blockIdx.x;
  __shared__ double red[kTrainBlock];
  const int n_terms = kGram;
  for (int term = 0; term < n_terms; ++term) {
    double acc = 0.0;
    for (int i = threadIdx.x; i < P * K; i += blockDim.x) {
      const int p = i / K;
      const double tgt = (p == 0 || p == 3 || p == 5) ? 1.0 : 0.0;
      const double* s = Sp + 2 * ((size_t)r * P * K + i);
      const double dr = s[0] - tgt, di = s[1];
      if (term == 0) {
        acc += dr * dr + di * di;
      } else if (term <= kO) {
        const int c = term - 1;
        const double* gc = G + 2 * (((size_t)r * kO + c) * P * K + i);
        acc += dr * gc[0] + di * gc[1];
      } else {
        const int c = (term - 1 - kO) / kO, c2 = (term - 1 - kO) % kO;
        const double* ga = G + 2 * (((size_t)r * kO + c) * P * K + i);
        const double* gb = G + 2 * (((size_t)r * kO + c2) * P * K + i);
        acc += ga[0] * gb[0] + ga[1] * gb[1];
      }
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
      if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
      __syncthreads();
    }
    if (threadIdx.x == 0) out[(size_t)r * kGram + term] = red[0];
    __syncthreads();
  }
}

// The network in shared memory: rows of W1 with their bias (one 16-byte read per hidden
// unit), W2 and W3 row-major.
struct TrainNet {
  float4 w1[kH];
  float w2[kH][kH];
  float w3[kO][kH];
  float b2[kH], b3[kO];

  __device__ void load(const float* __restrict__ W) {
    for (int i = threadIdx.x; i < kH; i += blockDim.x) {
      const float* r = W + kOffW1 + 3 * i;
      w1[i] = make_float4(r[0], r[1], r[2], W[kOffB1 + i]);
      b2[i] = W[kOffB2 + i];
    }
    for (int i = threadIdx.x; i < kH * kH; i += blockDim.x) w2[i / kH][i % kH] = W[kOffW2 + i];
    for (int i = threadIdx.x; i < kO * kH; i += blockDim.x) w3[i / kH][i % kH] = W[kOffW3 + i];
    for (int i = threadIdx.x; i < kO; i += blockDim.x) b3[i] = W[kOffB3 + i];
  }
};

// Forward of one input, everything in registers: every unit's sum starts at its bias and
// adds its inputs in index order; eight units' chains run side by side.
__device__ __forceinline__ void forward(const TrainNet& W, const float (&x)[3], float (&h1)[kH], float (&h2)[kH],
                                        float (&s)[kO]) {
#pragma unroll
  for (int h = 0; h < kH; ++h) {
    const float4 w = W.w1[h];
    h1[h] = fmaxf(fmaf(w.z, x[2], fmaf(w.y, x[1], fmaf(w.x, x[0], w.w))), 0.f);
  }
#pragma unroll
  for (int h0 = 0; h0 < kH; h0 += 8) {
    float z[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) z[j] = W.b2[h0 + j];
#pragma unroll
    for (int k = 0; k < kH; k += 4)
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float4 w = *reinterpret_cast<const float4*>(&W.w2[h0 + j][k]);
        z[j] = fmaf(w.w, h1[k + 3], fmaf(w.z, h1[k + 2], fmaf(w.y, h1[k + 1], fmaf(w.x, h1[k], z[j]))));
      }
#pragma unroll
    for (int j = 0; j < 8; ++j) h2[h0 + j] = fmaxf(z[j], 0.f);
  }
#pragma unroll
  for (int c = 0; c < kO; ++c) s[c] = W.b3[c];
#pragma unroll
  for (int h = 0; h < kH; h += 4)
#pragma unroll
    for (int c = 0; c < kO; ++c) {
      const float4 w = *reinterpret_cast<const float4*>(&W.w3[c][h]);
      s[c] = fmaf(w.w, h2[h + 3], fmaf(w.z, h2[h + 2], fmaf(w.y, h2[h + 1], fmaf(w.x, h2[h], s[c]))));
    }
#pragma unroll
  for (int c = 0; c < kO; ++c) s[c] = 1.f + s[c];
}

// Pass 1: forward of every sample, block partial sums of s_c^2 per run.
// grid = R * blocks_per_run; block b of run r covers samples [b*256, b*256+256).
// FP32 issue-bound (1312 multiply-adds a sample, weights by 16-byte shared reads).  The
// FP64 sums go through shared memory, 8 values a thread and then 32 a channel: a warp
// shuffle tree would spend every lane's slot of GB300's 2-per-clock FP64 pipe on each add.
__global__ void __launch_bounds__(kTrainBlock)
k_mlp_fwd_stats(const float* __restrict__ Wg, const float* __restrict__ X, int B, int blocks_per_run,
                double* __restrict__ partial) {
  __shared__ __align__(16) TrainNet W;
  __shared__ float s_sh[kO][kTrainBlock];
  __shared__ double red[kO][32];
  W.load(Wg);
  __syncthreads();
  const int r = blockIdx.x / blocks_per_run, bb = blockIdx.x % blocks_per_run;
  const int b = bb * blockDim.x + threadIdx.x;
  float s[kO] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  if (b < B) {
    const float* xp = X + 3 * ((size_t)r * B + b);
    const float x[3] = {xp[0], xp[1], xp[2]};
    float h1[kH], h2[kH];
    forward(W, x, h1, h2, s);
  }
#pragma unroll
  for (int c = 0; c < kO; ++c) s_sh[c][threadIdx.x] = s[c];
  __syncthreads();
  if (threadIdx.x < 32 * kO) {
    const int c = threadIdx.x >> 5, j = threadIdx.x & 31;
    double v = 0.0;
#pragma unroll
    for (int i = 0; i < kTrainBlock / 32; ++i) {
      const double q = (double)s_sh[c][j + 32 * i];
      v = fma(q, q, v);
    }
    red[c][j] = v;
  }
  __syncthreads();
  if (threadIdx.x < kO) {
    double v = 0.0;
    for (int j = 0; j < 32; ++j) v += red[threadIdx.x][j];
    partial[(size_t)blockIdx.x * kO + threadIdx.x] = v;
  }
}

// Pass 2 (a warp per run; one block up to kLossRuns runs, which then also adds the losses): m_rc, the
// per-run loss and, from the Gram terms, dL/dm_rc 2 / B (the factor of s_c in dL/ds_c of a sample);
// thread 0 of a single block then adds the per-run losses in order.  Lane c + 8 j (c < 6, j < 4) sums
// channel c's partials j, j + 4, ..; all the loads of a run are in flight together.
constexpr int kLossBlock = 512, kLossRuns = 64;
__global__ void __launch_bounds__(kLossBlock)
k_mlp_loss(const double* __restrict__ partial, int R, int B, int blocks_per_run, const double* __restrict__ gram,
           double norm, double* __restrict__ m_out, double* __restrict__ dm, double* __restrict__ loss_r,
           double* __restrict__ loss) {
  const int lane = threadIdx.x & 31, c = lane & 7, j = lane >> 3;
  for (int64_t r = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); r < R;
       r += (int64_t)gridDim.x * (blockDim.x >> 5)) {
    const double* gm = gram + (size_t)r * kGram;
    double g = 0.0, H[kO] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    double m = 0.0;
    if (c < kO) {
      g = gm[1 + c];
#pragma unroll
      for (int c2 = 0; c2 < kO; ++c2) H[c2] = gm[1 + kO + c * kO + c2];
#pragma unroll 4
      for (int bb = j; bb < blocks_per_run; bb += 4) m += partial[((size_t)r * blocks_per_run + bb) * kO + c];
    }
    m += __shfl_xor_sync(0xffffffffu, m, 8);
    m += __shfl_xor_sync(0xffffffffu, m, 16);
    m /= B;
    double hd = 0.0;
#pragma unroll
    for (int c2 = 0; c2 < kO; ++c2) hd += H[c2] * (__shfl_sync(0xffffffffu, m, c2) - 1.0);
    const double term = 2.0 * g * (m - 1.0) + (m - 1.0) * hd;
    if (lane < kO) {
      m_out[r * kO + c] = m;
      dm[r * kO + c] = norm * (2.0 * g + 2.0 * hd) * 2.0 / B;
    }
    double L = gm[0];
#pragma unroll
    for (int c2 = 0; c2 < kO; ++c2) L += __shfl_sync(0xffffffffu, term, c2);
    if (lane == 0) loss_r[r] = L;
  }
  if (gridDim.x > 1) return;                // k_mlp_loss_sum
  __syncthreads();
  if (threadIdx.x == 0) {
    double L = 0.0;
    for (int r = 0; r < R; ++r) L += loss_r[r];
    *loss = norm * L;
  }
}

// The loss of many runs: strided sums of a block's threads, then those in order (20,000 runs: the whole step
// 11.2 ms with all of pass 2 in one block, 0.53 so).
__global__ void __launch_bounds__(kTrainBlock)
k_mlp_loss_sum(const double* __restrict__ loss_r, int R, double norm, double* __restrict__ loss) {
  __shared__ double part[kTrainBlock];
  double L = 0.0;
  for (int64_t r = threadIdx.x; r < R; r += kTrainBlock) L += loss_r[r];
  part[threadIdx.x] = L;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < kTrainBlock; ++i) L += part[i];
    *loss = norm * L;
  }
}

// Dot product term a b added to the unevaluated sum s + c: the product and the sum are
// split into their rounded value and the exact rounding error (two-product by fused
// multiply-add, two-sum by Knuth), and the errors collected in c -- the Dot2 scheme of
// Ogita, Rump & Oishi (SIAM J. Sci. Comput. 26, 2005), whose result is as accurate as one
// computed in twice the working precision.  That is 48 bits in FP32's exponent range, less than
// FP64: the error of n = 108 terms (a thread's share of 16 x 4096 samples) is 5e-15 of the sum of their
// magnitudes in the root mean square, 1.1e-13 at most in 2000 sums (FP64 3e-17 and 2e-16), and bounded
// by (n 2^-24)^2; the rounding of the gradient to FP32 covers it unless the terms cancel to 10^-7 of their
// magnitudes.  Products below 2^-102 lose part of their error term, and a partial sum beyond FP32's
// range is infinite.
__device__ __forceinline__ void dot2_add(float a, float b, float& s, float& c) {
  const float p = __fmul_rn(a, b), e = __fmaf_rn(a, b, -p);
  const float t = __fadd_rn(s, p), z = __fsub_rn(t, s);
  const float q = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));
  c = __fadd_rn(c, __fadd_rn(q, e));
  s = t;
}
__device__ __forceinline__ double dot2_value(float s, float c) {
  return isfinite(s) && isfinite(c) ? (double)s + (double)c : (double)s;   // the split of an infinity is a NaN
}

// Pass 3: backward of every sample and the gradient sums of the block's samples.
//
// The gradient is 1382 sums over all samples, 1024 of them the products dz2_h h1_k.  As
// one block per parameter with FP64 multiply-adds over intermediates in memory it was
// bound by GB300's FP64 pipe (2 per clock per SM) and by reading the 36 MB of
// intermediates hundreds of times from L2: 541 us of a 630 us step at 16 x 4096 samples.
// Here a block takes a contiguous range of samples in tiles.  Each thread runs one sample
// forward and backward in registers and leaves the factors of its products in shared
// memory; then every thread adds a 4 x 4 patch of products over the tile's samples with
// the two-FP32 sums of dot2_add (10 FP32 operations a term on a pipe 64 times as wide as
// the FP64 one): 69 us, FP32 issue-bound, and 98 us for the whole step.  The sums stay in registers over the tiles; each
// block then writes one FP64 partial per parameter.
//
// kGradGroup threads cover all 1382 sums once; a block has kGradGroups such groups, which
// take every other four samples.  Factor rows in shared memory, kGradStride floats apart
// (rows 4 banks x 5 apart: eight threads reading eight consecutive rows by float4 hit
// every bank once).
constexpr int kGradGroup = 96, kGradGroups = 2, kGradThreads = kGradGroup * kGradGroups;
constexpr int kGradTile = 176, kGradStride = 180;
constexpr int kRowDz1 = 0, kRowDz2 = kRowDz1 + kH, kRowDo = kRowDz2 + kH, kRowX = kRowDo + 8, kRowOne = kRowX + 3;
constexpr int kRowH1 = kRowOne + 1, kRowH2 = kRowH1 + kH, kGradRows = kRowH2 + kH;
constexpr int kGradMaxBlocks = 304;          // two blocks on each of GB300's 152 SMs; a constant, so that the
                                             // scratch size and the order of the sums do not follow the device
constexpr size_t kGradSmem = sizeof(TrainNet) + sizeof(float) * kGradRows * kGradStride;
static_assert(2 * (kGradSmem + 1024) <= 228 * 1024, "two blocks per SM");
static_assert(kGradTile <= kGradThreads && kGradTile % 8 == 0 && kGradTile <= kGradStride, "one sample per thread");

// blocks and samples per block of the gradient pass
__host__ __device__ inline int grad_blocks(int64_t n) {
  const int64_t per = 64;                    // no fewer samples than this in a block
  const int64_t g = (n + per - 1) / per;
  return (int)(g < kGradMaxBlocks ? g : kGradMaxBlocks);
}

__global__ void __launch_bounds__(kGradThreads, 2)
k_mlp_grad(const float* __restrict__ Wg, const float* __restrict__ X, int R, int B, const double* __restrict__ dm,
           double* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* rows = reinterpret_cast<float*>(smem_raw + sizeof(TrainNet));
  reinterpret_cast<TrainNet*>(smem_raw)->load(Wg);
  unsigned int w_off = 0;
  const int tid = threadIdx.x, grp = tid / kGradGroup, g = tid % kGradGroup;
  // this thread's patch: factor rows a_r (r < 4) times rows b_q (q < 4)
  //   g < 64:  dz2[g % 8 + 8 r] h1[g / 8 + 8 q]
  //   64..71:  dz1[u + 8 r] (x_0, x_1, x_2, 1)_q, u = g - 64        (W1 and b1)
  //   72..87:  do[u % 2 + 2 r] h2[u / 2 + 8 q], u = g - 72          (W3; rows 6, 7 of do are zero)
  //   88..95:  dz2[u + 8 r] (1, .., ..)_q, u = g - 88              (b2)
  // and, for 88..95, the plain sum of do[u] (b3)
  int a0, as, b0, bs;
  if (g < 64) { a0 = kRowDz2 + (g & 7); as = 8; b0 = kRowH1 + (g >> 3); bs = 8; }
  else if (g < 72) { a0 = kRowDz1 + (g - 64); as = 8; b0 = kRowX; bs = 1; }
  else if (g < 88) { a0 = kRowDo + (g & 1); as = 2; b0 = kRowH2 + ((g - 72) >> 1); bs = 8; }
  else { a0 = kRowDz2 + (g - 88); as = 8; b0 = kRowOne; bs = 0; }
  const float* pa = rows + a0 * kGradStride;
  const float* pb = rows + b0 * kGradStride;
  const float* pd = rows + (kRowDo + (g & 7)) * kGradStride;
  as *= kGradStride; bs *= kGradStride;
  float s[4][4], c[4][4], s3 = 0.f, c3 = 0.f;
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) { s[r][q] = 0.f; c[r][q] = 0.f; }

  // the block's samples in equal tiles of at most kGradTile (a multiple of 8 rows wide)
  const int64_t n = (int64_t)R * B, per = (n + gridDim.x - 1) / gridDim.x;
  const int64_t i0 = blockIdx.x * per, i1 = i0 + per < n ? i0 + per : n;
  const int tiles = (int)((per + kGradTile - 1) / kGradTile);
  const int tile = (int)((per + tiles - 1) / tiles);
  for (int64_t t0 = i0; t0 < i1; t0 += tile) {
    const int cnt = (int)(i1 - t0 < tile ? i1 - t0 : tile), cnt8 = (cnt + 7) & ~7;
    __syncthreads();                        // W is loaded; the previous tile's rows are used
    asm volatile("" : "+r"(w_off));         // opaque: no weight is kept across tiles (1376 of them spill)
    const TrainNet& W = *reinterpret_cast<const TrainNet*>(smem_raw + w_off);
    if (tid < cnt) {
      const int64_t i = t0 + tid;
      const int run = (int)(i / B);
      const float x[3] = {X[3 * i], X[3 * i + 1], X[3 * i + 2]};
      float h1[kH], h2[kH], sc[kO], dout[kO];
      forward(W, x, h1, h2, sc);
      float* o = rows + tid;
#pragma unroll
      for (int k = 0; k < 3; ++k) o[(kRowX + k) * kGradStride] = x[k];
      o[kRowOne * kGradStride] = 1.f;
#pragma unroll
      for (int k = 0; k < kO; ++k) {
        // in FP64: dL/dm alone may leave FP32's range (s = 1 + o is never subnormal, widen is exact)
        dout[k] = (float)(dm[run * kO + k] * widen(sc[k]));
        o[(kRowDo + k) * kGradStride] = dout[k];
      }
      o[(kRowDo + 6) * kGradStride] = 0.f;
      o[(kRowDo + 7) * kGradStride] = 0.f;
      float dz1[kH];
#pragma unroll
      for (int k = 0; k < kH; ++k) dz1[k] = 0.f;
#pragma unroll
      for (int h = 0; h < kH; ++h) {
        o[(kRowH2 + h) * kGradStride] = h2[h];
        float v = 0.f;
#pragma unroll
        for (int k = 0; k < kO; ++k) v = fmaf(W.w3[k][h], dout[k], v);
        const float dz2 = h2[h] > 0.f ? v : 0.f;
        o[(kRowDz2 + h) * kGradStride] = dz2;
#pragma unroll
        for (int k = 0; k < kH; k += 4) {
          const float4 w = *reinterpret_cast<const float4*>(&W.w2[h][k]);
          dz1[k] = fmaf(w.x, dz2, dz1[k]);
          dz1[k + 1] = fmaf(w.y, dz2, dz1[k + 1]);
          dz1[k + 2] = fmaf(w.z, dz2, dz1[k + 2]);
          dz1[k + 3] = fmaf(w.w, dz2, dz1[k + 3]);
        }
      }
#pragma unroll
      for (int k = 0; k < kH; ++k) {
        o[(kRowH1 + k) * kGradStride] = h1[k];
        o[(kRowDz1 + k) * kGradStride] = h1[k] > 0.f ? dz1[k] : 0.f;
      }
    } else if (tid < cnt8) {                // pad the tile with zero samples
      for (int k = 0; k < kGradRows; ++k) rows[k * kGradStride + tid] = 0.f;
    }
    __syncthreads();
    for (int i = 4 * grp; i < cnt8; i += 4 * kGradGroups) {
      float4 av[4], bv[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        av[r] = *reinterpret_cast<const float4*>(pa + r * as + i);
        bv[r] = *reinterpret_cast<const float4*>(pb + r * bs + i);
      }
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          dot2_add(av[r].x, bv[q].x, s[r][q], c[r][q]);
          dot2_add(av[r].y, bv[q].y, s[r][q], c[r][q]);
          dot2_add(av[r].z, bv[q].z, s[r][q], c[r][q]);
          dot2_add(av[r].w, bv[q].w, s[r][q], c[r][q]);
        }
      if (g >= 64) {                        // the last warp of the group
        const float4 d = *reinterpret_cast<const float4*>(pd + i);
        dot2_add(d.x, 1.f, s3, c3);
        dot2_add(d.y, 1.f, s3, c3);
        dot2_add(d.z, 1.f, s3, c3);
        dot2_add(d.w, 1.f, s3, c3);
      }
    }
  }
  // the two groups' sums in FP64, group 1 first into shared memory
  __syncthreads();
  double* sum = reinterpret_cast<double*>(rows);           // [kNParams]
  double* out = part + (size_t)blockIdx.x * kNParams;
  for (int pass = kGradGroups - 1; pass >= 0; --pass) {
    if (grp == pass) {
      auto put = [&](int p, float hi, float lo) {
        const double v = dot2_value(hi, lo) + (pass == kGradGroups - 1 ? 0.0 : sum[p]);
        if (pass) sum[p] = v;
        else out[p] = v;
      };
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (g < 64) put(kOffW2 + kH * ((g & 7) + 8 * r) + (g >> 3) + 8 * q, s[r][q], c[r][q]);
          else if (g < 72) put(q < 3 ? kOffW1 + 3 * (g - 64 + 8 * r) + q : kOffB1 + g - 64 + 8 * r, s[r][q], c[r][q]);
          else if (g < 88) {
            const int o = (g & 1) + 2 * r;
            if (o < kO) put(kOffW3 + kH * o + ((g - 72) >> 1) + 8 * q, s[r][q], c[r][q]);
          } else if (q == 0) put(kOffB2 + g - 88 + 8 * r, s[r][q], c[r][q]);
        }
      if (g >= 88 && g - 88 < kO) put(kOffB3 + g - 88, s3, c3);
    }
    __syncthreads();
  }
}

// Pass 4: the gradient from the blocks' partials (fixed order: 16 interleaved sums per
// parameter, then those in order) and, with lr > 0, Adam (Kingma & Ba, 2015) with bias
// correction.
constexpr int kFinishSlices = 16;
__global__ void __launch_bounds__(kTrainBlock)
k_mlp_grad_finish(const double* __restrict__ part, int blocks, float* __restrict__ grad, float* __restrict__ W,
                  float* __restrict__ m, float* __restrict__ v, float lr, float b1, float b2, float eps, float c1,
                  float c2) {
  constexpr int kCols = kTrainBlock / kFinishSlices;
  __shared__ double red[kFinishSlices][kCols];
  const int col = threadIdx.x % kCols, sl = threadIdx.x / kCols;
  const int i = blockIdx.x * kCols + col;
  double acc = 0.0;
  if (i < kNParams) {
#pragma unroll 10
    for (int b = sl; b < blocks; b += kFinishSlices) acc += part[(size_t)b * kNParams + i];
  }
  red[sl][col] = acc;
  __syncthreads();
  if (sl != 0 || i >= kNParams) return;
  for (int k = 1; k < kFinishSlices; ++k) acc += red[k][col];
  const float g = (float)acc;
  grad[i] = g;
  if (!(lr > 0.f)) return;
  const float mi = fmaf(b1, m[i], (1.f - b1) * g);
  const float vi = fmaf(b2, v[i], (1.f - b2) * g * g);
  m[i] = mi;
  v[i] = vi;
  W[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

static int64_t a256(int64_t x) { return (x + 255) & ~int64_t(255); }

struct TrainLayout {
  int blocks_per_run;
  int64_t off_partial, off_dm, off_lossr, off_part, off_grad, total;
};

static TrainLayout train_layout(int R, int B) {
  TrainLayout t;
  t.blocks_per_run = (B + kTrainBlock - 1) / kTrainBlock;
  int64_t off = 0;
  t.off_partial = off; off = a256(off + 8 * (int64_t)R * t.blocks_per_run * kO);
  t.off_dm = off; off = a256(off + 8 * (int64_t)R * kO);
  t.off_lossr = off; off = a256(off + 8 * (int64_t)R);
  t.off_grad = off; off = a256(off + 4 * (int64_t)kNParams);
  t.off_part = off; off = a256(off + 8 * (int64_t)kNParams * grad_blocks((int64_t)R * B));
  t.total = off;
  return t;
}

}  // namespace flb

using namespace flb;

extern "C" {

int flb_mlp_param_count(void) { return kNParams; }

int flb_mlp_gram(const double* splain_dev, const double* g_dev, int R, int P, int K, double* gram_dev,
                 void* cuda_stream) {
  if (R < 1 || P != kPairs || K < 1) return set_error(FLB_EINVAL, "need R >= 1, P = 6 pairs, K >= 1");
  if (!splain_dev || !g_dev || !gram_dev) return set_error(FLB_EINVAL, "NULL pointer");
  k_mlp_gram<<<R, kTrainBlock, 0, static_cast<cudaStream_t>(cuda_stream)>>>(splain_dev, g_dev, P, K, gram_dev);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? FLB_OK : set_error(FLB_ECUDA, "flb_mlp_gram: %s", cudaGetErrorString(e));
}

int flb_mlp_scratch_bytes(int R, int B, size_t* bytes) {
  if (R < 1 || B < 1 || !bytes) return set_error(FLB_EINVAL, "need R, B >= 1");
  *bytes = (size_t)train_layout(R, B).total;
  return FLB_OK;
}

int flb_mlp_train_step(float* w_dev, float* adam_m_dev, float* adam_v_dev, int t, float lr, float beta1,
                       float beta2, float eps, const float* x_dev, int R, int B, const double* gram_dev,
                       int P, int K, double* loss_dev, double* m_dev, float* grad_dev, void* scratch_dev,
                       size_t scratch_bytes, void* cuda_stream) {
  if (!w_dev || !x_dev || !gram_dev || !loss_dev || !m_dev || !scratch_dev) return set_error(FLB_EINVAL, "NULL pointer");
  if (R < 1 || B < 1 || P != kPairs || K < 1) return set_error(FLB_EINVAL, "need R, B, K >= 1 and P = 6");
  if (lr > 0.f && (!adam_m_dev || !adam_v_dev || t < 1)) return set_error(FLB_EINVAL, "Adam needs m, v and t >= 1");
  const TrainLayout T = train_layout(R, B);
  if (scratch_bytes < (size_t)T.total) return set_error(FLB_ENOMEM, "scratch %zu < %lld bytes", scratch_bytes, (long long)T.total);
  if (((uintptr_t)scratch_dev) & 255) return set_error(FLB_EINVAL, "scratch must be 256-byte aligned");
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  char* s = static_cast<char*>(scratch_dev);
  double* partial = reinterpret_cast<double*>(s + T.off_partial);
  double* dm = reinterpret_cast<double*>(s + T.off_dm);
  double* part = reinterpret_cast<double*>(s + T.off_part);
  float* grad = grad_dev ? grad_dev : reinterpret_cast<float*>(s + T.off_grad);
  const double norm = 1.0 / ((double)R * P * K);
  cudaError_t e = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGradSmem);
  if (e != cudaSuccess) return set_error(FLB_ECUDA, "flb_mlp_train_step: %s", cudaGetErrorString(e));
  k_mlp_fwd_stats<<<R * T.blocks_per_run, kTrainBlock, 0, st>>>(w_dev, x_dev, B, T.blocks_per_run, partial);
  double* loss_r = reinterpret_cast<double*>(s + T.off_lossr);
  const int loss_blocks = R <= kLossRuns ? 1 : std::min((R + kLossBlock / 32 - 1) / (kLossBlock / 32), 1216);
  k_mlp_loss<<<loss_blocks, R < kLossBlock / 32 ? 32 * R : kLossBlock, 0, st>>>(partial, R, B, T.blocks_per_run, gram_dev,
                                                                                norm, m_dev, dm, loss_r, loss_dev);
  if (loss_blocks > 1) k_mlp_loss_sum<<<1, kTrainBlock, 0, st>>>(loss_r, R, norm, loss_dev);
  const int blocks = grad_blocks((int64_t)R * B);
  k_mlp_grad<<<blocks, kGradThreads, kGradSmem, st>>>(w_dev, x_dev, R, B, dm, part);
  const float c1 = lr > 0.f ? 1.f - powf(beta1, (float)t) : 1.f, c2 = lr > 0.f ? 1.f - powf(beta2, (float)t) : 1.f;
  constexpr int kCols = kTrainBlock / kFinishSlices;
  k_mlp_grad_finish<<<(kNParams + kCols - 1) / kCols, kTrainBlock, 0, st>>>(part, blocks, grad, w_dev, adam_m_dev,
                                                                            adam_v_dev, lr, beta1, beta2, eps, c1, c2);
  e = cudaGetLastError();
  return e == cudaSuccess ? FLB_OK : set_error(FLB_ECUDA, "flb_mlp_train_step: %s", cudaGetErrorString(e));
}

}  // extern "C"
