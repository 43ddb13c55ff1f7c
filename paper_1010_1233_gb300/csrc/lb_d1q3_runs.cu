// Runs of D1Q3 steps in FP64 with their correlator sampling.
//
// The lattices are small (L = 64 in the D1Q3 workload) and each step needs the one before, so a
// run is a chain; what can be taken off the chain decides its time (all of it in one block: 10 - 12 us
// a step at L = 64 with every step sampled, nearly all latency between barriers).  Only the step itself is
// serial here, and the rest runs on the whole GPU before and after it, a chunk of steps at a time:
//   k_d1q3_noise   the noise of every (step, site) of the chunk
//   k_d1q3_steps   one block per replica: pull and collide, 15 FP64 instructions a site, one barrier
//                  a step; the noise is loaded two steps ahead; at a sample the pulled
//                  populations go to memory
//   k_d1q3_sample  row transforms of all samples (radix-2 passes of fft_common.cuh, two fields
//                  packed per complex row) and their pair products
//   k_d1q3_sums    adds the products to the replica's sums, sample by sample (k_d1q3_sums_many on large
//                  batches; on small ones blocks of the next k_d1q3_steps do it while there is one)
// Every sum takes the samples' products one at a time in the order of the steps, as the per-step
// launches add them, so it does not depend on how runs are cut into calls and chunks or on the other
// replicas of the context.
// k_d1q3_steps is bound by its warps' FP64 instructions, one in 64 cycles (15 x 64 = 960 of the 1240
// cycles of a step up to 128 sites, four warps on four schedulers): L = 64, 0.60 us a step, 0.64 with
// every step sampled.
#include <algorithm>
#include "d1q3_common.cuh"
#include "fft_common.cuh"

namespace flb {

constexpr int kD1SampleThreads = 256;
constexpr int kD1SamplePoints = 2048;        // points of packed rows in one block's batch, at most
constexpr size_t kD1SampleSmem = 80 * 1024;  // shared memory of a batch of more than one sample

__host__ __device__ inline int d1_rows(int F) { return (F + 1) / 2; }           // packed rows per sample
// shared memory of one sample: its packed rows with their pad slots and the half spectra of its fields
__host__ __device__ inline size_t d1_sample_bytes(int nx, int F) {
  return ((size_t)d1_rows(F) * (nx + 33) + (size_t)F * (nx / 2 + 1)) * sizeof(double2);
}
// samples of a batch of k_d1q3_sample: as many as kD1SamplePoints and kD1SampleSmem hold (below 32 sites
// the pad slots take most of a row), and no more than an even share of the ns samples (a batch's
// transforms are FP64-bound, 0.5 us a sample at L = 64)
__host__ __device__ inline int d1_batch(int nx, int F) {
  if (F < 1) return 1;
  const int pts = kD1SamplePoints / (nx * d1_rows(F)), fit = (int)(kD1SampleSmem / d1_sample_bytes(nx, F));
  const int b = pts < fit ? pts : fit;
  return b < 1 ? 1 : b;
}
__device__ __forceinline__ int d1_batch_of(int nx, int F, uint32_t ns, int blocks) {
  const int share = (int)((ns + blocks - 1) / blocks);
  return min(d1_batch(nx, F), max(share, 1));
}

size_t d1q3_steps_smem(int nx) { return 6 * (size_t)nx * sizeof(double); }
size_t d1q3_sample_smem(int nx, int F) { return d1_batch(nx, F) * d1_sample_bytes(nx, F); }

// A replica's scratch: noise, pulled populations, and products in the order of its sums: the pairs (one
// double a wave vector for a field with itself, two for two fields), then the k = 0 value of every field.
__device__ __forceinline__ double* d1_noise(const ReplicaDesc& d, char* ws, const D1Scratch& sc) {
  return reinterpret_cast<double*>(ws + sc.noise) + (d.d1_site0 - sc.site0) * sc.steps;
}
__device__ __forceinline__ double* d1_raw(const ReplicaDesc& d, char* ws, const D1Scratch& sc) {
  return reinterpret_cast<double*>(ws + sc.raw) + (d.d1_site0 - sc.site0) * 3 * sc.samples;
}
__device__ __forceinline__ double* d1_products(const ReplicaDesc& d, char* ws, const D1Scratch& sc) {
  return reinterpret_cast<double*>(ws + sc.products) + (d.d1_product0 - sc.product0) * sc.samples;
}

__global__ void __launch_bounds__(256)
k_d1q3_noise(const ReplicaDesc* __restrict__ descs, char* __restrict__ ws, const D1Scratch sc, uint64_t t0,
             uint32_t n_steps) {
  const ReplicaDesc& d = descs[blockIdx.x];
  const int nx = d.nx;
  double* out = d1_noise(d, ws, sc);
  const uint32_t n = n_steps * (uint32_t)nx;
  for (uint32_t i = blockIdx.y * blockDim.x + threadIdx.x; i < n; i += gridDim.y * blockDim.x) {
    const uint32_t s = i / (uint32_t)nx;
    out[i] = d1q3_noise(d, (int)(i - s * nx), (uint32_t)(t0 + s));
  }
}

// The sum of product i (lb_d1q3_runs.cu's order).
__device__ __forceinline__ double* d1_sum(const ReplicaDesc& d, char* __restrict__ ws, int64_t i, int64_t np) {
  const int nx = d.nx;
  if (i >= np - d.n_fields) return reinterpret_cast<double*>(ws + d.off_mean0) + (i - (np - d.n_fields));
  int pr = d.n_pairs - 1;
  while (pr > 0 && i < d1q3_pair_first(nx, pr, d.pair_a[pr], d.pair_b[pr])) --pr;
  return reinterpret_cast<double*>(ws + d.pair_off[pr]) + (i - d1q3_pair_first(nx, pr, d.pair_a[pr], d.pair_b[pr]));
}

// The ns samples' products added to a replica's sums, a thread per product, by block `part` of `parts`:
// beside steps, or in many blocks, so a few loads ahead in registers do (58 ns a sample).
__device__ __forceinline__ void d1q3_add_products(const ReplicaDesc& d, char* __restrict__ ws, const D1Scratch& sc,
                                                  uint32_t ns, int part, int parts) {
  if (!d.n_fields) return;
  const int64_t np = d1q3_products(d.nx, (int)d.n_fields);
  for (int64_t i = (int64_t)part * blockDim.x + threadIdx.x; i < np; i += (int64_t)parts * blockDim.x) {
    double* sum = d1_sum(d, ws, i, np);
    const double* p = d1_products(d, ws, sc) + i;
    double acc = *sum;
    uint32_t s = 0;
    for (; s + 8 <= ns; s += 8) {
      double v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = p[(s + u) * np];
#pragma unroll
      for (int u = 0; u < 8; ++u) acc = __dadd_rn(acc, v[u]);
    }
    for (; s < ns; ++s) acc = __dadd_rn(acc, p[s * np]);
    *sum = acc;
  }
}

// SPT sites per thread (x = tid + k blockDim): steps t0 .. t0 + n_steps - 1 of replica blockIdx.x,
// state from the buffer of parity t0 & 1 to that of (t0 + n_steps) & 1.  The blocks from n_reps on add
// the products of the chunk before (its sum_ns samples), sum_parts of them a replica: 60 us of a chain
// for 1024 samples, beside the 620 us of 1024 steps (2000 steps at L = 64, two fields, every step sampled:
// 1.41 ms with the additions after each chunk, 1.34 here, 1.32 with a short last chunk).
template <int SPT>
__global__ void __launch_bounds__(1024)
k_d1q3_steps(const ReplicaDesc* __restrict__ descs, char* __restrict__ ws, const D1Scratch sc, uint32_t every,
             uint64_t t0, uint32_t n_steps, int n_reps, uint32_t sum_ns, int sum_parts) {
  extern __shared__ __align__(16) double pop[];              // [2][3][nx]
  if ((int)blockIdx.x >= n_reps) {
    const int b = (int)blockIdx.x - n_reps;
    d1q3_add_products(descs[b / sum_parts], ws, sc, sum_ns, b % sum_parts, sum_parts);
    return;
  }
  const ReplicaDesc& d = descs[blockIdx.x];
  const int nx = d.nx, tid = (int)threadIdx.x, nt = (int)blockDim.x;
  const double* src = reinterpret_cast<const double*>(ws + d.off_pop[t0 & 1]);
  for (int i = tid; i < 3 * nx; i += nt) pop[i] = src[i];
  const D1Coef coef(d);
  const double* noise = d1_noise(d, ws, sc) + (int64_t)sc.noise_first * nx;
  double* raw = d1_raw(d, ws, sc);
  int xs[SPT], xl[SPT], xr[SPT];
  double n0[SPT], n1[SPT];                                    // noise of this step and the next
#pragma unroll
  for (int k = 0; k < SPT; ++k) {
    xs[k] = tid + k * nt;
    const bool in = xs[k] < nx;
    xl[k] = nx + (xs[k] == 0 ? nx - 1 : xs[k] - 1);
    xr[k] = 2 * nx + (xs[k] == nx - 1 ? 0 : xs[k] + 1);
    n0[k] = in ? noise[xs[k]] : 0.0;
    n1[k] = in && n_steps > 1 ? noise[nx + xs[k]] : 0.0;
  }
  // steps until the next sample (never without sampled fields)
  uint32_t wait = every && d.n_fields ? (uint32_t)((every - t0 % every) % every) : 0xFFFFFFFFu;
  __syncthreads();
  for (uint32_t s = 0; s < n_steps; ++s) {
    const double* in = pop + (s & 1) * 3 * nx;
    double* out = pop + ((s & 1) ^ 1) * 3 * nx;
    const bool sample = wait == 0;
    wait = sample ? every - 1 : wait - 1;
    const double* nn = noise + (int64_t)(s + 2) * nx;
#pragma unroll
    for (int k = 0; k < SPT; ++k) {
      const int x = xs[k];
      if (x >= nx) continue;
      double g[3] = {in[x], in[xl[k]], in[xr[k]]};
      const double h = n0[k];
      n0[k] = n1[k];
      if (s + 2 < n_steps) n1[k] = nn[x];
      if (sample) {
        raw[x] = g[0];
        raw[nx + x] = g[1];
        raw[2 * nx + x] = g[2];
      }
      d1q3_collide(g, coef, h);
      if (FLB_INB(x >= 0 && xr[k] < 3 * nx && xl[k] < 2 * nx, 181)) {
        out[x] = g[0];
        out[nx + x] = g[1];
        out[2 * nx + x] = g[2];
      }
    }
    if (sample) raw += 3 * nx;
    __syncthreads();
  }
  double* dst = reinterpret_cast<double*>(ws + d.off_pop[(t0 + n_steps) & 1]);
  const double* fin = pop + (n_steps & 1) * 3 * nx;
  for (int i = tid; i < 3 * nx; i += nt) dst[i] = fin[i];
}

// Block g = blockIdx.y of replica blockIdx.x takes the sample batches g, g + G, .. (G = gridDim.y) of the
// chunk's ns samples and leaves their products; the block of the last batch writes its fields.
__global__ void __launch_bounds__(kD1SampleThreads)
k_d1q3_sample(const ReplicaDesc* __restrict__ descs, char* __restrict__ ws, const D1Scratch sc, uint32_t ns) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const ReplicaDesc& d = descs[blockIdx.x];
  const int nx = d.nx, logn = d.log2nx, F = (int)d.n_fields, hn1 = nx / 2 + 1, tid = (int)threadIdx.x;
  const int nt = (int)blockDim.x;
  if (!F) return;
  const int rows = d1_rows(F), SB = d1_batch_of(nx, F, ns, (int)gridDim.y), ss = nx + 33;
  const int ps = logn > 5 ? logn - 5 : 31;
  double2* z = reinterpret_cast<double2*>(smem_raw);
  double2* X = z + SB * rows * ss;
  const double2* tw = reinterpret_cast<const double2*>(ws + d.off_tw_x);
  const double* raw = d1_raw(d, ws, sc);
  double* prod = d1_products(d, ws, sc);
  const int64_t np = d1q3_products(nx, F);
  for (uint32_t b0 = blockIdx.y * SB; b0 < ns; b0 += gridDim.y * SB) {
    const int nb = (int)min((uint32_t)SB, ns - b0), nq = nb * rows;             // samples, packed rows
    const bool last = b0 + nb == ns;
    // bit-reversed load of the packed rows (and, in the last batch, the fields of the last sample)
    for (int i = tid; i < nq * nx; i += nt) {
      const int q = i >> logn, x = i & (nx - 1), b = q / rows, fa = 2 * (q - b * rows);
      const double* g = raw + (int64_t)(b0 + b) * 3 * nx + x;
      const double g0 = g[0], g1 = g[nx], g2 = g[2 * nx];
      double2 v;
      v.x = d1q3_field(d, d.field_id[fa], g0, g1, g2);
      v.y = fa + 1 < F ? d1q3_field(d, d.field_id[fa + 1], g0, g1, g2) : 0.0;
      if (last && b == nb - 1) {
        double* f = reinterpret_cast<double*>(ws + d.off_fields) + (int64_t)fa * nx + x;
        f[0] = v.x;
        if (fa + 1 < F) f[nx] = v.y;
      }
      const int e = brev(x, logn);
      if (FLB_INB(q < SB * rows && e < nx, 181)) z[q * ss + e + (e >> ps)] = v;
    }
    __syncthreads();
    dit_fft<double>(z, logn, nq, ss, tw, 1, ps);
    // X_f(k) of every sample: [b][F][hn1]
    for (int i = tid; i < nq * hn1; i += nt) {
      const int q = i / hn1, k = i - q * hn1, b = q / rows, fa = 2 * (q - b * rows);
      const int km = (nx - k) & (nx - 1);
      const double2 Zk = z[q * ss + k + (k >> ps)], Zm = z[q * ss + km + (km >> ps)];
      double2* o = X + ((int64_t)b * F + fa) * hn1 + k;
      o[0] = make_double2(0.5 * (Zk.x + Zm.x), 0.5 * (Zk.y - Zm.y));
      if (fa + 1 < F) o[hn1] = make_double2(0.5 * (Zk.y + Zm.y), 0.5 * (Zm.x - Zk.x));
    }
    __syncthreads();
    // one item per (pair, sample, k), then the k = 0 values
    const int body = d.n_pairs * nb * hn1;
    for (int it = tid; it < body + nb * F; it += nt) {
      if (it < body) {
        const int row = it / hn1, k = it - row * hn1, pr = row / nb, b = row - pr * nb;
        const int fa = d.pair_a[pr], fb = d.pair_b[pr];
        if (!FLB_INB(fa < F && fb < F, 182)) continue;
        const double2 A = X[((int64_t)b * F + fa) * hn1 + k], B = X[((int64_t)b * F + fb) * hn1 + k];
        double* o = prod + (b0 + b) * np + d1q3_pair_first(nx, pr, fa, fb);
        if (fa == fb) {
          o[k] = A.x * A.x + A.y * A.y;
        } else {                                                                 // X_a X_b^*
          o[2 * k] = A.x * B.x + A.y * B.y;
          o[2 * k + 1] = A.y * B.x - A.x * B.y;
        }
      } else {
        const int b = (it - body) / F, f = it - body - b * F;
        prod[(b0 + b + 1) * np - F + f] = X[((int64_t)b * F + f) * hn1].x;
      }
    }
    __syncthreads();
  }
}

// The same for large batches, whose warps hide each other's loads.
constexpr int kD1SumThreads = 64, kD1SumBatch = 32, kD1SumStages = 3;
__global__ void __launch_bounds__(kD1SumThreads)
k_d1q3_sums_many(const ReplicaDesc* __restrict__ descs, char* __restrict__ ws, const D1Scratch sc, uint32_t ns) {
  d1q3_add_products(descs[blockIdx.x], ws, sc, ns, (int)blockIdx.y, (int)gridDim.y);
}

// The same for the last chunk of a small batch, where the time is a thread's chain of dependent additions,
// 31 ns each at best: their products come by asynchronous copies up to 64 samples ahead into slots of the
// thread's own.  About 43 ns a sample (loads into registers 8 ahead 58, 32 ahead 50); its shared memory
// leaves an SM 8 warps, so that batches of 2000 x 1024 sites, four fields, would take 861 us a step for 730.
__global__ void __launch_bounds__(kD1SumThreads)
k_d1q3_sums(const ReplicaDesc* __restrict__ descs, char* __restrict__ ws, const D1Scratch sc, uint32_t ns) {
  __shared__ double ring[kD1SumStages][kD1SumBatch][kD1SumThreads];
  const ReplicaDesc& d = descs[blockIdx.x];
  const int64_t np = d1q3_products(d.nx, (int)d.n_fields);
  const int64_t i = (int64_t)blockIdx.y * kD1SumThreads + threadIdx.x;
  if (!d.n_fields || i >= np) return;
  const double* p = d1_products(d, ws, sc) + i;
  const uint32_t batches = (ns + kD1SumBatch - 1) / kD1SumBatch;
  auto fetch = [&](uint32_t b) {                    // (one group per batch, empty past the end)
    if (b < batches) {
#pragma unroll
      for (int u = 0; u < kD1SumBatch; ++u) {
        const uint32_t s = b * kD1SumBatch + u;
        if (s < ns)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::
                       "r"((uint32_t)__cvta_generic_to_shared(&ring[b % kD1SumStages][u][threadIdx.x])), "l"(p + s * np) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (uint32_t b = 0; b < kD1SumStages - 1; ++b) fetch(b);
  double* sum = d1_sum(d, ws, i, np);
  double acc = *sum;
  for (uint32_t b = 0; b < batches; ++b) {
    fetch(b + kD1SumStages - 1);                    // into the slots that batch b - 1 has left
    asm volatile("cp.async.wait_group %0;" :: "n"(kD1SumStages - 1) : "memory");
    const double (*r)[kD1SumThreads] = ring[b % kD1SumStages];
    const uint32_t left = ns - b * kD1SumBatch;
    if (left >= kD1SumBatch) {
      double v[kD1SumBatch];
#pragma unroll
      for (int u = 0; u < kD1SumBatch; ++u) v[u] = r[u][threadIdx.x];
#pragma unroll
      for (int u = 0; u < kD1SumBatch; ++u) acc = __dadd_rn(acc, v[u]);
    } else {
      for (uint32_t u = 0; u < left; ++u) acc = __dadd_rn(acc, r[u][threadIdx.x]);
    }
  }
  *sum = acc;
}

cudaError_t set_d1q3_runs_smem() {
  const int m = 200 * 1024;
  cudaError_t e = cudaFuncSetAttribute(k_d1q3_steps<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, m);
  if (!e) e = cudaFuncSetAttribute(k_d1q3_steps<kD1SitesPerThread>, cudaFuncAttributeMaxDynamicSharedMemorySize, m);
  if (!e) e = cudaFuncSetAttribute(k_d1q3_sample, cudaFuncAttributeMaxDynamicSharedMemorySize, m);
  return e;
}

// additions by themselves: a run's last chunk where d1q3_sums_beside, every chunk of a large batch
cudaError_t launch_d1q3_sums(const ReplicaDesc* descs, const D1Group& g, char* ws, const D1Scratch& sc, uint32_t ns,
                             bool beside, cudaStream_t st, int* launches) {
  if (!ns) return cudaSuccess;
  const dim3 grid(g.n, (unsigned)((g.max_products + kD1SumThreads - 1) / kD1SumThreads));
  if (beside) k_d1q3_sums<<<grid, kD1SumThreads, 0, st>>>(descs + g.first, ws, sc, ns);
  else k_d1q3_sums_many<<<grid, kD1SumThreads, 0, st>>>(descs + g.first, ws, sc, ns);
  const cudaError_t e = cudaGetLastError();
  if (!e) ++*launches;
  return e;
}

static int d1_block(const D1Group& g) { return g.max_nx <= 1024 ? (g.max_nx + 31) & ~31 : 1024; }
static int64_t d1_sum_parts(const D1Group& g) { return (g.max_products + d1_block(g) - 1) / d1_block(g); }
// do a chunk's additions run beside the next chunk's steps (on SMs that the steps leave idle)?
bool d1q3_sums_beside(const D1Group& g, int sms) { return g.n * (1 + d1_sum_parts(g)) <= sms; }

// One chunk: steps t0 .. t0 + n_steps - 1 of a group (max_nx <= kD1MaxSites), with the noise of noise_steps
// steps drawn before them (at most sc.steps; 0: the noise area has it from sc.noise_first on), sampled
// every `every` (0: not), and the additions of the group's chunk before (*pending samples).  With `beside`
// (the context's only group, and d1q3_sums_beside) the chunk leaves its own additions in *pending, for
// the next one or launch_d1q3_sums; else they follow at once.  Adds the launches to *launches.  Replicas are in the grids' x
// (up to 2^31 - 1; y ends at 65535).  A launch that is refused ends the chunk: its first kernel writes
// scratch alone, so the state stays as it was when that one fails.
cudaError_t launch_d1q3_chunk(const ReplicaDesc* descs, const D1Group& g, char* ws, const D1Scratch& sc, uint32_t every,
                              uint64_t t0, uint32_t n_steps, uint32_t noise_steps, bool beside, int sms,
                              cudaStream_t st, uint32_t* pending, int* launches) {
  descs += g.first;
  cudaError_t e;
  if (noise_steps) {
    const int64_t most = (int64_t)noise_steps * g.max_nx;
    k_d1q3_noise<<<dim3(g.n, (unsigned)std::min<int64_t>((most + 255) / 256, 8 * (int64_t)sms)), 256, 0, st>>>(
        descs, ws, sc, t0, noise_steps);
    if ((e = cudaGetLastError())) return e;
    ++*launches;
  }
  const size_t smem = d1q3_steps_smem(g.max_nx);
  const int block = d1_block(g), parts = (int)d1_sum_parts(g);
  const int grid = g.n + (*pending ? g.n * parts : 0);              // (left pending only where that is at most sms)
  if (g.max_nx <= 1024)
    k_d1q3_steps<1><<<grid, block, smem, st>>>(descs, ws, sc, every, t0, n_steps, g.n, *pending, parts);
  else
    k_d1q3_steps<kD1SitesPerThread><<<grid, block, smem, st>>>(descs, ws, sc, every, t0, n_steps, g.n, *pending, parts);
  if ((e = cudaGetLastError())) return e;
  ++*launches;
  *pending = 0;
  uint32_t ns = 0;
  if (every && g.sample_smem) {             // samples at the steps t in [t0, t0 + n_steps) with t % every == 0
    const uint64_t first = (t0 + every - 1) / every * every;
    if (first < t0 + n_steps) ns = (uint32_t)((t0 + n_steps - 1 - first) / every + 1);
  }
  if (!ns) return cudaSuccess;
  const int blocks = std::max(1, sms / g.n);                   // of the sampling kernel, per replica
  k_d1q3_sample<<<dim3(g.n, blocks), kD1SampleThreads, g.sample_smem, st>>>(descs, ws, sc, ns);
  if ((e = cudaGetLastError())) return e;
  ++*launches;
  if (!beside) return launch_d1q3_sums(descs - g.first, g, ws, sc, ns, false, st, launches);
  *pending = ns;
  return cudaSuccess;
}

}  // namespace flb
