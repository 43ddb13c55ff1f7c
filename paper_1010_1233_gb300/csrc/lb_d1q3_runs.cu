// Runs of D1Q3 steps in FP64 with their correlator sampling.
//
// The lattices are small (L = 64 in the D1Q3 workload) and each step needs the one before, so a
// run is a chain; what can be taken off the chain decides its time.  One block that did the
// noise, the step, the row transforms and the pair sums of every step in turn took 10 - 12 us a
// step at L = 64 with every step sampled, nearly all of it latency between barriers.  Here only
// the step itself is serial, and the rest runs on the whole GPU before and after it, a chunk of
// steps at a time:
//   k_d1q3_noise   the noise of every (step, site) of the chunk
//   k_d1q3_steps   one block per replica: pull and collide, 15 FP64 instructions a site, one barrier
//                  a step; the noise is loaded two steps ahead; at a sample the pulled
//                  populations go to memory
//   k_d1q3_sample  row transforms of all samples (radix-2 passes of fft_common.cuh, two fields
//                  packed per complex row) and per-block sums of the pair products
//   k_d1q3_finish  adds the blocks' sums to the replica's, in block order
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

// Scratch of a replica (ReplicaDesc::off_d1_*): noise [chunk][nx], pulled populations [samples][3][nx],
// partial sums [run.blocks][items] (double2).
__global__ void __launch_bounds__(256)
k_d1q3_noise(const ReplicaDesc* __restrict__ descs, char* __restrict__ ws, uint64_t t0, uint32_t n_steps) {
  const ReplicaDesc& d = descs[blockIdx.x];
  const int nx = d.nx;
  double* out = reinterpret_cast<double*>(ws + d.off_d1_noise);
  const uint32_t n = n_steps * (uint32_t)nx;
  for (uint32_t i = blockIdx.y * blockDim.x + threadIdx.x; i < n; i += gridDim.y * blockDim.x) {
    const uint32_t s = i / (uint32_t)nx;
    out[i] = d1q3_noise(d, (int)(i - s * nx), (uint32_t)(t0 + s));
  }
}

// SPT sites per thread (x = tid + k blockDim): steps t0 .. t0 + n_steps - 1 of replica blockIdx.x,
// state from the buffer of parity t0 & 1 to that of (t0 + n_steps) & 1.
template <int SPT>
__global__ void __launch_bounds__(1024)
k_d1q3_steps(const ReplicaDesc* __restrict__ descs, char* __restrict__ ws, D1Run run, uint64_t t0, uint32_t n_steps) {
  extern __shared__ __align__(16) double pop[];              // [2][3][nx]
  const ReplicaDesc& d = descs[blockIdx.x];
  const int nx = d.nx, tid = (int)threadIdx.x, nt = (int)blockDim.x;
  const double* src = reinterpret_cast<const double*>(ws + d.off_pop[t0 & 1]);
  for (int i = tid; i < 3 * nx; i += nt) pop[i] = src[i];
  const D1Coef coef(d);
  const double* noise = reinterpret_cast<const double*>(ws + d.off_d1_noise);
  double* raw = reinterpret_cast<double*>(ws + d.off_d1_raw);
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
  uint32_t wait = run.every && d.n_fields ? (uint32_t)((run.every - t0 % run.every) % run.every) : 0xFFFFFFFFu;
  __syncthreads();
  for (uint32_t s = 0; s < n_steps; ++s) {
    const double* in = pop + (s & 1) * 3 * nx;
    double* out = pop + ((s & 1) ^ 1) * 3 * nx;
    const bool sample = wait == 0;
    wait = sample ? run.every - 1 : wait - 1;
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
// chunk's ns samples and leaves its sums in partial row g; the block of the last batch writes its fields.
__global__ void __launch_bounds__(kD1SampleThreads)
k_d1q3_sample(const ReplicaDesc* __restrict__ descs, char* __restrict__ ws, uint32_t ns) {
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
  const double* raw = reinterpret_cast<const double*>(ws + d.off_d1_raw);
  const int items = (int)d1q3_items(d);
  double2* part = reinterpret_cast<double2*>(ws + d.off_d1_part) + (int64_t)blockIdx.y * items;
  bool first = true;
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
    for (int it = tid; it < items; it += nt) {
      double2 acc = first ? make_double2(0.0, 0.0) : part[it];
      const int pr = it / hn1, k = it - pr * hn1;
      if (pr < d.n_pairs) {
        const double2* xa = X + (int64_t)d.pair_a[pr] * hn1 + k;
        const double2* xb = X + (int64_t)d.pair_b[pr] * hn1 + k;
        const bool cross = d.pair_a[pr] != d.pair_b[pr];
        if (!FLB_INB(d.pair_a[pr] < F && d.pair_b[pr] < F, 182)) continue;
        for (int b = 0; b < nb; ++b) {
          const double2 A = xa[(int64_t)b * F * hn1], Bv = xb[(int64_t)b * F * hn1];
          acc.x += A.x * Bv.x + A.y * Bv.y;                                      // X_a X_b^*
          if (cross) acc.y += A.y * Bv.x - A.x * Bv.y;
        }
      } else {                                                                   // X_f(0) of field it - n_pairs hn1
        const int f = it - d.n_pairs * hn1;
        for (int b = 0; b < nb; ++b) acc.x += X[((int64_t)b * F + f) * hn1].x;
      }
      part[it] = acc;
    }
    first = false;
    __syncthreads();
  }
}

// The partial sums of blocks 0 .. used - 1 (used: the blocks that had a batch), a warp per item, added
// to the replica's sums.
__global__ void __launch_bounds__(256)
k_d1q3_finish(const ReplicaDesc* __restrict__ descs, char* __restrict__ ws, uint32_t ns, int blocks) {
  const ReplicaDesc& d = descs[blockIdx.x];
  const int F = (int)d.n_fields, hn1 = d.nx / 2 + 1, lane = (int)threadIdx.x & 31;
  if (!F) return;
  const int SB = d1_batch_of(d.nx, F, ns, blocks), items = (int)d1q3_items(d);
  const int used = (int)min((uint32_t)blocks, (ns + SB - 1) / SB);
  const double2* part = reinterpret_cast<const double2*>(ws + d.off_d1_part);
  for (int it = (int)(blockIdx.y * blockDim.x + threadIdx.x) >> 5; it < items; it += (int)(gridDim.y * blockDim.x) >> 5) {
    double2 v = make_double2(0.0, 0.0);
    for (int g = lane; g < used; g += 32) {
      const double2 p = part[(int64_t)g * items + it];
      v.x += p.x;
      v.y += p.y;
    }
    for (int o = 16; o > 0; o >>= 1) {
      v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
      v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    if (lane) continue;
    const int pr = it / hn1, k = it - pr * hn1;
    if (pr < d.n_pairs) {
      if (d.pair_a[pr] == d.pair_b[pr]) {
        reinterpret_cast<double*>(ws + d.pair_off[pr])[k] += v.x;
      } else {
        double2* a = reinterpret_cast<double2*>(ws + d.pair_off[pr]) + k;
        const double2 s = *a;
        *a = make_double2(s.x + v.x, s.y + v.y);
      }
    } else {
      reinterpret_cast<double*>(ws + d.off_mean0)[it - d.n_pairs * hn1] += v.x;
    }
  }
}

cudaError_t set_d1q3_runs_smem() {
  const int m = 200 * 1024;
  cudaError_t e = cudaFuncSetAttribute(k_d1q3_steps<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, m);
  if (!e) e = cudaFuncSetAttribute(k_d1q3_steps<kD1SitesPerThread>, cudaFuncAttributeMaxDynamicSharedMemorySize, m);
  if (!e) e = cudaFuncSetAttribute(k_d1q3_sample, cudaFuncAttributeMaxDynamicSharedMemorySize, m);
  return e;
}

// One chunk: steps t0 .. t0 + n_steps - 1 (n_steps <= run.chunk) of all replicas (run.max_nx <=
// kD1MaxSites); adds the launches to *launches.  Replicas are in the grids' x (up to 2^31 - 1; y ends at
// 65535).  A launch that is refused ends the chunk: its first kernel writes scratch alone, so the
// state stays as it was when that one fails.
cudaError_t launch_d1q3_chunk(const ReplicaDesc* descs, int n_reps, char* ws, const D1Run& run, uint64_t t0,
                              uint32_t n_steps, int sms, cudaStream_t st, int* launches) {
  const int64_t most = (int64_t)n_steps * run.max_nx;
  cudaError_t e;
  k_d1q3_noise<<<dim3(n_reps, (unsigned)std::min<int64_t>((most + 255) / 256, 8 * (int64_t)sms)), 256, 0, st>>>(
      descs, ws, t0, n_steps);
  if ((e = cudaGetLastError())) return e;
  ++*launches;
  const size_t smem = d1q3_steps_smem(run.max_nx);
  if (run.max_nx <= 1024)
    k_d1q3_steps<1><<<n_reps, (run.max_nx + 31) & ~31, smem, st>>>(descs, ws, run, t0, n_steps);
  else
    k_d1q3_steps<kD1SitesPerThread><<<n_reps, 1024, smem, st>>>(descs, ws, run, t0, n_steps);
  if ((e = cudaGetLastError())) return e;
  ++*launches;
  uint32_t ns = 0;
  if (run.every) {             // samples at the steps t in [t0, t0 + n_steps) with t % every == 0
    const uint64_t first = (t0 + run.every - 1) / run.every * run.every;
    if (first < t0 + n_steps) ns = (uint32_t)((t0 + n_steps - 1 - first) / run.every + 1);
  }
  if (!ns || !run.sample_smem) return cudaSuccess;
  k_d1q3_sample<<<dim3(n_reps, run.blocks), kD1SampleThreads, run.sample_smem, st>>>(descs, ws, ns);
  if ((e = cudaGetLastError())) return e;
  ++*launches;
  k_d1q3_finish<<<dim3(n_reps, (unsigned)((run.max_items + 7) / 8)), 256, 0, st>>>(descs, ws, ns, run.blocks);
  if ((e = cudaGetLastError())) return e;
  ++*launches;
  return cudaSuccess;
}

}  // namespace flb
