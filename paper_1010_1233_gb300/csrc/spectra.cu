// Correlator sampling (Eqs. 11-12): 2D discrete Fourier transform of the
// sampled real fields with a hand-written radix-2 FFT, and FP64 accumulation
// of X_a(k) X_b(k)^* for every sampled field pair on the half spectrum
// kx in [0, nx/2] (the other half follows from X(-k) = X(k)^* for real fields).
//
// Pass 1 (rows): two real rows (consecutive (field, row) units) are packed as one
// complex row z = X_a + i X_b, transformed along x in shared memory, and unpacked
// into the transforms of both rows, X_a(kx) = (Z(kx) + Z(-kx)^*)/2,
// X_b(kx) = (Z(kx) - Z(-kx)^*)/(2i).
// Pass 2 (columns): tiles of columns of every field are transformed along y in
// shared memory and the pair products are added to the FP64 sums.  Columns too
// long for shared memory use the four-step split ny = N1 N2, y = N2 y1 + y2,
// ky = k1 + N1 k2:  X(ky) = sum_y2 W_N2^(y2 k2) W_N^(y2 k1) sum_y1 W_N1^(y1 k1) x(y);
// pass 2a does the inner length-N1 transforms and the W_N^(y2 k1) twiddle in
// place (rows N2 y1 + y2 -> N2 k1 + y2), pass 2b the outer length-N2 transforms.
#include <algorithm>
#include "spectra_acc.cuh"

namespace flb {

// Pass 1: one block per (replica, group of rows_per_block(nx, most) packed pairs of row units).
//
// Each pass of the transform is a few dozen instructions between two barriers, so what
// bounds it is how many rows an SM works on at a time.  With one pair per block of nx / 2
// threads only nx / 8 threads had work in the radix-8 and radix-16 passes, and a batched
// launch sized its blocks for the longest row.  256 threads and up to 2048 points per block
// keep every thread busy and 4 blocks on an SM (64 registers): 64 replicas of 64^2 .. 512^2
// (3 fields) 153 -> 70 us, 3 x 1024 x 2048 42 -> 24 us.
template <typename R>
__global__ void __launch_bounds__(kRowsBlock, sizeof(R) == 4 ? 4 : 2)
k_fft_rows(const ReplicaDesc* __restrict__ descs, const int64_t* __restrict__ vb_begin,
                           int n_reps, int64_t n_vblocks, char* __restrict__ ws, int slot, int most) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C<R>* z = reinterpret_cast<C<R>*>(smem_raw);
  const int tid = (int)threadIdx.x, nt = (int)blockDim.x;
  for (int64_t vb = blockIdx.x; vb < n_vblocks; vb += gridDim.x) {
    const int r = find_rep(vb_begin, n_reps, vb);
    const ReplicaDesc& d = descs[r];
    if (sizeof(R) == 4 && rows16_nx(d.nx)) continue;   // k_fft_rows16's row
    // pair p packs the row units u = 2 p and u + 1 (unit u: field u / ny, row u % ny; ny is a
    // power of two), so an odd field count leaves at most one half-empty transform
    const int nx = d.nx, logn = d.log2nx, hn = nx >> 1;
    const int64_t units = (int64_t)d.n_fields << d.log2ny, pairs = (units + 1) >> 1;
    const int P = rows_per_block(nx, most);
    const int64_t p0 = (vb - vb_begin[r]) * P;
    const int np = (int)min((int64_t)P, pairs - p0);           // this block's pairs, sequences of z
    const int ss = rows_seq_stride(nx);
    const R* fields = reinterpret_cast<const R*>(ws + d.off_fields) + 2 * p0 * nx;   // unit u starts at u nx
    const int n_units = (int)min((int64_t)2 * np, units - 2 * p0);
    const int ps = logn > 5 ? logn - 5 : 31;        // 32 pad slots per row
    const C<R>* tw = reinterpret_cast<const C<R>*>(ws + d.off_tw_x);
    // the rows of this block's next group into L2 while this one is transformed
    if (tid == 0 && vb + gridDim.x < n_vblocks) {
      const int64_t vbn = vb + gridDim.x;
      const int rn = find_rep(vb_begin, n_reps, vbn);
      const ReplicaDesc& dn = descs[rn];
      const int64_t un = 2 * (vbn - vb_begin[rn]) * rows_per_block(dn.nx, most);
      const int64_t left = ((int64_t)dn.n_fields << dn.log2ny) - un;
      const R* fn = reinterpret_cast<const R*>(ws + dn.off_fields) + un * dn.nx;
      const int64_t bytes = min((int64_t)2 * rows_per_block(dn.nx, most), left) * dn.nx * (int64_t)sizeof(R);
      if (left > 0 && bytes % 16 == 0 && (reinterpret_cast<uintptr_t>(fn) & 15) == 0)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(fn), "r"((uint32_t)bytes) : "memory");
    }
    if (logn >= 3) {
      // item (pair, x0), x0 < nx/8, loads x0 + j nx/8 (j < 8, coalesced): after bit reversal
      // these are elements t = brev3(j) of the group m = brev(x0) of the first three stages,
      // which run in registers before the group is stored
      const int n8 = nx >> 3;
      for (int it = tid; it < np * n8; it += nt) {
        const int k = it >> (logn - 3), x0 = it & (n8 - 1);
        const R* xa = fields + (int64_t)(2 * k) * nx;
        const bool has_b = 2 * k + 1 < n_units;
        C<R> v[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          const int x = x0 + (((t & 1) << 2) | (t & 2) | ((t >> 2) & 1)) * n8;
          const bool in = FLB_INB(x >= 0 && x < nx && 2 * k < n_units, 131);
          v[t].x = in ? xa[x] : (R)0;
          v[t].y = has_b && in ? xa[nx + x] : (R)0;
        }
        dit_group<R, 3>(v, logn, 0, 0, tw, 1);
        const int i0 = brev(x0, logn - 3) << 3;
#pragma unroll
        for (int t = 0; t < 8; ++t)
          if (FLB_INB(i0 + t < nx, 132)) z[k * ss + i0 + t + ((i0 + t) >> ps)] = v[t];
      }
      __syncthreads();
      dit_fft<R, sizeof(R) == 4 ? 4 : 3>(z, logn, np, ss, tw, 1, ps, 3);   // FP32: four stages per pass
    } else {
      for (int it = tid; it < np << logn; it += nt) {
        const int k = it >> logn, x = it & (nx - 1);
        const R* xa = fields + (int64_t)(2 * k) * nx;
        C<R> v; v.x = xa[x]; v.y = 2 * k + 1 < n_units ? xa[nx + x] : (R)0;
        const int i = brev(x, logn);
        if (FLB_INB(i < nx && 2 * k < n_units, 132)) z[k * ss + i + (i >> ps)] = v;
      }
      __syncthreads();
      dit_fft<R>(z, logn, np, ss, tw, 1, ps);
    }
    // row u's half spectrum starts at u wpitch (the rows of all fields are contiguous)
    C<R>* spec = reinterpret_cast<C<R>*>(ws + d.off_spec + slot * d.spec_slot) + 2 * p0 * d.wpitch;
    const bool rows_ok = FLB_INB(2 * p0 + n_units <= units && hn < d.wpitch, 133);
    // items (pair, k < nx/2), then k = nx/2 of every pair
    const int body = np << (logn - 1);
    for (int it = tid; it < body + np && rows_ok; it += nt) {
      const int q = it < body ? it >> (logn - 1) : it - body, k = it < body ? it & (hn - 1) : hn;
      const int km = (nx - k) & (nx - 1);
      const C<R> Z = z[q * ss + k + (k >> ps)];
      const C<R> Zm = z[q * ss + km + (km >> ps)];
      C<R>* ra = spec + (int64_t)(2 * q) * d.wpitch + k;
      C<R> A; A.x = (R)0.5 * (Z.x + Zm.x); A.y = (R)0.5 * (Z.y - Zm.y);
      *ra = A;
      if (2 * q + 1 < n_units) {            // (Z - conj(Zm)) / (2i)
        C<R> B; B.x = (R)0.5 * (Z.y + Zm.y); B.y = (R)0.5 * (Zm.x - Z.x);
        ra[d.wpitch] = B;
      }
    }
    __syncthreads();
  }
}

// Pass 2a (four-step only): one block per (replica, y2, tile of ncol columns).
template <typename R>
__global__ void __launch_bounds__(kColsBlock, sizeof(R) == 4 ? 4 : 2)
k_fft_cols_a(const ReplicaDesc* __restrict__ descs, const int64_t* __restrict__ vb_begin,
                             int n_reps, int64_t n_vblocks, char* __restrict__ ws, int ncol, int slot) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C<R>* s = reinterpret_cast<C<R>*>(smem_raw);
  for (int64_t vb = blockIdx.x; vb < n_vblocks; vb += gridDim.x) {
    const int r = find_rep(vb_begin, n_reps, vb);
    const ReplicaDesc& d = descs[r];
    if (sizeof(R) == 4 && cols16_b(1 << d.log2n1)) continue;        // a register-resident kernel's block
    const int lc = 31 - __clz(ncol);                    // ncol is a power of two
    const int tiles = (d.half_nx + ncol - 1) >> lc;
    const int64_t local = vb - vb_begin[r];
    const int y2 = (int)(local / tiles);
    const int kx0 = (int)(local - (int64_t)y2 * tiles) << lc;
    const int ncl = min(ncol, d.half_nx - kx0);
    const int logn1 = d.log2n1, n1 = 1 << logn1, n2 = d.ny >> logn1, F = (int)d.n_fields;
    C<R>* spec = reinterpret_cast<C<R>*>(ws + d.off_spec + slot * d.spec_slot);
    const int64_t fplane = (int64_t)d.ny * d.wpitch;
    const int total = F * n1 * ncol;
    // the next tile of this block into L2 (one bulk prefetch per (field, y1) segment)
    if (vb + gridDim.x < n_vblocks) {
      const int64_t vbn = vb + gridDim.x;
      const int rn = find_rep(vb_begin, n_reps, vbn);
      const ReplicaDesc& dn = descs[rn];
      const int tn = (dn.half_nx + ncol - 1) >> lc;
      const int64_t ln = vbn - vb_begin[rn];
      const int y2n = (int)(ln / tn);
      const int kxn = (int)(ln - (int64_t)y2n * tn) << lc;
      const int ncn = min(ncol, dn.half_nx - kxn);
      const int l1n = dn.log2n1, n2n = dn.ny >> l1n;
      const uint32_t bytes = (uint32_t)(((ncn * (int)sizeof(C<R>)) + 15) & ~15);
      const C<R>* sp = reinterpret_cast<const C<R>*>(ws + dn.off_spec + slot * dn.spec_slot);
      const int64_t fpn = (int64_t)dn.ny * dn.wpitch;
      const int segs = (int)dn.n_fields << l1n;
      for (int i = threadIdx.x; i < segs; i += blockDim.x) {
        const int f = i >> l1n, y1 = i & ((1 << l1n) - 1);
        const C<R>* a = sp + f * fpn + (int64_t)(n2n * y1 + y2n) * dn.wpitch + kxn;
        if ((reinterpret_cast<uintptr_t>(a) & 15) == 0)
          asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(a), "r"(bytes) : "memory");
      }
    }
    // gather, four loads in flight per thread
    for (int i0 = threadIdx.x; i0 < total; i0 += 4 * blockDim.x) {
      C<R> v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * blockDim.x;
        const int c = i & (ncol - 1), y1 = (i >> lc) & (n1 - 1), f = i >> (lc + logn1);
        v[u].x = (R)0; v[u].y = (R)0;
        if (i < total && c < ncl && FLB_INB(f < F && n2 * y1 + y2 < d.ny && kx0 + c < d.half_nx, 151))
          v[u] = spec[f * fplane + (int64_t)(n2 * y1 + y2) * d.wpitch + kx0 + c];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * blockDim.x;
        const int c = i & (ncol - 1), y1 = (i >> lc) & (n1 - 1), f = i >> (lc + logn1);
        if (i < total && FLB_INB(f < F && c < ncol && brev(y1, logn1) < n1, 152))
          s[(f * ncol + c) * (n1 + 1) + brev(y1, logn1)] = v[u];
      }
    }
    __syncthreads();
    const C<R>* tw = reinterpret_cast<const C<R>*>(ws + d.off_tw_y);
    dit_fft<R>(s, logn1, F * ncol, n1 + 1, tw, n2);
    const int hn = d.ny >> 1;
    for (int i = threadIdx.x; i < total; i += blockDim.x) {
      const int c = i & (ncol - 1);
      const int k1 = (i >> lc) & (n1 - 1);
      const int f = i >> (lc + logn1);
      if (c >= ncl || !FLB_INB(f < F && n2 * k1 + y2 < d.ny && kx0 + c < d.half_nx, 151)) continue;
      const int e = y2 * k1;                       // < ny
      C<R> w = tw[e < hn ? e : e - hn];
      if (e >= hn) { w.x = -w.x; w.y = -w.y; }
      spec[f * fplane + (int64_t)(n2 * k1 + y2) * d.wpitch + kx0 + c] = cmul<R>(s[(f * ncol + c) * (n1 + 1) + k1], w);
    }
    __syncthreads();
  }
}

// Pass 2b: one block per (replica, k1, tile of w columns, group of pairs); all fields of the
// tile.  One-pass columns are the case N1 = 1.  vb_begin counts the layout's tiles of ncol
// columns, each cut as sp says (ColsSplit); split: one-pass replicas are k_pair_sums'.
template <typename R>
__global__ void __launch_bounds__(cols_block_max(sizeof(R)), 1)
k_fft_cols_acc(const ReplicaDesc* __restrict__ descs, const int64_t* __restrict__ vb_begin,
                               int n_reps, int64_t n_vblocks, char* __restrict__ ws, int ncol, ColsSplit sp,
                               TimeCorr tc, bool split) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C<R>* s = reinterpret_cast<C<R>*>(smem_raw);
  const int w = sp.w, lc = 31 - __clz(w), lsub = 31 - __clz(ncol) - lc;      // powers of two
  const int n_sub = sp.ps << lsub;
  for (int64_t v = blockIdx.x; v < n_vblocks * n_sub; v += gridDim.x) {
    const int64_t vb = v / n_sub;
    const int sub = (int)(v - vb * n_sub), pg = sub >> lsub;
    const int r = find_rep(vb_begin, n_reps, vb);
    const ReplicaDesc& d = descs[r];
    if (sizeof(R) == 4 && cols16_b(d.ny >> d.log2n1)) continue;     // a register-resident kernel's block
    if (split && !d.log2n1) continue;                               // k_pair_sums' replica
    const int tiles = (d.half_nx + ncol - 1) >> (lc + lsub);
    const int64_t local = vb - vb_begin[r];
    const int k1 = (int)(local / tiles);
    const int kx0 = ((int)(local - (int64_t)k1 * tiles) << (lc + lsub)) + ((sub & ((1 << lsub) - 1)) << lc);
    if (kx0 >= d.half_nx) continue;                     // past the last column
    const int logn1 = d.log2n1, n1 = 1 << logn1, logn2 = d.log2ny - logn1, n2 = d.ny >> logn1;
    const int F = (int)d.n_fields;
    const int ncl = min(w, d.half_nx - kx0);
    const C<R>* spec = reinterpret_cast<const C<R>*>(ws + d.off_spec);
    const int64_t fplane = (int64_t)d.ny * d.wpitch;
    // blocked pair sums: the layout tile's sums of every pair are one contiguous range, pulled
    // into L2 by bulk prefetches while the columns are loaded and transformed
    if (d.acc_ncol && sub == 0) prefetch_sums(d, ws, k1, kx0, ncol, tiles, n2);
    // smem layout: [field][column][n2]
    const int total = F * n2 * w;
    for (int i0 = threadIdx.x; i0 < total; i0 += 4 * blockDim.x) {   // four loads in flight
      C<R> v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * blockDim.x;
        const int c = i & (w - 1), y2 = (i >> lc) & (n2 - 1), f = i >> (lc + logn2);
        v[u].x = (R)0; v[u].y = (R)0;
        if (i < total && c < ncl && FLB_INB(f < F && n2 * k1 + y2 < d.ny && kx0 + c < d.half_nx, 161))
          v[u] = spec[f * fplane + (int64_t)(n2 * k1 + y2) * d.wpitch + kx0 + c];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * blockDim.x;
        const int c = i & (w - 1), y2 = (i >> lc) & (n2 - 1), f = i >> (lc + logn2);
        if (i < total && FLB_INB(f < F && c < w && brev(y2, logn2) < n2, 162))
          s[(f * w + c) * (n2 + 1) + brev(y2, logn2)] = v[u];
      }
    }
    __syncthreads();
    dit_fft<R>(s, logn2, F * w, n2 + 1, reinterpret_cast<const C<R>*>(ws + d.off_tw_y), n1);
    accumulate_tile<R, 0>(d, ws, s, n2 + 1, k1, kx0, ncl, w, ncol, tiles, pg, sp.ps);
    if (pg == 0) tile_tail<R, 0>(d, ws, s, n2 + 1, r, k1, kx0, ncl, w, tc, 1, 0);
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// One-pass columns (N1 = 1) of lattices with kSplitPoints or more half-spectrum points in the launch:
// the column transforms in place (k_fft_cols_t here, k_fft_cols_t16 in spectra_cols.cu), then the pair
// sums point by point (k_pair_sums).  The fused pass holds all fields of a tile in shared memory
// through the FP64 additions, so few warps were left to keep the sums' reads and writes in flight;
// apart, the transforms run one field per block and the sums stream at whole lines, for one more
// write and read of the spectrum.  us per sample, fused and apart: FP64 256^2 with 9 fields 70 -> 57,
// the 64-replica sweep 286 -> 231, 3 x 1024 x 2048 96 -> 73; whole runs: 256^2 with 9 fields FP32, 2000
// steps with 200 samples, 11.5 -> 10.5 ms.

// One block per (replica, field, tile of columns, cols_t_log2): the columns transformed over y in place.
template <typename R>
__global__ void __launch_bounds__(kColsBlock, sizeof(R) == 4 ? 4 : 2)
k_fft_cols_t(const ReplicaDesc* __restrict__ descs, const int64_t* __restrict__ vb_begin, int n_reps,
             int64_t n_vblocks, char* __restrict__ ws, int slot) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C<R>* s = reinterpret_cast<C<R>*>(smem_raw);
  for (int64_t vb = blockIdx.x; vb < n_vblocks; vb += gridDim.x) {
    const int r = find_rep(vb_begin, n_reps, vb);
    const ReplicaDesc& d = descs[r];
    if (d.log2n1 || (sizeof(R) == 4 && cols16_b(d.ny))) continue;      // another kernel's replica
    const int lw = cols_t_log2(d.ny, d.half_nx), w = 1 << lw, tiles = (d.half_nx + w - 1) >> lw;
    const int local = (int)(vb - vb_begin[r]), f = local / tiles;
    const int kx0 = (local - f * tiles) << lw, ncl = min(w, d.half_nx - kx0);
    const int logn = d.log2ny, n = d.ny, total = n << lw;
    C<R>* col = reinterpret_cast<C<R>*>(ws + d.off_spec + slot * d.spec_slot) + (int64_t)f * n * d.wpitch + kx0;
    for (int i0 = threadIdx.x; i0 < total; i0 += 4 * blockDim.x) {     // four loads in flight
      C<R> v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * blockDim.x, c = i & (w - 1), y = i >> lw;
        v[u].x = (R)0; v[u].y = (R)0;
        if (i < total && c < ncl && FLB_INB(y < n && kx0 + c < d.half_nx, 151)) v[u] = col[(int64_t)y * d.wpitch + c];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * blockDim.x, c = i & (w - 1), y = i >> lw;
        if (i < total && FLB_INB(brev(y, logn) < n, 152)) s[c * (n + 1) + brev(y, logn)] = v[u];
      }
    }
    __syncthreads();
    dit_fft<R>(s, logn, w, n + 1, reinterpret_cast<const C<R>*>(ws + d.off_tw_y), 1);
    for (int i = threadIdx.x; i < total; i += blockDim.x) {
      const int c = i & (w - 1), y = i >> lw;
      if (c < ncl) col[(int64_t)y * d.wpitch + c] = s[c * (n + 1) + y];
    }
    __syncthreads();
  }
}

// Pair sums of transformed fields: thread = one point of the sums' layout (and one group of field rows),
// X_f of all fields in registers, then per field a the pairs (a, b >= a), kPairBatch sums in flight.
// gs groups: group g takes the rows a = g, 2 gs - 1 - g, 2 gs + g, .. (rows a and F - 1 - a together
// have F + 1 pairs).  The first block of a replica also records the time-correlator ring entries and
// adds the k = 0 values.
// FM: the most fields of a replica the kernel is compiled for (its registers).
constexpr int kPairBatch = 4;
template <typename R, int FM>
__global__ void __launch_bounds__(kColsBlock, FM <= 3 ? (sizeof(R) == 4 ? 4 : 3) : 2)
k_pair_sums(const ReplicaDesc* __restrict__ descs, const int64_t* __restrict__ vb_begin, int n_reps,
            int64_t n_vblocks, char* __restrict__ ws, int ncol, int gs, int nslots, TimeCorr tc) {
  for (int64_t v = blockIdx.x; v < n_vblocks * gs; v += gridDim.x) {
    const int64_t vb = v / gs;
    const int grp = (int)(v - vb * gs);
    const int r = find_rep(vb_begin, n_reps, vb);
    const ReplicaDesc& d = descs[r];
    if (d.log2n1) continue;                             // the fused pass's replica
    const int F = (int)d.n_fields, hn = d.half_nx, ny = d.ny;
    const int64_t pt = (vb - vb_begin[r]) * kColsBlock + threadIdx.x;
    const C<R>* spec = reinterpret_cast<const C<R>*>(ws + d.off_spec);
    // (either spectrum layout, spec_index)
    const int64_t fplane = spec_index(d, 1, 0, 0), slot = d.spec_slot / (int64_t)sizeof(C<R>);
    if (vb == vb_begin[r] && grp == 0) {
      if (tc.base) {
        const int rs = (int)(tc.count[r] % (uint64_t)tc.n_lags);
        double2* ring = reinterpret_cast<double2*>(tc.base + d.off_tc_ring);
        for (int i = threadIdx.x; i < tc.n_k * F; i += blockDim.x) {
          const int j = i % tc.n_k, f = i / tc.n_k;
          if (!FLB_INB(tc.kx[j] < hn && tc.ky[j] < ny, 164)) continue;
          const C<R> X = spec[spec_index(d, f, tc.ky[j], tc.kx[j])];
          ring[((int64_t)rs * F + f) * tc.n_k + j] = make_double2((double)X.x, (double)X.y);
        }
      }
      if (threadIdx.x < F) {
        double* m0 = reinterpret_cast<double*>(ws + d.off_mean0) + threadIdx.x;
        double m = *m0;
        for (int k = 0; k < nslots; ++k) m += (double)spec[k * slot + threadIdx.x * fplane].x;
        *m0 = m;
      }
    }
    // the point's (ky, kx): blocked layout [tile][ky][c] (N1 = 1) or [ky][kx]
    int ky, kx;
    bool in;
    if (d.acc_ncol) {
      const int lc = 31 - __clz(ncol);
      const int64_t row = pt >> lc;
      const int tile = (int)(row >> d.log2ny);
      ky = (int)(row & (ny - 1));
      kx = (tile << lc) + (int)(pt & (ncol - 1));
      in = kx < hn;
    } else {
      ky = (int)((uint32_t)pt / (uint32_t)hn);          // fewer than 2^31 points
      kx = (int)(pt - (int64_t)ky * hn);
      in = ky < ny;
    }
    if (!in || !FLB_INB(ky < ny && kx < d.wpitch && pt < sum_limit(d, ncol, (hn + ncol - 1) / ncol), 165)) continue;
    const C<R>* p = spec + spec_index(d, 0, ky, kx);
    C<R> X0[FM], X1[FM];
#pragma unroll
    for (int f = 0; f < FM; ++f)
      if (f < F) {
        X0[f] = p[f * fplane];
        if (sizeof(R) == 4 && nslots > 1) X1[f] = p[slot + f * fplane];
      }
    int pr0 = 0;                                        // index of pair (a, a)
#pragma unroll
    for (int a = 0; a < FM; ++a) {
      if (a >= F) break;
      const int am = a % (2 * gs);
      if (am == grp || am == 2 * gs - 1 - grp) {
#pragma unroll
        for (int b0 = a; b0 < FM; b0 += kPairBatch) {
          double2 acc[kPairBatch];
#pragma unroll
          for (int u = 0; u < kPairBatch; ++u) {
            const int b = b0 + u;
            if (b >= FM || b >= F) break;
            const double* q = reinterpret_cast<const double*>(ws + d.pair_off[pr0 + b - a]);
            if (b == a) acc[u].x = q[pt];
            else acc[u] = load_sum2(q + 2 * pt);
          }
#pragma unroll
          for (int u = 0; u < kPairBatch; ++u) {
            const int b = b0 + u;
            if (b >= FM || b >= F) break;
            double* q = reinterpret_cast<double*>(ws + d.pair_off[pr0 + b - a]);
            // the product in the transform's precision, the sums in FP64, sample by sample
#pragma unroll
            for (int k = 0; k < (sizeof(R) == 4 ? 2 : 1); ++k) {
              if (k >= nslots) break;
              const C<R> Xa = k ? X1[a] : X0[a], Xb = k ? X1[b] : X0[b];
              if (b == a) {
                acc[u].x += widen(Xa.x * Xa.x + Xa.y * Xa.y);
              } else {
                acc[u].x += widen(Xa.x * Xb.x + Xa.y * Xb.y);     // X_a X_b^*
                acc[u].y += widen(Xa.y * Xb.x - Xa.x * Xb.y);
              }
            }
            if (b == a) q[pt] = acc[u].x;
            else store_sum2(q + 2 * pt, acc[u]);
          }
        }
      }
      pr0 += F - a;
    }
  }
}

// Time correlators, after the column pass of a sample: sums[tau][a][b][j] +=
// X_a(k_j, s) X_b(k_j, s - tau)^* for every lag with a sample s - tau in the ring
// (s = count), then (k_time_corr_advance) count += 1.  One item per (tau, a, b, j);
// blockIdx.y is the replica.
__global__ void k_time_corr(const ReplicaDesc* __restrict__ descs, TimeCorr tc) {
  const int r = blockIdx.y;
  const ReplicaDesc& d = descs[r];
  const int F = (int)d.n_fields, T = tc.n_lags, nk = tc.n_k;
  const uint64_t cnt = tc.count[r];
  const int slot = (int)(cnt % (uint64_t)T);
  const double2* ring = reinterpret_cast<const double2*>(tc.base + d.off_tc_ring);
  double2* sums = reinterpret_cast<double2*>(tc.base + d.off_tc_sums);
  const int64_t items = (int64_t)T * F * F * nk;
  for (int64_t it = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; it < items; it += (int64_t)gridDim.x * blockDim.x) {
    const int j = (int)(it % nk);
    const int64_t rest = it / nk;
    const int b = (int)(rest % F), a = (int)((rest / F) % F), tau = (int)(rest / ((int64_t)F * F));
    if ((uint64_t)tau > cnt) continue;                         // no sample s - tau yet
    const int old = (slot - tau + T) % T;
    const double2 xa = ring[((int64_t)slot * F + a) * nk + j];
    const double2 xb = ring[((int64_t)old * F + b) * nk + j];
    double2 v = sums[it];
    v.x += xa.x * xb.x + xa.y * xb.y;                          // X_a X_b^*
    v.y += xa.y * xb.x - xa.x * xb.y;
    sums[it] = v;
  }
}

__global__ void k_time_corr_advance(TimeCorr tc, int n_reps) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r < n_reps) tc.count[r] += 1;
}

template <typename R>
__global__ void k_twiddles(C<R>* tw, int n) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= n / 2) return;
  double sn, cs;
  sincospi(2.0 * (double)m / (double)n, &sn, &cs);
  C<R> v; v.x = (R)cs; v.y = (R)(-sn);
  tw[m] = v;
}

// ---------------------------------------------------------------------------
void launch_fft_cols_a16(int mask, const ReplicaDesc* descs, const int64_t* vb_begin, int n_reps, int64_t n_vblocks,
                         char* ws, int grid, cudaStream_t st, int slot);
void launch_fft_cols_acc16(int mask, const ReplicaDesc* descs, const int64_t* vb_begin, int n_reps, int64_t n_vblocks,
                           char* ws, int ncol, const ColsSplit& sp, int sms, int max_fields, cudaStream_t st,
                           const TimeCorr& tc, int nslots, bool split);
cudaError_t set_fft16_smem_limits();
void launch_fft_rows16(const ReplicaDesc* descs, const int64_t* vb_begin, int n_reps, int64_t n_vblocks, char* ws,
                       int grid, int nx, cudaStream_t st, int slot);
cudaError_t set_rows16_smem_limits();

void launch_twiddles(int precision, void* tw, int n, cudaStream_t st) {
  if (n < 2) return;
  const int half = n / 2;
  if (precision == FLB_FP64)
    k_twiddles<double><<<(half + 255) / 256, 256, 0, st>>>(reinterpret_cast<double2*>(tw), n);
  else
    k_twiddles<float><<<(half + 255) / 256, 256, 0, st>>>(reinterpret_cast<float2*>(tw), n);
}

// shared memory of the row pass for rows of nx: k_fft_rows16 holds nx / 2 complex values
// (one pad slot per 16), k_fft_rows its group of rows
int fft_rows_smem(int precision, int nx, int most) {
  if (rows16(precision, nx)) return (nx / 2 + nx / 32) * 8;
  return rows_per_block(nx, most) * rows_seq_stride(nx) * (precision == FLB_FP64 ? 16 : 8);
}
// the columns of every field of a tile, plus a table of up to 256 roots of unity
// (the register-resident passes of spectra_cols.cu)
int fft_cols_smem(int precision, int F, int ny, int ncol) { return (F * (ny + 1) * ncol + 256) * (precision == FLB_FP64 ? 16 : 8); }

cudaError_t set_fft_smem_limits() {
  cudaError_t e;
  const int maxb = 227 * 1024;
  // the transforms want shared memory, not L1 (a preference the CUDA runtime rounds to a supported split)
  const int carve = (int)cudaSharedmemCarveoutMaxShared;
  if ((e = cudaFuncSetAttribute(k_fft_rows<float>, cudaFuncAttributePreferredSharedMemoryCarveout, carve))) return e;
  if ((e = cudaFuncSetAttribute(k_fft_cols_a<float>, cudaFuncAttributePreferredSharedMemoryCarveout, carve))) return e;
  if ((e = cudaFuncSetAttribute(k_fft_cols_acc<float>, cudaFuncAttributePreferredSharedMemoryCarveout, carve))) return e;
  if ((e = cudaFuncSetAttribute(k_fft_rows<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, maxb))) return e;
  if ((e = cudaFuncSetAttribute(k_fft_rows<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, maxb))) return e;
  if ((e = cudaFuncSetAttribute(k_fft_cols_acc<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, maxb))) return e;
  if ((e = cudaFuncSetAttribute(k_fft_cols_a<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, maxb))) return e;
  if ((e = cudaFuncSetAttribute(k_fft_cols_a<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, maxb))) return e;
  if ((e = cudaFuncSetAttribute(k_fft_cols_acc<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, maxb))) return e;
  if ((e = cudaFuncSetAttribute(k_fft_cols_t<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, maxb))) return e;
  if ((e = cudaFuncSetAttribute(k_fft_cols_t<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, maxb))) return e;
  if ((e = set_rows16_smem_limits())) return e;
  return set_fft16_smem_limits();
}

// slot: the spectrum slot (0 or 1) the sample's transforms go to.  paths: kColsGeneric
// for the shared-memory kernel, bit b for k_fft_rows16 on rows of nx = 4096 << b (FP32).
// grid: blocks of the shared-memory kernel; the Stockham kernel takes at most two blocks
// per SM of the sms SMs (its blocks loop over their rows)
void launch_fft_rows(int precision, const ReplicaDesc* descs, const int64_t* vb_begin, int n_reps,
                     int64_t n_vblocks, char* ws, int grid, int smem, int most, cudaStream_t st, int slot, int paths,
                     int sms) {
  const int block = kRowsBlock;
  if (precision == FLB_FP64) {
    k_fft_rows<double><<<grid, block, smem, st>>>(descs, vb_begin, n_reps, n_vblocks, ws, slot, most);
    return;
  }
  if (paths & kColsGeneric) k_fft_rows<float><<<grid, block, smem, st>>>(descs, vb_begin, n_reps, n_vblocks, ws, slot, most);
  const int g16 = (int)std::min<int64_t>((int64_t)grid, 2 * (int64_t)sms);
  for (int b = 0; b < 4; ++b)
    if (paths & (1 << b)) launch_fft_rows16(descs, vb_begin, n_reps, n_vblocks, ws, g16, 4096 << b, st, slot);
}

// paths: kColsGeneric for the shared-memory kernel, bit B for the register-resident
// kernel of columns of 16 B (FP32 only; see cols16_b).  The register-resident pass-2a
// kernel takes one block per field of a (y2, tile) unit (cols_a_units), tiles of kColsA16
// columns; the shared-memory kernel tiles of ncol.
void launch_fft_cols_a(int precision, const ReplicaDesc* descs, const int64_t* vb_begin, int n_reps,
                       int64_t n_vblocks, char* ws, int ncol, int grid, int block, int smem, cudaStream_t st,
                       int paths, int slot, int sms) {
  if (precision == FLB_FP64) {
    k_fft_cols_a<double><<<grid, block, smem, st>>>(descs, vb_begin, n_reps, n_vblocks, ws, ncol, slot);
    return;
  }
  if (paths & kColsGeneric)
    k_fft_cols_a<float><<<grid, block, smem, st>>>(descs, vb_begin, n_reps, n_vblocks, ws, ncol, slot);
  // the pipelined kernel: its resident blocks (4 per SM) loop over their units
  launch_fft_cols_a16(paths & (kColsGeneric - 1), descs, vb_begin, n_reps, n_vblocks, ws,
                      (int)std::min<int64_t>((int64_t)grid, 4 * (int64_t)sms), st, slot);
}

void launch_fft_cols_t16(int mask, const ReplicaDesc* descs, const int64_t* vb_begin, int n_reps, int64_t n_vblocks,
                         char* ws, int grid, cudaStream_t st, int slot);

// Column transforms in place of the one-pass replicas (paths: the lengths among them, as in
// launch_fft_cols; smem: of the shared-memory kernel, cols_t_smem); returns the launches.
int launch_fft_cols_t(int precision, const ReplicaDesc* descs, const int64_t* vb_begin, int n_reps, int64_t n_vblocks,
                      char* ws, cudaStream_t st, int paths, int slot, int smem, int sms) {
  const int grid = (int)std::min<int64_t>(n_vblocks, 16 * (int64_t)sms);
  int launches = 0;
  if (precision == FLB_FP64 || (paths & kColsGeneric)) {
    if (precision == FLB_FP64)
      k_fft_cols_t<double><<<grid, kColsBlock, smem, st>>>(descs, vb_begin, n_reps, n_vblocks, ws, slot);
    else
      k_fft_cols_t<float><<<grid, kColsBlock, smem, st>>>(descs, vb_begin, n_reps, n_vblocks, ws, slot);
    ++launches;
  }
  if (precision != FLB_FP64) {
    launch_fft_cols_t16(paths & (kColsGeneric - 1), descs, vb_begin, n_reps, n_vblocks, ws, grid, st, slot);
    launches += __builtin_popcount(paths & (kColsGeneric - 1));
  }
  return launches;
}

void launch_pair_sums(int precision, const ReplicaDesc* descs, const int64_t* vb_begin, int n_reps, int64_t n_vblocks,
                      char* ws, int ncol, int max_fields, int nslots, cudaStream_t st, const TimeCorr& tc, int sms) {
  // groups of field rows where the points alone do not fill the GPU (half the fields at most)
  int gs = 1;
  while (2 * gs < max_fields && n_vblocks * gs < 4 * (int64_t)sms) ++gs;
  const int grid = (int)std::min<int64_t>(n_vblocks * gs, 32 * (int64_t)sms);
#define FLB_L(R, FM) k_pair_sums<R, FM><<<grid, kColsBlock, 0, st>>>(descs, vb_begin, n_reps, n_vblocks, ws, ncol, gs, nslots, tc)
#define FLB_LR(R) { if (max_fields <= 3) FLB_L(R, 3); else if (max_fields <= 6) FLB_L(R, 6); else FLB_L(R, kMaxFields); }
  if (precision == FLB_FP64) FLB_LR(double) else FLB_LR(float)
#undef FLB_LR
#undef FLB_L
}

// max_fields, max_len: the most fields and the longest column transform of a replica (the
// shared-memory kernel's launch holds them)
void launch_fft_cols(int precision, const ReplicaDesc* descs, const int64_t* vb_begin, int n_reps,
                     int64_t n_vblocks, char* ws, int ncol, cudaStream_t st, const TimeCorr& tc, int paths,
                     int nslots, int max_fields, int max_len, int max_pairs, int sms, bool split) {
  const ColsSplit sp = cols_split(precision, n_vblocks, ncol, max_fields * max_len, max_pairs, sms);
  if (precision == FLB_FP64 || (paths & kColsGeneric)) {    // one slot (the host folds samples only without it)
    const int smem = fft_cols_smem(precision, max_fields, max_len, sp.w);
    const int64_t nb = n_vblocks * (ncol / sp.w) * sp.ps;
    const int grid = (int)std::min<int64_t>(nb, 8 * (int64_t)sms);
    const int block = std::min(cols_threads(nb, sms, sp.w * max_len, smem), cols_block_max(precision == FLB_FP64 ? 8 : 4));
    if (precision == FLB_FP64)
      k_fft_cols_acc<double><<<grid, block, smem, st>>>(descs, vb_begin, n_reps, n_vblocks, ws, ncol, sp, tc, split);
    else
      k_fft_cols_acc<float><<<grid, block, smem, st>>>(descs, vb_begin, n_reps, n_vblocks, ws, ncol, sp, tc, split);
  }
  if (precision != FLB_FP64)
    launch_fft_cols_acc16(paths & (kColsGeneric - 1), descs, vb_begin, n_reps, n_vblocks, ws, ncol, sp, sms,
                          max_fields, st, tc, nslots, split);
}

void launch_time_corr(const ReplicaDesc* descs, int n_reps, int max_fields, const TimeCorr& tc, cudaStream_t st) {
  const int64_t items = (int64_t)tc.n_lags * max_fields * max_fields * tc.n_k;
  const int gx = (int)std::min<int64_t>((items + 255) / 256, 4096);
  k_time_corr<<<dim3(gx, n_reps), 256, 0, st>>>(descs, tc);
  k_time_corr_advance<<<(n_reps + 127) / 128, 128, 0, st>>>(tc, n_reps);
}

}  // namespace flb
