// Device-pointer entry point of the correlator sampler (Eqs. 11-12): FFT and FP64
// pair accumulation of caller-provided real fields, without a simulation context.
// Uses the kernels of spectra.cu; the per-call plan (descriptor, block tables,
// twiddles, row-transformed spectra) lives in caller-provided scratch memory.
#include <algorithm>
#include <cstring>

#include "flb_internal.cuh"
#include "spectra_plan.cuh"

namespace flb {

int fft_rows_smem(int precision, int nx, int most);
int fft_cols_smem(int precision, int F, int ny, int ncol);
cudaError_t set_fft_smem_limits();
void launch_fft_rows(int precision, const ReplicaDesc* descs, const int64_t* vb_begin, int n_reps,
                     int64_t n_vblocks, char* ws, int grid, int smem, int most, cudaStream_t st, int slot, int paths,
                     int sms);
void launch_fft_cols(int precision, const ReplicaDesc* descs, const int64_t* vb_begin, int n_reps,
                     int64_t n_vblocks, char* ws, int ncol, cudaStream_t st, const TimeCorr& tc, int paths,
                     int nslots, int max_fields, int max_len, int max_pairs, int sms, bool split);
int launch_fft_cols_t(int precision, const ReplicaDesc* descs, const int64_t* vb_begin, int n_reps, int64_t n_vblocks,
                      char* ws, cudaStream_t st, int paths, int slot, int smem, int sms);
void launch_pair_sums(int precision, const ReplicaDesc* descs, const int64_t* vb_begin, int n_reps, int64_t n_vblocks,
                      char* ws, int ncol, int max_fields, int nslots, cudaStream_t st, const TimeCorr& tc, int sms);
void launch_fft_cols_a(int precision, const ReplicaDesc* descs, const int64_t* vb_begin, int n_reps,
                       int64_t n_vblocks, char* ws, int ncol, int grid, int block, int smem, cudaStream_t st,
                       int paths, int slot, int sms);

static inline int64_t a256(int64_t x) { return (x + 255) & ~int64_t(255); }

int spectra_plan(int precision, int nx, int ny, int F, SpectraPlan& P) {
  memset(&P, 0, sizeof P);
  if (precision != FLB_FP64 && precision != FLB_FP32_DEV) return set_error(FLB_EINVAL, "unknown precision %d", precision);
  if (F < 1 || F > kMaxFields) return set_error(FLB_EINVAL, "n_fields must be in 1..%d", kMaxFields);
  auto pow2 = [](int v) { return v > 0 && (v & (v - 1)) == 0; };
  if (!pow2(nx) || !pow2(ny) || nx < 2) return set_error(FLB_EINVAL, "nx, ny must be powers of two, nx >= 2");
  if (fft_rows_smem(precision, nx, kRowsPairs) > 227 * 1024) return set_error(FLB_EINVAL, "nx = %d too long for the row FFT", nx);
  const int l1 = column_split(precision, F, ny);
  int ly = 0;
  while ((1 << ly) < ny) ++ly;
  int lx = 0;
  while ((1 << lx) < nx) ++lx;
  const int len = std::max(1 << l1, ny >> l1);
  if (fft_cols_smem(precision, F, len, 1) > kColsSmemBudget)
    return set_error(FLB_EINVAL, "ny = %d too long for the column FFT with %d fields", ny, F);
  const int64_t rs = precision == FLB_FP64 ? 8 : 4;
  const int cs = (int)(2 * rs);
  ReplicaDesc& d = P.desc;
  d.nx = nx; d.ny = ny; d.log2nx = lx; d.log2ny = ly; d.q = 9;
  d.n_fields = F;
  for (int f = 0; f < F; ++f) d.field_id[f] = f;
  int np = 0;
  for (int a = 0; a < F; ++a)
    for (int b = a; b < F; ++b) { d.pair_a[np] = a; d.pair_b[np] = b; ++np; }
  d.n_pairs = np;
  d.half_nx = nx / 2 + 1;
  d.wpitch = (d.half_nx + 1) & ~1;
  d.log2n1 = l1;
  P.ncol = kColsMax;
  while (P.ncol > 1 && fft_cols_smem(precision, F, len, P.ncol) > kColsSmemBudget) P.ncol >>= 1;
  P.rows_most = kRowsPairs;
  while (P.rows_most > 1 && rows_blocks(precision, nx, F, ny, P.rows_most) < kRowsMinBlocks) P.rows_most >>= 1;
  P.rows_smem = fft_rows_smem(precision, nx, P.rows_most);
  P.cols_smem = fft_cols_smem(precision, F, len, P.ncol);
  const int64_t tiles = (d.half_nx + P.ncol - 1) / P.ncol;
  P.n_vb_rows = rows_blocks(precision, nx, F, ny, P.rows_most);
  P.n_vb_cols = tiles << l1;
  P.n_vb_cols_a = cols_a_blocks(precision, l1, F, d.half_nx, ny, P.ncol);
  int64_t off = 0;
  P.off_desc = off; off = a256(off + (int64_t)sizeof(ReplicaDesc));
  P.off_vb = off; off = a256(off + 8 * 3);
  P.off_tw_x = off; off = a256(off + (int64_t)(nx / 2) * cs + 16);
  P.off_tw_y = off; off = a256(off + (int64_t)(ny / 2) * cs + 16);
  d.spec_tiled = spec_tiled_ok(precision, nx, ny, l1) ? 1 : 0;
  P.off_spec = off; off = a256(off + spec_elems(d) * cs);
  P.scratch_bytes = (size_t)off;
  int64_t sums = 0;
  for (int pr = 0; pr < np; ++pr) sums += (int64_t)ny * d.half_nx * (d.pair_a[pr] == d.pair_b[pr] ? 1 : 2);
  P.n_sum_doubles = sums;
  return FLB_OK;
}

// One launch prepares a call: block 0 stores the plan's descriptor and block tables (so no
// host-to-device copy and no host staging buffer is involved), the others the twiddle tables
// exp(-2 pi i m / n), m < n / 2, of nx and ny.
template <typename R>
__global__ void __launch_bounds__(256) k_store_plan(const __grid_constant__ ReplicaDesc d, ReplicaDesc* dst, int64_t* vb) {
  if (blockIdx.x == 0) {
    const uint4* src = reinterpret_cast<const uint4*>(&d);
    for (int i = threadIdx.x; i < (int)(sizeof(ReplicaDesc) / 16); i += blockDim.x) reinterpret_cast<uint4*>(dst)[i] = src[i];
    if (threadIdx.x < 3) vb[threadIdx.x] = 0;
    return;
  }
  char* base = reinterpret_cast<char*>(dst);              // offsets are relative to the scratch
  const int hx = d.nx / 2, hy = d.ny / 2;
  const int m = ((int)blockIdx.x - 1) * (int)blockDim.x + (int)threadIdx.x;
  if (m >= hx + hy) return;
  cplx<R>* tw = reinterpret_cast<cplx<R>*>(base + (m < hx ? d.off_tw_x : d.off_tw_y));
  const int k = m < hx ? m : m - hx, n = m < hx ? d.nx : d.ny;
  double sn, cs;
  sincospi(2.0 * (double)k / (double)n, &sn, &cs);
  tw[k].x = (R)cs;
  tw[k].y = (R)(-sn);
}

int spectra_launch(int precision, SpectraPlan& P, char* scratch, const void* fields, double* pair_sums,
                   double* mean0, cudaStream_t st) {
  ReplicaDesc& d = P.desc;
  // offsets are relative to the scratch base
  const uintptr_t base = (uintptr_t)scratch;
  d.off_fields = (int64_t)((uintptr_t)fields - base);
  d.off_spec = P.off_spec;
  d.off_tw_x = P.off_tw_x;
  d.off_tw_y = P.off_tw_y;
  d.off_mean0 = (int64_t)((uintptr_t)mean0 - base);
  int64_t doff = 0;
  for (int pr = 0; pr < d.n_pairs; ++pr) {
    d.pair_off[pr] = (int64_t)((uintptr_t)(pair_sums + doff) - base);
    doff += (int64_t)d.ny * d.half_nx * (d.pair_a[pr] == d.pair_b[pr] ? 1 : 2);
  }
  cudaError_t e = set_fft_smem_limits();
  if (e != cudaSuccess) return set_error(FLB_ECUDA, "smem limits: %s", cudaGetErrorString(e));
  ReplicaDesc* ddesc = reinterpret_cast<ReplicaDesc*>(scratch + P.off_desc);     // (off_desc = 0: the scratch's start)
  int64_t* vb = reinterpret_cast<int64_t*>(scratch + P.off_vb);
  const int prep = 1 + (d.nx / 2 + d.ny / 2 + 255) / 256;
  if (precision == FLB_FP64) k_store_plan<double><<<prep, 256, 0, st>>>(d, ddesc, vb);
  else k_store_plan<float><<<prep, 256, 0, st>>>(d, ddesc, vb);
  int sms = 1, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int gr = (int)std::min<int64_t>(P.n_vb_rows, (int64_t)sms * 8);
  launch_fft_rows(precision, ddesc, vb, 1, P.n_vb_rows, scratch, gr, P.rows_smem, P.rows_most, st, 0,
                  rows16(precision, d.nx) ? 1 << (d.log2nx - 12) : kColsGeneric, sms);
  if (P.n_vb_cols_a) {
    const int ga = (int)std::min<int64_t>(P.n_vb_cols_a, (int64_t)sms * 8);
    launch_fft_cols_a(precision, ddesc, vb + 1, 1, P.n_vb_cols_a, scratch, P.ncol, ga, kColsBlock, P.cols_smem, st,
                      cols16_b(1 << d.log2n1) ? cols16_b(1 << d.log2n1) : kColsGeneric, 0, sms);
  }
  const int paths = precision != FLB_FP64 && cols16_b(d.ny >> d.log2n1) ? cols16_b(d.ny >> d.log2n1) : kColsGeneric;
  if (!d.log2n1 && (int64_t)d.ny * d.half_nx >= kSplitPoints) {
    launch_fft_cols_t(precision, ddesc, vb + 2, 1, cols_t_blocks(precision, d), scratch, st, paths, 0, cols_t_smem(precision, d), sms);
    launch_pair_sums(precision, ddesc, vb + 2, 1, pair_blocks(d, P.ncol), scratch, P.ncol, (int)d.n_fields, 1, st,
                     TimeCorr{}, sms);
  } else {
    launch_fft_cols(precision, ddesc, vb + 2, 1, P.n_vb_cols, scratch, P.ncol, st, TimeCorr{}, paths, 1,
                    (int)d.n_fields, std::max(1 << d.log2n1, d.ny >> d.log2n1), d.n_pairs, sms, false);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return set_error(FLB_ECUDA, "spectra launch: %s", cudaGetErrorString(e));
  return FLB_OK;
}

}  // namespace flb

using namespace flb;

extern "C" {

int flb_spectra_scratch_bytes(int precision, int nx, int ny, int n_fields, size_t* bytes_out, size_t* n_sums_out) {
  SpectraPlan P;
  const int rc = spectra_plan(precision, nx, ny, n_fields, P);
  if (rc) return rc;
  if (bytes_out) *bytes_out = P.scratch_bytes;
  if (n_sums_out) *n_sums_out = (size_t)P.n_sum_doubles;
  return FLB_OK;
}

int flb_spectra_accumulate(int precision, int nx, int ny, int n_fields, const void* fields_dev,
                           double* pair_sums_dev, double* mean0_dev, void* scratch_dev, size_t scratch_bytes,
                           void* cuda_stream) {
  SpectraPlan P;
  int rc = spectra_plan(precision, nx, ny, n_fields, P);
  if (rc) return rc;
  if (!fields_dev || !pair_sums_dev || !mean0_dev || !scratch_dev) return set_error(FLB_EINVAL, "NULL pointer");
  if (((uintptr_t)scratch_dev) & 255) return set_error(FLB_EINVAL, "scratch must be 256-byte aligned");
  if (scratch_bytes < P.scratch_bytes)
    return set_error(FLB_ENOMEM, "scratch %zu bytes < required %zu", scratch_bytes, P.scratch_bytes);
  return spectra_launch(precision, P, static_cast<char*>(scratch_dev), fields_dev, pair_sums_dev, mean0_dev,
                        static_cast<cudaStream_t>(cuda_stream));
}

}  // extern "C"
