// The D1Q3 step of one site, shared by the per-step kernel (lb_step.cu), the fused FP32
// multi-step kernel (lb_d1q3_fused.cu) and the FP64 run kernels (lb_d1q3_runs.cu).
//
// D1Q3: v = (0, +1, -1), w = (2/3, 1/6, 1/6), moments 1, sqrt3 v, (3 v^2 - 1)/sqrt2 (the
// projection of the D2Q9 basis).  Pull streaming (Eq. 1) from src, relaxation of the one
// non-conserved moment M^2 towards its equilibrium (Eqs. 5, 10) plus the noise of Eq. 8
// (noise mode 2: with the local density), back transform into dst; src and dst hold the
// populations as [3][nx].  With SAMPLE the pre-collision fields (moment minus its
// reference, or u - u0) of the replica's slots go to fields[slot * nx + x].
//
// FP64: the same update with every operation spelled out (d1q3_collide), so that the run kernels
// (lb_d1q3_runs.cu) and the per-step kernel give the same states.
#pragma once
#include "flb_internal.cuh"

namespace flb {

// Collision of one FP64 site.  With S = sqrt2, M^2 = S (g1 + g2) - g0 / S and M^{2,0} = 3 rho u^2 / S,
// the moment change is D = (M^{2,0} - M^2) / tau + xi, and the populations move by -2 H, H, H with
// H = S D / 6 = (j^2 / rho / 2 - (g1 + g2) / 3 + g0 / 6) / tau + S xi / 6.  GB300 issues an FP64
// instruction of a warp every 64 cycles, so their number is the time of a step: 15 here.  The
// quotient is j^2 y (1 + e + e^2) with y the hardware's FP32 reciprocal of rho (22 bits, from the FP32
// sum of the narrowed populations, beside the FP64 sums) and e = 1 - rho y: e^3 < 2^-63.
struct D1Coef {
  double a, b, c;          // 1 / (2 tau), -1 / (3 tau), 1 / (6 tau)
  double local;            // noise mode 2: sqrt(1 / rho0), else 0
  bool is_local;
  __device__ __forceinline__ explicit D1Coef(const ReplicaDesc& d) {
    const double it = d.dco[kCoInvTau + 2];
    a = 0.5 * it;
    b = -(1.0 / 3.0) * it;
    c = (1.0 / 6.0) * it;
    is_local = d.noise_mask && d.noise_mode == 2;
    local = is_local ? sqrt(1.0 / d.dco[kCoRho0]) : 0.0;
  }
};

// FP64 to FP32 and back on the integer pipes, for magnitudes of 2^-100 .. 2^100 (truncating)
__device__ __forceinline__ float narrow64(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  return __uint_as_float((hi & 0x80000000u) | (((hi & 0x7FFFFFFFu) - 0x38000000u) << 3) | (lo >> 29));
}
// 2^-100 <= x < 2^100 (positive), an integer comparison
__device__ __forceinline__ bool ordinary64(double x) {
  return (uint32_t)__double2hiint(x) - ((1023u - 100u) << 20) < (200u << 20);
}
__device__ __forceinline__ double widen64(float x) {
  const uint32_t b = __float_as_uint(x);
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + 0x38000000u)), (int)(b << 29));
}

// out of line, like divide64
static __device__ __noinline__ double d1q3_sqrt(double a) { return sqrt(a); }

// q / rho, rho = g0 + s.  The estimate needs populations and their FP32 sum of ordinary size (and
// a sum without cancellation, so that it is good to 22 bits); anything else divides.
__device__ __forceinline__ double d1q3_quotient(double q, double rho, double g0, double g1, double g2) {
  const float f = narrow64(g0) + (narrow64(g1) + narrow64(g2));
  if (!(ordinary64(g0) && ordinary64(g1) && ordinary64(g2))) return divide64(q, rho);
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
  const double y0 = widen64(y);
  const double e = __fma_rn(-rho, y0, 1.0), qy = __dmul_rn(q, y0);
  return __fma_rn(qy, __fma_rn(e, e, e), qy);
}

// h = S amp N / 6 (d1q3_noise)
__device__ __forceinline__ void d1q3_collide(double (&g)[3], const D1Coef& k, double h) {
  const double s = __dadd_rn(g[1], g[2]), rho = __dadd_rn(g[0], s), j = __dsub_rn(g[1], g[2]);
  if (k.is_local) h *= d1q3_sqrt(rho) * k.local;
  const double r = __fma_rn(k.b, s, __fma_rn(k.c, g[0], h));
  const double H = __fma_rn(k.a, d1q3_quotient(__dmul_rn(j, j), rho, g[0], g[1], g[2]), r);
  g[0] = __fma_rn(-2.0, H, g[0]);
  g[1] = __dadd_rn(g[1], H);
  g[2] = __dadd_rn(g[2], H);
}

// sqrt2 / 6 of the noise amp N of site x at a step
__device__ __forceinline__ double d1q3_noise(const ReplicaDesc& d, int x, uint32_t step) {
  if (!d.noise_mask) return 0.0;
  const uint4 w = philox4x32_10((uint32_t)x, step, 0u, d.stream, d.seed_lo, d.seed_hi);
  double n0, n1;
  box_muller(w.x, w.y, n0, n1);
  return __dmul_rn(__dmul_rn(1.4142135623730950488 / 6.0, d.dco[kCoAmp + 2]), n0);
}

// sampled field fid (minus its reference) of the pre-collision populations
__device__ __forceinline__ double d1q3_field(const ReplicaDesc& d, int fid, double g0, double g1, double g2) {
  const double s = __dadd_rn(g1, g2), j = __dsub_rn(g1, g2);
  switch (fid) {
    case 0: return __dsub_rn(__dadd_rn(g0, s), d.dco[kCoMref]);
    case 1: return __fma_rn(1.7320508075688772935, j, -d.dco[kCoMref + 1]);
    case 2: return __dsub_rn(__fma_rn(1.4142135623730950488, s, __dmul_rn(-0.70710678118654752440, g0)),
                             d.dco[kCoMref + 2]);
    default: return __dsub_rn(d1q3_quotient(j, __dadd_rn(g0, s), g0, g1, g2), d.dco[kCoU0x]);
  }
}

template <typename R, bool DEV, bool SAMPLE>
__device__ __forceinline__ void d1q3_site(const ReplicaDesc& d, const R* __restrict__ src, R* __restrict__ dst,
                                          R* __restrict__ fields, int nx, int x, uint32_t step) {
  if (!FLB_INB(x >= 0 && x < nx, 111)) return;
  if constexpr (sizeof(R) == 8) {
    double g[3] = {src[x], src[nx + (x == 0 ? nx - 1 : x - 1)], src[2 * nx + (x == nx - 1 ? 0 : x + 1)]};
    if constexpr (SAMPLE)
      for (int slot = 0; slot < (int)d.n_fields && FLB_INB(slot < kMaxFields, 111); ++slot)
        fields[(int64_t)slot * nx + x] = d1q3_field(d, d.field_id[slot], g[0], g[1], g[2]);
    d1q3_collide(g, D1Coef(d), d1q3_noise(d, x, step));
    dst[x] = g[0];
    dst[nx + x] = g[1];
    dst[2 * nx + x] = g[2];
    return;
  }
  const R g0 = src[x];
  const R g1 = src[nx + (x == 0 ? nx - 1 : x - 1)];
  const R g2 = src[2 * nx + (x == nx - 1 ? 0 : x + 1)];
  const R sum = g0 + (g1 + g2);
  const R rho = DEV ? coef<R>(d, kCoRho0) + sum : sum;
  const R j = g1 - g2;
  const R u = j / rho;
  const R S2 = (R)1.4142135623730950488, IS2 = (R)0.70710678118654752440;
  const R M2 = S2 * (g1 + g2) - IS2 * g0;
  const R E2 = (R)3 * IS2 * rho * u * u;
  if constexpr (SAMPLE) {
    const R mom[3] = {sum, (R)1.7320508075688772935 * j, M2};
    for (int slot = 0; slot < (int)d.n_fields; ++slot) {
      if (!FLB_INB(slot < kMaxFields, 111)) break;
      const int fid = d.field_id[slot];
      const R val = fid < 3 ? mom[fid] - coef<R>(d, kCoMref + fid) : u - coef<R>(d, kCoU0x);
      fields[(int64_t)slot * nx + x] = val;
    }
  }
  R D2 = (E2 - M2) * coef<R>(d, kCoInvTau + 2);
  if (d.noise_mask) {
    const uint4 w = philox4x32_10((uint32_t)x, step, 0u, d.stream, d.seed_lo, d.seed_hi);
    R n0, n1;
    box_muller(w.x, w.y, n0, n1);
    if (d.noise_mode == 2) n0 *= sqrt(rho / coef<R>(d, kCoRho0));    // local density in Eq. 8
    D2 += coef<R>(d, kCoAmp + 2) * n0;
  }
  dst[x] = g0 - (R)(2.0 / 3.0) * IS2 * D2;
  const R side = (R)(1.0 / 6.0) * S2 * D2;
  dst[nx + x] = g1 + side;
  dst[2 * nx + x] = g2 + side;
}

}  // namespace flb
