// Per-cell arithmetic of the fused step (moments, pseudopotential, force,
// collision), shared by every step kernel.
#pragma once
#include "lbm_internal.cuh"

namespace lbm {
namespace {

constexpr float kW1 = 1.0f / 9.0f, kW5 = 1.0f / 36.0f, kW0 = 4.0f / 9.0f;

// The per-cell arithmetic is written once for V = float (one cell) and
// V = float2 (two neighbouring cells, packed FP32 instructions), with every
// operation an explicitly rounded add, multiply or fused multiply-add, so all
// kernels produce bitwise the same populations.

__device__ __forceinline__ float exp2_approx(float a) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ float rcp_approx(float a) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
// 1 / rho for a density 0 < rho < 2^102, given as b = 2^24 rho, by two
// Newton-Raphson steps r <- r + r (1 - b r) on the hardware's approximation. The
// residual is exact in a fused operation, so the second step rounds correctly
// (Markstein, IBM J. Res. Dev. 34, 1990): equal to __frcp_rn(rho) for every such
// density, without its branch. The approximation flushes subnormal arguments, and
// b is none; powers of two change no rounding, and the second one stands in for
// the sign. (Other densities are faults, see report_faults.)
constexpr float kRhoScale = 16777216.0f;

__device__ __forceinline__ float recip(float b) {
  float n = rcp_approx(-b);
  n = __fmaf_rn(n, __fmaf_rn(b, n, 1.0f), n);
  n = __fmaf_rn(n, __fmaf_rn(b, n, 1.0f), n);
  return __fmul_rn(n, -kRhoScale);
}

template <typename V>
struct VOps;

template <>
struct VOps<float> {
  static __device__ __forceinline__ float set(float a) { return a; }
  static __device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
  static __device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
  static __device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
  static __device__ __forceinline__ float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
  static __device__ __forceinline__ float rcp(float b) { return recip(b); }
  static __device__ __forceinline__ float ex2(float a) { return exp2_approx(a); }
  static __device__ __forceinline__ void note(float b, uint32_t& worst) { worst = __viaddmax_u32(__float_as_uint(b), 0xffffffffu, worst); }
};

// The pair type uses the packed two-wide FP32 instructions of sm_100 and
// later, whose rounding per component is that of the scalar intrinsics; a
// difference is the fused b * (-1) + a, which rounds once, exactly as a - b.
template <>
struct VOps<float2> {
  static __device__ __forceinline__ float2 set(float a) { return make_float2(a, a); }
  static __device__ __forceinline__ float2 add(float2 a, float2 b) { return __fadd2_rn(a, b); }
  static __device__ __forceinline__ float2 sub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
  static __device__ __forceinline__ float2 mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
  static __device__ __forceinline__ float2 fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
  static __device__ __forceinline__ float2 rcp(float2 b) {
    // the negative of the reciprocal throughout: a sign flips no rounding,
    // and 1 - b r is then one fused operation
    const float2 one = set(1.f);
    float2 n = make_float2(rcp_approx(-b.x), rcp_approx(-b.y));
    n = fma(n, fma(b, n, one), n);
    n = fma(n, fma(b, n, one), n);
    return mul(n, set(-kRhoScale));
  }
  static __device__ __forceinline__ float2 ex2(float2 a) { return make_float2(exp2_approx(a.x), exp2_approx(a.y)); }
  static __device__ __forceinline__ void note(float2 b, uint32_t& worst) {
    VOps<float>::note(b.x, worst);
    VOps<float>::note(b.y, worst);
  }
};

// Eq. 11: rho and j from the nine incoming populations.
template <typename V>
__device__ __forceinline__ void moments9(const V f[Q], V& rho, V& jx, V& jy) {
  using O = VOps<V>;
  rho = O::add(O::add(O::add(f[0], f[1]), O::add(f[2], f[3])), O::add(O::add(f[4], f[5]), O::add(f[6], f[7])));
  rho = O::add(rho, f[8]);
  const V d57 = O::sub(f[5], f[7]), d86 = O::sub(f[8], f[6]);
  jx = O::add(O::sub(f[1], f[3]), O::add(d57, d86));
  jy = O::add(O::sub(f[2], f[4]), O::sub(d57, d86));
}

// Full density from the summed stored values: for 16-bit storage (DEV) the
// stored values are deviations g_i = f_i - w_i rho_ref, whose sum is
// rho - rho_ref (the weights sum to one).
template <bool DEV, typename V>
__device__ __forceinline__ V full_rho(V rho_raw, const StepParams& p) {
  return DEV ? VOps<V>::add(VOps<V>::set(p.rho_ref), rho_raw) : rho_raw;
}

// Eq. 30, e^x as 2^(x log2 e): psi is what it is with __expf, for every density.
template <typename V>
__device__ __forceinline__ V psi_of(V rho, const StepParams& p) {
  using O = VOps<V>;
  const V x = O::mul(rho, O::set(-p.inv_rho0));
  return O::mul(O::set(p.rho0), O::sub(O::set(1.0f), O::ex2(O::mul(x, O::set(1.4426950408889634f)))));
}

// Eq. 22 with the barrier substitution: s[i] holds psi(x + e_i), or psi(x)
// where the edge is blocked.
template <typename V>
__device__ __forceinline__ void force_of(const V s[Q], V psi_c, float G, V& Fx, V& Fy) {
  using O = VOps<V>;
  const V w1 = O::set(kW1), w5 = O::set(kW5);
  const V d57 = O::sub(s[5], s[7]), d86 = O::sub(s[8], s[6]);
  const V sx = O::fma(w1, O::sub(s[1], s[3]), O::mul(w5, O::add(d57, d86)));
  const V sy = O::fma(w1, O::sub(s[2], s[4]), O::mul(w5, O::sub(d57, d86)));
  const V gp = O::mul(O::set(-G), psi_c);
  Fx = O::mul(gp, sx);
  Fy = O::mul(gp, sy);
}

// Eqs. 39-40 (u_eq = (j + tau F)/rho), Eq. 14 evaluated by opposite pairs,
// Eq. 18 (BGK). f holds the incoming stored values and receives the outgoing
// ones. With DEV the values are deviations from w_i rho_ref: j is unchanged
// (sum e_i w_i = 0) and the equilibrium deviation is
// w_i (rho - rho_ref - 1.5 rho u^2 + rho (3 e.u + 4.5 (e.u)^2)).
// The density enters as b = 2^24 rho (recip); with DEV one fused operation gives
// it from the summed deviations in place of rho, so the scale costs nothing there.
template <bool TAU_ONE, bool DEV, typename V>
__device__ __forceinline__ void collide(V f[Q], V rho_raw, V jx, V jy, V Fx, V Fy, const StepParams& p, uint32_t& worst) {
  using O = VOps<V>;
  const V b = DEV ? O::fma(rho_raw, O::set(kRhoScale), O::set(p.rho_ref * kRhoScale)) : O::mul(rho_raw, O::set(kRhoScale));
  const V ir = O::rcp(b);
  // tau stays a multiplier at tau = 1 too: a packed add of the product gp s
  // (force_of) and j would be contracted to one rounding, unlike the scalar one
  const V tau = O::set(p.tau);
  const V ux = O::mul(O::fma(tau, Fx, jx), ir);
  const V uy = O::mul(O::fma(tau, Fy, jy), ir);
  O::note(b, worst);
  const V uu = O::fma(ux, ux, O::mul(uy, uy));
  constexpr float k = DEV ? 1.0f / kRhoScale : 1.0f;
  const V rho = DEV ? b : rho_raw;  // times k
  const V a = DEV ? O::fma(O::mul(O::set(-1.5f * k), rho), uu, rho_raw) : O::mul(rho, O::fma(O::set(-1.5f), uu, O::set(1.0f)));
  const V r3 = O::mul(O::set(3.0f * k), rho), r45 = O::mul(O::set(4.5f * k), rho);
  const V w1 = O::set(kW1), w5 = O::set(kW5);
  V feq[Q];
  feq[0] = O::mul(O::set(kW0), a);
  {
    const V s = O::fma(O::mul(r45, ux), ux, a), t = O::mul(r3, ux);
    feq[1] = O::mul(w1, O::add(s, t));
    feq[3] = O::mul(w1, O::sub(s, t));
  }
  {
    const V s = O::fma(O::mul(r45, uy), uy, a), t = O::mul(r3, uy);
    feq[2] = O::mul(w1, O::add(s, t));
    feq[4] = O::mul(w1, O::sub(s, t));
  }
  {
    const V e = O::add(ux, uy);
    const V s = O::fma(O::mul(r45, e), e, a), t = O::mul(r3, e);
    feq[5] = O::mul(w5, O::add(s, t));
    feq[7] = O::mul(w5, O::sub(s, t));
  }
  {
    const V e = O::sub(uy, ux);
    const V s = O::fma(O::mul(r45, e), e, a), t = O::mul(r3, e);
    feq[6] = O::mul(w5, O::add(s, t));
    feq[8] = O::mul(w5, O::sub(s, t));
  }
  const V om = O::set(p.inv_tau);
#pragma unroll
  for (int i = 0; i < Q; ++i) f[i] = TAU_ONE ? feq[i] : O::fma(O::sub(feq[i], f[i]), om, f[i]);
}

// A step kernel tracks `worst`, the largest bits(b) - 1 (as unsigned) of the
// scaled densities b it collided: a density that is not in (0, 1e30) - zero,
// negative, NaN or infinite - has the largest values, at one operation per cell.
__device__ __forceinline__ void report_faults(uint32_t worst, int* flags) {
  if (worst >= __float_as_uint(1e30f * kRhoScale) - 1u) atomicOr(flags + FLAG_NUMERIC, 1);
}

}  // namespace
}  // namespace lbm
