// fsmp_pe_kernel.cuh -- device code of the PE-space chain kernel, compiled by fsmp_pe.cu (the
// dynode charge model) and fsmp_pe_mix.cu (the MCP charge mixture), each instantiating its own
// kernels so that the two build in parallel.
//
// The FSMP chain in PE space, a warp or half warp per chain (arXiv 2403.03156, Sec. 2.4 and
// Appendix A.1, with the Woodbury identity applied to the whole of A).
//
// Sigma(z) = sigma_eps^2 I + sigma_q^2 A A^T with A = [a_1 .. a_N] (n x N). With
// r = sigma_eps^2 / sigma_q^2 and the N x N capacitance matrix C = r I + A^T A,
//   Sigma^-1 = (I - A C^-1 A^T) / sigma_eps^2,   log|Sigma| = n log sigma_eps^2 + log|C| - N log r.
// A chain keeps C^-1, v = C^-1 A^T y and the residual y = w - mu_q sum_k a_k. For a move with the
// columns a_- = a_k (a PE of z) and a_+ (a new position), and b = A^T a_+,
//   a_+^T Sigma^-1 a_+ = (|a_+|^2 - b^T C^-1 b) / sigma_eps^2,   a_+^T Sigma^-1 y = (a_+^T y - b^T v) / sigma_eps^2,
//   1 - sigma_q^2 a_k^T Sigma^-1 a_k = r C^-1_kk,                a_k^T Sigma^-1 y = v_k / sigma_q^2,
//   a_k^T Sigma^-1 a_+ = (C^-1 b)_k / sigma_q^2,
// the 2x2 quantities of Eqs. (16)-(18). With the MCP charge mixture (Appendix A.2) each PE k has
// its own mean mu_k, variance sigma_k^2 and r_k = sigma_eps^2 / sigma_k^2: C = diag(r_k) + A^T A,
// log|Sigma| = n log sigma_eps^2 + log|C| - sum_k log r_k, and sigma_q^2, r above become those of
// the PE concerned (the dynode model is the one-component case). Only the p PEs whose support
// overlaps a_+ have b != 0, so a
// proposal reads p^2 + O(p) entries of C^-1 and no n-vector beyond a_+'s support. An accepted move
// updates C^-1 by bordering (birth), a Schur-complement downdate (death) or both in one pass
// (update): O(N^2) instead of the O(n^2) of Sigma^-1. The charge summary is
// E[Q | z, w] = sum_k (mu_k + v_k). Inner products a_i^T a_j over the window come from the SER
// cross-correlation prefix table.
//
// Layout: a chain runs on a group of L consecutive lanes (L = 32: a warp; L = 16: two chains per
// warp, for chains with few PEs, where most of a step is work that every lane repeats); a CTA
// holds several independent chains and a group takes chains from a launch-wide counter. A chain of
// up to 32 PEs scores four steps at once (kSpec below). C^-1 sits
// in a per-chain shared-memory tile (the packed triangle of Ns PEs) while N <= Ns and moves to the
// chain's global slot (n_cap PEs) when a birth would exceed the tile. The counts of N after
// burn-in (for lambda_FSMP) sit in a global slot per chain.
//
// Precision. For PEs close in time C is nearly singular (eigenvalues down to r) and C^-1 holds
// entries near 1/r that cancel in b^T C^-1 b; stored in FP32 they cost about 1e-2 in log alpha per
// step. C^-1, v and b therefore carry twice the working precision: in FP32 mode float-float pairs
// (hi + lo, Dekker's exact product and Knuth's TwoSum) that run on the FP32 pipe -- an FP64
// instruction costs this part as much as 64 FP32 ones -- and in FP64 mode double-double pairs
// built the same way, so that a_+^T Sigma^-1 a_+ = (|a_+|^2 - b^T C^-1 b) / sigma_eps^2 keeps FP64
// accuracy where |a_+|^2 and b^T C^-1 b nearly cancel (chains with many overlapping PEs, and
// small r when a mixture component is wide). In FP32 mode the residual y,
// the SER and phi tables, the random draws and the 2x2 algebra are FP32, and C^-1, v, y, log|Sigma|
// and the log-likelihood are rebuilt from z in FP64 (Gauss-Jordan inversion of C, which is
// symmetric positive definite) every refresh_every accepted moves and at the end. Per step the
// random draws, proposal rules and acceptance tests are those of the Sigma^-1 kernel.
#pragma once
#include <math.h>

#include "fsmp_internal.h"

namespace fsmp {
namespace {

constexpr int kPeMaxThreads = 128;  // warps per CTA: at most 4
constexpr int kSub = 4;  // subgroups of a chain's lanes that score a step each (see kSpec)

// x, unknown to the compiler: keeps it from cloning a loop per value of a flag that is the same in
// all of its passes (the clones tripled the accept's code, and code size is what binds here).
__device__ __forceinline__ bool opaque(bool x) {
  int v = x;
  asm volatile("" : "+r"(v));
  return v != 0;
}

// The lanes of one chain: L consecutive lanes of a warp. Exchanges and reductions stay inside the
// group; gm is its lane mask. A step draws the random numbers of the next L steps (one per lane).
template <int L> struct Lanes {
  int sl;       // lane within the group
  int g;        // group within the warp
  unsigned gm;  // lane mask of the group
};
template <> struct Lanes<32> {  // a whole warp: the mask is a constant, which its shuffles need no code for
  int sl;
  static constexpr int g = 0;
  static constexpr unsigned gm = 0xffffffffu;
};
template <int L> __device__ __forceinline__ Lanes<L> pe_lanes() {
  static_assert(L == 32 || L == 16, "a chain runs on 32 or 16 lanes");
  const int lane = threadIdx.x & 31;
  Lanes<L> r;
  r.sl = lane & (L - 1);
  if constexpr (L != 32) {
    r.g = lane / L;
    r.gm = ((1u << L) - 1u) << (r.g * L);
  }
  return r;
}
// the group's lanes with p set, as bits 0 .. L-1
template <int L> __device__ __forceinline__ unsigned gballot(bool p, const Lanes<L> ln) {
  const unsigned b = __ballot_sync(ln.gm, p);
  if constexpr (L == 32) return b;
  else return (b >> (ln.g * L)) & ((1u << L) - 1u);
}

// ---------------------------------------------------------------- float-float / double-double arithmetic
// A value hi + lo with |lo| <= ulp(hi) / 2. TwoSum (Knuth) and the FMA-based exact product
// (Dekker) give the rounding error of one FP32 operation exactly; the pair operations below are
// the usual "sloppy" double-float forms (relative error about 2^-44).
struct ff {
  float hi, lo;
};
__device__ __forceinline__ ff ff_quick(float a, float b) {  // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return ff{s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ ff ff_add(ff x, ff y) {
  const float s = __fadd_rn(x.hi, y.hi);
  const float bb = __fsub_rn(s, x.hi);
  const float e = __fadd_rn(__fsub_rn(x.hi, __fsub_rn(s, bb)), __fsub_rn(y.hi, bb));
  return ff_quick(s, __fadd_rn(e, __fadd_rn(x.lo, y.lo)));
}
__device__ __forceinline__ ff ff_mul(ff x, ff y) {
  const float p = __fmul_rn(x.hi, y.hi);
  float e = __fmaf_rn(x.hi, y.hi, -p);
  e = __fmaf_rn(x.hi, y.lo, e);
  e = __fmaf_rn(x.lo, y.hi, e);
  return ff_quick(p, e);
}
__device__ __forceinline__ ff ff_neg(ff x) { return ff{-x.hi, -x.lo}; }

// The same pair arithmetic in FP64 (double-double, about 2^-100 relative error).
struct dd {
  double hi, lo;
};
__device__ __forceinline__ dd dd_quick(double a, double b) {  // |a| >= |b|
  const double s = __dadd_rn(a, b);
  return dd{s, __dsub_rn(b, __dsub_rn(s, a))};
}
__device__ __forceinline__ dd dd_add(dd x, dd y) {
  const double s = __dadd_rn(x.hi, y.hi);
  const double bb = __dsub_rn(s, x.hi);
  const double e = __dadd_rn(__dsub_rn(x.hi, __dsub_rn(s, bb)), __dsub_rn(y.hi, bb));
  return dd_quick(s, __dadd_rn(e, __dadd_rn(x.lo, y.lo)));
}
__device__ __forceinline__ dd dd_mul(dd x, dd y) {
  const double p = __dmul_rn(x.hi, y.hi);
  double e = __fma_rn(x.hi, y.hi, -p);
  e = __fma_rn(x.hi, y.lo, e);
  e = __fma_rn(x.lo, y.hi, e);
  return dd_quick(p, e);
}
__device__ __forceinline__ dd dd_neg(dd x) { return dd{-x.hi, -x.lo}; }

// The state arithmetic: C = dd (FP64 mode) or ff (FP32 mode). The plain FP64 forms serve the
// FP64 refresh.
__device__ __forceinline__ double cadd(double a, double b) { return a + b; }
__device__ __forceinline__ double csub(double a, double b) { return a - b; }
__device__ __forceinline__ double cmul(double a, double b) { return a * b; }
__device__ __forceinline__ double cfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double cneg(double a) { return -a; }
__device__ __forceinline__ double crcp(double a) { return 1.0 / a; }
__device__ __forceinline__ double cnum(double a) { return a; }   // to the scoring precision
__device__ __forceinline__ double c64(double a) { return a; }    // to FP64
__device__ __forceinline__ bool cnz(double a) { return a != 0.0; }
template <int L> __device__ __forceinline__ double cshfl_xor(double a, int o, unsigned gm) {
  return __shfl_xor_sync(gm, a, o, L);
}
template <int L> __device__ __forceinline__ double cshfl(double a, int src, unsigned gm) {
  return __shfl_sync(gm, a, src, L);
}
template <typename C> __device__ __forceinline__ C czero();
template <> __device__ __forceinline__ double czero<double>() { return 0.0; }

__device__ __forceinline__ dd cadd(dd a, dd b) { return dd_add(a, b); }
__device__ __forceinline__ dd csub(dd a, dd b) { return dd_add(a, dd_neg(b)); }
__device__ __forceinline__ dd cmul(dd a, dd b) { return dd_mul(a, b); }
__device__ __forceinline__ dd cfma(dd a, dd b, dd c) { return dd_add(dd_mul(a, b), c); }
__device__ __forceinline__ dd cneg(dd a) { return dd_neg(a); }
__device__ __forceinline__ dd crcp(dd a) {  // one Newton step on the FP64 reciprocal
  const double r = 1.0 / a.hi;
  const dd e = dd_add(dd{1.0, 0.0}, dd_neg(dd_mul(a, dd{r, 0.0})));
  return dd_add(dd{r, 0.0}, dd_mul(e, dd{r, 0.0}));
}
__device__ __forceinline__ double cnum(dd a) { return __dadd_rn(a.hi, a.lo); }
__device__ __forceinline__ double c64(dd a) { return __dadd_rn(a.hi, a.lo); }
__device__ __forceinline__ bool cnz(dd a) { return a.hi != 0.0; }
template <int L> __device__ __forceinline__ dd cshfl_xor(dd a, int o, unsigned gm) {
  return dd{__shfl_xor_sync(gm, a.hi, o, L), __shfl_xor_sync(gm, a.lo, o, L)};
}
template <int L> __device__ __forceinline__ dd cshfl(dd a, int src, unsigned gm) {
  return dd{__shfl_sync(gm, a.hi, src, L), __shfl_sync(gm, a.lo, src, L)};
}
template <> __device__ __forceinline__ dd czero<dd>() { return dd{0.0, 0.0}; }

__device__ __forceinline__ ff cadd(ff a, ff b) { return ff_add(a, b); }
__device__ __forceinline__ ff csub(ff a, ff b) { return ff_add(a, ff_neg(b)); }
__device__ __forceinline__ ff cmul(ff a, ff b) { return ff_mul(a, b); }
__device__ __forceinline__ ff cfma(ff a, ff b, ff c) { return ff_add(ff_mul(a, b), c); }
__device__ __forceinline__ ff cneg(ff a) { return ff_neg(a); }
__device__ __forceinline__ ff crcp(ff a) {  // one Newton step on the FP32 reciprocal
  const float r = __frcp_rn(a.hi);
  const ff e = ff_add(ff{1.0f, 0.0f}, ff_neg(ff_mul(a, ff{r, 0.0f})));
  return ff_add(ff{r, 0.0f}, ff_mul(e, ff{r, 0.0f}));
}
__device__ __forceinline__ float cnum(ff a) { return __fadd_rn(a.hi, a.lo); }
__device__ __forceinline__ double c64(ff a) { return (double)a.hi + (double)a.lo; }
__device__ __forceinline__ bool cnz(ff a) { return a.hi != 0.0f; }
template <int L> __device__ __forceinline__ ff cshfl_xor(ff a, int o, unsigned gm) {
  return ff{__shfl_xor_sync(gm, a.hi, o, L), __shfl_xor_sync(gm, a.lo, o, L)};
}
template <int L> __device__ __forceinline__ ff cshfl(ff a, int src, unsigned gm) {
  return ff{__shfl_sync(gm, a.hi, src, L), __shfl_sync(gm, a.lo, src, L)};
}
// Two state values side by side. The float-float operations run on both at once with this part's
// packed FP32 instructions (one instruction for two lanes' worth of the same rounding): half the
// instructions of the loops over C^-1, which wait on instruction supply. Every half rounds as the
// single operation does.
template <typename C> struct Pk;
template <> struct Pk<dd> {
  dd a, b;
};
template <> struct Pk<ff> {
  unsigned long long hi, lo;  // (hi of the first, hi of the second), the same of lo
};
__device__ __forceinline__ unsigned long long f2(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float f2_first(unsigned long long p) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p));
  return a;
}
__device__ __forceinline__ float f2_second(unsigned long long p) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p));
  return b;
}
__device__ __forceinline__ unsigned long long f2_add(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long f2_mul(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long f2_fma(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// a - b, as b (-1) + a: the product is exact, so one rounding
__device__ __forceinline__ unsigned long long f2_sub(unsigned long long a, unsigned long long b) {
  return f2_fma(b, 0xbf800000bf800000ull, a);
}
__device__ __forceinline__ Pk<dd> pk2(dd a, dd b) { return Pk<dd>{a, b}; }
__device__ __forceinline__ Pk<ff> pk2(ff a, ff b) { return Pk<ff>{f2(a.hi, b.hi), f2(a.lo, b.lo)}; }
__device__ __forceinline__ dd pk_first(Pk<dd> x) { return x.a; }
__device__ __forceinline__ dd pk_second(Pk<dd> x) { return x.b; }
__device__ __forceinline__ ff pk_first(Pk<ff> x) { return ff{f2_first(x.hi), f2_first(x.lo)}; }
__device__ __forceinline__ ff pk_second(Pk<ff> x) { return ff{f2_second(x.hi), f2_second(x.lo)}; }
__device__ __forceinline__ Pk<dd> pk_add(Pk<dd> x, Pk<dd> y) { return Pk<dd>{cadd(x.a, y.a), cadd(x.b, y.b)}; }
__device__ __forceinline__ Pk<dd> pk_mul(Pk<dd> x, Pk<dd> y) { return Pk<dd>{cmul(x.a, y.a), cmul(x.b, y.b)}; }
__device__ __forceinline__ Pk<ff> pk_quick(unsigned long long a, unsigned long long b) {
  const unsigned long long s = f2_add(a, b);
  return Pk<ff>{s, f2_sub(b, f2_sub(s, a))};
}
__device__ __forceinline__ Pk<ff> pk_add(Pk<ff> x, Pk<ff> y) {  // ff_add on both
  const unsigned long long s = f2_add(x.hi, y.hi);
  const unsigned long long bb = f2_sub(s, x.hi);
  const unsigned long long e = f2_add(f2_sub(x.hi, f2_sub(s, bb)), f2_sub(y.hi, bb));
  return pk_quick(s, f2_add(e, f2_add(x.lo, y.lo)));
}
__device__ __forceinline__ Pk<ff> pk_mul(Pk<ff> x, Pk<ff> y) {  // ff_mul on both
  const unsigned long long p = f2_mul(x.hi, y.hi);
  unsigned long long e = f2_fma(x.hi, y.hi, f2_mul(p, 0xbf800000bf800000ull));
  e = f2_fma(x.hi, y.lo, e);
  e = f2_fma(x.lo, y.hi, e);
  return pk_quick(p, e);
}
template <typename C> __device__ __forceinline__ Pk<C> pk_fma(Pk<C> x, Pk<C> y, Pk<C> z) {
  return pk_add(pk_mul(x, y), z);
}

// a scoring-precision value (T) as a state value
__device__ __forceinline__ ff cfromf(float a) { return ff{a, 0.0f}; }
__device__ __forceinline__ dd cfromf(double a) { return dd{a, 0.0}; }
// a table entry as a value of type C: cross-correlation tables are FP64 (refresh, FP64 mode)
// or float-float (FP32 mode)
template <typename C> __device__ __forceinline__ C cload(double a);
template <> __device__ __forceinline__ double cload<double>(double a) { return a; }
template <> __device__ __forceinline__ dd cload<dd>(double a) { return dd{a, 0.0}; }
template <typename C> __device__ __forceinline__ C cload(ff a);
template <> __device__ __forceinline__ ff cload<ff>(ff a) { return a; }
template <> __device__ __forceinline__ ff czero<ff>() { return ff{0.0f, 0.0f}; }
// FP64 -> state value (refresh only)
template <typename C> __device__ __forceinline__ C cfrom64(double a);
template <> __device__ __forceinline__ dd cfrom64<dd>(double a) { return dd{a, 0.0}; }
template <> __device__ __forceinline__ ff cfrom64<ff>(double a) {
  const float h = (float)a;
  return ff{h, (float)(a - (double)h)};
}
// mean and r = sigma_eps^2 / sigma_e^2 of charge component e as state values (split into
// pairs on the host)
template <typename C> __device__ __forceinline__ C c_mu(const DevModel& M, int e);
template <> __device__ __forceinline__ dd c_mu<dd>(const DevModel& M, int e) { return dd{M.cm_mu[e], 0.0}; }
template <> __device__ __forceinline__ ff c_mu<ff>(const DevModel& M, int e) { return ff{M.cm_mu_hi[e], M.cm_mu_lo[e]}; }
template <typename C> __device__ __forceinline__ C c_r(const DevModel& M, int e);
template <> __device__ __forceinline__ dd c_r<dd>(const DevModel& M, int e) { return dd{M.cm_r[e], 0.0}; }
template <> __device__ __forceinline__ ff c_r<ff>(const DevModel& M, int e) { return ff{M.cm_r_hi[e], M.cm_r_lo[e]}; }

// A charge component's constant in the scoring precision T: the FP32 copies in FP32 mode, so
// that the step loop converts nothing from FP64 (an FP64 instruction costs this part as much as
// 64 FP32 ones).
template <typename T> struct CmT;
template <> struct CmT<float> {
  __device__ static float mu(const DevModel& M, int e) { return M.cmf_mu[e]; }
  __device__ static float q(const DevModel& M, int e) { return M.cmf_q[e]; }
  __device__ static float iq(const DevModel& M, int e) { return M.cmf_iq[e]; }
  __device__ static float r(const DevModel& M, int e) { return M.cmf_r[e]; }
};
template <> struct CmT<double> {
  __device__ static double mu(const DevModel& M, int e) { return M.cm_mu[e]; }
  __device__ static double q(const DevModel& M, int e) { return M.cm_q[e]; }
  __device__ static double iq(const DevModel& M, int e) { return M.cm_iq[e]; }
  __device__ static double r(const DevModel& M, int e) { return M.cm_r[e]; }
};

// Component of a born or updated PE, e+ ~ G (Sec. 2.4): the smallest e whose cumulative
// probability exceeds the uniform u, else the last component with G > 0. The comparison is
// in FP64 in both modes, so the draw is the same as the FP64 reference's.
__device__ __forceinline__ int pe_draw_comp(const DevModel& M, double u) {
#pragma unroll 1
  for (int e = 0; e < M.n_comp; ++e)
    if (M.cm_cum[e] > u) return e;
  return M.cm_last;
}

// group sum of a state value
template <int L, typename C> __device__ __forceinline__ C csum(C v, const Lanes<L> ln) {
#pragma unroll 1
  for (int o = L / 2; o > 0; o >>= 1) v = cadd(v, cshfl_xor<L>(v, o, ln.gm));
  return v;
}

// twice a state value (exact)
__device__ __forceinline__ double ctwice(double a) { return 2.0 * a; }
__device__ __forceinline__ dd ctwice(dd a) { return dd{2.0 * a.hi, 2.0 * a.lo}; }
__device__ __forceinline__ ff ctwice(ff a) { return ff{2.0f * a.hi, 2.0f * a.lo}; }

// The first offset of a butterfly over values that are zero on lanes >= m (m >= 0): the levels
// above it would add zeros only, which leaves a normalised pair as it is.
template <int L> __device__ __forceinline__ int first_level(int m) {
  return m > L / 2 ? L / 2 : (m > 1 ? 1 << (31 - __clz(m - 1)) : 0);
}
// one or two group sums of state values that are zero on lanes >= m, the result on every lane
template <int L, typename C> __device__ __forceinline__ C csum_m(C v, int m, const Lanes<L> ln) {
#pragma unroll 1
  for (int o = first_level<L>(m); o > 0; o >>= 1) v = cadd(v, cshfl_xor<L>(v, o, ln.gm));
  return m > L / 2 ? v : cshfl<L>(v, 0, ln.gm);
}
template <int L, typename C> __device__ __forceinline__ void csum2_m(C& a, C& b, int m, const Lanes<L> ln) {
  Pk<C> p = pk2(a, b);
#pragma unroll 1
  for (int o = first_level<L>(m); o > 0; o >>= 1)
    p = pk_add(p, pk2(cshfl_xor<L>(pk_first(p), o, ln.gm), cshfl_xor<L>(pk_second(p), o, ln.gm)));
  a = pk_first(p);
  b = pk_second(p);
  if (m <= L / 2) {
    a = cshfl<L>(a, 0, ln.gm);
    b = cshfl<L>(b, 0, ln.gm);
  }
}

// four group sums in one butterfly (two state values, two scoring-precision values), so that
// their shuffles and additions overlap
// (over the group's L lanes, or within its subgroups of GW lanes)
template <int L, int GW, typename C, typename T>
__device__ __forceinline__ void gsum4(C& a, C& b, T& x, T& y, const Lanes<L> ln) {
  Pk<C> p = pk2(a, b);
#pragma unroll 1
  for (int o = GW / 2; o > 0; o >>= 1) {
    const C a2 = cshfl_xor<L>(pk_first(p), o, ln.gm), b2 = cshfl_xor<L>(pk_second(p), o, ln.gm);
    const T x2 = __shfl_xor_sync(ln.gm, x, o, L), y2 = __shfl_xor_sync(ln.gm, y, o, L);
    p = pk_add(p, pk2(a2, b2));
    x += x2;
    y += y2;
  }
  a = pk_first(p);
  b = pk_second(p);
}

// C^-1 is symmetric and stored as its lower triangle, row by row: entry (i, j), j <= i, at
// tri(i) + j. The storage has no row stride, so a chain's C^-1 moves from the shared tile to
// its global slot by a plain copy.
__host__ __device__ __forceinline__ int tri(int i) { return i * (i + 1) / 2; }
__device__ __forceinline__ int pk(int i, int j) { return i >= j ? tri(i) + j : tri(j) + i; }
// (i, j) of packed position e (j <= i); the FP32 square root is exact enough below 2^22
__device__ __forceinline__ void untri(int e, int& i, int& j) {
  i = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
  if (tri(i + 1) <= e) ++i;
  if (tri(i) > e) --i;
  j = e - tri(i);
}

// A lane's walk over the packed triangle, entries e = first, first + L, ...: (i, j) from the
// block's table below kTriTab entries (the rows of a chain of up to 32 PEs, nearly all of the
// accepts of the uneven windows), one row carry per step beyond it (rows there have more than L
// entries). The table replaces a square root and its corrections, about 25 instructions of the
// 90 that an entry of the accept's pass took.
constexpr int kTriRows = 32;
constexpr int kTriTab = kTriRows * (kTriRows + 1) / 2;
template <int L> struct TriWalk {
  int i = 0, j = 0;
  __device__ __forceinline__ void at(const unsigned short* __restrict__ tij, int e) {
    if (e < kTriTab) {
      const int t = tij[e];
      i = t >> 8;
      j = t & 255;
    } else {
      j += L;
      if (j > i) {
        j -= i + 1;
        ++i;
      }
    }
  }
};

// sum_a C^-1[q][idx[a]] b[a] over a < m, C^-1 in global memory: four independent partial sums so
// that the gathers of consecutive terms overlap
template <typename C>
__device__ __forceinline__ C dot_row4(const C* __restrict__ Cp, int q, const int* __restrict__ idx,
                                      const C* __restrict__ b, int m) {
  Pk<C> s01 = pk2(czero<C>(), czero<C>()), s23 = s01;
  int a = 0;
#pragma unroll 1
  for (; a + 3 < m; a += 4) {
    C r[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) r[u] = Cp[pk(q, idx[a + u])];
    s01 = pk_fma(pk2(r[0], r[1]), pk2(b[a], b[a + 1]), s01);
    s23 = pk_fma(pk2(r[2], r[3]), pk2(b[a + 2], b[a + 3]), s23);
  }
  C s0 = cadd(cadd(cadd(pk_first(s01), pk_second(s01)), pk_first(s23)), pk_second(s23));
#pragma unroll 1
  for (; a < m; ++a) s0 = cfma(Cp[pk(q, idx[a])], b[a], s0);
  return s0;
}

template <int L, typename T> __device__ __forceinline__ T wsum(T v, const Lanes<L> ln) {
#pragma unroll 1
  for (int o = L / 2; o > 0; o >>= 1) v += __shfl_xor_sync(ln.gm, v, o, L);
  return v;
}
template <int L, typename T> __device__ __forceinline__ T wmax(T v, const Lanes<L> ln) {
#pragma unroll 1
  for (int o = L / 2; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(ln.gm, v, o, L));
  return v;
}

// ---------------------------------------------------------------- model tables
template <typename T> struct PeTab;
template <> struct PeTab<double> {
  using C = dd;
  __device__ static const double* V(const DevModel& M) { return M.V64; }
  __device__ static const double* logphi(const DevModel& M) { return M.logphi; }
  __device__ static const double* cphi(const DevModel& M) { return M.cphi; }
  __device__ static const double* tc(const DevModel& M) { return M.tc64; }
};
template <> struct PeTab<float> {
  using C = ff;
  __device__ static const float* V(const DevModel& M) { return M.V32; }
  __device__ static const float* logphi(const DevModel& M) { return M.logphi32; }
  __device__ static const float* cphi(const DevModel& M) { return M.cphi32; }
  __device__ static const ff* tc(const DevModel& M) { return reinterpret_cast<const ff*>(M.tcff); }
};

template <typename T> __device__ __forceinline__ T pe_logphi(const DevModel& M, int d) {
  return (d < -M.D || d > M.D) ? (T)-INFINITY : __ldg(PeTab<T>::logphi(M) + (d + M.D));
}
template <typename T> __device__ __forceinline__ T pe_cphi(const DevModel& M, int d) {
  if (d < -M.D) return (T)0;
  if (d > M.D) return __ldg(PeTab<T>::cphi(M) + 2 * M.D);
  return __ldg(PeTab<T>::cphi(M) + (d + M.D));
}

// Support of the PE at grid index j in a window of n samples: its first sample w0 = ceil(j / R),
// the phase ph = w0 R - j of that sample, and the range [ilo, ihi) of its support samples
// (sample w0 + i, SER index ph + i R) that lie in the window.
struct Sup {
  int w0, ph, ilo, ihi;
};
__device__ __forceinline__ Sup pe_sup(const DevModel& M, int n, int j) {
  Sup s;
  // w0 = ceil(j / R) = floor((j + R - 1) / R): an FP32 estimate (off by at most one for
  // |j| < 2^22) corrected by one integer step, instead of a division
  const int num = j + M.R - 1;
  int q = __float2int_rd((float)num * M.inv_Rf);
  if (q * M.R > num) --q;
  else if ((q + 1) * M.R <= num) ++q;
  s.w0 = q;
  s.ph = q * M.R - j;
  s.ilo = max(0, -q);
  s.ihi = min(M.L_V, n - q);  // every phase ph < R covers L_V samples (Lt = L_V R)
  if (s.ihi <= s.ilo) s.ilo = s.ihi = 0;  // no sample of the window: an all-zero column
  return s;
}

// a_x^T a_q over the window, for x with support s and q = x - o (|o| < Lt), from the prefix table.
template <typename C, typename TT>
__device__ __forceinline__ C xcorr(const DevModel& M, const TT* __restrict__ tc, const Sup& s, int o) {
  const unsigned O = 2 * M.Lt - 1, row = s.ph * M.tcM;  // at most 64 x 129 x 16383 entries
  C v = cload<C>(tc[(row + s.ihi) * O + (o + M.Lt - 1)]);
  if (s.ilo > 0) v = csub(v, cload<C>(tc[(row + s.ilo) * O + (o + M.Lt - 1)]));
  return v;
}

// Smallest j in [T_lo, T_hi) with cphi(j - k0) - base > target (L-ary group search; cphi is
// non-decreasing, so the answer does not depend on L); if rounding leaves none, the last j of T
// with phi > 0.
template <typename T, int L>
__device__ int pe_birth_search(const DevModel& M, int T_lo, int T_hi, int k0, T base, T target, const Lanes<L> ln) {
  int lo = T_lo, hi = T_hi - 1;
  if ((pe_cphi<T>(M, hi - k0) - base) > target) {
#pragma unroll 1
    while (lo < hi) {
      const int len = hi - lo + 1;
      const int step = (len + L - 1) / L;
      const int p = min(hi, lo + (ln.sl + 1) * step - 1);
      const bool pred = (pe_cphi<T>(M, p - k0) - base) > target;
      const unsigned b = gballot(pred, ln);
      const int f = __ffs(b) - 1;
      const int new_lo = lo + f * step;
      hi = min(hi, lo + (f + 1) * step - 1);
      lo = new_lo;
    }
    return lo;
  }
  int last = -1;
#pragma unroll 1
  for (int top = T_hi - 1; top >= T_lo; top -= L) {
    const int j = top - ln.sl;
    const bool ok = j >= T_lo && pe_logphi<T>(M, j - k0) > (T)-INFINITY;
    const unsigned b = gballot(ok, ln);
    if (b) { last = top - (__ffs(b) - 1); break; }
  }
  return last;
}

// cphi(d) without branches (the same values as pe_cphi)
template <typename T> __device__ __forceinline__ T pe_cphi_clamped(const DevModel& M, int d) {
  const T v = __ldg(PeTab<T>::cphi(M) + min(max(d + M.D, 0), 2 * M.D));
  return d < -M.D ? (T)0 : v;
}
// The last j of T with phi > 0 for the subgroups with want set, -1 if there is none (a birth search
// that rounding left without an answer: it runs next to never, so out of line).
template <typename T, int L>
__device__ __noinline__ int pe_birth_last(const DevModel& M, int T_lo, int T_hi, int k0, bool want, const Lanes<L> ln) {
  constexpr int w = L / kSub;
  const int gi = ln.sl / w, m = ln.sl % w;
  int last = -1;
#pragma unroll 1
  for (int top = T_hi - 1; gballot(want && last < 0 && top >= T_lo, ln); top -= w) {
    const int j = top - m;
    const bool ok = want && last < 0 && j >= T_lo && pe_logphi<T>(M, j - k0) > (T)-INFINITY;
    const unsigned b = (gballot(ok, ln) >> (gi * w)) & ((1u << w) - 1u);
    if (b) last = top - (__ffs(b) - 1);
  }
  return last;
}
// The birth search for every subgroup of w lanes at once (subgroups with want = false idle): each
// lane tests kSub points per round, so that their table loads overlap. u4 is the uniform of the
// proposal: the target is u4 tot, tot = cphi(T_hi - 1 - k0) - base the mass of T. All lanes of the
// chain call.
template <typename T, int L>
__device__ __forceinline__ int pe_birth_search_sub(const DevModel& M, int T_lo, int T_hi, int k0, T u4, bool want,
                                                   const Lanes<L> ln) {
  constexpr int w = L / kSub, P = w * kSub;
  const int gi = ln.sl / w, m = ln.sl % w;
  const unsigned sm = ((1u << w) - 1u) << (gi * w);
  int lo = T_lo, hi = T_hi - 1;
  const T base = pe_cphi_clamped<T>(M, T_lo - 1 - k0), tot = pe_cphi_clamped<T>(M, hi - k0) - base, target = u4 * tot;
  const bool found = tot > target;
#pragma unroll 1
  while (gballot(want && found && lo < hi, ln)) {
    const int step = (hi - lo + P) / P;
    int nf = 0;  // points that are not beyond the target: the first ones
    T c[kSub];
#pragma unroll
    for (int u = 0; u < kSub; ++u)
      c[u] = pe_cphi_clamped<T>(M, min(hi, lo + (m * kSub + u + 1) * step - 1) - k0);
#pragma unroll
    for (int u = 0; u < kSub; ++u) nf += __popc(gballot(!(c[u] - base > target), ln) & sm);
    lo += nf * step;
    hi = min(hi, lo + step - 1);
  }
  if (gballot(want && !found, ln)) {
    const int last = pe_birth_last<T, L>(M, T_lo, T_hi, k0, want && !found, ln);
    if (!found) lo = last;
  }
  return lo;
}

template <typename T, bool MIX> struct PeRand {
  T z1, lu0, u3, u4, z2, lu;  // t0 shift normal, log u2, jump type, PE choice, shift normal, log u7
};
template <typename T> struct PeRand<T, true> {
  T z1, lu0, u3, u4, z2, lu;
  int ep;  // charge component of a born or updated PE
};
template <typename T, bool MIX> __host__ __device__ constexpr size_t pe_rand_bytes() { return sizeof(PeRand<T, MIX>); }

// FP32 value of the uniform ((x >> 11) + 0.5) 2^-53: the odd 54-bit integer 2 (x >> 11) + 1
// rounded to FP32, times 2^-54 (exact), i.e. the FP64 uniform rounded to FP32 without FP64 work.
__device__ __forceinline__ float u01_float(uint64_t x) {
  return __ull2float_rn(((x >> 11) << 1) | 1ull) * 0x1.0p-54f;
}

// Per-chain statistics (shared memory, written by the group's first lane).
struct PeStats {
  // of the state: the charge summary and the Wasserstein scalars of the PE times and components
  // (they hold from step q_from on: they change only with z); the sums over the samples of each
  // and of its square, then log|Sigma| and log L
  double cur[3], sum[8];
  static constexpr int kLogdet = 6, kLogL = 7;
  long long St, Se;  // sum of |t_k| (grid units) and of e_k over the PEs of the state
  double drift_max, wsq;
  int n_refresh, status, q_from, n_acc_refresh, refresh_fail, pad;
};

// Speculative batches. A chain's step depends on the step before it only where that step was
// accepted, and most steps are not (accepted: 4 % at one PE, 13 % over the uneven windows, 33 % at
// 30 PEs). So a chain of up to kSpecPes PEs scores kSpec consecutive steps at once, step i on the
// i-th of kSpec subgroups of its lanes, all from the same state (each with its own t0: those moves
// come first, one after the other); the steps up to and including the first accepted one count, the
// ones behind it are scored again from the new state. Everything a step does with the same values on
// every lane (the 2x2 algebra, the proposal, the bookkeeping) then runs once per batch instead of
// once per step: 1077 instead of 1630 warp instructions a step at 8 PEs, and half the code fetched.
// The decisions and every rounding are those of the one-by-one steps: a subgroup adds up the L
// lanes' partial sums in the same order (each of its lanes holds kSpec of them). Four steps: with
// eight the batch's loops are twice as long, and wait for instructions too (low occupancy 106 ms
// against 104, one event 5.97 against 5.22). Up to 32 PEs: beyond, the entries scored for steps
// that do not count cost what the batch saves. In FP64 mode, where the entries' pair arithmetic is
// most of a step, that is so from 12 PEs on (x 300 steps, batches up to 32 PEs and up to 12: 608
// chains of 24 PEs 15.1 ms and 13.1, of 8 PEs 8.0 and 7.2, 16 of 4 PEs 4.35 and 4.35; with batches up to
// 8 those 16 take 4.48, with batches up to 4 256 chains of 2 PEs x 1000 13.6 instead of 11.6). 20 000
// uneven windows x 2000 steps: 120 -> 110 ms, 100 000 low-occupancy chains x 1000: 134 -> 103 ms, 256
// FP64 chains x 1000: 13.7 -> 9.8 ms.
constexpr int kSpec = kSub;
constexpr int kSpecPes = 32;   // most PEs of a chain scored this way (indices in W.ix())
template <typename T> __host__ __device__ constexpr int spec_pes() { return sizeof(T) == 4 ? kSpecPes : 12; }
constexpr int kCounts = 8;     // integer counts of a chain, per subgroup (PeChain::cnt)

// A step's addition to count q: sums over the samples after burn-in of N, N^2, k0 and k0^2, the
// algorithmic words, then pairs of counters: proposed births | deaths, accepted births | deaths,
// accepted updates | accepted t0 moves (a chain's other proposals follow from its step count).
__device__ __forceinline__ unsigned long long count_of(int q, int N, int k0, bool past, unsigned words, int jump,
                                                       bool applied, bool t0_acc) {
  const int a = (q & 2) ? k0 : N, b = (q & 1) ? a : 1;
  const unsigned long long jp = jump == 0 ? 1ull : (jump == 1 ? 1ull << 32 : 0ull);
  const unsigned long long tail = q == 4 ? (unsigned long long)words
                                  : q == 5 ? jp
                                  : q == 6 ? (applied ? jp : 0ull)
                                           : (applied && jump == 2 ? 1ull : 0ull) + (t0_acc ? 1ull << 32 : 0ull);
  return q < 4 ? (past ? (unsigned long long)((long long)a * (long long)b) : 0ull) : tail;
}

__host__ __device__ inline size_t a16(size_t x) { return (x + 15) & ~(size_t)15; }

// The CTA's dynamic shared memory: the block tables, then a block per chain. Everything in it is
// addressed by 32-bit offsets from this symbol, so that the compiler sees shared memory also in
// the out-of-line functions (generic 64-bit pointers there cost two registers each and about a
// third more code, which is what binds chains with few PEs: the step has to stay in the SM's
// 32 KB instruction cache).
extern __shared__ __align__(16) unsigned char pe_smem[];

// Block tables: (i, j) of the first packed entries, the SER, log(i) and 1 / i (i <= n_cap + 1).
constexpr unsigned kTabBytes = (sizeof(unsigned short) * kTriTab + 15) & ~15u;
template <typename T> __host__ __device__ inline size_t pe_block_bytes(const DevModel& M) {
  return kTabBytes + a16(sizeof(T) * M.Lt) + a16(sizeof(T) * (M.n_cap + 2)) + a16(sizeof(double) * (M.n_cap + 2));
}
__device__ __forceinline__ unsigned short* pe_tij() { return reinterpret_cast<unsigned short*>(pe_smem); }
template <typename T> __device__ __forceinline__ T* pe_V() { return reinterpret_cast<T*>(pe_smem + kTabBytes); }

// Per-chain shared memory. C is the state type (16 bytes in FP64 mode, 8 in FP32 mode).
template <typename T, bool BIG, int L, bool MIX> struct PeChain {
  using C = typename PeTab<T>::C;
  unsigned o;    // the chain's block
  unsigned vb;   // bytes of a vector of n_cap state values
  unsigned lb;   // bytes of the PE list
  unsigned yb;   // bytes of the residual
  unsigned pb;   // bytes of log Phi
  static constexpr unsigned kCnt = (sizeof(PeStats) + 15) & ~15u, kIx = kCnt + 8 * kSpec * kCounts,
                            kRnd = kIx + (BIG ? 0 : kSpec * kSpecPes),
                            kVec = (kRnd + (unsigned)sizeof(PeRand<T, MIX>) * L + 15) & ~15u;
  template <typename E> __device__ __forceinline__ E* at(unsigned b) const {
    return reinterpret_cast<E*>(pe_smem + (o + b));
  }
  __device__ __forceinline__ PeStats& st() const { return *at<PeStats>(0); }
  // counts [kSpec][kCounts]
  __device__ __forceinline__ unsigned long long* cnt() const { return at<unsigned long long>(kCnt); }
  // batch: PEs overlapping each subgroup's proposed one [kSpec][kSpecPes]
  __device__ __forceinline__ unsigned char* ix() const { return at<unsigned char>(kIx); }
  // draws of the next L steps
  __device__ __forceinline__ PeRand<T, MIX>* rnd() const { return at<PeRand<T, MIX>>(kRnd); }
  __device__ __forceinline__ C* v() const { return at<C>(kVec); }  // C^-1 A^T y
  // four work vectors (BIG: three and a list of indices). In a batch, subgroup i keeps the
  // proposed PE's inner products b in the i-th. Otherwise: b over the overlapping PEs (the accept
  // then keeps u' / delta there), row k of C^-1, C^-1 b, and b's indices (then c / -gamma)
  __device__ __forceinline__ C* work(int i) const { return at<C>(kVec + (1 + i) * vb); }
  __device__ __forceinline__ C* ovb() const { return work(0); }
  __device__ __forceinline__ C* cv() const { return work(1); }
  __device__ __forceinline__ C* uv() const { return work(2); }
  __device__ __forceinline__ int* ovi() const { return at<int>(kVec + 4 * vb); }
  __device__ __forceinline__ C* cvn() const { return work(3); }  // not BIG
  __device__ __forceinline__ int* list() const { return at<int>(tail()); }  // PE grid indices [n_cap]
  __device__ __forceinline__ unsigned tail() const { return kVec + 4 * vb + (BIG ? lb : vb); }
  // residual [n_alloc], then log(Phi_T(t0) g) on the chain's t0 grid [win_extra], the C^-1 tile
  // (packed triangle of Ns PEs) and the PEs' charge components [n_cap] (mixture only)
  __device__ __forceinline__ T* y() const { return at<T>(tail() + lb); }
  __device__ __forceinline__ T* lPhi() const { return at<T>(tail() + lb + yb); }
  __device__ __forceinline__ unsigned char* le() const { return at<unsigned char>(tail() + lb + yb + pb); }
  __device__ __forceinline__ C* Cs(int n_cap) const {
    return at<C>(tail() + lb + yb + pb + (MIX ? (unsigned)a16((size_t)n_cap) : 0u));
  }
};
template <typename T, bool BIG, int L, bool MIX>
__host__ __device__ inline size_t pe_chain_bytes(int n_cap, int n_alloc, int win_extra, int Ns) {
  constexpr size_t cs = sizeof(typename PeTab<T>::C);
  return PeChain<T, BIG, L, MIX>::kVec + 4 * a16(cs * (size_t)n_cap) + a16((BIG ? sizeof(int) : cs) * (size_t)n_cap) +
         a16(sizeof(int) * n_cap) + a16(sizeof(T) * n_alloc) + a16(sizeof(T) * win_extra) +
         (MIX ? a16((size_t)n_cap) : 0) + a16(cs * (size_t)tri(Ns));
}

// Global per-chain slots (one per resident chain of the launch).
struct PeSlots {
  void* C;             // C^-1 slots (state entries): the packed triangle of n_cap PEs
  size_t c_stride;     // entries per slot
  double* ws;          // FP64 refresh workspace slots (FP32 mode)
  size_t ws_stride;    // doubles per slot
  int* hist;           // N histogram slots, n_cap + 1 counts each
  int* counter;        // next chain of the launch (zeroed before the launch)
  int Ns;              // shared-memory tile of C^-1 (0: always global)
};

// FP64 refresh workspace of one chain: C (n_cap x n_cap), h and v (n_cap each), a sweep block's
// rows before and after its sweep (n_cap x kSweepBlock each; together they also hold an FP64
// copy of the window while the residual is rebuilt) and the block's pivot factors
// (kSweepBlock x kSweepBlock); every part starts on a 16-byte boundary.
constexpr int kSweepBlock = 8;
__host__ __device__ inline size_t pe_ws_a2(size_t n) { return (n + 1) & ~(size_t)1; }
__host__ __device__ inline size_t pe_ws_doubles(int n_cap) {
  return pe_ws_a2((size_t)n_cap * n_cap) + (2 + 2 * kSweepBlock) * pe_ws_a2(n_cap) + kSweepBlock * kSweepBlock;
}

// Close the hold of the state's summaries at step s and, where a move was accepted (dT, dnu: its
// changes of log|Sigma| and log L), add these: a lane per sum, so that the FP64 operations (64
// issue cycles each on this part, however few lanes take part) are done once for all of them.
template <typename T>
__device__ __forceinline__ void close_hold(PeStats& S, int s, int burn_in, bool accepted, T dT, T dnu, int sl) {
  if (sl < 8) {
    const int held = s - max(S.q_from, burn_in);
    double x = sl < 6 ? S.cur[sl >> 1] : (double)(sl == 6 ? dT : dnu);
    if (sl < 6 && (sl & 1)) x = x * x;
    if (sl < 6 ? held > 0 : accepted) S.sum[sl] = fma(x, sl < 6 ? (double)held : 1.0, S.sum[sl]);
  }
}
// The summaries of a state with N PEs, a lane per value: the charge sum_k (mu_k + v_k), given
// qs = sum v_k and ms = mu (dynode: times N) or sum_k mu_k (mixture), and the Wasserstein scalars
// (the convergence check of Sec. 3.2): with a dummy PE at t = 0, e = 0 added, the 1-Wasserstein
// distance from the sequence to the dummy alone is the mean of |t| (or of e) over the N + 1
// points. inv1[i] = 1 / i (a block table, so that no FP64 division runs in the step loop).
template <bool MIX>
__device__ __forceinline__ void set_summaries(PeStats& S, double g, int N, double ms, double qs, const double* inv1,
                                              int sl) {
  if (sl < 3) {
    const long long n = sl == 0 ? (MIX ? 1 : N) : (sl == 1 ? S.St : S.Se);
    const double x = fma((double)n, sl == 0 ? ms : (sl == 1 ? g : 1.0), sl == 0 ? qs : 0.0);
    S.cur[sl] = sl == 0 ? x : x * inv1[N + 1];
  }
}

// lambda_FSMP at the chain end, out of line: the estimator's code stays out of the step loop's
// instruction stream
template <int L>
__device__ __noinline__ double pe_lambda_mle(const int* h, int n_max, double lambda0, int sl, unsigned gm) {
  return group_lambda_mle<L>(h, n_max, lambda0, sl, gm);
}

struct RefreshOut {
  int ok;
  double logdet, logL, drift;
};

// Teams. A chain of more than kSpecPes PEs spends nearly all of its step waiting for C^-1: one
// warp keeps some hundred gathers in flight, and a launch of few chains ends when its longest one
// does. With TW = kTeam the CTA is one chain: warp 0 runs it, and the other warps take part where a
// step reads or writes all of C^-1 or rebuilds it. They wait at a barrier for the next command,
// do their share, and meet again. Entries, rows and sums keep their operations and their order
// (a sum of the scoring stays the sum of 32 partial sums), so the results are the same bit for bit.
// 1000 pile-up chains x 2000 steps: 600 ms with a warp per chain, 255 with a team; a burst of 64
// events of up to 100 PEs a channel: 104 and 51; 777 uneven windows x 1000 steps: 16.9 and 10.7.
// Bound now: the latency of C^-1's gathers from L2 and of the sums' dependent additions, and the
// FP64 pipe of the rebuilds. 4 CTAs per SM (128 registers): with 3, 3000 uneven windows take 18.8
// ms against 16.4 and pile-up the same.
constexpr int kTeam = 4;
enum TeamOp { kOpExit, kOpScore, kOpRows, kOpUpdate, kOpRefresh };
template <typename C> struct PeTeam {
  C part[32];          // scoring: the partial sums of b^T C^-1 b
  double red[kTeam][2];  // refresh: the warps' largest drift and entry
  C* Cp;
  double* ws;
  const float* w;
  double wsq;
  C nig, idl;
  int op, N, np, jump, kk, n, ok;
};
constexpr unsigned kTeamBytes = 640;
// the command block: behind the block tables, before the chain
template <typename T> __device__ __forceinline__ PeTeam<typename PeTab<T>::C>& pe_team(const DevModel& M) {
  static_assert(sizeof(PeTeam<typename PeTab<T>::C>) <= kTeamBytes || sizeof(T) == 8, "the command block");
  return *reinterpret_cast<PeTeam<typename PeTab<T>::C>*>(pe_smem + pe_block_bytes<T>(M));
}
__device__ __forceinline__ void team_bar() {
  __syncwarp();
  asm volatile("bar.sync 1, %0;" ::"n"(kTeam * 32) : "memory");
}
// the team's threads (TW = 1: the chain's lanes) meet
template <int TW, int L> __device__ __forceinline__ void team_sync(const Lanes<L> ln) {
  if constexpr (TW > 1) team_bar();
  else __syncwarp(ln.gm);
}
// (i, j) of packed entries e, e + S, e + 2 S, ... (rows beyond the table are longer than 32)
template <int S> struct TeamWalk {
  int i = 0, j = 0;
  __device__ __forceinline__ void at(const unsigned short* __restrict__ tij, int e) {
    if (e < kTriTab) {
      const int t = tij[e];
      i = t >> 8;
      j = t & 255;
    } else {
      j += S;
      while (j > i) {
        j -= i + 1;
        ++i;
      }
    }
  }
};

// b^T C^-1 b: partial sum l (of entries l, l + 32, ..) on four neighbouring threads, each of which
// takes every fourth product; all four add them up in order.
template <typename T, bool BIG, int L, bool MIX>
__device__ __noinline__ void team_score(const DevModel& M, const PeChain<T, BIG, L, MIX> W) {
  using C = typename PeTab<T>::C;
  PeTeam<C>& tm = pe_team<T>(M);
  const unsigned short* const tij = pe_tij();
  const C* const Cp = tm.Cp;
  const int nt = tri(tm.np), lane = threadIdx.x & 31, r = lane & 3, l = (threadIdx.x >> 5) * 8 + (lane >> 2);
  constexpr int U = 4;  // products of a thread per pass, their loads ahead of the sums
  TeamWalk<128> tw;
  C acc = czero<C>();
#pragma unroll 1
  for (int base = 0; base < nt; base += U * 128) {
    C t[U];
    int dg = 0;
    {
      C cq[U], ba[U], bb[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = base + u * 128 + r * 32 + l;
        const bool in = e < nt;  // beyond the triangle: zero terms
        if (in) tw.at(tij, e);
        const C c = Cp[tri(W.ovi()[tw.i]) + W.ovi()[tw.j]];
        cq[u] = in ? c : czero<C>();
        ba[u] = W.ovb()[tw.i];
        bb[u] = W.ovb()[tw.j];
        dg |= (tw.i == tw.j) << u;
      }
#pragma unroll
      for (int u = 0; u < U; u += 2) {
        const Pk<C> p = pk_mul(pk2(cq[u], cq[u + 1]), pk_mul(pk2(ba[u], ba[u + 1]), pk2(bb[u], bb[u + 1])));
        const C t0 = pk_first(p), t1 = pk_second(p);
        t[u] = (dg >> u) & 1 ? t0 : ctwice(t0);
        t[u + 1] = (dg >> (u + 1)) & 1 ? t1 : ctwice(t1);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc = cadd(acc, cshfl<4>(t[u], q, 0xffffffffu));
  }
  if (r == 0) tm.part[l] = acc;
}

// u' before the removed PE's term: row i of C^-1 times b~, a thread per row
template <typename T, bool BIG, int L, bool MIX>
__device__ __noinline__ void team_rows(const DevModel& M, const PeChain<T, BIG, L, MIX> W) {
  using C = typename PeTab<T>::C;
  const PeTeam<C>& tm = pe_team<T>(M);
  const C* const Cp = tm.Cp;
  const int N = tm.N, np = tm.np;
#pragma unroll 1
  for (int i = threadIdx.x; i < N; i += kTeam * 32) {
    if constexpr (BIG) {
      W.uv()[i] = dot_row4<C>(Cp, i, W.ovi(), W.ovb(), np);
    } else {
      C acc = czero<C>();
      int a = 0;
#pragma unroll 1
      for (; a + 3 < np; a += 4) {
        C x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = Cp[pk(i, W.ovi()[a + u])];
#pragma unroll
        for (int u = 0; u < 4; ++u) acc = cfma(x[u], W.ovb()[a + u], acc);
      }
#pragma unroll 1
      for (; a < np; ++a) acc = cfma(Cp[pk(i, W.ovi()[a])], W.ovb()[a], acc);
      W.uv()[i] = acc;
    }
  }
}

// The accepted move's pass over C^-1 (see pe_accept), entries over the team's threads. A pass
// reads an entry only where it writes it, or in the last row for a death (which is not written).
template <typename T, bool BIG, int L, bool MIX>
__device__ __noinline__ void team_update(const DevModel& M, const PeChain<T, BIG, L, MIX> W) {
  using C = typename PeTab<T>::C;
  const PeTeam<C>& tm = pe_team<T>(M);
  const unsigned short* const tij = pe_tij();
  C* const Cp = tm.Cp;
  const int N = tm.N, jump = tm.jump, kk = tm.kk;
  const bool has_m = jump != 0, has_p = jump != 1;
  const int Nout = N + (jump == 0 ? 1 : (jump == 1 ? -1 : 0)), last = N - 1;
  const int s = jump == 0 ? N : (jump == 2 ? kk : -1), kmap = jump == 1 ? kk : -1;
  const int ne = tri(Nout);
  const C nig = tm.nig, idl = tm.idl;
  const C* const cv = W.cv();
  const C* const cvn = BIG ? W.cv() : W.cvn();
  const C* const uv = W.uv();
  const C* const uvd = W.ovb();
  constexpr int U = 4, S = kTeam * 32;
  TeamWalk<S> tw;
#pragma unroll 1
  for (int e = threadIdx.x; e < ne; e += U * S) {
    int ii[U], jj[U];
    C x[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (e + u * S < ne) tw.at(tij, e + u * S);
      ii[u] = tw.i;
      jj[u] = tw.j;
      x[u] = Cp[pk(tw.i == kmap ? last : tw.i, tw.j == kmap ? last : tw.j)];
    }
#pragma unroll
    for (int u = 0; u < U; u += 2) {
      const int i = ii[u], j = jj[u], i2 = ii[u + 1], j2 = jj[u + 1];
      Pk<C> y = pk2(x[u], x[u + 1]);
      if (has_m) {
        Pk<C> cj = pk2(cvn[j == kmap ? last : j], cvn[j2 == kmap ? last : j2]);
        if constexpr (BIG) cj = pk_mul(cj, pk2(nig, nig));
        y = pk_fma(pk2(cv[i == kmap ? last : i], cv[i2 == kmap ? last : i2]), cj, y);
      }
      if (has_p) y = pk_fma(pk2(uv[i], uv[i2]), pk2(uvd[j], uvd[j2]), y);
      C y0 = pk_first(y), y1 = pk_second(y);
      if (has_p) {
        if (i == s || j == s) y0 = i == j ? idl : cneg(uvd[i == s ? j : i]);
        if (i2 == s || j2 == s) y1 = i2 == j2 ? idl : cneg(uvd[i2 == s ? j2 : i2]);
      }
      if (e + u * S < ne) Cp[e + u * S] = y0;
      if (e + (u + 1) * S < ne) Cp[e + (u + 1) * S] = y1;
    }
  }
}

// FP64 rebuild of C^-1, v, y, log|Sigma| and the log-likelihood from the PE list (FP32 mode).
// ok = 0 (state untouched) if C is not numerically positive definite. Arguments are passed by
// value (no address of the caller's locals escapes, so they stay in registers). TW > 1: every warp
// of the team calls (see PeTeam); the outputs are warp 0's.
template <typename T, bool BIG, int L, bool MIX, int TW>
__device__ __noinline__ RefreshOut pe_refresh_part(const DevModel& M, const PeChain<T, BIG, L, MIX> W, typename PeTab<T>::C* Cp,
                                              double* ws, int n_cap, const float* w, double wsq, int n,
                                              int N, const Lanes<L> ln) {
  using C = typename PeTab<T>::C;
  RefreshOut out{0, 0.0, 0.0, 0.0};
  const int wp = TW > 1 ? (int)(threadIdx.x >> 5) : 0, tl = wp * L + ln.sl;  // warp and thread of the team
  constexpr int LT = L * TW;
  const int ws_ld = N > 0 ? N : 1;
  constexpr int SB = BIG ? kSweepBlock : kSweepBlock / 2;  // fewer registers in the compact variant
  const size_t lv = pe_ws_a2(n_cap);
  double* A = ws;                                 // C, then -C^-1 (row-major N x N, lower triangle)
  double* h = A + pe_ws_a2((size_t)n_cap * n_cap);  // A^T y
  double* rowk = h + lv;                          // v
  double* P = rowk + lv;                          // a sweep block's rows before its sweep (N x SB)
  double* Pn = P + (size_t)kSweepBlock * lv;      // the same rows during and after it
  // the block's pivot factors: F[q SB + r] = A_rp / pivot (r != q), F[q SB + q] = 1 / pivot
  double* F = Pn + (size_t)kSweepBlock * lv;
  const double* V = M.V64;
  constexpr bool mix = MIX;
  const double mu = M.cm_mu[0], r = M.cm_r[0];  // the dynode model's (one component)
  // C = diag(r_k) + A^T A (its lower triangle, row-major: entry (i, j) at i N + j for j <= i);
  // lanes over columns, RC rows at a time so that the
  // table loads of the rows overlap. The unrolled forms (BIG: many PEs per chain) cost the
  // caller registers around the call, which the compact variant cannot spare.
  constexpr int RC = BIG ? 4 : 1, RG = BIG ? 4 : 1;
#pragma unroll 1
  for (int j = tl; j < N; j += LT) {
    const int jj = W.list()[j];
#pragma unroll 1
    for (int i0 = j; i0 < N; i0 += RC) {
      double c[RC];
#pragma unroll
      for (int q = 0; q < RC; ++q) {
        const int i = min(i0 + q, N - 1);
        const int ji = W.list()[i];
        const int o = ji - jj;
        c[q] = (o > -M.Lt && o < M.Lt) ? xcorr<double>(M, M.tc64, pe_sup(M, n, ji), o) : 0.0;
      }
#pragma unroll
      for (int q = 0; q < RC; ++q) {
        const int i = i0 + q;
        if (i < N) A[(size_t)i * ws_ld + j] = c[q] + (j == i ? (mix ? M.cm_r[W.le()[i]] : r) : 0.0);
      }
    }
  }
  team_sync<TW>(ln);
  // With y = w - sum_k mu_k a_k: h = A^T y = A^T w - (A^T A) m (m the PEs' means), and
  // y^T y = w^T w - 2 m^T A^T w + m^T A^T A m -- no FP64 copy of y is needed. The dynode
  // model factors its single mean out.
  double awt = 0.0, rst = 0.0;
#pragma unroll 1
  for (int k = tl; k < N; k += LT) {
    const Sup s = pe_sup(M, n, W.list()[k]);
    // the loops' loads go four at a time ahead of their (unchanged) sums
    double a0 = 0.0, a1 = 0.0;
    int i = s.ilo;
#pragma unroll 1
    for (; i + 3 < s.ihi; i += 4) {
      double vv[4], ww[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        vv[u] = V[s.ph + (i + u) * M.R];
        ww[u] = (double)w[s.w0 + i + u];
      }
      a0 = fma(vv[0], ww[0], a0);
      a1 = fma(vv[1], ww[1], a1);
      a0 = fma(vv[2], ww[2], a0);
      a1 = fma(vv[3], ww[3], a1);
    }
#pragma unroll 1
    for (; i + 1 < s.ihi; i += 2) {
      a0 = fma(V[s.ph + i * M.R], (double)w[s.w0 + i], a0);
      a1 = fma(V[s.ph + (i + 1) * M.R], (double)w[s.w0 + i + 1], a1);
    }
    if (i < s.ihi) a0 = fma(V[s.ph + i * M.R], (double)w[s.w0 + i], a0);
    const double aw = a0 + a1;
    auto c_kj = [&](int j) { return *(j <= k ? A + (size_t)k * ws_ld + j : A + (size_t)j * ws_ld + k); };
    int j = 0;
    if (mix) {
      const int ek = W.le()[k];
      const double mk = M.cm_mu[ek];
      double hs = -M.cm_r[ek] * mk;  // (A^T A m)_k = sum_j C_kj m_j - r_k m_k
#pragma unroll 1
      for (; j + 3 < N; j += 4) {
        double cc[4], mm[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          cc[u] = c_kj(j + u);
          mm[u] = M.cm_mu[W.le()[j + u]];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) hs = fma(cc[u], mm[u], hs);
      }
#pragma unroll 1
      for (; j < N; ++j) hs = fma(c_kj(j), M.cm_mu[W.le()[j]], hs);
      h[k] = aw - hs;
      if constexpr (TW > 1) {
        rowk[k] = aw;
        P[k] = hs;
      } else {
        awt = fma(mk, aw, awt);
        rst = fma(mk, hs, rst);
      }
    } else {
      double rs = -r;
#pragma unroll 1
      for (; j + 3 < N; j += 4) {
        double cc[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) cc[u] = c_kj(j + u);
#pragma unroll
        for (int u = 0; u < 4; ++u) rs += cc[u];
      }
#pragma unroll 1
      for (; j < N; ++j) rs += c_kj(j);
      h[k] = fma(-mu, rs, aw);
      if constexpr (TW > 1) {
        rowk[k] = aw;
        P[k] = rs;
      } else {
        awt += aw;
        rst += rs;
      }
    }
  }
  if constexpr (TW > 1) {  // the sums in the order in which one warp adds them
    team_bar();
#pragma unroll 1
    for (int k = ln.sl; k < N; k += L) {
      const double aw = rowk[k], rs = P[k];
      if (mix) {
        const double mk = M.cm_mu[W.le()[k]];
        awt = fma(mk, aw, awt);
        rst = fma(mk, rs, rst);
      } else {
        awt += aw;
        rst += rs;
      }
    }
  }
  awt = wsum(awt, ln);
  rst = wsum(rst, ln);
  // (roundings written out, so that every instance of this function gives the same bits)
  const double yy = mix ? fma(-2.0, awt, wsq) + rst : fma(mu * mu, rst, fma(-2.0 * mu, awt, wsq));
  // the FP32 residual, each sample summed in FP64 over the PEs that cover it, in list order: PE
  // by PE with lanes over its support samples, into an FP64 copy of the window held in the
  // sweep's panel buffers (free until the sweep); sample by sample where the window does not fit
  // (and by a team, whose threads have few samples each)
  if (TW == 1 && n <= 2 * kSweepBlock * (int)lv) {
    double* yd = P;  // P and Pn are contiguous
#pragma unroll 1
    for (int x = ln.sl; x < n; x += L) yd[x] = (double)w[x];
    __syncwarp(ln.gm);
#pragma unroll 1
    for (int k = 0; k < N; ++k) {
      const Sup s = pe_sup(M, n, W.list()[k]);
      const double mk = mix ? -M.cm_mu[W.le()[k]] : -mu;
#pragma unroll 1
      for (int i = s.ilo + ln.sl; i < s.ihi; i += L) yd[s.w0 + i] = fma(mk, V[s.ph + i * M.R], yd[s.w0 + i]);
      __syncwarp(ln.gm);
    }
#pragma unroll 1
    for (int x = ln.sl; x < n; x += L) W.y()[x] = (T)yd[x];
  } else {
#pragma unroll 1
    for (int x = tl; x < n; x += LT) {
      double yv = (double)w[x];
#pragma unroll 1
      for (int k = 0; k < N; ++k) {
        const int idx = x * M.R - W.list()[k];
        if (idx >= 0 && idx < M.Lt) yv = fma(mix ? -M.cm_mu[W.le()[k]] : -mu, V[idx], yv);
      }
      W.y()[x] = (T)yv;
    }
  }
  team_sync<TW>(ln);
  // Inversion by the symmetric sweep operator (Gauss-Jordan with diagonal pivots, kept
  // symmetric): sweeping pivot p maps A_pp -> -1/A_pp, A_pj -> A_pj/A_pp, A_ip -> A_ip/A_pp and
  // A_ij -> A_ij - A_ip A_pj/A_pp. Sweeps commute, sweeping every index leaves -C^-1, and only
  // the lower triangle is kept. The pivots are C's LDL^T pivots (all positive for SPD C):
  // log|C| = sum log pivot, kept as mantissa x 2^exponent. Pivots go SB at a time with one pass
  // over the matrix per block K = [k0, k1): the block's rows A_K. (the panel) are swept first --
  // they change only through their own entries -- then every other entry (i, j), i, j outside K,
  // takes the rank-SB update A_ij -= sum_q P_iq G_qj, with P_i. = A_Ki before the sweep and
  // G_.j = A_Kj after it. Within the panel, the diagonal block A_KK depends on nothing else, so
  // it is swept first and its pivots and factors recorded; each other column A_Kj then takes
  // them in turn (the same operations in the same order as sweeping the panel pivot by pivot).
  double pm = 1.0;
  int pe = 0;
#pragma unroll 1
  for (int k0 = 0; k0 < N; k0 += SB) {
    const int nb = min(SB, N - k0), k1 = k0 + nb;
    // the diagonal block A_KK swept on its own, lane r holding its row r in full; each pivot's
    // row goes to the other lanes by shuffles
    const int rl = ln.sl;
    if (TW == 1 || wp == 0) {
      bool bad = false;
      double kr[SB];
#pragma unroll
      for (int c = 0; c < SB; ++c)
        kr[c] = (rl < nb && c < nb)
                    ? *(c <= rl ? A + (size_t)(k0 + rl) * ws_ld + k0 + c : A + (size_t)(k0 + c) * ws_ld + k0 + rl)
                    : 0.0;
#pragma unroll
      for (int q = 0; q < SB; ++q) {
        if (q < nb) {
          const double piv = __shfl_sync(ln.gm, kr[q], q, L);
          if (!(piv > 0.0) || !isfinite(piv)) {
            if constexpr (TW == 1) return out;
            bad = true;
            break;
          }
          const double ip = 1.0 / piv;
          int ex;
          pm *= frexp(piv, &ex);
          pe += ex;
          pm = frexp(pm, &ex);
          pe += ex;
          const double fr = kr[q] * ip;  // A_rp / pivot for this lane's row r
          double aq[SB];
#pragma unroll
          for (int c = 0; c < SB; ++c) aq[c] = __shfl_sync(ln.gm, kr[c], q, L);
#pragma unroll
          for (int c = 0; c < SB; ++c)
            kr[c] = (rl == q) ? (c == q ? -ip : aq[c] * ip) : (c == q ? fr : fma(-fr, aq[c], kr[c]));
          if (rl < nb) F[q * SB + rl] = (rl == q) ? ip : fr;
        }
      }
      if (rl < nb) {
#pragma unroll
        for (int c = 0; c < SB; ++c)
          if (c <= rl) A[(size_t)(k0 + rl) * ws_ld + k0 + c] = kr[c];
      }
      if constexpr (TW > 1) {
        if (ln.sl == 0) pe_team<T>(M).ok = !bad;
      }
    }
    team_sync<TW>(ln);
    if constexpr (TW > 1) {
      if (!pe_team<T>(M).ok) return out;
    }
    // the panel A_Kj of every column j outside the block: P_j. keeps it as it was, then the
    // block's pivots are applied to it in registers and it goes to Pn_j. and back into A
#pragma unroll 1
    for (int j = tl; j < N; j += LT) {
      if (j >= k0 && j < k1) continue;
      double b[SB];
#pragma unroll
      for (int q = 0; q < SB; ++q)
        b[q] = q < nb ? *(j > k0 ? A + (size_t)j * ws_ld + k0 + q : A + (size_t)(k0 + q) * ws_ld + j) : 0.0;
#pragma unroll
      for (int q = 0; q < SB; ++q) P[(size_t)j * SB + q] = b[q];
#pragma unroll
      for (int q = 0; q < SB; ++q) {
        if (q < nb) {
          const double apj = b[q];
#pragma unroll
          for (int r = 0; r < SB; ++r)
            if (r < nb) b[r] = (r == q) ? apj * F[q * SB + q] : fma(-F[q * SB + r], apj, b[r]);
        }
      }
#pragma unroll
      for (int q = 0; q < SB; ++q) {
        Pn[(size_t)j * SB + q] = b[q];
        if (q < nb) *(j < k0 ? A + (size_t)(k0 + q) * ws_ld + j : A + (size_t)j * ws_ld + k0 + q) = b[q];
      }
    }
    team_sync<TW>(ln);
    // every entry (i, j), i >= j, outside the block's rows and columns: lanes over a group of L
    // columns, the rows in step across the lanes (a row's loads coalesce and its P row is one
    // broadcast), RG rows at a time so that their loads overlap
#pragma unroll 1
    for (int j0 = 0; j0 < N; j0 += L) {
      const int j = j0 + ln.sl;
      const bool jv = j < N && (j < k0 || j >= k1);
      double g[SB];
#pragma unroll
      for (int q = 0; q < SB; ++q) g[q] = jv ? Pn[(size_t)j * SB + q] : 0.0;
      // the column group's rows: [j0, k0) above the block, then [max(j0, k1), N) below it; the
      // next RG rows' entries are loaded while the current ones are updated
      const int nA = max(0, k0 - j0), s2 = max(j0, k1), nr = nA + max(0, N - s2);
      auto row = [&](int t) { return t < nA ? j0 + t : s2 + (t - nA); };
      double xn[RG];
#pragma unroll
      for (int t = 0; t < RG; ++t) {
        const int t1 = wp * RG + t, r = row(t1);
        xn[t] = (jv && t1 < nr && r >= j) ? A[(size_t)r * ws_ld + j] : 0.0;
      }
#pragma unroll 1
      for (int t0 = wp * RG; t0 < nr; t0 += TW * RG) {
        double x[RG];
        int rr[RG];
#pragma unroll
        for (int t = 0; t < RG; ++t) {
          x[t] = xn[t];
          rr[t] = row(min(t0 + t, nr - 1));
          const int tt = t0 + TW * RG + t, r = row(tt);
          xn[t] = (jv && tt < nr && r >= j) ? A[(size_t)r * ws_ld + j] : 0.0;
        }
#pragma unroll
        for (int t = 0; t < RG; ++t) {
          const double2* Pi = reinterpret_cast<const double2*>(P + (size_t)rr[t] * SB);
#pragma unroll
          for (int q = 0; q < SB / 2; ++q) {
            const double2 pq = Pi[q];
            x[t] = fma(-pq.x, g[2 * q], x[t]);
            x[t] = fma(-pq.y, g[2 * q + 1], x[t]);
          }
        }
#pragma unroll
        for (int t = 0; t < RG; ++t)
          if (jv && t0 + t < nr && rr[t] >= j) A[(size_t)rr[t] * ws_ld + j] = x[t];
      }
    }
    team_sync<TW>(ln);
  }
  const double logdetC = fma((double)pe, 0.6931471805599453, log(pm));
  // v = C^-1 h = -A h (entry (i, j) of the symmetric A from the lower triangle; lanes over rows;
  // BIG: four partial sums)
#pragma unroll 1
  for (int i = tl; i < N; i += LT) {
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    auto a_ij = [&](int j) { return *(j < i ? A + (size_t)i * ws_ld + j : A + (size_t)j * ws_ld + i); };
    int j = 0;
#pragma unroll 1
    for (; BIG && j + 3 < N; j += 4) {
      s0 = fma(a_ij(j), h[j], s0);
      s1 = fma(a_ij(j + 1), h[j + 1], s1);
      s2 = fma(a_ij(j + 2), h[j + 2], s2);
      s3 = fma(a_ij(j + 3), h[j + 3], s3);
    }
#pragma unroll 1
    for (; j < N; ++j) s0 = fma(a_ij(j), h[j], s0);
    rowk[i] = -((s0 + s1) + (s2 + s3));
  }
  team_sync<TW>(ln);
  double hv = 0.0;
#pragma unroll 1
  for (int i = ln.sl; i < N; i += L) hv = fma(h[i], rowk[i], hv);
  hv = wsum(hv, ln);
  // drift of the incremental state, then the refreshed state (packed lower triangle)
  double dmax = 0.0, amax = 0.0;
  constexpr int RD = BIG ? 4 : 1;  // entries per lane at a time, their loads ahead of their stores
  const int nt = tri(N);
#pragma unroll 1
  for (int e0 = tl; e0 < nt; e0 += RD * LT) {
    double nv[RD], ov[RD];
#pragma unroll
    for (int u = 0; u < RD; ++u) {
      const int e = e0 + u * LT;
      nv[u] = ov[u] = 0.0;
      if (e < nt) {
        int i, j;
        untri(e, i, j);
        nv[u] = -A[(size_t)i * ws_ld + j];
        ov[u] = c64(Cp[e]);
      }
    }
#pragma unroll
    for (int u = 0; u < RD; ++u) {
      const int e = e0 + u * LT;
      if (e < nt) {
        dmax = fmax(dmax, fabs(nv[u] - ov[u]));
        amax = fmax(amax, fabs(nv[u]));
        Cp[e] = cfrom64<C>(nv[u]);
      }
    }
  }
  if constexpr (TW > 1) {  // the warps' largest drift and entry; what follows is warp 0's
    PeTeam<C>& tm = pe_team<T>(M);
    dmax = wmax(dmax, ln); amax = wmax(amax, ln);
    if (ln.sl == 0) {
      tm.red[wp][0] = dmax;
      tm.red[wp][1] = amax;
    }
    team_bar();
    if (wp > 0) return out;
#pragma unroll 1
    for (int q = 1; q < TW; ++q) {
      dmax = fmax(dmax, tm.red[q][0]);
      amax = fmax(amax, tm.red[q][1]);
    }
  }
  double vd = 0.0, va = 0.0;
#pragma unroll 1
  for (int i = ln.sl; i < N; i += L) {
    vd = fmax(vd, fabs(rowk[i] - c64(W.v()[i])));
    va = fmax(va, fabs(rowk[i]));
    W.v()[i] = cfrom64<C>(rowk[i]);
  }
  dmax = wmax(dmax, ln); amax = wmax(amax, ln); vd = wmax(vd, ln); va = wmax(va, ln);
  __syncwarp(ln.gm);
  // sum_k log r_k
  double lrs = N * M.cm_lr[0];
  if (mix) {
    lrs = 0.0;
#pragma unroll 1
    for (int k = ln.sl; k < N; k += L) lrs += M.cm_lr[W.le()[k]];
    lrs = wsum(lrs, ln);
  }
  out.ok = 1;
  out.drift = fmax(amax > 0.0 ? dmax / amax : 0.0, va > 0.0 ? vd / fmax(va, 1.0) : 0.0);
  out.logdet = fma((double)n, M.log_se2, logdetC) - lrs;
  out.logL = -0.5 * (fma((double)n, kLog2Pi, out.logdet) + (yy - hv) / M.se2);
  return out;
}

template <typename T, bool BIG, int L, bool MIX>
__device__ __noinline__ void team_refresh(const DevModel& M, const PeChain<T, BIG, L, MIX> W, const Lanes<L> ln) {
  const PeTeam<typename PeTab<T>::C>& tm = pe_team<T>(M);
  pe_refresh_part<T, BIG, L, MIX, kTeam>(M, W, tm.Cp, tm.ws, M.n_cap, tm.w, tm.wsq, tm.n, tm.N, ln);
}
// The rebuild as the chain's first warp calls it.
template <typename T, bool BIG, int L, bool MIX, int TW>
__device__ __forceinline__ RefreshOut pe_refresh(const DevModel& M, const PeChain<T, BIG, L, MIX> W, typename PeTab<T>::C* Cp,
                                                 double* ws, int n_cap, const float* w, double wsq, int n, int N,
                                                 const Lanes<L> ln) {
  if constexpr (TW > 1) {
    PeTeam<typename PeTab<T>::C>& tm = pe_team<T>(M);
    if (ln.sl == 0) {
      tm.op = kOpRefresh;
      tm.Cp = Cp; tm.ws = ws; tm.w = w; tm.wsq = wsq; tm.n = n; tm.N = N;
    }
    team_bar();
    const RefreshOut ro = pe_refresh_part<T, BIG, L, MIX, TW>(M, W, Cp, ws, n_cap, w, wsq, n, N, ln);
    team_bar();
    return ro;
  } else {
    return pe_refresh_part<T, BIG, L, MIX, 1>(M, W, Cp, ws, n_cap, w, wsq, n, N, ln);
  }
}
// The other warps of a team, until the CTA has no chain left.
template <typename T, bool BIG, int L, bool MIX>
__device__ __noinline__ void team_help(const DevModel& M, const PeChain<T, BIG, L, MIX> W, const Lanes<L> ln) {
  const PeTeam<typename PeTab<T>::C>& tm = pe_team<T>(M);
  for (;;) {
    team_bar();
    const int op = tm.op;
    if (op == kOpExit) return;
    if (op == kOpScore) team_score<T, BIG, L, MIX>(M, W);
    else if (op == kOpRows) team_rows<T, BIG, L, MIX>(M, W);
    else if (op == kOpUpdate) team_update<T, BIG, L, MIX>(M, W);
    else team_refresh<T, BIG, L, MIX>(M, W, ln);
    team_bar();
  }
}

// Scalars of an accepted move, from the proposal and its scoring.
template <typename C> struct PeMove {
  int jump, kk, jp, jm, np;
  int em, ep;  // charge components of the removed and the new PE
  C aa, vk, ay;
  Sup sp;
};

template <typename C> struct AcceptOut {
  C* Cp;
  int cap, N;
  unsigned long long words;
  C idl;  // 1 / delta, delta the Schur complement of the new PE (birth, update)
};

// Apply an accepted move to C^-1, v, y and the PE list. Returns the new N, and the new C^-1 storage
// when it moves from the shared tile (capacity cap PEs) to the global slot (n_cap PEs). Inlined in
// the step loop (the call's moves and the model constants' generic loads cost it 4 %).
template <typename T, bool BIG, int L, bool MIX, int TW>
__device__ __forceinline__ AcceptOut<typename PeTab<T>::C> pe_accept(const DevModel& M, const PeChain<T, BIG, L, MIX> W,
                                                                  typename PeTab<T>::C* Cp, int cap,
                                                                  typename PeTab<T>::C* Cg,
                                                                  const PeMove<typename PeTab<T>::C> mv, int n, int N,
                                                                  const Lanes<L> ln) {
  // With c = row k of C^-1 (death, update), gamma = c_k, and u' = C_-^-1 b~ (birth, update: C_- is
  // C without PE k for an update, C itself for a birth; b~ is b without its k entry),
  // delta = r + |a_+|^2 - b~^T u':
  //   C'_ij = C_{m(i) m(j)} - c_m(i) c_m(j) / gamma + u'_i u'_j / delta   (i, j != s),
  //   C'_is = -u'_i / delta,  C'_ss = 1 / delta,
  // where s is the slot of the new PE (N for a birth, k for an update; none for a death) and
  // m moves the last PE into slot k for a death (identity otherwise). A birth has no c term, a
  // death no u' term. v changes the same way.
  // The removed PE has mean mu_- (component em), the new one mean mu_+ and r_+ (component ep).
  using C = typename PeTab<T>::C;
  const int em = MIX ? mv.em : 0, ep = MIX ? mv.ep : 0;
  const C mum = c_mu<C>(M, em), mup = c_mu<C>(M, ep), rrp = c_r<C>(M, ep);
  const T mumT = CmT<T>::mu(M, em), mupT = CmT<T>::mu(M, ep);
  const int R = M.R, np = mv.np, kk = mv.kk, jump = mv.jump;
  const bool has_m = jump != 0, has_p = jump != 1;
  const int Nout = N + (jump == 0 ? 1 : (jump == 1 ? -1 : 0));
  const int s = jump == 0 ? N : (jump == 2 ? kk : -1);
  const int last = N - 1;
  C* const cvn = BIG ? W.cv() : W.cvn();  // c / -gamma (BIG has no room for it: taken per entry)
  C* const uvd = W.ovb();  // u' / delta, once b is no longer read
  const T* const Vs = pe_V<T>();
  const unsigned short* const tij = pe_tij();
  const bool team = TW > 1 && N > kSpecPes;  // the team's warps take part in the passes over C^-1
  C ig = czero<C>(), idl = czero<C>(), t = czero<C>(), fv = czero<C>(), nig = czero<C>();
  C bvf = czero<C>(), bk = czero<C>(), wk = czero<C>();
  if (has_p) {
    // b^T v in full state precision (the scoring used an FP32 sum) and, for an update, the
    // entry of b for PE k, in one butterfly; then b~ in b's place
#pragma unroll 1
    for (int a = ln.sl; a < np; a += L) {
      bvf = cfma(W.ovb()[a], W.v()[W.ovi()[a]], bvf);
      if (opaque(jump == 2) && W.ovi()[a] == kk) {
        bk = W.ovb()[a];
        W.ovb()[a] = czero<C>();
      }
    }
    csum2_m(bvf, bk, np, ln);
    if (team) {
      if constexpr (TW > 1) {
        PeTeam<C>& tm = pe_team<T>(M);
        if (ln.sl == 0) { tm.op = kOpRows; tm.Cp = Cp; tm.N = N; tm.np = np; }
        team_bar();
        team_rows<T, BIG, L, MIX>(M, W);
        team_bar();
      }
    } else if constexpr (BIG) {
      __syncwarp(ln.gm);
#pragma unroll 1
      for (int i = ln.sl; i < N; i += L) W.uv()[i] = dot_row4<C>(Cp, i, W.ovi(), W.ovb(), np);
    } else if (N > L) {
      // two rows per lane, i and i + L
      __syncwarp(ln.gm);
#pragma unroll 1
      for (int i = ln.sl; i < N; i += 2 * L) {
        const int i2 = min(i + L, N - 1);
        Pk<C> acc = pk2(czero<C>(), czero<C>());
#pragma unroll 1
        for (int a = 0; a < np; ++a) {
          const int q = W.ovi()[a];
          const C b = W.ovb()[a];
          acc = pk_fma(pk2(Cp[pk(i, q)], Cp[pk(i2, q)]), pk2(b, b), acc);
        }
        W.uv()[i] = pk_first(acc);
        if (i + L < N) W.uv()[i + L] = pk_second(acc);
      }
    } else {
      // 2^ls lanes per row (2^ls N <= L), each summing every 2^ls-th term of the row's product with
      // b~, then a butterfly over them: the dependent chain of a row is np / 2^ls terms long
      int ls = 0;
#pragma unroll 1
      while (ls < 3 && (2 * N << ls) <= L) ++ls;
      const int rq = ln.sl >> ls, qq = ln.sl & ((1 << ls) - 1), rpp = L >> ls;
      __syncwarp(ln.gm);
#pragma unroll 1
      for (int i0 = 0; i0 < N; i0 += rpp) {
        const int i = i0 + rq;
        C acc = czero<C>();
        if (i < N) {
#pragma unroll 1
          for (int a = qq; a < np; a += 1 << ls) acc = cfma(Cp[pk(i, W.ovi()[a])], W.ovb()[a], acc);
        }
#pragma unroll 1
        for (int o = 1; o < 1 << ls; o <<= 1) acc = cadd(acc, cshfl_xor<L>(acc, o, ln.gm));
        if (i < N && qq == 0) W.uv()[i] = acc;
      }
    }
    if (ln.sl == 0 && jump == 0) W.uv()[N] = czero<C>();  // slot N of a birth (N < n_cap)
  }
  if (has_m) {
#pragma unroll 1
    for (int i = ln.sl; i < N; i += L) W.cv()[i] = Cp[pk(kk, i)];
    __syncwarp(ln.gm);
    ig = crcp(W.cv()[kk]);
    nig = cneg(ig);
    fv = cmul(cadd(mv.vk, mum), ig);
  } else {
    __syncwarp(ln.gm);
  }
  if (has_p) {
    if (jump == 2) {
      // u' = w - c w_k / gamma on the system without PE k
      wk = W.uv()[kk];
      const C wkg = cneg(cmul(wk, ig));
      __syncwarp(ln.gm);  // every lane has read w_k
#pragma unroll 1
      for (int i = ln.sl; i < N; i += L) W.uv()[i] = (i == kk) ? czero<C>() : cfma(W.cv()[i], wkg, W.uv()[i]);
      __syncwarp(ln.gm);
    }
    C bu = czero<C>();
#pragma unroll 1
    for (int a = ln.sl; a < np; a += L) bu = cfma(W.ovb()[a], W.uv()[W.ovi()[a]], bu);
    bu = csum_m(bu, np, ln);
    idl = crcp(csub(cadd(rrp, mv.aa), bu));
    // t = (b~^T v_- - mu_+ b~^T u' - h_new) / delta with v_- = v after removing PE k and h_new
    // the new PE's a^T y on the final residual (PE k removed, the new PE added)
    const C bvm = jump == 2 ? csub(csub(bvf, cmul(bk, mv.vk)), cmul(wk, fv)) : bvf;
    const C hnew = csub(cadd(mv.ay, cmul(mum, bk)), cmul(mup, mv.aa));
    t = cmul(csub(csub(bvm, cmul(mup, bu)), hnew), idl);
  }
  // the factors c / -gamma and u' / delta, once per PE instead of once per entry
  __syncwarp(ln.gm);  // b and its indices are read
#pragma unroll 1
  for (int i = ln.sl; i <= N; i += L) {
    if (!BIG && opaque(has_m) && i < N) cvn[i] = cmul(W.cv()[i], nig);
    if (opaque(has_p) && i < Nout) uvd[i] = cmul(W.uv()[i], idl);
  }
  if (jump == 0 && N + 1 > cap && Cp != Cg) {  // the tile is full: move C^-1 to the global slot
#pragma unroll 1
    for (int e = ln.sl; e < tri(N); e += L) Cg[e] = Cp[e];
    Cp = Cg;
    cap = M.n_cap;
  }
  __syncwarp(ln.gm);
  // C^-1 in place over the packed triangle, all lanes on consecutive entries. A pass reads an
  // entry only where it writes it, or in the last row for a death (which it does not write).
  const int kmap = jump == 1 ? kk : -1;  // the slot the last PE moves into
  const int ne = tri(Nout);               // rows 0 .. Nout-1
  auto src = [&](int i, int j) { return pk(i == kmap ? last : i, j == kmap ? last : j); };
  auto update2 = [&](int i, int j, C& x, int i2, int j2, C& x2) {
    Pk<C> y = pk2(x, x2);
    if (opaque(has_m)) {
      Pk<C> cj = pk2(cvn[j == kmap ? last : j], cvn[j2 == kmap ? last : j2]);
      if constexpr (BIG) cj = pk_mul(cj, pk2(nig, nig));
      y = pk_fma(pk2(W.cv()[i == kmap ? last : i], W.cv()[i2 == kmap ? last : i2]), cj, y);
    }
    if (opaque(has_p)) y = pk_fma(pk2(W.uv()[i], W.uv()[i2]), pk2(uvd[j], uvd[j2]), y);
    x = pk_first(y);
    x2 = pk_second(y);
    if (opaque(has_p)) {
      if (i == s || j == s) x = i == j ? idl : cneg(uvd[i == s ? j : i]);
      if (i2 == s || j2 == s) x2 = i2 == j2 ? idl : cneg(uvd[i2 == s ? j2 : i2]);
    }
  };
  TriWalk<L> tw;
  int e = ln.sl;
  if (team) {
    if constexpr (TW > 1) {
      PeTeam<C>& tm = pe_team<T>(M);
      if (ln.sl == 0) { tm.op = kOpUpdate; tm.Cp = Cp; tm.N = N; tm.jump = jump; tm.kk = kk; tm.nig = nig; tm.idl = idl; }
      team_bar();
      team_update<T, BIG, L, MIX>(M, W);
      team_bar();
      e = ne;
    }
  } else if constexpr (BIG) {
    // C^-1 in the global slot: four entries per lane and pass, all read before any is written
    // (each read is the entry itself or one in the unwritten last row), so that the loads of a
    // pass overlap
#pragma unroll 1
    for (; e - ln.sl + 4 * L <= ne; e += 4 * L) {
      int ii[4], jj[4];
      C x[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        tw.at(tij, e + q * L);
        ii[q] = tw.i;
        jj[q] = tw.j;
        x[q] = Cp[src(tw.i, tw.j)];
      }
#pragma unroll
      for (int q = 0; q < 4; q += 2) update2(ii[q], jj[q], x[q], ii[q + 1], jj[q + 1], x[q + 1]);
#pragma unroll
      for (int q = 0; q < 4; ++q) Cp[e + q * L] = x[q];
    }
  }
  // entries e and e + L of a lane, both read before either is written
#pragma unroll 1
  for (; e < ne; e += 2 * L) {
    tw.at(tij, e);
    const int i = tw.i, j = tw.j;
    const bool two = e + L < ne;
    if (two) tw.at(tij, e + L);
    C x = Cp[src(i, j)], x2 = Cp[src(tw.i, tw.j)];
    update2(i, j, x, tw.i, tw.j, x2);
    Cp[e] = x;
    if (two) Cp[e + L] = x2;
  }
  // v' = v_m - c_m fv + (t - mu_+) u', v'_s = -t
  const C tm = csub(t, mup), nfv = cneg(fv);
#pragma unroll 1
  for (int i = ln.sl; i < Nout; i += L) {
    const int mi = (i == kmap) ? last : i;
    C x = i < N ? W.v()[mi] : czero<C>();
    if (opaque(has_m)) x = cfma(W.cv()[mi], nfv, x);
    if (opaque(has_p)) x = i == s ? cneg(t) : cfma(tm, W.uv()[i], x);
    W.v()[i] = x;
  }
  // residual and PE list
  unsigned long long wds = (unsigned long long)N * np + 2ull * tri(Nout) + 2ull * Nout;
  if (has_m) {
    const Sup sm = pe_sup(M, n, mv.jm);
#pragma unroll 1
    for (int i = sm.ilo + ln.sl; i < sm.ihi; i += L) W.y()[sm.w0 + i] += mumT * Vs[sm.ph + i * R];
    wds += 2 * (sm.ihi - sm.ilo) + N;
    __syncwarp(ln.gm);
  }
  if (has_p) {
    const Sup sp = mv.sp;
#pragma unroll 1
    for (int i = sp.ilo + ln.sl; i < sp.ihi; i += L) W.y()[sp.w0 + i] -= mupT * Vs[sp.ph + i * R];
    wds += 2 * (sp.ihi - sp.ilo);
  }
  if (ln.sl == 0) {
    if (jump == 0) {
      W.list()[N] = mv.jp;
      if constexpr (MIX) W.le()[N] = (unsigned char)ep;
    } else if (jump == 1) {
      W.list()[kk] = W.list()[last];
      if constexpr (MIX) W.le()[kk] = W.le()[last];
    } else {
      W.list()[kk] = mv.jp;
      if constexpr (MIX) W.le()[kk] = (unsigned char)ep;
    }
  }
  __syncwarp(ln.gm);
  return AcceptOut<C>{Cp, cap, Nout, wds, idl};
}

// The same out of line, for the births of an initial state.
template <typename T, bool BIG, int L, bool MIX>
__device__ __noinline__ AcceptOut<typename PeTab<T>::C> pe_accept_call(const DevModel& M, const PeChain<T, BIG, L, MIX> W,
                                                                       typename PeTab<T>::C* Cp, int cap,
                                                                       typename PeTab<T>::C* Cg,
                                                                       const PeMove<typename PeTab<T>::C> mv, int n,
                                                                       int N, const Lanes<L> ln) {
  return pe_accept<T, BIG, L, MIX, 1>(M, W, Cp, cap, Cg, mv, n, N, ln);
}

// The 2x2 algebra of Eqs. (16)-(18) in the scoring precision: log D, Delta nu and the status bits
// of a move with components em (removed) and ep (new); r1 = 1 - q_- m_--.
template <typename T> struct PeScore {
  T dT, dnu;
  int st;
  bool ok;
};
template <typename T, bool MIX>
__device__ __forceinline__ PeScore<T> pe_score(const DevModel& M, int e_m, int e_p, T em, T mmm, T mmp, T mpp, T gm, T gp) {
  PeScore<T> o;
  o.dT = (T)0; o.dnu = (T)NAN; o.st = 0; o.ok = false;
  // det(I + Lambda M), Lambda = diag(-q_-, q_+) (q = sigma_e^2 of the PE concerned), with
  // 1 - q_- m_-- = em; lambda = (-mu_-, mu_+) (Eq. (DeltaU), Appendix A.2)
  const T qm = CmT<T>::q(M, e_m), qp = CmT<T>::q(M, e_p);
  const T mum = CmT<T>::mu(M, e_m), mup = CmT<T>::mu(M, e_p);
  const T Dd = em * ((T)1 + qp * mpp) + qm * qp * mmp * mmp;
  if (!(Dd > (T)0)) {
    o.st = FSMP_ST_BADDET;
  } else {
    const T iD = (T)1 / Dd;
    const T B11 = -qm * ((T)1 + qp * mpp) * iD, B12 = qm * qp * mmp * iD, B22 = qp * em * iD;
    // rho = g - M lambda; dR = -2 lambda^T g + lambda^T M lambda - rho^T B rho
    const T rm = gm + mum * mmm - mup * mmp, rp = gp + mum * mmp - mup * mpp;
    // (rho^T B rho with its roundings written out: which products a compiler fuses depends on the
    // code around them, and a chain's decisions follow the last bit; results stay those of the
    // forms it chose when each mode was checked)
    const T b1 = B11 * rm, b2 = (T)2 * B12 * rm;
    const T rBr = fma(B22 * rp, rp, sizeof(T) == 4 && !MIX ? fma(b1, rm, b2 * rp) : fma(b2, rp, b1 * rm));
    const T dR = (T)-2 * (mup * gp - mum * gm) + (mum * mum * mmm - (T)2 * mum * mup * mmp + mup * mup * mpp) - rBr;
    o.dT = log(Dd);
    o.dnu = (T)-0.5 * (o.dT + dR);
    if (!isfinite(o.dnu)) o.st = FSMP_ST_NONFINITE;
    else o.ok = true;
  }
  return o;
}

// Random draws of the L steps from `step` on, lane l taking step + l (Philox4x64-10 keyed by
// (seed, waveform), counter (step, block, 0, 0); Box-Muller for the two shifts). Out of line:
// it runs once per L steps, and keeping it out of the step loop keeps the loop's code compact.
// FP32 mode takes cos(2 pi u) as cospif(2u), whose argument reduction is exact.
template <typename T, bool BIG, int L, bool MIX>
__device__ __noinline__ void pe_draw(const DevModel& M, const PeChain<T, BIG, L, MIX> W, uint64_t seed, uint64_t wf_id, int step,
                                     const Lanes<L> ln) {
  constexpr bool fp32 = sizeof(T) == 4;
  PeRand<T, MIX> rd;
#pragma unroll 1
  for (int blk = 0; blk < (MIX ? 3 : 2); ++blk) {
    uint64_t c[4] = {(uint64_t)(step + ln.sl), (uint64_t)blk, 0, 0};
    philox4x64_10(c, seed, wf_id);
    if (blk == 2) {  // MCP component of a born or updated PE
      if constexpr (MIX) rd.ep = pe_draw_comp(M, u01_from_bits(c[0]));
    } else if constexpr (fp32) {
      const float a = u01_float(c[0]), b = u01_float(c[1]), d = u01_float(c[2]), e = u01_float(c[3]);
      if (blk == 0) {
        rd.z1 = (T)(sqrtf(-2.0f * logf(a)) * cospif(2.0f * b));
        rd.lu0 = (T)logf(d);
        rd.u3 = (T)e;
      } else {
        rd.u4 = (T)a;
        rd.z2 = (T)(sqrtf(-2.0f * logf(b)) * cospif(2.0f * d));
        rd.lu = (T)logf(e);
      }
    } else {
      const double a = u01_from_bits(c[0]), b = u01_from_bits(c[1]), d = u01_from_bits(c[2]), e = u01_from_bits(c[3]);
      if (blk == 0) {
        rd.z1 = (T)(sqrt(-2.0 * log(a)) * cos(kTwoPi * b));
        rd.lu0 = (T)log(d);
        rd.u3 = (T)e;
      } else {
        rd.u4 = (T)a;
        rd.z2 = (T)(sqrt(-2.0 * log(b)) * cos(kTwoPi * d));
        rd.lu = (T)log(e);
      }
    }
  }
  W.rnd()[ln.sl] = rd;
  __syncwarp(ln.gm);
}

// Out-of-line pieces of the step that run only when the caller asked for them (a trace record,
// the PE-time histogram), so that their code stays out of the step loop's instruction stream.
__device__ __noinline__ void pe_trace_record(fsmp_trace* t, double la0, double lu0, double la, double lu, double dnu,
                                             int N, int k0, int jump, int flags) {
  fsmp_trace tr;
  tr.la0 = la0; tr.lu0 = lu0; tr.la = la; tr.lu = lu; tr.dnu = dnu;
  tr.N = N; tr.k0 = k0; tr.jump = jump; tr.flags = flags;
  *t = tr;
}
template <typename T, bool BIG, int L, bool MIX>
__device__ __noinline__ void pe_hist_add(const PeChain<T, BIG, L, MIX> W, uint32_t* peh, int N, int T_lo, int width,
                                         uint32_t times, const Lanes<L> ln) {
#pragma unroll 1
  for (int k = ln.sl; k < N; k += L) {
    const int c = W.list()[k] - T_lo;
    if (c >= 0 && c < width) atomicAdd(peh + c, times);
  }
}

// Resident CTAs per SM the registers are cut for. A chain waits on instruction supply (the code it
// runs through is larger than a scheduler's instruction cache, which refills at 16 bytes in 2.6
// cycles), so cut for 2 CTAs a launch does as many steps per second as cut for 4 (uneven windows,
// 20 000 chains x 1000 steps: 58.96 ms against 58.78), each chain faster: that takes the tail off a
// launch that has few chains (MCP mixture, 3000 chains: 18.2 ms against 25.7; pile-up, 600 chains:
// 85.6 against 95.2). The instances then take, in FP32 mode, 168 registers (dynode: 3 CTAs, 12 warps
// on an SM), 213 (its pile-up variant) and 180 (mixture: 2 CTAs each), in FP64 mode 168 to 204, and
// spill nothing. With two chains per warp (L = 16) the half warps wait on each other, and 16 warps are
// better (30 000 low-occupancy chains: 31.5 ms cut for 4 CTAs, 42.9 for 2), although at 128 registers
// a step spills (92 bytes stored, 184 loaded); a team's 4 CTAs too (kTeam; pile-up 252 and 520).
//
// The mixture's chains of more than 40 PEs gain from the L1 that 2 CTAs leave (608 of 50 PEs x 600
// steps: 9.7 ms against 13.6 with 3 CTAs, 5000 of 0.5 to 50 PEs 11.4 against 13.9), but where an SM has
// enough light chains, 12 warps do more steps than 8: so it comes in both (MORE: 168 registers, 3
// CTAs; 16 000 chains: 2 PEs 16.2 -> 13.2 ms, 8 PEs 27.9 -> 23.7, 24 PEs 62.9 -> 58.9, 0.5 to 50
// 33.6 -> 30.9; n_cap 48, 6000 of 16 PEs 17.2 -> 15.2).
constexpr int pe_min_ctas(int L, int TW, bool MORE) { return L == 16 || TW > 1 ? 4 : (MORE ? 3 : 2); }

template <typename T, bool BIG, int L, bool MIX, int TW = 1, bool MORE = false>
__global__ void __launch_bounds__(kPeMaxThreads, pe_min_ctas(L, TW, MORE))
    pe_kernel(const __grid_constant__ DevModel M, const __grid_constant__ BatchView B, const __grid_constant__ PeSlots G) {
  using C = typename PeTab<T>::C;
  constexpr bool fp32 = sizeof(T) == 4;
  const Lanes<L> ln = pe_lanes<L>();
  constexpr int kGroups = 32 / L;  // chains per warp
  static_assert(TW == 1 || (TW == kTeam && L == 32), "a team is the CTA's warps");
  const int cw = TW > 1 ? 0 : (threadIdx.x >> 5) * kGroups + ln.g, nchains = TW > 1 ? 1 : (blockDim.x >> 5) * kGroups;
  const int n_alloc = B.n_max, n_cap = M.n_cap, Ns = G.Ns;
  unsigned short* const tij = pe_tij();
  T* const Vs = pe_V<T>();
  T* const lgN = reinterpret_cast<T*>(pe_smem + (kTabBytes + (unsigned)a16(sizeof(T) * M.Lt)));
  double* const inv1 = reinterpret_cast<double*>(
      pe_smem + (kTabBytes + (unsigned)a16(sizeof(T) * M.Lt) + (unsigned)a16(sizeof(T) * (n_cap + 2))));
#pragma unroll 1
  for (int e = threadIdx.x; e < kTriTab; e += blockDim.x) {
    int i, j;
    untri(e, i, j);
    tij[e] = (unsigned short)(i << 8 | j);
  }
#pragma unroll 1
  for (int m = threadIdx.x; m < M.Lt; m += blockDim.x) Vs[m] = PeTab<T>::V(M)[m];
#pragma unroll 1
  for (int i = threadIdx.x; i < n_cap + 2; i += blockDim.x) {
    lgN[i] = i > 0 ? (fp32 ? (T)logf((float)i) : (T)log((double)i)) : (T)0;
    inv1[i] = i > 0 ? 1.0 / (double)i : 0.0;
  }
  __syncthreads();
  PeChain<T, BIG, L, MIX> W;
  W.vb = (unsigned)a16(sizeof(C) * (size_t)n_cap);
  W.lb = (unsigned)a16(sizeof(int) * (size_t)n_cap);
  W.yb = (unsigned)a16(sizeof(T) * (size_t)n_alloc);
  W.pb = (unsigned)a16(sizeof(T) * (size_t)M.win_extra);
  W.o = (unsigned)(pe_block_bytes<T>(M) + (TW > 1 ? kTeamBytes : 0u) + (size_t)cw * pe_chain_bytes<T, BIG, L, MIX>(n_cap, n_alloc, M.win_extra, Ns));
  if constexpr (TW > 1) {
    if (threadIdx.x >= 32) {
      team_help<T, BIG, L, MIX>(M, W, ln);
      return;
    }
  }
  PeStats& S = W.st();
  const size_t slot = (size_t)blockIdx.x * nchains + cw;
  int* const hist = G.hist + slot * (size_t)(n_cap + 1);
  C* const Cg = G.C ? reinterpret_cast<C*>(G.C) + slot * G.c_stride : nullptr;
  double* const ws = G.ws ? G.ws + slot * G.ws_stride : nullptr;
  const auto* __restrict__ tc = PeTab<T>::tc(M);
  const T ise2T = (T)M.inv_se2;
  constexpr bool mix = MIX;  // MCP charge mixture: per-PE components (else the one dynode model)
  const T Jt = (T)M.J, logJ = (T)M.log_J, inv_gT = (T)M.inv_g;
  const int R = M.R;

  for (;;) {
    int ci = 0;
    if (ln.sl == 0) ci = atomicAdd(G.counter, 1);
    ci = __shfl_sync(ln.gm, ci, 0, L);
    if (ci >= B.n_waveforms) break;
    const int wi = B.order ? B.order[ci] : ci;
    // ------------------------------------------------------------- chain set-up
    const int o0 = B.offsets[wi], n = B.offsets[wi + 1] - o0;
    const float* __restrict__ w = B.samples + o0;
    const double lambda0 = B.lambda0[wi];
    const double t_origin = B.t_origin ? B.t_origin[wi] : 0.0;
    const int T_lo = B.T_lo ? B.T_lo[wi] : 0;
    const int T_hi = B.T_hi ? B.T_hi[wi] : n * R;
    const int k0_lo = (int)ceil((M.t0_lo - t_origin) / M.g - 1e-9);
    const int k0_hi = (int)floor((M.t0_hi - t_origin) / M.g + 1e-9);
    const uint64_t seed = B.seeds ? B.seeds[wi] : B.seed;
    const uint64_t wf_id = B.wf_ids ? B.wf_ids[wi] : B.index_base + (uint64_t)wi;
    const int n_steps = B.n_steps_arr ? B.n_steps_arr[wi] : B.n_steps;
    const int burn_in = B.burn_in_arr ? B.burn_in_arr[wi] : B.burn_in;
    fsmp_summary* out = B.out + wi;
    uint32_t* const peh = B.pe_hist ? B.pe_hist + (size_t)wi * B.pe_hist_width : nullptr;
    fsmp_trace* trace = B.trace ? B.trace + (B.trace_off ? B.trace_off[wi] : (int64_t)wi * n_steps) : nullptr;
    const bool invalid = n < 1 || n > n_alloc || T_hi <= T_lo || k0_hi < k0_lo || !(lambda0 > 0.0) || n_steps < 0 ||
                         burn_in < 0 || ((fp32 || B.z_init) && ws == nullptr) || k0_hi - k0_lo + 1 > M.win_extra ||
                         (Cg == nullptr && Ns < n_cap);
    if (invalid) {
      if (ln.sl == 0) {
        fsmp_summary o;
        o.mean_N = o.var_N = o.mean_t0 = o.var_t0 = o.mean_Q = o.var_Q = o.logL = o.logdet = NAN;
        o.drift_max = 0.0; o.alg_bytes = 0.0; o.lambda_hat = NAN;
        o.mean_wt = o.var_wt = o.mean_we = o.var_we = NAN;
        for (int k = 0; k < 3; ++k) { o.acc[k] = 0; o.prop[k] = 0; }
        o.acc_t0 = o.prop_t0 = o.N_final = o.k0_final = o.n_samples = o.n_refresh = o.reserved = 0;
        o.status = FSMP_ST_INVALID;
        *out = o;
        note_chain_done(B, wi);
      }
      __syncwarp(ln.gm);
      continue;
    }
    int k0;
    {
      const double t0i = B.t0_init ? B.t0_init[wi] : NAN;
      if (!isnan(t0i)) {
        double kq = rint((t0i - t_origin) / M.g);
        kq = fmin(fmax(kq, (double)k0_lo), (double)k0_hi);
        k0 = (int)kq;
      } else {
        k0 = k0_lo + (k0_hi - k0_lo) / 2;
      }
    }
    // log(Phi_T(t0) g) on the t0 grid (-inf where Phi_T = 0), from the FP64 tables
#pragma unroll 1
    for (int k = ln.sl; k <= k0_hi - k0_lo; k += L) {
      const int kq = k0_lo + k;
      const double tot = pe_cphi<double>(M, T_hi - 1 - kq) - pe_cphi<double>(M, T_lo - 1 - kq);
      W.lPhi()[k] = tot > 0.0 ? (fp32 ? (T)logf((float)(tot * M.g)) : (T)log(tot * M.g)) : (T)-INFINITY;
    }
#pragma unroll 1
    for (int k = ln.sl; k <= n_cap; k += L) hist[k] = 0;
#pragma unroll 1
    for (int q = ln.sl; q < kSpec * kCounts; q += L) W.cnt()[q] = 0;
    // empty z: y = w
    double wsq = 0.0;
#pragma unroll 1
    for (int x = ln.sl; x < n; x += L) {
      const float wx = w[x];
      W.y()[x] = (T)wx;
      wsq += (double)wx * (double)wx;
    }
    wsq = wsum(wsq, ln);
    if (ln.sl == 0) {
      for (int k = 0; k < 3; ++k) S.cur[k] = S.sum[2 * k] = S.sum[2 * k + 1] = 0.0;
      S.St = S.Se = 0; S.q_from = 0;
      S.sum[PeStats::kLogdet] = n * M.log_se2;
      S.sum[PeStats::kLogL] = -0.5 * (n * kLog2Pi + S.sum[PeStats::kLogdet] + wsq * M.inv_se2);
      S.wsq = wsq;
      S.drift_max = 0.0;
      S.n_refresh = S.status = S.n_acc_refresh = S.refresh_fail = 0;
    }
    __syncwarp(ln.gm);
    const T log_lambda0 = fp32 ? (T)logf((float)lambda0) : (T)log(lambda0);
    C* Cp = Ns > 0 ? W.Cs(n_cap) : Cg;  // C^-1 (packed), room for cap PEs
    int cap = Ns > 0 ? Ns : n_cap;
    int N = 0;
    if (B.z_init) {
      // a given initial state (LucyDDM, Sec. 2.3): the PE list, each PE of the most probable
      // component, then C^-1, v, y, log|Sigma| and log L from it by the FP64 rebuild
      int ni = min(B.n_init[wi], B.z_stride);
      const bool cut = ni > n_cap;
      if (cut) ni = n_cap;
#pragma unroll 1
      for (int k = ln.sl; k < ni; k += L) {
        W.list()[k] = B.z_init[(size_t)wi * B.z_stride + k];
        if constexpr (MIX) W.le()[k] = (unsigned char)M.cm_mode;
      }
      __syncwarp(ln.gm);
      if (ni > cap) { Cp = Cg; cap = n_cap; }
      if (ni > 0) {
        bool ok = true;
        double ms = 0.0;
        C qs = czero<C>();
        if constexpr (fp32) {
          // FP32 mode: the FP64 rebuild
          const RefreshOut ro = pe_refresh<T, BIG, L, MIX, TW>(M, W, Cp, ws, n_cap, w, S.wsq, n, ni, ln);
          ok = ro.ok != 0;
          if (ok && ln.sl == 0) { S.sum[PeStats::kLogdet] = ro.logdet; S.sum[PeStats::kLogL] = ro.logL; }
        } else {
          // FP64 mode: the PEs born one by one through the accepted-move update in double-double
          // (the FP64 rebuild would leave C^-1 only as accurate as FP64 times its condition
          // number); log|C| is the sum of the log Schur complements
          double lC = 0.0;
#pragma unroll 1
          for (int k = 0; k < ni; ++k) {
            PeMove<C> mv;
            mv.jump = 0; mv.kk = -1; mv.jp = W.list()[k]; mv.jm = -1;
            mv.em = mv.ep = MIX ? M.cm_mode : 0;
            const Sup sp = pe_sup(M, n, mv.jp);
            mv.sp = sp;
            int np = 0;
#pragma unroll 1
            for (int base = 0; base < N; base += L) {
              const int qi = base + ln.sl;
              C bq = czero<C>();
              if (qi < N) {
                const int o = mv.jp - W.list()[qi];
                if (o > -M.Lt && o < M.Lt) bq = xcorr<C>(M, tc, sp, o);
              }
              const bool ov = cnz(bq);
              const unsigned m = gballot(ov, ln);
              if (ov) {
                const int pos = np + __popc(m & ((1u << ln.sl) - 1u));
                W.ovi()[pos] = qi;
                W.ovb()[pos] = bq;
              }
              np += __popc(m);
            }
            __syncwarp(ln.gm);
            mv.np = np;
            mv.aa = xcorr<C>(M, tc, sp, 0);
            T ayp = (T)0;
#pragma unroll 1
            for (int i = sp.ilo + ln.sl; i < sp.ihi; i += L) ayp += Vs[sp.ph + i * R] * W.y()[sp.w0 + i];
            mv.ay = cfromf(wsum(ayp, ln));
            mv.vk = czero<C>();
            const AcceptOut<C> ao = pe_accept_call<T, BIG, L, MIX>(M, W, Cp, cap, Cg, mv, n, N, ln);
            Cp = ao.Cp;
            cap = ao.cap;
            N = ao.N;
            const double dl = c64(ao.idl);
            if (!(dl > 0.0) || !isfinite(dl)) ok = false;
            lC -= log(dl);
          }
          N = 0;
          // log|Sigma| = n log se2 + log|C| - sum_k log r_k; y^T Sigma^-1 y = (y^T y - h^T v) / se2
          double lr = 0.0, yy = 0.0, hv = 0.0;
#pragma unroll 1
          for (int k = ln.sl; k < ni; k += L) {
            lr += M.cm_lr[MIX ? M.cm_mode : 0];
            const Sup s = pe_sup(M, n, W.list()[k]);
            double hk = 0.0;
#pragma unroll 1
            for (int i = s.ilo; i < s.ihi; ++i) hk = fma((double)Vs[s.ph + i * R], (double)W.y()[s.w0 + i], hk);
            hv = fma(hk, c64(W.v()[k]), hv);
          }
#pragma unroll 1
          for (int x = ln.sl; x < n; x += L) yy = fma((double)W.y()[x], (double)W.y()[x], yy);
          lr = wsum(lr, ln); yy = wsum(yy, ln); hv = wsum(hv, ln);
          if (ok && ln.sl == 0) {
            S.sum[PeStats::kLogdet] = n * M.log_se2 + lC - lr;
            S.sum[PeStats::kLogL] = -0.5 * (n * kLog2Pi + S.sum[PeStats::kLogdet] + (yy - hv) * M.inv_se2);
          }
        }
#pragma unroll 1
        for (int i = ln.sl; i < ni; i += L) {
          qs = cadd(qs, W.v()[i]);
          if (mix) ms += M.cm_mu[W.le()[i]];
        }
        qs = csum(qs, ln);
        ms = mix ? wsum(ms, ln) : M.cm_mu[0];
        if (ok) {
          N = ni;
        } else {  // C not numerically positive definite: start empty
#pragma unroll 1
          for (int x = ln.sl; x < n; x += L) W.y()[x] = (T)w[x];
          Cp = Ns > 0 ? W.Cs(n_cap) : Cg;
          cap = Ns > 0 ? Ns : n_cap;
        }
        long long st = 0;
#pragma unroll 1
        for (int k = ln.sl; k < ni; k += L) st += abs(W.list()[k]);
        st = wsum(st, ln);
        if (ln.sl == 0) {
          if (ok) {
            S.St = st;
            S.Se = MIX ? (long long)ni * M.cm_mode : 0;
          } else {
            S.status |= FSMP_ST_BADDET;
          }
        }
        __syncwarp(ln.gm);
        if (ok) set_summaries<MIX>(S, M.g, ni, ms, c64(qs), inv1, ln.sl);
      }
      if (ln.sl == 0 && cut) S.status |= FSMP_ST_CAPACITY;
      __syncwarp(ln.gm);
    }

    for (int step = 0; step < n_steps;) {
      // ---- random draws of the next L steps: lane l takes step step + l
      PeRand<T, MIX>* const rnd = W.rnd();
      if ((step & (L - 1)) == 0) pe_draw<T, BIG, L, MIX>(M, W, seed, wf_id, step, ln);
      // The accepted move of this round (or, one by one, the step made), filled in below
      PeMove<C> mv;
      T dT = (T)0, dnu = (T)NAN;
      int jump = 0, e_m = 0;   // of the step last = step + counted - 1
      bool apply = false, t0_acc = false;
      bool one = true;         // that step is still to be counted
      unsigned words = 0;
      int last;
      if (!BIG && N <= spec_pes<T>()) {
        // ---------------------------------------------- a batch of steps, one per subgroup
        constexpr int gw = L / kSpec;  // lanes of a subgroup
        const int gi = ln.sl / gw, m = ln.sl % gw;
        const int g = min(min(kSpec, n_steps - step), L - (step & (L - 1)));  // steps of the batch
        const bool mine = gi < g;
        const PeRand<T, MIX> rd = rnd[(step + min(gi, g - 1)) & (L - 1)];
        // ---- Gibbs part 1: MH on t0 (Sec. 2.4), the steps in turn; a subgroup keeps its step's k0
        int k0i = k0;
        T la0 = (T)NAN;
        unsigned t0a = 0;  // accepted t0 moves of the batch
        if (M.sample_t0) {
          int kr = k0;
#pragma unroll 1
          for (int i = 0; i < g; ++i) {
            const PeRand<T, MIX>& ri = rnd[(step + i) & (L - 1)];
            const T z1 = ri.z1;
            const int Dm = fp32 ? __float2int_rn((float)(z1 * inv_gT)) : __double2int_rn((double)(z1 * inv_gT));
            const int k0p = kr + Dm;
            T la = (T)0;
            if (Dm != 0) {
              if (k0p < k0_lo || k0p > k0_hi) {
                la = (T)-INFINITY;
              } else {
                T part = (T)0;
#pragma unroll 1
                for (int k = ln.sl; k < N; k += L) {
                  const int j = W.list()[k];
                  part += pe_logphi<T>(M, j - k0p) - pe_logphi<T>(M, j - kr);
                }
                la = wsum(part, ln);
              }
            }
            if (ri.lu0 < la) { kr = k0p; t0a |= 1u << i; }
            if (gi == i) { k0i = kr; la0 = la; }
          }
        }
        // ---- Gibbs part 2: one RJMCMC jump (Sec. 2.4)
        jump = (N == 0) ? 0 : (rd.u3 < Jt ? 0 : (rd.u3 < (T)2 * Jt ? 1 : 2));
        int st = 0, kk = -1, jp = -1, jm = -1, e_p = 0;
        if constexpr (MIX) { e_m = rd.ep; e_p = rd.ep; }
        bool valid = false, noop = false;
        T la_prior = (T)0, la_fixed = (T)-INFINITY;
        const T lphi_t0 = W.lPhi()[k0i - k0_lo];
        const bool birth = mine && jump == 0 && N < n_cap && lphi_t0 > (T)-INFINITY;
        if (jump == 0 && N >= n_cap) st = FSMP_ST_CAPACITY;
        if (gballot(birth, ln)) {
          const int jb = pe_birth_search_sub<T, L>(M, T_lo, T_hi, k0i, rd.u4, birth, ln);
          if (birth) {
            jp = jb;
            valid = jp >= T_lo;
            la_prior = log_lambda0 + lphi_t0 - lgN[N + 1] + (N == 0 ? logJ : (T)0);
          }
        }
        if (mine && jump != 0) {
          kk = fp32 ? __float2int_rd((float)(rd.u4 * (T)N)) : __double2int_rd((double)(rd.u4 * (T)N));
          if (kk >= N) kk = N - 1;
          jm = W.list()[kk];
          if constexpr (MIX) e_m = W.le()[kk];
          if (jump == 1) {
            valid = true;
            e_p = e_m;
            la_prior = -log_lambda0 - lphi_t0 + lgN[N] - (N == 1 ? logJ : (T)0);
          } else {
            const int Dm = fp32 ? __float2int_rn((float)(rd.z2 * inv_gT)) : __double2int_rn((double)(rd.z2 * inv_gT));
            const int jpl = jm + Dm;
            if (Dm == 0 && (!MIX || e_p == e_m)) {  // same time and component: an accepted no-op
              noop = true;
              la_fixed = (T)0;
            } else if (jpl >= T_lo && jpl < T_hi) {
              const T lp = pe_logphi<T>(M, jpl - k0i);
              if (!(lp == (T)-INFINITY)) {
                jp = jpl;
                valid = true;
                la_prior = lp - pe_logphi<T>(M, jm - k0i);
              }
            }
          }
        }
        // ---- scoring: PEs overlapping a_+, with b_q = a_q^T a_+
        const bool new_pe = valid && jump != 1;
        Sup sp{0, 0, 0, 0};
        C aa = czero<C>();
        if (new_pe) {
          sp = pe_sup(M, n, jp);
          aa = xcorr<C>(M, tc, sp, 0);
        }
        C* const bs = W.work(gi);
        unsigned char* const ix = W.ix() + gi * kSpecPes;
        int np = 0;
#pragma unroll 1
        for (int base = 0; base < N; base += gw) {
          const int qi = base + m;
          C bq = czero<C>();
          if (new_pe && qi < N) {
            const int o = jp - W.list()[qi];
            if (o > -M.Lt && o < M.Lt) bq = xcorr<C>(M, tc, sp, o);
          }
          const bool ov = cnz(bq);
          const unsigned b = (gballot(ov, ln) >> (gi * gw)) & ((1u << gw) - 1u);
          if (ov) {
            const int pos = np + __popc(b & ((1u << m) - 1u));
            ix[pos] = (unsigned char)qi;
            bs[pos] = bq;
          }
          np += __popc(b);
        }
        __syncwarp(ln.gm);
        // b^T C^-1 b, (C^-1 b)_k of an update, b^T v and a_+^T y: the partial sums x_u that lanes
        // m + u gw (u < 4) of a step made alone have, two at a time, added as its butterfly adds
        // them: (x_0 + x_2) + (x_1 + x_3)
        static_assert(kSpec == 4, "the sums below are of four lanes' partial sums");
        C qp, ck;
        T bvp, ayp;
        {
          const int nt = tri(np);
          Pk<C> hq = pk2(czero<C>(), czero<C>()), hc = hq;
          T ha0 = (T)0, ha1 = (T)0, hb0 = (T)0, hb1 = (T)0;
#pragma unroll 1
          for (int vl = m; vl < L; vl += 2 * gw) {
            T xa0 = (T)0, xa1 = (T)0, xb0 = (T)0, xb1 = (T)0;
            Pk<C> xq = pk2(czero<C>(), czero<C>()), xc = xq;
#pragma unroll 1
            for (int i = sp.ilo + vl; i < sp.ihi; i += L) {
              xa0 += Vs[sp.ph + i * R] * W.y()[sp.w0 + i];
              if (i + gw < sp.ihi) xa1 += Vs[sp.ph + (i + gw) * R] * W.y()[sp.w0 + i + gw];
            }
#pragma unroll 1
            for (int e = vl; e < nt; e += L) {
              const int ij = tij[e], a = ij >> 8, b2 = ij & 255;
              const bool two = e + gw < nt;  // else a zero term
              if constexpr (!fp32) {  // FP64 operations are not packed: no zero terms
                const C t0 = cmul(Cp[tri(ix[a]) + ix[b2]], cmul(bs[a], bs[b2]));
                xq.a = cadd(xq.a, a == b2 ? t0 : ctwice(t0));
                if (two) {
                  const int ij1 = tij[e + gw], a1 = ij1 >> 8, b21 = ij1 & 255;
                  const C t1 = cmul(Cp[tri(ix[a1]) + ix[b21]], cmul(bs[a1], bs[b21]));
                  xq.b = cadd(xq.b, a1 == b21 ? t1 : ctwice(t1));
                }
                continue;
              }
              const int ij1 = tij[two ? e + gw : e], a1 = ij1 >> 8, b21 = ij1 & 255;
              const C c1 = Cp[tri(ix[a1]) + ix[b21]];
              const Pk<C> t = pk_mul(pk2(Cp[tri(ix[a]) + ix[b2]], two ? c1 : czero<C>()),
                                     pk_mul(pk2(bs[a], bs[a1]), pk2(bs[b2], bs[b21])));
              const C t0 = pk_first(t), t1 = pk_second(t);
              xq = pk_add(xq, pk2(a == b2 ? t0 : ctwice(t0), a1 == b21 ? t1 : ctwice(t1)));
            }
#pragma unroll 1
            for (int a = vl; a < np; a += L) {
              const bool two = a + gw < np;
              const int a1 = two ? a + gw : a;
              const C ba = bs[a], ba1 = two ? bs[a1] : czero<C>();
              const int q = ix[a], q1 = ix[a1];
              xb0 += (T)cnum(ba) * (T)cnum(W.v()[q]);
              xb1 += (T)cnum(ba1) * (T)cnum(W.v()[q1]);
              if (opaque(jump == 2)) {
                if constexpr (fp32) {
                  xc = pk_fma(pk2(Cp[pk(kk, q)], Cp[pk(kk, q1)]), pk2(ba, ba1), xc);
                } else {
                  xc.a = cfma(Cp[pk(kk, q)], ba, xc.a);
                  if (two) xc.b = cfma(Cp[pk(kk, q1)], ba1, xc.b);
                }
              }
            }
            ha0 += xa0; ha1 += xa1; hb0 += xb0; hb1 += xb1;
            hq = pk_add(hq, xq); hc = pk_add(hc, xc);
          }
          ayp = ha0 + ha1; bvp = hb0 + hb1;
          qp = cadd(pk_first(hq), pk_second(hq)); ck = cadd(pk_first(hc), pk_second(hc));
        }
        __syncwarp(ln.gm);
        gsum4<L, gw>(qp, ck, bvp, ayp, ln);
        T mmm = 0, mmp = 0, mpp = 0, gm = 0, gp = 0, em = 1;
        if (new_pe) {
          const T bvT = bvp;  // b^T v at the scoring precision (the accept recomputes it)
          const T ayT = ayp;
          mpp = (T)cnum(csub(aa, qp)) * ise2T;
          gp = (ayT - bvT) * ise2T;
          mmp = (T)cnum(ck);  // times 1 / sigma_-^2 below (update only)
          words += (unsigned)(N + 2 * np + 2 * (sp.ihi - sp.ilo) + np * np + np);
        }
        if (valid && jump != 0) {
          const T iqm = CmT<T>::iq(M, e_m);
          em = CmT<T>::r(M, e_m) * (T)cnum(Cp[tri(kk) + kk]);
          mmm = ((T)1 - em) * iqm;
          gm = (T)cnum(W.v()[kk]) * iqm;
          mmp *= iqm;
          words += 2;
        }
        T la = la_fixed;
        if (valid) {
          const PeScore<T> sc = pe_score<T, MIX>(M, e_m, e_p, em, mmm, mmp, mpp, gm, gp);
          dT = sc.dT;
          dnu = sc.dnu;
          st |= sc.st;
          la = sc.ok ? dnu + la_prior : (T)-INFINITY;
        }
        const bool acc = mine && rd.lu < la;
        apply = acc && valid && isfinite(la);
        // ---- the steps that count: up to and including the first accepted move
        const unsigned first = gballot(apply, ln);
        const int f = first ? (__ffs(first) - 1) / gw : g - 1;
        const bool counted = gi <= f;
        const bool t0m = (t0a >> gi) & 1u;
        if (m == 0 && counted) {
          if (st) atomicOr(&S.status, st);
          if (trace)
            pe_trace_record(trace + step + gi, (double)la0, (double)rd.lu0, (double)la, (double)rd.lu, (double)dnu,
                            N + (apply ? (jump == 0 ? 1 : (jump == 1 ? -1 : 0)) : 0), k0i, jump,
                            (M.sample_t0 ? 1 : 0) | (t0m ? 2 : 0) | (acc ? 4 : 0) | ((acc && noop) ? 8 : 0));
        }
        if (counted && !apply) {
#pragma unroll
          for (int q = m; q < kCounts; q += gw)
            W.cnt()[gi * kCounts + q] += count_of(q, N, k0i, step + gi >= burn_in, words, jump, false, t0m);
        }
        const int rejected = first ? f : g;
        const int past = max(0, rejected - max(0, burn_in - step));  // of them after burn-in
        if (past > 0) {
          if (ln.sl == 0) atomicAdd(hist + N, past);  // no value returned: the lane does not wait on it
          if (peh) pe_hist_add(W, peh, N, T_lo, B.pe_hist_width, (uint32_t)past, ln);
        }
        last = step + f;
        k0 = __shfl_sync(ln.gm, k0i, f * gw, L);
        one = apply = first != 0;
        if (apply) {
          // the accepted move on every lane; its overlapping PEs as the accept reads them
          const int src = f * gw;
          jump = __shfl_sync(ln.gm, jump, src, L);
          kk = __shfl_sync(ln.gm, kk, src, L);
          mv.np = __shfl_sync(ln.gm, np, src, L);
          mv.jp = __shfl_sync(ln.gm, jp, src, L);
          mv.jm = __shfl_sync(ln.gm, jm, src, L);
          if constexpr (MIX) { e_m = __shfl_sync(ln.gm, e_m, src, L); e_p = __shfl_sync(ln.gm, e_p, src, L); }
          dT = __shfl_sync(ln.gm, dT, src, L);
          dnu = __shfl_sync(ln.gm, dnu, src, L);
          words = __shfl_sync(ln.gm, words, src, L);
          mv.ay = cfromf(__shfl_sync(ln.gm, ayp, src, L));
          mv.aa = cshfl<L>(aa, src, ln.gm);
          t0_acc = (t0a >> f) & 1u;
          mv.jump = jump; mv.kk = kk; mv.em = e_m; mv.ep = e_p;
          mv.vk = jump != 0 ? W.v()[kk] : czero<C>();
          mv.sp = jump != 1 ? pe_sup(M, n, mv.jp) : Sup{0, 0, 0, 0};
          if (jump != 1) {
            if (f > 0) {
#pragma unroll 1
              for (int a = ln.sl; a < mv.np; a += L) W.ovb()[a] = W.work(f)[a];
              __syncwarp(ln.gm);
            }
#pragma unroll 1
            for (int a = ln.sl; a < mv.np; a += L) W.ovi()[a] = W.ix()[f * kSpecPes + a];
          }
          __syncwarp(ln.gm);
        }
      } else {
        // ---------------------------------------------- one step on all lanes
        last = step;
        const PeRand<T, MIX> rd = rnd[step & (L - 1)];
        // ---- Gibbs part 1: MH on t0 (Sec. 2.4), uniform prior on its grid range
        T la0 = (T)NAN;
        const T lu0 = rd.lu0;
        if (M.sample_t0) {
          const int Dm = fp32 ? __float2int_rn((float)(rd.z1 * inv_gT)) : __double2int_rn((double)(rd.z1 * inv_gT));
          const int k0p = k0 + Dm;
          if (Dm == 0) {
            la0 = (T)0;
          } else if (k0p < k0_lo || k0p > k0_hi) {
            la0 = (T)-INFINITY;
          } else {
            T part = (T)0;
#pragma unroll 1
            for (int k = ln.sl; k < N; k += L) {
              const int j = W.list()[k];
              part += pe_logphi<T>(M, j - k0p) - pe_logphi<T>(M, j - k0);
            }
            la0 = wsum(part, ln);
          }
          t0_acc = lu0 < la0;
          if (t0_acc) k0 = k0p;
        }
        // ---- Gibbs part 2: one RJMCMC jump (Sec. 2.4)
        jump = (N == 0) ? 0 : (rd.u3 < Jt ? 0 : (rd.u3 < (T)2 * Jt ? 1 : 2));
        int st = 0, valid = 0, noop = 0, kk = -1, jp = -1, jm = -1;
        if constexpr (MIX) e_m = rd.ep;
        T la_prior = (T)0, la_fixed = (T)-INFINITY;
        const T lu = rd.lu;
        const T lphi_t0 = W.lPhi()[k0 - k0_lo];
        if (jump == 0) {
          if (N >= n_cap) {
            st |= FSMP_ST_CAPACITY;
          } else if (lphi_t0 > (T)-INFINITY) {
            const T base = pe_cphi<T>(M, T_lo - 1 - k0), tot = pe_cphi<T>(M, T_hi - 1 - k0) - base;
            jp = pe_birth_search<T, L>(M, T_lo, T_hi, k0, base, rd.u4 * tot, ln);
            valid = jp >= T_lo;
            la_prior = log_lambda0 + lphi_t0 - lgN[N + 1] + (N == 0 ? logJ : (T)0);
          }
        } else {
          kk = fp32 ? __float2int_rd((float)(rd.u4 * (T)N)) : __double2int_rd((double)(rd.u4 * (T)N));
          if (kk >= N) kk = N - 1;
          jm = W.list()[kk];
          if constexpr (MIX) e_m = W.le()[kk];
          if (jump == 1) {
            valid = 1;
            la_prior = -log_lambda0 - lphi_t0 + lgN[N] - (N == 1 ? logJ : (T)0);
          } else {
            const int Dm = fp32 ? __float2int_rn((float)(rd.z2 * inv_gT)) : __double2int_rn((double)(rd.z2 * inv_gT));
            const int jpl = jm + Dm;
            bool same = Dm == 0;
            if constexpr (MIX) same = same && rd.ep == e_m;
            if (same) {  // same time and component: an accepted no-op
              noop = 1;
              la_fixed = (T)0;
            } else if (jpl < T_lo || jpl >= T_hi || pe_logphi<T>(M, jpl - k0) == (T)-INFINITY) {
              la_fixed = (T)-INFINITY;
            } else {
              jp = jpl;
              valid = 1;
              la_prior = pe_logphi<T>(M, jp - k0) - pe_logphi<T>(M, jm - k0);
            }
          }
        }
        // ---- scoring: the 2x2 quantities in PE space, then the 2x2 algebra in T
        mv.jump = jump; mv.kk = kk; mv.jp = jp; mv.jm = jm; mv.np = 0;
        // components of a_- and a_+; the absent one of a birth or death takes the other's values
        // (its terms vanish)
        mv.em = e_m;
        mv.ep = 0;
        if constexpr (MIX) mv.ep = jump == 1 ? e_m : rd.ep;
        mv.aa = mv.vk = mv.ay = czero<C>();
        mv.sp = Sup{0, 0, 0, 0};
        T mmm = 0, mmp = 0, mpp = 0, gm = 0, gp = 0, em = 1;
        if (valid) {
          if (jump != 1) {
            const Sup sp = pe_sup(M, n, jp);
            mv.sp = sp;
            mv.aa = xcorr<C>(M, tc, sp, 0);  // issued first: its table load overlaps the scan's
            // PEs overlapping a_+, with b_q = a_q^T a_+
            int np = 0;
#pragma unroll 1
            for (int base = 0; base < N; base += L) {
              const int qi = base + ln.sl;
              C bq = czero<C>();
              if (qi < N) {
                const int o = jp - W.list()[qi];
                if (o > -M.Lt && o < M.Lt) bq = xcorr<C>(M, tc, sp, o);
              }
              const bool ov = cnz(bq);
              const unsigned b = gballot(ov, ln);
              if (ov) {
                const int pos = np + __popc(b & ((1u << ln.sl) - 1u));
                W.ovi()[pos] = qi;
                W.ovb()[pos] = bq;
              }
              np += __popc(b);
            }
            __syncwarp(ln.gm);
            mv.np = np;
            // b^T C^-1 b over the lower triangle of the overlap block (lanes over its entries, the
            // off-diagonal ones counted twice), b^T v, (C^-1 b)_k of an update and a_+^T y, then one
            // reduction of the four over the group
            T ayp = (T)0;
#pragma unroll 1
            for (int i = sp.ilo + ln.sl; i < sp.ihi; i += L) ayp += Vs[sp.ph + i * R] * W.y()[sp.w0 + i];
            C qp = czero<C>(), ck = czero<C>();
            T bvp = (T)0;
            const bool team = TW > 1 && np > kSpecPes;
            const int nt = team ? 0 : tri(np);
            TriWalk<L> tw;
            int e = ln.sl;
            if constexpr (TW > 1) {
              if (team) {  // the helpers start; this warp's share comes after the sums below
                PeTeam<C>& tm = pe_team<T>(M);
                if (ln.sl == 0) { tm.op = kOpScore; tm.Cp = Cp; tm.np = np; }
                team_bar();
              }
            }
            // the products of two entries e, e + L at a time (BIG, C^-1 in the global slot: two
            // such pairs, their loads ahead of their sums), added in order
            constexpr int PE = BIG ? 4 : 2;
#pragma unroll 1
            for (; e < nt; e += PE * L) {
              C cq[PE], ba[PE], bb[PE];
              bool dg[PE];
#pragma unroll
              for (int u = 0; u < PE; ++u) {
                const bool in = e + u * L < nt;  // beyond the triangle: zero terms
                if (in) tw.at(tij, e + u * L);
                const C c = Cp[tri(W.ovi()[tw.i]) + W.ovi()[tw.j]];
                cq[u] = in ? c : czero<C>();
                ba[u] = W.ovb()[tw.i];
                bb[u] = W.ovb()[tw.j];
                dg[u] = tw.i == tw.j;
              }
#pragma unroll
              for (int u = 0; u < PE; u += 2) {
                const Pk<C> t = pk_mul(pk2(cq[u], cq[u + 1]), pk_mul(pk2(ba[u], ba[u + 1]), pk2(bb[u], bb[u + 1])));
                const C t0 = pk_first(t), t1 = pk_second(t);
                qp = cadd(qp, dg[u] ? t0 : ctwice(t0));
                qp = cadd(qp, dg[u + 1] ? t1 : ctwice(t1));
              }
            }
#pragma unroll 1
            for (int a = ln.sl; a < np; a += L) {
              const C ba = W.ovb()[a];
              bvp += (T)cnum(ba) * (T)cnum(W.v()[W.ovi()[a]]);
              if (opaque(jump == 2)) ck = cfma(Cp[pk(kk, W.ovi()[a])], ba, ck);
            }
            if constexpr (TW > 1) {
              if (team) {
                team_score<T, BIG, L, MIX>(M, W);
                team_bar();
                qp = pe_team<T>(M).part[ln.sl];
              }
            }
            gsum4<L, L>(qp, ck, bvp, ayp, ln);
            const T bvT = bvp;  // b^T v at the scoring precision (the accept recomputes it)
            const T ayT = ayp;
            mv.ay = cfromf(ayT);
            mpp = (T)cnum(csub(mv.aa, qp)) * ise2T;
            gp = (ayT - bvT) * ise2T;
            mmp = (T)cnum(ck);  // times 1 / sigma_-^2 below (update only)
            words += (unsigned)(N + 2 * np + 2 * (sp.ihi - sp.ilo) + np * np + np);
          }
          if (jump != 0) {
            const T iqm = CmT<T>::iq(M, mv.em);
            mv.vk = W.v()[kk];
            em = CmT<T>::r(M, mv.em) * (T)cnum(Cp[tri(kk) + kk]);
            mmm = ((T)1 - em) * iqm;
            gm = (T)cnum(mv.vk) * iqm;
            mmp *= iqm;
            words += 2;
          }
        }
        T la = la_fixed;
        if (valid) {
          const PeScore<T> sc = pe_score<T, MIX>(M, mv.em, mv.ep, em, mmm, mmp, mpp, gm, gp);
          dT = sc.dT;
          dnu = sc.dnu;
          st |= sc.st;
          la = sc.ok ? dnu + la_prior : (T)-INFINITY;
        }
        const bool acc = lu < la;
        apply = acc && valid && isfinite(la);
        if (ln.sl == 0) {
          if (st) S.status |= st;
          if (trace)
            pe_trace_record(trace + step, (double)la0, (double)lu0, (double)la, (double)lu, (double)dnu,
                            N + (apply ? (jump == 0 ? 1 : (jump == 1 ? -1 : 0)) : 0), k0, jump,
                            (M.sample_t0 ? 1 : 0) | (t0_acc ? 2 : 0) | (acc ? 4 : 0) | ((acc && noop) ? 8 : 0));
        }
      }

      // ---- accepted move: C^-1, v, y and the PE list
      if (apply) {
        {
          const AcceptOut<C> ao = pe_accept<T, BIG, L, MIX, TW>(M, W, Cp, cap, Cg, mv, n, N, ln);
          Cp = ao.Cp;
          cap = ao.cap;
          N = ao.N;
          words += (unsigned)ao.words;
        }
        close_hold(S, last, burn_in, true, dT, dnu, ln.sl);
        C qs = czero<C>();
        double ms = M.cm_mu[0];  // the PEs' mean charge (the mixture: the sum of them)
        if constexpr (MIX) ms = 0.0;
#pragma unroll 1
        for (int i = ln.sl; i < N; i += L) {
          qs = cadd(qs, W.v()[i]);
          if constexpr (MIX) ms += M.cm_mu[W.le()[i]];
        }
        qs = csum_m(qs, N, ln);
        if constexpr (MIX) ms = wsum(ms, ln);
        if (ln.sl == 0) {
          S.q_from = last;
          // the PE removed (death, update) and the one added (birth, update)
          if (jump != 1) { S.St += abs(mv.jp); S.Se += mv.ep; }
          if (jump != 0) { S.St -= abs(mv.jm); S.Se -= mv.em; }
          S.n_acc_refresh++;
        }
        __syncwarp(ln.gm);
        set_summaries<MIX>(S, M.g, N, ms, c64(qs), inv1, ln.sl);
        __syncwarp(ln.gm);
        if (fp32 && M.refresh_every > 0 && S.n_acc_refresh >= M.refresh_every) {
          const RefreshOut ro = pe_refresh<T, BIG, L, MIX, TW>(M, W, Cp, ws, n_cap, w, S.wsq, n, N, ln);
          C qr = czero<C>();
#pragma unroll 1
          for (int i = ln.sl; i < N; i += L) qr = cadd(qr, W.v()[i]);
          qr = csum(qr, ln);
          if (ln.sl == 0) {
            S.n_acc_refresh = 0;
            if (ro.ok) {
              S.sum[PeStats::kLogdet] = ro.logdet; S.sum[PeStats::kLogL] = ro.logL;
              S.drift_max = fmax(S.drift_max, ro.drift);
              if (ro.drift > M.drift_tol) S.status |= FSMP_ST_DRIFT;
              S.n_refresh++;
              S.cur[0] = fma(MIX ? 1.0 : (double)N, ms, c64(qr));
            } else {
              S.status |= FSMP_ST_DRIFT;
              S.refresh_fail++;
            }
          }
          __syncwarp(ln.gm);
        }
      }

      // ---- bookkeeping of the accepted step (of a batch) or of the step made alone
      if (one) {
        if (ln.sl < kCounts)
          W.cnt()[ln.sl] += count_of(ln.sl, N, k0, last >= burn_in, words, jump, apply, t0_acc);
        if (last >= burn_in) {
          if (ln.sl == 0) atomicAdd(hist + N, 1);  // no value returned: the lane does not wait on it
          if (peh) pe_hist_add(W, peh, N, T_lo, B.pe_hist_width, 1u, ln);
        }
      }
      step = last + 1;
      __syncwarp(ln.gm);
    }

    // ------------------------------------------------------------- chain end
    if (fp32 && M.refresh_every > 0 && S.n_acc_refresh > 0) {
      // the reported log-likelihood and log|Sigma| come from an FP64 rebuild
      const RefreshOut ro = pe_refresh<T, BIG, L, MIX, TW>(M, W, Cp, ws, n_cap, w, S.wsq, n, N, ln);
      if (ln.sl == 0) {
        if (ro.ok) {
          S.sum[PeStats::kLogdet] = ro.logdet; S.sum[PeStats::kLogL] = ro.logL;
          S.drift_max = fmax(S.drift_max, ro.drift);
          if (ro.drift > M.drift_tol) S.status |= FSMP_ST_DRIFT;
          S.n_refresh++;
        } else {
          S.status |= FSMP_ST_DRIFT;
        }
      }
    }
    if (ln.sl < kCounts) {  // the subgroups' counts together
      unsigned long long t = W.cnt()[ln.sl];
#pragma unroll 1
      for (int i = 1; i < kSpec; ++i) t += W.cnt()[i * kCounts + ln.sl];
      W.cnt()[ln.sl] = t;
    }
    __syncwarp(ln.gm);
    close_hold(S, n_steps, burn_in, false, (T)0, (T)0, ln.sl);
    __syncwarp(ln.gm);
    const double lam_hat = pe_lambda_mle<L>(hist, n_cap, lambda0, ln.sl, ln.gm);
    if (ln.sl == 0) {
      fsmp_summary o;
      o.lambda_hat = lam_hat;
      int ns = n_steps - burn_in;
      if (ns < 0) ns = 0;
      const double inv = ns > 0 ? 1.0 / ns : NAN;
      const long long* const cnt = reinterpret_cast<const long long*>(W.cnt());
      const double mN = (double)cnt[0] * inv, mK = (double)cnt[2] * inv;
      o.mean_N = mN; o.var_N = (double)cnt[1] * inv - mN * mN;
      o.mean_t0 = t_origin + M.g * mK; o.var_t0 = M.g * M.g * ((double)cnt[3] * inv - mK * mK);
      o.mean_Q = S.sum[0] * inv; o.var_Q = S.sum[1] * inv - o.mean_Q * o.mean_Q;
      o.mean_wt = S.sum[2] * inv; o.var_wt = S.sum[3] * inv - o.mean_wt * o.mean_wt;
      o.mean_we = S.sum[4] * inv; o.var_we = S.sum[5] * inv - o.mean_we * o.mean_we;
      o.logL = S.sum[PeStats::kLogL]; o.logdet = S.sum[PeStats::kLogdet];
      o.drift_max = S.drift_max; o.alg_bytes = (double)W.cnt()[4] * 8.0;
      o.prop[0] = (int)(unsigned)W.cnt()[5]; o.prop[1] = (int)(W.cnt()[5] >> 32);
      o.prop[2] = n_steps - o.prop[0] - o.prop[1];
      o.acc[0] = (int)(unsigned)W.cnt()[6]; o.acc[1] = (int)(W.cnt()[6] >> 32); o.acc[2] = (int)(unsigned)W.cnt()[7];
      o.acc_t0 = (int)(W.cnt()[7] >> 32); o.prop_t0 = M.sample_t0 ? n_steps : 0; o.N_final = N; o.k0_final = k0;
      o.status = S.status; o.n_samples = ns; o.n_refresh = S.n_refresh; o.reserved = 0;
      *out = o;
      note_chain_done(B, wi);
    }
    __syncwarp(ln.gm);
  }
  if constexpr (TW > 1) {
    if (ln.sl == 0) pe_team<T>(M).op = kOpExit;
    team_bar();
  }
}

// Float-float copy of an FP64 table: hi = fl(x), lo = fl(x - hi).
__global__ void split_ff_kernel(const double* a, float* out, size_t n) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float h = (float)a[i];
  out[2 * i] = h;
  out[2 * i + 1] = (float)(a[i] - (double)h);
}


// The kernel instance for (precision, BIG, lanes) of a charge model; f receives its address.
// The mixture has no BIG instance (its chains use the compact loops at any n_cap).
template <bool MIX, typename F> cudaError_t with_pe_kernel(int precision, bool big, int lanes, PeForm form, F f) {
  if (form == kPeTeam) {
    if (precision == FSMP_FP64 || lanes != 32) return cudaErrorInvalidValue;
    if constexpr (MIX) {
      return f(pe_kernel<float, false, 32, true, kTeam>);
    } else {
      return big ? f(pe_kernel<float, true, 32, false, kTeam>) : f(pe_kernel<float, false, 32, false, kTeam>);
    }
  }
  if (form == kPeWarpMore) {
    if constexpr (MIX) {
      if (precision != FSMP_FP64 && lanes == 32) return f(pe_kernel<float, false, 32, true, 1, true>);
    }
    return cudaErrorInvalidValue;
  }
  if constexpr (MIX) {
    if (precision == FSMP_FP64)
      return lanes == 16 ? f(pe_kernel<double, false, 16, true>) : f(pe_kernel<double, false, 32, true>);
    return lanes == 16 ? f(pe_kernel<float, false, 16, true>) : f(pe_kernel<float, false, 32, true>);
  } else {
    if (precision == FSMP_FP64) {
      if (big) return f(pe_kernel<double, true, 32, false>);
      return lanes == 16 ? f(pe_kernel<double, false, 16, false>) : f(pe_kernel<double, false, 32, false>);
    }
    if (big) return f(pe_kernel<float, true, 32, false>);
    return lanes == 16 ? f(pe_kernel<float, false, 16, false>) : f(pe_kernel<float, false, 32, false>);
  }
}

template <bool MIX> cudaError_t pe_set_attributes(int precision, int max_smem) {
  for (int big = 0; big < (MIX ? 1 : 2); ++big)
    for (int lanes : {32, 16}) {
      if (big && lanes == 16) continue;
      for (PeForm form : {kPeWarp, kPeWarpMore, kPeTeam}) {
        if (form != kPeWarp && (lanes != 32 || precision == FSMP_FP64)) continue;
        if (form == kPeWarpMore && !MIX) continue;
        const cudaError_t e = with_pe_kernel<MIX>(precision, big != 0, lanes, form, [&](auto k) {
          return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
        });
        if (e != cudaSuccess) return e;
      }
    }
  return cudaSuccess;
}

template <bool MIX> int pe_occupancy(int precision, int threads, size_t smem, bool big, int lanes, PeForm form) {
  int n = 0;
  const cudaError_t e = with_pe_kernel<MIX>(precision, big, lanes, form, [&](auto k) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, threads, smem);
  });
  return e == cudaSuccess ? n : 0;
}

template <bool MIX>
cudaError_t pe_launch(const DevModel& M, const BatchView& B, int warps, int lanes, int ctas, int Ns, size_t smem,
                      void* cinv, size_t c_stride, double* ws, size_t ws_stride, int* hist, int* counter,
                      bool big, PeForm form, cudaStream_t st) {
  PeSlots G;
  G.C = cinv;
  G.c_stride = c_stride;
  G.ws = ws;
  G.ws_stride = ws_stride;
  G.hist = hist;
  G.counter = counter;
  G.Ns = Ns;
  const cudaError_t e = with_pe_kernel<MIX>(M.precision, big, lanes, form, [&](auto k) {
    k<<<ctas, warps * 32, smem, st>>>(M, B, G);
    return cudaSuccess;
  });
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace
}  // namespace fsmp
