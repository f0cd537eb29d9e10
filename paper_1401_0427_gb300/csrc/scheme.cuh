// Device arithmetic of the D1Q3Q2 (section 2) and D2Q5Q4Q4 (section 3) schemes of
// Dubois' vectorial lattice Boltzmann method for the shallow-water equations.
//
// The equilibria are the derivatives of the potentials h_j^* of the dual entropy
// (f_j = dh_j^*/dtheta, g_j = dh_j^*/du ...), written here in closed form in the
// conserved variables W = (h, qx = h u, qy = h v).  With gamma = 2, p = g h^2/2,
// K = 1/(2g) and kappa = K theta = h/2 - (u^2 + v^2)/(4g):
//
//   2D  f0 = a kappa,  r = (h - f0)/4,
//       f1,3 = r +- qx/(2 lambda),            f2,4 = r +- qy/(2 lambda)
//       gx1,3 = qx/4 +- (qx u + p)/(2 lambda), gx2,4 = qx/4 +- qx qy/(h 2 lambda)
//       gy1,3 = qy/4 +- qx qy/(h 2 lambda),    gy2,4 = qy/4 +- (qy v + p)/(2 lambda)
//   1D  f0 = a kappa,  f+- = h/2 - a kappa/2 +- q/(2 lambda),
//       g+- = q/2 +- (q u + p)/(2 lambda)
//
// and the collision is the BGK form of Eq. 2-relaxation, f* = f + s (f^eq - f), evaluated
// as f* = (1 - s) f + s f^eq with s folded into the constants of each equilibrium term
// (collide13: two operations per population instead of three).
//
// Every operation is an explicitly rounded intrinsic (no compiler contraction), laid
// out so that mirror-image cells see mirror-image operations: a field with a
// symmetry of the square keeps it bit for bit, in FP32 and FP64.
#pragma once

#include <cuda_runtime.h>

namespace lbm {

__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float fmad(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmad(double a, double b, double c) { return __fma_rn(a, b, c); }
// FP32: the PTX approximation rcp.approx.ftz.f32 (1 ulp; the FP32 path is compared with the FP64
// oracle at 1e-5), the value of __fdividef(1, a) for every a but denormals, without its scaling of
// large arguments (five instructions more per cell).  FP64: the PTX approximation rcp.approx.ftz.f64 (relative error e of about
// 2^-20) and one step r <- r + r (e + e^2) (the geometric series of 1 / (1 - e) up to its second
// power; the rest, e^3 of about 2^-60, is below the rounding): three fused multiply-adds of the
// unit that bounds the FP64 kernels on GB300, where two Newton-Raphson steps take four.  Either is
// a fixed function of h, so mirror-image cells still round alike.
__device__ __forceinline__ float recip(float a) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ double recip(double a) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(a));
  const double e = __fma_rn(-a, r, 1.0);
  return __fma_rn(r, __fma_rn(e, e, e), r);
}
// x times 2^k (NEG: -2^k), exactly, by the exponent field: a few integer operations, where an FP64
// multiplication takes 64 cycles of a quarter of an SM.  Zeros keep their value; denormals,
// infinities, NaN and results out of the normal range take the multiplication.
template <int k, bool NEG>
__device__ __forceinline__ double times_pow2(double x) {
  constexpr int flip = NEG ? static_cast<int>(0x80000000u) : 0;
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int e = (hi >> 20) & 0x7ff;
  if (e > (k < 0 ? -k : 0) && e < (k < 0 ? 0x7ff : 0x7ff - k)) return __hiloint2double((hi + k * (1 << 20)) ^ flip, lo);
  if (((hi & 0x7fffffff) | lo) == 0) return __hiloint2double(hi ^ flip, 0);
  return __dmul_rn(x, (NEG ? -1.0 : 1.0) * (k < 0 ? 1.0 / (1 << -k) : static_cast<double>(1 << (k < 0 ? 0 : k))));
}

// Constants of the FP64 collisions in integers; FP32 kernels have none (they are parameters of every launch).
template <class T>
struct FixedConsts {};
template <>
struct FixedConsts<double> {
  // 1D: f0 = a_2 h + a_4g u^2
  double a_2, a_4g;
  // 2D (collide13_fixed): |1 - s| and s c in units of 2^-64, and whether they are below one
  unsigned long long x_om, x_sc;
  // the least difference of the families' exponents at which s c q stays below 2^62 units of the
  // depths' (q is below 2^62 of its own): s c 2^-least_sc <= 1
  int least_sc;
  // 2D MRT (collide13_mrt_fixed): m[0], m[1], m[2] / 4, m[3] / 4, m[4 .. 9] and c likewise
  unsigned long long x_m[10], x_c;
  int least_c;  // c 2^-least_c <= 1/2: c q stays below 2^61 units of the depths'
  // 1D (collide5_fixed): s / 2 likewise
  unsigned long long x_s2;
  bool om_neg, fixed_ok, fixed1_ok, fixed_mrt_ok;
};

// Scheme constants in the storage precision.
template <class T>
struct Consts : FixedConsts<T> {
  T s;       // relaxation rate
  T a;       // rest-potential weight
  T c;       // 1 / (2 lambda)
  T half_g;  // g / 2
  T inv4g;   // 1 / (4 g)
  T nz;      // -0, a value the compiler cannot see (products of the paired path, below)
  // Rates of the non-conserved moments for the MRT collision (Eq. 2-relaxation with
  // distinct s_l), in the order of the paper's moment bases:
  //   2D: J_x, J_y, eps, XX_rho | f_xx, f_xy, XX_u | f_yx, f_yy, XX_v   (r[0..9])
  //   1D: J_rho, eps_rho, J_q                                            (r[0..2])
  T r[10];
  // 2D: the same rates with the exact power-of-two factors of the moment transforms folded
  // in (collide13_mrt): J_x / 2, J_y / 2, eps, XX_rho | f_xx / 2, f_xy / 2, XX_u / 4 | f_yx / 2,
  // f_yy / 2, XX_v / 4.  Scaling by a power of two commutes with rounding, so each product
  // is exactly half (a quarter) of the unscaled one and the halvings that follow it vanish.
  T m[10];
  // BGK with the rate folded in (collide13): f* = om f + s f^eq, s f^eq built from
  //   z = -(s f0) / 4 = s_a2 h + s_a4g (u^2 + v^2)  (s_a2, s_a4g carry the -1/4),
  //   s f0 = -4 z,  s r = s (h - f0) / 4 = s_4 h + z  (one rounding),
  //   s c p = (s_p h) h,  s c q and s q / 4 = q s_c and q s_4.
  // om and s_4 are formed from s as stored (om = 1 - s and s_4 = s / 4 exactly for s in
  // [1/2, 2]), so om + 4 s_4 = 1 and the masses and momenta of om f and s f^eq add up to those
  // of f with no bias from the rounding of the constants.
  T om;     // 1 - s
  T s_a2;   // -s a / 8
  T s_a4g;  // s a / (16 g)
  T s_p;    // s c g / 2
  T s_c;    // s c
  T s_4;    // s / 4
};

// |v| <= 1 in units of 2^-64 (saturated)
inline __host__ unsigned long long in_2_64(double v) {
  const double a = v < 0 ? -v : v;
  return a >= 1.0 ? ~0ull : static_cast<unsigned long long>(a * 18446744073709551616.0);
}

// the least d from -31 to 1 with v 2^-d <= most (v <= 2 most)
inline __host__ int least_shift(double v, double most) {
  int d = 1;
  while (d > -31 && v * static_cast<double>(1LL << (1 - d)) <= most) --d;
  return d;
}

template <class T>
__host__ void set_mrt_folded(Consts<T>& k) {
  constexpr double scale[10] = {0.5, 0.5, 1.0, 1.0, 0.5, 0.5, 0.25, 0.5, 0.5, 0.25};
  for (int i = 0; i < 10; ++i) k.m[i] = static_cast<T>(static_cast<double>(k.r[i]) * scale[i]);
  if constexpr (sizeof(T) == 8) {
    k.x_c = in_2_64(k.c);
    k.least_c = least_shift(k.c, 0.5);
    k.fixed_mrt_ok = k.c > 0.0 && k.c <= 0.5;
    for (int i = 0; i < 10; ++i) {
      k.x_m[i] = in_2_64(k.m[i] * (i == 2 || i == 3 ? 0.25 : 1.0));
      k.fixed_mrt_ok = k.fixed_mrt_ok && k.r[i] >= 0.0 && k.r[i] <= 2.0;
    }
  }
}

template <class T>
__host__ Consts<T> make_consts(double g, double lambda, double s, double a) {
  Consts<T> k;
  k.s = static_cast<T>(s);
  k.a = static_cast<T>(a);
  k.c = static_cast<T>(1.0 / (2.0 * lambda));
  k.half_g = static_cast<T>(g / 2.0);
  k.inv4g = static_cast<T>(1.0 / (4.0 * g));
  k.nz = static_cast<T>(-0.0);
  const double c = 1.0 / (2.0 * lambda), st = static_cast<double>(k.s);  // s as stored
  k.om = static_cast<T>(1.0 - st);
  k.s_a2 = static_cast<T>(-st * a / 8.0);
  k.s_a4g = static_cast<T>(st * a / (16.0 * g));
  k.s_p = static_cast<T>(st * c * g / 2.0);
  k.s_c = static_cast<T>(st * c);
  k.s_4 = static_cast<T>(st / 4.0);
  if constexpr (sizeof(T) == 8) {
    k.a_2 = a / 2.0;
    k.a_4g = -a / (4.0 * g);
    k.x_om = in_2_64(1.0 - st);
    k.x_sc = in_2_64(st * c);
    k.least_sc = least_shift(st * c, 1.0);
    k.om_neg = st > 1.0;
    k.fixed_ok = st >= 0.0 && st <= 2.0 && st * c < 1.0;
    k.x_s2 = in_2_64(st / 2.0);
    k.fixed1_ok = st >= 0.0 && st <= 2.0 && c > 0.0 && c <= 1.0;
  }
  for (int i = 0; i < 10; ++i) k.r[i] = k.s;
  set_mrt_folded(k);
  return k;
}

// Constants with MRT rates (10 in 2D, 3 in 1D, in the order documented on Consts::r).
template <class T>
__host__ Consts<T> make_consts_mrt(double g, double lambda, double s, double a, const double* rates, int n) {
  Consts<T> k = make_consts<T>(g, lambda, s, a);
  for (int i = 0; i < n && i < 10; ++i) k.r[i] = static_cast<T>(rates[i]);
  set_mrt_folded(k);
  return k;
}

// Conserved moments, summed in mirror-symmetric pairs.
template <class T>
__device__ __forceinline__ void moments13(const T f[13], T& h, T& qx, T& qy) {
  h = add(f[0], add(add(f[1], f[3]), add(f[2], f[4])));
  qx = add(add(f[5], f[7]), add(f[6], f[8]));
  qy = add(add(f[9], f[11]), add(f[10], f[12]));
}

// ---- FP64 sums and relaxation in 64-bit integers ----
// An FP64 instruction takes 64 cycles of a quarter of an SM, in which its integer pipe takes 40 or
// so.  Values of like size are therefore added as 64-bit integers in units of 2^-59 of the
// power of two below the largest of them (`e`: that value's exponent field, in place) and rounded
// once to a double, to nearest even.  What an operand loses is below one unit.  Operations work on
// magnitudes and signs, so exact negatives give exact negatives (mirror-image cells), and sums
// do not depend on the order.
__device__ __forceinline__ int exp_field(double x) { return __double2hiint(x) & 0x7ff00000; }
// exponents for which every shift and result below stays inside the normal range
__device__ __forceinline__ bool exp_fits(int e) { return e >= (64 << 20) && e <= (2000 << 20); }
__device__ __forceinline__ unsigned long long mantissa(double x) {  // 53 bits (a zero: 2^52, shifted out by its exponent)
  return (static_cast<unsigned long long>((__double2hiint(x) & 0xfffff) | 0x100000) << 32) |
         static_cast<unsigned>(__double2loint(x));
}
// |x| in units of e's, for exponents up to e
__device__ __forceinline__ unsigned long long fix_mag(double x, int e) {
  return (mantissa(x) << 7) >> min((e - exp_field(x)) >> 20, 63);
}
__device__ __forceinline__ long long with_sign(unsigned long long m, int hi) {  // the sign bit of hi
  const long long s = hi >> 31;
  return (static_cast<long long>(m) ^ s) - s;
}
// x in units of e's, for exponents up to e + 1; ok: cleared beyond
__device__ __forceinline__ long long fix_one_more(double x, int e, bool& ok) {
  const int d = ((e - exp_field(x)) >> 20) + 1;
  ok = ok && d >= 0;
  return with_sign((mantissa(x) << 8) >> (d & 63) >> (d > 63 ? 63 : 0), __double2hiint(x));
}
// m from units of an exponent d below into units of e's; ok: cleared where d < least, the d down to
// which the result stays in range (below)
__device__ __forceinline__ unsigned long long to_units(unsigned long long m, int d, int least, bool& ok) {
  ok = ok && d >= least;
  return d >= 0 ? m >> min(d, 63) : m << (-d & 31);
}
// m c / 2^64 without the last partial product (less than 3 units too small)
__device__ __forceinline__ unsigned long long times_2_64(unsigned long long m, unsigned long long c) {
  const unsigned mh = static_cast<unsigned>(m >> 32), ml = static_cast<unsigned>(m);
  const unsigned ch = static_cast<unsigned>(c >> 32), cl = static_cast<unsigned>(c);
  return static_cast<unsigned long long>(mh) * ch + __umulhi(mh, cl) + __umulhi(ml, ch);
}
// m c / 2^64, rounded
__device__ __forceinline__ unsigned long long times_2_64_round(unsigned long long m, unsigned long long c) {
  return __umul64hi(m, c) + (m * c >> 63);
}
// v / 4, rounded to nearest even
__device__ __forceinline__ long long quarter(long long v) { return (v + 1 + (static_cast<unsigned>(v) >> 2 & 1)) >> 2; }
// the double of v (|v| < 2^63) in units of e's, rounded to nearest even
__device__ __forceinline__ double unfix(long long v, int e) {
  const int s = static_cast<int>(v >> 63);
  unsigned long long a = static_cast<unsigned long long>((v ^ s) - s);
  const int lz = __clzll(static_cast<long long>(a));
  a <<= (lz - 1) & 63;  // leading bit 62
  a += 0x1ff + (static_cast<unsigned>(a >> 10) & 1);
  const int hi = static_cast<int>(static_cast<unsigned>(a >> 42) + e + ((3 - lz) << 20)) | (s & static_cast<int>(0x80000000u));
  return v == 0 ? 0.0 : __hiloint2double(hi, static_cast<int>(a >> 10));
}

// The sum of N <= 5 values rounded once; infinities, NaN and sums near either end of the
// exponent's range are added in FP64.
template <int N>
__device__ __forceinline__ double sum_once(const double (&x)[N]) {
  int e = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) e = max(e, exp_field(x[i]));
  if (!exp_fits(e)) {
    const double s = add(add(x[0], x[1]), add(x[2], x[3]));
    return N == 5 ? add(x[N - 1], s) : s;
  }
  long long v = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) v += with_sign(fix_mag(x[i], e), __double2hiint(x[i]));
  return unfix(v, e);
}

__device__ __forceinline__ void moments13(const double f[13], double& h, double& qx, double& qy) {
  h = sum_once<5>({f[1], f[3], f[2], f[4], f[0]});
  qx = sum_once<4>({f[5], f[7], f[6], f[8]});
  qy = sum_once<4>({f[9], f[11], f[10], f[12]});
}

template <class T>
__device__ __forceinline__ void equilibrium13(T h, T qx, T qy, const Consts<T>& k, T e[13]) {
  const T rh = recip(h);
  const T u = mul(qx, rh);
  const T v = mul(qy, rh);
  const T uu = add(mul(u, u), mul(v, v));
  const T kap = fmad(-uu, k.inv4g, mul(T(0.5), h));
  const T f0 = mul(k.a, kap);
  const T hf = sub(h, f0);  // r = hf / 4
  const T p = mul(mul(k.half_g, h), h);
  const T ax = mul(qx, k.c);
  const T ay = mul(qy, k.c);
  const T pxx = mul(fmad(qx, u, p), k.c);
  const T pyy = mul(fmad(qy, v, p), k.c);
  const T pxy = mul(mul(mul(qx, qy), rh), k.c);
  // r +- a and q/4 +- b as one fused multiply-add each: the quarter is exact, so each is the
  // rounded sum of the exact quarter and the other term, as add(mul(., 1/4), +-b) would give
  const T q4 = T(0.25);
  e[0] = f0;
  e[1] = fmad(hf, q4, ax);
  e[2] = fmad(hf, q4, ay);
  e[3] = fmad(hf, q4, -ax);
  e[4] = fmad(hf, q4, -ay);
  e[5] = fmad(qx, q4, pxx);
  e[6] = fmad(qx, q4, pxy);
  e[7] = fmad(qx, q4, -pxx);
  e[8] = fmad(qx, q4, -pxy);
  e[9] = fmad(qy, q4, pxy);
  e[10] = fmad(qy, q4, pyy);
  e[11] = fmad(qy, q4, -pxy);
  e[12] = fmad(qy, q4, -pyy);
}

// Moments -> BGK relaxation, in place: f* = (1 - s) f + s f^eq, where s f^eq is formed from
// the terms of equilibrium13 each scaled by s through its constant (s f0 = s a kappa, s r,
// s q / 4, s c q, s c (q u + p), s c qx qy / h), so each population takes one add and one
// fused multiply-add.  s r is one fused multiply-add of h and -s f0 / 4: with s r rounded
// twice (s h / 4, then minus s f0 / 4) the FP32 depth drifted about 5 times as fast as with
// f + s (f^eq - f) on the 4096^2 dam-break; rounded once it drifts about as fast (+9e-7
// against +7e-7 relative over 1000 steps).  The moments (h, qx, qy) are returned too (the collision conserves
// them).  The operations stay mirror-symmetric: x -> -x flips the signs of qx, u, s c qx
// and s c qx qy / h exactly and leaves s c (qx u + p) unchanged.
template <class T>
__device__ __forceinline__ void collide13(T f[13], const Consts<T>& k, T& h, T& qx, T& qy) {
  moments13(f, h, qx, qy);
  const T rh = recip(h);
  const T u = mul(qx, rh);
  const T v = mul(qy, rh);
  const T uu = add(mul(u, u), mul(v, v));
  const T z = fmad(uu, k.s_a4g, mul(k.s_a2, h));  // -s f0^eq / 4
  const T f0 = mul(z, T(-4));                      // s f0^eq (exact)
  const T r = fmad(h, k.s_4, z);                   // s (h - f0^eq) / 4
  const T p = mul(mul(k.s_p, h), h);               // s c p
  const T ax = mul(qx, k.s_c);
  const T ay = mul(qy, k.s_c);
  const T x4 = mul(qx, k.s_4);
  const T y4 = mul(qy, k.s_4);
  const T pxx = fmad(ax, u, p);
  const T pyy = fmad(ay, v, p);
  const T pxy = mul(mul(mul(qx, qy), rh), k.s_c);
  const T om = k.om;
  f[0] = fmad(om, f[0], f0);
  f[1] = fmad(om, f[1], add(r, ax));
  f[2] = fmad(om, f[2], add(r, ay));
  f[3] = fmad(om, f[3], sub(r, ax));
  f[4] = fmad(om, f[4], sub(r, ay));
  f[5] = fmad(om, f[5], add(x4, pxx));
  f[6] = fmad(om, f[6], add(x4, pxy));
  f[7] = fmad(om, f[7], sub(x4, pxx));
  f[8] = fmad(om, f[8], sub(x4, pxy));
  f[9] = fmad(om, f[9], add(y4, pxy));
  f[10] = fmad(om, f[10], add(y4, pyy));
  f[11] = fmad(om, f[11], sub(y4, pxy));
  f[12] = fmad(om, f[12], sub(y4, pyy));
}

// FP64: the same operator in 42 operations of the FP64 unit instead of 59, the moments' 10 additions
// aside (sum_once).  The two terms of each equilibrium meet in one fused multiply-add, s r +- s c q
// and s q / 4 +- (s c h) t with t = u^2 + g h / 2, v^2 + g h / 2 or u v, so the products s c q and
// s c (q u + p) are not formed.  Mirror images still round alike.
__device__ __forceinline__ void collide13_fma(double f[13], const Consts<double>& k, double& h, double& qx, double& qy) {
  moments13(f, h, qx, qy);
  const double rh = recip(h);
  const double u = mul(qx, rh), v = mul(qy, rh);
  const double uu = mul(u, u), vv = mul(v, v), uv = mul(u, v);
  const double z = fmad(add(uu, vv), k.s_a4g, mul(k.s_a2, h));  // -s f0^eq / 4
  const double r = fmad(h, k.s_4, z);                           // s (h - f0^eq) / 4
  const double tx = fmad(k.half_g, h, uu), ty = fmad(k.half_g, h, vv);
  const double hc = mul(h, k.s_c), x4 = mul(qx, k.s_4), y4 = mul(qy, k.s_4);
  const double om = k.om;
  f[0] = fmad(om, f[0], times_pow2<2, true>(z));
  f[1] = fmad(om, f[1], fmad(k.s_c, qx, r));
  f[2] = fmad(om, f[2], fmad(k.s_c, qy, r));
  f[3] = fmad(om, f[3], fmad(-k.s_c, qx, r));
  f[4] = fmad(om, f[4], fmad(-k.s_c, qy, r));
  f[5] = fmad(om, f[5], fmad(hc, tx, x4));
  f[6] = fmad(om, f[6], fmad(hc, uv, x4));
  f[7] = fmad(om, f[7], fmad(-hc, tx, x4));
  f[8] = fmad(om, f[8], fmad(-hc, uv, x4));
  f[9] = fmad(om, f[9], fmad(hc, uv, y4));
  f[10] = fmad(om, f[10], fmad(hc, ty, y4));
  f[11] = fmad(om, f[11], fmad(-hc, uv, y4));
  f[12] = fmad(om, f[12], fmad(-hc, ty, y4));
}

// FP64, the usual case: the sums, s c q and the relaxation of the twelve moving populations in
// integers (above), each population rounded once: 18 operations of the FP64 unit.  The parts that
// the four populations of an equilibrium share, s (h - f0^eq) / 4 and s q / 4, are a quarter of what the relaxed
// populations leave of the integer sum (rounded to even), so the sums of depths and momenta
// keep their values but for the last rounding of each population, whatever the products lose.
// False, and nothing changed, where the values of a family differ too much in size (an equilibrium
// term more than twice the power of two of the largest population, as at the front of a
// jump; exponents near the ends of the range): collide13_fma takes the cell then.
// Bounds: the depths' units are 2^-59 of the power of two above their largest population, the
// momenta's of the one below, so populations are below 1/2 and 1 of 2^60 units and the remainders of
// the sums below 13/2 and 8; s c q is below 4; a relaxed population is below 25/4 (the
// integers' range is 8).
//
// 1536^2 cells, us per step: 278 with 59 operations in the FP64 unit, 218 with 52, 197 with the
// moments in integers, 144 this way (141 with s h / 4 and s q / 4 as truncated products, which lean one
// way; 158 with rounded ones).  Relative drift of the depths' sum of a dam break on 56^2
// cells after 20,000 steps, s = 1.8, 1.95 and 1.99: 8e-14, 1.8e-14 and 4e-15 with 59 operations, 5e-14,
// 3.3e-14 and 3.1e-14 with truncated products, at most 3e-16 this way.  Error against quadruple precision after
// 200 steps on 40^2 cells at s = 1.8: h 7.5e-16 and q 3.3e-15 with 59 operations, 1.1e-16 and 3.3e-16 (rates from
// 0.5 to 1.99, at rest, in a flow and in waves of 1e-2: 0.1 to 0.85 of the former error).
__device__ __forceinline__ bool collide13_fixed(double f[13], const Consts<double>& k, double& h, double& qx, double& qy) {
  int ef = exp_field(f[0]), ex = 0, ey = 0;
#pragma unroll
  for (int i = 1; i < 5; ++i) {
    ef = max(ef, exp_field(f[i]));
    ex = max(ex, exp_field(f[4 + i]));
    ey = max(ey, exp_field(f[8 + i]));
  }
  ef += 1 << 20;  // of the power of two above: the remainder of the sum, up to s h, has to fit
  if (!(k.fixed_ok && exp_fits(ef) && exp_fits(ex) && exp_fits(ey))) return false;
  unsigned long long m[13];
  long long v[3] = {0, 0, 0};
#pragma unroll
  for (int i = 0; i < 13; ++i) {
    m[i] = fix_mag(f[i], i < 5 ? ef : (i < 9 ? ex : ey));
    v[i < 5 ? 0 : (i < 9 ? 1 : 2)] += with_sign(m[i], __double2hiint(f[i]));
  }
  h = unfix(v[0], ef);
  qx = unfix(v[1], ex);
  qy = unfix(v[2], ey);
  const double rh = recip(h);
  const double u = mul(qx, rh), w = mul(qy, rh);
  const double uu = mul(u, u), ww = mul(w, w), uw = mul(u, w);
  const double z = fmad(add(uu, ww), k.s_a4g, mul(k.s_a2, h));  // -s f0^eq / 4
  const double hc = mul(h, k.s_c);
  const double pxx = mul(hc, fmad(k.half_g, h, uu)), pyy = mul(hc, fmad(k.half_g, h, ww)), pxy = mul(hc, uw);
  bool ok = true;
  const int sx = static_cast<int>(v[1] >> 32), sy = static_cast<int>(v[2] >> 32);  // their sign bits
  const unsigned long long ax = static_cast<unsigned long long>(v[1] < 0 ? -v[1] : v[1]);
  const unsigned long long ay = static_cast<unsigned long long>(v[2] < 0 ? -v[2] : v[2]);
  // s c q, in units of the f family's
  const long long cx = with_sign(to_units(times_2_64(ax, k.x_sc), (ef - ex) >> 20, k.least_sc, ok), sx);
  const long long cy = with_sign(to_units(times_2_64(ay, k.x_sc), (ef - ey) >> 20, k.least_sc, ok), sy);
  const double f0 = fmad(k.om, f[0], times_pow2<2, true>(z));  // relaxed
  const long long F0 = fix_one_more(f0, ef, ok);
  const long long fxx = fix_one_more(pxx, ex, ok), fxy = fix_one_more(pxy, ex, ok);
  const long long fyx = fix_one_more(pxy, ey, ok), fyy = fix_one_more(pyy, ey, ok);
  if (!ok) return false;
  const int flip = k.om_neg ? static_cast<int>(0x80000000u) : 0;
  long long t[13], rest[3] = {v[0] - F0, v[1], v[2]};
#pragma unroll
  for (int i = 1; i < 13; ++i) {
    t[i] = with_sign(times_2_64(m[i], k.x_om), __double2hiint(f[i]) ^ flip);
    rest[i < 5 ? 0 : (i < 9 ? 1 : 2)] -= t[i];
  }
  const long long fr = quarter(rest[0]), x4 = quarter(rest[1]), y4 = quarter(rest[2]);
  const long long eq[13] = {0,        fr + cx,  fr + cy,  fr - cx,  fr - cy,  x4 + fxx, x4 + fxy,
                            x4 - fxx, x4 - fxy, y4 + fyx, y4 + fyy, y4 - fyx, y4 - fyy};
  f[0] = f0;
#pragma unroll
  for (int i = 1; i < 13; ++i) f[i] = unfix(t[i] + eq[i], i < 5 ? ef : (i < 9 ? ex : ey));
  return true;
}

__device__ __forceinline__ void collide13(double f[13], const Consts<double>& k, double& h, double& qx, double& qy) {
  if (!collide13_fixed(f, k, h, qx, qy)) collide13_fma(f, k, h, qx, qy);
}

template <class T>
__device__ __forceinline__ void collide13(T f[13], const Consts<T>& k) {
  T h, qx, qy;
  collide13(f, k, h, qx, qy);
}

// MRT form: f* = f + M^-1 S M (f^eq - f), with M the 13 moments of section 3 (rho, J_x,
// J_y, eps, XX_rho; q_x, f_xx, f_xy, XX_u; q_y, f_yx, f_yy, XX_v), S = diag of the rates
// (0 on the conserved rho, q_x, q_y).  Family by family, with d = f^eq - f:
//   f:  dJx/lam = r0 (d1 - d3), dJy/lam = r1 (d2 - d4), deps = r2 (d1 + d2 + d3 + d4 - 4 d0),
//       dXX = r3 (d1 - d2 + d3 - d4); back: df0 = -deps/5, s13 = (deps/5 + dXX)/2,
//       s24 = (deps/5 - dXX)/2, df1,3 = (s13 +- dJx/lam)/2, df2,4 = (s24 +- dJy/lam)/2;
//   gx: dfxx/lam = r4 (g1 - g3), dfxy/lam = r5 (g2 - g4), dXX_u = r6 (g1 - g2 + g3 - g4);
//       back: dg1,3 = (dXX_u/2 +- dfxx/lam)/2, dg2,4 = (-dXX_u/2 +- dfxy/lam)/2;  gy alike (r7..r9).
// The halvings are folded into the rates (Consts::m) and into the quarter that forms s13/2
// and s24/2, which gives the same rounded values with 14 operations fewer per cell; the
// last correction of each momentum family is subtracted instead of negated and added.
template <class T>
__device__ __forceinline__ void mrt_family4(const T d[4], T ra2, T rb2, T rx4, T& g0, T& g1, T& g2, T& g3n) {
  const T ah = mul(ra2, sub(d[0], d[2]));  // (dfxx/lam) / 2
  const T bh = mul(rb2, sub(d[1], d[3]));  // (dfxy/lam) / 2
  const T xh = mul(rx4, sub(add(d[0], d[2]), add(d[1], d[3])));  // dXX_u / 4
  g0 = add(xh, ah);
  g2 = sub(xh, ah);
  g1 = sub(bh, xh);
  g3n = add(xh, bh);  // -dg4
}

template <class T>
__device__ __forceinline__ void collide13_mrt(T f[13], const Consts<T>& k, T& h, T& qx, T& qy) {
  moments13(f, h, qx, qy);
  T e[13];
  equilibrium13(h, qx, qy, k, e);
  T d[13];
#pragma unroll
  for (int j = 0; j < 13; ++j) d[j] = sub(e[j], f[j]);
  const T jxh = mul(k.m[0], sub(d[1], d[3]));
  const T jyh = mul(k.m[1], sub(d[2], d[4]));
  const T e5 = mul(mul(k.m[2], sub(add(add(d[1], d[2]), add(d[3], d[4])), mul(T(4), d[0]))), T(0.2));
  const T xx = mul(k.m[3], sub(add(d[1], d[3]), add(d[2], d[4])));
  const T s13q = mul(T(0.25), add(e5, xx)), s24q = mul(T(0.25), sub(e5, xx));
  f[0] = sub(f[0], e5);
  f[1] = add(f[1], add(s13q, jxh));
  f[3] = add(f[3], sub(s13q, jxh));
  f[2] = add(f[2], add(s24q, jyh));
  f[4] = add(f[4], sub(s24q, jyh));
  T g0, g1, g2, g3n;
  mrt_family4(d + 5, k.m[4], k.m[5], k.m[6], g0, g1, g2, g3n);
  f[5] = add(f[5], g0);
  f[6] = add(f[6], g1);
  f[7] = add(f[7], g2);
  f[8] = sub(f[8], g3n);
  mrt_family4(d + 9, k.m[7], k.m[8], k.m[9], g0, g1, g2, g3n);
  f[9] = add(f[9], g0);
  f[10] = add(f[10], g1);
  f[11] = add(f[11], g2);
  f[12] = sub(f[12], g3n);
}

// FP64, the usual case, in integers as collide13_fixed: 22 operations of the FP64 unit instead of
// 108 (the moments' sums aside).  The equilibria have no XX parts and conserve the depth, so the
// differences that the moments are made of are
//   d1 - d3 = 2 c qx - (f1 - f3),  d1 - d2 + d3 - d4 = -(f1 - f2 + f3 - f4),
//   d1 + d2 + d3 + d4 - 4 d0 = -5 d0,
// and likewise for the momenta's families: only d0, c qx, c qy and the three fluxes are formed.
// What one population gains from a moment another loses as the same integer, and a population
// of an equilibrium at rest keeps its bits (e0 and the pressure are evaluated as equilibrium13's).
// Bounds, with a family's largest population below one: 2 c q - (f1 - f3) below 6, a relaxed
// population below 8 (the integers' range).
//
// us per step, before and after: 480 x 120 19.7 and 6.3, 512^2 63.7 and 20.2, 1536^2 539 and 153 (BGK
// 144).  Error against extended precision after 300 steps of a dam break on 40^2 cells: h 8.8e-17 and
// 5.8e-17 (relative L1), q 4.2e-15 and 2.3e-15; no drift of the depths' sum over 10^5 steps in either.
__device__ __forceinline__ bool collide13_mrt_fixed(double f[13], const Consts<double>& k, double& h, double& qx,
                                                    double& qy) {
  int ef = exp_field(f[0]), ex = 0, ey = 0;
#pragma unroll
  for (int i = 1; i < 5; ++i) {
    ef = max(ef, exp_field(f[i]));
    ex = max(ex, exp_field(f[4 + i]));
    ey = max(ey, exp_field(f[8 + i]));
  }
  if (!(k.fixed_mrt_ok && exp_fits(ef) && exp_fits(ex) && exp_fits(ey))) return false;
  long long F[13], v[3] = {0, 0, 0};
#pragma unroll
  for (int i = 0; i < 13; ++i) {
    F[i] = with_sign(fix_mag(f[i], i < 5 ? ef : (i < 9 ? ex : ey)), __double2hiint(f[i]));
    v[i < 5 ? 0 : (i < 9 ? 1 : 2)] += F[i];
  }
  h = unfix(v[0], ef);
  qx = unfix(v[1], ex);
  qy = unfix(v[2], ey);
  const double rh = recip(h);
  const double u = mul(qx, rh), w = mul(qy, rh);
  const double uu = add(mul(u, u), mul(w, w));
  const double d0 = sub(mul(k.a, fmad(-uu, k.inv4g, times_pow2<-1, false>(h))), f[0]);
  const double p = mul(mul(k.half_g, h), h);
  const double pxx = mul(fmad(qx, u, p), k.c), pyy = mul(fmad(qy, w, p), k.c);
  const double pxy = mul(mul(mul(qx, qy), rh), k.c);
  bool ok = true;
  auto c_times = [&](long long q, int e) {  // c q, in units of the f family's
    const int s = static_cast<int>(q >> 32);
    return with_sign(to_units(times_2_64(static_cast<unsigned long long>(q < 0 ? -q : q), k.x_c), (ef - e) >> 20,
                              k.least_c, ok), s);
  };
  auto scaled = [&](long long x, unsigned long long c) {
    return with_sign(times_2_64(static_cast<unsigned long long>(x < 0 ? -x : x), c), static_cast<int>(x >> 32));
  };
  const long long cx = c_times(v[1], ex), cy = c_times(v[2], ey);
  const long long D0 = fix_one_more(d0, ef, ok);
  const long long fxx = fix_one_more(pxx, ex, ok), fxy = fix_one_more(pxy, ex, ok);
  const long long fyx = fix_one_more(pxy, ey, ok), fyy = fix_one_more(pyy, ey, ok);
  if (!ok) return false;
  // deps / 20, rounded: the depth's sum takes it four times
  const long long e4 = with_sign(times_2_64_round(static_cast<unsigned long long>(D0 < 0 ? -D0 : D0), k.x_m[2]),
                                 ~static_cast<int>(D0 >> 32));
  const long long xx = scaled(F[1] + F[3] - F[2] - F[4], k.x_m[3]);
  const long long jx = scaled(2 * cx - (F[1] - F[3]), k.x_m[0]), jy = scaled(2 * cy - (F[2] - F[4]), k.x_m[1]);
  f[0] = fmad(k.r[2], d0, f[0]);
  f[1] = unfix(F[1] + e4 - xx + jx, ef);
  f[2] = unfix(F[2] + e4 + xx + jy, ef);
  f[3] = unfix(F[3] + e4 - xx - jx, ef);
  f[4] = unfix(F[4] + e4 + xx - jy, ef);
#pragma unroll
  for (int i = 5; i < 13; i += 4) {
    const long long p1 = i == 5 ? fxx : fyx, p2 = i == 5 ? fxy : fyy;
    const unsigned long long* const m = k.x_m + (i == 5 ? 4 : 7);
    const int e = i == 5 ? ex : ey;
    const long long a = scaled(2 * p1 - (F[i] - F[i + 2]), m[0]), b = scaled(2 * p2 - (F[i + 1] - F[i + 3]), m[1]);
    const long long x = scaled(F[i] + F[i + 2] - F[i + 1] - F[i + 3], m[2]);
    f[i] = unfix(F[i] - x + a, e);
    f[i + 1] = unfix(F[i + 1] + x + b, e);
    f[i + 2] = unfix(F[i + 2] - x - a, e);
    f[i + 3] = unfix(F[i + 3] + x - b, e);
  }
  return true;
}

__device__ __forceinline__ void collide13_mrt(double f[13], const Consts<double>& k, double& h, double& qx, double& qy) {
  if (!collide13_mrt_fixed(f, k, h, qx, qy)) collide13_mrt<double>(f, k, h, qx, qy);
}

// Relaxation of either form.
template <class T, bool MRT>
__device__ __forceinline__ void collide13_any(T f[13], const Consts<T>& k, T& h, T& qx, T& qy) {
  if (MRT)
    collide13_mrt(f, k, h, qx, qy);
  else
    collide13(f, k, h, qx, qy);
}

// z = D(W)^T psi: vector-Jacobian product of the equilibria (closed forms of section 3
// in W = (h, qx, qy); kappa = h/2 - (qx^2 + qy^2)/(4 g h^2), c = 1/(2 lambda)).
template <class T>
__device__ __forceinline__ void equilibrium_vjp(T h, T qx, T qy, const T psi[13], const Consts<T>& K, T& zh,
                                                T& zx, T& zy) {
  const T rh = recip(h);
  const T u = qx * rh, v = qy * rh;
  const T gh = T(2) * K.half_g * h;
  const T inv2gh = T(2) * K.inv4g * rh;
  const T kh = T(0.5) + (u * u + v * v) * inv2gh;  // dkappa/dh
  const T kx = -u * inv2gh;                        // dkappa/dqx
  const T ky = -v * inv2gh;                        // dkappa/dqy
  const T Sf = (psi[1] + psi[3]) + (psi[2] + psi[4]);
  const T Af = psi[0] - T(0.25) * Sf;
  const T Df13 = psi[1] - psi[3], Df24 = psi[2] - psi[4];
  const T Sx = (psi[5] + psi[7]) + (psi[6] + psi[8]);
  const T Dx13 = psi[5] - psi[7], Dx24 = psi[6] - psi[8];
  const T Sy = (psi[9] + psi[11]) + (psi[10] + psi[12]);
  const T Dy13 = psi[9] - psi[11], Dy24 = psi[10] - psi[12];
  const T X = Dx24 + Dy13;
  const T c = K.c;
  zh = K.a * kh * Af + T(0.25) * Sf + c * (Dx13 * (gh - u * u) - X * u * v + Dy24 * (gh - v * v));
  zx = K.a * kx * Af + c * Df13 + T(0.25) * Sx + c * (T(2) * Dx13 * u + X * v);
  zy = K.a * ky * Af + c * Df24 + T(0.25) * Sy + c * (X * u + T(2) * Dy24 * v);
}

// ---- Two FP32 cells at once (the paired FP32 instructions of sm_100 and later) ----
// The same operations as collide13, in the same order, on (cell a, cell b) pairs, so each
// lane rounds exactly like the scalar code and the results are equal bit for bit.  The code
// generator contracts a paired multiply feeding a paired add into one fused multiply-add
// even when both carry an explicit rounding mode, which would change the rounding (and
// break the mirror symmetry of u u + v v).  So every paired product is formed as
// fma(a, b, nz) with nz = -0 read from the kernel's constants: exactly the rounded product
// a b (also for a zero product of either sign), in one instruction, and not a product
// the code generator can merge into the add that follows.
__device__ __forceinline__ unsigned long long pack2(float2 a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long r) {
  float2 a;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
  return a;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
  return unpack2(r);
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
  return unpack2(r);
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)), "l"(pack2(c)));
  return unpack2(r);
}
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }

// Moments and equilibria of two cells, as moments13 and equilibrium13.
__device__ __forceinline__ void moments_equilibrium13x2(const float2 f[13], const Consts<float>& k, float2& h,
                                                        float2& qx, float2& qy, float2 e[13]) {
  const float2 nz = dup2(k.nz);
  auto mul2 = [&](float2 a, float2 b) { return fma2(a, b, nz); };  // the rounded product a b
  h = add2(f[0], add2(add2(f[1], f[3]), add2(f[2], f[4])));
  qx = add2(add2(f[5], f[7]), add2(f[6], f[8]));
  qy = add2(add2(f[9], f[11]), add2(f[10], f[12]));
  const float2 rh = make_float2(recip(h.x), recip(h.y));
  const float2 u = mul2(qx, rh);
  const float2 v = mul2(qy, rh);
  const float2 uu = add2(mul2(u, u), mul2(v, v));
  // the sign on the constant instead of on uu: the same exact product, no negation per pair
  const float2 kap = fma2(uu, dup2(-k.inv4g), mul2(dup2(0.5f), h));
  const float2 f0 = mul2(dup2(k.a), kap);
  const float2 r = mul2(sub2(h, f0), dup2(0.25f));
  const float2 p = mul2(mul2(dup2(k.half_g), h), h);
  const float2 c = dup2(k.c);
  const float2 ax = mul2(qx, c);
  const float2 ay = mul2(qy, c);
  const float2 x4 = mul2(qx, dup2(0.25f));
  const float2 y4 = mul2(qy, dup2(0.25f));
  const float2 pxx = mul2(fma2(qx, u, p), c);
  const float2 pyy = mul2(fma2(qy, v, p), c);
  const float2 pxy = mul2(mul2(mul2(qx, qy), rh), c);
  e[0] = f0;
  e[1] = add2(r, ax);
  e[2] = add2(r, ay);
  e[3] = sub2(r, ax);
  e[4] = sub2(r, ay);
  e[5] = add2(x4, pxx);
  e[6] = add2(x4, pxy);
  e[7] = sub2(x4, pxx);
  e[8] = sub2(x4, pxy);
  e[9] = add2(y4, pxy);
  e[10] = add2(y4, pyy);
  e[11] = sub2(y4, pxy);
  e[12] = sub2(y4, pyy);
}

// collide13 on two cells, operation for operation; (h, qx, qy) receive the conserved
// moments of the pulled populations (as collide13's).
__device__ __forceinline__ void collide13x2(float2 f[13], const Consts<float>& k, float2& h, float2& qx, float2& qy) {
  const float2 nz = dup2(k.nz);
  auto mul2 = [&](float2 a, float2 b) { return fma2(a, b, nz); };  // the rounded product a b
  h = add2(f[0], add2(add2(f[1], f[3]), add2(f[2], f[4])));
  qx = add2(add2(f[5], f[7]), add2(f[6], f[8]));
  qy = add2(add2(f[9], f[11]), add2(f[10], f[12]));
  const float2 rh = make_float2(recip(h.x), recip(h.y));
  const float2 u = mul2(qx, rh);
  const float2 v = mul2(qy, rh);
  const float2 uu = add2(mul2(u, u), mul2(v, v));
  const float2 sc = dup2(k.s_c), s4 = dup2(k.s_4);
  const float2 z = fma2(uu, dup2(k.s_a4g), mul2(dup2(k.s_a2), h));
  const float2 f0 = mul2(z, dup2(-4.0f));
  const float2 r = fma2(h, s4, z);
  const float2 p = mul2(mul2(dup2(k.s_p), h), h);
  const float2 ax = mul2(qx, sc);
  const float2 ay = mul2(qy, sc);
  const float2 x4 = mul2(qx, s4);
  const float2 y4 = mul2(qy, s4);
  const float2 pxx = fma2(ax, u, p);
  const float2 pyy = fma2(ay, v, p);
  const float2 pxy = mul2(mul2(mul2(qx, qy), rh), sc);
  const float2 om = dup2(k.om);
  f[0] = fma2(om, f[0], f0);
  f[1] = fma2(om, f[1], add2(r, ax));
  f[2] = fma2(om, f[2], add2(r, ay));
  f[3] = fma2(om, f[3], sub2(r, ax));
  f[4] = fma2(om, f[4], sub2(r, ay));
  f[5] = fma2(om, f[5], add2(x4, pxx));
  f[6] = fma2(om, f[6], add2(x4, pxy));
  f[7] = fma2(om, f[7], sub2(x4, pxx));
  f[8] = fma2(om, f[8], sub2(x4, pxy));
  f[9] = fma2(om, f[9], add2(y4, pxy));
  f[10] = fma2(om, f[10], add2(y4, pyy));
  f[11] = fma2(om, f[11], sub2(y4, pxy));
  f[12] = fma2(om, f[12], sub2(y4, pyy));
}

__device__ __forceinline__ void collide13x2(float2 f[13], const Consts<float>& k) {
  float2 h, qx, qy;
  collide13x2(f, k, h, qx, qy);
}

// The MRT form of collide13_mrt on (cell a, cell b) pairs, operation for operation.
__device__ __forceinline__ void mrt_family4x2(const float2 d[4], float ra2, float rb2, float rx4, float2 nz,
                                              float2& g0, float2& g1, float2& g2, float2& g3n) {
  auto mul2 = [&](float2 a, float2 b) { return fma2(a, b, nz); };
  const float2 ah = mul2(dup2(ra2), sub2(d[0], d[2]));
  const float2 bh = mul2(dup2(rb2), sub2(d[1], d[3]));
  const float2 xh = mul2(dup2(rx4), sub2(add2(d[0], d[2]), add2(d[1], d[3])));
  g0 = add2(xh, ah);
  g2 = sub2(xh, ah);
  g1 = sub2(bh, xh);
  g3n = add2(xh, bh);
}

__device__ __forceinline__ void collide13x2_mrt(float2 f[13], const Consts<float>& k, float2& h, float2& qx,
                                                float2& qy) {
  const float2 nz = dup2(k.nz);
  auto mul2 = [&](float2 a, float2 b) { return fma2(a, b, nz); };
  float2 e[13];
  moments_equilibrium13x2(f, k, h, qx, qy, e);
  float2 d[13];
#pragma unroll
  for (int j = 0; j < 13; ++j) d[j] = sub2(e[j], f[j]);
  const float2 quarter = dup2(0.25f);
  const float2 jxh = mul2(dup2(k.m[0]), sub2(d[1], d[3]));
  const float2 jyh = mul2(dup2(k.m[1]), sub2(d[2], d[4]));
  const float2 e5 =
      mul2(mul2(dup2(k.m[2]), sub2(add2(add2(d[1], d[2]), add2(d[3], d[4])), mul2(dup2(4.0f), d[0]))), dup2(0.2f));
  const float2 xx = mul2(dup2(k.m[3]), sub2(add2(d[1], d[3]), add2(d[2], d[4])));
  const float2 s13q = mul2(quarter, add2(e5, xx)), s24q = mul2(quarter, sub2(e5, xx));
  f[0] = sub2(f[0], e5);
  f[1] = add2(f[1], add2(s13q, jxh));
  f[3] = add2(f[3], sub2(s13q, jxh));
  f[2] = add2(f[2], add2(s24q, jyh));
  f[4] = add2(f[4], sub2(s24q, jyh));
  float2 g0, g1, g2, g3n;
  mrt_family4x2(d + 5, k.m[4], k.m[5], k.m[6], nz, g0, g1, g2, g3n);
  f[5] = add2(f[5], g0);
  f[6] = add2(f[6], g1);
  f[7] = add2(f[7], g2);
  f[8] = sub2(f[8], g3n);
  mrt_family4x2(d + 9, k.m[7], k.m[8], k.m[9], nz, g0, g1, g2, g3n);
  f[9] = add2(f[9], g0);
  f[10] = add2(f[10], g1);
  f[11] = add2(f[11], g2);
  f[12] = sub2(f[12], g3n);
}

template <bool MRT>
__device__ __forceinline__ void collide13x2_any(float2 f[13], const Consts<float>& k, float2& h, float2& qx,
                                                float2& qy) {
  if constexpr (MRT)
    collide13x2_mrt(f, k, h, qx, qy);
  else
    collide13x2(f, k, h, qx, qy);
}

// ---- 1D: populations f0, f+, f-, g+, g- ----
template <class T>
__device__ __forceinline__ void moments5(const T f[5], T& h, T& q) {
  h = add(f[0], add(f[1], f[2]));
  q = add(f[3], f[4]);
}

template <class T>
__device__ __forceinline__ void equilibrium5(T h, T q, const Consts<T>& k, T e[5]) {
  const T rh = recip(h);
  const T u = mul(q, rh);
  const T kap = fmad(-mul(u, u), k.inv4g, mul(T(0.5), h));
  const T f0 = mul(k.a, kap);
  const T hf = sub(h, f0);  // half = hf / 2
  const T aq = mul(q, k.c);
  const T p = mul(mul(k.half_g, h), h);
  const T pq = mul(fmad(q, u, p), k.c);
  // exact halves folded into fused multiply-adds, as in equilibrium13
  e[0] = f0;
  e[1] = fmad(hf, T(0.5), aq);
  e[2] = fmad(hf, T(0.5), -aq);
  e[3] = fmad(q, T(0.5), pq);
  e[4] = fmad(q, T(0.5), -pq);
}

template <class T>
__device__ __forceinline__ void collide5(T f[5], const Consts<T>& k) {
  T h, q;
  moments5(f, h, q);
  T e[5];
  equilibrium5(h, q, k, e);
#pragma unroll
  for (int j = 0; j < 5; ++j) f[j] = fmad(k.s, sub(e[j], f[j]), f[j]);
}

// FP64 in 1D, where the integers do not fit: the same f + s (f^eq - f) with 26 operations of the FP64 unit instead of 32 (a
// line's steps are one warp's chain of them): the halves by the exponent field, the flux
// c (q u + p) as (c h) (u^2 + g h / 2) inside the fused multiply-adds of g+-.  The folded
// (1 - s) f + s f^eq would save four more, but its depth drifts: on 1000 cells after 500 steps
// the error of h against quadruple precision is 6e-16 in this form and the one above, 2e-15 folded.
__device__ __forceinline__ void collide5_fma(double f[5], const Consts<double>& k) {
  double h, q;
  moments5(f, h, q);
  const double u = mul(q, recip(h)), uu = mul(u, u);
  const double f0 = fmad(uu, k.a_4g, mul(h, k.a_2));
  const double r = times_pow2<-1, false>(sub(h, f0));  // (h - f0) / 2
  const double t = fmad(k.half_g, h, uu);
  const double hc = mul(h, k.c), q2 = times_pow2<-1, false>(q);
  const double e[5] = {f0, fmad(k.c, q, r), fmad(-k.c, q, r), fmad(hc, t, q2), fmad(-hc, t, q2)};
#pragma unroll
  for (int j = 0; j < 5; ++j) f[j] = fmad(k.s, sub(e[j], f[j]), f[j]);
}

// FP64 in 1D, the usual case, in integers as collide13_fixed: 10 operations of the FP64 unit.  It
// relaxes the differences f^eq - f, so a settled lake at rest keeps its bits, as in the form above;
// what one population gains others lose as the same integer.
// Bounds, with a family's largest population below one: c q below 1, an equilibrium term below 2, a
// relaxed population below 8 (the integers' range).
// 1000 cells, us per step: 1.43 with 32 operations of the FP64 unit, 1.18 with 26, 0.92 this way (0.94 folded, which
// moved 37 % of all lakes at rest by an ulp).
__device__ __forceinline__ bool collide5_fixed(double f[5], const Consts<double>& k) {
  const int ef = max(exp_field(f[0]), max(exp_field(f[1]), exp_field(f[2])));
  const int eg = max(exp_field(f[3]), exp_field(f[4]));
  if (!(k.fixed1_ok && exp_fits(ef) && exp_fits(eg))) return false;
  long long F[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) F[i] = with_sign(fix_mag(f[i], i < 3 ? ef : eg), __double2hiint(f[i]));
  const long long v = F[3] + F[4];
  const double h = unfix(F[0] + (F[1] + F[2]), ef), q = unfix(v, eg);
  const double u = mul(q, recip(h)), uu = mul(u, u);
  const double f0 = fmad(uu, k.a_4g, mul(h, k.a_2));
  const double pq = mul(mul(h, k.c), fmad(k.half_g, h, uu));
  bool ok = true;
  const long long c = with_sign(to_units(times_2_64(static_cast<unsigned long long>(v < 0 ? -v : v), k.x_c), (ef - eg) >> 20,
                                         k.least_c, ok), static_cast<int>(v >> 32));
  const long long e0 = fix_one_more(f0, ef, ok), p = fix_one_more(pq, eg, ok);
  if (!ok) return false;
  auto half_s_times = [&](long long d) {
    return with_sign(times_2_64(static_cast<unsigned long long>(d < 0 ? -d : d), k.x_s2), static_cast<int>(d >> 32));
  };
  const long long d0 = half_s_times(e0 - F[0]), df = half_s_times(2 * c - (F[1] - F[2])), dg = half_s_times(2 * p - (F[3] - F[4]));
  f[0] = unfix(F[0] + 2 * d0, ef);
  f[1] = unfix(F[1] - d0 + df, ef);
  f[2] = unfix(F[2] - d0 - df, ef);
  f[3] = unfix(F[3] + dg, eg);
  f[4] = unfix(F[4] - dg, eg);
  return true;
}

__device__ __forceinline__ void collide5(double f[5], const Consts<double>& k) {
  if (!collide5_fixed(f, k)) collide5_fma(f, k);
}

// MRT form in 1D on the moments of section 2 (rho, J_rho = lam (f+ - f-),
// eps_rho = lam^2 (f+ + f- - 2 f0), q, J_q = lam (g+ - g-)); with d = f^eq - f:
// dJ/lam = r0 (d+ - d-), deps/lam^2 = r1 (d+ + d- - 2 d0), dJq/lam = r2 (dg+ - dg-);
// back: sum = deps/(3 lam^2), df0 = -sum, df+- = (sum +- dJ/lam)/2, dg+- = +- dJq/(2 lam).
template <class T>
__device__ __forceinline__ void collide5_mrt(T f[5], const Consts<T>& k) {
  T h, q;
  moments5(f, h, q);
  T e[5];
  equilibrium5(h, q, k, e);
  T d[5];
#pragma unroll
  for (int j = 0; j < 5; ++j) d[j] = e[j] - f[j];
  const T j1 = k.r[0] * (d[1] - d[2]);
  const T sm = k.r[1] * ((d[1] + d[2]) - T(2) * d[0]) * T(1.0 / 3.0);
  const T jq = k.r[2] * (d[3] - d[4]) * T(0.5);
  f[0] = f[0] - sm;
  f[1] = f[1] + T(0.5) * (sm + j1);
  f[2] = f[2] + T(0.5) * (sm - j1);
  f[3] = f[3] + jq;
  f[4] = f[4] - jq;
}

template <class T, bool MRT>
__device__ __forceinline__ void collide5_any(T f[5], const Consts<T>& k) {
  if (MRT)
    collide5_mrt(f, k);
  else
    collide5(f, k);
}

}  // namespace lbm
