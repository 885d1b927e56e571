// lbm_fixed.cuh -- the parts of the FP64 step that are bounded by the pseudopotential's range, in
// 64-bit fixed point on the integer pipes.
//
// Why: this GPU's FP64 pipe takes 2 operations per SM per cycle, so one warp FP64 instruction
// holds it for 16 cycles, in which the SM's four schedulers issue 64 other instructions.  A 64-bit
// integer add is 2 of those and a 64 x 64 -> high 64 product about 12, so exact sums and bounded
// products cost a small fraction of their FP64 forms and run beside the FP64 work that is left.
// psi = 1 - exp(-rho / rho0) lies in [0, 1] for every density > 0, which gives its sums and
// products a range known beforehand; nothing here depends on the size of rho.
//
// Precision: psi is held with 2^-60 resolution (an FP64 psi in [1/2, 1) has 2^-53, one of 0.06 has
// 2^-57), sums and differences are exact, products are truncated at 2^-58 or below.  Measured
// against long double (tests/test_fixed_host.py): psi within 2^-56, forces and stresses no further
// off than the FP64 forms of lbm_core.cuh.
//
// Everything is __host__ __device__, so the same arithmetic is tested on the host.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#if defined(__CUDACC__)
#define LBM_FX __host__ __device__ __forceinline__
#else
#define LBM_FX inline
#endif

namespace lbm {

using i64 = long long;
using u64 = unsigned long long;

LBM_FX u64 mulhi_u(u64 a, u64 b) {
#if defined(__CUDA_ARCH__)
    return __umul64hi(a, b);
#else
    return (u64)(((unsigned __int128)a * b) >> 64);
#endif
}
LBM_FX i64 mulhi_s(i64 a, i64 b) {
#if defined(__CUDA_ARCH__)
    return __mul64hi(a, b);
#else
    return (i64)(((__int128)a * b) >> 64);
#endif
}
LBM_FX int clz64(u64 a) {
#if defined(__CUDA_ARCH__)
    return __clzll((i64)a);
#else
    return a ? __builtin_clzll(a) : 64;
#endif
}
LBM_FX u64 bits_of(double v) {
#if defined(__CUDA_ARCH__)
    return (u64)__double_as_longlong(v);
#else
    u64 b;
    memcpy(&b, &v, sizeof b);
    return b;
#endif
}
LBM_FX double of_bits(u64 b) {
#if defined(__CUDA_ARCH__)
    return __longlong_as_double((i64)b);
#else
    double v;
    memcpy(&v, &b, sizeof v);
    return v;
#endif
}

// v 2^e rounded to FP64 (to nearest, halves up), |v| < 2^63, the result a normal number or 0.
LBM_FX double scaled_double(i64 v, int e) {
    const u64 a = v < 0 ? (u64)0 - (u64)v : (u64)v;
    if (a == 0) return 0.0;
    const int lz = clz64(a);
    const u64 m = a << lz;                         // bit 63 set: |v| = m 2^-lz
    const u64 q = (m >> 11) + ((m >> 10) & 1);     // 2^52 .. 2^53; the carry of 2^53 moves into the exponent
    const u64 b = ((u64)(1085 + e - lz) << 52) + q;  // (1086 + e - lz) - 1: q holds the implicit bit
    return of_bits(b | (v < 0 ? (u64)1 << 63 : (u64)0));
}

// ---- exp(-rho / rho0) and psi -------------------------------------------------------------------

// log2(e) / rho0 = km 2^(ke - 63), 2^63 <= km < 2^64.
struct ExpFx {
    u64 km;
    int ke, pad;
};

inline ExpFx exp_fx_const(double rho0) {
    const long double k = 1.44269504088896340735992468100189214L / (long double)rho0;
    int e = 0;
    const long double m = frexpl(k, &e);  // k = m 2^e, 1/2 <= m < 1
    long double s = ldexpl(m, 64);
    ExpFx x;
    x.km = s >= 18446744073709551615.0L ? ~(u64)0 : (u64)s;
    x.ke = e - 1;
    x.pad = 0;
    return x;
}

// 2^63 2^(-j / 32), rounded
#define LBM_EXP2_TABLE                                                                              \
    0x8000000000000000ull, 0x7d41d96db915019dull, 0x7a92be8a92436616ull, 0x77f25ccdee6d7ae6ull,     \
    0x75606373ee921c97ull, 0x72dc8373be41a454ull, 0x70666f76154a7089ull, 0x6dfddbcbed791babull,     \
    0x6ba27e656b4eb57aull, 0x69540ec8f895722dull, 0x6712460a8fc24072ull, 0x64dcdec3371793d1ull,     \
    0x62b39508aa836d6full, 0x6096266533384a2bull, 0x5e8451cfac061b5full, 0x5c7dd7a3b17dcf75ull,     \
    0x5a827999fcef3242ull, 0x5891fac0e95612c8ull, 0x56ac1f752150a563ull, 0x54d0ad5a753e077cull,     \
    0x52ff6b54d8a89c75ull, 0x513821818624b40cull, 0x4f7a993048d088d7ull, 0x4dc69cdceaa72a9cull,     \
    0x4c1bf828c6dc54b8ull, 0x4a7a77d47f7b84b1ull, 0x48e1e9b9d588e19bull, 0x47521cc5a2e6a9e0ull,     \
    0x45cae0f1f545eb73ull, 0x444c0740496d4294ull, 0x42d561b3e6243d8aull, 0x4166c34c5615d0ecull
#if defined(__CUDACC__)
static __device__ const u64 exp2_table_dev[32] = {LBM_EXP2_TABLE};
#endif
static const u64 exp2_table_host[32] = {LBM_EXP2_TABLE};
#undef LBM_EXP2_TABLE

// Whether exp_fx takes rho: positive, finite, with room for the exponent arithmetic.
LBM_FX bool exp_fx_takes(double rho) { return rho > 1e-290 && rho < 1e290; }

// exp(-rho / rho0) 2^62 for such a rho, by table and polynomial in integers (the table-driven
// exponential of Tang, ACM TOMS 15(2), 1989, in base 2): t = rho log2(e) / rho0 with 57 fraction
// bits; its integer part is a shift, the next 5 bits a table entry, and 2^-r of the remaining
// r < 2^-5 is the Taylor polynomial of degree 8 (remainder below 2^-66).  About 110 integer
// instructions, against some 40 FP64 ones (640 cycles of the SM's FP64 pipe per warp) for the
// division and the library's exponential.
LBM_FX u64 exp_fx(double rho, const ExpFx& K) {
#if defined(__CUDA_ARCH__)
    const u64* const table = exp2_table_dev;
#else
    const u64* const table = exp2_table_host;
#endif
    const u64 b = bits_of(rho);
    const int ex = (int)(b >> 52) & 0x7ff;
    const u64 p = mulhi_u((b << 11) | (u64)1 << 63, K.km);  // t = p 2^(ex + ke - 1085)
    const int s = 1028 - ex - K.ke;
    if (s < 0) return 0;  // t >= 64: below 2^-63
    const u64 t = s < 64 ? p >> s : 0;
    const int n = (int)(t >> 57);
    if (n > 62) return 0;
    const u64 g = t << 7;                    // the fraction, 2^64 scale
    const u64 r = g & (((u64)1 << 59) - 1);  // below 2^-5
    // 1 - 2^-r = r (c1 - r (c2 - ...)), c_k = (ln 2)^k / k! on the 2^64 scale
    u64 v = 0x0000162c0223a5c8ull;
    v = 0x0000ffe5fe2c4586ull - mulhi_u(r, v);
    v = 0x000a184897c363c4ull - mulhi_u(r, v);
    v = 0x005761ff9e299cc4ull - mulhi_u(r, v);
    v = 0x0276556df749cee5ull - mulhi_u(r, v);
    v = 0x0e35846b82505fc6ull - mulhi_u(r, v);
    v = 0x3d7f7bff058b1d51ull - mulhi_u(r, v);
    v = 0xb17217f7d1cf79acull - mulhi_u(r, v);
    const u64 e = ((u64)1 << 63) - (mulhi_u(r, v) >> 1);  // 2^-r, 2^63 scale
    return mulhi_u(e, table[g >> 59]) >> n;
}

// psi on the 2^60 scale (0 for a density that exp_fx does not take: one that is <= 0, NaN or Inf
// has been flagged, and one that small has psi < 2^-900)
LBM_FX i64 psi_fx(double rho, const ExpFx& K) {
    if (!exp_fx_takes(rho)) return rho > 0.0 && rho >= 1e290 ? (i64)1 << 60 : 0;
    return (i64)((((u64)1 << 62) - exp_fx(rho, K) + 2) >> 2);
}

// ---- forces and stresses --------------------------------------------------------------------

// Coefficients c_k = v[k] 2^(e - 62), |v[k]| <= 2^62.
struct CoefFx {
    i64 v[5];
    double c[3];  // c_1, c_3, c_4 themselves
    int e, pad;
};
inline void coef_fx(CoefFx& F, const double* c) {
    F.c[0] = c[1];
    F.c[1] = c[3];
    F.c[2] = c[4];
    double top = 0.0;
    for (int k = 0; k < 5; ++k) top = fabs(c[k]) > top ? fabs(c[k]) : top;
    int e = 0;
    if (top > 0.0) (void)frexp(top, &e);  // top < 2^e
    for (int k = 0; k < 5; ++k) F.v[k] = (i64)ldexp(c[k], 62 - e);
    F.e = e;
    F.pad = 0;
}

// Eq. FORCE of one species from the 5 x 5 window p of psi on the 2^60 scale: intra_force of
// lbm_core.cuh with every sum exact.  K: K(1), K(2), 2 K(4), K(5), 2 K(8).  psi0: psi at the site.
// Every shell sum is at most 6, and their weighted sum at most 12 (coefficients <= 1): 12 2^58
// fits.  10 products and about 30 adds in integers and 4 FP64 instructions replace 34 FP64 ones.
LBM_FX void intra_force_fx(const CoefFx& K, const i64 (&p)[5][5], double psi0, double& fx, double& fz) {
#define LBM_Q(dx, dz) p[(dz) + 2][(dx) + 2]
    const i64 d10 = LBM_Q(1, 0) - LBM_Q(-1, 0), d01 = LBM_Q(0, 1) - LBM_Q(0, -1);
    const i64 d11 = LBM_Q(1, 1) - LBM_Q(-1, -1), e11 = LBM_Q(-1, 1) - LBM_Q(1, -1);
    const i64 d20 = LBM_Q(2, 0) - LBM_Q(-2, 0), d02 = LBM_Q(0, 2) - LBM_Q(0, -2);
    const i64 d21 = LBM_Q(2, 1) - LBM_Q(-2, -1), e21 = LBM_Q(-2, 1) - LBM_Q(2, -1);
    const i64 d12 = LBM_Q(1, 2) - LBM_Q(-1, -2), e12 = LBM_Q(-1, 2) - LBM_Q(1, -2);
    const i64 d22 = LBM_Q(2, 2) - LBM_Q(-2, -2), e22 = LBM_Q(-2, 2) - LBM_Q(2, -2);
    const i64 x5 = 2 * (d21 - e21) + (d12 - e12), z5 = 2 * (d12 + e12) + (d21 + e21);
    const i64 sx = mulhi_s(K.v[0], d10) + mulhi_s(K.v[1], d11 - e11) + mulhi_s(K.v[2], d20) + mulhi_s(K.v[3], x5) +
                   mulhi_s(K.v[4], d22 - e22) + 2;  // 5 truncated products: 2.5 low in the mean
    const i64 sz = mulhi_s(K.v[0], d01) + mulhi_s(K.v[1], d11 + e11) + mulhi_s(K.v[2], d02) + mulhi_s(K.v[3], z5) +
                   mulhi_s(K.v[4], d22 + e22) + 2;
    fx = -psi0 * scaled_double(sx, K.e - 58);
    fz = -psi0 * scaled_double(sz, K.e - 58);
#undef LBM_Q
}

// Appendix A's stresses of one species from the same window (intra_stress of lbm_core.cuh), added
// into (sxx, szz, sxz).  Q: sq(1), sq(2), 4 sq(4), sq(5), 4 sq(8).  Products of two psi are
// formed on the 2^58 scale; the shells' sums (at most 40 in shell 5) meet on the 2^57 scale, the
// weighted sums (at most 2 + 4 + 4 + 40 + 8) on the 2^55 scale.  33 products in integers and 6 FP64
// instructions replace about 65 FP64 ones.
LBM_FX void intra_stress_fx(const CoefFx& Q, const i64 (&p)[5][5], double& sxx, double& szz, double& sxz) {
#define LBM_P(dx, dz) p[(dz) + 2][(dx) + 2]
#define LBM_M(a, b) mulhi_s((a) * 4, (b))  // 2^62 x 2^k -> 2^(k - 2)
    const i64 p0 = LBM_P(0, 0) * 4;        // 2^62
    const i64 s10 = LBM_P(1, 0) + LBM_P(-1, 0), s01 = LBM_P(0, 1) + LBM_P(0, -1);
    const i64 d2 = LBM_P(1, 1) + LBM_P(-1, -1), a2 = LBM_P(-1, 1) + LBM_P(1, -1);
    const i64 x1 = mulhi_s(p0, s10) >> 1, z1 = mulhi_s(p0, s01) >> 1;
    const i64 t2 = mulhi_s(p0, d2 + a2) >> 1, u2 = mulhi_s(p0, d2 - a2) >> 1;
    // |c|^2 = 4
    const i64 x4 = (mulhi_s(p0, LBM_P(2, 0) + LBM_P(-2, 0)) >> 1) + LBM_M(LBM_P(-1, 0), LBM_P(1, 0));
    const i64 z4 = (mulhi_s(p0, LBM_P(0, 2) + LBM_P(0, -2)) >> 1) + LBM_M(LBM_P(0, -1), LBM_P(0, 1));
    // |c|^2 = 5: sums of up to 20 psi on the 2^58 scale
    const i64 a21 = (LBM_P(2, 1) + LBM_P(-2, -1)) >> 2, b21 = (LBM_P(-2, 1) + LBM_P(2, -1)) >> 2;
    const i64 a12 = (LBM_P(1, 2) + LBM_P(-1, -2)) >> 2, b12 = (LBM_P(-1, 2) + LBM_P(1, -2)) >> 2;
    const i64 t13 = LBM_M(LBM_P(1, 1), LBM_P(-1, 0)) + LBM_M(LBM_P(1, 0), LBM_P(-1, -1));
    const i64 t14 = LBM_M(LBM_P(1, 1), LBM_P(0, -1)) + LBM_M(LBM_P(0, 1), LBM_P(-1, -1));
    const i64 t15 = LBM_M(LBM_P(0, 1), LBM_P(1, -1)) + LBM_M(LBM_P(-1, 1), LBM_P(0, -1));
    const i64 t16 = LBM_M(LBM_P(-1, 1), LBM_P(1, 0)) + LBM_M(LBM_P(-1, 0), LBM_P(1, -1));
    const i64 o = t13 + t16, v = t14 + t15;
    const i64 x5 = 2 * mulhi_s(p0, 4 * (a21 + b21) + (a12 + b12)) + ((4 * o + v) >> 1);
    const i64 z5 = 2 * mulhi_s(p0, (a21 + b21) + 4 * (a12 + b12)) + ((o + 4 * v) >> 1);
    const i64 w5 = 4 * mulhi_s(p0, (a21 - b21) + (a12 - b12)) + ((t13 + t14) - (t15 + t16));
    // |c|^2 = 8
    const i64 a22 = LBM_P(2, 2) + LBM_P(-2, -2), b22 = LBM_P(-2, 2) + LBM_P(2, -2);
    const i64 ha = LBM_M(LBM_P(-1, -1), LBM_P(1, 1)), hb = LBM_M(LBM_P(-1, 1), LBM_P(1, -1));
    const i64 t8 = (mulhi_s(p0, a22 + b22) >> 1) + (ha + hb);
    const i64 u8 = (mulhi_s(p0, a22 - b22) >> 1) + (ha - hb);
    const i64 both = mulhi_s(Q.v[1], t2) + mulhi_s(Q.v[4], t8) + 2;  // as above
    sxx += scaled_double(mulhi_s(Q.v[0], x1) + mulhi_s(Q.v[2], x4) + mulhi_s(Q.v[3], x5) + both, Q.e - 55);
    szz += scaled_double(mulhi_s(Q.v[0], z1) + mulhi_s(Q.v[2], z4) + mulhi_s(Q.v[3], z5) + both, Q.e - 55);
    // xz, a difference of nearly equal sums, is small: weighted in FP64, whose rounding follows its size
    sxz += (Q.c[0] * scaled_double(u2, -57) + Q.c[1] * scaled_double(w5, -57)) + Q.c[2] * scaled_double(u8, -57);
#undef LBM_P
#undef LBM_M
}

}  // namespace lbm
