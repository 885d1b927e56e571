// lbm_fixed.cuh -- the parts of the FP64 step that are bounded by the pseudopotential's range, in
// 64-bit fixed point on the integer pipes.
//
// Why: this GPU's FP64 pipe takes 2 operations per SM per cycle, so one warp FP64 instruction
// holds it for 16 cycles, in which the SM's four schedulers issue 64 other instructions.  A 64-bit
// integer add is 2 of those, a 32 x 32 + 64 -> 64 multiply-add 1 or 2, a 64 x 64 -> high 64 product
// about 8, so exact sums and bounded products cost a small fraction of their FP64 forms and run
// beside the FP64 work that is left.
// psi = 1 - exp(-rho / rho0) lies in [0, 1] for every density > 0, which gives its sums and
// products a range known beforehand; nothing here depends on the size of rho.  A density <= 0 (a state
// that a run may pass through) has no psi in that range: the steps take the FP64 forms for it.
//
// Precision: psi is held with 2^-56 resolution (1 - exp(-x) in FP64 has an error of up to 2^-53
// whatever its size, that of the exponential), sums and differences are exact, the force is rounded
// once, the stresses' products are truncated at 2^-56 or below.  Measured against long double
// (tests/test_fixed_host.py): psi within 2^-56, forces and stresses no further off than the FP64
// forms of lbm_core.cuh.
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

// A float as a double by its bits: the conversion instruction takes the FP64 pipe 16 cycles a warp.
LBM_FX double widen_fx(float v) {
#if defined(__CUDA_ARCH__)
    const unsigned b = __float_as_uint(v);
    const unsigned e = b & 0x7f800000u;
    if (e != 0u && e != 0x7f800000u)  // normal: the exponent rebiased, the mantissa moved up
        return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
#endif
    return (double)v;
}

// 1 / x for a normal x with |x| in 2^-1000 .. 2^1000: a seed from the FP32 reciprocal of the mantissa
// (relative error below 2^-21), then one step of the third-order (Halley) iteration
// y (1 + d + d^2), d = 1 - x y, whose remainder d^3 is below 2^-63: 3 FP64 instructions, the error
// within an ulp (tests/test_fixed_host.py).
LBM_FX double rcp_fx(double x) {
    const u64 b = bits_of(x);
    const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
    const unsigned mb = 0x3f800000u | (hi & 0xfffffu) << 3 | lo >> 29;  // the mantissa, 1 <= m < 2
#if defined(__CUDA_ARCH__)
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(mb)));
    const unsigned rb = __float_as_uint(r);
#else
    float m, r;
    memcpy(&m, &mb, sizeof m);
    r = 1.0f / m;
    unsigned rb;
    memcpy(&rb, &r, sizeof rb);
#endif
    // r 2^(1023 - ex) with the sign of x: FP32's exponent moved to FP64's bias
    const unsigned ex = hi >> 20 & 0x7ff;
    const u64 yb = ((u64)rb << 29) + ((u64)(1023 - 127 + 1023 - (int)ex) << 52);
    const double y = of_bits(yb | (b & (u64)1 << 63));
    const double d = fma(-x, y, 1.0);
    return fma(y, fma(d, d, d), y);
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

// 2^63 2^(-j / 128), rounded
#define LBM_EXP2_TABLE                                                                              \
    0x8000000000000000ull, 0x7f4f08ae3dc7c426ull, 0x7e9f06067a4360baull, 0x7deff6b672f84e24ull,     \
    0x7d41d96db915019dull, 0x7c94acddaeea5d3aull, 0x7be86fb985689ddcull, 0x7b3d20b6399fc237ull,     \
    0x7a92be8a92436616ull, 0x79e947ef1d320d2dull, 0x7940bb9e2cffd89dull, 0x78991853d684a285ull,     \
    0x77f25ccdee6d7ae6ull, 0x774c87cc06d1812eull, 0x76a7980f6cca15c2ull, 0x76038c5b260e5eeeull,     \
    0x75606373ee921c97ull, 0x74be1c203627c62bull, 0x741cb5281e25ee34ull, 0x737c2d55770fe711ull,     \
    0x72dc8373be41a454ull, 0x723db6501b9ed447ull, 0x719fc4b95f452d29ull, 0x7102ad7fff41e9b4ull,     \
    0x70666f76154a7089ull, 0x6fcb096f5c782210ull, 0x6f307a412f074892ull, 0x6e96c0c284192610ull,     \
    0x6dfddbcbed791babull, 0x6d65ca379564e639ull, 0x6cce8ae13c57ebdbull, 0x6c381ca636d99642ull,     \
    0x6ba27e656b4eb57aull, 0x6b0daeff4fcde703ull, 0x6a79ad55e7f6fd10ull, 0x69e6784cc2cd61bdull,     \
    0x69540ec8f895722dull, 0x68c26fb128b4cd63ull, 0x683199ed779592caull, 0x67a18c678c8c8c61ull,     \
    0x6712460a8fc24072ull, 0x6683c5c3281ee6e9ull, 0x65f60a7f79393e2eull, 0x6569132f21483ba7ull,     \
    0x64dcdec3371793d1ull, 0x64516c2e47ff1623ull, 0x63c6ba6455dcd8aeull, 0x633cc85ad5122fbdull,     \
    0x62b39508aa836d6full, 0x622b1f66299a6599ull, 0x61a3666d124bb204ull, 0x611c69188f1eb339ull,     \
    0x6096266533384a2bull, 0x60109d50f86846d8ull, 0x5f8bccdb3d398841ull, 0x5f07b404c304c9f1ull,     \
    0x5e8451cfac061b5full, 0x5e01a53f7974fd86ull, 0x5d7fad59099f22feull, 0x5cfe69229605cef5ull,     \
    0x5c7dd7a3b17dcf75ull, 0x5bfdf7e546520f3eull, 0x5b7ec8f19468bbc9ull, 0x5b0049d42f6afbb6ull,     \
    0x5a827999fcef3242ull, 0x5a05575132a5cc20ull, 0x5988e20954889245ull, 0x590d18d3330c7f1eull,     \
    0x5891fac0e95612c8ull, 0x581786e5db7022c2ull, 0x579dbc56b48521baull, 0x57249a29651adc07ull,     \
    0x56ac1f752150a563ull, 0x56344b525f1ff495ull, 0x55bd1cdad49f699cull, 0x5546932976483b15ull,     \
    0x54d0ad5a753e077cull, 0x545b6a8b3d990704ull, 0x53e6c9da74b29ab5ull, 0x5372ca67f774358full,     \
    0x52ff6b54d8a89c75ull, 0x528cabc35f4f799dull, 0x521a8ad704f3404full, 0x51a907b474015dc9ull,     \
    0x513821818624b40cull, 0x50c7d76542a25b72ull, 0x50582887dcb8a7e1ull, 0x4fe91412b2006e83ull,     \
    0x4f7a993048d088d7ull, 0x4f0cb70c4ea39210ull, 0x4e9f6cd3967fdba8ull, 0x4e32b9b417619617ull,     \
    0x4dc69cdceaa72a9cull, 0x4d5b157e4a7fc325ull, 0x4cf022c9905bfd32ull, 0x4c85c3f13360c4d5ull,     \
    0x4c1bf828c6dc54b8ull, 0x4bb2bea4f8bd5847ull, 0x4b4a169b900c2d00ull, 0x4ae1ff436b663ff7ull,     \
    0x4a7a77d47f7b84b1ull, 0x4a137f87d58e025bull, 0x49ad159789f37496ull, 0x4947393eca98fcd6ull,     \
    0x48e1e9b9d588e19bull, 0x487d2645f7725895ull, 0x4818ee218a3358eeull, 0x47b5408bf36472e2ull,     \
    0x47521cc5a2e6a9e0ull, 0x46ef821011734e6bull, 0x468d6fadbf2dd4f3ull, 0x462be4e23237a6efull,     \
    0x45cae0f1f545eb73ull, 0x456a632296394492ull, 0x450a6abaa4b77ecdull, 0x44aaf701b0c72feeull,     \
    0x444c0740496d4294ull, 0x43ed9abffb4c6bc9ull, 0x438fb0cb4f468808ull, 0x433248adc91fdd02ull,     \
    0x42d561b3e6243d8aull, 0x4278fb2b1bce0d15ull, 0x421d1461d66f2023ull, 0x41c1aca777db771bull,     \
    0x4166c34c5615d0ecull, 0x410c57a1b9fe12f6ull, 0x40b268f9de0183baull, 0x4058f6a7ecccd5b6ull
#if defined(__CUDACC__)
static __device__ const u64 exp2_table_dev[128] = {LBM_EXP2_TABLE};
#endif
static const u64 exp2_table_host[128] = {LBM_EXP2_TABLE};
#undef LBM_EXP2_TABLE

LBM_FX unsigned mulhi32(unsigned a, unsigned b) {
#if defined(__CUDA_ARCH__)
    return __umulhi(a, b);
#else
    return (unsigned)(((u64)a * b) >> 32);
#endif
}

// exp(-rho / rho0) 2^62 for a normal rho > 0, by table and polynomial in integers (the table-driven
// exponential of Tang, ACM TOMS 15(2), 1989, in base 2): t = rho log2(e) / rho0 with 57 fraction
// bits; its integer part is a shift, the next 7 bits a table entry, and 2^-r of the remaining
// r = R 2^-7 is the Taylor polynomial of degree 6 (remainder below 2^-64).  With R in [0, 1) the
// coefficients shrink by 2^-7 each, so the upper terms fit 32 bits on the common 2^64 scale and
// take one-instruction products; five 64-bit products are left.  No branches: a thread's several
// exponentials interleave.  About 80 integer instructions, against some 40 FP64 ones (640 cycles
// of the SM's FP64 pipe per warp) for the division and the library's exponential.
//
// exp_parts: q and n with exp(-rho / rho0) = q 2^(-62 - n), 2^61 <= q <= 2^62, and n = 64 where t is 64 or
// more.  FINE keeps the fraction bits of t below 2^-57 too (within 2^-60 of the exponential then,
// relatively, instead of 2^-57 of 1), for callers that need it as a number of its own.
template <bool FINE>
LBM_FX u64 exp_parts(double rho, const ExpFx& K, int& n) {
#if defined(__CUDA_ARCH__)
    const u64* const table = exp2_table_dev;
#else
    const u64* const table = exp2_table_host;
#endif
    const u64 b = bits_of(rho);
    const int ex = (int)(b >> 52) & 0x7ff;
    const u64 p = mulhi_u((b << 11) | (u64)1 << 63, K.km);  // t = p 2^(ex + ke - 1085)
    const int s = 1028 - ex - K.ke;                         // < 0: t >= 64, exp below 2^-63
    const u64 t = (s > 63 ? 0 : p >> (s & 63));
    n = s < 0 ? 64 : (int)(t >> 57);
    u64 R = t << 14;
    if (FINE && s >= 0) R = s < 14 ? p << (14 - s) : (s - 14 > 63 ? 0 : p >> (s - 14));
    const unsigned R32 = (unsigned)(R >> 32);
    // 1 - 2^-r = R (c1 - R (c2 - ...)), c_k = (ln 2)^k / k! 2^(-7 k) on the 2^64 scale
    unsigned w = 0xaec40u - mulhi32(R32, 0x286u);
    w = 0x276556dfu - mulhi32(R32, w);
    u64 v = 0x71ac235c13ull - mulhi32(R32, w);
    v = 0xf5fdeffc162cull - mulhi_u(R, v);
    v = 0x162e42fefa39ef3ull - mulhi_u(R, v);
    const u64 e = ((u64)1 << 63) - (mulhi_u(R, v) >> 1);  // 2^-r, 2^63 scale
    return mulhi_u(e, table[(t >> 50) & 127]);
}
LBM_FX u64 exp_fx(double rho, const ExpFx& K) {
    int n;
    const u64 q = exp_parts<false>(rho, K, n);
    return n < 64 ? q >> n : 0;
}

// Whether exp_fx takes rho: positive, finite, with room for the exponent arithmetic.
LBM_FX bool exp_fx_takes(double rho) { return rho > 1e-290 && rho < 1e290; }

// exp(-rho / rho0) and psi as numbers of their own, good to the last bit or two whatever their size, as the
// library's exp and expm1 are (the fixed-point forms above are good to 2^-56 of 1): what a derivative
// multiplies.  Those are called where the fixed-point form would be short of bits: small psi, whose
// difference from 1 cancels, exponentials below 2^-64, and densities that exp_fx does not take.
LBM_FX double exp_number(double rho, double inv_rho0, const ExpFx& K) {
    if (exp_fx_takes(rho)) {
        int n;
        const u64 q = exp_parts<true>(rho, K, n);
        if (n < 64) return scaled_double((i64)q, -62 - n);
    }
    return exp(-rho * inv_rho0);
}
constexpr double PSI_SMALL = 0.03125;  // 2^-5
LBM_FX double psi_number(double rho, double inv_rho0, const ExpFx& K) {
    if (exp_fx_takes(rho)) {
        int n;
        const u64 q = exp_parts<true>(rho, K, n);
        const u64 v = ((u64)1 << 62) - (n < 64 ? q >> n : 0);
        if (v >= (u64)1 << 57) return scaled_double((i64)v, -62);
    }
    return -expm1(-rho * inv_rho0);
}
// A psi of PSI_SMALL .. 1 on the 2^57 scale, which its FP64 value is a multiple of: exact.
LBM_FX i64 psi_bits57(double psi) {
    const u64 b = bits_of(psi);
    return (i64)(((b & (((u64)1 << 52) - 1)) | (u64)1 << 52) << (((int)(b >> 52) - 1018) & 63));
}

// psi on the 2^56 scale; for a density that exp_fx does not take 1 or 0 (callers look at one that is <= 0
// or NaN themselves; one below 1e-290 has psi = 0 to any precision held here)
LBM_FX i64 psi_fx(double rho, const ExpFx& K) {
    const i64 v = (i64)((((u64)1 << 62) - exp_fx(rho, K) + 32) >> 6);
    const bool big = rho >= 1e290;
    return rho > 1e-290 && !big ? v : (big ? (i64)1 << 56 : 0);
}

// ---- forces and stresses --------------------------------------------------------------------

// N coefficients c_k = v[k] 2^(e - 62), |v[k]| <= 2^62, and c_k = (h[k] 2^29 + l[k]) 2^(e - 58) in two
// limbs, 0 <= l < 2^29, |h| <= 2^29.
template <int N>
struct CoefFx {
    i64 v[N];
    double c[N];  // the coefficients themselves
    int h[N], l[N];
    int e, pad;
};
// False, and all zero, for coefficients whose largest is not zero and outside 2^-900 .. 2^900 (or not
// finite): the sums' exponents would leave FP64's range.  Those go through the FP64 forms.
template <int N>
inline bool coef_fx(CoefFx<N>& F, const double* c) {
    F = CoefFx<N>{};
    double top = 0.0;
    for (int k = 0; k < N; ++k) {
        if (!isfinite(c[k])) return false;
        top = fabs(c[k]) > top ? fabs(c[k]) : top;
    }
    if (top != 0.0 && (top < 0x1p-900 || top > 0x1p900)) return false;
    int e = 0;
    if (top > 0.0) (void)frexp(top, &e);  // top < 2^e
    for (int k = 0; k < N; ++k) {
        F.c[k] = c[k];
        F.v[k] = (i64)ldexp(c[k], 62 - e);
        const i64 u = (i64)rint(ldexp(c[k], 58 - e));
        F.h[k] = (int)(u >> 29);
        F.l[k] = (int)(u & ((1 << 29) - 1));
    }
    F.e = e;
    return true;
}

// sum_k c_k S_k of a few sums |S_k| < 2^60, exact in three accumulators of 29-bit limb products (each a
// 32 x 32 -> 64 multiply-add), rounded once to the nearest: sum() 2^(e - 2) times the scale of S.
// Rounding every product down instead would push each site the same way, a drift that adds up over
// the steps; this is odd in S.  Room: with |c_k| <= 2^e and sum_k |S_k| <= 2^60.6 no accumulator
// passes 2^62.7.
struct DotFx {
    i64 hh = 0, mid = 0, ll = 0;
    template <int N>
    LBM_FX void add(const CoefFx<N>& K, int k, i64 S) {
        const int sh = (int)(S >> 29), sl = (int)(S & ((1 << 29) - 1));
        hh += (i64)sh * K.h[k];
        mid += (i64)sh * K.l[k];
        mid += (i64)sl * K.h[k];
        ll += (i64)sl * K.l[k];
    }
    LBM_FX i64 sum() const { return (hh << 2) + ((mid + (ll >> 29) + (1 << 26)) >> 27); }
};

// Eq. FORCE of one species from the 5 x 5 window p of psi on the 2^56 scale: intra_force of
// lbm_core.cuh with every sum exact.  K: K(1), K(2), 2 K(4), K(5), 2 K(8).  psi0: psi at the site.
// The shell sums are at most 1, 2, 1, 6 and 2, and their weighted sum at most 12 2^e, which fits.  40 multiply-adds
// and about 30 adds in integers and 4 FP64 instructions replace 34 FP64 ones.
LBM_FX void intra_force_fx(const CoefFx<5>& K, const i64 (&p)[5][5], double psi0, double& fx, double& fz) {
#define LBM_Q(dx, dz) p[(dz) + 2][(dx) + 2]
    const i64 d11 = LBM_Q(1, 1) - LBM_Q(-1, -1), e11 = LBM_Q(-1, 1) - LBM_Q(1, -1);
    const i64 d21 = LBM_Q(2, 1) - LBM_Q(-2, -1), e21 = LBM_Q(-2, 1) - LBM_Q(2, -1);
    const i64 d12 = LBM_Q(1, 2) - LBM_Q(-1, -2), e12 = LBM_Q(-1, 2) - LBM_Q(1, -2);
    const i64 d22 = LBM_Q(2, 2) - LBM_Q(-2, -2), e22 = LBM_Q(-2, 2) - LBM_Q(2, -2);
    DotFx x, z;
    x.add(K, 0, LBM_Q(1, 0) - LBM_Q(-1, 0));
    z.add(K, 0, LBM_Q(0, 1) - LBM_Q(0, -1));
    x.add(K, 1, d11 - e11);
    z.add(K, 1, d11 + e11);
    x.add(K, 2, LBM_Q(2, 0) - LBM_Q(-2, 0));
    z.add(K, 2, LBM_Q(0, 2) - LBM_Q(0, -2));
    x.add(K, 3, 2 * (d21 - e21) + (d12 - e12));
    z.add(K, 3, 2 * (d12 + e12) + (d21 + e21));
    x.add(K, 4, d22 - e22);
    z.add(K, 4, d22 + e22);
    fx = -psi0 * scaled_double(x.sum(), K.e - 58);
    fz = -psi0 * scaled_double(z.sum(), K.e - 58);
#undef LBM_Q
}

// Appendix A's stresses of one species from the same window (intra_stress of lbm_core.cuh), added
// into (sxx, szz, sxz), with psi shifted to the 2^60 scale.  Q: sq(1), sq(2), 4 sq(4), sq(5), 4 sq(8).  Products of two psi are
// formed on the 2^58 scale; the shells' sums (at most 40 in shell 5) meet on the 2^57 scale, the
// weighted sums (at most 2 + 4 + 4 + 40 + 8) on the 2^55 scale.  33 products in integers and 6 FP64
// instructions replace about 65 FP64 ones.
LBM_FX void intra_stress_fx(const CoefFx<5>& Q, const i64 (&p)[5][5], double& sxx, double& szz, double& sxz) {
#define LBM_P(dx, dz) (p[(dz) + 2][(dx) + 2] << 4)           // 2^60
#define LBM_M(a, b) (i64)mulhi_u((u64)(a) << 2, (u64)(b))    // 2^62 x 2^k -> 2^(k - 2), nothing negative
    const i64 p0 = p[2][2] << 6;                             // 2^62
    const i64 s10 = LBM_P(1, 0) + LBM_P(-1, 0), s01 = LBM_P(0, 1) + LBM_P(0, -1);
    const i64 d2 = LBM_P(1, 1) + LBM_P(-1, -1), a2 = LBM_P(-1, 1) + LBM_P(1, -1);
    const i64 x1 = (i64)mulhi_u(p0, s10) >> 1, z1 = (i64)mulhi_u(p0, s01) >> 1;
    const i64 t2 = (i64)mulhi_u(p0, d2 + a2) >> 1, u2 = mulhi_s(p0, d2 - a2) >> 1;
    // |c|^2 = 4
    const i64 x4 = ((i64)mulhi_u(p0, LBM_P(2, 0) + LBM_P(-2, 0)) >> 1) + LBM_M(LBM_P(-1, 0), LBM_P(1, 0));
    const i64 z4 = ((i64)mulhi_u(p0, LBM_P(0, 2) + LBM_P(0, -2)) >> 1) + LBM_M(LBM_P(0, -1), LBM_P(0, 1));
    // |c|^2 = 5: sums of up to 20 psi on the 2^58 scale
    const i64 a21 = (LBM_P(2, 1) + LBM_P(-2, -1)) >> 2, b21 = (LBM_P(-2, 1) + LBM_P(2, -1)) >> 2;
    const i64 a12 = (LBM_P(1, 2) + LBM_P(-1, -2)) >> 2, b12 = (LBM_P(-1, 2) + LBM_P(1, -2)) >> 2;
    const i64 t13 = LBM_M(LBM_P(1, 1), LBM_P(-1, 0)) + LBM_M(LBM_P(1, 0), LBM_P(-1, -1));
    const i64 t14 = LBM_M(LBM_P(1, 1), LBM_P(0, -1)) + LBM_M(LBM_P(0, 1), LBM_P(-1, -1));
    const i64 t15 = LBM_M(LBM_P(0, 1), LBM_P(1, -1)) + LBM_M(LBM_P(-1, 1), LBM_P(0, -1));
    const i64 t16 = LBM_M(LBM_P(-1, 1), LBM_P(1, 0)) + LBM_M(LBM_P(-1, 0), LBM_P(1, -1));
    const i64 o = t13 + t16, v = t14 + t15;
    const i64 x5 = 2 * (i64)mulhi_u(p0, 4 * (a21 + b21) + (a12 + b12)) + ((4 * o + v) >> 1);
    const i64 z5 = 2 * (i64)mulhi_u(p0, (a21 + b21) + 4 * (a12 + b12)) + ((o + 4 * v) >> 1);
    const i64 w5 = 4 * mulhi_s(p0, (a21 - b21) + (a12 - b12)) + ((t13 + t14) - (t15 + t16));
    // |c|^2 = 8
    const i64 a22 = LBM_P(2, 2) + LBM_P(-2, -2), b22 = LBM_P(-2, 2) + LBM_P(2, -2);
    const i64 ha = LBM_M(LBM_P(-1, -1), LBM_P(1, 1)), hb = LBM_M(LBM_P(-1, 1), LBM_P(1, -1));
    const i64 t8 = ((i64)mulhi_u(p0, a22 + b22) >> 1) + (ha + hb);
    const i64 u8 = (mulhi_s(p0, a22 - b22) >> 1) + (ha - hb);
    const i64 both = mulhi_s(Q.v[1], t2) + mulhi_s(Q.v[4], t8) + 2;  // 5 products rounded down: 2.5 low in the mean
    sxx += scaled_double(mulhi_s(Q.v[0], x1) + mulhi_s(Q.v[2], x4) + mulhi_s(Q.v[3], x5) + both, Q.e - 55);
    szz += scaled_double(mulhi_s(Q.v[0], z1) + mulhi_s(Q.v[2], z4) + mulhi_s(Q.v[3], z5) + both, Q.e - 55);
    // xz, a difference of nearly equal sums, is small: weighted in FP64, whose rounding follows its size
    sxz += (Q.c[1] * scaled_double(u2, -57) + Q.c[3] * scaled_double(w5, -57)) + Q.c[4] * scaled_double(u8, -57);
#undef LBM_P
#undef LBM_M
}

}  // namespace lbm
