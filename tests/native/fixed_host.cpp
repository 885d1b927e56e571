// Host build of the FP64 step's fixed-point arithmetic (lbm_fixed.cuh) beside the FP64 forms of
// lbm_core.cuh, and both in long double, for a site's window of densities.
#include "lbm_consts.h"

using namespace lbm;

namespace {

struct Ld {  // the forms of lbm_core.cuh in long double
    long double ps[25];
    const double *K, *q;
};

long double psi_l(double rho, double rho0) { return -expm1l(-(long double)rho / (long double)rho0); }

}  // namespace

extern "C" {

// psi of rho: out[0] fixed point, out[1] FP64 formula; returns |error| of the fixed-point value
// against long double, in units of 2^-56
double fixed_psi(double rho, double rho0, double* out) {
    const ExpFx K = exp_fx_const(rho0);
    const i64 v = psi_fx(rho, K);
    out[0] = scaled_double(v, -56);
    out[1] = 1.0 - exp(-rho / rho0);
    const long double got = (long double)v * 0x1p-56L;
    return (double)(fabsl(got - psi_l(rho, rho0)) * 0x1p56L);
}

double fixed_rcp(double x) { return rcp_fx(x); }

double fixed_scaled(long long v, int e) { return scaled_double(v, e); }

// Force and Appendix A stresses of one species over 25 densities: F, S (3) in fixed point, F64, S64
// in FP64 from FP64 psi, FL, SL by long double links.
void fixed_site(const lbm_params* p, int s, const double* rho25, double* F, double* S, double* F64, double* S64,
                double* FL, double* SL) {
    StepConst<double> C;
    const double rr[2] = {0.0, 0.0};
    fill_step_const<double>(C, *p, 8, 8, 32, 256, 2, 0, rr);
    i64 w[5][5];
    double d[5][5];
    long double l[5][5];
    for (int k = 0; k < 25; ++k) {
        w[k / 5][k % 5] = psi_fx(rho25[k], C.ex[s]);
        d[k / 5][k % 5] = psi_of(C, s, rho25[k]);
        l[k / 5][k % 5] = psi_l(rho25[k], p->rho0[s]);
    }
    intra_force_fx(C.kf[s], w, scaled_double(w[2][2], -56), F[0], F[1]);
    S[0] = S[1] = S[2] = S64[0] = S64[1] = S64[2] = 0.0;
    intra_stress_fx(C.sf[s], w, S[0], S[1], S[2]);
    intra_force(C, s, d, F64[0], F64[1]);
    intra_stress(C, s, d, S64[0], S64[1], S64[2]);
    long double K[9], f[2] = {0, 0}, t[3] = {0, 0, 0};
    for (int q = 0; q < 9; ++q) {
        const long double wa = p->weight_preset == LBM_WEIGHTS_CHEM09 ? w_belt1(q) : w_attr_paper(q);
        K[q] = (long double)p->weight_norm * ((long double)p->G1[s] * wa + (long double)p->G2[s] * w_rep(q));
    }
#define P(x, z) l[(z) + 2][(x) + 2]
    for (int z = -2; z <= 2; ++z)
        for (int x = -2; x <= 2; ++x) {
            const int q = x * x + z * z;
            if (q == 0) continue;
            f[0] -= P(0, 0) * K[q] * P(x, z) * x;
            f[1] -= P(0, 0) * K[q] * P(x, z) * z;
            long double v = (q <= 2 ? 0.5L : 0.25L) * K[q] * P(0, 0) * P(x, z);
            if (x > 0 || (x == 0 && z > 0)) {  // one of each antipodal pair
                if (q == 4 || q == 8) v += 0.25L * K[q] * 2 * P(x / 2, z / 2) * P(-x / 2, -z / 2);
                if (q == 5) {
                    const int mx = x / 2, mz = z / 2, kx = x - mx, kz = z - mz;
                    v += 0.25L * K[q] * (P(kx, kz) * P(-mx, -mz) + P(mx, mz) * P(-kx, -kz));
                }
            }
            t[0] += v * x * x;
            t[1] += v * z * z;
            t[2] += v * x * z;
        }
#undef P
    for (int k = 0; k < 2; ++k) FL[k] = (double)f[k];
    for (int k = 0; k < 3; ++k) SL[k] = (double)t[k];
}
}
