// Host build of the pseudopotential and its exponential as numbers of their own (lbm_fixed.cuh), each
// beside the FP64 formula, with their errors against long double in units of 2^-53 of the value.
#include "lbm_fixed.cuh"

using namespace lbm;

extern "C" {

// out: the number, the formula's value, the two errors
void number_psi(double rho, double rho0, double* out) {
    const long double want = -expm1l(-(long double)rho / (long double)rho0);
    out[0] = psi_number(rho, 1.0 / rho0, exp_fx_const(rho0));
    out[1] = -expm1(-rho * (1.0 / rho0));
    for (int k = 0; k < 2; ++k) out[2 + k] = (double)(fabsl(out[k] - want) / want * 0x1p53L);
}
void number_exp(double rho, double rho0, double* out) {
    const long double want = expl(-(long double)rho / (long double)rho0);
    out[0] = exp_number(rho, 1.0 / rho0, exp_fx_const(rho0));
    out[1] = exp(-rho * (1.0 / rho0));
    for (int k = 0; k < 2; ++k) out[2 + k] = (double)(fabsl(out[k] - want) / want * 0x1p53L);
}
long long number_bits57(double psi) { return psi_bits57(psi); }
}
extern "C" int coef_taken(const double* c) {
    CoefFx<5> F;
    return coef_fx(F, c);
}
