// lbm_adjoint.cu -- discrete adjoint of the time step (periodic lattice), in FP64 or FP32.
//
// The step maps the post-streaming populations f_n to f_{n+1} = S(f_n; theta):
//   rho_s = sum_l f_l, j_s = sum_l f_l c_l (Sec. II); psi_s = psi(rho_s) (Sec. IV);
//   F_s = -psi_s(x) sum_c (G1_s w(c) + G2_s p(c)) psi_s(x + c) c            (Eq. FORCE)
//         - G_AB rho_s(x) sum_c w8(c) rho_s'(x + c) c + rho_s g x            (Sec. IV);
//   u' = sum_s j_s / tau_s / sum_s rho_s / tau_s, u_s = u' + tau_s F_s / rho_s;
//   feq_l = W_l rho_s (1 + 3 c.u_s + 9/2 (c.u_s)^2 - 3/2 u_s.u_s);
//   g_l = f_l - (f_l - feq_l) / tau_s (Eq. LB);  f_{n+1}(x + c_l, l) = g_l(x).
// Given lam_{n+1} = dJ/df_{n+1}, three kernels form lam_n = dJ/df_n and the derivatives with
// respect to theta = (G1 A, G1 B, G2 A, G2 B, G_AB, tau A, tau B, g) by applying the transposed
// derivative of each stage in reverse order:
//   k_adj_moments  rho, j and psi of the state f_n (the linearisation point) -- for the first
//                  step of a sweep; for the others k_adj_final of the step before forms them;
//   k_adj_local    the force at the site (from its neighbours' psi and rho), then streaming
//                  transposed (a gather of lam_{n+1}), relaxation, equilibrium, shifted and
//                  common velocity transposed: dJ/dF_s, the site's own share of dJ/drho_s and
//                  dJ/dj_s, and every parameter derivative of the site;
//   k_adj_final    the neighbour shares of the force transposed (each site gathers what the
//                  forces at x - c owe to its psi and rho), the pseudopotential and the
//                  moments: lam_n; and the moments of f_{n-1} for the next step back.
// k_adj_local and k_adj_final work on tiles of 32 x ATZ sites and stage their neighbourhood fields
// (2 cells around the tile) in shared memory.  In FP64, bound by the FP64 pipe, antipodal links are
// gathered shell by shell as in the forward step, psi's sums in fixed point (lbm_fixed.cuh) on tiles
// where every psi is a multiple of its unit (2^-5 and above; elsewhere in FP64), and lam enters the collision's transpose through its six moments sum_l W_l lam_l (1, c, c c), formed of
// lam_l - lam_0.  In FP32, bound by latency, the sums stay link by link: the derivative of the body
// force is a small difference that a run's rounding fixes to 1e-6 .. 1e-5 of itself, and other sums,
// as exact, would land elsewhere in that range.
// In FP32 the kernels of a sweep follow one another by programmatic dependent launch.
// T is the precision of the states and of lam (FP64, or FP32 for FP32 forward runs).  The
// parameter derivatives are summed per block (FP64, or double-float pairs in FP32 mode), kept
// per block across the steps of a call, then summed over the blocks in FP64 in a fixed order.
#include "lbm_consts.h"
#include "lbm_internal.h"
#include "lbm_reduce.cuh"

namespace lbm {

namespace {

constexpr int AT = 256;  // threads per block of the objective and sum kernels
constexpr int NPAR = 8;
// Tiles of the per-step kernels: 32 columns (a warp a row) and, in FP64, whose pipe the SM with the
// most sites bounds, half the rows, for an even share of small lattices.
template <typename T>
struct Tile {
    static constexpr int Z = sizeof(T) == 4 ? 4 : 2, NT = 32 * Z;  // rows, threads
    static constexpr int W = 36, H = Z + 4;                        // with 2 cells around
};

// (dx, dz) of the 24 interaction links, first belt first (|c|^2 = 1, 2), then 4, 5, 8; constant
// expressions, so an unrolled loop over the links folds them
LBM_HD constexpr int LKX(int k) {
    constexpr int t[24] = {1, 0, -1, 0, 1, -1, -1, 1, 2, 0, -2, 0, 2, 1, -1, -2, -2, -1, 1, 2, 2, -2, -2, 2};
    return t[k];
}
LBM_HD constexpr int LKZ(int k) {
    constexpr int t[24] = {0, 1, 0, -1, 1, 1, -1, -1, 0, 2, 0, -2, 1, 2, 2, 1, -1, -2, -2, -1, 2, 2, -2, -2};
    return t[k];
}

// Periodic coordinate of v, -2 <= v: the position itself where it lies in the lattice.
__device__ __forceinline__ int wrap_t(int v, int n) {
    if (v >= 0 && v < n) return v;
    const int w = v < 0 ? v + n : v - n;
    if (w >= 0 && w < n) return w;
    return ((v % n) + n) % n;  // tiny lattices, and the columns past a ragged edge
}

// Programmatic dependent launch: nothing global is touched before the kernel before is complete.
__device__ __forceinline__ void pdl_enter() {
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
}

// FP64: by shell, the weights w(1), w(2), 2 w(4), w(5), 2 w(8) of the attraction and the repulsion and
// their sum K = G1 wa + G2 wr; the exponential and the weights in fixed point.
template <typename T>
struct AdjFixed {};
template <>
struct AdjFixed<double> {
    double sa[5], sr[5], K[2][5];
    ExpFx ex[2];
    CoefFx<5> fa, fr;  // of sa and sr
    int fixed;         // psi = 1 - exp(-rho / rho0) and the weights within coef_fx's range
};

template <typename T>
struct AdjC : AdjFixed<T> {
    int nx, nz, ns, psi_form;
    T wa[9], wr[9], wc[9];  // by |c|^2, weight_norm included
    T G1[2], G2[2], tau[2], itau[2], irho0[2];
    T G_AB, g;
};

// psi, and its derivative.
__device__ __forceinline__ float psi_t(const AdjC<float>& A, int s, float r) {
    return A.psi_form == 1 ? r : -expm1f(-r * A.irho0[s]);
}
__device__ __forceinline__ double psi_t(const AdjC<double>& A, int s, double r) {
    return A.psi_form == 1 ? r : psi_number(r, A.irho0[s], A.ex[s]);
}
__device__ __forceinline__ float dpsi_t(const AdjC<float>& A, int s, float r) {
    return A.psi_form == 1 ? 1.f : expf(-r * A.irho0[s]) * A.irho0[s];
}
__device__ __forceinline__ double dpsi_t(const AdjC<double>& A, int s, double r) {
    return A.psi_form == 1 ? 1.0 : exp_number(r, A.irho0[s], A.ex[s]) * A.irho0[s];
}

// Block accumulators: FP64, or a double-float pair (hi, lo) summed with TwoSum on the FP32 pipes.
template <typename T> struct Acc;
template <> struct Acc<double> {
    using A = double;
    __device__ static A from(double v) { return v; }
    __device__ static A add(A a, A b) { return a + b; }
    __device__ static A shfl(A a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
    __device__ static double wide(A a) { return a; }
};
template <> struct Acc<float> {
    using A = float2;
    __device__ static A from(float v) { return make_float2(v, 0.f); }
    __device__ static A add(A a, A b) { return ff_add(a, b); }
    __device__ static A shfl(A a, int o) {
        return make_float2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
    }
    __device__ static double wide(A a) { return (double)a.x + (double)a.y; }
};

// Sums over the warp of the eight values v[k]: each exchange halves what a lane still holds (9 adds,
// not 8 x 5), so lane 4 q' (q' = q with its bits reversed into lane bits 4, 3, 2) ends with sum q.
// Fixed order, so results repeat bit for bit.
template <typename R>
__device__ typename R::A warp_sum8(const typename R::A (&v)[NPAR], int& q) {
    using A = typename R::A;
    const int lane = threadIdx.x & 31;
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
    A v4[4], v2[2], v1;
#pragma unroll
    for (int k = 0; k < 4; ++k) v4[k] = R::add(b4 ? v[k + 4] : v[k], R::shfl(b4 ? v[k] : v[k + 4], 16));
#pragma unroll
    for (int k = 0; k < 2; ++k) v2[k] = R::add(b3 ? v4[k + 2] : v4[k], R::shfl(b3 ? v4[k] : v4[k + 2], 8));
    v1 = R::add(b2 ? v2[1] : v2[0], R::shfl(b2 ? v2[0] : v2[1], 4));
    v1 = R::add(v1, R::shfl(v1, 2));
    v1 = R::add(v1, R::shfl(v1, 1));
    q = (b4 ? 4 : 0) + (b3 ? 2 : 0) + (b2 ? 1 : 0);
    return v1;
}

// Block sums of the per-thread values v[k] (k < NPAR), stored to part[blk][k], or added to it
// (accumulate).
template <typename T>
__device__ void block_sum(const T (&v)[NPAR], typename Acc<T>::A* part, int blk, int accumulate) {
    using A = typename Acc<T>::A;
    constexpr int NW = Tile<T>::Z;
    __shared__ A red[NW][NPAR];
    A a[NPAR];
#pragma unroll
    for (int k = 0; k < NPAR; ++k) a[k] = Acc<T>::from(v[k]);
    int q;
    const A t1 = warp_sum8<Acc<T>>(a, q);
    if ((threadIdx.x & 3) == 0) red[threadIdx.y][q] = t1;
    __syncthreads();
    const int t = threadIdx.y * 32 + threadIdx.x;
    if (t < NPAR) {
        A s = red[0][t];
        for (int i = 1; i < NW; ++i) s = Acc<T>::add(s, red[i][t]);
        A* p = part + (long long)blk * NPAR + t;
        *p = accumulate ? Acc<T>::add(*p, s) : s;
    }
}

// grad[k] += sum over the nb blocks of part[b][k]: one block, FP64, fixed order (each thread's
// blocks in order, the warp, the warps in order).
template <typename T>
__global__ void __launch_bounds__(AT) k_adj_sum(const typename Acc<T>::A* __restrict__ part, long long nb,
                                                double* __restrict__ grad) {
    __shared__ double red[AT / 32][NPAR];
    pdl_enter();
    double t[NPAR];
#pragma unroll
    for (int k = 0; k < NPAR; ++k) t[k] = 0.0;
    for (long long b = threadIdx.x; b < nb; b += AT)
#pragma unroll
        for (int k = 0; k < NPAR; ++k) t[k] += Acc<T>::wide(part[b * NPAR + k]);
    int q;
    const double w1 = warp_sum8<Acc<double>>(t, q);
    if ((threadIdx.x & 3) == 0) red[threadIdx.x >> 5][q] = w1;
    __syncthreads();
    if (threadIdx.x < NPAR) {
        double a = 0.0;
        for (int w = 0; w < AT / 32; ++w) a += red[w][threadIdx.x];
        grad[threadIdx.x] += a;
    }
}

// Intermediate fields of one adjoint step, [ns][n] each.
template <typename T>
struct AdjBuf {
    T *rho, *jx, *jz, *psi;  // the state's moments and pseudopotential
    T *qx, *qz;              // psi_s dJ/dF_s: what the force at x owes to psi_s(x + c)
    T *rx, *rz;              // rho_s dJ/dF_s: what it owes to rho_s'(x + c)
    T *dloc, *djx, *djz;     // the site's own dJ/drho_s (psi' folded in), dJ/dj_s
    T* dps;                  // psi'(rho_s)
};

// 1 / v of a density
__device__ __forceinline__ float inverse(float v) { return 1.f / v; }
__device__ __forceinline__ double inverse(double v) { return rcp_fx(v); }

// rho, j and psi of the state f at site i, species s.
template <typename T>
__device__ __forceinline__ void moments_of(const T* __restrict__ f, const AdjC<T>& A, const AdjBuf<T>& B, int s,
                                           long long n, int i) {
    T v[9];
#pragma unroll
    for (int l = 0; l < 9; ++l) v[l] = f[(s * 9 + l) * n + i];
    T r = 0, mx = 0, mz = 0;
    if constexpr (sizeof(T) == 8) {
        r = sum9(v);
        momentum9(v, mx, mz);
    } else {
#pragma unroll
        for (int l = 0; l < 9; ++l) {
            r += v[l];
            mx += v[l] * (T)cx(l);
            mz += v[l] * (T)cz(l);
        }
    }
    B.rho[s * n + i] = r;
    B.jx[s * n + i] = mx;
    B.jz[s * n + i] = mz;
    B.psi[s * n + i] = psi_t(A, s, r);
}

// One thread per site and species (blockIdx.z = species).
template <typename T>
__global__ void __launch_bounds__(Tile<T>::NT) k_adj_moments(const T* __restrict__ f, const AdjC<T> A, AdjBuf<T> B) {
    pdl_enter();
    const int x = blockIdx.x * 32 + threadIdx.x, z = blockIdx.y * Tile<T>::Z + threadIdx.y;
    if (x < A.nx && z < A.nz) moments_of(f, A, B, blockIdx.z, (long long)A.nx * A.nz, z * A.nx + x);
}

// The shell sums of the differences v(x + c) - v(x - c) of antipodal links, weighted by c along x (sx)
// and z (sz): shells 1, 2, 4, 5, 8 (4 and 8 without the factor 2 of c).  w(dx, dz): the window.
template <typename V, typename W>
__device__ __forceinline__ void shell_sums(const W& w, V (&sx)[5], V (&sz)[5]) {
    const V d11 = w(1, 1) - w(-1, -1), e11 = w(-1, 1) - w(1, -1);
    const V d21 = w(2, 1) - w(-2, -1), e21 = w(-2, 1) - w(2, -1);
    const V d12 = w(1, 2) - w(-1, -2), e12 = w(-1, 2) - w(1, -2);
    const V d22 = w(2, 2) - w(-2, -2), e22 = w(-2, 2) - w(2, -2);
    sx[0] = w(1, 0) - w(-1, 0);
    sz[0] = w(0, 1) - w(0, -1);
    sx[1] = d11 - e11;
    sz[1] = d11 + e11;
    sx[2] = w(2, 0) - w(-2, 0);
    sz[2] = w(0, 2) - w(0, -2);
    sx[3] = V(2) * (d21 - e21) + (d12 - e12);
    sz[3] = V(2) * (d12 + e12) + (d21 + e21);
    sx[4] = d22 - e22;
    sz[4] = d22 + e22;
}
// The same contracted: sum over the antipodal pairs of c . (v(x + c) - v(x - c)) per shell, v = (p, q).
template <typename T, typename W1, typename W2>
__device__ __forceinline__ void shell_div(const W1& p, const W2& q, T (&t)[5]) {
    t[0] = (p(1, 0) - p(-1, 0)) + (q(0, 1) - q(0, -1));
    t[1] = ((p(1, 1) - p(-1, -1)) - (p(-1, 1) - p(1, -1))) + ((q(1, 1) - q(-1, -1)) + (q(-1, 1) - q(1, -1)));
    t[2] = (p(2, 0) - p(-2, 0)) + (q(0, 2) - q(0, -2));
    t[3] = (T(2) * ((p(2, 1) - p(-2, -1)) - (p(-2, 1) - p(2, -1))) + ((p(1, 2) - p(-1, -2)) - (p(-1, 2) - p(1, -2)))) +
           (T(2) * ((q(1, 2) - q(-1, -2)) + (q(-1, 2) - q(1, -2))) + ((q(2, 1) - q(-2, -1)) + (q(-2, 1) - q(2, -1))));
    t[4] = ((p(2, 2) - p(-2, -2)) - (p(-2, 2) - p(2, -2))) + ((q(2, 2) - q(-2, -2)) + (q(-2, 2) - q(2, -2)));
}

template <typename T, int NS>
__global__ void __launch_bounds__(Tile<T>::NT) k_adj_local(const T* __restrict__ f, const T* __restrict__ lam_next,
                                                           const AdjC<T> A, AdjBuf<T> B,
                                                           typename Acc<T>::A* __restrict__ part, int accumulate) {
    using TL = Tile<T>;
    __shared__ T ps[NS][TL::H][TL::W];
    __shared__ T rh[NS == 2 ? 2 : 1][TL::H][TL::W];
    pdl_enter();
    const long long n = (long long)A.nx * A.nz;
    const int x0 = blockIdx.x * 32, z0 = blockIdx.y * TL::Z;
    const int tx = threadIdx.x, tz = threadIdx.y, x = x0 + tx, z = z0 + tz;
    const bool live = x < A.nx && z < A.nz;
    const int i = z * A.nx + x;
    // the site's lam (streaming transposed: g_l(x) became f_l(x + c_l)), under way while the tile loads
    T m[NS][9], fl[NS][9], jx[NS], jz[NS];
    if (live) {
        const int xo[3] = {x == 0 ? A.nx - 1 : x - 1, x, x == A.nx - 1 ? 0 : x + 1};
        const int zo[3] = {(z == 0 ? A.nz - 1 : z - 1) * A.nx, z * A.nx, (z == A.nz - 1 ? 0 : z + 1) * A.nx};
#pragma unroll
        for (int s = 0; s < NS; ++s) {
#pragma unroll
            for (int l = 0; l < 9; ++l) m[s][l] = lam_next[(s * 9 + l) * n + (zo[cz(l) + 1] + xo[cx(l) + 1])];
#pragma unroll
            for (int l = 0; l < 9; ++l) fl[s][l] = f[(s * 9 + l) * n + i];
            jx[s] = B.jx[s * n + i];
            jz[s] = B.jz[s * n + i];
        }
    }
    bool small = false;  // a psi that the fixed-point sums would not hold exactly
    bool bits = false;   // whether to try them at all (uniform)
    if constexpr (sizeof(T) == 8) bits = A.fixed;
    for (int k = tz * 32 + tx; k < TL::H * TL::W; k += TL::NT) {
        const int r = k / TL::W, c = k - r * TL::W;
        const int j = wrap_t(z0 - 2 + r, A.nz) * A.nx + wrap_t(x0 - 2 + c, A.nx);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            T p = B.psi[s * n + j];
            if constexpr (sizeof(T) == 8) {
                if (bits) {
                    small = small || !(p >= PSI_SMALL);
                    p = of_bits((u64)psi_bits57(p));
                }
            }
            ps[s][r][c] = p;
            if (NS == 2) rh[s][r][c] = B.rho[s * n + j];
        }
    }
    bool fixed = false;  // the tile holds psi's bits on the 2^57 scale (uniform)
    if constexpr (sizeof(T) == 8) {
        fixed = !__syncthreads_or(small) && bits;
        if (bits && !fixed) {  // the numbers themselves
            for (int k = tz * 32 + tx; k < TL::H * TL::W; k += TL::NT) {
                const int r = k / TL::W, c = k - r * TL::W;
                const int j = wrap_t(z0 - 2 + r, A.nz) * A.nx + wrap_t(x0 - 2 + c, A.nx);
#pragma unroll
                for (int s = 0; s < NS; ++s) ps[s][r][c] = B.psi[s * n + j];
            }
            __syncthreads();
        }
    } else {
        __syncthreads();
    }
    T gp[NPAR] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (live) {
        // the force at the site, keeping its three sums (attraction a, repulsion p, cross b)
        T ax[NS], az[NS], px[NS], pz[NS], bx[NS], bz[NS];
        T rho[NS], psi[NS], Fx[NS], Fz[NS];
        T numx = 0, numz = 0, den = 0;
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const auto w = [&](int dx, int dz) { return ps[s][tz + 2 + dz][tx + 2 + dx]; };
            psi[s] = ps[s][tz + 2][tx + 2];
            if (NS == 2)
                rho[s] = rh[NS == 2 ? s : 0][tz + 2][tx + 2];
            else
                rho[s] = B.rho[s * n + i];
            ax[s] = az[s] = px[s] = pz[s] = bx[s] = bz[s] = 0;
            if constexpr (sizeof(T) == 8) {
                if (fixed) {
                    psi[s] = scaled_double((i64)bits_of(psi[s]), -57);
                    i64 sx[5], sz[5];
                    shell_sums([&](int dx, int dz) { return (i64)bits_of(w(dx, dz)); }, sx, sz);
                    DotFx dax, daz, dpx, dpz;
#pragma unroll
                    for (int q = 0; q < 5; ++q) {
                        if (q < 3) {  // the attraction's shells
                            dax.add(A.fa, q, sx[q]);
                            daz.add(A.fa, q, sz[q]);
                        }
                        dpx.add(A.fr, q, sx[q]);
                        dpz.add(A.fr, q, sz[q]);
                    }
                    ax[s] = scaled_double(dax.sum(), A.fa.e - 59);
                    az[s] = scaled_double(daz.sum(), A.fa.e - 59);
                    px[s] = scaled_double(dpx.sum(), A.fr.e - 59);
                    pz[s] = scaled_double(dpz.sum(), A.fr.e - 59);
                } else {
                    T sx[5], sz[5];
                    shell_sums(w, sx, sz);
                    ax[s] = (A.sa[0] * sx[0] + A.sa[1] * sx[1]) + A.sa[2] * sx[2];
                    az[s] = (A.sa[0] * sz[0] + A.sa[1] * sz[1]) + A.sa[2] * sz[2];
                    px[s] = ((A.sr[0] * sx[0] + A.sr[1] * sx[1]) + (A.sr[2] * sx[2] + A.sr[3] * sx[3])) + A.sr[4] * sx[4];
                    pz[s] = ((A.sr[0] * sz[0] + A.sr[1] * sz[1]) + (A.sr[2] * sz[2] + A.sr[3] * sz[3])) + A.sr[4] * sz[4];
                }
                Fx[s] = -psi[s] * (A.G1[s] * ax[s] + A.G2[s] * px[s]);
                Fz[s] = -psi[s] * (A.G1[s] * az[s] + A.G2[s] * pz[s]);
                if constexpr (NS == 2) {
                    const auto r = [&](int dx, int dz) { return rh[1 - s][tz + 2 + dz][tx + 2 + dx]; };
                    const T d11 = r(1, 1) - r(-1, -1), e11 = r(-1, 1) - r(1, -1);
                    bx[s] = A.wc[1] * (r(1, 0) - r(-1, 0)) + A.wc[2] * (d11 - e11);
                    bz[s] = A.wc[1] * (r(0, 1) - r(0, -1)) + A.wc[2] * (d11 + e11);
                    Fx[s] -= A.G_AB * rho[s] * bx[s];
                    Fz[s] -= A.G_AB * rho[s] * bz[s];
                }
                Fx[s] += rho[s] * A.g;
            } else {
                // FP32: link by link, in the links' order
#pragma unroll
                for (int k = 0; k < 24; ++k) {
                    const int q = LKX(k) * LKX(k) + LKZ(k) * LKZ(k);
                    const T ex = (T)LKX(k), ez = (T)LKZ(k);
                    const T p = w(LKX(k), LKZ(k));
                    ax[s] += A.wa[q] * p * ex;
                    az[s] += A.wa[q] * p * ez;
                    px[s] += A.wr[q] * p * ex;
                    pz[s] += A.wr[q] * p * ez;
                    if (NS == 2 && k < 8) {
                        const T ro = rh[NS == 2 ? 1 - s : 0][tz + 2 + LKZ(k)][tx + 2 + LKX(k)];
                        bx[s] += A.wc[q] * ro * ex;
                        bz[s] += A.wc[q] * ro * ez;
                    }
                }
                Fx[s] = -A.G1[s] * psi[s] * ax[s] - A.G2[s] * psi[s] * px[s] - A.G_AB * rho[s] * bx[s] + rho[s] * A.g;
                Fz[s] = -A.G1[s] * psi[s] * az[s] - A.G2[s] * psi[s] * pz[s] - A.G_AB * rho[s] * bz[s];
            }
            numx += jx[s] * A.itau[s];
            numz += jz[s] * A.itau[s];
            den += rho[s] * A.itau[s];
        }
        const T iden = inverse(den);
        const T upx = numx * iden, upz = numz * iden;
        T dupx = 0, dupz = 0, dr[NS], dFx[NS], dFz[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            if constexpr (sizeof(T) == 8) {
                const T r = rho[s], tau = A.tau[s], it = A.itau[s], ir = inverse(r), tir = tau * ir;
                const T ux = upx + Fx[s] * tir, uz = upz + Fz[s] * tir;
                // moments of lam_l - lam_0 with the rest weights: the part of lam common to all l, often the
                // largest, meets sum_l (f_l - feq_l) = 0 and would only multiply rounding; it adds lam_0 to
                // the zeroth moment and cancels in the velocity's derivative
                const T m0 = m[s][0];
                T q[9];
#pragma unroll
                for (int l = 1; l < 9; ++l) q[l] = m[s][l] - m0;
                // (36 times the moments: the weights 16, 4, 1 are exact)
                const T s13 = q[1] + q[3], s24 = q[2] + q[4], p57 = q[5] + q[7], p68 = q[6] + q[8], D = p57 + p68;
                const T d57 = q[5] - q[7], d86 = q[8] - q[6];
                const T a1x = T(4) * (q[1] - q[3]) + (d57 + d86), a1z = T(4) * (q[2] - q[4]) + (d57 - d86);
                const T axx = T(4) * s13 + D, azz = T(4) * s24 + D, axz = p57 - p68, a0 = T(4) * (s13 + s24) + D;
                const T hx = ux * axx + uz * axz, hz = ux * axz + uz * azz;  // second moments . u
                const T usq = ux * ux + uz * uz;
                // sum_l (lam_l - lam_0) feq_l / rho
                const T e1 = T(1.0 / 36.0) * ((a0 * (T(1) - T(1.5) * usq) + T(3) * (ux * a1x + uz * a1z)) + T(4.5) * (ux * hx + uz * hz));
                const T itr = it * r;
                const T aux = T(1.0 / 12.0) * (itr * ((a1x - ux * a0) + T(3) * hx)), auz = T(1.0 / 12.0) * (itr * ((a1z - uz * a0) + T(3) * hz));
                const T w1 = T(1.0 / 9.0), w2 = T(1.0 / 36.0);
                // d/dtau of g = f - (f - feq) / tau is (f - feq) / tau^2
                const T base = r * (T(1) - T(1.5) * usq);
                const T ea = w1 * base, ed = w2 * base;
                const T ca = T(0.5) * r, cd = T(0.125) * r, da = T(1.0 / 3.0) * r, dd = T(1.0 / 12.0) * r;
                const T cu[4] = {ux, uz, ux + uz, uz - ux};  // pairs (1,3), (2,4), (5,7), (6,8)
                T gt = 0;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const T e = k < 2 ? ea : ed, c = (k < 2 ? ca : cd) * cu[k], d = k < 2 ? da : dd;
                    const int lp = k < 2 ? k + 1 : k + 3;
                    gt += q[lp] * ((fl[s][lp] - e) - (c + d) * cu[k]);
                    gt += q[opp(lp)] * ((fl[s][opp(lp)] - e) - (c - d) * cu[k]);
                }
                // u_s = u' + tau F_s / rho_s
                dupx += aux;
                dupz += auz;
                dFx[s] = aux * tir;
                dFz[s] = auz * tir;
                const T fu = (aux * Fx[s] + auz * Fz[s]) * ir;
                dr[s] = it * (e1 + m0) - fu * tir;
                gp[5 + s] = gt * it * it + fu;
            } else {
                const T r = rho[s], tau = A.tau[s], it = A.itau[s], ir = inverse(r);
                const T ux = upx + tau * Fx[s] * ir, uz = upz + tau * Fz[s] * ir;
                const T usq = ux * ux + uz * uz;
                // d/dtau of g = f - (f - feq) / tau is (f - feq) / tau^2.  sum_l (f_l - feq_l) = 0
                // (the equilibrium keeps rho), so sum_l m_l (f_l - feq_l) = sum_l (m_l - m_0)(f_l - feq_l):
                // the part of lam common to all l, often the largest, would only multiply rounding
                T ar = 0, aux = 0, auz = 0, gt = 0;
                const T m0 = m[s][0];
#pragma unroll
                for (int l = 0; l < 9; ++l) {
                    const T ml = m[s][l];
                    const T ex = (T)cx(l), ez = (T)cz(l);
                    const T cu = ex * ux + ez * uz;
                    const T wr = wlb<T>(l) * r;
                    const T fe = wr * ((T)1 + (T)3 * cu + (T)4.5 * cu * cu - (T)1.5 * usq);
                    const T dfe = ml * it;  // g = f - (f - feq) / tau
                    gt += (ml - m0) * (fl[s][l] - fe);
                    ar += dfe * fe;
                    aux += dfe * wr * ((T)3 * ex + (T)9 * cu * ex - (T)3 * ux);
                    auz += dfe * wr * ((T)3 * ez + (T)9 * cu * ez - (T)3 * uz);
                }
                // u_s = u' + tau F_s / rho_s
                dupx += aux;
                dupz += auz;
                dFx[s] = aux * tau * ir;
                dFz[s] = auz * tau * ir;
                const T fu = (aux * Fx[s] + auz * Fz[s]) * ir;
                dr[s] = ar * ir - fu * tau * ir;
                gp[5 + s] += gt * it * it + fu;
            }
        }
        // u' = sum_k j_k / tau_k / sum_k rho_k / tau_k
        const T dnx = dupx * iden, dnz = dupz * iden, dden = -(dupx * upx + dupz * upz) * iden;
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const T it = A.itau[s];
            gp[5 + s] -= (jx[s] * dnx + jz[s] * dnz + rho[s] * dden) * it * it;
            dr[s] += dden * it;
            // the site's own terms of the force: F_s depends on psi_s(x), rho_s(x) and g
            const T ba = dFx[s] * ax[s] + dFz[s] * az[s], bp = dFx[s] * px[s] + dFz[s] * pz[s];
            const T bb = dFx[s] * bx[s] + dFz[s] * bz[s];
            const T dps = dpsi_t(A, s, rho[s]);
            gp[0 + s] -= psi[s] * ba;
            gp[2 + s] -= psi[s] * bp;
            if (NS == 2) gp[4] -= rho[s] * bb;
            gp[7] += rho[s] * dFx[s];
            B.dloc[s * n + i] = dr[s] - A.G_AB * bb + dFx[s] * A.g - dps * (A.G1[s] * ba + A.G2[s] * bp);
            B.djx[s * n + i] = dnx * it;
            B.djz[s * n + i] = dnz * it;
            B.dps[s * n + i] = dps;
            B.qx[s * n + i] = psi[s] * dFx[s];
            B.qz[s * n + i] = psi[s] * dFz[s];
            if (NS == 2) {
                B.rx[s * n + i] = rho[s] * dFx[s];
                B.rz[s * n + i] = rho[s] * dFz[s];
            }
        }
    }
    block_sum<T>(gp, part, blockIdx.y * gridDim.x + blockIdx.x, accumulate);
}

// One thread per site and species (blockIdx.z = species).  f_prev (may be null): the state of the
// step before, whose moments this kernel also forms for the next adjoint step (it reads none of
// the moment fields itself, so it may overwrite them).
template <typename T, int NS>
__global__ void __launch_bounds__(Tile<T>::NT) k_adj_final(const T* __restrict__ lam_next, const AdjC<T> A, AdjBuf<T> B,
                                                           T* __restrict__ lam, const T* __restrict__ f_prev) {
    using TL = Tile<T>;
    __shared__ T qs[2][TL::H][TL::W];
    __shared__ T rs[NS == 2 ? 2 : 1][TL::H][TL::W];
    pdl_enter();
    const long long n = (long long)A.nx * A.nz;
    const int s = blockIdx.z;
    const int x0 = blockIdx.x * 32, z0 = blockIdx.y * TL::Z;
    const int tx = threadIdx.x, tz = threadIdx.y, x = x0 + tx, z = z0 + tz;
    const bool live = x < A.nx && z < A.nz;
    const int i = z * A.nx + x;
    T m[9];
    T dloc = 0, dpsi = 0, djx = 0, djz = 0;
    if (live) {
        const int xo[3] = {x == 0 ? A.nx - 1 : x - 1, x, x == A.nx - 1 ? 0 : x + 1};
        const int zo[3] = {(z == 0 ? A.nz - 1 : z - 1) * A.nx, z * A.nx, (z == A.nz - 1 ? 0 : z + 1) * A.nx};
#pragma unroll
        for (int l = 0; l < 9; ++l) m[l] = lam_next[(s * 9 + l) * n + (zo[cz(l) + 1] + xo[cx(l) + 1])];
        dloc = B.dloc[s * n + i];
        dpsi = B.dps[s * n + i];
        djx = B.djx[s * n + i];
        djz = B.djz[s * n + i];
    }
    for (int k = tz * 32 + tx; k < TL::H * TL::W; k += TL::NT) {
        const int r = k / TL::W, c = k - r * TL::W;
        const int j = wrap_t(z0 - 2 + r, A.nz) * A.nx + wrap_t(x0 - 2 + c, A.nx);
        qs[0][r][c] = B.qx[s * n + j];
        qs[1][r][c] = B.qz[s * n + j];
        if constexpr (NS == 2) {
            rs[0][r][c] = B.rx[(1 - s) * n + j];
            rs[1][r][c] = B.rz[(1 - s) * n + j];
        }
    }
    __syncthreads();
    if (!live) return;
    // this site as the neighbour x + c of the sites x - c: their forces' dependence on its psi_s and,
    // through the cross term of the other species, on its rho_s: -sum_c K c . q(x - c), the
    // antipodal links together
    const T keep = (T)1 - A.itau[s];
    if constexpr (sizeof(T) == 8) {
        T t[5];
        shell_div([&](int dx, int dz) { return qs[0][tz + 2 + dz][tx + 2 + dx]; },
                  [&](int dx, int dz) { return qs[1][tz + 2 + dz][tx + 2 + dx]; }, t);
        const T* K = A.K[s];
        const T dps = ((K[0] * t[0] + K[1] * t[1]) + (K[2] * t[2] + K[3] * t[3])) + K[4] * t[4];
        T d = dloc + dpsi * dps;
        if constexpr (NS == 2) {
            const auto p = [&](int dx, int dz) { return rs[0][tz + 2 + dz][tx + 2 + dx]; };
            const auto q = [&](int dx, int dz) { return rs[1][tz + 2 + dz][tx + 2 + dx]; };
            const T t1 = (p(1, 0) - p(-1, 0)) + (q(0, 1) - q(0, -1));
            const T t2 = ((p(1, 1) - p(-1, -1)) - (p(-1, 1) - p(1, -1))) + ((q(1, 1) - q(-1, -1)) + (q(-1, 1) - q(1, -1)));
            d += A.G_AB * (A.wc[1] * t1 + A.wc[2] * t2);
        }
        const T jp = djx + djz, jm = djz - djx;
        const T add[9] = {d, d + djx, d + djz, d - djx, d - djz, d + jp, d + jm, d - jp, d - jm};
#pragma unroll
        for (int l = 0; l < 9; ++l) lam[(s * 9 + l) * n + i] = keep * m[l] + add[l];
    } else {  // link by link, in the links' order
        T dps = 0, dro = 0;
#pragma unroll
        for (int k = 0; k < 24; ++k) {
            const int q = LKX(k) * LKX(k) + LKZ(k) * LKZ(k);
            const T ex = (T)LKX(k), ez = (T)LKZ(k);
            const T qx = qs[0][tz + 2 - LKZ(k)][tx + 2 - LKX(k)], qz = qs[1][tz + 2 - LKZ(k)][tx + 2 - LKX(k)];
            dps -= (A.G1[s] * A.wa[q] + A.G2[s] * A.wr[q]) * (qx * ex + qz * ez);
            if constexpr (NS == 2) {
                if (k < 8) {
                    const T rx = rs[0][tz + 2 - LKZ(k)][tx + 2 - LKX(k)], rz = rs[1][tz + 2 - LKZ(k)][tx + 2 - LKX(k)];
                    dro -= A.G_AB * A.wc[q] * (rx * ex + rz * ez);
                }
            }
        }
        const T d = dloc + dro + dpsi * dps;
#pragma unroll
        for (int l = 0; l < 9; ++l) lam[(s * 9 + l) * n + i] = keep * m[l] + d + djx * (T)cx(l) + djz * (T)cz(l);
    }
    if (f_prev) moments_of(f_prev, A, B, s, n, i);
}

// Calibration objective: J = sum_z (ubar(z) - tu(z))^2 + (rhobar_A(z) - tr(z))^2, ubar the
// x-average of u = sum_s j_x,s / sum_s rho_s, rhobar_A the x-average of rho_A.  One block per
// row forms the averages (in T, widened to FP64); k_obj_total sums the rows' shares in a fixed
// order.
template <typename T>
__global__ void __launch_bounds__(AT) k_obj_rows(const T* __restrict__ f, const AdjC<T> A, double* __restrict__ ubar,
                                                 double* __restrict__ rbar) {
    const long long n = (long long)A.nx * A.nz;
    const int z = blockIdx.x;
    T su = 0, sr = 0;
    for (int x = threadIdx.x; x < A.nx; x += AT) {
        const long long i = (long long)z * A.nx + x;
        T rt = 0, mx = 0, ra = 0;
        for (int s = 0; s < A.ns; ++s)
            for (int l = 0; l < 9; ++l) {
                const T v = f[(s * 9 + l) * n + i];
                rt += v;
                mx += v * (T)cx(l);
                if (s == 0) ra += v;
            }
        su += mx / rt;
        sr += ra;
    }
    __shared__ T red[2][AT / 32];
    for (int o = 16; o > 0; o >>= 1) {
        su += __shfl_xor_sync(0xffffffffu, su, o);
        sr += __shfl_xor_sync(0xffffffffu, sr, o);
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = su;
        red[1][threadIdx.x >> 5] = sr;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0;
        for (int w = 0; w < AT / 32; ++w) {
            a += (double)red[0][w];
            b += (double)red[1][w];
        }
        ubar[z] = a / A.nx;
        rbar[z] = b / A.nx;
    }
}

__global__ void __launch_bounds__(AT) k_obj_total(int nz, const double* __restrict__ tu, const double* __restrict__ tr,
                                                  const double* __restrict__ ubar, const double* __restrict__ rbar,
                                                  double* __restrict__ J) {
    __shared__ double red[AT / 32];
    double t = 0.0;
    for (int z = threadIdx.x; z < nz; z += AT)
        t += (ubar[z] - tu[z]) * (ubar[z] - tu[z]) + (rbar[z] - tr[z]) * (rbar[z] - tr[z]);
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0;
        for (int w = 0; w < AT / 32; ++w) a += red[w];
        *J = a;
    }
}

// dJ/df of row z: 2 (ubar - tu) / nx (c_lx - u) / rho_tot + [s = A] 2 (rhobar_A - tr) / nx; the
// row's two coefficients are formed in FP64 and rounded to T once.
template <typename T>
__global__ void __launch_bounds__(AT) k_obj_grad(const T* __restrict__ f, const AdjC<T> A, const double* __restrict__ tu,
                                                 const double* __restrict__ tr, const double* __restrict__ ubar,
                                                 const double* __restrict__ rbar, T* __restrict__ g) {
    const long long n = (long long)A.nx * A.nz;
    const int z = blockIdx.x;
    const T cu = (T)(2.0 * (ubar[z] - tu[z]) / A.nx), cr = (T)(2.0 * (rbar[z] - tr[z]) / A.nx);
    for (int x = threadIdx.x; x < A.nx; x += AT) {
        const long long i = (long long)z * A.nx + x;
        T rt = 0, mx = 0;
        for (int s = 0; s < A.ns; ++s)
            for (int l = 0; l < 9; ++l) {
                const T v = f[(s * 9 + l) * n + i];
                rt += v;
                mx += v * (T)cx(l);
            }
        const T u = mx / rt, gu = cu / rt;
        for (int s = 0; s < A.ns; ++s)
            for (int l = 0; l < 9; ++l) g[(s * 9 + l) * n + i] = gu * ((T)cx(l) - u) + (s == 0 ? cr : (T)0);
    }
}

// The initial populations are W_l rho (equilibrium at rest): dJ/drho_s = sum_l W_l lam_0.
template <typename T>
__global__ void k_adj_initial(const T* __restrict__ lam0, const AdjC<T> A, double* __restrict__ g) {
    const long long n = (long long)A.nx * A.nz;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        for (int s = 0; s < A.ns; ++s) {
            T t = 0;
            for (int l = 0; l < 9; ++l) t += wlb<T>(l) * lam0[(s * 9 + l) * n + i];
            g[s * n + i] = (double)t;
        }
}

int grid_of(long long n) { return (int)((n + AT - 1) / AT); }

template <typename T>
AdjC<T> adj_const(const AdjConst& D) {
    AdjC<T> A;
    A.nx = D.nx;
    A.nz = D.nz;
    A.ns = D.ns;
    A.psi_form = D.psi_form;
    for (int q = 0; q < 9; ++q) {
        A.wa[q] = (T)D.wa[q];
        A.wr[q] = (T)D.wr[q];
        A.wc[q] = (T)D.wc[q];
    }
    if constexpr (sizeof(T) == 8) {
        const int at[5] = {1, 2, 4, 5, 8};
        for (int k = 0; k < 5; ++k) {
            const double c = at[k] == 4 || at[k] == 8 ? 2.0 : 1.0;  // the links' components
            A.sa[k] = c * D.wa[at[k]];
            A.sr[k] = c * D.wr[at[k]];
            for (int s = 0; s < 2; ++s) A.K[s][k] = D.G1[s] * A.sa[k] + D.G2[s] * A.sr[k];
        }
        const bool kept = coef_fx(A.fa, A.sa), rep = coef_fx(A.fr, A.sr);
        A.fixed = D.psi_form == 0 && kept && rep;
        for (int s = 0; s < 2; ++s) A.ex[s] = exp_fx_const(D.psi_form == 0 ? D.rho0[s] : 1.0);
    }
    for (int s = 0; s < 2; ++s) {
        A.G1[s] = (T)D.G1[s];
        A.G2[s] = (T)D.G2[s];
        A.tau[s] = (T)D.tau[s];
        A.itau[s] = (T)(1.0 / D.tau[s]);
        A.irho0[s] = (T)(1.0 / D.rho0[s]);
    }
    A.G_AB = (T)D.G_AB;
    A.g = (T)D.g;
    return A;
}

// Scratch of a context: the intermediate fields (12 ns n values, sized for FP64), then the block
// partials (NPAR 8-byte accumulators per block), then the objective's row averages (2 nz doubles).
size_t field_bytes(long long n, int ns) { return ((size_t)12 * ns * n * 8 + 255) & ~(size_t)255; }
template <typename T>
dim3 step_grid(int nx, int nz) {
    return dim3((nx + 31) / 32, (nz + Tile<T>::Z - 1) / Tile<T>::Z);
}
size_t part_bytes(int nx, int nz) {  // the FP64 tiles are the smaller ones
    const dim3 g = step_grid<double>(nx, nz);
    return ((size_t)NPAR * g.x * g.y * 8 + 255) & ~(size_t)255;
}

// pdl: the launch may start while the one before drains.  In FP32, whose launches are bound by
// latency; not in FP64, where CTAs placed early crowd the SMs that free first and the FP64 pipe of
// the fullest one bounds the launch (60 gradient steps of 150 x 90: 6.4 ms with, 4.5 without).
template <typename... K, typename... A>
void launch_pdl(bool pdl, void (*kernel)(K...), dim3 grid, dim3 block, cudaStream_t st, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<A&&>(args)...);  // the caller reads cudaGetLastError
}

template <typename T>
AdjBuf<T> adj_buf(void* scratch, long long n, int ns) {
    T* p = static_cast<T*>(scratch);
    const long long m = (long long)ns * n;
    AdjBuf<T> B;
    T** fields[] = {&B.rho, &B.jx, &B.jz, &B.psi, &B.qx, &B.qz, &B.rx, &B.rz, &B.dloc, &B.djx, &B.djz, &B.dps};
    for (int k = 0; k < 12; ++k) *fields[k] = p + k * m;
    return B;
}

template <typename T, int NS>
void enqueue_steps(const AdjC<T>& A, AdjBuf<T> B, typename Acc<T>::A* part, dim3 grid, int nsteps, const T* states,
                   long long stride, const T*& next, T* const bufs[2], cudaEvent_t* ev, cudaStream_t st) {
    const dim3 block(32, Tile<T>::Z), grid_s(grid.x, grid.y, NS);
    for (int k = nsteps - 1, t = 0; k >= 0; --k, ++t) {
        const T* f = states + (long long)k * stride;
        T* out = bufs[t & 1];
        cudaEvent_t* e = ev ? ev + 6 * t : nullptr;
        // the moments of f: its own kernel for the first step, else formed by the previous step's
        // final kernel
        if (e) cudaEventRecord(e[0], st);
        if (t == 0) launch_pdl(sizeof(T) == 4, k_adj_moments<T>, grid_s, block, st, f, A, B);
        if (e) cudaEventRecord(e[1], st), cudaEventRecord(e[2], st);
        launch_pdl(sizeof(T) == 4, k_adj_local<T, NS>, grid, block, st, f, next, A, B, part, t > 0 ? 1 : 0);
        if (e) cudaEventRecord(e[3], st), cudaEventRecord(e[4], st);
        const T* f_prev = k > 0 ? states + (long long)(k - 1) * stride : nullptr;
        launch_pdl(sizeof(T) == 4, k_adj_final<T, NS>, grid_s, block, st, next, A, B, out, f_prev);
        if (e) cudaEventRecord(e[5], st);
        next = out;
    }
}

}  // namespace

void fill_adj_const(AdjConst& A, const lbm_params& p, int nx, int nz, int ns, double body_force) {
    A.nx = nx;
    A.nz = nz;
    A.ns = ns;
    A.psi_form = p.psi_form;
    for (int q = 0; q < 9; ++q) {
        const double wa = p.weight_preset == LBM_WEIGHTS_CHEM09 ? w_belt1(q) : w_attr_paper(q);
        A.wa[q] = p.weight_norm * wa;
        A.wr[q] = p.weight_norm * w_rep(q);
        A.wc[q] = p.weight_norm * w_belt1(q);
    }
    for (int s = 0; s < 2; ++s) {
        const int ps = s < ns ? s : 0;
        A.G1[s] = p.G1[ps];
        A.G2[s] = p.G2[ps];
        A.tau[s] = p.tau[ps];
        A.rho0[s] = p.rho0[ps];
    }
    A.G_AB = ns == 2 ? p.G_AB : 0.0;
    A.g = body_force;
}

size_t adjoint_scratch_bytes(int nx, int nz, int ns) {
    const long long n = (long long)nx * nz;
    return field_bytes(n, ns) + part_bytes(nx, nz) + (size_t)2 * nz * sizeof(double);
}

template <typename T>
cudaError_t launch_adjoint_steps(const AdjConst& D, int nsteps, const T* states, long long stride, const T* lam_in,
                                 T* lam_a, T* lam_b, const T** lam_out, double* grad, void* scratch, cudaEvent_t* ev,
                                 cudaStream_t st) {
    const long long n = (long long)D.nx * D.nz;
    const AdjC<T> A = adj_const<T>(D);
    const AdjBuf<T> B = adj_buf<T>(scratch, n, D.ns);
    auto* part = reinterpret_cast<typename Acc<T>::A*>(static_cast<char*>(scratch) + field_bytes(n, D.ns));
    const dim3 grid = step_grid<T>(D.nx, D.nz);
    const T* next = lam_in;
    T* const bufs[2] = {lam_a, lam_b};
    if (D.ns == 2)
        enqueue_steps<T, 2>(A, B, part, grid, nsteps, states, stride, next, bufs, ev, st);
    else
        enqueue_steps<T, 1>(A, B, part, grid, nsteps, states, stride, next, bufs, ev, st);
    if (nsteps > 0) launch_pdl(sizeof(T) == 4, k_adj_sum<T>, dim3(1), dim3(AT), st, part, (long long)grid.x * grid.y, grad);
    *lam_out = next;
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_adjoint_objective(const AdjConst& D, const T* f, const double* tu, const double* tr, double* J,
                                     T* g, void* scratch, cudaStream_t st) {
    const long long n = (long long)D.nx * D.nz;
    const AdjC<T> A = adj_const<T>(D);
    double* ubar = reinterpret_cast<double*>(static_cast<char*>(scratch) + field_bytes(n, D.ns) + part_bytes(D.nx, D.nz));
    double* rbar = ubar + D.nz;
    k_obj_rows<T><<<D.nz, AT, 0, st>>>(f, A, ubar, rbar);
    k_obj_total<<<1, AT, 0, st>>>(D.nz, tu, tr, ubar, rbar, J);
    if (g) k_obj_grad<T><<<D.nz, AT, 0, st>>>(f, A, tu, tr, ubar, rbar, g);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_adjoint_initial(const AdjConst& D, const T* lam0, double* g, cudaStream_t st) {
    const long long n = (long long)D.nx * D.nz;
    const AdjC<T> A = adj_const<T>(D);
    k_adj_initial<T><<<grid_of(n) < 4096 ? grid_of(n) : 4096, AT, 0, st>>>(lam0, A, g);
    return cudaGetLastError();
}

#define LBM_ADJ_INST(T)                                                                                           \
    template cudaError_t launch_adjoint_steps<T>(const AdjConst&, int, const T*, long long, const T*, T*, T*,     \
                                                 const T**, double*, void*, cudaEvent_t*, cudaStream_t);         \
    template cudaError_t launch_adjoint_objective<T>(const AdjConst&, const T*, const double*, const double*,     \
                                                     double*, T*, void*, cudaStream_t);                          \
    template cudaError_t launch_adjoint_initial<T>(const AdjConst&, const T*, double*, cudaStream_t);
LBM_ADJ_INST(double)
LBM_ADJ_INST(float)

}  // namespace lbm
