// lbm3d.cu -- the three-dimensional extension of the two-belt Shan-Chen step (D3Q19; Eq. FORCE
// over the 3-D links of |c|^2 <= 8 with Appendix B's weights solved in three dimensions; the
// cross repulsion of Sec. IV over the first belt; the shifted-velocity BGK collision of
// Sec. II), behind the lbm3_* C ABI of include/lbm3d.h.
//
// A step is two kernels.
//  * k3_density reads each site's populations once and writes psi_s and rho_s into two
//    ghost-padded volumes (4 ghost columns in x, 2 ghost rows in y and z, holding the periodic
//    images, or beyond a wall the mirror images of the fluid), the two species of a site side
//    by side, so that a tile with its 2-cell halo is one in-bounds box.
//  * k3_step: a CTA of 32 x 4 x 2 sites loads the box of both volumes around its tile
//    (40 x 8 x 6 positions, x from x0 - 4 for 16-byte alignment) with one 4-D
//    cp.async.bulk.tensor on an mbarrier while every thread loads its own 19 populations per
//    species from HBM; then the force (46 antipodal link pairs, gathered shell by shell, both
//    species at once), the cross force, the collision, and the push of the new populations to
//    x + c_l (periodic in x and y, periodic or halfway bounce-back with Ladd's term in z).
// HBM traffic per site-update (FP32, two species): 152 B of populations read twice and written
// once plus the 16 B of the volumes written and read, 488 B; the method's own is 304 B
// (each population read and written once).  Populations are SoA f[s][l][z][y][x] (rows padded
// to 32), FP32 deviations f - W_l rho_ref,s or plain FP64.
//
// Full relaxation (two species in FP32, tau = 1 for both; lbm3_create says which lattices) needs no
// populations: the collision leaves f*_l = feq_l(rho_s, u_s), so the density and velocity after it (4
// numbers per species, held as 5) are the whole state, and a step only needs the density and
// momentum of what streams in.
//  * k3_stream evaluates, at every site, the 19 equilibria that stream in from the neighbours'
//    moments, and writes their density and momentum (and the psi / rho volumes);
//  * k3_step in its K3_RELAX form takes the force from the volumes and writes the new density and velocity.
// 144 B per site-update, and half the instructions.  Populations are formed where they are asked
// for (k3_expand).
#include <cuda.h>
#include <cudaTypedefs.h>
#include <stdarg.h>
#include <stdio.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "lbm3d.h"
#include "lbm_internal.h"

namespace lbm3 {

// ---- lattice -------------------------------------------------------------------------------

// D3Q19: rest, +-x, +-y, +-z, then the 12 edges; every velocity is followed by its opposite.
// Each velocity is coded as (cx + 1) + 3 (cy + 1) + 9 (cz + 1).
__host__ __device__ constexpr int code19(int l) {
    constexpr int k[19] = {13, 14, 12, 16, 10, 22, 4, 17, 9, 11, 15, 23, 3, 5, 21, 25, 1, 7, 19};
    return k[l];
}
__host__ __device__ constexpr int c3x(int l) { return code19(l) % 3 - 1; }
__host__ __device__ constexpr int c3y(int l) { return code19(l) / 3 % 3 - 1; }
__host__ __device__ constexpr int c3z(int l) { return code19(l) / 9 - 1; }
__host__ __device__ constexpr int opp19(int l) { return l == 0 ? 0 : (l % 2 ? l + 1 : l - 1); }
// The first velocity with a nonzero component along an axis (0: x, 1: y, 2: z).
__host__ __device__ constexpr int first19(int axis) {
    for (int l = 1; l < 19; ++l)
        if ((axis == 0 ? c3x(l) : (axis == 1 ? c3y(l) : c3z(l))) != 0) return l;
    return 0;
}
// Every odd velocity's first nonzero component is +1, so c_l . u can start from that component.
__host__ __device__ constexpr bool odd_velocities_lead_positive() {
    for (int l = 1; l < 19; l += 2)
        if ((c3x(l) ? c3x(l) : (c3y(l) ? c3y(l) : c3z(l))) != 1) return false;
    return true;
}
static_assert(odd_velocities_lead_positive(), "c_l . u of an odd velocity starts from a +1 component");
static_assert(c3x(first19(0)) == 1 && c3y(first19(1)) == 1 && c3z(first19(2)) == 1,
              "the momentum sums start from a +1 component");
template <typename T>
__host__ __device__ constexpr T w19(int l) {
    return l == 0 ? T(1) / T(3) : (l <= 6 ? T(1) / T(18) : T(1) / T(36));
}

// Interaction weights by shell |c|^2 (Appendix B's constraints solved in three dimensions).
inline double w_att3(int q) {
    switch (q) {
        case 1: return 2.0 / 15.0;
        case 2: return 1.0 / 15.0;
        case 3: return 1.0 / 60.0;
        case 4: return 1.0 / 120.0;
        default: return 0.0;
    }
}
inline double w_rep3(int q) {
    switch (q) {
        case 1: return 4.0 / 45.0;
        case 2: return 1.0 / 21.0;
        case 3: return 2.0 / 105.0;
        case 4: return 5.0 / 504.0;
        case 5: return 1.0 / 315.0;
        case 6: return 1.0 / 630.0;
        case 8: return 1.0 / 5040.0;
        default: return 0.0;
    }
}
inline double w_cross3(int q) { return q == 1 ? 1.0 / 6.0 : (q == 2 ? 1.0 / 12.0 : 0.0); }

// ---- pairs of the two species ----------------------------------------------------------------

// A site's two species side by side: float2 (FP32, packed instructions) or double2.
template <typename T> struct PairOf;
template <> struct PairOf<float> { using V = float2; };
template <> struct PairOf<double> { using V = double2; };

__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 vsplat(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 vswap(float2 a) { return make_float2(a.y, a.x); }
__device__ __forceinline__ double2 vadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 vsub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 vmul(double2 a, double2 b) { return make_double2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ double2 vfma(double2 a, double2 b, double2 c) {
    return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
__device__ __forceinline__ double2 vsplat(double a) { return make_double2(a, a); }
__device__ __forceinline__ double2 vswap(double2 a) { return make_double2(a.y, a.x); }

// Scalar operations whose rounding is fixed (the compiler neither contracts nor reorders them).
__device__ __forceinline__ float smul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double smul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float sadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double sadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float sfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double sfma(double a, double b, double c) { return __fma_rn(a, b, c); }

// v as FP64: of an FP32 value by its bits (the conversion instruction runs on the FP64 pipe).
__device__ __forceinline__ double wide3(float v) { return lbm::widen_fx(v); }
__device__ __forceinline__ double wide3(double v) { return v; }

// 1 / x of a density
__device__ __forceinline__ float rcp3(float x) { return 1.0f / x; }
__device__ __forceinline__ double rcp3(double x) { return lbm::rcp_fx(x); }

// ---- geometry and constants ----------------------------------------------------------------

constexpr int GX = 4, GY = 2, GZ = 2;         // ghosts of the psi / rho volumes
constexpr long long WAIT_LIMIT = 2000000000LL;  // clock cycles of the bounded wait (~1 s)
// The tile shapes (TY x TZ rows of TX sites, one thread per site) lbm3_autotune chooses from: the
// halo box of a tile is (TY + 4) x (TZ + 4) rows (x from x0 - 4: 16-byte aligned), so flatter tiles
// read more halo from L2 per site and taller ones hold fewer CTAs per SM.
//  * FP32: rows of 32 (a warp), 256 threads (shape 3: 512).
//  * FP64: rows of 16, two to a warp, 128 threads (shape 3: 256).  The pass is bound by the FP64
//    pipe, which a warp holds for 16 cycles an instruction however few of its sites are inside the
//    lattice, so a row's last tile should waste few: at nx = 65 rows of 16 keep 81 % of the lanes
//    at work, rows of 32 68 %; and the smaller CTAs leave a smaller last wave.
constexpr int NSHAPE = 4;
template <typename T>
struct Tile3 {
    static constexpr int TX = sizeof(T) == 4 ? 32 : 16;
    static constexpr int BX = TX + 2 * GX;  // box width
    static constexpr int ty(int shape) {
        constexpr int f[NSHAPE] = {4, 2, 8, 4}, d[NSHAPE] = {8, 4, 2, 8};
        return sizeof(T) == 4 ? f[shape] : d[shape];
    }
    static constexpr int tz(int shape) {
        constexpr int f[NSHAPE] = {2, 4, 1, 4}, d[NSHAPE] = {1, 2, 4, 2};
        return sizeof(T) == 4 ? f[shape] : d[shape];
    }
};

// FP64: the pseudopotential and Eq. FORCE's sums in fixed point (lbm_fixed.cuh).  psi is held on the
// 2^55 scale: a shell's sum reaches 16 (|c|^2 = 6), all seven 47.
constexpr int PSI3_BITS = 55;
template <typename T>
struct Fixed3 {};
template <>
struct Fixed3<double> {
    lbm::ExpFx ex[2];
    lbm::CoefFx<7> kf[2];  // K_s(1, 2, 3, 4, 5, 6, 8)
    int fixed;             // psi = 1 - exp(-rho / rho0): 1, or -1 with a coefficient beyond coef_fx's range; else 0
};

template <typename T>
struct Step3 : Fixed3<T> {
    int nx, ny, nz, ns, zbc, psi_form;
    int pitch;            // population row length (nx rounded up to 32)
    int gpitch;           // sites per row of a volume (nx + 2 GX rounded up to 4)
    long long plane;      // elements of one population volume (nz * ny * pitch)
    long long gvol;       // pairs in one psi / rho volume (gz * gy * gpitch)
    int gy, gz;           // rows and layers of a volume (ny + 2 GY, nz + 2 GZ)
    T omega[2], tau[2], rho_ref[2], inv_rho0[2], rho0[2];
    T g, wall_u[2];
    T kq[2][9];           // K_s(q) = weight_norm (G1_s w_att(q) + G2_s w_rep(q)) by shell q
    T kc[3];              // weight_norm G_AB w_cross(q), q = 1, 2 (zero for one species)
};

// psi as the volumes hold it: a value, or in FP64 with psi = 1 - exp(-rho / rho0) the bits of psi on the
// 2^PSI3_BITS scale.  A density <= 0 or NaN has no such bits (a run may pass through such states,
// reported but not stopped, and recover from them): its psi stands there as a number, whose bits
// are beyond the scale's 0 .. 2^PSI3_BITS, and psi3_number reads either.
__device__ __forceinline__ float psi3(const Step3<float>& C, int s, float rho) {
    return C.psi_form == 1 ? rho : 1.0f - __expf(-rho * C.inv_rho0[s]);
}
__device__ __forceinline__ double psi3(const Step3<double>& C, int s, double rho) {
    return C.psi_form == 1 ? rho : lbm::of_bits((lbm::u64)((lbm::psi_fx(rho, C.ex[s]) + 1) >> (56 - PSI3_BITS)));
}
__device__ __forceinline__ double psi3_number(double v) {
    const lbm::u64 b = lbm::bits_of(v);
    return b <= (lbm::u64)1 << PSI3_BITS ? lbm::scaled_double((lbm::i64)b, -PSI3_BITS) : v;
}
// Whether psi3 is to be the number: not > 0 and finite (its sign, or all of its exponent, set).
__device__ __forceinline__ bool psi3_beyond(double rho) {
    return (unsigned)(lbm::bits_of(rho) >> 32) - 1u >= 0x7fefffffu;
}

__device__ __forceinline__ int wrap3(int i, int n) {
    int r = i % n;
    return r < 0 ? r + n : r;
}
// reflection about the walls at -1/2 and n - 1/2 (the mirror reading of the ghost rows)
__device__ __forceinline__ int mirror3(int i, int n) {
    int m = i % (2 * n);
    if (m < 0) m += 2 * n;
    return m >= n ? 2 * n - 1 - m : m;
}

// The step's two kernels are launched with programmatic dependent launch: the next kernel's CTAs
// may be scheduled while this grid drains, and every thread waits for the previous grid in the
// stream (and the visibility of its writes) before its first global access.
__device__ __forceinline__ void pdl_enter() {
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
}

template <typename... K, typename... A>
cudaError_t launch_pdl(void (*kernel)(K...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<A&&>(args)...);
}

// ---- k3_density --------------------------------------------------------------------------

// The padded coordinates (own, then ghosts) that hold the value of coordinate v of an axis of
// n sites with g ghosts on each side: periodic images, or the mirror images with `mirror`.
__device__ __forceinline__ int ghost_list(int v, int n, int g, bool mirror, int* out) {
    int k = 0;
    out[k++] = v + g;
    if (v >= g && v < n - g) return k;
    for (int q = -g; q < n + g; ++q) {
        if (q >= 0 && q < n) {
            q = n - 1;  // skip the interior
            continue;
        }
        const int src = mirror ? mirror3(q, n) : wrap3(q, n);
        if (src == v && k < 2 * g + 1) out[k++] = q + g;
    }
    return k;
}

// A block of the density pass: 128 sites of a row; with the totals in FP32 32 columns of 4 rows, whose
// threads a narrow lattice keeps busy too (step_totals of one species at 32 x 32 x 128: 673 us for 24
// steps, 859 with rows of 128; at 128^3 2,527 and 2,550).  In FP64, bound by the FP64 pipe, the
// smaller blocks share small lattices out more evenly (32^3: 1,927 us for 24 steps, 2,038 in 32 x 4).
template <typename T, bool TOT>
struct DensityBlock {
    static constexpr int X = TOT && sizeof(T) == 4 ? 32 : 128, Y = 128 / X;
};

// The density pass: each site's sums over its 19 populations per species give rho_s and psi_s,
// written with their ghost images into the two volumes.  One thread per site: x and the row within
// the block (DensityBlock), y and z from the grid, looping when the grid is smaller than the lattice
// (the plain pass launches one block per row segment, so each loop runs once).  TOT: the block's
// FP64 partials of the totals of the state go to part[block] as well -- the sums over its sites of
// each species' density deviation sum_l f_l and of the lattice momentum: a site's sums (its two
// species' momenta added) in the context's precision, the sums over the sites in FP64 (the
// FP64 pipe is the scarce one), in a fixed order.
// 16 CTAs per SM for the plain FP32 pass (32 registers, as it ran fastest); 8 with the totals,
// whose FP64 accumulators need up to 64 registers, and in FP64, so that neither spills
// dn, jt (FP32, full relaxation, from populations; else null): the densities' deviations and the
// momentum (three planes) for K3_RELAX.  odd (FP64): set where a density's psi had to be a number; it
// stays set for the state's later steps, which take the FP64 forms then.
template <typename T, bool TOT, bool MOM = false>
__global__ void __launch_bounds__(128, TOT || MOM || sizeof(T) == 8 ? 8 : 16)
    k3_density(const T* __restrict__ f, T* __restrict__ vol, const Step3<T> C, double* __restrict__ part,
               float2* __restrict__ dn = nullptr, float* __restrict__ jt = nullptr, int* __restrict__ odd = nullptr) {
    using V = typename PairOf<T>::V;
    pdl_enter();
    using B = DensityBlock<T, TOT>;
    const int x = blockIdx.x * B::X + threadIdx.x % B::X;
    double mass0 = 0.0, mass1 = 0.0, momx = 0.0, momy = 0.0, momz = 0.0;
    V* const P = reinterpret_cast<V*>(vol);
    for (int z = blockIdx.z; z < C.nz; z += gridDim.z)
        for (int y = blockIdx.y * B::Y + threadIdx.x / B::X; y < C.ny; y += gridDim.y * B::Y) {
            if (x >= C.nx) continue;
            const long long i = ((long long)z * C.ny + y) * C.pitch + x;
            T rho[2] = {T(0), T(0)}, psi[2] = {T(0), T(0)};
            float2 dev = make_float2(0.f, 0.f);
            T d[9];  // TOT, MOM: f_l - f_opp(l) of the nine pairs, the species added
#pragma unroll
            for (int s = 0; s < 2; ++s) {  // unrolled, so that the per-species values stay in registers
                if (s >= C.ns) break;
                T a = f[(s * 19) * C.plane + i];
#pragma unroll
                for (int l = 1; l < 19; l += 2) {
                    const T u = f[(s * 19 + l) * C.plane + i], v = f[(s * 19 + l + 1) * C.plane + i];
                    a += u;
                    a += v;
                    if constexpr (TOT || MOM) d[l / 2] = s == 0 ? u - v : d[l / 2] + (u - v);
                }
                rho[s] = C.rho_ref[s] + a;
                psi[s] = psi3(C, s, rho[s]);
                if constexpr (sizeof(T) == 8) {
                    if (C.fixed != 0 && psi3_beyond(rho[s])) {
                        psi[s] = 1.0 - exp(-rho[s] / C.rho0[s]);
                        atomicOr(odd, 1);
                    }
                }
                if constexpr (TOT) {
                    if (s == 0)
                        mass0 += (double)a;
                    else
                        mass1 += (double)a;
                }
                if constexpr (MOM) (s == 0 ? dev.x : dev.y) = a;
            }
            if constexpr (TOT || MOM) {
                // velocities 1, 3, 5 along x, y, z, then (1,1,0), (1,-1,0), (1,0,1), (1,0,-1), (0,1,1), (0,1,-1)
                const T mx = d[0] + ((d[3] + d[4]) + (d[5] + d[6]));
                const T my = d[1] + ((d[3] - d[4]) + (d[7] + d[8]));
                const T mz = d[2] + ((d[5] - d[6]) + (d[7] - d[8]));
                if constexpr (TOT) {
                    momx += (double)mx;
                    momy += (double)my;
                    momz += (double)mz;
                }
                if constexpr (MOM) {
                    dn[i] = dev;
                    jt[i] = mx;
                    jt[C.plane + i] = my;
                    jt[2 * C.plane + i] = mz;
                }
            }
            V pv, rv;
            pv.x = psi[0];
            pv.y = psi[1];
            rv.x = rho[0];
            rv.y = rho[1];
            int xs[2 * GX + 1], ys[2 * GY + 1], zs[2 * GZ + 1];
            const int nxl = ghost_list(x, C.nx, GX, false, xs);
            const int nyl = ghost_list(y, C.ny, GY, false, ys);
            const int nzl = ghost_list(z, C.nz, GZ, C.zbc != 0, zs);
            for (int c = 0; c < nzl; ++c)
                for (int b = 0; b < nyl; ++b)
                    for (int a = 0; a < nxl; ++a) {
                        const long long o = ((long long)zs[c] * C.gy + ys[b]) * C.gpitch + xs[a];
                        P[o] = pv;
                        P[C.gvol + o] = rv;
                    }
        }
    if constexpr (TOT) {
        __shared__ double red[5][128];
        red[0][threadIdx.x] = mass0;
        red[1][threadIdx.x] = mass1;
        red[2][threadIdx.x] = momx;
        red[3][threadIdx.x] = momy;
        red[4][threadIdx.x] = momz;
        __syncthreads();
        for (int h = 64; h > 0; h >>= 1) {
            if ((int)threadIdx.x < h)
                for (int q = 0; q < 5; ++q) red[q][threadIdx.x] += red[q][threadIdx.x + h];
            __syncthreads();
        }
        const long long blk = ((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        if (threadIdx.x < 5) part[blk * 5 + threadIdx.x] = red[threadIdx.x][0];
    }
}

// out = mass A, mass B, momentum x, y, z: the sum of part[b][q] over the nblk blocks (64 threads per
// quantity, thread t adding blocks t, t + 64, ... in order, then a fixed tree; FP64, the same bits on
// every call), plus base[q] (the sites times rho_ref,s for the masses).
__global__ void __launch_bounds__(320)
    k3_totals_sum(const double* __restrict__ part, int nblk, double base0, double base1, double* __restrict__ out) {
    __shared__ double red[10];
    pdl_enter();
    const int q = threadIdx.x / 64, t = threadIdx.x % 64;
    double a = 0.0;
#pragma unroll 4
    for (int b = t; b < nblk; b += 64) a += part[b * 5 + q];
    for (int h = 16; h > 0; h >>= 1) a += __shfl_xor_sync(0xffffffffu, a, h);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x / 32] = a;
    __syncthreads();
    if (threadIdx.x < 5) {
        const double base = threadIdx.x == 0 ? base0 : (threadIdx.x == 1 ? base1 : 0.0);
        out[threadIdx.x] = (red[2 * threadIdx.x] + red[2 * threadIdx.x + 1]) + base;
    }
}

// ---- k3_step -----------------------------------------------------------------------------

// (FP32, tau = 1) K3_RELAX: the pass over moments; K3_LOOK: rho and u of a state held as moments
enum { K3_WRITE = 1, K3_FIELDS = 2, K3_RELAX = 4, K3_LOOK = 8 };

template <typename T, int TY, int TZ>
struct Smem3 {
    static constexpr int BX = Tile3<T>::BX, BY = TY + 2 * GY, BZ = TZ + 2 * GZ;
    typename PairOf<T>::V box[2][BZ][BY][BX];  // psi, rho pairs of the tile and its halo
    alignas(8) unsigned long long bar;
};

__device__ __forceinline__ unsigned su32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// The links of Eq. FORCE, one of each antipodal pair (first nonzero component positive), by
// shell |c|^2 = 1, 2, 3, 4, 5, 6, 8.
#define LBM3_SHELL1(L) L(0, 0, 1) L(0, 1, 0) L(1, 0, 0)
#define LBM3_SHELL2(L) L(0, 1, -1) L(0, 1, 1) L(1, -1, 0) L(1, 0, -1) L(1, 0, 1) L(1, 1, 0)
#define LBM3_SHELL3(L) L(1, -1, -1) L(1, -1, 1) L(1, 1, -1) L(1, 1, 1)
#define LBM3_SHELL4(L) L(0, 0, 2) L(0, 2, 0) L(2, 0, 0)
#define LBM3_SHELL5(L)                                                                                      \
    L(0, 1, -2) L(0, 1, 2) L(0, 2, -1) L(0, 2, 1) L(1, -2, 0) L(1, 0, -2) L(1, 0, 2) L(1, 2, 0) L(2, -1, 0) \
        L(2, 0, -1) L(2, 0, 1) L(2, 1, 0)
#define LBM3_SHELL6(L)                                                                                    \
    L(1, -2, -1) L(1, -2, 1) L(1, -1, -2) L(1, -1, 2) L(1, 1, -2) L(1, 1, 2) L(1, 2, -1) L(1, 2, 1)       \
        L(2, -1, -1) L(2, -1, 1) L(2, 1, -1) L(2, 1, 1)
#define LBM3_SHELL8(L) L(0, 2, -2) L(0, 2, 2) L(2, -2, 0) L(2, 0, -2) L(2, 0, 2) L(2, 2, 0)

// c * d added into an accumulator for a constant component c in -2..2
template <int C, typename V>
__device__ __forceinline__ V addc(V acc, V d) {
    if constexpr (C == 1) return vadd(acc, d);
    if constexpr (C == -1) return vsub(acc, d);
    if constexpr (C == 2 || C == -2) return vfma(vsplat(decltype(d.x)(C)), d, acc);
    return acc;
}

// Eq. FORCE of one species from psi on the 2^PSI3_BITS scale: the 46 antipodal differences gathered
// shell by shell in integers (exact), the seven shells' weighted sums rounded once (DotFx), the
// product with psi(x) in FP64.  The FP64 form takes about 170 FP64 instructions a species, this 3.
template <typename PSF>
__device__ __forceinline__ double3 force3_fx(const lbm::CoefFx<7>& K, const PSF& ps) {
    using lbm::i64;
    lbm::DotFx tx, ty, tz;
#define LBM3_ACC(dx, dy, dz)                                    \
    {                                                           \
        const i64 d_ = ps(dx, dy, dz) - ps(-(dx), -(dy), -(dz)); \
        sx += (dx) * d_;                                        \
        sy += (dy) * d_;                                        \
        sz += (dz) * d_;                                        \
    }
#define LBM3_SHELL(k, LIST)          \
    {                                \
        i64 sx = 0, sy = 0, sz = 0;  \
        LIST(LBM3_ACC)               \
        tx.add(K, k, sx);            \
        ty.add(K, k, sy);            \
        tz.add(K, k, sz);            \
    }
    LBM3_SHELL(0, LBM3_SHELL1)
    LBM3_SHELL(1, LBM3_SHELL2)
    LBM3_SHELL(2, LBM3_SHELL3)
    LBM3_SHELL(3, LBM3_SHELL4)
    LBM3_SHELL(4, LBM3_SHELL5)
    LBM3_SHELL(5, LBM3_SHELL6)
    LBM3_SHELL(6, LBM3_SHELL8)
#undef LBM3_SHELL
#undef LBM3_ACC
    const double m = -lbm::scaled_double(ps(0, 0, 0), -PSI3_BITS);
    const int e = K.e - 2 - PSI3_BITS;
    return make_double3(__dmul_rn(m, lbm::scaled_double(tx.sum(), e)), __dmul_rn(m, lbm::scaled_double(ty.sum(), e)),
                        __dmul_rn(m, lbm::scaled_double(tz.sum(), e)));
}

// Eq. FORCE over the 46 antipodal link pairs, shell by shell, both species at once, and the cross
// repulsion of Sec. IV over the first belt: F[s][axis] of the site whose psi and rho pairs at the
// offset (dx, dy, dz) are ps(dx, dy, dz) and rh(dx, dy, dz).  LINKS: the cross force's sums link by link
// from zero, as the two-species FP32 form on populations takes them: pairwise they are 18 additions
// fewer, but there, short of registers, cost 3 % of a step (65 x 48 x 33: 17.9 us, 17.5 link by link).
// fixed: psi's bits in fixed point (FP64; uniform).
template <typename T, int NS, bool LINKS, typename PSF, typename RHF>
__device__ __forceinline__ void force3(const Step3<T>& C, bool fixed, const PSF& ps, const RHF& rh, T (&F)[2][3]) {
    using V = typename PairOf<T>::V;
    const auto number = [&](int dx, int dy, int dz) {
        V v = ps(dx, dy, dz);
        if constexpr (sizeof(T) == 8) {
            if (C.fixed != 0) v.x = psi3_number(v.x), v.y = psi3_number(v.y);
        }
        return v;
    };
#define PS(dx, dy, dz) number(dx, dy, dz)
#define RH(dx, dy, dz) rh(dx, dy, dz)
    const V zero = vsplat(T(0));
    V Fx, Fy, Fz;
    if (sizeof(T) == 8 && fixed) {
        if constexpr (sizeof(T) == 8) {
            double3 f0 = force3_fx(C.kf[0], [&](int dx, int dy, int dz) { return (lbm::i64)lbm::bits_of(ps(dx, dy, dz).x); });
            Fx.x = f0.x, Fy.x = f0.y, Fz.x = f0.z;
            Fx.y = Fy.y = Fz.y = 0.0;
            if constexpr (NS == 2) {
                f0 = force3_fx(C.kf[1], [&](int dx, int dy, int dz) { return (lbm::i64)lbm::bits_of(ps(dx, dy, dz).y); });
                Fx.y = f0.x, Fy.y = f0.y, Fz.y = f0.z;
            }
        }
    } else {
    V ax = zero, ay = zero, az = zero;
#define LBM3_ACC(dx, dy, dz)                                \
    {                                                       \
        const V d_ = vsub(PS(dx, dy, dz), PS(-(dx), -(dy), -(dz))); \
        sx = addc<dx>(sx, d_);                              \
        sy = addc<dy>(sy, d_);                              \
        sz = addc<dz>(sz, d_);                              \
    }
#define LBM3_SHELL(q, LIST)                          \
    {                                                \
        V sx = zero, sy = zero, sz = zero;           \
        LIST(LBM3_ACC)                               \
        V kq_;                                       \
        kq_.x = C.kq[0][q];                          \
        kq_.y = C.kq[1][q];                          \
        ax = vfma(kq_, sx, ax);                      \
        ay = vfma(kq_, sy, ay);                      \
        az = vfma(kq_, sz, az);                      \
    }
    LBM3_SHELL(1, LBM3_SHELL1)
    LBM3_SHELL(2, LBM3_SHELL2)
    LBM3_SHELL(3, LBM3_SHELL3)
    LBM3_SHELL(4, LBM3_SHELL4)
    LBM3_SHELL(5, LBM3_SHELL5)
    LBM3_SHELL(6, LBM3_SHELL6)
    LBM3_SHELL(8, LBM3_SHELL8)
#undef LBM3_SHELL
#undef LBM3_ACC
    const V mp = vsub(zero, PS(0, 0, 0));
    Fx = vmul(mp, ax), Fy = vmul(mp, ay), Fz = vmul(mp, az);
    }
    if constexpr (NS == 2) {
        const V r0 = RH(0, 0, 0);
        // cross repulsion: F_s += -G_AB rho_s(x) sum_l w(|c|^2) rho_s'(x + c_l) c_l over the first belt
        V bx1 = zero, by1 = zero, bz1 = zero, bx2 = zero, by2 = zero, bz2 = zero;
#define LBM3_X(dx, dy, dz) vsub(RH(dx, dy, dz), RH(-(dx), -(dy), -(dz)))
        if constexpr (LINKS) {
#define LBM3_XACC(dx, dy, dz, SX, SY, SZ)     \
    {                                         \
        const V d_ = LBM3_X(dx, dy, dz);      \
        SX = addc<dx>(SX, d_);                \
        SY = addc<dy>(SY, d_);                \
        SZ = addc<dz>(SZ, d_);                \
    }
#define LBM3_X1(dx, dy, dz) LBM3_XACC(dx, dy, dz, bx1, by1, bz1)
#define LBM3_X2(dx, dy, dz) LBM3_XACC(dx, dy, dz, bx2, by2, bz2)
            LBM3_SHELL1(LBM3_X1)
            LBM3_SHELL2(LBM3_X2)
#undef LBM3_X1
#undef LBM3_X2
#undef LBM3_XACC
        } else {
            bx1 = LBM3_X(1, 0, 0), by1 = LBM3_X(0, 1, 0), bz1 = LBM3_X(0, 0, 1);
            const V xyp = LBM3_X(1, 1, 0), xym = LBM3_X(1, -1, 0), xzp = LBM3_X(1, 0, 1), xzm = LBM3_X(1, 0, -1),
                    yzp = LBM3_X(0, 1, 1), yzm = LBM3_X(0, 1, -1);
            bx2 = vadd(vadd(xyp, xym), vadd(xzp, xzm)), by2 = vadd(vsub(xyp, xym), vadd(yzp, yzm)),
            bz2 = vadd(vsub(xzp, xzm), vsub(yzp, yzm));
        }
#undef LBM3_X
        const V k1 = vsplat(C.kc[1]), k2 = vsplat(C.kc[2]);
        const V cx_ = vfma(k2, bx2, vmul(k1, bx1)), cy_ = vfma(k2, by2, vmul(k1, by1)),
                cz_ = vfma(k2, bz2, vmul(k1, bz1));
        const V mr = vsub(zero, r0);
        // species A sees the sums over rho_B, species B those over rho_A
        Fx = vfma(mr, vswap(cx_), Fx);
        Fy = vfma(mr, vswap(cy_), Fy);
        Fz = vfma(mr, vswap(cz_), Fz);
    }
    F[0][0] = Fx.x;
    F[0][1] = Fy.x;
    F[0][2] = Fz.x;
    F[1][0] = Fx.y;
    F[1][1] = Fy.y;
    F[1][2] = Fz.y;
#undef PS
#undef RH
}

// Where the fields of a state go (device memory, FP64; null: not wanted).
struct Fields3 {
    double *rho, *u, *f;
};

// The moments of the site's populations f, the body force along x, the common velocity of R5;
// then (K3_FIELDS) rho_s, u and the plain populations into `fields`, or (K3_WRITE) the
// shifted-velocity BGK of Sec. II and the push of the new populations to x + c_l.  Every scalar
// operation has its rounding fixed (smul, sadd, sfma), so a kernel that inlines this computes the
// same bits whatever the code around it.
template <typename T, int NS, int MODE>
__device__ __forceinline__ void site3(const Step3<T>& C, const T (&f)[NS][19], T (&F)[2][3], int x, int y, int z,
                                      long long i, T* __restrict__ fout, int* __restrict__ flag,
                                      const Fields3& fields) {
    using V = typename PairOf<T>::V;
    // ---- moments, body force, common velocity ----
    T rho[NS], ir[NS], jx[NS], jy[NS], jz[NS], drho[NS];
    bool bad = false;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        // each sum starts from its first term (no add of zero)
        T a = f[s][0], mx = f[s][first19(0)], my = f[s][first19(1)], mz = f[s][first19(2)];
#pragma unroll
        for (int l = 1; l < 19; ++l) {
            a = sadd(a, f[s][l]);
            if (c3x(l) && l != first19(0)) mx = sadd(mx, c3x(l) > 0 ? f[s][l] : -f[s][l]);
            if (c3y(l) && l != first19(1)) my = sadd(my, c3y(l) > 0 ? f[s][l] : -f[s][l]);
            if (c3z(l) && l != first19(2)) mz = sadd(mz, c3z(l) > 0 ? f[s][l] : -f[s][l]);
        }
        drho[s] = a;
        rho[s] = sadd(C.rho_ref[s], a);
        if (!(rho[s] > T(0)) || !(rho[s] < T(1e30))) bad = true;
        ir[s] = rcp3(rho[s]);
        jx[s] = mx;
        jy[s] = my;
        jz[s] = mz;
        F[s][0] = sfma(rho[s], C.g, F[s][0]);
    }
    if (bad) atomicOr(flag, 1);
    T nxu = T(0), nyu = T(0), nzu = T(0), den = T(0);
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        nxu = sfma(C.omega[s], jx[s], nxu);
        nyu = sfma(C.omega[s], jy[s], nyu);
        nzu = sfma(C.omega[s], jz[s], nzu);
        den = sfma(C.omega[s], rho[s], den);
    }
    const T iden = rcp3(den);
    const T upx = smul(nxu, iden), upy = smul(nyu, iden), upz = smul(nzu, iden);

    if constexpr ((MODE & K3_FIELDS) != 0) {
        // rho_s, the barycentric velocity (sum_s j_s + F_s / 2) / sum_s rho_s, plain populations
        const long long n = (long long)C.nx * C.ny * C.nz, k = ((long long)z * C.ny + y) * C.nx + x;
        T mxs = T(0), mys = T(0), mzs = T(0), rt = T(0);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            mxs += jx[s] + T(0.5) * F[s][0];
            mys += jy[s] + T(0.5) * F[s][1];
            mzs += jz[s] + T(0.5) * F[s][2];
            rt += rho[s];
            if (fields.rho) fields.rho[s * n + k] = (double)rho[s];
            if (fields.f) {
#pragma unroll
                for (int l = 0; l < 19; ++l)
                    fields.f[(s * 19 + l) * n + k] = wide3(f[s][l]) + w19<double>(l) * (double)C.rho_ref[s];
            }
        }
        if (fields.u) {
            fields.u[k] = (double)(mxs / rt);
            fields.u[n + k] = (double)(mys / rt);
            fields.u[2 * n + k] = (double)(mzs / rt);
        }
    }

    if constexpr ((MODE & K3_WRITE) != 0) {
        // ---- shifted-velocity BGK (Sec. II) and streaming ----
        // Destinations: the site's index plus one offset per axis, chosen by the sign of c_l; the
        // periodic wrap is folded into those offsets once per thread (walls in z are handled by
        // bounce-back below).
        const long long row = C.pitch, lay = (long long)C.ny * C.pitch;
        const bool wall_lo = C.zbc && z == 0, wall_hi = C.zbc && z == C.nz - 1;
        // FP32: the wrapped offsets of each axis precomputed; FP64 (short of registers): the
        // destination of each population wrapped where it is stored
        long long oxm = 0, oxp = 0, oym = 0, oyp = 0, ozm = 0, ozp = 0;
        if constexpr (sizeof(T) == 4) {
            oxm = x == 0 ? C.nx - 1 : -1;
            oxp = x == C.nx - 1 ? -(C.nx - 1) : 1;
            oym = y == 0 ? (C.ny - 1) * row : -row;
            oyp = y == C.ny - 1 ? -(C.ny - 1) * row : row;
            ozm = z == 0 ? (C.nz - 1) * lay : -lay;
            ozp = z == C.nz - 1 ? -(C.nz - 1) * lay : lay;
        }
        auto push = [&](int s, int l, T v) {
            const int cx_ = c3x(l), cy_ = c3y(l), cz_ = c3z(l);
            if ((cz_ < 0 && wall_lo) || (cz_ > 0 && wall_hi)) {  // halfway bounce-back with Ladd's term
                const T uw = cz_ < 0 ? C.wall_u[0] : C.wall_u[1];
                fout[(s * 19 + opp19(l)) * C.plane + i] = sadd(v, -smul(smul(T(6 * cx_) * w19<T>(l), rho[s]), uw));
                return;
            }
            if constexpr (sizeof(T) == 4) {
                const long long o = (cx_ < 0 ? oxm : (cx_ > 0 ? oxp : 0)) + (cy_ < 0 ? oym : (cy_ > 0 ? oyp : 0)) +
                                    (cz_ < 0 ? ozm : (cz_ > 0 ? ozp : 0));
                fout[(s * 19 + l) * C.plane + i + o] = v;
            } else {
                int xd = x + cx_, yd = y + cy_, zd = z + cz_;
                xd = xd < 0 ? xd + C.nx : (xd >= C.nx ? xd - C.nx : xd);
                yd = yd < 0 ? yd + C.ny : (yd >= C.ny ? yd - C.ny : yd);
                zd = zd < 0 ? zd + C.nz : (zd >= C.nz ? zd - C.nz : zd);
                fout[(s * 19 + l) * C.plane + ((long long)zd * C.ny + yd) * C.pitch + xd] = v;
            }
        };
        if constexpr (NS == 2 && sizeof(T) == 4) {
            // both species in lockstep, (A, B) pairs of packed FP32 instructions
            V fp[19];
#pragma unroll
            for (int l = 0; l < 19; ++l) {
                fp[l].x = f[0][l];
                fp[l].y = f[1][l];
            }
            V rh, drh, om, tau, fx, fy, fz;
            rh.x = rho[0], rh.y = rho[1];
            drh.x = drho[0], drh.y = drho[1];
            om.x = C.omega[0], om.y = C.omega[1];
            tau.x = smul(C.tau[0], ir[0]), tau.y = smul(C.tau[1], ir[1]);
            fx.x = F[0][0], fx.y = F[1][0];
            fy.x = F[0][1], fy.y = F[1][1];
            fz.x = F[0][2], fz.y = F[1][2];
            const V keep = vsub(vsplat(T(1)), om);
            const V ux = vfma(fx, tau, vsplat(upx)), uy = vfma(fy, tau, vsplat(upy)), uz = vfma(fz, tau, vsplat(upz));
            const V u15 = vmul(vsplat(T(1.5)), vfma(ux, ux, vfma(uy, uy, vmul(uz, uz))));
            const V b = vmul(om, rh);
            const V base = vsub(vmul(om, drh), vmul(b, u15));  // omega (drho - 3/2 rho u^2)
            push(0, 0, vfma(keep, fp[0], vmul(vsplat(w19<T>(0)), base)).x);
            push(1, 0, vfma(keep, fp[0], vmul(vsplat(w19<T>(0)), base)).y);
#pragma unroll
            for (int l = 1; l < 19; l += 2) {  // l and its opposite l + 1
                // c_l . u with the components +-1 or 0 of this l (the branches fold away unrolled)
                // from zero: starting from the first component, as the scalar path does, saves an
                // add but changed the register allocation of this build for the worse (measured)
                V cu = vsplat(T(0));
                if (c3x(l) > 0) cu = vadd(cu, ux);
                if (c3x(l) < 0) cu = vsub(cu, ux);
                if (c3y(l) > 0) cu = vadd(cu, uy);
                if (c3y(l) < 0) cu = vsub(cu, uy);
                if (c3z(l) > 0) cu = vadd(cu, uz);
                if (c3z(l) < 0) cu = vsub(cu, uz);
                const T w = w19<T>(l);
                const V wb = vmul(vsplat(w), b);
                const V even = vfma(vmul(vsplat(T(4.5)), wb), vmul(cu, cu), vmul(vsplat(w), base));
                const V odd = vmul(vmul(vsplat(T(3)), wb), cu);
                const V gp = vadd(vfma(keep, fp[l], even), odd);
                const V gm = vsub(vfma(keep, fp[l + 1], even), odd);
                push(0, l, gp.x);
                push(1, l, gp.y);
                push(0, l + 1, gm.x);
                push(1, l + 1, gm.y);
            }
        } else {
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                // the operations of the packed path, one species at a time
                const T om = C.omega[s], keep = T(1) - om, tir = smul(C.tau[s], ir[s]);
                const T ux = sfma(F[s][0], tir, upx), uy = sfma(F[s][1], tir, upy), uz = sfma(F[s][2], tir, upz);
                const T u15 = smul(T(1.5), sfma(ux, ux, sfma(uy, uy, smul(uz, uz))));
                const T b = smul(om, rho[s]);
                const T base = sadd(smul(om, drho[s]), -smul(b, u15));  // omega (drho - 3/2 rho u^2)
                // even part +- odd part = e + cu (4.5 w b cu +- 3 w b), per weight class; the kept
                // part (1 - omega) f vanishes at tau = 1
                const T wa = w19<T>(1), we = w19<T>(7);
                const T ea = smul(wa, base), ee = smul(we, base);
                const T ca = smul(T(4.5) * wa, b), ce = smul(T(4.5) * we, b);
                const T da = smul(T(3) * wa, b), de = smul(T(3) * we, b);
                const bool relaxed = keep == T(0);
                const T g0 = smul(w19<T>(0), base);
                push(s, 0, relaxed ? g0 : sfma(keep, f[s][0], g0));
#pragma unroll
                for (int l = 1; l < 19; l += 2) {  // l and its opposite l + 1
                    // starting from the first, +1, component (no add of zero)
                    T cu = c3x(l) ? ux : (c3y(l) ? uy : uz);
                    if (c3x(l) && c3y(l)) cu = sadd(cu, c3y(l) > 0 ? uy : -uy);
                    if ((c3x(l) || c3y(l)) && c3z(l)) cu = sadd(cu, c3z(l) > 0 ? uz : -uz);
                    const T e = l < 7 ? ea : ee, c = l < 7 ? ca : ce, d = l < 7 ? da : de;
                    const T ep = relaxed ? e : sfma(keep, f[s][l], e), em = relaxed ? e : sfma(keep, f[s][l + 1], e);
                    push(s, l, sfma(sfma(c, cu, d), cu, ep));
                    push(s, l + 1, sfma(sfma(c, cu, -d), cu, em));
                }
            }
        }
    }
}

// ---- full relaxation: the state as moments ------------------------------------------------------

// The state after a fully relaxed collision, as (A, B) pairs of FP32 in the layout of a population
// plane: the density deviation d (from rho_ref), the velocity u of the species' equilibrium, and
// base = d - 3/2 rho u.u, which its populations share:
//   f*_l - w_l rho_ref = w_l (base + rho c.u (3 + 9/2 c.u)).
// d has two copies (k3_stream reads the neighbours' old one while it writes the new).  jt holds the
// streamed-in lattice momentum, the species added (R5's common velocity needs no more at tau = 1).
struct Mom3 {
    float2* d[2];
    float2 *base, *ux, *uy, *uz;
    float *jx, *jy, *jz;
};

// That population over w_l; cu: c.u, or with sg = -1 its negative: (-cu) (3 - 9/2 cu) = cu (9/2 cu - 3)
// to the bit.
__device__ __forceinline__ float2 relaxed_pop(float2 base, float2 rho, float2 cu, int sg) {
    return vfma(vmul(rho, cu), vfma(vsplat(4.5f), cu, vsplat(sg > 0 ? 3.f : -3.f)), base);
}

// What has streamed into a site so far: density and momentum, species side by side, times 36 (the
// weights 12, 2 and 1 are exact, and a site is scaled once).
struct Sum3 {
    float2 r, x, y, z;
};

// v / 36 to the last rounding (1/36 in FP32 alone is 7e-9 too large: the same growth every step).
__device__ __forceinline__ float2 over36(float2 v) {
    constexpr float hi = (float)(1.0 / 36.0), lo = (float)(1.0 / 36.0 - (double)hi);
    return vfma(v, vsplat(hi), vmul(v, vsplat(lo)));
}

// Adds population 36 w g of velocity (CX, CY, CZ), w = 1/18 (axes: W2 = 2) or 1/36 (edges: 1).
template <int CX, int CY, int CZ>
__device__ __forceinline__ void gain(Sum3& S, float2 g) {
    constexpr float W2 = CX * CX + CY * CY + CZ * CZ == 1 ? 2.f : 1.f;
    const auto add = [&](float2 a, float sign) {
        if (W2 == 1.f) return sign > 0 ? vadd(a, g) : vsub(a, g);
        return vfma(vsplat(sign * W2), g, a);
    };
    S.r = add(S.r, 1.f);
    if constexpr (CX != 0) S.x = add(S.x, (float)CX);
    if constexpr (CY != 0) S.y = add(S.y, (float)CY);
    if constexpr (CZ != 0) S.z = add(S.z, (float)CZ);
}

constexpr int AHEAD = 2;
__device__ __forceinline__ void prefetch5(const Mom3& M, const float2* D, long long k) {
    asm volatile("prefetch.global.L1 [%0];" ::"l"(M.base + k));
    asm volatile("prefetch.global.L1 [%0];" ::"l"(D + k));
    asm volatile("prefetch.global.L1 [%0];" ::"l"(M.ux + k));
    asm volatile("prefetch.global.L1 [%0];" ::"l"(M.uy + k));
    asm volatile("prefetch.global.L1 [%0];" ::"l"(M.uz + k));
}

// One site of a neighbouring column: what its populations need.
struct Col3 {
    float2 base, rho, ux, uy, uz;
};
template <int CX, int CY, int CZ>
__device__ __forceinline__ void stream_in(Sum3& S, const Col3& c) {
    if constexpr (CX == 0 && CY == 0 && CZ == 0) {
        S.r = vfma(vsplat(12.f), c.base, S.r);
    } else {
        // c.u up to the sign of its first component, which relaxed_pop takes
        constexpr int sg = CX ? CX : (CY ? CY : CZ);
        float2 cu = CX ? c.ux : (CY ? c.uy : c.uz);
        if constexpr (CX != 0 && CY != 0) cu = CY * sg > 0 ? vadd(cu, c.uy) : vsub(cu, c.uy);
        if constexpr ((CX != 0 || CY != 0) && CZ != 0) cu = CZ * sg > 0 ? vadd(cu, c.uz) : vsub(cu, c.uz);
        gain<CX, CY, CZ>(S, relaxed_pop(c.base, c.rho, cu, sg));
    }
}
// The population (CX, CY, CZ) coming back from a wall: the site's own opposite one, with Ladd's term.
template <int CX, int CY, int CZ>
__device__ __forceinline__ void wall_in(Sum3& S, const Col3& c, float uw) {
    float2 cu = c.uz;  // of the opposite velocity, up to the sign of its z component
    if constexpr (CX != 0) cu = CX * CZ > 0 ? vadd(cu, c.ux) : vsub(cu, c.ux);
    if constexpr (CY != 0) cu = CY * CZ > 0 ? vadd(cu, c.uy) : vsub(cu, c.uy);
    float2 f = relaxed_pop(c.base, c.rho, cu, -CZ);
    if constexpr (CX != 0) f = vfma(vsplat(6.f * CX), vmul(c.rho, vsplat(uw)), f);
    gain<CX, CY, CZ>(S, f);
}

// The streaming pass.  A thread owns a column (x, y) of `chunk` layers and walks up it, one source
// layer at a time: each layer's nine columns around it are read once (37 pairs) and give to the
// three layers they stream to, so a site costs 37 (chunk + 2) / chunk reads instead of 67.  The
// order of the additions (from below, from the same layer, from above) is the same whatever the
// chunk.  With TOT the block's FP64 partials of the state's totals too (as k3_density's).
// About 240 instructions and 300 B of L1 reads per site with the whole state in L2 at 128^3, 66.6 us a
// step there; a block's layers are read one after the other, and the layer ahead prefetched.
template <bool TOT>
__global__ void __launch_bounds__(128, 4)
    k3_stream(const Mom3 M, int dc, float* __restrict__ vol, const Step3<float> C, int chunk, double* __restrict__ part) {
    pdl_enter();
    const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 4 + threadIdx.y;
    const bool live = x < C.nx && y < C.ny;
    const int z0 = blockIdx.z * chunk, z1 = min(z0 + chunk, C.nz);
    double tot[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    if (live) {
        const int xm = x == 0 ? C.nx - 1 : x - 1, xp = x == C.nx - 1 ? 0 : x + 1;
        // rows within a layer, whose sites number less than 2^31
        const int r0 = y * C.pitch, rm = (y == 0 ? C.ny - 1 : y - 1) * C.pitch, rp = (y == C.ny - 1 ? 0 : y + 1) * C.pitch;
        const long long lay = (long long)C.ny * C.pitch;
        const float2* const D = dc ? M.d[1] : M.d[0];
        float2* const Dn = dc ? M.d[0] : M.d[1];
        const float2 rref = make_float2(C.rho_ref[0], C.rho_ref[1]);
        float2* const P = reinterpret_cast<float2*>(vol);
        int xs[2 * GX + 1], ys[2 * GY + 1], zs_[2 * GZ + 1];
        const int nxl = ghost_list(x, C.nx, GX, false, xs);
        const int nyl = ghost_list(y, C.ny, GY, false, ys);
        const bool edge = nxl > 1 || nyl > 1;
        const Sum3 none = {vsplat(0.f), vsplat(0.f), vsplat(0.f), vsplat(0.f)};
        // layers zs - 1 (complete after this source layer), zs, zs + 1
        Sum3 below = none, here = none, above = none;
        const bool walls = C.zbc != 0;
        for (int zs = z0 - 1; zs <= z1; ++zs) {
            const bool in = zs >= 0 && zs < C.nz;
            if (zs + AHEAD < min(z1 + 1, C.nz)) {  // the block's part of a later layer into L1, its halo by its edge threads
                const long long o = lay * (zs + AHEAD);
                const int k = r0 + x;
                prefetch5(M, D, o + k);
                if (threadIdx.y == 0) prefetch5(M, D, o + rm + x);
                if (threadIdx.y == 3) prefetch5(M, D, o + rp + x);
            }
            if (in || !walls) {
                const long long o = lay * (in ? zs : (zs < 0 ? zs + C.nz : zs - C.nz));
                const float2 *const pb = M.base + o, *const pd = D + o, *const px = M.ux + o, *const py = M.uy + o,
                                   *const pz = M.uz + o;
#define LBM3_COL(name, off, X, Y, Z)  \
    Col3 name;                        \
    {                                 \
        const int k_ = (off);         \
        name.base = pb[k_];           \
        name.rho = vadd(rref, pd[k_]); \
        if (X) name.ux = px[k_];      \
        if (Y) name.uy = py[k_];      \
        if (Z) name.uz = pz[k_];      \
    }
                {
                    LBM3_COL(c, r0 + x, true, true, true)
                    stream_in<0, 0, -1>(below, c);
                    stream_in<0, 0, 0>(here, c);
                    stream_in<0, 0, 1>(above, c);
                    if (walls && zs == 0) {  // `here` is the bottom layer: nothing came from below
                        Sum3 own = none;
                        wall_in<0, 0, 1>(own, c, C.wall_u[0]);
                        wall_in<1, 0, 1>(own, c, C.wall_u[0]);
                        wall_in<-1, 0, 1>(own, c, C.wall_u[0]);
                        wall_in<0, 1, 1>(own, c, C.wall_u[0]);
                        wall_in<0, -1, 1>(own, c, C.wall_u[0]);
                        here.r = vadd(here.r, own.r);
                        here.x = vadd(here.x, own.x);
                        here.y = vadd(here.y, own.y);
                        here.z = vadd(here.z, own.z);
                    }
                    if (walls && zs == C.nz - 1) {  // `here` is the top layer: nothing will come from above
                        wall_in<0, 0, -1>(here, c, C.wall_u[1]);
                        wall_in<1, 0, -1>(here, c, C.wall_u[1]);
                        wall_in<-1, 0, -1>(here, c, C.wall_u[1]);
                        wall_in<0, 1, -1>(here, c, C.wall_u[1]);
                        wall_in<0, -1, -1>(here, c, C.wall_u[1]);
                    }
                }
                {
                    LBM3_COL(c, r0 + xm, true, false, true)
                    stream_in<1, 0, -1>(below, c);
                    stream_in<1, 0, 0>(here, c);
                    stream_in<1, 0, 1>(above, c);
                }
                {
                    LBM3_COL(c, r0 + xp, true, false, true)
                    stream_in<-1, 0, -1>(below, c);
                    stream_in<-1, 0, 0>(here, c);
                    stream_in<-1, 0, 1>(above, c);
                }
                {
                    LBM3_COL(c, rm + x, false, true, true)
                    stream_in<0, 1, -1>(below, c);
                    stream_in<0, 1, 0>(here, c);
                    stream_in<0, 1, 1>(above, c);
                }
                {
                    LBM3_COL(c, rp + x, false, true, true)
                    stream_in<0, -1, -1>(below, c);
                    stream_in<0, -1, 0>(here, c);
                    stream_in<0, -1, 1>(above, c);
                }
                if (zs >= z0 && zs < z1) {  // the diagonals stay in their layer
                    {
                        LBM3_COL(c, rm + xm, true, true, false)
                        stream_in<1, 1, 0>(here, c);
                    }
                    {
                        LBM3_COL(c, rp + xp, true, true, false)
                        stream_in<-1, -1, 0>(here, c);
                    }
                    {
                        LBM3_COL(c, rp + xm, true, true, false)
                        stream_in<1, -1, 0>(here, c);
                    }
                    {
                        LBM3_COL(c, rm + xp, true, true, false)
                        stream_in<-1, 1, 0>(here, c);
                    }
                }
#undef LBM3_COL
            }
            const int z = zs - 1;  // complete
            if (z >= z0) {
                const long long i = lay * z + r0 + x;
                const float2 dn = over36(below.r), px = over36(below.x), py = over36(below.y), pz = over36(below.z);
                Dn[i] = dn;
                const float jx = px.x + px.y, jy = py.x + py.y, jz = pz.x + pz.y;
                M.jx[i] = jx;
                M.jy[i] = jy;
                M.jz[i] = jz;
                const float2 rho = vadd(rref, dn);
                const float2 psi = make_float2(psi3(C, 0, rho.x), psi3(C, 1, rho.y));
                if constexpr (TOT) {
                    tot[0] += (double)dn.x;
                    tot[1] += (double)dn.y;
                    tot[2] += (double)jx;
                    tot[3] += (double)jy;
                    tot[4] += (double)jz;
                }
                float2* const own = P + ((long long)(z + GZ) * C.gy + (y + GY)) * C.gpitch + (x + GX);
                own[0] = psi;
                own[C.gvol] = rho;
                if (edge || z < GZ || z >= C.nz - GZ) {  // and where ghosts repeat the site
                    const int nzl = ghost_list(z, C.nz, GZ, walls, zs_);
                    for (int c = 0; c < nzl; ++c)
                        for (int b = 0; b < nyl; ++b)
                            for (int a = c == 0 && b == 0 ? 1 : 0; a < nxl; ++a) {
                                const long long k = ((long long)zs_[c] * C.gy + ys[b]) * C.gpitch + xs[a];
                                P[k] = psi;
                                P[C.gvol + k] = rho;
                            }
                }
            }
            below = here;
            here = above;
            above = none;
        }
    }
    if constexpr (TOT) {
        __shared__ double red[5][128];
        const int t = threadIdx.y * 32 + threadIdx.x;
#pragma unroll
        for (int q = 0; q < 5; ++q) red[q][t] = tot[q];
        __syncthreads();
        for (int h = 64; h > 0; h >>= 1) {
            if (t < h)
                for (int q = 0; q < 5; ++q) red[q][t] += red[q][t + h];
            __syncthreads();
        }
        const long long blk = ((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        if (t < 5) part[blk * 5 + t] = red[t][0];
    }
}

// Whether a density of the site is <= 0, NaN or Inf.
__device__ __forceinline__ bool bad_density(float2 rho) {
    return !(rho.x > 0.f) || !(rho.x < 1e30f) || !(rho.y > 0.f) || !(rho.y < 1e30f);
}

// The site update of the relaxing pass (k3_step, K3_RELAX): from the force, the streamed-in density
// and momentum, the species' velocities and base.
__device__ __forceinline__ void relax3(const Step3<float>& C, const Mom3& M, const float (&F)[2][3], float2 rho,
                                       long long i, float jx, float jy, float jz, float2 d, int* __restrict__ flag) {
    if (bad_density(rho)) atomicOr(flag, 1);
    const float iden = 1.f / sadd(rho.x, rho.y);
    const float2 ir = make_float2(1.f / rho.x, 1.f / rho.y);
    const float2 fx = make_float2(sfma(rho.x, C.g, F[0][0]), sfma(rho.y, C.g, F[1][0]));
    const float2 fy = make_float2(F[0][1], F[1][1]), fz = make_float2(F[0][2], F[1][2]);
    const float px = smul(jx, iden), py = smul(jy, iden), pz = smul(jz, iden);
    const float2 ux = vfma(fx, ir, vsplat(px)), uy = vfma(fy, ir, vsplat(py)), uz = vfma(fz, ir, vsplat(pz));
    const float2 u15 = vmul(vsplat(1.5f), vfma(ux, ux, vfma(uy, uy, vmul(uz, uz))));
    M.base[i] = vsub(d, vmul(rho, u15));
    M.ux[i] = ux;
    M.uy[i] = uy;
    M.uz[i] = uz;
}

// rho_s and the barycentric velocity (sum_s j_s + F_s / 2) / sum_s rho_s of a site (K3_LOOK), and, as
// every read of a state, the test of its densities.
__device__ __forceinline__ void look3(const Step3<float>& C, const float (&F)[2][3], float2 rho, long long k, float jx,
                                      float jy, float jz, int* __restrict__ flag, const Fields3& out) {
    if (bad_density(rho)) atomicOr(flag, 1);
    const long long n = (long long)C.nx * C.ny * C.nz;
    const float irt = 1.f / sadd(rho.x, rho.y);
    const float fx = sadd(sfma(rho.x, C.g, F[0][0]), sfma(rho.y, C.g, F[1][0])), fy = sadd(F[0][1], F[1][1]),
                fz = sadd(F[0][2], F[1][2]);
    if (out.rho) {
        out.rho[k] = wide3(rho.x);
        out.rho[n + k] = wide3(rho.y);
    }
    if (out.u) {
        out.u[k] = wide3(smul(sfma(0.5f, fx, jx), irt));
        out.u[n + k] = wide3(smul(sfma(0.5f, fy, jy), irt));
        out.u[2 * n + k] = wide3(smul(sfma(0.5f, fz, jz), irt));
    }
}

// Populations of the state after streaming, from the moments, into f: what streams into each site,
// population by population (k3_stream's terms).  O = float: the stored populations; double: the plain
// values of lbm3_get_fields.
template <typename O>
__global__ void __launch_bounds__(128) k3_expand(const Mom3 M, int dc, O* __restrict__ f, const Step3<float> C) {
    const int x = blockIdx.x * 128 + threadIdx.x;
    if (x >= C.nx) return;
    const float2 rref = make_float2(C.rho_ref[0], C.rho_ref[1]);
    for (int z = blockIdx.z; z < C.nz; z += gridDim.z)
        for (int y = blockIdx.y; y < C.ny; y += gridDim.y) {
            const long long i = ((long long)z * C.ny + y) * C.pitch + x;
#pragma unroll
            for (int l = 0; l < 19; ++l) {
                const int cx = c3x(l), cy = c3y(l), cz = c3z(l);
                int xs = x - cx, ys = y - cy, zs = z - cz;
                xs = xs < 0 ? xs + C.nx : (xs >= C.nx ? xs - C.nx : xs);
                ys = ys < 0 ? ys + C.ny : (ys >= C.ny ? ys - C.ny : ys);
                const bool wall = C.zbc && (zs < 0 || zs >= C.nz);
                zs = zs < 0 ? zs + C.nz : (zs >= C.nz ? zs - C.nz : zs);
                const long long k = wall ? i : ((long long)zs * C.ny + ys) * C.pitch + xs;
                const float2 base = M.base[k], rho = vadd(rref, (dc ? M.d[1] : M.d[0])[k]);
                const float2 ux = M.ux[k], uy = M.uy[k], uz = M.uz[k];
                float2 v;
                if (l == 0) {
                    v = vmul(vsplat(w19<float>(0)), base);
                } else if (!wall) {  // as stream_in
                    const int sg = cx ? cx : (cy ? cy : cz);
                    float2 cu = cx ? ux : (cy ? uy : uz);
                    if (cx && cy) cu = cy * sg > 0 ? vadd(cu, uy) : vsub(cu, uy);
                    if ((cx || cy) && cz) cu = cz * sg > 0 ? vadd(cu, uz) : vsub(cu, uz);
                    v = vmul(vsplat(w19<float>(l)), relaxed_pop(base, rho, cu, sg));
                } else {  // as wall_in
                    float2 cu = uz;
                    if (cx) cu = cx * cz > 0 ? vadd(cu, ux) : vsub(cu, ux);
                    if (cy) cu = cy * cz > 0 ? vadd(cu, uy) : vsub(cu, uy);
                    v = relaxed_pop(base, rho, cu, -cz);
                    if (cx) v = vfma(vsplat(6.f * cx), vmul(rho, vsplat(cz > 0 ? C.wall_u[0] : C.wall_u[1])), v);
                    v = vmul(vsplat(w19<float>(l)), v);
                }
                if constexpr (sizeof(O) == 4) {
                    f[l * C.plane + i] = v.x;
                    f[(19 + l) * C.plane + i] = v.y;
                } else {
                    const long long n = (long long)C.nx * C.ny * C.nz, q = ((long long)z * C.ny + y) * C.nx + x;
                    f[l * n + q] = lbm::widen_fx(v.x) + w19<double>(l) * (double)C.rho_ref[0];
                    f[(19 + l) * n + q] = lbm::widen_fx(v.y) + w19<double>(l) * (double)C.rho_ref[1];
                }
            }
        }
}

// FP32 tiles of 256 threads: 3 CTAs per SM (80 registers, 16 bytes of spills), measured faster than
// 2 CTAs at 110 registers without spills -- the kernel waits on memory and more warps hide it.
template <typename T, int MODE, int NS, int TY, int TZ>
__global__ void __launch_bounds__(Tile3<T>::TX* TY* TZ,
                                  Tile3<T>::TX* TY* TZ > 256 ? (MODE >= K3_RELAX ? 2 : 1)
                                                             : (sizeof(T) == 4 ? (MODE >= K3_RELAX ? 4 : 3)
                                                                               : 512 / (Tile3<T>::TX * TY * TZ)))
    k3_step(const __grid_constant__ CUtensorMap vmap, const T* __restrict__ fin, T* __restrict__ fout,
            const Step3<T> C, int* __restrict__ flag, const Fields3 fields, const Mom3 M, int dn) {
    constexpr int TX = Tile3<T>::TX;
    extern __shared__ __align__(1024) unsigned char smem3[];
    Smem3<T, TY, TZ>& S = *reinterpret_cast<Smem3<T, TY, TZ>*>(smem3);
    const int tx = threadIdx.x, ty = threadIdx.y, tz = threadIdx.z;
    const int tid = (tz * TY + ty) * TX + tx;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, z0 = blockIdx.z * TZ;
    const int x = x0 + tx, y = y0 + ty, z = z0 + tz;
    const bool live = x < C.nx && y < C.ny && z < C.nz;
    pdl_enter();
    if (tid == 0) {
        const unsigned bar = su32(&S.bar);
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        constexpr unsigned bytes = (unsigned)sizeof(S.box);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
        // box origin: padded (x0, y0, z0) = site (x0 - GX, y0 - GY, z0 - GZ); x counts values of T
        asm volatile(
            "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
            "%5}], [%6];\n" ::"r"(su32(&S.box[0][0][0][0])),
            "l"(&vmap), "r"(2 * x0), "r"(y0), "r"(z0), "r"(0), "r"(bar)
            : "memory");
    }
    // own populations from HBM while the box is on its way
    const long long i = ((long long)z * C.ny + y) * C.pitch + x;
    // (FP64, short of registers, loads them after the force: its other warps cover the wait)
    // K3_RELAX: the streamed-in density and momentum instead
    T f[MODE >= K3_RELAX ? 1 : NS][19];
    float jx = 0.f, jy = 0.f, jz = 0.f;
    float2 d = make_float2(0.f, 0.f);
    const auto load = [&]() {
        if constexpr (MODE >= K3_RELAX) {
            d = (dn ? M.d[1] : M.d[0])[i];
            jx = M.jx[i];
            jy = M.jy[i];
            jz = M.jz[i];
        } else {
#pragma unroll
            for (int s = 0; s < NS; ++s)
#pragma unroll
                for (int l = 0; l < 19; ++l) f[s][l] = fin[(s * 19 + l) * C.plane + i];
        }
    };
    if (sizeof(T) == 4 && live) load();
    __syncthreads();  // the barrier is initialised before anyone waits on it
    bool ok = true;
    {
        const unsigned bar = su32(&S.bar);
        const long long t0 = clock64();
        for (;;) {
            unsigned done;
            asm volatile(
                "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                : "=r"(done)
                : "r"(bar), "r"(0u)
                : "memory");
            if (done) break;
            if (clock64() - t0 > WAIT_LIMIT) {
                ok = false;
                break;
            }
        }
    }
    if (__syncthreads_or(!ok)) {
        if (tid == 0) {
            atomicOr(flag, 2);
            // the copy that did not arrive in time is waited for (bounded) before the CTA exits
            const unsigned bar = su32(&S.bar);
            const long long t0 = clock64();
            for (;;) {
                unsigned done;
                asm volatile(
                    "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, "
                    "p;\n}\n"
                    : "=r"(done)
                    : "r"(bar), "r"(0u)
                    : "memory");
                if (done || clock64() - t0 > WAIT_LIMIT) break;
            }
        }
        return;
    }
    if (!live) return;

    const int bx = tx + GX, by = ty + GY, bz = tz + GZ;
    T F[2][3];
    bool fixed = false;
    if constexpr (sizeof(T) == 8) fixed = C.fixed > 0 && __ldcg(flag + 1) == 0;
    force3<T, NS, sizeof(T) == 4 && MODE == K3_WRITE>(
        C, fixed, [&](int dx, int dy, int dz) { return S.box[0][bz + dz][by + dy][bx + dx]; },
        [&](int dx, int dy, int dz) { return S.box[1][bz + dz][by + dy][bx + dx]; }, F);
    if (sizeof(T) == 8) load();
    if constexpr (MODE == K3_LOOK)
        look3(C, F, S.box[1][bz][by][bx], ((long long)z * C.ny + y) * C.nx + x, jx, jy, jz, flag, fields);
    else if constexpr (MODE == K3_RELAX)
        relax3(C, M, F, S.box[1][bz][by][bx], i, jx, jy, jz, d, flag);
    else
        site3<T, NS, MODE>(C, f, F, x, y, z, i, fout, flag, fields);
}

// ---- equilibrium at rest, totals ---------------------------------------------------------------

template <typename T>
__global__ void k3_init(T* __restrict__ f, const double* __restrict__ rho, const Step3<T> C) {
    const long long n = (long long)C.nx * C.ny * C.nz;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(k % C.nx), y = (int)(k / C.nx % C.ny), z = (int)(k / ((long long)C.nx * C.ny));
        const long long i = ((long long)z * C.ny + y) * C.pitch + x;
        for (int s = 0; s < C.ns; ++s) {
            const double d = rho[s * n + k] - (double)C.rho_ref[s];
            for (int l = 0; l < 19; ++l) f[(s * 19 + l) * C.plane + i] = (T)(w19<double>(l) * d);
        }
    }
}

template <typename T, int MODE, int NS, int TY, int TZ>
cudaError_t launch_step3(const CUtensorMap& map, const T* fin, T* fout, const Step3<T>& C, int* flag, const Fields3& fields,
                         const Mom3& M, int dn, cudaStream_t st) {
    const size_t smem = sizeof(Smem3<T, TY, TZ>);
    static bool attr = false;  // per template instance
    if (!attr) {
        const cudaError_t e = cudaFuncSetAttribute(k3_step<T, MODE, NS, TY, TZ>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    constexpr int TX = Tile3<T>::TX;
    const dim3 grid((C.nx + TX - 1) / TX, (C.ny + TY - 1) / TY, (C.nz + TZ - 1) / TZ);
    return launch_pdl(k3_step<T, MODE, NS, TY, TZ>, grid, dim3(TX, TY, TZ), smem, st, map, fin, fout, C, flag, fields, M,
                      dn);
}

template <typename T, int MODE, int NS>
cudaError_t launch_shape(int shape, const CUtensorMap& map, const T* fin, T* fout, const Step3<T>& C, int* flag,
                         const Fields3& fields, const Mom3& M, int dn, cudaStream_t st) {
    switch (shape) {
        case 0: return launch_step3<T, MODE, NS, Tile3<T>::ty(0), Tile3<T>::tz(0)>(map, fin, fout, C, flag, fields, M, dn, st);
        case 1: return launch_step3<T, MODE, NS, Tile3<T>::ty(1), Tile3<T>::tz(1)>(map, fin, fout, C, flag, fields, M, dn, st);
        case 2: return launch_step3<T, MODE, NS, Tile3<T>::ty(2), Tile3<T>::tz(2)>(map, fin, fout, C, flag, fields, M, dn, st);
        case 3: return launch_step3<T, MODE, NS, Tile3<T>::ty(3), Tile3<T>::tz(3)>(map, fin, fout, C, flag, fields, M, dn, st);
        default: return cudaErrorInvalidValue;
    }
}

// the step pass in the chosen tile shape; the fields pass (lbm3_get_fields) in shape 0
template <typename T>
cudaError_t launch_step3_any(int mode, int ns, int shape, const CUtensorMap& map, const T* fin, T* fout,
                             const Step3<T>& C, int* flag, const Fields3& fields, const Mom3& M, int dn, cudaStream_t st) {
    if constexpr (sizeof(T) == 4) {
        if (mode == K3_RELAX) return launch_shape<T, K3_RELAX, 2>(shape, map, fin, fout, C, flag, fields, M, dn, st);
        if (mode == K3_LOOK)
            return launch_step3<T, K3_LOOK, 2, Tile3<T>::ty(0), Tile3<T>::tz(0)>(map, fin, fout, C, flag, fields, M, dn, st);
    }
    if (mode == K3_WRITE)
        return ns == 2 ? launch_shape<T, K3_WRITE, 2>(shape, map, fin, fout, C, flag, fields, M, dn, st)
                       : launch_shape<T, K3_WRITE, 1>(shape, map, fin, fout, C, flag, fields, M, dn, st);
    return ns == 2 ? launch_step3<T, K3_FIELDS, 2, Tile3<T>::ty(0), Tile3<T>::tz(0)>(map, fin, fout, C, flag, fields, M, dn, st)
                   : launch_step3<T, K3_FIELDS, 1, Tile3<T>::ty(0), Tile3<T>::tz(0)>(map, fin, fout, C, flag, fields, M, dn, st);
}

}  // namespace lbm3

// ---------------------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------------------
using namespace lbm3;

struct lbm3_ctx {
    lbm3_desc d{};
    lbm_params p{};
    bool have_params = false, have_fields = false;
    bool own_stream = false;
    cudaStream_t stream = nullptr;
    size_t esize = 4;
    int pitch = 0, gpitch = 0;
    long long plane = 0, gvol = 0, n = 0;
    void* f[2] = {nullptr, nullptr};
    int cur = 0;
    void* vol = nullptr;               // psi and rho volumes: [2][gz][gy][gpitch] pairs
    alignas(64) unsigned char map[NSHAPE][128] = {};  // TMA descriptors of vol, per tile shape
    int shape = 0;                     // tile shape of the step pass (lbm3_autotune)
    // FP32 at tau = 1: the state may be held as moments (Mom3), which live in f[cur ^ 1], and f[cur] is
    // stale; may_mom: this lattice does; mom: that is so now; dc: which copy of the densities is current; chunk: k3_stream's
    bool may_mom = false, mom = false;
    int dc = 0;
    int chunk = 1;
    int* flag = nullptr;               // [0] what lbm3_synchronize reports, [1] k3_density's odd
    double* staging = nullptr;         // lbm3_get_fields / lbm3_set_fields from the host
    size_t staging_bytes = 0;
    double* part = nullptr;            // the density pass's block partials of the totals
    double* tot = nullptr;             // lbm3_totals: the 5 totals on the device
    double* dcheck = nullptr;          // lbm3_set_fields: DCHECK_DOUBLES doubles (launch_density_check)
    int nblk_den = 0;                  // blocks of the density pass with totals
    int tot_grid[3] = {1, 1, 1};       // its grid
    double rho_ref[2] = {0.0, 0.0};
    Step3<float> c32{};
    Step3<double> c64{};
    bool profiling = false;
    std::vector<cudaEvent_t> ev;       // 4 per timed step
    size_t ev_used = 0;
    long long step = 0;
    cudaEvent_t tev[64] = {};          // lbm3_step_totals: an event per ticket (ring)
    long long tickets = 0;             // tickets issued
    std::string err;
};

static std::string g3_create_error;

static int fail3(lbm3_ctx* c, int code, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    if (c)
        c->err = buf;
    else
        g3_create_error = buf;
    return code;
}

#define CK3(call)                                                                                            \
    do {                                                                                                     \
        cudaError_t e_ = (call);                                                                             \
        if (e_ != cudaSuccess)                                                                               \
            return fail3(c, e_ == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA, "%s: %s (%s:%d)", #call, \
                         cudaGetErrorString(e_), __FILE__, __LINE__);                                        \
    } while (0)

template <typename T>
static void fill_step3(const lbm3_ctx* c, Step3<T>& C) {
    C = Step3<T>{};
    C.nx = c->d.nx;
    C.ny = c->d.ny;
    C.nz = c->d.nz;
    C.ns = c->d.n_species;
    C.zbc = c->d.z_boundary;
    C.psi_form = c->p.psi_form;
    C.pitch = c->pitch;
    C.gpitch = c->gpitch;
    C.plane = c->plane;
    C.gvol = c->gvol;
    C.gy = c->d.ny + 2 * GY;
    C.gz = c->d.nz + 2 * GZ;
    C.g = (T)c->p.body_force;
    C.wall_u[0] = (T)c->p.wall_u[0];
    C.wall_u[1] = (T)c->p.wall_u[1];
    const double wn = c->p.weight_norm;
    for (int s = 0; s < 2; ++s) {
        const bool on = s < c->d.n_species;
        const int ps = on ? s : 0;
        C.tau[s] = (T)c->p.tau[ps];
        C.omega[s] = (T)(1.0 / c->p.tau[ps]);
        C.rho0[s] = (T)c->p.rho0[ps];
        C.inv_rho0[s] = (T)(1.0 / c->p.rho0[ps]);
        C.rho_ref[s] = on ? (T)c->rho_ref[s] : T(0);
        for (int q = 0; q < 9; ++q)
            C.kq[s][q] = on ? (T)(wn * (c->p.G1[ps] * w_att3(q) + c->p.G2[ps] * w_rep3(q))) : T(0);
        if constexpr (sizeof(T) == 8) {
            C.ex[s] = lbm::exp_fx_const(c->p.psi_form == LBM_PSI_EXP ? c->p.rho0[ps] : 1.0);
            const double k[7] = {C.kq[s][1], C.kq[s][2], C.kq[s][3], C.kq[s][4], C.kq[s][5], C.kq[s][6], C.kq[s][8]};
            const bool kept = lbm::coef_fx(C.kf[s], k);
            if (c->p.psi_form == LBM_PSI_EXP) C.fixed = kept && C.fixed >= 0 ? 1 : -1;
        }
    }
    for (int q = 0; q < 3; ++q) C.kc[q] = c->d.n_species == 2 ? (T)(wn * c->p.G_AB * w_cross3(q)) : T(0);
}

static void refresh3(lbm3_ctx* c) {
    fill_step3<float>(c, c->c32);
    fill_step3<double>(c, c->c64);
}

extern "C" void lbm3_default_desc(lbm3_desc* d) {
    if (!d) return;
    *d = lbm3_desc{};
    d->nx = d->ny = d->nz = 64;
    d->n_species = 2;
    d->precision = LBM_FP32;
    d->z_boundary = LBM_PERIODIC;
}

static int check3(lbm3_ctx* c, const lbm3_desc* d) {
    if (!d) return fail3(c, LBM_EINVAL, "desc is NULL");
    if (d->nx < 1 || d->ny < 1 || d->nz < 1 || d->nx > 65536 || d->ny > 65535 || d->nz > 65535)
        return fail3(c, LBM_EINVAL, "nx, ny, nz must be >= 1 (nx <= 65536, ny, nz <= 65535)");
    if ((long long)d->nx * d->ny * d->nz > (1LL << 30)) return fail3(c, LBM_EINVAL, "nx * ny * nz > 2^30");
    if (d->n_species != 1 && d->n_species != 2) return fail3(c, LBM_EINVAL, "n_species must be 1 or 2");
    if (d->precision != LBM_FP32 && d->precision != LBM_FP64) return fail3(c, LBM_EINVAL, "bad precision");
    if (d->z_boundary != LBM_PERIODIC && d->z_boundary != LBM_BOUNCEBACK) return fail3(c, LBM_EINVAL, "bad z_boundary");
    if (d->device < 0) return fail3(c, LBM_EINVAL, "device < 0");
    return LBM_OK;
}

static void release3(lbm3_ctx* c) {
    for (int b = 0; b < 2; ++b) cudaFree(c->f[b]);
    cudaFree(c->vol);
    cudaFree(c->flag);
    cudaFree(c->staging);
    cudaFree(c->part);
    cudaFree(c->tot);
    cudaFree(c->dcheck);
    for (cudaEvent_t e : c->ev) cudaEventDestroy(e);
    for (cudaEvent_t e : c->tev)
        if (e) cudaEventDestroy(e);
    if (c->own_stream && c->stream) cudaStreamDestroy(c->stream);
}

static dim3 stream_grid3(const lbm3_ctx* c);

static int make_vol_map(lbm3_ctx* c, int shape) {
    const auto encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(lbm::tensor_map_encoder());
    if (!encode) return 1;
    const cuuint64_t es = c->esize;
    // dims: values of T along x (two per site), rows, layers, the two volumes
    const cuuint64_t dims[4] = {(cuuint64_t)2 * c->gpitch, (cuuint64_t)(c->d.ny + 2 * GY),
                                (cuuint64_t)(c->d.nz + 2 * GZ), 2};
    const cuuint64_t strides[3] = {(cuuint64_t)2 * c->gpitch * es, (cuuint64_t)2 * c->gpitch * (c->d.ny + 2 * GY) * es,
                                   (cuuint64_t)2 * c->gvol * es};
    const bool f32 = c->esize == 4;
    const int bx = f32 ? Tile3<float>::BX : Tile3<double>::BX;
    const int ty = f32 ? Tile3<float>::ty(shape) : Tile3<double>::ty(shape);
    const int tz = f32 ? Tile3<float>::tz(shape) : Tile3<double>::tz(shape);
    const cuuint32_t box[4] = {(cuuint32_t)(2 * bx), (cuuint32_t)(ty + 2 * GY), (cuuint32_t)(tz + 2 * GZ), 2};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUresult r = encode(reinterpret_cast<CUtensorMap*>(c->map[shape]),
                              c->esize == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 4,
                              c->vol, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                              CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? 0 : 2;
}

extern "C" int lbm3_create(lbm3_ctx** out, const lbm3_desc* d) {
    if (!out) return fail3(nullptr, LBM_EINVAL, "out is NULL");
    *out = nullptr;
    int rc = check3(nullptr, d);
    if (rc) return rc;
    lbm3_ctx* c = new (std::nothrow) lbm3_ctx();
    if (!c) return fail3(nullptr, LBM_ENOMEM, "host allocation failed");
    c->d = *d;
    lbm_default_params(&c->p);
    auto bail = [&](int code) {
        g3_create_error = c->err;
        release3(c);
        delete c;
        return code;
    };
#define CKC3(call)                                                                                       \
    do {                                                                                                 \
        cudaError_t e_ = (call);                                                                         \
        if (e_ != cudaSuccess)                                                                           \
            return bail(fail3(c, e_ == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA, "%s: %s", #call, \
                              cudaGetErrorString(e_)));                                                  \
    } while (0)
    CKC3(cudaSetDevice(d->device));
    if (d->stream) {
        c->stream = static_cast<cudaStream_t>(d->stream);
    } else {
        CKC3(cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking));
        c->own_stream = true;
    }
    const int nx = d->nx, ny = d->ny, nz = d->nz, ns = d->n_species;
    c->esize = d->precision == LBM_FP64 ? 8 : 4;
    c->pitch = (nx + 31) / 32 * 32;
    c->plane = (long long)nz * ny * c->pitch;
    c->gpitch = (nx + 2 * GX + 3) / 4 * 4;
    c->gvol = (long long)(nz + 2 * GZ) * (ny + 2 * GY) * c->gpitch;
    c->n = (long long)nx * ny * nz;
    const size_t fbytes = (size_t)ns * 19 * c->plane * c->esize;
    for (int b = 0; b < 2; ++b) {
        CKC3(cudaMalloc(&c->f[b], fbytes));
        CKC3(cudaMemsetAsync(c->f[b], 0, fbytes, c->stream));
    }
    const size_t vbytes = (size_t)2 * c->gvol * 2 * c->esize;
    CKC3(cudaMalloc(&c->vol, vbytes));
    CKC3(cudaMemsetAsync(c->vol, 0, vbytes, c->stream));
    CKC3(cudaMalloc(&c->flag, 2 * sizeof(int)));
    CKC3(cudaMemsetAsync(c->flag, 0, 2 * sizeof(int), c->stream));
    int nsm = 0;
    CKC3(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, d->device));
    {  // the density pass with totals: no more than the 8 CTAs that run on an SM, each looping over as many
       // rows (not one over two and the next over one); in FP64 also a CTA per row segment while those
       // are at most 16 per SM (FP32 there, 48^3: 963 us for 24 steps, 861 looping)
        const bool f32 = c->esize == 4;
        const int bx = f32 ? DensityBlock<float, true>::X : DensityBlock<double, true>::X;
        const int by = f32 ? DensityBlock<float, true>::Y : DensityBlock<double, true>::Y;
        const int gx = (nx + bx - 1) / bx, rows = (ny + by - 1) / by;
        const int target = !f32 && (long long)gx * rows * nz <= 16 * nsm ? 16 * nsm : 8 * nsm;
        int gy = std::max(1, std::min(rows, target / gx));
        int gz = std::max(1, std::min(nz, target / (gx * gy)));
        const int py = (rows + gy - 1) / gy, pz = (nz + gz - 1) / gz;
        gy = (rows + py - 1) / py;
        gz = (nz + pz - 1) / pz;
        c->tot_grid[0] = gx;
        c->tot_grid[1] = gy;
        c->tot_grid[2] = gz;
        c->nblk_den = gx * gy * gz;
    }
    // k3_stream: a block reads chunk + 2 layers, 4 blocks run on an SM: the chunk whose waves of
    // blocks read the fewest layers one after the other
    {
        const long long columns = (long long)((nx + 31) / 32) * ((ny + 3) / 4), slots = 4LL * nsm;
        long long best = -1;
        for (int k = 1; k <= 64; ++k) {
            const long long blocks = columns * ((nz + k - 1) / k), cost = (blocks + slots - 1) / slots * (k + 2);
            if (best < 0 || cost < best) best = cost, c->chunk = k;
        }
        // Which lattices are held as moments (a property of the lattice, so that the results' bits do not
        // depend on how a run is cut into calls).  One species: none, a pair's second half would be idle
        // (24 steps of 40^3 535 us as moments, 438 as populations; 128^3, 14 steps, 2,266 and 2,042).  Two:
        // all but those whose blocks of one layer are a little more than run at once, where two layers a
        // block leave a third of the slots empty and double its walk (24 steps of 36^3 533 and 508 us, 40^3
        // 543 and 505, 160 x 24 x 24 567 and 515; below, 33^3 496 and 505; above, 128 x 32 x 32 567 and 573,
        // 64^3 800 and 827, 96^3 1,823 and 2,374).
        const long long layers = columns * nz;
        c->may_mom = c->esize == 4 && ns == 2 && (layers <= slots || 2 * layers > 3 * slots);
    }
    const dim3 sg = stream_grid3(c);
    const size_t parts = std::max<size_t>(c->nblk_den, (size_t)sg.x * sg.y * sg.z);
    CKC3(cudaMalloc(&c->part, parts * 5 * sizeof(double)));
    CKC3(cudaMalloc(&c->tot, 5 * sizeof(double)));
    CKC3(cudaMalloc(&c->dcheck, lbm::DCHECK_DOUBLES * sizeof(double)));
    for (int k = 0; k < NSHAPE; ++k)
        if (make_vol_map(c, k) != 0)
            return bail(fail3(c, LBM_ECUDA, "cuTensorMapEncodeTiled failed for the psi / rho volumes"));
    CKC3(cudaStreamSynchronize(c->stream));
#undef CKC3
    refresh3(c);
    *out = c;
    return LBM_OK;
}

extern "C" void lbm3_destroy(lbm3_ctx* c) {
    if (!c) return;
    cudaSetDevice(c->d.device);
    if (c->stream) cudaStreamSynchronize(c->stream);
    release3(c);
    delete c;
}

extern "C" const char* lbm3_last_error(const lbm3_ctx* c) { return c ? c->err.c_str() : g3_create_error.c_str(); }

static cudaError_t expand3(lbm3_ctx* c, double* out = nullptr);

extern "C" int lbm3_set_params(lbm3_ctx* c, const lbm_params* p) {
    if (!c) return LBM_EINVAL;
    if (!p) return fail3(c, LBM_EINVAL, "params is NULL");
    if (lbm_validate_params(p, c->d.n_species) != LBM_OK)
        return fail3(c, LBM_EINVAL, "invalid parameters: %s", lbm_last_error(nullptr));
    if (p->weight_preset != LBM_WEIGHTS_PAPER) return fail3(c, LBM_EINVAL, "the 3-D step has the paper's weights only");
    if (p->psi_wall != LBM_WALL_MIRROR) return fail3(c, LBM_EINVAL, "the 3-D step has the mirror wall reading only");
    const lbm_params was = c->p;
    c->p = *p;
    c->have_params = true;
    // moments hold the state only under the relaxation times (all 1) and wall velocities it was formed
    // with (a population leaving through a wall is reflected by the step that sends it): under others
    // it goes on as the populations those give
    const bool keep = p->tau[0] == 1.0 && p->tau[1] == 1.0 &&
                      (c->d.z_boundary == LBM_PERIODIC || (p->wall_u[0] == was.wall_u[0] && p->wall_u[1] == was.wall_u[1]));
    if (c->mom && !keep) {
        CK3(cudaSetDevice(c->d.device));
        CK3(expand3(c));  // with the constants of the steps taken
        c->mom = false;
    }
    refresh3(c);
    return LBM_OK;
}

static int staging3(lbm3_ctx* c, size_t bytes) {
    if (c->staging_bytes >= bytes) return LBM_OK;
    cudaFree(c->staging);
    c->staging = nullptr;
    c->staging_bytes = 0;
    CK3(cudaMalloc(&c->staging, bytes));
    c->staging_bytes = bytes;
    return LBM_OK;
}

extern "C" int lbm3_set_fields(lbm3_ctx* c, const double* rho, int where) {
    if (!c) return LBM_EINVAL;
    if (!rho) return fail3(c, LBM_EINVAL, "rho is NULL");
    if (where != LBM_HOST && where != LBM_DEVICE) return fail3(c, LBM_EINVAL, "where must be LBM_HOST or LBM_DEVICE");
    if (!c->have_params) return fail3(c, LBM_EINVAL, "lbm3_set_params has not been called");
    CK3(cudaSetDevice(c->d.device));
    const int ns = c->d.n_species;
    const long long n = c->n;
    int rc = staging3(c, (size_t)ns * n * sizeof(double));
    if (rc) return rc;
    // the densities into the staging buffer, checked and summed there (the reference densities
    // need the sums on the host: one small read-back)
    CK3(cudaMemcpyAsync(c->staging, rho, (size_t)ns * n * sizeof(double),
                        where == LBM_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, c->stream));
    CK3(lbm::launch_density_check(c->staging, n, ns, c->dcheck, c->stream));
    double chk[3];
    CK3(cudaMemcpyAsync(chk, c->dcheck, sizeof chk, cudaMemcpyDeviceToHost, c->stream));
    CK3(cudaStreamSynchronize(c->stream));
    unsigned long long bad;
    memcpy(&bad, &chk[2], sizeof bad);
    if (bad != ~0ull) {
        double v = 0.0;
        CK3(cudaMemcpy(&v, c->staging + bad, sizeof v, cudaMemcpyDeviceToHost));
        return fail3(c, LBM_EINVAL, "rho must be > 0 and finite (rho[%d][%lld] = %g)", (int)(bad / n),
                     (long long)(bad % n), v);
    }
    for (int s = 0; s < 2; ++s)
        c->rho_ref[s] = c->d.precision == LBM_FP64 || s >= ns ? 0.0
                                                               : (c->p.rho_ref[s] >= 0.0 ? c->p.rho_ref[s] : chk[s] / n);
    refresh3(c);
    const int blocks = (int)std::min<long long>((n + 255) / 256, 4096);
    if (c->d.precision == LBM_FP64)
        lbm3::k3_init<double><<<blocks, 256, 0, c->stream>>>((double*)c->f[0], c->staging, c->c64);
    else
        lbm3::k3_init<float><<<blocks, 256, 0, c->stream>>>((float*)c->f[0], c->staging, c->c32);
    CK3(cudaGetLastError());
    CK3(cudaMemsetAsync(c->flag, 0, 2 * sizeof(int), c->stream));
    CK3(cudaStreamSynchronize(c->stream));
    c->cur = 0;
    c->mom = false;
    c->step = 0;
    c->have_fields = true;
    return LBM_OK;
}

// the density pass over f[cur] into the volumes; totals: its block partials of the totals of
// f[cur] summed into out (5 doubles, device memory) as well
static Mom3 moments3(const lbm3_ctx* c) {
    float* p = static_cast<float*>(c->f[c->cur ^ 1]);  // 15 planes of the 38
    const long long n = c->plane;
    Mom3 M;
    float2** pair[] = {&M.d[0], &M.d[1], &M.base, &M.ux, &M.uy, &M.uz};
    for (int k = 0; k < 6; ++k) *pair[k] = reinterpret_cast<float2*>(p + 2 * k * n);
    M.jx = p + 12 * n;
    M.jy = p + 13 * n;
    M.jz = p + 14 * n;
    return M;
}

// Whether a step relaxes every population fully to its equilibrium, on a lattice held as moments then.
static bool relaxed3(const lbm3_ctx* c) { return c->may_mom && c->c32.omega[0] == 1.0f && c->c32.omega[1] == 1.0f; }

static dim3 stream_grid3(const lbm3_ctx* c) {
    return dim3((c->d.nx + 31) / 32, (c->d.ny + 3) / 4, (c->d.nz + c->chunk - 1) / c->chunk);
}

// The populations of the state held as moments into f[cur], or (out) as plain values into the caller's
// device memory; the state stays what it is.
static cudaError_t expand3(lbm3_ctx* c, double* out) {
    const dim3 grid((c->d.nx + 127) / 128, c->d.ny, c->d.nz);
    const Mom3 M = moments3(c);
    float* const f = (float*)c->f[c->cur];
    if (out)
        k3_expand<double><<<grid, 128, 0, c->stream>>>(M, c->dc, out, c->c32);
    else
        k3_expand<float><<<grid, 128, 0, c->stream>>>(M, c->dc, f, c->c32);
    return cudaGetLastError();
}

// The density and momentum that stream into every site of a state held as moments (and psi and rho
// into the volumes), with the totals' partials.
static cudaError_t stream3(lbm3_ctx* c, bool totals) {
    const dim3 grid = stream_grid3(c), block(32, 4);
    const Mom3 M = moments3(c);
    float* vol = (float*)c->vol;
    return totals ? launch_pdl(k3_stream<true>, grid, block, 0, c->stream, M, c->dc, vol, c->c32, c->chunk, c->part)
                  : launch_pdl(k3_stream<false>, grid, block, 0, c->stream, M, c->dc, vol, c->c32, c->chunk,
                               (double*)nullptr);
}

// read: for a read of the state's densities only (no collision follows)
static cudaError_t density3(lbm3_ctx* c, double* totals = nullptr, bool read = false) {
    const dim3 grid = totals ? dim3(c->tot_grid[0], c->tot_grid[1], c->tot_grid[2])
                             : dim3((c->d.nx + 127) / 128, c->d.ny, c->d.nz);
    const dim3 block(128);
    cudaError_t e;
    if (c->d.precision == LBM_FP64)
        e = totals ? launch_pdl(lbm3::k3_density<double, true>, grid, block, 0, c->stream, (const double*)c->f[c->cur],
                                (double*)c->vol, c->c64, c->part, (float2*)nullptr, (float*)nullptr, c->flag + 1)
                   : launch_pdl(lbm3::k3_density<double, false>, grid, block, 0, c->stream,
                                (const double*)c->f[c->cur], (double*)c->vol, c->c64, (double*)nullptr,
                                (float2*)nullptr, (float*)nullptr, c->flag + 1);
    else if (c->mom && !read) {
        e = stream3(c, totals != nullptr);
    } else if (relaxed3(c) && !read) {  // populations, on the way to moments
        const Mom3 M = moments3(c);
        e = totals ? launch_pdl(lbm3::k3_density<float, true, true>, grid, block, 0, c->stream,
                                (const float*)c->f[c->cur], (float*)c->vol, c->c32, c->part, M.d[c->dc ^ 1], M.jx, (int*)nullptr)
                   : launch_pdl(lbm3::k3_density<float, false, true>, grid, block, 0, c->stream,
                                (const float*)c->f[c->cur], (float*)c->vol, c->c32, (double*)nullptr, M.d[c->dc ^ 1],
                                M.jx, (int*)nullptr);
    } else {
        e = totals ? launch_pdl(lbm3::k3_density<float, true>, grid, block, 0, c->stream, (const float*)c->f[c->cur],
                                (float*)c->vol, c->c32, c->part, (float2*)nullptr, (float*)nullptr, (int*)nullptr)
                   : launch_pdl(lbm3::k3_density<float, false>, grid, block, 0, c->stream, (const float*)c->f[c->cur],
                                (float*)c->vol, c->c32, (double*)nullptr, (float2*)nullptr, (float*)nullptr, (int*)nullptr);
    }
    if (e != cudaSuccess || !totals) return e;
    const dim3 sg = stream_grid3(c);
    const int nblk = c->mom && !read ? (int)(sg.x * sg.y * sg.z) : c->nblk_den;
    // the reference densities the FP32 deviations are taken from (zero in FP64, and for an absent
    // species), once per site
    const double n = (double)c->n;
    const double r0 = c->d.precision == LBM_FP64 ? 0.0 : (double)c->c32.rho_ref[0];
    const double r1 = c->d.precision == LBM_FP64 ? 0.0 : (double)c->c32.rho_ref[1];
    return launch_pdl(lbm3::k3_totals_sum, dim3(1), dim3(320), 0, c->stream, (const double*)c->part, nblk, n * r0, n * r1,
                      totals);
}

// The collide pass of a step (K3_WRITE, after density3: it makes the new state the current one), or
// K3_FIELDS.
static cudaError_t collide3(lbm3_ctx* c, int mode, const Fields3& fields = Fields3{}) {
    const bool relax = mode == K3_WRITE && relaxed3(c);
    const int shape = mode == K3_WRITE ? c->shape : 0;
    const CUtensorMap& map = *reinterpret_cast<const CUtensorMap*>(c->map[shape]);
    cudaError_t e;
    if (c->d.precision == LBM_FP64)
        e = launch_step3_any<double>(mode, c->d.n_species, shape, map, (const double*)c->f[c->cur],
                                     (double*)c->f[c->cur ^ 1], c->c64, c->flag, fields, Mom3{}, 0, c->stream);
    else
        e = launch_step3_any<float>(relax ? K3_RELAX : mode, c->d.n_species, shape, map, (const float*)c->f[c->cur],
                                    (float*)c->f[c->cur ^ 1], c->c32, c->flag, fields, moments3(c), c->dc ^ 1,
                                    c->stream);
    if (e == cudaSuccess && mode == K3_WRITE) {
        if (relax) {
            c->mom = true;
            c->dc ^= 1;
        } else {
            c->cur ^= 1;
        }
    }
    return e;
}

// one step: the density pass and the collide pass (bracketed by events while profiling)
static int one_step3(lbm3_ctx* c) {
    cudaEvent_t* e = nullptr;
    if (c->profiling) {
        if (c->ev_used + 4 > c->ev.size())
            for (int q = 0; q < 64; ++q) {
                cudaEvent_t ev;
                CK3(cudaEventCreate(&ev));
                c->ev.push_back(ev);
            }
        e = &c->ev[c->ev_used];
        c->ev_used += 4;
        CK3(cudaEventRecord(e[0], c->stream));
    }
    CK3(density3(c));
    if (e) {
        CK3(cudaEventRecord(e[1], c->stream));
        CK3(cudaEventRecord(e[2], c->stream));
    }
    CK3(collide3(c, K3_WRITE));
    if (e) CK3(cudaEventRecord(e[3], c->stream));
    c->step += 1;
    return LBM_OK;
}

extern "C" int lbm3_step(lbm3_ctx* c, int nsteps) {
    if (!c || nsteps < 0) return c ? fail3(c, LBM_EINVAL, "nsteps < 0") : LBM_EINVAL;
    if (!c->have_fields) return fail3(c, LBM_EINVAL, "lbm3_set_fields has not been called");
    CK3(cudaSetDevice(c->d.device));
    for (int k = 0; k < nsteps; ++k) {
        const int rc = one_step3(c);
        if (rc != LBM_OK) return rc;
    }
    return LBM_OK;
}

extern "C" int lbm3_step_totals(lbm3_ctx* c, int nsteps, double* dst, long long stride, long long* ticket) {
    if (!c) return LBM_EINVAL;
    if (nsteps < 0) return fail3(c, LBM_EINVAL, "nsteps < 0");
    if (!dst && nsteps > 0) return fail3(c, LBM_EINVAL, "dst is NULL");
    if (stride < 5 * (long long)sizeof(double) || stride % (long long)sizeof(double))
        return fail3(c, LBM_EINVAL, "stride must be a multiple of 8 bytes and at least 40");
    if (!c->have_fields) return fail3(c, LBM_EINVAL, "lbm3_set_fields has not been called");
    CK3(cudaSetDevice(c->d.device));
    // the kernels write the records themselves: device memory, or pinned host memory through its
    // device address
    double* out = nullptr;
    if (nsteps > 0) {
        cudaPointerAttributes pa{};
        const cudaError_t e = cudaPointerGetAttributes(&pa, dst);
        cudaGetLastError();  // an unregistered pointer may leave an error behind
        if (e == cudaSuccess && pa.type == cudaMemoryTypeDevice)
            out = dst;
        else if (e == cudaSuccess && pa.type == cudaMemoryTypeHost && pa.devicePointer)
            out = static_cast<double*>(pa.devicePointer);
        else
            return fail3(c, LBM_EINVAL, "dst must be device memory or pinned host memory");
    }
    // after each collide pass, the density pass of the next step forms the totals of the new state
    // too (so the populations are read once per step for both); the first step needs its own
    for (int k = 0; k < nsteps; ++k) {
        if (k == 0) CK3(density3(c));
        CK3(collide3(c, K3_WRITE));
        c->step += 1;
        CK3(density3(c, out + (long long)k * (stride / (long long)sizeof(double))));
    }
    if (nsteps > 0) {  // one event for the run: its last record
        cudaEvent_t& e = c->tev[c->tickets % 64];
        if (!e) CK3(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
        CK3(cudaEventRecord(e, c->stream));
        if (ticket) *ticket = c->tickets;
        c->tickets += 1;
    }
    return LBM_OK;
}

extern "C" int lbm3_wait(lbm3_ctx* c, long long ticket) {
    if (!c) return LBM_EINVAL;
    if (ticket < 0 || ticket >= c->tickets) return fail3(c, LBM_EINVAL, "ticket %lld was not issued", ticket);
    CK3(cudaSetDevice(c->d.device));
    if (ticket < c->tickets - 64)
        CK3(cudaStreamSynchronize(c->stream));  // its event was reused: wait for everything
    else
        CK3(cudaEventSynchronize(c->tev[ticket % 64]));
    return LBM_OK;
}

extern "C" int lbm3_synchronize(lbm3_ctx* c) {
    if (!c) return LBM_EINVAL;
    CK3(cudaSetDevice(c->d.device));
    CK3(cudaStreamSynchronize(c->stream));
    int flag = 0;
    CK3(cudaMemcpy(&flag, c->flag, sizeof(int), cudaMemcpyDeviceToHost));
    if (flag & 2) return fail3(c, LBM_ETIMEOUT, "a bounded device-side wait for a tile load gave up");
    if (flag & 1) return fail3(c, LBM_ENONFINITE, "a step met a density <= 0, NaN or Inf");
    return LBM_OK;
}

// Whether a kernel may write doubles at p: null, or aligned device memory of the context's device.
static bool writable3(const lbm3_ctx* c, const void* p) {
    if (!p) return true;
    cudaPointerAttributes a{};
    const cudaError_t e = cudaPointerGetAttributes(&a, p);
    cudaGetLastError();  // an unknown pointer may leave an error behind
    return e == cudaSuccess && a.type == cudaMemoryTypeDevice && a.device == c->d.device &&
           reinterpret_cast<size_t>(p) % sizeof(double) == 0;
}

extern "C" int lbm3_get_fields(lbm3_ctx* c, double* rho, double* u, double* f, int where) {
    if (!c) return LBM_EINVAL;
    if (where != LBM_HOST && where != LBM_DEVICE) return fail3(c, LBM_EINVAL, "where must be LBM_HOST or LBM_DEVICE");
    if (!c->have_fields) return fail3(c, LBM_EINVAL, "lbm3_set_fields has not been called");
    CK3(cudaSetDevice(c->d.device));
    const int ns = c->d.n_species;
    const long long n = c->n;
    // straight into the caller's device memory, or through the staging buffer (host memory, and
    // pointers that a kernel may not write)
    const size_t nrho = (size_t)ns * n, nu = (size_t)3 * n, nf = (size_t)19 * ns * n;
    Fields3 at{rho, u, f};
    const bool direct = where == LBM_DEVICE && writable3(c, rho) && writable3(c, u) && writable3(c, f);
    if (!direct) {
        const int rc = staging3(c, ((rho ? nrho : 0) + (u ? nu : 0) + (f ? nf : 0)) * sizeof(double));
        if (rc) return rc;
        double* p = c->staging;
        if (rho) at.rho = p, p += nrho;
        if (u) at.u = p, p += nu;
        if (f) at.f = p;
    }
    if (c->mom) {  // held as moments: no populations but those asked for; the densities are always looked at
        if (at.f) CK3(expand3(c, at.f));
        CK3(density3(c));
        CK3(collide3(c, K3_LOOK, at));
    } else {
        CK3(density3(c, nullptr, true));
        CK3(collide3(c, K3_FIELDS, at));
    }
    if (!direct) {
        const cudaMemcpyKind kind = where == LBM_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
        if (rho) CK3(cudaMemcpyAsync(rho, at.rho, nrho * sizeof(double), kind, c->stream));
        if (u) CK3(cudaMemcpyAsync(u, at.u, nu * sizeof(double), kind, c->stream));
        if (f) CK3(cudaMemcpyAsync(f, at.f, nf * sizeof(double), kind, c->stream));
    }
    return lbm3_synchronize(c);
}

extern "C" int lbm3_totals(lbm3_ctx* c, double* mass, double* momentum) {
    if (!c) return LBM_EINVAL;
    if (!c->have_fields) return fail3(c, LBM_EINVAL, "lbm3_set_fields has not been called");
    CK3(cudaSetDevice(c->d.device));
    CK3(density3(c, c->tot));  // the density pass with the totals of f[cur]
    double t[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    CK3(cudaMemcpyAsync(t, c->tot, sizeof t, cudaMemcpyDeviceToHost, c->stream));
    const int rc = lbm3_synchronize(c);
    if (rc) return rc;
    if (mass)
        for (int s = 0; s < c->d.n_species; ++s) mass[s] = t[s];
    if (momentum)
        for (int q = 0; q < 3; ++q) momentum[q] = t[2 + q];
    return LBM_OK;
}

extern "C" int lbm3_profile(lbm3_ctx* c, int enable) {
    if (!c) return LBM_EINVAL;
    CK3(cudaSetDevice(c->d.device));
    CK3(cudaStreamSynchronize(c->stream));
    c->profiling = enable != 0;
    c->ev_used = 0;
    return LBM_OK;
}

extern "C" int lbm3_profile_read(lbm3_ctx* c, double* ms, long long* steps) {
    if (!c) return LBM_EINVAL;
    CK3(cudaSetDevice(c->d.device));
    CK3(cudaStreamSynchronize(c->stream));
    double t[2] = {0.0, 0.0};
    for (size_t k = 0; k + 3 < c->ev_used; k += 4)
        for (int j = 0; j < 2; ++j) {
            float v = 0.f;
            CK3(cudaEventElapsedTime(&v, c->ev[k + 2 * j], c->ev[k + 2 * j + 1]));
            t[j] += v;
        }
    if (ms) {
        ms[0] = t[0];
        ms[1] = t[1];
    }
    if (steps) *steps = (long long)(c->ev_used / 4);
    return LBM_OK;
}

extern "C" int lbm3_autotune(lbm3_ctx* c, int steps, int* chosen, double* ms) {
    if (!c) return LBM_EINVAL;
    if (steps < 1 || steps > 10000) return fail3(c, LBM_EINVAL, "steps must be in 1 .. 10000");
    if (!c->have_fields) return fail3(c, LBM_EINVAL, "lbm3_set_fields has not been called");
    CK3(cudaSetDevice(c->d.device));
    // the state is kept aside and put back: the shapes change the schedule, not the arithmetic (held as
    // moments it is 15 planes of the other buffer)
    const int cur0 = c->cur, shape0 = c->shape, dc0 = c->dc;
    const bool mom0 = c->mom;
    void* const at = c->f[mom0 ? cur0 ^ 1 : cur0];
    const size_t fbytes = (mom0 ? (size_t)15 : (size_t)c->d.n_species * 19) * c->plane * c->esize;
    void* saved = nullptr;
    CK3(cudaMalloc(&saved, fbytes));
    cudaError_t e = cudaMemcpyAsync(saved, at, fbytes, cudaMemcpyDeviceToDevice, c->stream);
    const long long step0 = c->step;
    cudaEvent_t a = nullptr, b = nullptr;
    if (e == cudaSuccess) e = cudaEventCreate(&a);
    if (e == cudaSuccess) e = cudaEventCreate(&b);
    double t[NSHAPE] = {0.0, 0.0, 0.0, 0.0};
    int best = 0;
    for (int k = 0; k < NSHAPE && e == cudaSuccess; ++k) {
        c->shape = k;
        e = density3(c);  // one untimed step (module load, caches)
        if (e == cudaSuccess) e = collide3(c, K3_WRITE);
        if (e == cudaSuccess) e = cudaEventRecord(a, c->stream);
        for (int i = 0; i < steps && e == cudaSuccess; ++i) {
            e = density3(c);
            if (e == cudaSuccess) e = collide3(c, K3_WRITE);
        }
        if (e == cudaSuccess) e = cudaEventRecord(b, c->stream);
        if (e == cudaSuccess) e = cudaEventSynchronize(b);
        float v = 0.f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&v, a, b);
        t[k] = (double)v / steps;
        if (t[k] < t[best]) best = k;
        c->cur = cur0;
        c->mom = mom0;
        c->dc = dc0;
        if (e == cudaSuccess) e = cudaMemcpyAsync(at, saved, fbytes, cudaMemcpyDeviceToDevice, c->stream);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (a) cudaEventDestroy(a);
    if (b) cudaEventDestroy(b);
    cudaFree(saved);
    c->cur = cur0;
    c->mom = mom0;
    c->dc = dc0;
    c->step = step0;
    c->shape = e == cudaSuccess ? best : shape0;
    CK3(e);
    CK3(cudaMemsetAsync(c->flag, 0, 2 * sizeof(int), c->stream));
    if (chosen) *chosen = best;
    if (ms)
        for (int k = 0; k < NSHAPE; ++k) ms[k] = t[k];
    return LBM_OK;
}

extern "C" int lbm3_set_shape(lbm3_ctx* c, int shape) {
    if (!c) return LBM_EINVAL;
    if (shape < 0 || shape >= NSHAPE) return fail3(c, LBM_EINVAL, "shape must be in 0 .. %d", NSHAPE - 1);
    c->shape = shape;
    return LBM_OK;
}
