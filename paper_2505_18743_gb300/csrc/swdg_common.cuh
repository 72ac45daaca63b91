// swdg_common.cuh -- device data structures and warp helpers of the sm_103a
// sub-grid DG shallow-water hot path (arXiv 2505.18743).
//
// Layout in HBM (one context):
//   state   U[buf][field][cell][(r+1)^2]  float64, field = zeta, qx, qy, c
//   cmask   [buf][cell] uint8: bit f set when field f is constant on the cell
//           (such a field is evaluated as that constant, exactly)
//   resid   R[stage][6][cell][(r+1)^2] float64, 6 = F, Gx, Gy, R, Lx, Ly
//   tiles   [cell][P][P] float32|float64 bathymetry depth (mode S)
//   zpts    [cell][NV^2 + NM^2 + NG^2] float64: point samples (mode P) or
//           sub-cell mean depths sum_k w_k z_k (mode S)
// Small per-degree tables (1D interpolation matrices, quadrature weights) lie in
// device memory (Dev::tabs) and are copied to shared memory by the blocks that
// index them by lane; rarely run kernels take them as a parameter.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "swdg_fixed.cuh"

namespace swdg {

constexpr int MXP = 6;    // max quadrature points per direction (GL 5 for r = 3)
constexpr int MXN = 4;    // max nodes per direction (r + 1)
constexpr int MXPIX = 32; // max pixels per cell side in mode S
constexpr int MXTAG = 16;
constexpr int MXS = 4;    // max RK stages
constexpr int NBUF = 4;   // state buffers: v^n plus stages 2..4

// point sets
constexpr int SET_VOL = 0;  // volume Gauss-Legendre, floor(3r/2)+1 per direction
constexpr int SET_MASS = 1; // face / mass Gauss-Lobatto, r+2 per direction
constexpr int SET_MOM = 2;  // momentum mass Gauss-Legendre, r+1 per direction
constexpr int SET_HALF = 3; // coarse side of a 2:1 face: the GLL sub-intervals of each
                            // fine half face, h NM + al, in coarse coordinates
constexpr int NSET = 4;
constexpr int MXI = 2 * MXP; // max sub-intervals per set
constexpr int MXCLS = 4;     // max distinct pixel counts per cell side

// face info byte of a cell's face: FI_COARSE = this cell is the coarse side of
// a 2:1 face (two fine neighbours); FI_FINE | half << 2 = this cell is one of
// the two fine cells (half 0: lower tangential half of the coarse face)
constexpr int FI_COARSE = 1;
constexpr int FI_FINE = 2;

// pixel-overlap fractions of the sub-intervals of the four point sets for
// one pixel count P per cell side
struct OvTab {
    int P;
    int lo[NSET][MXI], cnt[NSET][MXI];
    double frac[NSET][MXI][MXPIX + 1];
    // the fractions of the first, the inner (all equal) and the last pixel as
    // digit pairs (swdg_fixed.cuh), exponent 0
    int2 ed[NSET][MXI][3];
};

// status bits
constexpr int ST_NAN = 1;

template <int R>
struct Sz {
    static constexpr int ND1 = R + 1, ND = ND1 * ND1;
    static constexpr int NV = (3 * R) / 2 + 1, NVP = NV * NV;
    static constexpr int NM = R + 2, NMP = NM * NM;
    static constexpr int NG = R + 1, NGP = NG * NG;
    static constexpr int NZP = NVP + NMP + NGP; // mode P samples per cell
};

// the basis tables as digit pairs (swdg_fixed.cuh), each with the exponent t*
// that bounds its rows' absolute sums; test tables are stored by node, and the
// volume ones carry the quadrature weight
struct FxTables {
    int2 Bv[MXP][MXN], Dv[MXP][MXN];                 // nodal -> volume (value, d/dxi)
    int2 WB[MXN][MXP], WD[MXN][MXP], WDB[MXN][MXP];  // wv Bv, wv Dv; wv Bv at the scale of wv Dv
    int2 BmT[MXN][MXP], BmHT[2][MXN][MXP];           // face test tables, one scale
    int tBv, tDv, tWB, tWD, tBmT;
};

// what the stage update and its adjoint take from the tables: digit pairs of
// the mass- and momentum-point contractions and of the inverse 1D matrices,
// with the plain weights and the FP32 basis
struct FxStage {
    int2 Bm[MXP][MXN], BmT[MXN][MXP]; // nodal -> mass points, its transpose
    int2 Bg[MXN][MXN], BgT[MXN][MXN]; // nodal -> momentum points, its transpose
    int2 Gi[MXN][MXN], GiT[MXN][MXN]; // inverse of Bg, its transpose
    int2 M1i[MXN][MXN];               // inverse 1D mass matrix
    double wm[MXP], wg[MXP], wn[MXN]; // wn: the nodes' weights in the momentum rule
    // the mass matrices' FP32 assembly: node scales 1 / |B_a| (2-norm over the
    // mass points, per direction) and products of the scaled basis, [pair][point]
    // with pair (a, c), c <= a, at a (a + 1) / 2 + c
    float sc[MXN], BB[MXN * (MXN + 1) / 2][MXP];
    int tBm, tBmT, tBg, tBgT, tGi, tGiT, tM1i, pad_;
};

// the face points' basis: nodal -> face GLL points, and those of half h of a
// 2:1 face (FP64 and FP32)
struct FaceTables {
    double Bm[MXP][MXN], BmH[2][MXP][MXN], wm[MXP];
    float BmF[MXP][MXN], BmHF[2][MXP][MXN];
};

// the basis tables in FP64, and the FP32 copies of the FP32-bulk kernels
struct BaseTables {
    double Bv[MXP][MXN], Dv[MXP][MXN], wv[MXP]; // nodal -> volume GL (value, d/dxi)
    double Bm[MXP][MXN], wm[MXP];               // nodal -> mass / face GLL
    double Bg[MXP][MXN], wg[MXP];               // nodal -> momentum GL (square)
    double Bginv[MXN][MXP];                     // inverse of Bg
    double M1inv[MXN][MXN];                     // inverse of the 1D GLL mass matrix
    double BmH[2][MXP][MXN];                    // nodal -> fine-face GLL points of half h
    float BvF[MXP][MXN], DvF[MXP][MXN], BmF[MXP][MXN], BmHF[2][MXP][MXN], BgF[MXP][MXN];
    float BginvF[MXN][MXP];
    float wvF[MXP];                             // volume GL weights (FP32-bulk residual)
    float wgF[MXP];                             // momentum GL weights (FP32-bulk stage update)
    double xs[MXN];                             // support nodes on [0, 1]
    double xq[3][MXP];                          // nodes of the three point sets on [0, 1]
};
struct Tables : BaseTables {
    FxTables fx;
    FxStage fs;
    FaceTables ft;
};

// clock of one ensemble member (a plain context is an ensemble of one)
struct Member {
    double t;                 // time at the start of the current step
    double dt_last;
    unsigned long long rmax;  // bits of max lambda l_Gamma / J_K over the member (non-negative double)
    double pad_;
};

// boundary table of one member: kind (SWDG_BC_*) and tide of every tag
struct Bc {
    int kind[MXTAG];
    double amp[MXTAG], per[MXTAG], ph[MXTAG];
};

struct Scalars {
    Member m0;                // the clock of a single-member context
    double fixed_dt;          // >= 0: fixed step, < 0: CFL
    int maxits, viol, fallback, status;
};

struct Dev {
    int64_t n;
    const Tables* tabs; // the tables in device memory (the kernels' copies to shared memory)
    const double* x0y0;
    const double* hxhy;
    const double* ihxhy; // 1/hx, 1/hy per cell (null: computed in the kernel)
    const int32_t* nbr;
    const void* tiles;
    const int64_t* tile_off; // first pixel of each cell's tile (null: k P^2)
    const uint8_t* pcls;     // pixel-count class of each cell (null: class 0)
    const OvTab* ov;         // overlap tables per class
    const uint8_t* finfo;    // [cell][4] face info (null: all conforming)
    const double* zhang;     // [cell][4][2][NM]: coarse-side strip means / samples
    const double* zpts;
    const double* zmax; // dry-start level of Eq. initial_guess (max z_b of the cell)
    const double* zmin; // min z_b of the cell: every pixel is wet when eta > -zmin
    const double* zabs; // max |z_b| of the cell (Newton tolerance scale)
    // [cell][NZP] (min, max) of the pixel depths of each sub-cell of the three
    // point sets (mode S; min rounded down, max up); null: the cell's bounds
    const float2* zsb;
    const double* manning;
    const double* nu_c; // tracer numerical diffusivity per cell (Eq. numdiff); null: none
    double* U;
    // FP32 copy of U in the same layout (FP32-bulk contexts; null otherwise),
    // written wherever U and its masks are written (k_masks, the step start,
    // the stage update), read by the FP32 face and residual arithmetic
    float* uF;
    uint8_t* cmask;
    double* res;
    double* llin;
    double* HN;
    double* CN;
    double* HNbar;
    double* CNbar;
    uint8_t* flag;
    // 1 where every mass point of the cell was fully wet at zeta^n (written by
    // the step start with H(zeta^n); null: unknown)
    uint8_t* wet0;
    // [cell][2][(r+1)^2]: qx, qy of v^n at the momentum points, written by the
    // step start (the same for every stage of the step; FP64 contexts); null:
    // interpolated by the stage update itself
    double* qpts;
    Scalars* sc;
    Member* mb;            // member clocks [nmemb] (a single member: &sc->m0)
    const int32_t* memb;   // member of each cell (null: every cell in member 0)
    const Bc* mbc;         // per-member boundary tables (null: the tables below)
    int nmemb;
    int mode; // 0 S, 1 P
    int s;    // stages
    double g, eps, hlim, eps0, cfl, newton_tol;
    double sg; // sqrt(g)
    int newton_max;
    int any_friction;
    int bc_kind[MXTAG];
    double bc_amp[MXTAG], bc_per[MXTAG], bc_ph[MXTAG];
    double a[MXS][MXS], at[MXS][MXS], b[MXS], bt[MXS], c[MXS];
    // face points evaluated once by k_faces (null fflux: the residual
    // integrates its faces itself)
    double* fflux;        // [cell][4 fields][4 faces][2 halves][NM]
    const int64_t* fjobs; // k << 8 | f | h << 2 | al << 3, k the lower index of the face
    int64_t njobs;
};

// ---------------------------------------------------------------------------
// warp helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_min(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
// sums over a team of TL lanes (the whole warp, or one of its two halves;
// tm = the team's lanes); for TL = 32 the same order as warp_sum
template <int TL>
__device__ __forceinline__ double team_sum(double v, unsigned tm) {
#pragma unroll
    for (int o = TL / 2; o > 0; o >>= 1) v += __shfl_xor_sync(tm, v, o);
    return v;
}
// two team sums at once, each bit for bit the team_sum of its value: the first
// level of the butterfly sums a on the team's lower half and b on its upper
// half (one addition per lane for both), the other levels run on both halves
// together, and a last exchange gives every lane both results.  Each level
// adds the same pairs as team_sum (addition commutes), so the tree is the
// same; the FP64 additions halve.  Teams are aligned groups of TL lanes.
template <int TL>
__device__ __forceinline__ void team_sum2(double& a, double& b, unsigned tm) {
    const bool hi = (threadIdx.x & (TL / 2)) != 0;
    double v = (hi ? b : a) + __shfl_xor_sync(tm, hi ? a : b, TL / 2);
#pragma unroll
    for (int o = TL / 4; o > 0; o >>= 1) v += __shfl_xor_sync(tm, v, o);
    const double w = __shfl_xor_sync(tm, v, TL / 2);
    a = hi ? w : v;
    b = hi ? v : w;
}
// maximum over the team of an order-preserving key (okey)
template <int TL>
__device__ __forceinline__ long long team_max_key(long long v, unsigned tm) {
#pragma unroll
    for (int o = TL / 2; o > 0; o >>= 1) {
        const long long w = __shfl_xor_sync(tm, v, o);
        v = w > v ? w : v;
    }
    return v;
}
// maxima of non-negative values (no NaN) over the team's lanes tm by their bit
// patterns, which order like the values: integer reductions, off the FP64 pipe
__device__ __forceinline__ float team_max_nonneg(float v, unsigned tm) {
    return __uint_as_float(__reduce_max_sync(tm, __float_as_uint(v)));
}
__device__ __forceinline__ double team_max_nonneg(double v, unsigned tm) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
    const unsigned mh = __reduce_max_sync(tm, hi);
    const unsigned ml = __reduce_max_sync(tm, hi == mh ? lo : 0u);
    return __longlong_as_double((long long)(((unsigned long long)mh << 32) | ml));
}
// equality and finiteness of doubles tested on their bit patterns, on the
// integer pipe (FP64 compares take the FP64 pipe).  same_bits differs from ==
// only for +0 against -0 and for NaN: a constant-field mask may treat those
// either way, since a field marked non-constant takes the general path.
__device__ __forceinline__ bool same_bits(double a, double b) {
    return __double_as_longlong(a) == __double_as_longlong(b);
}
__device__ __forceinline__ bool finite_bits(double v) {
    constexpr long long EXP = 0x7ff0000000000000ll;
    return (__double_as_longlong(v) & EXP) != EXP;
}
// v == 0.0 (either sign) on the bit pattern
__device__ __forceinline__ bool zero_bits(double v) {
    return (__double_as_longlong(v) << 1) == 0;
}
// Order-preserving integer key of a double that is not NaN: a > b exactly when
// okey(a) > okey(b), except that -0 keys below +0 (negative doubles have their
// non-sign bits flipped, so they order as negative integers).
__device__ __forceinline__ long long okey(double v) {
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double of_okey(long long b) {
    return __longlong_as_double(b ^ ((b >> 63) & 0x7fffffffffffffffll));
}
// the key of -z for a threshold -z, with -0 taken as +0, so that
// okey(eta) > nkey_neg(z) is exactly eta > -z for every eta that is not NaN
// (for eta = +-0 and -z = -0 both are false)
__device__ __forceinline__ long long nkey_neg(double z) {
    long long b = __double_as_longlong(z) ^ (long long)0x8000000000000000ull;
    if (b == (long long)0x8000000000000000ull) b = 0;
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ bool nan_bits(double v) {
    return (__double_as_longlong(v) & 0x7fffffffffffffffll) > 0x7ff0000000000000ll;
}
__device__ __forceinline__ double* ufield(const Dev& d, int buf, int f, int nd) {
    return d.U + ((size_t)buf * 4 + f) * (size_t)d.n * nd;
}
__device__ __forceinline__ float* ufieldF(const Dev& d, int buf, int f, int nd) {
    return d.uF + ((size_t)buf * 4 + f) * (size_t)d.n * nd;
}
__device__ __forceinline__ double* rfield(const Dev& d, int stage, int f, int nd) {
    return d.res + ((size_t)stage * 6 + f) * (size_t)d.n * nd;
}

// a block's copy of a table (or part of one) in shared memory, from device
// memory: the kernel's parameter bank would serialise the lanes' reads
template <typename T>
__device__ __forceinline__ void copy_table(T& dst, const T* __restrict__ src) {
    static_assert(sizeof(T) % 8 == 0, "8-byte words");
    for (int i = threadIdx.x; i < (int)(sizeof(T) / 8); i += blockDim.x)
        ((unsigned long long*)&dst)[i] = ((const unsigned long long*)src)[i];
    __syncthreads();
}

__device__ __forceinline__ int member_of(const Dev& d, int64_t k) {
    return d.memb ? d.memb[k] : 0;
}

__device__ __forceinline__ double get_dt(const Dev& d, int m) {
    // dt = cfl min J/(lambda l) = cfl / max(lambda l / J) over the member's
    // cells, Eq. deltat_fe
    return d.sc->fixed_dt >= 0.0 ? d.sc->fixed_dt : d.cfl / __longlong_as_double(d.mb[m].rmax);
}

// FP32 value of a positive double in the FP32 normal range and the double of a
// positive FP32 normal, by bit patterns on the integer pipe (conversions run
// on the FP64 pipe: 9 and 17 clocks per warp against 1-2); the first truncates
__device__ __forceinline__ bool f32_range(double x) {
    const unsigned h = (unsigned)__double2hiint(x);
    return h - 0x39e00000u < 0x46000000u - 0x39e00000u; // 2^-97 <= x < 2^97
}
__device__ __forceinline__ float f32_trunc(double x) {
    const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
    return __uint_as_float(((h - 0x38000000u) << 3) | (l >> 29));
}
// the nearest FP32 value of any double (ties to even, as a conversion rounds), the
// same way; outside the FP32 normal range by conversion
__device__ __forceinline__ float f32_of(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned h = (unsigned)(b >> 32) & 0x7fffffffu;
    if (h - 0x38100000u < 0x47e00000u - 0x38100000u) {
        const unsigned m = (unsigned)(((b & 0x7fffffffffffffffull) + 0xfffffffull +
                                       ((b >> 29) & 1ull)) >> 29);
        return __uint_as_float((m - 0xc0000000u) | ((unsigned)(b >> 32) & 0x80000000u));
    }
    return b << 1 ? (float)x : 0.0f;
}
__device__ __forceinline__ double f64_of(float v) {
    const unsigned b = __float_as_uint(v);
    return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}

// x^(-1/3) of a positive double: an FP32 reciprocal-cube-root seed (~2^-22)
// refined by one third-order (Halley) step for z^-3 = x in FP64,
// z (1 + e/3 + 2/9 e^2), e = 1 - x z^3 (no division).  Values outside the FP32
// seed's comfortable range take 1 / cbrt(x).
__device__ __noinline__ inline double inv_cbrt_any(double x) { return 1.0 / cbrt(x); }
__device__ __noinline__ inline double sqrt_any(double x) { return sqrt(x); }
__device__ __forceinline__ double inv_cbrt(double x) {
    if (!f32_range(x)) return inv_cbrt_any(x);
    const double z = f64_of(rcbrtf(f32_trunc(x)));
    const double e = fma(-x, z * z * z, 1.0);
    return fma(fma(e, 2.0 / 9.0, 1.0 / 3.0), z * e, z);
}

// sqrt(x), x >= 0, in five FP64 instructions (CUDA's takes nine): the same kind
// of step from an FP32 seed y of x^(-1/2), x y (1 + e/2 + 3/8 e^2),
// e = 1 - x y^2 (within 1 ulp).  Values outside the FP32 seed's comfortable
// range, 0 and NaN among them, take sqrt itself.
__device__ __forceinline__ double sqrt_fast(double x) {
    if (!f32_range(x)) return zero_bits(x) ? 0.0 : sqrt_any(x);
    const double y = f64_of(rsqrtf(f32_trunc(x)));
    const double t = x * y, e = fma(-t, y, 1.0);
    return fma(t * e, fma(e, 0.375, 0.5), t);
}

// 1/h and sqrt(g h) of a wet depth (h >= eps) from one root y = h^(-1/2): an
// FP32 seed (~2^-22) and one third-order (Halley) step y (1 + e/2 + 3/8 e^2),
// e = 1 - h y^2; then 1/h = y^2 with one Newton correction.  Ten FP64
// instructions where a division and a square root take fifteen.
__device__ __forceinline__ void inv_and_wave(double h, double g, double sg, double& rh, double& cw) {
    if (!f32_range(h)) {
        rh = 1.0 / h;
        cw = sqrt(g * h);
        return;
    }
    const double y0 = f64_of(rsqrtf(f32_trunc(h)));
    const double e = fma(-(h * y0), y0, 1.0);
    const double y = fma(fma(e, 0.375, 0.5), y0 * e, y0);
    const double y2 = y * y;
    rh = fma(fma(-h, y2, 1.0), y2, y2);
    cw = sg * (h * y);
}

// desingularised velocity factor u = f q, Eq. velocity (T = double or float)
template <typename T>
__device__ __forceinline__ T vel_factor(T h, T eps) {
    if (h <= T(0)) return T(0);
    if (h >= eps) return T(1) / h; // max(h^4, eps^4) = h^4: sqrt(2) h / sqrt(2 h^4) = 1/h
    T h4 = (h * h) * (h * h), e4 = (eps * eps) * (eps * eps);
    return sqrt(T(2)) * h / sqrt(e4 + h4);
}
// Manning coefficient gamma = g n^2 |q| / h_des^(7/3), Eqs. manning, discharge_rhs_implicit
template <typename T>
__device__ __forceinline__ T gamma_manning(T n, T h, T qx, T qy, T g, T eps) {
    if (n == T(0) || h <= T(0)) return T(0);
    T hdes = h; // h_des = h when h >= eps
    if (h < eps) {
        T h4 = (h * h) * (h * h), e4 = (eps * eps) * (eps * eps);
        hdes = sqrt(e4 + h4) / (sqrt(T(2)) * h);
    }
    if constexpr (std::is_same<T, double>::value) {
        // h_des^(-7/3) = z^7 with z = h_des^(-1/3): no division, no cbrt
        const double z = inv_cbrt(hdes), z3 = z * z * z;
        return g * n * n * sqrt(qx * qx + qy * qy) * (z3 * z3 * z);
    } else {
        return g * n * n * sqrt(qx * qx + qy * qy) / (hdes * hdes * cbrt(hdes));
    }
}

// the velocity factor of one point and, with friction, |q| h_des^(-7/3) (the
// Manning coefficient without g n^2), in FP64
// (h < eps, or no friction: rare, not inlined)
struct VelGam {
    double fv, gm;
};
__device__ __noinline__ inline VelGam vel_friction_any(double h, double qx, double qy, bool friction,
                                                       double eps) {
    if (h >= eps) return {1.0 / h, 0.0};
    return {vel_factor<double>(h, eps), friction ? gamma_manning<double>(1.0, h, qx, qy, 1.0, eps) : 0.0};
}
__device__ __forceinline__ void vel_friction(double h, double qx, double qy, bool friction, double eps,
                                             double& fv, double& gm) {
    // h >= eps on the bit patterns (h is not negative, eps > 0; a NaN depth stays
    // on this branch), off the FP64 pipe
    if (friction && __double_as_longlong(h) >= __double_as_longlong(eps)) {
        // 1/h = z^3 from z = h^(-1/3) (a few ulp from the rounded quotient, no
        // FP64 division); h^(-7/3) = z^7
        const double z = inv_cbrt(h), rh = z * z * z;
        fv = rh;
        gm = sqrt_fast(qx * qx + qy * qy) * (rh * rh) * z;
    } else {
        const VelGam r = vel_friction_any(h, qx, qy, friction, eps);
        fv = r.fv;
        gm = r.gm;
    }
}

// sub-grid wet depth V and wet area A of sub-cell (ia, ib) of point sets setx,
// sety (mode S): V = sum_k w_k max(eta + z_k, 0), A = sum_k w_k [eta + z_k > 0]
struct SubV {
    double V, A;
    bool full;
};
// in FP64
template <typename Pix>
__device__ __forceinline__ SubV subgrid_f64(const Pix* __restrict__ tile, const OvTab& ov, int setx,
                                            int ia, int sety, int ib, double eta) {
    const int P = ov.P;
    const int lox = ov.lo[setx][ia], cx = ov.cnt[setx][ia];
    const int loy = ov.lo[sety][ib], cy = ov.cnt[sety][ib];
    double v = 0.0, a = 0.0;
    bool f = true;
    for (int j = 0; j < cy; ++j) {
        const Pix* row = tile + (size_t)(loy + j) * P + lox;
        double vr = 0.0, ar = 0.0;
        for (int i = 0; i < cx; ++i) {
            double dd = eta + (double)row[i];
            if (dd > 0.0) {
                double fx = ov.frac[setx][ia][i];
                vr += fx * dd;
                ar += fx;
            } else {
                f = false;
            }
        }
        double fy = ov.frac[sety][ib][j];
        v += fy * vr;
        a += fy * ar;
    }
    return {v, a, f};
}

// a pixel is wet (eta + z > 0, that is z > -eta) exactly: against the largest FP32
// value up to -eta, or by order-preserving keys; a NaN pixel is dry
struct WetF {
    float t;
    __device__ __forceinline__ WetF(double eta) { t = __double2float_rd(-eta); }
    __device__ __forceinline__ bool operator()(float z) const { return z > t; }
};
struct WetD {
    unsigned long long t, span; // wet: the key is in (-eta, inf], as one comparison
    __device__ __forceinline__ WetD(double eta) {
        t = (unsigned long long)nkey_neg(eta) + 1;
        span = 0x7ff0000000000001ull - t;
    }
    __device__ __forceinline__ bool operator()(double z) const {
        return (unsigned long long)okey(z) - t < span;
    }
};
template <typename Pix>
using Wet = std::conditional_t<std::is_same<Pix, float>::value, WetF, WetD>;
// the larger of two depths (a NaN z: m), and a bound of one in FP32
__device__ __forceinline__ float deeper(float m, float z) { return z > m ? z : m; }
__device__ __forceinline__ double deeper(double m, double z) { return okey(z) > okey(m) && !nan_bits(z) ? z : m; }
__device__ __forceinline__ float bound_f(float z) { return z; }
__device__ __forceinline__ float bound_f(double z) { return __double2float_ru(z); }
template <typename Pix>
__device__ __noinline__ Pix deepest(const Pix* __restrict__ t, int P, int cx, int cy) {
    Pix m = (Pix)-INFINITY;
#pragma unroll 1
    for (int j = 0; j < cy; ++j, t += P)
#pragma unroll 1
        for (int i = 0; i < cx; ++i) m = deeper(m, t[i]);
    return m;
}
// a sub-cell with depths past FP32's range (rare: not inlined)
template <typename Pix>
__device__ __noinline__ SubV subgrid_inf(const Pix* __restrict__ tile, const OvTab* __restrict__ ov, int setx,
                                         int ia, int sety, int ib, double eta) {
    return subgrid_f64<Pix>(tile, *ov, setx, ia, sety, ib, eta);
}
__device__ __forceinline__ long long fx_pixel(float z, int e) { return fx::from_float(z, e); }
__device__ __forceinline__ long long fx_pixel(double z, int e) { return fx::from_double(z, e); }

// The same with the pixels summed as integers (swdg_fixed.cuh): in FP64 a pixel costs
// five instructions of the FP64 pipe (80 clocks per warp), here about 15 of the
// integer pipe, and the weights enter once per row, since w_k = fy fx with fx
// equal for all but the first and last pixel of a row.
// zhi is a bound of the sub-cell's pixel depths (NaN: found here).  A wet pixel lies
// between -eta and zhi, so the block exponent is that of the larger of the two, and
// dry pixels, however high, have no part in it.  With room for the sum of a row
// (cx <= 2^lg pixels), eta and the wet pixels keep 2^-(58 - lg) of it: exactly what
// they are where eta + z cancels, and below the rounding of eta + z where it does
// not.  The rows' sums are then moved up to the bound eta + zhi of a pixel's depth, so
// that a film of water at a great height, or beside a deep cell, has its own
// relative accuracy (59 places of cx times that bound).  Not inlined: most cells never
// get here, and the callers' code stays small.  Measured, a step of the lagoon (r = 2,
// 8 to 32 pixels a side): 3543 us with FP64 pixel sums, 2104 with integers; without the
// move up 10 us less, and with a branch around the conversion of a dry pixel 150 more.
template <typename Pix>
__device__ __noinline__ SubV subgrid_S(const Pix* __restrict__ tile, const OvTab* __restrict__ ov,
                                       int setx, int ia, int sety, int ib, double eta, float zhi) {
    const int P = ov->P;
    const int lox = ov->lo[setx][ia], cx = ov->cnt[setx][ia];
    const int loy = ov->lo[sety][ib], cy = ov->cnt[sety][ib];
    if (fx::mag(eta) >= 0x7ff00000u) { // an infinity or a NaN reads as entirely wet or dry
        const bool wet = eta > 0.0;
        return {wet ? eta : 0.0, wet ? 1.0 : 0.0, wet};
    }
    const Wet<Pix> is_wet(eta);
    const int lg = 32 - __clz(cx - 1); // ceil(log2(cx))
    int es;
    long long E, D1;
    // the block of a bound, and the bound of a pixel's depth in it
    auto block = [&]() {
        es = max(fx::block_exp(fx::mag(eta)), fx::block_exp_f(__float_as_uint(zhi) & 0x7fffffffu)) + lg + 2;
        E = fx::from_double(eta, es);
        D1 = E + fx::from_float(zhi, es);
    };
    const bool given = zhi == zhi;
    if (given) block();
    // no bound, or (FP64 pixels) one that its rounding to FP32 may leave far above the depths
    if (!given || (sizeof(Pix) == sizeof(double) && D1 < 1ll << 36)) {
        const Pix m = deepest<Pix>(tile + loy * P + lox, P, cx, cy);
        if (!is_wet(m)) return {0.0, 0.0, false};
        zhi = bound_f(m);
        block();
        if (sizeof(Pix) == sizeof(double)) D1 = E + fx_pixel(m, es);
    }
    if (fx::fbits(zhi) == 0x7f800000u) return subgrid_inf<Pix>(tile, ov, setx, ia, sety, ib, eta);
    const int up = D1 > 0 ? fx::clz64((unsigned long long)D1) - (64 - fx::FB) - lg : 0;
    fx::Acc v, a;
    int wet = 0;
#pragma unroll 1
    for (int j = 0; j < cy; ++j) {
        const Pix* row = tile + (loy + j) * P + lox;
        // the row's sum, its first and its last pixel (0 where it has only one)
        // (a dry pixel's integer means nothing; it is selected out, without a branch)
        const long long D0 = E + fx_pixel(row[0], es);
        const int cf = is_wet(row[0]);
        const long long first = cf ? D0 : 0;
        long long T = first, last = 0;
        int c = cf, cl = 0;
#pragma unroll 2
        for (int i = 1; i < cx; ++i) {
            const Pix z = row[i];
            const long long D = E + fx_pixel(z, es);
            cl = is_wet(z);
            last = cl ? D : 0;
            T += last;
            c += cl;
        }
        wet += c;
        const int2 f0 = ov->ed[setx][ia][0], f1 = ov->ed[setx][ia][1], f2 = ov->ed[setx][ia][2];
        const int2 fy = ov->ed[sety][ib][j == 0 ? 0 : j == cy - 1 ? 2 : 1];
        fx::Acc r;
        r.mac(f0, fx::split(first << up));
        r.mac(f1, fx::split((T - first - last) << up));
        r.mac(f2, fx::split(last << up));
        v.mac(fy, fx::split(r.get()));
        // the row's wet width, exactly (at most 1)
        a.mac(fy, fx::split((cf ? fx::join(f0) : 0) + (cl ? fx::join(f2) : 0) + (c - cf - cl) * fx::join(f1)));
    }
    const bool full = wet == cx * cy;
    const long long X = v.get(); // a wet pixel of less than a place may have rounded below 0
    return {fx::to_double(X > 0 ? X : 0, es - up),
            full ? 1.0 : wet ? fx::to_double(a.get(), 1022) : 0.0, full};
}

__device__ __forceinline__ void subgrid_P(double z, double eta, double& V, double& A) {
    double dd = eta + z;
    if (dd > 0.0) { V = dd; A = 1.0; }
    else { V = 0.0; A = 0.0; }
}

} // namespace swdg
