// swdg_kernels.cuh -- sm_103a kernels of the sub-grid DG shallow-water hot
// path (arXiv 2505.18743): residual (Sec. 3.2), degree switch (Eq.
// criteria_p), stage update (Sec. 3.1) and auxiliary reductions.
//
// Mapping: one cell per team of 8, 16 or 32 lanes, a launch-time number of warps
// per block (1..8), grid-stride over cells; one launch covers every member of an
// ensemble.  Each team stages its cell in shared memory and evaluates the
// tensor-product operators by sum factorisation (1D contractions, in block fixed
// point), one quadrature point or degree of freedom per lane; the face points
// are one per lane over the whole mesh (k_faces).
#pragma once
#include "swdg_common.cuh"

#include <utility>

namespace swdg {

constexpr int WPB = 4;    // default warps per block
constexpr int MAXWPB = 8; // largest block the kernels are compiled for

// ---------------------------------------------------------------------------
// small tensor contractions on a warp (all arrays in shared memory, x fastest)
// ---------------------------------------------------------------------------
// out[q1 NO + q0] = sum_b B[q1][b] sum_a B[q0][a] in[b NI + a]
template <int NI, int NO, typename T = double, int TL = 32>
__device__ __forceinline__ void tens_interp(const T (*B)[MXN], const T* in, T* tmp, T* out,
                                            int lane, unsigned tm = 0xffffffffu) {
    for (int i = lane; i < NI * NO; i += TL) {
        int b = i / NO, q0 = i % NO;
        T s = T(0);
#pragma unroll
        for (int a = 0; a < NI; ++a) s += B[q0][a] * in[b * NI + a];
        tmp[i] = s;
    }
    __syncwarp(tm);
    for (int i = lane; i < NO * NO; i += TL) {
        int q1 = i / NO, q0 = i % NO;
        T s = T(0);
#pragma unroll
        for (int b = 0; b < NI; ++b) s += B[q1][b] * tmp[b * NO + q0];
        out[i] = s;
    }
    __syncwarp(tm);
}

// out[b NI + a] = sum_q1 B[q1][b] sum_q0 B[q0][a] in[q1 NO + q0]   (transpose)
template <int NI, int NO, typename T = double, int TL = 32>
__device__ __forceinline__ void tens_test(const T (*B)[MXN], const T* in, T* tmp, T* out,
                                          int lane, unsigned tm = 0xffffffffu) {
    for (int i = lane; i < NO * NI; i += TL) {
        int q1 = i / NI, a = i % NI;
        T s = T(0);
#pragma unroll
        for (int q0 = 0; q0 < NO; ++q0) s += B[q0][a] * in[q1 * NO + q0];
        tmp[i] = s;
    }
    __syncwarp(tm);
    for (int i = lane; i < NI * NI; i += TL) {
        int b = i / NI, a = i % NI;
        T s = T(0);
#pragma unroll
        for (int q1 = 0; q1 < NO; ++q1) s += B[q1][b] * tmp[q1 * NI + a];
        out[i] = s;
    }
    __syncwarp(tm);
}

// out[b N + a] = scale * sum_d C(b,d) sum_c C(a,c) in[d N + c], C(i,j) = T ? M[j][i] : M[i][j]
template <int N, bool T, int LD, typename E = double, int TL = 32>
__device__ __forceinline__ void kron_apply(const E (*M)[LD], const E* in, E* tmp, E* out, E scale,
                                           int lane, unsigned tm = 0xffffffffu) {
    for (int i = lane; i < N * N; i += TL) {
        int d = i / N, a = i % N;
        E s = E(0);
#pragma unroll
        for (int c = 0; c < N; ++c) s += (T ? M[c][a] : M[a][c]) * in[d * N + c];
        tmp[i] = s;
    }
    __syncwarp(tm);
    for (int i = lane; i < N * N; i += TL) {
        int b = i / N, a = i % N;
        E s = E(0);
#pragma unroll
        for (int d = 0; d < N; ++d) s += (T ? M[d][b] : M[b][d]) * tmp[d * N + a];
        out[i] = scale * s;
    }
    __syncwarp(tm);
}

// The same contractions in block fixed point (swdg_fixed.cuh): T (NO x NI, by
// rows) applied along both directions of NI x NI digit pairs; f(it, i, X) takes
// the result at output i = q1 NO + q0 = lane + it TL, whose exponent is the
// input's plus twice the table's.  tmp: NI NO digit pairs.
template <int NI, int NO, int TL, int LD, typename F>
__device__ __forceinline__ void fx_tens(const int2 (*T)[LD], const int2* in, int2* tmp, int lane,
                                        unsigned tm, F f) {
    constexpr int M1 = NI * NO, M2 = NO * NO;
#pragma unroll
    for (int it = 0; it < (M1 + TL - 1) / TL; ++it) {
        const int i = lane + it * TL, b = i / NO, q0 = i % NO;
        if (i < M1) {
            fx::Acc s;
#pragma unroll
            for (int a = 0; a < NI; ++a) s.mac(T[q0][a], in[b * NI + a]);
            tmp[i] = fx::split(s.get());
        }
    }
    __syncwarp(tm);
#pragma unroll
    for (int it = 0; it < (M2 + TL - 1) / TL; ++it) {
        const int i = lane + it * TL, q1 = i / NO, q0 = i % NO;
        if (i < M2) {
            fx::Acc s;
#pragma unroll
            for (int b = 0; b < NI; ++b) s.mac(T[q1][b], tmp[b * NO + q0]);
            f(it, i, s.get());
        }
    }
}
// the block exponent of one value per lane of a team
__device__ __forceinline__ int team_exp(double v, unsigned tm) {
    return fx::block_exp(__reduce_max_sync(tm, fx::mag(v)));
}

// ---------------------------------------------------------------------------
// bathymetry sampling sites
// ---------------------------------------------------------------------------
// FX: partly wet sub-cells sum their pixels in fixed point (subgrid_S), else in FP64
// (subgrid_f64: the FP32-bulk path, the diagnostics and the refinement indicator)
template <int R, typename Pix, int MODE, bool FX = true>
struct Site {
    using S = Sz<R>;
    // zhi: a bound of the sub-cell's pixel depths (NaN: unknown)
    static __device__ __forceinline__ SubV pixels(const Dev& d, int64_t k, int setx, int ia, int sety,
                                                  int ib, double eta, float zhi) {
        const OvTab& o = tab(d, k);
        if constexpr (FX) return subgrid_S<Pix>(tile(d, o, k), &o, setx, ia, sety, ib, eta, zhi);
        else return subgrid_f64<Pix>(tile(d, o, k), o, setx, ia, sety, ib, eta);
    }
    static __device__ __forceinline__ int offset(int set) {
        return set == SET_VOL ? 0 : (set == SET_MASS ? S::NVP : S::NVP + S::NMP);
    }
    static __device__ __forceinline__ int count(int set) {
        return set == SET_VOL ? S::NV : (set == SET_MASS ? S::NM : S::NG);
    }
    static __device__ __forceinline__ const OvTab& tab(const Dev& d, int64_t k) {
        return d.ov[d.pcls ? d.pcls[k] : 0];
    }
    static __device__ __forceinline__ const Pix* tile(const Dev& d, const OvTab& o, int64_t k) {
        return (const Pix*)d.tiles + (d.tile_off ? d.tile_off[k] : (int64_t)k * o.P * o.P);
    }
    // mode S: a cell entirely wet (eta > -min z_b) gives V = eta + the sub-cell
    // mean depth and A = 1; entirely dry (eta <= -max z_b) gives V = A = 0;
    // otherwise the pixels are summed.  The per-cell bounds are optional (the
    // allocation-free residual has none): without them every sub-cell sums.
    // The two tests run on order-preserving integer keys (integer pipe); they
    // decide exactly as eta > -zmin and !(eta > -zmax), a NaN eta reading as
    // dry as under IEEE comparisons.
    static __device__ __forceinline__ bool shortcut(const Dev& d, int64_t k, double eta,
                                                    double zbar, double& V, double& A, bool& full) {
        if (d.zmin == nullptr) return false;
        return shortcut_b(eta, d.zmin[k], d.zmax[k], zbar, V, A, full);
    }
    // the same tests against the bounds zlo <= z_k <= zhi of a set of pixels
    static __device__ __forceinline__ bool shortcut_b(double eta, double zlo, double zhi,
                                                      double zbar, double& V, double& A,
                                                      bool& full) {
        const bool nan = nan_bits(eta);
        const long long ek = okey(eta);
        if (!nan && ek > nkey_neg(zlo)) {
            V = eta + zbar;
            A = 1.0;
            full = true;
            return true;
        }
        if (nan || !(ek > nkey_neg(zhi))) {
            V = 0.0;
            A = 0.0;
            full = false;
            return true;
        }
        return false;
    }
    // V, A of sub-cell (ia, ib) of point set `set` of cell k at elevation eta,
    // and whether every pixel of it is wet
    static __device__ __forceinline__ void VA(const Dev& d, const Tables& tb, int64_t k, int set,
                                              int ia, int ib, double eta, double& V, double& A,
                                              bool& full) {
        if (MODE == 0) {
            float zhi = NAN;
            if (d.zmin != nullptr) {
                const size_t ip = (size_t)k * S::NZP + offset(set) + ia + count(set) * ib;
                const double zbar = d.zpts[ip];
                // the cell's depth bounds first (one value per cell, cached); where
                // the waterline crosses the cell, the sub-cell's own bounds, so that
                // only the sub-cells it crosses sum their pixels
                if (shortcut_b(eta, d.zmin[k], d.zmax[k], zbar, V, A, full)) return;
                if (d.zsb != nullptr) {
                    const float2 b = d.zsb[ip];
                    if (shortcut_b(eta, (double)b.x, (double)b.y, zbar, V, A, full)) return;
                    zhi = b.y;
                }
            }
            const SubV r = pixels(d, k, set, ia, set, ib, eta, zhi);
            V = r.V;
            A = r.A;
            full = r.full;
        } else {
            subgrid_P(d.zpts[(size_t)k * S::NZP + offset(set) + ia + count(set) * ib], eta, V, A);
            full = A > 0.0;
        }
    }
    static __device__ __forceinline__ void VA(const Dev& d, const Tables& tb, int64_t k, int set,
                                              int ia, int ib, double eta, double& V, double& A) {
        bool full;
        VA(d, tb, k, set, ia, ib, eta, V, A, full);
    }
    // the strip of the coarse cell k on its face f under GLL point al of the
    // fine half face h (a 2:1 face): normal extent = its first/last mass
    // sub-interval, tangential extent = the fine point's sub-interval
    static __device__ __forceinline__ void VA_half(const Dev& d, int64_t k, int f, int h, int al,
                                                   double eta, double& V, double& A) {
        const double zh = d.zhang[(((size_t)k * 4 + f) * 2 + h) * S::NM + al];
        if (MODE == 0) {
            bool full;
            if (shortcut(d, k, eta, zh, V, A, full)) return;
            const int m = (f == 0 || f == 2) ? 0 : S::NM - 1, t = h * S::NM + al;
            const SubV r = pixels(d, k, f < 2 ? SET_MASS : SET_HALF, f < 2 ? m : t,
                                  f < 2 ? SET_HALF : SET_MASS, f < 2 ? t : m, eta, NAN);
            V = r.V;
            A = r.A;
        } else {
            subgrid_P(zh, eta, V, A);
        }
    }
};

// mass-point index of the strip of face f at face point al
template <int NM>
__device__ __forceinline__ void face_site_index(int f, int al, int& ia, int& ib) {
    if (f == 0) { ia = 0; ib = al; }
    else if (f == 1) { ia = NM - 1; ib = al; }
    else if (f == 2) { ia = al; ib = 0; }
    else { ia = al; ib = NM - 1; }
}
// node index (a + ND1 b) of the j-th node along face f
template <int ND1>
__device__ __forceinline__ int face_node(int f, int j) {
    if (f == 0) return ND1 * j;
    if (f == 1) return (ND1 - 1) + ND1 * j;
    if (f == 2) return j;
    return j + ND1 * (ND1 - 1);
}

// the four fields of a cell at face point al of face f: sum_j B[al][j] u(node(f, j));
// fields are fstride apart; a field constant on the cell is that constant
template <int ND1>
__device__ __forceinline__ void face_trace(const double* u, size_t fstride, unsigned cm, int f,
                                           const double (*B)[MXN], int al, double t[4]) {
#pragma unroll
    for (int fl = 0; fl < 4; ++fl) {
        const double* uf = u + fl * fstride;
        if (cm & (1u << fl)) {
            t[fl] = uf[0];
            continue;
        }
        double s = 0.0;
#pragma unroll
        for (int j = 0; j < ND1; ++j) s += B[al][j] * uf[face_node<ND1>(f, j)];
        t[fl] = s;
    }
}

__device__ __forceinline__ void atomic_max_pos(unsigned long long* addr, double v) {
    // non-negative doubles order like their bit patterns
    atomicMax(addr, (unsigned long long)__double_as_longlong(v));
}

// ---------------------------------------------------------------------------
// residual: volume terms on the volume Gauss-Legendre points, face terms on
// r+2 Gauss-Lobatto points per face (Eqs. mass_rhs, discharge_rhs,
// discharge_rhs_implicit, r_concentration)
// ---------------------------------------------------------------------------
// One face point (Sec. 3.2) in FP64: the Rusanov flux with the hydrostatic
// reconstruction at GLL point al of half h of face f of cell k, in the face's own
// frame: faces are axis-aligned, so the fluxes have an axis and a tangential component, normals are signs (applied to
// the sign bit) and one evaluation serves interior and boundary points.  flux =
// {F, G axis, G tangential, R} outward from side A (the lower cell index), pr
// the pressure vector's axis component g {{h*}} (h*A - h*B)/2 n_A, lam the wave
// speed bound.  uk: the cell's fields, ustride apart; Bm, BmH: the face basis.
__device__ __forceinline__ double flip(double v, unsigned sign) { // sign: 0 or 0x80000000
    return __hiloint2double(__double2hiint(v) ^ (int)sign, __double2loint(v));
}
// the smaller of two depths, on the bit patterns (they are not negative)
__device__ __forceinline__ double min_nonneg(double a, double b) {
    return __double_as_longlong(a) < __double_as_longlong(b) ? a : b;
}
// velocity factor and wave speed sqrt(g h) of a depth, as vel_factor below eps
__device__ __forceinline__ void vel_wave(double h, double g, double sg, double eps, double& f, double& w) {
    if (__double_as_longlong(h) >= __double_as_longlong(eps)) {
        inv_and_wave(h, g, sg, f, w);
    } else {
        f = vel_factor<double>(h, eps);
        w = h > 0.0 ? sqrt(g * h) : 0.0;
    }
}
// a side's wave speed bound as an integer that orders like it; a side whose velocity
// is NaN leaves the bound to the other one (as under fmax), both give a NaN
__device__ __forceinline__ long long wave_key(double l, double ut) {
    return nan_bits(l) || nan_bits(ut) ? -1 : __double_as_longlong(l);
}
struct FaceFlux {
    double flux[4], pr, lam;
    bool own_first, bnd;
    int64_t nb;
};
template <int ND1>
__device__ __forceinline__ void face_trace_axis(const double* u, size_t fstride, unsigned cm, int f,
                                                const double* B, double t[4]) {
    const int base = f == 1 ? ND1 - 1 : f == 3 ? ND1 * (ND1 - 1) : 0, st = f < 2 ? ND1 : 1;
    double b[ND1];
#pragma unroll
    for (int j = 0; j < ND1; ++j) b[j] = B[j];
#pragma unroll
    for (int fl = 0; fl < 4; ++fl) {
        const double* uf = u + fl * fstride + base;
        double s = 0.0;
#pragma unroll
        for (int j = 0; j < ND1; ++j) s += b[j] * uf[j * st];
        t[fl] = (cm & (1u << fl)) ? uf[0] : s;
    }
}
template <int R, typename Pix, int MODE>
__device__ __forceinline__ FaceFlux face_flux(const Dev& d, const FaceTables& ft, int64_t k,
                                              const double* uk, size_t ustride, unsigned cm, int buf,
                                              int f, int h, int al, unsigned info, int mem,
                                              double c_stage) {
    using S = Sz<R>;
    using ST = Site<R, Pix, MODE>;
    constexpr int ND1 = S::ND1, ND = S::ND, NM = S::NM;
    const int64_t n = d.n;
    const bool coarse = (info & 3) == FI_COARSE, fine = (info & 3) == FI_FINE;
    const int half = (int)(info >> 2), ax = f >> 1;
    FaceFlux out;
    const int32_t s0 = d.nbr[k * 8 + f * 2];
    out.bnd = s0 < 0;
    // a boundary's ghost takes the own cell's sub-grid operator
    const int64_t nb = out.bnd ? k : coarse && h ? (int64_t)d.nbr[k * 8 + f * 2 + 1] : (int64_t)s0;
    const int fo = out.bnd ? f : f ^ 1;
    out.nb = out.bnd ? -1 : nb;
    out.own_first = out.bnd || k < nb;
    double tm[4], tp[4];
    face_trace_axis<ND1>(uk, ustride, cm, f, coarse ? ft.BmH[h][al] : ft.Bm[al], tm);
    if (!out.bnd) {
        face_trace_axis<ND1>(ufield(d, buf, 0, ND) + nb * ND, (size_t)n * ND,
                             d.cmask[(size_t)buf * n + nb], fo, fine ? ft.BmH[half][al] : ft.Bm[al], tp);
    } else {
        const int tag = -1 - s0;
#pragma unroll
        for (int fl = 0; fl < 4; ++fl) tp[fl] = tm[fl];
        const bool tide = d.mbc ? d.mbc[mem].kind[tag] == 1 : d.bc_kind[tag] == 1;
        if (tide) {
            const double t = (c_stage == 0.0) ? d.mb[mem].t : d.mb[mem].t + c_stage * get_dt(d, mem);
            const double amp = d.mbc ? d.mbc[mem].amp[tag] : d.bc_amp[tag];
            const double per = d.mbc ? d.mbc[mem].per[tag] : d.bc_per[tag];
            const double ph = d.mbc ? d.mbc[mem].ph[tag] : d.bc_ph[tag];
            tp[0] = amp * sin(2.0 * M_PI * t / per + ph);
        } else { // mirrored: the normal discharge changes sign
            if (ax == 0) tp[1] = -tm[1];
            else tp[2] = -tm[2];
        }
    }
    // the sub-grid depths of both sides at both elevations, side by side in a loop
    // (one copy of the sampling code): hm, hp each side's own, hx V+(zeta-),
    // hy V-(zeta+)
    double hm = 0.0, hp = 0.0, hx = 0.0, hy = 0.0;
#pragma unroll 1
    for (int s = 0; s < (out.bnd ? 1 : 2); ++s) {
        const int64_t kc = s ? nb : k;
        const int fc = s ? fo : f;
        double Vm, Vp, A;
        if (s ? fine : coarse) {
            ST::VA_half(d, kc, fc, s ? half : h, al, tm[0], Vm, A);
            ST::VA_half(d, kc, fc, s ? half : h, al, tp[0], Vp, A);
        } else {
            int ia, ib;
            face_site_index<NM>(fc, al, ia, ib);
            ST::VA(d, *d.tabs, kc, SET_MASS, ia, ib, tm[0], Vm, A);
            ST::VA(d, *d.tabs, kc, SET_MASS, ia, ib, tp[0], Vp, A);
        }
        if (s == 0) { hm = Vm; hy = Vp; }
        else { hx = Vm; hp = Vp; }
    }
    // h*- = min(V-(zeta-), V+(zeta-)), h*+ = min(V+(zeta+), V-(zeta+)); a boundary's
    // ghost has the own operator
    double hsm, hsp;
    if (out.bnd) { hp = hy; hsm = hm; hsp = hp; }
    else { hsm = min_nonneg(hm, hx); hsp = min_nonneg(hp, hy); }
    const bool of = out.own_first;
    const double qnm = ax ? tm[2] : tm[1], qtm = ax ? tm[1] : tm[2];
    const double qnp = ax ? tp[2] : tp[1], qtp = ax ? tp[1] : tp[2];
    const double hA = of ? hm : hp, hB = of ? hp : hm, hsA = of ? hsm : hsp, hsB = of ? hsp : hsm;
    const double cA = of ? tm[3] : tp[3], cB = of ? tp[3] : tm[3];
    const unsigned sA = ((f & 1) != 0) == of ? 0u : 0x80000000u; // sign of A's outward normal
    double fA, fB, wA, wB;
    vel_wave(hA, d.g, d.sg, d.eps, fA, wA);
    vel_wave(hB, d.g, d.sg, d.eps, fB, wB);
    const double vA = fA * (of ? qnm : qnp), uA = fA * (of ? qtm : qtp);
    const double vB = fB * (of ? qnp : qnm), uB = fB * (of ? qtp : qtm);
    const double lam = __longlong_as_double(max(wave_key(fabs(vA) + wA, uA), wave_key(fabs(vB) + wB, uB)));
    const double hl = 0.5 * lam, dh = hsA - hsB;
    const double qsA = hsA * vA, qsB = hsB * vB, rsA = hsA * uA, rsB = hsB * uB;
    out.flux[0] = fma(hl, dh, flip(0.5 * (qsA + qsB), sA));
    out.flux[1] = fma(hl, qsA - qsB, flip(0.5 * fma(qsA, vA, qsB * vB), sA));
    out.flux[2] = fma(hl, rsA - rsB, flip(0.5 * fma(rsA, vA, rsB * vB), sA));
    out.flux[3] = fma(hl, fma(dh, cA, hsB * (cA - cB)), flip(0.5 * fma(qsA, cA, qsB * cB), sA));
    out.pr = flip(0.25 * d.g * (hsA + hsB) * dh, sA);
    out.lam = lam;
    return out;
}
// the four flux components (F, G_x, G_y, R) of a face flux seen from its own
// cell or (other) from the neighbour, times the weight w
__device__ __forceinline__ void side_values(const FaceFlux& q, int f, bool other, double w, double (&o)[4]) {
    const unsigned sg = q.own_first != other ? 0u : 0x80000000u;
    const double a = w * (flip(q.flux[1], sg) - q.pr), t = w * flip(q.flux[2], sg);
    o[0] = w * flip(q.flux[0], sg);
    o[1] = f < 2 ? a : t;
    o[2] = f < 2 ? t : a;
    o[3] = w * flip(q.flux[3], sg);
}

// The FP64 residual.  What bounds it is the FP64 pipe (one warp instruction
// per SM and 16 clocks, however few lanes are active), so only the pointwise
// physics runs there: every contraction is block fixed-point on the integer
// pipe (swdg_fixed.cuh), nodal values and point values being converted on the
// integer pipe too.  A team of TL lanes takes a cell, one volume point per
// lane: 32 lanes at r = 3 (25 points), 16 at r = 2 (16 points), 8 at r = 1
// (4 points), so that the FP64 instructions of the points serve 1, 2 or 4
// cells at once.  The products of the point values (fluxes, pressure, friction,
// tracer) are formed from digit pairs as well: the factors convert instead of
// the products, four values a point instead of twelve, and the FP64
// instructions of a cell fall from 60 to 30.  The test tables carry the
// quadrature weights; the geometric factors h_y of d/dxi and h_x of d/deta enter
// after the integration.  A launch of 65,536 cells (r = 3): 880 us with the sums in
// FP64, 328 so; 43,976 cells (r = 2): 156.
template <int R>
struct ResFx {
    using S = Sz<R>;
    static constexpr int TL = R == 3 ? 32 : (R == 2 ? 16 : 8);
    static constexpr int SUB = R == 1 ? 4 : 16; // lanes that load one field
    static constexpr int FPP = TL / SUB;        // fields loaded at once
    static constexpr int NE = S::ND1 * S::NV;
    // 8-byte words per team, two regions: nodal digits and x-contractions, then
    // the y-test sums; point values, then the face values (with the nodal values
    // where the faces are integrated inline)
    static constexpr int UD = 4 * S::ND, TX = 6 * NE, XP = 11 * S::NVP, SY = 11 * NE,
                         FD = 32 * S::NM;
    static constexpr int RA = UD + TX > SY ? UD + TX : SY, RB = XP > FD + UD ? XP : FD + UD;
    static constexpr int words = RA + RB + 12; // and 4 nodal values, 16 block exponents
    static_assert(S::NVP <= TL && S::ND <= SUB, "one point per lane");
};

// the face fluxes of a conforming cell F [4 fields][4 faces][2 halves][NM], slots
// i = (face, point) spread over the team's lanes
template <int NM, int TL>
__device__ __forceinline__ void face_load(const double* F, double (&fv)[(4 * NM + TL - 1) / TL][4],
                                          int lane) {
#pragma unroll
    for (int j = 0; j < (4 * NM + TL - 1) / TL; ++j) {
        const int i = lane + j * TL;
        const double* Fi = F + (i / NM) * 2 * NM + i % NM;
#pragma unroll
        for (int cf = 0; cf < 4; ++cf) fv[j][cf] = i < 4 * NM ? Fi[cf * 8 * NM] : 0.0;
    }
}
// ... to digits, field by field: fd [4 fields][2 halves][4 faces][NM], block exponents es
template <int NM, int TL>
__device__ __forceinline__ void face_digits(const double (&fv)[(4 * NM + TL - 1) / TL][4], int2* fd,
                                            int* es, int lane, unsigned tm) {
    constexpr int SL = (4 * NM + TL - 1) / TL;
#pragma unroll
    for (int cf = 0; cf < 4; ++cf) {
        unsigned m = 0;
#pragma unroll
        for (int j = 0; j < SL; ++j) m = max(m, fx::mag(fv[j][cf]));
        const int e = fx::block_exp(__reduce_max_sync(tm, m));
#pragma unroll
        for (int j = 0; j < SL; ++j)
            if (lane + j * TL < 4 * NM)
                fd[cf * 8 * NM + lane + j * TL] = fx::split(fx::from_double(fv[j][cf], e));
        if (lane == 0) es[cf] = e;
    }
}
// the same where faces have second halves (or were integrated inline): slot(cf, i),
// i = (half, face, point) < nslot
template <int NM, int TL, typename F>
__device__ __forceinline__ void face_digits_any(F slot, int nslot, int2* fd, int* es, int lane, unsigned tm) {
#pragma unroll 1
    for (int cf = 0; cf < 4; ++cf) {
        unsigned m = 0;
#pragma unroll 1
        for (int i = lane; i < nslot; i += TL) m = max(m, fx::mag(slot(cf, i)));
        const int e = fx::block_exp(__reduce_max_sync(tm, m));
#pragma unroll 1
        for (int i = lane; i < nslot; i += TL) fd[cf * 8 * NM + i] = fx::split(fx::from_double(slot(cf, i), e));
        if (lane == 0) es[cf] = e;
    }
}
// one field's face fluxes lifted onto node (a, b) (a node takes part in at most one
// x face and one y face)
template <int ND1, int NM, typename T>
__device__ __forceinline__ long long face_lift(const T& tx, const int2* fd, int a, int b,
                                               const bool (&c_f)[4]) {
    long long sf = 0;
    auto lift = [&](int f, int tn, bool coarse) {
        fx::Acc q;
        const int2* v = fd + f * NM;
        if (!coarse) {
#pragma unroll
            for (int al = 0; al < NM; ++al) q.mac(tx.BmT[tn][al], v[al]);
        } else {
#pragma unroll
            for (int al = 0; al < NM; ++al) {
                q.mac(tx.BmHT[0][tn][al], v[al]);
                q.mac(tx.BmHT[1][tn][al], v[4 * NM + al]);
            }
        }
        sf += q.get();
    };
    if (a == 0 || a == ND1 - 1) lift(a == 0 ? 0 : 1, b, a == 0 ? c_f[0] : c_f[1]);
    if (b == 0 || b == ND1 - 1) lift(b == 0 ? 2 : 3, a, b == 0 ? c_f[2] : c_f[3]);
    return sf;
}

// INL: the cell integrates its faces itself (the allocation-free entry, which has
// no slot buffer); a kernel of its own, so that the other's code stays small
template <int R, typename Pix, int MODE, bool INL = false>
__global__ void __maxnreg__(64)
    k_residual(const __grid_constant__ Dev d, int buf, int stage, double c_stage, int want_dt) {
    // the tables in shared memory: the contractions index them by lane, which
    // the constant cache would serialise
    __shared__ FxTables tx;
    copy_table(tx, &d.tabs->fx);
    const Tables& tb = *d.tabs;
    using S = Sz<R>;
    using L = ResFx<R>;
    using ST = Site<R, Pix, MODE>;
    constexpr int ND1 = S::ND1, ND = S::ND, NV = S::NV, NVP = S::NVP, NM = S::NM, NE = L::NE;
    constexpr int TL = L::TL;
    extern __shared__ double smem[];
    const int team = threadIdx.x / TL, lane = threadIdx.x % TL, tpb = blockDim.x / TL;
    const unsigned tm =
        TL == 32 ? 0xffffffffu : ((1u << (TL & 31)) - 1u) << (threadIdx.x & 31 & ~(TL - 1));
    int2* ud = (int2*)(smem + team * L::words); // [4][ND]
    int2* sx = ud + L::UD;                      // [6][ND1][NV]: zeta (Bv, Dv), qx, qy, c (Bv), c (Dv)
    int2* sy = ud;                              // [11][NV][ND1]
    int2* xp = ud + L::RA;                      // [11][NVP]
    int2* fd = xp;                              // [4 fields][2 halves][4 faces][NM]
    double* c0 = (double*)(xp + L::RB);         // [4] first nodal value of each field
    int* es = (int*)(c0 + 4); // block exponents: fields 0..3, faces 4..7, xi-parts 8..11, eta-parts 12..15
    double* fh = (double*)fd;                   // the face values before their conversion
    double* su = fh + L::FD;                    // [4][ND] (inline faces only)
    const double g = d.g, eps = d.eps;
    const int64_t n = d.n;
    const int tBB = 2 * tx.tBv, tBD = tx.tBv + tx.tDv, tW = tx.tWB + tx.tWD;
    // the lane's volume point (idle lanes take point 0 and store nothing)
    const bool pt = lane < NVP;
    const int pl = pt ? lane : 0, pal = pl % NV, pbe = pl / NV;

    for (int64_t k = (int64_t)blockIdx.x * tpb + team; k < n; k += (int64_t)gridDim.x * tpb) {
        const unsigned cm = d.cmask[(size_t)buf * n + k];
        const double hx = d.hxhy[2 * k], hy = d.hxhy[2 * k + 1];
#pragma unroll 1
        for (int ps = 0; ps < 4 / L::FPP; ++ps) {
            const int sub = lane / L::SUB, f = ps * L::FPP + sub, node = lane % L::SUB;
            const double v = node < ND ? ufield(d, buf, f, ND)[k * ND + node] : 0.0;
            unsigned m = fx::mag(v);
#pragma unroll
            for (int o = 1; o < L::SUB; o <<= 1) m = max(m, __shfl_xor_sync(tm, m, o));
            const int e = fx::block_exp(m);
            if (node < ND) {
                ud[f * ND + node] = fx::split(fx::from_double(v, e));
                if (node == 0) {
                    c0[f] = v;
                    es[f] = e;
                }
            }
        }
        unsigned fi[4]; // indexed by constants only (registers)
#pragma unroll
        for (int f = 0; f < 4; ++f) fi[f] = d.finfo ? d.finfo[k * 4 + f] : 0;
        const bool c_f[4] = {(fi[0] & 3) == FI_COARSE, (fi[1] & 3) == FI_COARSE,
                             (fi[2] & 3) == FI_COARSE, (fi[3] & 3) == FI_COARSE};
        const int nslot = (c_f[0] || c_f[1] || c_f[2] || c_f[3]) ? 8 * NM : 4 * NM;
        __syncwarp(tm);
        // x-contractions: zeta (value, d/dxi), qx, qy, c, and c's d/dxi for the
        // tracer numerical diffusion (Eq. numdiff)
        const double nu = d.nu_c ? d.nu_c[k] : 0.0;
#pragma unroll 1
        for (int i = lane; i < (nu != 0.0 ? 6 : 5) * NE; i += TL) {
            const int f = i / NE, r_ = i % NE, b = r_ / NV, al = r_ % NV;
            const int2* T = (f == 1 || f == 5) ? tx.Dv[al] : tx.Bv[al];
            const int2* u = ud + (f < 2 ? 0 : f < 5 ? f - 1 : 3) * ND + ND1 * b;
            fx::Acc s;
#pragma unroll
            for (int a = 0; a < ND1; ++a) s.mac(T[a], u[a]);
            sx[i] = fx::split(s.get());
        }
        __syncwarp(tm);
        // y-contraction and pointwise physics, one volume point per lane.  Only the
        // depth's powers, |q| and the velocities are formed in FP64; the products
        // are products of digit pairs, with the exponents below
        const double man = d.manning[k];
        int eL[2]; // exponents of Lx, Ly
        {
            long long Z, ZX, ZY, QX, QY, C;
            {
                fx::Acc az, azx, azy, aqx, aqy, ac;
#pragma unroll
                for (int b = 0; b < ND1; ++b) {
                    const int2 Tb = tx.Bv[pbe][b], Td = tx.Dv[pbe][b];
                    const int2* s = sx + b * NV + pal;
                    az.mac(Tb, s[0]);
                    azy.mac(Td, s[0]);
                    azx.mac(Tb, s[NE]);
                    aqx.mac(Tb, s[2 * NE]);
                    aqy.mac(Tb, s[3 * NE]);
                    ac.mac(Tb, s[4 * NE]);
                }
                Z = az.get();
                ZX = azx.get();
                ZY = azy.get();
                QX = aqx.get();
                QY = aqy.get();
                C = ac.get();
            }
            const int eu0 = es[0], eu3 = es[3];
            int eD = eu0 + tBD, eX = es[1] + tBB, eY = es[2] + tBB, eC = eu3 + tBB;
            // a constant field is that constant exactly
            if (cm & 1u) ZX = ZY = 0;
            if (cm & 2u) QX = fx::from_double(c0[1], eX);
            if (cm & 4u) QY = fx::from_double(c0[2], eY);
            if (cm & 8u) C = fx::from_double(c0[3], eC);
            // the factors of products move up to the places that are free in their blocks:
            // the tables' bounds are a few places above the values, and far above the gradient
            auto up = [&](long long& x, int& e) {
                const int s = fx::headroom(__reduce_max_sync(tm, pt ? fx::high(x) : 0u));
                x <<= s;
                e -= s;
            };
            {
                const int s = fx::headroom(__reduce_max_sync(tm, pt ? max(fx::high(ZX), fx::high(ZY)) : 0u));
                ZX <<= s;
                ZY <<= s;
                eD -= s;
            }
            up(QX, eX);
            up(QY, eY);
            up(C, eC);
            const double z = (cm & 1u) ? c0[0] : fx::to_double(Z, eu0 + tBB);
            const double qx = fx::to_double(QX, eX), qy = fx::to_double(QY, eY);
            double h = 0.0, A;
            if (pt) ST::VA(d, tb, k, SET_VOL, pal, pbe, z, h, A);
            double fv, gm;
            vel_friction(h, qx, qy, !zero_bits(man), eps, fv, gm);
            const double ux = fv * qx, uy = fv * qy, gh = -g * h;
            auto block = [&](unsigned m) { return fx::block_exp(__reduce_max_sync(tm, pt ? m : 0u)); };
            const int eU = block(max(fx::mag(ux), fx::mag(uy))), eH = block(fx::mag(gh)),
                      eM = block(fx::mag(gm));
            const int2 dqx = fx::split(QX), dqy = fx::split(QY), dc = fx::split(C);
            const int2 dux = fx::split(fx::from_double(ux, eU)), duy = fx::split(fx::from_double(uy, eU));
            const int2 dgh = fx::split(fx::from_double(gh, eH)), dgm = fx::split(fx::from_double(gm, eM));
            // exponents of the products; -g h grad zeta joins the xi-part of Gx and
            // the eta-part of Gy
            const int eXU = fx::product_exp(eX, eU), eYU = fx::product_exp(eY, eU),
                      eHZ = fx::product_exp(eH, eD);
            const int eGx = max(eXU, eHZ), eGy = max(eYU, eHZ);
            int eRx = fx::product_exp(eC, eX), eRy = fx::product_exp(eC, eY);
            eL[0] = fx::product_exp(eM, eX);
            eL[1] = fx::product_exp(eM, eY);
            long long RX = fx::product(dc, dqx), RY = fx::product(dc, dqy);
            if (nu != 0.0 && !(cm & 8u)) {
                // -nu h grad c . grad psi: the reference derivatives of c at the point
                fx::Acc acx, acy;
#pragma unroll
                for (int b = 0; b < ND1; ++b) {
                    acx.mac(tx.Bv[pbe][b], sx[(5 * ND1 + b) * NV + pal]);
                    acy.mac(tx.Dv[pbe][b], sx[(4 * ND1 + b) * NV + pal]);
                }
                const double rx = fx::to_double(RX, eRx) - nu * h * fx::to_double(acx.get(), eu3 + tBD) / hx;
                const double ry = fx::to_double(RY, eRy) - nu * h * fx::to_double(acy.get(), eu3 + tBD) / hy;
                eRx = eRy = block(max(fx::mag(rx), fx::mag(ry)));
                RX = fx::from_double(rx, eRx);
                RY = fx::from_double(ry, eRx);
            }
            if (lane == 0) { // of F, Gx, Gy, R
                es[8] = eX;
                es[9] = eGx;
                es[10] = eYU;
                es[11] = eRx;
                es[12] = eY;
                es[13] = eYU;
                es[14] = eGy;
                es[15] = eRy;
            }
            if (pt) {
                int2* o = xp + pl;
                o[0 * NVP] = dqx;
                o[1 * NVP] = dqy;
                o[2 * NVP] = fx::split(RX);
                o[3 * NVP] = fx::split(RY);
                o[4 * NVP] = fx::split(fx::product(dqx, dux) >> min(eGx - eXU, 63));
                const long long yu = fx::product(dqy, dux); // = qx uy
                o[5 * NVP] = fx::split(yu);
                o[6 * NVP] = fx::split(fx::product(dqy, duy) >> min(eGy - eYU, 63));
                o[7 * NVP] = fx::split(fx::product(dgh, fx::split(ZX)) >> min(eGx - eHZ, 63));
                o[8 * NVP] = fx::split(fx::product(dgh, fx::split(ZY)) >> min(eGy - eHZ, 63));
                o[9 * NVP] = fx::split(fx::product(dgm, dqx));
                o[10 * NVP] = fx::split(fx::product(dgm, dqy));
            }
        }
        __syncwarp(tm);
        // the face fluxes of k_faces; where no face of the cell has a second half they
        // are loaded here, so that the y-contraction hides the latency
        const bool conforming = nslot == 4 * NM;
        double fv[(4 * NM + TL - 1) / TL][4];
        if (!INL && conforming) face_load<NM, TL>(d.fflux + k * (32 * NM), fv, lane);
        // test integration, y-contraction: jobs 0..3 the xi-parts of F, R, Gx, Gy
        // (wv Bv), 4, 5 Lx, Ly, 6..8 the eta-parts of F, R, Gx (wv Dv), 9 the value
        // part of Gx; then 10 the eta- and value parts of Gy
#pragma unroll 1
        for (int i = lane; i < 10 * NE; i += TL) {
            const int job = i / NE, r_ = i % NE, al = r_ / ND1, b = r_ % ND1;
            const int2* T = job < 6 ? tx.WB[b] : job < 9 ? tx.WD[b] : tx.WDB[b];
            const int2* X = xp + (int)((0x7531A95420ull >> (4 * job)) & 15u) * NVP + al;
            fx::Acc s;
#pragma unroll
            for (int be = 0; be < NV; ++be) s.mac(T[be], X[NV * be]);
            sy[i] = fx::split(s.get());
        }
#pragma unroll 1
        for (int i = lane; i < NE; i += TL) {
            const int al = i / ND1, b = i % ND1;
            const int2* X = xp + 6 * NVP + al;
            fx::Acc s;
#pragma unroll
            for (int be = 0; be < NV; ++be) {
                s.mac(tx.WD[b][be], X[NV * be]);
                s.mac(tx.WDB[b][be], X[2 * NVP + NV * be]);
            }
            sy[10 * NE + i] = fx::split(s.get());
        }
        __syncwarp(tm);
        if constexpr (INL) {
            // the allocation-free entry: the cell's faces here, one (sub)face
            // point per lane; the face points of faces 0..3 start at 0, b1, b2,
            // b3 (2 NM points on a coarse 2:1 face, else NM)
            const int mem = member_of(d, k);
            const double ihx = d.ihxhy ? d.ihxhy[2 * k] : 1.0 / hx;
            const double ihy = d.ihxhy ? d.ihxhy[2 * k + 1] : 1.0 / hy;
            for (int i = lane; i < 4 * ND; i += TL)
                su[i] = ufield(d, buf, i / ND, ND)[k * ND + (i % ND)];
            __syncwarp(tm);
            double dtl = 0.0;
            const int b1 = c_f[0] ? 2 * NM : NM, b2 = b1 + (c_f[1] ? 2 * NM : NM),
                      b3 = b2 + (c_f[2] ? 2 * NM : NM), b4 = b3 + (c_f[3] ? 2 * NM : NM);
            for (int it = lane; it < b4; it += TL) {
                const int f = (it >= b1) + (it >= b2) + (it >= b3);
                const int r_ = it - (f == 0 ? 0 : f == 1 ? b1 : f == 2 ? b2 : b3), h = r_ / NM,
                          al = r_ % NM;
                const unsigned info = f == 0 ? fi[0] : f == 1 ? fi[1] : f == 2 ? fi[2] : fi[3];
                const bool coarse = (info & 3) == FI_COARSE;
                const FaceFlux q = face_flux<R, Pix, MODE>(d, d.tabs->ft, k, su, ND, cm, buf, f, h, al,
                                                           info, mem, c_stage);
                double out[4];
                side_values(q, f, false, ((f < 2) ? hy : hx) * (coarse ? 0.5 : 1.0) * d.tabs->ft.wm[al],
                            out);
#pragma unroll
                for (int cf = 0; cf < 4; ++cf) fh[((cf * 2 + h) * 4 + f) * NM + al] = out[cf];
                // lambda l / J for the positivity step (l = L, J = hx hy)
                dtl = fmax(dtl, fmax(q.lam, 1e-12) * ((f < 2) ? ihx : ihy) * (coarse ? 0.5 : 1.0));
            }
            if (want_dt) {
                const double m = team_max_nonneg(dtl, tm);
                if (lane == 0) atomic_max_pos(&d.mb[mem].rmax, m);
            }
            __syncwarp(tm);
        }
        if (!INL && conforming) {
            face_digits<NM, TL>(fv, fd, es + 4, lane, tm);
        } else {
            face_digits_any<NM, TL>([&](int cf, int i) -> double { // 0 where a face has no second half
                const int h = i / (4 * NM), f = i / NM & 3, al = i % NM;
                const bool own = h == 0 || (f == 0 ? c_f[0] : f == 1 ? c_f[1] : f == 2 ? c_f[2] : c_f[3]);
                if (!own) return 0.0;
                return INL ? fh[cf * 8 * NM + i] : d.fflux[k * (32 * NM) + ((cf * 4 + f) * 2 + h) * NM + al];
            }, nslot, fd, es + 4, lane, tm);
        }
        __syncwarp(tm);
        // x-contraction of F, Gx, Gy, R, the xi-parts times h_y and the eta-parts
        // times h_x, minus the face fluxes lifted onto the nodes of their faces (a
        // node takes part in at most one x face and one y face)
        const int eh = fx::block_exp(max(fx::mag(hx), fx::mag(hy)));
        const int2 dhx = fx::split(fx::from_double(hx, eh)), dhy = fx::split(fx::from_double(hy, eh));
#pragma unroll 1
        for (int i = lane; i < 4 * ND; i += TL) {
            const int cf = i / ND, j = i % ND, a = j % ND1, b = j / ND1;
            const int2* s1 = sy + ((0x1320u >> (4 * cf)) & 15u) * NE + b;
            const int2* s2 = sy + ((0x7A86u >> (4 * cf)) & 15u) * NE + b;
            fx::Acc sa, sb;
#pragma unroll
            for (int al = 0; al < NV; ++al) {
                sa.mac(tx.WD[a][al], s1[al * ND1]);
                sb.mac(tx.WB[a][al], s2[al * ND1]);
            }
            if (cf == 1) {
#pragma unroll
                for (int al = 0; al < NV; ++al) sa.mac(tx.WB[a][al], sy[9 * NE + al * ND1 + b]);
            }
            const int e1 = es[8 + cf], e2 = es[12 + cf], ff = es[4 + cf];
            const int em = max(e1, e2);
            const long long vol = (fx::product(fx::split(sa.get()), dhy) >> min(em - e1, 63)) +
                                  (fx::product(fx::split(sb.get()), dhx) >> min(em - e2, 63));
            const long long sf = face_lift<ND1, NM>(tx, fd + cf * 8 * NM, a, b, c_f);
            rfield(d, stage, cf, ND)[k * ND + j] =
                fx::to_double(vol, fx::product_exp(em + tW, eh)) - fx::to_double(sf, ff + tx.tBmT);
        }
        const double kJ = -(g * man * man) * (hx * hy);
#pragma unroll 1
        for (int i = lane; i < 2 * ND; i += TL) { // Lx, Ly
            const int cl = i / ND, j = i % ND, a = j % ND1, b = j / ND1;
            fx::Acc s;
#pragma unroll
            for (int al = 0; al < NV; ++al) s.mac(tx.WB[a][al], sy[(4 + cl) * NE + al * ND1 + b]);
            rfield(d, stage, 4 + cl, ND)[k * ND + j] =
                kJ * fx::to_double(s.get(), (cl ? eL[1] : eL[0]) + 2 * tx.tWB);
        }
        __syncwarp(tm);
    }
}

// every face point of the mesh once (the residual's face integrals, Sec. 3.2):
// job j of d.fjobs is cell k = job >> 8 with face f, half h and GLL point al
// packed as f | h << 2 | al << 3, k the lower cell index of the face (or the
// cell of a boundary face).  The flux as seen from each side, times that
// side's quadrature weight, goes to the side's slots of d.fflux
// ([cell][4 fields][4 faces][2 halves][NM], the residual's fh layout);
// with want_dt the wave speed bound of each side (lambda l / J) raises its
// member's rmax, as the residual does when it integrates the faces itself.
// One job per lane.  65,536 cells at r = 3: 225 us in Cartesian components, 168 in the
// face's frame (the FP64 pipe bounds it).
template <int R, typename Pix, int MODE>
__global__ void __maxnreg__(72)
    k_faces(const __grid_constant__ Dev d, int buf, double c_stage, int want_dt) {
    __shared__ FaceTables ft; // its rows are indexed by lane
    copy_table(ft, &d.tabs->ft);
    using S = Sz<R>;
    constexpr int ND = S::ND, NM = S::NM, SL = 32 * NM;
    const int lane = threadIdx.x & 31;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t n = d.n;
    for (int64_t j0 = gw * 32; j0 < d.njobs; j0 += nw * 32) { // warp-uniform bounds
        const int64_t j = j0 + lane;
        double v = 0.0;
        int mem = -1;
        if (j < d.njobs) {
            const int64_t job = d.fjobs[j];
            const int64_t k = job >> 8;
            const int f = (int)(job & 3), h = (int)((job >> 2) & 1), al = (int)((job >> 3) & 31);
            const unsigned info = d.finfo ? d.finfo[k * 4 + f] : 0;
            mem = member_of(d, k);
            const FaceFlux q =
                face_flux<R, Pix, MODE>(d, ft, k, ufield(d, buf, 0, ND) + k * ND, (size_t)n * ND,
                                        d.cmask[(size_t)buf * n + k], buf, f, h, al, info, mem, c_stage);
            // max(lambda, 1e-12), a NaN counting as 1e-12
            const long long lb = __double_as_longlong(q.lam);
            const double lam = lb > __double_as_longlong(1e-12) && !nan_bits(q.lam) ? q.lam : 1e-12;
            // the own side, then the other one (the fine side of a 2:1 face has one
            // half) with its own weight; extent l_Gamma along the face, 1 / J l_Gamma
            // across it
#pragma unroll 1
            for (int s = 0; s < (q.bnd || q.nb == k ? 1 : 2); ++s) {
                const int64_t kc = s ? q.nb : k;
                const int fc = s ? f ^ 1 : f;
                const unsigned ci = s ? (d.finfo ? d.finfo[kc * 4 + fc] : 0) : info;
                const int hc = s ? ((info & 3) == FI_FINE ? (int)(info >> 2) : 0) : h;
                const double sc = (ci & 3) == FI_COARSE ? 0.5 : 1.0;
                double out[4];
                side_values(q, fc, s != 0, d.hxhy[2 * kc + (fc < 2 ? 1 : 0)] * sc * ft.wm[al], out);
                double* F = d.fflux + kc * SL + (fc * 2 + hc) * NM + al;
#pragma unroll
                for (int cf = 0; cf < 4; ++cf) F[cf * 8 * NM] = out[cf];
                if (want_dt) {
                    const double ih = d.ihxhy ? d.ihxhy[2 * kc + (fc < 2 ? 0 : 1)]
                                              : 1.0 / d.hxhy[2 * kc + (fc < 2 ? 0 : 1)];
                    v = fmax(v, lam * ih * sc);
                }
            }
        }
        if (want_dt) {
            // one atomic per warp when its jobs share a member, else per job
            const int m0 = __shfl_sync(0xffffffffu, mem, 0);
            if (__all_sync(0xffffffffu, mem == m0 || mem < 0)) {
                const double m = team_max_nonneg(v, 0xffffffffu); // v >= 0, never NaN
                if (lane == 0 && m0 >= 0) atomic_max_pos(&d.mb[m0].rmax, m);
            } else if (mem >= 0) {
                atomic_max_pos(&d.mb[mem].rmax, v);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// warp-cooperative scalar Newton for Hbar(e) = target (r_K = 0 cells,
// Eqs. newton, initial_guess); returns iterations
// ---------------------------------------------------------------------------
template <int R, typename Pix, int MODE, int TL = 32>
__device__ __forceinline__ void mass_scalar(const Dev& d, const Tables& tb, int64_t k, double J,
                                            double e, int lane, double& H, double& A,
                                            unsigned tm = 0xffffffffu) {
    using S = Sz<R>;
    double h = 0.0, a = 0.0;
#pragma unroll 1
    for (int p = lane; p < S::NMP; p += TL) {
        const int ia = p % S::NM, ib = p / S::NM;
        double V, Ap;
        Site<R, Pix, MODE>::VA(d, tb, k, SET_MASS, ia, ib, e, V, Ap);
        const double w = J * tb.wm[ia] * tb.wm[ib];
        h += w * V;
        a += w * Ap;
    }
    team_sum2<TL>(h, a, tm);
    H = h;
    A = a;
}

// The same mean depth and wet area for a constant elevation e, in mode S as
// one sum over the cell's pixels: the mass sub-cells tile the cell, so the
// pixel k of a P x P tile carries 1/P^2 of the area whatever sub-cells it
// is split among, and Hbar(e) = J / P^2 sum_k max(e + z_k, 0), Abar = J / P^2
// #{e + z_k > 0} (equal to mass_scalar up to rounding, with P^2 terms
// instead of the sub-cells' split pixels).  Cells wholly wet or dry, and mode
// P, take mass_scalar (its shortcut makes it cheap there), as does a cell with an
// infinite depth.  The wet depths are integers (as in subgrid_S, in the block of e
// and the deepest pixel) and their sum is exact.
// Not inlined: the scalar path calls it in three places, and its code shares the
// instruction cache with the other cells'.
struct Mass {
    double H, A;
};
template <int R, typename Pix, int MODE, int TL = 32>
__device__ __noinline__ Mass mass_scalar_pixels(const Dev& d, const Tables& tb, int64_t k, double J,
                                                double e, int lane, unsigned tm = 0xffffffffu) {
    using ST = Site<R, Pix, MODE>;
    const bool mixed = MODE == 0 && d.zmin != nullptr && !nan_bits(e) &&
                       !(okey(e) > nkey_neg(d.zmin[k])) && okey(e) > nkey_neg(d.zmax[k]) &&
                       finite_bits(d.zmax[k]);
    if (!mixed) {
        Mass m;
        mass_scalar<R, Pix, MODE, TL>(d, tb, k, J, e, lane, m.H, m.A, tm);
        return m;
    }
    const OvTab& o = ST::tab(d, k);
    const Pix* t = ST::tile(d, o, k);
    const int np = o.P * o.P;
    const int es = fx::block_exp(max(fx::mag(d.zmax[k]), fx::mag(e))) + 1;
    const long long E = fx::from_double(e, es);
    const Wet<Pix> is_wet(e);
    long long hi = 0;
    unsigned long long lo = 0;
    int a = 0;
#pragma unroll 1
    for (int i = lane; i < np; i += TL) {
        const Pix z = t[i];
        const long long D0 = E + fx_pixel(z, es), D = is_wet(z) ? D0 : 0;
        hi += D >> 32;
        lo += (unsigned)D;
        a += is_wet(z);
    }
    const double h = fx::to_double(hi, es + 32) + fx::to_double((long long)lo, es);
    const double w = J / (double)np;
    return {w * team_sum<TL>(h, tm), w * (double)__reduce_add_sync(tm, a)};
}

template <int R, typename Pix, int MODE, int TL = 32>
__device__ __noinline__ int scalar_newton(const Dev& d, const Tables& tb, int64_t k, double J, double target,
                             double& e, int lane, unsigned tm = 0xffffffffu) {
    constexpr int ND = Sz<R>::ND;
    Mass m = mass_scalar_pixels<R, Pix, MODE, TL>(d, tb, k, J, e, lane, tm);
    // the first iteration reuses this evaluation unless the start moves to the
    // dry start of Eq. initial_guess
    bool have = true;
    if (m.A == 0.0) {
        e = -d.zmax[k] + d.eps0;
        have = false;
    }
    int it = 0;
#pragma unroll 1
    for (int kk = 0; kk < d.newton_max; ++kk) {
        if (!have) m = mass_scalar_pixels<R, Pix, MODE, TL>(d, tb, k, J, e, lane, tm);
        have = false;
        if (m.A == 0.0) break;
        const double dd = (m.H - target) / m.A;
        e -= dd;
        ++it;
        if (ND * fabs(dd) <= d.newton_tol * (ND * (1.0 + fabs(e) + d.zabs[k]))) break;
    }
    return it;
}

// ---------------------------------------------------------------------------
// stage update for one cell: continuity Newton (Eq. newton, Eq. mass_matrix),
// momentum with the friction-modified mass matrix (Eq. mass_matrix_discharge)
// inverted as S^-1 D^-1 S^-T (Sec. 3.3), tracer with the depth-weighted mass
// matrix (Eq. mass_matrix_concentration) by Cholesky
// ---------------------------------------------------------------------------
struct StageArgs {
    int out_buf;   // state buffer written
    int prev_buf;  // state buffer of stage l-1 (friction coefficient)
    int nres;      // residual stages summed
    double wa[MXS], wat[MXS];
    double add;    // implicit diagonal a~_ll
    int use_llin;  // final: the last stage enters with its linearised friction term
    int make_llin; // this stage is the last one and implicit: store Llin
    int final_;    // final combination: update time and bookkeeping
};

// Cholesky of the SPD matrix M (ND x ND, lower part packed by rows) on a team, then M x = b in place by column-oriented forward and back
// substitution (one reciprocal per column, the updates spread over lanes);
// returns false on a non-positive pivot
__device__ __forceinline__ int tri(int i, int j) { return i * (i + 1) / 2 + j; } // j <= i
template <int ND, int TL = 32>
__device__ __noinline__ bool chol_solve(double* M, double* b, double* inv, int lane, unsigned tm = 0xffffffffu) {
#pragma unroll 1
    for (int j = 0; j < ND; ++j) {
        __syncwarp(tm);
        const double djj = M[tri(j, j)];
        if (!(djj > 0.0)) return false;
        const double ljj = sqrt(djj);
        const double r = 1.0 / ljj;
        __syncwarp(tm);
#pragma unroll 1
        for (int i = j + 1 + lane; i < ND; i += TL) M[tri(i, j)] *= r;
        if (lane == 0) {
            M[tri(j, j)] = ljj;
            inv[j] = r;
        }
        __syncwarp(tm);
        const int m = ND - j - 1;
#pragma unroll 1
        for (int idx = lane; idx < m * m; idx += TL) {
            const int i = j + 1 + idx / m, l = j + 1 + idx % m;
            if (l <= i) M[tri(i, l)] -= M[tri(i, j)] * M[tri(l, j)];
        }
    }
    __syncwarp(tm);
#pragma unroll 1
    for (int j = 0; j < ND; ++j) { // L y = b
        const double yj = b[j] * inv[j];
        __syncwarp(tm);
#pragma unroll 1
        for (int i = j + 1 + lane; i < ND; i += TL) b[i] -= M[tri(i, j)] * yj;
        if (lane == 0) b[j] = yj;
        __syncwarp(tm);
    }
#pragma unroll 1
    for (int j = ND - 1; j >= 0; --j) { // L^T x = y
        const double xj = b[j] * inv[j];
        __syncwarp(tm);
#pragma unroll 1
        for (int i = lane; i < j; i += TL) b[i] -= M[tri(j, i)] * xj;
        if (lane == 0) b[j] = xj;
        __syncwarp(tm);
    }
    return true;
}

// M_(a,b),(c,d) = sum_{al,be} c_{al,be} Bm[al][a] Bm[al][c] Bm[be][b] Bm[be][d],
// the lower part packed by rows (rarely reached: not inlined)
template <int ND1, int NM, int TL = 32>
__device__ __noinline__ void assemble_mass(const BaseTables& tb, const double* cw, double* Y,
                                              double* M, int lane, unsigned tm = 0xffffffffu) {
    constexpr int ND = ND1 * ND1;
#pragma unroll 1
    for (int i = lane; i < ND1 * ND1 * NM; i += TL) {
        const int a = i / (ND1 * NM), r_ = i % (ND1 * NM), c = r_ / NM, be = r_ % NM;
        double s = 0.0;
#pragma unroll
        for (int al = 0; al < NM; ++al) s += cw[al + NM * be] * tb.Bm[al][a] * tb.Bm[al][c];
        Y[i] = s;
    }
    __syncwarp(tm);
#pragma unroll 1
    for (int i = lane; i < ND * ND; i += TL) {
        const int r_ = i / ND, s_ = i % ND;
        if (s_ > r_) continue;
        const int a = r_ % ND1, b = r_ / ND1, c = s_ % ND1, dd = s_ / ND1;
        double s = 0.0;
#pragma unroll
        for (int be = 0; be < NM; ++be)
            s += Y[(a * ND1 + c) * NM + be] * tb.Bm[be][b] * tb.Bm[be][dd];
        M[tri(r_, s_)] = s;
    }
    __syncwarp(tm);
}

// FP32 inverse of H' = S B^T diag(cw') B S, one row per lane in a[] (ND <= TL):
// cw' = cw 2^-(ecw - 1022) <= 1 (given as FP32) and S scales the columns of B to
// norm 1, so the diagonal and every pivot of the elimination is at most 1.
// Gauss-Jordan in place: step J broadcasts row J through shared memory; with
// p = 1 / pivot, row i != J loses a_iJ p times it and row J is multiplied by p,
// written as r_l - (1 - p) r_l, which does not cancel since p >= 1.  The
// columns rotate by one per step, so that the pivot column is always a[0] and
// one loop body serves all steps (the unrolled Cholesky with its two
// substitutions per correction, which this replaces, was three times the
// instructions, and fetching them stalled the kernel).  buf: 16-byte aligned,
// 2 NDP + NMP + PR NM floats (NDP = ND rounded up to 4, PR = ND1 (ND1 + 1) / 2).
// Returns false on a non-positive pivot.
template <int N>
__device__ __forceinline__ void read_row(const float* b, float (&r)[N]) {
#pragma unroll
    for (int l = 0; l < N; l += 4) {
        const float4 v = *(const float4*)(b + l);
        r[l] = v.x;
        r[l + 1] = v.y;
        r[l + 2] = v.z;
        r[l + 3] = v.w;
    }
}
template <int ND1, int NM, int TL>
__device__ __forceinline__ bool mass_inverse_f(const FxStage& fs, float* buf, float (&a)[ND1 * ND1],
                                               int lane, unsigned tm) {
    constexpr int ND = ND1 * ND1, NDP = (ND + 3) / 4 * 4, PR = ND1 * (ND1 + 1) / 2;
    static_assert(ND <= TL, "one row per lane");
    const float* cwf = buf + 2 * NDP;  // [NMP], written by the caller
    float* Y = buf + 2 * NDP + NM * NM; // [PR][NM]: contracted over the points of a row
    __syncwarp(tm);
#pragma unroll 1
    for (int i = lane; i < PR * NM; i += TL) {
        const int pr = i / NM, be = i % NM;
        float s = 0.0f;
#pragma unroll
        for (int al = 0; al < NM; ++al) s += cwf[al + NM * be] * fs.BB[pr][al];
        Y[i] = s;
    }
    __syncwarp(tm);
    const int row = lane < ND ? lane : 0, ar = row % ND1, br = row / ND1;
    auto pair = [](int x, int y) { return x > y ? x * (x + 1) / 2 + y : y * (y + 1) / 2 + x; };
#pragma unroll
    for (int t = 0; t < ND; ++t) a[t] = 0.0f;
#pragma unroll
    for (int be = 0; be < NM; ++be) {
        float y[ND1], q[ND1];
#pragma unroll
        for (int c = 0; c < ND1; ++c) {
            y[c] = Y[pair(ar, c) * NM + be];
            q[c] = fs.BB[pair(br, c)][be];
        }
#pragma unroll
        for (int t = 0; t < ND; ++t) a[t] += y[t % ND1] * q[t / ND1];
    }
    bool ok = true;
#pragma unroll 1
    for (int J = 0; J < ND; ++J) {
        float* rb = buf + (J & 1) * NDP;
        if (lane == J) {
#pragma unroll
            for (int l = 0; l < NDP; l += 4)
                *(float4*)(rb + l) = make_float4(a[l], l + 1 < ND ? a[l + 1] : 0.0f,
                                                 l + 2 < ND ? a[l + 2] : 0.0f,
                                                 l + 3 < ND ? a[l + 3] : 0.0f);
        }
        __syncwarp(tm);
        float r[NDP];
        read_row<NDP>(rb, r);
        ok = ok && r[0] > 0.0f;
        const float p = __fdividef(1.0f, r[0]);
        const float f = lane == J ? 1.0f - p : a[0] * p;
#pragma unroll
        for (int l = 1; l < ND; ++l) a[l - 1] = fmaf(-f, r[l], a[l]);
        a[ND - 1] = lane == J ? p : -f;
    }
    __syncwarp(tm);
    return ok;
}

// Solve H x = b for the depth-weighted mass matrix H = B^T diag(cw) B (the
// tracer matrix of Eq. mass_matrix_concentration, or the masked Jacobian of
// Eq. mass_matrix) by mixed-precision iterative refinement: H is assembled and
// inverted in FP32, each correction is one FP32 product with the inverse, and
// the residual b - H x is formed matrix-free by sum factorisation in block fixed
// point (on the integer pipe; in FP64 arithmetic the two residuals were a third of
// the stage update's FP64 instructions), x being held as a fixed-point number too.
// The point values B x and cw B x move up to the top of their blocks, so that a
// residual keeps 57 places of the largest of them.  What goes through FP32 is scaled
// by the exponents of the blocks, so the magnitudes of b, cw and x do not matter.
// The sweeps stop when a correction, or the next one as predicted from the
// contraction of the last two, is below 1e-15 of x; if that does not happen within 6
// sweeps (an ill-conditioned near-dry cell), if the corrections grow or one is not
// finite, the FP64 Cholesky decides.  x in place of b on return.
// Scratch: buf (mass_inverse_f's, and 2 floats to align it), digit pairs xd [ND], qd [NMP], td [2 NMP], M,
// Y, inv (double, fallback: M may overlay buf, Y and inv xd, qd and td).
template <int ND1, int NM, int TL = 32>
__device__ __noinline__ bool solve_mass_mixed(const Tables& tb, const FxStage& fs, const double* cw, double* b,
                                 float* buf, int2* xd, int2* qd, int2* td, double* M, double* Y,
                                 double* inv, int lane, unsigned tm = 0xffffffffu) {
    constexpr int ND = ND1 * ND1, NMP = NM * NM, NDP = (ND + 3) / 4 * 4, PP = (NMP + TL - 1) / TL;
    buf = (float*)(((uintptr_t)buf + 15) & ~(uintptr_t)15);
    int2* cwd = td + NM * NM;
    const double bi = lane < ND ? b[lane] : 0.0;
    unsigned mc = 0;
#pragma unroll 1
    for (int p = lane; p < NMP; p += TL) mc = max(mc, fx::mag(cw[p]));
    const int ecw = fx::block_exp(__reduce_max_sync(tm, mc)), eb = team_exp(bi, tm);
#pragma unroll 1
    for (int p = lane; p < NMP; p += TL) {
        const long long c = fx::from_double(cw[p], ecw);
        cwd[p] = fx::split(c);
        buf[2 * NDP + p] = fx::to_float(c, 1022); // of cw 2^(1022 - ecw) <= 1
    }
    float a[ND]; // the lane's row of the inverse
    bool ok = mass_inverse_f<ND1, NM, TL>(fs, buf, a, lane, tm);
    long long X = 0; // the lane's component of x
    int ex = fx::EMIN;
    if (ok && eb >= fx::POISON_MIN) { // b holds an infinity or a NaN
        ex = fx::POISON;
    } else if (ok) {
        ok = false;
        const float si = lane < ND ? fs.sc[lane % ND1] * fs.sc[lane / ND1] : 0.0f;
        float rv = fx::to_float(fx::from_double(bi, eb), 1022); // the residual, 2^(1022 - er) of it
        int er = eb;
        float dprev = 0.0f; // max |correction| / max |x| of the previous sweep
#pragma unroll 1
        for (int sweep = 0; sweep < 6; ++sweep) {
            // the lane's component of the correction, 2^(ecw - er) of it:
            // H = 2^(ecw - 1022) S^-1 H' S^-1
            float* rb = buf + (sweep & 1) * NDP;
            if (lane < ND) rb[lane] = rv * si;
            __syncwarp(tm);
            float r[NDP], v = 0.0f;
            read_row<NDP>(rb, r);
#pragma unroll
            for (int j = 0; j < ND; ++j) v += a[j] * r[j];
            v *= si;
            const float da = lane < ND ? fabsf(v) : 0.0f;
            const unsigned dbits = __reduce_max_sync(tm, __float_as_uint(da)); // a NaN is the largest
            if (dbits >= 0x7f800000u) break;
            const int sc = er - ecw, ev = fx::block_exp_f(dbits) + sc;
            if (sweep == 0) ex = ev + 1; // a place of room for the corrections
            else if (ev > ex) break;
            X += fx::from_float(v, ex - sc);
            // max |x| and the ratio of the correction to it, for the stopping test
            const unsigned xm = __reduce_max_sync(
                tm, lane < ND ? (unsigned)((unsigned long long)(X < 0 ? -X : X) >> 31) : 0u);
            if (xm >= 1u << (fx::FB - 31)) break; // x has outgrown its block
            const float dmax = __uint_as_float(dbits);
            const float dr = dmax / fx::to_float((long long)xm << 31, ex - sc);
            // converged when this correction is below 1e-15 of x, or when the
            // next one is, as predicted from the contraction of the last two
            // (dr / dprev, at most 1/2)
            const bool next_small = sweep > 0 && dr <= 0.5f * dprev && dr * dr <= 1e-15f * dprev;
            if (dr <= 1e-15f || dmax == 0.0f || next_small) {
                ok = true;
                break;
            }
            dprev = dr;
            // r = b - H x, H x = B^T (cw (B x))
            if (lane < ND) xd[lane] = fx::split(X);
            __syncwarp(tm);
            long long q[PP];
            unsigned m = 0;
#pragma unroll
            for (int i = 0; i < PP; ++i) q[i] = 0;
            fx_tens<ND1, NM, TL>(fs.Bm, xd, td, lane, tm, [&](int it, int, long long v_) {
                q[it] = v_;
                m = max(m, fx::high(v_));
            });
            const int s1 = fx::headroom(__reduce_max_sync(tm, m));
            m = 0;
#pragma unroll
            for (int i = 0; i < PP; ++i) {
                const int p = lane + i * TL;
                if (p < NMP) q[i] = fx::product(fx::split(q[i] << s1), cwd[p]);
                m = max(m, fx::high(q[i]));
            }
            const int s2 = fx::headroom(__reduce_max_sync(tm, m));
#pragma unroll
            for (int i = 0; i < PP; ++i) {
                const int p = lane + i * TL;
                if (p < NMP) qd[p] = fx::split(q[i] << s2);
            }
            __syncwarp(tm);
            long long R = 0;
            fx_tens<NM, ND1, TL>(fs.BmT, qd, td, lane, tm, [&](int, int, long long v_) { R = v_; });
            const int eR = fx::product_exp(ex + 2 * fs.tBm - s1, ecw) - s2 + 2 * fs.tBmT;
            er = max(eR, eb);
            rv = lane < ND ? fx::to_float(fx::from_double(bi, er) - (R >> min(er - eR, 63)), 1022) : 0.0f;
        }
    }
    __syncwarp(tm);
    if (ok) {
        if (lane < ND) b[lane] = fx::to_double(X, ex);
        __syncwarp(tm);
        return true;
    }
    assemble_mass<ND1, NM, TL>(tb, cw, Y, M, lane, tm);
    return chol_solve<ND, TL>(M, b, inv, lane, tm);
}

// T (N x N) along both directions of NF fields of N x N values, one node per
// lane (N N <= team width), in block fixed point (t: the table's exponent): v[f] is
// the lane's value in and its result out.  w: 2 NF N N 8-byte words.
template <int N, int NF>
__device__ __forceinline__ void square(const int2 (*T)[MXN], int t, double (&v)[NF], int2* w, int lane,
                                       unsigned tm) {
    constexpr int NN = N * N;
    const bool act = lane < NN;
    const int i = act ? lane : NN - 1, r = i / N, c = i % N;
    int e[NF];
    int2* tmp = w + NF * NN;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        e[f] = team_exp(act ? v[f] : 0.0, tm);
        if (act) w[f * NN + i] = fx::split(fx::from_double(v[f], e[f]));
    }
    __syncwarp(tm);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        fx::Acc s;
#pragma unroll
        for (int a = 0; a < N; ++a) s.mac(T[c][a], w[f * NN + r * N + a]);
        if (act) tmp[f * NN + i] = fx::split(s.get());
    }
    __syncwarp(tm);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        fx::Acc s;
#pragma unroll
        for (int b = 0; b < N; ++b) s.mac(T[r][b], tmp[f * NN + b * N + c]);
        v[f] = fx::to_double(s.get(), e[f] + 2 * t);
    }
    __syncwarp(tm);
}
// one or two fields, not inlined: the stage update calls them in five places, and
// its hot code has to fit the instruction cache (32 KB)
struct Two {
    double a, b;
};
template <int N>
__device__ __noinline__ Two square_two(const int2 (*T)[MXN], int t, double a, double b, int2* w, int lane,
                                       unsigned tm) {
    double v[2] = {a, b};
    square<N, 2>(T, t, v, w, lane, tm);
    return {v[0], v[1]};
}
template <int N>
__device__ __noinline__ double square_one(const int2 (*T)[MXN], int t, double a, int2* w, int lane,
                                          unsigned tm) {
    double v[1] = {a};
    square<N, 1>(T, t, v, w, lane, tm);
    return v[0];
}
template <int N>
__device__ __forceinline__ void square2(const int2 (*T)[MXN], int t, double (&v)[2], int2* w, int lane,
                                        unsigned tm) {
    const Two r = square_two<N>(T, t, v[0], v[1], w, lane, tm);
    v[0] = r.a;
    v[1] = r.b;
}
// ---------------------------------------------------------------------------
// step start: degree switch (Eq. criteria_p) with mass-exact remap, then
// H_i(zeta^n), C~_i^n (Eqs. depth_rhs, concentration_rhs) and their sums
// ---------------------------------------------------------------------------
// One cell per team of 16 lanes, node i on lane i, mass points i and i + 16, as
// in the stage update; the contractions in block fixed point.  65,536 cells at r = 3:
// 300 us with FP64 sums and a cell per warp, 158 so.
template <int R>
struct BeginFx {
    using S = Sz<R>;
    static constexpr int TL = 16, PP = (S::NMP + TL - 1) / TL;
    // 8-byte words per team: digit pairs of nodal fields with scratch [4 ND], of
    // two mass-point fields [2 NMP], scratch [NMP]
    static constexpr int W = 4 * S::ND, words = W + 3 * S::NMP;
    static_assert(S::ND <= TL && S::ND1 * S::NM <= S::NMP, "one node per lane");
};

template <int R, typename Pix, int MODE>
__global__ void __maxnreg__(64)
    k_step_begin(const __grid_constant__ Dev d, int do_switch) {
    using S = Sz<R>;
    using L = BeginFx<R>;
    using ST = Site<R, Pix, MODE>;
    constexpr int ND1 = S::ND1, ND = S::ND, NM = S::NM, NMP = S::NMP, NGP = S::NGP;
    constexpr int TL = L::TL, PP = L::PP;
    __shared__ FxStage fs;
    copy_table(fs, &d.tabs->fs);
    const Tables& tb = *d.tabs;
    extern __shared__ double smem[];
    const int team = threadIdx.x / TL, lane = threadIdx.x % TL, tpb = blockDim.x / TL;
    const unsigned tm = 0xFFFFu << (threadIdx.x & 16);
    int2* w = (int2*)(smem + team * L::words);
    int2* qd = w + L::W; // [2][NMP]
    int2* qt = qd + 2 * NMP;
    const int64_t n = d.n;
    if (blockIdx.x == 0) {
        for (int i = threadIdx.x; i < d.nmemb; i += blockDim.x) d.mb[i].rmax = 0ull;
        if (threadIdx.x == 0) d.sc->maxits = 0;
    }
    const bool act = lane < ND;
    const int node = act ? lane : 0;
    const double wn = act ? fs.wn[node % ND1] * fs.wn[node / ND1] : 0.0;
    double wm2[PP];
#pragma unroll
    for (int j = 0; j < PP; ++j) {
        const int p = lane + j * TL;
        wm2[j] = p < NMP ? fs.wm[p % NM] * fs.wm[p / NM] : 0.0;
    }
    for (int64_t k = (int64_t)blockIdx.x * tpb + team; k < n; k += (int64_t)gridDim.x * tpb) {
        const size_t idx = (size_t)k * ND + node;
        double u[4];
#pragma unroll
        for (int f = 0; f < 4; ++f) u[f] = ufield(d, 0, f, ND)[idx];
        unsigned cm = d.cmask[k];
        const double J = d.hxhy[2 * k] * d.hxhy[2 * k + 1];
        // zeta and c at the lane's mass points
        double pe[PP], pc[PP], V[PP];
        {
            const int ez = team_exp(act ? u[0] : 0.0, tm), ec = team_exp(act ? u[3] : 0.0, tm);
            if (act) {
                w[lane] = fx::split(fx::from_double(u[0], ez));
                w[ND + lane] = fx::split(fx::from_double(u[3], ec));
            }
            const double z0 = __shfl_sync(tm, u[0], 0, TL), c0 = __shfl_sync(tm, u[3], 0, TL);
            __syncwarp(tm);
            fx_tens<ND1, NM, TL>(fs.Bm, w, qt, lane, tm, [&](int it, int, long long X) {
                pe[it] = (cm & 1u) ? z0 : fx::to_double(X, ez + 2 * fs.tBm);
            });
            fx_tens<ND1, NM, TL>(fs.Bm, w + ND, qd, lane, tm, [&](int it, int, long long X) {
                pc[it] = (cm & 8u) ? c0 : fx::to_double(X, ec + 2 * fs.tBm);
            });
        }
        bool allfull = true, low = false;
#pragma unroll
        for (int j = 0; j < PP; ++j) {
            const int p = lane + j * TL;
            V[j] = 0.0;
            if (p < NMP) {
                double A;
                bool full;
                ST::VA(d, tb, k, SET_MASS, p % NM, p / NM, pe[j], V[j], A, full);
                allfull = allfull && full && !zero_bits(A);
                // r_K = 0 where the smallest wet depth of the mass points is at most
                // h_lim (a NaN depth never counts, as under fmin)
                low = low || V[j] <= d.hlim;
            }
        }
        allfull = __all_sync(tm, allfull);
        low = __any_sync(tm, low);
        const int flag = (do_switch && low) ? 0 : R;
        if (flag == 0) {
            // remap to r_K = 0: mass-exact zeta, GL means of q, tracer-mass-exact c
            double m = 0.0, tr = 0.0;
            long long ek = (long long)0x8000000000000000ull;
#pragma unroll
            for (int j = 0; j < PP; ++j) {
                if (lane + j * TL >= NMP) continue;
                const double wv = J * wm2[j] * V[j];
                m += wv;
                tr += wv * pc[j];
                if (!nan_bits(pe[j])) ek = okey(pe[j]) > ek ? okey(pe[j]) : ek;
            }
            team_sum2<TL>(m, tr, tm);
            double mq[3] = {wn * u[1], wn * u[2], wn * u[3]};
            team_sum2<TL>(mq[0], mq[1], tm);
            mq[2] = team_sum<TL>(mq[2], tm);
            const double cnew = (m > 1e-14 * J * d.hlim) ? tr / m : mq[2];
            ek = team_max_key<TL>(ek, tm);
            if (!(cm & 8u)) u[3] = cnew;
            if (!(cm & 2u)) u[1] = mq[0];
            if (!(cm & 4u)) u[2] = mq[1];
            if (!(cm & 1u)) {
                double e = ek == (long long)0x8000000000000000ull ? -INFINITY : of_okey(ek);
                if (m <= 0.0) e = -d.zmax[k];
                else scalar_newton<R, Pix, MODE, TL>(d, tb, k, J, m, e, lane, tm);
                u[0] = e;
            }
            if (act) {
#pragma unroll
                for (int f = 0; f < 4; ++f) ufield(d, 0, f, ND)[idx] = u[f];
            }
            cm = 15u;
            const double z0 = __shfl_sync(tm, u[0], 0, TL), c0 = __shfl_sync(tm, u[3], 0, TL);
#pragma unroll
            for (int j = 0; j < PP; ++j) {
                const int p = lane + j * TL;
                pc[j] = c0;
                double A;
                if (p < NMP) ST::VA(d, tb, k, SET_MASS, p % NM, p / NM, z0, V[j], A);
            }
        }
        // H_i(zeta^n), C~_i^n and their sums
        double hb = 0.0, cb = 0.0, hv[PP];
        unsigned mh = 0, mc = 0;
#pragma unroll
        for (int j = 0; j < PP; ++j) {
            hv[j] = J * wm2[j] * V[j];
            if (lane + j * TL >= NMP) { hv[j] = 0.0; pc[j] = 0.0; }
            pc[j] *= hv[j]; // c is not needed beyond C~
            hb += hv[j];
            cb += pc[j];
            mh = max(mh, fx::mag(hv[j]));
            mc = max(mc, fx::mag(pc[j]));
        }
        team_sum2<TL>(hb, cb, tm);
        const int eh = fx::block_exp(__reduce_max_sync(tm, mh)), ec = fx::block_exp(__reduce_max_sync(tm, mc));
        __syncwarp(tm);
#pragma unroll
        for (int j = 0; j < PP; ++j) {
            if (lane + j * TL >= NMP) continue;
            qd[lane + j * TL] = fx::split(fx::from_double(hv[j], eh));
            qd[NMP + lane + j * TL] = fx::split(fx::from_double(pc[j], ec));
        }
        __syncwarp(tm);
        fx_tens<NM, ND1, TL>(fs.BmT, qd, qt, lane, tm, [&](int, int i, long long X) {
            d.HN[k * ND + i] = fx::to_double(X, eh + 2 * fs.tBmT);
        });
        __syncwarp(tm);
        fx_tens<NM, ND1, TL>(fs.BmT, qd + NMP, qt, lane, tm, [&](int, int i, long long X) {
            d.CN[k * ND + i] = fx::to_double(X, ec + 2 * fs.tBmT);
        });
        // the discharges of v^n at the momentum points, the same for every
        // stage of the step (the stage update reads them rather than
        // interpolating v^n again)
        if (d.qpts) {
            double q[2] = {u[1], u[2]};
            if ((cm & 6u) != 6u) square2<ND1>(fs.Bg, fs.tBg, q, w, lane, tm);
            if (act) {
                d.qpts[k * 2 * NGP + lane] = (cm & 2u) ? u[1] : q[0];
                d.qpts[k * 2 * NGP + NGP + lane] = (cm & 4u) ? u[2] : q[1];
            }
        }
        if (lane == 0) {
            d.HNbar[k] = hb;
            d.CNbar[k] = cb;
            d.flag[k] = (uint8_t)flag;
            d.cmask[k] = (uint8_t)cm;
            if (d.wet0) d.wet0[k] = (uint8_t)(flag != 0 && allfull);
        }
        __syncwarp(tm);
    }
}

// The stage update: one cell per team of 16 lanes, node i and momentum point i
// on lane i ((r+1)^2 <= 16), mass points i and i + 16.  The FP64 pipe bounds
// it, so every contraction (the Newton evaluations, the mass inverse, the
// momentum's S^-T, S^-1 and point values, the tracer's residuals) is block
// fixed-point on the integer pipe and a lane's nodal values stay in registers;
// FP64 is left with the right-hand sides, the pointwise physics and the sums
// that the mass balance needs.  65,536 cells at r = 3 (stage 2, 3, final): 790 / 860 /
// 660 us with FP64 sums, 513 / 545 / 449 so.
template <int R>
struct StageFx {
    using S = Sz<R>;
    static constexpr int TL = 16, PP = (S::NMP + TL - 1) / TL;
    // 8-byte words per team: digit pairs of nodal fields with scratch [6 ND] (the
    // fallback's Y), mass-point digits with the solve's scratch [2 NMP + NMP],
    // weights [NMP], right-hand side [ND], then the FP32 inverse's scratch or the
    // fallback's M
    static constexpr int W = 6 * S::ND, Q = 3 * S::NMP, CW = S::NMP, BV = S::ND;
    static constexpr int TRI = S::ND * (S::ND + 1) / 2;
    static constexpr int INV =
        (2 + 2 * ((S::ND + 3) / 4 * 4) + S::NMP + S::ND1 * (S::ND1 + 1) / 2 * S::NM + 1) / 2;
    static constexpr int words = W + Q + CW + BV + (TRI > INV ? TRI : INV);
    static_assert(S::ND <= TL && S::NGP == S::ND, "one node and one momentum point per lane");
    static_assert(S::ND1 * S::ND1 * S::NM <= W, "fallback Y");
};

// Newton's stopping test in FP64 (rare: not inlined)
template <int TL>
__device__ __noinline__ bool newton_done(double dz, double z, double zabs, double tol, bool act, unsigned tm) {
    double inc = act ? fabs(dz) : 0.0, scale = act ? 1.0 + fabs(z) + zabs : 0.0;
    team_sum2<TL>(inc, scale, tm);
    return inc <= tol * scale;
}

// the friction coefficient of v^(l-1) at the lane's momentum point (a constant
// field: its value).  w: the scratch of square.  Not inlined: both paths of the
// stage update call it.
template <int R, typename Pix, int MODE>
__device__ __noinline__ double stage_gamma(const Dev& d, const FxStage& fs, int buf, int64_t k, double man,
                                           int2* w, int lane, unsigned tm) {
    using S = Sz<R>;
    constexpr int ND1 = S::ND1, ND = S::ND, NG = S::NG;
    const bool act = lane < ND;
    const size_t idx = (size_t)k * ND + (act ? lane : 0);
    const unsigned cmp = d.cmask[(size_t)buf * d.n + k];
    const double q0 = ufield(d, buf, 1, ND)[idx], q1 = ufield(d, buf, 2, ND)[idx];
    double z = ufield(d, buf, 0, ND)[idx], V, A;
    double q[2] = {q0, q1}, gam = 0.0;
    if (!(cmp & 1u)) z = square_one<ND1>(fs.Bg, fs.tBg, z, w, lane, tm);
    if ((cmp & 6u) != 6u) square2<ND1>(fs.Bg, fs.tBg, q, w, lane, tm);
    if (cmp & 2u) q[0] = q0;
    if (cmp & 4u) q[1] = q1;
    if (act) {
        Site<R, Pix, MODE>::VA(d, *d.tabs, k, SET_MOM, lane % NG, lane / NG, z, V, A);
        gam = gamma_manning<double>(man, V, q[0], q[1], d.g, d.eps);
    }
    return gam;
}

// Position v of a launch -> group of cells: from both ends of the mesh inwards,
// STAGE_RUN groups from the end, then as many from the start, and so on: the cells
// that take several times as long (pixel sums, Newton steps) lie at the shore, and
// shores lie at the edge of a domain rather than in its middle, so the launch does
// not end on them, at whichever end they are.  A run is about what the chip holds
// at once: neighbours run at the same time, do much the same and share the
// instruction cache.  Measured, a stage of the lagoon (r = 2, 44,000 cells, the
// shore last): 405 us in the mesh's order, 320 so; groups from the two ends in turn
// 331, 61 stretches of the mesh interleaved 394.
constexpr unsigned STAGE_RUN = 1024;
__device__ __forceinline__ unsigned from_both_ends(unsigned v, unsigned ng) {
    const unsigned i = v / (2 * STAGE_RUN) * STAGE_RUN + v % STAGE_RUN;
    return v / STAGE_RUN & 1 ? i : ng - 1 - i;
}

template <int R, typename Pix, int MODE>
__global__ void __maxnreg__(72)
    k_stage(const __grid_constant__ Dev d, const __grid_constant__ StageArgs sa) {
    using S = Sz<R>;
    using L = StageFx<R>;
    using ST = Site<R, Pix, MODE>;
    constexpr int ND1 = S::ND1, ND = S::ND, NM = S::NM, NMP = S::NMP, NG = S::NG, NGP = S::NGP;
    constexpr int TL = L::TL, PP = L::PP;
    __shared__ FxStage fs;
    copy_table(fs, &d.tabs->fs);
    const Tables& tb = *d.tabs;
    extern __shared__ double smem[];
    const int team = threadIdx.x / TL, lane = threadIdx.x % TL, tpb = blockDim.x / TL;
    const unsigned tm = 0xFFFFu << (threadIdx.x & 16); // the team's lanes
    int2* w = (int2*)(smem + team * L::words); // digit pairs of nodal fields, and scratch
    int2* qd = w + L::W;                       // [NMP] mass-point digits, then scratch [2 NMP]
    int2* qt = qd + NMP;
    double* cw = (double*)(qd + L::Q); // [NMP] weights of a mass-matrix solve
    double* bv = cw + L::CW;           // [ND] its right-hand side and solution
    double* un = bv + L::BV;
    float* Mf = (float*)un;            // the FP32 inverse's scratch
    double* M = un;                    // the fallback's matrix, packed
    const int64_t n = d.n;
    const bool act = lane < ND;
    const int node = act ? lane : 0;
    int its_max = 0;
    int viol = 0, fb = 0, bad = 0;
    const double dt_all = d.memb ? 0.0 : get_dt(d, 0);
    const double w2 = fs.wg[node % NG] * fs.wg[node / NG]; // the lane's momentum weight
    double wm2[PP];                                        // its mass weights
#pragma unroll
    for (int j = 0; j < PP; ++j) {
        const int p = lane + j * TL;
        wm2[j] = p < NMP ? fs.wm[p % NM] * fs.wm[p / NM] : 0.0;
    }
    const float tolf = (float)d.newton_tol;

    const unsigned ng = (unsigned)((n + tpb - 1) / tpb);
#pragma unroll 1
    for (unsigned v = blockIdx.x; v < ng; v += gridDim.x) {
        const int64_t k = (int64_t)from_both_ends(v, ng) * tpb + team;
        if (k >= n) continue;
        const size_t idx = (size_t)k * ND + node;
        const unsigned cm0 = d.cmask[k];
        const double hx = d.hxhy[2 * k], hy = d.hxhy[2 * k + 1], J = hx * hy;
        const double man = d.manning[k];
        int flag = d.flag[k];
        const double dt = d.memb ? get_dt(d, d.memb[k]) : dt_all; // the member's step
        const double u0 = ufield(d, 0, 0, ND)[idx];               // zeta^n
        // right-hand sides of Eqs. algebraic_elevation, algebraic_discharge, algebraic_concentration
        const double hn = d.HN[idx], cn0 = d.CN[idx];
        double T, rq[2], rc, tsum = 0.0;
        {
            double sf = 0.0, sgx = 0.0, sgy = 0.0, sr = 0.0;
#pragma unroll 1
            for (int m = 0; m < sa.nres; ++m) {
                const bool lin = sa.use_llin && (m == sa.nres - 1);
                const double lx = lin ? d.llin[idx] : rfield(d, m, 4, ND)[idx];
                const double ly = lin ? d.llin[(size_t)n * ND + idx] : rfield(d, m, 5, ND)[idx];
                sf += sa.wa[m] * rfield(d, m, 0, ND)[idx];
                sgx += sa.wa[m] * rfield(d, m, 1, ND)[idx] + sa.wat[m] * lx;
                sgy += sa.wa[m] * rfield(d, m, 2, ND)[idx] + sa.wat[m] * ly;
                sr += sa.wa[m] * rfield(d, m, 3, ND)[idx];
            }
            sf *= dt;
            T = hn + sf;
            if (act) tsum = sf;
            rq[0] = dt * sgx;
            rq[1] = dt * sgy;
            rc = cn0 + dt * sr;
        }
        const double Tbar = d.HNbar[k] + team_sum<TL>(tsum, tm);
        if (Tbar < 0.0) viol++;
        bool scalar = (flag == 0);
        int its = 0;
        double z = u0;     // Newton iterate
        double V[PP], A[PP];
        // elevations at the lane's mass points of the nodal values v (cst: a constant field)
        auto mass_points = [&](double v, bool cst, double (&pe)[PP]) {
            const double v0 = __shfl_sync(tm, v, 0, TL);
            const int e = team_exp(act ? v : 0.0, tm);
            if (act) w[lane] = fx::split(fx::from_double(v, e));
            __syncwarp(tm);
            fx_tens<ND1, NM, TL>(fs.Bm, w, qt, lane, tm, [&](int it, int, long long X) {
                pe[it] = cst ? v0 : fx::to_double(X, e + 2 * fs.tBm);
            });
            __syncwarp(tm);
        };
        if (!scalar) {
            bool zc = (cm0 & 1u) != 0;
            bool prev_full = false;
            // every mass point fully wet at zeta^n (known from the step start,
            // which evaluated H(zeta^n) = HN from the same state): the first
            // Newton step needs no evaluation, since H(zeta^n) - T = HN - T and
            // M(zeta^n) is the constant mass matrix
            const bool full0 = d.wet0 != nullptr && d.wet0[k] != 0 && d.newton_max > 0;
            // each pass evaluates V, A at the current iterate; the last pass is
            // the evaluation at the result (for the tracer matrix and the
            // completely-dry test)
#pragma unroll 1
            for (int kk = 0;; ++kk) {
                int npart = 0;
                double o;
                if (kk == 0 && full0) {
                    o = hn - T;
                } else {
                    double pe[PP];
                    mass_points(z, zc, pe);
                    bool dry = false, part = false;
#pragma unroll
                    for (int j = 0; j < PP; ++j) {
                        const int p = lane + j * TL;
                        if (p < NMP) {
                            bool full;
                            ST::VA(d, tb, k, SET_MASS, p % NM, p / NM, pe[j], V[j], A[j], full);
                            if (zero_bits(A[j])) dry = true;
                            else if (!full) part = true;
                        }
                    }
                    if (__any_sync(tm, dry)) { scalar = true; break; }
                    npart = __any_sync(tm, part);
                    // every pixel wet at the previous and at this iterate: H is affine
                    // on the segment between them and M(previous) is its exact
                    // Jacobian, so this iterate solves H = T (the fully wet case of
                    // Sec. 3.4); no verification step is needed
                    if (kk > 0 && prev_full && npart == 0) break;
                    if (kk == d.newton_max) break;
                    // H_i(zeta_k)
                    double hv[PP];
                    unsigned m = 0;
#pragma unroll
                    for (int j = 0; j < PP; ++j) {
                        hv[j] = lane + j * TL < NMP ? J * wm2[j] * V[j] : 0.0;
                        m = max(m, fx::mag(hv[j]));
                    }
                    const int e = fx::block_exp(__reduce_max_sync(tm, m));
#pragma unroll
                    for (int j = 0; j < PP; ++j)
                        if (lane + j * TL < NMP) qd[lane + j * TL] = fx::split(fx::from_double(hv[j], e));
                    __syncwarp(tm);
                    double H = 0.0;
                    fx_tens<NM, ND1, TL>(fs.BmT, qd, qt, lane, tm, [&](int, int, long long X) {
                        H = fx::to_double(X, e + 2 * fs.tBmT);
                    });
                    o = H - T;
                    __syncwarp(tm);
                }
                double dz[1] = {o};
                if (npart == 0) {
                    // M is the constant mass matrix, inverted by its tensor factors
                    dz[0] = square_one<ND1>(fs.M1i, fs.tM1i, dz[0], w, lane, tm);
                    dz[0] *= d.ihxhy[2 * k] * d.ihxhy[2 * k + 1];
                } else {
                    if (act) bv[lane] = o;
#pragma unroll
                    for (int j = 0; j < PP; ++j)
                        if (lane + j * TL < NMP) cw[lane + j * TL] = J * wm2[j] * A[j];
                    __syncwarp(tm);
                    if (!solve_mass_mixed<ND1, NM, TL>(tb, fs, cw, bv, Mf, w, qd, qt, M, (double*)w,
                                                       (double*)qd, lane, tm)) {
                        scalar = true;
                        break;
                    }
                    dz[0] = bv[node];
                    __syncwarp(tm);
                }
                z -= dz[0];
                // the stopping test, sums of magnitudes against newton_tol of their scale, in
                // FP32 where that decides it (its error is below 1e-6 of either side)
                float inc = 0.0f, scale = 0.0f;
                if (act) {
                    inc = f32_of(fabs(dz[0]));
                    scale = 1.0f + f32_of(fabs(z)) + f32_of(d.zabs[k]);
                }
#pragma unroll
                for (int s = TL / 2; s > 0; s >>= 1) {
                    inc += __shfl_xor_sync(tm, inc, s);
                    scale += __shfl_xor_sync(tm, scale, s);
                }
                its++;
                prev_full = (npart == 0);
                const double z0 = __shfl_sync(tm, z, 0, TL);
                zc = __all_sync(tm, !act || same_bits(z, z0));
                const float lim = tolf * scale;
                bool done = inc <= lim;
                if (!(fabsf(inc - lim) > 1e-5f * lim && lim > 1e-30f))
                    done = newton_done<TL>(dz[0], z, d.zabs[k], d.newton_tol, act, tm);
                if (done) prev_full = false, kk = d.newton_max - 1;
            }
            if (scalar) {
                fb++;
                flag = 0;
                if (lane == 0) d.flag[k] = 0;
            }
        }
        // v^(l-1) at the lane's momentum point (a constant field: its value), the
        // discharges in T; then the friction coefficient there
        const bool need_gam = (sa.add != 0.0 || sa.make_llin) && !zero_bits(man);
        // v^n's discharges at the momentum point, interpolated
        auto q_points = [&](double (&v)[2]) {
            const double q0 = ufield(d, 0, 1, ND)[idx], q1 = ufield(d, 0, 2, ND)[idx];
            v[0] = q0;
            v[1] = q1;
            if ((cm0 & 6u) != 6u) square2<ND1>(fs.Bg, fs.tBg, v, w, lane, tm);
            if (cm0 & 2u) v[0] = q0;
            if (cm0 & 4u) v[1] = q1;
        };
        double oz, oq[2], oc, ll[2];
        const double gam =
            need_gam ? stage_gamma<R, Pix, MODE>(d, fs, sa.prev_buf, k, man, w, lane, tm) : 0.0;
        double qn[2]; // q^n at the point, from the step start
        if (d.qpts) {
            qn[0] = d.qpts[k * 2 * NGP + node];
            qn[1] = d.qpts[k * 2 * NGP + NGP + node];
        } else {
            q_points(qn);
        }
        const double wp = J * w2;
        if (scalar) {
            double e;
            if (cm0 & 1u) e = u0;
            else {
                double pe[PP], s = 0.0;
                mass_points(u0, false, pe);
#pragma unroll
                for (int j = 0; j < PP; ++j)
                    if (lane + j * TL < NMP) s += wm2[j] * pe[j];
                e = team_sum<TL>(s, tm);
            }
            its = scalar_newton<R, Pix, MODE, TL>(d, tb, k, J, Tbar, e, lane, tm);
            // momentum: sums of the rows of the friction-modified mass matrix
            double den = 0.0, num[2] = {0.0, 0.0}, rs0 = 0.0, rs1 = 0.0, rcs = 0.0;
            if (act) {
                den = wp * (1.0 + sa.add * dt * gam);
                num[0] = wp * qn[0];
                num[1] = wp * qn[1];
                rs0 = rq[0];
                rs1 = rq[1];
                rcs = rc - cn0;
            }
            team_sum2<TL>(den, rcs, tm);
            team_sum2<TL>(num[0], rs0, tm);
            team_sum2<TL>(num[1], rs1, tm);
            oz = e;
            oq[0] = (num[0] + rs0) / den;
            oq[1] = (num[1] + rs1) / den;
            const double Hs = mass_scalar_pixels<R, Pix, MODE, TL>(d, tb, k, J, e, lane, tm).H;
            oc = Hs > 1e-14 * J * d.hlim ? (d.CNbar[k] + rcs) / Hs : ufield(d, 0, 3, ND)[idx];
            if (sa.make_llin) {
                ll[0] = -(wp * gam) * oq[0];
                ll[1] = -(wp * gam) * oq[1];
                square2<ND1>(fs.BgT, fs.tBgT, ll, w, lane, tm);
            }
        } else {
            // momentum (Eq. algebraic_discharge with the friction-modified mass
            // matrix of Eq. mass_matrix_discharge on the (r+1)^2 Gauss-Legendre
            // points, inverted as S^-1 D^-1 S^-T): S Q = [D0 q^n + S^-T rq] / D,
            // D = D0 (1 + add dt gamma), D0 = J w, gamma from the previous stage;
            // optionally the linearised friction term Llin = -S^T (J w gamma S Q)
            double s[2] = {rq[0], rq[1]};
            square2<ND1>(fs.GiT, fs.tGiT, s, w, lane, tm);
            const double rD = 1.0 / (wp * (1.0 + sa.add * dt * gam));
            s[0] = (wp * qn[0] + s[0]) * rD;
            s[1] = (wp * qn[1] + s[1]) * rD;
            oq[0] = s[0];
            oq[1] = s[1];
            square2<ND1>(fs.Gi, fs.tGi, oq, w, lane, tm);
            if (sa.make_llin) {
                const double wl = wp * gam;
                ll[0] = -wl * s[0];
                ll[1] = -wl * s[1];
                square2<ND1>(fs.BgT, fs.tBgT, ll, w, lane, tm);
            }
            oz = z;
            // tracer: H(zeta^(l)) C = C~ + dt sum a R with the depth-weighted mass matrix
            if (act) bv[lane] = rc;
#pragma unroll
            for (int j = 0; j < PP; ++j)
                if (lane + j * TL < NMP) cw[lane + j * TL] = J * wm2[j] * V[j];
            __syncwarp(tm);
            solve_mass_mixed<ND1, NM, TL>(tb, fs, cw, bv, Mf, w, qd, qt, M, (double*)w, (double*)qd, lane,
                                          tm);
            oc = bv[node];
            __syncwarp(tm);
        }
        if (sa.make_llin && act) {
            d.llin[idx] = ll[0];
            d.llin[(size_t)n * ND + idx] = ll[1];
        }
        // write v^(l) and its constant-field mask
        const double ov[4] = {oz, oq[0], oq[1], oc};
        unsigned cmo = 0;
        bool fin = true;
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            const double v0 = __shfl_sync(tm, ov[f], 0, TL);
            if (__all_sync(tm, !act || same_bits(ov[f], v0))) cmo |= 1u << f;
            fin = fin && finite_bits(ov[f]);
            if (act) ufield(d, sa.out_buf, f, ND)[idx] = ov[f];
        }
        if (!__all_sync(tm, fin || !act)) bad = 1;
        if (lane == 0) d.cmask[(size_t)sa.out_buf * n + k] = (uint8_t)cmo;
        its_max = max(its_max, its);
        __syncwarp(tm);
    }
    if (lane == 0) {
        if (its_max) atomicMax(&d.sc->maxits, its_max);
        if (viol) atomicAdd(&d.sc->viol, viol);
        if (fb) atomicAdd(&d.sc->fallback, fb);
        if (bad) atomicOr(&d.sc->status, ST_NAN);
    }
    if (sa.final_ && blockIdx.x == 0) {
        // every member advances by its own step (rmax is not written here)
#pragma unroll 1
        for (int i = threadIdx.x; i < d.nmemb; i += blockDim.x) {
            const double dti = get_dt(d, i);
            d.mb[i].dt_last = dti;
            d.mb[i].t = d.mb[i].t + dti;
        }
    }
}

// ---------------------------------------------------------------------------
// constant-field masks of a state buffer
// ---------------------------------------------------------------------------
template <int R>
__global__ void k_masks(const __grid_constant__ Dev d, int buf) {
    constexpr int ND = Sz<R>::ND;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
    for (int64_t k = (int64_t)blockIdx.x * wpb + warp; k < d.n; k += (int64_t)gridDim.x * wpb) {
        unsigned cm = 0;
        for (int f = 0; f < 4; ++f) {
            const double* u = ufield(d, buf, f, ND) + k * ND;
            bool eq = true;
            for (int i = lane; i < ND; i += 32) eq = eq && same_bits(u[i], u[0]);
            if (__all_sync(0xffffffffu, eq)) cm |= (1u << f);
            if (d.uF)
                for (int i = lane; i < ND; i += 32) ufieldF(d, buf, f, ND)[k * ND + i] = (float)u[i];
        }
        if (lane == 0) d.cmask[(size_t)buf * d.n + k] = (uint8_t)cm;
    }
}

// ---------------------------------------------------------------------------
// diagnostics: per-cell wet mass (Eq. positivity-7), tracer mass, min depth
// ---------------------------------------------------------------------------
template <int R, typename Pix, int MODE>
__global__ void __launch_bounds__(32 * MAXWPB)
    k_cell_diag(const __grid_constant__ Dev d, const __grid_constant__ Tables tb, double* part) {
    using S = Sz<R>;
    constexpr int ND1 = S::ND1, ND = S::ND, NM = S::NM, NMP = S::NMP;
    extern __shared__ double smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
    double* su = smem + warp * (2 * ND + 2 * NMP + 2 * NM * NM);
    double* pe = su + 2 * ND;
    double* pc = pe + NMP;
    double* tmp = pc + NMP;
    for (int64_t k = (int64_t)blockIdx.x * wpb + warp; k < d.n; k += (int64_t)gridDim.x * wpb) {
        for (int i = lane; i < ND; i += 32) {
            su[i] = ufield(d, 0, 0, ND)[k * ND + i];
            su[ND + i] = ufield(d, 0, 3, ND)[k * ND + i];
        }
        const unsigned cm = d.cmask[k];
        const double J = d.hxhy[2 * k] * d.hxhy[2 * k + 1];
        __syncwarp();
        tens_interp<ND1, NM>(tb.Bm, su, tmp, pe, lane);
        tens_interp<ND1, NM>(tb.Bm, su + ND, tmp, pc, lane);
        double m = 0.0, tm = 0.0, hmin = INFINITY;
        for (int p = lane; p < NMP; p += 32) {
            const double e = (cm & 1u) ? su[0] : pe[p];
            const double c = (cm & 8u) ? su[ND] : pc[p];
            double V, A;
            Site<R, Pix, MODE, false>::VA(d, tb, k, SET_MASS, p % NM, p / NM, e, V, A);
            const double w = J * tb.wm[p % NM] * tb.wm[p / NM];
            m += w * V;
            tm += w * V * c;
            hmin = fmin(hmin, V);
        }
        m = warp_sum(m);
        tm = warp_sum(tm);
        hmin = warp_min(hmin);
        if (lane == 0) {
            part[4 * k + 0] = m;
            part[4 * k + 1] = tm;
            part[4 * k + 2] = hmin;
            part[4 * k + 3] = d.flag[k] ? 1.0 : 0.0;
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// zeta at gauge points (Lagrange product formula, Sec. 3.2)
// ---------------------------------------------------------------------------
template <int R>
__global__ void k_gauges(const __grid_constant__ Dev d, const __grid_constant__ Tables tb, int ng,
                         const double* xy, double* out, int64_t k0, int64_t k1,
                         const int32_t* cell) {
    constexpr int ND1 = R + 1, ND = ND1 * ND1;
    const int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= ng) return;
    const double x = xy[2 * gi], y = xy[2 * gi + 1];
    double v = NAN;
    // the cells searched: [k0, k1), or only the one located on the host (cell[gi], -1: none)
    if (cell) {
        k0 = cell[gi];
        k1 = k0 < 0 ? k0 : k0 + 1;
    }
    for (int64_t k = k0; k < k1; ++k) {
        const double x0 = d.x0y0[2 * k], y0 = d.x0y0[2 * k + 1], hx = d.hxhy[2 * k],
                     hy = d.hxhy[2 * k + 1];
        if (x >= x0 && x <= x0 + hx && y >= y0 && y <= y0 + hy) {
            const double* u = ufield(d, 0, 0, ND) + k * ND;
            if (d.cmask[k] & 1u) { v = u[0]; break; }
            const double xi = (x - x0) / hx, eta = (y - y0) / hy;
            double lx[ND1], ly[ND1];
            for (int a = 0; a < ND1; ++a) {
                double px = 1.0, py = 1.0;
                for (int b = 0; b < ND1; ++b)
                    if (b != a) {
                        px *= (xi - tb.xs[b]) / (tb.xs[a] - tb.xs[b]);
                        py *= (eta - tb.xs[b]) / (tb.xs[a] - tb.xs[b]);
                    }
                lx[a] = px;
                ly[a] = py;
            }
            double s = 0.0;
            for (int b = 0; b < ND1; ++b)
                for (int a = 0; a < ND1; ++a) s += u[a + ND1 * b] * lx[a] * ly[b];
            v = s;
            break;
        }
    }
    out[gi] = v;
}

} // namespace swdg
