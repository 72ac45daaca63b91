// swdg_degree.cuh -- launchers of one polynomial degree (included once by each
// swdg_r{1,2,3}.cu with SWDG_DEGREE defined).
#pragma once
#include "swdg_adjoint.cuh"
#include "swdg_bulk.cuh"
#include "swdg_amr.cuh"
#include "swdg_kernels.cuh"
#include "swdg_launch.h"

namespace swdg {

template <int R, typename Pix, int MODE, typename B>
struct Launchers {
    using S = Sz<R>;
    static constexpr bool F64 = sizeof(B) == sizeof(double);
    // shared memory per warp
    static constexpr size_t res_b =
        sizeof(double) * (F64 ? ResFx<R>::words : bulk::Res<R>::words) * (32 / ResFx<R>::TL);
    static constexpr int begin_cells = F64 ? 2 : 32 / bulk::begin_team<R>(); // per warp
    static constexpr size_t begin_b =
        sizeof(double) * begin_cells * (F64 ? BeginFx<R>::words : bulk::begin_smem<R>());
    static constexpr size_t stage_b =
        2 * sizeof(double) * (F64 ? StageFx<R>::words : bulk::stage_smem<R>());
    static auto residual_kernel() {
        if constexpr (F64) return k_residual<R, Pix, MODE>;
        else return bulk::k_residual<R, Pix, MODE>;
    }
    static auto begin_kernel() {
        if constexpr (F64) return k_step_begin<R, Pix, MODE>;
        else return bulk::k_step_begin<R, Pix, MODE>;
    }
    static auto stage_kernel() {
        if constexpr (F64) return k_stage<R, Pix, MODE>;
        else return bulk::k_stage<R, Pix, MODE>;
    }
    static constexpr size_t diag_b = sizeof(double) * (2 * S::ND + 2 * S::NMP + 2 * S::NM * S::NM);
    static constexpr size_t vjp_b = sizeof(double) * vjp_smem<R>() * (32 / VjpTeam<R>::TL); // per warp
    static constexpr size_t svjp_b = 2 * sizeof(double) * stage_vjp_smem<R>(); // two cells per warp
    static constexpr size_t bvjp_b = sizeof(double) * begin_vjp_smem<R>();
    static constexpr size_t ind_b = sizeof(double) * indicator_smem<R>();
    static constexpr size_t remap_b = sizeof(double) * remap_smem<R>();

    static void residual(const Dev& d, int buf, int stage, double c_stage,
                         int want_dt, Shape s, cudaStream_t st) {
        // 32 / TL cells per warp: no more blocks than their cells
        const int cpb = s.wpb * 32 / ResFx<R>::TL;
        const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(s.grid, (d.n + cpb - 1) / cpb));
        if constexpr (F64) {
            if (MODE == 0 && !d.fflux)
                k_residual<R, Pix, 0, true><<<grid, 32 * s.wpb, res_b * s.wpb, st>>>(d, buf, stage,
                                                                                     c_stage, want_dt);
            else
                k_residual<R, Pix, MODE><<<grid, 32 * s.wpb, res_b * s.wpb, st>>>(d, buf, stage, c_stage,
                                                                                  want_dt);
        } else {
            bulk::k_residual<R, Pix, MODE><<<grid, 32 * s.wpb, res_b * s.wpb, st>>>(d, buf, stage);
        }
    }
    static void faces(const Dev& d, int buf, double c_stage, int want_dt,
                      cudaStream_t st) {
        if (d.njobs <= 0) return;
        // one point per lane and one pass; 4 warps a block, so that small meshes spread
        // over the SMs (256 cells, r = 1: 14.2 us with 8 warps, 12.3 with 4; the FP32-bulk
        // ensemble 279 and 266)
        const int64_t blocks = (d.njobs + 127) / 128;
        if constexpr (F64)
            k_faces<R, Pix, MODE><<<(int)blocks, 128, 0, st>>>(d, buf, c_stage, want_dt);
        else
            bulk::k_faces<R, Pix, MODE><<<(int)blocks, 128, 0, st>>>(d, buf, c_stage, want_dt);
    }
    static void step_begin(const Dev& d, int do_switch, Shape s, cudaStream_t st) {
        const int cpb = begin_cells * s.wpb;
        const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(s.grid, (d.n + cpb - 1) / cpb));
        if constexpr (F64)
            k_step_begin<R, Pix, MODE><<<grid, 32 * s.wpb, begin_b * s.wpb, st>>>(d, do_switch);
        else
            bulk::k_step_begin<R, Pix, MODE><<<grid, 32 * s.wpb, begin_b * s.wpb, st>>>(d, do_switch);
    }
    static void stage(const Dev& d, const StageArgs& sa, Shape s, cudaStream_t st) {
        // two cells per warp: no more blocks than 2 wpb cells each
        const int64_t need = (d.n + 2 * s.wpb - 1) / (2 * s.wpb);
        const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(s.grid, need));
        if constexpr (F64)
            k_stage<R, Pix, MODE><<<grid, 32 * s.wpb, stage_b * s.wpb, st>>>(d, sa);
        else
            bulk::k_stage<R, Pix, MODE><<<grid, 32 * s.wpb, stage_b * s.wpb, st>>>(d, sa);
    }
    static void masks(const Dev& d, int buf, Shape s, cudaStream_t st) {
        k_masks<R><<<s.grid, 32 * s.wpb, 0, st>>>(d, buf);
    }
    static void cell_diag(const Dev& d, const Tables& tb, double* part, Shape s, cudaStream_t st) {
        k_cell_diag<R, Pix, MODE><<<s.grid, 32 * s.wpb, diag_b * s.wpb, st>>>(d, tb, part);
    }
    static void gauges(const Dev& d, const Tables& tb, int ng, const double* xy, double* out,
                       int64_t k0, int64_t k1, const int32_t* cell, cudaStream_t st) {
        k_gauges<R><<<(ng + 63) / 64, 64, 0, st>>>(d, tb, ng, xy, out, k0, k1, cell);
    }
    static void gauges_vjp(const Dev& d, const Tables& tb, int ng, const double* xy,
                           const double* gbar, double* zb, const int32_t* cell, cudaStream_t st) {
        k_gauges_vjp<R><<<(ng + 63) / 64, 64, 0, st>>>(d, tb, ng, xy, gbar, zb, cell);
    }
    static void residual_vjp(const Dev& d, const double* u, const uint8_t* cm,
                             const double* rbar, double* ubar, double* nbar, double* dbar,
                             int accumulate, Shape s, cudaStream_t st) {
        const int cpb = s.wpb * 32 / VjpTeam<R>::TL;
        const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(s.grid, (d.n + cpb - 1) / cpb));
        k_residual_vjp<R, Pix, MODE><<<grid, 32 * s.wpb, vjp_b * s.wpb, st>>>(
            d, u, cm, rbar, ubar, nbar, dbar, accumulate);
    }
    static void stage_vjp(const Dev& d, const StageVjpArgs& a, Shape s,
                          cudaStream_t st) {
        const int64_t need = (d.n + 2 * s.wpb - 1) / (2 * s.wpb);
        const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(s.grid, need));
        k_stage_vjp<R, Pix, MODE><<<grid, 32 * s.wpb, svjp_b * s.wpb, st>>>(d, a);
    }
    static void begin_vjp(const Dev& d, const BeginVjpArgs& a, Shape s,
                          cudaStream_t st) {
        k_begin_vjp<R, Pix, MODE><<<s.grid, 32 * s.wpb, bvjp_b * s.wpb, st>>>(d, a);
    }
    static void indicator(const Dev& d, const Tables& tb, int kind, double* eta, Shape s,
                          cudaStream_t st) {
        k_indicator<R, Pix, MODE><<<s.grid, 32 * s.wpb, ind_b * s.wpb, st>>>(d, tb, kind, eta);
    }
    static void remap(const Tables& tb, const RemapArgs& a, Shape s, cudaStream_t st) {
        k_remap<R><<<s.grid, 32 * s.wpb, remap_b * s.wpb, st>>>(tb, a);
    }
    template <typename K>
    static bool opt_in(K kern, size_t per_warp) {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)(per_warp * MAXWPB)) == cudaSuccess;
    }
    static bool prepare() {
        if constexpr (F64)
            if (!opt_in(k_residual<R, Pix, 0, true>, res_b)) return false;
        return opt_in(residual_kernel(), res_b) &&
               opt_in(begin_kernel(), begin_b) &&
               opt_in(stage_kernel(), stage_b) &&
               opt_in(k_cell_diag<R, Pix, MODE>, diag_b) &&
               opt_in(k_residual_vjp<R, Pix, MODE>, vjp_b) &&
               opt_in(k_stage_vjp<R, Pix, MODE>, svjp_b) &&
               opt_in(k_begin_vjp<R, Pix, MODE>, bvjp_b);
    }
    template <typename K>
    static int occ(K kern, int wpb, size_t per_warp) {
        int nb = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, 32 * wpb, per_warp * wpb) !=
            cudaSuccess)
            return 0;
        return nb;
    }
    static int occupancy(int kind, int wpb) {
        if (wpb < 1 || wpb > MAXWPB) return 0;
        switch (kind) {
        case KK_BEGIN: return occ(begin_kernel(), wpb, begin_b);
        case KK_RESIDUAL: return occ(residual_kernel(), wpb, res_b);
        case KK_STAGE: return occ(stage_kernel(), wpb, stage_b);
        default: return occ(k_cell_diag<R, Pix, MODE>, wpb, diag_b);
        }
    }
    static void fill(Launch* L) {
        L->residual = &residual;
        L->faces = &faces;
        L->step_begin = &step_begin;
        L->stage = &stage;
        L->masks = &masks;
        L->cell_diag = &cell_diag;
        L->gauges = &gauges;
        L->gauges_vjp = &gauges_vjp;
        L->residual_vjp = &residual_vjp;
        L->stage_vjp = &stage_vjp;
        L->begin_vjp = &begin_vjp;
        L->indicator = &indicator;
        L->remap = &remap;
        L->prepare = &prepare;
        L->occupancy = &occupancy;
        L->nzp = Sz<R>::NZP;
    }
};

template <int R, typename B>
bool get_launch_prec(int mode, int pix, Launch* L) {
    if (mode == 1) Launchers<R, double, 1, B>::fill(L);
    else if (pix == 0) Launchers<R, float, 0, B>::fill(L);
    else if (pix == 1) Launchers<R, double, 0, B>::fill(L);
    else return false;
    return true;
}

// precision 0: FP64; 1: FP32-bulk residual arithmetic
template <int R>
bool get_launch_degree(int mode, int pix, int prec, Launch* L) {
    if (prec == 0) return get_launch_prec<R, double>(mode, pix, L);
    if (prec == 1) return get_launch_prec<R, float>(mode, pix, L);
    return false;
}

} // namespace swdg
