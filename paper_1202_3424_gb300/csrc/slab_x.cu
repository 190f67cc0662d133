// The slab matvec (slab.cuh): its x passes, its copy of the Green tensor, and
// the launcher.
#include "slab.h"

#include "slab.cuh"

namespace dda {

namespace {

// Radix plan variants of the warp-local rows (XwPlan), by the fused mode of the
// matvec: plan 0 (fewer points per lane) or plan 1 (fewer exchanges through
// shared memory), us per launch with plan 0 / 1 by row length:
//                                    128a       192b       256c       512d
//   forward, plain gather          16.4/14.6   110/114    54/42      55/46
//   forward, in a solve            19.8/22.7   167/198    68/72      69/-
//   inverse, plain                 14.3/14.3   184/170    84/71      93/99
//   inverse, in a solve            20.1/20.9   220/182    86/86      88/103
// (a 64^3 sphere, 2 RHS; b 96x64x32 ellipsoid, 32 RHS; c 128x48x24, 16 RHS; d
// 256x48x24, 8 RHS.)  A plain gather takes plan 1 up to 256 points; the BiCGstab
// gathers, which hold up to seven operands per point, plan 0; the inverse plan 1
// at 192 and 256 points.  (512 points still gather with plan 0.)
template <int LX, int MODE> constexpr int kPlanFwd = MODE == 0 && (LX == 128 || LX == 192 || LX == 256) ? 1 : 0;
template <int LX> constexpr int kPlanInv = LX == 192 || LX == 256 ? 1 : 0;

template <int LX, int MODE>
cudaError_t xfwd_mode(const Geom& g, int R, float2* x, float2* u, const DevTarget& tg, const float2* tw,
                      const int* active, const FusedKrylov<float>& fk, cudaStream_t st) {
    constexpr int V = kPlanFwd<LX, MODE>;
    using PL = XwPlan<LX, V>;
    const size_t sm = xw_tile_bytes<PL>(xw_rows<PL>()) + (xw_shared_twiddles<LX>() ? LX * sizeof(float2) : 0);
    const int nrows = g.ny * g.nz;
    dim3 grid((nrows + xw_rows<PL>() - 1) / xw_rows<PL>(), 3, R);
    RowMap rm = row_map(g);
    rm.pitch = nrows;
    cudaError_t e = allow_smem(k_xfwd_w<LX, V, MODE, true>, sm);
    if (e != cudaSuccess) return e;
    PROF_BEGIN(st);
    k_xfwd_w<LX, V, MODE, true><<<grid, kXwThreads, sm, st>>>(x, u, rm, tg.site_of, nrows, g.N, tw, active,
                                                              fwd_vecs(fk));
    PROF_END(KK_XFWD_C64, R, st);
    return cudaGetLastError();
}
template <int LX>
cudaError_t xfwd(const Geom& g, int R, float2* x, float2* u, const DevTarget& tg, const float2* tw, const int* active,
                 const FusedKrylov<float>& fk, cudaStream_t st) {
    if (fk.mode == 0) return xfwd_mode<LX, 0>(g, R, x, u, tg, tw, active, fk, st);
    if (fk.mode == 1) return xfwd_mode<LX, 1>(g, R, x, u, tg, tw, active, fk, st);
    if (fk.mode == 2) return xfwd_mode<LX, 2>(g, R, x, u, tg, tw, active, fk, st);
    return xfwd_mode<LX, 3>(g, R, x, u, tg, tw, active, fk, st);
}

template <int LX, int MODE, int DIAG>
cudaError_t xinv_mode(const Geom& g, int R, const float2* u, float2* y, const float2* x, const DevTarget& tg,
                      const float2* beta, int beta_stride, const float2* tw, int* active,
                      const FusedKrylov<float>& fk, cudaStream_t st) {
    constexpr int V = kPlanInv<LX>;
    using PL = XwPlan<LX, V>;
    constexpr int rows = xwi_rows<PL, true>();
    const size_t sm = xw_tile_bytes<PL>(rows);
    const int nrows = tg.rows != nullptr ? tg.nrows : g.ny * g.nz;
    dim3 grid((nrows + rows - 1) / rows, 3, R);
    RowMap rm = row_map(g);
    rm.pitch = g.ny * g.nz;
    cudaError_t e = allow_smem(k_xinv_w<LX, V, MODE, DIAG, true>, sm);
    if (e != cudaSuccess) return e;
    PROF_BEGIN(st);
    k_xinv_w<LX, V, MODE, DIAG, true><<<grid, xwi_threads<PL, true>(), sm, st>>>(u, rm, y, x, tg.site_of, tg.comp_of, beta,
                                                                     beta_stride, tg.rows, nrows, g.N, tw, active,
                                                                     fk.rhat, fk.st, fk.part, fk.cnt, fk.part_stride);
    PROF_END(KK_XINV_C64, R, st);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return fused_finalize<float>(fk.mode, R, (int)(grid.x * grid.y), fk, active, st);
}
template <int LX>
cudaError_t xinv(const Geom& g, int R, const float2* u, float2* y, const float2* x, const DevTarget& tg,
                 const float2* beta, int beta_stride, const float2* tw, int* active, const FusedKrylov<float>& fk,
                 cudaStream_t st) {
    auto by_mode = [&](auto d) -> cudaError_t {
        constexpr int D = decltype(d)::value;
        const int mode = inverse_mode(fk.mode);
        if (mode == 0) return xinv_mode<LX, 0, D>(g, R, u, y, x, tg, beta, beta_stride, tw, active, fk, st);
        if (mode == 1) return xinv_mode<LX, 1, D>(g, R, u, y, x, tg, beta, beta_stride, tw, active, fk, st);
        return xinv_mode<LX, 2, D>(g, R, u, y, x, tg, beta, beta_stride, tw, active, fk, st);
    };
    // (anisotropic materials keep the separate passes)
    if (tg.comp_of == nullptr) return by_mode(std::integral_constant<int, kDiagSite>{});
    return by_mode(std::integral_constant<int, kDiagComp>{});
}

using SlabFn = cudaError_t (*)(const Geom&, int, float2*, const float4*, const Twiddles<float>&, const int*,
                               cudaStream_t);
SlabFn slab_fn(const Geom& g) {
    switch (g.Ly) {
        case 16: return slab_fn_16(g.Lz);
        case 32: return slab_fn_32(g.Lz);
        case 48: return slab_fn_48(g.Lz);
        case 64: return slab_fn_64(g.Lz);
        case 96: return slab_fn_96(g.Lz);
        case 128: return slab_fn_128(g.Lz);
        default: return nullptr;
    }
}

}  // namespace

bool slab_built(const Geom& g) { return slab_fn(g) != nullptr; }

int64_t slab_green_size(const Geom& g) { return slab_green_all(g.hx(), g.Ly, g.Lz); }

cudaError_t launch_slab_green(const Geom& g, const double2* gh64, float4* out, cudaStream_t st) {
    auto go = [&](auto kern) {
        kern<<<grid1d(slab_green_size(g), 256), 256, 0, st>>>(gh64, out, g.hx(), g.Ly);
        return cudaGetLastError();
    };
    switch (g.Lz) {
        case 16: return go(k_slab_green<16>);
        case 32: return go(k_slab_green<32>);
        case 48: return go(k_slab_green<48>);
        case 64: return go(k_slab_green<64>);
        case 96: return go(k_slab_green<96>);
        case 128: return go(k_slab_green<128>);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_slab_matvec(const Geom& g, int R, float2* x, float2* y, const PadWork<float>& w, const DevTarget& tg,
                               const float2* beta, int beta_stride, const Twiddles<float>& tw, int* active,
                               const FusedKrylov<float>& fk, cudaStream_t st) {
    SlabFn slab = slab_fn(g);
    if (slab == nullptr || w.beta_tensor) return cudaErrorInvalidValue;
    auto fwdx = [&]() -> cudaError_t { DDA_DISPATCH_L(g.Lx, xfwd, g, R, x, w.u2, tg, tw.x, active, fk, st); };
    auto invx = [&]() -> cudaError_t {
        DDA_DISPATCH_L(g.Lx, xinv, g, R, w.u2, y, x, tg, beta, beta_stride, tw.x, active, fk, st);
    };
    cudaError_t e;
    if ((e = fwdx()) != cudaSuccess) return e;
    if ((e = slab(g, R, w.u2, w.slab, tw, active, st)) != cudaSuccess) return e;
    return invx();
}

}  // namespace dda
