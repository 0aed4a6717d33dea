// Instantiation helpers shared by the per-precision translation units.
#pragma once

#include <algorithm>
#include <utility>
#include <vector>

#include "mhd_adjoint.cuh"
#include "mhd_aux.cuh"
#include "mhd_launch.h"
#include "mhd_step.cuh"

namespace mhd {

template <typename R>
static StepArgs<R> to_args(const StepHostArgs& h) {
    StepArgs<R> a;
    a.U = static_cast<const R*>(h.U);
    a.Unew = static_cast<R*>(h.Unew);
    a.slice = h.slice;
    a.dt_patch = h.dt_patch;
    a.patches = h.patches;
    a.tiles = h.tiles;
    a.ntiles = h.ntiles;
    a.nzb = h.nzb;
    a.ntiles_dev = h.ntiles_dev;
    a.dynamic = h.dynamic;
    a.work = h.work;
    a.dt_ptr = h.dt_ptr;
    a.dt_val = h.dt_val;
    a.gamma = R(h.gamma);
    a.gm1 = R(h.gamma - 1.0);
    a.gm1i = R(1.0 / (h.gamma - 1.0));
    a.eps = R(h.eps);
    for (int d = 0; d < 3; ++d) {
        a.dxi[d] = h.dxi[d];
        a.dxir[d] = R(h.dxi[d]);
    }
    a.limiter = h.limiter;
    a.riemann = h.riemann;
    a.err = h.err;
    return a;
}

// The chunks of a 3D plane shared out to the warps (StepPlan), longest first to the least loaded warp:
// in phase A the edges, the z-faces and the conversion, in phase B the prep, the other faces and the
// update.  Costs: cycles of a chunk with four warps per scheduler running, measured (FP32, 32x8); FP64
// operations (FP64, bound by that pipe).  False: a list is too long.
template <typename C>
static bool make_plan(StepPlan& plan) {
    constexpr bool F64 = C::EQ == 2;
    constexpr int PREP = F64 ? 330 : 2480, FACE = F64 ? 220 : 1450, EDGE = F64 ? 260 : 1400, CONV = F64 ? 40 : 620,
                  UPD = F64 ? 45 : 700;
    using Tasks = std::vector<std::pair<int, int>>;   // (cost, chunk)
    auto share = [&](Tasks tasks, int phase) {
        std::stable_sort(tasks.begin(), tasks.end(), [](const auto& x, const auto& y) { return x.first > y.first; });
        int load[C::NWARP] = {};
        Tasks list[C::NWARP];
        for (const auto& t : tasks) {
            const int w = (int)(std::min_element(load, load + C::NWARP) - load);
            list[w].push_back(t);
            load[w] += t.first;
        }
        for (int w = 0; w < C::NWARP; ++w) {
            // the short, latency-bound chunks at another place in the list of each warp of a
            // scheduler (warps w, w + 4, ...), so that the others have work meanwhile
            auto& L = list[w];
            if (L.size() > 1) std::rotate(L.begin(), L.end() - (w / 4) % (int)L.size(), L.end());
            if ((int)L.size() > 8 * C::NQ - (C::NQ > 1)) return false;
            plan.t[phase][w][0] = plan.t[phase][w][1] = ~0ull;
            for (size_t k = 0; k < L.size(); ++k)
                plan.t[phase][w][k / 8] ^= (255ull ^ (unsigned long long)L[k].second) << (8 * (k % 8));
        }
        return true;
    };
    Tasks A, B;
    for (int q = 0; q < C::NZ; ++q) A.emplace_back(q < C::IFZ::N ? FACE : EDGE, C::NI + q);
    for (int q = 0; q < C::IEZ::N; ++q) A.emplace_back(EDGE, C::IFX::N + C::IFY::N + q);
    for (int q = 0; q < C::ICV::N; ++q) A.emplace_back(CONV, C::NI + C::NZ + C::IPR::N + q);
    for (int q = 0; q < C::IPR::N; ++q) B.emplace_back(PREP, C::NI + C::NZ + q);
    for (int q = 0; q < C::IFX::N + C::IFY::N; ++q) B.emplace_back(FACE, q);
    for (int q = 0; q < C::IUP::N; ++q) B.emplace_back(UPD, C::NI + C::NZ + C::IPR::N + C::ICV::N + q);
    return share(A, 0) && share(B, 1);
}

template <typename R, int NDIM, int TX, int TY, int NT, int MINB = 1>
struct StepInst {
    using C = StepCfg<R, NDIM, TX, TY, NT, MINB>;
    static_assert((C::SMEM_BYTES + 1024) * MINB <= 228 * 1024, "tile too large for shared memory");
    static_assert(C::NI + C::NZ + C::IPR::N + C::ICV::N + C::IUP::N < 255 && C::NWARP >= 4 * (NDIM == 3) &&
                      C::NWARP <= StepPlan::MAXW,
                  "chunk numbers are bytes");
    // whole columns, z-blocks (3D), asynchronous stepping (which may use z-blocks)
    static constexpr auto whole = &step_kernel<R, NDIM, TX, TY, NT, MINB, false, false>;
    static constexpr auto split = &step_kernel<R, NDIM, TX, TY, NT, MINB, NDIM == 3, false>;
    static constexpr auto async = &step_kernel<R, NDIM, TX, TY, NT, MINB, NDIM == 3, true>;
    static const StepPlan* plan() {   // null: none
        static StepPlan p{};
        static const bool ok = NDIM != 3 || make_plan<C>(p);
        return ok ? &p : nullptr;
    }
    static cudaError_t prepare() {
        if (!plan()) return cudaErrorInvalidConfiguration;
        for (auto k : {whole, split, async}) {
            const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM_BYTES);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    }
    static cudaError_t occupancy(int* blocks) {
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, whole, NT, C::SMEM_BYTES);
    }
    static cudaError_t launch(const void* args, int grid, cudaStream_t s) {
        const StepArgs<R> a = to_args<R>(*static_cast<const StepHostArgs*>(args));
        const StepPlan& plan = *StepInst::plan();
        if (a.slice) launch_pdl(async, grid, NT, C::SMEM_BYTES, s, a, plan);
        else (a.nzb > 1 ? split : whole)<<<grid, NT, C::SMEM_BYTES, s>>>(a, plan);
        return cudaGetLastError();
    }
    static StepLaunch entry(float plane_us = 1, float alone_us = 1) {
        return StepLaunch{NDIM, C::TX, C::TY, NT, C::SMEM_BYTES, &prepare, &occupancy, &launch, plane_us, alone_us};
    }
};

template <typename R>
static cudaError_t launch_fill(void* U, const PatchDev* patches, int npatch, const FillGeom& fg,
                               const int64_t* nboff, int Zp, unsigned* err, cudaStream_t s) {
    if (nboff) {
        fill_grid_kernel<R><<<(unsigned)npatch * (unsigned)Zp, 128, 0, s>>>(static_cast<R*>(U), patches, nboff, Zp);
    } else {
        dim3 grid(8, npatch < 65535 ? npatch : 65535);
        fill_kernel<R><<<grid, 256, 0, s>>>(static_cast<R*>(U), patches, npatch, fg, err);
    }
    return cudaGetLastError();
}

template <typename R>
static cudaError_t prepare_fill_cfl() {
    return cudaFuncSetAttribute(fill_cfl_staged_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)FILL_CFL_STAGED_MAX_SMEM);
}

// the staged pass where the plane fits its shared-memory cap, else the register version
template <typename R>
static cudaError_t launch_fill_cfl(void* U, const PatchDev* patches, const PatchDev& h0, int npatch,
                                  const int64_t* nboff, int Zp, double gamma, double courant, const double dxi[3],
                                  const int act[3], void* partial, unsigned* counter, double* dt_out, unsigned* err,
                                  cudaStream_t s) {
    const unsigned grid = (unsigned)npatch * (unsigned)Zp;
    const size_t smem = fill_cfl_staged_smem<R>(h0.X, h0.Y, h0.nx, h0.ny, h0.gx, h0.gy);
    // constants in the kernel's precision, rounded here once (as the kernel would round them)
    const R g = R(gamma), gm1 = R(gamma - 1.0), d0 = R(dxi[0]), d1 = R(dxi[1]), d2 = R(dxi[2]);
    if (fill_cfl_staged_fits<R>(h0))
        fill_cfl_staged_kernel<R><<<grid, 256, smem, s>>>(static_cast<R*>(U), patches, nboff, Zp, g, gm1, courant, d0,
                                                          d1, d2, act[1], act[2], static_cast<R*>(partial), counter,
                                                          dt_out, err);
    else
        fill_cfl_grid_kernel<R><<<grid, 128, 0, s>>>(static_cast<R*>(U), patches, nboff, Zp, g, gm1, courant, d0, d1,
                                                     d2, act[1], act[2], static_cast<R*>(partial), counter, dt_out,
                                                     err);
    return cudaGetLastError();
}

template <typename R>
static cudaError_t launch_fill_interp(void* U0, void* U1, const PatchDev* patches, int npatch, const int* list,
                                     int nlist, const int* nlist_dev, int grid_y, const int* slice,
                                     const double* t_old, const double* t_cur, const FillGeom& fg,
                                     const int64_t* nboff, int Zp, int64_t pstride, unsigned* err, cudaStream_t s) {
    if (nlist <= 0) return cudaSuccess;
    if (nboff) {
        launch_pdl(fill_interp_grid_kernel<R>, interp_grid(nlist, Zp, grid_y), 128, 0, s, static_cast<R*>(U0), static_cast<R*>(U1), patches, nboff,
                   list, nlist, nlist_dev, pstride, Zp, slice, t_old, t_cur);
        return cudaGetLastError();
    }
    dim3 grid(32, std::min(std::min(nlist, grid_y > 0 ? grid_y : nlist), 65535));
    launch_pdl(fill_interp_kernel<R>, grid, 256, 0, s, static_cast<R*>(U0), static_cast<R*>(U1), patches, npatch, list, nlist,
                                               nlist_dev, slice, t_old, t_cur, fg, err);
    return cudaGetLastError();
}

template <typename R>
static cudaError_t launch_cfl_patch(const void* U0, const void* U1, const PatchDev* patches, const int* list,
                                   int nlist, const int* nlist_dev, int grid_y, const int* slice, double gamma,
                                   const double dxi[3], const int act[3], unsigned long long* rate_max,
                                   unsigned* err, cudaStream_t s) {
    if (nlist <= 0) return cudaSuccess;
    const unsigned grid = (unsigned)std::min<int64_t>((int64_t)16 * nlist, (int64_t)8 * (grid_y > 0 ? grid_y : nlist));
    launch_pdl(cfl_patch_kernel<R>, grid, 256, 0, s, static_cast<const R*>(U0), static_cast<const R*>(U1), patches, list,
                                             nlist, nlist_dev, slice, gamma, dxi[0], dxi[1], dxi[2], act[1], act[2],
                                             rate_max, err);
    return cudaGetLastError();
}

template <typename R>
static cudaError_t launch_cfl(const void* U, const PatchDev* patches, int npatch, double gamma, double courant,
                              const double dxi[3], const int act[3], void* partial, int grid, unsigned* counter,
                              double* dt_out, unsigned* err, cudaStream_t s) {
    CflArgs<R> a;
    a.U = static_cast<const R*>(U);
    a.patches = patches;
    a.npatch = npatch;
    a.gamma = gamma;
    a.courant = courant;
    for (int d = 0; d < 3; ++d) {
        a.dxi[d] = dxi[d];
        a.act[d] = act[d];
    }
    a.partial = static_cast<R*>(partial);
    a.counter = counter;
    a.dt_out = dt_out;
    a.err = err;
    cfl_kernel<R><<<grid, 256, 0, s>>>(a);
    return cudaGetLastError();
}

template <typename R>
static cudaError_t launch_adjoint(const AdjHostArgs& h, const FillGeom& fg, unsigned* err, cudaStream_t s,
                                  int* nlaunch) {
    AdjArgs<R> a;
    a.U = static_cast<const R*>(h.U);
    a.lam_next = static_cast<const R*>(h.lam_next);
    a.lam = static_cast<R*>(h.lam);
    a.F = static_cast<R*>(h.F);
    a.G = static_cast<R*>(h.G);
    a.ncell = h.ncell;
    a.patches = h.patches;
    a.npatch = h.npatch;
    a.gamma = h.gamma;
    a.eps = h.eps;
    a.dt = h.dt;
    for (int d = 0; d < 3; ++d) a.dxi[d] = h.dxi[d];
    a.limiter = h.limiter;
    a.riemann = h.riemann;
    // x-blocks per patch: 64, or (FP64, whose kernels are longer) enough for ~8 blocks per
    // SM on small bunches; never more than one thread per padded cell
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        sms = 0;
    const int bcap = (h.max_cells + 255) / 256;
    const int bwant = sizeof(R) == 8 ? std::max(64, (8 * sms + h.npatch - 1) / h.npatch) : 64;
    const int bx = std::max(1, std::min(bcap, bwant));
    const dim3 grid(bx, h.npatch < 65535 ? h.npatch : 65535), blk(256);
    const dim3 fgrid(bx, h.npatch < 65535 ? h.npatch : 65535);
    const unsigned pgrid = (unsigned)h.npatch * (unsigned)h.Zp;   // planes (regular grids)
    int n = 0;
    if (h.nboff)
        fill_grid_kernel<R><<<pgrid, 128, 0, s>>>(static_cast<R*>(h.U), h.patches, h.nboff, h.Zp);
    else
        fill_kernel<R><<<fgrid, 256, 0, s>>>(static_cast<R*>(h.U), h.patches, h.npatch, fg, err);
    ++n;
    adj_fwd_prim<R><<<grid, blk, 0, s>>>(a); ++n;
    adj_fwd_slopes<R><<<grid, blk, 0, s>>>(a); ++n;
    adj_fwd_en<R><<<grid, blk, 0, s>>>(a); ++n;
    adj_fwd_bh<R><<<grid, blk, 0, s>>>(a); ++n;
    adj_fwd_wh<R><<<grid, blk, 0, s>>>(a); ++n;
    adj_init<R><<<grid, blk, 0, s>>>(a); ++n;
    adj_faces<R><<<dim3(grid.x, grid.y, 3), blk, 0, s>>>(a); ++n;
    adj_edges<R><<<dim3(grid.x, grid.y, 3), blk, 0, s>>>(a); ++n;
    adj_pred<R><<<grid, blk, 0, s>>>(a); ++n;
    adj_bh<R><<<grid, blk, 0, s>>>(a); ++n;
    adj_en<R><<<grid, blk, 0, s>>>(a); ++n;
    adj_slopes<R><<<grid, blk, 0, s>>>(a); ++n;
    adj_prim<R><<<grid, blk, 0, s>>>(a); ++n;
    if (h.nboff)
        adj_fill_transpose_grid<R><<<pgrid, 128, 0, s>>>(static_cast<R*>(h.lam), h.patches, h.nboff, h.Zp);
    else
        adj_fill_transpose<R><<<fgrid, 256, 0, s>>>(static_cast<R*>(h.lam), h.patches, h.npatch, fg, err);
    ++n;
    if (nlaunch) *nlaunch = n;
    return cudaGetLastError();
}

}  // namespace mhd
