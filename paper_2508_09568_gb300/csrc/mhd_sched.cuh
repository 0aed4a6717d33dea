// Device-side scheduler of asynchronous per-patch time stepping (mhd_bunch_advance_async).
//
// Every round of the asynchronous advance (DISPATCH's patches at their own times, Sec. 2.2,
// updated in bunches of ready patches, Sec. 2.4) is a sequence of stream-ordered launches
// with no host round trip:
//   async_ready_kernel     a flag per patch: short of t_span and no neighbour (an owner of
//                          a cell of its guard zone) at an earlier time;
//   async_list_kernel      the slices of the previous round's patches flipped; the flagged patches
//                          in ascending order and their tiles (one CTA, block-wide scans);
//   fill_interp_kernel     guard zones of the listed patches at their own times;
//   cfl_patch_kernel       each listed patch's maximum CFL rate;
//   async_clamp_kernel     dt = courant / rate, clipped to what is left of t_span, recorded;
//                          t_old <- t_cur, t_cur <- t_cur + dt (t_span for a patch that arrived);
//   step_kernel (ASYNC)    the update of the listed tiles, each patch by its own dt.
// The host enqueues rounds in batches and reads each batch's record afterwards.  The update reads
// slices and dt but no times, so the times advance before it and the readiness test of the next
// round finds them as a host scheduler would between rounds.
//
// A round of a few dozen patches is a chain of latencies, each launch some microseconds of which a
// few dependent loads are most: hence a warp per patch in the readiness test, no launch for the
// commit, and fill and CFL grids that fit the chip at once and share out what is listed (a grid of
// all planes of as many patches as twice the SMs took 7.6 us to find an empty list).  256^3 box of 512
// patches, 64 rounds: 10.8 -> 9.9 ms.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "mhd_common.cuh"

namespace mhd {

constexpr int kSchedThreads = 1024;   // async_list_kernel: one CTA of 32 warps

// Exclusive scan of v over the 1024 threads of the block; *total receives the sum.
// ws: 32 ints of shared memory, free again on return.
__device__ __forceinline__ int block_exscan(int v, int* ws, int* total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int s = ws[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        ws[lane] = s;
    }
    __syncthreads();
    const int prefix = (wid ? ws[wid - 1] : 0) + x - v;
    *total = ws[31];
    __syncthreads();
    return prefix;
}

// ready[p] = 1 when patch p is short of t_span and no neighbour is at an earlier time
// (nothing is ready once a round has failed: *abort != 0); one warp per patch, 256 threads
__global__ void __launch_bounds__(256) async_ready_kernel(int npatch, const int* __restrict__ nb_off,
                                                          const int* __restrict__ nb_idx, const double* t_cur,
                                                          double t_span, const unsigned* abort, int* ready) {
    pdl_begin();
    const int p = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (p >= npatch) return;
    const double tp = t_cur[p];
    bool ok = (*abort == 0u) && tp < t_span;
    const int k1 = nb_off[p + 1];
    for (int k = nb_off[p] + lane; k < k1; k += 32) ok &= t_cur[nb_idx[k]] >= tp;
    ok = __all_sync(0xffffffffu, ok);
    if (lane == 0) ready[p] = ok;
}

// slice flipped for the n patches of a list
__device__ __forceinline__ void flip_slices(const int* list, int n, int* slice) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) slice[list[i]] ^= 1;
}
__global__ void async_flip_kernel(const int* list, const int* n_ptr, int* slice) {
    pdl_begin();
    flip_slices(list, *n_ptr, slice);
}

// The ready patches in ascending order (list, *n_out), their tiles patch by patch in the
// natural tile order (tiles, *ntiles_out), and their rate maxima zeroed.  One CTA.  Before that the
// slices of the previous round's patches (prev, *n_prev; n_prev null: none) are flipped.
__global__ void __launch_bounds__(kSchedThreads) async_list_kernel(int npatch, const int* ready,
                                                                   const int* __restrict__ tfirst,
                                                                   const int* __restrict__ tcount,
                                                                   const int4* __restrict__ tnat, int* list,
                                                                   int* n_out, int4* tiles, int* ntiles_out,
                                                                   unsigned long long* rate_max, const int* prev,
                                                                   const int* n_prev, int* slice) {
    pdl_begin();
    if (n_prev) flip_slices(prev, *n_prev, slice);
    __syncthreads();   // (prev may be the row that is written next)
    __shared__ int ws[32];
    int count = 0, tcnt = 0;
    for (int base = 0; base < npatch; base += blockDim.x) {
        const int p = base + threadIdx.x;
        const int r = p < npatch ? ready[p] : 0;
        int tot = 0, ttot = 0;
        const int pos = block_exscan(r, ws, &tot);
        const int nt = r ? tcount[p] : 0;
        const int tpos = block_exscan(nt, ws, &ttot);
        if (r) {
            list[count + pos] = p;
            rate_max[p] = 0ull;
            const int f = tfirst[p];
            for (int j = 0; j < nt; ++j) tiles[tcnt + tpos + j] = tnat[f + j];
        }
        count += tot;
        tcnt += ttot;
    }
    if (threadIdx.x == 0) {
        *n_out = count;
        *ntiles_out = tcnt;
    }
}

// dt of each listed patch: courant / its maximum CFL rate (rate_max, the bits of a
// non-negative double from cfl_patch_kernel), clipped to what is left of t_span, written to dtp for
// the update and recorded in the round's row; the patch's times advance by it.  A
// non-positive or non-finite dt sets ERR_PHYS and the abort flag (later rounds schedule
// nothing) and is replaced by 0 so that the update leaves the patch unchanged.
__global__ void async_clamp_kernel(const int* list, const int* n_ptr,
                                   const unsigned long long* rate_max, double courant,
                                   double* t_old, double* t_cur, double t_span, double* dtp, double* dt_row,
                                   unsigned* abort, unsigned* err) {
    pdl_begin();
    const int n = *n_ptr;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int p = list[i];
        double d = courant / __longlong_as_double((long long)rate_max[p]);
        const double t = t_cur[p], rem = t_span - t;
        bool last = false;
        if (!(d > 0.0) || !isfinite(d)) {
            atomicOr(abort, 1u);
            atomicOr(err, ERR_PHYS);
            d = 0.0;
        } else if (d >= rem) {
            d = rem;
            last = true;
        }
        dtp[p] = d;
        dt_row[i] = d;
        t_old[p] = t;
        t_cur[p] = last ? t_span : t + d;
    }
}

// The final slice of every patch into the buffer `to`: a patch whose current slice is 1
// (held by `from`) is copied whole (8 variables of its padded block), as 4-byte words.
__global__ void async_gather_kernel(unsigned* to, const unsigned* from,
                                    const PatchDev* __restrict__ patches, int npatch, const int* slice,
                                    int real_words) {
    pdl_begin();
    for (int p = blockIdx.y; p < npatch; p += gridDim.y) {
        if (!slice[p]) continue;
        const PatchDev pt = patches[p];
        const int64_t w0 = pt.off * real_words;
        const int64_t nw = (int64_t)8 * pt.X * pt.Y * pt.Z * real_words;
        for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nw; k += (int64_t)gridDim.x * blockDim.x)
            to[w0 + k] = from[w0 + k];
    }
}

}  // namespace mhd
