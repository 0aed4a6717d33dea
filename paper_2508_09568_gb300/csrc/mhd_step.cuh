// Fused bunch-update kernel: steps a3-a9 of one time step for tiles of patches.
//
// One CTA owns a tile of TX x TY columns of one patch and marches through its z-planes.
// Per plane it stages, in shared memory:
//   W ring   : primitive variables + face fields of the three planes c-1, c, c+1
//              over the tile plus a halo of 2 cells (+1 face on the high side);
//   prep     : predicted state W^{n+1/2}, limited slopes, predicted low-face fields and
//              their transverse slopes of planes c-1 and c, over the tile plus 1 halo;
//   fluxes   : HLLD fluxes of the x-, y-faces and the z-edge EMF of the plane, and the
//              z-faces / x-, y-edge EMFs between planes c-1 and c (double buffered);
// and writes the interior cells and owned faces of plane c-1 of U^{n+1}.  Every face
// flux and edge EMF of the tile is computed once; faces and edges on tile borders are
// recomputed by the neighbouring tile with the same code and inputs, so shared values
// agree bit for bit (exact conservation and div B across tiles and patches).
//
// Scheme: Sec. 2.1 (Eq. 6 flux, EOS), Sec. 2.1.2 (HLLD), Sec. 2.1.3 (Eqs. 7-12, Fig. 3),
// Sec. 2.1.4 (MUSCL-Hancock).  See mhd_math.cuh for the per-element arithmetic.
#pragma once

#include <type_traits>

#include "mhd_common.cuh"
#include "mhd_math.cuh"

namespace mhd {

// Items of a stage (an NI x NJ rectangle) in warp-sized chunks.  Three lane maps:
//   MAP_ROWS    one row of 32 per chunk, the columns from 32 on gathered in chunks of their own
//               (tiles 32 wide: no index division, almost no idle lanes, and a warp's reads of
//               a row are contiguous: no bank conflicts);
//   MAP_PITCH   rows of the pitch P of the arrays read, idle lanes at the row ends (other
//               single-precision tiles: contiguous reads);
//   MAP_PACKED  rows of NI (double precision: fewest idle lanes; its shared memory is idle).
enum { MAP_ROWS, MAP_PITCH, MAP_PACKED };

template <int NI, int NJ, int P, int MAP>
struct Items {
    static constexpr int XTRA = MAP == MAP_ROWS && NI > 32 ? NI - 32 : 0;
    static constexpr int N = MAP == MAP_ROWS ? NJ + (XTRA * NJ + 31) / 32
                                             : ((MAP == MAP_PITCH ? P : NI) * NJ + 31) / 32;   // chunks
    // one dimension: chunk q holds no item with i <= imax (a tile that reaches past its patch: of the
    // 64 columns of a tile a 16-cell patch needs one chunk in three, and each costs the FP64 pipe the
    // same; 1D step of 256 cells 50 -> 24 us).  In 2D and 3D the test costs more than the rows of
    // ragged tiles that it saves (512^3 +1 %, 21x28x17 patches no change).
    __device__ static __forceinline__ bool beyond(int q, int imax) { return NJ == 1 && q * 32 > imax; }
    // item (i, j) of lane `lane` of chunk q; false: idle lane
    __device__ static __forceinline__ bool at(int q, int lane, int& i, int& j) {
        if constexpr (MAP == MAP_ROWS) {
            if (XTRA == 0 || q < NJ) {
                i = lane;
                j = q;
                return NI >= 32 || lane < NI;
            }
            const int k = (q - NJ) * 32 + lane;
            i = 32 + k / NJ;
            j = k - (i - 32) * NJ;
            return i < NI;
        } else {
            constexpr int W = MAP == MAP_PITCH ? P : NI;
            const int k = q * 32 + lane;
            j = k / W;
            i = k - j * W;
            return i < NI && j < NJ;
        }
    }
};

// Which chunks each warp of the CTA runs in the two phases of a plane (see step_kernel): a list of
// chunk numbers, one per byte from the low end, closed by 255.
struct StepPlan {
    static constexpr int MAXW = 24;
    unsigned long long t[2][MAXW][2];
};

template <typename R, int NDIM_, int TX_, int TY_, int NT_, int MINB_>
struct StepCfg {
    static constexpr int NDIM = NDIM_, TX = TX_, TY = (NDIM_ >= 2 ? TY_ : 1), NT = NT_;
    static constexpr bool AY = NDIM >= 2, AZ = NDIM >= 3;
    // W ring: tile-local i in [-2, TX+2], j in [-2, TY+2] (y collapsed: j = 0)
    static constexpr int LOX = 2, LOY = AY ? 2 : 0;
    static constexpr int LX = TX + 5, LY = AY ? TY + 5 : 1;
    static constexpr int LSZ = LX * LY;
    static constexpr int NWV = 11;          // 8 primitives + 3 face fields
    static constexpr int NWSLOT = AZ ? 3 : 1;
    // prep: i in [-1, TX], j in [-1, TY]
    static constexpr int POX = 1, POY = AY ? 1 : 0;
    static constexpr int PX = TX + 2, PY = AY ? TY + 2 : 1;
    static constexpr int PSZ = PX * PY;
    static constexpr int NPV = 38;          // Wh(8) + dW(21) + bh(3) + face slopes(6)
    static constexpr int NPSLOT = AZ ? 2 : 1;
    // flux buffers
    static constexpr int FXN = (TX + 1) * TY;
    static constexpr int FYN = AY ? TX * (TY + 1) : 0;
    static constexpr int EZN = (TX + 1) * (AY ? TY + 1 : 1);
    static constexpr int FZN = AZ ? TX * TY : 0;
    static constexpr int EXN = AY ? TX * (TY + 1) : 0;
    static constexpr int EYN = (TX + 1) * TY;
    static constexpr int INB = 5 * FXN + 5 * FYN + EZN;     // in-plane buffer
    static constexpr int ZB = 5 * FZN + EXN + EYN;          // inter-plane buffer
    static constexpr int NINB = AZ ? 2 : 1, NZB = AZ ? 2 : 1;
    // raw plane staging (3D, single precision): 8 variables and the next plane's Bz; whole padded
    // rows of patches up to RAWX wide, as one block per variable rounded out to 16-byte bounds
    static constexpr int EQ = 16 / (int)sizeof(R);
    static constexpr bool STAGED = AZ && sizeof(R) == 4 && MINB_ != 2;   // (two 16x8 CTAs have no room)
    static constexpr int RAWX = MINB_ == 1 && LX < 37 ? 38 : LX + 1;
    static constexpr int RAWV = (LY * RAWX + 2 * EQ - 2) / EQ * EQ, RAWN = STAGED ? 9 * RAWV : 0;
    static_assert(!STAGED || 3 * RAWN <= NPSLOT * NPV * PSZ, "the first three planes are staged in the prep slots");
    // raw planes first: the bulk copies want 16-byte aligned rows
    static constexpr size_t PREP_OFF = (RAWN + 3) / 4 * 4;
    static constexpr size_t PREP_REALS = ((size_t)NPSLOT * NPV * PSZ + 3) / 4 * 4;
    static constexpr size_t SMEM_REALS = PREP_OFF + PREP_REALS + (size_t)NWSLOT * NWV * LSZ + (size_t)NINB * INB +
                                         (size_t)NZB * ZB;
    static constexpr size_t SMEM_BYTES = SMEM_REALS * sizeof(R) + 16;
    // chunks of the stages
    static constexpr int MAP = sizeof(R) == 8 ? MAP_PACKED : (TX == 32 ? MAP_ROWS : MAP_PITCH);
    using ICV = Items<LX, LY, LX, MAP>;
    using IPR = Items<PX, PY, LX, MAP>;
    using IFX = Items<TX + 1, TY, PX, MAP>;
    using IFY = Items<TX, AY ? TY + 1 : 0, PX, MAP>;
    using IEZ = Items<TX + 1, AY ? TY + 1 : 1, PX, MAP>;
    using IFZ = Items<TX, AZ ? TY : 0, PX, MAP>;
    using IEX = Items<TX, AY ? TY + 1 : 0, PX, MAP>;
    using IEY = Items<TX + 1, TY, PX, MAP>;
    using IUP = Items<TX, TY, TX + 1, MAP>;
    static constexpr int NI = IFX::N + IFY::N + IEZ::N, NZ = IFZ::N + IEX::N + IEY::N;
    static constexpr int NWARP = NT / 32;
    static constexpr int NQ = NWARP >= 12 ? 1 : 2;   // words of a warp's chunk list
};

// prep slot variable indices
#define PV_WH(k) (k)
// slope of primitive k along d (the slope of the normal field component along its own
// axis is never used and not stored)
#define PV_DW(d, k) (8 + 7 * (d) + ((k) < 5 + (d) ? (k) : (k) - 1))
#define PV_BH(c) (29 + (c))
#define PV_FS(c, k) (32 + 2 * (c) + (k))   // slope of face field c along (c+k+1)%3

template <typename R, typename C>
struct StepSmem {
    R* raw;   // [9][LY][RAWP] one plane as it came (STAGED)
    R* w;     // [NWSLOT][NWV][LSZ]
    R* prep;  // [NPSLOT][NPV][PSZ]
    R* inb;   // [NINB][INB]
    R* zb;    // [NZB][ZB]
    __device__ __forceinline__ R* W(int slot) const { return w + (size_t)slot * C::NWV * C::LSZ; }
    __device__ __forceinline__ R* P(int slot) const { return prep + (size_t)slot * C::NPV * C::PSZ; }
    __device__ __forceinline__ R* I(int slot) const { return inb + (size_t)slot * C::INB; }
    __device__ __forceinline__ R* Z(int slot) const { return zb + (size_t)slot * C::ZB; }
};

template <typename C>
__device__ __forceinline__ int lidx(int i, int j) {   // W ring cell index
    return (j + C::LOY) * C::LX + (i + C::LOX);
}
template <typename C>
__device__ __forceinline__ int pidx(int i, int j) {   // prep cell index
    return (j + C::POY) * C::PX + (i + C::POX);
}

// ---------------------------------------------------------------------------------------
// stages 1 and 2: plane m of U^n into the W ring, conserved -> primitive (a3), and its face
// fields.  Staged (single precision, 3D): the plane's rows come into shared memory one phase
// ahead (stage_plane), so that the DRAM latency is not seen; else straight from global memory.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ unsigned smem_addr(const void* p) { return static_cast<unsigned>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned arrivals) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(arrivals) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
// wait for the phase of the given parity; false: it did not complete within a second
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity) {
    const unsigned b = smem_addr(bar);
    uint64_t t0 = 0;
    for (;;) {
        unsigned done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(b), "r"(parity), "r"(20000u)
            : "memory");
        if (done) return true;
        uint64_t t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t0 == 0) t0 = t;
        else if (t - t0 > 1000000000ull) return false;
    }
}

// How a tile's planes are staged.  bulk: one bulk copy per variable and plane, the padded rows of
// the tile's halo whole (a warp spends a few instructions per plane, element copies some forty per
// cell), for patches whose rows fit RAWX; the copied block starts at the 16-byte bound at or below
// its first element, (s + v * vm + z * zm) mod EQ elements before it.  Otherwise element copies of
// the tile's own columns (pitch LX, no offset).  Row 0, column 0 of the tile's halo is element
// r0 + z * X * Y of each variable of the patch.
struct Stage {
    bool bulk;
    int P, rows, r0, s, vm, zm;
};

template <typename R, typename C>
__device__ __forceinline__ Stage stage_of(const PatchDev& pt, int x0, int y0) {
    Stage g;
    const int ys = y0 - C::LOY + pt.gy;
    g.rows = min(C::LY, pt.Y - ys);
    g.bulk = pt.X <= C::RAWX;
    g.P = g.bulk ? pt.X : C::LX;
    g.r0 = ys * pt.X;
    // the offset of column 0 (the halo starts at x0 - 2 + gx) stays in the index of the block
    g.s = g.bulk ? (int)((pt.off + g.r0) & (C::EQ - 1)) : 0;
    g.vm = g.bulk ? (int)(((int64_t)pt.X * pt.Y * pt.Z) & (C::EQ - 1)) : 0;
    g.zm = g.bulk ? (pt.X * pt.Y) & (C::EQ - 1) : 0;
    return g;
}

// Plane m (its 8 variables and the Bz of plane m+1) on its way into raw.  Bulk: copy v is issued by
// one lane of warp (w0 + v) mod NWARP and completes on bar (9 arrivals).  The blocks lie inside the
// patch's variable, rounded out to 16 bytes: inside the state, whose patches start and whose end
// lies at 16-byte bounds.  Planes m and m+1 are planes of the padded patch.
template <typename R, typename C>
__device__ __forceinline__ void stage_plane(const R* __restrict__ U, const PatchDev& pt, const Stage& g, int x0, int m,
                                            R* raw, uint64_t* bar, int w0) {
    const int64_t vol = (int64_t)pt.X * pt.Y * pt.Z;
    const int z = m + pt.gz, XY = pt.X * pt.Y;
    if (g.bulk) {
        const int wid = threadIdx.x >> 5;
        for (int v = (wid + C::NWARP - w0 % C::NWARP) % C::NWARP; v < 9; v += C::NWARP) {
            if ((threadIdx.x & 31) == 0) {
                // what the CTA's threads did here before the barrier comes before the copy
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                const int64_t e0 = pt.off + (v == 8 ? 7 * vol + XY : v * vol) + (int64_t)z * XY + g.r0;
                const int64_t e = e0 & ~(int64_t)(C::EQ - 1);
                const unsigned bytes = (unsigned)(((int)(e0 - e) + g.rows * pt.X + C::EQ - 1) / C::EQ * 16);
                mbar_expect(bar, bytes);
                asm volatile(
                    "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                        smem_addr(raw + v * C::RAWV)),
                    "l"(U + e), "r"(bytes), "r"(smem_addr(bar))
                    : "memory");
            }
        }
    } else {
        const R* base = U + pt.off + (int64_t)z * XY + g.r0 + (x0 - C::LOX + pt.gx);
        const int n = min(C::LX, pt.X - (x0 - C::LOX + pt.gx));
        for (int w = threadIdx.x; w < C::LSZ; w += C::NT) {
            const int lj = w / C::LX, li = w - lj * C::LX;
            if (lj >= g.rows || li >= n) continue;
            const R* u = base + (int64_t)lj * pt.X + li;
#pragma unroll
            for (int v = 0; v < 9; ++v) {
                const R* src = v == 8 ? u + 7 * vol + XY : u + v * vol;
                asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(smem_addr(raw + v * C::RAWV + w)),
                             "l"(src), "n"((int)sizeof(R))
                             : "memory");
            }
        }
    }
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// The tile a CTA works on.
template <typename R>
struct Tile {
    PatchDev pt;
    int x0, y0, wx, wy;   // low corner in the patch, columns inside the patch
    int z0, z1;           // planes updated (the z-block)
    const R* Uc;          // state read
    R* Un;                // state written
    R hdt, dtdx[3];
    Stage g;
};

// One chunk q of plane m into ring slot Wslot, from the staged rows (raw) or from U.
template <typename R, typename C>
__device__ __forceinline__ void convert_chunk(const Tile<R>& T, const R* raw, int m, R* Wslot, int q, R gm1) {
    int li, lj;
    if (C::ICV::beyond(q, T.wx + 2 + C::LOX) || !C::ICV::at(q, threadIdx.x & 31, li, lj)) return;
    const PatchDev& pt = T.pt;
    const int x0 = T.x0, y0 = T.y0;
    const int w = lj * C::LX + li;
    const int x = x0 + li - C::LOX + pt.gx, y = C::AY ? y0 + lj - C::LOY + pt.gy : 0, z = m + pt.gz;
    R p[8], bf[3];
    if (x >= 0 && x < pt.X && y >= 0 && y < pt.Y && z >= 0 && z < pt.Z) {
        const int64_t vol = (int64_t)pt.X * pt.Y * pt.Z;
        // high faces: 0 past the end of the padded patch and of the tile's halo (cells that feed
        // no owned output)
        const bool hx = li + 1 < C::LX && x + 1 < pt.X, hy = lj + 1 < C::LY && y + 1 < pt.Y, hz = z + 1 < pt.Z;
        R v[8], bx1, by1, bz1;
        if constexpr (C::STAGED) {
            constexpr int M = C::EQ - 1;
            const Stage& g = T.g;
            const int sz = g.s + z * g.zm;
            const R* r = raw + lj * g.P + li + (g.bulk ? x0 - C::LOX + pt.gx : 0);
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = r[k * C::RAWV + ((sz + k * g.vm) & M)];
            bx1 = hx ? r[5 * C::RAWV + ((sz + 5 * g.vm) & M) + 1] : R(0);
            by1 = hy ? r[6 * C::RAWV + ((sz + 6 * g.vm) & M) + g.P] : R(0);
            bz1 = hz ? r[8 * C::RAWV + ((sz + 7 * g.vm + g.zm) & M)] : R(0);
        } else {
            const R* u = T.Uc + pt.off + ((int64_t)z * pt.Y + y) * pt.X + x;
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = u[k * vol];
            bx1 = hx ? u[5 * vol + 1] : R(0);
            by1 = C::AY ? (hy ? u[6 * vol + pt.X] : R(0)) : v[6];
            bz1 = C::AZ ? (hz ? u[7 * vol + (int64_t)pt.X * pt.Y] : R(0)) : v[7];
        }
        cons_to_prim(v[0], v[1], v[2], v[3], v[4], R(0.5) * (v[5] + bx1), R(0.5) * (v[6] + by1), R(0.5) * (v[7] + bz1),
                     gm1, p);
#pragma unroll
        for (int c = 0; c < 3; ++c) bf[c] = v[5 + c];
    } else {
        // outside the padded patch: a benign state, never used by owned outputs
#pragma unroll
        for (int k = 0; k < 8; ++k) p[k] = R(0);
        p[Q_RHO] = R(1);
        p[Q_P] = gm1;
#pragma unroll
        for (int c = 0; c < 3; ++c) bf[c] = R(0);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) Wslot[k * C::LSZ + w] = p[k];
#pragma unroll
    for (int c = 0; c < 3; ++c) Wslot[(8 + c) * C::LSZ + w] = bf[c];
}

// ---------------------------------------------------------------------------------------
// stage 3: prep (a4 slopes, time-n edge EMF, predicted faces, a5 Hancock predictor)
// ---------------------------------------------------------------------------------------
template <typename R, typename C>
struct PrepCtx {
    const R* Wm;   // plane c-1
    const R* W0;   // plane c
    const R* Wp;   // plane c+1
    R hdt, gamma, dxi[3];
};

// value of W-ring variable k at (i+di, j+dj) on plane c+dk (dk in -1..1)
template <typename R, typename C>
__device__ __forceinline__ R wv(const PrepCtx<R, C>& X, int k, int i, int j, int dk) {
    const R* s = (!C::AZ || dk == 0) ? X.W0 : (dk < 0 ? X.Wm : X.Wp);
    return s[k * C::LSZ + lidx<C>(i, C::AY ? j : 0)];
}

// time-n edge EMF (Eqs. 7-11) times 8: E_e = <v_a><B_b> - <v_b><B_a> on the edge low in (a, b) of
// cell (i, j, dk).  <v> averages the four cells around the edge, <B_a> the two a-faces,
// <B_b> the two b-faces.  Collapsed axes map the -1 neighbour onto the cell itself.
template <typename R, typename C>
__device__ __forceinline__ R emf_n(const PrepCtx<R, C>& X, int e, int i, int j, int dk) {
    const int a = (e + 1) % 3, b = (e + 2) % 3;
    // offsets of the "-1" neighbour along a and b in (i, j, k)
    auto off = [&](int d, int& oi, int& oj, int& ok) {
        oi = (d == 0) ? -1 : 0;
        oj = (d == 1 && C::AY) ? -1 : 0;
        ok = (d == 2 && C::AZ) ? -1 : 0;
    };
    int ai, aj, ak, bi, bj, bk;
    off(a, ai, aj, ak);
    off(b, bi, bj, bk);
    const int qa = Q_U + a, qb = Q_U + b;
    // (pairwise sums: two dependent additions instead of three; sums instead of means: the
    // caller's factor h / dx carries their 1/4 * 1/2, a power of two, so nothing rounds)
    const R va = (wv(X, qa, i, j, dk) + wv(X, qa, i + ai, j + aj, dk + ak)) +
                 (wv(X, qa, i + bi, j + bj, dk + bk) + wv(X, qa, i + ai + bi, j + aj + bj, dk + ak + bk));
    const R vb = (wv(X, qb, i, j, dk) + wv(X, qb, i + ai, j + aj, dk + ak)) +
                 (wv(X, qb, i + bi, j + bj, dk + bk) + wv(X, qb, i + ai + bi, j + aj + bj, dk + ak + bk));
    const R Ba = wv(X, 8 + a, i, j, dk) + wv(X, 8 + a, i + bi, j + bj, dk + bk);
    const R Bb = wv(X, 8 + b, i, j, dk) + wv(X, 8 + b, i + ai, j + aj, dk + ak);
    return va * Bb - vb * Ba;
}

template <typename R, typename C, int LIM>
__device__ __forceinline__ void prep_cell(const PrepCtx<R, C>& X, int i, int j, R* Pslot, int pid) {
    const int li = lidx<C>(i, C::AY ? j : 0);
    R q[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) q[k] = X.W0[k * C::LSZ + li];
    // a4: limited slopes of the primitives along each active axis
    R dW[3][8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        dW[0][k] = limited(q[k] - wv(X, k, i - 1, j, 0), wv(X, k, i + 1, j, 0) - q[k], LIM);
        dW[1][k] = C::AY ? limited(q[k] - wv(X, k, i, j - 1, 0), wv(X, k, i, j + 1, 0) - q[k], LIM) : R(0);
        dW[2][k] = C::AZ ? limited(q[k] - wv(X, k, i, j, -1), wv(X, k, i, j, 1) - q[k], LIM) : R(0);
    }
    // transverse slopes of the low face fields of this cell
    const R bx = wv(X, 8, i, j, 0), by = wv(X, 9, i, j, 0), bz = wv(X, 10, i, j, 0);
    const R fs_bx_y = C::AY ? limited(bx - wv(X, 8, i, j - 1, 0), wv(X, 8, i, j + 1, 0) - bx, LIM) : R(0);
    const R fs_bx_z = C::AZ ? limited(bx - wv(X, 8, i, j, -1), wv(X, 8, i, j, 1) - bx, LIM) : R(0);
    const R fs_by_z = C::AZ ? limited(by - wv(X, 9, i, j, -1), wv(X, 9, i, j, 1) - by, LIM) : R(0);
    const R fs_by_x = limited(by - wv(X, 9, i - 1, j, 0), wv(X, 9, i + 1, j, 0) - by, LIM);
    const R fs_bz_x = limited(bz - wv(X, 10, i - 1, j, 0), wv(X, 10, i + 1, j, 0) - bz, LIM);
    const R fs_bz_y = C::AY ? limited(bz - wv(X, 10, i, j - 1, 0), wv(X, 10, i, j + 1, 0) - bz, LIM) : R(0);

    // time-n edge EMFs around the cell (Eqs. 7-11); edge index = low corner cell
    const int jy = C::AY ? 1 : 0;
    const int kz = C::AZ ? 1 : 0;
    // Ez at (i-1/2 + di, j-1/2 + dj) for di, dj in {0, 1}
    const R ez00 = emf_n(X, 2, i, j, 0), ez10 = emf_n(X, 2, i + 1, j, 0);
    const R ez01 = emf_n(X, 2, i, j + jy, 0), ez11 = emf_n(X, 2, i + 1, j + jy, 0);
    // Ex at (i, j-1/2 + dj, k-1/2 + dk)
    const R ex00 = emf_n(X, 0, i, j, 0), ex10 = emf_n(X, 0, i, j + jy, 0);
    const R ex01 = emf_n(X, 0, i, j, kz), ex11 = emf_n(X, 0, i, j + jy, kz);
    // Ey at (i-1/2 + di, j, k-1/2 + dk)
    const R ey00 = emf_n(X, 1, i, j, 0), ey10 = emf_n(X, 1, i + 1, j, 0);
    const R ey01 = emf_n(X, 1, i, j, kz), ey11 = emf_n(X, 1, i + 1, j, kz);

    // face fields predicted to t + dt/2 by Eq. 12 over dt/2 (with EMF = u x B):
    // dBx/dt = d_y Ez - d_z Ey, dBy/dt = d_z Ex - d_x Ez, dBz/dt = d_x Ey - d_y Ex
    const R h = R(0.125) * X.hdt;   // emf_n returns 8 E
    R tx0 = R(0), tx1 = R(0), ty0 = R(0), ty1 = R(0), tz0 = R(0), tz1 = R(0);
    if (C::AY) {
        tx0 += h * X.dxi[1] * (ez01 - ez00);
        tx1 += h * X.dxi[1] * (ez11 - ez10);
        tz0 -= h * X.dxi[1] * (ex10 - ex00);
        tz1 -= h * X.dxi[1] * (ex11 - ex01);
    }
    if (C::AZ) {
        tx0 -= h * X.dxi[2] * (ey01 - ey00);
        tx1 -= h * X.dxi[2] * (ey11 - ey10);
        ty0 += h * X.dxi[2] * (ex01 - ex00);
        ty1 += h * X.dxi[2] * (ex11 - ex10);
    }
    ty0 -= h * X.dxi[0] * (ez10 - ez00);
    ty1 -= h * X.dxi[0] * (ez11 - ez01);
    tz0 += h * X.dxi[0] * (ey10 - ey00);
    tz1 += h * X.dxi[0] * (ey11 - ey01);
    const R bxh0 = bx + tx0, bxh1 = wv(X, 8, i + 1, j, 0) + tx1;
    const R byh0 = by + ty0, byh1 = (C::AY ? wv(X, 9, i, j + 1, 0) : by) + ty1;
    const R bzh0 = bz + tz0, bzh1 = (C::AZ ? wv(X, 10, i, j, 1) : bz) + tz1;

    // a5: Hancock predictor
    R hq[5];
    hancock_dw<C::NDIM>(q, dW, X.dxi, X.hdt, X.gamma, hq);

#pragma unroll
    for (int k = 0; k < 5; ++k) Pslot[PV_WH(k) * C::PSZ + pid] = hq[k];
    Pslot[PV_WH(5) * C::PSZ + pid] = R(0.5) * (bxh0 + bxh1);
    Pslot[PV_WH(6) * C::PSZ + pid] = R(0.5) * (byh0 + byh1);
    Pslot[PV_WH(7) * C::PSZ + pid] = R(0.5) * (bzh0 + bzh1);
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (k != 5 + d) Pslot[PV_DW(d, k) * C::PSZ + pid] = dW[d][k];
    Pslot[PV_BH(0) * C::PSZ + pid] = bxh0;
    Pslot[PV_BH(1) * C::PSZ + pid] = byh0;
    Pslot[PV_BH(2) * C::PSZ + pid] = bzh0;
    Pslot[PV_FS(0, 0) * C::PSZ + pid] = fs_bx_y;
    Pslot[PV_FS(0, 1) * C::PSZ + pid] = fs_bx_z;
    Pslot[PV_FS(1, 0) * C::PSZ + pid] = fs_by_z;
    Pslot[PV_FS(1, 1) * C::PSZ + pid] = fs_by_x;
    Pslot[PV_FS(2, 0) * C::PSZ + pid] = fs_bz_x;
    Pslot[PV_FS(2, 1) * C::PSZ + pid] = fs_bz_y;
}

// ---------------------------------------------------------------------------------------
// stage 4: fluxes (a6 face states + a7 HLLD) and edge EMFs (a8)
// ---------------------------------------------------------------------------------------
template <typename R, typename C>
__device__ __forceinline__ R pv(const R* P, int v, int pid) { return P[v * C::PSZ + pid]; }

// flux through the low d-face of cell (pidR) with left cell (pidL) (possibly in another
// slot for d = z).  F receives (rho, mx, my, mz, E) fluxes.
template <typename R, typename C>
__device__ __forceinline__ void face_flux(const R* PL, int pidL, const R* PR, int pidR, int d, R gamma,
                                          R gm1i, R eps, int riemann, R F[5]) {
    const int t1 = (d + 1) % 3, t2 = (d + 2) % 3;
    R L[7], Rr[7];
    const int ks[7] = {Q_RHO, Q_U + d, Q_U + t1, Q_U + t2, Q_P, Q_BX + t1, Q_BX + t2};
#pragma unroll
    for (int n = 0; n < 7; ++n) {
        const int k = ks[n];
        L[n] = pv<R, C>(PL, PV_WH(k), pidL) + R(0.5) * pv<R, C>(PL, PV_DW(d, k), pidL);
        Rr[n] = pv<R, C>(PR, PV_WH(k), pidR) - R(0.5) * pv<R, C>(PR, PV_DW(d, k), pidR);
    }
    const R bn = pv<R, C>(PR, PV_BH(d), pidR);
    R f[5];
    if (riemann == 1) hll(L, Rr, bn, gamma, gm1i, f);
    else hlld(L, Rr, bn, gamma, gm1i, eps, f);
    F[0] = f[0];
    F[4] = f[4];
    F[1 + d] = f[1];
    F[1 + t1] = f[2];
    F[1 + t2] = f[3];
}

// corner state (sa, sb) of a cell for edge direction e with (a, b) = ((e+1)%3, (e+2)%3).
// Ba: the a-face on side sa (value and its slope along b), Bb: the b-face on side sb.
template <typename R, typename C>
__device__ __forceinline__ Corner<R> corner(const R* P, int pid, int e, R sa, R sb, R ba_face,
                                            R ba_slope, R bb_face, R bb_slope) {
    const int a = (e + 1) % 3, b = (e + 2) % 3;
    auto ext = [&](int k) {
        return pv<R, C>(P, PV_WH(k), pid) +
               R(0.5) * (sa * pv<R, C>(P, PV_DW(a, k), pid) + sb * pv<R, C>(P, PV_DW(b, k), pid));
    };
    Corner<R> s;
    s.rho = ext(Q_RHO);
    s.p = ext(Q_P);
    s.ua = ext(Q_U + a);
    s.ub = ext(Q_U + b);
    s.Be = ext(Q_BX + e);
    s.Ba = ba_face + R(0.5) * sb * ba_slope;
    s.Bb = bb_face + R(0.5) * sa * bb_slope;
    return s;
}

// The EMF on an edge along e whose transverse axis o is collapsed, between the cells pid0 and pid1 along
// the other, d (the face between them is the low face of pid1): each cell's state at that face.
template <typename R, typename C>
__device__ __forceinline__ R line_emf(const R* P, int pid0, int pid1, int e, int d, R gamma) {
    const int o = 3 - e - d, k = d == (o + 1) % 3 ? 0 : 1;   // PV_FS(o, k): slope along d of the o-face field
    const bool along_a = d == (e + 1) % 3;
    const R bd = pv<R, C>(P, PV_BH(d), pid1);
    auto state = [&](int pid, R s) {
        auto ext = [&](int v) { return pv<R, C>(P, PV_WH(v), pid) + R(0.5) * (s * pv<R, C>(P, PV_DW(d, v), pid)); };
        const R ud = ext(Q_U + d), uo = ext(Q_U + o);
        const R bo = pv<R, C>(P, PV_BH(o), pid) + R(0.5) * s * pv<R, C>(P, PV_FS(o, k), pid);
        Corner<R> c;
        c.rho = ext(Q_RHO);
        c.p = ext(Q_P);
        c.ua = along_a ? ud : uo;
        c.ub = along_a ? uo : ud;
        c.Be = ext(Q_BX + e);
        c.Ba = along_a ? bd : bo;
        c.Bb = along_a ? bo : bd;
        return c;
    };
    return emf_line(state(pid0, R(1)), state(pid1, R(-1)), along_a, gamma);
}

// ---------------------------------------------------------------------------------------
// the kernel
// ---------------------------------------------------------------------------------------
template <typename R>
struct StepArgs {
    const R* U;
    R* Unew;
    // asynchronous stepping (both null otherwise): patch p reads its current time slice
    // from buffer slice[p] (U when 0, Unew when 1) and writes the new one into the other
    // buffer, advancing by its own dt_patch[p]
    const int* slice;
    const double* dt_patch;
    const PatchDev* __restrict__ patches;
    const int4* tiles;
    int ntiles;
    int nzb;              // 3D: z-blocks of a tile, each a work item (ASYNC: chosen from the tile count)
    const int* ntiles_dev;  // ASYNC: tile count written by the device scheduler (null: ntiles)
    int dynamic;          // 1: pull tiles from *work (persistent), 0: one tile per CTA
    int* work;            // [0] next tile, [1] finished CTAs
    const double* dt_ptr; // device dt (if not null)
    double dt_val;
    // scheme constants in the kernel's precision, rounded on the host: instructions take them
    // from the parameter bank, no register holds them
    R gamma, gm1, gm1i, eps;
    double dxi[3];
    R dxir[3];
    int limiter;
    int riemann;          // face flux: 0 HLLD, 1 HLL
    unsigned* err;
};

// a9 for one chunk q of plane u of the tile: conservative update and constrained transport
// (Eq. 12) from the in-plane buffer of plane u and the inter-plane buffers of levels u-1/2,
// u+1/2.
template <typename R, typename C>
__device__ __forceinline__ void update_chunk(const StepSmem<R, C>& S, const Tile<R>& T, int u, unsigned* err, int q) {
    const PatchDev& pt = T.pt;
    const R dtdx0 = T.dtdx[0], dtdx1 = T.dtdx[1], dtdx2 = T.dtdx[2];
    const R* IB = S.I(C::AZ ? (u & 1) : 0);
    const R* Fx = IB;
    const R* Fy = IB + 5 * C::FXN;
    const R* Ez = Fy + 5 * C::FYN;
    const R* ZL = S.Z(C::AZ ? (u & 1) : 0);        // level u-1/2
    const R* ZH = S.Z(C::AZ ? ((u + 1) & 1) : 0);  // level u+1/2
    const R* FzL = ZL;
    const R* FzH = ZH;
    const R* ExL = ZL + 5 * C::FZN;
    const R* ExH = ZH + 5 * C::FZN;
    const R* EyL = ExL + C::EXN;
    const R* EyH = ExH + C::EXN;
    const int64_t vol = (int64_t)pt.X * pt.Y * pt.Z;
    int i, j;
    if (!C::IUP::at(q, threadIdx.x & 31, i, j) || i >= T.wx || j >= T.wy) return;
    const int x = T.x0 + i + pt.gx, y = C::AY ? T.y0 + j + pt.gy : 0, z = u + pt.gz;
    const int64_t o = pt.off + ((int64_t)z * pt.Y + y) * pt.X + x;
    const int fx = j * (C::TX + 1) + i;   // x-faces, Ez, Ey: pitch TX+1
    const int fy = j * C::TX + i;         // y-faces, z-faces, Ex: pitch TX
    R du[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        R d = dtdx0 * (Fx[v * C::FXN + fx + 1] - Fx[v * C::FXN + fx]);
        if (C::AY) d += dtdx1 * (Fy[v * C::FYN + fy + C::TX] - Fy[v * C::FYN + fy]);
        if (C::AZ) d += dtdx2 * (FzH[v * C::FZN + fy] - FzL[v * C::FZN + fy]);
        du[v] = -d;
    }
    R dbx = R(0), dby, dbz;
    if (C::AY) dbx += dtdx1 * (Ez[fx + (C::TX + 1)] - Ez[fx]);
    if (C::AZ) dbx -= dtdx2 * (EyH[fx] - EyL[fx]);
    dby = -dtdx0 * (Ez[fx + 1] - Ez[fx]);
    if (C::AZ) dby += dtdx2 * (ExH[fy] - ExL[fy]);
    dbz = dtdx0 * (EyL[fx + 1] - EyL[fx]);
    if (C::AY) dbz -= dtdx1 * (ExL[fy + C::TX] - ExL[fy]);
    const R* Ub = T.Uc + o;
    R* Un = T.Un + o;
    R nv[8];
#pragma unroll
    for (int v = 0; v < 5; ++v) nv[v] = Ub[v * vol] + du[v];
    nv[5] = Ub[5 * vol] + dbx;
    nv[6] = Ub[6 * vol] + dby;
    nv[7] = Ub[7 * vol] + dbz;
#pragma unroll
    for (int v = 0; v < 8; ++v) Un[v * vol] = nv[v];
    if (!(nv[0] > R(0)) || !finite_(nv[4])) atomicOr(err, ERR_PHYS);
}

// The EMF at (i-1/2, j-1/2) of plane c, chunk q of IEZ: i in [0, TX], j in [0, TY]
template <typename R, typename C>
__device__ __forceinline__ void flux_ez(const R* P0, R* IB, int q, int wx, R gamma) {
    R* Ez = IB + 5 * C::FXN + 5 * C::FYN;
    int i, j;
    if (!C::IEZ::beyond(q, wx) && C::IEZ::at(q, threadIdx.x & 31, i, j)) {
        if constexpr (!C::AY) {
            Ez[i] = line_emf<R, C>(P0, pidx<C>(i - 1, j), pidx<C>(i, j), 2, 0, gamma);
            return;
        }
        const int jm = j - 1;
        // cells: SW=(i-1,j-1) RT, SE=(i,j-1) LT, NW=(i-1,j) RB, NE=(i,j) LB
        const int pSW = pidx<C>(i - 1, jm), pSE = pidx<C>(i, jm);
        const int pNW = pidx<C>(i - 1, j), pNE = pidx<C>(i, j);
        // Ba = Bx face on side sa (+ slope along y): the x-face between cells i-1 and i is
        // the low face of cell i; Bb = By face on side sb (+ slope along x): the low y-face
        // of row j
        const R bxS = pv<R, C>(P0, PV_BH(0), pSE), bxN = pv<R, C>(P0, PV_BH(0), pNE);
        const R sxS = pv<R, C>(P0, PV_FS(0, 0), pSE), sxN = pv<R, C>(P0, PV_FS(0, 0), pNE);
        const R byW = pv<R, C>(P0, PV_BH(1), pNW), byE = pv<R, C>(P0, PV_BH(1), pNE);
        const R syW = pv<R, C>(P0, PV_FS(1, 1), pNW), syE = pv<R, C>(P0, PV_FS(1, 1), pNE);
        const Corner<R> SW = corner<R, C>(P0, pSW, 2, R(1), R(1), bxS, sxS, byW, syW);
        const Corner<R> SE = corner<R, C>(P0, pSE, 2, R(-1), R(1), bxS, sxS, byE, syE);
        const Corner<R> NW = corner<R, C>(P0, pNW, 2, R(1), R(-1), bxN, sxN, byW, syW);
        const Corner<R> NE = corner<R, C>(P0, pNE, 2, R(-1), R(-1), bxN, sxN, byE, syE);
        Ez[j * (C::TX + 1) + i] = emf2d(SW, SE, NW, NE, gamma);
    }
}

// The x- and y-faces of plane c (slot P0 into IB), one chunk q of IFX::N + IFY::N.
template <typename R, typename C>
__device__ __forceinline__ void flux_faces(const R* P0, R* IB, int q, int wx, R gamma, R gm1i, R eps, int riemann) {
    R* Fx = IB;
    R* Fy = IB + 5 * C::FXN;
    const int lane = threadIdx.x & 31;
    int i, j;
    if (q < C::IFX::N) {   // x-face i-1/2 of cell (i, j): i in [0, TX], j in [0, TY)
        if (!C::IFX::beyond(q, wx) && C::IFX::at(q, lane, i, j)) {
            R F[5];
            face_flux<R, C>(P0, pidx<C>(i - 1, j), P0, pidx<C>(i, j), 0, gamma, gm1i, eps, riemann, F);
            const int o = j * (C::TX + 1) + i;
#pragma unroll
            for (int v = 0; v < 5; ++v) Fx[v * C::FXN + o] = F[v];
        }
        return;
    }
    q -= C::IFX::N;
    if (q < C::IFY::N) {   // y-face j-1/2 of cell (i, j): i in [0, TX), j in [0, TY]
        if (C::AY && !C::IFY::beyond(q, wx) && C::IFY::at(q, lane, i, j)) {
            R F[5];
            face_flux<R, C>(P0, pidx<C>(i, j - 1), P0, pidx<C>(i, j), 1, gamma, gm1i, eps, riemann, F);
            const int o = j * C::TX + i;
#pragma unroll
            for (int v = 0; v < 5; ++v) Fy[v * C::FYN + o] = F[v];
        }
    }
}

// Fluxes between planes c-1 (slot Pm) and c (slot P0) into ZB, one chunk q of NZ.
template <typename R, typename C>
__device__ __forceinline__ void flux_interplane(const R* Pm, const R* P0, R* ZB, int q, int wx, R gamma,
                                                R gm1i, R eps, int riemann) {
    R* Fz = ZB;
    R* Ex = ZB + 5 * C::FZN;
    R* Ey = Ex + C::EXN;
    const int lane = threadIdx.x & 31;
    int i, j;
    if (q < C::IFZ::N) {   // z-face c-1/2 of cell (i, j): i in [0, TX), j in [0, TY)
        if (C::AZ && !C::IFZ::beyond(q, wx) && C::IFZ::at(q, lane, i, j)) {
            const int p = pidx<C>(i, j);
            R F[5];
            face_flux<R, C>(Pm, p, P0, p, 2, gamma, gm1i, eps, riemann, F);
            const int o = j * C::TX + i;
#pragma unroll
            for (int v = 0; v < 5; ++v) Fz[v * C::FZN + o] = F[v];
        }
        return;
    }
    q -= C::IFZ::N;
    if (q < C::IEX::N) {   // Ex at (i, j-1/2, c-1/2): a = y, b = z; i in [0, TX), j in [0, TY]
        if (C::AY && !C::IEX::beyond(q, wx) && C::IEX::at(q, lane, i, j)) {
            const int pS = pidx<C>(i, j - 1), pN = pidx<C>(i, j);
            if constexpr (!C::AZ) {
                Ex[j * C::TX + i] = line_emf<R, C>(P0, pS, pN, 0, 1, gamma);
                return;
            }
            // SW = (j-1, c-1) corner (+y,+z); SE = (j, c-1) (-y,+z);
            // NW = (j-1, c) (+y,-z); NE = (j, c) (-y,-z)
            // Ba = By face at side sy: the low y-face of row j (both planes)
            const R byB = pv<R, C>(Pm, PV_BH(1), pN), byT = pv<R, C>(P0, PV_BH(1), pN);
            const R syB = pv<R, C>(Pm, PV_FS(1, 0), pN), syT = pv<R, C>(P0, PV_FS(1, 0), pN);
            // Bb = Bz face at side sz: the face between c-1 and c = low face of plane c
            const R bzW = pv<R, C>(P0, PV_BH(2), pS), bzE = pv<R, C>(P0, PV_BH(2), pN);
            const R szW = pv<R, C>(P0, PV_FS(2, 1), pS), szE = pv<R, C>(P0, PV_FS(2, 1), pN);
            const Corner<R> SW = corner<R, C>(Pm, pS, 0, R(1), R(1), byB, syB, bzW, szW);
            const Corner<R> SE = corner<R, C>(Pm, pN, 0, R(-1), R(1), byB, syB, bzE, szE);
            const Corner<R> NW = corner<R, C>(P0, pS, 0, R(1), R(-1), byT, syT, bzW, szW);
            const Corner<R> NE = corner<R, C>(P0, pN, 0, R(-1), R(-1), byT, syT, bzE, szE);
            Ex[j * C::TX + i] = emf2d(SW, SE, NW, NE, gamma);
        }
        return;
    }
    q -= C::IEX::N;
    {   // Ey at (i-1/2, j, c-1/2): a = z, b = x; i in [0, TX], j in [0, TY)
        if (!C::IEY::beyond(q, wx) && C::IEY::at(q, lane, i, j)) {
            const int pW = pidx<C>(i - 1, j), pE = pidx<C>(i, j);
            if constexpr (!C::AZ) {
                Ey[j * (C::TX + 1) + i] = line_emf<R, C>(P0, pW, pE, 1, 0, gamma);
                return;
            }
            // SW = (x=i-1, c-1) corner (+z,+x); SE = (i-1, c) (-z,+x);
            // NW = (i, c-1) (+z,-x); NE = (i, c) (-z,-x)
            // Ba = Bz face at side sz: low face of plane c (shared); slope along x
            const R bzS = pv<R, C>(P0, PV_BH(2), pW), bzN = pv<R, C>(P0, PV_BH(2), pE);
            const R szS = pv<R, C>(P0, PV_FS(2, 0), pW), szN = pv<R, C>(P0, PV_FS(2, 0), pE);
            // Bb = Bx face at side sx: low face of cell i (shared); slope along z
            const R bxW = pv<R, C>(Pm, PV_BH(0), pE), bxE = pv<R, C>(P0, PV_BH(0), pE);
            const R sxW = pv<R, C>(Pm, PV_FS(0, 1), pE), sxE = pv<R, C>(P0, PV_FS(0, 1), pE);
            const Corner<R> SW = corner<R, C>(Pm, pW, 1, R(1), R(1), bzS, szS, bxW, sxW);
            const Corner<R> SE = corner<R, C>(P0, pW, 1, R(-1), R(1), bzS, szS, bxE, sxE);
            const Corner<R> NW = corner<R, C>(Pm, pE, 1, R(1), R(-1), bzN, szN, bxW, sxW);
            const Corner<R> NE = corner<R, C>(P0, pE, 1, R(-1), R(-1), bzN, szN, bxE, sxE);
            Ey[j * (C::TX + 1) + i] = emf2d(SW, SE, NW, NE, gamma);
        }
    }
}

// prep of one chunk q of a plane
template <typename R, typename C>
__device__ __forceinline__ void prep_chunk(const PrepCtx<R, C>& X, R* Ps, int q, int limiter, int wx) {
    int i, j;
    if (C::IPR::beyond(q, wx + C::POX) || !C::IPR::at(q, threadIdx.x & 31, i, j)) return;
    i -= C::POX;
    j -= C::POY;
    if (limiter == 0) prep_cell<R, C, 0>(X, i, j, Ps, pidx<C>(i, j));
    else prep_cell<R, C, 1>(X, i, j, Ps, pidx<C>(i, j));
}

// a warp's chunk list, held in registers
template <int NQ>
struct ChunkList {
    unsigned long long w[NQ];
    __device__ __forceinline__ ChunkList(const unsigned long long* t) {
#pragma unroll
        for (int k = 0; k < NQ; ++k) w[k] = t[k];
    }
    __device__ __forceinline__ int next() {
        const int q = (int)(w[0] & 255u);
#pragma unroll
        for (int k = 0; k < NQ; ++k) w[k] = (w[k] >> 8) | ((k + 1 < NQ ? w[k + 1] : ~0ull) << 56);
        return q;
    }
};

// The 3D step marches a tile through its planes in two phases per plane c, a barrier after each:
//   A: the fluxes between planes c-1 and c (prep slots c-1 and c), and plane c+2 into the ring
//      slot of plane c-1, which the prep of plane c was the last to read;
//   B: the prep of plane c+1 into the slot of plane c-1, which phase A was the last to read,
//      beside the fluxes inside plane c, which read slot c only, and the update of plane c-1,
//      whose last fluxes came in phase A.
// The EMFs inside plane c run in phase A of plane c+1 (slot c is still there): the two phases are even
// then, and the edge solvers' code is in A alone, that of the prep and of the x- and y-faces in B.
// Every warp has a fixed list of chunks in each phase.  The tile is copied to registers and the
// lists come from the parameter bank: with the lists decoded chunk by chunk from memory, or shared out
// through a counter, the step took 24.7 and 25.7 ms.
//
// What bounds it (FP32): the issue slots (70 % busy with 32x8 tiles on 32^3 patches, 64 % with 24x8 on
// 24^3; 16 warps, the registers allow no more).  Of 5.6 warps waiting per issued instruction 1.5 (24x8:
// 1.3) lost the slot to another, 1.0 (1.1) wait for a fixed latency, 0.6 (0.8) for instructions (the code
// of a phase's solvers and prep is more than the instruction cache holds) and 0.6 (1.2) at the ends of
// the phases; neither HBM (9 %) nor the FP32 pipes (34 %) bound it.  Measured on the 512^3 box, 32x8,
// step and fill: part of the EMFs inside the plane in either phase, a little more even but with their
// solver in both (instruction waits 1.4 with 24x8), 21.36 ms; as it is 20.64; one solver per phase behind the state loads of all directions 21.12 (24^3
// patches -1 %), one with offsets chosen at run time 23.5 (a third more instructions); one chunk list
// per warp and plane with two mbarrier points instead of the barriers, no waits at the ends (then 1.02 ->
// 0.04) but all code at once (instruction stalls 2.7), 30.4.  The form before this one, three phases
// (load + update + conversion / prep / fluxes) whose flux phase ended on a half-filled pass and whose
// prep left four of sixteen warps idle, took 21.0 ms for the step alone, this one 17.9.  FP64 is bound
// by the FP64 pipe (see mhd_math.cuh).
//
// ZB: work items are z-blocks of tiles (a launch of fewer tiles than SMs: the 64^3 box of 32^3
// patches, 32 tiles, took 172 us and takes 58); an instantiation of its own, whose block bounds cost
// the whole-column step 1.5 %.
//
// ASYNC: asynchronous stepping (a.slice, a.dt_patch): per-tile slice choice and dt; a
// separate instantiation so that the synchronous step keeps its kernel-wide constants.
template <typename R, int NDIM, int TX, int TY, int NT, int MINB, bool ZB, bool ASYNC>
__global__ void __launch_bounds__(NT, MINB) step_kernel(StepArgs<R> a, StepPlan plan) {
    using C = StepCfg<R, NDIM, TX, TY, NT, MINB>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    StepSmem<R, C> S;
    S.raw = reinterpret_cast<R*>(smem_raw);
    S.prep = S.raw + C::PREP_OFF;
    S.w = S.prep + C::PREP_REALS;
    S.inb = S.w + (size_t)C::NWSLOT * C::NWV * C::LSZ;
    S.zb = S.inb + (size_t)C::NINB * C::INB;
    __shared__ Tile<R> sT;
    __shared__ int s_tile, s_fail;
    __shared__ __align__(8) uint64_t s_bar[2];   // copies of a tile's first three planes; of the later ones

    const int wid = threadIdx.x >> 5;

    if (threadIdx.x == 0) {
        s_fail = 0;
        if constexpr (C::STAGED) {
            mbar_init(&s_bar[0], 27);
            mbar_init(&s_bar[1], 9);
            asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        }
    }
    if constexpr (ASYNC) pdl_begin();
    if (threadIdx.x == 0) s_tile = a.dynamic ? atomicAdd(&a.work[0], 1) : (int)blockIdx.x;
    __syncthreads();
    int t = s_tile;
    int ntiles = a.ntiles, nzb = ZB ? a.nzb : 1;
    if constexpr (ASYNC) {
        if (a.ntiles_dev) ntiles = min(*a.ntiles_dev, a.ntiles);
        // a round of few tiles: as many z-blocks as fill the grid (a.nzb: the most a patch takes)
        if constexpr (ZB) nzb = max(1, min(a.nzb, (int)gridDim.x / max(ntiles, 1)));
    }
    ntiles *= nzb;   // work items: z-block item % nzb of tile item / nzb
    // first plane of z-block k
    auto zblock = [&](int nz, int k) { return ZB ? nz * k / nzb : nz * k; };
    // the state that holds U^n of a patch
    auto source = [&](int p) -> const R* {
        if constexpr (ASYNC) return a.slice[p] ? a.Unew : a.U;
        else return a.U;
    };
    // the first planes of a tile on their way: -2, -1 and 0 into the prep slots, which no phase
    // reads between the last phase A of one tile and the first phase B of the next, 1 into raw
    auto begin = [&](int item) {
        if constexpr (C::STAGED) {
            if (item < ntiles) {
                const int4 tl = a.tiles[ZB ? item / nzb : item];
                const PatchDev pt = a.patches[tl.x];
                const R* U = source(tl.x);
                const Stage g = stage_of<R, C>(pt, tl.y, tl.z);
                const int z0 = zblock(pt.nz, ZB ? item % nzb : 0);
                for (int k = 0; k < 3; ++k)
                    stage_plane<R, C>(U, pt, g, tl.y, z0 + k - 2, S.prep + k * C::RAWN, &s_bar[0], 9 * k);
                stage_plane<R, C>(U, pt, g, tl.y, z0 + 1, S.raw, &s_bar[1], 27);
            }
        }
    };
    begin(t);
    unsigned par0 = 0, par1 = 0;   // phase parities of s_bar
    bool fail = false;
    while (t < ntiles && !fail) {
        // what the tile's chunks need of it, in shared memory (they would hold some forty
        // registers through every chunk)
        if (threadIdx.x == 0) {
            const int4 tl = a.tiles[ZB ? t / nzb : t];
            Tile<R>& T = sT;
            T.pt = a.patches[tl.x];
            T.x0 = tl.y;
            T.z0 = zblock(T.pt.nz, ZB ? t % nzb : 0);
            T.z1 = zblock(T.pt.nz, ZB ? t % nzb + 1 : 1);
            T.y0 = tl.z;
            T.wx = min(C::TX, T.pt.nx - tl.y);
            T.wy = C::AY ? min(C::TY, T.pt.ny - tl.z) : 1;
            T.Uc = source(tl.x);
            T.Un = T.Uc == a.U ? a.Unew : const_cast<R*>(a.U);
            if constexpr (C::STAGED) T.g = stage_of<R, C>(T.pt, tl.y, tl.z);
            double dt;
            if constexpr (ASYNC) dt = a.dt_patch[tl.x];
            else dt = a.dt_ptr ? *a.dt_ptr : a.dt_val;
            T.hdt = R(0.5 * dt);
            for (int d = 0; d < 3; ++d) T.dtdx[d] = R(dt * a.dxi[d]);
        }
        __syncthreads();
        const Tile<R> T = sT;

        if constexpr (C::AZ) {
            const int z0 = ZB ? T.z0 : 0, z1 = ZB ? T.z1 : T.pt.nz;
            const bool bulk = C::STAGED && T.g.bulk;
            int tnext = ntiles;
            if constexpr (C::STAGED) {
                if (bulk) {
                    if (!mbar_wait(&s_bar[0], par0)) s_fail = 1;
                    par0 ^= 1;
                } else {
                    cp_async_wait_all();
                    __syncthreads();
                }
            }
            for (int q = wid; q < 3 * C::ICV::N; q += C::NWARP) {
                const int k = q / C::ICV::N;   // plane z0 + k - 2
                convert_chunk<R, C>(T, S.prep + k * C::RAWN, z0 + k - 2, S.W((z0 + k + 1) % 3), q - k * C::ICV::N, a.gm1);
            }
            __syncthreads();
            auto phase = [&](int c, auto Bc) -> bool {
                constexpr bool B = decltype(Bc)::value;
                if (!B) {
                    if (a.dynamic && c == z1 && threadIdx.x == 0) s_tile = atomicAdd(&a.work[0], 1);
                } else if (c == z1) {
                    if (a.dynamic) tnext = s_tile;
                    begin(tnext);
                } else if constexpr (C::STAGED) {
                    if (c >= z0 - 1 && c + 3 <= z1 + 1) stage_plane<R, C>(T.Uc, T.pt, T.g, T.x0, c + 3, S.raw, &s_bar[1], 0);
                }
                const int ci = B ? c : c - 1;   // plane of the in-plane chunks
                ChunkList<C::NQ> list(plan.t[B][wid]);
                bool waited = false;
                for (int q; (q = list.next()) != 255;) {
                    if (q < C::NI) {
                        if (ci >= z0 && ci < z1) {
                            if constexpr (B) flux_faces<R, C>(S.P(ci & 1), S.I(ci & 1), q, T.wx, a.gamma, a.gm1i, a.eps, a.riemann);
                            else flux_ez<R, C>(S.P(ci & 1), S.I(ci & 1), q - C::IFX::N - C::IFY::N, T.wx, a.gamma);
                        }
                    } else if (q < C::NI + C::NZ) {
                        if (c >= z0)
                            flux_interplane<R, C>(S.P((c + 1) & 1), S.P(c & 1), S.Z(c & 1), q - C::NI, T.wx, a.gamma, a.gm1i,
                                                  a.eps, a.riemann);
                    } else if (q < C::NI + C::NZ + C::IPR::N) {
                        if (c < z1) {
                            PrepCtx<R, C> X;
                            X.Wm = S.W((c + 3) % 3);
                            X.W0 = S.W((c + 4) % 3);
                            X.Wp = S.W((c + 5) % 3);
                            X.hdt = T.hdt;
                            X.gamma = a.gamma;
                            for (int d = 0; d < 3; ++d) X.dxi[d] = a.dxir[d];
                            prep_chunk<R, C>(X, S.P((c + 1) & 1), q - C::NI - C::NZ, a.limiter, T.wx);
                        }
                    } else if (q < C::NI + C::NZ + C::IPR::N + C::ICV::N) {
                        if (c < z1) {
                            if constexpr (C::STAGED) {
                                if (bulk && !waited && !mbar_wait(&s_bar[1], par1)) s_fail = 1;
                                waited = true;
                            }
                            convert_chunk<R, C>(T, S.raw, c + 2, S.W((c + 5) % 3), q - C::NI - C::NZ - C::IPR::N, a.gm1);
                        }
                    } else if (c > z0) {
                        update_chunk<R, C>(S, T, c - 1, a.err, q - C::NI - C::NZ - C::IPR::N - C::ICV::N);
                    }
                }
                if (!B) {
                    par1 ^= c < z1 && bulk;
                } else if (c == z1) {
                    return true;
                } else if constexpr (C::STAGED) {
                    if (!bulk) cp_async_wait_all();
                }
                __syncthreads();
                if constexpr (C::STAGED) {
                    if (!B && s_fail) {
                        fail = true;
                        return true;
                    }
                }
                return false;
            };
            if (!phase(z0 - 2, std::true_type()))
#pragma unroll 1
                for (int c = z0 - 1; c <= z1; ++c) {
                    if (phase(c, std::false_type())) break;
                    if (phase(c, std::true_type())) break;
                }
            if (C::STAGED && !bulk) cp_async_wait_all();
            __syncthreads();   // (T is rewritten)
            t = tnext;
        } else {
            // one plane: convert, prep, fluxes, update (Ex and Ey with the collapsed z)
            for (int q = wid; q < C::ICV::N; q += C::NWARP) convert_chunk<R, C>(T, S.raw, 0, S.W(0), q, a.gm1);
            __syncthreads();
            PrepCtx<R, C> X;
            X.W0 = X.Wm = X.Wp = S.W(0);
            X.hdt = T.hdt;
            X.gamma = a.gamma;
            for (int d = 0; d < 3; ++d) X.dxi[d] = a.dxir[d];
            for (int q = wid; q < C::IPR::N; q += C::NWARP) prep_chunk<R, C>(X, S.P(0), q, a.limiter, T.wx);
            __syncthreads();
            for (int q = wid; q < C::NI + C::NZ; q += C::NWARP) {
                constexpr int NF = C::IFX::N + C::IFY::N;
                if (q < NF) flux_faces<R, C>(S.P(0), S.I(0), q, T.wx, a.gamma, a.gm1i, a.eps, a.riemann);
                else if (q < C::NI) flux_ez<R, C>(S.P(0), S.I(0), q - NF, T.wx, a.gamma);
                else flux_interplane<R, C>(S.P(0), S.P(0), S.Z(0), q - C::NI, T.wx, a.gamma, a.gm1i, a.eps, a.riemann);
            }
            if (a.dynamic && threadIdx.x == 0) s_tile = atomicAdd(&a.work[0], 1);
            __syncthreads();
            for (int q = wid; q < C::IUP::N; q += C::NWARP) update_chunk<R, C>(S, T, 0, a.err, q);
            t = a.dynamic ? s_tile : ntiles;
            __syncthreads();   // (T is rewritten)
        }
    }
    if constexpr (C::STAGED) {
        if (fail && threadIdx.x == 0) {
            // copies that did not land in time: wait once more (bounded) so that none is still
            // writing this CTA's shared memory when it exits, and report
            mbar_wait(&s_bar[0], par0 ^ 1);
            mbar_wait(&s_bar[1], par1 ^ 1);
            atomicOr(a.err, ERR_TIMEOUT);
        }
    }
    if (a.dynamic && threadIdx.x == 0) {
        // the last CTA to finish resets the work counters for the next launch
        __threadfence();
        if (atomicAdd(&a.work[1], 1) == (int)gridDim.x - 1) {
            a.work[0] = 0;
            a.work[1] = 0;
            __threadfence();
        }
    }
}

}  // namespace mhd
