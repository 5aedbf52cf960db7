// bottom_kernel.cu -- the bottom of the FAS V-cycle (the small grids and the coarsest solve) in
// one block.
//
// On the small grids (here at most 64 x 64 cells) every kernel of the V-cycle is latency-bound:
// a launch costs far more than its few thousand cells of work.  This kernel runs the whole
// sub-cycle from grid `lb` down to the coarsest and back in a single 1024-thread block, with
// every grid resident in shared memory.  It executes, cell by cell, exactly the arithmetic of
// the per-grid kernels (the snapshot, the per-phase smoother, the residual, the transfers and the
// coarsest solve share their device functions), so the V-cycle's results do not change.
// Used for the FP32 / mixed storage and the Spencer-Chen model when the grids fit in shared
// memory; the host falls back to the per-grid kernels otherwise.
#include <cooperative_groups.h>

#include "arith.cuh"
#include "coarse_body.cuh"
#include "reduce.cuh"
#include "tma.cuh"

#include <algorithm>

namespace segmg {

namespace {

constexpr int kBT = kCoarseThreads;   // threads of the block (the coarsest solve uses them all)
static_assert(kBT == kBottomThreads, "the host's default first grid assumes this block size");

// One grid in shared memory.  The row pitch P is odd where there is room for it (bottom_pitch): a
// column piece's 32 cells then lie in 32 different banks.
struct BGrid {
    int n, m, P, npm, npn;
    float cdiff, inv_tau, Sigma, inv_2h, beta;
    int pn, u, w, F, rhs, G, f, u0;   // places in smf (floats)
    int mrow, mcol;                   // ... of the masks [2][n][npm], [2][m][npn] (32-bit words)
    int has_rhs;
};

// The block's dynamic shared memory.  The grids' arrays are addressed by their place in it, not by
// pointers kept in a structure: the compiler then knows them to be shared memory.  Little of the
// SM's first-level cache is left beside the 200 KB that these kernels take, so anything a thread
// keeps in local memory (a spilled register, a structure on the stack, a function call's saved
// registers) is a round trip to L2: the code of each step of the sub-cycle therefore stands inline
// at one place.
extern __shared__ __align__(16) float smf[];
__device__ __forceinline__ uint32_t *smw() { return reinterpret_cast<uint32_t *>(smf); }

// Scratch of tile_smooth: the tile's jump classes, its column masks and which sweeps have members.
struct TileScratch {
    uint8_t star[32][36];
    uint32_t mcol[2][32];
    unsigned any;          // bit k: a member cell of sweep k in this tile
    unsigned anyr[16];     // cluster: every tile's `any`, pushed by its CTA
};

// Thread layout over an array with `cols` columns: TX = the power of two >= cols (at most the
// block size) threads along a row, kBT / TX rows at a time; no integer division per cell.
struct Map2 {
    int tx, ty, TX, TY;
};
__device__ __forceinline__ Map2 map_for(int cols) {
    int lg = cols <= 1 ? 0 : 32 - __clz(cols - 1);
    lg = min(lg, 10);
    Map2 r;
    r.TX = 1 << lg;
    r.TY = kBT >> lg;
    r.tx = threadIdx.x & (r.TX - 1);
    r.ty = threadIdx.x >> lg;
    return r;
}
#define FOR_CELLS(M, n, m, i, j)                                                              \
    for (int i = (M).ty; i < (n); i += (M).TY)                                                \
        for (int j = (M).tx; j < (m); j += (M).TX)

// G = w / |grad phi|_beta of every cell at phi = pn + uu (mirror-clamped neighbours), as the
// tile kernels form it.
__device__ __forceinline__ void b_G(const BGrid &B, int uu_) {
    const int n = B.n, m = B.m, P = B.P;
    const float *pn = smf + B.pn, *uu = smf + uu_, *W = smf + B.w;
    const Map2 M = map_for(m);
    FOR_CELLS(M, n, m, i, j) {
        const int q = i * P + j;
        const int s = (i + 1 < n ? i + 1 : n - 1) * P + j, nn = (i > 0 ? i - 1 : 0) * P + j;
        const int e = q + (j + 1 < m ? 1 : 0), w = q - (j > 0 ? 1 : 0);
        stc(smf + B.G, q, (size_t)n * P, kDbgBottom,
            cell_G(W[q], pn[s], pn[nn], pn[e], pn[w], uu[s], uu[nn], uu[e], uu[w], B.inv_2h, B.beta));
    }
    __syncthreads();
}

// Snapshot (as k_snapshot): G, f, jump class and the member masks of every piece.
__device__ __forceinline__ void b_snapshot(const BGrid &B, uint8_t *star) {
    const int n = B.n, m = B.m, P = B.P;
    b_G(B, B.u);
    const Map2 M = map_for(m);
    FOR_CELLS(M, n, m, i, j) {
        const int q = i * P + j;
        const bool hS = i + 1 < n, hN = i > 0, hE = j + 1 < m, hW = j > 0;
        const int oS = hS ? q + P : q, oN = hN ? q - P : q, oE = hE ? q + 1 : q, oW = hW ? q - 1 : q;
        const float gc = (smf + B.G)[q];
        const float aS = face(gc, (smf + B.G)[oS], hS), aN = face(gc, (smf + B.G)[oN], hN);
        const float aE = face(gc, (smf + B.G)[oE], hE), aW = face(gc, (smf + B.G)[oW], hW);
        const float pc = (smf + B.pn)[q];
        float ds = mul_rn(aS, sub_rn((smf + B.pn)[oS], pc));
        ds = fma_rn(aN, sub_rn((smf + B.pn)[oN], pc), ds);
        ds = fma_rn(aE, sub_rn((smf + B.pn)[oE], pc), ds);
        ds = fma_rn(aW, sub_rn((smf + B.pn)[oW], pc), ds);
        float base = add_rn((smf + B.F)[q], 0.0f);
        if (B.has_rhs) base = add_rn(base, (smf + B.rhs)[q]);
        stc(smf + B.f, q, (size_t)n * P, kDbgBottom, fma_rn(-B.cdiff, ds, base));
        const float big = 3.0e38f;
        const float vS = hS ? aS : big, vN = hN ? aN : big, vE = hE ? aE : big, vW = hW ? aW : big;
        const float mn = fminf(fminf(vS, vN), fminf(vE, vW));
        const float mx = fmaxf(fmaxf(hS ? aS : -1.f, hN ? aN : -1.f), fmaxf(hE ? aE : -1.f, hW ? aW : -1.f));
        const int am = vS == mn ? 0 : (vN == mn ? 1 : (vE == mn ? 2 : 3));
        const int cnt = (int)hS + (int)hN + (int)hE + (int)hW;
        stc(star, q, (size_t)n * P, kDbgBottom, (cnt >= 2 && mx > mul_rn(B.Sigma, mn)) ? (uint8_t)(1u << am) : (uint8_t)0);
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = warp; i < n; i += kBT / 32)                  // row pieces: sweeps A, B
        for (int pc = 0; pc < B.npm; ++pc) {
            const int j = pc * 32 + lane, len = min(32, m - pc * 32);
            const uint8_t s = lane < len ? star[i * P + j] : 0;
            const uint32_t mA = members_of(__ballot_sync(0xffffffffu, s & 1u), len);
            const uint32_t mB = members_of(__ballot_sync(0xffffffffu, s & 2u), len);
            if (lane == 0) {
                stc(smw() + B.mrow, (size_t)(0 * n + i) * B.npm + pc, (size_t)2 * n * B.npm, kDbgBottom, mA);
                stc(smw() + B.mrow, (size_t)(1 * n + i) * B.npm + pc, (size_t)2 * n * B.npm, kDbgBottom, mB);
            }
        }
    for (int j = warp; j < m; j += kBT / 32)                  // column pieces: sweeps C, D
        for (int pc = 0; pc < B.npn; ++pc) {
            const int i = pc * 32 + lane, len = min(32, n - pc * 32);
            const uint8_t s = lane < len ? star[i * P + j] : 0;
            const uint32_t mC = members_of(__ballot_sync(0xffffffffu, s & 4u), len);
            const uint32_t mD = members_of(__ballot_sync(0xffffffffu, s & 8u), len);
            if (lane == 0) {
                stc(smw() + B.mcol, (size_t)(0 * m + j) * B.npn + pc, (size_t)2 * m * B.npn, kDbgBottom, mC);
                stc(smw() + B.mcol, (size_t)(1 * m + j) * B.npn + pc, (size_t)2 * m * B.npn, kDbgBottom, mD);
            }
        }
    __syncthreads();
}

__device__ __forceinline__ bool b_member(const BGrid &B, int sweep, int i, int j) {
    if (sweep < 2) return ((smw() + B.mrow)[(sweep * B.n + i) * B.npm + (j >> 5)] >> (j & 31)) & 1u;
    return ((smw() + B.mcol)[((sweep - 2) * B.m + j) * B.npn + (i >> 5)] >> (i & 31)) & 1u;
}

// The two partial-line phases of one directional sweep (as k_seg): one warp per line of the
// phase's parity.  Lines of one parity do not interact, and the cells just outside a piece lie
// on the same line, so a warp reads the end values of all its pieces before it solves any run:
// no block-wide barrier is needed within a phase.
__device__ __forceinline__ void b_lines(const BGrid &B, int sweep, float *endv) {
    const int n = B.n, m = B.m, P = B.P;
    const bool rev = sweep & 1, rowwise = sweep < 2;
    const int nlines = rowwise ? n : m, llen = rowwise ? m : n, npieces = rowwise ? B.npm : B.npn;
    const int step = rowwise ? 1 : P;                 // stride along a line
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int ph = 0; ph < 2; ++ph) {
        const int parity = rev ? 1 - ph : ph;
        const int nl = (nlines - parity + 1) / 2;
        for (int li = warp; li < nl; li += kBT / 32) {
            const int line = parity + 2 * li;
            const int base = rowwise ? line * P : line;   // cell of position 0 on the line
            const uint32_t *mks = smw() + (rowwise ? B.mrow + (sweep * n + line) * B.npm
                                          : B.mcol + ((sweep - 2) * m + line) * B.npn);
            float *ev = endv + 2 * li * npieces;
            for (int pc = lane; pc < npieces; pc += 32) {
                const int t0 = pc * 32, len = min(32, llen - t0);
                ev[2 * pc] = t0 > 0 ? (smf + B.u)[base + (t0 - 1) * step] : 0.f;
                ev[2 * pc + 1] = t0 + len < llen ? (smf + B.u)[base + (t0 + len) * step] : 0.f;
            }
            __syncwarp();
            for (int pc = 0; pc < npieces; ++pc) {
                const uint32_t mk = mks[pc];
                if (!mk) continue;   // the whole warp
                const int t0 = pc * 32, len = min(32, llen - t0), tt = t0 + lane;
                const float own = lane < len ? (smf + B.u)[base + tt * step] : 0.f;
                auto at = [&](int r) -> RunCell<float> {
                    const int o = base + (t0 + r) * step;
                    const int i = rowwise ? line : t0 + r, j = rowwise ? t0 + r : line;
                    const bool hS = i + 1 < n, hN = i > 0, hE = j + 1 < m, hW = j > 0;
                    const int oS = hS ? o + P : o, oN = hN ? o - P : o, oE = hE ? o + 1 : o, oW = hW ? o - 1 : o;
                    const float gc = (smf + B.G)[o];
                    const float aS = face(gc, (smf + B.G)[oS], hS), aN = face(gc, (smf + B.G)[oN], hN);
                    const float aE = face(gc, (smf + B.G)[oE], hE), aW = face(gc, (smf + B.G)[oW], hW);
                    RunCell<float> c;
                    if (rowwise) { c.ap = aW; c.an = aE; c.ax1 = aS; c.ax2 = aN; c.ux1 = (smf + B.u)[oS]; c.ux2 = (smf + B.u)[oN]; }
                    else         { c.ap = aN; c.an = aS; c.ax1 = aE; c.ax2 = aW; c.ux1 = (smf + B.u)[oE]; c.ux2 = (smf + B.u)[oW]; }
                    c.f = (smf + B.f)[o];
                    return c;
                };
                float x;
                if (pcr_piece<float>(mk, len, B.cdiff, B.inv_tau, own, ev[2 * pc], ev[2 * pc + 1], at, x))
                    stc(smf + B.u, (size_t)(base + tt * step), (size_t)n * P, kDbgBottom, x);
            }
            __syncwarp();
        }
        __syncthreads();
    }
}

// One directional sweep of Hybrid Smoother 2 in the parallel ordering (as k_rb + k_seg).
__device__ __forceinline__ void b_sweep(const BGrid &B, int sweep, float *endv) {
    const int n = B.n, m = B.m, P = B.P;
    const bool rev = sweep & 1;
    // checkerboard phases: the cells of one colour, two per row pair of threads' columns
    const int mh = (m + 1) >> 1;
    const Map2 MH = map_for(mh);
    for (int ph = 0; ph < 2; ++ph) {
        const int colour = rev ? 1 - ph : ph;
        FOR_CELLS(MH, n, mh, i, k) {
            const int j = 2 * k + ((i + colour) & 1);
            if (j >= m || b_member(B, sweep, i, j)) continue;
            const int q = i * P + j;
            const bool hS = i + 1 < n, hN = i > 0, hE = j + 1 < m, hW = j > 0;
            const int oS = hS ? q + P : q, oN = hN ? q - P : q, oE = hE ? q + 1 : q, oW = hW ? q - 1 : q;
            const float gc = (smf + B.G)[q];
            const float aS = face(gc, (smf + B.G)[oS], hS), aN = face(gc, (smf + B.G)[oN], hN);
            const float aE = face(gc, (smf + B.G)[oE], hE), aW = face(gc, (smf + B.G)[oW], hW);
            stc(smf + B.u, q, (size_t)n * P, kDbgBottom,
                point_relax(B.cdiff, B.inv_tau, aS, aN, aE, aW, (smf + B.u)[oS], (smf + B.u)[oN], (smf + B.u)[oE], (smf + B.u)[oW], (smf + B.f)[q]));
        }
        __syncthreads();
    }
    b_lines(B, sweep, endv);
}

// One outer smoothing iteration (snapshot and four sweeps) of a grid with at most one cell per
// thread that is longer than 32 cells on a side (tile_smooth takes the others).  The cell's four face values, the denominator of its point update, f and its member
// bits are formed once after the snapshot and kept in registers, so a checkerboard phase reads
// only the four neighbouring values of u from shared memory.  The update is point_relax's
// sequence of operations, so the results equal those of b_snapshot and four b_sweep calls; a
// sweep with no member cell on the grid skips its (empty) line phases.
__device__ __forceinline__ void b_smooth_small(const BGrid &B, uint8_t *star, float *endv) {
    __shared__ unsigned s_any;   // bit k: sweep k has a member cell somewhere on the grid
    if (threadIdx.x == 0) s_any = 0;
    b_snapshot(B, star);         // ends with a barrier
    const int n = B.n, m = B.m, P = B.P;
    const bool own = threadIdx.x < n * m;
    const int ci = threadIdx.x / m, cj = threadIdx.x - ci * m, q = own ? ci * P + cj : 0;
    float aS = 0.f, aN = 0.f, aE = 0.f, aW = 0.f, dv = 1.f, fq = 0.f;
    int oS = q, oN = q, oE = q, oW = q, colour = 0;
    unsigned mem = 0;
    if (own) {
        const int i = ci, j = cj;
        const bool hS = i + 1 < n, hN = i > 0, hE = j + 1 < m, hW = j > 0;
        oS = hS ? q + P : q; oN = hN ? q - P : q; oE = hE ? q + 1 : q; oW = hW ? q - 1 : q;
        const float gc = (smf + B.G)[q];
        aS = face(gc, (smf + B.G)[oS], hS); aN = face(gc, (smf + B.G)[oN], hN);
        aE = face(gc, (smf + B.G)[oE], hE); aW = face(gc, (smf + B.G)[oW], hW);
        dv = fma_rn(B.cdiff, add_rn(add_rn(aS, aN), add_rn(aE, aW)), B.inv_tau);
        fq = (smf + B.f)[q];
        colour = (i + j) & 1;
        for (int k = 0; k < 4; ++k) mem |= (unsigned)b_member(B, k, i, j) << k;
    }
    const unsigned wm = __reduce_or_sync(0xffffffffu, mem);
    if ((threadIdx.x & 31) == 0 && wm) atomicOr(&s_any, wm);
    __syncthreads();
    const unsigned any = s_any;
    for (int k = 0; k < 4; ++k) {
        const bool rev = k & 1;
        for (int ph = 0; ph < 2; ++ph) {
            if (own && colour == (rev ? 1 - ph : ph) && !((mem >> k) & 1u)) {
                float num = mul_rn(aS, (smf + B.u)[oS]);
                num = fma_rn(aN, (smf + B.u)[oN], num);
                num = fma_rn(aE, (smf + B.u)[oE], num);
                num = fma_rn(aW, (smf + B.u)[oW], num);
                stc(smf + B.u, q, (size_t)n * P, kDbgBottom, div_relax(fma_rn(B.cdiff, num, -fq), dv));
            }
            __syncthreads();
        }
        if ((any >> k) & 1u) b_lines(B, k, endv);
    }
}

// out = rhs - L(pn + uu) (mode 0) or out += L(pn + uu) (mode 1), as k_residual.
__device__ __forceinline__ void b_residual(const BGrid &B, int uu_, int out_, int mode) {
    const int n = B.n, m = B.m, P = B.P;
    b_G(B, uu_);
    const float *uu = smf + uu_;
    float *out = smf + out_;
    const Map2 M = map_for(m);
    FOR_CELLS(M, n, m, i, j) {
        const int q = i * P + j;
        const bool hS = i + 1 < n, hN = i > 0, hE = j + 1 < m, hW = j > 0;
        const int oS = hS ? q + P : q, oN = hN ? q - P : q, oE = hE ? q + 1 : q, oW = hW ? q - 1 : q;
        const float gc = (smf + B.G)[q];
        const float aS = face(gc, (smf + B.G)[oS], hS), aN = face(gc, (smf + B.G)[oN], hN);
        const float aE = face(gc, (smf + B.G)[oE], hE), aW = face(gc, (smf + B.G)[oW], hW);
        const float pc = (smf + B.pn)[q], uc = uu[q];
        float fl = mul_rn(aS, add_rn(sub_rn((smf + B.pn)[oS], pc), sub_rn(uu[oS], uc)));
        fl = fma_rn(aN, add_rn(sub_rn((smf + B.pn)[oN], pc), sub_rn(uu[oN], uc)), fl);
        fl = fma_rn(aE, add_rn(sub_rn((smf + B.pn)[oE], pc), sub_rn(uu[oE], uc)), fl);
        fl = fma_rn(aW, add_rn(sub_rn((smf + B.pn)[oW], pc), sub_rn(uu[oW], uc)), fl);
        const float Lv = sub_rn(fma_rn(B.cdiff, fl, -add_rn((smf + B.F)[q], 0.0f)), mul_rn(B.inv_tau, uc));
        if (mode == 0) stc(out, q, (size_t)n * P, kDbgBottom, B.has_rhs ? sub_rn((smf + B.rhs)[q], Lv) : -Lv);
        else stc(out, q, (size_t)n * P, kDbgBottom, add_rn(out[q], Lv));
    }
    __syncthreads();
}

// Full weighting of r = fine.f and of fine.u onto the coarse grid C (rhs; u and u0), as k_restrict:
// three taps per axis, or two of weight 1/2 at the last coarse cell of an even axis.
__device__ __forceinline__ void b_restrict(const BGrid &F, const BGrid &C) {
    const Map2 M = map_for(C.m);
    FOR_CELLS(M, C.n, C.m, I, J) {
        const bool r3 = 2 * I + 2 < F.n, c3 = 2 * J + 2 < F.m;
        const float rw = r3 ? 0.25f : 0.5f, cw = c3 ? 0.25f : 0.5f;
        const int o = 2 * I * F.P + 2 * J;
        auto weigh = [&](const float *src) {
            float s = 0.f;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if (a == 2 && !r3) break;
                const size_t oa = (size_t)(o + a * F.P), lim = (size_t)F.n * F.P;
                float row = fma_rn(cw, ldc(src, oa, lim, kDbgBottom), 0.f);
                row = fma_rn(0.5f, ldc(src, oa + 1, lim, kDbgBottom), row);
                if (c3) row = fma_rn(cw, ldc(src, oa + 2, lim, kDbgBottom), row);
                s = fma_rn(a == 1 ? 0.5f : rw, row, s);
            }
            return s;
        };
        const float sr = weigh(smf + F.f), su = weigh(smf + F.u);
        const int q = I * C.P + J;
        const size_t lim = (size_t)C.n * C.P;
        stc(smf + C.rhs, q, lim, kDbgBottom, sr);
        stc(smf + C.u, q, lim, kDbgBottom, su);
        stc(smf + C.u0, q, lim, kDbgBottom, su);
    }
    __syncthreads();
}

// fine.u += P (coarse.u - coarse.u0), as k_interp_add.
__device__ __forceinline__ void b_interp_add(const BGrid &F, const BGrid &C) {
    const Map2 M = map_for(F.m);
    FOR_CELLS(M, F.n, F.m, i, j) {
        int ri[2], ci[2];
        float rw[2], cw[2];
        const int nr = bl_taps(i, C.n, ri, rw), nk = bl_taps(j, C.m, ci, cw);
        float s = 0.f;
        for (int a = 0; a < nr; ++a)
            for (int b = 0; b < nk; ++b) {
                const int o = ri[a] * C.P + ci[b];
                const size_t lc = (size_t)C.n * C.P;
                s = fma_rn(rw[a] * cw[b], sub_rn(ldc(smf + C.u, o, lc, kDbgBottom), ldc(smf + C.u0, o, lc, kDbgBottom)), s);
            }
        const int q = i * F.P + j;
        stc(smf + F.u, q, (size_t)F.n * F.P, kDbgBottom, add_rn((smf + F.u)[q], s));
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------------------
// Smoothing of one 32 x 32 tile by 1024 threads, one cell per thread (warp w: tile row w, lane l:
// tile column l): a whole grid of at most 32 x 32 cells, or one CTA's tile of a grid spread over a
// cluster (CL).
//
// Everything here is a chain of short dependent phases, so what is kept out of them decides the
// time.  After the snapshot a thread holds in registers the faces, diagonal and f of its own cell
// (w, l), which its warp needs for the checkerboard phases and for tile row w's partial lines: those
// phases then read only values of u.  For tile column w's partial lines it forms them again for the
// transposed cell (l, w) (kept as well, they do not fit the 64 registers a thread has, and a spilled
// register is a round trip to L2 here).  Row masks are warp votes and stay in registers, column masks
// go through shared memory once.  A grid's arrays have an odd pitch, so that a column's cells lie in different banks
// (with the pitch equal to a row of 32 or 64 cells a column read took 32 turns).
//
// CL: pn, u and G carry a ring of the neighbouring tiles' edge cells.  A thread that changes an
// edge cell stores the value into the neighbours' rings (distributed shared memory) and the cluster
// barrier after the phase publishes it.  The store may land while a neighbour is still in the same
// phase.  Checkerboard phases read only cells of the other colour.  Partial-line phases read lines
// of the other parity and, in a line's own ring cells, the end values as the sweep's first line
// phase starts: every CTA reads those of both phases there, the second phase's lines push theirs at
// once, and the first phase's lines push the ones that lie on the line's ends (which nothing reads
// before the next sweep) only after the barrier.  A sweep so needs two cluster barriers for its line
// phases (about 600 cycles each).
// ---------------------------------------------------------------------------------------
constexpr int kHP = 34;        // the 32 x 32 tile and its ring
constexpr int kTP = 35;        // ... with an odd pitch
constexpr int kTW = 33;        // pitch of the tile's fields without a ring

struct CTile {
    float P[kHP][kTP], U[kHP][kTP], G[kHP][kTP];            // pn, u, G; tile cell (a, b) at [a + 1][b + 1]
    float W[32][kTW], F[32][kTW], R[32][kTW], Fv[32][kTW], Res[32][kTW];   // w, F, rhs, f, residual
    TileScratch S;
};
constexpr size_t kTileBytes = (sizeof(CTile) + 127) / 128 * 128;

// A tile as tile_smooth sees it: cell (a, b) of the tile at off + a * pu + b of P, U and G and at
// a * pw + b of W, F, R and Fv (places in smf); i0, j0: the tile's place in the n x m grid.
struct TileArgs {
    int n, m, i0, j0, pu, off, pw;
    float cdiff, inv_tau, Sigma, inv_2h, beta;
    int has_rhs;
    int P, U, G, W, F, R, Fv;
};

// Where a tile cell's value goes when it changes: the same cell in the ring of the tile above or below
// (v) and of the tile to the left or right (h), as distributed shared-memory addresses of u (0: no such
// tile, or the cell is not on that edge).  pn and G lie at a fixed distance from u.
struct Push {
    uint32_t v = 0, h = 0;
    __device__ __forceinline__ void to_v(float x, int field = 0) const { if (v) put(v + field, x); }
    __device__ __forceinline__ void to_h(float x, int field = 0) const { if (h) put(h + field, x); }
    static __device__ __forceinline__ void put(uint32_t at, float x) {
        asm volatile("st.shared::cluster.f32 [%0], %1;\n" ::"r"(at), "f"(x) : "memory");
    }
};
constexpr int kPushP = (int)offsetof(CTile, P) - (int)offsetof(CTile, U);
constexpr int kPushG = (int)offsetof(CTile, G) - (int)offsetof(CTile, U);

// Address of `p`, a place in this CTA's shared memory, in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t remote(const void *p, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return r;
}

// The pushes of tile cell (a, b); tile (i0, j0) of an n x m grid, TX tiles a row.
__device__ __forceinline__ Push push_of(CTile &T, int a, int b, int i0, int j0, int n, int m, int rank, int TX) {
    Push p;
    if (a == 0 && i0 > 0) p.v = remote(&T.U[33][b + 1], rank - TX);
    if (a == 31 && i0 + 32 < n) p.v = remote(&T.U[0][b + 1], rank + TX);
    if (b == 0 && j0 > 0) p.h = remote(&T.U[a + 1][33], rank - 1);
    if (b == 31 && j0 + 32 < m) p.h = remote(&T.U[a + 1][0], rank + 1);
    return p;
}

// This thread's number, recomputed wherever it is called for: what a step of the cycle derives from it
// is then not kept (and spilled) across the other steps.
__device__ __forceinline__ int fresh_tid() {
    int t = threadIdx.x;
    asm volatile("" : "+r"(t));
    return t;
}

// All threads of the cluster, with the stores made before it visible after it.
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// The barrier of a tile's threads: the cluster (CL), or the first `nt` threads of the block.
template <bool CL>
__device__ __forceinline__ void tile_sync(int nt) {
    if (CL) cluster_sync();
    else asm volatile("bar.sync 1, %0;\n" ::"r"(nt) : "memory");
}

// One outer smoothing iteration: the snapshot and the four sweeps.  fas: the grid's first
// snapshot after the restriction (u = u0) also completes the FAS right-hand side, rhs += L(pn + u0).
// Not CL: run by the warps that own a row or a column of the grid (w < max(n, m)); the caller's
// other warps wait at the block barrier after it.
template <bool CL>
__device__ __forceinline__ void tile_smooth(const TileArgs &A, TileScratch &S, CTile *T, int TX, int rank, int ntiles,
                                            bool fas) {
    const int n = A.n, m = A.m, i0 = A.i0, j0 = A.j0, pu = A.pu, pw = A.pw;
    const int nt = CL ? kBT : 32 * max(n, m);
    float *const U = smf + A.U + A.off, *const P = smf + A.P + A.off, *const G = smf + A.G + A.off;
    const float cdiff = A.cdiff, inv_tau = A.inv_tau;
    const int tid = fresh_tid(), w = tid >> 5, lane = tid & 31;
    // the own cell (w, lane) and, clamped into the grid (the mirror ghosts), its neighbours: a
    // neighbour outside the grid has the cell's own place
    const bool own = i0 + w < n && j0 + lane < m;
    const int o = own ? w * pu + lane : 0, oc = own ? w * pw + lane : 0;
    const int oS = own && i0 + w + 1 < n ? o + pu : o, oN = own && i0 + w > 0 ? o - pu : o;
    const int oE = own && j0 + lane + 1 < m ? o + 1 : o, oW = own && j0 + lane > 0 ? o - 1 : o;
    if (tid == 0) S.any = 0;
    // CL: where the changes of the own cell and of the transposed cell (lane, w) go
    Push own_push, line_push;
    if (CL) {
        own_push = push_of(*T, w, lane, i0, j0, n, m, rank, TX);
        line_push = push_of(*T, lane, w, i0, j0, n, m, rank, TX);
    }
    // G at pn + u of the own cell; fas: the differences of pn + u to the neighbours too, since after the
    // next barrier a neighbouring tile may be at its first checkerboard phase, whose pushes change this
    // tile's ring of u
    float uc = 0.f, dS = 0.f, dN = 0.f, dE = 0.f, dW = 0.f;
    {
        if (fas) {
            const float pc = P[o];
            uc = U[o];
            dS = add_rn(sub_rn(P[oS], pc), sub_rn(U[oS], uc));
            dN = add_rn(sub_rn(P[oN], pc), sub_rn(U[oN], uc));
            dE = add_rn(sub_rn(P[oE], pc), sub_rn(U[oE], uc));
            dW = add_rn(sub_rn(P[oW], pc), sub_rn(U[oW], uc));
        }
        const float g = cell_G(smf[A.W + oc], P[oS], P[oN], P[oE], P[oW], U[oS], U[oN], U[oE], U[oW], A.inv_2h, A.beta);
        if (own) {
            G[o] = g;
            if (CL) { own_push.to_v(g, kPushG); own_push.to_h(g, kPushG); }
        }
    }
    tile_sync<CL>(nt);
    float aS, aN, aE, aW, dv, fq;
    uint32_t star;
    {
        const bool hS = oS != o, hN = oN != o, hE = oE != o, hW = oW != o;
        const float gc = G[o];
        aS = face(gc, G[oS], hS); aN = face(gc, G[oN], hN);
        aE = face(gc, G[oE], hE); aW = face(gc, G[oW], hW);
        const float pc = P[o], pS = P[oS], pN = P[oN], pE = P[oE], pW = P[oW];
        float ds = mul_rn(aS, sub_rn(pS, pc));
        ds = fma_rn(aN, sub_rn(pN, pc), ds);
        ds = fma_rn(aE, sub_rn(pE, pc), ds);
        ds = fma_rn(aW, sub_rn(pW, pc), ds);
        float base = add_rn(smf[A.F + oc], 0.0f);
        if (fas) {   // as b_residual, mode 1, with uu = u (= u0 here)
            float fl = mul_rn(aS, dS);
            fl = fma_rn(aN, dN, fl);
            fl = fma_rn(aE, dE, fl);
            fl = fma_rn(aW, dW, fl);
            const float rn = add_rn(smf[A.R + oc], sub_rn(fma_rn(cdiff, fl, -base), mul_rn(inv_tau, uc)));
            if (own) smf[A.R + oc] = rn;
            base = add_rn(base, rn);
        } else if (A.has_rhs) {
            base = add_rn(base, smf[A.R + oc]);
        }
        fq = fma_rn(-cdiff, ds, base);
        if (own) smf[A.Fv + oc] = fq;
        const float big = 3.0e38f;
        const float vS = hS ? aS : big, vN = hN ? aN : big, vE = hE ? aE : big, vW = hW ? aW : big;
        const float mn = fminf(fminf(vS, vN), fminf(vE, vW));
        const float mx = fmaxf(fmaxf(hS ? aS : -1.f, hN ? aN : -1.f), fmaxf(hE ? aE : -1.f, hW ? aW : -1.f));
        const int am = vS == mn ? 0 : (vN == mn ? 1 : (vE == mn ? 2 : 3));
        const int cnt = (int)hS + (int)hN + (int)hE + (int)hW;
        star = (own && cnt >= 2 && mx > mul_rn(A.Sigma, mn)) ? (1u << am) : 0u;
        dv = fma_rn(cdiff, add_rn(add_rn(aS, aN), add_rn(aE, aW)), inv_tau);
    }
    // member masks of tile row w (sweeps A, B) and tile column w (C, D)
    const int lenr = min(32, m - j0), lenc = min(32, n - i0);
    S.star[w][lane] = (uint8_t)star;
    const uint32_t mA = members_of(__ballot_sync(0xffffffffu, star & 1u), lenr);
    const uint32_t mB = members_of(__ballot_sync(0xffffffffu, star & 2u), lenr);
    if (CL) __syncthreads();
    else tile_sync<false>(nt);
    const bool town = i0 + lane < n && j0 + w < m;
    const uint32_t st = town ? S.star[lane][w] : 0;
    const uint32_t mC = members_of(__ballot_sync(0xffffffffu, st & 4u), lenc);
    const uint32_t mD = members_of(__ballot_sync(0xffffffffu, st & 8u), lenc);
    if (lane == 0) {
        S.mcol[0][w] = mC;
        S.mcol[1][w] = mD;
        const unsigned a = (mA ? 1u : 0u) | (mB ? 2u : 0u) | (mC ? 4u : 0u) | (mD ? 8u : 0u);
        if (a) atomicOr(&S.any, a);
    }
    if (CL) __syncthreads();
    else tile_sync<false>(nt);
    // the sweeps in which the own cell is a member; bits 8 and up: the sweeps with members anywhere
    unsigned mem = ((mA >> lane) & 1u) | (((mB >> lane) & 1u) << 1);
    if (own) mem |= (((S.mcol[0][lane] >> w) & 1u) << 2) | (((S.mcol[1][lane] >> w) & 1u) << 3);
    unsigned any = S.any;
    if (CL && tid < ntiles) Push::put(remote(&S.anyr[rank], tid), __uint_as_float(any));
    // checkerboard phase of the own cell (i0 and j0 are even); 2: never
    const int colour = own ? (w + lane) & 1 : 2;
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {
        const int rev = k & 1;
#pragma unroll 1
        for (int ph = 0; ph < 2; ++ph) {
            if (colour == (ph ^ rev) && !((mem >> k) & 1u)) {
                float num = mul_rn(aS, U[oS]);
                num = fma_rn(aN, U[oN], num);
                num = fma_rn(aE, U[oE], num);
                num = fma_rn(aW, U[oW], num);
                const float v = div_relax(fma_rn(cdiff, num, -fq), dv);
                U[o] = v;
                if (CL) { own_push.to_v(v); own_push.to_h(v); }
            }
            tile_sync<CL>(nt);
            if (CL && k == 0 && ph == 0)
                for (int r = 0; r < ntiles; ++r) any |= S.anyr[r];   // every tile's bits
        }
        if (!((any >> k) & 1u)) continue;
        // partial lines: this warp's line is tile row w (A, B) or tile column w (C, D)
        const bool rowwise = k < 2;
        const uint32_t mk = k == 0 ? mA : (k == 1 ? mB : (k == 2 ? mC : mD));   // 0 outside the grid
        const int len = rowwise ? lenr : lenc;
        // the line's end values in the neighbouring tiles (no coupling where there is none)
        float e0 = 0.f, e1 = 0.f;
        if (CL && mk) {
            const int t0 = rowwise ? j0 : i0, first = rowwise ? w * pu : w, step = rowwise ? 1 : pu;
            if (t0 > 0) e0 = U[first - step];
            if (t0 + len < (rowwise ? m : n)) e1 = U[first + len * step];
        }
        const bool member = (mk >> lane) & 1u;
        float xn = 0.f;
#pragma unroll 1
        for (int ph = 0; ph < 2; ++ph) {
            if (CL && ph == 1 && member && (w & 1) == rev) {   // the first phase's lines: their end cells
                if (rowwise) own_push.to_h(xn);
                else line_push.to_v(xn);
            }
            if (mk && (w & 1) == (ph ^ rev)) {
                // position `lane` of the line: the own cell, or (columns) the transposed cell (lane, w)
                int lo_ = o, x1 = oS, x2 = oN;
                float ap = aW, an = aE, ax1 = aS, ax2 = aN, dg = dv, fl = fq;
                if (!rowwise) {
                    lo_ = town ? lane * pu + w : 0;
                    const int tS = town && i0 + lane + 1 < n ? lo_ + pu : lo_, tN = town && i0 + lane > 0 ? lo_ - pu : lo_;
                    x1 = town && j0 + w + 1 < m ? lo_ + 1 : lo_;
                    x2 = town && j0 + w > 0 ? lo_ - 1 : lo_;
                    const float tg = G[lo_];
                    an = face(tg, G[tS], tS != lo_);
                    ap = face(tg, G[tN], tN != lo_);
                    ax1 = face(tg, G[x1], x1 != lo_);
                    ax2 = face(tg, G[x2], x2 != lo_);
                    dg = fma_rn(cdiff, add_rn(add_rn(an, ap), add_rn(ax1, ax2)), inv_tau);
                    fl = smf[A.Fv + (town ? lane * pw + w : 0)];
                }
                const float ownv = lane < len ? U[lo_] : 0.f;
                float prevv = __shfl_up_sync(0xffffffffu, ownv, 1), nextv = __shfl_down_sync(0xffffffffu, ownv, 1);
                if (lane == 0) prevv = e0;
                if (lane == len - 1) nextv = e1;
                xn = pcr_cell<float>(mk, len, cdiff, ap, an, ax1, ax2, dg, U[x1], U[x2], fl, prevv, nextv);
                if (member) {
                    U[lo_] = xn;
                    if (CL) {
                        if (rowwise || ph) (rowwise ? own_push : line_push).to_v(xn);
                        if (!rowwise || ph) (rowwise ? own_push : line_push).to_h(xn);
                    }
                }
            }
            tile_sync<CL>(nt);
        }
    }
}

}  // namespace

// Row pitch of a bottom grid of m columns: odd when `pad` (rows of fewer than 16 cells stay dense: a
// column of theirs meets few bank conflicts, and the padding would weigh most).
__host__ __device__ inline int bottom_pitch(int m, int pad) { return pad && m >= 16 ? m | 1 : m; }

// Shared-memory bytes the bottom kernel needs for grids lb .. L-1 (pad: odd row pitches).
size_t bottom_smem_bytes(const int *n, const int *m, int lb, int L, int coarse_fp64, int pad) {
    size_t b = 0;
    int maxN = 0, maxTask = 0;
    for (int l = lb; l < L; ++l) {
        const size_t N = (size_t)n[l] * bottom_pitch(m[l], pad);
        const int npm = (m[l] + 31) / 32, npn = (n[l] + 31) / 32;
        b += 8 * N * sizeof(float);
        b += sizeof(uint32_t) * (2 * (size_t)n[l] * npm + 2 * (size_t)m[l] * npn);
        maxN = std::max(maxN, (int)N);
        maxTask = std::max(maxTask, std::max((n[l] + 1) / 2 * npm, (m[l] + 1) / 2 * npn));
    }
    b += (size_t)maxN;                                   // star bytes
    b = (b + 15) / 16 * 16;
    b += sizeof(float) * 2 * (size_t)maxTask;           // end values
    b = (b + 15) / 16 * 16;
    b += (coarse_fp64 ? sizeof(double) : sizeof(float)) * coarse_scratch_elems(n[L - 1], m[L - 1]);
    return b;
}

// The sub-cycle from grid lb (its u and rhs already in shared memory) down to the coarsest and
// back, run by the whole block: smoothing, residual, restriction, coarse right-hand side, the
// coarsest solve, interpolation, post-smoothing (Algorithm 1).  fas: grid lb's right-hand side still
// lacks L(pn + u0).  One step of the cycle a turn of the loop, so that each step's code stands once.
__device__ __forceinline__ void bottom_subcycle(const BottomArgs &A, const BGrid *Bs, int lb, bool fas, uint8_t *star,
                                                float *endv, TileScratch &S, unsigned char *scratch, double *red,
                                                int *s_err) {
    bool down = true;
    int l = lb, t = 0;   // the grid; smoothing iterations done on it (-1: not yet interpolated)
#pragma unroll 1
    while (l >= lb) {
        const BGrid &B = Bs[l];
        const bool coarsest = l == A.L - 1, one_tile = B.n <= 32 && B.m <= 32;
        const bool smooth = !coarsest && t >= 0 && t < (down ? A.nu1 : A.nu2);
        // a grid's first snapshot completes its right-hand side where tile_smooth takes it
        if (fas && !(smooth && one_tile)) {
            b_residual(B, B.u0, B.rhs, 1);
            fas = false;
        }
        if (smooth) {
            if (one_tile) {
                const TileArgs ta{B.n, B.m, 0, 0, B.P, 0, B.P, B.cdiff, B.inv_tau, B.Sigma, B.inv_2h, B.beta, B.has_rhs,
                                  B.pn, B.u, B.G, B.w, B.F, B.rhs, B.f};
                if ((int)(threadIdx.x >> 5) < max(B.n, B.m)) tile_smooth<false>(ta, S, nullptr, 1, 0, 1, fas);
                __syncthreads();
            } else if (B.n * B.m <= kBT) {
                b_smooth_small(B, star, endv);
            } else {
                b_snapshot(B, star);
#pragma unroll 1
                for (int k = 0; k < 4; ++k) b_sweep(B, k, endv);
            }
            fas = false;
            ++t;
        } else if (coarsest) {
            CoarseGrid<float> cg{B.n, B.m, B.P, smf + B.pn, smf + B.u, smf + B.w, nullptr, smf + B.F, smf + B.rhs,
                                 B.has_rhs, B.inv_2h, B.inv_tau, B.beta};
            int it;
            double res;
            if (A.coarse_fp64)
                coarse_solve_block<float, double>(cg, A.mp, A.sc->A1frac, A.h2nm_coarse, A.coarse_maxit, A.coarse_tol,
                                                  reinterpret_cast<double *>(scratch), red, s_err, &it, &res,
                                                  A.coarse_aos, A.aos_dt);
            else
                coarse_solve_block<float, float>(cg, A.mp, A.sc->A1frac, A.h2nm_coarse, A.coarse_maxit, A.coarse_tol,
                                                 reinterpret_cast<float *>(scratch), red, s_err, &it, &res,
                                                 A.coarse_aos, A.aos_dt);
            if (threadIdx.x == 0) {
                A.sc->picard = it;
                A.sc->coarse_res = res;
                if (*s_err) A.sc->err = 1;
            }
            down = false;
            --l;
            t = -1;
        } else if (down) {
            b_residual(B, B.u, B.f, 0);
            b_restrict(B, Bs[l + 1]);
            fas = true;
            ++l;
            t = 0;
        } else if (t < 0) {
            b_interp_add(B, Bs[l + 1]);
            t = 0;
        } else {
            --l;
            t = -1;
        }
    }
}

// Carves the shared memory of grids lb .. L-1 (thread 0) and loads pn, w and F of every grid and,
// when load_first, u and rhs of grid lb.  s_off: bytes to the star bytes, end values, coarsest-solve
// scratch.
__device__ __forceinline__ void bottom_setup(const BottomArgs &A, BGrid *Bs, int lb, bool load_first, size_t first_byte,
                                             size_t *s_off) {
    if (threadIdx.x == 0) {
        size_t off = first_byte;
        int maxN = 0, maxTask = 0;
        for (int l = lb; l < A.L; ++l) {
            const LevelView<float> &G = A.g[l];
            BGrid &B = Bs[l];
            B.n = G.n; B.m = G.m; B.npm = (G.m + 31) / 32; B.npn = (G.n + 31) / 32;
            B.P = bottom_pitch(G.m, A.pad);
            B.cdiff = G.cdiff; B.inv_tau = G.inv_tau; B.Sigma = G.Sigma; B.inv_2h = G.inv_2h; B.beta = G.beta;
            B.has_rhs = G.has_rhs;
            const int N = G.n * B.P;
            int at = (int)(off / sizeof(float));
            auto take = [&](int words) { const int a = at; at += words; return a; };
            B.pn = take(N); B.u = take(N); B.w = take(N); B.F = take(N);
            B.rhs = take(N); B.G = take(N); B.f = take(N); B.u0 = take(N);
            B.mrow = take(2 * G.n * B.npm);
            B.mcol = take(2 * G.m * B.npn);
            off = sizeof(float) * (size_t)at;
            maxN = max(maxN, N);
            maxTask = max(maxTask, max((G.n + 1) / 2 * B.npm, (G.m + 1) / 2 * B.npn));
        }
        s_off[0] = off;                                 // star bytes
        off += maxN;
        off = (off + 15) / 16 * 16;
        s_off[1] = off;                                 // end values
        off += sizeof(float) * 2 * maxTask;
        off = (off + 15) / 16 * 16;
        s_off[2] = off;                                 // coarsest-solve scratch
    }
    __syncthreads();
    for (int l = lb; l < A.L; ++l) {
        const LevelView<float> &G = A.g[l];
        const BGrid &B = Bs[l];
        const Map2 M = map_for(B.m);
        FOR_CELLS(M, B.n, B.m, i, j) {
            const int q = i * B.P + j;
            const size_t o = (size_t)i * G.pitch + j, lim = (size_t)G.n * G.pitch;
            smf[B.pn + q] = ldc(G.pn, o, lim, kDbgBottom);
            smf[B.w + q] = weight_at(G, o);
            smf[B.F + q] = ldc(G.F, o, lim, kDbgBottom);
        }
    }
    pdl_wait();      // what lies above is fixed during a step; grid lb's u and rhs come from the
    pdl_trigger();   // kernel before
    if (load_first) {
        const LevelView<float> &G = A.first;
        const BGrid &B = Bs[lb];
        const Map2 M = map_for(B.m);
        FOR_CELLS(M, B.n, B.m, i, j) {
            const int q = i * B.P + j;
            const size_t o = (size_t)i * G.pitch + j, lim = (size_t)G.n * G.pitch;
            if (!MG_DBG_OK(o, lim, kDbgBottom)) continue;
            const float u = __ldcg(G.u + o);
            smf[B.u + q] = u;
            smf[B.u0 + q] = u;
            smf[B.rhs + q] = G.has_rhs ? __ldcg(G.rhs + o) : 0.f;
        }
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kBT) k_bottom(const __grid_constant__ BottomArgs A) {
    __shared__ double red[33];
    __shared__ int s_err;
    __shared__ BGrid Bs[kMaxLevels];
    __shared__ size_t s_off[3];
    __shared__ TileScratch ts;
    unsigned char *sm = reinterpret_cast<unsigned char *>(smf);
    bottom_setup(A, Bs, A.lb, true, 0, s_off);
    bottom_subcycle(A, Bs, A.lb, A.fas != 0, sm + s_off[0], reinterpret_cast<float *>(sm + s_off[1]), ts, sm + s_off[2], red,
                    &s_err);
    // ---- grid lb's increment back to global memory
    {
        const LevelView<float> &G = A.g[A.lb];
        const BGrid &B = Bs[A.lb];
        const Map2 M = map_for(B.m);
        FOR_CELLS(M, B.n, B.m, i, j)
            stc(G.u, (size_t)i * G.pitch + j, (size_t)G.n * G.pitch, kDbgBottom, smf[B.u + i * B.P + j]);
    }
}

// ---------------------------------------------------------------------------------------
// The bottom of the V-cycle from a grid spread over a thread-block cluster.  On grids of about
// 64^2 every per-grid launch is latency-bound (a V-cycle spends about 23 launches per grid) while
// one block is too little for the grid.  Here one 1024-thread CTA owns each 32 x 32 tile of grid
// lc (one cell per thread, at most 16 tiles: one cluster) in its shared memory and smooths it with
// tile_smooth.  CTA 0 also holds grids lc+1 .. L-1 and runs their sub-cycle (bottom_subcycle)
// between the restriction and the interpolation.  Every cell performs the per-grid kernels'
// operations, so the results are the same.
// ---------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kBT) k_cluster(const __grid_constant__ BottomArgs A) {
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    __shared__ double red[33];
    __shared__ int s_err;
    __shared__ BGrid Bs[kMaxLevels];
    __shared__ size_t s_off[3];
    __shared__ CTile *tp[16];
    unsigned char *sm = reinterpret_cast<unsigned char *>(smf);
    CTile &T = *reinterpret_cast<CTile *>(smf);
    const int lc = A.lb;
    const LevelView<float> &Lg = A.first;   // grid lc: at a fixed place of the arguments, read without registers
    const int n = Lg.n, m = Lg.m, TX = (m + 31) / 32;
    const float cdiff = Lg.cdiff, inv_tau = Lg.inv_tau, inv_2h = Lg.inv_2h, beta = Lg.beta;
    const bool has_rhs = Lg.has_rhs != 0;
    const int rank = (int)cl.block_rank(), ntiles = (int)cl.num_blocks();
    const int ty = rank / TX, tx = rank - ty * TX, i0 = ty * 32, j0 = tx * 32;
    if ((int)threadIdx.x < ntiles) tp[threadIdx.x] = cl.map_shared_rank(&T, threadIdx.x);
    auto place_of = [&](const float *a) { return (int)(a - smf); };
    // the thread's cell: its tile row and column, its grid row and column, its place in the padded
    // arrays and its neighbours' (clamped into the grid: the mirror ghosts)
    struct Cell {
        int ti, lane, i, j, r0, c0, rS, rN, cE, cW;
        bool own, hS, hN, hE, hW;
    };
    auto cell_of_thread = [&]() {
        Cell c;
        const int q = fresh_tid();
        c.ti = q >> 5; c.lane = q & 31; c.i = i0 + c.ti; c.j = j0 + c.lane;
        c.own = c.i < n && c.j < m;
        c.r0 = c.ti + 1; c.c0 = c.lane + 1;
        c.hS = c.i + 1 < n; c.hN = c.i > 0; c.hE = c.j + 1 < m; c.hW = c.j > 0;
        c.rS = c.hS ? c.r0 + 1 : c.r0; c.rN = c.hN ? c.r0 - 1 : c.r0;
        c.cE = c.hE ? c.c0 + 1 : c.c0; c.cW = c.hW ? c.c0 - 1 : c.c0;
        return c;
    };
    const TileArgs ta{n, m, i0, j0, kTP, kTP + 1, kTW, cdiff, inv_tau, Lg.Sigma, inv_2h, beta, Lg.has_rhs,
                      place_of(&T.P[0][0]), place_of(&T.U[0][0]), place_of(&T.G[0][0]), place_of(&T.W[0][0]),
                      place_of(&T.F[0][0]), place_of(&T.R[0][0]), place_of(&T.Fv[0][0])};
    {
        const Cell c = cell_of_thread();
        if (c.own) {
            const size_t o = (size_t)c.i * Lg.pitch + c.j, lim = (size_t)n * Lg.pitch;
            T.P[c.r0][c.c0] = ldc(Lg.pn, o, lim, kDbgBottom);
            T.W[c.ti][c.lane] = weight_at(Lg, o);
            T.F[c.ti][c.lane] = ldc(Lg.F, o, lim, kDbgBottom);
        }
    }
    // grids lc+1 .. L-1: every CTA carves the same offsets (CTA 0's arrays are then reached by
    // mapping this CTA's addresses); their pn, w, F are loaded
    bottom_setup(A, Bs, lc + 1, false, kTileBytes, s_off);   // (waits for the kernel before)
    {
        const Cell c = cell_of_thread();
        const size_t o = (size_t)c.i * Lg.pitch + c.j, lim = (size_t)n * Lg.pitch;
        if (c.own && MG_DBG_OK(o, lim, kDbgBottom)) {
            T.U[c.r0][c.c0] = __ldcg(Lg.u + o);
            T.R[c.ti][c.lane] = has_rhs ? __ldcg(Lg.rhs + o) : 0.f;
        }
    }
    cluster_sync();   // every CTA of the cluster runs: its shared memory may be written
    {
        const Cell c = cell_of_thread();
        if (c.own) {
            const Push push = push_of(T, c.ti, c.lane, i0, j0, n, m, rank, TX);
            push.to_v(T.P[c.r0][c.c0], kPushP);
            push.to_h(T.P[c.r0][c.c0], kPushP);
            push.to_v(T.U[c.r0][c.c0]);
            push.to_h(T.U[c.r0][c.c0]);
        }
    }
    cluster_sync();
    // ---- pre-smoothing, the coarse-grid correction, post-smoothing (each step's code once)
#pragma unroll 1
    for (int up = 0; up < 2; ++up) {
#pragma unroll 1
        for (int t = 0; t < (up ? A.nu2 : A.nu1); ++t)
            tile_smooth<true>(ta, T.S, &T, TX, rank, ntiles, A.fas && !up && t == 0);
        if (up) break;
        // ---- residual r = rhs - L(pn + u) of the own cell (as b_residual, mode 0)
        {
            const Cell c = cell_of_thread();
            const int r0 = c.r0, c0 = c.c0;
            if (c.own) {
                const float g = cell_G(T.W[c.ti][c.lane], T.P[c.rS][c0], T.P[c.rN][c0], T.P[r0][c.cE], T.P[r0][c.cW],
                                       T.U[c.rS][c0], T.U[c.rN][c0], T.U[r0][c.cE], T.U[r0][c.cW], inv_2h, beta);
                T.G[r0][c0] = g;
                const Push push = push_of(T, c.ti, c.lane, i0, j0, n, m, rank, TX);
                push.to_v(g, kPushG);
                push.to_h(g, kPushG);
            }
            cluster_sync();
            if (c.own) {
                const float gc = T.G[r0][c0];
                const float aS = face(gc, T.G[c.rS][c0], c.hS), aN = face(gc, T.G[c.rN][c0], c.hN);
                const float aE = face(gc, T.G[r0][c.cE], c.hE), aW = face(gc, T.G[r0][c.cW], c.hW);
                const float pcv = T.P[r0][c0], uc = T.U[r0][c0];
                float fl = mul_rn(aS, add_rn(sub_rn(T.P[c.rS][c0], pcv), sub_rn(T.U[c.rS][c0], uc)));
                fl = fma_rn(aN, add_rn(sub_rn(T.P[c.rN][c0], pcv), sub_rn(T.U[c.rN][c0], uc)), fl);
                fl = fma_rn(aE, add_rn(sub_rn(T.P[r0][c.cE], pcv), sub_rn(T.U[r0][c.cE], uc)), fl);
                fl = fma_rn(aW, add_rn(sub_rn(T.P[r0][c.cW], pcv), sub_rn(T.U[r0][c.cW], uc)), fl);
                const float Lv = sub_rn(fma_rn(cdiff, fl, -add_rn(T.F[c.ti][c.lane], 0.0f)), mul_rn(inv_tau, uc));
                T.Res[c.ti][c.lane] = has_rhs ? sub_rn(T.R[c.ti][c.lane], Lv) : -Lv;
            }
            cluster_sync();
        }
        // ---- CTA 0: restriction of the residual and of u (as b_restrict), the coarse right-hand
        // side, and the sub-cycle of grids lc+1 .. L-1
        if (rank == 0) {
            const BGrid &C = Bs[lc + 1];
            auto fine = [&](bool res, int a, int b) -> float {   // a fine cell inside the grid
                const CTile *t = tp[(a >> 5) * TX + (b >> 5)];
                return res ? t->Res[a & 31][b & 31] : t->U[(a & 31) + 1][(b & 31) + 1];
            };
            const Map2 M = map_for(C.m);
            FOR_CELLS(M, C.n, C.m, I, J) {
                int ri[3], ci[3];
                float rw[3], cw[3];
                const int nr = fw_taps(I, n, ri, rw), nk = fw_taps(J, m, ci, cw);
                float sr = 0.f, su = 0.f;
                for (int a = 0; a < nr; ++a) {
                    float rr = 0.f, ru = 0.f;
                    for (int b = 0; b < nk; ++b) {
                        rr = fma_rn(cw[b], fine(true, ri[a], ci[b]), rr);
                        ru = fma_rn(cw[b], fine(false, ri[a], ci[b]), ru);
                    }
                    sr = fma_rn(rw[a], rr, sr);
                    su = fma_rn(rw[a], ru, su);
                }
                const int o = I * C.P + J;
                smf[C.rhs + o] = sr;
                smf[C.u + o] = su;
                smf[C.u0 + o] = su;
            }
            __syncthreads();
            bottom_subcycle(A, Bs, lc + 1, true, sm + s_off[0], reinterpret_cast<float *>(sm + s_off[1]), T.S, sm + s_off[2],
                            red, &s_err);
        }
        cluster_sync();
        // ---- interpolation of CTA 0's coarse correction (as b_interp_add)
        {
            const BGrid &C = Bs[lc + 1];
            const float *Cu = cl.map_shared_rank(smf + C.u, 0), *Cu0 = cl.map_shared_rank(smf + C.u0, 0);
            const Cell c = cell_of_thread();
            if (c.own) {
                int ri[2], ci[2];
                float rw[2], cw[2];
                const int nr = bl_taps(c.i, C.n, ri, rw), nk = bl_taps(c.j, C.m, ci, cw);
                float sum = 0.f;
                for (int a = 0; a < nr; ++a)
                    for (int b = 0; b < nk; ++b) {
                        const int o = ri[a] * C.P + ci[b];
                        sum = fma_rn(rw[a] * cw[b], sub_rn(Cu[o], Cu0[o]), sum);
                    }
                const float v = add_rn(T.U[c.r0][c.c0], sum);
                T.U[c.r0][c.c0] = v;
                const Push push = push_of(T, c.ti, c.lane, i0, j0, n, m, rank, TX);
                push.to_v(v);
                push.to_h(v);
            }
        }
        cluster_sync();
    }
    const Cell c = cell_of_thread();
    if (c.own) stc(Lg.u, (size_t)c.i * Lg.pitch + c.j, (size_t)n * Lg.pitch, kDbgBottom, T.U[c.r0][c.c0]);
    cluster_sync();   // no CTA leaves while another may still read its shared memory
}

void prepare_bottom_kernel() {
    cudaFuncSetAttribute(k_bottom, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBottomSmemPad);
    // a refused attribute leaves the cluster kernel unusable: cluster_fits then reports no fit
    if (cudaFuncSetAttribute(k_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClusterSmemMax) != cudaSuccess ||
        cudaFuncSetAttribute(k_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
        cudaGetLastError();
}

void launch_bottom(const BottomArgs &A, size_t smem, cudaStream_t st) {
    launch_pdl(k_bottom, dim3(1), dim3(kBT), smem, st, A);
}

size_t cluster_smem_bytes(size_t bottom_bytes) { return kTileBytes + bottom_bytes; }

int cluster_fits(int tiles, size_t smem) {
    if (tiles < 1 || tiles > kClusterMaxTiles || smem > kClusterSmemMax) return 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(tiles);
    cfg.blockDim = dim3(kBT);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = tiles;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int nc = 0;
    const cudaError_t e = cudaOccupancyMaxActiveClusters(&nc, k_cluster, &cfg);
    if (e != cudaSuccess) {
        cudaGetLastError();   // the query's error is reported through the return value
        return -(int)e;
    }
    return nc;
}

void launch_cluster(const BottomArgs &A, int tiles, size_t smem, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(tiles);
    cfg.blockDim = dim3(kBT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = tiles;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    cudaLaunchKernelEx(&cfg, k_cluster, A);
}

}  // namespace segmg
