// tail_kernel.cu -- the smallest grids of the V-cycle in one block, for the paths whose bottom
// bottom_kernel.cu does not run: FP64 storage and the Rada-Chen model.
//
// On these grids a launch costs 4 to 7 us and a grid takes about 25 of them a V-cycle (with the
// Rada-Chen area terms 35) for a few hundred cells of work.  One block of 256 threads runs them from
// the first grid that fits down to the coarsest and back, every grid in shared memory, with the
// per-grid kernels' operations in their order (cell_G, face, point_relax, pcr_piece, the transfer
// taps, the area sum's order, the coarsest solve): the results are the same numbers.  517x700 Rada-Chen
// step 7.05 -> 5.97 ms, 128x128 FP64 step 29.4 -> 26.2 ms.
//
// First grid: at most 32 x 32 cells in FP32, one 32-cell piece a line and one area partial.  In FP64 at
// most 256 cells: one SM does two FP64 multiply-adds a cycle, so a larger grid's cells cost more here
// than the launches that spread them over more SMs.
#include "arith.cuh"
#include "coarse_body.cuh"
#include "reduce.cuh"
#include "tma.cuh"

#include <algorithm>

namespace segmg {

namespace {

constexpr int kNT = 256, kWarps = kNT / 32;

extern __shared__ __align__(16) unsigned char smem_tail[];
template <typename T>
__device__ __forceinline__ T *sm() { return reinterpret_cast<T *>(smem_tail); }

// Odd row pitch: a column's cells lie in different banks.
__host__ __device__ inline int tail_pitch(int m) { return m | 1; }

template <typename T>
struct TGrid {
    int n, m, P, has_rhs;
    T cdiff, inv_tau, Sigma, inv_2h, beta;
    double h2nm;
    int pn, u, w, F, rhs, G, f, u0;   // places in the shared memory (values of T)
};

struct TailShared {
    double red[33];
    uint8_t star[32][32];
    uint32_t mrow[2][32], mcol[2][32];   // member masks of the lines of sweeps A, B and C, D
    int s_err;
    unsigned any;                        // bit k: sweep k has a member cell
};

// Cells (i, j) of an n x m grid (m <= 32): a power of two >= m threads a row.
#define TAIL_CELLS(n_, m_, i, j)                                                                       \
    for (int lg_ = (m_) <= 1 ? 0 : 32 - __clz((m_) - 1), j = (int)threadIdx.x & ((1 << lg_) - 1),       \
             i = (int)threadIdx.x >> lg_;                                                              \
         i < (n_); i += kNT >> lg_)                                                                    \
        if (j < (m_))

// G at pn + uu.
template <typename T>
__device__ __forceinline__ void t_G(const TGrid<T> &B, int uu) {
    const T *pn = sm<T>() + B.pn, *u = sm<T>() + uu, *w = sm<T>() + B.w;
    const int n = B.n, m = B.m, P = B.P;
    TAIL_CELLS(n, m, i, j) {
        const int q = i * P + j;
        const int s = i + 1 < n ? q + P : q, nn = i > 0 ? q - P : q, e = j + 1 < m ? q + 1 : q, x = j > 0 ? q - 1 : q;
        sm<T>()[B.G + q] = cell_G(w[q], pn[s], pn[nn], pn[e], pn[x], u[s], u[nn], u[e], u[x], B.inv_2h, B.beta);
    }
    __syncthreads();
}

// The Rada-Chen area term at pn + uu (as k_area_partials and k_area_final on one tile).
template <typename T>
__device__ __forceinline__ T t_area(const TGrid<T> &B, int uu, const ModelParams &mp, double A1frac, double *red) {
    const T eps = T(mp.eps);
    T s = T(0);
    for (int q = threadIdx.x; q < 1024; q += kNT) {
        const int i = q / 32, j = q % 32;
        if (i >= B.n || j >= B.m) continue;
        const int o = i * B.P + j;
        s += T(0.5) + atan((sm<T>()[B.pn + o] + sm<T>()[uu + o]) / eps) * T(M_1_PI);
    }
    const double v = block_sum_warps(s, red);
    return T(2.0 * mp.nu * (B.h2nm * v - A1frac));
}

template <typename T>
struct TFaces {
    T S, N, E, W;
    int oS, oN, oE, oW;
    bool hS, hN, hE, hW;
};
template <typename T>
__device__ __forceinline__ TFaces<T> t_faces(const TGrid<T> &B, int i, int j) {
    const T *G = sm<T>() + B.G;
    const int q = i * B.P + j;
    TFaces<T> a;
    a.hS = i + 1 < B.n; a.hN = i > 0; a.hE = j + 1 < B.m; a.hW = j > 0;
    a.oS = a.hS ? q + B.P : q; a.oN = a.hN ? q - B.P : q; a.oE = a.hE ? q + 1 : q; a.oW = a.hW ? q - 1 : q;
    const T gc = G[q];
    a.S = face(gc, G[a.oS], a.hS); a.N = face(gc, G[a.oN], a.hN);
    a.E = face(gc, G[a.oE], a.hE); a.W = face(gc, G[a.oW], a.hW);
    return a;
}

// Snapshot: G, f, the jump classes and the member masks.
template <typename T>
__device__ __forceinline__ void t_snapshot(const TGrid<T> &B, T ar, TailShared &S) {
    if (threadIdx.x == 0) S.any = 0;
    t_G(B, B.u);
    const T *pn = sm<T>() + B.pn;
    const int n = B.n, m = B.m;
    TAIL_CELLS(n, m, i, j) {
        const int q = i * B.P + j;
        const TFaces<T> a = t_faces(B, i, j);
        const T pc = pn[q];
        T ds = mul_rn(a.S, sub_rn(pn[a.oS], pc));
        ds = fma_rn(a.N, sub_rn(pn[a.oN], pc), ds);
        ds = fma_rn(a.E, sub_rn(pn[a.oE], pc), ds);
        ds = fma_rn(a.W, sub_rn(pn[a.oW], pc), ds);
        T base = add_rn(sm<T>()[B.F + q], ar);
        if (B.has_rhs) base = add_rn(base, sm<T>()[B.rhs + q]);
        sm<T>()[B.f + q] = fma_rn(-B.cdiff, ds, base);
        const T big = T(3.0e38);
        const T vS = a.hS ? a.S : big, vN = a.hN ? a.N : big, vE = a.hE ? a.E : big, vW = a.hW ? a.W : big;
        const T mn = fmin(fmin(vS, vN), fmin(vE, vW));
        const T mx = fmax(fmax(a.hS ? a.S : T(-1), a.hN ? a.N : T(-1)), fmax(a.hE ? a.E : T(-1), a.hW ? a.W : T(-1)));
        const int am = vS == mn ? 0 : (vN == mn ? 1 : (vE == mn ? 2 : 3));
        const int cnt = (int)a.hS + (int)a.hN + (int)a.hE + (int)a.hW;
        S.star[i][j] = (cnt >= 2 && mx > mul_rn(B.Sigma, mn)) ? (uint8_t)(1u << am) : (uint8_t)0;
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = warp; i < n; i += kWarps) {
        const unsigned s = lane < m ? S.star[i][lane] : 0u;
        const uint32_t a = members_of(__ballot_sync(0xffffffffu, s & 1u), m);
        const uint32_t b = members_of(__ballot_sync(0xffffffffu, s & 2u), m);
        if (lane == 0) {
            S.mrow[0][i] = a;
            S.mrow[1][i] = b;
            if (a | b) atomicOr(&S.any, (a ? 1u : 0u) | (b ? 2u : 0u));
        }
    }
    for (int j = warp; j < m; j += kWarps) {
        const unsigned s = lane < n ? S.star[lane][j] : 0u;
        const uint32_t a = members_of(__ballot_sync(0xffffffffu, s & 4u), n);
        const uint32_t b = members_of(__ballot_sync(0xffffffffu, s & 8u), n);
        if (lane == 0) {
            S.mcol[0][j] = a;
            S.mcol[1][j] = b;
            if (a | b) atomicOr(&S.any, (a ? 4u : 0u) | (b ? 8u : 0u));
        }
    }
    __syncthreads();
}

// The two checkerboard phases of a sweep.
template <typename T>
__device__ __forceinline__ void t_points(const TGrid<T> &B, int sweep, const TailShared &S) {
    T *u = sm<T>() + B.u;
    const T *f = sm<T>() + B.f;
#pragma unroll 1
    for (int ph = 0; ph < 2; ++ph) {
        const int colour = (sweep & 1) ? 1 - ph : ph;
        TAIL_CELLS(B.n, B.m, i, j) {
            if (((i + j) & 1) != colour) continue;
            const uint32_t mk = sweep < 2 ? S.mrow[sweep][i] >> j : S.mcol[sweep - 2][j] >> i;
            if (mk & 1u) continue;
            const TFaces<T> a = t_faces(B, i, j);
            const int q = i * B.P + j;
            u[q] = point_relax(B.cdiff, B.inv_tau, a.S, a.N, a.E, a.W, u[a.oS], u[a.oN], u[a.oE], u[a.oW], f[q]);
        }
        __syncthreads();
    }
}

// The two partial-line phases of a sweep (one piece a line: nothing lies before or after it).
template <typename T>
__device__ __forceinline__ void t_lines(const TGrid<T> &B, int sweep, const TailShared &S) {
    const int n = B.n, m = B.m;
    const bool rev = sweep & 1, rowwise = sweep < 2;
    T *u = sm<T>() + B.u;
    const T *f = sm<T>() + B.f;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nlines = rowwise ? n : m, len = rowwise ? m : n;
#pragma unroll 1
    for (int ph = 0; ph < 2; ++ph) {
        for (int line = (rev ? 1 - ph : ph) + 2 * warp; line < nlines; line += 2 * kWarps) {
            const uint32_t mk = rowwise ? S.mrow[sweep][line] : S.mcol[sweep - 2][line];
            if (!mk) continue;   // the whole warp
            auto place = [&](int t) { return rowwise ? line * B.P + t : t * B.P + line; };
            const T own = lane < len ? u[place(lane)] : T(0);
            auto at = [&](int t) -> RunCell<T> {
                const TFaces<T> a = t_faces(B, rowwise ? line : t, rowwise ? t : line);
                RunCell<T> c;
                if (rowwise) { c.ap = a.W; c.an = a.E; c.ax1 = a.S; c.ax2 = a.N; c.ux1 = u[a.oS]; c.ux2 = u[a.oN]; }
                else         { c.ap = a.N; c.an = a.S; c.ax1 = a.E; c.ax2 = a.W; c.ux1 = u[a.oE]; c.ux2 = u[a.oW]; }
                c.f = f[place(t)];
                return c;
            };
            T x;
            if (pcr_piece<T>(mk, len, B.cdiff, B.inv_tau, own, T(0), T(0), at, x)) u[place(lane)] = x;
        }
        __syncthreads();
    }
}

// The four sweeps of Hybrid Smoother 2 after the snapshot.  On a grid of one cell a thread the cell's
// faces, diagonal, f and member bits stay in registers over all of them: FP64 face sums and diagonals
// are then formed once, not in each of eight phases (128x128 FP64 step 27.6 -> 26.2 ms).  Line phases
// without a member are skipped.
template <typename T>
__device__ __forceinline__ void t_sweeps(const TGrid<T> &B, const TailShared &S) {
    const unsigned any = S.any;
    const int lg = B.m <= 1 ? 0 : 32 - __clz(B.m - 1), i = (int)threadIdx.x >> lg, j = (int)threadIdx.x & ((1 << lg) - 1);
    if (B.n > kNT >> lg) {
#pragma unroll 1
        for (int k = 0; k < 4; ++k) {
            t_points(B, k, S);
            if ((any >> k) & 1u) t_lines(B, k, S);
        }
        return;
    }
    const bool own = i < B.n && j < B.m;
    T *u = sm<T>() + B.u;
    TFaces<T> a{};
    T dv = T(1), fq = T(0);
    int q = 0, colour = 2;
    unsigned mem = 0;
    if (own) {
        a = t_faces(B, i, j);
        q = i * B.P + j;
        dv = fma_rn(B.cdiff, add_rn(add_rn(a.S, a.N), add_rn(a.E, a.W)), B.inv_tau);
        fq = sm<T>()[B.f + q];
        colour = (i + j) & 1;
        mem = ((S.mrow[0][i] >> j) & 1u) | (((S.mrow[1][i] >> j) & 1u) << 1) | (((S.mcol[0][j] >> i) & 1u) << 2) |
              (((S.mcol[1][j] >> i) & 1u) << 3);
    }
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {
#pragma unroll 1
        for (int ph = 0; ph < 2; ++ph) {
            if (colour == (ph ^ (k & 1)) && !((mem >> k) & 1u)) {
                T num = mul_rn(a.S, u[a.oS]);
                num = fma_rn(a.N, u[a.oN], num);
                num = fma_rn(a.E, u[a.oE], num);
                num = fma_rn(a.W, u[a.oW], num);
                u[q] = div_relax(fma_rn(B.cdiff, num, -fq), dv);
            }
            __syncthreads();
        }
        if ((any >> k) & 1u) t_lines(B, k, S);
    }
}

// out = rhs - L(pn + uu) (mode 0) or out += L(pn + uu) (mode 1).
template <typename T>
__device__ __forceinline__ void t_residual(const TGrid<T> &B, int uu_, int out_, int mode, T ar) {
    t_G(B, uu_);
    const T *pn = sm<T>() + B.pn, *uu = sm<T>() + uu_;
    T *out = sm<T>() + out_;
    TAIL_CELLS(B.n, B.m, i, j) {
        const int q = i * B.P + j;
        const TFaces<T> a = t_faces(B, i, j);
        const T pc = pn[q], uc = uu[q];
        T fl = mul_rn(a.S, add_rn(sub_rn(pn[a.oS], pc), sub_rn(uu[a.oS], uc)));
        fl = fma_rn(a.N, add_rn(sub_rn(pn[a.oN], pc), sub_rn(uu[a.oN], uc)), fl);
        fl = fma_rn(a.E, add_rn(sub_rn(pn[a.oE], pc), sub_rn(uu[a.oE], uc)), fl);
        fl = fma_rn(a.W, add_rn(sub_rn(pn[a.oW], pc), sub_rn(uu[a.oW], uc)), fl);
        const T Lv = sub_rn(fma_rn(B.cdiff, fl, -add_rn(sm<T>()[B.F + q], ar)), mul_rn(B.inv_tau, uc));
        if (mode == 0) out[q] = B.has_rhs ? sub_rn(sm<T>()[B.rhs + q], Lv) : -Lv;
        else out[q] = add_rn(out[q], Lv);
    }
    __syncthreads();
}

// Full weighting of the residual (in f) and of u of grid B onto grid C (rhs; u and u0).
template <typename T>
__device__ __forceinline__ void t_restrict(const TGrid<T> &B, const TGrid<T> &C) {
    TAIL_CELLS(C.n, C.m, I, J) {
        int ri[3], ci[3];
        float rw[3], cw[3];
        const int nr = fw_taps(I, B.n, ri, rw), nk = fw_taps(J, B.m, ci, cw);
        auto weigh = [&](const T *src) {
            T s = T(0);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if (a >= nr) break;
                T row = T(0);
#pragma unroll
                for (int b = 0; b < 3; ++b)
                    if (b < nk) row = fma_rn(T(cw[b]), src[ri[a] * B.P + ci[b]], row);
                s = fma_rn(T(rw[a]), row, s);
            }
            return s;
        };
        const int q = I * C.P + J;
        sm<T>()[C.rhs + q] = weigh(sm<T>() + B.f);
        const T su = weigh(sm<T>() + B.u);
        sm<T>()[C.u + q] = su;
        sm<T>()[C.u0 + q] = su;
    }
    __syncthreads();
}

// B.u += P (C.u - C.u0).
template <typename T>
__device__ __forceinline__ void t_interp(const TGrid<T> &B, const TGrid<T> &C) {
    TAIL_CELLS(B.n, B.m, i, j) {
        int ri[2], ci[2];
        float rw[2], cw[2];
        const int nr = bl_taps(i, C.n, ri, rw), nk = bl_taps(j, C.m, ci, cw);
        T s = T(0);
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b)
                if (a < nr && b < nk) {
                    const int o = ri[a] * C.P + ci[b];
                    s = fma_rn(T(rw[a] * cw[b]), sub_rn(sm<T>()[C.u + o], sm<T>()[C.u0 + o]), s);
                }
        T &x = sm<T>()[B.u + i * B.P + j];
        x = add_rn(x, s);
    }
    __syncthreads();
}

template <typename T, typename C>
__global__ void __launch_bounds__(kNT) k_tail(const __grid_constant__ TailArgs<T> A) {
    __shared__ TailShared S;
    __shared__ TGrid<T> Bs[kMaxLevels];
    __shared__ int s_scratch;
    const int first = A.first, last = A.L - 1;
    if (threadIdx.x == 0) {
        int at = 0;
        for (int l = first; l < A.L; ++l) {
            const LevelView<T> &G = A.g[l];
            TGrid<T> &B = Bs[l];
            B.n = G.n; B.m = G.m; B.P = tail_pitch(G.m); B.has_rhs = G.has_rhs;
            B.cdiff = G.cdiff; B.inv_tau = G.inv_tau; B.Sigma = G.Sigma; B.inv_2h = G.inv_2h; B.beta = G.beta;
            B.h2nm = A.h2nm[l];
            const int N = B.n * B.P;
            int *place[8] = {&B.pn, &B.u, &B.w, &B.F, &B.rhs, &B.G, &B.f, &B.u0};
            for (int k = 0; k < 8; ++k, at += N) *place[k] = at;
        }
        s_scratch = (int)((at * sizeof(T) + 15) / 16 * 16);
    }
    __syncthreads();
    for (int l = first; l <= last; ++l) {   // fixed during a step: read before the dependent launch's wait
        const LevelView<T> &G = A.g[l];
        const TGrid<T> &B = Bs[l];
        TAIL_CELLS(B.n, B.m, i, j) {
            const size_t o = (size_t)i * G.pitch + j, lim = (size_t)G.n * G.pitch;
            const int q = i * B.P + j;
            sm<T>()[B.pn + q] = ldc(G.pn, o, lim, kDbgBottom);
            sm<T>()[B.w + q] = weight_at(G, o);
            sm<T>()[B.F + q] = ldc(G.F, o, lim, kDbgBottom);
        }
    }
    pdl_wait();
    pdl_trigger();
    {
        const LevelView<T> &G = A.g[first];
        const TGrid<T> &B = Bs[first];
        TAIL_CELLS(B.n, B.m, i, j) {
            const size_t o = (size_t)i * G.pitch + j, lim = (size_t)G.n * G.pitch;
            const int q = i * B.P + j;
            const T u = ldl2(G.u, o, lim, kDbgBottom);
            sm<T>()[B.u + q] = u;
            sm<T>()[B.u0 + q] = u;
            sm<T>()[B.rhs + q] = ldl2(G.rhs, o, lim, kDbgBottom);
        }
    }
    const double A1frac = __ldcg(&A.sc->A1frac);
    const bool rc = A.mp.model == 1;
    __syncthreads();
    bool down = true, fas = A.fas != 0;
    int l = first, t = 0;   // the grid; smoothing iterations done on it (-1: not yet interpolated)
#pragma unroll 1
    while (l >= first) {
        const TGrid<T> &B = Bs[l];
        if (l == last) {
            CoarseGrid<T> cg{B.n, B.m, B.P, sm<T>() + B.pn, sm<T>() + B.u, sm<T>() + B.w, nullptr, sm<T>() + B.F,
                             sm<T>() + B.rhs, B.has_rhs, B.inv_2h, B.inv_tau, B.beta};
            if (fas) {
                t_residual(B, B.u0, B.rhs, 1, rc ? t_area(B, B.u0, A.mp, A1frac, S.red) : T(0));
                fas = false;
            }
            int it;
            double res;
            coarse_solve_block<T, C>(cg, A.mp, A1frac, B.h2nm, A.coarse_maxit, A.coarse_tol,
                                     reinterpret_cast<C *>(smem_tail + s_scratch), S.red, &S.s_err, &it, &res,
                                     A.coarse_aos, A.aos_dt);
            if (threadIdx.x == 0) {
                A.sc->picard = it;
                A.sc->coarse_res = res;
                if (S.s_err) A.sc->err = 1;
            }
            __syncthreads();
            down = false;
            --l;
            t = -1;
        } else if (t < 0) {
            t_interp(B, Bs[l + 1]);
            t = 0;
        } else if (t < (down ? A.nu1 : A.nu2)) {
            const T ar = rc ? t_area(B, B.u, A.mp, A1frac, S.red) : T(0);
            if (fas) {   // the first snapshot after the restriction: u = u0, so the area term is the same
                t_residual(B, B.u0, B.rhs, 1, ar);
                fas = false;
            }
            t_snapshot(B, ar, S);
            t_sweeps(B, S);
            ++t;
        } else if (down) {
            t_residual(B, B.u, B.f, 0, rc ? t_area(B, B.u, A.mp, A1frac, S.red) : T(0));
            t_restrict(B, Bs[l + 1]);
            fas = true;
            ++l;
            t = 0;
        } else {
            --l;
            t = -1;
        }
    }
    // what the per-grid kernels leave on these grids: u, the right-hand side, the last snapshot's G
    for (int k = first; k <= last; ++k) {
        const LevelView<T> &G = A.g[k];
        const TGrid<T> &B = Bs[k];
        TAIL_CELLS(B.n, B.m, i, j) {
            const size_t o = (size_t)i * G.pitch + j, lim = (size_t)G.n * G.pitch;
            const int q = i * B.P + j;
            stc(G.u, o, lim, kDbgBottom, sm<T>()[B.u + q]);
            stc(G.rhs, o, lim, kDbgBottom, sm<T>()[B.rhs + q]);
            if (k < last) stc(G.G, o, lim, kDbgBottom, sm<T>()[B.G + q]);
        }
    }
}

template <typename T, typename C>
void set_tail_attr() {
    cudaFuncSetAttribute(k_tail<T, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTailSmemMax);
}

}  // namespace

void prepare_tail_kernel() {
    set_tail_attr<float, float>();
    set_tail_attr<float, double>();
    set_tail_attr<double, double>();
}

// Shared memory of grids first .. L-1, or 0 where the block does not take them.
template <typename T>
size_t tail_smem_bytes(const int *n, const int *m, int first, int L, int coarse_fp64) {
    if (first < 1 || first > L - 2 || n[first] > 32 || m[first] > 32 || n[L - 1] * m[L - 1] > kWarpCoarseMax) return 0;
    if (sizeof(T) == 8 && n[first] * m[first] > kNT) return 0;
    size_t b = 0;
    for (int l = first; l < L; ++l) b += 8 * sizeof(T) * (size_t)n[l] * tail_pitch(m[l]);
    b = (b + 15) / 16 * 16;
    b += (coarse_fp64 || sizeof(T) == 8 ? sizeof(double) : sizeof(float)) * coarse_scratch_elems(n[L - 1], m[L - 1]);
    return b <= kTailSmemMax ? b : 0;
}

template <typename T>
void launch_tail(const TailArgs<T> &A, int coarse_fp64, size_t smem, cudaStream_t st) {
    if constexpr (sizeof(T) == 4) {
        if (!coarse_fp64) {
            launch_pdl(k_tail<T, float>, dim3(1), dim3(kNT), smem, st, A);
            return;
        }
    }
    launch_pdl(k_tail<T, double>, dim3(1), dim3(kNT), smem, st, A);
}

#define INST(T)                                                                           \
    template size_t tail_smem_bytes<T>(const int *, const int *, int, int, int);         \
    template void launch_tail<T>(const TailArgs<T> &, int, size_t, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace segmg
