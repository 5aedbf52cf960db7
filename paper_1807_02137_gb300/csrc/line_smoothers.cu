// line_smoothers.cu -- the paper's other two smoothers on the GPU: GSLINE-I (Sec. 3.2, the
// smoother of Algorithm 1) and Hybrid Smoother 1 (Sec. 4.2, Algorithm 2), in parallel orderings.
//
// GSLINE-I: every column is one tridiagonal system (eq. system) coupling the column's cells
// through A and B, with C and D terms from the current values.  The columns of one parity are
// not neighbours, so all even columns are solved at once, then all odd ones (zebra), each by the
// Thomas algorithm down and up its rows, with the eliminated diagonal (its reciprocal in FP32) and
// right-hand side kept in two scratch grids.
//
// Hybrid Smoother 1: after GSLINE-I, every cell P of the set D (from the coefficient snapshot:
// class byte = 1 << index of the smallest coefficient) and its neighbours other than the lagged
// one solve their own equations exactly (the arrow systems of eqs. caseAlagged - caseDlagged).
// Cells are visited in 16 classes (i mod 4, j mod 4): two blocks of one class are 4 or more
// cells apart, so neither reads what the other writes, and one launch does one class.
//
// Rows are in the row-scaled form of the solver (divided by delta): the coefficient of
// neighbour X in the row of a cell is mu/h^2 times the face value of G, S is their sum plus
// 1/tau and f is the snapshot's right-hand side.  A face on the domain boundary is zero.
#include "arith.cuh"

namespace segmg {

namespace {

// ---------------------------------------------------------------------------------------
// GSLINE-I, one parity of columns: a block solves 32 of them.
//
// A column's elimination and substitution are serial recurrences, and a grid has few columns (512
// of a parity at 1024^2): the recurrence's chain sets the time, about 45 cycles a row down (a
// reciprocal, a product, a multiply-add) and 12 up, if nothing else stands in it.  So one warp
// runs the 32 recurrences from values in shared memory, and the block's other warps form those
// values (faces, products, right-hand sides) and store the results, a chunk of kGR rows ahead and
// behind.  (One thread a column that also loaded and formed its values took about 250 cycles a row
// each way: 4.2 ms a V-cycle at 1024^2.)  A forming warp takes neighbouring rows with all their loads
// in flight: 1024^2 step 40.4 -> 39.7 ms against one row at a time; the chain is what is left.
// dg / rg: scratch for what the eliminated rows leave (the reciprocal of the diagonal, or in FP64 the
// diagonal, and the right-hand side), row by row at the columns' own order (pitched like the grid).
// ---------------------------------------------------------------------------------------
constexpr int kGF = 8, kGW = 1 + kGF;   // warps that form values; with the solving one

template <typename T>
__global__ void __launch_bounds__(32 * kGW) k_gsline(LevelView<T> L, int parity, T *__restrict__ dg, T *__restrict__ rg) {
    constexpr int kGR = 128 / sizeof(T);   // rows of a chunk (32 KB of values in two chunks)
    constexpr int kFR = kGR / kGF;         // neighbouring rows of a chunk that a forming warp takes
    // down: lo, up, diagonal, right-hand side; up: up, reciprocal, right-hand side
    __shared__ T val[2][4][kGR][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n = L.n, m = L.m, p = L.pitch;
    const int c = blockIdx.x * 32 + lane, j = parity + 2 * c;   // this lane's column
    const bool on = j < m;
    const int jc = on ? j : parity;                             // a lane past the last column reads the first
    const bool hE = jc + 1 < m, hW = jc > 0;
    const int chunks = (n + kGR - 1) / kGR;
    const size_t lim = (size_t)n * p;
    // the coefficients and the right-hand side of rows i0 .. i0 + kGR - 1 into val[b]
    // (every load of a warp's rows is issued before the first is used; a row past the last is the last)
    auto form = [&](int k, int b) {
        const int r0 = (warp - 1) * kFR, i0 = k * kGR + r0;
        if (i0 >= n) return;
        T g[kFR + 2], gE[kFR], gW[kFR], uE[kFR], uW[kFR], f[kFR];
        const size_t eE = hE ? 1 : 0, eW = hW ? 1 : 0;
        g[0] = __ldg(L.G + (size_t)max(i0 - 1, 0) * p + jc);
        g[kFR + 1] = __ldg(L.G + (size_t)min(i0 + kFR, n - 1) * p + jc);
#pragma unroll
        for (int r = 0; r < kFR; ++r) {
            const size_t o = (size_t)min(i0 + r, n - 1) * p + jc;
            g[r + 1] = __ldg(L.G + o);
            gE[r] = __ldg(L.G + o + eE);
            gW[r] = __ldg(L.G + o - eW);
            uE[r] = __ldg(L.u + o + eE);
            uW[r] = __ldg(L.u + o - eW);
            f[r] = __ldg(L.f + o);
        }
#pragma unroll
        for (int r = 0; r < kFR; ++r) {
            const bool hS = i0 + r + 1 < n, hN = i0 + r > 0;
            const T aS = face(g[r + 1], g[r + 2], hS), aN = face(g[r + 1], g[r], hN);
            const T aE = face(g[r + 1], gE[r], hE), aW = face(g[r + 1], gW[r], hW);
            const T sum = add_rn(add_rn(aN, aS), add_rn(aE, aW));
            const T across = fma_rn(aW, uW[r], mul_rn(aE, uE[r]));
            val[b][0][r0 + r][lane] = mul_rn(L.cdiff, aN);
            val[b][1][r0 + r][lane] = mul_rn(L.cdiff, aS);
            val[b][2][r0 + r][lane] = -fma_rn(L.cdiff, sum, L.inv_tau);
            val[b][3][r0 + r][lane] = fma_rn(-L.cdiff, across, f[r]);
        }
    };
    // ---- elimination, downwards
    if (warp > 0) form(0, 0);
    __syncthreads();
    T up_prev = T(0), rec_prev = T(0), rhs_prev = T(0);
    for (int k = 0; k < chunks; ++k) {
        const int b = k & 1, rows = min(kGR, n - k * kGR);
        if (warp > 0) {
            if (k + 1 < chunks) form(k + 1, b ^ 1);
        } else {
            for (int r0 = 0; r0 < rows; r0 += 8) {
                T lo[8], up[8], di[8], rh[8];
#pragma unroll
                for (int r = 0; r < 8; ++r) {   // (rows past the grid's last are read and not used)
                    lo[r] = val[b][0][r0 + r][lane]; up[r] = val[b][1][r0 + r][lane];
                    di[r] = val[b][2][r0 + r][lane]; rh[r] = val[b][3][r0 + r][lane];
                }
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    if (r0 + r >= rows) break;
                    if (k > 0 || r0 + r > 0) {
                        const T wgt = div_by(lo[r], rec_prev);
                        di[r] = fma_rn(-wgt, up_prev, di[r]);
                        rh[r] = fma_rn(-wgt, rhs_prev, rh[r]);
                    }
                    up_prev = up[r];
                    rec_prev = recip_relax(di[r]);
                    rhs_prev = rh[r];
                    if (on) {
                        const size_t o = (size_t)(k * kGR + r0 + r) * p + c;
                        stc(dg, o, lim, kDbgOther, rec_prev);
                        stc(rg, o, lim, kDbgOther, rhs_prev);
                    }
                }
            }
        }
        __syncthreads();
    }
    // ---- substitution, upwards: chunk k from its last row
    auto fetch = [&](int k, int b) {
        const int r0 = (warp - 1) * kFR, i0 = k * kGR + r0;
        if (i0 >= n) return;
        T g[kFR + 1], rec[kFR], rh[kFR];
        g[kFR] = __ldg(L.G + (size_t)min(i0 + kFR, n - 1) * p + jc);
#pragma unroll
        for (int r = 0; r < kFR; ++r) {
            const size_t row = (size_t)min(i0 + r, n - 1) * p, q = row + (on ? c : 0);
            g[r] = __ldg(L.G + row + jc);
            rec[r] = dg[q];
            rh[r] = rg[q];
        }
#pragma unroll
        for (int r = 0; r < kFR; ++r) {
            val[b][0][r0 + r][lane] = i0 + r + 1 < n ? mul_rn(L.cdiff, face(g[r], g[r + 1], true)) : T(0);
            val[b][1][r0 + r][lane] = rec[r];
            val[b][2][r0 + r][lane] = rh[r];
        }
    };
    if (warp > 0) fetch(chunks - 1, (chunks - 1) & 1);
    __syncthreads();
    T x = T(0);
    for (int k = chunks - 1; k >= 0; --k) {
        const int b = k & 1, rows = min(kGR, n - k * kGR);
        if (warp > 0) {
            if (k > 0) fetch(k - 1, b ^ 1);
        } else {
            for (int r1 = rows - 1; r1 >= 0; r1 -= 8) {
                T up[8], rec[8], rh[8];
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const int q = max(r1 - r, 0);
                    up[r] = val[b][0][q][lane]; rec[r] = val[b][1][q][lane]; rh[r] = val[b][2][q][lane];
                }
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    if (r1 - r < 0) break;
                    const int i = k * kGR + r1 - r;
                    x = i == n - 1 ? div_by(rh[r], rec[r]) : div_by(fma_rn(-up[r], x, rh[r]), rec[r]);
                    if (on) stc(L.u, (size_t)i * p + j, lim, kDbgOther, x);
                }
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------------------
// Hybrid Smoother 1 blocks of one class (ci, cj): cells i = ci + 4I, j = cj + 4J.
// ---------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) k_hs1(LevelView<T> L, int ci, int cj) {
    const int i = ci + 4 * (blockIdx.y * blockDim.y + threadIdx.y);
    const int j = cj + 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    const int n = L.n, m = L.m, p = L.pitch;
    if (i >= n || j >= m) return;
    const size_t o = (size_t)i * p + j;
    const unsigned cls = L.cls[o];
    if (!cls) return;
    const int lag = __ffs(cls) - 1;                 // 0..3 = A (south), B (north), C (east), D (west)
    const int di[4] = {1, -1, 0, 0}, dj[4] = {0, 0, 1, -1};
    auto inside = [&](int a, int b) { return a >= 0 && a < n && b >= 0 && b < m; };
    // row coefficients of a cell: c[t] = mu/h^2 G_face toward neighbour t (0 if none), S
    auto row = [&](int a, int b, T *c, T &S) {
        const size_t q = (size_t)a * p + b;
        const T gc = L.G[q];
        T s = T(0);
        for (int t = 0; t < 4; ++t) {
            const int a2 = a + di[t], b2 = b + dj[t];
            c[t] = inside(a2, b2) ? L.cdiff * face(gc, L.G[(size_t)a2 * p + b2], true) : T(0);
            s += c[t];
        }
        S = s + L.inv_tau;
    };
    T cP[4], SP;
    row(i, j, cP, SP);
    // P's row: -S_P x_P + sum over leaves c_Pl x_l = f_P - c_P,lag u_lag
    T rP = L.f[o];
    {
        const int a2 = i + di[lag], b2 = j + dj[lag];
        rP -= cP[lag] * L.u[(size_t)a2 * p + b2];
    }
    T num = T(0), den = -SP;
    T rl[4], cl[4], Sl[4];
    bool leaf[4];
    for (int t = 0; t < 4; ++t) {
        const int a = i + di[t], b = j + dj[t];
        leaf[t] = t != lag && inside(a, b);
        if (!leaf[t]) continue;
        T c[4], S;
        row(a, b, c, S);
        const int back = t ^ 1;                     // the direction from the leaf back to P
        T r = L.f[(size_t)a * p + b];
        for (int u = 0; u < 4; ++u) {
            if (u == back || c[u] == T(0)) continue;
            r -= c[u] * L.u[(size_t)(a + di[u]) * p + (b + dj[u])];
        }
        rl[t] = r;
        cl[t] = c[back];
        Sl[t] = S;
        num += cP[t] * r / S;
        den += cP[t] * c[back] / S;
    }
    const T xP = (rP + num) / den;
    stc(L.u, o, (size_t)n * p, kDbgOther, xP);
    for (int t = 0; t < 4; ++t) {
        if (!leaf[t]) continue;
        stc(L.u, (size_t)(i + di[t]) * p + (j + dj[t]), (size_t)n * p, kDbgOther, (cl[t] * xP - rl[t]) / Sl[t]);
    }
}

}  // namespace

template <typename T>
void launch_gsline(const LevelView<T> &L, cudaStream_t st) {
    for (int par = 0; par < 2; ++par) {
        const int cols = (L.m - par + 1) / 2;
        if (cols <= 0) continue;
        k_gsline<T><<<(cols + 31) / 32, 32 * kGW, 0, st>>>(L, par, L.r, L.t);
    }
}

template <typename T>
void launch_hs1_blocks(const LevelView<T> &L, cudaStream_t st) {
    for (int c = 0; c < 16; ++c) {
        const int ci = c / 4, cj = c % 4;
        const int ni = (L.n - ci + 3) / 4, nj = (L.m - cj + 3) / 4;
        if (ni <= 0 || nj <= 0) continue;
        dim3 block(32, 8), grid((nj + 31) / 32, (ni + 7) / 8);
        k_hs1<T><<<grid, block, 0, st>>>(L, ci, cj);
    }
}

template void launch_gsline<float>(const LevelView<float> &, cudaStream_t);
template void launch_gsline<double>(const LevelView<double> &, cudaStream_t);
template void launch_hs1_blocks<float>(const LevelView<float> &, cudaStream_t);
template void launch_hs1_blocks<double>(const LevelView<double> &, cudaStream_t);

}  // namespace segmg
