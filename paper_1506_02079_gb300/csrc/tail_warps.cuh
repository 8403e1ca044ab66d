// Coarse tail with the cells in registers (FP32).
//
// The levels of one slice from kc (the first with both sides <= kTailMax = 64) down to 1 x 1 are run
// by one CTA.  Only level kc touches global memory: its right-hand side (and, continuing at level 0,
// its iterate) is read at the start and its final iterate written at the end, where the UP leg of
// level kc - 1 (or the residual kernel, at kc = 0) reads it.  The per-cell arithmetic and its order
// are those of every other schedule.
//
// Bound by the latency of about 70 dependent passes (half-sweeps, restrictions, prolongations)
// over few cells, so each pass is kept short, with the cells in registers:
//   levels of 33 .. 64 cells a side: 16 warps of 4 rows, a lane holds columns 2 lane, 2 lane + 1;
//   17 .. 32: 16 warps of 2 rows, a lane holds one column: exactly the coarse cells of what the
//            same lane holds of the finer level, so the restriction stays in the lane;
//   9 .. 16: one warp, 2 lanes a column of 8 rows each; <= 8: one warp, 4 lanes of 2 rows each;
//            neighbours by shuffles alone, no barriers.
// Warps exchange edge rows through shared memory, double buffered, one barrier per half-sweep.
// Cells outside the level are kept at exactly 0 (their 1 / D is 0), a missing neighbour adds
// nothing, and a cell's stencil depends on its column only, except on the first and last row
// (another diagonal) and on rows of partial cells (the level's table).
// 16 slices of 64 x 64, 2 + 2 sweeps: 23 us per launch, 60 x 60 25, 16 x 16 17; passes
// over cells in shared memory (tail_cells.cuh) take 33, 33 and 19, with stencils formed in every pass
// they took 137.  Both blocks' state at once (the 64- and 32-levels') is a few registers more than the 128 of
// 512 threads: 88 bytes a thread spill, written and read between the legs.  FP64 keeps those: one warp's FP64 instructions take 16 cycles each, so few warps
// with every second lane idle are slower there (170 against 80 us).
#pragma once
#include <cuda_runtime.h>

#include "fused_impl.cuh"

namespace emfuse {
namespace fused_detail {

constexpr int kTailWarps = 16;
static_assert(kTailThreads == 32 * kTailWarps, "one warp per group of rows");
constexpr int kTailSides = 128;    // sum of a side over the levels, at most 64 + 32 + .. + 1

// What a half-sweep needs of a column.
template <class T>
struct ColCoefs {
    T cw, ce, cy;
};

// The tables of the tail's levels, one level after another.
template <class T>
struct TailTables {
    TailCoef<T> coef[kTailMaxLevels][16];  // [class of y][class of x]
    ColStencil<T> col[kTailSides];
    AxisCoef<T> ax[kTailSides], ay[kTailSides];
    T wx[kTailSides], wy[kTailSides];      // interpolation weights toward the other coarse cell
    unsigned char mode[kTailSides];        // row modes
};

// One level as its passes see it.
template <class T>
struct TailLevel {
    const TailCoef<T>* coef;
    const ColStencil<T>* col;
    const AxisCoef<T> *ax, *ay;
    const T *wx, *wy;
    const unsigned char* mode;
    T sk;
    int nx, ny;
};

// Gauss-Seidel update of a cell of a row of full cells, from its column's stencil (id = 1 / D).
template <class T>
__device__ __forceinline__ T tail_update(const ColCoefs<T>& q, T id, T b, T w, T e, T n, T s) {
    Coef<T> c;
    c.cw = q.cw; c.ce = q.ce; c.cn = c.cs = q.cy; c.iD = id;
    return gs_update<T>(c, b, w, e, n, s);
}
// The faces of any cell from the axis coefficients of its column and row (make_coef's products; the
// level-0 ones are plain factors, and sk is 1 there).
template <class T>
__device__ __forceinline__ Coef<T> tail_faces(const AxisCoef<T>& ax, const AxisCoef<T>& ay, T sk) {
    Coef<T> c;
    c.cw = sk * (ay.w * ax.gm);
    c.ce = sk * (ay.w * ax.gp);
    c.cn = sk * (ax.w * ay.gm);
    c.cs = sk * (ax.w * ay.gp);
    return c;
}
// 1 / D of a cell of column x (stencil q) on a row of full cells of mode m; 0 outside the level: such
// a cell stays 0.
template <class T>
__device__ __forceinline__ T tail_id(const ColStencil<T>& q, unsigned m) {
    return m == kRowInner ? q.iD : (m == kRowEdge ? q.iDb : T(0));
}
// The stencil of a cell in the level from the level's table (any row).
template <class T>
__device__ __forceinline__ const TailCoef<T>& tail_entry(const TailLevel<T>& L, int x, int y) {
    return L.coef[4 * tail_class(y, L.ny) + tail_class(x, L.nx)];
}
// Residual of a cell (0 outside the level): FULL rows from the column's stencil, else from the table.
template <class T, bool FULL>
__device__ __forceinline__ T tail_residual(const TailLevel<T>& L, const ColCoefs<T>& q, int x, int y, T u, T b, T w, T e, T n,
                                           T s) {
    if (x >= L.nx || y >= L.ny) return T(0);
    Coef<T> c;
    if (FULL) {
        c.cw = q.cw; c.ce = q.ce; c.cn = c.cs = q.cy;
        c.D = L.mode[y] == kRowInner ? L.col[x].D : L.col[x].Db;
    } else {
        c = tail_coef<T>(&tail_entry<T>(L, x, y));
    }
    return residual_at<T>(c, b, u, w, e, n, s);
}
// Interpolated coarse correction at (x, y) from coarse values `c` with row pitch `p` (see k_wave for
// which coarse cell is the other one; a weight of 0 marks that there is none).
template <class T>
__device__ __forceinline__ T tail_interp(const TailLevel<T>& L, const T* c, int p, int x, int y) {
    const T wx = L.wx[x], wy = L.wy[y];
    const int I = x >> 1, J = wx == T(0) ? I : ((x & 1) ? I + 1 : I - 1);
    const int Y = y >> 1, Z = wy == T(0) ? Y : ((y & 1) ? Y + 1 : Y - 1);
    const T *r0 = c + Y * p, *r1 = c + Z * p;
    return bilinear<T>(r0[I], r0[J], r1[I], r1[J], wx, wy);
}

// The block's part of a level: R rows of C columns per lane (R = 4, C = 2 or R = 2, C = 1).
template <class T, int R, int C>
struct TailBlock {
    TailLevel<T> L;
    T u[R][C], b[R][C], id[R][C];
    ColCoefs<T> col[C];
    bool partial;  // the warp holds a row of partial cells
    int x, y;      // first cell

    __device__ __forceinline__ void init(const TailLevel<T>& lev, int lane, int warp) {
        L = lev;
        x = C * lane;
        y = R * warp;
        partial = false;
#pragma unroll
        for (int r = 0; r < R; ++r) partial |= y + r < L.ny && L.mode[y + r] == kRowPartial;
#pragma unroll
        for (int i = 0; i < C; ++i) {
            col[i] = ColCoefs<T>{T(0), T(0), T(0)};
            ColStencil<T> q{T(0), T(0), T(0), T(0), T(0), T(0), T(0)};
            if (x + i < L.nx) q = L.col[x + i];
            col[i] = ColCoefs<T>{q.cw, q.ce, q.cy};
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const unsigned m = y + r < L.ny ? L.mode[y + r] : kRowOut;
                id[r][i] = tail_id<T>(q, m);
                if (partial && m == kRowPartial && x + i < L.nx) id[r][i] = tail_entry<T>(L, x + i, y + r).iD;
            }
        }
    }
    __device__ __forceinline__ AxisCoef<T> column(int i) const {
        return x + i < L.nx ? L.ax[x + i] : AxisCoef<T>{T(0), T(0), T(0)};
    }
    __device__ __forceinline__ AxisCoef<T> row(int r) const {
        return y + r < L.ny ? L.ay[y + r] : AxisCoef<T>{T(0), T(0), T(0)};
    }
    // The rows above and below the warp's (edge: [2][kTailWarps][2][64], buf alternates).
    __device__ __forceinline__ void exchange(T* edge, int& buf, int lane, int warp, T (&no)[C], T (&so)[C]) {
        T* e = edge + buf * (kTailWarps * 2 * 64);
#pragma unroll
        for (int i = 0; i < C; ++i) {
            e[(warp * 2) * 64 + C * lane + i] = u[0][i];
            e[(warp * 2 + 1) * 64 + C * lane + i] = u[R - 1][i];
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < C; ++i) {
            no[i] = warp > 0 ? e[(warp * 2 - 1) * 64 + C * lane + i] : T(0);
            so[i] = warp + 1 < kTailWarps ? e[(warp * 2 + 2) * 64 + C * lane + i] : T(0);
        }
        buf ^= 1;
    }
    __device__ __forceinline__ void relax(T* edge, int& buf, int lane, int warp, int sweeps) {
#pragma unroll 1
        for (int h = 0; h < 2 * sweeps; h += 2) {
            half_sweep<0>(edge, buf, lane, warp);
            half_sweep<1>(edge, buf, lane, warp);
        }
    }
    // (all rows from the old values: a half-sweep only reads the other colour)
    template <int COLOUR>
    __device__ __forceinline__ void half_sweep(T* edge, int& buf, int lane, int warp) {
        T no[C], so[C];
        exchange(edge, buf, lane, warp, no, so);
        if (partial) rows<COLOUR, true>(lane, no, so);
        else rows<COLOUR, false>(lane, no, so);
    }
    template <int COLOUR, bool PARTIAL>
    __device__ __forceinline__ void rows(int lane, const T (&no)[C], const T (&so)[C]) {
        T v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            // C = 2: cell i of the lane has the colour (y is even); C = 1: every second lane's cell
            const int i = C == 2 ? (r + COLOUR) & 1 : 0;
            T w, e;
            if (C == 2) {
                const T o = i == 0 ? __shfl_up_sync(0xffffffffu, u[r][C - 1], 1) : __shfl_down_sync(0xffffffffu, u[r][0], 1);
                w = i == 0 ? o : u[r][0];
                e = i == 0 ? u[r][C - 1] : o;
            } else {
                w = __shfl_up_sync(0xffffffffu, u[r][0], 1);
                e = __shfl_down_sync(0xffffffffu, u[r][0], 1);
            }
            const T n = r > 0 ? u[r > 0 ? r - 1 : 0][i % C] : no[i % C];
            const T s = r + 1 < R ? u[r + 1 < R ? r + 1 : 0][i % C] : so[i % C];
            if (PARTIAL) {
                Coef<T> c = tail_faces<T>(column(i % C), row(r), L.sk);
                c.iD = id[r][i % C];
                v[r] = gs_update<T>(c, b[r][i % C], w, e, n, s);
            } else {
                v[r] = tail_update<T>(col[i % C], id[r][i % C], b[r][i % C], w, e, n, s);
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (C == 2) u[r][((r + COLOUR) & 1) % C] = v[r];
            else if (((lane + r + COLOUR) & 1) == 0) u[r][0] = v[r];
        }
    }
    __device__ __forceinline__ void residual(T* edge, int& buf, int lane, int warp, T (&res)[R][C]) {
        T no[C], so[C];
        exchange(edge, buf, lane, warp, no, so);
        if (partial) residual_rows<false>(no, so, res);
        else residual_rows<true>(no, so, res);
    }
    template <bool FULL>
    __device__ __forceinline__ void residual_rows(const T (&no)[C], const T (&so)[C], T (&res)[R][C]) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const T wo = __shfl_up_sync(0xffffffffu, u[r][C - 1], 1), eo = __shfl_down_sync(0xffffffffu, u[r][0], 1);
#pragma unroll
            for (int i = 0; i < C; ++i) {
                const T w = i == 0 ? wo : u[r][0], e = i == C - 1 ? eo : u[r][C - 1];
                const T n = r > 0 ? u[r > 0 ? r - 1 : 0][i] : no[i], s = r + 1 < R ? u[r + 1 < R ? r + 1 : 0][i] : so[i];
                res[r][i] = tail_residual<T, FULL>(L, col[i], x + i, y + r, u[r][i], b[r][i], w, e, n, s);
            }
        }
    }
    __device__ __forceinline__ void prolong(const T* c, int p) {
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int i = 0; i < C; ++i)
                if (x + i < L.nx && y + r < L.ny) u[r][i] += tail_interp<T>(L, c, p, x + i, y + r);
    }
};

// The CTA's shared memory.
template <class T>
struct alignas(16) TailShared {
    TailTables<T> tab;
    int off[2][kTailMaxLevels];        // where a level's columns and rows start in the tables
    int size[2][kTailMaxLevels];       // its sides
    T sk[kTailMaxLevels];              // 4^-k
    T edge[2 * kTailWarps * 2 * 64];
    T uc[32 * 32];                     // iterate of the 32-level for the prolongation
    T us[5][16 * 16], bs[5][16 * 16];  // levels of at most 16 x 16
};

// Level q of the tail.
template <class T>
__device__ __forceinline__ TailLevel<T> tail_view(TailShared<T>& sh, int q) {
    TailLevel<T> L;
    const int ox = sh.off[0][q], oy = sh.off[1][q];
    L.coef = sh.tab.coef[q];
    L.col = sh.tab.col + ox;
    L.ax = sh.tab.ax + ox;
    L.ay = sh.tab.ay + oy;
    L.wx = sh.tab.wx + ox;
    L.wy = sh.tab.wy + oy;
    L.mode = sh.tab.mode + oy;
    L.nx = sh.size[0][q];
    L.ny = sh.size[1][q];
    L.sk = sh.sk[q];
    return L;
}

// One warp's level: 2^LC columns, 32 / 2^LC lanes per column with R rows each (LC = 4, R = 8 or
// LC = 3, R = 2); u and b are dense arrays of row pitch 16 in shared memory.
template <class T, int LC, int R>
struct TailWarp {
    // All rows of a half-sweep are formed from its old values before any is written (it only reads
    // the other colour), so they do not wait for one another.
    template <bool PARTIAL>
    static __device__ __forceinline__ void relax(const TailLevel<T>& L, const ColCoefs<T>& col, const AxisCoef<T>& ax,
                                                 T (&u)[R], const T (&b)[R], const T (&id)[R], int x, int y,
                                                 int half_sweeps) {
        const int lane = threadIdx.x & 31;
        constexpr int W = 1 << LC;
#pragma unroll 1
        for (int h = 0; h < half_sweeps; ++h) {
            const T no = __shfl_up_sync(0xffffffffu, u[R - 1], W), so = __shfl_down_sync(0xffffffffu, u[0], W);
            T v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const T w = __shfl_up_sync(0xffffffffu, u[r], 1), e = __shfl_down_sync(0xffffffffu, u[r], 1);
                const T n = r > 0 ? u[r > 0 ? r - 1 : 0] : (lane < W ? T(0) : no);
                const T s = r + 1 < R ? u[r + 1 < R ? r + 1 : 0] : (lane >= 32 - W ? T(0) : so);
                if (PARTIAL) {
                    Coef<T> c = tail_faces<T>(ax, y + r < L.ny ? L.ay[y + r] : AxisCoef<T>{T(0), T(0), T(0)}, L.sk);
                    c.iD = id[r];
                    v[r] = gs_update<T>(c, b[r], w, e, n, s);
                } else {
                    v[r] = tail_update<T>(col, id[r], b[r], w, e, n, s);
                }
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (((x + y + r + h) & 1) == 0) u[r] = v[r];
        }
    }
    // DOWN: relax from zero (or us), keep u, restrict into cb (null on the last level).  UP: add the
    // correction interpolated from cu, relax.  q: the tail's level, i: its arrays.  Out of line, one
    // function per form, so that a launch fetches only the forms it runs.
    template <bool PARTIAL>
    static __device__ __noinline__ void leg(int q, int i, int next, bool down, bool from_us, int sweeps) {
        extern __shared__ __align__(16) unsigned char tail_smem[];
        TailShared<T>& sh = *reinterpret_cast<TailShared<T>*>(tail_smem);
        const TailLevel<T> L = tail_view<T>(sh, q);
        T* const us = sh.us[i];
        const T* const bs = sh.bs[i];
        T* const cb = down && next != i ? sh.bs[next] : nullptr;
        const T* const cu = down ? nullptr : sh.us[next];
        const int lane = threadIdx.x & 31;
        constexpr int W = 1 << LC;
        const int x = lane & (W - 1), y = (lane >> LC) * R;
        ColCoefs<T> col{T(0), T(0), T(0)};
        AxisCoef<T> ax{T(0), T(0), T(0)};
        ColStencil<T> cs{T(0), T(0), T(0), T(0), T(0), T(0), T(0)};
        if (x < L.nx) {
            cs = L.col[x];
            if (PARTIAL) ax = L.ax[x];
        }
        col = ColCoefs<T>{cs.cw, cs.ce, cs.cy};
        T u[R], b[R], id[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const bool in = x < L.nx && y + r < L.ny;
            const unsigned m = y + r < L.ny ? L.mode[y + r] : kRowOut;
            id[r] = tail_id<T>(cs, m);
            if (PARTIAL && m == kRowPartial && x < L.nx) id[r] = tail_entry<T>(L, x, y + r).iD;
            b[r] = in ? bs[(y + r) * 16 + x] : T(0);
            u[r] = in && from_us ? us[(y + r) * 16 + x] : T(0);
            if (cu && in) u[r] += tail_interp<T>(L, cu, 16, x, y + r);
        }
        // a 1 x 1 level has no neighbours: one half-sweep is the solution, the others repeat it
        const int half_sweeps = L.nx * L.ny == 1 ? 1 : 2 * sweeps;
        relax<PARTIAL>(L, col, ax, u, b, id, x, y, half_sweeps);
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (x < L.nx && y + r < L.ny) us[(y + r) * 16 + x] = u[r];
        if (cb) {
            const T no = __shfl_up_sync(0xffffffffu, u[R - 1], W), so = __shfl_down_sync(0xffffffffu, u[0], W);
            T res[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const T w = __shfl_up_sync(0xffffffffu, u[r], 1), e = __shfl_down_sync(0xffffffffu, u[r], 1);
                const T n = r > 0 ? u[r > 0 ? r - 1 : 0] : (lane < W ? T(0) : no);
                const T s = r + 1 < R ? u[r + 1 < R ? r + 1 : 0] : (lane >= 32 - W ? T(0) : so);
                res[r] = tail_residual<T, !PARTIAL>(L, col, x, y + r, u[r], b[r], w, e, n, s);
            }
#pragma unroll
            for (int r = 0; r < R; r += 2) {
                const T e0 = __shfl_down_sync(0xffffffffu, res[r], 1), e1 = __shfl_down_sync(0xffffffffu, res[r + 1], 1);
                const T c = ((res[r] + e0) + res[r + 1]) + e1;
                if ((x & 1) == 0 && x < L.nx && y + r < L.ny) cb[((y + r) >> 1) * 16 + (x >> 1)] = c * T(0.25);
            }
        }
        __syncwarp();
    }
};

template <class T>
__global__ void __launch_bounds__(kTailThreads) k_tail(TailArgs<T> a) {
    extern __shared__ __align__(16) unsigned char tail_smem[];
    TailShared<T>& sh = *reinterpret_cast<TailShared<T>*>(tail_smem);
    TailTables<T>& tab = sh.tab;
    T* const edge = sh.edge;
    T* const uc = sh.uc;
    auto& us = sh.us;
    auto& bs = sh.bs;
    const int j = blockIdx.x;
    if (a.active && !a.active[j]) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int kc = a.kc[j];
    const LSlice<T>* lv = a.table + a.level_off[j];
    const int nl = a.nlev[j] - kc;  // levels of the tail
    if (nl > kTailMaxLevels || nl < 1) return;  // never: a 64 x 64 level has 6 levels below it
    const LSlice<T> G = lv[kc];
    const int n0x = G.n0x, n0y = G.n0y;
    auto scale = [&](int q) { return T(1) / T(1ll << (2 * (kc + q))); };  // 4^-k, exact: kc + q < 31
    if (tid >= kTailThreads - 2) {
        const int ax = kTailThreads - 1 - tid;
        int o = 0;
        for (int q = 0; q < nl; ++q) {
            const int n = level_size(ax == 0 ? n0x : n0y, kc + q);
            sh.off[ax][q] = o;
            sh.size[ax][q] = n;
            if (ax == 0) sh.sk[q] = scale(q);
            o += n;
        }
    }
    for (int t = tid; t < kTailSides * 2 + nl * 16; t += kTailThreads) {
        if (t < 2 * kTailSides) {
            const bool ax = t < kTailSides;  // columns, then rows
            const int n0 = ax ? n0x : n0y;
            int i = ax ? t : t - kTailSides, q = 0;
            const int at = i;
            while (q < nl && i >= level_size(n0, kc + q)) i -= level_size(n0, kc + q++);
            if (q < nl) {
                const int k = kc + q, n = level_size(n0, k);
                T w = T(0);
                if (q + 1 < nl) {
                    int I, J;
                    interp_axis<T>(i, n0, k, level_size(n0, k + 1), I, J, w);
                }
                (ax ? tab.ax : tab.ay)[at] = axis_coef<T>(i, n, n0, k);
                if (ax) {
                    tab.col[at] = col_stencil<T>(i, n, n0, k, a.alpha, scale(q));
                    tab.wx[at] = w;
                } else {
                    tab.mode[at] = row_mode<T>(i, n, n0, k);
                    tab.wy[at] = w;
                }
            }
        } else {
            const int p = t - 2 * kTailSides, q = p >> 4, k = kc + q, nx = level_size(n0x, k), ny = level_size(n0y, k);
            const Coef<T> c = coef_at<T>(tail_class_rep(p & 3, nx), tail_class_rep((p >> 2) & 3, ny), nx, ny, n0x, n0y, k,
                                         a.alpha, scale(q));
            TailCoef<T>& o = tab.coef[q][p & 15];
            o.cw = c.cw; o.ce = c.ce; o.cn = c.cn; o.cs = c.cs; o.iD = c.iD; o.D = c.D;
        }
    }
    const bool cont = a.cont && kc == 0;
    const int side = max(G.nx, G.ny);
    const bool hasA = side > 32, hasB = nl > (hasA ? 1 : 0) && (hasA || side > 16);
    const int qB = hasA ? 1 : 0, qC = qB + (hasB ? 1 : 0);  // levels of the second and third stage
    TailBlock<T, 4, 2> A;
    TailBlock<T, 2, 1> B;
    int buf = 0;
    // level kc from global memory
    auto load = [&](int x, int y, T& u, T& b) {
        u = b = T(0);
        if (x < G.nx && y < G.ny) {
            const int64_t g = (int64_t)y * G.pitch + x;
            b = G.b[g];
            if (cont) u = G.u[g];  // else zero: coarse levels solve for a correction
        }
    };
    if (hasA) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int i = 0; i < 2; ++i) load(2 * lane + i, 4 * warp + r, A.u[r][i], A.b[r][i]);
    } else if (hasB) {
#pragma unroll
        for (int r = 0; r < 2; ++r) load(lane, 2 * warp + r, B.u[r][0], B.b[r][0]);
    } else if (tid < 256) {
        load(tid & 15, tid >> 4, us[0][tid], bs[0][tid]);
    }
    __syncthreads();
    // Each stage runs twice, on the way down and on the way up, through the same code (rolled loops:
    // most of it is executed a few times only, so fetching it is a sizeable part of the launch).
    if (hasA) A.init(tail_view<T>(sh, 0), lane, warp);
    if (hasB) B.init(tail_view<T>(sh, qB), lane, warp);
#pragma unroll 1
    for (int pa = 0; pa < 2; ++pa) {
        if (hasA) {
            if (pa) A.prolong(uc, 32);
            A.relax(edge, buf, lane, warp, pa ? a.nu_post : a.nu_pre);
        }
        if (pa) break;
        if (hasA) {
            T res[4][2];
            A.residual(edge, buf, lane, warp, res);
            // the reference restriction's order; children outside the level add 0
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                B.b[r][0] = (((res[2 * r][0] + res[2 * r][1]) + res[2 * r + 1][0]) + res[2 * r + 1][1]) * T(0.25);
                B.u[r][0] = T(0);
            }
        }
#pragma unroll 1
        for (int pb = 0; pb < 2; ++pb) {
            if (hasB) {
                if (pb) B.prolong(us[0], 16);
                B.relax(edge, buf, lane, warp, pb ? a.nu_post : a.nu_pre);
            }
            if (pb) break;
            if (hasB) {
                T res[2][1];
                B.residual(edge, buf, lane, warp, res);
                const T e0 = __shfl_down_sync(0xffffffffu, res[0][0], 1), e1 = __shfl_down_sync(0xffffffffu, res[1][0], 1);
                const T c = ((res[0][0] + e0) + res[1][0]) + e1;
                if ((lane & 1) == 0) bs[0][warp * 16 + (lane >> 1)] = c * T(0.25);
                __syncthreads();
            }
            if (warp == 0) {
                const int nc = nl - qC;
#pragma unroll 1
                for (int t = 0; t < 2 * nc - 1; ++t) {  // levels qC .. nl - 1, then back to qC
                    const bool down = t < nc;
                    const int i = down ? t : 2 * nc - 2 - t;
                    const int q = qC + i, next = i + 1 < nc ? i + 1 : i;
                    const bool from_us = !down || (cont && q == 0);
                    const int sweeps = down ? a.nu_pre : a.nu_post;
                    const int ny = sh.size[1][q], mode = ny > 1 ? max(sh.tab.mode[sh.off[1][q] + ny - 1], sh.tab.mode[sh.off[1][q] + ny - 2])
                                                                : kRowPartial;  // one row: both its faces are missing
                    const bool partial = mode == kRowPartial, wide = max(sh.size[0][q], ny) > 8;
                    if (wide && partial) TailWarp<T, 4, 8>::template leg<true>(q, i, next, down, from_us, sweeps);
                    else if (wide) TailWarp<T, 4, 8>::template leg<false>(q, i, next, down, from_us, sweeps);
                    else if (partial) TailWarp<T, 3, 2>::template leg<true>(q, i, next, down, from_us, sweeps);
                    else TailWarp<T, 3, 2>::template leg<false>(q, i, next, down, from_us, sweeps);
                }
            }
            __syncthreads();
        }
        if (hasA) {  // B's iterate for A's prolongation
#pragma unroll
            for (int r = 0; r < 2; ++r) uc[(2 * warp + r) * 32 + lane] = B.u[r][0];
            __syncthreads();
        }
    }
    // the final iterate of level kc back to global memory
    auto store = [&](int x, int y, T u) {
        if (x < G.nx && y < G.ny) G.u[(int64_t)y * G.pitch + x] = u;
    };
    if (hasA) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int i = 0; i < 2; ++i) store(2 * lane + i, 4 * warp + r, A.u[r][i]);
    } else if (hasB) {
#pragma unroll
        for (int r = 0; r < 2; ++r) store(lane, 2 * warp + r, B.u[r][0]);
    } else if (tid < 256) {
        store(tid & 15, tid >> 4, us[0][tid]);
    }
}

}  // namespace fused_detail
}  // namespace emfuse
