// Tile kernels: the V-cycle legs of the middle levels (too large for one CTA, too small to fill
// the chip with the wavefront kernel's long marches).
//
// A CTA takes one tile of a level, 128 columns x 4 rows per warp, into registers: a lane holds 4
// consecutive cells of 4 rows, its right-hand sides included.  All half-sweeps of a leg then run
// without another look at global memory.  Neighbours along x inside a lane are registers, across
// lanes one shuffle per row; along y inside a warp registers, across warps the edge rows are
// exchanged through shared memory, double buffered, one barrier per half-sweep.  The outermost
// cells of the tile lack their neighbours, and every half-sweep carries the wrong values one cell
// further in, so a tile's output is the loaded area less a halo of S cells (UP) or S + 1 (DOWN,
// whose residual reaches one further); halos are recomputed by the neighbouring tiles.
//
//   DOWN: S half-sweeps (from zero, or from the previous V-cycle's iterate), u written, residual
//         summed 2 x 2 / 4 into the next level's right-hand side.
//   UP:   the interpolated coarse correction added while loading, S half-sweeps, uo written.
//
// The per-cell arithmetic and its order are those of every other schedule (the results are the
// same bit for bit).  Three ways to a cell's stencil, chosen per warp and row: the interior one
// from registers (all cells of the warp interior); per-column stencils from a table in shared
// memory for rows whose cells have full height, where cells outside the level are kept at exactly
// 0 (their 1 / D is 0), so that a missing neighbour adds nothing and only the diagonal differs on
// the first and last row; and the table of a level's stencils for rows of partial cells.
//
// Bound by latency and barriers (two CTAs of 16 warps per SM): one 128 x 128 level of 16 slices
// takes 8 us where the wavefront kernel's march took 25; 64 registers hold the 32 values and
// their neighbours (the UP leg's coarse rows spill 52 bytes while it loads), taller warps would leave
// one CTA per SM.
#pragma once
#include <cuda_runtime.h>

#include "fused_impl.cuh"

namespace emfuse {
namespace fused_detail {

constexpr int kTileRows = 4;  // rows per lane

// Warps per CTA: 16 (64 rows; two CTAs per SM at 64 registers) for float, 8 for double.
template <class T>
struct TileShape {
    static constexpr int kWarps = sizeof(T) == 4 ? 16 : 8;
    static constexpr int kRows = kWarps * kTileRows;
};

// Stencil of cell (x, y), which must be in the level.
template <class T>
__device__ __forceinline__ Coef<T> tile_coef(const TailCoef<T>* tab, int x, int y, int nx, int ny) {
    return tail_coef<T>(tab + 4 * tail_class(y, ny) + tail_class(x, nx));
}

// Stencils of a column (col_stencil), split for vector loads.
template <class T>
struct alignas(16) ColCoef {
    T cw, ce, cy, iD;
};
template <class T>
struct ColDiag {
    T iDb, D, Db;
};

template <class T, bool ZERO, bool UP>
__global__ void __launch_bounds__(TileShape<T>::kWarps * 32, 2) k_tile(TileArgs<T> a) {
    constexpr int NW = TileShape<T>::kWarps, R = kTileRows;
    __shared__ __align__(16) T edge[2][NW][2][kWaveWidth];  // first and last row of every warp
    __shared__ TailCoef<T> tab[16];
    __shared__ ColCoef<T> col[4][32];        // column 4 lane + i at [i][lane]
    __shared__ ColDiag<T> diag[4][32];
    __shared__ T colw[4][32], roww[TileShape<T>::kRows];  // interpolation weights (UP)
    __shared__ __align__(4) unsigned char rowm[TileShape<T>::kRows];
    const int64_t t = blockIdx.x;
    const int j = find_item_warp(a.tile_start, a.nsl, t);
    const LSlice<T> L = a.sl[j];
    if (a.active && !a.active[L.slice]) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nx = L.nx, ny = L.ny, k = a.k;
    const int lt = int(t - a.tile_start[j]);
    const int ow = kWaveWidth - 2 * a.hx, oh = TileShape<T>::kRows - 2 * a.hy;
    const int tiles_x = (nx + ow - 1) / ow;
    const int X0 = (lt % tiles_x) * ow, Y0 = (lt / tiles_x) * oh;  // multiples of 4 and 2
    const int x = X0 - a.hx + 4 * lane;                           // first cell of the lane
    const int y = Y0 - a.hy + R * warp;                           // first row of the warp (even)
    // stencils and interpolation weights of the tile's columns and rows, one per thread
    if (tid < kWaveWidth) {
        const int xc = X0 - a.hx + tid, q = tid & 3, l = tid >> 2;
        T w = T(0);
        const ColStencil<T> st = col_stencil<T>(xc, nx, L.n0x, k, a.alpha, a.sk);
        const ColCoef<T> c{st.cw, st.ce, st.cy, st.iD};
        const ColDiag<T> d{st.iDb, st.D, st.Db};
        if (UP && xc >= 0 && xc < nx) {
            int I, J;
            interp_axis<T>(xc, L.n0x, k, L.ncx, I, J, w);
        }
        col[q][l] = c;
        diag[q][l] = d;
        if (UP) colw[q][l] = w;
    } else if (tid < kWaveWidth + TileShape<T>::kRows) {
        const int q = tid - kWaveWidth, yr = Y0 - a.hy + q;
        T w = T(0);
        if (UP && yr >= 0 && yr < ny) {
            int I, J;
            interp_axis<T>(yr, L.n0y, k, L.ncy, I, J, w);
        }
        rowm[q] = row_mode<T>(yr, ny, L.n0y, k);
        if (UP) roww[q] = w;
    } else if (tid >= TileShape<T>::kWarps * 32 - 16) {
        const int q = tid & 15;
        const Coef<T> c = coef_at<T>(tail_class_rep(q & 3, nx), tail_class_rep(q >> 2, ny), nx, ny, L.n0x, L.n0y, k, a.alpha, a.sk);
        TailCoef<T>& o = tab[q];
        o.cw = c.cw; o.ce = c.ce; o.cn = c.cn; o.cs = c.cs; o.iD = c.iD; o.D = c.D;
    }
    T u[R][4], b[R][4];
    const bool lane_in = x >= 0 && x < nx;  // x is a multiple of 4
    const T* const usrc = a.from_uo ? L.uo : L.u;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const bool in = lane_in && y + r >= 0 && y + r < ny;
#pragma unroll
        for (int i = 0; i < 4; ++i) b[r][i] = u[r][i] = T(0);
        if (in) {  // rows are padded to 128 bytes, so the vector stays inside the row
            const int64_t p = (int64_t)(y + r) * L.pitch + x;
            Vec4<T>::load(L.b + p, b[r]);
            if (!ZERO) Vec4<T>::load(usrc + p, u[r]);
        }
#pragma unroll
        for (int i = 1; i < 4; ++i)
            if (x + i >= nx) {  // padding
                b[r][i] = T(0);
                u[r][i] = T(0);
            }
    }
    if (UP) {
        // coarse rows y/2 - 1 .. y/2 + 2, columns x/2 - 1 .. x/2 + 2 (those outside the level are
        // met with weight 0).  A fine cell's other coarse cell is the previous one for even
        // cells and the next one for odd cells, or its weight is 0 (interp_axis).
        const int cx = x >> 1, cy = y >> 1;  // y may be negative: arithmetic shift
        T c[R / 2 + 2][4];
#pragma unroll
        for (int q = 0; q < R / 2 + 2; ++q) {
            const int Y = cy - 1 + q;
            const bool row = Y >= 0 && Y < L.ncy;
            const T* src = L.uco + (int64_t)Y * L.pitchc;
            T m0 = T(0), m1 = T(0);
            if (row && cx >= 0 && cx < L.ncx) Vec2<T>::load(src + cx, m0, m1);
            if (cx + 1 >= L.ncx) m1 = T(0);
            T w = __shfl_up_sync(0xffffffffu, m1, 1), e = __shfl_down_sync(0xffffffffu, m0, 1);
            if (lane == 0) w = row && cx >= 1 && cx - 1 < L.ncx ? src[cx - 1] : T(0);
            if (lane == 31) e = row && cx + 2 >= 0 && cx + 2 < L.ncx ? src[cx + 2] : T(0);
            c[q][0] = w; c[q][1] = m0; c[q][2] = m1; c[q][3] = e;
        }
        __syncthreads();  // colw, roww
        T wx[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) wx[i] = colw[i][lane];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (y + r < 0 || y + r >= ny) continue;  // warp-uniform
            const T wy = roww[R * warp + r];
            const int q0 = r / 2 + 1, q1 = (r & 1) ? q0 + 1 : q0 - 1;
            const T v0 = bilinear<T>(c[q0][1], c[q0][0], c[q1][1], c[q1][0], wx[0], wy);
            const T v1 = bilinear<T>(c[q0][1], c[q0][2], c[q1][1], c[q1][2], wx[1], wy);
            const T v2 = bilinear<T>(c[q0][2], c[q0][1], c[q1][2], c[q1][1], wx[2], wy);
            const T v3 = bilinear<T>(c[q0][2], c[q0][3], c[q1][2], c[q1][3], wx[3], wy);
            if (lane_in) {
                u[r][0] += v0;
                if (x + 1 < nx) u[r][1] += v1;
                if (x + 2 < nx) u[r][2] += v2;
                if (x + 3 < nx) u[r][3] += v3;
            }
        }
    }
    // every cell of the warp interior along x and y: class 1 for all, in the level
    const int last = k == 0 ? 1 : 2;  // cells from the end whose stencil may differ
    const bool fast = __all_sync(0xffffffffu, x >= 1 && x + 3 < nx - last) && y >= 1 && y + R - 1 < ny - last;
    Coef<T> ci;
    {
        AxisCoef<T> one;
        one.w = T(1); one.gm = T(1); one.gp = T(1);
        ci = make_coef<T>(one, one, k, a.alpha, a.sk);
    }
    unsigned modes = 0;  // rowm of the warp's rows, one byte each (read after the first barrier)
    int buf = 0;
    T no[4], so[4];  // the rows above and below the warp's
    auto exchange = [&]() {
        Vec4<T>::store(&edge[buf][warp][0][4 * lane], u[0]);
        Vec4<T>::store(&edge[buf][warp][1][4 * lane], u[R - 1]);
        __syncthreads();
        if (warp > 0) Vec4<T>::load(&edge[buf][warp - 1][1][4 * lane], no);
        else no[0] = no[1] = no[2] = no[3] = T(0);
        if (warp + 1 < NW) Vec4<T>::load(&edge[buf][warp + 1][0][4 * lane], so);
        else so[0] = so[1] = so[2] = so[3] = T(0);
        buf ^= 1;
    };
    // one cell on a row of full cells, mode inner, edge or outside
    auto update = [&](int i, unsigned mode, T bv, T w, T e, T n, T s) -> T {
        const ColCoef<T> q = col[i][lane];
        Coef<T> c;
        c.cw = q.cw; c.ce = q.ce; c.cn = c.cs = q.cy;
        c.iD = mode == kRowInner ? q.iD : (mode == kRowEdge ? diag[i][lane].iDb : T(0));
        return gs_update<T>(c, bv, w, e, n, s);
    };
    auto half_sweep = [&](auto colour_tag) {
        constexpr int C = decltype(colour_tag)::value;
        exchange();
        if (!fast) modes = *reinterpret_cast<const unsigned*>(&rowm[R * warp]);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const T(&n)[4] = r > 0 ? u[r > 0 ? r - 1 : 0] : no;
            const T(&s)[4] = r + 1 < R ? u[r + 1 < R ? r + 1 : 0] : so;
            const int f = (r + C) & 1;  // y is even and x a multiple of 4
            const T o = f == 0 ? __shfl_up_sync(0xffffffffu, u[r][3], 1) : __shfl_down_sync(0xffffffffu, u[r][0], 1);
            const T w0 = f == 0 ? o : u[r][0], e0 = f == 0 ? u[r][1] : u[r][2];
            const T w1 = f == 0 ? u[r][1] : u[r][2], e1 = f == 0 ? u[r][3] : o;
            const unsigned mode = (modes >> (8 * r)) & 0xffu;
            if (fast) {
                u[r][f] = gs_update<T>(ci, b[r][f], w0, e0, n[f], s[f]);
                u[r][f + 2] = gs_update<T>(ci, b[r][f + 2], w1, e1, n[f + 2], s[f + 2]);
            } else if (mode != kRowPartial) {
                u[r][f] = update(f, mode, b[r][f], w0, e0, n[f], s[f]);
                u[r][f + 2] = update(f + 2, mode, b[r][f + 2], w1, e1, n[f + 2], s[f + 2]);
            } else if (lane_in) {
                if (x + f < nx)
                    u[r][f] = gs_update<T>(tile_coef<T>(tab, x + f, y + r, nx, ny), b[r][f], w0, e0, n[f], s[f]);
                if (x + f + 2 < nx)
                    u[r][f + 2] = gs_update<T>(tile_coef<T>(tab, x + f + 2, y + r, nx, ny), b[r][f + 2], w1, e1,
                                               n[f + 2], s[f + 2]);
            }
        }
    };
#pragma unroll 1
    for (int s = 0; s < a.nu; ++s) {
        half_sweep(std::integral_constant<int, 0>{});
        half_sweep(std::integral_constant<int, 1>{});
    }
    const bool lane_out = lane_in && 4 * lane >= a.hx && 4 * lane < kWaveWidth - a.hx;
    T* const dst = UP ? L.uo : L.u;
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (lane_out && y + r >= Y0 && y + r < min(Y0 + oh, ny))
            Vec4<T>::store(dst + (int64_t)(y + r) * L.pitch + x, u[r]);
    if (!UP) {
        exchange();
        T res[R][4];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const T(&n)[4] = r > 0 ? u[r > 0 ? r - 1 : 0] : no;
            const T(&s)[4] = r + 1 < R ? u[r + 1 < R ? r + 1 : 0] : so;
            const T w = __shfl_up_sync(0xffffffffu, u[r][3], 1), e = __shfl_down_sync(0xffffffffu, u[r][0], 1);
            const unsigned mode = (modes >> (8 * r)) & 0xffu;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const T uw = i == 0 ? w : u[r][i > 0 ? i - 1 : 0], ue = i == 3 ? e : u[r][i < 3 ? i + 1 : 0];
                res[r][i] = T(0);
                if (fast) {
                    res[r][i] = residual_at<T>(ci, b[r][i], u[r][i], uw, ue, n[i], s[i]);
                } else if (mode <= kRowEdge) {
                    const ColCoef<T> q = col[i][lane];
                    Coef<T> c;
                    c.cw = q.cw; c.ce = q.ce; c.cn = c.cs = q.cy;
                    c.D = mode == kRowInner ? diag[i][lane].D : diag[i][lane].Db;
                    res[r][i] = residual_at<T>(c, b[r][i], u[r][i], uw, ue, n[i], s[i]);
                } else if (mode == kRowPartial && lane_in && x + i < nx) {
                    res[r][i] = residual_at<T>(tile_coef<T>(tab, x + i, y + r, nx, ny), b[r][i], u[r][i], uw, ue, n[i],
                                               s[i]);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < R / 2; ++q) {
            const int Y = (y >> 1) + q, X = x >> 1;
            if (lane_out && 2 * Y >= Y0 && 2 * Y < min(Y0 + oh, ny)) {
                // the reference restriction's order; children outside the level add 0
                const T c0 = ((res[2 * q][0] + res[2 * q][1]) + res[2 * q + 1][0]) + res[2 * q + 1][1];
                const T c1 = ((res[2 * q][2] + res[2 * q][3]) + res[2 * q + 1][2]) + res[2 * q + 1][3];
                Vec2<T>::store(L.bc + (int64_t)Y * L.pitchc + X, c0 * T(0.25), c1 * T(0.25));
            }
        }
    }
}

template <class T>
void tile_extent_impl(int halo, int& hx, int& hy, int& out_x, int& out_y) {
    hx = (halo + 3) / 4 * 4;
    hy = (halo + 1) / 2 * 2;
    out_x = kWaveWidth - 2 * hx;
    out_y = TileShape<T>::kRows - 2 * hy;
}

// One CTA per tile.
template <class T>
int launch_tile_impl(const TileArgs<T>& a, bool zero_init, bool up, cudaStream_t st, double bytes) {
    if (a.ntiles == 0) return EMFUSE_OK;
    static const char* const kUp[] = {"tile_up_l0", "tile_up_l1", "tile_up_l2", "tile_up_l3", "tile_up_l4",
                                      "tile_up_l5+"};
    static const char* const kDown[] = {"tile_down_l0", "tile_down_l1", "tile_down_l2", "tile_down_l3",
                                        "tile_down_l4", "tile_down_l5+"};
    KernelScope ks((up ? kUp : kDown)[a.k < 5 ? a.k : 5], st, bytes);
    const unsigned grid = (unsigned)a.ntiles, threads = TileShape<T>::kWarps * 32;
    if (up) k_tile<T, false, true><<<grid, threads, 0, st>>>(a);
    else if (zero_init) k_tile<T, true, false><<<grid, threads, 0, st>>>(a);
    else k_tile<T, false, false><<<grid, threads, 0, st>>>(a);
    EMF_CHECK_LAUNCH();
    return EMFUSE_OK;
}

}  // namespace fused_detail
}  // namespace emfuse
