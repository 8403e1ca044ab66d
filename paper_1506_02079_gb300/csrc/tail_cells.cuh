// Coarse tail on copies in shared memory (FP64; tail_warps.cuh says when which).
//
// The levels of one slice from kc (the first with both sides <= kTailMax) down to 1 x 1 are run by
// one CTA: at most 64 x 64 + 32 x 32 + ... cells, u and b each.  Only level kc touches global memory:
// its right-hand side (and, continuing at level 0, its iterate) is read at the start and its final
// iterate written at the end.  The per-cell arithmetic and its order are those of every other
// schedule.
//
// Bound by the latency of about 70 dependent passes and by the FP64 pipe, so all warps share the
// coloured cells of a pass: the iterate has a border of zeros (no range checks: a missing neighbour
// has coefficient 0), the stencils come from a table of the at most 4 x 4 different ones of a level,
// the interpolation weights from tables, a thread loads the inputs of up to four cells before it
// stores any, and levels of at most 8 x 8 cells are run by one warp without block barriers.
#pragma once
#include <cuda_runtime.h>

#include "fused_impl.cuh"

namespace emfuse {
namespace fused_detail {

// Shared-memory bytes of the tail of a slice whose sides are all at most kTailMax (u with a border of
// one cell, and b, of every level down to 1 x 1).
template <class T>
constexpr int cells_smem_bytes() {
    int cells = 0;
    for (int n = kTailMax; n >= 1; n /= 2) cells += n * n + (n + 2) * (n + 2);
    return cells * (int)sizeof(T);
}

template <class T>
struct CellLevel {
    T* u;        // cell (0, 0) of the bordered iterate (row pitch nx + 2)
    T* b;        // right-hand side (row pitch nx)
    const TailCoef<T>* coef;  // [class of y][class of x]
    const T *wx, *wy;         // interpolation weights of this level's cells toward J
    const signed char *jx, *jy;  // J - I along each axis (0, -1 or 1)
    int nx, ny;
};

// Where a level's arrays start in the CTA's shared memory (offsets, not pointers, so that the
// accesses stay shared-memory ones).
struct CellOffsets {
    int u, b, x, y, nx, ny;
};

// `threads` threads (a power of two) on the cells of one colour: 2^sh lanes across the row.
__device__ __forceinline__ int cells_shift(int cells_x, int threads) {
    int sh = 0;
    while ((1 << sh) < cells_x && (1 << sh) < 32 && (1 << sh) < threads) ++sh;
    return sh;
}

template <class T, class Sync>
__device__ __forceinline__ void cells_relax(const CellLevel<T>& L, int sweeps, int tid, int threads, Sync sync) {
    const int nx = L.nx, ny = L.ny, pu = nx + 2;
    const int sh = cells_shift((nx + 1) >> 1, threads);
    const int lx = tid & ((1 << sh) - 1), ly = tid >> sh, rows = threads >> sh;
    constexpr int B = 4;  // cells in flight per thread
    for (int h = 0; h < 2 * sweeps; ++h) {
        for (int y0 = ly; y0 < ny; y0 += B * rows) {
            T v[B];
#pragma unroll
            for (int i = 0; i < B; ++i) {
                const int y = y0 + i * rows;
                const int x = 2 * lx + ((y + h) & 1);
                if (y < ny && x < nx) {
                    const Coef<T> c = tail_coef<T>(L.coef + 4 * tail_class(y, ny) + tail_class(x, nx));
                    const T* q = L.u + y * pu + x;
                    v[i] = gs_update<T>(c, L.b[y * nx + x], q[-1], q[1], q[-pu], q[pu]);
                }
            }
#pragma unroll
            for (int i = 0; i < B; ++i) {
                const int y = y0 + i * rows;
                const int x = 2 * lx + ((y + h) & 1);
                if (y < ny && x < nx) L.u[y * pu + x] = v[i];
            }
        }
        sync();
    }
}

// C.b = sum of the child residuals / 4 (C.u is zero already: it was cleared at the start).
template <class T, class Sync>
__device__ __forceinline__ void cells_restrict(const CellLevel<T>& L, const CellLevel<T>& C, int tid, int threads,
                                              Sync sync) {
    const int nx = L.nx, ny = L.ny, pu = nx + 2;
    const int sh = cells_shift(C.nx, threads);
    const int lx = tid & ((1 << sh) - 1), ly = tid >> sh, rows = threads >> sh;
    if (lx < C.nx)
        for (int J = ly; J < C.ny; J += rows) {
            T sum = T(0);
#pragma unroll
            for (int dy = 0; dy < 2; ++dy)
#pragma unroll
                for (int dx = 0; dx < 2; ++dx) {
                    const int x = 2 * lx + dx, y = 2 * J + dy;
                    if (x < nx && y < ny) {
                        const Coef<T> c = tail_coef<T>(L.coef + 4 * tail_class(y, ny) + tail_class(x, nx));
                        const T* q = L.u + y * pu + x;
                        sum += residual_at<T>(c, L.b[y * nx + x], q[0], q[-1], q[1], q[-pu], q[pu]);
                    }
                }
            C.b[J * C.nx + lx] = sum * T(0.25);
        }
    sync();
}

// L.u += interpolated C.u.
template <class T, class Sync>
__device__ __forceinline__ void cells_prolong(const CellLevel<T>& L, const CellLevel<T>& C, int tid, int threads,
                                             Sync sync) {
    const int nx = L.nx, ny = L.ny, pu = nx + 2, pc = C.nx + 2;
    const int sh = cells_shift(nx, threads);
    const int lx = tid & ((1 << sh) - 1), ly = tid >> sh, rows = threads >> sh;
    for (int x = lx; x < nx; x += 1 << sh) {
        const T wx = L.wx[x];
        const int I = x >> 1, J = I + L.jx[x];
        for (int y = ly; y < ny; y += rows) {
            const T wy = L.wy[y];
            const int Iy = y >> 1;
            const T* r0 = C.u + Iy * pc;
            const T* r1 = r0 + L.jy[y] * pc;
            L.u[y * pu + x] += bilinear<T>(r0[I], r0[J], r1[I], r1[J], wx, wy);
        }
    }
    sync();
}

// The V-cycle legs of levels q0 .. q1 - 1 (down; the last level of all is `last`) and q1 - 1 .. q0
// (up) of the tail; view(q) is level q.
template <class T, class View, class Sync>
__device__ __forceinline__ void cells_down(View view, int q0, int q1, int last, int nu, int tid, int threads,
                                          Sync sync) {
    for (int q = q0; q < q1; ++q) {
        cells_relax<T>(view(q), nu, tid, threads, sync);
        if (q < last) cells_restrict<T>(view(q), view(q + 1), tid, threads, sync);
    }
}
template <class T, class View, class Sync>
__device__ __forceinline__ void cells_up(View view, int q0, int q1, int nu, int tid, int threads, Sync sync) {
    for (int q = q1 - 1; q >= q0; --q) {
        cells_prolong<T>(view(q), view(q + 1), tid, threads, sync);
        cells_relax<T>(view(q), nu, tid, threads, sync);
    }
}

template <class T>
__global__ void __launch_bounds__(kTailThreads) k_tail_cells(TailArgs<T> a) {
    extern __shared__ __align__(16) unsigned char tail_smem[];
    __shared__ TailCoef<T> coef[kTailMaxLevels][16];
    __shared__ CellOffsets sl[kTailMaxLevels];
    __shared__ T wtab[2][4 * kTailMax];            // per axis, the levels one after another
    __shared__ signed char jtab[2][4 * kTailMax];
    const int j = blockIdx.x;
    if (a.active && !a.active[j]) return;
    const int tid = threadIdx.x;
    const int kc = a.kc[j];
    const LSlice<T>* lv = a.table + a.level_off[j];
    const int nl = a.nlev[j] - kc;  // levels of the tail
    if (nl > kTailMaxLevels || nl < 1) return;  // never: a 64 x 64 level has 6 levels below it
    const LSlice<T> G = lv[kc];
    const int n0x = G.n0x, n0y = G.n0y;
    // shared-memory layout: the bordered iterates of all levels, then their right-hand sides
    T* const base = reinterpret_cast<T*>(tail_smem);
    int ucells = 0;
    for (int q = 0; q < nl; ++q) ucells += (level_size(n0x, kc + q) + 2) * (level_size(n0y, kc + q) + 2);
    for (int p = tid; p < ucells; p += kTailThreads) base[p] = T(0);
    if (tid < nl) {
        CellOffsets L{0, ucells, 0, 0, 0, 0};
        for (int q = 0;; ++q) {
            L.nx = level_size(n0x, kc + q);
            L.ny = level_size(n0y, kc + q);
            if (q == tid) break;
            L.u += (L.nx + 2) * (L.ny + 2);
            L.b += L.nx * L.ny;
            L.x += L.nx;
            L.y += L.ny;
        }
        sl[tid] = L;
    }
    auto view = [&](int q) {
        const CellOffsets o = sl[q];
        CellLevel<T> L;
        L.u = base + o.u + (o.nx + 2) + 1;
        L.b = base + o.b;
        L.coef = coef[q];
        L.wx = wtab[0] + o.x;
        L.wy = wtab[1] + o.y;
        L.jx = jtab[0] + o.x;
        L.jy = jtab[1] + o.y;
        L.nx = o.nx;
        L.ny = o.ny;
        return L;
    };
    for (int p = tid; p < nl * 16; p += kTailThreads) {
        const int k = kc + (p >> 4), nx = level_size(n0x, k), ny = level_size(n0y, k);
        const int x = tail_class_rep(p & 3, nx), y = tail_class_rep((p >> 2) & 3, ny);
        const Coef<T> c = coef_at<T>(x, y, nx, ny, n0x, n0y, k, a.alpha, T(ldexp(1.0, -2 * k)));
        TailCoef<T>& t = coef[p >> 4][p & 15];
        t.cw = c.cw; t.ce = c.ce; t.cn = c.cn; t.cs = c.cs; t.iD = c.iD; t.D = c.D;
    }
    __syncthreads();
    {   // interpolation tables (every level but the last), and level kc from global memory: its
        // rhs, and its iterate when continuing at level 0
        for (int q = 0; q + 1 < nl; ++q)
            for (int p = tid; p < sl[q].nx + sl[q].ny; p += kTailThreads) {
                const bool ax = p < sl[q].nx;
                const int i = ax ? p : p - sl[q].nx;
                int I, J;
                T w;
                interp_axis<T>(i, ax ? n0x : n0y, kc + q, ax ? sl[q + 1].nx : sl[q + 1].ny, I, J, w);
                const int at = (ax ? sl[q].x : sl[q].y) + i;
                wtab[ax ? 0 : 1][at] = w;
                jtab[ax ? 0 : 1][at] = (signed char)(J - I);
            }
        const CellLevel<T> L = view(0);
        const bool cont = a.cont && kc == 0;
        const int sh = cells_shift(L.nx, kTailThreads);
        for (int x = tid & ((1 << sh) - 1); x < L.nx; x += 1 << sh)
            for (int y = tid >> sh; y < L.ny; y += kTailThreads >> sh) {
                const int64_t g = (int64_t)y * G.pitch + x;
                L.b[y * L.nx + x] = G.b[g];
                if (cont) L.u[y * (L.nx + 2) + x] = G.u[g];  // else zero: coarse levels solve for a correction
            }
    }
    __syncthreads();
    int qs = 0;  // first level that one warp runs alone (the last level is 1 x 1)
    while (sl[qs].nx > 8 || sl[qs].ny > 8) ++qs;
    auto block_sync = [] { __syncthreads(); };
    auto warp_sync = [] { __syncwarp(); };
    cells_down<T>(view, 0, qs, nl - 1, a.nu_pre, tid, kTailThreads, block_sync);
    if (tid < 32) {
        cells_down<T>(view, qs, nl, nl - 1, a.nu_pre, tid, 32, warp_sync);
        cells_up<T>(view, qs, nl - 1, a.nu_post, tid, 32, warp_sync);
    }
    __syncthreads();
    cells_up<T>(view, 0, qs, a.nu_post, tid, kTailThreads, block_sync);
    {   // the final iterate of level kc back to global memory
        const CellLevel<T> L = view(0);
        const int sh = cells_shift(L.nx, kTailThreads);
        for (int x = tid & ((1 << sh) - 1); x < L.nx; x += 1 << sh)
            for (int y = tid >> sh; y < L.ny; y += kTailThreads >> sh)
                G.u[(int64_t)y * G.pitch + x] = L.u[y * (L.nx + 2) + x];
    }
}

}  // namespace fused_detail
}  // namespace emfuse
