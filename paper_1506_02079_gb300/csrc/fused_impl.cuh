// Fused multigrid schedule.
//
// Wavefront kernel (k_wave).  One warp owns a strip of 128 cells (32 lanes x 4 consecutive
// cells) and marches down a chunk of rows two at a time.  All nu red-black sweeps are
// pipelined in one pass: at step T the warp receives row pair T (rows 2T, 2T+1) and applies
// half-sweep s (s = 1..S, S = 2 nu) to pair T - s.  Half-sweep s only reads the other colour,
// whose latest update (half-sweep s - 1) reached pairs T-s-1 .. T-s+1 before half-sweep s + 1
// touches them, so the result is exactly that of S global half-sweeps (Gauss-Seidel
// red-black, colour (x + y) mod 2).  Row pairs arrive by TMA (one 128 x 2 box per array) into
// a per-warp shared-memory ring guarded by mbarriers with bounded waits; u moves into a
// register window of S + 3 pairs, b is read from the ring when a half-sweep needs it.
// Neighbours along x come from warp shuffles, so strip edges are recomputed by the adjacent
// strips (8-cell overlap on each side).
//
//   DOWN (restriction leg): optional zero initial guess (the first half-sweep then needs no
//        load of u), S half-sweeps, the residual of the pair S + 1 behind, and its 2x2 sums / 4
//        written as one row of the next level's right-hand side.  One read of b
//        (and u), one write of u and of the coarse rhs per cell.
//   UP   (prolongation leg): the interpolated coarse correction is added as each row
//        arrives, then S half-sweeps; one read of u, b and the coarse iterate, one write of
//        the result into a second buffer (uo): the warps read u on their halos, so no warp may
//        overwrite it in place.
//
// Rows of a step: see `step` in k_wave for its three bodies.  Running the steps at the top of a
// chunk by the same range-check-free bodies as the rest, and strips of any width by cached
// stencils, took level 0 of 64 x 2048 x 2048 from 0.556 to 0.507 ms per UP leg, of 96 ragged slices
// (291 M cells) from 1.08 to 0.66 ms, on average over solves in whose last V-cycles most slices have
// converged.  With every slice at work: 0.59 ms (5.9 TB/s, 0.87 of the copy rate) and 0.81 ms (5.7); DOWN
// legs 0.54 to 0.56 (5.3) and 0.76 (5.2).
//
// Levels whose larger side is <= 64 are run by one CTA per slice: tail_warps.cuh (FP32),
// tail_cells.cuh (FP64).
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

#include "emfuse_common.cuh"
#include "mg_fused.cuh"
#include "tma.cuh"

namespace emfuse {
namespace fused_detail {

template <class T>
struct Vec4;
template <>
struct Vec4<float> {
    static __device__ __forceinline__ void load(const float* p, float (&v)[4]) {
        const float4 q = *reinterpret_cast<const float4*>(p);
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    }
    static __device__ __forceinline__ void store(float* p, const float (&v)[4]) {
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    }
};
template <>
struct Vec4<double> {
    static __device__ __forceinline__ void load(const double* p, double (&v)[4]) {
        const double2 a = *reinterpret_cast<const double2*>(p);
        const double2 b = *reinterpret_cast<const double2*>(p + 2);
        v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    }
    static __device__ __forceinline__ void store(double* p, const double (&v)[4]) {
        *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
        *reinterpret_cast<double2*>(p + 2) = make_double2(v[2], v[3]);
    }
};

template <class T>
struct Vec2;
template <>
struct Vec2<float> {
    static __device__ __forceinline__ void load(const float* p, float& a, float& b) {
        const float2 q = *reinterpret_cast<const float2*>(p);
        a = q.x; b = q.y;
    }
    static __device__ __forceinline__ void store(float* p, float a, float b) {
        *reinterpret_cast<float2*>(p) = make_float2(a, b);
    }
};
template <>
struct Vec2<double> {
    static __device__ __forceinline__ void load(const double* p, double& a, double& b) {
        const double2 q = *reinterpret_cast<const double2*>(p);
        a = q.x; b = q.y;
    }
    static __device__ __forceinline__ void store(double* p, double a, double b) {
        *reinterpret_cast<double2*>(p) = make_double2(a, b);
    }
};

constexpr int kWaveWarps = 4;  // warps (strips) per CTA


__host__ __device__ constexpr int wmod(int a, int w) { return ((a % w) + w) % w; }

// CTAs per SM the register budget is sized for: the register window grows with the sweeps (S + 3
// row pairs) and FP64 windows take twice the registers (the continuing DOWN leg in FP64 at S = 4, once a
// solve, spills 24 bytes).
template <class T, int S>
struct WaveOcc { static constexpr int value = (sizeof(T) == 4 && S <= 4) ? 4 : 2; };

// ---------------------------------------------------------------- per-cell stencils
// Interior cells (full cells with full neighbours) all share one stencil.  Cells on a slice
// edge, a partial coarse cell or outside the level take per-cell stencils: selects at level 0
// (alpha + degree and its reciprocal formed when needed, so that nothing of these rare paths
// stays live in registers across the march), the general finite-volume formula out of line on
// coarse levels.
template <class T>
struct StencilTab {
    Coef<T> ci;   // interior stencil
};

// Per-lane diagonal of the interior body (see "ghost strips" in k_wave): 1 / D of cell 0, of
// cells 1 and 2 and of cell 3 of the lane, and D of cells 0 and 3 (cells 1 and 2 always have the
// interior D).  Interior lanes hold the interior values; lanes outside the level 1 / D = 0.
template <class T>
struct LaneDiag {
    T iD0, iD12, iD3;
    T D0, D3;
};

// gs_update with the reciprocal diagonal given separately (same operations, same order).
template <class T>
__device__ __forceinline__ T gs_update_iD(const Coef<T>& c, T iD, T b, T uw, T ue, T un, T us) {
    T acc = fma_t(c.cw, uw, b);
    acc = fma_t(c.ce, ue, acc);
    acc = fma_t(c.cn, un, acc);
    acc = fma_t(c.cs, us, acc);
    return mul_t(acc, iD);
}

// residual_at with the diagonal given separately (same operations, same order).
template <class T>
__device__ __forceinline__ T residual_at_D(const Coef<T>& c, T D, T b, T u, T uw, T ue, T un, T us) {
    T acc = fma_t(c.cw, uw, b);
    acc = fma_t(c.ce, ue, acc);
    acc = fma_t(c.cn, un, acc);
    acc = fma_t(c.cs, us, acc);
    return fma_t(-D, u, acc);
}

template <class T>
__device__ __forceinline__ void make_stencil_tab(StencilTab<T>& tab, int k, T alpha, T sk) {
    AxisCoef<T> one;
    one.w = T(1); one.gm = T(1); one.gp = T(1);
    tab.ci = make_coef<T>(one, one, k, alpha, sk);
}

// Level-0 stencil of cell (x, r) from selects; equal to make_coef at level 0.
template <class T>
__device__ __forceinline__ Coef<T> level0_coef(int x, int r, int nx, int ny, T alpha) {
    Coef<T> c;
    const bool in = x >= 0 && x < nx && r >= 0 && r < ny;
    const int w = in && x > 0, e = in && x + 1 < nx, n = in && r > 0, s = in && r + 1 < ny;
    c.cw = T(w); c.ce = T(e); c.cn = T(n); c.cs = T(s);
    // alpha + (((cw + ce) + cn) + cs) for 0/1 coefficients; outside the level the cell is
    // decoupled (the w = 1 cell of axis_coef): D = alpha
    c.D = alpha + T(w + e + n + s);
    c.iD = rcp_t(c.D);
    return c;
}

template <class T>
__device__ __noinline__ Coef<T> coarse_cell_coef(int x, int r, int nx, int ny, int n0x, int n0y, int k, T alpha,
                                                 T sk) {
    return make_coef<T>(axis_coef<T>(x, nx, n0x, k), axis_coef<T>(r, ny, n0y, k), k, alpha, sk);
}

template <class T>
__device__ __forceinline__ Coef<T> edge_coef(const StencilTab<T>& tab, int x, int r, int nx, int ny, int n0x,
                                             int n0y, int k, T alpha, T sk) {
    return k == 0 ? level0_coef<T>(x, r, nx, ny, alpha) : coarse_cell_coef<T>(x, r, nx, ny, n0x, n0y, k, alpha, sk);
}

// Stencil of cell i of the lane on an interior row, from the lane's shared-memory cache
// (cw, ce, cn = cs, 1/D per cell, as make_coef returns them on such a row, in one vector load
// without bank conflicts; D apart, only the residual needs it).  `cache`: the lane's first vector.
template <class T>
__device__ __forceinline__ Coef<T> cached_coef(uint32_t cache, int i) {
    Coef<T> c;
    T q[4];
    lds4(cache + i * 128 * (uint32_t)sizeof(T), q);
    c.cw = q[0]; c.ce = q[1]; c.cn = q[2]; c.cs = q[2]; c.iD = q[3];
    return c;
}
template <class T>
__device__ __forceinline__ T cached_diag(uint32_t cache, int lane, int i) {
    return lds1(cache - lane * 3 * (uint32_t)sizeof(T) + (512 + 32 * i) * (uint32_t)sizeof(T), T(0));
}

// Half-sweep of one colour on one row of the lane's 4 cells (cells f and f + 2).  FAST: interior
// stencils (with the lane's diagonals); ROWS: an interior row, known when compiled.
template <class T, bool FAST, bool ROWS>
__device__ __forceinline__ void sweep_row(T (&row)[4], const T (&brow)[4], const T (&nrow)[4], const T (&srow)[4],
                                          int f, T west, T east, bool fast, bool irow, uint32_t cache,
                                          const StencilTab<T>& tab, const LaneDiag<T>& g, int xlane, int r, int nx,
                                          int ny, int n0x, int n0y, int k, T alpha, T sk) {
    if (FAST || fast) {
        if (f == 0) {
            row[0] = gs_update_iD<T>(tab.ci, g.iD0, brow[0], west, row[1], nrow[0], srow[0]);
            row[2] = gs_update_iD<T>(tab.ci, g.iD12, brow[2], row[1], row[3], nrow[2], srow[2]);
        } else {
            row[1] = gs_update_iD<T>(tab.ci, g.iD12, brow[1], row[0], row[2], nrow[1], srow[1]);
            row[3] = gs_update_iD<T>(tab.ci, g.iD3, brow[3], row[2], east, nrow[3], srow[3]);
        }
    } else {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = 2 * h + f;
            const T uw = i == 0 ? west : row[i - 1];
            const T ue = i == 3 ? east : row[i + 1];
            const Coef<T> c = ROWS || irow ? cached_coef<T>(cache, i)
                                           : edge_coef<T>(tab, xlane + i, r, nx, ny, n0x, n0y, k, alpha, sk);
            row[i] = gs_update<T>(c, brow[i], uw, ue, nrow[i], srow[i]);
        }
    }
}

// Residuals of one row of the lane's 4 cells.
template <class T, bool FAST, bool ROWS>
__device__ __forceinline__ void residual_row(T (&res)[4], const T (&row)[4], const T (&brow)[4], const T (&nrow)[4],
                                             const T (&srow)[4], T west, T east, bool fast, bool irow,
                                             uint32_t cache, const StencilTab<T>& tab, const LaneDiag<T>& g,
                                             int xlane, int r, int nx, int ny, int n0x, int n0y, int k, T alpha,
                                             T sk) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const T uw = i == 0 ? west : row[i - 1];
        const T ue = i == 3 ? east : row[i + 1];
        if (FAST || fast) {
            const T D = i == 0 ? g.D0 : (i == 3 ? g.D3 : tab.ci.D);
            res[i] = residual_at_D<T>(tab.ci, D, brow[i], row[i], uw, ue, nrow[i], srow[i]);
        } else {
            Coef<T> c;
            if (ROWS || irow) {
                c = cached_coef<T>(cache, i);
                c.D = cached_diag<T>(cache, threadIdx.x & 31, i);
            } else {
                c = edge_coef<T>(tab, xlane + i, r, nx, ny, n0x, n0y, k, alpha, sk);
            }
            res[i] = residual_at<T>(c, brow[i], row[i], uw, ue, nrow[i], srow[i]);
        }
    }
}

// Shared-memory rings of one warp, in units of row pairs.  b: one slot per pair from the
// oldest pair still needed (the residual pair, S + 1 behind the newest) to the newest pair in
// flight; u and the coarse rows (UP) are consumed when their pair arrives, so kAhead slots.
template <class T, int S, bool ZERO, bool UP>
struct WaveRing {
    static constexpr int kAhead = 2;                                         // pairs in flight
    static constexpr int kNB = kAhead + S + (UP ? 1 : 2);                    // b slots = barriers
    static constexpr int kPairBytes = 2 * kWaveWidth * (int)sizeof(T);
    static constexpr int kCoarseBytes = UP ? (kWaveCoarseW * 3 * (int)sizeof(T) + 127) / 128 * 128 : 0;
    static constexpr int kUSlotBytes = (ZERO ? 0 : kPairBytes) + kCoarseBytes;
    static constexpr int kBRingBytes = kNB * kPairBytes;
    static constexpr int kURingBytes = kAhead * kUSlotBytes;
    // per-lane cache: stencils, and for UP the interpolation weights along x
    static constexpr int kCoefBytes = 32 * 4 * (UP ? 6 : 5) * (int)sizeof(T);
    static constexpr int kWarpBytes = kBRingBytes + kURingBytes + kCoefBytes + (kNB * 8 + 127) / 128 * 128;
};

template <class T, int S, bool ZERO, bool UP>
constexpr int wave_smem_bytes() { return kWaveWarps * WaveRing<T, S, ZERO, UP>::kWarpBytes; }

template <class T, int S, bool ZERO, bool UP>
__global__ void __launch_bounds__(kWaveWarps * 32, WaveOcc<T, S>::value) k_wave(WaveArgs<T> a) {
    using R = WaveRing<T, S, ZERO, UP>;
    constexpr int NB = R::kNB;
    constexpr int AHEAD = R::kAhead;
    constexpr int NR = UP ? S + 2 : S + 3;      // window: pairs T-NR+1 .. T (slot NR-1 = pair T)
    constexpr int HP = UP ? (S + 1) / 2 : (S + 2) / 2;  // halo pairs above the chunk
    constexpr uint32_t kRowB = kWaveWidth * sizeof(T);
    extern __shared__ __align__(128) unsigned char wave_smem[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    // ---- rings and barriers of this warp, set up once: the warp runs work items back to back
    // through them, taking the next item from the launch's work counter (items are independent,
    // so the order does not change any result)
    unsigned char* ring = wave_smem + (size_t)warp * R::kWarpBytes;
    const uint32_t ring_s = smem_addr(ring);
    const uint32_t uring_s = ring_s + R::kBRingBytes;
    const uint32_t coef_s = uring_s + R::kURingBytes + lane * 4 * (uint32_t)sizeof(T);
    const uint32_t bar_s = uring_s + R::kURingBytes + R::kCoefBytes;
    if (lane == 0) {
        for (int q = 0; q < NB; ++q) mbar_init(bar_s + 8 * q, 1);
        mbar_init_fence();
    }
    __syncwarp();
    int bs = 0, us = 0;  // ring slots of the next pair
    uint32_t phase = 0;  // parity of the b-slot barriers in the current lap

    // One work item: a strip of 128 columns and a chunk of rows of one slice.  Returns false
    // when a bounded wait gave up.
    auto run_item = [&](const int64_t item) -> bool {
    const int j = find_item(a.item_start, a.nsl, item);
    const LSlice<T> L = a.sl[j];
    if (a.active && !a.active[L.slice]) return true;
    const CUtensorMap* map_b = a.maps + 4 * j + 1;
    const CUtensorMap* map_c = a.maps + 4 * j + 2;
    const CUtensorMap* map_u = a.maps + 4 * j + a.u_map;
    const int li = int(item - a.item_start[j]);
    // consecutive items walk down one strip; the two edge strips (slower: per-cell stencils on
    // all their lanes) are handed out first, so that they do not finish last
    const int nchunks = (L.ny + a.ch - 1) / a.ch;
    const int sidx = li / nchunks;
    const int strip = L.fstrips < 2 || sidx == 0 ? sidx : (sidx == 1 ? L.fstrips - 1 : sidx - 1);
    const int chunk = li - sidx * nchunks;
    const int X0 = strip * kWaveIW - kWaveHalo;
    const int Y0 = chunk * a.ch;                  // even
    const int Y1 = min(Y0 + a.ch, L.ny);
    const int P0 = Y0 >> 1, P1 = (Y1 + 1) >> 1;   // output pairs [P0, P1)
    const int pb = P0 - HP;                       // first pair of the march
    const int te = UP ? P1 - 1 + S : P1 + S;      // last pair (each pair is loaded once)
    const int k = a.k;
    const T alpha = a.alpha, sk = a.sk;
    const int nx = L.nx, ny = L.ny;

    const int xlane = X0 + 4 * lane;
    const bool lane_in = xlane >= 0 && xlane < nx;  // X0 is a multiple of 4: all-or-none
    const bool interior_lane = lane >= kWaveHalo / 4 && lane < 32 - kWaveHalo / 4;
    StencilTab<T> tab;
    make_stencil_tab<T>(tab, k, alpha, sk);

    // Ghost strips.  A strip whose lanes are each wholly inside or wholly outside the level, and
    // whose in-level cells are all interior along x except the level's first cell (cell 0 of a
    // lane) and last cell (cell 3 of a lane) with their one-sided stencils (and for UP, there,
    // the injection from the coarse cell), runs its interior rows with the interior body too.
    // Cells outside the level are kept at exactly 0 there: their 1 / D is 0 and no coarse
    // correction is added to them (weight pm = 0; TMA fills them with 0 on every load).  A
    // boundary cell's missing neighbour then enters the interior stencil as 0, which adds
    // nothing (fma(c, 0, acc) = acc), and only its diagonal differs from the interior one: the
    // lane's iD0 / D0 or iD3 / D3 (LaneDiag), and its interpolation weight along x is 0 (wx0 /
    // wx3).  The operations and their order are those of the per-cell stencils, so the results
    // are the same bit for bit.  Every strip of a level whose width is a multiple of 4 and whose
    // coarse cells are full qualifies; others take the general body.
    const bool all_in = xlane >= 0 && xlane + 3 < nx;
    const bool all_out = xlane + 3 < 0 || xlane >= nx;
    bool ghost_ok = all_in || all_out;
    LaneDiag<T> g;
    g.iD0 = g.iD12 = g.iD3 = all_out ? T(0) : tab.ci.iD;
    g.D0 = g.D3 = tab.ci.D;
    T wx0 = T(0.25), wx3 = T(0.25);
    const T pm = all_out ? T(0) : T(1);
    if (all_in) {
        AxisCoef<T> one;
        one.w = T(1); one.gm = T(1); one.gp = T(1);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const AxisCoef<T> q = axis_coef<T>(xlane + i, nx, L.n0x, k);
            if (q.w == T(1) && q.gm == T(1) && q.gp == T(1)) continue;
            const bool first = i == 0 && xlane == 0 && q.w == T(1) && q.gm == T(0) && q.gp == T(1);
            const bool last = i == 3 && xlane + 3 == nx - 1 && q.w == T(1) && q.gm == T(1) && q.gp == T(0);
            if (!(first || last)) {
                ghost_ok = false;
                continue;
            }
            const Coef<T> c = make_coef<T>(q, one, k, alpha, sk);
            if (i == 0) { g.iD0 = c.iD; g.D0 = c.D; }
            if (i == 3) { g.iD3 = c.iD; g.D3 = c.D; }
        }
    }

    // prolongation geometry along x (UP): coarse columns cx0-1 .. cx0+2 around the lane
    const int cx0 = X0 / 2 + 2 * lane;
    const int cbox_x = X0 / 2 - 4;  // first staged coarse column (x * size stays 16-B aligned)
    const bool has_coarse = UP && L.uco != nullptr;
    T wxl[4] = {T(0), T(0), T(0), T(0)};  // weight of each cell toward its other coarse column
    if (UP) {
        // A cell's other coarse column is the previous one for even cells and the next one for
        // odd cells, or its weight is 0 (interp_axis: a cell's centre lies left of its coarse
        // cell's centre if it is the left one of two).
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (!has_coarse || xlane + i < 0 || xlane + i >= nx) continue;
            int I, J;
            interp_axis<T>(xlane + i, L.n0x, k, L.ncx, I, J, wxl[i]);
            if (wxl[i] == T(0.25)) continue;
            // weight 0 at the level's first / last cell keeps a ghost strip
            const bool edge_cell = (i == 0 && xlane == 0) || (i == 3 && xlane + 3 == nx - 1);
            if (edge_cell && wxl[i] == T(0)) {
                if (i == 0) wx0 = T(0);
                if (i == 3) wx3 = T(0);
            } else {
                ghost_ok = false;
            }
        }
    }

    {  // cache this lane's stencils for interior rows (read when the row pair is not all-interior)
        AxisCoef<T> one;
        one.w = T(1); one.gm = T(1); one.gp = T(1);
        T* cc = reinterpret_cast<T*>(ring + (coef_s - ring_s));
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const Coef<T> c = make_coef<T>(axis_coef<T>(xlane + i, nx, L.n0x, k), one, k, alpha, sk);
            cc[128 * i + 0] = c.cw;
            cc[128 * i + 1] = c.ce;
            cc[128 * i + 2] = c.cn;
            cc[128 * i + 3] = c.iD;
            cc[512 + 32 * i - 3 * lane] = c.D;
            if (UP) cc[640 + i] = wxl[i];
        }
    }
    __syncwarp();
    // TMA loads of pair P (lane 0): b (and u) rows 2P, 2P+1; coarse rows P-1 .. P+1 (UP)
    auto issue = [&](int P, int bslot, int uslot) {
        const uint32_t bar = bar_s + 8 * bslot;
        const uint32_t udst = uring_s + uslot * R::kUSlotBytes;
        const bool coarse = has_coarse && 2 * P < ny && 2 * P + 1 >= 0;
        const uint32_t bytes = R::kPairBytes + (ZERO ? 0u : (uint32_t)R::kPairBytes) +
                               (coarse ? (uint32_t)(kWaveCoarseW * 3 * sizeof(T)) : 0u);
        mbar_expect_tx(bar, bytes);
        tma_load_2d(ring_s + bslot * R::kPairBytes, map_b, X0, 2 * P, bar);
        if (!ZERO) tma_load_2d(udst, map_u, X0, 2 * P, bar);
        if (coarse) tma_load_2d(udst + (ZERO ? 0 : R::kPairBytes), map_c, cbox_x, P - 1, bar);
    };
    // the ring's slots were last read by the previous item: order those reads before the
    // copies that overwrite them
    fence_proxy_async();
    if (lane == 0)
        for (int p = 0; p < AHEAD && pb + p <= te; ++p) {
            const int b2 = bs + p, u2 = us + p;
            issue(pb + p, b2 >= NB ? b2 - NB : b2, u2 >= AHEAD ? u2 - AHEAD : u2);
        }

    T w[NR][2][4];  // window of u pairs in registers
#pragma unroll
    for (int q = 0; q < NR; ++q)
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < 4; ++i) w[q][h][i] = T(0);
    auto bslot_of = [&](int bs, int back) { const int q = bs - back; return q < 0 ? q + NB : q; };
    auto load_b = [&](int bslot, int h, T (&v)[4]) {
        lds4(ring_s + bslot * R::kPairBytes + h * kRowB + 4 * lane * (uint32_t)sizeof(T), v);
    };

    // Steps whose every updated row is an interior row run a body without range checks along y:
    // in a strip whose lanes all take the interior stencil along x (and for UP the regular
    // 1/4-3/4 prolongation pattern) one specialised to the interior stencil (FAST), in the others
    // one with the lanes' cached stencils (ROWS).  The remaining steps (the first and last rows of
    // a level) run the general body.  The choice is warp-uniform, so each step executes exactly
    // one of the three.  The first steps of a chunk, whose older pairs were never loaded, need no
    // body of their own: what they compute for those pairs only reaches the rows that the chunk's
    // halo is there for, and is not stored.
    const bool x_ghost = __all_sync(0xffffffffu, ghost_ok);

    auto step = [&](auto fast_tag, auto rows_tag, const int T_) {
        constexpr bool FAST = decltype(fast_tag)::value;
        constexpr bool ROWS = decltype(rows_tag)::value;  // FAST implies ROWS
        {
            // shift the window and bring in pair T
#pragma unroll
            for (int q = 0; q < NR - 1; ++q)
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int i = 0; i < 4; ++i) w[q][h][i] = w[q + 1][h][i];
            const uint32_t us_addr = uring_s + us * R::kUSlotBytes;
            if (ZERO) {
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int i = 0; i < 4; ++i) w[NR - 1][h][i] = T(0);
            } else {
                lds4(us_addr + 4 * lane * (uint32_t)sizeof(T), w[NR - 1][0]);
                lds4(us_addr + kRowB + 4 * lane * (uint32_t)sizeof(T), w[NR - 1][1]);
            }
            // UP: add the interpolated coarse correction to rows 2T and 2T+1
            if (has_coarse && (ROWS || (2 * T_ < ny && 2 * T_ + 1 >= 0))) {
                const uint32_t cb = us_addr + (ZERO ? 0 : R::kPairBytes);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int r = 2 * T_ + h;
                    if (!ROWS && (r < 0 || r >= ny)) continue;
                    int Iy, Jy;
                    T wy;
                    if (ROWS) {  // interior pattern along y (the step's rows are >= 2 and below the last two coarse rows)
                        Iy = T_;
                        Jy = h ? T_ + 1 : T_ - 1;
                        wy = T(0.25);
                    } else {
                        interp_axis<T>(r, L.n0y, k, L.ncy, Iy, Jy, wy);
                    }
                    // coarse row q sits at box row q - (T - 1); columns cx0-1 .. cx0+2 at 2l+3 .. 2l+6
                    const uint32_t c0 = cb + ((Iy - T_ + 1) * kWaveCoarseW + 2 * lane + 2) * (uint32_t)sizeof(T);
                    const uint32_t c1 = cb + ((Jy - T_ + 1) * kWaveCoarseW + 2 * lane + 2) * (uint32_t)sizeof(T);
                    T a0[6], a1[6];  // columns 2l+2 .. 2l+7 of the box (8-byte aligned pairs)
#pragma unroll
                    for (int m = 0; m < 6; m += 2) {
                        lds2(c0 + m * sizeof(T), a0[m], a0[m + 1]);
                        lds2(c1 + m * sizeof(T), a1[m], a1[m + 1]);
                    }
                    const T v0[4] = {a0[1], a0[2], a0[3], a0[4]};
                    const T v1[4] = {a1[1], a1[2], a1[3], a1[4]};
                    if (!FAST && !lane_in) continue;
                    T(&row)[4] = w[NR - 1][h];
                    const T q4 = T(0.25);
                    if (FAST) {
                        // interior pattern, with the ghost-strip weights (fma(1, p, u) = u + p)
                        row[0] = fma_t(pm, bilinear<T>(v0[1], v0[0], v1[1], v1[0], wx0, wy), row[0]);
                        row[1] = fma_t(pm, bilinear<T>(v0[1], v0[2], v1[1], v1[2], q4, wy), row[1]);
                        row[2] = fma_t(pm, bilinear<T>(v0[2], v0[1], v1[2], v1[1], q4, wy), row[2]);
                        row[3] = fma_t(pm, bilinear<T>(v0[2], v0[3], v1[2], v1[3], wx3, wy), row[3]);
                    } else {
                        T wv[4];
                        lds4(coef_s + 640 * (uint32_t)sizeof(T), wv);
                        row[0] = row[0] + bilinear<T>(v0[1], v0[0], v1[1], v1[0], wv[0], wy);
                        if (xlane + 1 < nx) row[1] = row[1] + bilinear<T>(v0[1], v0[2], v1[1], v1[2], wv[1], wy);
                        if (xlane + 2 < nx) row[2] = row[2] + bilinear<T>(v0[2], v0[1], v1[2], v1[1], wv[2], wy);
                        if (xlane + 3 < nx) row[3] = row[3] + bilinear<T>(v0[2], v0[3], v1[2], v1[3], wv[3], wy);
                    }
                }
            }
            // refill: pair T + AHEAD into the b slot of pair T + AHEAD - NB (no longer needed)
            // and the u/coarse slot of pair T (just consumed)
            __syncwarp();
            {
                int nbs = bs + AHEAD;
                if (nbs >= NB) nbs -= NB;
                if (lane == 0 && T_ + AHEAD <= te) issue(T_ + AHEAD, nbs, us);
            }

            // half-sweeps: stage s updates pair T - s (window slot NR-1-s) with colour (s - 1) & 1
#pragma unroll
            for (int s = 1; s <= S; ++s) {
                const int m = T_ - s;
                const int r0 = 2 * m, r1 = 2 * m + 1;
                if (!ROWS && (m < pb || r0 >= ny || r1 < 0)) continue;
                T(&p0)[4] = w[NR - 1 - s][0];
                T(&p1)[4] = w[NR - 1 - s][1];
                const T(&north)[4] = w[NR - 2 - s][1];  // row 2m - 1
                const T(&south)[4] = w[NR - s][0];      // row 2m + 2
                const int bq = bslot_of(bs, s);
                T b0[4], b1[4];
                load_b(bq, 0, b0);
                load_b(bq, 1, b1);
                const int f0 = (r0 + ((s - 1) & 1)) & 1;  // first cell of the colour on row r0
                // Row r0 updates cells {0, 2} (needs cell 3 of lane-1) when f0 == 0, else {1, 3}
                // (needs cell 0 of lane+1); row r1 the other way round.  One shuffle per row.
                const int d0 = f0 == 0 ? -1 : 1;
                const T x0 = __shfl_sync(0xffffffffu, f0 == 0 ? p0[3] : p0[0], lane + d0);
                const T x1 = __shfl_sync(0xffffffffu, f0 == 0 ? p1[0] : p1[3], lane - d0);
                const bool ir0 = ROWS || interior_row(r0, ny, k), ir1 = ROWS || interior_row(r1, ny, k);
                // warp-uniform: in a strip with edge lanes every lane reads its cached stencil
                // (an interior lane's cached stencil is the interior one), so no lane diverges
                const bool fast = FAST || (!ROWS && x_ghost && ir0 && ir1);
                sweep_row<T, FAST, ROWS>(p0, b0, north, p1, f0, x0, x0, fast, ir0, coef_s, tab, g, xlane, r0, nx, ny,
                                   L.n0x, L.n0y, k, alpha, sk);
                if (ROWS || r1 < ny)
                    sweep_row<T, FAST, ROWS>(p1, b1, p0, south, f0 ^ 1, x1, x1, fast, ir1, coef_s, tab, g, xlane, r1, nx,
                                       ny, L.n0x, L.n0y, k, alpha, sk);
            }
            // output of the pair that completed all half-sweeps
            {
                const int m = T_ - S;
                if (interior_lane && lane_in && m >= P0 && m < P1) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int r = 2 * m + h;
                        if (!ROWS && r >= Y1) continue;
                        const T(&orow)[4] = w[NR - 1 - S][h];
                        T* dst = (UP ? L.uo : L.u) + (int64_t)r * L.pitch + xlane;
                        if (FAST || xlane + 3 < nx) {
                            Vec4<T>::store(dst, orow);
                        } else {
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                if (xlane + i < nx) dst[i] = orow[i];
                        }
                    }
                }
            }
            if (!UP) {
                // residual of pair m = T - S - 1 (slot 1; neighbours in slots 0 and 2) and its
                // 2x2 restriction: rows 2m and 2m+1 form coarse row m
                const int m = T_ - S - 1;
                const T(&q0)[4] = w[1][0];
                const T(&q1)[4] = w[1][1];
                const T w0 = __shfl_up_sync(0xffffffffu, q0[3], 1);
                const T e0 = __shfl_down_sync(0xffffffffu, q0[0], 1);
                const T w1 = __shfl_up_sync(0xffffffffu, q1[3], 1);
                const T e1 = __shfl_down_sync(0xffffffffu, q1[0], 1);
                if (L.bc && m >= P0 && m < P1 && (FAST || lane_in)) {
                    const int r0 = 2 * m, r1 = 2 * m + 1;
                    const int bq = bslot_of(bs, S + 1);
                    T b0[4], b1[4];
                    load_b(bq, 0, b0);
                    load_b(bq, 1, b1);
                    const bool ir0 = ROWS || interior_row(r0, ny, k), ir1 = ROWS || interior_row(r1, ny, k);
                    const bool fast = FAST || (!ROWS && x_ghost && ir0 && ir1);
                    T res0[4], res1[4] = {T(0), T(0), T(0), T(0)};
                    residual_row<T, FAST, ROWS>(res0, q0, b0, w[0][1], q1, w0, e0, fast, ir0, coef_s, tab, g, xlane, r0,
                                          nx, ny, L.n0x, L.n0y, k, alpha, sk);
                    const bool has_r1 = ROWS || r1 < ny;
                    if (has_r1)
                        residual_row<T, FAST, ROWS>(res1, q1, b1, q0, w[2][0], w1, e1, fast, ir1, coef_s, tab, g, xlane,
                                              r1, nx, ny, L.n0x, L.n0y, k, alpha, sk);
                    // same summation order as the reference restriction: (((0 + r00) + r01) + r10) + r11
                    T c0 = T(0), c1 = T(0);
                    if (FAST || xlane + 0 < nx) c0 = c0 + res0[0];
                    if (FAST || xlane + 1 < nx) c0 = c0 + res0[1];
                    if (FAST || xlane + 2 < nx) c1 = c1 + res0[2];
                    if (FAST || xlane + 3 < nx) c1 = c1 + res0[3];
                    if (has_r1) {
                        if (FAST || xlane + 0 < nx) c0 = c0 + res1[0];
                        if (FAST || xlane + 1 < nx) c0 = c0 + res1[1];
                        if (FAST || xlane + 2 < nx) c1 = c1 + res1[2];
                        if (FAST || xlane + 3 < nx) c1 = c1 + res1[3];
                    }
                    if (interior_lane && m < L.ncy) {
                        T* dst = L.bc + (int64_t)m * L.pitchc + cx0;
                        const T v0 = c0 * T(0.25), v1 = c1 * T(0.25);
                        if (cx0 + 1 < L.ncx) Vec2<T>::store(dst, v0, v1);
                        else if (cx0 < L.ncx) dst[0] = v0;
                    }
                }
            }
        }
    };
#pragma unroll 1
    for (int T_ = pb; T_ <= te; ++T_) {
        if (!mbar_wait_warp(bar_s + 8 * bs, phase)) {
            // give up: flag the host, let the copies already issued land, leave
            if (lane == 0) atomicExch(a.err, 1);
            int b2 = bs, ph2 = phase;
            for (int tt = T_ + 1; tt <= te && tt < T_ + AHEAD; ++tt) {
                if (++b2 == NB) { b2 = 0; ph2 ^= 1; }
                mbar_wait_warp(bar_s + 8 * b2, ph2);
            }
            return false;
        }
        // The bodies without range checks along y are taken where every row the step updates
        // (pairs T - S - 1 .. T - 1) is an interior row (interior rows form one contiguous range)
        // and, for UP, the prolongation rows 2T, 2T + 1 lie in the level with the interior
        // interpolation pattern along y (coarse rows T - 1 .. T + 1 all full: T + 2 < the coarse
        // level's rows).
        const int rlo = 2 * (T_ - S - (UP ? 0 : 1)), rhi = 2 * T_ - 1;
        const bool rows = interior_row(rlo, ny, k) && interior_row(rhi, ny, k) &&
                          (!UP || (2 * T_ + 1 < ny && (!has_coarse || T_ + 2 < L.ncy)));
        if (rows && x_ghost) step(std::true_type{}, std::true_type{}, T_);
        else if (rows) step(std::false_type{}, std::true_type{}, T_);
        else step(std::false_type{}, std::false_type{}, T_);
        if (++bs == NB) { bs = 0; phase ^= 1; }
        if (++us == AHEAD) us = 0;
    }
    return true;
    };

    for (;;) {
        unsigned int item = 0;
        if (lane == 0) item = atomicAdd(a.work, 1u);
        item = __shfl_sync(0xffffffffu, item, 0);
        if ((int64_t)item >= a.nitems) break;
        if (!run_item((int64_t)item)) return;  // the host sees the error word and resets the counters
    }
    // the last warp of the launch to finish resets the counters for the next launch on this stream
    if (lane == 0) {
        const unsigned int total = gridDim.x * (unsigned int)kWaveWarps;
        if (atomicAdd(a.work + 1, 1u) == total - 1) {
            atomicExch(a.work, 0u);
            atomicExch(a.work + 1, 0u);
        }
    }
}

// ---------------------------------------------------------------- stencils of small levels
// (tile_impl.cuh, tail_warps.cuh, tail_cells.cuh)
constexpr int kTailMaxLevels = 8;  // levels of the coarse tail: 64, 32, .. 1
constexpr int kTailThreads = 512;

// One of the stencils of a level, 16-byte aligned for vector loads.
template <class T>
struct alignas(16) TailCoef {
    T cw, ce, cn, cs, iD, D, pad0, pad1;
};

template <class T>
__device__ __forceinline__ Coef<T> tail_coef(const TailCoef<T>* t) {
    Coef<T> c;
    T q[4];
    Vec4<T>::load(&t->cw, q);
    c.cw = q[0]; c.ce = q[1]; c.cn = q[2]; c.cs = q[3];
    Vec2<T>::load(&t->iD, c.iD, c.D);
    return c;
}

// Class of index i of an axis of n cells: 0 first, 1 inner (all three cells full), 2 last but one,
// 3 last; axis_coef is the same for all inner cells.
__device__ __forceinline__ int tail_class(int i, int n) {
    return i >= 1 && i + 2 < n ? 1 : (i == 0 ? 0 : (i == n - 1 ? 3 : 2));
}
// A cell of class c (if the axis has one).
__device__ __forceinline__ int tail_class_rep(int c, int n) {
    return c == 0 ? 0 : (c == 1 ? min(1, n - 1) : max(0, n - 4 + c));
}

// Stencil of a column on inner rows (iD, D) and on a full first or last row (iDb, Db), where one
// face less enters the diagonal; all 0 outside the level.
template <class T>
struct ColStencil {
    T cw, ce, cy, iD, iDb, D, Db;
};
template <class T>
__device__ __forceinline__ ColStencil<T> col_stencil(int x, int nx, int n0x, int k, T alpha, T sk) {
    ColStencil<T> c{T(0), T(0), T(0), T(0), T(0), T(0), T(0)};
    if (x < 0 || x >= nx) return c;
    const AxisCoef<T> ax = axis_coef<T>(x, nx, n0x, k);
    AxisCoef<T> ay;
    ay.w = T(1); ay.gm = T(1); ay.gp = T(1);
    const Coef<T> m = make_coef<T>(ax, ay, k, alpha, sk);
    ay.gm = T(0);
    const Coef<T> e = make_coef<T>(ax, ay, k, alpha, sk);
    c.cw = m.cw; c.ce = m.ce; c.cy = m.cn; c.iD = m.iD; c.iDb = e.iD; c.D = m.D; c.Db = e.D;
    return c;
}

// Rows: inner, first / last of full cells, outside the level, of partial cells.
enum : unsigned char { kRowInner = 0, kRowEdge = 1, kRowOut = 2, kRowPartial = 3 };
template <class T>
__device__ __forceinline__ unsigned char row_mode(int y, int ny, int n0y, int k) {
    if (y < 0 || y >= ny) return kRowOut;
    const AxisCoef<T> ay = axis_coef<T>(y, ny, n0y, k);
    const bool n1 = ay.gm == T(1), s1 = ay.gp == T(1), n0 = ay.gm == T(0), s0 = ay.gp == T(0);
    if (ay.w != T(1) || !(n0 || n1) || !(s0 || s1) || (n0 && s0)) return kRowPartial;
    return n1 && s1 ? kRowInner : kRowEdge;
}

}  // namespace fused_detail
}  // namespace emfuse
