// 3-D multigrid for the gradient-domain smoothing of the earlier method (Sec. 3 "Alternate
// Solutions": the target gradient field is the stack's gradient with its z-components set to
// zero), screened as in Eq. (1):
//     (alpha I + L_xy + L_z) f = alpha I0 + L_xy I0
// on the 6-neighbour graph of the stack (Neumann boundaries, unit spacing on every axis).  The
// paper solved this problem with a streaming multigrid; this is a multigrid on the stack held in
// HBM, the 3-D counterpart of the slice solver:
//   * correction form f = I0 + d, so the right-hand side of the correction equation is
//     alpha I0 + L_xy I0 - A I0 = -L_z I0 (z differences only), and A d = -L_z I0;
//   * cell-centred coarsening to 1 x 1 x 1 (an axis that reaches one cell stays at one), the
//     finite-volume operator of each level on its true (possibly partial) cells, face
//     coefficients 2 / (w_I + w_{I+1}) times the face area, scaled by 4^-k;
//   * restriction: the sum of the (up to 8) child residuals / 8; prolongation: trilinear
//     interpolation between true cell centres; red-black Gauss-Seidel (colour = parity of
//     x + y + z) with nu_pre / nu_post sweeps;
//   * V-cycles in FP32 on the correction equation, outer defect-correction passes: d += e,
//     r = -L_z I0 - A d, out = I0 + d, until ||r|| / ||alpha I0 + L_xy I0|| <= tol; d and A d in
//     two floats per value (48 bits, split.cuh), in FP64 for tol < 1e-7 or alpha < 1e-5.
//
// A leg of a level is one pass over memory (k3_leg: the red-black half-sweeps pipelined along z,
// with the prolongation before or the restriction after them); levels of at most kTail3 cells
// run in one CTA (k3_tail).  The host checks the residual norm after every defect pass.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include "emfuse_common.cuh"
#include "emfuse_internal.cuh"
#include "fpconv.cuh"
#include "mg_fused.cuh"
#include "split.cuh"

namespace emfuse {
namespace {

constexpr int kThreads3 = 256;

struct Lev3 {
    float* u;       // iterate of the V-cycle
    float* v;       // second iterate: a leg reads one and writes the other
    float* b;       // right-hand side
    int nx, ny, nz;
    int pitch;      // row pitch of u and b (even); v has its own
    int vpitch;
};

struct Geo3 {
    int n0x, n0y, n0z;  // finest sizes (fix the cell geometry of every level)
};

// The 7-point finite-volume stencil of level k at a cell.
struct alignas(16) Coef3 {
    float cw, ce, cn, cs, cd, cu, iD, D;
};

__device__ __forceinline__ Coef3 coef3(int x, int y, int z, int nx, int ny, int nz, const Geo3& g, int k, float alpha,
                                       float sk) {
    const AxisCoef<float> ax = axis_coef<float>(x, nx, g.n0x, k);
    const AxisCoef<float> ay = axis_coef<float>(y, ny, g.n0y, k);
    const AxisCoef<float> az = axis_coef<float>(z, nz, g.n0z, k);
    Coef3 c;
    const float ayz = ay.w * az.w, axz = ax.w * az.w, axy = ax.w * ay.w;
    c.cw = sk * (ayz * ax.gm);
    c.ce = sk * (ayz * ax.gp);
    c.cn = sk * (axz * ay.gm);
    c.cs = sk * (axz * ay.gp);
    c.cd = sk * (axy * az.gm);
    c.cu = sk * (axy * az.gp);
    c.D = fmaf(alpha, axy * az.w, ((c.cw + c.ce) + (c.cn + c.cs)) + (c.cd + c.cu));
    c.iD = 1.f / c.D;
    return c;
}

// Class of index i of an axis of n cells: 0 first, 1 inner, 2 last but one, 3 last.  axis_coef is
// the same for all inner cells, so a level has at most 4 x 4 x 4 different stencils.
__device__ __forceinline__ int class3(int i, int n) {
    return i >= 1 && i + 2 < n ? 1 : (i == 0 ? 0 : (i == n - 1 ? 3 : 2));
}
__device__ __forceinline__ int class_rep(int c, int n) {  // a cell of class c (if the axis has one)
    return c == 0 ? 0 : (c == 1 ? min(1, n - 1) : max(0, n - 4 + c));
}
// Entry t of a level's table, [class of z][class of y][class of x].
__device__ __forceinline__ Coef3 table_entry(int t, int nx, int ny, int nz, const Geo3& g, int k, float alpha, float sk) {
    return coef3(class_rep(t & 3, nx), class_rep((t >> 2) & 3, ny), class_rep(t >> 4, nz), nx, ny, nz, g, k, alpha, sk);
}

// ---------------------------------------------------------------- one leg of a level
// A CTA owns a tile of 64 x 64 cells in x and y (16 warps of 4 rows; a lane holds 2 cells of each
// row) and marches along z.  At step T plane T arrives and half-sweep s (s = 1 .. S) updates plane
// T - s: it reads the other colour of planes T - s - 1 .. T - s + 1, all of which half-sweep s - 1
// has updated, in plane T - s + 1 earlier in this step and in plane T - s in the step before.  So
// the S half-sweeps of a leg are one pass over memory, exactly S global half-sweeps, with one
// barrier per plane: neighbours along z are the thread's own registers, along x in the lane or
// one shuffle away, along y in registers or, across warps, edge rows in shared memory, written
// in one step and read in the next.  Wrong values enter at the tile's rim (no neighbours there)
// and move in by one cell per half-sweep: a halo of S cells (S + 1 under a residual) is
// recomputed by the neighbouring tiles, and likewise S planes at the ends of a chunk along z.
//
//   DOWN  optionally from zero; after the sweeps the residual, summed 2 x 2 x 2 / 8 into the next
//         level's right-hand side (where cb is given).
//   UP    the interpolated coarse correction is added as a plane arrives (where cu is given); the
//         result is stored, or added to the correction d (where d is given).
//
// The source and destination differ: tiles read their halo while neighbours write.
//
// Bound by instruction issue (about 50 per cell at S = 4, halo included; 65 % of the slots) at one CTA of
// 16 warps per SM; S = 4 keeps 6 or 7 planes in registers.  What is on its way (iterate,
// right-hand side, coarse plane, correction) goes to shared memory by asynchronous copies: prefetched
// into registers it made the UP leg spill, and the correction was read where it was needed (0.53 ms).
// 32 x 1024 x 1024: DOWN 0.25 ms, UP with the addition to d 0.36 ms; one kernel per half-sweep,
// restriction and prolongation took 0.89 and 0.84 (and 0.11 for the addition).
constexpr int kWarps3 = 16, kRows3 = 4, kTile3 = 64;

struct Leg3 {
    const float* src;      // initial iterate (not read from zero)
    float* dst;
    const float* b;
    float* cb;             // next level's right-hand side (DOWN) or null
    const float* cu;       // next level's iterate (UP) or null
    Split* d;              // UP: the correction the result is added to, instead of dst; or null
    int sp, dp, bp, cp, pitch_d;  // row pitches
    int svec, dvec;        // src / dst pairs are 8-byte aligned
    int d_first;           // d = result instead of d += result
    int nx, ny, nz, ncx, ncy, ncz;
    int k, halo, zch;      // halo in x and y (even); planes per chunk (even)
    unsigned tx, ty;       // tiles along x and y (block = (chunk * ty + tile row) * tx + tile column)
    Geo3 g;
    float alpha, sk;
};

constexpr int kCoarse3 = kRows3 / 2 + 2, kCoarseW3 = kTile3 / 2 + 2;  // coarse rows and columns of a warp

// Shared memory of a leg: right-hand sides of S + 2 (residual: S + 3) planes and two planes of the
// iterate, the ones on their way included, edge rows of S + 2 planes, and for UP a plane of the
// correction and the warps' rows of a coarse plane on their way.
template <int S, bool UP>
constexpr int leg3_smem() {
    return ((UP ? S + 6 : S + 5) * kTile3 * kTile3 + (S + 2) * kWarps3 * 2 * kTile3 +
            (UP ? kWarps3 * kCoarse3 * kCoarseW3 : 0)) * (int)sizeof(float);
}

// 8 bytes to shared memory (the last 8 - bytes of them zeros), 4 or 16 bytes; complete after copies_done().
__device__ __forceinline__ void copy8(float* to, const float* from, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"((unsigned)__cvta_generic_to_shared(to)), "l"(from),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void copy4(float* to, const float* from) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(to)), "l"(from)
                 : "memory");
}
__device__ __forceinline__ void copy16(float* to, const void* from) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(to)), "l"(from)
                 : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

constexpr int kOut3 = 8;  // "missing neighbours" of a column or row outside the level

// Missing neighbours along one axis at index i.
__device__ __forceinline__ int missing3(int i, int n) { return i < 0 || i >= n ? kOut3 : int(i == 0) + int(i == n - 1); }
// All cells of an axis of n0 fine cells are full at level k.
__device__ __forceinline__ bool full3(int n0, int k) { return (n0 & ((1 << k) - 1)) == 0; }

// b + sum_q c_pq u_q by a table entry (in shared memory).
__device__ __noinline__ float general_sum(const Coef3* q, float b, float uw, float ue, float un, float us, float ud,
                                          float uu) {
    float acc = fmaf(q->cw, uw, fmaf(q->ce, ue, b));
    acc = fmaf(q->cn, un, fmaf(q->cs, us, acc));
    return fmaf(q->cd, ud, fmaf(q->cu, uu, acc));
}

template <int S, bool ZERO, bool UP>
__global__ void __launch_bounds__(kWarps3 * 32, 1) k3_leg(const Leg3 a) {
    constexpr int NS = S + 2;                 // planes of edge rows
    constexpr int NB = UP ? S + 2 : S + 3;    // planes of right-hand sides (a residual is one plane behind)
    constexpr int NP = UP ? S + 2 : S + 3;    // planes in registers: T - NP + 1 .. T
    constexpr int R = kRows3;
    extern __shared__ __align__(16) float smem3[];
    float* const bring = smem3;                            // [NB][64][64] right-hand sides, own cells only
    float* const edge = smem3 + NB * kTile3 * kTile3;      // [NS][warp][first, last row][64]
    float* const uplane = edge + NS * kWarps3 * 2 * kTile3;  // [2][64][64] of the iterate, own cells only
    float* const dplane = uplane + 2 * kTile3 * kTile3;      // UP: [64][64] of the correction, own cells only
    float* const cplane = dplane + 2 * kTile3 * kTile3;      // UP: [warp][kCoarse3][kCoarseW3]
    __shared__ Coef3 tab[64];
    // levels of full cells: 1 / D and D of a cell with c missing neighbours, 0 for cells outside
    __shared__ float itab[kOut3 + kOut3 + 3], dtab[kOut3 + kOut3 + 3];
    __shared__ float roww[kTile3];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nx = a.nx, ny = a.ny, nz = a.nz, k = a.k;
    const int ox = kTile3 - 2 * a.halo;
    const unsigned tile = blockIdx.x / a.tx, chunk = tile / a.ty;
    const int X0 = int(blockIdx.x - tile * a.tx) * ox, Y0 = int(tile - chunk * a.ty) * ox;  // even
    const int x = X0 - a.halo + 2 * lane;                  // first of the lane's two columns (even)
    const int row0 = R * warp;
    const int y = Y0 - a.halo + row0;                      // first of the warp's rows (even)
    const int z0 = int(chunk) * a.zch, z1 = min(z0 + a.zch, nz);
    const int HZ = UP ? S : S + 1;
    const int Tb = max(0, z0 - HZ);
    const int Te = UP ? z1 - 1 + S : z1 + S;
    if (tid < 64) tab[tid] = table_entry(tid, nx, ny, nz, a.g, k, a.alpha, a.sk);
    if (tid < kOut3 + kOut3 + 3) {
        const float D = a.alpha + a.sk * float(6 - min(tid, 6));
        itab[tid] = tid < 7 ? 1.f / D : 0.f;
        dtab[tid] = tid < 7 ? D : 0.f;
    }
    if (UP && tid < kTile3) {
        const int yr = Y0 - a.halo + tid;
        float w = 0.f;
        if (a.cu && yr >= 0 && yr < ny) {
            int I, J;
            interp_axis<float>(yr, a.g.n0y, k, a.ncy, I, J, w);
        }
        roww[tid] = w;
    }
    float wx0 = 0.f, wx1 = 0.f;
    if (UP && a.cu) {
        int I, J;
        if (x >= 0 && x < nx) interp_axis<float>(x, a.g.n0x, k, a.ncx, I, J, wx0);
        if (x + 1 >= 0 && x + 1 < nx) interp_axis<float>(x + 1, a.g.n0x, k, a.ncx, I, J, wx1);
    }
    const bool col0 = x >= 0 && x < nx, col1 = x >= 0 && x + 1 < nx;  // x is even
    // Where a warp's cells are all full, the stencil is the interior one with cells outside the
    // level kept at exactly 0 (1 / D = 0): a missing neighbour adds nothing, and only the diagonal
    // differs.  Warps and planes with partial cells (the last cell of an axis, and its neighbour)
    // take the level's table, out of line.
    const bool full_z = full3(a.g.n0z, k);
    const bool full_warp = (full3(a.g.n0x, k) || X0 - a.halo + kTile3 - 1 < nx - 2) && (full3(a.g.n0y, k) || y + R - 1 < ny - 2);
    const int mx[2] = {missing3(x, nx), missing3(x + 1, nx)};
    unsigned my = 0;  // one nibble per row
#pragma unroll
    for (int r = 0; r < R; ++r) my |= (unsigned)missing3(y + r, ny) << (4 * r);
    const bool lane_out = col0 && 2 * lane >= a.halo && 2 * lane < kTile3 - a.halo;
    const int ylim = min(Y0 + ox, ny);
    unsigned rows_in = 0, rows_out = 0;  // rows of the warp in the level / among the tile's output
#pragma unroll
    for (int r = 0; r < R; ++r) {
        rows_in |= (y + r >= 0 && y + r < ny ? 1u : 0u) << r;
        rows_out |= (y + r >= Y0 && y + r < ylim ? 1u : 0u) << r;
    }

    float w[NP][R][2];
#pragma unroll
    for (int q = 0; q < NP; ++q)
#pragma unroll
        for (int r = 0; r < R; ++r) w[q][r][0] = w[q][r][1] = 0.f;
    // Plane T + 1 is on its way while plane T is worked on, by asynchronous copies: registers are short.
    // Right-hand sides of cells outside the level stay 0, of planes outside are not used.
    const int64_t first_row = (int64_t)Tb * ny + y;
    const float* bsrc = a.b + first_row * a.bp + x;     // next plane to fetch, this lane's first cell
    const float* usrc = ZERO ? nullptr : a.src + first_row * a.sp + x;
    const int64_t bstep = (int64_t)ny * a.bp, ustep = (int64_t)ny * a.sp;
    float* const own = bring + row0 * kTile3 + 2 * lane;
#pragma unroll
    for (int q = 0; q < NB; ++q)
#pragma unroll
        for (int r = 0; r < R; ++r) *reinterpret_cast<float2*>(own + (q * kTile3 + r) * kTile3) = make_float2(0.f, 0.f);
    __syncthreads();
    int bslot = Tb % NB;         // ring slot of the next plane to fetch
    auto fetch = [&](int z) {
        const bool in = z < nz && col0;
        float* const to = own + bslot * kTile3 * kTile3;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            float* const ut = uplane + (((z & 1) * kTile3 + row0 + r) * kTile3 + 2 * lane);
            if (in && (rows_in >> r & 1)) {
                copy8(to + r * kTile3, bsrc + r * a.bp, col1 ? 8 : 4);
                if (!ZERO) {
                    const float* p = usrc + r * a.sp;
                    if (a.svec) {
                        copy8(ut, p, col1 ? 8 : 4);
                    } else {
                        copy4(ut, p);
                        if (col1) copy4(ut + 1, p + 1);
                        else ut[1] = 0.f;
                    }
                }
            } else if (!ZERO) {
                *reinterpret_cast<float2*>(ut) = make_float2(0.f, 0.f);
            }
        }
        bslot = bslot + 1 == NB ? 0 : bslot + 1;
        bsrc += bstep;
        if (!ZERO) usrc += ustep;
    };
    fetch(Tb);
    // UP: coarse planes zp = (T - 1) / 2 (rounded down) in h0 and zp + 1 in h1, interpolated along x at
    // the lane's two columns, rows y/2 - 1 .. y/2 + 2; plane zp + 2 on its way in cplane, zeros outside the
    // level.  The other coarse cell of a fine cell is the previous one for even cells and the next
    // one for odd cells, or its weight is 0.
    constexpr int Q = kCoarse3;
    float h0[Q][2], h1[Q][2];
    const int cx = x >> 1, cy = y >> 1;  // arithmetic shifts: y may be negative
    float* const crow = cplane + warp * Q * kCoarseW3;  // a row: the column before the warp's, its 32, the one behind
    auto fetch_coarse = [&](int Z) {
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int Y = cy - 1 + q;
            const bool in = Z >= 0 && Z < a.ncz && Y >= 0 && Y < a.ncy;
            const float* p = a.cu + ((int64_t)Z * a.ncy + Y) * a.cp;
            float* to = crow + q * kCoarseW3 + 1 + lane;
            if (in && cx >= 0 && cx < a.ncx) copy4(to, p + cx);
            else *to = 0.f;
            if (lane == 0 || lane == 31) {
                const int e = lane == 0 ? -1 : 1;
                if (in && cx + e >= 0 && cx + e < a.ncx) copy4(to + e, p + (cx + e));
                else to[e] = 0.f;
            }
        }
    };
    auto take_coarse = [&](float (&h)[Q][2]) {
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const float* from = crow + q * kCoarseW3 + 1 + lane;
            const float v = from[0];
            h[q][0] = fmaf(wx0, from[-1] - v, v);
            h[q][1] = fmaf(wx1, from[1] - v, v);
        }
    };
    if (UP && a.cu) {
        const int zp = (Tb >> 1) - 1;  // Tb is even
        fetch_coarse(zp);
        copies_done();
        __syncthreads();
        take_coarse(h0);
        __syncthreads();
        fetch_coarse(zp + 1);
        copies_done();
        __syncthreads();
        take_coarse(h1);
    }
    const int64_t out_row = (int64_t)z0 * ny + y;  // next output plane, this lane's first cell
    float* odst = a.dst + out_row * a.dp + x;
    Split* odst_d = a.d + out_row * a.pitch_d + x;
    const int64_t ostep = (int64_t)ny * a.dp, ostep_d = (int64_t)ny * a.pitch_d;
    float part[2] = {0.f, 0.f};  // restriction: the even plane's 2 x 2 sums of the two coarse rows
    int slot = Tb % NS;          // ring slot of plane T (edge rows)
    auto slot_of = [&](int back) { const int q = slot - back; return q < 0 ? q + NS : q; };
    int slot_b = Tb % NB;        // ring slot of plane T (right-hand sides)
    auto rhs_of = [&](int back) { const int q = slot_b - back; return own + (q < 0 ? q + NB : q) * kTile3 * kTile3; };
    // UP: plane z of the correction on its way to dplane
    auto fetch_d = [&](int z) {
        if (a.d && !a.d_first && lane_out && z >= z0 && z < z1) {
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (rows_out >> r & 1) copy16(dplane + ((row0 + r) * (kTile3 / 2) + lane) * 4, odst_d + r * a.pitch_d);
        }
    };
    auto edge_at = [&](int sl, int wr, int which) { return edge + ((sl * kWarps3 + wr) * 2 + which) * kTile3 + 2 * lane; };

#pragma unroll 1
    for (int T = Tb; T <= Te; ++T) {
        copies_done();    // a thread reads only what it copied itself
        __syncthreads();  // edge rows of the last step are visible, those of the oldest plane are free
#pragma unroll
        for (int q = 0; q + 1 < NP; ++q)
#pragma unroll
            for (int r = 0; r < R; ++r) {
                w[q][r][0] = w[q + 1][r][0];
                w[q][r][1] = w[q + 1][r][1];
            }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            float2 t = make_float2(0.f, 0.f);
            if (!ZERO) t = *reinterpret_cast<const float2*>(uplane + (((T & 1) * kTile3 + row0 + r) * kTile3 + 2 * lane));
            w[NP - 1][r][0] = t.x;
            w[NP - 1][r][1] = t.y;
        }
        if (T < Te) fetch(T + 1);
        if (UP) fetch_d(T - S);
        if (UP && a.cu && T < nz) {
            if ((T & 1) && T > Tb) {  // planes (T - 1) / 2 and the next one
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    h0[q][0] = h1[q][0];
                    h0[q][1] = h1[q][1];
                }
                take_coarse(h1);
            }
            if ((T & 1) == 0) fetch_coarse((T >> 1) + 1);  // a barrier after the last reads of cplane
            int Iz, Jz;
            float wz;
            interp_axis<float>(T, a.g.n0z, k, a.ncz, Iz, Jz, wz);
            if ((T & 1) == 0) wz = 1.f - wz;  // weight of h1: T's own coarse plane is h1 for even T
            float h[Q][2];
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                h[q][0] = fmaf(wz, h1[q][0] - h0[q][0], h0[q][0]);
                h[q][1] = fmaf(wz, h1[q][1] - h0[q][1], h0[q][1]);
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (!(rows_in >> r & 1)) continue;
                const float wy = roww[row0 + r];
                const int q0 = r / 2 + 1, q1 = (r & 1) ? q0 + 1 : q0 - 1;
                if (col0) w[NP - 1][r][0] += fmaf(wy, h[q1][0] - h[q0][0], h[q0][0]);
                if (col1) w[NP - 1][r][1] += fmaf(wy, h[q1][1] - h[q0][1], h[q0][1]);
            }
        }
        if (S > 0 || !UP) {
            *reinterpret_cast<float2*>(edge_at(slot, warp, 0)) = make_float2(w[NP - 1][0][0], w[NP - 1][0][1]);
            *reinterpret_cast<float2*>(edge_at(slot, warp, 1)) = make_float2(w[NP - 1][R - 1][0], w[NP - 1][R - 1][1]);
        }
        // half-sweep s of plane T - s: colour (s - 1) & 1 of x + y + z; with x and y even for cell 0 of
        // row 0, that row's cell is I0 = (s - 1 + z) & 1 and every second row's the other
        // (BODY 0: full cells, inner rows; 1: full cells; 2: partial cells)
        auto half_sweep = [&](auto stage_tag, auto i_tag, auto body_tag, int m) {
            constexpr int s = decltype(stage_tag)::value, I0 = decltype(i_tag)::value;
            constexpr int BODY = decltype(body_tag)::value;
            constexpr int P = NP - 1 - s;
            const int sl = slot_of(s);
            const float no = warp > 0 ? edge_at(sl, warp - 1, 1)[I0] : 0.f;
            constexpr int IL = (I0 + R - 1) & 1;
            const float so = warp + 1 < kWarps3 ? edge_at(sl, warp + 1, 0)[IL] : 0.f;
            const int mz = int(m == 0) + int(m == nz - 1);
            float iD[2] = {0.f, 0.f};
            if (BODY == 0) {
                iD[0] = itab[mx[0] + mz];
                iD[1] = itab[mx[1] + mz];
            }
            const float* bp = rhs_of(s);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int i = (I0 + r) & 1;
                float(&u)[2] = w[P][r];
                const float o = i == 0 ? __shfl_up_sync(0xffffffffu, u[1], 1) : __shfl_down_sync(0xffffffffu, u[0], 1);
                const float uw = i == 0 ? o : u[0], ue = i == 0 ? u[1] : o;
                const float un = r > 0 ? w[P][r > 0 ? r - 1 : 0][i] : no;
                const float us = r + 1 < R ? w[P][r + 1 < R ? r + 1 : 0][i] : so;
                const float ud = w[P - 1][r][i], uu = w[P + 1][r][i];
                const float bv = bp[r * kTile3 + i];
                if (BODY < 2) {
                    const float acc = fmaf(a.sk, ((uw + ue) + (un + us)) + (ud + uu), bv);
                    u[i] = acc * (BODY == 0 ? iD[i] : itab[mx[i] + int(my >> (4 * r) & 15u) + mz]);
                } else if ((i == 0 ? col0 : col1) && (rows_in >> r & 1)) {
                    const Coef3* q = tab + class3(m, nz) * 16 + class3(y + r, ny) * 4 + class3(x + i, nx);
                    u[i] = general_sum(q, bv, uw, ue, un, us, ud, uu) * q->iD;
                }
                if (r == 0) edge_at(sl, warp, 0)[i] = u[i];
                if (r == R - 1) edge_at(sl, warp, 1)[i] = u[i];
            }
        };
        auto stage = [&](auto stage_tag) {
            constexpr int s = decltype(stage_tag)::value;
            const int m = T - s;
            if (m < Tb || m >= nz) return;
            const bool full = full_warp && (full_z || m + 2 < nz);
            auto run = [&](auto i_tag) {
                if (full && my == 0) half_sweep(stage_tag, i_tag, std::integral_constant<int, 0>{}, m);
                else if (full) half_sweep(stage_tag, i_tag, std::integral_constant<int, 1>{}, m);
                else half_sweep(stage_tag, i_tag, std::integral_constant<int, 2>{}, m);
            };
            if (((s - 1 + m) & 1) == 0) run(std::integral_constant<int, 0>{});
            else run(std::integral_constant<int, 1>{});
        };
        if constexpr (S >= 1) stage(std::integral_constant<int, 1>{});
        if constexpr (S >= 2) stage(std::integral_constant<int, 2>{});
        if constexpr (S >= 3) stage(std::integral_constant<int, 3>{});
        if constexpr (S >= 4) stage(std::integral_constant<int, 4>{});
        {   // the plane that completed all half-sweeps
            const int m = T - S;
            const bool mine = m >= z0 && m < z1;
            if (UP && a.d && !a.d_first) copies_done();
            if (mine && lane_out) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if (!(rows_out >> r & 1)) continue;
                    const float v0 = w[NP - 1 - S][r][0], v1 = w[NP - 1 - S][r][1];
                    if (UP && a.d) {
                        Split* q = odst_d + r * a.pitch_d;  // 16-byte aligned, the padding included
                        Split e[2] = {{v0, 0.f}, {v1, 0.f}};
                        if (!a.d_first) {
                            const float4 t =
                                *reinterpret_cast<const float4*>(dplane + ((row0 + r) * (kTile3 / 2) + lane) * 4);
                            e[0] = split_add(Split{t.x, t.y}, v0);
                            e[1] = split_add(Split{t.z, t.w}, v1);
                        }
                        *reinterpret_cast<float4*>(q) = make_float4(e[0].hi, e[0].lo, e[1].hi, e[1].lo);
                    } else {
                        float* q = odst + r * a.dp;
                        if (a.dvec) {
                            *reinterpret_cast<float2*>(q) = make_float2(v0, v1);
                        } else {
                            q[0] = v0;
                            if (col1) q[1] = v1;
                        }
                    }
                }
            }
            if (mine) {
                odst += ostep;
                if (UP) odst_d += ostep_d;
            }
        }
        if (!UP && a.cb) {
            const int m = T - S - 1;
            if (m >= z0 && m < z1) {
                const int sl = slot_of(S + 1);
                const float* bp = rhs_of(S + 1);
                float2 no = make_float2(0.f, 0.f), so = no;
                if (warp > 0) no = *reinterpret_cast<const float2*>(edge_at(sl, warp - 1, 1));
                if (warp + 1 < kWarps3) so = *reinterpret_cast<const float2*>(edge_at(sl, warp + 1, 0));
                const bool full = full_warp && (full_z || m + 2 < nz);
                const int mz = int(m == 0) + int(m == nz - 1);
                float sum[R / 2];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    constexpr int P = UP ? 1 : NP - 2 - S;  // plane T - S - 1 (never used for UP)
                    const float2 bv = *reinterpret_cast<const float2*>(bp + r * kTile3);
                    const float u0 = w[P][r][0], u1 = w[P][r][1];
                    const float uw = __shfl_up_sync(0xffffffffu, u1, 1), ue = __shfl_down_sync(0xffffffffu, u0, 1);
                    const float n0 = r > 0 ? w[P][r > 0 ? r - 1 : 0][0] : no.x, n1 = r > 0 ? w[P][r > 0 ? r - 1 : 0][1] : no.y;
                    const float s0 = r + 1 < R ? w[P][r + 1 < R ? r + 1 : 0][0] : so.x;
                    const float s1 = r + 1 < R ? w[P][r + 1 < R ? r + 1 : 0][1] : so.y;
                    const float d0 = w[P - 1][r][0], d1 = w[P - 1][r][1], t0 = w[P + 1][r][0], t1 = w[P + 1][r][1];
                    float res = 0.f;
                    if (full) {
                        const float q0 = fmaf(a.sk, ((uw + u1) + (n0 + s0)) + (d0 + t0), bv.x);
                        const float q1 = fmaf(a.sk, ((u0 + ue) + (n1 + s1)) + (d1 + t1), bv.y);
                        const int c = int(my >> (4 * r) & 15u) + mz;
                        if (mx[0] + c < 7) res = fmaf(-dtab[mx[0] + c], u0, q0);
                        if (mx[1] + c < 7) res += fmaf(-dtab[mx[1] + c], u1, q1);
                    } else if (rows_in >> r & 1) {
                        const Coef3* t = tab + class3(m, nz) * 16 + class3(y + r, ny) * 4;
                        if (col0) {
                            const Coef3* q = t + class3(x, nx);
                            res = fmaf(-q->D, u0, general_sum(q, bv.x, uw, u1, n0, s0, d0, t0));
                        }
                        if (col1) {
                            const Coef3* q = t + class3(x + 1, nx);
                            res += fmaf(-q->D, u1, general_sum(q, bv.y, u0, ue, n1, s1, d1, t1));
                        }
                    }
                    sum[r / 2] = (r & 1) ? sum[r / 2] + res : res;
                }
#pragma unroll
                for (int q = 0; q < R / 2; ++q) {
                    if ((m & 1) == 0) part[q] = sum[q];
                    else part[q] += sum[q];
                    const int yy = y + 2 * q;
                    if (((m & 1) || m == nz - 1) && lane_out && (rows_out >> (2 * q) & 1))
                        a.cb[((int64_t)(m >> 1) * a.ncy + (yy >> 1)) * a.cp + (x >> 1)] = part[q] * 0.125f;
                }
            }
        }
        if (++slot == NS) slot = 0;
        if (++slot_b == NB) slot_b = 0;
    }
}

// ---------------------------------------------------------------- the small levels
// Levels kt .. of at most kTail3 cells on copies in shared memory, one CTA: the rest of the
// V-cycle in one launch (bound by the latency of its passes, one barrier each).
constexpr int kTail3 = 8192, kTailThreads3 = 1024, kTailLevels3 = 14;

struct Tail3 {
    const float* b;   // right-hand side of level kt (dense rows of `pitch`)
    float* u;         // its iterate: read if cont, written at the end
    int pitch, nx, ny, nz, kt, nlev;
    int nu_pre, nu_post, cont;
    Geo3 g;
    float alpha;
};

// Division by a small number known at run time: exact for 0 <= p, d < 2^16.
struct SmallDiv {
    unsigned d, m;
    __device__ __forceinline__ explicit SmallDiv(int v) : d(v), m(v == 1 ? 0u : 0xffffffffu / (unsigned)v + 1u) {}
    __device__ __forceinline__ int of(int p) const { return d == 1 ? p : (int)__umulhi((unsigned)p, m); }
};

struct TailLev3 {
    float *u, *b;
    const Coef3* tab;
    const float *wx, *wy, *wz;  // interpolation weights toward the other coarse cell (see k3_leg)
    int nx, ny, nz;
};

// Cell p of the half-lattice of one colour (p over ceil(nx / 2) x ny x nz); false past the row's end.
__device__ __forceinline__ bool tail3_cell(const TailLev3& L, const SmallDiv& dx, const SmallDiv& dy, int p, int colour,
                                           int& x, int& y, int& z) {
    const int hx = (L.nx + 1) >> 1;
    const int row = dx.of(p);
    z = dy.of(row);
    y = row - z * L.ny;
    x = 2 * (p - row * hx) + ((y + z + colour) & 1);
    return x < L.nx;
}

__device__ __forceinline__ float tail3_sum(const TailLev3& L, const Coef3& c, int p, int x, int y, int z, float b) {
    const int sy = L.nx, sz = L.nx * L.ny;
    float acc = b;
    if (x > 0) acc = fmaf(c.cw, L.u[p - 1], acc);
    if (x + 1 < L.nx) acc = fmaf(c.ce, L.u[p + 1], acc);
    if (y > 0) acc = fmaf(c.cn, L.u[p - sy], acc);
    if (y + 1 < L.ny) acc = fmaf(c.cs, L.u[p + sy], acc);
    if (z > 0) acc = fmaf(c.cd, L.u[p - sz], acc);
    if (z + 1 < L.nz) acc = fmaf(c.cu, L.u[p + sz], acc);
    return acc;
}

__device__ __forceinline__ const Coef3& tail3_coef(const TailLev3& L, int x, int y, int z) {
    return L.tab[class3(z, L.nz) * 16 + class3(y, L.ny) * 4 + class3(x, L.nx)];
}

__device__ __forceinline__ void tail3_relax(const TailLev3& L, int half_sweeps) {
    const int n = ((L.nx + 1) >> 1) * L.ny * L.nz;
    const SmallDiv dx((L.nx + 1) >> 1), dy(L.ny);
    for (int h = 0; h < half_sweeps; ++h) {
        for (int q = threadIdx.x; q < n; q += kTailThreads3) {
            int x, y, z;
            if (!tail3_cell(L, dx, dy, q, h & 1, x, y, z)) continue;
            const int p = (z * L.ny + y) * L.nx + x;
            const Coef3& c = tail3_coef(L, x, y, z);
            L.u[p] = tail3_sum(L, c, p, x, y, z, L.b[p]) * c.iD;
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kTailThreads3) k3_tail(const Tail3 a) {
    extern __shared__ __align__(16) float smem3[];
    __shared__ int off[kTailLevels3 + 1], woff[kTailLevels3 + 1];
    Coef3* const tabs = reinterpret_cast<Coef3*>(smem3);  // 64 per level
    float* const base = smem3 + a.nlev * 64 * (int)(sizeof(Coef3) / sizeof(float));
    const int tid = threadIdx.x;
    auto size = [&](int n0, int q) { return level_size(n0, a.kt + q); };
    if (tid == 0) {
        int o = 0, wo = 0;
        for (int q = 0; q < a.nlev; ++q) {
            off[q] = o;
            woff[q] = wo;
            o += 2 * size(a.g.n0x, q) * size(a.g.n0y, q) * size(a.g.n0z, q);
            wo += size(a.g.n0x, q) + size(a.g.n0y, q) + size(a.g.n0z, q);
        }
        off[a.nlev] = o;
        woff[a.nlev] = wo;
    }
    for (int t = tid; t < 64 * a.nlev; t += kTailThreads3) {
        const int q = t >> 6, k = a.kt + q;
        tabs[t] = table_entry(t & 63, size(a.g.n0x, q), size(a.g.n0y, q), size(a.g.n0z, q), a.g, k, a.alpha,
                              ldexpf(1.f, -2 * k));
    }
    __syncthreads();
    auto view = [&](int q) {
        TailLev3 L;
        L.nx = size(a.g.n0x, q);
        L.ny = size(a.g.n0y, q);
        L.nz = size(a.g.n0z, q);
        L.u = base + off[q];
        L.b = L.u + L.nx * L.ny * L.nz;
        L.tab = tabs + 64 * q;
        L.wx = base + off[a.nlev] + woff[q];
        L.wy = L.wx + L.nx;
        L.wz = L.wy + L.ny;
        return L;
    };
    for (int p = tid; p < off[a.nlev]; p += kTailThreads3) base[p] = 0.f;
    for (int q = 0; q + 1 < a.nlev; ++q) {
        const TailLev3 L = view(q), C = view(q + 1);
        for (int p = tid; p < L.nx + L.ny + L.nz; p += kTailThreads3) {
            const int ax = p < L.nx ? 0 : (p < L.nx + L.ny ? 1 : 2);
            const int i = ax == 0 ? p : (ax == 1 ? p - L.nx : p - L.nx - L.ny);
            int I, J;
            float w;
            interp_axis<float>(i, ax == 0 ? a.g.n0x : (ax == 1 ? a.g.n0y : a.g.n0z), a.kt + q,
                               ax == 0 ? C.nx : (ax == 1 ? C.ny : C.nz), I, J, w);
            base[off[a.nlev] + woff[q] + p] = w;
        }
    }
    __syncthreads();
    {
        const TailLev3 L = view(0);
        for (int p = tid; p < L.nx * L.ny * L.nz; p += kTailThreads3) {
            const int row = p / L.nx;
            const int64_t g = (int64_t)row * a.pitch + (p - row * L.nx);
            L.b[p] = a.b[g];
            if (a.cont) L.u[p] = a.u[g];
        }
        __syncthreads();
    }
    for (int q = 0; q + 1 < a.nlev; ++q) {
        const TailLev3 L = view(q), C = view(q + 1);
        tail3_relax(L, 2 * a.nu_pre);
        const SmallDiv dx(C.nx), dy(C.ny);
        for (int p = tid; p < C.nx * C.ny * C.nz; p += kTailThreads3) {
            const int row = dx.of(p), X = p - row * C.nx, Z = dy.of(row), Y = row - Z * C.ny;
            float sum = 0.f;
            for (int o = 0; o < 8; ++o) {
                const int x = 2 * X + (o & 1), y = 2 * Y + ((o >> 1) & 1), z = 2 * Z + (o >> 2);
                if (x >= L.nx || y >= L.ny || z >= L.nz) continue;
                const int f = (z * L.ny + y) * L.nx + x;
                const Coef3& c = tail3_coef(L, x, y, z);
                sum += fmaf(-c.D, L.u[f], tail3_sum(L, c, f, x, y, z, L.b[f]));
            }
            C.b[p] = sum * 0.125f;
        }
        __syncthreads();
    }
    tail3_relax(view(a.nlev - 1), 1);  // 1 x 1 x 1: one half-sweep solves it
    for (int q = a.nlev - 2; q >= 0; --q) {
        const TailLev3 L = view(q), C = view(q + 1);
        const SmallDiv dx(L.nx), dy(L.ny);
        for (int p = tid; p < L.nx * L.ny * L.nz; p += kTailThreads3) {
            const int row = dx.of(p), x = p - row * L.nx, z = dy.of(row), y = row - z * L.ny;
            const float wx = L.wx[x], wy = L.wy[y], wz = L.wz[z];
            auto other = [](int i, float w2) { return w2 == 0.f ? i >> 1 : ((i & 1) ? (i >> 1) + 1 : (i >> 1) - 1); };
            const int Ix = x >> 1, Iy = y >> 1, Iz = z >> 1;
            const int Jx = other(x, wx), Jy = other(y, wy), Jz = other(z, wz);
            const float* u0 = C.u + Iz * C.ny * C.nx;
            const float* u1 = C.u + Jz * C.ny * C.nx;
            const float e = bilinear<float>(u0[Iy * C.nx + Ix], u0[Iy * C.nx + Jx], u0[Jy * C.nx + Ix], u0[Jy * C.nx + Jx],
                                            wx, wy);
            const float f = bilinear<float>(u1[Iy * C.nx + Ix], u1[Iy * C.nx + Jx], u1[Jy * C.nx + Ix], u1[Jy * C.nx + Jx],
                                            wx, wy);
            L.u[p] += fmaf(wz, f - e, e);
        }
        __syncthreads();
        tail3_relax(L, 2 * a.nu_post);
    }
    const TailLev3 L = view(0);
    for (int p = tid; p < L.nx * L.ny * L.nz; p += kTailThreads3) {
        const int row = p / L.nx;
        a.u[(int64_t)row * a.pitch + (p - row * L.nx)] = L.u[p];
    }
}

// Block sum of two doubles into sums[0], sums[1] (shuffle tree, one atomic per block).
__device__ __forceinline__ void block_sum2(double a, double b, double* sums) {
    __shared__ double red[2][kThreads3 / 32];
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, m);
        b += __shfl_xor_sync(0xffffffffu, b, m);
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) { red[0][w] = a; red[1][w] = b; }
    __syncthreads();
    if (w == 0) {
        a = l < kThreads3 / 32 ? red[0][l] : 0.0;
        b = l < kThreads3 / 32 ? red[1][l] : 0.0;
#pragma unroll
        for (int m = 4; m > 0; m >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, m);
            b += __shfl_xor_sync(0xffffffffu, b, m);
        }
        if (l == 0) {
            atomicAdd(&sums[0], a);
            if (b != 0.0) atomicAdd(&sums[1], b);  // only the first pass has the second sum
        }
    }
}

// d += e (or d = e where `first`), e = the level-0 result of the last V-cycle, over the padded rows.
template <class D>
__global__ void __launch_bounds__(kThreads3) k3_update(D* __restrict__ d, const float* __restrict__ e, int64_t n,
                                                       int first) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        if constexpr (sizeof(D) == sizeof(Split) && !std::is_same<D, double>::value)
            d[t] = first ? Split{e[t], 0.f} : split_add(d[t], e[t]);
        else
            d[t] = (first ? 0.0 : d[t]) + f2d_ieee(e[t]);
    }
}

// Defect pass on the finest level: r = -L_z I0 - A d (A = alpha I + L, 7-point, Neumann), out =
// I0 + d; r goes to the level-0 right-hand side (FP32).  sums[0] += ||r||^2; with FIRST (d = 0, not
// read) also sums[1] += ||alpha I0 + L_xy I0||^2.  Three forms of d: Split (two floats, tolerances
// from 1e-7 and alpha from 1e-5): A d carries the rounding errors of its sums and product and is rounded once to FP32
// before it is taken from the FP32-formed -L_z I0 (exact for 8-bit input; its own rounding bounds
// what more bits could add there); double with everything in FP64, -L_z I0 and the subtraction
// included (smaller tolerances, where that rounding would cap the reachable residual).
//
// A thread marches along z over a chunk of kDefectZ planes of one pixel column, so that the
// neighbours along z stay in registers; those along y and x are L1 hits of a 32 x 8 tile.  A block takes
// `per` such items, several where the stack has few planes: with one each, the sums' atomics
// bounded the pass (a call on 1 x 2048 x 2048: 168 us, now 95).  Bound
// by instruction issue (about 145 per cell): 32 x 1024 x 1024, a pass 509 -> 201 us against FP64
// evaluation (bound by that pipe).  The norms' conversions on the integer units: 223 us with the
// hardware's, which go to the FP64 pipe.
constexpr int kDefectZ = 16;

template <class D>
struct Adeg3 {
    D v[7];  // alpha + q, q = 0..6 (the diagonal of A for a cell with q neighbours)
};

template <class D>
__device__ __forceinline__ D at_degree3(const Adeg3<D>& t, int q) {
    return q == 6 ? t.v[6] : q == 5 ? t.v[5] : q == 4 ? t.v[4] : q == 3 ? t.v[3] : q == 2 ? t.v[2] : q == 1 ? t.v[1] : t.v[0];
}

// a c - (sum of the six neighbours), rounded once to binary32 (see split_apply of split.cuh).
__device__ __forceinline__ float split_apply7(Split a, Split c, Split w, Split e, Split n, Split s, Split d, Split u) {
    float s1, e1, s2, e2, s3, e3, s4, e4, s5, e5;
    two_sum(w.hi, e.hi, s1, e1);
    two_sum(n.hi, s.hi, s2, e2);
    two_sum(d.hi, u.hi, s3, e3);
    two_sum(s1, s2, s4, e4);
    two_sum(s4, s3, s5, e5);
    const float lo = (((w.lo + e.lo) + (n.lo + s.lo)) + (d.lo + u.lo)) + (((e1 + e2) + (e3 + e4)) + e5);
    return split_finish(a, c, s5, lo);
}

template <class Tin, class D, bool FIRST>
__global__ void __launch_bounds__(kThreads3) k3_defect(const Tin* __restrict__ I0, const D* __restrict__ d,
                                                       float* __restrict__ r0, float* __restrict__ out, int nx, int ny,
                                                       int nz, int pitch, unsigned items, unsigned per, float alpha,
                                                       Adeg3<D> adeg, double* __restrict__ sums) {
    constexpr bool SPLIT = std::is_same<D, Split>::value;
    const unsigned tx = (unsigned)((nx - 1) / 32 + 1), ty = (unsigned)((ny - 1) / 8 + 1);
    const unsigned end = min((blockIdx.x + 1) * per, items);
    double rr = 0.0, bb = 0.0;
    for (unsigned item = blockIdx.x * per; item < end; ++item) {
        const unsigned tile = item / tx, chunk = tile / ty;
        const int x = int(item - tile * tx) * 32 + (threadIdx.x & 31);
        const int y = int(tile - chunk * ty) * 8 + (threadIdx.x >> 5), zc = int(chunk) * kDefectZ;
        if (x >= nx || y >= ny) continue;
        const int64_t sz = (int64_t)nx * ny, pz = (int64_t)pitch * ny;
        int64_t t = ((int64_t)zc * ny + y) * nx + x, q = ((int64_t)zc * ny + y) * pitch + x;
        const bool hw = x > 0, he = x + 1 < nx, hn = y > 0, hs = y + 1 < ny;
        const int degxy = int(hw) + int(he) + int(hn) + int(hs);
        float im = zc > 0 ? (float)I0[t - sz] : 0.f, ip = (float)I0[t];
        D dm{}, dp{};
        if (!FIRST) {
            if (zc > 0) dm = d[q - pz];
            dp = d[q];
        }
        const int ze = min(zc + kDefectZ, nz);
        for (int z = zc; z < ze; ++z, t += sz, q += pz) {
            const bool hd = z > 0, hu = z + 1 < nz;
            const float in = hu ? (float)I0[t + sz] : 0.f;
            // -L_z I0: the z neighbours minus the cell
            float rhs = 0.f;
            if (hd) rhs += im - ip;
            if (hu) rhs += in - ip;
            float r = rhs, o = ip;
            if (!FIRST) {
                const D zero{};
                const D dn = hu ? d[q + pz] : zero;
                const D w = hw ? d[q - 1] : zero, e = he ? d[q + 1] : zero;
                const D n = hn ? d[q - pitch] : zero, s = hs ? d[q + pitch] : zero;
                const D a = at_degree3(adeg, degxy + int(hd) + int(hu));
                if constexpr (SPLIT) {
                    r = rhs - split_apply7(a, dp, w, e, n, s, dm, dn);
                    o = ip + dp.hi;
                } else {
                    const double id = f2d_ieee(ip);
                    double rd = 0.0;
                    if (hd) rd += f2d_ieee(im) - id;
                    if (hu) rd += f2d_ieee(in) - id;
                    rd -= fma(a, dp, -((((w + e) + n) + s) + (dm + dn)));
                    r = d2f_ieee(rd);
                    rr = fma(rd, rd, rr);
                    o = ip + d2f_ieee(dp);
                }
                dm = dp;
                dp = dn;
            } else {
                float lxy = 0.f;  // L_xy I0
                if (hw) lxy += ip - (float)I0[t - 1];
                if (he) lxy += ip - (float)I0[t + 1];
                if (hn) lxy += ip - (float)I0[t - nx];
                if (hs) lxy += ip - (float)I0[t + nx];
                const float b = fmaf(alpha, ip, lxy);
                const double bd = f2d_ieee(b);
                bb = fma(bd, bd, bb);
            }
            // squares in FP64: in FP32 they leave its range (1e-23, 1e19) long before r and b do
            if (SPLIT || FIRST) {
                const double rd = f2d_ieee(r);
                rr = fma(rd, rd, rr);
            }
            r0[q] = r;
            out[t] = o;
            im = ip;
            ip = in;
        }
    }
    block_sum2(rr, bb, sums);
}

unsigned grid_for(int64_t n) {
    const int64_t blocks = (n + kThreads3 - 1) / kThreads3;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(blocks, (int64_t)kNumSMs * 16));
}

}  // namespace

namespace {

// Sweeps of the kernels of one leg: an odd number of passes of at most two sweeps each (a leg
// reads one iterate buffer and ends in the other; see gd_multigrid).
std::vector<int> leg_sweeps(int nu) {
    int n = std::max(1, (nu + 1) / 2);
    if (n % 2 == 0) ++n;
    std::vector<int> v(n, 1);
    if (nu == 0) v[0] = 0;
    for (int i = 0; i < nu - n; ++i) v[i] = 2;
    return v;
}

template <int S, bool ZERO, bool UP>
int launch_leg3_one(const Leg3& a, dim3 grid, cudaStream_t st) {
    static std::mutex mu;
    static bool done[64] = {false};
    int dev = 0;
    EMF_CUDA(cudaGetDevice(&dev));
    if (dev >= 0 && dev < 64) {
        std::lock_guard<std::mutex> lk(mu);
        if (!done[dev]) {
            EMF_CUDA(cudaFuncSetAttribute(k3_leg<S, ZERO, UP>, cudaFuncAttributeMaxDynamicSharedMemorySize, leg3_smem<S, UP>()));
            done[dev] = true;
        }
    }
    k3_leg<S, ZERO, UP><<<grid, kWarps3 * 32, leg3_smem<S, UP>(), st>>>(a);
    EMF_CHECK_LAUNCH();
    return EMFUSE_OK;
}

template <int S>
int launch_leg3_s(const Leg3& a, bool zero, bool up, dim3 grid, cudaStream_t st) {
    if (up) return launch_leg3_one<S, false, true>(a, grid, st);
    if (zero) return launch_leg3_one<S, true, false>(a, grid, st);
    return launch_leg3_one<S, false, false>(a, grid, st);
}

// One pass of `sweeps` sweeps (0, 1 or 2) over a level.
int launch_leg3(Leg3 a, int sweeps, bool zero, bool up, const char* name, double bytes, cudaStream_t st) {
    const int halo = 2 * sweeps + (a.cb ? 1 : 0);
    a.halo = (halo + 1) / 2 * 2;
    const int ox = kTile3 - 2 * a.halo;
    const int64_t tx = ceil_div(a.nx, ox), ty = ceil_div(a.ny, ox);
    // one chunk along z, unless the tiles leave SMs idle: then chunks of at least 8 planes (each
    // end of a chunk recomputes 2 * sweeps planes)
    const int64_t chunks = std::max<int64_t>(1, std::min<int64_t>(kNumSMs / (tx * ty), a.nz / 8));
    a.zch = (int)round_up(ceil_div(a.nz, chunks), 2);
    const int64_t cz = ceil_div(a.nz, a.zch);
    a.tx = (unsigned)tx;
    a.ty = (unsigned)ty;
    const dim3 grid((unsigned)(tx * ty * cz));
    KernelScope ks(name, st, bytes);
    switch (sweeps) {
        case 0: return launch_leg3_s<0>(a, zero, up, grid, st);
        case 1: return launch_leg3_s<2>(a, zero, up, grid, st);
        default: return launch_leg3_s<4>(a, zero, up, grid, st);
    }
}

// cells and sides: summed over the tail's levels
int launch_tail3(const Tail3& a, size_t cells, size_t sides, cudaStream_t st) {
    const int smem = a.nlev * 64 * (int)sizeof(Coef3) + (int)((2 * cells + sides) * sizeof(float));
    static std::mutex mu;
    static int set[64] = {0};
    int dev = 0;
    EMF_CUDA(cudaGetDevice(&dev));
    if (dev >= 0 && dev < 64) {
        std::lock_guard<std::mutex> lk(mu);
        if (set[dev] < smem) {
            EMF_CUDA(cudaFuncSetAttribute(k3_tail, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
            set[dev] = smem;
        }
    }
    KernelScope ks("gd3_tail", st, 8.0 * (double)cells);
    k3_tail<<<1, kTailThreads3, smem, st>>>(a);
    EMF_CHECK_LAUNCH();
    return EMFUSE_OK;
}

}  // namespace

int gd_multigrid(const void* in, int dt, float* out, int64_t nx, int64_t ny, int64_t nz, double alpha,
                 const emfuse_solve_opts& opts, emfuse_slice_stats* stats, cudaStream_t st) {
    // levels: ceil halving per axis down to 1 x 1 x 1
    std::vector<Lev3> lev;
    for (int k = 0;; ++k) {
        Lev3 L{};
        L.nx = level_size((int)nx, k);
        L.ny = level_size((int)ny, k);
        L.nz = level_size((int)nz, k);
        L.pitch = (int)round_up(L.nx, 2);
        lev.push_back(L);
        if (L.nx == 1 && L.ny == 1 && L.nz == 1) break;
    }
    const int nlev = (int)lev.size();
    auto padded = [&](int k) { return (size_t)lev[k].pitch * lev[k].ny * lev[k].nz; };
    auto cells = [&](int k) { return (size_t)lev[k].nx * lev[k].ny * lev[k].nz; };
    int kt = 0;  // first level of the tail kernel
    while (cells(kt) > (size_t)kTail3) ++kt;
    size_t tail_cells = 0, tail_sides = 0, all = 0;
    for (int k = 0; k < nlev; ++k) {
        all += padded(k);
        if (k >= kt) {
            tail_cells += cells(k);
            tail_sides += (size_t)lev[k].nx + lev[k].ny + lev[k].nz;
        }
    }
    const size_t coarse = all - padded(0), n0p = padded(0);
    // d and A d in two floats, unless the tolerance or alpha asks for more: 48 bits of 6 + alpha hold alpha
    // itself to 2^-46 / alpha, which reaches d's smooth part as that share of it.  Root-mean-square error of
    // 24 x 300 x 301 (0 .. 255) at tol 1e-6, d in FP64 with A d rounded to FP32 / two floats: alpha = 1e-4 1.4e-4 /
    // 1.4e-4, 1e-5 2.1e-4 / 1.5e-4, 1e-6 1.7e-4 / 6.0e-4.
    const bool split = opts.tol >= 1e-7 && alpha >= 1e-5;
    // Iterate buffers.  A leg reads one buffer and ends in the other: DOWN u -> v (from u only when
    // a V-cycle continues from the last one), UP v -> u.  The finest level's v is the caller's
    // `out`, which every defect pass rewrites; and between its two legs the finest level's u is
    // free and holds the v of the coarse levels.
    DeviceBuffer ub, bbuf, dbuf, sums;
    EMF_TRY(ub.alloc((std::max(n0p, coarse) + coarse) * sizeof(float), st));
    EMF_TRY(bbuf.alloc(all * sizeof(float), st));
    EMF_TRY(dbuf.alloc(n0p * sizeof(double), st));
    EMF_TRY(sums.alloc(2 * sizeof(double), st));
    {
        float *u = ub.as<float>() + std::max(n0p, coarse), *v = ub.as<float>(), *b = bbuf.as<float>();
        for (int k = 0; k < nlev; ++k) {
            lev[k].b = b;
            b += padded(k);
            lev[k].u = k == 0 ? ub.as<float>() : u;
            lev[k].v = k == 0 ? out : v;
            lev[k].vpitch = k == 0 ? (int)nx : lev[k].pitch;
            if (k > 0) {
                u += padded(k);
                v += padded(k);
            }
        }
    }
    const Geo3 g{(int)nx, (int)ny, (int)nz};
    const float af = (float)alpha;
    void* const d = dbuf.as<void>();

    double hs[2] = {0.0, 0.0};
    auto defect = [&](bool first) -> int {
        EMF_CUDA(cudaMemsetAsync(sums.as<double>(), 0, 2 * sizeof(double), st));
        {
            const double n0 = (double)nx * ny * nz;
            KernelScope ks("gd3_defect", st, n0 * ((dt == EMFUSE_U8 ? 1.0 : 4.0) + (first ? 0.0 : 8.0) + 8.0),
                           first || split ? 0.0 : n0 * 8.0);
            const unsigned items = (unsigned)(ceil_div(nx, 32) * ceil_div(ny, 8) * ceil_div(nz, kDefectZ));
            const unsigned per = (unsigned)std::max<int64_t>(1, kDefectZ / nz);
            const unsigned grid = (items - 1) / per + 1;
            auto run = [&](auto tin, auto dd, auto first_tag) {
                using Tin = decltype(tin);
                using D = decltype(dd);
                Adeg3<D> adeg;
                for (int q = 0; q <= 6; ++q) {
                    const double v = alpha + (double)q;
                    if constexpr (std::is_same<D, Split>::value) {
                        adeg.v[q].hi = (float)v;
                        adeg.v[q].lo = (float)(v - (double)adeg.v[q].hi);
                    } else {
                        adeg.v[q] = v;
                    }
                }
                k3_defect<Tin, D, decltype(first_tag)::value><<<grid, kThreads3, 0, st>>>(
                    (const Tin*)in, (const D*)d, lev[0].b, out, (int)nx, (int)ny, (int)nz, lev[0].pitch, items, per, af, adeg,
                    sums.as<double>());
            };
            auto run_d = [&](auto tin) {
                if (first) run(tin, Split{}, std::true_type{});
                else if (split) run(tin, Split{}, std::false_type{});
                else run(tin, 0.0, std::false_type{});
            };
            if (dt == EMFUSE_U8) run_d(uint8_t{});
            else run_d(float{});
            EMF_CHECK_LAUNCH();
        }
        EMF_CUDA(cudaMemcpyAsync(hs, sums.as<double>(), 2 * sizeof(double), cudaMemcpyDeviceToHost, st));
        EMF_CUDA(cudaStreamSynchronize(st));
        return EMFUSE_OK;
    };
    auto vec = [](const float* p, int pitch) { return pitch % 2 == 0 && (reinterpret_cast<uintptr_t>(p) & 7) == 0 ? 1 : 0; };
    const std::vector<int> dn = leg_sweeps(opts.nu_pre), up = leg_sweeps(opts.nu_post);
    // One V-cycle from zero or (cont) from the last result; `add`: the result is added to d (or
    // becomes it, d_first) instead of staying in lev[0].u.
    auto vcycle = [&](bool cont, bool add, bool d_first) -> int {
        auto leg = [&](int k) {
            const Lev3& F = lev[k];
            Leg3 a{};
            a.b = F.b;
            a.bp = F.pitch;
            a.nx = F.nx;
            a.ny = F.ny;
            a.nz = F.nz;
            a.k = k;
            a.g = g;
            a.alpha = af;
            a.sk = std::ldexp(1.f, -2 * k);
            if (k + 1 < nlev) {
                a.ncx = lev[k + 1].nx;
                a.ncy = lev[k + 1].ny;
                a.ncz = lev[k + 1].nz;
                a.cp = lev[k + 1].pitch;
            }
            return a;
        };
        // pass i of a leg: odd passes u -> v (DOWN) or v -> u (UP), the others back
        auto buffers = [&](Leg3& a, int k, bool from_u) {
            const Lev3& F = lev[k];
            a.src = from_u ? F.u : F.v;
            a.sp = from_u ? F.pitch : F.vpitch;
            a.dst = from_u ? F.v : F.u;
            a.dp = from_u ? F.vpitch : F.pitch;
            a.svec = vec(a.src, a.sp);
            a.dvec = vec(a.dst, a.dp);
        };
        for (int k = 0; k < kt; ++k) {
            for (size_t i = 0; i < dn.size(); ++i) {
                Leg3 a = leg(k);
                buffers(a, k, i % 2 == 0);
                const bool zero = i == 0 && !(cont && k == 0), last = i + 1 == dn.size();
                if (last) a.cb = lev[k + 1].b;
                EMF_TRY(launch_leg3(a, dn[i], zero, false, k == 0 ? "gd3_down_l0" : "gd3_down",
                                    (double)cells(k) * ((zero ? 8.0 : 12.0) + (last ? 0.5 : 0.0)), st));
            }
        }
        {
            Tail3 t{};
            t.b = lev[kt].b;
            t.u = lev[kt].u;
            t.pitch = lev[kt].pitch;
            t.nx = lev[kt].nx;
            t.ny = lev[kt].ny;
            t.nz = lev[kt].nz;
            t.kt = kt;
            t.nlev = nlev - kt;
            t.nu_pre = opts.nu_pre;
            t.nu_post = opts.nu_post;
            t.cont = cont && kt == 0;
            t.g = g;
            t.alpha = af;
            EMF_TRY(launch_tail3(t, tail_cells, tail_sides, st));
        }
        for (int k = kt - 1; k >= 0; --k)
            for (size_t i = 0; i < up.size(); ++i) {
                Leg3 a = leg(k);
                buffers(a, k, i % 2 != 0);
                if (i == 0) a.cu = lev[k + 1].u;
                if (k == 0 && add && split && i + 1 == up.size()) {
                    a.d = (Split*)d;
                    a.pitch_d = lev[0].pitch;
                    a.d_first = d_first;
                }
                EMF_TRY(launch_leg3(a, up[i], false, true, k == 0 ? "gd3_up_l0" : "gd3_up",
                                    (double)cells(k) * (8.0 + (a.d ? (d_first ? 8.0 : 16.0) : 4.0) + (i == 0 ? 0.5 : 0.0)),
                                    st));
            }
        if (add && (kt == 0 || !split)) {
            KernelScope ks("gd3_update", st, (double)n0p * (d_first ? 12.0 : 20.0));
            if (split) k3_update<Split><<<grid_for((int64_t)n0p), kThreads3, 0, st>>>((Split*)d, lev[0].u, (int64_t)n0p, d_first);
            else k3_update<double><<<grid_for((int64_t)n0p), kThreads3, 0, st>>>((double*)d, lev[0].u, (int64_t)n0p, d_first);
            EMF_CHECK_LAUNCH();
        }
        return EMFUSE_OK;
    };

    // relative residual; a NaN or Inf anywhere in the input makes a norm non-finite
    auto relres = [&](double bnorm) {
        if (!std::isfinite(hs[0]) || !std::isfinite(bnorm)) return std::nan("");
        return bnorm > 0.0 ? std::sqrt(hs[0]) / bnorm : (hs[0] > 0.0 ? HUGE_VAL : 0.0);
    };
    EMF_TRY(defect(true));
    const double bnorm = std::sqrt(hs[1]);
    double rel = relres(bnorm);
    int v = 0;
    bool finite = std::isfinite(rel);
    while (finite && rel > opts.tol && v < opts.max_vcycles) {
        // before the first defect pass, further FP32 V-cycles continue from the last iterate (their
        // fine residual is formed in FP32 inside the cycle), as in the slice solver
        const bool first = v == 0;
        const int n = first ? std::max(1, std::min(opts.first_vcycles, opts.max_vcycles)) : 1;
        for (int i = 0; i < n; ++i, ++v) EMF_TRY(vcycle(i > 0, i + 1 == n, first));
        EMF_TRY(defect(false));
        rel = relres(bnorm);
        finite = std::isfinite(rel);
    }
    if (stats) {
        stats->vcycles = v;
        stats->converged = finite && rel <= opts.tol ? 1 : 0;
        stats->rel_residual = rel;
        stats->b_norm = bnorm;
        stats->rel_residual_check = -1.0;
    }
    if (!finite) {
        set_error("emfuse_smooth_gradient_domain_mg: non-finite residual (NaN or Inf in the input?)");
        return EMFUSE_EINVAL;
    }
    if (rel > opts.tol) {
        set_error("emfuse_smooth_gradient_domain_mg: tolerance not reached within max_vcycles");
        return EMFUSE_ENOCONV;
    }
    return EMFUSE_OK;
}

}  // namespace emfuse
