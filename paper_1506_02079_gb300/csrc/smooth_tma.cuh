// The TMA-staged smoothing kernel (see smooth.cu for what the smoothing is and which kernel runs
// when), instantiated in smooth.cu for stacks whose rows TMA can read and in smooth_packed.cu for
// packed copies of stacks whose rows it cannot.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include <mutex>

#include "emfuse_common.cuh"
#include "tma.cuh"

namespace emfuse {
namespace smooth_detail {

constexpr int kTX = 64;   // tile width (outputs)
constexpr int kTY = 16;   // tile height (outputs)
constexpr int kThreads = 256;
constexpr int kMaxRxy = 8;

struct SmoothParams {
    float wxy[2 * kMaxRxy + 1];  // taps w(d), d = -Rxy..Rxy
    float wz[19];                // wz[j] = w(Rz - j), j = 0..2Rz (zero beyond)
    int Rxy, Rz;
    float kappa2;                // robust averaging: squared threshold in standard deviations
};

// Robust z-average of one voxel (Sec. 3, the outlier example: only values within kappa
// weighted standard deviations of the window's weighted mean are averaged).  v[j] are the
// xy-smoothed window values, w[j] their tap weights (0 for taps outside the stack).
template <int P>
__device__ __forceinline__ float robust_window(const float (&v)[P], const float (&w)[P], float kappa2) {
    float W = 0.f, m = 0.f;
#pragma unroll
    for (int j = 0; j < P; ++j) {
        W += w[j];
        m = fmaf(w[j], v[j], m);
    }
    const float mu = m / W;
    float s2 = 0.f;
#pragma unroll
    for (int j = 0; j < P; ++j) {
        const float dv = v[j] - mu;
        s2 = fmaf(w[j] * dv, dv, s2);
    }
    const float thr = kappa2 * (s2 / W);
    float sk = 0.f, wk = 0.f;
#pragma unroll
    for (int j = 0; j < P; ++j) {
        const float dv = v[j] - mu;
        const float wj = dv * dv <= thr ? w[j] : 0.f;
        wk += wj;
        sk = fmaf(wj, v[j], sk);
    }
    return sk / wk;
}

// One launch of the kernel.
struct SmoothTmaCall {
    CUtensorMap map;
    float* out;
    int nx, ny, nz;
    int64_t pitch;
    int z0, z1;
    const float *inv_x, *inv_y, *inv_z;
    SmoothParams prm;
    int ybase, yend;  // output rows
    int ymap, zmap;   // first row and plane of the map
    int* err;
};

// The kernel in smooth_fused_kernel's arithmetic (smooth_packed.cu), 1 <= prm.Rxy <= 4 and
// 1 <= prm.Rz <= 9.
int smooth_tma_packed(const SmoothTmaCall& c, int dt, bool robust, cudaStream_t st);

// ---------------------------------------------------------------- TMA-staged kernel
// Shared-memory layout of the TMA kernel for input type Tin and xy radius R.
template <class Tin, int R>
struct SmTile {
    static constexpr int HX = sizeof(Tin) == 1 ? 16 : 4;   // staged columns left of the tile: the
                                                          // copy's x-start stays 16-byte aligned
    static constexpr int HXR = sizeof(Tin) == 1 ? 16 : 8;  // right: a float row of 76 words is
                                                          // 304 B, so 8 consecutive rows start in
                                                          // 8 different 16-B bank groups
    static constexpr int BX = kTX + HX + HXR;
    static constexpr int BY = kTY + 2 * R;
    static constexpr int kPlaneBytes = BX * BY * (int)sizeof(Tin);
    static constexpr int kPlaneStride = (kPlaneBytes + 127) / 128 * 128;  // TMA destinations 128-B aligned
    // plane buffers, all in flight except the one being blurred (about 64 KiB of copies in
    // flight per SM with two CTAs per SM for float input)
    static constexpr int NBUF = sizeof(Tin) == 1 ? 8 : 5;
    static constexpr int SXW = kTX + 4;                    // x-blurred row stride (words): 272 B,
                                                          // 8 rows -> 8 different bank groups
    static constexpr int kRowBlocks = (BY + 7) / 8;        // x-blur items: 8 rows x 8 groups each
    static constexpr int kXItems = 64 * kRowBlocks;        // <= 256 for R <= 4
    static constexpr int kSmemBytes = NBUF * kPlaneStride + 2 * BY * SXW * 4 + NBUF * 8;
};

// 16 consecutive staged values (as float) starting at p.
template <class Tin>
__device__ __forceinline__ void load16(const Tin* p, float (&s)[16]);
template <>
__device__ __forceinline__ void load16<float>(const float* p, float (&s)[16]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float4 q = reinterpret_cast<const float4*>(p)[k];
        s[4 * k] = q.x; s[4 * k + 1] = q.y; s[4 * k + 2] = q.z; s[4 * k + 3] = q.w;
    }
}
template <>
__device__ __forceinline__ void load16<uint8_t>(const uint8_t* p, float (&s)[16]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uchar4 q = reinterpret_cast<const uchar4*>(p)[k];
        s[4 * k] = q.x; s[4 * k + 1] = q.y; s[4 * k + 2] = q.z; s[4 * k + 3] = q.w;
    }
}

// One HBM pass of the separable smoothing.  A CTA owns a 64 x 16 xy-tile and marches along z.
// Per input plane (arriving by TMA into a ring of NBUF shared-memory buffers, zero-filled
// outside the stack):
//   x blur   items of 8 outputs on one staged row (rows tile + y halo), written to one of two
//            x-blurred planes; 8 consecutive lanes take 8 rows, so the vector loads and
//            stores of a quarter-warp fall in distinct banks;
//   barrier  the only one per plane: the x-blurred plane is complete, the staged buffer is
//            free and is refilled with the plane NBUF ahead;
//   y blur   each thread 2 columns x 2 rows into a register ring of the last 19 planes;
//   z blur   the plane Rz behind is emitted from the ring, scaled by the product of the three
//            inverse normalisers.
// The taps are kernel parameters with compile-time indices, i.e. constant-bank operands of the
// FMAs.  With SCALED the blurs along x and y are scaled by their inverse normalisers as they are
// formed, with P taps along z: the operations of smooth_fused_kernel in its order, so the results
// are the same bit for bit.  Without, one scale by the product at the end and P = 19: results
// agree with the other implementations to rounding.  Bound by latency at 16 warps per SM: 65 % of the issue
// slots, FMA pipe 36 %, DRAM 30 % (16 x 2048 x 2048 float, 0.21 ms); the per-plane barrier and the shared-memory
// loads behind it are the stalls that work of other planes could hide.  ROB instances are at the cap of 128
// registers and spill 108 to 124 bytes.  The tensor map may hold a slab of the stack
// (rows from ymap, planes from zmap); output rows are ybase .. yend - 1.
template <class Tin, int R, bool ROB, bool SCALED, int P>
__global__ void __launch_bounds__(kThreads, 2)
smooth_tma_kernel(const __grid_constant__ CUtensorMap map, float* __restrict__ out, int nx, int ny, int nz,
                  int64_t pitch, int z0, int z1, const float* __restrict__ inv_nx,
                  const float* __restrict__ inv_ny, const float* __restrict__ inv_nz, SmoothParams prm,
                  int ybase, int yend, int ymap, int zmap, int* __restrict__ err) {
    using G = SmTile<Tin, R>;
    constexpr int NB = G::NBUF;
    extern __shared__ __align__(128) unsigned char smem[];
    unsigned char* s_raw = smem;
    float* s_x = reinterpret_cast<float*>(smem + NB * G::kPlaneStride);  // [2][BY][SXW]
    uint64_t* s_bar = reinterpret_cast<uint64_t*>(smem + NB * G::kPlaneStride + 2 * G::BY * G::SXW * 4);
    const int tid = threadIdx.x;
    __shared__ __align__(16) float s_ix[SCALED ? kTX : 4];  // inverse normalisers of the columns
    const int x0 = blockIdx.x * kTX, y0 = ybase + blockIdx.y * kTY;
    if (SCALED && tid < kTX) s_ix[tid] = inv_nx[min(x0 + tid, nx - 1)];
    const int Rz = prm.Rz;
    const int zin_lo = max(0, z0 - Rz), zin_hi = min(nz, z1 + Rz), zi_end = z1 + Rz;
    const uint32_t bar0 = smem_addr(&s_bar[0]);
    if (tid == 0) {
        for (int q = 0; q < NB; ++q) mbar_init(bar0 + 8 * q, 1);
        mbar_init_fence();
    }
    __syncthreads();
    // thread 0: plane zi into buffer slot (zi - zin_lo) mod NB; a slot is refilled only after
    // the barrier that ended the x blur of the plane it held
    auto issue = [&](int zi, int slot) {
        fence_proxy_async();
        mbar_expect_tx(bar0 + 8 * slot, G::kPlaneBytes);
        tma_load_3d(smem_addr(s_raw + slot * G::kPlaneStride), &map, x0 - G::HX, y0 - R - ymap, zi - zmap, bar0 + 8 * slot);
    };
    if (tid == 0)
        for (int q = 0; q < NB && zin_lo + q < zin_hi; ++q) issue(zin_lo + q, q);

    // x-blur item of this thread (warp-uniform participation: kXItems is a multiple of 64)
    const bool xw = tid < G::kXItems;
    const int xr = (tid >> 6) * 8 + (tid & 7);  // staged row
    const int xg = (tid >> 3) & 7;              // group of 8 output columns
    const bool xitem = xw && xr < G::BY;
    const Tin* const s_in0 = reinterpret_cast<const Tin*>(s_raw) + xr * G::BX + 8 * xg + G::HX - 4;
    float* const sx_item = s_x + xr * G::SXW + 8 * xg;
    // y/z outputs of this thread: columns 2 lane, 2 lane + 1 of rows 2 warp, 2 warp + 1
    const int lane = tid & 31, wrp = tid >> 5;
    const int gx = x0 + 2 * lane;
    const int gy0 = y0 + 2 * wrp, gy1 = gy0 + 1;
    const float* const sy_col = s_x + (2 * wrp) * G::SXW + 2 * lane;
    // inv_x * inv_y of the 4 outputs (row 0 x, row 0 x+1, row 1 x, row 1 x+1); SCALED: inv_y
    float sxy[4];
    if (SCALED) {
        sxy[0] = sxy[1] = inv_ny[min(gy0, ny - 1)];
        sxy[2] = sxy[3] = inv_ny[min(gy1, ny - 1)];
    } else {
        const float ix0 = inv_nx[min(gx, nx - 1)], ix1 = inv_nx[min(gx + 1, nx - 1)];
        const float iy0 = inv_ny[min(gy0, ny - 1)], iy1 = inv_ny[min(gy1, ny - 1)];
        sxy[0] = ix0 * iy0; sxy[1] = ix1 * iy0; sxy[2] = ix0 * iy1; sxy[3] = ix1 * iy1;
    }
    const bool st0 = gy0 < yend, st1 = gy1 < yend;
    const bool vec2 = (pitch & 1) == 0 && (reinterpret_cast<uintptr_t>(out) & 7) == 0 && gx + 1 < nx;
    float* const dst0 = out + (int64_t)min(gy0, ny - 1) * pitch + gx;
    float* const dst1 = out + (int64_t)min(gy1, ny - 1) * pitch + gx;

    // z ring: slots 0 .. P-2 hold the P-1 planes before the current block of U planes, slots
    // P-1 .. P-2+U the block; the ring moves by U slots once per block (the loop over a block is
    // unrolled, so every slot index is a constant)
    constexpr int U = ROB ? 2 : 4;  // the robust window needs more registers of its own
    float ring[P - 1 + U][4];
#pragma unroll
    for (int q = 0; q < P - 1 + U; ++q)
#pragma unroll
        for (int c = 0; c < 4; ++c) ring[q][c] = 0.f;
    const int64_t plane = pitch * (int64_t)ny;

    int slot = 0;        // buffer slot of plane zi
    uint32_t phase = 0;  // barrier parity of the current lap over the slots
    int buf = 0;         // x-blurred plane buffer (0 or 1)
#pragma unroll 1
    for (int zb = zin_lo; zb < zi_end; zb += U) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int zi = zb + u;
            float v[4] = {0.f, 0.f, 0.f, 0.f};
            if (zi < zin_hi) {  // uniform across the CTA
                bool ok = true;
                const int boff = buf * (G::BY * G::SXW);
                if (xw) {
                    ok = mbar_wait_warp(bar0 + 8 * slot, phase);
                    if (ok && xitem) {
                        float s[16];
                        load16<Tin>(s_in0 + slot * (G::kPlaneStride / (int)sizeof(Tin)), s);
                        // output i sits at s[4 + i]
                        float o[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            float acc = prm.wxy[0] * s[4 + i - R];
#pragma unroll
                            for (int d = -R + 1; d <= R; ++d) acc = fmaf(prm.wxy[d + R], s[4 + i + d], acc);
                            o[i] = acc;
                        }
                        if (SCALED) {
                            float q[8];
                            *reinterpret_cast<float4*>(q) = *reinterpret_cast<const float4*>(s_ix + 8 * xg);
                            *reinterpret_cast<float4*>(q + 4) = *reinterpret_cast<const float4*>(s_ix + 8 * xg + 4);
#pragma unroll
                            for (int i = 0; i < 8; ++i) o[i] *= q[i];
                        }
                        float4* dst = reinterpret_cast<float4*>(sx_item + boff);
                        dst[0] = make_float4(o[0], o[1], o[2], o[3]);
                        dst[1] = make_float4(o[4], o[5], o[6], o[7]);
                    }
                }
                if (!__syncthreads_and(ok)) {
                    // give up: flag the host, let the copies in flight land, leave
                    if (tid == 0) {
                        atomicExch(err, 1);
                        for (int zz = zi; zz < zin_hi && zz < zi + NB; ++zz) {
                            const int k = zz - zin_lo;
                            const uint32_t b = bar0 + 8 * (k % NB), ph = (uint32_t)((k / NB) & 1);
                            for (int it = 0; it < kWaitLimit; ++it)
                                if (mbar_try_wait(b, ph)) break;
                        }
                    }
                    __syncthreads();
                    return;
                }
                if (tid == 0 && zi + NB < zin_hi) issue(zi + NB, slot);
                // y blur of rows 2 warp, 2 warp + 1 (x-blurred rows 2 warp .. 2 warp + 2R + 1)
#pragma unroll
                for (int t = 0; t <= 2 * R + 1; ++t) {
                    const float2 q = *reinterpret_cast<const float2*>(sy_col + boff + t * G::SXW);
                    if (t == 0) {
                        v[0] = prm.wxy[0] * q.x;
                        v[1] = prm.wxy[0] * q.y;
                    } else if (t <= 2 * R) {
                        v[0] = fmaf(prm.wxy[t], q.x, v[0]);
                        v[1] = fmaf(prm.wxy[t], q.y, v[1]);
                    }
                    if (t == 1) {
                        v[2] = prm.wxy[0] * q.x;
                        v[3] = prm.wxy[0] * q.y;
                    } else if (t >= 2) {
                        v[2] = fmaf(prm.wxy[t - 1], q.x, v[2]);
                        v[3] = fmaf(prm.wxy[t - 1], q.y, v[3]);
                    }
                }
                if (R == 0) {  // 2R + 1 = 1 row per output
                    const float2 q = *reinterpret_cast<const float2*>(sy_col + boff + G::SXW);
                    v[2] = prm.wxy[0] * q.x;
                    v[3] = prm.wxy[0] * q.y;
                }
                if (SCALED) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) v[c] *= sxy[c];
                }
                if (++slot == NB) { slot = 0; phase ^= 1u; }
                buf ^= 1;
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) ring[P - 1 + u][c] = v[c];
            // emit plane zi - Rz from ring slots u .. u + P - 1 (slot u + P - 1 = plane zi)
            const int zo = zi - Rz;
            if (zo >= z0 && zo < z1) {  // uniform across the CTA
                float o[4];
                if constexpr (ROB) {
                    float wv[P];
#pragma unroll
                    for (int jj = 0; jj < P; ++jj) wv[jj] = (zi - jj >= 0 && zi - jj < nz) ? prm.wz[jj] : 0.f;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        float vv[P];
#pragma unroll
                        for (int jj = 0; jj < P; ++jj) vv[jj] = ring[u + P - 1 - jj][c];
                        o[c] = robust_window<P>(vv, wv, prm.kappa2);
                        if (!SCALED) o[c] *= sxy[c];
                    }
                } else {
                    const float inz = inv_nz[zo];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        float acc = prm.wz[0] * ring[u + P - 1][c];
#pragma unroll
                        for (int jj = 1; jj < P; ++jj) acc = fmaf(prm.wz[jj], ring[u + P - 1 - jj][c], acc);
                        o[c] = acc * (SCALED ? inz : sxy[c] * inz);
                    }
                }
                const int64_t zoff = (int64_t)(zo - z0) * plane;
                if (vec2) {
                    if (st0) *reinterpret_cast<float2*>(dst0 + zoff) = make_float2(o[0], o[1]);
                    if (st1) *reinterpret_cast<float2*>(dst1 + zoff) = make_float2(o[2], o[3]);
                } else {
                    if (st0 && gx < nx) dst0[zoff] = o[0];
                    if (st0 && gx + 1 < nx) dst0[zoff + 1] = o[1];
                    if (st1 && gx < nx) dst1[zoff] = o[2];
                    if (st1 && gx + 1 < nx) dst1[zoff + 1] = o[3];
                }
            }
        }
#pragma unroll
        for (int q = 0; q < P - 1; ++q)
#pragma unroll
            for (int c = 0; c < 4; ++c) ring[q][c] = ring[q + U][c];
    }
}

// Opt in to the kernel's dynamic shared memory once per instantiation and device, and launch.
template <class Tin, int R, bool ROB, bool SCALED, int P>
int smooth_tma_launch(const SmoothTmaCall& c, cudaStream_t st) {
    static std::mutex mu;
    static bool done[64] = {false};
    int dev = 0;
    EMF_CUDA(cudaGetDevice(&dev));
    auto* kernel = smooth_tma_kernel<Tin, R, ROB, SCALED, P>;
    constexpr int smem = SmTile<Tin, R>::kSmemBytes;
    if (dev >= 0 && dev < 64) {
        std::lock_guard<std::mutex> lk(mu);
        if (!done[dev]) {
            EMF_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
            done[dev] = true;
        }
    }
    const dim3 grid((unsigned)ceil_div(c.nx, kTX), (unsigned)ceil_div(c.yend - c.ybase, kTY));
    kernel<<<grid, kThreads, smem, st>>>(c.map, c.out, c.nx, c.ny, c.nz, c.pitch, c.z0, c.z1, c.inv_x, c.inv_y, c.inv_z,
                                         c.prm, c.ybase, c.yend, c.ymap, c.zmap, c.err);
    EMF_CHECK_LAUNCH();
    return EMFUSE_OK;
}

}  // namespace smooth_detail
}  // namespace emfuse
