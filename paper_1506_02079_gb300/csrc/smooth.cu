// Phase 1 of the method: anisotropic Gaussian smoothing I1 = I0 * G_{sigma_xy, sigma_z}
// (Sec. 3 "Anisotropic Smoothing"), with the Gaussian cut off beyond three standard deviations
// (Sec. 3 "Implementation") and the weights renormalised over the taps inside the stack.
//
// Three implementations:
//   * smooth_tma_kernel (default): one HBM pass.  A CTA owns a 64x16 xy-tile and marches
//     along z.  Input planes (tile plus xy halo) arrive by TMA bulk tensor copies into a ring of
//     shared-memory buffers, all but one in flight while a plane is blurred; the hardware
//     zero-fills the halo outside the stack.  x blur in items of 8 outputs, one barrier per
//     plane, y blur of 2 x 2 outputs per thread, then a 19-plane register ring along z (moved
//     once per block of planes, so the march stays a small rolled loop).  Needs rows whose
//     byte pitch is a multiple of 16; others are packed to such a pitch first.
//   * smooth_fused_kernel: the same data flow with plain loads, for any pitch.
//     Each input plane is staged in shared memory with its xy halo, blurred in x then y,
//     and pushed into a per-thread ring of the last P planes held in registers; the z-blur of
//     the plane R behind is emitted from the ring.  The ring index is a compile-time constant
//     (the z loop is unrolled by the ring period P), so the ring never leaves registers.
//     Reads I0 once (plus L2-resident halo) and writes I1 once.
//   * axis_x_kernel, axis_yz_kernel: one renormalised 1-D pass along an axis with optional pre/post
//     scaling.  Used for large supports, for the transpose K^T and for dK/dsigma_z in the
//     adjoint, and as an independent cross-check of the fused kernel.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include "emfuse_common.cuh"
#include "emfuse_internal.cuh"
#include "smooth_tma.cuh"
#include "tma.cuh"

namespace emfuse {

namespace {

using namespace smooth_detail;

template <class Tin>
__device__ __forceinline__ float load_in(const Tin* p) { return float(*p); }

template <class Tin, int P, bool ROB>
__global__ void __launch_bounds__(kThreads, 2)
smooth_fused_kernel(const Tin* __restrict__ in, float* __restrict__ out, int nx, int ny, int nz,
                    int64_t pitch, int z0, int z1, const float* __restrict__ inv_nx,
                    const float* __restrict__ inv_ny, const float* __restrict__ inv_nz,
                    SmoothParams prm) {
    constexpr int MAXH = kTY + 2 * kMaxRxy;
    __shared__ float s_in[MAXH][kTX + 2 * kMaxRxy + 1];
    __shared__ float s_x[MAXH][kTX];

    const int R = prm.Rxy;
    const int Rz = prm.Rz;
    const int x0 = blockIdx.x * kTX;
    const int y0 = blockIdx.y * kTY;
    const int tid = threadIdx.x;
    const int tx = tid % 16;  // 4 consecutive x per thread
    const int ty = tid / 16;  // one row per thread
    const int W = kTX + 2 * R;
    const int H = kTY + 2 * R;
    const int64_t plane = pitch * (int64_t)ny;

    float ring[P][4];
#pragma unroll
    for (int q = 0; q < P; ++q)
#pragma unroll
        for (int i = 0; i < 4; ++i) ring[q][i] = 0.f;

    // input planes that influence outputs [z0, z1)
    const int zin_lo = max(0, z0 - Rz);
    const int zin_hi = min(nz, z1 + Rz);  // exclusive
    // zi runs from zin_lo to z1 - 1 + Rz; output zo = zi - Rz
    const int zi_end = z1 + Rz;

    for (int zb = zin_lo; zb < zi_end; zb += P) {
#pragma unroll
        for (int q = 0; q < P; ++q) {
            const int zi = zb + q;
            if (zi >= zi_end) break;  // uniform across the CTA
            float v[4] = {0.f, 0.f, 0.f, 0.f};
            if (zi < zin_hi) {
                const Tin* src = in + (int64_t)zi * plane;
                __syncthreads();
                for (int e = tid; e < W * H; e += kThreads) {
                    const int r = e / W, c = e - r * W;
                    const int gy = y0 - R + r, gx = x0 - R + c;
                    float val = 0.f;
                    if (gy >= 0 && gy < ny && gx >= 0 && gx < nx) val = load_in(src + (int64_t)gy * pitch + gx);
                    s_in[r][c] = val;
                }
                __syncthreads();
                for (int e = tid; e < kTX * H; e += kThreads) {
                    const int r = e / kTX, c = e - r * kTX;
                    float acc = 0.f;
                    for (int d = -R; d <= R; ++d) acc = fmaf(prm.wxy[d + R], s_in[r][c + R + d], acc);
                    const int gx = min(x0 + c, nx - 1);
                    s_x[r][c] = acc * inv_nx[gx];
                }
                __syncthreads();
                const int gy = min(y0 + ty, ny - 1);
                const float iny = inv_ny[gy];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float acc = 0.f;
                    for (int d = -R; d <= R; ++d) acc = fmaf(prm.wxy[d + R], s_x[ty + R + d][4 * tx + i], acc);
                    v[i] = acc * iny;
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) ring[q][i] = v[i];
            const int zo = zi - Rz;
            if (zo >= z0 && zo < z1) {
                float o4[4] = {0.f, 0.f, 0.f, 0.f};
                float inz = 1.f;
                if constexpr (ROB) {
                    float wv[P];
#pragma unroll
                    for (int j = 0; j < P; ++j) wv[j] = (zi - j >= 0 && zi - j < nz) ? prm.wz[j] : 0.f;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        float vv[P];
#pragma unroll
                        for (int j = 0; j < P; ++j) vv[j] = ring[(q - j + P * 4) % P][i];
                        o4[i] = robust_window<P>(vv, wv, prm.kappa2);
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < P; ++j) {
                        const float w = prm.wz[j];
                        const int slot = (q - j + P * 4) % P;
#pragma unroll
                        for (int i = 0; i < 4; ++i) o4[i] = fmaf(w, ring[slot][i], o4[i]);
                    }
                    inz = inv_nz[zo];
                }
                const int gy = y0 + ty;
                if (gy < ny) {
                    float* dst = out + (int64_t)(zo - z0) * plane + (int64_t)gy * pitch;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int gx = x0 + 4 * tx + i;
                        if (gx < nx) dst[gx] = o4[i] * inz;
                    }
                }
            }
        }
    }
}

// Largest packed slab (see smooth_stack).
constexpr int64_t kPackBytes = (int64_t)1 << 29;

// Rows y0 .. y0 + ny_slab - 1 of planes z0 .. of `in` (any pitch) to rows of `ppitch` elements, a block
// per row, or gridDim.y blocks where the rows do not fill the chip (15 rows of 1,200,001 floats: the
// call takes 3.2 ms with a block each, now 1.2); the padding is not written (TMA reads only nx elements of a row).
template <class T>
__global__ void __launch_bounds__(256)
k_pack(const T* __restrict__ in, T* __restrict__ out, int nx, int y0, int ny_slab, int64_t ny, int64_t z0, int64_t pitch,
       int64_t ppitch, int64_t rows) {
    const int first = int(blockIdx.y * blockDim.x + threadIdx.x), step = int(gridDim.y * blockDim.x);
    for (int64_t row = blockIdx.x; row < rows; row += gridDim.x) {
        const int64_t z = row / ny_slab, y = row - z * ny_slab;
        const T* src = in + ((z0 + z) * ny + y0 + y) * pitch;
        T* dst = out + row * ppitch;
        if (sizeof(T) == 1) {  // 4 bytes per store; the last store stays inside the padded row
#pragma unroll 1  // one or two rounds on most rows: unrolled it costs 2 us of 28
            for (int x = 4 * first; x < nx; x += 4 * step) {
                uint32_t v = 0;
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (x + i < nx) v |= (uint32_t)(uint8_t)src[x + i] << (8 * i);
                *reinterpret_cast<uint32_t*>(dst + x) = v;
            }
        } else {
            for (int x = first; x < nx; x += step) dst[x] = src[x];
        }
    }
}

constexpr int kAxisGroup = 8;     // cells of a lane along y or z
constexpr int kAxisMaxRadius = 32;

// Taps d = -R .. R at w[kAxisGroup - 1 ...], zeros beside them.
struct AxisParams {
    float w[2 * kAxisMaxRadius + 1 + 3 * kAxisGroup];
    int R;
};

// One 1-D pass of the general smoothing and of its adjoint:
//   out[p] = post[c] * sum_{|d| <= R, c + d inside} w(d) pre[c + d] in[p + d],  c = the index of p along the axis,
// pre / post may be null (= 1).  The taps of a cell are added in ascending order of d, those outside the stack
// are left out.  Both kernels give a warp whole lines of a row, so that one division per item, not three
// per cell, finds the cell: a pass over 32 x 512 x 512 cells took 105 us with one cell per thread and
// index divisions in 64 bits, now 26 us along x and 24 along y (R = 3), 32 along z (R = 7, two sets of taps).
// Bound by instruction issue at small radii (80 % of the slots), with 10 us of memory traffic.

// Rows narrower than so many cells are taken as one line of cells (FLAT): a lane finds the row of its
// cells by divisions of its own, where a warp to a row would leave most lanes without one.  The whole
// smoothing (sigma 4 and 5, float), a warp to a row / as one line: 40 x 5001 x 3 353 / 199 us, 40 x 1000 x 20
// 139 / 115, x 48 151 / 137, x 63 156 / 142.
constexpr int kAxisFlat = 64;

// Along x: a warp makes 128 cells of a row, a lane every 32nd; the taps' loads hit L1.
template <class Tin, bool FLAT>
__global__ void __launch_bounds__(256)
axis_x_kernel(const Tin* __restrict__ in, float* __restrict__ out, int nx, int64_t rows, int64_t pitch_in, int64_t pitch_out,
              const float* __restrict__ pre, const float* __restrict__ post, AxisParams prm) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * 8;
    if constexpr (FLAT) {
        const int64_t cells = rows * nx;
        for (int64_t item = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); item * 128 < cells; item += warps) {
            int c[4];
            const Tin* src[4];
            float* dst[4];
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int64_t q = item * 128 + lane + 32 * t, row = index_div(q, nx);
                c[t] = q < cells ? (int)(q - row * nx) : nx + kAxisMaxRadius;  // past the end: no tap lies inside
                src[t] = in + row * pitch_in;
                dst[t] = out + row * pitch_out + c[t];
            }
            for (int d = -prm.R; d <= prm.R; ++d) {
                const float w = prm.w[kAxisGroup - 1 + d + prm.R];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int e = c[t] + d;
                    if (e < 0 || e >= nx) continue;
                    float v = float(src[t][e]);
                    if (pre) v *= pre[e];
                    acc[t] = fmaf(w, v, acc[t]);
                }
            }
#pragma unroll
            for (int t = 0; t < 4; ++t)
                if (c[t] < nx) *dst[t] = post ? acc[t] * post[c[t]] : acc[t];
        }
        return;
    }
    const int64_t segs = (nx + 127) / 128;
    for (int64_t item = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); item < segs * rows; item += warps) {
        const int64_t row = index_div(item, segs);
        const int x0 = (int)(item - row * segs) * 128, x = x0 + lane;
        const Tin* src = in + row * pitch_in;
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        if (x0 >= prm.R && x0 + 128 <= nx - prm.R) {
            const Tin* p = src + (x - prm.R);
            if (pre) {
                const float* f = pre + (x - prm.R);
                for (int k = 0; k <= 2 * prm.R; ++k, ++p, ++f) {
#pragma unroll
                    for (int t = 0; t < 4; ++t)
                        acc[t] = fmaf(prm.w[kAxisGroup - 1 + k], __fmul_rn(float(p[32 * t]), f[32 * t]), acc[t]);
                }
            } else {
#pragma unroll 2
                for (int k = 0; k <= 2 * prm.R; ++k, ++p) {
#pragma unroll
                    for (int t = 0; t < 4; ++t) acc[t] = fmaf(prm.w[kAxisGroup - 1 + k], float(p[32 * t]), acc[t]);
                }
            }
        } else {
            for (int d = -prm.R; d <= prm.R; ++d) {
                const float w = prm.w[kAxisGroup - 1 + d + prm.R];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int c = x + 32 * t + d;
                    if (c < 0 || c >= nx) continue;
                    float v = float(src[c]);
                    if (pre) v *= pre[c];
                    acc[t] = fmaf(w, v, acc[t]);
                }
            }
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int c = x + 32 * t;
            if (c < nx) out[row * pitch_out + c] = post ? acc[t] * post[c] : acc[t];
        }
    }
}

// Along y or z (`stride` cells apart, `len` of them): a lane makes kAxisGroup consecutive cells of
// the axis from one read of their common inputs, so R = 7 reads 22 values for 8 cells, not 120.
// The groups of a column run next to each other and share their halos in L1 and L2.  `outer` counts
// the other of the two axes.  DUAL: out = post * (w taps) + post2 * (w2 taps), from the same reads.
// The z passes take a plane as one row.
template <bool DUAL, bool FLAT>
__global__ void __launch_bounds__(256, DUAL ? 3 : 4)
axis_yz_kernel(const float* __restrict__ in, float* __restrict__ out, int nx, int len, int64_t stride, int64_t outer,
               int64_t outer_stride, const float* __restrict__ pre, const float* __restrict__ post,
               const float* __restrict__ post2, const __grid_constant__ AxisParams prm,
               const __grid_constant__ AxisParams prm2) {
    constexpr int G = kAxisGroup;
    const int lane = threadIdx.x & 31, R = prm.R;
    const int64_t groups = (len + G - 1) / G, segs = (nx + 31) / 32, warps = (int64_t)gridDim.x * 8;
    const int64_t items = FLAT ? (groups * nx * outer + 31) / 32 : groups * segs * outer;
    for (int64_t item = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); item < items; item += warps) {
        int64_t q;
        int c0, x;
        if constexpr (FLAT) {
            const int64_t t = item * 32 + lane, col = index_div(t, nx);
            q = index_div(col, groups);
            c0 = (int)(col - q * groups) * G;
            x = (int)(t - col * nx);
            if (q >= outer) continue;
        } else {
            const int64_t col = index_div(item, groups);
            q = index_div(col, segs);
            c0 = (int)(item - col * groups) * G;
            x = (int)(col - q * segs) * 32 + lane;
            if (x >= nx) continue;
        }
        const float* p = in + (q * outer_stride + x + (int64_t)(c0 - R) * stride);
        float acc[G], acc2[G];
#pragma unroll
        for (int j = 0; j < G; ++j) acc[j] = acc2[j] = 0.f;
        // inputs c0 - R + k, k = 0 .. 2 R + G - 1; cell j takes k - j = 0 .. 2 R.  The taps beside these
        // are 0 in the padded table, so finite values pass them without a test (a zero's sign aside).
        for (int k0 = 0; k0 < 2 * R + G; k0 += G) {
            const int cb = c0 - R + k0;
            float v[G], w[2 * G - 1], w2[2 * G - 1];
            bool finite = true;
            if (cb >= 0 && cb + G <= len) {
#pragma unroll
                for (int i = 0; i < G; ++i, p += stride) v[i] = *p;
                if (pre) {
#pragma unroll
                    for (int i = 0; i < G; ++i) v[i] *= pre[cb + i];
                }
            } else {
#pragma unroll
                for (int i = 0; i < G; ++i, p += stride) {
                    v[i] = 0.f;
                    if (cb + i >= 0 && cb + i < len) v[i] = pre ? *p * pre[cb + i] : *p;
                }
            }
#pragma unroll
            for (int i = 0; i < G; ++i) finite = finite && fabsf(v[i]) <= 3.4028235e38f;
#pragma unroll
            for (int i = 0; i < 2 * G - 1; ++i) {
                w[i] = prm.w[k0 + i];
                w2[i] = DUAL ? prm2.w[k0 + i] : 0.f;
            }
            if (finite) {
#pragma unroll
                for (int i = 0; i < G; ++i)
#pragma unroll
                    for (int j = 0; j < G; ++j) {
                        acc[j] = fmaf(w[G - 1 + i - j], v[i], acc[j]);
                        if (DUAL) acc2[j] = fmaf(w2[G - 1 + i - j], v[i], acc2[j]);
                    }
            } else {
#pragma unroll
                for (int i = 0; i < G; ++i)
#pragma unroll
                    for (int j = 0; j < G; ++j) {
                        const int t = k0 + i - j;
                        if (t < 0 || t > 2 * R || cb + i < 0 || cb + i >= len) continue;
                        acc[j] = fmaf(w[G - 1 + i - j], v[i], acc[j]);
                        if (DUAL) acc2[j] = fmaf(w2[G - 1 + i - j], v[i], acc2[j]);
                    }
            }
        }
        float* o = out + (q * outer_stride + x + (int64_t)c0 * stride);
#pragma unroll
        for (int j = 0; j < G; ++j, o += stride) {
            if (c0 + j >= len) break;
            float r = post ? __fmul_rn(acc[j], post[c0 + j]) : acc[j];
            if (DUAL) r = __fadd_rn(r, __fmul_rn(acc2[j], post2[c0 + j]));
            *o = r;
        }
    }
}

}  // namespace

int support_radius(float sigma) {
    if (!(sigma > 0.f)) return 0;
    return (int)std::floor(3.0 * (double)sigma + 1e-9);
}

std::vector<float> gaussian_taps(float sigma, int R) {
    std::vector<float> w(2 * R + 1, 1.f);
    if (sigma > 0.f)
        for (int d = -R; d <= R; ++d) w[d + R] = (float)std::exp(-(double)d * d / (2.0 * (double)sigma * sigma));
    return w;
}

// 1 / (sum of in-range taps) for every index 0..n-1 of an axis of length n.  The same for all
// indexes with every tap in range, so formed once for them: an axis of 1,200,000 cells with 7 taps took 5 ms
// of host time.
std::vector<float> inverse_norms(const std::vector<float>& w, int n) {
    const int R = ((int)w.size() - 1) / 2;
    auto at = [&](int i) {
        double s = 0.0;
        for (int d = std::max(-R, -i); d <= std::min(R, n - 1 - i); ++d) s += w[d + R];
        return (float)(1.0 / s);
    };
    std::vector<float> inv(n, n > 2 * R ? at(R) : 0.f);
    for (int i = 0; i < n; ++i) {
        if (i == R && n > 2 * R) i = n - R;  // the inner ones are done
        if (i < n) inv[i] = at(i);
    }
    return inv;
}

static int axis_params(const std::vector<float>& w, AxisParams* prm) {
    prm->R = ((int)w.size() - 1) / 2;
    if (prm->R > kAxisMaxRadius) {
        set_error("smoothing support radius above 32 taps is not supported");
        return EMFUSE_EINVAL;
    }
    for (size_t i = 0; i < w.size(); ++i) prm->w[kAxisGroup - 1 + i] = w[i];
    return EMFUSE_OK;
}

static unsigned axis_blocks(int64_t items) { return (unsigned)std::min<int64_t>(ceil_div(items, 8), (int64_t)kNumSMs * 64); }

static int launch_axis_x(const void* in, int dt, float* out, int64_t nx, int64_t ny, int64_t nz, int64_t pin,
                         const std::vector<float>& w, const float* pre, const float* post, cudaStream_t st) {
    AxisParams prm{};
    EMF_TRY(axis_params(w, &prm));
    const int64_t rows = ny * nz;
    KernelScope ks("smooth_axis", st, (double)nx * rows * ((dt == EMFUSE_U8 ? 1.0 : 4.0) + 4.0));
    const bool flat = nx < kAxisFlat;
    const unsigned blocks = axis_blocks(flat ? ceil_div(nx * rows, 128) : ceil_div(nx, 128) * rows);
    auto launch = [&](auto tin, auto flat_tag) {
        using Tin = decltype(tin);
        axis_x_kernel<Tin, decltype(flat_tag)::value><<<blocks, 256, 0, st>>>((const Tin*)in, out, (int)nx, rows, pin, nx, pre,
                                                                               post, prm);
    };
    auto launch_as = [&](auto tin) {
        if (flat) launch(tin, std::true_type{});
        else launch(tin, std::false_type{});
    };
    if (dt == EMFUSE_U8) launch_as(uint8_t{});
    else launch_as(float{});
    EMF_CHECK_LAUNCH();
    return EMFUSE_OK;
}

// Along y (axis 1) or z (axis 2) of a dense stack; w2 / post2: second set of taps, null if there is none.
static int launch_axis_yz(const float* in, float* out, int64_t nx, int64_t ny, int64_t nz, int axis,
                          const std::vector<float>& w, const float* pre, const float* post,
                          const std::vector<float>* w2, const float* post2, cudaStream_t st) {
    AxisParams prm{}, prm2{};
    EMF_TRY(axis_params(w, &prm));
    if (w2) EMF_TRY(axis_params(*w2, &prm2));
    KernelScope ks("smooth_axis", st, 8.0 * nx * ny * nz);
    if (axis == 2 && nx * ny <= INT32_MAX) {  // a plane as one row
        nx *= ny;
        ny = 1;
    }
    const int64_t len = axis == 1 ? ny : nz, stride = axis == 1 ? nx : nx * ny;
    const int64_t outer = axis == 1 ? nz : ny, outer_stride = axis == 1 ? nx * ny : nx;
    const int64_t groups = ceil_div(len, kAxisGroup);
    const bool flat = nx < kAxisFlat && !w2;
    const unsigned blocks = axis_blocks(flat ? ceil_div(groups * nx * outer, 32) : groups * ceil_div(nx, 32) * outer);
    auto launch = [&](auto dual_tag, auto flat_tag) {
        axis_yz_kernel<decltype(dual_tag)::value, decltype(flat_tag)::value><<<blocks, 256, 0, st>>>(
            in, out, (int)nx, (int)len, stride, outer, outer_stride, pre, post, post2, prm, prm2);
    };
    if (w2) launch(std::true_type{}, std::false_type{});
    else if (flat) launch(std::false_type{}, std::true_type{});
    else launch(std::false_type{}, std::false_type{});
    EMF_CHECK_LAUNCH();
    return EMFUSE_OK;
}

// Device table of the inverse normalisers of the three axes: [inv_x | inv_y | inv_z].
static int upload_norms(DeviceBuffer& buf, const std::vector<float>& ix, const std::vector<float>& iy,
                        const std::vector<float>& iz, cudaStream_t st, std::vector<float>& host) {
    host.clear();
    host.insert(host.end(), ix.begin(), ix.end());
    host.insert(host.end(), iy.begin(), iy.end());
    host.insert(host.end(), iz.begin(), iz.end());
    EMF_TRY(buf.alloc(host.size() * sizeof(float), st));
    EMF_CUDA(cudaMemcpyAsync(buf.as<float>(), host.data(), host.size() * sizeof(float),
                             cudaMemcpyHostToDevice, st));
    return EMFUSE_OK;
}

int smooth_stack(const void* in, int dt, float* out, int64_t nx, int64_t ny, int64_t nz,
                 int64_t pitch, int64_t z0, int64_t z1, float sigma_xy, float sigma_z,
                 cudaStream_t st, int force_path, float kappa) {
    const int Rxy = support_radius(sigma_xy);
    const int Rz = support_radius(sigma_z);
    const bool rob = kappa > 0.f;
    if (rob && (Rxy > kMaxRxy || Rz > 9 || force_path == 1)) {
        set_error("robust averaging needs floor(3 sigma_xy) <= 8 and floor(3 sigma_z) <= 9");
        return EMFUSE_EINVAL;
    }
    const auto wxy = gaussian_taps(sigma_xy, Rxy);
    const auto wz = gaussian_taps(sigma_z, Rz);
    std::vector<float> host;
    DeviceBuffer norms;
    EMF_TRY(upload_norms(norms, inverse_norms(wxy, (int)nx), inverse_norms(wxy, (int)ny),
                         inverse_norms(wz, (int)nz), st, host));
    const float* inv_x = norms.as<float>();
    const float* inv_y = inv_x + nx;
    const float* inv_z = inv_y + ny;

    const size_t esz = dt == EMFUSE_U8 ? 1 : 4;
    const bool tma_ok = Rxy <= 4 && Rz <= 9 && force_path == 0;
    const bool aligned = (pitch * (int64_t)esz) % 16 == 0 && (reinterpret_cast<uintptr_t>(in) & 15) == 0;
    const int64_t zin0 = std::max<int64_t>(0, z0 - Rz), zin1 = std::min<int64_t>(nz, z1 + Rz), nzin = zin1 - zin0;
    // Unaligned rows: packed (below), or by plain loads.  The copy's launch, its memory and the tensor map are
    // 7 us of host time, which marches of a plane or two over small planes do not earn back (us a call,
    // packed / plain, float: 1 x 100 x 101 24.9 / 17.4 one after another and 35.8 / 31.2 alone, 1 x 600 x 601 25.4 / 20.3
    // and 41.2 / 38.2, 1 x 1000 x 1001 26.9 / 26.7 and 48.6 / 47.6, 2 x 600 x 601 26.4 / 25.4 and 43.4 / 47.6, 3 x 300 x 301
    // 24.6 / 19.2 and 38.6 / 40.4, robust 24.8 / 29.9 and 48.5 / 50.4).  Supports below one cell, which no one
    // smooths by, have no packed instances.
    const bool few = nzin <= (rob ? 2 : 3) && nx * ny * nzin <= 400000;
    const bool packed = !aligned && Rxy >= 1 && Rz >= 1 && !few;
    if (tma_ok && (aligned || packed)) {
        SmoothTmaCall c{};
        c.prm.Rxy = Rxy;
        c.prm.Rz = Rz;
        for (int d = 0; d < 2 * Rxy + 1; ++d) c.prm.wxy[d] = wxy[d];
        for (int j = 0; j < 2 * Rz + 1; ++j) c.prm.wz[j] = wz[2 * Rz - j];
        c.prm.kappa2 = kappa * kappa;
        c.out = out;
        c.nx = (int)nx;
        c.ny = (int)ny;
        c.nz = (int)nz;
        c.pitch = pitch;
        c.z0 = (int)z0;
        c.z1 = (int)z1;
        c.inv_x = inv_x;
        c.inv_y = inv_y;
        c.inv_z = inv_z;
        c.yend = (int)ny;
        c.err = device_error_flag();
        const int hx = dt == EMFUSE_U8 ? 16 : 4, hxr = dt == EMFUSE_U8 ? 16 : 8;
        if (!c.err) {
            set_error("could not allocate the device error word");
            return EMFUSE_ECUDA;
        }
        const double bytes = (double)nx * ((zin1 - zin0) * (double)esz + (z1 - z0) * 4.0);  // per row
        if (aligned) {
            EMF_TRY(encode_tensor_map_3d(&c.map, in, (int)esz, nx, ny, nz, pitch, kTX + hx + hxr, kTY + 2 * Rxy));
            KernelScope ks(rob ? "smooth_tma_robust" : "smooth_tma", st, bytes * ny);
            auto run = [&](auto radius) -> int {
                constexpr int R = decltype(radius)::value;
                if (dt == EMFUSE_U8)
                    return rob ? smooth_tma_launch<uint8_t, R, true, false, 19>(c, st)
                               : smooth_tma_launch<uint8_t, R, false, false, 19>(c, st);
                return rob ? smooth_tma_launch<float, R, true, false, 19>(c, st)
                           : smooth_tma_launch<float, R, false, false, 19>(c, st);
            };
            switch (Rxy) {
                case 0: return run(std::integral_constant<int, 0>{});
                case 1: return run(std::integral_constant<int, 1>{});
                case 2: return run(std::integral_constant<int, 2>{});
                case 3: return run(std::integral_constant<int, 3>{});
                default: return run(std::integral_constant<int, 4>{});
            }
            // a timed-out wait is reported by the next call that synchronises (the solves)
        }
        // Rows that TMA cannot read (a byte pitch or base that is no multiple of 16): slabs of rows
        // of the needed planes, with their halo rows, are copied to an aligned pitch first.  The
        // copy costs 2 (uint8) or 8 bytes per voxel: 32 x 2047 x 2049 uint8 0.10 ms and the kernel 0.44
        // where smooth_fused_kernel took 2.32 (float 0.29 and 0.45 for 2.52; robust 1.68 for 3.73
        // and 1.95 for 4.06, copy included).  A slab is at most kPackBytes; where not even one
        // tile's rows fit, or there is no memory for it, smooth_fused_kernel still runs.
        const int64_t ppitch = round_up(nx, 16 / (int64_t)esz);
        const int64_t row_bytes = nzin * ppitch * (int64_t)esz;
        int64_t rows = std::min<int64_t>(ny, kPackBytes / row_bytes - 2 * Rxy);  // output rows of a slab
        if (rows < ny) rows = rows / kTY * kTY;
        DeviceBuffer slab;
        if (rows >= 1 && slab.alloc((size_t)(std::min<int64_t>(ny, rows + 2 * Rxy) * row_bytes), st) == EMFUSE_OK) {
            for (int64_t ya = 0; ya < ny; ya += rows) {
                const int64_t yb = std::min(ny, ya + rows);
                const int64_t ra = std::max<int64_t>(0, ya - Rxy), rb = std::min<int64_t>(ny, yb + Rxy);
                {
                    KernelScope ks("smooth_pack", st, (double)(2 * esz) * nx * (rb - ra) * nzin);
                    const int64_t n = nzin * (rb - ra);
                    constexpr int64_t full = (int64_t)kNumSMs * 32;
                    const int64_t per_block = 256 * (esz == 1 ? 4 : 1);
                    const dim3 grid((unsigned)std::min(n, full),
                                    (unsigned)std::min(std::max<int64_t>(1, full / n), ceil_div(nx, per_block)));
                    if (dt == EMFUSE_U8)
                        k_pack<uint8_t><<<grid, 256, 0, st>>>((const uint8_t*)in, slab.as<uint8_t>(), (int)nx, (int)ra,
                                                              (int)(rb - ra), ny, zin0, pitch, ppitch, n);
                    else
                        k_pack<float><<<grid, 256, 0, st>>>((const float*)in, slab.as<float>(), (int)nx, (int)ra,
                                                            (int)(rb - ra), ny, zin0, pitch, ppitch, n);
                    EMF_CHECK_LAUNCH();
                }
                EMF_TRY(encode_tensor_map_3d(&c.map, slab.as<char>(), (int)esz, nx, rb - ra, nzin, ppitch, kTX + hx + hxr,
                                             kTY + 2 * Rxy));
                c.ybase = (int)ya;
                c.yend = (int)yb;
                c.ymap = (int)ra;
                c.zmap = (int)zin0;
                KernelScope ks(rob ? "smooth_packed_robust" : "smooth_packed", st, bytes * (yb - ya));
                EMF_TRY(smooth_tma_packed(c, dt, rob, st));
            }
            return EMFUSE_OK;
        }
        cudaGetLastError();  // no memory for the copy: not an error of this call
        set_error("");
    }
    const bool fused_ok = Rxy <= kMaxRxy && Rz <= 9 && force_path != 1;
    if (fused_ok) {
        SmoothParams prm{};
        prm.Rxy = Rxy;
        prm.Rz = Rz;
        for (int d = 0; d < 2 * Rxy + 1; ++d) prm.wxy[d] = wxy[d];
        for (int j = 0; j < 2 * Rz + 1; ++j) prm.wz[j] = wz[2 * Rz - j];
        prm.kappa2 = kappa * kappa;
        dim3 grid((unsigned)ceil_div(nx, kTX), (unsigned)ceil_div(ny, kTY));
        const int P = 2 * Rz + 1;
        KernelScope ks(rob ? "smooth_fused_robust" : "smooth_fused", st,
                       (double)nx * ny * ((zin1 - zin0) * (dt == EMFUSE_U8 ? 1.0 : 4.0) + (z1 - z0) * 4.0));
#define EMF_SMOOTH_LAUNCH1(PP, RB)                                                             \
    do {                                                                                       \
        if (dt == EMFUSE_U8)                                                                   \
            smooth_fused_kernel<uint8_t, PP, RB><<<grid, kThreads, 0, st>>>(                   \
                (const uint8_t*)in, out, (int)nx, (int)ny, (int)nz, pitch, (int)z0, (int)z1,   \
                inv_x, inv_y, inv_z, prm);                                                     \
        else                                                                                   \
            smooth_fused_kernel<float, PP, RB><<<grid, kThreads, 0, st>>>(                     \
                (const float*)in, out, (int)nx, (int)ny, (int)nz, pitch, (int)z0, (int)z1,     \
                inv_x, inv_y, inv_z, prm);                                                     \
    } while (0)
#define EMF_SMOOTH_LAUNCH(PP)                                                                  \
    do {                                                                                       \
        if (rob) EMF_SMOOTH_LAUNCH1(PP, true);                                                 \
        else EMF_SMOOTH_LAUNCH1(PP, false);                                                    \
    } while (0)
        if (P <= 1) EMF_SMOOTH_LAUNCH(1);
        else if (P <= 7) EMF_SMOOTH_LAUNCH(7);
        else EMF_SMOOTH_LAUNCH(19);
#undef EMF_SMOOTH_LAUNCH
#undef EMF_SMOOTH_LAUNCH1
        EMF_CHECK_LAUNCH();
        return EMFUSE_OK;
    }
    // Three renormalised 1-D passes (x, y over the needed input planes; then z).
    DeviceBuffer t1, t2;
    EMF_TRY(t1.alloc((size_t)(nzin * ny * nx) * sizeof(float), st));
    EMF_TRY(t2.alloc((size_t)(nzin * ny * nx) * sizeof(float), st));
    const void* in0 = (const char*)in + (size_t)(zin0 * ny * pitch) * esz;
    EMF_TRY(launch_axis_x(in0, dt, t1.as<float>(), nx, ny, nzin, pitch, wxy, nullptr, inv_x, st));
    EMF_TRY(launch_axis_yz(t1.as<float>(), t2.as<float>(), nx, ny, nzin, 1, wxy, nullptr, inv_y, nullptr, nullptr, st));
    // z pass: only the requested output planes, normaliser indexed by absolute z
    DeviceBuffer tz;
    EMF_TRY(tz.alloc((size_t)(nzin * ny * nx) * sizeof(float), st));
    std::vector<float> iz_local(host.begin() + nx + ny + zin0, host.begin() + nx + ny + zin1);
    // renormalisation by the absolute-z table: recompute in local coordinates would be wrong
    // when the slab is a sub-range, so scale with the global table slice.
    DeviceBuffer izb;
    EMF_TRY(izb.alloc(iz_local.size() * sizeof(float), st));
    EMF_CUDA(cudaMemcpyAsync(izb.as<float>(), iz_local.data(), iz_local.size() * sizeof(float),
                             cudaMemcpyHostToDevice, st));
    EMF_TRY(launch_axis_yz(t2.as<float>(), tz.as<float>(), nx, ny, nzin, 2, wz, nullptr, izb.as<float>(), nullptr, nullptr,
                           st));
    EMF_CUDA(cudaMemcpy2DAsync(out, pitch * sizeof(float),
                               tz.as<float>() + (z0 - zin0) * ny * nx, nx * sizeof(float),
                               nx * sizeof(float), (size_t)((z1 - z0) * ny), cudaMemcpyDeviceToDevice, st));
    EMF_CUDA(cudaStreamSynchronize(st));  // host vectors above must outlive the async copies
    return EMFUSE_OK;
}

// K^T g for K = Kz Ky Kx (dense float stack, pitch nx):  (K_a^T v)(q) = sum_p w(p-q) v(p)/N(p).
int smooth_transpose(const float* g, float* out, int64_t nx, int64_t ny, int64_t nz,
                     float sigma_xy, float sigma_z, cudaStream_t st) {
    const int Rxy = support_radius(sigma_xy), Rz = support_radius(sigma_z);
    const auto wxy = gaussian_taps(sigma_xy, Rxy);
    const auto wz = gaussian_taps(sigma_z, Rz);
    std::vector<float> host;
    DeviceBuffer norms;
    EMF_TRY(upload_norms(norms, inverse_norms(wxy, (int)nx), inverse_norms(wxy, (int)ny),
                         inverse_norms(wz, (int)nz), st, host));
    const float* inv_x = norms.as<float>();
    const float* inv_y = inv_x + nx;
    const float* inv_z = inv_y + ny;
    DeviceBuffer t1;
    EMF_TRY(t1.alloc((size_t)(nx * ny * nz) * sizeof(float), st));
    EMF_TRY(launch_axis_yz(g, out, nx, ny, nz, 2, wz, inv_z, nullptr, nullptr, nullptr, st));
    EMF_TRY(launch_axis_yz(out, t1.as<float>(), nx, ny, nz, 1, wxy, inv_y, nullptr, nullptr, nullptr, st));
    EMF_TRY(launch_axis_x(t1.as<float>(), EMFUSE_F32, out, nx, ny, nz, nx, wxy, inv_x, nullptr, st));
    EMF_CUDA(cudaStreamSynchronize(st));
    return EMFUSE_OK;
}

// (dK/dsigma_z) I0 with the support radius fixed at floor(3 sigma_z):
//   Kz' v = (sum w' v) / N - (sum w v) N' / N^2,  w'(d) = w(d) d^2 / sigma^3.
int smooth_dsigma_z(const void* in, int dt, float* out, int64_t nx, int64_t ny, int64_t nz,
                    float sigma_xy, float sigma_z, cudaStream_t st) {
    const int Rxy = support_radius(sigma_xy), Rz = support_radius(sigma_z);
    const auto wxy = gaussian_taps(sigma_xy, Rxy);
    const auto wz = gaussian_taps(sigma_z, Rz);
    std::vector<float> dwz(wz.size());
    for (int d = -Rz; d <= Rz; ++d)
        dwz[d + Rz] = sigma_z > 0.f ? (float)((double)wz[d + Rz] * d * d / std::pow((double)sigma_z, 3)) : 0.f;
    const auto ix = inverse_norms(wxy, (int)nx), iy = inverse_norms(wxy, (int)ny), iz = inverse_norms(wz, (int)nz);
    std::vector<float> c1(nz), c2(nz);  // 1/N and -N'/N^2 per plane
    for (int z = 0; z < nz; ++z) {
        double N = 0, dN = 0;
        for (int d = -Rz; d <= Rz; ++d)
            if (z + d >= 0 && z + d < nz) { N += wz[d + Rz]; dN += dwz[d + Rz]; }
        c1[z] = (float)(1.0 / N);
        c2[z] = (float)(-dN / (N * N));
    }
    std::vector<float> host;
    DeviceBuffer norms, cz;
    EMF_TRY(upload_norms(norms, ix, iy, iz, st, host));
    std::vector<float> hc(c1);
    hc.insert(hc.end(), c2.begin(), c2.end());
    EMF_TRY(cz.alloc(hc.size() * sizeof(float), st));
    EMF_CUDA(cudaMemcpyAsync(cz.as<float>(), hc.data(), hc.size() * sizeof(float), cudaMemcpyHostToDevice, st));
    DeviceBuffer t1, t2;
    EMF_TRY(t1.alloc((size_t)(nx * ny * nz) * sizeof(float), st));
    EMF_TRY(t2.alloc((size_t)(nx * ny * nz) * sizeof(float), st));
    const float* inv_x = norms.as<float>();
    const float* inv_y = inv_x + nx;
    EMF_TRY(launch_axis_x(in, dt, t1.as<float>(), nx, ny, nz, nx, wxy, nullptr, inv_x, st));
    EMF_TRY(launch_axis_yz(t1.as<float>(), t2.as<float>(), nx, ny, nz, 1, wxy, nullptr, inv_y, nullptr, nullptr, st));
    EMF_TRY(launch_axis_yz(t2.as<float>(), out, nx, ny, nz, 2, dwz, nullptr, cz.as<float>(), &wz, cz.as<float>() + nz, st));
    EMF_CUDA(cudaStreamSynchronize(st));
    return EMFUSE_OK;
}

// ---------------------------------------------------------------- allocation-free variant
// emfuse_smooth_z_noalloc runs smooth_fused_kernel with its only scratch, the three per-axis
// tables of inverse normalisers, in a file-scope device array instead of memory from the CUDA
// allocator.  It exists for callers that cannot allocate device memory while they run: a host
// that has handed all device memory to its own pool or works under a fixed memory budget, and
// code on a latency-critical path where cudaMalloc / cudaFree would synchronise the device.
// Every GPU that loads this library holds the array (kNoAllocMaxNorms floats, 384 KiB) until
// the process exits.
constexpr int64_t kNoAllocMaxNorms = 3 * 32768;  // nx + ny + nz of one call
static __device__ __align__(256) float g_noalloc_norms[kNoAllocMaxNorms];

namespace {

// Fills the table [inv_x | inv_y | inv_z] of the allocation-free variant on the device, from the
// taps passed by value: entry i of an axis of length n is 1 / (sum of the taps w(d), |d| <= R,
// with 0 <= i + d < n), summed in double over d = -R..R and rounded once to float, i.e. the
// values inverse_norms() forms on the host.  (prm.wz holds w(R_z - j); the taps are symmetric,
// so prm.wz[d + R_z] = w(d).)
__global__ void k_noalloc_norms(float* __restrict__ tab, int nx, int ny, int nz, SmoothParams prm) {
    const int total = nx + ny + nz;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        const bool zax = t >= nx + ny;
        const int i = t < nx ? t : (zax ? t - nx - ny : t - nx);
        const int n = t < nx ? nx : (zax ? nz : ny);
        const int R = zax ? prm.Rz : prm.Rxy;
        double sum = 0.0;
        for (int d = -R; d <= R; ++d)
            if (i + d >= 0 && i + d < n) sum += (double)(zax ? prm.wz[d + R] : prm.wxy[d + R]);
        tab[t] = (float)(1.0 / sum);
    }
}

std::mutex g_noalloc_mu;
float* g_noalloc_ptr[64] = {nullptr};

// Device address of g_noalloc_norms on the current device, looked up once per device with
// that device current (in host code the array's name is only a host-side stand-in).
int noalloc_norms(float** out) {
    int dev = 0;
    EMF_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) {
        set_error("emfuse_smooth_z_noalloc: device ordinal out of range");
        return EMFUSE_EINVAL;
    }
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void* p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_norms);
        if (e != cudaSuccess || !p) {
            set_error(std::string("emfuse_smooth_z_noalloc: cudaGetSymbolAddress failed: ") +
                      cudaGetErrorString(e));
            return EMFUSE_ECUDA;
        }
        g_noalloc_ptr[dev] = static_cast<float*>(p);
    }
    *out = g_noalloc_ptr[dev];
    return EMFUSE_OK;
}

}  // namespace

}  // namespace emfuse

extern "C" int emfuse_smooth_z_noalloc(const void* in, int dt, float* out, int64_t nx, int64_t ny, int64_t nz,
                                       int64_t pitch, int64_t z0, int64_t z1, float sigma_xy, float sigma_z,
                                       void* stream) {
    using namespace emfuse;
    set_error("");
    if (!in || !out) {
        set_error("emfuse_smooth_z_noalloc: null pointer");
        return EMFUSE_EINVAL;
    }
    if (dt != EMFUSE_U8 && dt != EMFUSE_F32) {
        set_error("emfuse_smooth_z_noalloc: dtype must be EMFUSE_U8 or EMFUSE_F32");
        return EMFUSE_EINVAL;
    }
    if (nx < 1 || ny < 1 || nz < 1 || pitch < nx || z0 < 0 || z1 > nz || z0 >= z1) {
        set_error("emfuse_smooth_z_noalloc: need sizes >= 1, pitch >= nx and 0 <= z0 < z1 <= nz");
        return EMFUSE_EINVAL;
    }
    if (nx + ny + nz > kNoAllocMaxNorms) {
        set_error("emfuse_smooth_z_noalloc: nx + ny + nz = " + std::to_string(nx + ny + nz) +
                  " exceeds the static scratch of " + std::to_string(kNoAllocMaxNorms) +
                  " entries; use emfuse_smooth_z");
        return EMFUSE_EINVAL;
    }
    if (!std::isfinite(sigma_xy) || !std::isfinite(sigma_z) || sigma_xy < 0.f || sigma_z < 0.f) {
        set_error("emfuse_smooth_z_noalloc: sigma_xy and sigma_z must be finite and >= 0");
        return EMFUSE_EINVAL;
    }
    const int Rxy = support_radius(sigma_xy), Rz = support_radius(sigma_z);
    if (Rxy > kMaxRxy || Rz > 9) {
        set_error("emfuse_smooth_z_noalloc: needs floor(3 sigma_xy) <= 8 and floor(3 sigma_z) <= 9; wider "
                  "supports need temporaries, use emfuse_smooth_z");
        return EMFUSE_EINVAL;
    }
    const cudaStream_t st = (cudaStream_t)stream;
    float* norms = nullptr;
    EMF_TRY(noalloc_norms(&norms));
    const auto wxy = gaussian_taps(sigma_xy, Rxy);
    const auto wz = gaussian_taps(sigma_z, Rz);
    SmoothParams prm{};
    prm.Rxy = Rxy;
    prm.Rz = Rz;
    for (int d = 0; d < 2 * Rxy + 1; ++d) prm.wxy[d] = wxy[d];
    for (int j = 0; j < 2 * Rz + 1; ++j) prm.wz[j] = wz[2 * Rz - j];
    // The normaliser tables are written on the device, stream-ordered before the smoothing
    // kernel, from the taps in `prm` (no host buffer is involved).  Every entry the smoothing
    // kernel reads is rewritten by each call.
    {
        const int total = (int)(nx + ny + nz);
        KernelScope ks("smooth_noalloc_norms", st, 4.0 * total);
        k_noalloc_norms<<<(unsigned)ceil_div(total, 256), 256, 0, st>>>(norms, (int)nx, (int)ny, (int)nz, prm);
        EMF_CHECK_LAUNCH();
    }
    const float* inv_x = norms;
    const float* inv_y = inv_x + nx;
    const float* inv_z = inv_y + ny;
    const dim3 grid((unsigned)ceil_div(nx, kTX), (unsigned)ceil_div(ny, kTY));
    const int P = 2 * Rz + 1;
    const int64_t zin0 = std::max<int64_t>(0, z0 - Rz), zin1 = std::min<int64_t>(nz, z1 + Rz);
    KernelScope ks("smooth_noalloc", st,
                   (double)nx * ny * ((zin1 - zin0) * (dt == EMFUSE_U8 ? 1.0 : 4.0) + (z1 - z0) * 4.0));
#define EMF_NOALLOC_LAUNCH(PP)                                                               \
    do {                                                                                     \
        if (dt == EMFUSE_U8)                                                                 \
            smooth_fused_kernel<uint8_t, PP, false><<<grid, kThreads, 0, st>>>(              \
                (const uint8_t*)in, out, (int)nx, (int)ny, (int)nz, pitch, (int)z0, (int)z1, \
                inv_x, inv_y, inv_z, prm);                                                   \
        else                                                                                 \
            smooth_fused_kernel<float, PP, false><<<grid, kThreads, 0, st>>>(                \
                (const float*)in, out, (int)nx, (int)ny, (int)nz, pitch, (int)z0, (int)z1,   \
                inv_x, inv_y, inv_z, prm);                                                   \
    } while (0)
    if (P <= 1) EMF_NOALLOC_LAUNCH(1);
    else if (P <= 7) EMF_NOALLOC_LAUNCH(7);
    else EMF_NOALLOC_LAUNCH(19);
#undef EMF_NOALLOC_LAUNCH
    EMF_CHECK_LAUNCH();
    return EMFUSE_OK;
}
