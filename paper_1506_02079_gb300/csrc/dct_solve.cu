// Direct solve of Eq. (1) by fast Fourier transforms: the frequency-space interpretation of
// Sec. 3 ("Frequency-Space Interpretation": every frequency of the result is a weighted average
// of the two inputs' frequencies) turned into a solver.  Sec. 3 "Alternate Solutions" weighs an
// FFT solver against multigrid and rejects it for out-of-core CPUs (log-linear work and an
// out-of-core transpose); with a slice in HBM neither objection holds, so it serves here as an
// exact second GPU solver to compare the multigrid against.
//
// The Neumann graph Laplacian of an ny x nx slice is diagonal in the cosine modes (DCT-II), with
// eigenvalues 4 sin^2(pi k / 2ny) + 4 sin^2(pi l / 2nx).  In correction form f = o + d,
// (alpha I + L) d = alpha (s - o), so  d = IDCT( DCT(s - o) * alpha / (alpha + lambda) ).
//
// The cosine transforms run as real Fourier transforms of the slice's own size (J. Makhoul, "A
// Fast Cosine Transform in One and Two Dimensions", IEEE Trans. ASSP 28, 1980): along each axis
// the even samples in order, then the odd ones in reverse; the DCT coefficients are the real
// parts of the rotated transform.  A mode couples with its mirror images along both axes, so one
// thread takes the two spectrum entries (k, l) and (ny - k, l), forms the four coefficients
// they hold, scales them, and writes the two entries of the inverse transform's input: the
// spectrum is read and written once.  The transforms are cuFFT (R2C / C2R, batched over the
// slices); permutation, scaling and extraction are the kernels below.  All passes are bound by
// memory (64 B per cell in FP32, the two transforms' passes included).  Transforming the mirror
// extension (2ny x 2nx) instead, four times the points, took 0.99 ms for 16 x 1024 x 1024 in FP32
// where this takes 0.25 ms (3-D gradient domain, 32 x 1024 x 1024 uint8: 2.25 -> 0.63 ms).
#include <cuda_runtime.h>
#include <cublas_v2.h>
#include <cufft.h>

#include <algorithm>
#include <cmath>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <tuple>
#include <utility>
#include <vector>

#include "emfuse_common.cuh"
#include "emfuse_internal.cuh"

namespace emfuse {
namespace {

template <class T>
struct Fft;
template <>
struct Fft<float> {
    using C = cufftComplex;
    static constexpr cufftType kR2C = CUFFT_R2C, kC2R = CUFFT_C2R;
    static cufftResult fwd(cufftHandle p, float* in, C* out) { return cufftExecR2C(p, in, out); }
    static cufftResult inv(cufftHandle p, C* in, float* out) { return cufftExecC2R(p, in, out); }
};
template <>
struct Fft<double> {
    using C = cufftDoubleComplex;
    static constexpr cufftType kR2C = CUFFT_D2Z, kC2R = CUFFT_Z2D;
    static cufftResult fwd(cufftHandle p, double* in, C* out) { return cufftExecD2Z(p, in, out); }
    static cufftResult inv(cufftHandle p, C* in, double* out) { return cufftExecZ2D(p, in, out); }
};

inline unsigned grid_of(int64_t n) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, 256), (int64_t)kNumSMs * 32));
}

// Position of sample i of an axis of n in the transform's order: even samples first, then the odd
// ones from the end.
__device__ __forceinline__ int dct_place(int i, int n) { return (i & 1) ? n - 1 - (i >> 1) : i >> 1; }

// A thread's first cell of a row and its step, gridDim.y blocks to the row (row_blocks).
__device__ __forceinline__ int first_of_row() { return int(blockIdx.y * blockDim.x + threadIdx.x); }
__device__ __forceinline__ int row_step() { return int(gridDim.y * blockDim.x); }

// v = s - o (o may be null) in the transform's order.  One block per row, or gridDim.y of them.
template <class T, class Tin>
__global__ void __launch_bounds__(256)
k_permute(const Tin* __restrict__ s, const float* __restrict__ o, T* __restrict__ v, int nx, int ny, int64_t rows) {
    for (int64_t row = blockIdx.x; row < rows; row += gridDim.x) {
        const int64_t j = row / ny;
        const int y = int(row - j * ny);
        const Tin* sr = s + row * nx;
        const float* orow = o ? o + row * nx : nullptr;
        T* dst = v + (j * ny + dct_place(y, ny)) * nx;
        for (int x = first_of_row(); x < nx; x += row_step())
            dst[dct_place(x, nx)] = orow ? T(sr[x]) - T(orow[x]) : T(sr[x]);
    }
}

// f = o + v taken from the transform's order.
template <class T, class To>
__global__ void __launch_bounds__(256)
k_extract(const T* __restrict__ v, const To* __restrict__ o, float* __restrict__ f, int nx, int ny, int64_t rows) {
    for (int64_t row = blockIdx.x; row < rows; row += gridDim.x) {
        const int64_t j = row / ny;
        const int y = int(row - j * ny);
        const T* src = v + (j * ny + dct_place(y, ny)) * nx;
        const To* orow = o + row * nx;
        float* dst = f + row * nx;
        for (int x = first_of_row(); x < nx; x += row_step()) dst[x] = float(T(orow[x]) + src[dct_place(x, nx)]);
    }
}

// Device tables of a slice size: rotations e^{-i pi k / 2n} for k = 0 .. n / 2 and eigenvalues
// 4 sin^2(pi k / 2n) for k = 0 .. n - 1 of both axes.
template <class T, class C>
struct DctTables {
    const C *rot_y, *rot_x;
    const T *lam_y, *lam_x;
};

// Scales the cosine coefficients (k, l) of every slice by alpha / (alpha + lam_y[k] + lam_x[l])
// * norm, or with lam_z by -lam_z[j] / (alpha + lam_z[j] + lam_y[k] + lam_x[l]) * norm, in the half
// spectrum of the permuted slices (ny rows of nx / 2 + 1).  With A, B the entries of rows k and
// ny - k, a, b the rotations of k and l, P = b A and Q = b B:
//     X(k, l)           =  Re a (P + Q*) / 2        X(ny - k, l)      = Im a* (Q + P*) / 2
//     X(k, nx - l)      = -Im a (P - Q*) / 2        X(ny - k, nx - l) = Re a* (Q - P*) / 2
// (from cos u cos v and the Hermitian symmetry of a real transform), and back, with X(ny, .) =
// X(., nx) = 0,
//     row k:       a* b* ((X(k, l) - X(ny-k, nx-l)) - i (X(ny-k, l) + X(k, nx-l)))
//     row ny - k:  a  b* ((X(k, l) + X(ny-k, nx-l)) + i (X(ny-k, l) - X(k, nx-l)))
// GAIN: the gain first, for an alpha whose product with a coefficient leaves the type's range where the
// gain does not.  Not needed for 1e-20 <= alpha <= 1e20 (coefficients of 2^29 cells a side and values of
// 1e-10 .. 1e10 stay in FP32's range there), and 3 % slower in FP64 (20 x 400 x 700 217 -> 223 us).
template <class T, class C, bool GAIN>
__global__ void __launch_bounds__(256)
k_scale(C* __restrict__ spec, DctTables<T, C> tab, const T* __restrict__ lam_z, T alpha, T norm, int nx, int ny,
        int64_t nslices) {
    const int cols = nx / 2 + 1, half = ny / 2 + 1;
    const int64_t rows = nslices * half;
    for (int64_t row = blockIdx.x; row < rows; row += gridDim.x) {
        const int64_t j = row / half;
        const int k = int(row - j * half), r = k == 0 ? 0 : ny - k;
        C* rk = spec + (j * ny + k) * cols;
        C* rr = spec + (j * ny + r) * cols;
        const C a = tab.rot_y[k];
        const T lz = lam_z ? lam_z[j] : T(0);
        const T num = lam_z ? -lz : alpha;
        const T y0 = alpha + lz + tab.lam_y[k], y1 = k == 0 ? T(1) : alpha + lz + tab.lam_y[ny - k];
        const T h = GAIN ? T(0.5) * norm : T(0.5) * norm * num;
        for (int l = first_of_row(); l < cols; l += row_step()) {
            const C A = rk[l], B = rr[l], b = tab.rot_x[l];
            const T px = b.x * A.x - b.y * A.y, py = b.x * A.y + b.y * A.x;
            const T qx = b.x * B.x - b.y * B.y, qy = b.x * B.y + b.y * B.x;
            const T l0 = tab.lam_x[l], l1 = l == 0 ? T(0) : tab.lam_x[nx - l];
            // P + Q* = (px + qx, py - qy), Q + P* its conjugate; P - Q* = (px - qx, py + qy),
            // Q - P* = (qx - px, qy + py)
            const T sx = px + qx, sy = py - qy, dx = px - qx, dy = py + qy;
            auto scaled = [&](T sum, T den) {
                if constexpr (GAIN) return h * (num / den) * sum;
                else return h * sum / den;
            };
            const T x00 = scaled(a.x * sx - a.y * sy, y0 + l0);
            const T x10 = k == 0 ? T(0) : scaled(-a.x * sy - a.y * sx, y1 + l0);
            const T x01 = l == 0 ? T(0) : -scaled(a.x * dy + a.y * dx, y0 + l1);
            const T x11 = k == 0 || l == 0 ? T(0) : scaled(a.y * dy - a.x * dx, y1 + l1);
            // a b* and a* b*
            const T ux = a.x * b.x + a.y * b.y, uy = a.y * b.x - a.x * b.y;
            const T wx = a.x * b.x - a.y * b.y, wy = -(a.x * b.y + a.y * b.x);
            const T e = x00 - x11, g = -(x10 + x01);
            C o0;
            o0.x = wx * e - wy * g;
            o0.y = wx * g + wy * e;
            rk[l] = o0;
            if (r != k) {
                const T e1 = x00 + x11, g1 = x10 - x01;
                C o1;
                o1.x = ux * e1 - uy * g1;
                o1.y = ux * g1 + uy * e1;
                rr[l] = o1;
            }
        }
    }
}

// Real parts into / out of the spectrum of 1 x 1 slices (the transform of length 1).
template <class T, class C>
__global__ void k_single(T* __restrict__ v, C* __restrict__ spec, int64_t n, int forward) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (forward) {
            spec[i].x = v[i];
            spec[i].y = T(0);
        } else {
            v[i] = spec[i].x;
        }
    }
}

// cuFFT plans (forward R2C and inverse C2R over a batch) and the tables of their size, kept per
// device, size, batch and precision until emfuse_release_cache.
struct FftPlans {
    cufftHandle fwd = 0, inv = 0;  // none for 1 x 1 slices
    DeviceBuffer tables;           // DctTables, then the z transform's matrix and eigenvalues
    size_t rot_x = 0, lam_y = 0, lam_x = 0, z_mat = 0, z_lam = 0;  // byte offsets
    size_t work = 0;               // bytes of the transforms' work area, which each call brings
    std::mutex mu;  // held around cufftSetStream, cufftSetWorkArea and exec: one plan, several callers
    ~FftPlans() {
        if (fwd) cufftDestroy(fwd);
        if (inv) cufftDestroy(inv);
    }
};
// key: device, batch, ny, nx, element size, z transform
using FftKey = std::tuple<int, int64_t, int64_t, int64_t, int, bool>;
std::mutex g_fft_mu;
std::map<FftKey, std::shared_ptr<FftPlans>>& g_fft = *new std::map<FftKey, std::shared_ptr<FftPlans>>();

int fft_error(const char* what, cufftResult r) {
    set_error(std::string("cuFFT ") + what + " failed (cufftResult " + std::to_string((int)r) + ")");
    return r == CUFFT_ALLOC_FAILED ? EMFUSE_ENOMEM : EMFUSE_ECUDA;
}

// Tables of a plan, formed in FP64 on the host and on the device before the plan is handed out:
// callers on any stream may use it next, and a copy from pageable memory may return before it has
// reached the device, so it is waited for.  On a stream of its own, which waits for nothing else.
template <class T>
int make_tables(FftPlans& p, int64_t nx, int64_t ny, int64_t nz, bool z) {
    using C = typename Fft<T>::C;
    std::vector<char> host;
    auto rotations = [&](int64_t n) {
        const size_t at = host.size();
        host.resize(at + (size_t)round_up((n / 2 + 1) * (int64_t)sizeof(C), 256));
        C* c = reinterpret_cast<C*>(host.data() + at);
        for (int64_t k = 0; k <= n / 2; ++k) {
            c[k].x = T(std::cos(M_PI * (double)k / (2.0 * (double)n)));
            c[k].y = T(-std::sin(M_PI * (double)k / (2.0 * (double)n)));
        }
        return at;
    };
    auto eigenvalues = [&](int64_t n) {
        const size_t at = host.size();
        host.resize(at + (size_t)round_up(n * (int64_t)sizeof(T), 256));
        T* t = reinterpret_cast<T*>(host.data() + at);
        for (int64_t k = 0; k < n; ++k) {
            const double sn = std::sin(M_PI * (double)k / (2.0 * (double)n));
            t[k] = T(4.0 * sn * sn);
        }
        return at;
    };
    rotations(ny);
    p.rot_x = rotations(nx);
    p.lam_y = eigenvalues(ny);
    p.lam_x = eigenvalues(nx);
    if (z) {
        p.z_lam = eigenvalues(nz);
        p.z_mat = host.size();
        host.resize(p.z_mat + (size_t)(nz * nz) * sizeof(T));
        T* m = reinterpret_cast<T*>(host.data() + p.z_mat);
        for (int64_t k = 0; k < nz; ++k) {
            const double ck = std::sqrt((k == 0 ? 1.0 : 2.0) / (double)nz);
            for (int64_t q = 0; q < nz; ++q)
                m[k * nz + q] = T(ck * std::cos(M_PI * (double)k * (double)(2 * q + 1) / (2.0 * (double)nz)));
        }
    }
    EMF_TRY(p.tables.alloc_persistent(host.size()));
    cudaStream_t up = nullptr;
    EMF_CUDA(cudaStreamCreateWithFlags(&up, cudaStreamNonBlocking));
    cudaError_t e = cudaMemcpyAsync(p.tables.as<char>(), host.data(), host.size(), cudaMemcpyHostToDevice, up);
    const cudaError_t es = cudaStreamSynchronize(up);
    cudaStreamDestroy(up);
    if (e == cudaSuccess) e = es;
    EMF_CUDA(e);
    return EMFUSE_OK;
}

// n transforms of ny x nx (1-D ones along the longer axis where a side is 1; none for 1 x 1)
template <class T>
int get_plans(int64_t nx, int64_t ny, int64_t n, bool z, std::shared_ptr<FftPlans>& out) {
    int dev = 0;
    EMF_CUDA(cudaGetDevice(&dev));
    const FftKey key = std::make_tuple(dev, n, ny, nx, (int)sizeof(T), z);
    std::lock_guard<std::mutex> lk(g_fft_mu);
    auto it = g_fft.find(key);
    if (it != g_fft.end()) {
        out = it->second;
        return EMFUSE_OK;
    }
    auto p = std::make_shared<FftPlans>();
    if (nx * ny > 1) {
        const int rank = ny == 1 ? 1 : 2;
        long long dims[2] = {(long long)ny, (long long)nx};
        long long* d = rank == 1 ? dims + 1 : dims;
        const long long rdist = nx * ny, cdist = ny * (nx / 2 + 1);
        size_t work[2] = {0, 0};
        cufftResult r = cufftCreate(&p->fwd);
        if (r == CUFFT_SUCCESS) r = cufftSetAutoAllocation(p->fwd, 0);
        if (r == CUFFT_SUCCESS)
            r = cufftMakePlanMany64(p->fwd, rank, d, nullptr, 1, rdist, nullptr, 1, cdist, Fft<T>::kR2C, n, &work[0]);
        if (r != CUFFT_SUCCESS) return fft_error("forward plan", r);
        r = cufftCreate(&p->inv);
        if (r == CUFFT_SUCCESS) r = cufftSetAutoAllocation(p->inv, 0);
        if (r == CUFFT_SUCCESS)
            r = cufftMakePlanMany64(p->inv, rank, d, nullptr, 1, cdist, nullptr, 1, rdist, Fft<T>::kC2R, n, &work[1]);
        if (r != CUFFT_SUCCESS) return fft_error("inverse plan", r);
        p->work = std::max(work[0], work[1]);
    }
    EMF_TRY((make_tables<T>(*p, nx, ny, n, z)));
    g_fft[key] = p;
    out = p;
    return EMFUSE_OK;
}

// forward / inverse transform of the batch on stream st, in the caller's work area (p.work bytes).
// Transforms of one plan run asynchronously and at the same time on several streams, so a work area of
// the plan's own would be shared by them; the lock covers what the plan holds until they are queued.
template <class T>
int fft_run(FftPlans& p, T* v, typename Fft<T>::C* spec, void* work, int64_t n, bool forward, cudaStream_t st) {
    if (!p.fwd) {
        k_single<T, typename Fft<T>::C><<<grid_of(n), 256, 0, st>>>(v, spec, n, forward ? 1 : 0);
        EMF_CHECK_LAUNCH();
        return EMFUSE_OK;
    }
    std::lock_guard<std::mutex> lk(p.mu);
    cufftResult r = cufftSetStream(forward ? p.fwd : p.inv, st);
    if (r == CUFFT_SUCCESS && work) r = cufftSetWorkArea(forward ? p.fwd : p.inv, work);
    if (r == CUFFT_SUCCESS) r = forward ? Fft<T>::fwd(p.fwd, v, spec) : Fft<T>::inv(p.inv, spec, v);
    return r == CUFFT_SUCCESS ? EMFUSE_OK : fft_error(forward ? "forward transform" : "inverse transform", r);
}

// Threads and blocks of a pass over `rows` rows of `cells` cells: a block per row while the rows
// fill the chip (loops beyond that), several blocks to a row where they do not.  Two rows of 200,000
// cells in FP64: 2.67 ms with a block per row, in which each thread takes 800 cells one after another,
// 0.28 with the chip filled (FP32 0.63 and 0.10).
inline unsigned row_threads(int64_t cells) {
    return (unsigned)std::min<int64_t>(256, round_up(std::max<int64_t>(cells, 1), 32));
}
inline dim3 row_blocks(int64_t rows, int64_t cells) {
    constexpr int64_t full = (int64_t)kNumSMs * 32;
    const int64_t gx = std::max<int64_t>(1, std::min(rows, full));
    const int64_t gy = std::min(std::max<int64_t>(1, full / gx), ceil_div(std::max<int64_t>(cells, 1), row_threads(cells)));
    return dim3((unsigned)gx, (unsigned)gy);
}

// v -> cosine coefficients scaled -> v, in the transform's order (lam_z: see k_scale)
template <class T>
int dct_filter(FftPlans& p, T* v, typename Fft<T>::C* spec, void* work, int64_t nx, int64_t ny, int64_t n, double alpha, bool z,
               const char* name, cudaStream_t st) {
    using C = typename Fft<T>::C;
    EMF_TRY((fft_run<T>(p, v, spec, work, n, true, st)));
    {
        const char* t = p.tables.as<char>();
        DctTables<T, C> tab;
        tab.rot_y = reinterpret_cast<const C*>(t);
        tab.rot_x = reinterpret_cast<const C*>(t + p.rot_x);
        tab.lam_y = reinterpret_cast<const T*>(t + p.lam_y);
        tab.lam_x = reinterpret_cast<const T*>(t + p.lam_x);
        const int64_t cols = nx / 2 + 1;
        KernelScope ks(name, st, (double)n * ny * cols * 2.0 * sizeof(C));
        const bool gain = !z && (alpha < 1e-20 || alpha > 1e20);
        auto* kernel = gain ? k_scale<T, C, true> : k_scale<T, C, false>;
        kernel<<<row_blocks(n * (ny / 2 + 1), cols), row_threads(cols), 0, st>>>(
            spec, tab, z ? reinterpret_cast<const T*>(t + p.z_lam) : nullptr, T(alpha),
            T(1.0 / ((double)nx * (double)ny)), (int)nx, (int)ny, n);
        EMF_CHECK_LAUNCH();
    }
    return fft_run<T>(p, v, spec, work, n, false, st);
}

template <class T>
int dct_solve(const float* s, const float* o, float* f, int64_t n, int64_t nx, int64_t ny, double alpha,
              cudaStream_t st) {
    using C = typename Fft<T>::C;
    if (nx == 1) std::swap(nx, ny);  // a column is a row in memory
    std::shared_ptr<FftPlans> plans;
    EMF_TRY((get_plans<T>(nx, ny, n, false, plans)));
    // one allocation: the spectra (first, for their alignment), the slices, cuFFT's work area
    const size_t nspec = round_up(n * ny * (nx / 2 + 1) * (int64_t)sizeof(C), 256);
    const size_t nv = round_up(n * nx * ny * (int64_t)sizeof(T), 256);
    DeviceBuffer tmp;
    EMF_TRY(tmp.alloc(nspec + nv + plans->work, st));
    C* const spec = tmp.as<C>();
    T* const v = reinterpret_cast<T*>(tmp.as<char>() + nspec);
    void* const work = plans->work ? tmp.as<char>() + nspec + nv : nullptr;
    {
        KernelScope ks("dct_permute", st, (double)n * nx * ny * (8.0 + sizeof(T)));
        k_permute<T, float><<<row_blocks(n * ny, nx), row_threads(nx), 0, st>>>(s, o, v, (int)nx, (int)ny, n * ny);
        EMF_CHECK_LAUNCH();
    }
    EMF_TRY((dct_filter<T>(*plans, v, spec, work, nx, ny, n, alpha, false, "dct_scale", st)));
    {
        KernelScope ks("dct_extract", st, (double)n * nx * ny * (4.0 + 4.0 + sizeof(T)));
        k_extract<T, float><<<row_blocks(n * ny, nx), row_threads(nx), 0, st>>>(v, o, f, (int)nx, (int)ny, n * ny);
        EMF_CHECK_LAUNCH();
    }
    // the temporaries go back to the pool stream-ordered; the caller's stream orders f
    return EMFUSE_OK;
}

// ---------------------------------------------------------------- 3-D gradient-domain smoothing
// The smoothing of the earlier method (Sec. 3 "Alternate Solutions"): the stack f minimising
// alpha |f - I0|^2 + |grad_xy f - grad_xy I0|^2 + |d_z f|^2 on the 6-neighbour graph with
// Neumann boundaries, (alpha I + L_xy + L_z) f = alpha I0 + L_xy I0.  In correction form
// f = I0 + d, (alpha I + L_xy + L_z) d = -L_z I0.  The orthonormal DCT-II along z,
// C[k][z] = c_k cos(pi k (2z + 1) / 2nz), diagonalises L_z (eigenvalues lam_z[k] =
// 4 sin^2(pi k / 2nz)), so with I~ = C I0 and d~ = C d (per pixel column) the problem falls
// apart into nz independent slice problems
//     (alpha + lam_z[k]) d~_k + L_xy d~_k = -lam_z[k] I~_k,
// each a screened Poisson equation of the kind of Eq. (1) with its own screening, solved
// exactly by the cosine transforms of the 2-D direct solver above.  The two z transforms are
// dense nz x nz contractions over all pixels: cuBLAS GEMMs; they act on pixel columns, so the
// slices are permuted into the transform's order before the first and back after the second, in
// the passes that convert the input and add the result to it.

// cuBLAS handles, one per device, kept until emfuse_release_cache.  As with the transforms, a call
// brings its own workspace (the handle's would be shared by GEMMs on several streams), and the lock
// covers cublasSetStream, cublasSetWorkspace and the GEMM's launch.
constexpr size_t kBlasWorkspace = (size_t)32 << 20;  // what cuBLAS itself takes on this architecture
struct BlasHandle {
    cublasHandle_t h = nullptr;
    std::mutex mu;
    ~BlasHandle() {
        if (h) cublasDestroy(h);
    }
};
std::mutex g_blas_mu;
std::map<int, std::shared_ptr<BlasHandle>>& g_blas = *new std::map<int, std::shared_ptr<BlasHandle>>();

int get_blas(std::shared_ptr<BlasHandle>& out) {
    int dev = 0;
    EMF_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(g_blas_mu);
    auto it = g_blas.find(dev);
    if (it != g_blas.end()) {
        out = it->second;
        return EMFUSE_OK;
    }
    auto b = std::make_shared<BlasHandle>();
    const cublasStatus_t s = cublasCreate(&b->h);
    if (s != CUBLAS_STATUS_SUCCESS) {
        b->h = nullptr;
        set_error("cuBLAS handle creation failed (cublasStatus " + std::to_string((int)s) + ")");
        return s == CUBLAS_STATUS_ALLOC_FAILED ? EMFUSE_ENOMEM : EMFUSE_ECUDA;
    }
    g_blas[dev] = b;
    out = b;
    return EMFUSE_OK;
}

template <class T>
struct Gemm;
template <>
struct Gemm<float> {
    static cublasStatus_t run(cublasHandle_t h, cublasOperation_t tb, int64_t m, int64_t n, const float* A,
                              const float* B, float* Cm) {
        const float one = 1.f, zero = 0.f;
        return cublasSgemm_64(h, CUBLAS_OP_N, tb, m, n, n, &one, A, m, B, n, &zero, Cm, m);
    }
};
template <>
struct Gemm<double> {
    static cublasStatus_t run(cublasHandle_t h, cublasOperation_t tb, int64_t m, int64_t n, const double* A,
                              const double* B, double* Cm) {
        const double one = 1.0, zero = 0.0;
        return cublasDgemm_64(h, CUBLAS_OP_N, tb, m, n, n, &one, A, m, B, n, &zero, Cm, m);
    }
};

// The stack x as [nz][P] row-major is the P x nz column-major matrix X; the row-major DCT
// matrix C[k][z] read column-major is C^T.  Forward: Y = X C^T (Y[k][p] = sum_z C[k][z] x[z][p]);
// inverse: Y = X C (Y[z][p] = sum_k C[k][z] x[k][p]).
template <class T>
int z_transform(BlasHandle& b, void* work, const T* x, const T* cmat, T* y, int64_t P, int64_t nz, bool inverse,
                cudaStream_t st) {
    std::lock_guard<std::mutex> lk(b.mu);
    cublasStatus_t s = cublasSetStream(b.h, st);  // also resets the handle's workspace
    if (s == CUBLAS_STATUS_SUCCESS) s = cublasSetWorkspace(b.h, work, kBlasWorkspace);
    if (s == CUBLAS_STATUS_SUCCESS) s = Gemm<T>::run(b.h, inverse ? CUBLAS_OP_T : CUBLAS_OP_N, P, nz, x, cmat, y);
    if (s != CUBLAS_STATUS_SUCCESS) {
        set_error("cuBLAS GEMM of the z transform failed (cublasStatus " + std::to_string((int)s) + ")");
        return EMFUSE_ECUDA;
    }
    return EMFUSE_OK;
}

template <class T, class Tin>
int gd_smooth(const Tin* in, float* out, int64_t nx, int64_t ny, int64_t nz, double alpha, cudaStream_t st) {
    using C = typename Fft<T>::C;
    if (nx == 1) std::swap(nx, ny);  // a column is a row in memory
    const int64_t P = nx * ny, N = P * nz;
    std::shared_ptr<FftPlans> plans;
    std::shared_ptr<BlasHandle> blas;
    EMF_TRY((get_plans<T>(nx, ny, nz, true, plans)));
    EMF_TRY(get_blas(blas));
    // one allocation: the spectra (first, for their alignment), the stack twice, and one work area for
    // the transforms and the GEMMs, which follow one another on the stream
    const size_t nspec = round_up(nz * ny * (nx / 2 + 1) * (int64_t)sizeof(C), 256);
    const size_t nstack = round_up(N * (int64_t)sizeof(T), 256);
    DeviceBuffer tmp;
    EMF_TRY(tmp.alloc(nspec + 2 * nstack + std::max(plans->work, kBlasWorkspace), st));
    C* const spec = tmp.as<C>();
    T* const x = reinterpret_cast<T*>(tmp.as<char>() + nspec);
    T* const y = reinterpret_cast<T*>(tmp.as<char>() + nspec + nstack);
    void* const work = tmp.as<char>() + nspec + 2 * nstack;
    const T* cmat = reinterpret_cast<const T*>(plans->tables.as<char>() + plans->z_mat);
    {
        KernelScope ks("gd_permute", st, (double)N * (sizeof(Tin) + sizeof(T)));
        k_permute<T, Tin><<<row_blocks(nz * ny, nx), row_threads(nx), 0, st>>>(in, nullptr, x, (int)nx, (int)ny,
                                                                          nz * ny);
        EMF_CHECK_LAUNCH();
    }
    EMF_TRY(z_transform<T>(*blas, work, x, cmat, y, P, nz, false, st));
    EMF_TRY((dct_filter<T>(*plans, y, spec, work, nx, ny, nz, alpha, true, "gd_scale", st)));
    EMF_TRY(z_transform<T>(*blas, work, y, cmat, x, P, nz, true, st));
    {
        KernelScope ks("gd_out", st, (double)N * (sizeof(Tin) + sizeof(T) + 4.0));
        k_extract<T, Tin><<<row_blocks(nz * ny, nx), row_threads(nx), 0, st>>>(x, in, out, (int)nx, (int)ny, nz * ny);
        EMF_CHECK_LAUNCH();
    }
    return EMFUSE_OK;
}

}  // namespace

int smooth_gradient_domain(const void* in, int dt, float* out, int64_t nx, int64_t ny, int64_t nz, double alpha,
                           int precision, cudaStream_t st) {
    if (dt == EMFUSE_U8) {
        const uint8_t* p = static_cast<const uint8_t*>(in);
        return precision == EMFUSE_PREC_FP32 ? gd_smooth<float>(p, out, nx, ny, nz, alpha, st)
                                             : gd_smooth<double>(p, out, nx, ny, nz, alpha, st);
    }
    const float* p = static_cast<const float*>(in);
    return precision == EMFUSE_PREC_FP32 ? gd_smooth<float>(p, out, nx, ny, nz, alpha, st)
                                         : gd_smooth<double>(p, out, nx, ny, nz, alpha, st);
}

int solve_dct_batch(const float* s, const float* o, float* f, int64_t n, int64_t nx, int64_t ny, double alpha,
                    int precision, cudaStream_t st) {
    return precision == EMFUSE_PREC_FP32 ? dct_solve<float>(s, o, f, n, nx, ny, alpha, st)
                                         : dct_solve<double>(s, o, f, n, nx, ny, alpha, st);
}

void release_fft_plans() {
    {
        std::lock_guard<std::mutex> lk(g_fft_mu);
        g_fft.clear();
    }
    std::lock_guard<std::mutex> lk(g_blas_mu);
    g_blas.clear();
}

}  // namespace emfuse
