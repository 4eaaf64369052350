// Translation stage of the FMM-FFT (Sec. II.A, between Eqs. 3 and 5; refs. [7, 8]),
// with the translation operator of the addition theorem (ref. [25]):
//
//   g_v(k_i) = c sum_{v' far from v} T_L(k_i, r_v - r_v') F_v'(k_i),
//   T_L(k, X) = sum_{l=0}^{L} (-j)^l (2l + 1) h_l^(2)(k |X|) P_l(k . X / |X|),
//   c = -j k / (16 pi^2),
//
// for every box v, direction i and component alpha; boxes are far when their grid
// indices differ by 2 or more in some coordinate (touching boxes belong to the near
// field).  T depends on the boxes only through their index difference, so for each
// direction the sum is a discrete 3-D convolution over the box grid: the spectra are
// scattered into a zero-padded grid of N_x x N_y x N_z >= (2K - 1)^3 points,
// transformed, multiplied by the transform of c T (built once, FP64, then stored
// FP32, N_dir x N_grid) and transformed back.
//
// Two forms.  Near-cubic grids of up to 36 points a side run cube_translate_kernel: one
// CTA does a whole transform in shared memory and registers, so that HBM sees the spectra and
// the operator only.  Other grids run cuFFT over a work array in HBM holding the 2 N_dir
// transforms of one right-hand side one after the other (transform j = alpha N_dir + i, grid
// point s at j N_grid + s), with the scatter, product and gather kernels here.
#include <cufft.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "internal.h"

namespace tfmm {

namespace {

#define CUFFT_CHECK(call)                                                                           \
    do {                                                                                            \
        cufftResult r_ = (call);                                                                    \
        if (r_ != CUFFT_SUCCESS)                                                                    \
            fail(r_ == CUFFT_ALLOC_FAILED ? TFMM_OOM : TFMM_CUDA,                                    \
                 std::string(#call) + " failed with cuFFT status " + std::to_string((int)r_));     \
    } while (0)

constexpr int kMaxL = 512;

// c T_L(k_i, X(s)) for the grid point s (signed index differences d, far ones only), FP64:
// h_l^(2)(k|X|) by the upward three-term recurrence of the spherical Bessel functions
// (stable for h^(2) = j - i y, whose magnitude grows with l), P_l(cos) by Bonnet's recurrence.
__global__ void translation_kernel(const double* __restrict__ khat, int n_dir, int L, double k, double a, int Nx,
                                   int Ny, int Nz, int Kx, int Ky, int Kz, int64_t Ns, double2* __restrict__ T) {
    __shared__ double2 h[kMaxL + 1];
    __shared__ double xh[3];
    __shared__ int far;
    const int64_t s = blockIdx.x;
    const int sx = (int)(s % Nx), sy = (int)((s / Nx) % Ny), sz = (int)(s / ((int64_t)Nx * Ny));
    const int dx = sx < Nx - sx ? sx : sx - Nx, dy = sy < Ny - sy ? sy : sy - Ny, dz = sz < Nz - sz ? sz : sz - Nz;
    if (threadIdx.x == 0) {
        const int m = max(abs(dx), max(abs(dy), abs(dz)));
        far = (m >= 2 && abs(dx) < Kx && abs(dy) < Ky && abs(dz) < Kz) ? 1 : 0;
        if (far) {
            const double X[3] = {dx * a, dy * a, dz * a};
            const double r = sqrt(X[0] * X[0] + X[1] * X[1] + X[2] * X[2]);
            for (int c = 0; c < 3; ++c) xh[c] = X[c] / r;
            const double x = k * r, sn = sin(x), cs = cos(x);
            // h_0 = j_0 - i y_0, h_1 = j_1 - i y_1
            h[0] = make_double2(sn / x, cs / x);
            if (L >= 1) h[1] = make_double2(sn / (x * x) - cs / x, cs / (x * x) + sn / x);
            for (int l = 1; l < L; ++l) {
                const double f = (2.0 * l + 1.0) / x;
                h[l + 1] = make_double2(f * h[l].x - h[l - 1].x, f * h[l].y - h[l - 1].y);
            }
        }
    }
    __syncthreads();
    const double2 c = make_double2(0.0, -k / (16.0 * 3.14159265358979323846 * 3.14159265358979323846));
    for (int i = threadIdx.x; i < n_dir; i += blockDim.x) {
        double2 acc = make_double2(0.0, 0.0);
        if (far) {
            const double ct = khat[3 * i] * xh[0] + khat[3 * i + 1] * xh[1] + khat[3 * i + 2] * xh[2];
            double pm = 0.0, p = 1.0;  // P_{l-1}, P_l
            for (int l = 0; l <= L; ++l) {
                if (l == 1) {
                    pm = 1.0;
                    p = ct;
                } else if (l >= 2) {
                    const double pn = ((2.0 * l - 1.0) * ct * p - (l - 1.0) * pm) / l;
                    pm = p;
                    p = pn;
                }
                // (-j)^l (2l + 1) P_l h_l
                const double w = (2.0 * l + 1.0) * p;
                double2 t = make_double2(w * h[l].x, w * h[l].y);
                switch (l & 3) {
                    case 1: t = make_double2(t.y, -t.x); break;   // * (-j)
                    case 2: t = make_double2(-t.x, -t.y); break;  // * (-1)
                    case 3: t = make_double2(-t.y, t.x); break;   // * (+j)
                    default: break;
                }
                acc.x += t.x;
                acc.y += t.y;
            }
            acc = make_double2(c.x * acc.x - c.y * acc.y, c.x * acc.y + c.y * acc.x);
        }
        T[(int64_t)i * Ns + s] = acc;
    }
}

__global__ void to_f32_kernel(const double2* __restrict__ in, int64_t n, float2* __restrict__ out) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        out[e] = make_float2((float)in[e].x, (float)in[e].y);
}

// grid[j][cell(g)] = spectra[g][j] for every group g and j < 2 N_dir (the rest of the
// grid was zeroed)
__global__ void scatter_kernel(const float2* __restrict__ spec, const int* __restrict__ group_cell, int G, int nb,
                               int64_t Ns, float2* __restrict__ grid) {
    const int64_t total = (int64_t)G * nb;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int g = (int)(e / nb), j = (int)(e - (int64_t)g * nb);
        grid[(int64_t)j * Ns + group_cell[g]] = spec[e];
    }
}

// grid[alpha N_dir + i][s] *= That[i][s]
__global__ void multiply_kernel(float2* __restrict__ grid, const float2* __restrict__ That, int64_t Ns, int n_dir) {
    const int64_t per = (int64_t)n_dir * Ns, total = 2 * per;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const float2 t = That[e < per ? e : e - per], v = grid[e];
        grid[e] = make_float2(v.x * t.x - v.y * t.y, v.x * t.y + v.y * t.x);
    }
}

// spectra_in[g][j] = grid[j][cell(g)] / Ns (the inverse transform is unnormalised)
__global__ void gather_kernel(const float2* __restrict__ grid, const int* __restrict__ group_cell, int G, int nb,
                              int64_t Ns, float scale, float2* __restrict__ spec) {
    const int64_t total = (int64_t)G * nb;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int g = (int)(e / nb), j = (int)(e - (int64_t)g * nb);
        const float2 v = grid[(int64_t)j * Ns + group_cell[g]];
        spec[e] = make_float2(scale * v.x, scale * v.y);
    }
}

// ------------------------------------------------------------ whole transforms on the SM
// Register FFTs: a thread transforms one line of N = A B points (A, B <= 8) held in
// registers, X[k1 + A k2] = sum_b W_B^(b k2) W_N^(b k1) sum_a W_A^(a k1) x[B a + b].  Every
// loop unrolls, so that the line stays in registers and the twiddles are constant operands.
// (no 4: for up to two boxes a side its volume is past twice cuFFT's grid; no 16: 15 serves eight boxes, 18 nine)
constexpr int kCubeSizes[] = {6, 8, 10, 12, 15, 18, 20, 24, 25, 30, 32, 36};
constexpr int kCubeMax = 36;
__constant__ float2 c_tw[kCubeMax * (kCubeMax + 1) / 2];  // W_n^k = exp(-2 pi i k / n) at n (n - 1) / 2 + k

template <int N>
__device__ __forceinline__ float2 twiddle(int k) { return c_tw[N * (N - 1) / 2 + k % N]; }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }

// v <- its DFT (natural order): 2 and 4 by butterflies, 3 and 5 by the symmetric and
// antisymmetric halves of each pair, 6 and 8 as 2 x 3 and 2 x 4
template <int R>
__device__ __forceinline__ void dft(float2 (&v)[R]) {
    if constexpr (R == 2) {
        const float2 a = v[0];
        v[0] = cadd(a, v[1]);
        v[1] = csub(a, v[1]);
    } else if constexpr (R == 4) {
        const float2 a = cadd(v[0], v[2]), b = csub(v[0], v[2]), c = cadd(v[1], v[3]), d = csub(v[1], v[3]);
        v[0] = cadd(a, c);
        v[2] = csub(a, c);
        v[1] = make_float2(b.x + d.y, b.y - d.x);  // b - i d
        v[3] = make_float2(b.x - d.y, b.y + d.x);
    } else if constexpr (R == 3 || R == 5) {
        constexpr int H = R / 2;
        float2 s[H], d[H], o[R];
        o[0] = v[0];
#pragma unroll
        for (int j = 0; j < H; ++j) {
            s[j] = cadd(v[j + 1], v[R - 1 - j]);
            d[j] = csub(v[j + 1], v[R - 1 - j]);
            o[0] = cadd(o[0], s[j]);
        }
#pragma unroll
        for (int k = 1; k <= H; ++k) {
            float2 e = v[0], f = make_float2(0.f, 0.f);  // e + (+-)i f
#pragma unroll
            for (int j = 0; j < H; ++j) {
                const float2 w = twiddle<R>(k * (j + 1));  // (cos, -sin)
                e.x = fmaf(w.x, s[j].x, e.x);
                e.y = fmaf(w.x, s[j].y, e.y);
                f.x = fmaf(w.y, d[j].x, f.x);
                f.y = fmaf(w.y, d[j].y, f.y);
            }
            o[k] = make_float2(e.x - f.y, e.y + f.x);
            o[R - k] = make_float2(e.x + f.y, e.y - f.x);
        }
#pragma unroll
        for (int k = 0; k < R; ++k) v[k] = o[k];
    } else if constexpr (R == 6 || R == 8) {
        constexpr int B = R / 2;
        float2 lo[B], hi[B];
#pragma unroll
        for (int b = 0; b < B; ++b) {
            lo[b] = cadd(v[b], v[b + B]);
            hi[b] = cmul(csub(v[b], v[b + B]), twiddle<R>(b));
        }
        dft<B>(lo);
        dft<B>(hi);
#pragma unroll
        for (int b = 0; b < B; ++b) {
            v[2 * b] = lo[b];
            v[2 * b + 1] = hi[b];
        }
    }
}

template <int N>
__host__ __device__ constexpr int fft_a() {  // first factor of N
    return N == 6 ? 2 : N == 8 ? 2 : N == 10 ? 2 : N == 12 ? 3 : N == 15 ? 3 : N == 18 ? 3 : N == 20 ? 4 : N == 24 ? 4 : N == 25 ? 5 : N == 30 ? 5 : N == 32 ? 4 : 6;
}

template <int N>
__device__ __forceinline__ void fft_line(float2 (&x)[N]) {
    constexpr int A = fft_a<N>(), B = N / A;
    static_assert(A * B == N && B <= 8, "line length");
#pragma unroll
    for (int b = 0; b < B; ++b) {
        float2 t[A];
#pragma unroll
        for (int a = 0; a < A; ++a) t[a] = x[B * a + b];
        dft<A>(t);
#pragma unroll
        for (int a = 0; a < A; ++a) x[B * a + b] = (a && b) ? cmul(t[a], twiddle<N>(a * b)) : t[a];
    }
    float2 o[N];
#pragma unroll
    for (int a = 0; a < A; ++a) {
        float2 t[B];
#pragma unroll
        for (int b = 0; b < B; ++b) t[b] = x[B * a + b];
        dft<B>(t);
#pragma unroll
        for (int b = 0; b < B; ++b) o[a + A * b] = t[b];
    }
#pragma unroll
    for (int k = 0; k < N; ++k) x[k] = o[k];
}
__device__ __forceinline__ float2 swapped(float2 v) { return make_float2(v.y, v.x); }

// Threads per CTA: 256 while two CTAs share an SM (128 registers a thread either way), 512
// once the grid leaves room for one; small grids have fewer lines than that.
template <int N>
__host__ __device__ constexpr int cube_threads() { return N <= 8 ? 64 : N <= 12 ? 128 : N <= 30 ? 256 : 512; }
template <int N>
constexpr size_t cube_smem(int K) { return sizeof(float2) * (size_t)(N | 1) * N * K; }

// One direction i and right-hand side r: the spectra of every group scattered into a K^3
// corner of the N^3 grid, transformed, multiplied by That[i], transformed back and gathered,
// first component 0, then 1.  Both ends of the convolution live in the corner, so the lines
// are pruned: x lines of K x K, y lines of N x K and z lines of N x N, the z line going
// forward, through the product and back without leaving registers, and shared memory holds
// N x N x K points (rows padded to an odd length against bank conflicts in the x lines).
// Inverse transforms are forward ones with real and imaginary parts swapped before and after.
// What bounds it: issue and shared-memory passes on the SM, with That (the only large stream,
// N^3 per direction) pulled into L2 meanwhile.  30^3 grid, 3200 directions, 1034 groups: cuFFT's
// six passes over a 1.38 GB array, scatter, product and gather took 4.40 ms; this 0.65 ms
// (0.73 GB, 0.11 ms at the copy rate).
template <int N>
__global__ void __launch_bounds__(cube_threads<N>(), N <= 30 ? 2 : 1)
    cube_translate_kernel(const float2* __restrict__ spec, const int* __restrict__ cells,
                          const float2* __restrict__ That, int G, int n_dir, int K, int R, float scale,
                          float2* __restrict__ out) {
    constexpr int LD = N | 1, NT = cube_threads<N>();
    extern __shared__ float2 g[];  // [z < K][y < N][x < LD]
    const int i = blockIdx.x / R, r = blockIdx.x % R, tid = threadIdx.x;
    const float2* T = That + (int64_t)i * (N * N * N);
    if (tid == 0) {
        const uint32_t bytes = (uint32_t)(sizeof(float2) * N * N * N) & ~15u;
        const char* p = reinterpret_cast<const char*>(T);
        p -= reinterpret_cast<uintptr_t>(p) & 15;  // inside the same allocation
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
    }
    for (int alpha = 0; alpha < 2; ++alpha) {
        const int64_t j = (int64_t)r * G * 2 * n_dir + (int64_t)alpha * n_dir + i;
        for (int e = tid; e < K * K * K; e += NT) {
            const int x = e % K, q = e / K;
            g[x + LD * (q % K + N * (q / K))] = make_float2(0.f, 0.f);
        }
        __syncthreads();
        for (int v = tid; v < G; v += NT) g[cells[v]] = spec[j + (int64_t)v * 2 * n_dir];
        __syncthreads();
        for (int e = tid; e < K * K; e += NT) {  // x lines
            float2* p = g + LD * (e % K + N * (e / K));
            float2 x[N];
#pragma unroll
            for (int k = 0; k < N; ++k) x[k] = k < K ? p[k] : make_float2(0.f, 0.f);
            fft_line<N>(x);
#pragma unroll
            for (int k = 0; k < N; ++k) p[k] = x[k];
        }
        __syncthreads();
        for (int e = tid; e < N * K; e += NT) {  // y lines
            float2* p = g + e % N + LD * N * (e / N);
            float2 x[N];
#pragma unroll
            for (int k = 0; k < N; ++k) x[k] = k < K ? p[LD * k] : make_float2(0.f, 0.f);
            fft_line<N>(x);
#pragma unroll
            for (int k = 0; k < N; ++k) p[LD * k] = x[k];
        }
        __syncthreads();
        for (int e = tid; e < N * N; e += NT) {  // z lines: forward, product, back
            float2* p = g + e % N + LD * (e / N);
            float2 x[N];
#pragma unroll
            for (int k = 0; k < N; ++k) x[k] = k < K ? p[LD * N * k] : make_float2(0.f, 0.f);
            fft_line<N>(x);
#pragma unroll
            for (int k = 0; k < N; ++k) x[k] = swapped(cmul(x[k], __ldg(T + e + N * N * k)));
            fft_line<N>(x);
#pragma unroll
            for (int k = 0; k < N; ++k)
                if (k < K) p[LD * N * k] = x[k];  // stays swapped through the y and x lines
        }
        __syncthreads();
        for (int e = tid; e < N * K; e += NT) {
            float2* p = g + e % N + LD * N * (e / N);
            float2 x[N];
#pragma unroll
            for (int k = 0; k < N; ++k) x[k] = p[LD * k];
            fft_line<N>(x);
#pragma unroll
            for (int k = 0; k < N; ++k)
                if (k < K) p[LD * k] = x[k];
        }
        __syncthreads();
        for (int e = tid; e < K * K; e += NT) {
            float2* p = g + LD * (e % K + N * (e / K));
            float2 x[N];
#pragma unroll
            for (int k = 0; k < N; ++k) x[k] = p[k];
            fft_line<N>(x);
#pragma unroll
            for (int k = 0; k < N; ++k)
                if (k < K) p[k] = x[k];
        }
        __syncthreads();
        for (int v = tid; v < G; v += NT) {
            const float2 u = g[cells[v]];
            out[j + (int64_t)v * 2 * n_dir] = make_float2(scale * u.y, scale * u.x);
        }
        __syncthreads();
    }
}

// Calls f(std::integral_constant<int, N>) for a cube size N.
template <class F>
void with_cube_size(int n, F&& f) {
    switch (n) {
#define TFMM_CUBE(N) case N: f(std::integral_constant<int, N>{}); break;
        TFMM_CUBE(6) TFMM_CUBE(8) TFMM_CUBE(10) TFMM_CUBE(12) TFMM_CUBE(15) TFMM_CUBE(18) TFMM_CUBE(20)
        TFMM_CUBE(24) TFMM_CUBE(25) TFMM_CUBE(30) TFMM_CUBE(32) TFMM_CUBE(36)
#undef TFMM_CUBE
        default: fail(TFMM_CUDA, "no cube kernel of this size");
    }
}

int grid_blocks(int64_t total) { return (int)std::max<int64_t>(1, std::min<int64_t>((total + 255) / 256, 152 * 64)); }

// smallest n >= m whose prime factors are 2, 3, 5 or 7 (fast cuFFT sizes)
int fft_size(int m) {
    for (int n = std::max(m, 1);; ++n) {
        int v = n;
        for (int p : {2, 3, 5, 7})
            while (v % p == 0) v /= p;
        if (v == 1) return n;
    }
}

}  // namespace

TransPlan::~TransPlan() {
    if (fft) cufftDestroy((cufftHandle)fft);
}

void build_translation(Plan& P, cudaStream_t s) {
    if (P.trans) return;
    TFMM_REQUIRE(P.has_geometry && !P.centres.empty(), "translation needs box centres: a plan made by tfmm_plan_create");
    TFMM_REQUIRE(P.L <= kMaxL, "bandwidth L too large for the translation kernel");
    auto T = std::make_unique<TransPlan>();
    const double a = P.params.box;
    // integer box coordinates relative to the lowest centre (differences are what matter)
    double lo[3] = {INFINITY, INFINITY, INFINITY};
    for (int g = 0; g < P.G; ++g)
        for (int c = 0; c < 3; ++c) lo[c] = std::min(lo[c], P.centres[3 * (size_t)g + c]);
    std::vector<int> bi((size_t)P.G * 3);
    int K[3] = {1, 1, 1};
    for (int g = 0; g < P.G; ++g)
        for (int c = 0; c < 3; ++c) {
            const int v = (int)std::lround((P.centres[3 * (size_t)g + c] - lo[c]) / a);
            bi[3 * (size_t)g + c] = v;
            K[c] = std::max(K[c], v + 1);
        }
    for (int c = 0; c < 3; ++c) T->N[c] = fft_size(2 * K[c] - 1);
    // The cube kernel runs N^3 lines whatever the grid: taken while the cube is at most twice the
    // grid cuFFT would transform (a sphere's or a trihedral's box grid is a cube already; a plate's is
    // not, and cuFFT's passes over the smaller grid win there) and the corner fits shared memory.
    const int Kmax = std::max(K[0], std::max(K[1], K[2]));
    int cube = 0;
    for (int n : kCubeSizes)
        if (!cube && n >= 2 * Kmax - 1) cube = n;
    if (cube && (int64_t)cube * cube * cube <= 2 * (int64_t)T->N[0] * T->N[1] * T->N[2]) {
        int dev = 0, opt_in = 0;
        TFMM_CUDA_CHECK(cudaGetDevice(&dev));
        TFMM_CUDA_CHECK(cudaDeviceGetAttribute(&opt_in, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
        with_cube_size(cube, [&](auto n) {
            constexpr int N = decltype(n)::value;
            if (cube_smem<N>(Kmax) > (size_t)opt_in) return;
            // the most this device allows: another plan may run the same side with a larger corner
            TFMM_CUDA_CHECK(cudaFuncSetAttribute(cube_translate_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 opt_in));
            T->cube = N;
            T->K = Kmax;
        });
    }
    if (T->cube) {
        for (int c = 0; c < 3; ++c) T->N[c] = T->cube;
        std::vector<float2> tw((size_t)kCubeMax * (kCubeMax + 1) / 2);
        for (int n = 1; n <= kCubeMax; ++n)
            for (int k = 0; k < n; ++k) {
                const double t = 2.0 * 3.14159265358979323846 * k / n;
                tw[(size_t)n * (n - 1) / 2 + k] = make_float2((float)std::cos(t), (float)-std::sin(t));
            }
        TFMM_CUDA_CHECK(cudaMemcpyToSymbolAsync(c_tw, tw.data(), sizeof(float2) * tw.size(), 0, cudaMemcpyHostToDevice, s));
        TFMM_CUDA_CHECK(cudaStreamSynchronize(s));
    }
    T->Ns = (int64_t)T->N[0] * T->N[1] * T->N[2];
    const int nd = P.n_dir;
    T->nb = 2 * nd;
    std::vector<int> group_cell(P.G);
    for (int g = 0; g < P.G; ++g) {
        const int64_t row = T->cube ? T->cube | 1 : T->N[0];  // the cube kernel pads its rows
        const int64_t cell = bi[3 * (size_t)g] + row * (bi[3 * (size_t)g + 1] + (int64_t)T->N[1] * bi[3 * (size_t)g + 2]);
        group_cell[g] = (int)cell;
    }
    TFMM_CUDA_CHECK(device_malloc(&T->group_cell.p, sizeof(int) * std::max(P.G, 1)));
    TFMM_CUDA_CHECK(cudaMemcpy(T->group_cell.p, group_cell.data(), sizeof(int) * P.G, cudaMemcpyHostToDevice));
    // directions k_i
    std::vector<double> kh((size_t)nd * 3);
    for (int ip = 0; ip < P.n_phi; ++ip)
        for (int it = 0; it < P.n_theta; ++it) {
            const double t = P.theta[it], ph = P.phi[ip];
            double* d = &kh[3 * ((size_t)it + (size_t)P.n_theta * ip)];
            d[0] = std::sin(t) * std::cos(ph);
            d[1] = std::sin(t) * std::sin(ph);
            d[2] = std::cos(t);
        }
    {
        DeviceBuffer d_kh, d_T;
        TFMM_CUDA_CHECK(device_malloc(&d_kh.p, sizeof(double) * kh.size()));
        TFMM_CUDA_CHECK(cudaMemcpy(d_kh.p, kh.data(), sizeof(double) * kh.size(), cudaMemcpyHostToDevice));
        TFMM_CUDA_CHECK(device_malloc(&d_T.p, sizeof(double2) * T->Ns * nd));
        translation_kernel<<<(unsigned)T->Ns, 128, 0, s>>>(static_cast<const double*>(d_kh.p), nd, P.L, P.k, a,
                                                           T->N[0], T->N[1], T->N[2], K[0], K[1], K[2], T->Ns,
                                                           static_cast<double2*>(d_T.p));
        TFMM_CUDA_CHECK(cudaGetLastError());
        // forward transform of every direction's kernel over the grid (FP64), then FP32
        int n[3] = {T->N[2], T->N[1], T->N[0]};
        cufftHandle h64 = 0;
        CUFFT_CHECK(cufftPlanMany(&h64, 3, n, n, 1, (int)T->Ns, n, 1, (int)T->Ns, CUFFT_Z2Z, nd));
        cufftSetStream(h64, s);
        const cufftResult r64 = cufftExecZ2Z(h64, static_cast<cufftDoubleComplex*>(d_T.p),
                                             static_cast<cufftDoubleComplex*>(d_T.p), CUFFT_FORWARD);
        cufftDestroy(h64);
        CUFFT_CHECK(r64);
        TFMM_CUDA_CHECK(device_malloc(&T->That.p, sizeof(float2) * T->Ns * nd));
        to_f32_kernel<<<grid_blocks(T->Ns * nd), 256, 0, s>>>(static_cast<const double2*>(d_T.p), T->Ns * nd,
                                                              static_cast<float2*>(T->That.p));
        TFMM_CUDA_CHECK(cudaGetLastError());
        TFMM_CUDA_CHECK(cudaStreamSynchronize(s));
    }
    if (T->cube) {
        P.trans = std::move(T);
        return;
    }
    TFMM_CUDA_CHECK(device_malloc(&T->grid.p, sizeof(float2) * T->Ns * T->nb));
    int n[3] = {T->N[2], T->N[1], T->N[0]};
    cufftHandle h = 0;
    CUFFT_CHECK(cufftPlanMany(&h, 3, n, n, 1, (int)T->Ns, n, 1, (int)T->Ns, CUFFT_C2C, T->nb));
    T->fft = (int)h;
    P.trans = std::move(T);
}

void launch_translate(Plan& P, const float2* spec_out, int R, float2* spec_in, cudaStream_t s) {
    build_translation(P, s);
    TransPlan& T = *P.trans;
    if (T.cube) {
        with_cube_size(T.cube, [&](auto n) {
            constexpr int N = decltype(n)::value;
            constexpr int kCols = 4096;  // right-hand sides per launch (the grid is directions x these)
            for (int r0 = 0; r0 < R; r0 += kCols) {
                const int nr = std::min(kCols, R - r0);
                const int64_t off = (int64_t)r0 * P.G * T.nb;
                cube_translate_kernel<N><<<(unsigned)P.n_dir * nr, cube_threads<N>(), cube_smem<N>(T.K), s>>>(
                    spec_out + off, static_cast<const int*>(T.group_cell.p), static_cast<const float2*>(T.That.p), P.G,
                    P.n_dir, T.K, nr, 1.0f / (float)T.Ns, spec_in + off);
            }
        });
        TFMM_CUDA_CHECK(cudaGetLastError());
        return;
    }
    float2* grid = static_cast<float2*>(T.grid.p);
    CUFFT_CHECK(cufftSetStream((cufftHandle)T.fft, s));
    for (int r = 0; r < R; ++r) {
        const int64_t off = (int64_t)r * P.G * T.nb;
        TFMM_CUDA_CHECK(cudaMemsetAsync(grid, 0, sizeof(float2) * T.Ns * T.nb, s));
        scatter_kernel<<<grid_blocks((int64_t)P.G * T.nb), 256, 0, s>>>(
            spec_out + off, static_cast<const int*>(T.group_cell.p), P.G, T.nb, T.Ns, grid);
        TFMM_CUDA_CHECK(cudaGetLastError());
        CUFFT_CHECK(cufftExecC2C((cufftHandle)T.fft, reinterpret_cast<cufftComplex*>(grid),
                                 reinterpret_cast<cufftComplex*>(grid), CUFFT_FORWARD));
        multiply_kernel<<<grid_blocks(T.Ns * T.nb), 256, 0, s>>>(grid, static_cast<const float2*>(T.That.p), T.Ns,
                                                                 P.n_dir);
        TFMM_CUDA_CHECK(cudaGetLastError());
        CUFFT_CHECK(cufftExecC2C((cufftHandle)T.fft, reinterpret_cast<cufftComplex*>(grid),
                                 reinterpret_cast<cufftComplex*>(grid), CUFFT_INVERSE));
        gather_kernel<<<grid_blocks((int64_t)P.G * T.nb), 256, 0, s>>>(
            grid, static_cast<const int*>(T.group_cell.p), P.G, T.nb, T.Ns, 1.0f / (float)T.Ns, spec_in + off);
        TFMM_CUDA_CHECK(cudaGetLastError());
    }
}

}  // namespace tfmm
