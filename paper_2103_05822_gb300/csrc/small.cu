// Aggregation and disaggregation of small groups (Figs. 2b, 3b), any number of right-hand
// sides, FP32 on CUDA cores: one CTA per (group, component) keeps all its factors and every
// intermediate in shared memory.
//
// Half-wavelength boxes give thousands of groups of about 60 RWGs whose factors are 40 to 90 KB.
// The persistent kernels stream such an item phase by phase, each phase waiting for the
// previous one's barrier and for its own first bytes, and the grouped-GEMM chain spends one
// launch per phase on 64 x 64 tiles that the ranks (9, 13, 35) leave mostly empty.  Here the
// four factors are requested at once (cp.async), a phase starts when its factor is there,
// and kCols columns at a time go through all phases; factors are read once for all columns.
// Every product is a register-tiled GEMM from shared memory (tile_gemm), with the contraction
// split over neighbouring lanes where a phase has fewer outputs than the CTA has threads.
// Bound: FP32 issue and shared-memory wavefronts, about one of each per four multiply-adds, at
// the half to two thirds of the issue slots that three CTAs' barriers leave.  20-lambda sphere in
// half-wavelength boxes (7240 groups, 16 columns, ranks to (9, 13, 35)): aggregation 3.59 -> 0.86 ms,
// disaggregation 4.01 -> 1.46 ms (0.18 ms each for the bytes).  One column of the 2-lambda sphere
// (56 groups), both stages in a graph: 25.9 -> 20.0 us.
#include <cooperative_groups.h>

#include <algorithm>
#include <numeric>

#include "internal.h"

namespace tfmm {

namespace {

namespace cg = cooperative_groups;

constexpr int kThreads = 256;
constexpr int kSpecCols = 4;  // columns of the spectra staged at once (disaggregation)

__device__ __forceinline__ void cfma(float2& acc, float2 a, float2 b) {
    acc.x = fmaf(a.x, b.x, acc.x);
    acc.x = fmaf(-a.y, b.y, acc.x);
    acc.y = fmaf(a.x, b.y, acc.y);
    acc.y = fmaf(a.y, b.x, acc.y);
}

// Division of indexes below 2^16 by a size below 2^16 through the high half of a product (the
// run-time divisions of the staging loops and of the outputs' indexes cost as much issue as the
// multiply-adds of these short contractions).
struct FastDiv {
    uint32_t d, m;
    __host__ __device__ FastDiv() : d(1), m(0) {}
    __host__ __device__ explicit FastDiv(int n) : d((uint32_t)n), m(0xffffffffu / (uint32_t)n + 1u) {}
    __device__ __forceinline__ int div(int e) const { return d == 1 ? e : (int)__umulhi((uint32_t)e, m); }
    __device__ __forceinline__ int mod(int e, int q) const { return e - q * (int)d; }
};

// Requests n complex elements (rounded up to 16 bytes; the packed factors are zero-padded) as
// one cp.async group.
__device__ __forceinline__ void fetch(float2* dst, const float2* src, int n) {
    for (int e = 2 * (int)threadIdx.x; e < n; e += 2 * kThreads)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst + e)),
                     "l"(src + e));
    asm volatile("cp.async.commit_group;");
}
// Rows of U_beta^T and C_(3) sit smem_ld(ld) apart: the long contractions read four rows by four
// neighbouring columns per half warp, and a row length of 4 modulo 8 puts those 16 words (8 bytes
// each) into different banks; at 96 or 64, the lengths that occur, they took eight turns.
__host__ __device__ __forceinline__ int smem_ld(int ld) { return ((ld + 3) & ~7) + 4; }
__device__ __forceinline__ void fetch_rows(float2* dst, const float2* src, int rows, int ld) {
    const int h = ld / 2, lds = smem_ld(ld);
    const FastDiv by_h(h);
    for (int e = threadIdx.x; e < rows * h; e += kThreads) {
        const int r = by_h.div(e), c = by_h.mod(e, r);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(dst + r * lds + 2 * c)),
                     "l"(src + 2 * e));
    }
    asm volatile("cp.async.commit_group;");
}
template <int LEFT>
__device__ __forceinline__ void fetched() {  // all but the last LEFT groups are in shared memory
    asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
    __syncthreads();
}

// C(m, n) = sum_{k < K} a(m, k) b(k, n): every thread holds a TM x TN block of outputs with
// rows and columns mt and nt apart (so that lanes read neighbouring rows), KS neighbouring
// lanes share a block's k and add up by shuffles.  emit(m, n, v) once per output.
template <int TM, int TN, int KS, class LA, class LB, class Emit>
__device__ __forceinline__ void tile_gemm(int M, int N, int K, LA a, LB b, Emit emit) {
    const int mt = (M + TM - 1) / TM, nt = (N + TN - 1) / TN, tasks = mt * nt * KS;
    const FastDiv by_mt(mt);
    for (int t = threadIdx.x; t < ((tasks + 31) & ~31); t += kThreads) {  // whole warps: shuffles below
        const bool live = t < tasks;
        const int k0 = t % KS, u = live ? t / KS : 0, n0 = by_mt.div(u), m0 = by_mt.mod(u, n0);
        float2 acc[TM][TN];
        int mi[TM], nj[TN];
#pragma unroll
        for (int i = 0; i < TM; ++i) mi[i] = min(m0 + i * mt, M - 1);
#pragma unroll
        for (int j = 0; j < TN; ++j) nj[j] = min(n0 + j * nt, N - 1);
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) acc[i][j] = make_float2(0.f, 0.f);
        if constexpr (TM * TN == 1) {
            // One output a thread: two sums side by side.  With one, the 2-lambda sphere's error against 64 bits
            // was 2.1e-7 instead of 1.7e-7 (and its captured matvec 18.4 us instead of 19.2).
            float2 odd = make_float2(0.f, 0.f);
#pragma unroll 2
            for (int k = k0; k < K; k += 2 * KS) {
                cfma(acc[0][0], a(mi[0], k), b(k, nj[0]));
                if (k + KS < K) cfma(odd, a(mi[0], k + KS), b(k + KS, nj[0]));
            }
            acc[0][0].x += odd.x;
            acc[0][0].y += odd.y;
        } else {
#pragma unroll 4
            for (int k = k0; k < K; k += KS) {
                float2 av[TM], bv[TN];
#pragma unroll
                for (int i = 0; i < TM; ++i) av[i] = a(mi[i], k);
#pragma unroll
                for (int j = 0; j < TN; ++j) bv[j] = b(k, nj[j]);
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < TN; ++j) cfma(acc[i][j], av[i], bv[j]);
            }
        }
#pragma unroll
        for (int o = KS / 2; o > 0; o >>= 1)
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    acc[i][j].x += __shfl_xor_sync(0xffffffffu, acc[i][j].x, o);
                    acc[i][j].y += __shfl_xor_sync(0xffffffffu, acc[i][j].y, o);
                }
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j)
                if (live && (i * TN + j) % KS == k0 && m0 + i * mt < M && n0 + j * nt < N)
                    emit(m0 + i * mt, n0 + j * nt, acc[i][j]);
    }
}

// Tiles of the phases for one column and for a block of columns.
template <int COLS>
struct Tile {
    static constexpr int TM = 2, TN = 4, KS_LONG = 4, KS_SHORT = 1;  // long: K = n_beta, r_theta r_phi
};
template <>
struct Tile<1> {
    static constexpr int TM = 1, TN = 1, KS_LONG = 8, KS_SHORT = 2;
};
// stride of the column index in X, T, M, H, S and y: odd, so that columns of neighbouring rows
// fall into different banks
template <int COLS>
__host__ __device__ constexpr int col_ld() { return COLS == 1 ? 1 : COLS + 1; }

struct SmallArgs {
    const TuckerItem* items;
    const int* order;     // this launch's groups
    const float2* fac;
    const int* grp_rwg;
    const float2* x;      // aggregation input
    const float* w;       // disaggregation weights or null
    const float2* spec_in;
    float2* spec;         // aggregation output
    float2* y;            // disaggregation output
    int64_t ld;
    float2 beta;
    int n_theta, n_phi, n_dir, G, R;
    FastDiv by_theta, by_phi, by_dir;
    int o_work;           // complex elements of the largest item's factors
    int o_a, o_b, o_c, o_d;  // regions of the work area behind them
};

struct SmallFactors {
    float2 *ub, *core, *uphi, *uth;
};
__device__ __forceinline__ int even(int n) { return (n + 1) & ~1; }
__device__ __forceinline__ SmallFactors carve(float2* sm, const TuckerItem& d, int n_phi) {
    SmallFactors f;
    f.ub = sm;
    f.core = f.ub + d.rb * smem_ld(d.ld_nb);
    f.uphi = f.core + d.rb * smem_ld(d.ld_ab);
    f.uth = f.uphi + even(n_phi * d.rp);
    return f;
}

// One (group, component) per CTA: T = U_beta^T X, M = C_(3)^T T, V = U_phi M', F = U_theta V'.
template <int COLS>
__global__ void __launch_bounds__(kThreads) small_aggregate_kernel(const __grid_constant__ SmallArgs a) {
    constexpr int LC = col_ld<COLS>();
    using L = Tile<COLS>;
    extern __shared__ float4 smem4[];
    float2* sm = reinterpret_cast<float2*>(smem4);
    const TuckerItem d = a.items[2 * a.order[blockIdx.x / 2] + (blockIdx.x & 1)];
    const SmallFactors f = carve(sm, d, a.n_phi);
    fetch_rows(f.ub, a.fac + d.ub, d.rb, d.ld_nb);
    fetch_rows(f.core, a.fac + d.core, d.rb, d.ld_ab);
    fetch(f.uphi, a.fac + d.uphi, a.n_phi * d.rp);
    fetch(f.uth, a.fac + d.uth, a.n_theta * d.rt);
    float2* sM = sm + a.o_work + a.o_a;  // [a + r_t b][col]
    float2* sX = sm + a.o_work + a.o_b;  // [n][col]; V over X and T once they are used
    float2* sT = sm + a.o_work + a.o_c;  // [c][col]
    float2* sV = sX;                     // [a][i_phi + n_phi col]
    const int rt = d.rt, np = a.n_phi, nt = a.n_theta, ldn = smem_ld(d.ld_nb), lda = smem_ld(d.ld_ab);
    const FastDiv by_beta(d.n_beta);
    for (int r0 = 0; r0 < a.R; r0 += COLS) {
        const int nc = min(COLS, a.R - r0);
        for (int e = threadIdx.x; e < d.n_beta * COLS; e += kThreads) {
            const int c = by_beta.div(e), n = by_beta.mod(e, c);
            sX[n * LC + c] = c < nc ? a.x[(int64_t)a.grp_rwg[d.rwg + n] + a.ld * (r0 + c)] : make_float2(0.f, 0.f);
        }
        fetched<3>();
        tile_gemm<L::TM, L::TN, L::KS_LONG>(
            d.rb, COLS, d.n_beta, [&](int c, int n) { return f.ub[c * ldn + n]; },
            [&](int n, int r) { return sX[n * LC + r]; }, [&](int c, int r, float2 v) { sT[c * LC + r] = v; });
        fetched<2>();
        tile_gemm<L::TM, L::TN, L::KS_SHORT>(
            rt * d.rp, COLS, d.rb, [&](int ab, int c) { return f.core[c * lda + ab]; },
            [&](int c, int r) { return sT[c * LC + r]; }, [&](int ab, int r, float2 v) { sM[ab * LC + r] = v; });
        fetched<1>();
        tile_gemm<L::TM, L::TN, 1>(
            np, rt * COLS, d.rp, [&](int ip, int b) { return f.uphi[ip + np * b]; },
            [&](int b, int n) { return sM[(n / COLS + rt * b) * LC + n % COLS]; },
            [&](int ip, int n, float2 v) { sV[(n / COLS) * (np * COLS) + ip + np * (n % COLS)] = v; });
        fetched<0>();
        float2* out = a.spec + (((int64_t)r0 * a.G + d.g) * 2 + d.alpha) * a.n_dir;
        const int64_t rs = (int64_t)a.G * 2 * a.n_dir;
        tile_gemm<L::TM, L::TN, 1>(
            nt, np * nc, rt, [&](int it, int aa) { return f.uth[it + nt * aa]; },
            [&](int aa, int n) { return sV[aa * (np * COLS) + n]; },
            [&](int it, int n, float2 v) {
                const int r = a.by_phi.div(n);
                out[it + nt * a.by_phi.mod(n, r) + rs * r] = v;
            });
        __syncthreads();
    }
}

// One group per cluster of two CTAs, one component each: P = U_theta^T conj(W g), H = P U_phi,
// S = C_(3) H, then U_beta S; the two parts of y_g meet through distributed shared memory, each
// CTA finishing half of the group's RWGs.
template <int COLS>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 3)
    small_disaggregate_kernel(const __grid_constant__ SmallArgs a) {
    constexpr int LC = col_ld<COLS>(), SC = COLS < kSpecCols ? COLS : kSpecCols, LS = col_ld<SC>();
    using L = Tile<COLS>;
    extern __shared__ float4 smem4[];
    float2* sm = reinterpret_cast<float2*>(smem4);
    cg::cluster_group cluster = cg::this_cluster();
    const int half = (int)cluster.block_rank();
    const TuckerItem d = a.items[2 * a.order[blockIdx.x / 2] + half];
    const SmallFactors f = carve(sm, d, a.n_phi);
    fetch(f.uth, a.fac + d.uth, a.n_theta * d.rt);
    fetch(f.uphi, a.fac + d.uphi, a.n_phi * d.rp);
    fetch_rows(f.core, a.fac + d.core, d.rb, d.ld_ab);
    fetch_rows(f.ub, a.fac + d.ub, d.rb, d.ld_nb);
    float2* sH = sm + a.o_work + a.o_a;  // [a + r_t b][col]
    float2* sS = sm + a.o_work + a.o_b;  // [c][col]
    float2* sP = sm + a.o_work + a.o_c;  // [i_phi][a][SC columns], then conj(W g) of these columns
    float2* sG = sP + a.n_phi * d.rt * LS;
    float2* sy = sP;                     // y_g [n][col] over both
    const int rt = d.rt, np = a.n_phi, nt = a.n_theta, ldn = smem_ld(d.ld_nb), lda = smem_ld(d.ld_ab);
    const int ldg = nt | 1;
    const float2* spec = a.spec_in + ((int64_t)d.g * 2 + d.alpha) * a.n_dir;
    const int64_t rs = (int64_t)a.G * 2 * a.n_dir;
    const int mid = d.n_beta / 2, n0 = half ? mid : 0, cnt = half ? d.n_beta - mid : mid;
    int* ids = reinterpret_cast<int*>(sm + a.o_work + a.o_d);
    for (int n = threadIdx.x; n < cnt; n += kThreads) ids[n] = a.grp_rwg[d.rwg + n0 + n];
    const FastDiv by_cnt(max(cnt, 1));
    for (int r0 = 0; r0 < a.R; r0 += COLS) {
        const int nc = min(COLS, a.R - r0);
        for (int s0 = 0; s0 < COLS; s0 += SC) {
            for (int e = threadIdx.x; e < a.n_dir * SC; e += kThreads) {
                const int c = a.by_dir.div(e), i = a.by_dir.mod(e, c), ip = a.by_theta.div(i);
                float2 v = make_float2(0.f, 0.f);
                if (s0 + c < nc) {
                    const float2 g = spec[rs * (r0 + s0 + c) + i];
                    const float wt = a.w ? a.w[i] : 1.0f;
                    v = make_float2(wt * g.x, -wt * g.y);
                }
                sG[(c * np + ip) * ldg + a.by_theta.mod(i, ip)] = v;
            }
            fetched<3>();
            tile_gemm<L::TM, L::TN, 1>(
                np * SC, rt, nt, [&](int m, int it) { return sG[m * ldg + it]; },
                [&](int it, int aa) { return f.uth[it + nt * aa]; },
                [&](int m, int aa, float2 v) {
                    const int c = a.by_phi.div(m);
                    sP[(a.by_phi.mod(m, c) * rt + aa) * LS + c] = v;
                });
            fetched<2>();
            tile_gemm<L::TM, L::TN, L::KS_LONG>(
                rt * SC, d.rp, np, [&](int m, int ip) { return sP[(ip * rt + m / SC) * LS + m % SC]; },
                [&](int ip, int b) { return f.uphi[ip + np * b]; },
                [&](int m, int b, float2 v) { sH[(m / SC + rt * b) * LC + s0 + m % SC] = v; });
            __syncthreads();
        }
        fetched<1>();
        tile_gemm<L::TM, L::TN, L::KS_LONG>(
            d.rb, COLS, rt * d.rp, [&](int c, int ab) { return f.core[c * lda + ab]; },
            [&](int ab, int r) { return sH[ab * LC + r]; }, [&](int c, int r, float2 v) { sS[c * LC + r] = v; });
        fetched<0>();
        tile_gemm<L::TM, L::TN, L::KS_SHORT>(
            d.n_beta, COLS, d.rb, [&](int n, int c) { return f.ub[c * ldn + n]; },
            [&](int c, int r) { return sS[c * LC + r]; }, [&](int n, int r, float2 v) { sy[n * LC + r] = v; });
        cluster.sync();
        const float2* other = cluster.map_shared_rank(sy, half ^ 1);
        for (int e = threadIdx.x; e < cnt * nc; e += kThreads) {
            const int c = by_cnt.div(e), i = by_cnt.mod(e, c), n = n0 + i;
            const float2 p = sy[n * LC + c], q = other[n * LC + c];
            float2 v = make_float2(p.x + q.x, -(p.y + q.y));
            float2* dst = a.y + ids[i] + a.ld * (r0 + c);
            if (a.beta.x != 0.f || a.beta.y != 0.f) {
                const float2 old = *dst;
                v.x += a.beta.x * old.x - a.beta.y * old.y;
                v.y += a.beta.x * old.y + a.beta.y * old.x;
            }
            *dst = v;
        }
        cluster.sync();  // the other CTA has read this one's part
    }
}

int even_host(int n) { return (n + 1) & ~1; }

// Work regions (complex elements) of one pass over `cols` columns and the total with the factors.
struct SmallLayout {
    int a, b, c, d, total;
};
SmallLayout agg_work(const Plan& P, const SmallClass& k, int cols) {
    const int lc = cols == 1 ? 1 : cols + 1;
    SmallLayout l{};
    l.b = even_host(k.max_m * lc);
    l.c = l.b + even_host(k.max_nb * lc);
    l.total = std::max(l.c + k.max_rb * lc, l.b + k.max_rt * P.n_phi * cols);
    l.total = even_host(l.total) + k.elems;
    return l;
}
SmallLayout dis_work(const Plan& P, const SmallClass& k, int cols) {
    const int lc = cols == 1 ? 1 : cols + 1, sc = std::min(cols, kSpecCols);
    SmallLayout l{};
    l.b = even_host(k.max_m * lc);
    l.c = l.b + even_host(k.max_rb * lc);
    const int ls = sc == 1 ? 1 : sc + 1;
    l.d = l.c + even_host(std::max(P.n_phi * k.max_rt * ls + sc * P.n_phi * (P.n_theta | 1), k.max_nb * lc));
    l.total = l.d + even_host(k.max_nb / 4 + 1) + k.elems;  // RWG ids of half a group, two per element
    return l;
}

constexpr int kClasses = 4;
constexpr int kBlocks[] = {16, 8, 4, 1};  // columns per pass
// dynamic shared memory of which three, two CTAs fit an SM
constexpr size_t kThirdSM = 75 * 1024, kHalfSM = 113 * 1024;

template <class F>
void with_cols(int cols, F&& f) {
    switch (cols) {
        case 16: f(std::integral_constant<int, 16>{}); break;
        case 8: f(std::integral_constant<int, 8>{}); break;
        case 4: f(std::integral_constant<int, 4>{}); break;
        default: f(std::integral_constant<int, 1>{}); break;
    }
}

// Columns per pass: the most, up to R, with which three CTAs fit an SM, else two, else one.
struct SmallPass {
    int cols, per_sm;
};
template <class Work>
SmallPass pick_pass(const Plan& P, const SmallClass& k, int R, Work work) {
    if (R == 1 || P.params.mrhs_precision == 1) return {1, 1};  // 1: every column as a call of its own
    const size_t room[3] = {kThirdSM, kHalfSM, P.small_room};
    for (int i = 0; i < 3; ++i)
        for (int c : kBlocks)
            if ((c < 2 * R || c == 4) && c > 1 && sizeof(float2) * work(P, k, c).total <= room[i]) return {c, 3 - i};
    return {1, 1};
}

// Columns in blocks pay where a pass takes four at least: with one, a pass costs as much as a column of
// the persistent kernels and more.  Past 48 columns the passes of one CTA also lose to the chain where
// the CTAs do not fill the SMs, or where four columns fill an SM's shared memory.  Measured (us, this /
// chain), one column a pass: 300 groups of 200 KB disaggregation, 16 columns 567 / 264, 100 3446 / 1325;
// 40 groups of 54 KB, 48 columns 68 + 77 / 60 + 77, 100 136 + 169 / 93 + 110 (110 groups 181 + 229 /
// 207 + 239); four columns to an SM: 80 groups of 198 KB aggregation, 12 columns 71 / 75, 48 257 / 205, 100
// 560 / 361, 400 of 161 KB disaggregation, 8 columns 252 / 250, 48 1392 / 975, 100 2884 / 1886.
template <class Work>
bool blocks_pay(const Plan& P, int R, Work work) {
    for (const SmallClass& k : P.small_classes) {
        const SmallPass p = pick_pass(P, k, R, work);
        if (p.cols == 1) return false;
        if (R > 48 && (2 * P.G <= P.num_sms || (p.cols <= 4 && p.per_sm == 1))) return false;
    }
    return true;
}

SmallArgs small_args(const Plan& P, const SmallClass& k, int R, const SmallLayout& l) {
    SmallArgs a{};
    a.items = P.d_items;
    a.order = static_cast<const int*>(P.small_order.p) + k.first;
    a.fac = P.d_factors;
    a.grp_rwg = P.d_grp_rwg;
    a.n_theta = P.n_theta;
    a.n_phi = P.n_phi;
    a.n_dir = P.n_dir;
    a.by_theta = FastDiv(P.n_theta);
    a.by_phi = FastDiv(P.n_phi);
    a.by_dir = FastDiv(P.n_dir);
    a.G = P.G;
    a.R = R;
    a.o_work = k.elems;
    a.o_a = l.a;
    a.o_b = l.b;
    a.o_c = l.c;
    a.o_d = l.d;
    return a;
}

}  // namespace

void configure_small(Plan& P, cudaStream_t s) {
    P.small_ok = P.small_one = false;
    P.small_classes.clear();
    if (plan_is_svd(P)) return;
    int dev = 0, opt_in = 0;
    TFMM_CUDA_CHECK(cudaGetDevice(&dev));
    TFMM_CUDA_CHECK(cudaDeviceGetAttribute(&opt_in, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    P.small_room = (size_t)opt_in;
    std::vector<int64_t> need(P.G, 0);  // factors of the larger component
    for (const TuckerItem& d : P.items)
        need[d.g] = std::max<int64_t>(need[d.g], (int64_t)d.rb * (smem_ld(d.ld_nb) + smem_ld(d.ld_ab)) +
                                                     even_host(P.n_phi * d.rp) +
                                                     even_host(P.n_theta * d.rt));
    std::vector<int> order(P.G);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return need[a] > need[b]; });
    if (need[order[0]] * (int64_t)sizeof(float2) > opt_in) return;
    // FastDiv's range: the largest index (columns x directions or RWGs, or a phase's tasks)
    if ((int64_t)kBlocks[0] * std::max({P.n_dir, P.max_nb, P.max_rank[0] * P.n_phi}) > 65535) return;
    // A launch's CTAs all get the shared memory its largest item needs.  Plans with many groups
    // launch kClasses size classes, largest first, so that the smaller items run more columns per
    // pass and more CTAs per SM (7240 groups x 16 columns, one class / four: aggregation 0.86 / 0.84 ms,
    // disaggregation 1.67 / 1.62 ms when it was brought in).
    const int n = P.G >= 4 * P.num_sms ? kClasses : 1;
    for (int c = 0; c < n; ++c) {
        SmallClass k;
        k.first = (int)((int64_t)P.G * c / n);
        k.groups = (int)((int64_t)P.G * (c + 1) / n) - k.first;
        k.elems = (int)need[order[k.first]];
        for (int i = k.first; i < k.first + k.groups; ++i)
            for (int al = 0; al < 2; ++al) {
                const TuckerItem& d = P.items[2 * (size_t)order[i] + al];
                k.max_nb = std::max(k.max_nb, d.n_beta);
                k.max_rt = std::max(k.max_rt, d.rt);
                k.max_rb = std::max(k.max_rb, d.rb);
                k.max_m = std::max(k.max_m, d.rt * d.rp);
            }
        // one column at a time is the least either stage needs
        if (sizeof(float2) * std::max(agg_work(P, k, 1).total, dis_work(P, k, 1).total) > P.small_room) {
            P.small_classes.clear();
            return;
        }
        P.small_classes.push_back(k);
    }
    for (int c : kBlocks)
        with_cols(c, [&](auto n) {
            constexpr int COLS = decltype(n)::value;
            TFMM_CUDA_CHECK(cudaFuncSetAttribute(small_aggregate_kernel<COLS>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, opt_in));
            TFMM_CUDA_CHECK(cudaFuncSetAttribute(small_disaggregate_kernel<COLS>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, opt_in));
        });
    if (!P.small_order.p) TFMM_CUDA_CHECK(device_malloc(&P.small_order.p, sizeof(int) * P.G));
    TFMM_CUDA_CHECK(cudaMemcpyAsync(P.small_order.p, order.data(), sizeof(int) * P.G, cudaMemcpyHostToDevice, s));
    TFMM_CUDA_CHECK(cudaStreamSynchronize(s));
    P.small_ok = true;
    // One column: taken while the SMs hold all items in at most a round and a half, where one launch
    // with everything requested at once wins; with more, the persistent kernels keep DRAM busy through
    // each other's phases.  Measured (aggregation + disaggregation, persistent kernels / this, us): 56
    // groups of up to 90 KB 27 / 20, 271 of 120 KB 36 / 37, 631 of 60 KB 50 / 76, 1391 of 120 KB 105 / 193,
    // 7240 of 60 KB 440 / 448.
    P.small_one = 2 * P.G <= 3 * P.num_sms;
}

bool small_takes(const Plan& P, bool aggregation, int R) {
    if (R <= 1 || P.params.mrhs_precision == 1) return P.small_one;
    return P.small_ok && P.params.mrhs_precision == 0 &&
           (aggregation ? blocks_pay(P, R, agg_work) : blocks_pay(P, R, dis_work));
}

void launch_small_aggregate(const Plan& P, const float2* x, int R, int64_t ldx, float2* spec, cudaStream_t s) {
    for (const SmallClass& k : P.small_classes)
        with_cols(pick_pass(P, k, R, agg_work).cols, [&](auto n) {
            constexpr int COLS = decltype(n)::value;
            const SmallLayout l = agg_work(P, k, COLS);
            SmallArgs a = small_args(P, k, R, l);
            a.x = x;
            a.ld = ldx;
            a.spec = spec;
            small_aggregate_kernel<COLS><<<2 * k.groups, kThreads, sizeof(float2) * l.total, s>>>(a);
        });
    TFMM_CUDA_CHECK(cudaGetLastError());
}

void launch_small_disaggregate(const Plan& P, const float2* spec, int R, int weights, float2 beta, float2* y,
                               int64_t ldy, cudaStream_t s) {
    for (const SmallClass& k : P.small_classes)
        with_cols(pick_pass(P, k, R, dis_work).cols, [&](auto n) {
            constexpr int COLS = decltype(n)::value;
            const SmallLayout l = dis_work(P, k, COLS);
            SmallArgs a = small_args(P, k, R, l);
            a.spec_in = spec;
            a.w = weights ? P.d_weights : nullptr;
            a.y = y;
            a.ld = ldy;
            a.beta = beta;
            small_disaggregate_kernel<COLS><<<2 * k.groups, kThreads, sizeof(float2) * l.total, s>>>(a);
        });
    TFMM_CUDA_CHECK(cudaGetLastError());
}

}  // namespace tfmm
