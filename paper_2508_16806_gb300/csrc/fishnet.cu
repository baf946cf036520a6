// Algorithm 7 (fishnet casting, Section 2.5) on the GPU: P candidate points
// advanced together by fixed-step PDHG, so each product with K or K^T is a
// sparse-times-dense product over a row-major n x P (m x P) point block instead
// of P separate SpMVs; cull by duality gap and convex repopulation between
// rounds.  T = double keeps the point blocks and products in FP64 (the cull
// compares gaps, so its decisions are then taken as in the FP64 oracle);
// T = float keeps them in FP32 (GB300's FP64 pipe makes the FP64 block products
// arithmetic-bound: P fused multiply-adds per nonzero), with FP64 gap
// reductions.
//
// Readings shared with the oracle: points x~_p = (||K~||_2 / sqrt(n)) g_p on the
// scaled problem, Y^0 = K~ X^0, k fixed steps of Algorithm 1 per round with the
// solver's initial eta and omega, cull to the half with the smallest |gap|
// (stable by index, survivors in their old order), repopulation at odd rounds
// while more than two columns entered the round, with weights |z| / sum |z|.
#include <algorithm>
#include <cmath>
#include <numeric>
#include <vector>

#include "common.cuh"
#include "control.cuh"

namespace pdhg {
namespace {

constexpr int kFW = 8;             // warps per block of the block-SpMM kernels
constexpr int kFGrid = 152 * 16;   // grid cap of the block-SpMM kernels (persistent rows loop)

// A side of up to kWarpRows rows, or of more than kLaneAvg nonzeros a row on average, takes
// a warp per row (k_spmm_warp), any other lanes (k_spmm).  Products of all rounds of a step
// from 2 / from 64 points down, us, warp | lanes.  Few rows, 12.5 nonzeros a row of K and 6.25
// of K^T: FP64, 500 x 1,000 7.6 / 124 | 18.3 / 187, 2,000 x 4,000 13.2 / 164 | 21.6 / 206, the
// K side of 5,000 rows 18.6 / 250 | 22.1 / 260, of 8,000 rows 20.4 / 317 | 22.4 / 303; FP32,
// 500 rows 8.0 / 104 | 10.3 / 102, 2,000 10.1 / 114 | 11.5 / 116, the K side of 5,000
// 12.1 / 128 | 12.2 / 125.  Long rows: 4,000 x 8,000, 129 to 256 a row, FP32 19.9 / 391 |
// 34.7 / 508; 30,000 x 60,000, 80 a row, the K side 39.7 / 653 | 40.6 / 561, FP64 72 / 2,695 |
// 61 / 2,075; 50,000 x 100,000, 40 a row, FP32 48 / 791 | 38 / 478.
constexpr int64_t kLaneAvg = 48;
template <typename T> constexpr int64_t kWarpRows = sizeof(T) == 4 ? 4096 : 6144;

// Rows with more nonzeros than this go to k_spmm_long (a block per row), so that no lane
// (kLaneRow) and no warp (kWarpRow) walks a power-law row of thousands of nonzeros alone.
// kLaneRow at 64 | 128, the same figures, FP32: power-law rows of 4 to 2,000 35.0 / 678 |
// 35.2 / 676, 1 % of the rows with 80 to 100 23.8 / 369 | 23.1 / 351, all with 80
// 42.9 / 727 | 39.7 / 653; 2 % with 129 to 256 by lanes 34 / 505, by blocks 25 / 414.
constexpr int64_t kLaneRow = 128, kWarpRow = 256;

// V consecutive columns of a point block's row
template <typename T, int V>
struct alignas(sizeof(T) * V) Vec {
    T v[V];
};

// Accumulates the batches b0, b0 + stride, ... (32 nonzeros each) of row [s, e)
// into a0 (and a1 for P = 64); every lane of the warp calls it.
template <typename T>
__device__ __forceinline__ void spmm_row_part(const int32_t* __restrict__ ci,
                                              const T* __restrict__ val, int64_t b0, int64_t e,
                                              int64_t stride, int P, const T* __restrict__ X,
                                              int lane, int G, int g, int p, bool two, T& a0,
                                              T& a1)
{
    const unsigned full = 0xffffffffu;
    for (int64_t b = b0; b < e; b += stride) {
        const int64_t k = b + lane;
        const int c = k < e ? ci[k] : 0;
        const T v = k < e ? val[k] : T(0);
        const int cnt = e - b < 32 ? (int)(e - b) : 32;
#pragma unroll 8
        for (int t0 = 0; t0 < cnt; t0 += G) {
            const int t = t0 + g;   // <= 31; lanes past the row's end hold v = 0
            const int ct = __shfl_sync(full, c, t);
            const T vt = __shfl_sync(full, v, t);
            const T* xr = X + (int64_t)ct * P;
            a0 += vt * xr[p];
            if (two) a1 += vt * xr[p + 32];
        }
    }
}

// out[r, p] = sum_k val_k X[col_k, p] for the rows r of a CSR matrix; X is row major with
// P columns (a power of two, 1..64).  P / V lanes take a row, V columns (16 bytes where
// P allows) each, and walk its nonzeros in order, eight gathers in flight (past the end:
// the last entry again, times zero).  G sums per column, one for every G-th nonzero, added
// up in pairs: 32 / P of them below 32 points, the sums of k_spmm_warp to the bit (one sum
// for up to 128 nonzeros: up to 32 times as many roundings in a chain; FP64 steps, 50,000
// rows, 64 points and fewer: 1,037 us instead of 1,090, FP32 289 instead of 288).
// What bounds it is the chain start -> column -> gather -> epilogue and, for many columns,
// the L2 bytes of the gathers; so many rows at once and few instructions each.  50,000 x
// 100,000 LP, 625,000 nonzeros, P from 32 to 2, averages: a warp per row 34 us (K^T side)
// and 24 us (K side); so 12.6 us and 13.0 us, a call 11.4 -> 7.9 ms.
template <typename T, int V, int G, class Epi>
__global__ void __launch_bounds__(kFW * 32)
k_spmm(const int64_t* __restrict__ rp, const int32_t* __restrict__ ci,
       const T* __restrict__ val, int64_t rows, int P, const T* __restrict__ X, Epi epi)
{
    using W = Vec<T, V>;
    constexpr int S = G < 8 ? 8 : G;    // nonzeros of a round
    const int lr = P / V, per = kFW * 32 / lr;
    const int p = (int)(threadIdx.x & (lr - 1)) * V;
    for (int64_t r = (int64_t)blockIdx.x * per + threadIdx.x / lr; r < rows;
         r += (int64_t)gridDim.x * per) {
        const int64_t s = rp[r], e = rp[r + 1];
        if (e - s > kLaneRow) continue;
        const auto pre = epi.template load<V>(r, p);
        W a[G];
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int i = 0; i < V; ++i) a[g].v[i] = T(0);
        // FP32: the columns and values of the next eight are fetched while eight are gathered
        // (10,000 x 20,000, 64 points and fewer: 167 -> 135 us; FP64 is bound by its unit
        // instead, and slower so: 50,000 rows 1,090 -> 1,165 us)
        constexpr bool AHEAD = sizeof(T) == 4;
        int c[8];
        T v[8];
        const auto fetch = [&](int64_t k) {
#pragma unroll
            for (int u = 0; u < 8; ++u) c[u] = ci[k + u < e ? k + u : e - 1];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = k + u < e ? val[k + u] : T(0);
        };
        if (AHEAD && s < e) fetch(s);
        for (int64_t k0 = s; k0 < e; k0 += S) {
#pragma unroll
            for (int h = 0; h < S; h += 8) {
                const int64_t k = k0 + h;
                if (h > 0 && k >= e) break;
                W x[8];
                T w[8];
                if (!AHEAD) fetch(k);
#pragma unroll
                for (int u = 0; u < 8; ++u) x[u] = *reinterpret_cast<const W*>(X + (int64_t)c[u] * P + p);
#pragma unroll
                for (int u = 0; u < 8; ++u) w[u] = v[u];
                if (AHEAD && k + 8 < e) fetch(k + 8);
#pragma unroll
                for (int u = 0; u < 8; ++u)
#pragma unroll
                    for (int i = 0; i < V; ++i)
                        a[(h + u) % G].v[i] = fma(w[u], x[u].v[i], a[(h + u) % G].v[i]);
            }
        }
#pragma unroll
        for (int o = 1; o < G; o <<= 1)
#pragma unroll
            for (int g = 0; g < G; g += 2 * o)
#pragma unroll
                for (int i = 0; i < V; ++i) a[g].v[i] += a[g + o].v[i];
        epi.template row<V>(r, p, a[0], pre);
    }
}

// The same sums with a warp per row: lane l serves column l % P (and l + 32 when P = 64),
// the G = 32 / P lane groups take every G-th nonzero of each batch of 32.  A row's columns
// and values come in one load and its sums take few instructions of the FP64 unit: the
// better form while a wave of warps holds the rows, and for long ones.
template <typename T, class Epi>
__global__ void __launch_bounds__(kFW * 32)
k_spmm_warp(const int64_t* __restrict__ rp, const int32_t* __restrict__ ci,
            const T* __restrict__ val, int64_t rows, int P, const T* __restrict__ X, Epi epi)
{
    const int lane = threadIdx.x & 31;
    const int Pl = P < 32 ? P : 32;
    const int G = 32 / Pl;
    const int g = lane / Pl, p = lane % Pl;
    const bool two = P == 64;
    for (int64_t r = (int64_t)blockIdx.x * kFW + (threadIdx.x >> 5); r < rows;
         r += (int64_t)gridDim.x * kFW) {
        const int64_t s = rp[r], e = rp[r + 1];
        if (e - s > kWarpRow) continue;
        T a0 = 0, a1 = 0;
        spmm_row_part(ci, val, s, e, 32, P, X, lane, G, g, p, two, a0, a1);
        for (int o = Pl; o < 32; o <<= 1) a0 += __shfl_xor_sync(0xffffffffu, a0, o);
        if (g == 0) {
            epi.template row<1>(r, p, Vec<T, 1>{{a0}}, epi.template load<1>(r, p));
            if (two) epi.template row<1>(r, p + 32, Vec<T, 1>{{a1}}, epi.template load<1>(r, p + 32));
        }
    }
}

// The longest rows (listed in `rows`): one block per row, warp w
// takes the row's batches w, w + kFW, ...; the warps' sums are added in warp
// order (fixed) before the epilogue.
template <typename T, class Epi>
__global__ void __launch_bounds__(kFW * 32)
k_spmm_long(const int64_t* __restrict__ rp, const int32_t* __restrict__ ci,
            const T* __restrict__ val, const int32_t* __restrict__ rows, int count, int P,
            const T* __restrict__ X, Epi epi)
{
    __shared__ T sh[kFW][64];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int Pl = P < 32 ? P : 32;
    const int G = 32 / Pl;
    const int g = lane / Pl, p = lane % Pl;
    const bool two = P == 64;
    for (int i = blockIdx.x; i < count; i += gridDim.x) {
        const int64_t r = rows[i];
        const int64_t s = rp[r], e = rp[r + 1];
        T a0 = 0, a1 = 0;
        spmm_row_part(ci, val, s + 32 * (int64_t)warp, e, 32 * (int64_t)kFW, P, X, lane, G, g,
                      p, two, a0, a1);
        for (int o = Pl; o < 32; o <<= 1) a0 += __shfl_xor_sync(full, a0, o);
        if (g == 0) {
            sh[warp][p] = a0;
            if (two) sh[warp][p + 32] = a1;
        }
        __syncthreads();
        if (warp == 0 && g == 0) {
            T t0 = 0, t1 = 0;
            for (int w = 0; w < kFW; ++w) {
                t0 += sh[w][p];
                if (two) t1 += sh[w][p + 32];
            }
            epi.template row<1>(r, p, Vec<T, 1>{{t0}}, epi.template load<1>(r, p));
            if (two) epi.template row<1>(r, p + 32, Vec<T, 1>{{t1}}, epi.template load<1>(r, p + 32));
        }
        __syncthreads();
    }
}

// Epilogues: load<V> fetches the row's operands ahead of the sums, row<V> takes the sums
// of columns p .. p + V - 1.
template <typename T>
struct FStore {
    T* out;
    int P;
    template <int V> __device__ int load(int64_t, int) const { return 0; }
    template <int V> __device__ void row(int64_t r, int p, const Vec<T, V>& s, int) const
    {
        *reinterpret_cast<Vec<T, V>*>(out + r * P + p) = s;
    }
};

// x' = proj_X(x - tau (c - K^T y)) per column (Algorithm 1, theta = 1)
template <typename T>
struct FPrimal {
    const T* X;
    T* Xn;
    const T *c, *l, *u;
    T tau;
    int P;
    template <int V> struct Pre { Vec<T, V> x; T c, l, u; };
    template <int V> __device__ Pre<V> load(int64_t j, int p) const
    {
        return {*reinterpret_cast<const Vec<T, V>*>(X + j * P + p), c[j], l[j], u[j]};
    }
    template <int V> __device__ void row(int64_t j, int p, const Vec<T, V>& s, const Pre<V>& o) const
    {
        Vec<T, V> w;
#pragma unroll
        for (int i = 0; i < V; ++i) {
            T v = o.x.v[i] - tau * (o.c - s.v[i]);
            if (v < o.l) v = o.l;
            if (v > o.u) v = o.u;
            w.v[i] = v;
        }
        *reinterpret_cast<Vec<T, V>*>(Xn + j * P + p) = w;
    }
};

// y' = proj_Y(y + sigma (q - (2 K x' - K x))); K x' replaces K x
template <typename T>
struct FDual {
    const T* Y;
    T* Yn;
    T* KX;
    const T* q;
    const uint8_t* sense;
    T sigma;
    int P;
    template <int V> struct Pre { Vec<T, V> y, kx; T q; bool ge; };
    template <int V> __device__ Pre<V> load(int64_t i, int p) const
    {
        return {*reinterpret_cast<const Vec<T, V>*>(Y + i * P + p),
                *reinterpret_cast<const Vec<T, V>*>(KX + i * P + p), q[i], sense[i] != 0};
    }
    template <int V> __device__ void row(int64_t i, int p, const Vec<T, V>& s, const Pre<V>& o) const
    {
        Vec<T, V> w;
#pragma unroll
        for (int k = 0; k < V; ++k) {
            T v = o.y.v[k] + sigma * (o.q - (T(2) * s.v[k] - o.kx.v[k]));
            if (o.ge && v < T(0)) v = T(0);
            w.v[k] = v;
        }
        *reinterpret_cast<Vec<T, V>*>(Yn + i * P + p) = w;
        *reinterpret_cast<Vec<T, V>*>(KX + i * P + p) = s;
    }
};

template <typename T>
__global__ void k_cast(int64_t n, int P, double rad, const double* G, T* X)
{
    const int64_t total = n * P;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x)
        X[t] = (T)(rad * G[t]);
}

// Per-column sums over the rows of a point block, fixed order: thread t of a
// block serves column t % P and rows blockIdx.x * (256 / P) + t / P, ... .
// part[q * P * gridDim.x + p * gridDim.x + block] for the NQ sums.
constexpr int kGapNT = 256;

template <int NQ>
__device__ void column_partials(const double (&v)[NQ], int P, double* part)
{
    __shared__ double sh[NQ][kGapNT];
#pragma unroll
    for (int q = 0; q < NQ; ++q) sh[q][threadIdx.x] = v[q];
    __syncthreads();
    if ((int)threadIdx.x < P) {
        const int per = kGapNT / P;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            double s = 0.0;
            for (int k = 0; k < per; ++k) s += sh[q][k * P + threadIdx.x];
            part[((size_t)q * P + threadIdx.x) * gridDim.x + blockIdx.x] = s;
        }
    }
}

// c~^T x_p and l~^T lambda_p^+ + u~^T lambda_p^-, lambda_p = proj_Lambda(c~ - K~^T y_p)
template <typename T>
__global__ void __launch_bounds__(kGapNT)
k_gap_cols(int64_t n, int P, const T* X, const T* KTY, const T* c, const T* l, const T* u,
           double* part)
{
    const int p = threadIdx.x % P, per = kGapNT / P;
    T a[2] = {T(0), T(0)};
    for (int64_t j = (int64_t)blockIdx.x * per + threadIdx.x / P; j < n;
         j += (int64_t)gridDim.x * per) {
        const int64_t t = j * P + p;
        const T cj = c[j], lj = l[j], uj = u[j];
        a[0] += cj * X[t];
        const T lam = proj_lambda(cj - KTY[t], isfinite(lj), isfinite(uj));
        if (lam > T(0)) a[1] += lj * lam;
        if (lam < T(0)) a[1] += uj * lam;
    }
    const double v[2] = {(double)a[0], (double)a[1]};
    column_partials<2>(v, P, part);
}

// q~^T y_p
template <typename T>
__global__ void __launch_bounds__(kGapNT)
k_gap_rows(int64_t m, int P, const T* Y, const T* q, double* part)
{
    const int p = threadIdx.x % P, per = kGapNT / P;
    T a = T(0);
    for (int64_t i = (int64_t)blockIdx.x * per + threadIdx.x / P; i < m;
         i += (int64_t)gridDim.x * per)
        a += q[i] * Y[i * P + p];
    const double v[1] = {(double)a};
    column_partials<1>(v, P, part);
}

// |pobj_p - dobj_p|, a block per column (one block over all 64 columns: 109 us for
// 391 + 196 partials a column, serial sums; now 5 us)
__global__ void __launch_bounds__(kGapNT)
k_gap_final(int P, const double* partC, int nbC, const double* partR, int nbR, double* gap)
{
    const int p = blockIdx.x;
    const double pobj = block_sum_array<kGapNT>(partC + (size_t)p * nbC, nbC);
    const double lt = block_sum_array<kGapNT>(partC + ((size_t)P + p) * nbC, nbC);
    const double qy = block_sum_array<kGapNT>(partR + (size_t)p * nbR, nbR);
    if (threadIdx.x == 0) gap[p] = fabs(pobj - (qy + lt));
}

// dst (rows x Pn) from src (rows x Po): columns t < keep copy src column
// kept[t]; column t >= keep is sum_a W[(t - keep) * keep + a] * src column kept[a].
template <typename T>
__global__ void k_combine(int64_t rows, int Po, int Pn, int keep, const int* kept,
                          const double* W, const T* src, T* dst)
{
    const int64_t total = rows * Pn;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = e / Pn;
        const int t = (int)(e - r * Pn);
        const T* s = src + r * Po;
        if (t < keep) {
            dst[e] = s[kept[t]];
        } else {
            const double* w = W + (size_t)(t - keep) * keep;
            T v = T(0);
            for (int a = 0; a < keep; ++a) v += (T)w[a] * s[kept[a]];
            dst[e] = v;
        }
    }
}

template <typename T>
__global__ void k_unscale(int64_t count, const T* v, const double* f, double* out)
{
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < count;
         t += (int64_t)gridDim.x * blockDim.x)
        out[t] = f[t] * (double)v[t];
}

int ew_blocks(int64_t count)
{
    int64_t g = (count + 255) / 256;
    if (g < 1) g = 1;
    if (g > kEWGrid * 4) g = kEWGrid * 4;
    return (int)g;
}

// The form of one side's products, and its rows that take a block each.
template <typename T>
struct Side {
    bool warp;
    std::vector<int32_t> rows;
    int32_t* dev = nullptr;
    explicit Side(const std::vector<int64_t>& rp)
    {
        const int64_t count = (int64_t)rp.size() - 1;
        warp = count <= kWarpRows<T> || rp.back() > kLaneAvg * count;
        for (int64_t r = 0; r < count; ++r)
            if (rp[(size_t)r + 1] - rp[(size_t)r] > (warp ? kWarpRow : kLaneRow)) rows.push_back((int32_t)r);
    }
};

// One block product: the short rows, then the long ones (a block each).
template <typename T, class Epi>
void spmm(Handle* h, const int64_t* rp, const int32_t* ci, const T* val, int64_t rows, int P,
          const T* X, const Side<T>& L, const Epi& epi)
{
    constexpr int W = 16 / sizeof(T);   // columns of a 16-byte load
    const int64_t per = L.warp ? kFW : kFW * 32 / (P / (P < W ? P : W));   // rows of a block
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((rows + per - 1) / per, kFGrid));
    const auto go = [&](auto kernel) {
        kernel<<<grid, kFW * 32, 0, h->stream>>>(rp, ci, val, rows, P, X, epi);
    };
    if (L.warp) go(k_spmm_warp<T, Epi>);
    else if (P >= 32) go(k_spmm<T, W, 1, Epi>);
    else if (P == 16) go(k_spmm<T, W, 2, Epi>);
    else if (P == 8) go(k_spmm<T, W, 4, Epi>);
    else if (P == 4) go(k_spmm<T, W, 8, Epi>);
    else if (P == 2) go(k_spmm<T, 2, 16, Epi>);
    else go(k_spmm<T, 1, 32, Epi>);
    ++h->launches;
    if (!L.rows.empty()) {
        k_spmm_long<T, Epi><<<(int)std::min<size_t>(L.rows.size(), kFGrid), kFW * 32, 0, h->stream>>>(
            rp, ci, val, L.dev, (int)L.rows.size(), P, X, epi);
        ++h->launches;
    }
}

// device buffers owned by one fishnet call
struct Scratch {
    std::vector<void*> ptrs;
    ~Scratch()
    {
        for (void* p : ptrs) cudaFree(p);
    }
    template <typename T>
    lp_status get(T** p, size_t count)
    {
        *p = nullptr;
        cudaError_t e = cudaMalloc((void**)p, std::max<size_t>(count, 1) * sizeof(T));
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            *p = nullptr;
            return e == cudaErrorMemoryAllocation ? LP_OUT_OF_MEMORY : LP_CUDA_ERROR;
        }
        ptrs.push_back(*p);
        return LP_OK;
    }
};

}  // namespace

int64_t fishnet_draws(int P)
{
    int64_t total = 0;
    int cols = P, i = 0;
    while (cols > 1) {
        const int keep = cols / 2;
        if ((i & 1) == 1 && cols > 2) {
            total += (int64_t)keep * keep;
            cols = 2 * keep;
        } else {
            cols = keep;
        }
        ++i;
    }
    return total;
}

namespace {

template <typename T>
lp_status fishnet_t(Handle* h, double eta, double omega, double normK, int P, int k_steps,
                    const double* G, const double* Z_host, int64_t nZ, double* x0, double* y0,
                    double* gaps_host, int32_t* rounds_out, int space)
{
    const int64_t m = h->m, n = h->n;
    const Engine<T>& E = engine_of<T>(h);
    cudaStream_t st = h->stream;
    if (fishnet_draws(P) > nZ) return LP_INVALID_ARGUMENT;
    Scratch S;
    T *X, *Xn, *KTY, *Y, *Yn, *KX, *KX2;
    double *Gd = nullptr, *gap, *W, *partC, *partR;
    int* kept_d;
    LP_TRY(S.get(&X, (size_t)n * P));
    LP_TRY(S.get(&Xn, (size_t)n * P));
    LP_TRY(S.get(&KTY, (size_t)n * P));
    LP_TRY(S.get(&Y, (size_t)m * P));
    LP_TRY(S.get(&Yn, (size_t)m * P));
    LP_TRY(S.get(&KX, (size_t)m * P));
    LP_TRY(S.get(&KX2, (size_t)m * P));
    LP_TRY(S.get(&gap, (size_t)P));
    LP_TRY(S.get(&W, (size_t)P * P));
    LP_TRY(S.get(&kept_d, (size_t)P));
    const int nbC = ew_blocks(n), nbR = ew_blocks(m);
    LP_TRY(S.get(&partC, (size_t)2 * P * nbC));
    LP_TRY(S.get(&partR, (size_t)P * nbR));
    if (space == LP_MEM_HOST) {
        LP_TRY(S.get(&Gd, (size_t)n * P));
        LP_CUDA_TRY(cudaMemcpyAsync(Gd, G, sizeof(double) * (size_t)n * P,
                                    cudaMemcpyHostToDevice, st));
        G = Gd;
    }
    Side<T> lk(h->h_rp), lt(h->h_trp);
    for (Side<T>* q : {&lk, &lt}) {
        LP_TRY(S.get(&q->dev, q->rows.size()));
        if (!q->rows.empty())
            LP_CUDA_TRY(cudaMemcpyAsync(q->dev, q->rows.data(), q->rows.size() * sizeof(int32_t),
                                        cudaMemcpyHostToDevice, st));
    }
    const T tau = (T)(eta / omega), sigma = (T)(eta * omega);
    // spectral casting, Y^0 = K~ X^0 (also the first K x)
    k_cast<T><<<ew_blocks(n * P), 256, 0, st>>>(n, P, normK / std::sqrt((double)n), G, X);
    ++h->launches;
    spmm<T>(h, h->rp, h->ci, E.val, m, P, X, lk, FStore<T>{Y, P});
    LP_CUDA_TRY(cudaMemcpyAsync(KX, Y, sizeof(T) * (size_t)m * P, cudaMemcpyDeviceToDevice, st));
    LP_CUDA_TRY(cudaGetLastError());

    std::vector<double> gh(P), wh((size_t)P * P);
    std::vector<int> order(P), kept(P);
    int cols = P, round = 0;
    int64_t zpos = 0;
    while (cols > 1) {
        const int j_top = cols;
        for (int t = 0; t < k_steps; ++t) {
            spmm<T>(h, h->trp, h->tci, E.tval, n, cols, Y, lt,
                    FPrimal<T>{X, Xn, E.c, E.l, E.u, tau, cols});
            spmm<T>(h, h->rp, h->ci, E.val, m, cols, Xn, lk,
                    FDual<T>{Y, Yn, KX, E.q, h->sense, sigma, cols});
            std::swap(X, Xn);
            std::swap(Y, Yn);
        }
        // |duality gap| of every column
        spmm<T>(h, h->trp, h->tci, E.tval, n, cols, Y, lt, FStore<T>{KTY, cols});
        k_gap_cols<T><<<nbC, kGapNT, 0, st>>>(n, cols, X, KTY, E.c, E.l, E.u, partC);
        k_gap_rows<T><<<nbR, kGapNT, 0, st>>>(m, cols, Y, E.q, partR);
        k_gap_final<<<cols, kGapNT, 0, st>>>(cols, partC, nbC, partR, nbR, gap);
        h->launches += 3;
        LP_CUDA_TRY(cudaGetLastError());
        LP_CUDA_TRY(cudaMemcpyAsync(gh.data(), gap, sizeof(double) * cols,
                                    cudaMemcpyDeviceToHost, st));
        LP_CUDA_TRY(cudaStreamSynchronize(st));
        if (gaps_host)
            for (int p = 0; p < cols; ++p) gaps_host[(int64_t)round * P + p] = gh[p];
        // cull_points: the half with the smallest gaps, in their old order
        std::iota(order.begin(), order.begin() + cols, 0);
        std::stable_sort(order.begin(), order.begin() + cols,
                         [&](int a, int b) { return gh[a] < gh[b]; });
        const int keep = cols / 2;
        std::copy(order.begin(), order.begin() + keep, kept.begin());
        std::sort(kept.begin(), kept.begin() + keep);
        int ncols = keep;
        // repopulate: one convex combination of the survivors per survivor
        if ((round & 1) == 1 && j_top > 2) {
            for (int t = 0; t < keep; ++t) {
                double sw = 0.0;
                for (int a = 0; a < keep; ++a) {
                    wh[(size_t)t * keep + a] = std::fabs(Z_host[zpos + (int64_t)t * keep + a]);
                    sw += wh[(size_t)t * keep + a];
                }
                for (int a = 0; a < keep; ++a)
                    wh[(size_t)t * keep + a] =
                        sw > 0.0 ? wh[(size_t)t * keep + a] / sw : 1.0 / keep;
            }
            zpos += (int64_t)keep * keep;
            ncols = 2 * keep;
            LP_CUDA_TRY(cudaMemcpyAsync(W, wh.data(), sizeof(double) * (size_t)keep * keep,
                                        cudaMemcpyHostToDevice, st));
        }
        LP_CUDA_TRY(cudaMemcpyAsync(kept_d, kept.data(), sizeof(int) * keep,
                                    cudaMemcpyHostToDevice, st));
        k_combine<T><<<ew_blocks(n * ncols), 256, 0, st>>>(n, cols, ncols, keep, kept_d, W, X, Xn);
        k_combine<T><<<ew_blocks(m * ncols), 256, 0, st>>>(m, cols, ncols, keep, kept_d, W, Y, Yn);
        k_combine<T><<<ew_blocks(m * ncols), 256, 0, st>>>(m, cols, ncols, keep, kept_d, W, KX,
                                                           KX2);
        h->launches += 3;
        LP_CUDA_TRY(cudaGetLastError());
        std::swap(X, Xn);
        std::swap(Y, Yn);
        std::swap(KX, KX2);
        // the host vectors above are reused next round: wait for the copies
        LP_CUDA_TRY(cudaStreamSynchronize(st));
        cols = ncols;
        ++round;
    }
    // the survivor, unscaled (x = C x~, y = R y~)
    double *xo = x0, *yo = y0, *xd = nullptr, *yd = nullptr;
    if (space == LP_MEM_HOST) {
        LP_TRY(S.get(&xd, (size_t)n));
        LP_TRY(S.get(&yd, (size_t)m));
        xo = xd;
        yo = yd;
    }
    k_unscale<T><<<ew_blocks(n), 256, 0, st>>>(n, X, h->C, xo);
    k_unscale<T><<<ew_blocks(m), 256, 0, st>>>(m, Y, h->R, yo);
    h->launches += 2;
    LP_CUDA_TRY(cudaGetLastError());
    if (space == LP_MEM_HOST) {
        LP_CUDA_TRY(cudaMemcpyAsync(x0, xd, sizeof(double) * n, cudaMemcpyDeviceToHost, st));
        LP_CUDA_TRY(cudaMemcpyAsync(y0, yd, sizeof(double) * m, cudaMemcpyDeviceToHost, st));
    }
    LP_CUDA_TRY(cudaStreamSynchronize(st));
    if (rounds_out) *rounds_out = round;
    return LP_OK;
}

}  // namespace

lp_status run_fishnet(Handle* h, int precision, double eta, double omega, double normK, int P,
                      int k_steps, const double* G, const double* Z_host, int64_t nZ, double* x0,
                      double* y0, double* gaps_host, int32_t* rounds_out, int space)
{
    if (precision == LP_PREC_MIXED)
        return fishnet_t<float>(h, eta, omega, normK, P, k_steps, G, Z_host, nZ, x0, y0,
                                gaps_host, rounds_out, space);
    return fishnet_t<double>(h, eta, omega, normK, P, k_steps, G, Z_host, nZ, x0, y0, gaps_host,
                             rounds_out, space);
}

}  // namespace pdhg
