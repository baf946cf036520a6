// Setup of the sliced rows (sliced.cuh) on the device.
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "sliced.cuh"

namespace pdhg {

namespace {

// The rows of one window (wst: first rows; at most W) by falling length (ties: the lower row first) and its slices,
// one block of W threads per window.  Count only (slice = nullptr): cnt[w] =
// (slices, steps, entries of the row list, 0).  Else the records and the row list go to
// their places off[w] = (first slice, first step, first entry of the row list, 0).
template <int W>
__global__ void __launch_bounds__(W)
k_slice_rows(const int32_t* wst, const int64_t* rp, int4* cnt, const int4* off, int4* slice, int32_t* list)
{
    __shared__ int len[W], srt[W], who[W];
    const int t = threadIdx.x;
    const int r0 = wst[blockIdx.x], n = wst[blockIdx.x + 1] - r0;
    const int64_t r = r0 + t;
    len[t] = t < n ? (int)(rp[r + 1] - rp[r]) : -1;
    __syncthreads();
    int k = 0;
    for (int j = 0; j < W; ++j) k += len[j] > len[t] || (len[j] == len[t] && j < t);
    srt[k] = len[t];
    who[k] = t;
    __syncthreads();
    if (t != 0) return;
    const int4 o = slice ? off[blockIdx.x] : make_int4(0, 0, 0, 0);
    int ns = 0, steps = 0, nl = 0;
    for (int i = 0; i < n;) {
        int lg = 0;
        while (lg < 5 && (srt[i] + (1 << lg) - 1) >> lg > kSliceRow) ++lg;
        const int st = (srt[i] + (1 << lg) - 1) >> lg, per = 32 >> lg;
        if (slice) {
            slice[o.x + ns] = make_int4(o.y + steps, st, lg, o.z + nl);
            for (int j = 0; j < per; ++j)
                list[o.z + nl + j] = i + j < n ? r0 + who[i + j] : -1;
        }
        ++ns;
        steps += st;
        nl += per;
        i += per;
    }
    if (!slice) cnt[blockIdx.x] = make_int4(ns, steps, nl, 0);
}

// Column indices of the slices (-1: padding) and the nonzero of each entry, a warp per slice.
__global__ void k_slice_fill(int nslice, const int4* slice, const int32_t* list, const int64_t* rp,
                             const int32_t* ci, int32_t* idx, int32_t* perm)
{
    const int lane = threadIdx.x & 31;
    for (int s = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); s < nslice;
         s += (int)((gridDim.x * blockDim.x) >> 5)) {
        const int4 d = slice[s];
        const int row = list[d.w + (lane >> d.z)];
        const int g = lane & ((1 << d.z) - 1);
        const int64_t p0 = row >= 0 ? rp[row] : 0, p1 = row >= 0 ? rp[row + 1] : 0;
        const size_t base = (size_t)d.x * 32 + lane;
        for (int k = 0; k < d.y; ++k) {
            const int64_t p = p0 + g + ((int64_t)k << d.z);
            idx[base + 32 * (size_t)k] = p < p1 ? ci[p] : -1;
            perm[base + 32 * (size_t)k] = p < p1 ? (int32_t)p : -1;
        }
    }
}

template <typename T>
__global__ void k_slice_values(int64_t entries, const int32_t* perm, const T* val, T* out)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < entries;
         i += (int64_t)gridDim.x * blockDim.x)
        out[i] = perm[i] >= 0 ? val[perm[i]] : T(0);
}

}  // namespace

// Whether a side's products are faster in slices than in the CSR ring (spmv.cuh), which
// cuts long rows across warps and deals out nonzeros evenly.  steps: nonzeros of a lane if
// all warps had the same.  A vector that L1 holds keeps the ring (its gathers hit there).
//
// The longest row: a slice takes it with 32 lanes, and the product waits for that warp.
// Iterations (K and K^T) with one row of 20 | 2,048 | 4,096 | 8,000 nonzeros among rows of 5
// to 20, us: FP64, 60,000 x 120,000 in slices 28 | 33 | 41 | 56, in the ring 41 for all;
// 250,000 x 500,000 63 | 68 | 79 | 99 against 103; FP32, 100,000 x 200,000 24 | 24 | 34 | 48
// against 24 | 24 | 29 | 30; 400,000 x 800,000 64 | 66 | 78 | 96 against 65 | 65 | 64 | 67.  The
// 1M x 2M LP (rows of up to 5,000, 20M nonzeros) hides it: FP64 K side 220 -> 142 us, FP32
// 116 -> 107.
//
// The average: FP64 slices were faster up to the 130 nonzeros a row that were tried (120,000
// rows, ring -> slices: 20 a row 71 -> 47 us, 48 140 -> 75, 64 196 -> 93, 130 316 -> 155); the
// line is at 48, above it nothing has moved.  FP32 gains little (1,000,000 rows of 12, K
// side: 66.4 -> 63.7 us; 200,000 rows of 5 to 20: 26.5 -> 24.1) and loses where rows are
// longer and warps few steps (100,000 rows of 22 to 66: 34.2 -> 36.5 us; the K^T side of
// 150,000 rows of 20: 22.6 -> 24.7; with 300,000 rows of 22 to 66 72.7 -> 71.3).
template <typename T>
bool slices_pay(int64_t rows, int64_t nnz, int64_t maxrow, int64_t x_len, double steps, bool batch)
{
    const double avg = (double)nnz / (double)rows;
    if (avg > 48.0 || maxrow > 8192 || x_len * (int64_t)sizeof(T) <= kL1GatherBytes) return false;
    if (batch) return true;   // its ring cuts no rows
    if (sizeof(T) == 4 && avg >= 16.0 && steps < 32.0) return false;
    const double longest = (double)maxrow / 32.0;
    return sizeof(T) == 4 ? longest <= std::max(64.0, 2.0 * steps) : longest <= std::max(128.0, 8.0 * steps);
}

template <typename T>
lp_status slice_side(Handle* h, const std::vector<int64_t>& hrp, const int64_t* rp, const int32_t* ci,
                     int64_t x_len, const std::vector<int64_t>* lp0, SlicedSide* out)
{
    constexpr int W = kSliceWin<T>;
    SlicedSide S;
    *out = S;
    const int64_t rows = (int64_t)hrp.size() - 1, nnz = h->nnz;
    if (nnz == 0 || rows >= ((int64_t)1 << 31)) return LP_OK;
    int64_t maxrow = 0;
    for (int64_t r = 0; r < rows; ++r) maxrow = std::max(maxrow, hrp[(size_t)r + 1] - hrp[(size_t)r]);
    cudaStream_t st = h->stream;
    int sms = 0;
    LP_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device));
    if (!slices_pay<T>(rows, nnz, maxrow, x_len,
                       (double)nnz / 32.0 / (double)(sms * kSliceBlocks<T> * (kSpmvNT / 32)), lp0 != nullptr))
        return LP_OK;
    // windows of W rows, none across two LPs
    const size_t B = lp0 ? lp0->size() - 1 : 1;
    std::vector<int32_t> wst, wfirst(B + 1);
    for (size_t k = 0; k < B; ++k) {
        wfirst[k] = (int32_t)wst.size();
        const int64_t e = lp0 ? (*lp0)[k + 1] : rows;
        for (int64_t r = lp0 ? (*lp0)[k] : 0; r < e; r += W) wst.push_back((int32_t)r);
    }
    const int nwin = wfirst[B] = (int32_t)wst.size();
    wst.push_back((int32_t)rows);
    std::vector<int4> w((size_t)nwin);
    // the windows' lists lie in the handle's scratch: 20 bytes for 128 rows and an LP, of
    // 16 for every row and column
    int4* dw = reinterpret_cast<int4*>(h->scratch);
    int32_t* dst = reinterpret_cast<int32_t*>(dw + nwin);
    LP_CUDA_TRY(cudaMemcpyAsync(dst, wst.data(), wst.size() * 4, cudaMemcpyHostToDevice, st));
    k_slice_rows<W><<<nwin, W, 0, st>>>(dst, rp, dw, nullptr, nullptr, nullptr);
    LP_CUDA_TRY(cudaGetLastError());
    LP_CUDA_TRY(cudaMemcpyAsync(w.data(), dw, (size_t)nwin * sizeof(int4), cudaMemcpyDeviceToHost, st));
    LP_CUDA_TRY(cudaStreamSynchronize(st));
    int64_t ns = 0, steps = 0, nl = 0;
    for (int4& q : w) {
        const int4 c = q;
        q = make_int4((int)ns, (int)steps, (int)nl, 0);
        ns += c.x;
        steps += c.y;
        nl += c.z;
    }
    // A second copy of the matrix: at most a sixteenth of the device's memory, so a quarter
    // for both sides in both precisions.  (By what is free, the same LP summed in another
    // order when something else held the card.)
    size_t avail = 0, total = 0;
    LP_CUDA_TRY(cudaMemGetInfo(&avail, &total));
    const size_t need = (size_t)ns * sizeof(int4) + (size_t)nl * 4 + (size_t)steps * 32 * (8 + sizeof(T));
    if (steps * 32 >= ((int64_t)1 << 31) || nl >= ((int64_t)1 << 31) || need > total / 16) return LP_OK;
    // one allocation: values, records, columns, nonzeros, rows; without room the ring stays
    T* val = nullptr;
    const lp_status as = dev_alloc(h, (void**)&val, need);
    if (as == LP_OUT_OF_MEMORY) return LP_OK;
    LP_TRY(as);
    int4* raw = reinterpret_cast<int4*>(val + steps * 32);
    int32_t* idx = reinterpret_cast<int32_t*>(raw + ns);
    int32_t* perm = idx + steps * 32;
    int32_t* list = perm + steps * 32;
    LP_CUDA_TRY(cudaMemcpyAsync(dw, w.data(), (size_t)nwin * sizeof(int4), cudaMemcpyHostToDevice, st));
    k_slice_rows<W><<<nwin, W, 0, st>>>(dst, rp, nullptr, dw, raw, list);
    k_slice_fill<<<4 * 1216, 256, 0, st>>>((int)ns, raw, list, rp, ci, idx, perm);
    LP_CUDA_TRY(cudaGetLastError());
    h->launches += 3;
    // the longest first (a counting sort: stable)
    std::vector<int4> rec((size_t)ns), ord((size_t)ns);
    LP_CUDA_TRY(cudaMemcpyAsync(rec.data(), raw, (size_t)ns * sizeof(int4), cudaMemcpyDeviceToHost, st));
    LP_CUDA_TRY(cudaStreamSynchronize(st));
    int mx = 0;
    for (const int4& q : rec) mx = std::max(mx, q.y);
    std::vector<int64_t> at((size_t)mx + 2, 0);
    for (const int4& q : rec) ++at[(size_t)(mx - q.y) + 1];
    for (int k = 0; k <= mx; ++k) at[(size_t)k + 1] += at[(size_t)k];
    std::vector<int32_t> tag((size_t)ns);
    for (int64_t i = 0; i < ns; ++i) {
        const int64_t p = at[(size_t)(mx - rec[(size_t)i].y)]++;
        ord[(size_t)p] = rec[(size_t)i];
        tag[(size_t)p] = (int32_t)i;
    }
    LP_CUDA_TRY(cudaMemcpyAsync(raw, ord.data(), (size_t)ns * sizeof(int4), cudaMemcpyHostToDevice, st));
    std::vector<int32_t> lp, lps(B + 1, (int32_t)ns);
    if (lp0) {
        lp.resize((size_t)ns);
        for (size_t k = 0; k < B; ++k)
            lps[k] = wfirst[k] < nwin ? w[(size_t)wfirst[k]].x : (int32_t)ns;
        for (size_t k = 0; k < B; ++k)
            std::fill(lp.begin() + lps[k], lp.begin() + lps[k + 1], (int32_t)k);
        int32_t *dtag = nullptr, *dlp = nullptr, *dlp0 = nullptr;
        LP_TRY(dev_alloc_n(h, &dtag, (size_t)ns));
        LP_TRY(dev_alloc_n(h, &dlp, (size_t)ns));
        LP_TRY(dev_alloc_n(h, &dlp0, B + 1));
        LP_TRY(dev_alloc_n(h, &S.part, 2 * (size_t)ns));
        LP_TRY(dev_alloc_n(h, &S.slice_live, (size_t)ns));
        LP_TRY(dev_alloc_n(h, &S.tag_live, (size_t)ns));
        LP_TRY(dev_alloc_n(h, &S.live, 2));
        LP_CUDA_TRY(cudaMemcpyAsync(dtag, tag.data(), (size_t)ns * 4, cudaMemcpyHostToDevice, st));
        LP_CUDA_TRY(cudaMemcpyAsync(dlp, lp.data(), (size_t)ns * 4, cudaMemcpyHostToDevice, st));
        LP_CUDA_TRY(cudaMemcpyAsync(dlp0, lps.data(), (B + 1) * 4, cudaMemcpyHostToDevice, st));
        S.tag = dtag;
        S.lp = dlp;
        S.lp0 = dlp0;
    }
    LP_CUDA_TRY(cudaStreamSynchronize(st));
    S.slice = raw;
    S.row = list;
    S.idx = idx;
    S.perm = perm;
    S.val = val;
    S.entries = steps * 32;
    S.nslice = (int)ns;
    S.grid = (int)std::min<int64_t>((int64_t)sms * kSliceBlocks<T>, (ns + 7) / 8);
    S.on = true;
    *out = S;
    return LP_OK;
}

template <typename T>
lp_status slice_plan(Handle* h)
{
    Engine<T>& E = engine_of<T>(h);
    LP_TRY(slice_side<T>(h, h->h_rp, h->rp, h->ci, h->n, nullptr, &E.slK));
    LP_TRY(slice_side<T>(h, h->h_trp, h->trp, h->tci, h->m, nullptr, &E.slT));
    return LP_OK;
}

template <typename T>
lp_status slice_refresh(Handle* h, const SlicedSide& S, const T* val)
{
    if (!S.on) return LP_OK;
    const int64_t g = std::min<int64_t>(4 * 1216, (S.entries + 255) / 256);
    k_slice_values<T><<<(int)g, 256, 0, h->stream>>>(S.entries, S.perm, val, static_cast<T*>(S.val));
    ++h->launches;
    LP_CUDA_TRY(cudaGetLastError());
    return LP_OK;
}

template <typename T>
lp_status slice_values(Handle* h)
{
    Engine<T>& E = engine_of<T>(h);
    LP_TRY(slice_refresh<T>(h, E.slK, E.val));
    return slice_refresh<T>(h, E.slT, E.tval);
}

template lp_status slice_plan<double>(Handle*);
template lp_status slice_plan<float>(Handle*);
template lp_status slice_values<double>(Handle*);
template lp_status slice_values<float>(Handle*);
template lp_status slice_side<double>(Handle*, const std::vector<int64_t>&, const int64_t*, const int32_t*,
                                      int64_t, const std::vector<int64_t>*, SlicedSide*);
template lp_status slice_side<float>(Handle*, const std::vector<int64_t>&, const int64_t*, const int32_t*,
                                     int64_t, const std::vector<int64_t>*, SlicedSide*);
template lp_status slice_refresh<double>(Handle*, const SlicedSide&, const double*);
template lp_status slice_refresh<float>(Handle*, const SlicedSide&, const float*);

}  // namespace pdhg
