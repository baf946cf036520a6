// Setup of the sliced rows (sliced.cuh) on the device.
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "sliced.cuh"

namespace pdhg {

namespace {

// The rows of one window by falling length (ties: the lower row first) and its slices,
// one block of W threads per window.  Count only (slice = nullptr): cnt[w] =
// (slices, steps, entries of the row list, 0).  Else the records and the row list go to
// their places off[w] = (first slice, first step, first entry of the row list, 0).
template <int W>
__global__ void __launch_bounds__(W)
k_slice_rows(int64_t rows, const int64_t* rp, int4* cnt, const int4* off, int4* slice, int32_t* list)
{
    __shared__ int len[W], srt[W], who[W];
    const int t = threadIdx.x;
    const int64_t r = (int64_t)blockIdx.x * W + t;
    const int n = (int)(rows - (int64_t)blockIdx.x * W < W
                            ? rows - (int64_t)blockIdx.x * W
                            : W);
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
                list[o.z + nl + j] =
                    i + j < n ? (int32_t)((int64_t)blockIdx.x * W + who[i + j]) : -1;
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

template <typename T>
lp_status slice_side(Handle* h, const std::vector<int64_t>& hrp, const int64_t* rp, const int32_t* ci,
                     int64_t x_len, int sms, SlicedSide* out)
{
    constexpr int W = kSliceWin<T>;
    SlicedSide S;
    *out = S;
    const int64_t rows = (int64_t)hrp.size() - 1, nnz = h->nnz;
    // Long rows keep the CSR form, which cuts them across warps where its lists would be
    // unbalanced; so does a vector that L1 holds (its gathers hit there)
    if (nnz == 0 || (double)nnz > 48.0 * (double)rows) return LP_OK;
    int64_t maxrow = 0;
    for (int64_t r = 0; r < rows; ++r) maxrow = std::max(maxrow, hrp[(size_t)r + 1] - hrp[(size_t)r]);
    if (maxrow > 8192 || x_len * (int64_t)sizeof(T) <= kL1GatherBytes) return LP_OK;
    cudaStream_t st = h->stream;
    const int nwin = (int)((rows + W - 1) / W);
    std::vector<int4> w((size_t)nwin);
    int4 *dw = nullptr, *raw = nullptr;
    LP_TRY(dev_alloc_n(h, &dw, (size_t)nwin));
    k_slice_rows<W><<<nwin, W, 0, st>>>(rows, rp, dw, nullptr, nullptr, nullptr);
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
    // a second copy of the matrix: only where memory is plentiful
    size_t avail = 0, total = 0;
    LP_CUDA_TRY(cudaMemGetInfo(&avail, &total));
    const size_t need = (size_t)ns * sizeof(int4) + (size_t)nl * 4 + (size_t)steps * 32 * (8 + sizeof(T));
    if (steps * 32 >= ((int64_t)1 << 31) || nl >= ((int64_t)1 << 31) || need > avail / 4) {
        dev_free(h, dw);
        return LP_OK;
    }
    int32_t *list = nullptr, *idx = nullptr, *perm = nullptr;
    T* val = nullptr;
    LP_TRY(dev_alloc_n(h, &raw, (size_t)ns));
    LP_TRY(dev_alloc_n(h, &list, (size_t)nl));
    LP_TRY(dev_alloc_n(h, &idx, (size_t)steps * 32));
    LP_TRY(dev_alloc_n(h, &perm, (size_t)steps * 32));
    LP_TRY(dev_alloc_n(h, &val, (size_t)steps * 32));
    LP_CUDA_TRY(cudaMemcpyAsync(dw, w.data(), (size_t)nwin * sizeof(int4), cudaMemcpyHostToDevice, st));
    k_slice_rows<W><<<nwin, W, 0, st>>>(rows, rp, nullptr, dw, raw, list);
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
    for (const int4& q : rec) ord[(size_t)at[(size_t)(mx - q.y)]++] = q;
    LP_CUDA_TRY(cudaMemcpyAsync(raw, ord.data(), (size_t)ns * sizeof(int4), cudaMemcpyHostToDevice, st));
    LP_CUDA_TRY(cudaStreamSynchronize(st));
    dev_free(h, dw);
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

}  // namespace

template <typename T>
lp_status slice_plan(Handle* h)
{
    Engine<T>& E = engine_of<T>(h);
    int sms = 0;
    LP_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device));
    LP_TRY(slice_side<T>(h, h->h_rp, h->rp, h->ci, h->n, sms, &E.slK));
    LP_TRY(slice_side<T>(h, h->h_trp, h->trp, h->tci, h->m, sms, &E.slT));
    return LP_OK;
}

template <typename T>
lp_status slice_values(Handle* h)
{
    Engine<T>& E = engine_of<T>(h);
    for (int side = 0; side < 2; ++side) {
        const SlicedSide& S = side ? E.slT : E.slK;
        if (!S.on) continue;
        const int64_t g = std::min<int64_t>(4 * 1216, (S.entries + 255) / 256);
        k_slice_values<T><<<(int)g, 256, 0, h->stream>>>(S.entries, S.perm, side ? E.tval : E.val,
                                                         static_cast<T*>(S.val));
        ++h->launches;
    }
    LP_CUDA_TRY(cudaGetLastError());
    return LP_OK;
}

template lp_status slice_plan<double>(Handle*);
template lp_status slice_plan<float>(Handle*);
template lp_status slice_values<double>(Handle*);
template lp_status slice_values<float>(Handle*);

}  // namespace pdhg
