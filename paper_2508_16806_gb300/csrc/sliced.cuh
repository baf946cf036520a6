// Products with K and K^T in sliced rows (SELL-C-sigma: Kreutzer et al., 2014): the form for
// short rows.
//
// Rows are taken kSliceWin at a time, sorted by length, and cut into slices: 32
// lanes that serve 32 / G rows with G lanes each (G = 1 up to kSliceRow nonzeros),
// the nonzeros stored transposed (step k of the 32 lanes side by side, padded to the
// slice's longest row with column -1).  A warp takes a slice: values and columns
// come coalesced and without conditions, eight steps in flight, each lane gathers
// its own row's entries (none for padding) and sums them by fused multiply-adds in a
// fixed order, and the epilogue runs on the row's owner lane.  No shared memory, no row
// starts, no hand-over between warps: what is left of the time is the gathers (an SM
// issues about one 32-byte sector request a cycle) and in FP64 the multiply-adds (16
// cycles of an SM for a warp's 32 lanes, however few are active: the sorted slices
// keep them busy).  Slices go to the warps longest first, round robin: a fixed
// order, so results are bitwise reproducible.
//
// 1M x 2M power-law LP (20M nonzeros), CSR ring (spmv.cuh) -> sliced: FP64 K side
// 226 -> 147 us, K^T side 173 -> 113 us; FP32 118 -> 106 us, 103 -> 101 us.  Windows: wide
// ones pad less (entries per nonzero of the K side: 64 rows 1.69, 128 1.40, 256 1.23, 512
// 1.13), narrow ones keep a slice's rows in fewer sectors; FP64 K + K^T 280 / 265 / 260 /
// 261 us, FP32 207 / 207 / 219 / 225 us.  Windows dealt to blocks whole, so that the rows
// of a window meet in one L1, were slower (FP32 K side 126 us, FP64 163 us: uneven warps).
#pragma once

#include "spmv.cuh"

namespace pdhg {

constexpr int kSliceRow = 32;      // steps of a slice, where a row's lanes allow it
// rows sorted together, resident blocks per SM
template <typename T> constexpr int kSliceWin = sizeof(T) == 4 ? 128 : 256;
template <typename T> constexpr int kSliceBlocks = sizeof(T) == 4 ? 5 : 3;

// the vector's entry c (none for padding: c < 0), as a load that is skipped, not
// branched around
__device__ __forceinline__ float gather_if(const float* x, int c)
{
    float v = 0.0f;
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ge.s32 p, %2, 0;\n\t"
        "@p ld.global.nc.L1::no_allocate.f32 %0, [%1];\n\t}"
        : "+f"(v)
        : "l"(x + c), "r"(c));
    return v;
}
__device__ __forceinline__ double gather_if(const double* x, int c)
{
    double v = 0.0;
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ge.s32 p, %2, 0;\n\t"
        "@p ld.global.nc.L1::no_allocate.f64 %0, [%1];\n\t}"
        : "+d"(v)
        : "l"(x + c), "r"(c));
    return v;
}

template <int U, int M, int C, typename T>
__device__ __forceinline__ void slice_steps(const int32_t* __restrict__ si, const T* __restrict__ sv,
                                            const T* x, T (&a)[C])
{
    int c[U];
    T v[U], xv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) c[u] = __ldcs(si + 32 * u);
#pragma unroll
    for (int u = 0; u < U; ++u) v[u] = __ldcs(sv + 32 * u);
#pragma unroll
    for (int u = 0; u < U; ++u) xv[u] = gather_if(x, c[u]);
#pragma unroll
    for (int u = 0; u < U; ++u) a[u % M] = fma(v[u], xv[u], a[u % M]);
}

// A lane's n steps in C sums, one for every C-th step of the groups of eight (what is left
// in two of them), which then meet in pairs: chains as short as those of the ring's lane
// groups.  Rounding error of an FP64 row sum (root mean square, in 2^-52 of the terms'
// magnitudes), one chain | four sums, eight from 16 steps | the ring: 6 nonzeros 0.20 | 0.19 |
// 0.20, 12 0.20 | 0.17 | 0.17, 24 0.20 | 0.13 | 0.13, 32 0.20 | 0.12 | 0.12; FP32 with four: 12
// 0.17 | 0.19 (ring), 24 0.14 | 0.15, 32 0.13 | 0.13.  The 1M x 2M LP, K and K^T side, one chain ->
// so: FP64 146 + 110 -> 154 + 112 us, FP32 111 + 99 -> 113 + 98 (116 with sums for two, four and
// eight chosen by a branch).
template <int C, typename T>
__device__ __forceinline__ T slice_sum(const int32_t* __restrict__ si, const T* __restrict__ sv, int n,
                                       const T* x)
{
    T a[C];
#pragma unroll
    for (int k = 0; k < C; ++k) a[k] = T(0);
    for (; n >= 8; n -= 8, si += 256, sv += 256) slice_steps<8, C, C, T>(si, sv, x, a);
    if (n >= 4) {
        slice_steps<4, 2, C, T>(si, sv, x, a);
        n -= 4, si += 128, sv += 128;
    }
    if (n >= 2) {
        slice_steps<2, 2, C, T>(si, sv, x, a);
        n -= 2, si += 64, sv += 64;
    }
    if (n >= 1) slice_steps<1, 2, C, T>(si, sv, x, a);
#pragma unroll
    for (int o = 1; o < C; o <<= 1)
#pragma unroll
        for (int k = 0; k < C; k += 2 * o) a[k] += a[k + o];
    return a[0];
}

// One slice: the rows' sums and, on each row's owner lane, their epilogue.
template <typename T, class Epi>
__device__ __forceinline__ void slice_run(const SlicedSide& S, const T* __restrict__ val, const int4 d,
                                          const T* __restrict__ x, Epi& epi, typename Epi::Acc& acc)
{
    const int lane = threadIdx.x & 31;
    const int row = __ldg(S.row + d.w + (lane >> d.z));
    const bool own = row >= 0 && (lane & ((1 << d.z) - 1)) == 0;
    const int32_t* __restrict__ si = S.idx + (size_t)d.x * 32 + lane;
    const T* __restrict__ sv = val + (size_t)d.x * 32 + lane;
    typename Epi::Pre pre;
    if (own) pre = epi.load(row);
    T a;
    if (sizeof(T) == 8 && d.y >= 16) a = slice_sum<8, T>(si, sv, d.y, x);
    else a = slice_sum<4, T>(si, sv, d.y, x);
    for (int o = (1 << d.z) >> 1; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (own) epi.row(row, a, pre, acc);
}

template <typename T, class Epi>
__global__ void __launch_bounds__(kSpmvNT, kSliceBlocks<T>)
k_sliced(const SlicedSide S, const T* __restrict__ val, Epi epi)
{
    if (!epi.begin()) return;
    const T* __restrict__ x = epi.xin();
    typename Epi::Acc acc;
    const int nw = gridDim.x * (kSpmvNT / 32), s1 = S.nslice;
    int s = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    // first entry / 32, steps, log2 of the lanes per row, first row of the list
    int4 d = make_int4(0, 0, 0, 0);
    if (s < s1) d = __ldg(S.slice + s);
    while (s < s1) {
        s += nw;
        int4 dn = d;
        if (s < s1) dn = __ldg(S.slice + s);
        slice_run<T, Epi>(S, val, d, x, epi, acc);
        d = dn;
    }
    epi.finish(acc);
}

// The same for a batch: a slice lies within one LP, whose state the epilogue takes
// (and whose finish skips it); its partials go to the slice's place in row order, so
// they are the same bits from whichever list the slice comes.  live: the list of the
// unfinished LPs instead of the whole one.
template <typename T, class Epi>
__global__ void __launch_bounds__(kSpmvNT, kSliceBlocks<T>)
k_sliced_lp(const SlicedSide S, const T* __restrict__ val, Epi epi, bool live)
{
    typename Epi::Acc acc;
    const int4* __restrict__ rec = live ? S.slice_live : S.slice;
    const int32_t* __restrict__ tag = live ? S.tag_live : S.tag;
    const int nw = gridDim.x * (kSpmvNT / 32), s1 = live ? __ldg(S.live) : S.nslice;
    int s = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    int4 d = make_int4(0, 0, 0, 0);
    int t = 0;
    if (s < s1) {
        d = __ldg(rec + s);
        t = __ldg(tag + s);
    }
    while (s < s1) {
        s += nw;
        int4 dn = d;
        int tn = t;
        if (s < s1) {
            dn = __ldg(rec + s);
            tn = __ldg(tag + s);
        }
        if (epi.live(t)) {
            epi.task_start(t);
            slice_run<T, Epi>(S, val, d, epi.xin(), epi, acc);
            epi.task_done(t, acc);
        }
        d = dn;
        t = tn;
    }
}

// K x (side_t = false) or K^T y with an epilogue: sliced rows where the engine has
// them for that side, else the CSR form.
template <typename T, class Epi>
inline void launch_product(Handle* h, Engine<T>& E, bool side_t, cudaStream_t st, const Epi& epi,
                           bool pdl = false)
{
    const SlicedSide& S = side_t ? E.slT : E.slK;
    if (S.on) {
        k_sliced<T, Epi><<<S.grid, kSpmvNT, 0, st>>>(S, static_cast<const T*>(S.val), epi);
        return;
    }
    if (side_t)
        launch_spmv<T>(E.gT, st, E.bcol, E.bnzT, E.ntblk, E.wbegT, E.permT, h->trp, h->tci, E.tval,
                       h->dev_err, h->m, epi, pdl, E.splitT);
    else
        launch_spmv<T>(E.gK, st, E.brow, E.bnzK, E.nblk, E.wbegK, E.permK, h->rp, h->ci, E.val,
                       h->dev_err, h->n, epi, pdl, E.splitK);
}

}  // namespace pdhg
