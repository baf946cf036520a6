// Resident iterations for LPs that fit the chip's shared memory: one launch runs
// every step attempt of a check period, instead of two or three launches per
// attempt.
//
// What bounds a small LP is not bytes but the chain of dependent steps: with one
// launch per product an attempt of a 5,000 x 10,000 LP (62,000 nonzeros) took
// 17.5 us, of which the data movement is less than one.  Here every row (of K and
// of K^T) has one owner for the whole launch; a block keeps its rows' nonzeros
// and their state in shared memory, and the two products of an attempt are
// separated by a barrier that also carries the reductions of Algorithm 5: every
// block adds the blocks' partial sums in the same order and takes the same
// decision, so no block waits for a deciding one.  (Left in global memory, the
// nonzeros came from L2 in every product, since the barrier's fence empties L1:
// 300 cycles and more for each dependent load.)
//
// Two forms (ResPlan::cluster): where x and y fit beside that in every block's
// shared memory, the blocks of one cluster (1 to 16) each keep a whole copy of
// the gathered vectors; a block sends its new entries to the others by bulk
// copies that complete on the receivers' mbarriers, which is the barrier.
// Otherwise a cooperative grid gathers through L2 and meets at a barrier in
// global memory.  An attempt takes (launches per product -> resident,
// a check per 1,024): 200 x 400, FP64 19.2 -> 3.9 us; 5,000 x 10,000, FP32 15.1 -> 4.2 us,
// FP64 20.5 -> 8.0 us; 20,000 x 40,000, FP64 with adaptive steps 31.5 -> 12.6 us; 50,000 x
// 100,000, FP64 37.6 -> 16.4 us; 100,000 x 200,000, FP32 26.6 -> 22.1 us.  The
// cluster form is bound by its barriers (two of about 1,200 cycles an attempt) and
// the latency of a slice; the grid form by its gathers (a 32-byte sector each, one
// a cycle and SM) and barriers (2,500 cycles each).
//
// GB300's FP64 unit takes 64 cycles of an SM quarter for a warp instruction
// however few lanes are active (measured; a division takes 1,500, a comparison
// about 100), so a row's nonzeros are dealt to G lanes (few where rows abound),
// rows of similar length sit together, and a slice of 32 / G rows is stored
// transposed, padded to its longest row, so that its loads are free of conflicts
// and of conditions (with a condition per nonzero the compiler made one branch
// each: 300 cycles a nonzero).  Padding repeats the row's first column with the
// value 0.  All orders are fixed: results are bitwise reproducible.
#pragma once

#include "common.cuh"
#include "control.cuh"

namespace pdhg {

constexpr int kResNT = 1024;
constexpr int kResMaxWarps = kResNT / 32;
constexpr int kResSteps = 16;        // nonzeros of a row per lane of its slice, at most (up to 32 lanes)
constexpr int kResMaxRow = 8192;     // longest row of a resident LP
constexpr int kResMaxCluster = 16;
constexpr int kResMaxGrid = 160;
constexpr unsigned long long kResWaitNs = 1000ull * 1000 * 1000;   // bound of a barrier's wait

// One orientation (rows of K, or of K^T): global arrays, and the layout of a
// block's share in shared memory.
template <typename T>
struct ResMat {
    const T* sval;
    ResSide s;
};

// A block's share in shared memory.
template <typename T>
struct ResTile {
    T* val;
    int* idx;
    int4* slice;     // first entry, steps, log2 of the lanes per row, first slot
    int* row;        // row of each slot (-1: none)
    int nslice, nslot;
};

extern __shared__ __align__(16) unsigned char res_dyn[];

// Copies a block's share into shared memory at p (advanced).
template <typename T>
__device__ __forceinline__ ResTile<T> res_tile(const ResMat<T>& A, unsigned char*& p)
{
    const int c = blockIdx.x;
    const int e0 = A.s.eptr[c], ne = A.s.eptr[c + 1] - e0;
    const int s0 = A.s.cptr[c], r0 = A.s.rptr[c];
    ResTile<T> t;
    t.nslice = A.s.cptr[c + 1] - s0;
    t.nslot = A.s.rptr[c + 1] - r0;
    t.val = reinterpret_cast<T*>(p);
    p += sizeof(T) * (size_t)A.s.max_entry;
    t.idx = reinterpret_cast<int*>(p);
    p += sizeof(int) * (size_t)A.s.max_entry;
    t.slice = reinterpret_cast<int4*>(p);
    p += sizeof(int4) * (size_t)A.s.max_slice;
    t.row = reinterpret_cast<int*>(p);
    p += sizeof(int) * (size_t)A.s.max_slot;
    // entries come in multiples of 32: whole 16-byte words
    const int4* gi = reinterpret_cast<const int4*>(A.s.sidx + e0);
    for (int i = threadIdx.x; i < ne / 4; i += blockDim.x)
        reinterpret_cast<int4*>(t.idx)[i] = __ldg(gi + i);
    const int4* gv = reinterpret_cast<const int4*>(A.sval + e0);
    for (int i = threadIdx.x; i < ne / (int)(16 / sizeof(T)); i += blockDim.x)
        reinterpret_cast<int4*>(t.val)[i] = __ldg(gv + i);
    for (int i = threadIdx.x; i < t.nslice; i += blockDim.x) t.slice[i] = __ldg(A.s.slice + s0 + i);
    for (int i = threadIdx.x; i < t.nslot; i += blockDim.x) t.row[i] = __ldg(A.s.row + r0 + i);
    return t;
}

// A block's arrival at the grid barrier: 16-byte words of a partial sum and the
// barrier's number, written and read as a whole.  Two sets, used in turn: a
// block reaches barrier n + 1 only after it has read the arrivals of barrier n,
// so set n % 2 is free at barrier n + 2.
struct __align__(64) ResSlot {
    ulonglong2 w[4];        // (bits, number); w[3]: block 0's device clock
};

__device__ __forceinline__ ulonglong2 ld_relaxed_b128(const ulonglong2* p)
{
    ulonglong2 v;
    asm volatile(
        "{\n\t.reg .b128 t;\n\t"
        "ld.relaxed.gpu.global.b128 t, [%2];\n\t"
        "mov.b128 {%0, %1}, t;\n\t}"
        : "=l"(v.x), "=l"(v.y)
        : "l"(p)
        : "memory");
    return v;
}

__device__ __forceinline__ void st_relaxed_b128(ulonglong2* p, unsigned long long a,
                                                unsigned long long b)
{
    asm volatile(
        "{\n\t.reg .b128 t;\n\t"
        "mov.b128 t, {%1, %2};\n\t"
        "st.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
        "l"(a), "l"(b)
        : "memory");
}

__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ uint32_t res_smem(const void* p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ uint32_t res_mapa(uint32_t a, int rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

__device__ __forceinline__ void res_cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                     : "memory");
}

// Shared memory of this block to the same place of block `rank`, completing on
// its mbarrier (addresses and size in multiples of 16 bytes).
__device__ __forceinline__ void res_bulk(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t mbar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, "
        "[%3];" ::"r"(dst),
        "r"(src), "r"(bytes), "r"(mbar)
        : "memory");
}

// The sum of 32 floats, exact to 2^-78 of the largest's binade: the mantissas, shifted to
// the largest exponent, add up as integers (a fixed-point accumulator, as Kulisch's) in
// three pieces of 26 bits, which 32 lanes cannot overflow.  Lane 0 keeps the pieces and
// the exponent; fixed_value turns them into a double.
__device__ __forceinline__ int4 warp_fixed_sum(float v)
{
    const unsigned b = __float_as_uint(v);
    const unsigned ex = (b >> 23) & 255u;
    const int e = max((int)__reduce_max_sync(0xffffffffu, ex), 1);
    const unsigned long long m = (b & 0x7fffffu) | (ex ? 0x800000u : 0u);
    const int s = 54 - (e - max((int)ex, 1));        // m moves up by s bits, to 78 in all
    const int hi = s >= 52 ? (int)(m << (s - 52)) : (int)(m >> min(52 - s, 63));
    const int mi = (int)((s >= 26 ? m << (s - 26) : m >> min(26 - s, 63)) & 0x3ffffffu);
    const int lo = (int)((s >= 0 ? m << s : m >> min(-s, 63)) & 0x3ffffffu);
    const bool neg = b >> 31;
    return make_int4(__reduce_add_sync(0xffffffffu, neg ? -hi : hi),
                     __reduce_add_sync(0xffffffffu, neg ? -mi : mi),
                     __reduce_add_sync(0xffffffffu, neg ? -lo : lo), e);
}
__device__ __forceinline__ double fixed_value(const int4 p)
{
    if (p.w == 255) return __longlong_as_double(0x7ff8000000000000ll);   // an infinity or a NaN
    const double unit = __longlong_as_double((long long)(1023 + p.w - 204) << 52);
    return fma((double)(((long long)p.x << 26) + p.y), 67108864.0, (double)p.z) * unit;
}

// Sums over the block of NV per-thread values, valid in lane 0 of warp q for value
// q.  FP32 values: as integers within a warp (with a tree of doubles the FP64 unit would
// take 5 instructions of every warp for a value), the 32 warps' sums in doubles, 32 to an
// instruction (5,000 x 10,000, 512 FP32 iterations: 4.16 ms a solve; 4.25 ms with pairs of
// floats, which also kept 48 bits only).  FP64 values: through shared memory, so that every FP64 instruction adds 32
// of them (1,024 values: 41 warp instructions instead of 165).  lg[q]: only lanes that are
// a multiple of 2^lg[q] hold a value of v[q].
template <typename T, int NV>
__device__ __forceinline__ double res_block_sums(const T (&v)[NV], const int (&lg)[NV])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    double t = 0.0;
    if constexpr (sizeof(T) == 4) {
        __shared__ int4 red[NV][kResMaxWarps];
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const int4 p = warp_fixed_sum(v[q]);
            if (lane == 0) red[q][warp] = p;
        }
        __syncthreads();
        if (warp < NV) t = warp_sum(lane < nw ? fixed_value(red[warp][lane]) : 0.0);
    } else {
        __shared__ double all[NV][kResNT];
        __shared__ double part[NV][4][32];
#pragma unroll
        for (int q = 0; q < NV; ++q)
            if ((lane & ((1 << lg[q]) - 1)) == 0) all[q][threadIdx.x >> lg[q]] = v[q];
        __syncthreads();
        for (int k = warp; k < 4 * NV; k += nw) {
            const int q = k >> 2, p = k & 3;
            int n = 0;
#pragma unroll
            for (int j = 0; j < NV; ++j)
                if (j == q) n = (nw << 5) >> lg[j];
            double a = 0.0;
            for (int i = p * 32 + lane; i < n; i += 128) a += all[q][i];
            part[q][p][lane] = a;
        }
        __syncthreads();
        if (warp < NV)
            t = warp_sum((part[warp][0][lane] + part[warp][1][lane]) +
                         (part[warp][2][lane] + part[warp][3][lane]));
    }
    return t;
}

// Values that one block hands to all at a barrier: up to three sums and block 0's
// device clock.
struct __align__(16) ResPay {
    double v[3];
    unsigned long long clk;
};

// Shared state of the barriers.
struct ResShared {
    uint64_t mbar[2];                  // cluster form: arrivals of the x and of the y parts
    ResPay out[2];                     // this block's sums, two sets used in turn
    ResPay in[2][kResMaxCluster];      // every block's sums, two sets used in turn
    double tot[4];
    unsigned long long clk;
    int failed;
};

// The barrier between two products, called by every thread.  `side`: which
// vector the blocks have just written (0: x, 1: y); vec, chunk: this block's copy
// of it and the bytes of a block's own part.  NV > 0 or CLOCK: `decide` runs in
// thread 0 of every block with the sums over all threads of v[0..NV) and block
// 0's device clock (the same bits in every block).  The other threads do not wait
// for it: they go on with what does not depend on the decision (warp 0 has no
// rows) and meet it at the caller's next __syncthreads.  When a wait runs out,
// sh.failed is set (and the error flag).
//
// Why nothing is overwritten while it may still be read (cluster form): a block
// that has passed barrier b has every block's arrival at b, so every block has
// passed b - 1: it has received this block's words of b - 1 (their bulk copies have
// read their source), decided on b - 1 and done its product after b - 1.  A block
// may therefore write, for barrier b + 1, over what it last sent at barrier b - 1 or
// before, here and in the others' memory.  The sums take the two sets in turn by deciding
// barriers alone, so a set comes back after one deciding barrier at least, whether
// plain barriers lie between (the iterations) or not (the last two of the power
// iteration); the parts of x and of y are sent at every other barrier (`side`
// alternates), which also keeps the phases of the two mbarriers apart.
struct ResBarrier {
    ResShared& sh;
    ResSlot* slots;            // grid form: [2][gridDim.x]
    unsigned long long* arrived;   // grid form: arrivals at barriers without sums, ever
    unsigned int seq;              // deciding barriers met
    unsigned long long plain;      // arrivals awaited
    unsigned int par;          // parities of the mbarriers' next waits
    int* err;
    bool cluster;

    __device__ __forceinline__ void init()
    {
        if (threadIdx.x == 0) {
            sh.failed = 0;
            // a launch adds whole rounds, and none ends before this block arrives
            if (!cluster) plain = ld_relaxed_u64(arrived) / gridDim.x * gridDim.x;
            for (int k = 0; k < 2; ++k)
                asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(res_smem(&sh.mbar[k]))
                             : "memory");
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncthreads();
        // every block runs, its mbarriers are ready: the others may write to it
        if (cluster && gridDim.x > 1) res_cluster_sync();
    }
    // no block leaves while its shared memory can be read or written by others
    __device__ __forceinline__ void end()
    {
        if (cluster && gridDim.x > 1) res_cluster_sync();
    }
    __device__ __forceinline__ void fail()
    {
        sh.failed = 1;
        atomicOr(err, 1);
    }
    // whether a spinning thread goes on: checks the clock every 64 spins
    __device__ __forceinline__ bool spin(int& spins, unsigned long long& t0)
    {
        if ((++spins & 63) != 0) return true;
        const unsigned long long n = global_ns();
        if (t0 == 0) t0 = n;
        return n - t0 <= kResWaitNs;
    }

    template <typename T, int NV, bool CLOCK, class D>
    __device__ __forceinline__ void meet(int side, T* vec, int chunk, const T (&v)[NV > 0 ? NV : 1],
                                         const int (&lg)[NV > 0 ? NV : 1], D&& decide)
    {
        constexpr int NT_ = NV > 0 ? NV : 1;
        constexpr bool DEC = NV > 0 || CLOCK;
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const int nb = gridDim.x;
        double mine = 0.0;     // warp q < NV, lane 0: the block's sum of v[q]
        if constexpr (NV > 0) mine = res_block_sums<T, NV>(v, lg);
        if (nb == 1) {
            if (NV > 0 && warp < NV && lane == 0) sh.tot[warp] = mine;
            __syncthreads();
            if (DEC && threadIdx.x == 0) decide(sh.tot, CLOCK ? global_ns() : 0ull);
            return;
        }
        if (cluster) {
            if (DEC) ++seq;
            ResPay* in = sh.in[seq & 1];
            ResPay& out = sh.out[seq & 1];
            const uint32_t mb = res_smem(&sh.mbar[side]);
            if (NV > 0 && warp < NV && lane == 0) out.v[warp] = in[blockIdx.x].v[warp] = mine;
            if (CLOCK && warp == 0 && lane == 0 && blockIdx.x == 0)
                out.clk = in[0].clk = global_ns();
            // this thread's entries are in the copy before the bulk copies read it
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncthreads();
            if (warp == 0) {
                if (lane == 0) {
                    const uint32_t bytes = (uint32_t)((nb - 1) * (chunk + (DEC ? 32 : 0)));
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb),
                                 "r"(bytes)
                                 : "memory");
                }
                if (lane < nb && lane != (int)blockIdx.x) {
                    const uint32_t rm = res_mapa(mb, lane);
                    const uint32_t src = res_smem(vec) + (uint32_t)blockIdx.x * (uint32_t)chunk;
                    res_bulk(res_mapa(src, lane), src, (uint32_t)chunk, rm);
                    if (DEC)
                        res_bulk(res_mapa(res_smem(&in[blockIdx.x]), lane), res_smem(&out), 32u, rm);
                }
            }
            const uint32_t want = (par >> side) & 1u;
            par ^= 1u << side;
            unsigned long long t0 = 0;
            int spins = 0;
            for (;;) {
                uint32_t done;
                asm volatile(
                    "{\n\t.reg .pred p;\n\t"
                    "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                    "selp.u32 %0, 1, 0, p;\n\t}"
                    : "=r"(done)
                    : "r"(mb), "r"(want)
                    : "memory");
                if (done) break;
                if (!spin(spins, t0)) {
                    fail();
                    break;
                }
            }
            if (DEC && warp == 0) {
                // the sums of the blocks in a fixed order, one quantity after another
#pragma unroll
                for (int q = 0; q < NV; ++q) {
                    const double x = warp_sum(lane < nb ? in[lane].v[q] : 0.0);
                    if (lane == 0) sh.tot[q] = x;
                }
                if (lane == 0) decide(sh.tot, CLOCK ? in[0].clk : 0ull);
            }
            return;
        }
        __syncthreads();
        if (!DEC) {
            // a count of arrivals: one address instead of one per block (with NV
            // sums: the words below)
            plain += (unsigned int)nb;
            if (threadIdx.x == 0) {
                asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(arrived) : "memory");
                unsigned long long t0 = 0;
                int spins = 0;
                for (;;) {
                    unsigned long long a;
                    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(a) : "l"(arrived) : "memory");
                    if (a >= plain) break;
                    if (!spin(spins, t0)) {
                        fail();
                        break;
                    }
                }
            }
            __syncthreads();
            return;
        }
        ++seq;
        ResSlot* set = slots + (size_t)(seq & 1) * nb;
        constexpr int PER = kResMaxGrid / 32;
        if (warp < NT_) {
            // a warp per quantity: its block's arrival, then every block's, all loads
            // in flight
            if (lane == 0) {
                ResSlot* me = set + blockIdx.x;
                __threadfence();
                st_relaxed_b128(&me->w[warp], (unsigned long long)__double_as_longlong(mine), seq);
                if (CLOCK && threadIdx.x == 0 && blockIdx.x == 0)
                    st_relaxed_b128(&me->w[3], global_ns(), seq);
            }
            unsigned long long x[PER], c3 = 0, t0 = 0;
            int spins = 0;
            for (;;) {
                bool ready = true;
#pragma unroll
                for (int j = 0; j < PER; ++j) {
                    const int i = lane + 32 * j;
                    if (i < nb) {
                        const ulonglong2 w = ld_relaxed_b128(&set[i].w[warp]);
                        x[j] = w.x;
                        ready = ready && (unsigned int)w.y == seq;
                    }
                }
                if (CLOCK && threadIdx.x == 0) {
                    const ulonglong2 w = ld_relaxed_b128(&set[0].w[3]);
                    c3 = w.x;
                    ready = ready && (unsigned int)w.y == seq;
                }
                if (__all_sync(0xffffffffu, ready)) break;
                if (__any_sync(0xffffffffu, !spin(spins, t0))) {
                    if (lane == 0) fail();
                    break;
                }
            }
            __threadfence();   // what the other blocks wrote is read after this
            if constexpr (NV > 0) {
                double s = 0.0;
#pragma unroll
                for (int j = 0; j < PER; ++j)
                    if (lane + 32 * j < nb) s += __longlong_as_double((long long)x[j]);
                s = warp_sum(s);
                if (lane == 0) sh.tot[warp] = s;
            }
            if (CLOCK && threadIdx.x == 0) sh.clk = c3;
        }
        __syncthreads();
        if (threadIdx.x == 0) decide(sh.tot, CLOCK ? sh.clk : 0ull);
    }

    template <typename T>
    __device__ __forceinline__ bool wait_all(int side, T* vec, int chunk)
    {
        const T none[1] = {T(0)};
        const int lg[1] = {0};
        meet<T, 0, false>(side, vec, chunk, none, lg, [](const double*, unsigned long long) {});
        if (cluster) __syncthreads();   // every thread's wait is over (or its failure known)
        return !sh.failed;
    }
};

// The gathered vector: each block's copy in shared memory (SM), or global memory
// through L2 (its entries are written during the launch, by any block).
template <typename T, bool SM>
struct ResVec {
    const T* g;
    const T* s;
    __device__ __forceinline__ T operator()(int c) const
    {
        if constexpr (SM) return s[c];
        else return __ldcg(g + c);
    }
};

// U gathers of a slice, all in flight
template <int U, typename T, bool SM>
__device__ __forceinline__ void res_gather(const int* si, const ResVec<T, SM>& x, T (&xv)[U])
{
    int c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) c[u] = si[32 * u];
#pragma unroll
    for (int u = 0; u < U; ++u) xv[u] = x(c[u]);
}
template <int U, int C, typename T>
__device__ __forceinline__ void res_fma(const T* sv, const T (&xv)[U], T (&a)[C])
{
#pragma unroll
    for (int u = 0; u < U; ++u) a[u % C] = fma(sv[32 * u], xv[u], a[u % C]);
}
// A lane's n nonzeros of a slice in C sums, one for every C-th, which then meet in pairs
// (two, four from 8 nonzeros, two lanes from 17: the rounding of the CSR ring's lane groups,
// the figures beside slice_sum; 200 x 400 FP64 4 % slower than with one chain, FP32 as fast);
// the gathers of the next four are in flight while four are multiplied (the FP64
// additions would otherwise wait for the gathers and the gathers for them)
template <int C, typename T, bool SM>
__device__ __forceinline__ T res_sum(const int* si, const T* sv, int n, const ResVec<T, SM>& x)
{
    T a[C];
#pragma unroll
    for (int k = 0; k < C; ++k) a[k] = T(0);
    if (n >= 4) {
        T x0[4], x1[4];
        res_gather<4, T, SM>(si, x, x0);
        for (;;) {
            if (n < 8) {
                res_fma<4, C, T>(sv, x0, a);
                n -= 4, si += 128, sv += 128;
                break;
            }
            res_gather<4, T, SM>(si + 128, x, x1);
            res_fma<4, C, T>(sv, x0, a);
            if (n < 12) {
                res_fma<4, C, T>(sv + 128, x1, a);
                n -= 8, si += 256, sv += 256;
                break;
            }
            res_gather<4, T, SM>(si + 256, x, x0);
            res_fma<4, C, T>(sv + 128, x1, a);
            n -= 8, si += 256, sv += 256;
        }
    }
    if (n >= 2) {
        T xv[2];
        res_gather<2, T, SM>(si, x, xv);
        res_fma<2, C, T>(sv, xv, a);
        n -= 2, si += 64, sv += 64;
    }
    if (n >= 1) {
        T xv[1];
        res_gather<1, T, SM>(si, x, xv);
        res_fma<1, C, T>(sv, xv, a);
    }
#pragma unroll
    for (int o = 1; o < C; o <<= 1)
#pragma unroll
        for (int k = 0; k < C; k += 2 * o) a[k] += a[k + o];
    return a[0];
}
template <typename T, bool SM>
__device__ __forceinline__ T res_dot(const int* si, const T* sv, int n, const ResVec<T, SM>& x)
{
    return n >= 8 ? res_sum<4, T, SM>(si, sv, n, x) : res_sum<2, T, SM>(si, sv, n, x);
}

// The products of the block's rows with x and the epilogue f.row(slot, row, sum) of
// each, by one lane; warp w > 0 takes the slices w - 1, w - 1 + (warps - 1), ...
// `ready` runs between the product of a warp's first slice and the first epilogue,
// in every thread once (a __syncthreads for what the epilogue waits for); false:
// nothing more is done.  product = false: the epilogues alone, with sum 0.
template <typename T, bool SM, class F, class R>
__device__ __forceinline__ bool res_phase(const ResTile<T>& A, const ResVec<T, SM>& x, F& f,
                                          bool product, R&& ready)
{
    const int lane = threadIdx.x & 31, step = (blockDim.x >> 5) - 1, warp = threadIdx.x >> 5;
    const int first = warp > 0 ? warp - 1 : A.nslice;
    auto dot = [&](const int4& d) {
        T a = res_dot<T, SM>(A.idx + d.x + lane, A.val + d.x + lane, d.y, x);
        for (int o = (1 << d.z) >> 1; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        return a;
    };
    // d: first entry, steps, log2 of the lanes per row, first slot
    int4 d = make_int4(0, 0, 0, 0);
    T a = T(0);
    if (first < A.nslice) {
        d = A.slice[first];
        if (product) a = dot(d);
    }
    if (!ready()) return false;
    for (int b = first; b < A.nslice;) {
        const int slot = d.w + (lane >> d.z);
        const int r = A.row[slot];
        if (r >= 0 && (lane & ((1 << d.z) - 1)) == 0) f.row(slot, r, a);
        __syncwarp();
        b += step;
        if (b < A.nslice) {
            d = A.slice[b];
            if (product) a = dot(d);
        }
    }
    return true;
}
template <typename T, bool SM, class F>
__device__ __forceinline__ void res_phase(const ResTile<T>& A, const ResVec<T, SM>& x, F& f,
                                          bool product = true)
{
    (void)res_phase<T, SM>(A, x, f, product, [] { return true; });
}

}  // namespace pdhg
