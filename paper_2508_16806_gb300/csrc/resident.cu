// The resident kernels (see resident.cuh): a check period of restarted PDHG or
// of Halpern iterations, and the power iteration of Algorithm 2, each in one
// launch; and the host plan that chooses them.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include <cuda.h>

#include "resident.cuh"

namespace pdhg {

namespace {

template <typename T>
struct ResArgs {
    ResMat<T> K, KT;
    T *X0, *X1, *Y0, *Y1, *KX0, *KX1, *KTY0, *KTY1, *XS, *YS, *XA, *YA, *XH;
    const T *XANC, *YANC, *KXANC;
    const T *c, *q, *l, *u;
    const uint8_t* sense;
    Ctrl* ctrl;
    ResSlot* slots;
    unsigned int* seq;
    int* err;
};

// The state of a block's rows and columns in shared memory, by slot; the arrays
// with two halves follow Ctrl::cur.
template <typename T>
struct ResRows {
    T* p;
    int n;
    uint8_t* ge;
    __device__ __forceinline__ T* y(int k) const { return p + k * n; }
    __device__ __forceinline__ T* kx(int k) const { return p + (2 + k) * n; }
    __device__ __forceinline__ T* q() const { return p + 4 * n; }
    __device__ __forceinline__ T* ys() const { return p + 5 * n; }    // Halpern: the anchor's y
    __device__ __forceinline__ T* kxa() const { return p + 6 * n; }   // Halpern: the anchor's K x
};
template <typename T>
struct ResCols {
    T* p;
    int n;
    __device__ __forceinline__ T* x(int k) const { return p + k * n; }
    __device__ __forceinline__ T* kty(int k) const { return p + (2 + k) * n; }
    __device__ __forceinline__ T* c() const { return p + 4 * n; }
    __device__ __forceinline__ T* l() const { return p + 5 * n; }
    __device__ __forceinline__ T* u() const { return p + 6 * n; }
    __device__ __forceinline__ T* xs() const { return p + 7 * n; }    // Halpern: the anchor's x
};
constexpr int kResRowT = 7, kResColT = 8;   // values of T per slot

// What one thread decides for the block after a barrier.
template <typename T>
struct ResStep {
    T tau, sigma, pw, a, b, g;
    int cur, mode, hat, pend;   // pend: pw is not 0; mode as Ctrl::t_mode: 0 stop, 1 accepted, 2
                                // accepted and a check or the end follows, 3 rejected
};

// Everything of a block: the gathered copies (cluster form), its share of K and
// K^T, the state of its rows and columns.
template <typename T, bool SM>
struct ResBlock {
    T *sx, *sy;
    int cx, cy;             // bytes of a block's part of x, of y
    ResTile<T> K, KT;
    ResRows<T> R;
    ResCols<T> C;

    __device__ __forceinline__ void load(const ResArgs<T>& A, bool halpern)
    {
        unsigned char* p = res_dyn;
        cx = A.KT.s.chunk * (int)sizeof(T);
        cy = A.K.s.chunk * (int)sizeof(T);
        sx = reinterpret_cast<T*>(p);
        if (SM) p += (size_t)cx * gridDim.x;
        sy = reinterpret_cast<T*>(p);
        if (SM) p += (size_t)cy * gridDim.x;
        K = res_tile<T>(A.K, p);
        KT = res_tile<T>(A.KT, p);
        R.p = reinterpret_cast<T*>(p);
        R.n = A.K.s.max_slot;
        p += sizeof(T) * (size_t)(kResRowT * R.n);
        C.p = reinterpret_cast<T*>(p);
        C.n = A.KT.s.max_slot;
        R.ge = p + sizeof(T) * (size_t)(kResColT * C.n);
        __syncthreads();
        for (int s = threadIdx.x; s < K.nslot; s += blockDim.x) {
            const int r = K.row[s];
            if (r < 0) continue;
            R.y(0)[s] = A.Y0[r];
            R.y(1)[s] = A.Y1[r];
            R.kx(0)[s] = A.KX0[r];
            R.kx(1)[s] = A.KX1[r];
            R.q()[s] = A.q[r];
            R.ys()[s] = halpern ? A.YANC[r] : A.YS[r];
            if (halpern) R.kxa()[s] = A.KXANC[r];
            R.ge[s] = A.sense[r];
        }
        for (int s = threadIdx.x; s < KT.nslot; s += blockDim.x) {
            const int j = KT.row[s];
            if (j < 0) continue;
            C.x(0)[s] = A.X0[j];
            C.x(1)[s] = A.X1[j];
            C.kty(0)[s] = A.KTY0[j];
            C.kty(1)[s] = A.KTY1[j];
            C.c()[s] = A.c[j];
            C.l()[s] = A.l[j];
            C.u()[s] = A.u[j];
            C.xs()[s] = halpern ? A.XANC[j] : A.XS[j];
        }
    }
    // the iterates go back to global memory
    __device__ __forceinline__ void store(const ResArgs<T>& A, bool halpern)
    {
        for (int s = threadIdx.x; s < K.nslot; s += blockDim.x) {
            const int r = K.row[s];
            if (r < 0) continue;
            A.Y0[r] = R.y(0)[s];
            A.Y1[r] = R.y(1)[s];
            A.KX0[r] = R.kx(0)[s];
            A.KX1[r] = R.kx(1)[s];
            if (!halpern) A.YS[r] = R.ys()[s];
        }
        for (int s = threadIdx.x; s < KT.nslot; s += blockDim.x) {
            const int j = KT.row[s];
            if (j < 0) continue;
            A.X0[j] = C.x(0)[s];
            A.X1[j] = C.x(1)[s];
            A.KTY0[j] = C.kty(0)[s];
            A.KTY1[j] = C.kty(1)[s];
            if (!halpern) A.XS[j] = C.xs()[s];
        }
    }
};

// y' = proj_Y(y + sigma (q - (2 K x' - K x))) of one row; the pending weight of y
// enters the y sums
template <typename T, bool SM>
struct RDual {
    const T *y, *kx, *q;
    const uint8_t* ge;
    T *yn, *kxn, *ys;
    T* put;                 // where y' is gathered from
    T sigma, pw;
    bool pend, adapt;       // pw != 0; the sums of Algorithm 5 are needed
    T dy2, inter;
    __device__ void row(int s, int i, T p) {
        const T y0 = y[s], k0 = kx[s];
        if (pend) ys[s] = ys[s] + pw * y0;
        T v = y0 + sigma * (q[s] - (T(2) * p - k0));
        if (ge[s]) v = res_pos(v);
        yn[s] = v;
        put[i] = v;
        kxn[s] = p;
        if (adapt) {
            const T d = v - y0;
            dy2 += d * d;
            inter += d * (p - k0);
        }
    }
};

// K^T y' of one column (mode 1, 2: kept, and x' enters the x sums) and the next
// candidate x'' = clamp(x' - tau (c - K^T y'), l, u) (mode 1; mode 3: from the kept
// K^T y)
template <typename T, bool SM>
struct RPrimal {
    const T *x, *c, *l, *u;
    T *xn, *kty, *xs;
    T* put;                 // where x'' is gathered from
    T tau, pw;
    bool pend, adapt;
    int mode;
    T dx2;
    __device__ void row(int s, int j, T prod) {
        const T x0 = x[s];
        T k = prod;
        if (mode == 3) {
            k = kty[s];
        } else {
            kty[s] = prod;
            if (pend) xs[s] = xs[s] + pw * x0;
        }
        if (mode != 2) {
            const T v = res_clamp(x0 - tau * (c[s] - k), l[s], u[s]);
            xn[s] = v;
            put[j] = v;
            if (adapt) dx2 += (v - x0) * (v - x0);
        }
    }
};

// Copies the control block into shared memory; false when there is nothing to do.
__device__ __forceinline__ bool res_begin(const Ctrl* g, Ctrl& c)
{
    if (g->skip) return false;
    const unsigned int* src = reinterpret_cast<const unsigned int*>(g);
    unsigned int* dst = reinterpret_cast<unsigned int*>(&c);
    for (int i = threadIdx.x; i < (int)(sizeof(Ctrl) / 4); i += blockDim.x) dst[i] = src[i];
    __syncthreads();
    return true;
}

// The control block goes back to global memory (block 0), with the scalars that
// the lazy decisions left out.
__device__ __forceinline__ void res_end(Ctrl* g, Ctrl& c, unsigned int seq, unsigned int* seq_out)
{
    if (blockIdx.x != 0) return;
    if (threadIdx.x == 0) {
        if (c.W > 0.0) c.Winv = 1.0 / c.W;
        c.t_mode = 0;
        c.tick = 0;
        refresh_scalars(c);
        *seq_out = seq;
    }
    __syncthreads();
    unsigned int* dst = reinterpret_cast<unsigned int*>(g);
    const unsigned int* src = reinterpret_cast<const unsigned int*>(&c);
    for (int i = threadIdx.x; i < (int)(sizeof(Ctrl) / 4); i += blockDim.x) dst[i] = src[i];
}

// A wait ran out: the loop ends.
__device__ __forceinline__ void res_fail(Ctrl* g)
{
    if (threadIdx.x == 0) {
        g->status = LP_NUMERICAL_ERROR;
        g->want_check = 0;
        g->skip = 1;
        g->done = 1;
    }
}

// The step attempts of restarted PDHG up to the next check (or the end).
template <typename T, bool SM>
__global__ void __launch_bounds__(kResNT, 1) k_res_pdhg(const ResArgs<T> A)
{
    __shared__ Ctrl c;
    __shared__ ResStep<T> st;
    __shared__ ResShared sh;
    if (!res_begin(A.ctrl, c)) return;
    ResBlock<T, SM> B;
    B.load(A, false);
    ResBarrier bar{sh, A.slots, reinterpret_cast<unsigned long long*>(A.seq + 2), A.seq[0], 0ull, 0u,
                   A.err, SM};
    if (threadIdx.x == 0) {
        const StepScalars<T>& sc = step_scalars<T>(c);
        st = ResStep<T>{sc.tau, sc.sigma, sc.pw, T(0), T(0), T(0), c.cur, 1, 0, c.pend_w != 0.0};
    }
    bar.init();
    const bool adapt = c.adaptive != 0;
    const int lgs[3] = {A.KT.s.lgmin, A.K.s.lgmin, A.K.s.lgmin};
    auto primal = [&](int cur, int mode) {
        return RPrimal<T, SM>{B.C.x(cur), B.C.c(), B.C.l(), B.C.u(), B.C.x(cur ^ 1), B.C.kty(cur), B.C.xs(),
                              SM ? B.sx : (cur ? A.X0 : A.X1), st.tau, st.pw, st.pend != 0, adapt,
                              mode, T(0)};
    };
    // the first candidate, from the kept K^T y
    RPrimal<T, SM> fp = primal(st.cur, 3);
    res_phase<T, SM>(B.KT, ResVec<T, SM>{nullptr, B.sy}, fp, false);
    bool ok = bar.wait_all(0, B.sx, B.cx);
    while (ok) {
        const int cur = st.cur;
        RDual<T, SM> fd{B.R.y(cur), B.R.kx(cur), B.R.q(), B.R.ge, B.R.y(cur ^ 1), B.R.kx(cur ^ 1),
                        B.R.ys(), SM ? B.sy : (cur ? A.Y0 : A.Y1), st.sigma, st.pw, st.pend != 0,
                        adapt, T(0), T(0)};
        res_phase<T, SM>(B.K, ResVec<T, SM>{cur ? A.X0 : A.X1, B.sx}, fd);
        // one thread: the Algorithm 5 decision and what the K^T product does next
        auto decide = [&](double dx2, double dy2, double inter, unsigned long long now) {
            const long long k0 = c.k;
            const double eta = c.eta, omega = c.omega;
            double eta_bar = NAN;
            step_decide(&c, adapt, dy2, dx2, inter, &eta_bar, now, true);
            log_attempt(&c, k0, eta, eta_bar, omega, adapt, dx2, dy2, inter, blockIdx.x == 0);
            int mode = 0;
            if (!c.done) mode = c.k != k0 ? (c.want_check ? 2 : 1) : 3;
            st.mode = mode;
            st.cur = c.cur;
            st.pw = (T)c.pend_w;
            st.pend = mode == 1 || mode == 2;
            if (adapt) {
                st.tau = (T)div_by(c.eta, c.omega, c.romega);
                st.sigma = (T)(c.eta * c.omega);
            }
        };
        if (adapt) {
            const T v[3] = {fp.dx2, fd.dy2, fd.inter};
            bar.template meet<T, 3, true>(1, B.sy, B.cy, v, lgs,
                                          [&](const double* t, unsigned long long now) {
                                              decide(t[0], t[1], t[2], now);
                                          });
        } else {
            const T v[1] = {T(0)};
            const int none[1] = {0};
            bar.template meet<T, 0, true>(1, B.sy, B.cy, v, none,
                                          [&](const double*, unsigned long long now) {
                                              decide(0.0, 0.0, 0.0, now);
                                          });
        }
        // K^T y', and the decision before its first epilogue
        int mode = 0;
        res_phase<T, SM>(B.KT, ResVec<T, SM>{cur ? A.Y0 : A.Y1, B.sy}, fp, true, [&] {
            __syncthreads();
            ok = !sh.failed;
            mode = ok ? st.mode : 0;
            if (mode != 0) fp = primal(st.cur, mode);
            return mode != 0;
        });
        if (mode == 0 || mode == 2) break;
        ok = bar.wait_all(0, B.sx, B.cx);
    }
    __syncthreads();
    B.store(A, false);
    if (ok) res_end(A.ctrl, c, bar.seq, A.seq);
    else res_fail(A.ctrl);
    bar.end();
}

// K x^ of one row of a Halpern iteration (EpiHalpernDual)
template <typename T, bool SM>
struct RHalpernDual {
    const T *y, *kx, *q, *yanc, *kxanc;
    const uint8_t* ge;
    T *yn, *kxn, *yh;
    T* put;                 // where y+ is gathered from
    T sigma, a, b, g;
    int hat;
    T dy2, inter;
    __device__ void row(int s, int i, T kxh) {
        const T y0 = y[s], k0 = kx[s];
        T v = y0 + sigma * (q[s] - (T(2) * kxh - k0));
        if (ge[s]) v = res_pos(v);
        const T d = v - y0;
        dy2 += d * d;
        inter += d * (kxh - k0);
        const T yp = a * v - b * y0 + g * yanc[s];
        yn[s] = yp;
        put[i] = yp;
        kxn[s] = a * kxh - b * k0 + g * kxanc[s];
        if (hat) yh[i] = v;
    }
};

// K^T y+ of one column and the primal half of the next Halpern iteration
// (k_primal_halpern); stored: the primal half from the kept K^T y; last: no next
// iteration in this launch
template <typename T, bool SM>
struct RHalpernPrimal {
    const T *x, *c, *l, *u, *xanc;
    T *xn, *kty, *xa;
    T* put;                  // where x^ is gathered from
    T tau, a, b, g;
    int hat, stored, last;
    T dx2;
    __device__ void row(int s, int j, T prod) {
        T k = prod;
        if (stored) k = kty[s];
        else kty[s] = prod;
        if (last) return;
        const T x0 = x[s];
        const T v = res_clamp(x0 - tau * (c[s] - k), l[s], u[s]);
        put[j] = v;
        if (hat) xa[j] = v;
        xn[s] = a * v - b * x0 + g * xanc[s];
        dx2 += (v - x0) * (v - x0);
    }
};

// The Halpern iterations up to the next check (or the end).
template <typename T, bool SM>
__global__ void __launch_bounds__(kResNT, 1) k_res_halpern(const ResArgs<T> A)
{
    __shared__ Ctrl c;
    __shared__ ResStep<T> st;
    __shared__ double lam_next;
    __shared__ ResShared sh;
    if (!res_begin(A.ctrl, c)) return;
    ResBlock<T, SM> B;
    B.load(A, true);
    ResBarrier bar{sh, A.slots, reinterpret_cast<unsigned long long*>(A.seq + 2), A.seq[0], 0ull, 0u,
                   A.err, SM};
    // the scalars of the coming iteration, by one thread
    auto scalars = [&](double lam) {
        const long long k1 = c.k + 1;
        st.a = (T)(lam * (1.0 + c.reflect));
        st.b = (T)(lam * c.reflect);
        st.g = (T)(1.0 - lam);
        st.cur = c.cur;
        st.hat = k1 >= c.next_check || k1 >= c.max_iters;
    };
    if (threadIdx.x == 0) {
        st.tau = (T)div_by(c.eta, c.omega, c.romega);
        st.sigma = (T)(c.eta * c.omega);
        st.mode = 1;
        scalars((double)(c.epoch_k + 1) / (double)(c.epoch_k + 2));
    }
    bar.init();
    const int lgs[3] = {A.KT.s.lgmin, A.K.s.lgmin, A.K.s.lgmin};
    auto primal = [&](int stored) {
        const int cur = st.cur;
        return RHalpernPrimal<T, SM>{B.C.x(cur), B.C.c(), B.C.l(), B.C.u(), B.C.xs(), B.C.x(cur ^ 1),
                                     B.C.kty(cur), A.XA, SM ? B.sx : A.XH, st.tau, st.a, st.b, st.g,
                                     st.hat, stored, st.mode == 2, T(0)};
    };
    RHalpernPrimal<T, SM> fp = primal(1);
    res_phase<T, SM>(B.KT, ResVec<T, SM>{nullptr, B.sy}, fp, false);
    bool ok = bar.wait_all(0, B.sx, B.cx);
    while (ok) {
        const int cur = st.cur;
        if (threadIdx.x == 0)
            lam_next = (double)(c.epoch_k + 2) / (double)(c.epoch_k + 3);
        RHalpernDual<T, SM> fd{B.R.y(cur), B.R.kx(cur), B.R.q(), B.R.ys(), B.R.kxa(), B.R.ge,
                               B.R.y(cur ^ 1), B.R.kx(cur ^ 1), A.YA,
                               SM ? B.sy : (cur ? A.Y0 : A.Y1), st.sigma, st.a, st.b, st.g, st.hat,
                               T(0), T(0)};
        res_phase<T, SM>(B.K, ResVec<T, SM>{A.XH, B.sx}, fd);
        const T v[3] = {fp.dx2, fd.dy2, fd.inter};
        bar.template meet<T, 3, true>(
            1, B.sy, B.cy, v, lgs, [&](const double* t, unsigned long long now) {
                const long long k0 = c.k;
                const double eta = c.eta, omega = c.omega;
                double eta_bar = NAN;
                // the weight of the coming iteration: formed in the shadow of the
                // products (a division takes 1,500 cycles)
                const double lam = lam_next;
                step_decide(&c, 0, t[1], t[0], t[2], &eta_bar, now, true);
                log_attempt(&c, k0, eta, eta_bar, omega, true, t[0], t[1], t[2],
                            blockIdx.x == 0);
                st.mode = c.done && c.k == k0 ? 0 : (c.want_check || c.done ? 2 : 1);
                scalars(lam);
            });
        // K^T y+, and the decision before its first epilogue
        int mode = 0;
        res_phase<T, SM>(B.KT, ResVec<T, SM>{cur ? A.Y0 : A.Y1, B.sy}, fp, true, [&] {
            __syncthreads();
            ok = !sh.failed;
            mode = ok ? st.mode : 0;
            if (mode != 0) fp = primal(0);
            return mode != 0;
        });
        if (mode == 0 || mode == 2) break;
        ok = bar.wait_all(0, B.sx, B.cx);
    }
    __syncthreads();
    B.store(A, true);
    if (ok) res_end(A.ctrl, c, bar.seq, A.seq);
    else res_fail(A.ctrl);
    bar.end();
}

// Algorithm 2: t = K (b / ||b||), b = K^T t, repeated; out[0] = ||K b / ||b||||^2.
// Between the first and the last product b is divided by the power of two next to
// its norm (an exact scaling) instead of by the norm itself: the directions, and
// the last quotient, are the same, and the square root and division (4,000
// cycles, on every iteration's critical path) are left out.
template <bool SQ>
struct RPower {
    double* put;
    double scale;
    double s2;          // SQ: sum of the results' squares
    __device__ void row(int, int r, double v) {
        v *= scale;
        put[r] = v;
        if (SQ) s2 += v * v;
    }
};

template <bool SM>
__global__ void __launch_bounds__(kResNT, 1)
k_res_power(const ResArgs<double> A, int n, int iters, double* out)
{
    __shared__ double inv;
    __shared__ int go;
    __shared__ ResShared sh;
    unsigned char* p = res_dyn;
    const int cx = A.KT.s.chunk * 8, cy = A.K.s.chunk * 8;
    double* sb = SM ? reinterpret_cast<double*>(p) : A.XA;
    if (SM) p += (size_t)cx * gridDim.x;
    double* st = SM ? reinterpret_cast<double*>(p) : A.YA;
    if (SM) p += (size_t)cy * gridDim.x;
    const ResTile<double> K = res_tile<double>(A.K, p), KT = res_tile<double>(A.KT, p);
    ResBarrier bar{sh, A.slots, reinterpret_cast<unsigned long long*>(A.seq + 2), A.seq[0], 0ull, 0u,
                   A.err, SM};
    if (threadIdx.x == 0) {
        inv = 1.0;
        go = 1;
    }
    if (SM)
        for (int j = threadIdx.x; j < n; j += blockDim.x) sb[j] = 1.0;
    else
        for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x)
            sb[j] = 1.0;
    bar.init();
    bool ok = SM || bar.wait_all(0, sb, cx);
    const int lgT[1] = {A.KT.s.lgmin}, lgK[1] = {A.K.s.lgmin};
    for (int it = 0; ok && it < iters && go; ++it) {
        RPower<false> f{st, inv, 0.0};
        res_phase<double, SM>(K, ResVec<double, SM>{sb, sb}, f);
        ok = bar.wait_all(1, st, cy);
        if (!ok) break;
        RPower<true> fb{sb, 1.0, 0.0};
        res_phase<double, SM>(KT, ResVec<double, SM>{st, st}, fb);
        const double v[1] = {fb.s2};
        const bool last = it == iters - 1;
        bar.template meet<double, 1, false>(
            0, sb, cx, v, lgT, [&](const double* s, unsigned long long) {
                if (!(s[0] > 0.0)) {
                    go = 0;
                } else if (last) {
                    inv = 1.0 / sqrt(s[0]);
                } else {
                    // 2^-floor(e / 2), e the exponent of ||b||^2
                    const int e = (int)(__double_as_longlong(s[0]) >> 52) - 1023;
                    inv = __longlong_as_double((long long)(1023 - (e >> 1)) << 52);
                }
            });
        __syncthreads();
        ok = !sh.failed;
    }
    if (ok) {
        RPower<true> f{st, inv, 0.0};
        res_phase<double, SM>(K, ResVec<double, SM>{sb, sb}, f);
        const double v[1] = {f.s2};
        bar.template meet<double, 1, false>(
            1, st, cy, v, lgK, [&](const double* s, unsigned long long) {
                if (blockIdx.x == 0) {
                    *out = s[0];
                    A.seq[0] = bar.seq;
                }
            });
    }
    bar.end();
}

// Entries of the slices of one orientation: values, and (once) column indices.
template <typename T>
__global__ void k_res_fill(const int64_t* rp, const int32_t* ci, const T* val, ResSide s, int nb,
                           int32_t* sidx, T* sval)
{
    const int lane = threadIdx.x & 31;
    // a warp per slice: the slices of block c follow one another
    for (int b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; b < s.nslice;
         b += (gridDim.x * blockDim.x) >> 5) {
        int lo = 0, hi = nb - 1;   // the block of slice b
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s.cptr[mid] <= b) lo = mid;
            else hi = mid - 1;
        }
        const int4 d = s.slice[b];
        const int row = s.row[s.rptr[lo] + d.w + (lane >> d.z)];
        const int g = lane & ((1 << d.z) - 1);
        const size_t base = (size_t)s.eptr[lo] + d.x + lane;
        const int64_t p0 = row >= 0 ? rp[row] : 0, p1 = row >= 0 ? rp[row + 1] : 0;
        const int pad = p1 > p0 && sidx ? ci[p0] : 0;
        for (int k = 0; k < d.y; ++k) {
            const int64_t p = p0 + g + ((int64_t)k << d.z);
            if (sidx) sidx[base + 32 * (size_t)k] = p < p1 ? ci[p] : pad;
            if (sval) sval[base + 32 * (size_t)k] = p < p1 ? val[p] : T(0);
        }
    }
}

template <typename T>
ResArgs<T> res_args(Handle* h, Engine<T>& E)
{
    ResArgs<T> A;
    A.K = ResMat<T>{static_cast<T*>(E.res.svalK), E.res.K};
    A.KT = ResMat<T>{static_cast<T*>(E.res.svalT), E.res.T};
    A.X0 = E.X[0]; A.X1 = E.X[1]; A.Y0 = E.Y[0]; A.Y1 = E.Y[1];
    A.KX0 = E.KX[0]; A.KX1 = E.KX[1]; A.KTY0 = E.KTY[0]; A.KTY1 = E.KTY[1];
    A.XS = E.XS; A.YS = E.YS; A.XA = E.XA; A.YA = E.YA; A.XH = E.XH;
    A.XANC = E.XANC; A.YANC = E.YANC; A.KXANC = E.KXANC;
    A.c = E.c; A.q = E.q; A.l = E.l; A.u = E.u;
    A.sense = h->sense;
    A.ctrl = E.ctrl;
    A.slots = static_cast<ResSlot*>(E.res.slots);
    A.seq = E.res.seq;
    A.err = h->dev_err;
    return A;
}

// The slices of one orientation, by block (see resident.cuh).
struct SidePlan {
    std::vector<int4> slice;
    std::vector<int32_t> cptr, eptr, rptr, row;
    int chunk = 0, lgmin = 5, max_entry = 0, max_slice = 0, max_slot = 0;
};

// A row takes one lane up to kResSteps nonzeros, else as many as leave kResSteps each
// (with more lanes per short row an attempt of the 5,000 x 10,000 LP took 6.0 us instead of
// 5.4, one of the 200 x 400 LP 4.1 instead of 4.6).  cluster: block c owns the rows
// [c chunk, (c + 1) chunk); otherwise slices of rows sorted within windows of 512 go round the blocks,
// those of long rows to the block with the fewest steps.
SidePlan plan_rows(const std::vector<int64_t>& rp, int nb, bool cluster)
{
    SidePlan P;
    const int rows = (int)rp.size() - 1;
    auto len = [&](int r) { return (int)(rp[(size_t)r + 1] - rp[(size_t)r]); };
    struct Slice { int first, n, lg, steps; };
    std::vector<int32_t> order((size_t)rows);
    std::vector<std::vector<Slice>> own((size_t)nb);
    P.chunk = ((rows + nb - 1) / nb + 7) & ~7;
    const int W = cluster ? P.chunk : 512;
    std::vector<int64_t> load((size_t)nb, 0);
    std::vector<int> cnt;
    std::vector<int32_t> tmp;
    int next = 0;
    for (int w = 0; (int64_t)w * W < rows; ++w) {
        const int r0 = w * W, r1 = std::min(rows, r0 + W);
        // rows by falling length (a counting sort: stable)
        int mx = 0;
        for (int r = r0; r < r1; ++r) mx = std::max(mx, len(r));
        cnt.assign((size_t)mx + 2, 0);
        for (int r = r0; r < r1; ++r) ++cnt[(size_t)(mx - len(r)) + 1];
        for (int k = 0; k <= mx; ++k) cnt[(size_t)k + 1] += cnt[(size_t)k];
        for (int r = r0; r < r1; ++r) order[(size_t)(r0 + cnt[(size_t)(mx - len(r))]++)] = r;
        for (int i = r0; i < r1;) {
            int l = 0;
            const int n0 = len(order[(size_t)i]);
            while (l < 5 && (n0 + (1 << l) - 1) >> l > kResSteps) ++l;
            const int n = std::min(32 >> l, r1 - i), steps = (n0 + (1 << l) - 1) >> l;
            int c = w;
            if (!cluster) {
                if (steps > kResSteps / 2) {
                    c = (int)(std::min_element(load.begin(), load.end()) - load.begin());
                } else {
                    c = next;
                    next = next + 1 == nb ? 0 : next + 1;
                }
            }
            own[(size_t)c].push_back(Slice{i, n, l, steps});
            load[(size_t)c] += steps;
            P.lgmin = std::min(P.lgmin, l);
            i += n;
        }
    }
    P.cptr.push_back(0);
    P.eptr.push_back(0);
    P.rptr.push_back(0);
    for (int c = 0; c < nb; ++c) {
        int e = 0, s = 0;
        for (const Slice& sl : own[(size_t)c]) {
            P.slice.push_back(make_int4(e, sl.steps, sl.lg, s));
            for (int k = 0; k < 32 >> sl.lg; ++k)
                P.row.push_back(k < sl.n ? order[(size_t)(sl.first + k)] : -1);
            e += 32 * sl.steps;
            s += 32 >> sl.lg;
        }
        P.cptr.push_back((int32_t)P.slice.size());
        P.eptr.push_back(P.eptr.back() + e);
        P.rptr.push_back((int32_t)P.row.size());
        P.max_entry = std::max(P.max_entry, e);
        P.max_slot = std::max(P.max_slot, (s + 15) & ~15);
        P.max_slice = std::max(P.max_slice, (int)own[(size_t)c].size());
    }
    return P;
}

lp_status upload_side(Handle* h, const SidePlan& P, ResSide* s)
{
    auto up = [&](const auto& v, auto** out) -> lp_status {
        using E = typename std::decay<decltype(v[0])>::type;
        E* d = nullptr;
        LP_TRY(dev_alloc_n(h, &d, v.size() + 1));
        if (!v.empty())
            LP_CUDA_TRY(cudaMemcpyAsync(d, v.data(), v.size() * sizeof(E),
                                        cudaMemcpyHostToDevice, h->stream));
        *out = d;
        return LP_OK;
    };
    LP_TRY(up(P.slice, &s->slice));
    LP_TRY(up(P.cptr, &s->cptr));
    LP_TRY(up(P.eptr, &s->eptr));
    LP_TRY(up(P.rptr, &s->rptr));
    LP_TRY(up(P.row, &s->row));
    s->chunk = P.chunk;
    s->lgmin = P.lgmin;
    s->nslice = (int)P.slice.size();
    s->max_entry = P.max_entry;
    s->max_slice = P.max_slice;
    s->max_slot = P.max_slot;
    LP_CUDA_TRY(cudaStreamSynchronize(h->stream));   // the host lists go out of scope
    return LP_OK;
}

template <typename T>
size_t side_bytes(const SidePlan& P, int values)
{
    return (size_t)P.max_entry * (sizeof(T) + 4) + (size_t)P.max_slice * 16 +
           (size_t)P.max_slot * (4 + (size_t)values * sizeof(T) + 1);
}

int fill_grid(int nslice) { return std::max(1, std::min(nslice / 8 + 1, 1216)); }

template <typename T>
const void* res_kernel(int what, bool sm)
{
    switch (what) {
    case 0: return sm ? (const void*)k_res_pdhg<T, true> : (const void*)k_res_pdhg<T, false>;
    case 1: return sm ? (const void*)k_res_halpern<T, true> : (const void*)k_res_halpern<T, false>;
    default: return sm ? (const void*)k_res_power<true> : (const void*)k_res_power<false>;
    }
}

// Launch of a resident kernel: a cooperative grid, or one cluster.
cudaLaunchConfig_t res_config(const ResPlan& R, cudaStream_t st, cudaLaunchAttribute* at)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)R.ncta);
    cfg.blockDim = dim3((unsigned)R.threads);
    cfg.dynamicSmemBytes = R.smem;
    cfg.stream = st;
    if (R.cluster) {
        at->id = cudaLaunchAttributeClusterDimension;
        at->val.clusterDim.x = (unsigned)R.ncta;
        at->val.clusterDim.y = 1;
        at->val.clusterDim.z = 1;
    } else {
        at->id = cudaLaunchAttributeCooperative;
        at->val.cooperative = 1;
    }
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

lp_status res_launch(const ResPlan& R, cudaStream_t st, const void* f, void** args)
{
    cudaLaunchAttribute at;
    const cudaLaunchConfig_t cfg = res_config(R, st, &at);
    LP_CUDA_TRY(cudaLaunchKernelExC(&cfg, f, args));
    return LP_OK;
}

constexpr size_t kResSmem = 227 * 1024 - 4096;   // of a block, less the kernels' static part

// SMs that the kernels of a stream may use: those of its green context, or of its context
// (the device's where the driver does not say).
int stream_sms(cudaStream_t st, int device_sms)
{
    const auto entry = [](const char* name, unsigned version) {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult r = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion(name, &f, version, cudaEnableDefault, &r) != cudaSuccess)
            (void)cudaGetLastError();
        return r == cudaDriverEntryPointSuccess ? f : nullptr;
    };
    const auto get = reinterpret_cast<decltype(&cuStreamGetCtx_v2)>(entry("cuStreamGetCtx", 12050));
    const auto of_green =
        reinterpret_cast<decltype(&cuGreenCtxGetDevResource)>(entry("cuGreenCtxGetDevResource", 12040));
    const auto of_ctx = reinterpret_cast<decltype(&cuCtxGetDevResource)>(entry("cuCtxGetDevResource", 12040));
    CUcontext ctx = nullptr;
    CUgreenCtx green = nullptr;
    CUdevResource res;
    if (!get || !of_green || !of_ctx || get(st, &ctx, &green) != CUDA_SUCCESS) return device_sms;
    const CUresult r = green ? of_green(green, &res, CU_DEV_RESOURCE_TYPE_SM)
                             : of_ctx(ctx, &res, CU_DEV_RESOURCE_TYPE_SM);
    return r == CUDA_SUCCESS ? (int)res.sm.smCount : device_sms;
}

}  // namespace

template <typename T>
lp_status res_plan(Handle* h)
{
    Engine<T>& E = engine_of<T>(h);
    E.res = ResPlan{};
    ResPlan& R = E.res;
    const int64_t m = h->m, n = h->n, nnz = h->nnz;
    const size_t dyn = kResSmem - (sizeof(T) == 8 ? 28 * 1024 : 0);
    int sms = 0, coop = 0;
    LP_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device));
    LP_CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, h->device));
    // the blocks of a launch wait for one another: on a part of the device, which may not
    // hold them all at once, the launches per product stay
    if (stream_sms(h->stream, sms) < sms) return LP_OK;
    sms = std::min(sms, kResMaxGrid);
    // Resident only where nonzeros and state fit the chip's shared memory (34 MB: about
    // 1.2M nonzeros in FP32 at 12 a row): with the nonzeros left in L2 an attempt of the
    // 100,000 x 200,000 LP (1.25M nonzeros, FP32, Halpern) took 27 us, as the launches
    // per product do.  Within it the grid form is the better one up to its largest size
    // (50,000 x 100,000 in FP64: 16.4 us an attempt against 37.6), the cluster form
    // wherever it fits (5,000 x 10,000 in FP32: 5.0 us against 10.8 for the grid).
    const double need = 2.0 * (double)nnz * (sizeof(T) + 4) + (double)m * (4 + kResRowT * sizeof(T) + 1) +
                        (double)n * (4 + kResColT * sizeof(T) + 1);
    if (need > (double)dyn * sms) return LP_OK;
    for (const std::vector<int64_t>* rp : {&h->h_rp, &h->h_trp})
        for (size_t r = 0; r + 1 < rp->size(); ++r)
            if ((*rp)[r + 1] - (*rp)[r] > kResMaxRow) return LP_OK;
    SidePlan pk, pt;
    auto plan = [&](int nb, bool cluster) {
        R.ncta = nb;
        R.cluster = cluster;
        pk = plan_rows(h->h_rp, nb, cluster);
        pt = plan_rows(h->h_trp, nb, cluster);
        const size_t vec = cluster ? (size_t)nb * (pk.chunk + pt.chunk) * sizeof(T) : 0;
        R.smem = vec + side_bytes<T>(pk, kResRowT) + side_bytes<T>(pt, kResColT) + 64;
        return R.smem <= dyn;
    };
    bool fits = false;
    const int64_t slices = (std::max(m, n) + 31) / 32;
    if ((double)(m + n) * sizeof(T) + need / kResMaxCluster <= (double)dyn) {
        // a slice a block or more: the 200 x 400 LP (13 slices of columns) takes 4.5 us
        // an attempt on 8 or 16 blocks, 9.2 on one
        int nb = 1;
        while (nb < kResMaxCluster && nb < slices) nb *= 2;
        fits = plan(nb, true);
    }
    if (!fits && coop) fits = plan((int)std::min<int64_t>(sms, std::max<int64_t>(1, slices)), false);
    if (!fits) return LP_OK;
    R.threads = 32 * std::min(kResMaxWarps, std::max(4, 1 + std::max(pk.max_slice, pt.max_slice)));
    for (int what = 0; what < (std::is_same<T, double>::value ? 3 : 2); ++what) {
        const void* f = res_kernel<T>(what, R.cluster);
        LP_CUDA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn));
        if (R.cluster) {
            LP_CUDA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
            // a device (or a part of one) without room for such a cluster keeps the launches
            // per product
            int fit = 0;
            cudaLaunchAttribute at;
            const cudaLaunchConfig_t cfg = res_config(R, h->stream, &at);
            if (cudaOccupancyMaxActiveClusters(&fit, f, &cfg) != cudaSuccess || fit < 1) {
                (void)cudaGetLastError();
                return LP_OK;
            }
        } else {
            int occ = 0;
            LP_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, f, R.threads, R.smem));
            if (occ < 1) return LP_OK;
        }
    }
    LP_TRY(upload_side(h, pk, &R.K));
    LP_TRY(upload_side(h, pt, &R.T));
    int32_t *ik = nullptr, *it = nullptr;
    T *vk = nullptr, *vt = nullptr;
    LP_TRY(dev_alloc_n(h, &ik, (size_t)pk.eptr.back()));
    LP_TRY(dev_alloc_n(h, &it, (size_t)pt.eptr.back()));
    LP_TRY(dev_alloc_n(h, &vk, (size_t)pk.eptr.back()));
    LP_TRY(dev_alloc_n(h, &vt, (size_t)pt.eptr.back()));
    k_res_fill<T><<<fill_grid(R.K.nslice), 256, 0, h->stream>>>(h->rp, h->ci, nullptr, R.K, R.ncta, ik, nullptr);
    k_res_fill<T><<<fill_grid(R.T.nslice), 256, 0, h->stream>>>(h->trp, h->tci, nullptr, R.T, R.ncta, it, nullptr);
    LP_CUDA_TRY(cudaGetLastError());
    R.K.sidx = ik;
    R.T.sidx = it;
    R.svalK = vk;
    R.svalT = vt;
    ResSlot* slots = nullptr;
    LP_TRY(dev_alloc_n(h, &slots, 2 * (size_t)R.ncta));
    LP_TRY(dev_alloc_n(h, &R.seq, 4));
    LP_CUDA_TRY(cudaMemsetAsync(slots, 0, 2 * (size_t)R.ncta * sizeof(ResSlot), h->stream));
    LP_CUDA_TRY(cudaMemsetAsync(R.seq, 0, 4 * sizeof(unsigned int), h->stream));
    R.slots = slots;
    R.on = true;
    return LP_OK;
}

template <typename T>
lp_status res_values(Handle* h)
{
    Engine<T>& E = engine_of<T>(h);
    const ResPlan& R = E.res;
    if (!R.on) return LP_OK;
    k_res_fill<T><<<fill_grid(R.K.nslice), 256, 0, h->stream>>>(
        h->rp, h->ci, E.val, R.K, R.ncta, nullptr, static_cast<T*>(R.svalK));
    k_res_fill<T><<<fill_grid(R.T.nslice), 256, 0, h->stream>>>(
        h->trp, h->tci, E.tval, R.T, R.ncta, nullptr, static_cast<T*>(R.svalT));
    h->launches += 2;
    LP_CUDA_TRY(cudaGetLastError());
    return LP_OK;
}

template <typename T>
lp_status launch_res_period(Handle* h, cudaStream_t st, bool halpern)
{
    Engine<T>& E = engine_of<T>(h);
    ResArgs<T> A = res_args<T>(h, E);
    void* args[] = {&A};
    return res_launch(E.res, st, res_kernel<T>(halpern ? 1 : 0, E.res.cluster), args);
}

lp_status launch_res_power(Handle* h, cudaStream_t st, int iters, double* out)
{
    Engine<double>& E = h->e64;
    ResArgs<double> A = res_args<double>(h, E);
    int n = (int)h->n;
    void* args[] = {&A, &n, &iters, &out};
    LP_TRY(res_launch(E.res, st, res_kernel<double>(2, E.res.cluster), args));
    ++h->launches;
    return LP_OK;
}

template lp_status res_plan<double>(Handle*);
template lp_status res_plan<float>(Handle*);
template lp_status res_values<double>(Handle*);
template lp_status res_values<float>(Handle*);
template lp_status launch_res_period<double>(Handle*, cudaStream_t, bool);
template lp_status launch_res_period<float>(Handle*, cudaStream_t, bool);

}  // namespace pdhg
