// Unrolled fixed-step PDHG and its reverse-mode derivative.
//
// Forward (Algorithm 1, theta = 1, unscaled problem): x' = clamp(x - tau (c - K^T y), l, u),
// y' = proj_Y(y + sigma (q - K (2 x' - x))) for K_iters steps from x = proj_X(0), y = 0.
// Reverse: for one step with v_x = x - tau (c - K^T y), v_y = y + sigma (q - K xbar),
// xbar = 2 x' - x, masks M_x = [l < v_x < u], M_y = [equality row or v_y > 0], and
// incoming adjoints (gx', gy'):
//   gv_y = M_y gy';   gq += sigma gv_y;   gxbar = -sigma K^T gv_y
//   gv_x = M_x (gx' + 2 gxbar);   gc += -tau gv_x
//   gx = gv_x - gxbar;   gy = gv_y + tau K gv_x
//   gK_ij += -sigma gv_y_i xbar_j + tau y_i gv_x_j
// tau and sigma are held constant.  Iterates are checkpointed every ckpt steps;
// the reverse pass recomputes one segment at a time into a ring (x, y and the
// two projection masks of every step of the segment).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "common.cuh"
#include "control.cuh"
#include "sliced.cuh"

namespace pdhg {

namespace {

inline int ew_grid_g(int64_t count)
{
    int64_t g = (count + kEW - 1) / kEW;
    if (g < 1) g = 1;
    if (g > kEWGrid) g = kEWGrid;
    return (int)g;
}

// What bounds an unrolled step of a mid-size LP is its chain of short launches and, in the
// derivative of the nonzeros, gathers and FP64 instructions.  The elementwise parts
// therefore ride on the products' epilogues (two launches a forward step, two a reverse
// step), and the derivative of the nonzeros is taken kGSteps reverse steps at a time
// (k_g_pack, k_g_sddmm).  100,000 x 200,000, 1.25M nonzeros, FP64: a product with its
// epilogue 12 to 16 us (12.2 us without one), the derivative 61 us for eight steps; a call
// of 500 iterations 85.5 -> 68.8 ms (three launches a forward and five a reverse step before).

// K^T y + primal step: x' = clamp(x - tau (c - K^T y), l, u); mask of the strict interior
template <typename T>
struct EpiGPrimal {
    PDHG_SINGLE_LP_TASK_HOOKS
    const T* y;          // being multiplied
    const T* x;
    const T *c, *l, *u;
    const double* coef;  // [0] = tau
    T* xn;
    uint8_t* mx;
    struct Pre { T x = 0, c = 0, l = 0, u = 0; };
    struct Acc {};
    __device__ bool begin() const { return true; }
    __device__ const T* xin() const { return y; }
    __device__ Pre load(int j) const { return Pre{x[j], c[j], l[j], u[j]}; }
    __device__ void row(int j, T k, const Pre& p, Acc&) const {
        const T v = p.x - (T)coef[0] * (p.c - k);
        xn[j] = res_clamp(v, p.l, p.u);
        if (mx) mx[j] = res_inside(v, p.l, p.u) ? 1 : 0;
    }
    __device__ void finish(Acc&) const {}
};

// K x' + dual step of the unrolled forward, with the dual mask
template <typename T>
struct EpiGDual {
    PDHG_SINGLE_LP_TASK_HOOKS
    const T* x;          // x' (being multiplied)
    const T* y;          // y
    const T* kx;         // K x
    const T* q;
    const uint8_t* sense;
    const double* coef;  // [1] = sigma
    T* yn;
    T* kxn;
    uint8_t* my;
    struct Pre { T y = 0, kx = 0, q = 0; uint8_t ge = 0; };
    struct Acc {};
    __device__ bool begin() const { return true; }
    __device__ const T* xin() const { return x; }
    __device__ Pre load(int i) const { return Pre{y[i], kx[i], q[i], sense[i]}; }
    __device__ void row(int i, T v, const Pre& p, Acc&) const {
        const T sigma = (T)coef[1];
        const T w = p.y + sigma * (p.q - (T(2) * v - p.kx));
        yn[i] = p.ge ? res_pos(w) : w;
        kxn[i] = v;
        if (my) my[i] = (!p.ge || res_positive(w)) ? 1 : 0;
    }
    __device__ void finish(Acc&) const {}
};

// reverse, last step of a segment: gv_y = M_y gy; dq += sigma gv_y
template <typename T>
__global__ void k_g_gvy(const uint8_t* my, const T* gy, const double* coef, T* gvy, double* dq,
                        int64_t m)
{
    const double sigma = coef[1];
    for (int64_t i = (int64_t)blockIdx.x * kEW + threadIdx.x; i < m; i += (int64_t)gridDim.x * kEW) {
        const T g = my[i] ? gy[i] : T(0);
        gvy[i] = g;
        dq[i] += sigma * (double)g;
    }
}

// reverse: gxbar = -sigma K^T gv_y; gv_x = M_x (gx + 2 gxbar); dc += -tau gv_x;
// gx <- gv_x - gxbar (epilogue of the K^T gv_y product)
template <typename T>
struct EpiGvx {
    PDHG_SINGLE_LP_TASK_HOOKS
    const T* gvy;        // being multiplied
    const uint8_t* mx;
    const double* coef;  // [0] = tau, [2] = -sigma
    T* gx;
    T* gvx;
    double* dc;
    struct Pre { T gx = 0; uint8_t in = 0; };
    struct Acc {};
    __device__ bool begin() const { return true; }
    __device__ const T* xin() const { return gvy; }
    __device__ Pre load(int j) const { return Pre{gx[j], mx[j]}; }
    __device__ void row(int j, T v, const Pre& p, Acc&) const {
        const T gb = (T)__dmul_rn((double)v, coef[2]);   // one value in both places below
        const T g = p.in ? p.gx + T(2) * gb : T(0);
        gvx[j] = g;
        dc[j] += -coef[0] * (double)g;
        gx[j] = g - gb;
    }
    __device__ void finish(Acc&) const {}
};

// reverse: gy = gv_y + tau K gv_x (epilogue of the K gv_x product) and, unless the segment
// ends, the first half of the step before: gv_y = M_y gy; dq += sigma gv_y
template <typename T>
struct EpiGy {
    PDHG_SINGLE_LP_TASK_HOOKS
    const T* gvx;        // being multiplied
    const T* gvy;
    const double* coef;  // [0] = tau, [1] = sigma
    T* gy;               // kept where the segment ends (my = nullptr)
    const uint8_t* my;   // of the step before
    T* gvyn;
    double* dq;
    struct Pre { T g = 0; uint8_t in = 0; };
    struct Acc {};
    __device__ bool begin() const { return true; }
    __device__ const T* xin() const { return gvx; }
    __device__ Pre load(int i) const { return Pre{gvy[i], my ? my[i] : (uint8_t)0}; }
    __device__ void row(int i, T v, const Pre& p, Acc&) const {
        const T g = p.g + (T)coef[0] * v;
        if (!my) {
            gy[i] = g;
            return;
        }
        const T w = p.in ? g : T(0);
        gvyn[i] = w;
        dq[i] += coef[1] * (double)w;
    }
    __device__ void finish(Acc&) const {}
};

// Reverse steps whose derivative of the nonzeros is taken together, at most.
constexpr int kGSteps = 8;

// The factors of cnt reverse steps (t, t - 1, ...) side by side, for k_g_sddmm:
// P[j][k] = (xbar_j, gv_x_j), Q[i][k] = (-sigma gv_y_i, tau y_i).  X, Y: the iterates of
// step t (X + n: those of t + 1); gvx, gvy: a vector per step.
template <typename T>
__global__ void k_g_pack(int cnt, int stride, const T* X, const T* Y, const T* gvx, const T* gvy,
                         const double* coef, double2* P, double2* Q, int64_t n, int64_t m)
{
    const double tau = coef[0], sigma = coef[1];
    for (int64_t r = (int64_t)blockIdx.x * kEW + threadIdx.x; r < n + m;
         r += (int64_t)gridDim.x * kEW) {
        if (r < n) {
            double xn = (double)X[n + r];
            for (int k = 0; k < cnt; ++k) {
                const double x = (double)X[r - k * n];
                P[r * stride + k] = make_double2(2.0 * xn - x, (double)gvx[k * n + r]);
                xn = x;
            }
        } else {
            const int64_t i = r - n;
            for (int k = 0; k < cnt; ++k)
                Q[i * stride + k] = make_double2(-sigma * (double)gvy[k * m + i],
                                                 tau * (double)Y[i - k * m]);
        }
    }
}

// reverse: dA_p += -sigma gv_y_i xbar_j + tau y_i gv_x_j for every nonzero p = (i, j),
// the packed steps one after the other.  A step by itself took five gathers of a 32-byte
// sector, 32 bytes of indices and sums, and seven FP64 instructions a nonzero; eight packed
// steps gather two 128-byte lines and take three instructions a step.  (Two, with the
// steps' terms added up before they meet dA, were 1 % faster a call, with an error against
// 64 bits of 1.3e-14 instead of 1.1e-14.)
__global__ void k_g_sddmm(const int32_t* krow, const int32_t* ci, const double2* P, const double2* Q,
                          int cnt, int stride, double* dvals, int64_t nnz)
{
    for (int64_t p = (int64_t)blockIdx.x * kEW + threadIdx.x; p < nnz;
         p += (int64_t)gridDim.x * kEW) {
        const double2* q = Q + (int64_t)krow[p] * stride;
        const double2* c = P + (int64_t)ci[p] * stride;
        double t = dvals[p];
        if (cnt == kGSteps) {
            double2 a[kGSteps], b[kGSteps];
#pragma unroll
            for (int k = 0; k < kGSteps; ++k) b[k] = c[k];
#pragma unroll
            for (int k = 0; k < kGSteps; ++k) a[k] = q[k];
#pragma unroll
            for (int k = 0; k < kGSteps; ++k) t += fma(a[k].x, b[k].x, a[k].y * b[k].y);
        } else {
            for (int k = 0; k < cnt; ++k) t += fma(q[k].x, c[k].x, q[k].y * c[k].y);
        }
        dvals[p] = t;
    }
}

template <typename T>
__global__ void k_g_init(const T* l, const T* u, T* x, T* y, int64_t n, int64_t m)
{
    for (int64_t t = (int64_t)blockIdx.x * kEW + threadIdx.x; t < n + m;
         t += (int64_t)gridDim.x * kEW) {
        if (t < n) {
            T v = T(0);
            if (v < l[t]) v = l[t];
            if (v > u[t]) v = u[t];
            x[t] = v;
        } else {
            y[t - n] = T(0);
        }
    }
}

template <typename T>
__global__ void k_g_from_double(const double* src, T* dst, int64_t count)
{
    for (int64_t t = (int64_t)blockIdx.x * kEW + threadIdx.x; t < count;
         t += (int64_t)gridDim.x * kEW)
        dst[t] = (T)src[t];
}

template <typename T>
__global__ void k_g_to_double(const T* src, double* dst, int64_t count)
{
    for (int64_t t = (int64_t)blockIdx.x * kEW + threadIdx.x; t < count;
         t += (int64_t)gridDim.x * kEW)
        dst[t] = (double)src[t];
}

// Everything one unrolled run needs, allocated per call and released at its end.
template <typename T>
struct GradBufs {
    Handle* h = nullptr;
    std::vector<void*> mem;
    lp_status alloc(void** p, size_t bytes)
    {
        cudaError_t e = cudaMalloc(p, bytes + 64);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            return e == cudaErrorMemoryAllocation ? LP_OUT_OF_MEMORY : LP_CUDA_ERROR;
        }
        mem.push_back(*p);
        return LP_OK;
    }
    ~GradBufs()
    {
        if (h) cudaStreamSynchronize(h->stream);
        for (void* p : mem) cudaFree(p);
    }
};

// Unscaled data for the unrolled iterations: no Ruiz scaling, so the engine's
// "scaled" copies are the problem itself; step sizes from Algorithm 2 on K.
template <typename T>
lp_status grad_prepare(Handle* h, const lp_opts* o, double* tau, double* sigma)
{
    lp_opts o2 = *o;
    o2.ruiz_iters = 0;
    o2.pock_chambolle = 0;
    LP_TRY(setup_engine<double>(h, &o2));
    double normK = 0.0;
    LP_TRY(setup_scale(h, &o2, &normK));
    if (std::is_same<T, float>::value) LP_TRY(setup_engine<float>(h, &o2));
    double eta = normK > 0.0 ? o->eta_scale / normK : 1.0;
    if (o->eta0 > 0.0) eta = o->eta0;
    double omega = (h->cnorm > o->eps_zero && h->qnorm > o->eps_zero) ? h->cnorm / h->qnorm : 1.0;
    if (o->omega0 > 0.0) omega = o->omega0;
    *tau = eta / omega;
    *sigma = eta * omega;
    LP_CUDA_TRY((spmv_prepare<T, EpiGPrimal<T>>()));
    LP_CUDA_TRY((spmv_prepare<T, EpiGDual<T>>()));
    LP_CUDA_TRY((spmv_prepare<T, EpiStore<T>>()));
    LP_CUDA_TRY((spmv_prepare<T, EpiGvx<T>>()));
    LP_CUDA_TRY((spmv_prepare<T, EpiGy<T>>()));
    return LP_OK;
}

// One forward step from (x, y, kx) into (xn, yn, kxn), with masks.
template <typename T>
void forward_step(Handle* h, Engine<T>& E, const double* coef, const T* x, const T* y, const T* kx,
                  T* xn, T* yn, T* kxn, uint8_t* mx, uint8_t* my)
{
    EpiGPrimal<T> ep{y, x, E.c, E.l, E.u, coef, xn, mx};
    launch_product<T>(h, E, true, h->stream, ep);
    EpiGDual<T> ed{xn, y, kx, E.q, h->sense, coef, yn, kxn, my};
    launch_product<T>(h, E, false, h->stream, ed);
    h->launches += 2;
}

// K x
template <typename T>
lp_status product(Handle* h, Engine<T>& E, const T* x, T* kx)
{
    EpiStore<T> e1{x, kx, nullptr, nullptr, nullptr};
    launch_product<T>(h, E, false, h->stream, e1);
    ++h->launches;
    LP_CUDA_TRY(cudaGetLastError());
    return LP_OK;
}

lp_status copy_out(Handle* h, double* dst, const double* src_dev, int64_t count, int space)
{
    LP_CUDA_TRY(cudaMemcpyAsync(dst, src_dev, sizeof(double) * (size_t)count,
                                space == LP_MEM_DEVICE ? cudaMemcpyDeviceToDevice
                                                       : cudaMemcpyDeviceToHost,
                                h->stream));
    return LP_OK;
}

template <typename T>
lp_status grad_impl(Handle* h, const lp_opts* o, int K, int ckpt, const double* gxK, double* dc,
                    double* dq, double* dvals, double* xK, double* yK, int space,
                    double* tau_sigma, bool backward)
{
    const int64_t m = h->m, n = h->n, nnz = h->nnz;
    cudaStream_t st = h->stream;
    double tau = 0, sigma = 0;
    LP_TRY(grad_prepare<T>(h, o, &tau, &sigma));
    if (tau_sigma) {
        tau_sigma[0] = tau;
        tau_sigma[1] = sigma;
    }
    Engine<T>& E = engine_of<T>(h);
    GradBufs<T> B;
    B.h = h;
    double* coef = nullptr;   // [tau, sigma, -sigma]
    LP_TRY(B.alloc((void**)&coef, 4 * sizeof(double)));
    const double hc[4] = {tau, sigma, -sigma, 0.0};
    LP_CUDA_TRY(cudaMemcpyAsync(coef, hc, sizeof(hc), cudaMemcpyHostToDevice, st));
    const int nseg = ckpt > 0 ? (K + ckpt - 1) / ckpt : 0;
    // checkpoints: (x, y) at t = 0, ckpt, 2 ckpt, ... (< K)
    T *CX = nullptr, *CY = nullptr;
    LP_TRY(B.alloc((void**)&CX, sizeof(T) * (size_t)std::max(1, nseg) * n));
    LP_TRY(B.alloc((void**)&CY, sizeof(T) * (size_t)std::max(1, nseg) * m));
    // forward with checkpointing
    T* x = E.X[0];
    T* y = E.Y[0];
    k_g_init<T><<<ew_grid_g(n + m), kEW, 0, st>>>(E.l, E.u, x, y, n, m);
    ++h->launches;
    LP_TRY(product<T>(h, E, x, E.KX[0]));
    int cur = 0;
    for (int t = 0; t < K; ++t) {
        if (backward && t % ckpt == 0) {
            const int c = t / ckpt;
            LP_CUDA_TRY(cudaMemcpyAsync(CX + (size_t)c * n, E.X[cur], sizeof(T) * n,
                                        cudaMemcpyDeviceToDevice, st));
            LP_CUDA_TRY(cudaMemcpyAsync(CY + (size_t)c * m, E.Y[cur], sizeof(T) * m,
                                        cudaMemcpyDeviceToDevice, st));
        }
        forward_step<T>(h, E, coef, E.X[cur], E.Y[cur], E.KX[cur], E.X[cur ^ 1], E.Y[cur ^ 1],
                        E.KX[cur ^ 1], nullptr, nullptr);
        cur ^= 1;
    }
    LP_CUDA_TRY(cudaGetLastError());
    double* dtmp = nullptr;   // FP64 staging of outputs [max(n, m, nnz)]
    LP_TRY(B.alloc((void**)&dtmp, sizeof(double) * (size_t)std::max({n, m, nnz})));
    if (xK) {
        k_g_to_double<T><<<ew_grid_g(n), kEW, 0, st>>>(E.X[cur], dtmp, n);
        LP_TRY(copy_out(h, xK, dtmp, n, space));
        LP_CUDA_TRY(cudaStreamSynchronize(st));
    }
    if (yK) {
        k_g_to_double<T><<<ew_grid_g(m), kEW, 0, st>>>(E.Y[cur], dtmp, m);
        LP_TRY(copy_out(h, yK, dtmp, m, space));
        LP_CUDA_TRY(cudaStreamSynchronize(st));
    }
    if (!backward) {
        int derr = 0;
        LP_CUDA_TRY(cudaMemcpyAsync(&derr, h->dev_err, sizeof(int), cudaMemcpyDeviceToHost, st));
        LP_CUDA_TRY(cudaStreamSynchronize(st));
        return derr ? LP_DEVICE_TIMEOUT : LP_OK;
    }

    // reverse pass
    T *RX = nullptr, *RY = nullptr, *gx = nullptr, *gy = nullptr, *gvx = nullptr, *gvy = nullptr;
    double2 *P = nullptr, *Q = nullptr;
    const int S = h->lean ? 1 : std::min(kGSteps, ckpt);   // reverse steps packed together
    uint8_t *RMX = nullptr, *RMY = nullptr;
    double *ddc = nullptr, *ddq = nullptr, *ddv = nullptr;
    LP_TRY(B.alloc((void**)&RX, sizeof(T) * (size_t)(ckpt + 1) * n));
    LP_TRY(B.alloc((void**)&RY, sizeof(T) * (size_t)(ckpt + 1) * m));
    LP_TRY(B.alloc((void**)&RMX, (size_t)ckpt * n));
    LP_TRY(B.alloc((void**)&RMY, (size_t)ckpt * m));
    LP_TRY(B.alloc((void**)&gx, sizeof(T) * n));
    LP_TRY(B.alloc((void**)&gy, sizeof(T) * m));
    LP_TRY(B.alloc((void**)&gvx, sizeof(T) * (size_t)S * n));
    LP_TRY(B.alloc((void**)&gvy, sizeof(T) * (size_t)S * m));
    LP_TRY(B.alloc((void**)&P, sizeof(double2) * (size_t)S * n));
    LP_TRY(B.alloc((void**)&Q, sizeof(double2) * (size_t)S * m));
    LP_TRY(B.alloc((void**)&ddc, sizeof(double) * n));
    LP_TRY(B.alloc((void**)&ddq, sizeof(double) * m));
    LP_TRY(B.alloc((void**)&ddv, sizeof(double) * (size_t)std::max<int64_t>(nnz, 1)));
    LP_CUDA_TRY(cudaMemsetAsync(ddc, 0, sizeof(double) * n, st));
    LP_CUDA_TRY(cudaMemsetAsync(ddq, 0, sizeof(double) * m, st));
    LP_CUDA_TRY(cudaMemsetAsync(ddv, 0, sizeof(double) * (size_t)std::max<int64_t>(nnz, 1), st));
    LP_CUDA_TRY(cudaMemsetAsync(gy, 0, sizeof(T) * m, st));
    // incoming adjoint of x_K
    {
        double* g64 = dtmp;
        LP_CUDA_TRY(cudaMemcpyAsync(g64, gxK, sizeof(double) * n,
                                    space == LP_MEM_DEVICE ? cudaMemcpyDeviceToDevice
                                                           : cudaMemcpyHostToDevice,
                                    st));
        k_g_from_double<T><<<ew_grid_g(n), kEW, 0, st>>>(g64, gx, n);
        ++h->launches;
    }
    for (int sgi = nseg - 1; sgi >= 0; --sgi) {
        const int t0 = sgi * ckpt;
        const int len = std::min(ckpt, K - t0);
        // recompute the segment: ring slot s holds iterate t0 + s, masks of step t0 + s
        LP_CUDA_TRY(cudaMemcpyAsync(RX, CX + (size_t)sgi * n, sizeof(T) * n,
                                    cudaMemcpyDeviceToDevice, st));
        LP_CUDA_TRY(cudaMemcpyAsync(RY, CY + (size_t)sgi * m, sizeof(T) * m,
                                    cudaMemcpyDeviceToDevice, st));
        LP_TRY(product<T>(h, E, RX, E.KX[0]));
        int c = 0;
        for (int s = 0; s < len; ++s) {
            forward_step<T>(h, E, coef, RX + (size_t)s * n, RY + (size_t)s * m, E.KX[c],
                            RX + (size_t)(s + 1) * n, RY + (size_t)(s + 1) * m, E.KX[c ^ 1],
                            RMX + (size_t)s * n, RMY + (size_t)s * m);
            c ^= 1;
        }
        // reverse through the segment; slot k of gvx and gvy: step s of the pack begun
        // at step s + k
        k_g_gvy<T><<<ew_grid_g(m), kEW, 0, st>>>(RMY + (size_t)(len - 1) * m, gy, coef, gvy, ddq, m);
        ++h->launches;
        for (int s = len - 1, k = 0; s >= 0; --s) {
            const T* gvy_s = gvy + (size_t)k * m;
            T* gvx_s = gvx + (size_t)k * n;
            EpiGvx<T> eg{gvy_s, RMX + (size_t)s * n, coef, gx, gvx_s, ddc};
            launch_product<T>(h, E, true, st, eg);
            const bool full = ++k == S || s == 0;
            // before the K product, which may write the first slot anew
            if (full && nnz > 0) {
                const int t = s + k - 1;
                k_g_pack<T><<<ew_grid_g(n + m), kEW, 0, st>>>(k, S, RX + (size_t)t * n,
                                                              RY + (size_t)t * m, gvx, gvy, coef, P, Q,
                                                              n, m);
                k_g_sddmm<<<ew_grid_g(nnz), kEW, 0, st>>>(h->krow, h->ci, P, Q, k, S, ddv, nnz);
                h->launches += 2;
            }
            if (full) k = 0;
            EpiGy<T> ey{gvx_s, gvy_s, coef, gy, s > 0 ? RMY + (size_t)(s - 1) * m : nullptr,
                        gvy + (size_t)k * m, ddq};
            launch_product<T>(h, E, false, st, ey);
            h->launches += 2;
        }
        LP_CUDA_TRY(cudaGetLastError());
    }
    LP_TRY(copy_out(h, dc, ddc, n, space));
    LP_TRY(copy_out(h, dq, ddq, m, space));
    if (nnz > 0) LP_TRY(copy_out(h, dvals, ddv, nnz, space));
    int derr = 0;
    LP_CUDA_TRY(cudaMemcpyAsync(&derr, h->dev_err, sizeof(int), cudaMemcpyDeviceToHost, st));
    LP_CUDA_TRY(cudaStreamSynchronize(st));
    return derr ? LP_DEVICE_TIMEOUT : LP_OK;
}

}  // namespace

lp_status run_grad(Handle* h, const lp_opts* o, int K_iters, int ckpt, const double* gxK,
                   double* dc, double* dq, double* dvals, double* xK, int space, double* tau_sigma)
{
    if (o->precision == LP_PREC_MIXED)
        return grad_impl<float>(h, o, K_iters, ckpt, gxK, dc, dq, dvals, xK, nullptr, space,
                                tau_sigma, true);
    return grad_impl<double>(h, o, K_iters, ckpt, gxK, dc, dq, dvals, xK, nullptr, space,
                             tau_sigma, true);
}

lp_status run_unroll(Handle* h, const lp_opts* o, int K_iters, double* xK, double* yK, int space,
                     double* tau_sigma)
{
    if (o->precision == LP_PREC_MIXED)
        return grad_impl<float>(h, o, K_iters, 1, nullptr, nullptr, nullptr, nullptr, xK, yK, space,
                                tau_sigma, false);
    return grad_impl<double>(h, o, K_iters, 1, nullptr, nullptr, nullptr, nullptr, xK, yK, space,
                             tau_sigma, false);
}

}  // namespace pdhg
