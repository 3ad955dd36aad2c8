// surrogate.cu -- deep ensemble of multilayer perceptrons that map scenario
// parameters to the statistics of the final aggregate (fractal dimension and
// RDF), trained and evaluated on the GPU by the BF16 tcgen05 kernels of
// mlp.cu.  The paper has no learned component; the plain simulation is the
// surrogate's fallback and the measure of its error.
//
// Network: n_in inputs (padded to 16) -> n_layers hidden layers of width H
// with SiLU -> n_out outputs (padded to a multiple of 16).  Weights and
// activations are BF16, accumulation and the pre-activations FP32, master
// weights and the AdamW moments FP32.  Padded weight rows and columns are
// masked and stay zero.  Inputs and targets are standardised with the
// (mean, std) vectors set by npsim_surr_set_norm.
//
// Parameter layout of one network (npsim_surr_get_params): for each layer l
// in order, W_l (out_pad x in_pad, row-major) then b_l (out_pad).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "npsim_internal.cuh"

using namespace npsim;

namespace {

int round16(int x) { return (x + 15) / 16 * 16; }

int pow2_at_least(int x)
{
    int p = 32;
    while (p < x)
        p <<= 1;
    return p;
}

template <class T> cudaError_t dmalloc(T **p, size_t n)
{
    *p = nullptr;
    return cudaMalloc((void **)p, sizeof(T) * (n ? n : 1));
}

template <class T> void dfree2(T *&p)
{
    if (p)
        cudaFree((void *)p);
    p = nullptr;
}

} // namespace

struct npsim_surr {
    int n_in = 0, n_in_p = 0, H = 0, NL = 0, n_out = 0, n_out_p = 0, n_nets = 0, sms = 0;
    // parameters of all networks as flat vectors [n_nets][n_params] (the layout of
    // npsim_surr_get_params): FP32 master weights, gradients, AdamW moments; BF16
    // copies and transposes per layer, all networks in one block (D.Wb, D.Wt)
    NetDims D{};
    float *W = nullptr, *G = nullptr, *mom = nullptr, *var = nullptr;
    unsigned char *mask = nullptr; // [n_params] bit 0: a parameter (not padding), bit 1: decays
    std::vector<float> xm, xs, ym, ys; // normalisation
    cudaStream_t st = nullptr;
    // prediction of a batch of up to bcap rows
    int bcap = 0;
    float *xin = nullptr;          // raw FP32 inputs (staging)
    __nv_bfloat16 *xb = nullptr;   // normalised, padded, BF16
    float *y_all = nullptr;        // outputs of every network [n_nets][bcap][n_out_p]
    float *ystat = nullptr;        // ensemble mean and spread [2][bcap][n_out]
    // activations and gradients of the layer-by-layer passes, networks stacked:
    // network k of a pass at rows k bp; rcap rows in all.  T: transposed copies
    // ([width][bp] per network), the operands of the weight gradients
    size_t rcap = 0, tcap = 0;
    std::vector<__nv_bfloat16 *> a, aT; // NL + 1 (a[0] = input)
    std::vector<float *> z;             // NL pre-activations
    float *y = nullptr, *yt = nullptr, *dyf = nullptr;
    __nv_bfloat16 *dyb = nullptr, *dyT = nullptr;
    __nv_bfloat16 *dz[2] = {nullptr, nullptr}, *dzT[2] = {nullptr, nullptr};
    std::vector<float *> dzf;           // NL (the column sums read them at the end)
    float *loss = nullptr;              // [n_nets]
    float *outw = nullptr;
    float *d_ym = nullptr, *d_ys = nullptr; // output normalisation (n_out)
    float *d_xm = nullptr, *d_xs = nullptr; // input normalisation (n_in)
    int *flags = nullptr;
    int *h_flags = nullptr; // page-locked copy of the flags
    long long adam_t = 0;
    // dataset on the device, its staging and the shuffled orders (kept between calls)
    size_t ds_cap = 0;
    __nv_bfloat16 *dsx = nullptr;
    float *dsy = nullptr, *ds_tmp = nullptr;
    int *d_idx = nullptr;

    ~npsim_surr()
    {
        for (int l = 0; l < kMaxLayers; ++l) {
            dfree2(D.Wb[l]);
            dfree2(D.Wt[l]);
        }
        for (float **p : {&W, &G, &mom, &var, &xin, &y_all, &ystat, &y, &yt, &dyf, &loss, &outw,
                          &d_ym, &d_ys, &d_xm, &d_xs, &dsy, &ds_tmp})
            dfree2(*p);
        for (__nv_bfloat16 **p : {&xb, &dyb, &dyT, &dz[0], &dz[1], &dzT[0], &dzT[1], &dsx})
            dfree2(*p);
        for (auto *v : {&a, &aT})
            for (auto *&p : *v)
                dfree2(p);
        for (auto *v : {&z, &dzf})
            for (auto *&p : *v)
                dfree2(p);
        dfree2(mask);
        dfree2(d_idx);
        dfree2(flags);
        if (h_flags)
            cudaFreeHost(h_flags);
        if (st)
            cudaStreamDestroy(st);
    }
};

namespace {

#define SR_CUDA(call)                                                                   \
    do {                                                                                \
        cudaError_t e_ = (call);                                                        \
        if (e_ != cudaSuccess)                                                          \
            return report_error(e_ == cudaErrorMemoryAllocation ? NPSIM_ERR_OOM         \
                                                                 : NPSIM_ERR_CUDA,      \
                                "%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), \
                                __FILE__, __LINE__);                                    \
    } while (0)

// Rows (networks x minibatch) of a training pass.
constexpr int kTrainRows = 65536;

// Columns per tile: at most 64, the width the epilogue handles two columns per lane
// (an output layer of 80 columns as one tile took 11.1 us, as 48 + 32 8.5, cold
// caches), and at most 32, then 16, while the product still has no more CTAs than
// SMs: a shorter epilogue per CTA, on SMs that had none (4 networks, 256 columns, at
// most 64 / 32 / 16: a minibatch of 256 rows 88 / 77 / 74 us, of 32 81 / 68 / 63).
int n_tile_for(int M, int N, int nz, int sms)
{
    const int mt = (M + 127) / 128 * nz;
    const int most = mt * ((N + 15) / 16) <= sms ? 16 : mt * ((N + 31) / 32) <= sms ? 32 : 64;
    const int tiles = (N + most - 1) / most;
    return ((N + tiles - 1) / tiles + 15) / 16 * 16;
}

// Bound of the GEMM kernel's main-loop waits set by npsim_test_wait_cycles
// (0: the kernel's default).
std::atomic<long long> g_wait_cycles{0};

// A product of nk networks (operand rows za / zb, outputs zc elements apart).
GemmArgs gemm(npsim_surr *s, int mode, const __nv_bfloat16 *A, int lda, int za,
              const __nv_bfloat16 *B, int ldb, int zb, int M, int N, int K, int ldc, size_t zc, int nk)
{
    GemmArgs g{};
    g.A = A;
    g.B = B;
    g.M = M;
    g.N = N;
    g.K = K;
    g.lda = lda;
    g.ldb = ldb;
    g.ldc = ldc;
    g.n_tile = n_tile_for(M, N, nk, s->sms);
    g.tmem_cols = pow2_at_least(g.n_tile);
    g.mode = mode;
    g.flags = s->flags;
    g.wait_cycles = g_wait_cycles.load();
    g.nz = nk;
    g.za = za;
    g.zb = zb;
    g.zc = zc;
    return g;
}

// Buffers of a prediction of bp rows.
int alloc_batch(npsim_surr *s, int bp)
{
    if (bp <= s->bcap)
        return NPSIM_OK;
    s->bcap = 0;
    dfree2(s->xin);
    dfree2(s->xb);
    dfree2(s->y_all);
    dfree2(s->ystat);
    SR_CUDA(dmalloc(&s->xin, (size_t)bp * s->n_in_p));
    SR_CUDA(dmalloc(&s->xb, (size_t)bp * s->n_in_p));
    SR_CUDA(dmalloc(&s->y_all, (size_t)s->n_nets * bp * s->n_out_p));
    SR_CUDA(dmalloc(&s->ystat, (size_t)2 * bp * s->n_out));
    s->bcap = bp;
    return NPSIM_OK;
}

// Buffers of a layer-by-layer pass of `rows` rows (networks x batch), and with
// `train` those of the backward pass.
int alloc_rows(npsim_surr *s, size_t rows, bool train)
{
    if (rows > s->rcap) {
        s->rcap = 0;
        s->a.resize(s->NL + 1, nullptr);
        s->z.resize(s->NL, nullptr);
        for (auto *&p : s->a)
            dfree2(p);
        for (auto *&p : s->z)
            dfree2(p);
        dfree2(s->y);
        SR_CUDA(dmalloc(&s->a[0], rows * s->n_in_p));
        for (int l = 0; l < s->NL; ++l) {
            SR_CUDA(dmalloc(&s->a[l + 1], rows * s->H));
            SR_CUDA(dmalloc(&s->z[l], rows * s->H));
        }
        SR_CUDA(dmalloc(&s->y, rows * s->n_out_p));
        s->rcap = rows;
    }
    if (train && rows > s->tcap) {
        s->tcap = 0;
        s->aT.resize(s->NL + 1, nullptr);
        s->dzf.resize(s->NL, nullptr);
        for (auto *&p : s->aT)
            dfree2(p);
        for (auto *&p : s->dzf)
            dfree2(p);
        for (float **p : {&s->yt, &s->dyf})
            dfree2(*p);
        for (__nv_bfloat16 **p : {&s->dyb, &s->dyT, &s->dz[0], &s->dz[1], &s->dzT[0], &s->dzT[1]})
            dfree2(*p);
        SR_CUDA(dmalloc(&s->aT[0], rows * s->n_in_p));
        for (int l = 0; l < s->NL; ++l) {
            SR_CUDA(dmalloc(&s->aT[l + 1], rows * s->H));
            SR_CUDA(dmalloc(&s->dzf[l], rows * s->H));
        }
        SR_CUDA(dmalloc(&s->yt, rows * s->n_out_p));
        SR_CUDA(dmalloc(&s->dyf, rows * s->n_out_p));
        SR_CUDA(dmalloc(&s->dyb, rows * s->n_out_p));
        SR_CUDA(dmalloc(&s->dyT, rows * s->n_out_p));
        for (int k = 0; k < 2; ++k) {
            SR_CUDA(dmalloc(&s->dz[k], rows * s->H));
            SR_CUDA(dmalloc(&s->dzT[k], rows * s->H));
        }
        s->tcap = rows;
    }
    return NPSIM_OK;
}

// Forward pass of networks k0 .. k0 + nk - 1 on bp rows each (a multiple of 128),
// the inputs at x (network k's xz rows further): hidden layers write z (FP32) and a
// (BF16; with `train` its transpose too), the output layer writes y_out (FP32).
int forward(npsim_surr *s, int k0, int nk, int bp, const __nv_bfloat16 *x, int xz, float *y_out,
            bool train)
{
    const NetDims &D = s->D;
    for (int l = 0; l <= s->NL; ++l) {
        const int N = D.out_p[l], K = D.in_p[l];
        const bool out = l == s->NL;
        GemmArgs g = gemm(s, out ? GEMM_F32 : GEMM_ACT, l == 0 ? x : s->a[l], K, l == 0 ? xz : bp,
                          D.Wb[l] + (size_t)k0 * N * K, K, N, bp, N, K, N, (size_t)bp * N, nk);
        g.bias = s->W + (size_t)k0 * D.n_params + D.off[l] + N * K;
        g.zbias = (size_t)D.n_params;
        if (out) {
            g.Cf = y_out;
        } else {
            g.act = 1;
            g.Z = s->z[l];
            g.Cb = s->a[l + 1];
            if (train) {
                g.CbT = s->aT[l + 1];
                g.ldt = bp;
                g.zt = (size_t)bp * N;
            }
        }
        SR_CUDA(launch_gemm(g, nullptr, s->st));
    }
    return NPSIM_OK;
}

// Back-propagation of the mean-squared error on rows < m_valid of the batch for
// networks k0 .. k0 + nk - 1: weight gradients gW = dZ^T A_prev (from the
// transposed copies the producing kernels wrote), dZ_prev = (dZ W) * SiLU'(Z_prev)
// beside it in the same launch, bias gradients = column sums of every dZ at the
// end.  loss[0 .. nk) must be zero.
int backward(npsim_surr *s, int k0, int nk, int bp, int m_valid)
{
    const NetDims &D = s->D;
    SR_CUDA(launch_mse_grad(s->y, s->yt, s->outw, bp, m_valid, s->n_out, s->n_out_p, nk, s->dyf,
                            s->dyb, s->dyT, s->loss, s->st));
    // current gradient wrt the pre-activation of layer l, and its transpose
    const __nv_bfloat16 *d = s->dyb, *dT = s->dyT;
    ColsumArgs cs{};
    cs.M = bp;
    cs.nz = nk;
    cs.G[s->NL] = s->dyf;
    int ping = 0;
    for (int l = s->NL; l >= 0; --l) {
        const int N = D.out_p[l], K = D.in_p[l];
        // gW (N x K) = dZ^T (N x bp) * (A_prev^T (K x bp))^T
        GemmArgs gw = gemm(s, GEMM_F32, dT, bp, N, s->aT[l], bp, K, N, K, bp, K,
                           (size_t)D.n_params, nk);
        gw.Cf = s->G + (size_t)k0 * D.n_params + D.off[l];
        if (l == 0) {
            SR_CUDA(launch_gemm(gw, nullptr, s->st));
            break;
        }
        // dZ_prev (bp x K) = dZ (bp x N) * (W^T (K x N))^T
        GemmArgs gx = gemm(s, GEMM_DACT, d, N, bp, D.Wt[l] + (size_t)k0 * N * K, N, K, bp, K, N, K,
                           (size_t)bp * K, nk);
        gx.Z = s->z[l - 1];
        gx.Cf = s->dzf[l - 1];
        gx.Cb = s->dz[ping];
        gx.CbT = s->dzT[ping];
        gx.ldt = bp;
        gx.zt = (size_t)bp * K;
        SR_CUDA(launch_gemm(gx, &gw, s->st));
        cs.G[l - 1] = s->dzf[l - 1];
        d = s->dz[ping];
        dT = s->dzT[ping];
        ping ^= 1;
    }
    SR_CUDA(launch_colsum(cs, D, s->G + (size_t)k0 * D.n_params, s->st));
    return NPSIM_OK;
}

int adamw_step(npsim_surr *s, int k0, int nk, float lr, float wd)
{
    AdamArgs a{};
    a.lr = lr;
    a.b1 = 0.9f;
    a.b2 = 0.999f;
    a.eps = 1e-8f;
    a.wd = wd;
    const double t = (double)s->adam_t;
    a.bc1 = (float)(1.0 - std::pow(0.9, t));
    a.bc2 = (float)(1.0 - std::pow(0.999, t));
    SR_CUDA(launch_adamw(s->W, s->G, s->mom, s->var, s->mask, s->D, k0, nk, a, s->st));
    return NPSIM_OK;
}

// (v - mean) / std of rows x n raw values, padded with zeros to rows_p x n_p, as
// BF16 (ob) or FP32 (of).
__global__ void k_normalise(const float *__restrict__ v, int rows, int n, int rows_p, int n_p,
                            const float *__restrict__ mean, const float *__restrict__ std,
                            __nv_bfloat16 *__restrict__ ob, float *__restrict__ of)
{
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (size_t)rows_p * n_p)
        return;
    const int r = (int)(e / n_p), c = (int)(e - (size_t)r * n_p);
    const float q =
        r < rows && c < n ? __fdiv_rn(__fsub_rn(v[(size_t)r * n + c], mean[c]), std[c]) : 0.f;
    if (ob)
        ob[e] = __float2bfloat16_rn(q);
    else
        of[e] = q;
}

// Raw host rows to the device (staged in raw) and normalised there.
int upload_rows(npsim_surr *s, const float *v, int rows, int n, int rows_p, int n_p, float *raw,
                const float *mean, const float *std, __nv_bfloat16 *ob, float *of)
{
    SR_CUDA(cudaMemcpyAsync(raw, v, sizeof(float) * (size_t)rows * n, cudaMemcpyHostToDevice, s->st));
    const size_t e = (size_t)rows_p * n_p;
    k_normalise<<<(unsigned)((e + 255) / 256), 256, 0, s->st>>>(raw, rows, n, rows_p, n_p, mean, std,
                                                                ob, of);
    SR_CUDA(cudaGetLastError());
    return NPSIM_OK;
}

// The error flags behind everything queued so far: copied with the call's last
// copies, looked at after the stream has been waited for.
cudaError_t fetch_flags(npsim_surr *s)
{
    return cudaMemcpyAsync(s->h_flags, s->flags, sizeof(int), cudaMemcpyDeviceToHost, s->st);
}

int flags_status(npsim_surr *s)
{
    const int h = *s->h_flags;
    if (h) {
        SR_CUDA(cudaMemsetAsync(s->flags, 0, sizeof(int), s->st));
        return report_error(NPSIM_ERR_TIMEOUT, "a tensor-core wait expired (flags 0x%x)", h);
    }
    return NPSIM_OK;
}

int check_flags(npsim_surr *s)
{
    SR_CUDA(fetch_flags(s));
    SR_CUDA(cudaStreamSynchronize(s->st));
    return flags_status(s);
}

// One minibatch of every network of a group: rows idx[0 .. rows) of network
// blockIdx.y (its indices idx_ld further) into x, its transpose and y; rows beyond
// are zero.  Clears the networks' losses.
__global__ void k_gather_rows(const __nv_bfloat16 *__restrict__ sx, const float *__restrict__ sy,
                              const int *__restrict__ idx, int idx_ld, int rows, int bp, int nx,
                              int ny, __nv_bfloat16 *__restrict__ x,
                              __nv_bfloat16 *__restrict__ xT, float *__restrict__ y,
                              float *__restrict__ loss)
{
    const int r = blockIdx.x, k = (int)blockIdx.y + after_previous();
    const size_t row = (size_t)k * bp + r;
    const bool ok = r < rows;
    const int src = ok ? idx[(size_t)k * idx_ld + r] : 0;
    if (r == 0 && threadIdx.x == 0)
        loss[k] = 0.f;
    for (int c = threadIdx.x; c < nx; c += blockDim.x) {
        const __nv_bfloat16 v = ok ? sx[(size_t)src * nx + c] : __float2bfloat16_rn(0.f);
        x[row * nx + c] = v;
        xT[((size_t)k * nx + c) * bp + r] = v;
    }
    for (int c = threadIdx.x; c < ny; c += blockDim.x)
        y[row * ny + c] = ok ? sy[(size_t)src * ny + c] : 0.f;
}

// float(sqrt(x)) for x >= 0 without the float64 square root: the float32 root r of x,
// corrected by the float64 residual x - r^2 (exact to 2^-53 of x): r + e / (2 r) is
// within 2^-47 of the root before its one rounding.  Values whose float32 image is not
// an ordinary number take the float64 root.
__device__ __forceinline__ float sqrt_to_float(double x)
{
    const float xf = (float)x;
    if (!(xf > 1e-30f && xf < 1e30f))
        return (float)sqrt(x);
    const float r = sqrtf(xf);
    const float e = (float)fma(-(double)r, (double)r, x);
    return fmaf(e, 0.5f / r, r);
}

// Mean and spread (population standard deviation) over the networks of the
// de-normalised outputs y * ys + ym, for rows < B and the n_out valid columns, in
// float64.  inv: 1 / n_nets where that is exact (a power of two), else 0.  The float64
// unit bounds it: two divisions and a square root were three quarters of its
// operations (4096 x 65 outputs of 4 networks: 27 us, now 18.6).
__global__ void k_ens_stats(const float *__restrict__ y_all, int n_nets, double inv, int bp, int ldy,
                            int B, int n_out, const float *__restrict__ ym,
                            const float *__restrict__ ys, float *__restrict__ mean,
                            float *__restrict__ spread)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x + after_previous();
    if (idx >= B * n_out)
        return;
    const int r = idx / n_out, c = idx - r * n_out;
    const double sc = ys[c], of = ym[c];
    double s1 = 0.0, s2 = 0.0;
    for (int k = 0; k < n_nets; ++k) {
        const double v = (double)y_all[((size_t)k * bp + r) * ldy + c] * sc + of;
        s1 += v;
        s2 += v * v;
    }
    const double m = inv != 0.0 ? __dmul_rn(s1, inv) : s1 / n_nets;
    const double q = inv != 0.0 ? __dmul_rn(s2, inv) : s2 / n_nets;
    mean[idx] = (float)m;
    spread[idx] = sqrt_to_float(fmax(0.0, q - m * m));
}

} // namespace

extern "C" {

int npsim_surr_create(int32_t n_in, int32_t n_hidden, int32_t n_layers, int32_t n_out,
                      int32_t n_nets, uint64_t seed, npsim_surr_t *out)
{
    NP_TRACE();
    if (!out)
        return report_error(NPSIM_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (n_in < 1 || n_in > 64 || n_hidden < 16 || n_hidden > 256 || n_hidden % 16 ||
        n_layers < 1 || n_layers > 8 || n_out < 1 || n_out > 256 || n_nets < 1 || n_nets > 64)
        return report_error(NPSIM_ERR_INVALID_ARG,
                            "surrogate shape out of range (n_in <= 64, hidden 16..256 step 16, "
                            "1..8 layers, n_out <= 256, 1..64 nets)");
    int count = 0;
    if (cudaGetDeviceCount(&count) != cudaSuccess || count < 1)
        return report_error(NPSIM_ERR_NO_DEVICE, "no CUDA device visible");
    npsim_surr *s = new npsim_surr();
    auto bail = [&](int rc) {
        delete s;
        return rc;
    };
    s->n_in = n_in;
    s->n_in_p = round16(n_in);
    s->H = n_hidden;
    s->NL = n_layers;
    s->n_out = n_out;
    s->n_out_p = round16(n_out);
    s->n_nets = n_nets;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&s->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return bail(report_error(NPSIM_ERR_CUDA, "no SM count"));
    s->xm.assign(n_in, 0.f);
    s->xs.assign(n_in, 1.f);
    s->ym.assign(n_out, 0.f);
    s->ys.assign(n_out, 1.f);
    if (cudaStreamCreateWithFlags(&s->st, cudaStreamNonBlocking) != cudaSuccess)
        return bail(report_error(NPSIM_ERR_CUDA, "stream create failed"));
    NetDims &D = s->D;
    D.n_layers = n_layers + 1;
    std::vector<unsigned char> mask;
    for (int l = 0; l <= n_layers; ++l) {
        const int in = l == 0 ? n_in : n_hidden, out = l == n_layers ? n_out : n_hidden;
        D.in_p[l] = l == 0 ? s->n_in_p : n_hidden;
        D.out_p[l] = l == n_layers ? s->n_out_p : n_hidden;
        D.off[l] = (int)mask.size();
        for (int r = 0; r < D.out_p[l]; ++r)
            for (int c = 0; c < D.in_p[l]; ++c)
                mask.push_back(r < out && c < in ? 3 : 0);
        for (int r = 0; r < D.out_p[l]; ++r)
            mask.push_back(r < out ? 1 : 0);
        const size_t nw = (size_t)n_nets * D.out_p[l] * D.in_p[l];
        if (dmalloc(&D.Wb[l], nw) != cudaSuccess || dmalloc(&D.Wt[l], nw) != cudaSuccess)
            return bail(report_error(NPSIM_ERR_OOM, "surrogate weights"));
    }
    D.n_params = (int)mask.size();
    const size_t np = (size_t)n_nets * D.n_params;
    if (dmalloc(&s->W, np) != cudaSuccess || dmalloc(&s->G, np) != cudaSuccess ||
        dmalloc(&s->mom, np) != cudaSuccess || dmalloc(&s->var, np) != cudaSuccess ||
        dmalloc(&s->mask, mask.size()) != cudaSuccess)
        return bail(report_error(NPSIM_ERR_OOM, "surrogate weights"));
    // He-uniform initialisation on the valid block, zero padding and biases
    std::mt19937_64 rng(seed);
    std::vector<float> w(np, 0.f);
    for (int k = 0; k < n_nets; ++k)
        for (int l = 0; l <= n_layers; ++l) {
            const int in = l == 0 ? n_in : n_hidden, out = l == n_layers ? n_out : n_hidden;
            const float lim = std::sqrt(6.0f / (float)in);
            std::uniform_real_distribution<float> U(-lim, lim);
            float *wl = w.data() + (size_t)k * D.n_params + D.off[l];
            for (int r = 0; r < out; ++r)
                for (int c = 0; c < in; ++c)
                    wl[(size_t)r * D.in_p[l] + c] = U(rng);
        }
    cudaError_t ce = cudaMemcpy(s->W, w.data(), sizeof(float) * np, cudaMemcpyHostToDevice);
    for (float *q : {s->G, s->mom, s->var})
        if (ce == cudaSuccess)
            ce = cudaMemset(q, 0, sizeof(float) * np);
    if (ce == cudaSuccess)
        ce = cudaMemcpy(s->mask, mask.data(), mask.size(), cudaMemcpyHostToDevice);
    for (int k = 0; k < n_nets && ce == cudaSuccess; ++k)
        ce = launch_weights_bf16(s->W, D, k, s->st);
    if (ce != cudaSuccess)
        return bail(report_error(NPSIM_ERR_CUDA, "surrogate weights: %s", cudaGetErrorString(ce)));
    if (dmalloc(&s->loss, (size_t)n_nets) != cudaSuccess || dmalloc(&s->flags, 1) != cudaSuccess ||
        dmalloc(&s->outw, (size_t)s->n_out_p) != cudaSuccess ||
        dmalloc(&s->d_ym, (size_t)n_out) != cudaSuccess ||
        dmalloc(&s->d_ys, (size_t)n_out) != cudaSuccess ||
        dmalloc(&s->d_xm, (size_t)n_in) != cudaSuccess ||
        dmalloc(&s->d_xs, (size_t)n_in) != cudaSuccess ||
        cudaHostAlloc((void **)&s->h_flags, sizeof(int), cudaHostAllocDefault) != cudaSuccess)
        return bail(report_error(NPSIM_ERR_OOM, "surrogate scratch"));
    cudaMemcpy(s->d_ym, s->ym.data(), sizeof(float) * n_out, cudaMemcpyHostToDevice);
    cudaMemcpy(s->d_ys, s->ys.data(), sizeof(float) * n_out, cudaMemcpyHostToDevice);
    cudaMemcpy(s->d_xm, s->xm.data(), sizeof(float) * n_in, cudaMemcpyHostToDevice);
    cudaMemcpy(s->d_xs, s->xs.data(), sizeof(float) * n_in, cudaMemcpyHostToDevice);
    std::vector<float> ow(s->n_out_p, 0.f);
    for (int c = 0; c < n_out; ++c)
        ow[c] = 1.f;
    cudaMemcpy(s->outw, ow.data(), sizeof(float) * ow.size(), cudaMemcpyHostToDevice);
    cudaMemsetAsync(s->flags, 0, sizeof(int), s->st);
    int rc = alloc_batch(s, 512);
    if (rc)
        return bail(rc);
    if (cudaStreamSynchronize(s->st) != cudaSuccess)
        return bail(report_error(NPSIM_ERR_CUDA, "surrogate init failed"));
    *out = s;
    return NPSIM_OK;
}

void npsim_surr_destroy(npsim_surr_t s)
{
    if (!s)
        return;
    cudaStreamSynchronize(s->st);
    delete s;
}

int npsim_surr_set_norm(npsim_surr_t s, const float *x_mean, const float *x_std,
                        const float *y_mean, const float *y_std)
{
    if (!s)
        return report_error(NPSIM_ERR_INVALID_ARG, "surrogate is NULL");
    for (int c = 0; c < s->n_in; ++c) {
        s->xm[c] = x_mean ? x_mean[c] : 0.f;
        s->xs[c] = x_std ? x_std[c] : 1.f;
        if (!(s->xs[c] > 0.f))
            return report_error(NPSIM_ERR_INVALID_ARG, "x_std[%d] must be positive", c);
    }
    for (int c = 0; c < s->n_out; ++c) {
        s->ym[c] = y_mean ? y_mean[c] : 0.f;
        s->ys[c] = y_std ? y_std[c] : 1.f;
        if (!(s->ys[c] > 0.f))
            return report_error(NPSIM_ERR_INVALID_ARG, "y_std[%d] must be positive", c);
    }
    SR_CUDA(cudaMemcpyAsync(s->d_ym, s->ym.data(), sizeof(float) * s->n_out,
                            cudaMemcpyHostToDevice, s->st));
    SR_CUDA(cudaMemcpyAsync(s->d_ys, s->ys.data(), sizeof(float) * s->n_out,
                            cudaMemcpyHostToDevice, s->st));
    SR_CUDA(cudaMemcpyAsync(s->d_xm, s->xm.data(), sizeof(float) * s->n_in,
                            cudaMemcpyHostToDevice, s->st));
    SR_CUDA(cudaMemcpyAsync(s->d_xs, s->xs.data(), sizeof(float) * s->n_in,
                            cudaMemcpyHostToDevice, s->st));
    SR_CUDA(cudaStreamSynchronize(s->st));
    return NPSIM_OK;
}

int npsim_surr_param_count(npsim_surr_t s, int64_t *count)
{
    if (!s || !count)
        return report_error(NPSIM_ERR_INVALID_ARG, "surrogate and count are required");
    *count = s->D.n_params;
    return NPSIM_OK;
}

int npsim_surr_get_params(npsim_surr_t s, int32_t net, float *flat, float *grads)
{
    if (!s || net < 0 || net >= s->n_nets)
        return report_error(NPSIM_ERR_INVALID_ARG, "bad surrogate or net index");
    SR_CUDA(cudaStreamSynchronize(s->st));
    const size_t np = (size_t)s->D.n_params, off = (size_t)net * np;
    if (flat)
        SR_CUDA(cudaMemcpy(flat, s->W + off, sizeof(float) * np, cudaMemcpyDeviceToHost));
    if (grads)
        SR_CUDA(cudaMemcpy(grads, s->G + off, sizeof(float) * np, cudaMemcpyDeviceToHost));
    return NPSIM_OK;
}

int npsim_surr_set_params(npsim_surr_t s, int32_t net, const float *flat)
{
    if (!s || !flat || net < 0 || net >= s->n_nets)
        return report_error(NPSIM_ERR_INVALID_ARG, "bad surrogate, net index or params");
    const size_t np = (size_t)s->D.n_params;
    SR_CUDA(cudaMemcpy(s->W + (size_t)net * np, flat, sizeof(float) * np, cudaMemcpyHostToDevice));
    SR_CUDA(launch_weights_bf16(s->W, s->D, net, s->st));
    SR_CUDA(cudaStreamSynchronize(s->st));
    return NPSIM_OK;
}

int npsim_surr_grads(npsim_surr_t s, int32_t net, const float *X, const float *Y, int32_t B,
                     float *grads, float *loss, float *Yhat)
{
    if (!s || !X || !Y || B < 1 || net < 0 || net >= s->n_nets)
        return report_error(NPSIM_ERR_INVALID_ARG, "bad surrogate, net, inputs or batch");
    const int bp = (B + 127) / 128 * 128;
    int rc = alloc_batch(s, bp);
    if (!rc)
        rc = alloc_rows(s, (size_t)bp, true);
    if (!rc)
        rc = upload_rows(s, X, B, s->n_in, bp, s->n_in_p, s->xin, s->d_xm, s->d_xs, s->xb, nullptr);
    if (!rc) // the targets' raw rows pass through the gradient buffer
        rc = upload_rows(s, Y, B, s->n_out, bp, s->n_out_p, s->dyf, s->d_ym, s->d_ys, nullptr, s->yt);
    if (rc)
        return rc;
    SR_CUDA(launch_transpose_bf16(s->xb, bp, s->n_in_p, s->n_in_p, s->aT[0], bp, s->st));
    SR_CUDA(cudaMemsetAsync(s->loss, 0, sizeof(float), s->st));
    rc = forward(s, net, 1, bp, s->xb, 0, s->y, true);
    if (!rc)
        rc = backward(s, net, 1, bp, B);
    if (rc)
        return rc;
    rc = check_flags(s);
    if (rc)
        return rc;
    if (loss)
        SR_CUDA(cudaMemcpy(loss, s->loss, sizeof(float), cudaMemcpyDeviceToHost));
    if (Yhat) {
        std::vector<float> yy((size_t)bp * s->n_out_p);
        SR_CUDA(cudaMemcpy(yy.data(), s->y, sizeof(float) * yy.size(), cudaMemcpyDeviceToHost));
        for (int r = 0; r < B; ++r)
            for (int c = 0; c < s->n_out; ++c)
                Yhat[(size_t)r * s->n_out + c] = yy[(size_t)r * s->n_out_p + c];
    }
    return npsim_surr_get_params(s, net, nullptr, grads);
}

int npsim_surr_train(npsim_surr_t s, const float *X, const float *Y, int32_t n_samples,
                     int32_t epochs, int32_t batch, float lr, float wd, uint64_t shuffle_seed,
                     float *final_loss)
{
    NP_TRACE();
    if (!s || !X || !Y || n_samples < 1 || epochs < 0 || batch < 1 || batch > 8192)
        return report_error(NPSIM_ERR_INVALID_ARG, "bad training arguments");
    const int bp = (batch + 127) / 128 * 128;
    // networks trained side by side: all of them, while their minibatches stay
    // below kTrainRows rows (their activations and gradients are kept together)
    const int group = std::max(1, std::min(s->n_nets, kTrainRows / bp));
    int rc = alloc_rows(s, (size_t)group * bp, true);
    if (rc)
        return rc;
    // dataset on the device, normalised and padded
    if ((size_t)n_samples > s->ds_cap) {
        s->ds_cap = 0;
        dfree2(s->dsx);
        dfree2(s->dsy);
        dfree2(s->ds_tmp);
        dfree2(s->d_idx);
        SR_CUDA(dmalloc(&s->dsx, (size_t)n_samples * s->n_in_p));
        SR_CUDA(dmalloc(&s->ds_tmp, (size_t)n_samples * std::max(s->n_in, s->n_out)));
        SR_CUDA(dmalloc(&s->dsy, (size_t)n_samples * s->n_out_p));
        SR_CUDA(dmalloc(&s->d_idx, (size_t)n_samples * s->n_nets));
        s->ds_cap = (size_t)n_samples;
    }
    rc = upload_rows(s, X, n_samples, s->n_in, n_samples, s->n_in_p, s->ds_tmp, s->d_xm, s->d_xs,
                     s->dsx, nullptr);
    if (!rc)
        rc = upload_rows(s, Y, n_samples, s->n_out, n_samples, s->n_out_p, s->ds_tmp, s->d_ym,
                         s->d_ys, nullptr, s->dsy);
    if (rc)
        return rc;
    // every network's shuffled order of an epoch, drawn network by network; the next
    // epoch's is drawn while this one runs
    std::vector<int> order[2];
    order[0].resize((size_t)s->n_nets * n_samples);
    order[1].resize(epochs > 1 ? order[0].size() : 0);
    std::mt19937_64 rng(shuffle_seed);
    auto shuffle = [&](std::vector<int> &ord) {
        for (int k = 0; k < s->n_nets; ++k) {
            int *o = ord.data() + (size_t)k * n_samples;
            for (int i = 0; i < n_samples; ++i)
                o[i] = i;
            std::shuffle(o, o + n_samples, rng);
        }
    };
    int *d_idx = s->d_idx;
    const int nb = (n_samples + batch - 1) / batch;
    float last = 0.f;
    cudaError_t e = cudaSuccess;
    if (epochs > 0)
        shuffle(order[0]);
    for (int ep = 0; ep < epochs && !rc && e == cudaSuccess; ++ep) {
        e = cudaMemcpyAsync(d_idx, order[ep & 1].data(), sizeof(int) * order[0].size(),
                            cudaMemcpyHostToDevice, s->st);
        int kl = 0; // first network of the group that ran last
        for (int b = 0; b < nb && !rc && e == cudaSuccess; ++b) {
            const int r0 = b * batch, rows = std::min(batch, n_samples - r0);
            ++s->adam_t;
            for (int k0 = 0; k0 < s->n_nets && !rc && e == cudaSuccess; k0 += group) {
                const int nk = std::min(group, s->n_nets - k0);
                kl = k0;
                e = launch_after(k_gather_rows, dim3(bp, nk), 96, 0, s->st, s->dsx, s->dsy,
                                 d_idx + (size_t)k0 * n_samples + r0, n_samples, rows, bp,
                                 s->n_in_p, s->n_out_p, s->a[0], s->aT[0], s->yt, s->loss);
                if (e == cudaSuccess)
                    rc = forward(s, k0, nk, bp, s->a[0], bp, s->y, true);
                if (!rc && e == cudaSuccess)
                    rc = backward(s, k0, nk, bp, rows);
                if (!rc && e == cudaSuccess)
                    rc = adamw_step(s, k0, nk, lr, wd);
            }
        }
        if (!rc && e == cudaSuccess && ep + 1 < epochs)
            shuffle(order[(ep + 1) & 1]);
        if (!rc && e == cudaSuccess)
            rc = check_flags(s); // waits for the epoch
        if (!rc && e == cudaSuccess && ep + 1 == epochs)
            e = cudaMemcpy(&last, s->loss + (s->n_nets - 1 - kl), sizeof(float),
                           cudaMemcpyDeviceToHost);
    }
    if (rc)
        return rc;
    if (e == cudaSuccess && epochs == 0)
        e = cudaStreamSynchronize(s->st); // X and Y are the caller's again
    if (e != cudaSuccess)
        return report_error(NPSIM_ERR_CUDA, "training: %s", cudaGetErrorString(e));
    if (final_loss)
        *final_loss = last;
    return NPSIM_OK;
}

int npsim_surr_predict(npsim_surr_t s, const float *X, int32_t B, float *Y_mean, float *Y_spread)
{
    NP_TRACE();
    if (!s || !X || !Y_mean || B < 1 || B > 65536)
        return report_error(NPSIM_ERR_INVALID_ARG, "bad prediction arguments");
    const int bp = (B + 127) / 128 * 128;
    int rc = alloc_batch(s, bp);
    if (rc)
        return rc;
    rc = upload_rows(s, X, B, s->n_in, bp, s->n_in_p, s->xin, s->d_xm, s->d_xs, s->xb, nullptr);
    if (rc)
        return rc;
    // NPSIM_SURR_LAYERED selects the layer-by-layer GEMM path (same arithmetic)
    const bool layered = getenv("NPSIM_SURR_LAYERED") != nullptr;
    if (!layered && mlp_infer_supported(s->NL, s->n_in_p, s->H, s->n_out_p)) {
        // every layer of every network in one launch
        MlpInferArgs f{};
        f.X = s->xb;
        for (int l = 0; l <= s->NL; ++l) {
            f.W[l] = s->D.Wb[l];
            f.b[l] = s->W + s->D.off[l] + s->D.out_p[l] * s->D.in_p[l];
        }
        f.b_stride = s->D.n_params;
        f.NL = s->NL;
        f.in_p = s->n_in_p;
        f.H = s->H;
        f.out_p = s->n_out_p;
        f.bp = bp;
        f.n_nets = s->n_nets;
        f.y = s->y_all;
        f.flags = s->flags;
        SR_CUDA(launch_mlp_infer(f, s->st));
    } else {
        rc = alloc_rows(s, (size_t)bp, false);
        for (int k = 0; k < s->n_nets && !rc; ++k)
            rc = forward(s, k, 1, bp, s->xb, 0, s->y_all + (size_t)k * bp * s->n_out_p, false);
        if (rc)
            return rc;
    }
    float *d_mean = s->ystat, *d_spread = s->ystat + (size_t)B * s->n_out;
    const int ne = B * s->n_out;
    const double inv = (s->n_nets & (s->n_nets - 1)) == 0 ? 1.0 / s->n_nets : 0.0;
    SR_CUDA(launch_after(k_ens_stats, dim3((ne + 255) / 256), 256, 0, s->st, s->y_all, s->n_nets, inv, bp,
                         s->n_out_p, B, s->n_out, s->d_ym, s->d_ys, d_mean, d_spread));
    SR_CUDA(fetch_flags(s));
    cudaError_t joined = cudaErrorInvalidValue;
    if (Y_spread == Y_mean + ne) // back to back on the host too: one copy
        joined = copy_joined(Y_mean, d_mean, sizeof(float) * 2 * (size_t)ne, s->st);
    if (joined != cudaErrorInvalidValue) {
        SR_CUDA(joined);
    } else {
        SR_CUDA(cudaMemcpyAsync(Y_mean, d_mean, sizeof(float) * ne, cudaMemcpyDeviceToHost, s->st));
        if (Y_spread)
            SR_CUDA(cudaMemcpyAsync(Y_spread, d_spread, sizeof(float) * ne, cudaMemcpyDeviceToHost,
                                    s->st));
    }
    SR_CUDA(cudaStreamSynchronize(s->st));
    return flags_status(s);
}

int npsim_test_wait_cycles(int64_t cycles)
{
    if (cycles < 0)
        return report_error(NPSIM_ERR_INVALID_ARG, "cycles must be >= 0");
    g_wait_cycles.store((long long)cycles);
    return NPSIM_OK;
}

// Test hook: C = A B^T for host BF16 matrices (bit patterns), C in FP32.
int npsim_gemm_bf16(const uint16_t *A, const uint16_t *B, int32_t M, int32_t N, int32_t K,
                    int32_t n_tile, float *C)
{
    NP_TRACE();
    if (!A || !B || !C || M < 1 || N < 16 || K < 16 || N % 16 || K % 16 || n_tile % 16 ||
        n_tile < 16 || n_tile > 256)
        return report_error(NPSIM_ERR_INVALID_ARG, "gemm shape: N, K, n_tile multiples of 16");
    __nv_bfloat16 *dA = nullptr, *dB = nullptr;
    float *dC = nullptr;
    int *dflag = nullptr;
    SR_CUDA(dmalloc(&dA, (size_t)M * K));
    SR_CUDA(dmalloc(&dB, (size_t)N * K));
    SR_CUDA(dmalloc(&dC, (size_t)M * N));
    SR_CUDA(dmalloc(&dflag, 1));
    SR_CUDA(cudaMemcpy(dA, A, sizeof(uint16_t) * (size_t)M * K, cudaMemcpyHostToDevice));
    SR_CUDA(cudaMemcpy(dB, B, sizeof(uint16_t) * (size_t)N * K, cudaMemcpyHostToDevice));
    SR_CUDA(cudaMemset(dflag, 0, sizeof(int)));
    GemmArgs g{};
    g.A = dA;
    g.B = dB;
    g.M = M;
    g.N = N;
    g.K = K;
    g.lda = K;
    g.ldb = K;
    g.ldc = N;
    g.n_tile = n_tile;
    g.tmem_cols = pow2_at_least(n_tile);
    g.mode = GEMM_F32;
    g.Cf = dC;
    g.flags = dflag;
    g.wait_cycles = g_wait_cycles.load();
    g.nz = 1;
    cudaError_t e = launch_gemm(g, nullptr, 0);
    if (e == cudaSuccess)
        e = cudaDeviceSynchronize();
    int flag = 0;
    if (e == cudaSuccess)
        e = cudaMemcpy(&flag, dflag, sizeof(int), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess)
        e = cudaMemcpy(C, dC, sizeof(float) * (size_t)M * N, cudaMemcpyDeviceToHost);
    cudaFree(dA);
    cudaFree(dB);
    cudaFree(dC);
    cudaFree(dflag);
    if (e != cudaSuccess)
        return report_error(NPSIM_ERR_CUDA, "gemm: %s", cudaGetErrorString(e));
    if (flag)
        return report_error(NPSIM_ERR_TIMEOUT, "gemm: a tensor-core wait expired");
    return NPSIM_OK;
}

} // extern "C"
