// Learned warm start: a coordinate MLP 4 -> 256 -> 256 -> 256 -> 6 (exact-erf GELU) that
// maps (x, y, log Kn, u_w) to the six normalised moments of the steady state, trained
// and evaluated on the fifth-generation tensor cores in BF16 with FP32 accumulation.  A
// training step is three launches: the row-local chain (forward pass, loss, input gradients;
// mlp_chain.cu), the weight gradients, and their reduction with Adam on FP32 master weights
// (mlp_grad.cu); a forward pass is the chain alone.  As one launch per product, activation,
// transposition, column sum and array update a training step of 8192 rows took 390 us.  The
// warm-start kernel then builds the initial distribution
// from the predicted moments by the second-order Hermite expansion
//   h_a = w_a [rho' + xi_a . j' + 1/2 sum_ij (P'_ij - rho' delta_ij)(xi_i xi_j - delta_ij)].
// The paper has no learned component; this follows the warm-start configuration of
// the project's workloads.
#include <cuda_bf16.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "../../include/lbm.h"
#include "hermite_state.cuh"
#include "lbm_internal.h"
#include "mlp_internal.h"
#include "umma.cuh"

lbm_status lbm_norms_fail(lbm_status s, const char *msg);

using namespace mlpk;

namespace {

// both BF16 copies of a layer's weights W [N][K]: q [N][ldq] and its transpose qt [K][ldt]
__global__ void refresh_kernel(const float *W, int n, int k, __nv_bfloat16 *q, int ldq, __nv_bfloat16 *qt, int ldt)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n * k; i += gridDim.x * blockDim.x) {
        const __nv_bfloat16 v = __float2bfloat16_rn(W[i]);
        q[(i / k) * ldq + i % k] = v;
        qt[(i % k) * ldt + i / k] = v;
    }
}

// features of cell c of an nx x ny cavity: (2x-1, 2y-1, (2 log10 Kn + 1)/3, (u_w - 0.0125)/0.0075)
__global__ void features_kernel(int nx, int ny, float f2, float f3, float *x)
{
    const long n = (long)nx * ny;
    for (long c = (long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long)gridDim.x * blockDim.x) {
        const int yy = (int)(c / nx), xx = (int)(c - (long)yy * nx);
        x[c * 4 + 0] = 2.f * ((xx + 0.5f) / nx) - 1.f;
        x[c * 4 + 1] = 2.f * ((yy + 0.5f) / ny) - 1.f;
        x[c * 4 + 2] = f2;
        x[c * 4 + 3] = f3;
    }
}

// state from normalised predicted moments
// pred[c][0..5] = ((rho-1)/u_w, u_x/u_w, u_y/u_w, (P_xx-1)/u_w, P_xy/u_w, (P_yy-1)/u_w)
template <typename T>
__global__ void warm_state_kernel(const float *pred, int nx, int ny, long pa, long py, int m, const double *xi1,
                                  const double *w1, double uw_over_uref, T *h, bool tiled32)
{
    __shared__ double c[LBM_MAX_M][3];
    hermite::row_table(c, xi1, w1, m);
    const int iy = threadIdx.x >> 5;
    const long cell = (long)blockIdx.x * 32 + (threadIdx.x & 31);
    if (cell >= (long)nx * ny) return;
    const double s = uw_over_uref;              // rho u / u_ref, linearised rho = 1
    const float *p = pred + cell * 6;
    const hermite::Cell q = {s * p[0], s * p[1], s * p[2], s * p[3], s * p[4], s * p[5]};
    hermite::put_row(q, c, xi1[iy], w1[iy], iy, m, (int)(cell % nx), (int)(cell / nx), ny, pa, py, h, tiled32);
}

lbm_status mfail(lbm_status s, const std::string &m) { return lbm_norms_fail(s, m.c_str()); }

}  // namespace

struct lbm_mlp {
    int max_batch;
    cudaStream_t stream;
    void *base;
    // flat parameters (W_0, b_0, W_1, ...), Adam moments and gradient; BF16 copies per layer
    float *p, *m, *v, *grad;
    __nv_bfloat16 *wq[NL];    // [N][PADW[l]]
    __nv_bfloat16 *wqT[NL];   // [K][PADW[l+1]]
    float *x32;               // staging of a forward pass in place
    __nv_bfloat16 *aT[NL], *gT[NL];
    float *gp, *colpart, *part;
    double *loss_part;
    double *host_loss;
    int *status;              // set by a kernel whose bounded wait gave up
    ChainMaps chain;
    GradMaps grads;           // of grad_tiles row tiles
    int grad_tiles;
    long step;
};

namespace {

size_t al(size_t v) { return (v + 255) & ~(size_t)255; }

constexpr long nparams()
{
    long n = 0;
    for (int l = 0; l < NL; ++l) n += (long)WIDTH[l + 1] * WIDTH[l] + WIDTH[l + 1];
    return n;
}

// offset of layer l's weights in the flat arrays; its biases follow them
long weights_at(int l)
{
    long o = 0;
    for (int q = 0; q < l; ++q) o += (long)WIDTH[q + 1] * WIDTH[q] + WIDTH[q + 1];
    return o;
}
long biases_at(int l) { return weights_at(l) + (long)WIDTH[l + 1] * WIDTH[l]; }

int row_tiles(int rows) { return (rows + ROWS - 1) / ROWS; }

// layout of all device arrays of one MLP; returns total bytes, fills pointers if base != nullptr
size_t mlp_layout(lbm_mlp *p, char *base, int M)
{
    size_t off = 0;
    const long tiles = row_tiles(M), rows = tiles * ROWS;
    auto take = [&](size_t bytes) -> char * {
        char *r = base ? base + off : nullptr;
        off = al(off + bytes);
        return r;
    };
    lbm_mlp dummy;
    lbm_mlp &q = p ? *p : dummy;
    for (float **f : {&q.p, &q.m, &q.v, &q.grad}) *f = (float *)take(4 * nparams());
    for (int l = 0; l < NL; ++l) {
        q.wq[l] = (__nv_bfloat16 *)take(2 * (size_t)WIDTH[l + 1] * PADW[l]);
        q.wqT[l] = (__nv_bfloat16 *)take(2 * (size_t)WIDTH[l] * PADW[l + 1]);
        q.aT[l] = (__nv_bfloat16 *)take(2 * (size_t)WIDTH[l] * rows);
        q.gT[l] = (__nv_bfloat16 *)take(2 * (size_t)WIDTH[l + 1] * rows);
    }
    q.x32 = (float *)take(16 * (size_t)M);
    q.gp = (float *)take(4 * (size_t)3 * 256 * rows);
    q.colpart = (float *)take(4 * (size_t)COLS * tiles);
    q.part = (float *)take(4 * (size_t)WTILES * SPLITS * 128 * 128);
    q.loss_part = (double *)take(8 * (size_t)tiles);
    q.status = (int *)take(16);
    return off;
}

int blocks_for(long n) { long b = (n + 255) / 256; return (int)(b < 1 ? 1 : (b > 1216 ? 1216 : b)); }

cudaError_t refresh_bf16(lbm_mlp *p, int l)
{
    const int n = WIDTH[l + 1], k = WIDTH[l];
    refresh_kernel<<<blocks_for((long)n * k), 256, 0, p->stream>>>(p->p + weights_at(l), n, k, p->wq[l], PADW[l], p->wqT[l],
                                                                   PADW[l + 1]);
    return cudaGetLastError();
}

bool make_chain_maps(lbm_mlp *p)
{
    bool ok = true;
    for (int l = 0; l < NL; ++l)
        ok = ok && umma::make_map(&p->chain.w[l], p->wq[l], WIDTH[l + 1], PADW[l], PADW[l], l == 3 ? 16 : 128);
    for (int l = NL - 1; l > 0; --l)
        ok = ok && umma::make_map(&p->chain.w[7 - l], p->wqT[l], WIDTH[l], PADW[l + 1], PADW[l + 1], 128);
    return ok;
}

// the weight gradients sum over whole row tiles: their maps end at the batch's last one
bool make_grad_maps(lbm_mlp *p, int tiles)
{
    if (p->grad_tiles == tiles) return true;
    p->grad_tiles = 0;
    bool ok = true;
    for (int l = 0; l < NL; ++l)
        ok = ok && umma::make_map(&p->grads.g[l], p->gT[l], WIDTH[l + 1], ROWS, ROWS, 128, tiles) &&
             umma::make_map(&p->grads.a[l], p->aT[l], WIDTH[l], ROWS, ROWS, l == 0 ? 16 : 128, tiles);
    if (ok) p->grad_tiles = tiles;
    return ok;
}

ChainArgs chain_args(lbm_mlp *p, const float *x, int M)
{
    ChainArgs a;
    std::memset(&a, 0, sizeof a);
    a.x = x;
    for (int l = 0; l < NL; ++l) {
        a.b[l] = p->p + biases_at(l);
        a.aT[l] = p->aT[l];
        a.gT[l] = p->gT[l];
    }
    a.gp = p->gp;
    a.colpart = p->colpart;
    a.loss = p->loss_part;
    a.M = M;
    a.status = p->status;
    return a;
}

// splitmix64-based uniform numbers for the default initialisation
double u01(uint64_t &state)
{
    uint64_t z = (state += 0x9E3779B97F4A7C15ULL);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    z ^= z >> 31;
    return (double)(z >> 11) * (1.0 / 9007199254740992.0);
}

}  // namespace

extern "C" {

lbm_status lbm_mlp_param_count(long *count)
{
    if (!count) return mfail(LBM_EINVAL, "count is NULL");
    *count = nparams();
    return LBM_OK;
}

lbm_status lbm_mlp_create(int max_batch, unsigned long long seed, void *stream, lbm_mlp **out)
{
    if (!out || max_batch < 1 || max_batch > (1 << 24)) return mfail(LBM_EINVAL, "invalid MLP arguments");
    *out = nullptr;
    lbm_mlp *p = new (std::nothrow) lbm_mlp;
    if (!p) return mfail(LBM_ENOMEM, "host allocation failed");
    std::memset(p, 0, sizeof *p);
    p->max_batch = max_batch;
    p->stream = (cudaStream_t)stream;
    const size_t bytes = mlp_layout(nullptr, nullptr, max_batch);
    cudaError_t e = cudaMalloc(&p->base, bytes);
    if (e != cudaSuccess) {
        delete p;
        return mfail(LBM_ENOMEM, std::string("cudaMalloc for the MLP: ") + cudaGetErrorString(e));
    }
    mlp_layout(p, (char *)p->base, max_batch);
    e = cudaMemsetAsync(p->base, 0, bytes, p->stream);
    if (e == cudaSuccess) e = cudaMallocHost(&p->host_loss, sizeof(double) * row_tiles(max_batch));
    if (e == cudaSuccess) e = prepare_chain();
    if (e == cudaSuccess) e = prepare_grads();
    if (e == cudaSuccess && !make_chain_maps(p)) e = cudaErrorInvalidValue;
    if (e != cudaSuccess) {
        lbm_mlp_destroy(p);
        return mfail(LBM_ECUDA, cudaGetErrorString(e));
    }
    // default initialisation: U(-1/sqrt(fan_in), 1/sqrt(fan_in))
    uint64_t st = seed;
    std::vector<float> flat;
    for (int l = 0; l < NL; ++l) {
        const double bound = 1.0 / std::sqrt((double)WIDTH[l]);
        for (long i = 0; i < (long)WIDTH[l + 1] * WIDTH[l] + WIDTH[l + 1]; ++i)
            flat.push_back((float)((2.0 * u01(st) - 1.0) * bound));
    }
    lbm_status s2 = lbm_mlp_set_params(p, flat.data());
    if (s2 != LBM_OK) {
        lbm_mlp_destroy(p);
        return s2;
    }
    *out = p;
    return LBM_OK;
}

void lbm_mlp_destroy(lbm_mlp *p)
{
    if (!p) return;
    if (p->stream) cudaStreamSynchronize(p->stream);
    else cudaDeviceSynchronize();
    if (p->base) cudaFree(p->base);
    if (p->host_loss) cudaFreeHost(p->host_loss);
    delete p;
}

lbm_status lbm_mlp_set_params(lbm_mlp *p, const float *flat)
{
    if (!p || !flat) return mfail(LBM_EINVAL, "NULL argument");
    cudaError_t e = cudaMemcpyAsync(p->p, flat, 4 * nparams(), cudaMemcpyHostToDevice, p->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(p->m, 0, 4 * nparams(), p->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(p->v, 0, 4 * nparams(), p->stream);
    for (int l = 0; l < NL && e == cudaSuccess; ++l) e = refresh_bf16(p, l);
    if (e == cudaSuccess) e = cudaStreamSynchronize(p->stream);
    p->step = 0;
    return e == cudaSuccess ? LBM_OK : mfail(LBM_ECUDA, cudaGetErrorString(e));
}

lbm_status lbm_mlp_get_params(lbm_mlp *p, float *flat)
{
    if (!p || !flat) return mfail(LBM_EINVAL, "NULL argument");
    cudaError_t e = cudaMemcpyAsync(flat, p->p, 4 * nparams(), cudaMemcpyDeviceToHost, p->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(p->stream);
    return e == cudaSuccess ? LBM_OK : mfail(LBM_ECUDA, cudaGetErrorString(e));
}

lbm_status lbm_mlp_forward(lbm_mlp *p, const float *x_dev, int M, float *y_dev)
{
    if (!p || !x_dev || !y_dev || M < 1 || M > p->max_batch) return mfail(LBM_EINVAL, "invalid forward arguments");
    // row tiles write y while others still read x: overlapping buffers go through a copy of x
    const uintptr_t x0 = (uintptr_t)x_dev, y0 = (uintptr_t)y_dev;
    cudaError_t e = cudaSuccess;
    if (x0 < y0 + 24L * M && y0 < x0 + 16L * M) {
        e = cudaMemcpyAsync(p->x32, x_dev, 16L * M, cudaMemcpyDeviceToDevice, p->stream);
        x_dev = p->x32;
    }
    ChainArgs a = chain_args(p, x_dev, M);
    a.y = y_dev;
    if (e == cudaSuccess) e = launch_chain(false, p->chain, a, p->stream);
    return e == cudaSuccess ? LBM_OK : mfail(LBM_ECUDA, cudaGetErrorString(e));
}

// Chain, weight gradients and their reduction: the gradient into p->grad (lr = 0) or one Adam
// step; the loss (may be NULL) of the parameters before it.
static lbm_status train(lbm_mlp *p, const float *x_dev, const float *t_dev, int M, float lr, double *loss)
{
    const int tiles = row_tiles(M), ktiles = tiles * (ROWS / umma::UK), splits = ktiles < SPLITS ? ktiles : SPLITS;
    if (!make_grad_maps(p, tiles)) return mfail(LBM_ECUDA, "encoding a tensor map failed");
    ChainArgs c = chain_args(p, x_dev, M);
    c.t = t_dev;
    cudaError_t e = launch_chain(true, p->chain, c, p->stream);
    if (e == cudaSuccess) e = launch_grads(p->grads, ktiles, splits, p->part, p->status, p->stream);
    if (e != cudaSuccess) return mfail(LBM_ECUDA, cudaGetErrorString(e));
    if (loss) {
        int stw = 0;
        e = cudaMemcpyAsync(p->host_loss, p->loss_part, 8L * tiles, cudaMemcpyDeviceToHost, p->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&stw, p->status, sizeof(int), cudaMemcpyDeviceToHost, p->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(p->stream);
        if (e != cudaSuccess) return mfail(LBM_ECUDA, cudaGetErrorString(e));
        if (stw != 0) return mfail(LBM_ETIMEOUT, "a bounded wait of a tensor-core kernel gave up");
        double s = 0.0;
        for (int i = 0; i < tiles; ++i) s += p->host_loss[i];
        *loss = s / ((double)M * WIDTH[NL]);
    }
    AdamArgs a;
    std::memset(&a, 0, sizeof a);
    a.part = p->part;
    a.colpart = p->colpart;
    a.splits = splits;
    a.tiles = tiles;
    if (lr > 0) {
        p->step += 1;
        a.p = p->p;
        a.m = p->m;
        a.v = p->v;
        for (int l = 0; l < NL; ++l) {
            a.wq[l] = p->wq[l];
            a.wqT[l] = p->wqT[l];
        }
        a.lr = lr;
        a.c1 = 1.f - std::pow(0.9f, (float)p->step);
        a.c2 = 1.f - std::pow(0.999f, (float)p->step);
    } else {
        a.grad = p->grad;
    }
    e = launch_reduce_adam(a, p->stream);
    return e == cudaSuccess ? LBM_OK : mfail(LBM_ECUDA, cudaGetErrorString(e));
}

lbm_status lbm_mlp_loss_grad(lbm_mlp *p, const float *x_dev, const float *t_dev, int M, double *loss, float *grad_flat)
{
    if (!p || !x_dev || !t_dev || M < 1 || M > p->max_batch) return mfail(LBM_EINVAL, "invalid arguments");
    lbm_status st = train(p, x_dev, t_dev, M, 0.f, loss);
    if (st != LBM_OK || !grad_flat) return st;
    cudaError_t e = cudaMemcpyAsync(grad_flat, p->grad, 4 * nparams(), cudaMemcpyDeviceToHost, p->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(p->stream);
    return e == cudaSuccess ? LBM_OK : mfail(LBM_ECUDA, cudaGetErrorString(e));
}

lbm_status lbm_mlp_train_step(lbm_mlp *p, const float *x_dev, const float *t_dev, int M, float lr, double *loss)
{
    if (!p || !x_dev || !t_dev || M < 1 || M > p->max_batch || !(lr > 0)) return mfail(LBM_EINVAL, "invalid arguments");
    return train(p, x_dev, t_dev, M, lr, loss);
}

lbm_status lbm_mlp_features(lbm_mlp *p, int nx, int ny, double kn, double u_w, float *x_dev)
{
    if (!p || !x_dev || nx < 1 || ny < 1 || !(kn > 0)) return mfail(LBM_EINVAL, "invalid feature arguments");
    const float f2 = (float)((2.0 * std::log10(kn) + 1.0) / 3.0);
    const float f3 = (float)((u_w - 0.0125) / 0.0075);
    features_kernel<<<blocks_for((long)nx * ny), 256, 0, p->stream>>>(nx, ny, f2, f3, x_dev);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? LBM_OK : mfail(LBM_ECUDA, cudaGetErrorString(e));
}

}  // extern "C"

cudaError_t launch_warm_state(const float *pred, int nx, int ny, long pa, long py, int m, const double *xi1,
                              const double *w1, double uw_over_uref, void *h, int prec, cudaStream_t s, bool tiled32)
{
    const unsigned nb = (unsigned)(((long)nx * ny + 31) / 32);
    if (prec == LBM_FP64)
        warm_state_kernel<double><<<nb, 32 * m, 0, s>>>(pred, nx, ny, pa, py, m, xi1, w1, uw_over_uref, (double *)h, tiled32);
    else
        warm_state_kernel<float><<<nb, 32 * m, 0, s>>>(pred, nx, ny, pa, py, m, xi1, w1, uw_over_uref, (float *)h, tiled32);
    return cudaGetLastError();
}

cudaStream_t mlp_stream(const lbm_mlp *p) { return p->stream; }
