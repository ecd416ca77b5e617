// Shared by the warm-start network's host code (mlp.cu) and its kernels (mlp_chain.cu, mlp_grad.cu).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace mlpk {

constexpr int NL = 4;                                 // layers
constexpr int WIDTH[NL + 1] = {4, 256, 256, 256, 6};
constexpr int PADW[NL + 1] = {8, 256, 256, 256, 8};   // row lengths of the BF16 copies, padded to 16 bytes
constexpr int ROWS = 128;                             // rows of the batch a CTA pair takes
constexpr int COLS = 3 * 256 + 8;                     // bias gradients of a row tile: layers 0-2, then 3
constexpr int WTILES = 12;                            // 128 x 128 tiles of the four weight gradients
constexpr int SPLITS = 12;                            // K-splits of a weight gradient at most

// tensor maps of the chain kernel: W_0..W_3 (forward) and W_3^T, W_2^T, W_1^T (input gradients)
struct ChainMaps {
    CUtensorMap w[7];
};

struct ChainArgs {
    const float *x;            // [M][4]
    const float *t;            // targets [M][6] (training)
    float *y;                  // [M][6] (inference)
    const float *b[NL];
    // training: what the weight gradients need, transposed ([tile][column][ROWS]), and per row
    // tile the bias gradients and the squared error
    __nv_bfloat16 *aT[NL], *gT[NL];
    float *gp;                 // GELU'(z) of the hidden layers [tiles][3][256][ROWS]
    float *colpart;            // [tiles][COLS]
    double *loss;              // [tiles]
    int M;
    int *status;
};

// tensor maps of the weight gradients: g_l^T and a_l^T, three-dimensional (row of the tile, column, tile)
struct GradMaps {
    CUtensorMap g[NL], a[NL];
};

// Device arrays of the parameters for the reduction and Adam (layer l: W [N][K], b [N])
struct AdamArgs {
    const float *part;         // [WTILES][splits][columns][128] partial weight gradients
    const float *colpart;
    int splits, tiles;
    float *grad;               // flat gradient out, or NULL
    float *p, *m, *v;          // flat parameters and Adam moments (NULL: no update)
    __nv_bfloat16 *wq[NL], *wqT[NL];
    float lr, c1, c2;          // step size, 1 - beta^t
};

// Launch as a programmatic dependent of the stream's last kernel (the kernels of this network wait
// for it themselves); a plain launch on the legacy stream.
template <typename... P, typename... A>
cudaError_t launch_after(void (*fn)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, const A &...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = s != nullptr ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, fn, args...);
}

cudaError_t prepare_chain();
cudaError_t launch_chain(bool train, const ChainMaps &maps, const ChainArgs &a, cudaStream_t s);
cudaError_t prepare_grads();
cudaError_t launch_grads(const GradMaps &maps, int ktiles, int splits, float *part, int *status, cudaStream_t s);
cudaError_t launch_reduce_adam(const AdamArgs &a, cudaStream_t s);

}  // namespace mlpk
