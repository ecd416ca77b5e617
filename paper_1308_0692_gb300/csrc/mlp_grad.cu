// Weight gradients of the warm-start network, their reduction and Adam (sm_103a).
//
// mlp_grad_kernel: dW_l = g_l^T a_l for the four layers in one launch, K = the batch rows
// (128-row tiles padded with zero gradients).  A CTA takes one 128 x 128 tile (128 x 16 for the
// 4-wide input layer) of one layer and one of the K-splits: a TMA producer, one thread issuing
// tcgen05.mma, a ring of four stages, the accumulators in tensor memory -- and stores its partial
// tile column by column (lane = row: contiguous).  Twelve tiles times at most twelve splits are
// 144 CTAs, one wave of the 152 SMs.  The CTA's steps go to four accumulators, a quarter of them
// each: FP32 additions in tensor memory lose half an ulp on average, so the error grows with the
// length of a chain, and 48 chains are shorter than twelve (128 rows over and over, 8192 and 32768 in
// all: relative error of the gradients 1.2e-7 and 6.1e-7; with one accumulator 6.2e-7 and 2.8e-6).
// They fill the tensor memory; no other kernel of the network fits on the SM beside this one's
// shared memory.
//
// mlp_reduce_adam_kernel: adds the splits in ascending order, turns the 32 x 32 block through
// shared memory, applies Adam on the FP32 master weights and refreshes both BF16 copies
// (W and W^T); the last blocks do the biases from the row tiles' column sums.  Replaces a
// reduction, an Adam, a conversion and a transposition launch per array.
#include <algorithm>

#include "mlp_internal.h"
#include "umma.cuh"

using namespace umma;

namespace mlpk {

namespace {

constexpr int STAGES = 4;
constexpr int STAGE = 2 * UM * 128;                 // bytes: A and B tiles of one K step
constexpr int SMEM = STAGES * STAGE + 1024;
constexpr int ACCS = 4, ACC = 128;                  // accumulators of a CTA, 128 columns each

// tile t of the list: layer, first row (of N_l), first column (of K_l), columns
struct Tile {
    int l, m0, n0, n;
};
__host__ __device__ constexpr Tile tile_of(int t)
{
    if (t < 4) return {1, (t & 1) * 128, (t >> 1) * 128, 128};
    if (t < 8) return {2, (t & 1) * 128, ((t - 4) >> 1) * 128, 128};
    if (t < 10) return {3, 0, (t - 8) * 128, 128};
    return {0, (t - 10) * 128, 0, 16};
}
// tile that holds row n (of N_l), column k (of K_l) of layer l
__device__ __forceinline__ int tile_at(int l, int n, int k)
{
    if (l == 1) return (n >> 7) + 2 * (k >> 7);
    if (l == 2) return 4 + (n >> 7) + 2 * (k >> 7);
    if (l == 3) return 8 + (k >> 7);
    return 10 + (n >> 7);
}

__global__ void __launch_bounds__(256, 1)
    mlp_grad_kernel(const __grid_constant__ GradMaps maps, int ktiles, int kper, float *part, int *status)
{
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], accf;
    __shared__ uint32_t s_tmem;
    unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const Tile t = tile_of(blockIdx.x);
    const int kt0 = blockIdx.y * kper, kt1 = min(ktiles, kt0 + kper);
    const int chain = max(1, (kt1 - kt0 + ACCS - 1) / ACCS);      // steps of an accumulator

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            bar_init(&full[s], 1);
            bar_init(&empty[s], 1);
        }
        bar_init(&accf, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 0) tmem_alloc(&s_tmem, ACCS * ACC);
    asm volatile("griddepcontrol.launch_dependents;\n griddepcontrol.wait;\n" ::: "memory");
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = s_tmem;

    if (warp == 0 && lane == 0) {
        // ---- producer ----
        int issued = 0;
        for (int kt = kt0; kt < kt1; ++kt, ++issued) {
            const int s = issued % STAGES;
            if (issued >= STAGES && !bar_wait(&empty[s], ((issued / STAGES) - 1) & 1)) {
                atomicExch(status, 1);
                break;
            }
            unsigned char *st = smem + s * STAGE;
            bar_expect(&full[s], (unsigned)((UM + t.n) * 128));
            const int x = (kt & 1) * UK, z = kt >> 1;          // ROWS = 2 UK
            tma_load_3d(st, &maps.g[t.l], x, t.m0, z, &full[s]);
            tma_load_3d(st + UM * 128, &maps.a[t.l], x, t.n0, z, &full[s]);
        }
        // the copies still in flight land before the CTA can exit
        for (int j = issued > STAGES ? issued - STAGES : 0; j < issued; ++j) bar_wait(&full[j % STAGES], (j / STAGES) & 1);
    } else if (warp == 1 && lane == 0) {
        // ---- MMA issuer ----
        const uint32_t idesc = instr_desc(t.n);
        int done = 0;
        for (int kt = kt0; kt < kt1; ++kt, ++done) {
            const int s = done % STAGES;
            if (!bar_wait(&full[s], (done / STAGES) & 1)) {
                atomicExch(status, 1);
                break;
            }
            fence_after_sync();
            const unsigned char *st = smem + s * STAGE;
            const uint64_t da = smem_desc(st), db = smem_desc(st + UM * 128);
#pragma unroll
            for (int k = 0; k < UK / 16; ++k)   // advance 16 BF16 = 32 bytes along K inside the swizzle row
                mma_bf16(tmem + (uint32_t)(done / chain * ACC), da + 2 * k, db + 2 * k, idesc, (done % chain | k) ? 1u : 0u);
            mma_commit(&empty[s]);
        }
        mma_commit(&accf);
    }
    __syncwarp();
    const bool ok = bar_wait(&accf, 0);
    if (!ok && lane == 0) atomicExch(status, 1);
    fence_after_sync();
    // ---- epilogue: warp w takes rows 32 (w % 4).., columns 64 (w / 4)..; column-major partial tile
    float *out = part + ((long)blockIdx.x * gridDim.y + blockIdx.y) * (128 * 128) + (warp & 3) * 32 + lane;
    const int accs = kt1 > kt0 ? (kt1 - kt0 + chain - 1) / chain : 0;
    __syncwarp();
#pragma unroll 1
    for (int c0 = (warp >> 2) * 64; c0 < (warp >> 2) * 64 + 64 && c0 < t.n; c0 += 32) {
        float v[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = 0.f;
        for (int q = 0; q < accs; ++q) {
            float u[32];
            tmem_ld32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(q * ACC + c0), u);
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] += u[j];
        }
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (c0 + j < t.n) out[(c0 + j) * 128] = v[j];
    }
    fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        fence_after_sync();
        tmem_free(tmem, ACCS * ACC);
    }
}

// 32 x 32 blocks of the weight arrays, layers in order, then the biases
struct Blocks {
    int first[NL + 1];
};
__host__ __device__ constexpr Blocks weight_blocks()
{
    Blocks b{};
    int at = 0;
    for (int l = 0; l < NL; ++l) {
        b.first[l] = at;
        at += ((WIDTH[l + 1] + 31) / 32) * ((WIDTH[l] + 31) / 32);
    }
    b.first[NL] = at;
    return b;
}
constexpr int BIASES = 3 * 256 + 6;

__device__ __forceinline__ float adam(const AdamArgs &a, long i, float g)
{
    constexpr float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float mi = b1 * a.m[i] + (1.f - b1) * g;
    const float vi = b2 * a.v[i] + (1.f - b2) * g * g;
    a.m[i] = mi;
    a.v[i] = vi;
    const float pi = a.p[i] - a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + eps);
    a.p[i] = pi;
    return pi;
}

__global__ void __launch_bounds__(256) mlp_reduce_adam_kernel(const __grid_constant__ AdamArgs a)
{
    constexpr Blocks B = weight_blocks();
    constexpr int N[NL] = {WIDTH[1], WIDTH[2], WIDTH[3], WIDTH[4]}, K[NL] = {WIDTH[0], WIDTH[1], WIDTH[2], WIDTH[3]};
    constexpr int LDQ[NL] = {PADW[0], PADW[1], PADW[2], PADW[3]}, LDT[NL] = {PADW[1], PADW[2], PADW[3], PADW[4]};
    __shared__ float tile[32][33];
    const int bid = blockIdx.x;
    asm volatile("griddepcontrol.launch_dependents;\n griddepcontrol.wait;\n" ::: "memory");
    if (bid >= B.first[NL]) {
        // biases: the row tiles' column sums, 32 columns a block, 8 groups of tiles in turn, then
        // the groups in order
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        const int c = (bid - B.first[NL]) * 32 + lane;
        float s = 0.f;
        if (c < BIASES)
            for (int t = w; t < a.tiles; t += 8) s += a.colpart[(long)t * COLS + c];
        tile[w][lane] = s;
        __syncthreads();
        if (w == 0 && c < BIASES) {
            float g = 0.f;
#pragma unroll
            for (int q = 0; q < 8; ++q) g += tile[q][lane];
            int l = c < 768 ? c >> 8 : 3;
            long at = c < 768 ? (c & 255) : c - 768;
            for (int q = 0; q < l; ++q) at += (long)N[q] * K[q] + N[q];
            at += (long)N[l] * K[l];
            if (a.grad) a.grad[at] = g;
            if (a.p) adam(a, at, g);
        }
        return;
    }
    int l = 0;
    while (l + 1 < NL && bid >= B.first[l + 1]) ++l;
    long base = 0;
    for (int q = 0; q < l; ++q) base += (long)N[q] * K[q] + N[q];
    const int nl = N[l], kl = K[l], kb = (kl + 31) / 32;
    const int n0 = ((bid - B.first[l]) / kb) * 32, k0 = ((bid - B.first[l]) % kb) * 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // sums with lane = row n (the partial tiles' order)
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    const int n = n0 + lane;
    if (n < nl) {
        // the block's 32 columns lie in one partial tile; eight splits of loads in flight
        const float *src = a.part + (long)tile_at(l, n, k0) * a.splits * (128 * 128) + ((k0 & 127) + w) * 128 + (n & 127);
        const int nq = kl - k0 - w > 0 ? min(4, (kl - k0 - w + 7) / 8) : 0;
#pragma unroll 8
        for (int z = 0; z < a.splits; ++z)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (q < nq) s[q] += src[(long)z * (128 * 128) + q * 8 * 128];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) tile[w + 8 * q][lane] = s[q];
    __syncthreads();
    // parameters with lane = column k
    const int k = k0 + lane;
#pragma unroll
    for (int q = 0; q < 4; ++q) s[q] = tile[lane][w + 8 * q];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int nn = n0 + w + 8 * q;
        float v = 0.f;
        if (nn < nl && k < kl) {
            const long at = base + (long)nn * kl + k;
            if (a.grad) a.grad[at] = s[q];
            if (a.p) {
                v = adam(a, at, s[q]);
                a.wq[l][(long)nn * LDQ[l] + k] = __float2bfloat16_rn(v);
            }
        }
        tile[w + 8 * q][lane] = v;
    }
    if (!a.p) return;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int kk = k0 + w + 8 * q;
        if (kk < kl && n < nl) a.wqT[l][(long)kk * LDT[l] + n] = __float2bfloat16_rn(tile[lane][w + 8 * q]);
    }
}

}  // namespace

cudaError_t prepare_grads() { return cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM); }

cudaError_t launch_grads(const GradMaps &maps, int ktiles, int splits, float *part, int *status, cudaStream_t s)
{
    return launch_after(mlp_grad_kernel, dim3(WTILES, splits), 256, SMEM, s, maps, ktiles, (ktiles + splits - 1) / splits, part,
                        status);
}

cudaError_t launch_reduce_adam(const AdamArgs &a, cudaStream_t s)
{
    const int blocks = weight_blocks().first[NL] + (BIASES + 31) / 32;
    return launch_after(mlp_reduce_adam_kernel, dim3(blocks), 256, 0, s, a);
}

}  // namespace mlpk
