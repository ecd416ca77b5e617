// The row-local part of the warm-start network in one launch (sm_103a): the forward pass
//   z_l = a_l W_l^T + b_l, a_{l+1} = bf16(GELU(z_l)), y = z_3,
// and in training also the loss and the chain of input gradients
//   g_3 = 2 (y - t) / (6 M), g_{l-1} = (g_l W_l) GELU'(z_{l-1}),
// every product BF16 x BF16 into FP32 on the fifth-generation tensor cores.
//
// A cluster of two CTAs takes 128 rows of the batch; each CTA computes 128 of the 256 columns
// of every hidden product (M = 128, N = 128, K = 256 in steps of 64) and writes its columns of
// the next layer's BF16 operand into its own and, through distributed shared memory, into its
// partner's operand buffer (two buffers in turn, K-major with the 128-byte swizzle the product
// reads).  Activations and gradients thus never leave the chip between layers.  The weights
// stream in by TMA: a layer's slice (up to 64 KB) replaces the last one as soon as its products
// have read it, behind the epilogue.  The 6-wide output layer is computed by both CTAs.
//
// What bounds it: not the products (5 us of tensor time over the whole chip at 8192 rows is
// 2 us) but the elementwise work of the epilogues, erff above all, and the chain of seven
// products, each behind a cluster barrier.  Two CTAs per 128 rows put that work on 128 SMs at
// 8192 rows instead of 64, and sixteen warps per CTA keep each SM quarter's issue slots busy.
//
// Training leaves for the weight gradients the transposed operands a_l^T, g_l^T, row tile by row
// tile ([tile][column][128]: lane = row, so a warp's store of one column is contiguous and needs
// no transposition pass, and the columns are a fixed distance apart), and per tile the column
// sums of the FP32 g_l in a fixed order (a butterfly over the lanes, then the four row groups).
// Those stores, GELU' and the column sums come after the arrival at the cluster barrier, behind
// the next product: before it, the barrier's release waited for every one of the stores.
#include <cstring>

#include "mlp_internal.h"
#include "umma.cuh"

using namespace umma;

namespace mlpk {

namespace {

constexpr int THREADS = 512;
constexpr int BN = 128;                             // columns a CTA computes of a hidden product
constexpr int SUB = ROWS * 128;                     // bytes of one 64-wide K step of an operand
constexpr int SMEM_A = 4 * SUB, SMEM = 2 * SMEM_A + 4 * SUB + 1024;

// GELU(z) = z e / 2 with e = 1 + erf(z / sqrt 2), and its derivative
__device__ __forceinline__ float gelu_e(float z) { return 1.0f + erff(z * 0.70710678118654752f); }
__device__ __forceinline__ float gelu_grad(float z, float e) { return 0.5f * e + z * expf(-0.5f * z * z) * 0.39894228040143268f; }

__device__ __forceinline__ unsigned peer_address(unsigned addr, unsigned rank)
{
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }

__device__ __forceinline__ unsigned pack(float lo, float hi)
{
    const __nv_bfloat162 v = __halves2bfloat162(__float2bfloat16_rn(lo), __float2bfloat16_rn(hi));
    return *reinterpret_cast<const unsigned *>(&v);
}

// Sum over the warp's 32 lanes of each of 32 values: lane j returns column j's sum
__device__ __forceinline__ float column_sum(float (&v)[32], int lane)
{
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
#pragma unroll
        for (int i = 0; i < s; ++i) {
            const float send = (lane & s) ? v[i] : v[i + s], keep = (lane & s) ? v[i + s] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
        }
    }
    return v[0];
}

template <bool TRAIN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
    mlp_chain_kernel(const __grid_constant__ ChainMaps maps, const __grid_constant__ ChainArgs p)
{
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full, done;
    __shared__ uint32_t s_tmem;
    __shared__ float s_col[2][4][BN];                // by product parity: read after the next barrier
    __shared__ double s_loss[4];
    unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char *const wbuf = smem + 2 * SMEM_A;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rg = warp & 3, cg = warp >> 2;           // 32 rows, 32 columns of a warp's part
    const int rank = blockIdx.x & 1, tile = blockIdx.x >> 1;
    const int row = rg * 32 + lane;
    const long grow = (long)tile * ROWS + row;
    const bool valid = grow < p.M;

    if (tid == 0) {
        bar_init(&full, 1);
        bar_init(&done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 0) tmem_alloc(&s_tmem, BN);
    // the kernels of a step are set up while the one before runs and wait for it here
    asm volatile("griddepcontrol.launch_dependents;\n griddepcontrol.wait;\n" ::: "memory");
    // layer 0's operand: the four features, zeros up to K = 16
    if (cg == 0) {
        float f[4] = {0.f, 0.f, 0.f, 0.f};
        if (valid)
#pragma unroll
            for (int c = 0; c < 4; ++c) f[c] = p.x[grow * 4 + c];
        uint4 *at = reinterpret_cast<uint4 *>(smem + row * 128);
        at[0 ^ (row & 7)] = make_uint4(pack(f[0], f[1]), pack(f[2], f[3]), 0u, 0u);
        at[1 ^ (row & 7)] = make_uint4(0u, 0u, 0u, 0u);
        if (TRAIN && rank == 0)
#pragma unroll
            for (int c = 0; c < 4; ++c) p.aT[0][((long)tile * 4 + c) * ROWS + row] = __float2bfloat16_rn(f[c]);
    }
    asm volatile("fence.proxy.async;\n" ::: "memory");
    fence_before_sync();
    __syncthreads();
    cluster_arrive();
    cluster_wait();                                    // the partner's buffers may be written from here on
    fence_after_sync();
    const uint32_t tmem = s_tmem;

    // products in order: forward layers 0-3, then the input gradients of layers 3, 2, 1
    constexpr int NPROD = TRAIN ? 7 : 4;
    auto rows_of = [](int i) { return i == 3 ? 16 : BN; };
    auto ksteps_of = [](int i) { return (i == 0 || i == 4) ? 1 : 4; };
    auto fetch = [&](int i) {                          // weights of product i (one thread)
        const int n = rows_of(i), nk = ksteps_of(i);
        bar_expect(&full, (unsigned)(nk * n * 128));
        for (int k = 0; k < nk; ++k) tma_load_2d(wbuf + k * n * 128, &maps.w[i], k * UK, i == 3 ? 0 : rank * BN, &full);
    };
    bool ok = true;
    if (tid == 0) fetch(0);
    __syncwarp();
    // products of one thread: operand i in abuf, weights i in wbuf
    auto multiply = [&](int i) {
        ok = bar_wait(&full, i & 1) && ok;
        fence_after_sync();
        asm volatile("fence.proxy.async;\n" ::: "memory");
        const unsigned char *abuf = smem + (i & 1) * SMEM_A;
        const uint32_t idesc = instr_desc(rows_of(i));
        const int nk = ksteps_of(i), ks = nk == 1 ? 1 : UK / 16;       // K = 16 of layer 0's and 3's operands
        for (int k = 0; k < nk; ++k) {
            const uint64_t da = smem_desc(abuf + k * SUB), db = smem_desc(wbuf + k * rows_of(i) * 128);
            for (int q = 0; q < ks; ++q) mma_bf16(tmem, da + 2 * q, db + 2 * q, idesc, (k | q) ? 1u : 0u);
        }
        mma_commit(&done);
    };
    if (tid == 0) multiply(0);
    __syncwarp();
#pragma unroll 1
    for (int i = 0; i < NPROD; ++i) {
        const bool fwd = i < 4;
        const int l = fwd ? i : 6 - i;                 // layer of z (forward) or of g_l (backward)
        const int n0 = rank * BN + cg * 32;            // this warp's first column of a hidden product
        unsigned char *anext = smem + ((i + 1) & 1) * SMEM_A;
        float *gpt = TRAIN ? p.gp + (((long)tile * 3 + (l < 3 ? l : 0)) * 256 + n0) * ROWS + row : nullptr;
        float gp[TRAIN ? 32 : 1];
        if (TRAIN && !fwd) {                           // GELU' of this thread's values, stored by it before
#pragma unroll
            for (int j = 0; j < 32; ++j) gp[TRAIN ? j : 0] = gpt[j * ROWS];
        }
        ok = bar_wait(&done, i & 1) && ok;
        __syncwarp();
        fence_after_sync();
        if (tid == 0 && i + 1 < NPROD) fetch(i + 1);   // the products have read the last weights
        __syncwarp();
        const uint32_t lanes = tmem + ((uint32_t)(rg * 32) << 16);
        float v[32], z[TRAIN ? 32 : 1];
        float g[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        double acc = 0.0;
        // ---- the next product's operand, here and at the partner ----
        if (i != 3) {
            tmem_ld32(lanes + (uint32_t)(cg * 32), v);
            if (fwd) {
                const float *bias = p.b[i];            // (no read-only path: the step before updates them while this grid is set up)
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const float zj = v[j] + bias[n0 + j], e = gelu_e(zj);
                    if (TRAIN) {
                        z[TRAIN ? j : 0] = zj;
                        gp[TRAIN ? j : 0] = e;
                    }
                    v[j] = 0.5f * zj * e;
                }
            } else {
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] *= gp[TRAIN ? j : 0];
            }
            if (i + 1 < NPROD) {
                const unsigned base = su32(anext + (n0 >> 6) * SUB + row * 128);
                const unsigned far = peer_address(base, (unsigned)(rank ^ 1));
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const unsigned off = (unsigned)(((((n0 & 32) >> 3) + c) ^ (row & 7)) << 4);
                    const unsigned a = pack(v[8 * c], v[8 * c + 1]), b = pack(v[8 * c + 2], v[8 * c + 3]);
                    const unsigned d = pack(v[8 * c + 4], v[8 * c + 5]), e = pack(v[8 * c + 6], v[8 * c + 7]);
                    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(base + off), "r"(a), "r"(b), "r"(d), "r"(e) : "memory");
                    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(far + off), "r"(a), "r"(b), "r"(d), "r"(e) : "memory");
                }
            }
        } else if (cg == 0) {
            float y[8];
            tmem_ld8(lanes, y);
            const float scale = 2.0f / ((float)p.M * 6.0f);
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                y[c] += p.b[3][c];
                if (!TRAIN) {
                    if (valid && rank == 0) p.y[grow * 6 + c] = y[c];
                } else if (valid) {
                    const float d = y[c] - p.t[grow * 6 + c];
                    acc += (double)d * d;
                    g[c] = scale * d;
                }
            }
            if (TRAIN) {
                uint4 *at = reinterpret_cast<uint4 *>(anext + row * 128);
                at[0 ^ (row & 7)] = make_uint4(pack(g[0], g[1]), pack(g[2], g[3]), pack(g[4], g[5]), 0u);
                at[1 ^ (row & 7)] = make_uint4(0u, 0u, 0u, 0u);
            }
        }
        asm volatile("fence.proxy.async;\n" ::: "memory");
        fence_before_sync();
        __syncwarp();
        cluster_arrive();                              // operands written and the accumulator read
        if (warp == 0) {
            cluster_wait();
            fence_after_sync();
            if (tid == 0 && i + 1 < NPROD) multiply(i + 1);
            __syncwarp();
        }
        // ---- what the weight gradients need, behind the next product ----
        if (TRAIN && i != 3) {
            __nv_bfloat16 *out = (fwd ? p.aT[fwd ? i + 1 : 0] : p.gT[l]) + ((long)tile * 256 + n0) * ROWS + row;
#pragma unroll
            for (int j = 0; j < 32; ++j) out[j * ROWS] = __float2bfloat16_rn(v[j]);
            if (fwd) {
#pragma unroll
                for (int j = 0; j < 32; ++j) gpt[j * ROWS] = gelu_grad(z[TRAIN ? j : 0], gp[TRAIN ? j : 0]);
            } else {
                s_col[i & 1][rg][cg * 32 + lane] = column_sum(v, lane);
            }
        } else if (TRAIN && cg == 0) {
            if (rank == 0)
#pragma unroll
                for (int c = 0; c < 6; ++c) p.gT[3][((long)tile * 6 + c) * ROWS + row] = __float2bfloat16_rn(g[c]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                acc += __shfl_xor_sync(0xffffffffu, acc, o);
#pragma unroll
                for (int c = 0; c < 6; ++c) g[c] += __shfl_xor_sync(0xffffffffu, g[c], o);
            }
            if (lane == 0) {
                s_loss[rg] = acc;
#pragma unroll
                for (int c = 0; c < 6; ++c) s_col[i & 1][rg][c] = g[c];
            }
        }
        if (warp != 0) {
            __syncwarp();
            cluster_wait();
            fence_after_sync();
        }
        if (TRAIN && i >= 3) {
            __syncthreads();
            if (i == 3 ? (rank == 0 && tid < 6) : tid < BN) {
                float t = 0.f;
#pragma unroll
                for (int q = 0; q < 4; ++q) t += s_col[i & 1][q][tid];
                p.colpart[(long)tile * COLS + (i == 3 ? 768 : l * 256 + rank * BN) + tid] = t;
                if (i == 3 && tid == 0) p.loss[tile] = (s_loss[0] + s_loss[1]) + (s_loss[2] + s_loss[3]);
            }
            __syncwarp();
        }
    }
    if (!ok) {
        atomicExch(p.status, 1);
        if (tid == 0) bar_wait(&full, (NPROD - 1) & 1);   // no copy outlives the CTA
    }
    fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        fence_after_sync();
        tmem_free(tmem, BN);
    }
}

}  // namespace

cudaError_t prepare_chain()
{
    cudaError_t e = cudaFuncSetAttribute(mlp_chain_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(mlp_chain_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
}

cudaError_t launch_chain(bool train, const ChainMaps &maps, const ChainArgs &a, cudaStream_t s)
{
    const int grid = 2 * ((a.M + ROWS - 1) / ROWS);
    if (train) return launch_after(mlp_chain_kernel<true>, dim3(grid), THREADS, SMEM, s, maps, a);
    mlp_chain_kernel<false><<<grid, THREADS, SMEM, s>>>(maps, a);     // a single launch: nothing to overlap
    return cudaGetLastError();
}

}  // namespace mlpk
