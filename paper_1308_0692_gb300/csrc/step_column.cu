// Several time steps of a one-column Couette channel in one launch (sm_103a): a cluster of 16
// CTAs keeps the channel's whole state on chip, FP64 or FP32, first-order transport
// (Ghiroldi & Gibelli, arXiv:1308.0692, Eqs. 1, 5-9).
//
// What bounds a channel's step launched by itself (step_tile.cuh) is latency: the launch, two
// trips to the L2 and, in FP64, the 64 cycles every FP64 instruction of a warp holds its SM
// quarter.  Here the cells are dealt to the CTAs of one cluster, S threads a cell -- thread =
// (velocity row, part of the row), M / P velocities in registers -- so that a channel of 100
// cells spreads its FP64 work over 60 SM quarters in warps of a few instructions.  Per step:
//   * every thread has put its values into shared memory, the first and last cell of a CTA
//     also into the neighbouring CTA's (distributed shared memory), double-buffered: one
//     cluster barrier a step;
//   * transport: a0 h + nu h_up with the neighbour's value, or at a wall G1 rho_w + G0 with the
//     ghost's coefficients (Eq. 8) in the places of nu and zero: no extra operations;
//   * the moments as sums over the cell's threads in two stages of at most four terms;
//   * rho_w (Eq. 9) from the row sums of the state itself, which the wall cells' threads leave in
//     shared memory before the step's barrier: the same bits wherever a launch begins.  (A recurrence
//     from the sums of the step before, which made the last bits depend on how the steps were dealt
//     to calls, took as long: 100 cells, M = 8, FP64 2.88 us a step against 2.80, FP32 1.55
//     against 1.51.)
// FP32 keeps the wall sums in FP64, as the other FP32 kernels do.
#include <cstring>

#include "lbm_internal.h"

namespace {

template <int M>
struct Shape {
    static constexpr int P = M % 2 ? 1 : 2, V = M / P, S = M * P, HALF = M / 2;
    static constexpr int GS = M == 3 ? 1 : M == 6 ? 3 : 4, NG = S / GS;    // first-stage groups; S / 2 is whole groups
};

constexpr int CLUSTER = 16;

__device__ __forceinline__ unsigned peer(const void *p, unsigned rank)
{
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void put(unsigned at, double v) { asm volatile("st.shared::cluster.f64 [%0], %1;\n" ::"r"(at), "d"(v) : "memory"); }
__device__ __forceinline__ void put(unsigned at, float v) { asm volatile("st.shared::cluster.f32 [%0], %1;\n" ::"r"(at), "f"(v) : "memory"); }

template <typename T>
struct Coef;      // the tables of StepArgs in the arithmetic type
template <>
struct Coef<double> {
    static __device__ __forceinline__ double xi(const StepArgs &a, int i) { return a.xi[i]; }
    static __device__ __forceinline__ double w(const StepArgs &a, int i) { return a.w1[i]; }
    static __device__ __forceinline__ double nuy(const StepArgs &a, int i) { return a.nuy_s[i]; }
    static __device__ __forceinline__ double omw(const StepArgs &a, int i) { return a.omw[i]; }
};
template <>
struct Coef<float> {
    static __device__ __forceinline__ float xi(const StepArgs &a, int i) { return a.xi_f[i]; }
    static __device__ __forceinline__ float w(const StepArgs &a, int i) { return a.w1_f[i]; }
    static __device__ __forceinline__ float nuy(const StepArgs &a, int i) { return a.nuy_f[i]; }
    static __device__ __forceinline__ float omw(const StepArgs &a, int i) { return a.omega_f * a.w1_f[i]; }
};

// Pairwise sum of N values: an FP64 operation is a hundred cycles and more to the next one that
// needs it, so the chains of a step are kept short
template <int N, typename T, typename F>
__device__ __forceinline__ T tree(F f, int first = 0)
{
    if constexpr (N == 1) return f(first);
    else return tree<N / 2, T>(f, first) + tree<N - N / 2, T>(f, first + N / 2);
}

// Shared memory of a CTA of nc cells: values [2][nc + 2][M * M], partial sums [nc][S] of rho, j_x
// and (FP64) xi_y R, first-stage groups and totals
template <typename T, int M>
__host__ __device__ constexpr size_t column_smem(int nc)
{
    using Sh = Shape<M>;
    return sizeof(T) * ((size_t)2 * (nc + 2) * M * M + (size_t)nc * (2 * Sh::S + 2 * Sh::NG + 2)) +
           sizeof(double) * ((size_t)nc * (Sh::S + Sh::NG + 1) + 64 + 1);
}

template <typename T, int M>
__global__ void __launch_bounds__(1024) column_kernel(const __grid_constant__ StepArgs a, int nc, int steps, int resid)
{
    using Sh = Shape<M>;
    cluster_arrive();                              // waited for before the first write into a neighbour
    constexpr int P = Sh::P, V = Sh::V, S = Sh::S, HALF = Sh::HALF, GS = Sh::GS, NG = Sh::NG, NV = M * M;
    constexpr bool DP = sizeof(T) == 8;
    extern __shared__ __align__(16) unsigned char smem[];
    double *const s_j = reinterpret_cast<double *>(smem);            // [nc][S]
    double *const s_jg = s_j + (size_t)nc * S;                       // [nc][NG]
    double *const s_jt = s_jg + (size_t)nc * NG;                     // [nc]
    double *const s_red = s_jt + nc;                                 // [2][32]
    T *const s_v = reinterpret_cast<T *>(s_red + 64);                // [2][nc + 2][NV]
    T *const s_m = s_v + (size_t)2 * (nc + 2) * NV;                  // [2][nc][S]
    T *const s_mg = s_m + (size_t)2 * nc * S;                        // [2][nc][NG]
    T *const s_mt = s_mg + (size_t)2 * nc * NG;                      // [nc][2]
    __shared__ double s_out[2][M];                                   // |xi_y| R of the bottom and the top cell's rows
    unsigned rank;
    asm("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(rank));
    const int ny = a.ny, y0 = (int)rank * nc, nloc = max(0, min(nc, ny - y0));
    const int t = threadIdx.x, cl = t / S, s = t - cl * S, iy = s / P, k0 = (s - iy * P) * V;
    const bool act = cl < nc, on = cl < nloc;
    const int y = y0 + cl;
    const bool up = iy >= M - HALF, down = iy < HALF;
    const bool wall = on && ((up && y == 0) || (down && y == ny - 1));
    const T xiy = Coef<T>::xi(a, iy), omw = Coef<T>::omw(a, iy), nuy = Coef<T>::nuy(a, iy);
    const T a0 = DP ? (T)a.a0[iy * M] : T(0);                        // no x transport: the same for the whole row
    // the wall's populations in the upwind place: g1 rho_w + g0 (Eq. 8), FP64 times the Courant number
    T c1[V], c0[V], xi[V], w[V], wxi[V];
    {
        const double u = up ? a.u_bottom : a.u_top;
#pragma unroll
        for (int k = 0; k < V; ++k) {
            const int ix = k0 + k;
            xi[k] = Coef<T>::xi(a, ix);
            w[k] = Coef<T>::w(a, ix);
            wxi[k] = (T)a.wxi[ix];
            const double wa = a.w1[ix] * a.w1[iy], f = DP ? (double)nuy : 1.0;
            c1[k] = wall ? (T)(f * (wa * (1.0 + a.xi[ix] * u))) : nuy;
            c0[k] = wall ? (T)(f * (wa * (a.xi[ix] * u * a.inv_u_ref))) : T(0);
        }
    }
    const bool edge = on && (y == 0 || y == ny - 1);
    const double out = fabs(a.xi[iy]) * a.inv_dy_wall;
    const T xo = omw * xiy;
    T rho_w = 0;
    const unsigned below = rank > 0 && act && cl == 0 && on && down ? peer(s_v + ((size_t)(nc + 1) * NV + iy * M + k0), rank - 1) : 0;
    const unsigned above = act && on && cl == nloc - 1 && y < ny - 1 && up ? peer(s_v + (iy * M + k0), rank + 1) : 0;
    const unsigned flip = (unsigned)((nc + 2) * NV * sizeof(T));     // bytes from buffer 0 to buffer 1

    const size_t plane = (size_t)a.ncells;
    const T *src = static_cast<const T *>(a.h) + (size_t)(iy * M + k0) * plane + y;
    T h[V];
#pragma unroll
    for (int k = 0; k < V; ++k) h[k] = on ? src[k * plane] : T(0);

    auto publish = [&](int b) {
        if (on) {
            T *at = s_v + ((size_t)b * (nc + 2) + cl + 1) * NV + iy * M + k0;
#pragma unroll
            for (int k = 0; k < V; ++k) at[k] = h[k];
            if (below)
#pragma unroll
                for (int k = 0; k < V; ++k) put(below + b * flip + k * (unsigned)sizeof(T), h[k]);
            if (above)
#pragma unroll
                for (int k = 0; k < V; ++k) put(above + b * flip + k * (unsigned)sizeof(T), h[k]);
        }
        __syncwarp();
        cluster_arrive();
        cluster_wait();
    };
    // what the wall cells' rows carry towards a wall, before the barrier; behind it, Eq. 9
    auto leave = [&] {
        if (__any_sync(0xffffffffu, edge)) {
            double p = out * (double)tree<V, T>([&](int k) { return h[k]; });
            if (P == 2) p += __shfl_xor_sync(0xffffffffu, p, 1);
            if (edge && k0 == 0) s_out[y == 0 ? 0 : 1][iy] = p;
        }
    };
    auto density = [&] { return (T)tree<HALF, double>([&](int i) { return s_out[up ? 0 : 1][up ? i : M - HALF + i]; }); };
    // sums over a cell's threads of v, xi_x v and xi_y v
    auto sums = [&](const T (&v)[V], T &rho, T &jx, T &jy) {
        const T R = tree<V, T>([&](int k) { return v[k]; });
        const T X = tree<V, T>([&](int k) { return xi[k] * v[k]; });
        if (act) {
            s_m[cl * S + s] = R;
            s_m[(nc + cl) * S + s] = X;
            s_j[cl * S + s] = (double)xiy * (double)R;
        }
        __syncthreads();
        const int q = s / NG, g = s - q * NG;
        if (act && (GS > 1 ? q < 3 : true)) {
            if (GS == 1) {                         // three threads a cell: no first stage
                if (s == 0) s_mt[cl * 2] = s_m[cl * S] + s_m[cl * S + 1] + s_m[cl * S + 2];
                if (s == 1) s_mt[cl * 2 + 1] = s_m[(nc + cl) * S] + s_m[(nc + cl) * S + 1] + s_m[(nc + cl) * S + 2];
                if (s == 2) s_jt[cl] = s_j[cl * S] + s_j[cl * S + 2];
            } else if (q < 2) {
                const T *p = s_m + (size_t)(q * nc + cl) * S + g * GS;
                s_mg[(q * nc + cl) * NG + g] = tree<GS, T>([&](int k) { return p[k]; });
            } else {
                const double *p = s_j + (size_t)cl * S + g * GS;
                s_jg[cl * NG + g] = tree<GS, double>([&](int k) { return p[k]; });
            }
        }
        __syncthreads();
        if (GS > 1) {
            if (act && s < 2) {
                const T *p = s_mg + (size_t)(s * nc + cl) * NG;
                s_mt[cl * 2 + s] = tree<NG, T>([&](int k) { return p[k]; });
            } else if (act && s == 2) {
                const double *p = s_jg + (size_t)cl * NG;
                s_jt[cl] = tree<NG, double>([&](int k) { return p[k]; });
            }
            __syncthreads();
        }
        rho = act ? s_mt[cl * 2] : T(0);
        jx = act ? s_mt[cl * 2 + 1] : T(0);
        jy = act ? (T)s_jt[cl] : T(0);
    };

    leave();
    __syncwarp();
    cluster_wait();                                // every CTA of the cluster runs: its shared memory may be written
    publish(0);
    T psd = 0, psn = 0;
    for (int n = 0; n < steps; ++n) {
        const int b = n & 1;
        const T *nb = s_v + ((size_t)b * (nc + 2) + (act ? (up ? cl : down ? cl + 2 : cl + 1) : 0)) * NV + iy * M + k0;
        if (wall) rho_w = density();
        T v[V];
#pragma unroll
        for (int k = 0; k < V; ++k) {
            if (DP) {
                const T op = wall ? rho_w : nb[k];
                v[k] = c1[k] * op + (a0 * h[k] + c0[k]);
            } else {
                const T op = wall ? c1[k] * rho_w + c0[k] : nb[k];
                v[k] = h[k] + nuy * (op - h[k]);
            }
        }
        T rho, jx, jy;
        sums(v, rho, jx, jy);
        const T q = DP ? omw * rho + xo * jy : omw * (rho + xiy * jy), jj = omw * jx;
        const bool last = resid && n == steps - 1;
#pragma unroll
        for (int k = 0; k < V; ++k) {
            T o;
            if (DP) {
                if (!a.fold) v[k] *= (T)a.b;
                o = w[k] * q + (wxi[k] * jj + v[k]);
            } else {
                o = (T)a.b_f * v[k] + w[k] * (q + xi[k] * jj);
            }
            if (last) {
                const T d = o - h[k];
                psd += d * d;
                psn += o * o;
            }
            h[k] = o;
        }
        if (n + 1 < steps) {
            leave();
            publish(b ^ 1);
        }
    }
    T *dst = static_cast<T *>(a.hn) + (size_t)(iy * M + k0) * plane + y;
    if (on)
#pragma unroll
        for (int k = 0; k < V; ++k) dst[k * plane] = h[k];
    if (resid) {
        double d = on ? (double)psd : 0.0, e = on ? (double)psn : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            d += __shfl_xor_sync(0xffffffffu, d, o);
            e += __shfl_xor_sync(0xffffffffu, e, o);
        }
        if ((t & 31) == 0) {
            s_red[t >> 5] = d;
            s_red[32 + (t >> 5)] = e;
        }
        __syncthreads();
        if (t == 0) {
            for (int k = 1; k < (int)blockDim.x / 32; ++k) {
                d += s_red[k];
                e += s_red[32 + k];
            }
            a.partials[2 * blockIdx.x] = d;
            a.partials[2 * blockIdx.x + 1] = e;
        }
    }
    // no CTA leaves while a neighbour may still write into it
    __syncwarp();
    cluster_arrive();
    cluster_wait();
}

template <typename T, int M>
void column_config(int ny, cudaLaunchConfig_t &cfg, cudaLaunchAttribute *at)
{
    const int nc = (ny + CLUSTER - 1) / CLUSTER;
    std::memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3(CLUSTER);
    cfg.blockDim = dim3((nc * Shape<M>::S + 31) / 32 * 32);
    cfg.dynamicSmemBytes = column_smem<T, M>(nc);
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CLUSTER;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
}

// whether the device runs a cluster of this channel; opts the kernel into its launch shape
template <typename T, int M>
bool prepare(int ny)
{
    const int nc = (ny + CLUSTER - 1) / CLUSTER;
    if (nc * Shape<M>::S > 1024) return false;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    column_config<T, M>(ny, cfg, at);
    int n = 0;
    const bool ok = cudaFuncSetAttribute(column_kernel<T, M>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                    cudaFuncSetAttribute(column_kernel<T, M>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024) == cudaSuccess &&
                    cfg.dynamicSmemBytes <= 160 * 1024 &&
                    cudaOccupancyMaxActiveClusters(&n, column_kernel<T, M>, &cfg) == cudaSuccess && n >= 1;
    if (!ok) cudaGetLastError();
    return ok;
}

template <typename T, int M>
cudaError_t launch(const StepArgs &a, int steps, int resid, cudaStream_t s)
{
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    column_config<T, M>(a.ny, cfg, at);
    cfg.stream = s;
    return cudaLaunchKernelEx(&cfg, column_kernel<T, M>, a, (a.ny + CLUSTER - 1) / CLUSTER, steps, resid);
}

}  // namespace

int column_blocks() { return CLUSTER; }

bool prepare_column(bool dp, int m, int ny)
{
    switch (m) {
    case 3: return dp ? prepare<double, 3>(ny) : prepare<float, 3>(ny);
    case 4: return dp ? prepare<double, 4>(ny) : prepare<float, 4>(ny);
    case 6: return dp ? prepare<double, 6>(ny) : prepare<float, 6>(ny);
    case 8: return dp ? prepare<double, 8>(ny) : prepare<float, 8>(ny);
    case 12: return dp ? prepare<double, 12>(ny) : prepare<float, 12>(ny);
    default: return false;
    }
}

cudaError_t launch_column(bool dp, int m, const StepArgs &a, int steps, int resid, cudaStream_t s)
{
    switch (m) {
    case 3: return dp ? launch<double, 3>(a, steps, resid, s) : launch<float, 3>(a, steps, resid, s);
    case 4: return dp ? launch<double, 4>(a, steps, resid, s) : launch<float, 4>(a, steps, resid, s);
    case 6: return dp ? launch<double, 6>(a, steps, resid, s) : launch<float, 6>(a, steps, resid, s);
    case 8: return dp ? launch<double, 8>(a, steps, resid, s) : launch<float, 8>(a, steps, resid, s);
    case 12: return dp ? launch<double, 12>(a, steps, resid, s) : launch<float, 12>(a, steps, resid, s);
    default: return cudaErrorInvalidValue;
    }
}
