// Fused time step on the planar state, any grid (sm_103a): the kernel of load paths 0 and 1
// and of the refinement (defect and correction steps).
//
// One launch = one step of the paper's fully discrete scheme (Ghiroldi & Gibelli,
// arXiv:1308.0692, Eqs. 1, 5-9): first-order upwind transport with the Maxwell diffuse-wall
// ghosts, then relaxation towards w_a (rho + xi_a . j), wall cells included.
//
// Work decomposition.  A block holds W x R cells -- W consecutive places of a row-major walk
// over columns of R rows, R rows each, so any nx fills the lanes -- times NS velocity slices:
// thread (x, y, z) = (place, slice, row) owns the M / NS velocity rows iy of its slice of one
// cell.  W and R are launch dimensions (blockDim), M and NS template parameters.  A lane
// loads the own value and the two upwind neighbours of each of its velocities (the neighbours
// of other lanes and of the row above come from L1), keeps the transported values in
// registers and exchanges the moments through shared memory in a fixed order.
//
// Walls.  Blocks that hold a wall cell (block-uniform) also form Eq. 9's wall densities from
// the own values already in registers -- products and sums within a velocity row in the
// arithmetic type, across rows and slices in FP64 -- and take a copy of the transport loop
// that puts Eq. 8's ghost in the upwind place.
//
// FP64 arithmetic.  GB300 retires about two FP64 lanes per cycle and SM, so the FP64 form
// counts its operations, seven per velocity and a few per row: transport as
// s [(1 - nu_x - nu_y) h + nu_x h_x + nu_y h_y] with s = 1 - omega (three, the coefficients host
// tables), two for the moment sums, two for the relaxation, which only adds
// w_x q + w_x xi_x J to the scaled transported value.  (Where 1 - omega is below 1/16, s = 1 and
// the factor is applied after the moments.)  The FP32 form
// keeps h + nu_x (h_x - h) + nu_y (h_y - h), which moves a constant state without rounding.
#pragma once

#include <type_traits>

#include "step_kernel.cuh"

namespace lbmk {

// cells of a block: W * R at most
template <int NS>
__host__ __device__ constexpr int tile_cells() { return NS >= 6 ? 32 : 64; }

template <typename TS, typename TC, int M, int NS, bool RESID, bool SOURCE, bool DEFECT, bool WIDE = false>
__global__ void __launch_bounds__(tile_cells<NS>() * NS) step_tile_kernel(const __grid_constant__ StepArgs a)
{
    constexpr int RPL = M / NS, HALF = M / 2, CELLS = tile_cells<NS>();
    constexpr bool ACC = RESID || DEFECT;
    constexpr bool DP = sizeof(TC) == 8;
    constexpr bool TWO = DP && NS >= 4;       // moments summed by three slices, then read back
    static_assert(M % NS == 0, "slices must divide the velocity rows");
    __shared__ TC s_mom[3][NS][CELLS];
    __shared__ double s_wall[4][NS][CELLS];
    __shared__ TC s_tot[TWO ? 3 : 1][CELLS];
    __shared__ double s_red[2][(CELLS * NS + 31) / 32];

    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    const int W = blockDim.x, g = threadIdx.y;
    const int cl = threadIdx.x + W * threadIdx.z;
    const int nx = a.nx, ny = a.ny;
    const long ncells = a.ncells;
    const unsigned ncol = (unsigned)nx * (unsigned)((ny + (int)blockDim.z - 1) / (int)blockDim.z);
    const unsigned place = blockIdx.x * (unsigned)W + threadIdx.x;
    const unsigned col = place < ncol ? place : ncol - 1;
    const unsigned Y = col / (unsigned)nx;
    const int x = (int)(col - Y * (unsigned)nx);
    const int yr = (int)(Y * blockDim.z + threadIdx.z);
    const int y = yr < ny ? yr : ny - 1;      // lanes past the grid mirror a cell and store nothing
    const bool valid = place < ncol && yr < ny;
    const bool cav = a.cavity != 0;
    const bool wl = cav && x == 0, wr = cav && x == nx - 1, wb = y == 0, wt = y == ny - 1;
    const long c = (long)y * nx + x;
    const long dl = x > 0 ? -1 : (cav ? 0 : nx - 1);          // periodic in Couette
    const long dr = x < nx - 1 ? 1 : (cav ? 0 : 1 - nx);
    const long dn = y > 0 ? -(long)nx : 0, up = y < ny - 1 ? nx : 0;
    const bool walls = __syncthreads_or((int)(wl || wr || wb || wt)) != 0;

    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    const TS *hp = reinterpret_cast<const TS *>(a.h) + (long)(g * RPL * M) * ncells + c;
    TC hs[RPL * M];
#pragma unroll
    for (int k = 0; k < RPL * M; ++k) hs[k] = (TC)hp[k * ncells];
    // the source beside them: read where it is added, its latency stood after the moment exchange
    [[maybe_unused]] TC sv[SOURCE ? RPL * M : 1];
    if constexpr (SOURCE) {
        const TS *hsrc = reinterpret_cast<const TS *>(a.src) + (long)(g * RPL * M) * ncells + c;
#pragma unroll
        for (int k = 0; k < RPL * M; ++k) sv[k] = (TC)hsrc[k * ncells];
    }

    // ---- wall densities of the faces this cell touches (Eq. 9) ----
    TC rb = 0, rt = 0, rl = 0, rr = 0;
    if (walls) {
        double sb = 0.0, st = 0.0, sl = 0.0, sr = 0.0;
        if (wb || wt) {
#pragma unroll
            for (int r = 0; r < RPL; ++r) {
                const int iy = g * RPL + r;
                TC sum = 0;
#pragma unroll
                for (int ix = 0; ix < M; ++ix) sum += hs[r * M + ix];
                if (iy < HALF) sb -= a.xi[iy] * (double)sum;
                if (iy >= M - HALF) st += a.xi[iy] * (double)sum;
            }
        }
        if (wl) {
#pragma unroll
            for (int r = 0; r < RPL; ++r) {
                TC sum = 0;
#pragma unroll
                for (int ix = 0; ix < HALF; ++ix) sum -= pick<TC>(a.xi, a.xi_f, ix) * hs[r * M + ix];
                sl += (double)sum;
            }
        }
        if (wr) {
#pragma unroll
            for (int r = 0; r < RPL; ++r) {
                TC sum = 0;
#pragma unroll
                for (int ix = M - HALF; ix < M; ++ix) sum += pick<TC>(a.xi, a.xi_f, ix) * hs[r * M + ix];
                sr += (double)sum;
            }
        }
        if (NS > 1) {
            s_wall[0][g][cl] = sb;
            s_wall[1][g][cl] = st;
            s_wall[2][g][cl] = sl;
            s_wall[3][g][cl] = sr;
            __syncthreads();
            auto total = [&](int f) {
                double t = 0.0;
#pragma unroll
                for (int q = 0; q < NS; ++q) t += s_wall[f][q][cl];
                return t;
            };
            if (wb) sb = total(0);
            if (wt) st = total(1);
            if (wl) sl = total(2);
            if (wr) sr = total(3);
        }
        rb = (TC)(sb * a.inv_dy_wall);
        rt = (TC)(st * a.inv_dy_wall);
        rl = (TC)(sl * a.inv_dx_wall);
        rr = (TC)(sr * a.inv_dx_wall);
    }

    // ---- transport (upwind) + moment sums, transported values in registers ----
    TC rho = 0, jx = 0, jy = 0;
    auto transport = [&](auto xwalls_tag, auto ywalls_tag) {
        constexpr bool XW = decltype(xwalls_tag)::value, YW = decltype(ywalls_tag)::value;
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
            const int iy = g * RPL + r;
            const bool ypos = iy >= M - HALF, yneg = iy < HALF;
            const long dy = ypos ? dn : (yneg ? up : 0);
            const TC nuy = pick<TC>(a.nuy_s, a.nuy_f, iy), wy = pick<TC>(a.w1, a.w1_f, iy);
            const bool ywall = YW && ((ypos && wb) || (yneg && wt));
            TC gy0 = 0, gy1 = 0;                       // ghost w_x (gy0 + xi_x gy1) of a y wall
            if (YW) {
                const TC d = ypos ? rb : rt, u = (TC)(ypos ? a.u_bottom : a.u_top);
                const TC drive = a.homogeneous ? TC(0) : (TC)((ypos ? a.u_bottom : a.u_top) * a.inv_u_ref);
                gy0 = wy * d;
                gy1 = wy * (d * u + drive);
            }
            TC R = 0;
            [[maybe_unused]] TC X = 0;                 // FP32: the row's sum first
            // a row's upwind values ahead of its arithmetic (FP32: 300 x 250, M = 6, 7.1 to 6.0 us a step;
            // M = 12 loses by its registers, 6.6 to 7.8).  WIDE: at the side walls too, which pays on
            // grids of many cells (333 x 251, M = 8: three at once 8.9 us a step each against 9.5) but not
            // on small ones (128^2 4.4 against 3.9)
            constexpr bool AHEAD = !DP && !YW && (!XW || WIDE) && M <= 8;
            [[maybe_unused]] TC hxr[M], hyr[M];
            if constexpr (AHEAD) {
#pragma unroll
                for (int ix = 0; ix < M; ++ix) {
                    const TS *hv = hp + (long)(r * M + ix) * ncells;
                    hyr[ix] = (TC)hv[dy];
                    if (ix >= M - HALF || ix < HALF) hxr[ix] = (TC)hv[ix >= M - HALF ? dl : dr];
                }
            }
#pragma unroll
            for (int ix = 0; ix < M; ++ix) {
                const TS *hv = hp + (long)(r * M + ix) * ncells;
                const TC hc = hs[r * M + ix], xix = pick<TC>(a.xi, a.xi_f, ix), wx = pick<TC>(a.w1, a.w1_f, ix);
                TC hx = hc, hy;
                if constexpr (AHEAD) {
                    hy = hyr[ix];
                    if (ix >= M - HALF || ix < HALF) hx = hxr[ix];
                    if (XW && ix >= M - HALF && wl) hx = wx * (wy * rl);
                    if (XW && ix < HALF && wr) hx = wx * (wy * rr);
                } else {
                    hy = (TC)hv[dy];
                    if (ix >= M - HALF) hx = (XW && wl) ? wx * (wy * rl) : (TC)hv[dl];
                    else if (ix < HALF) hx = (XW && wr) ? wx * (wy * rr) : (TC)hv[dr];
                    if (YW && ywall) hy = wx * (gy0 + xix * gy1);
                }
                TC v;
                if constexpr (DP) {
                    v = a.a0[iy * M + ix] * hc;
                    if (ix >= M - HALF || ix < HALF) v += a.nux_s[ix] * hx;
                    v += nuy * hy;
                } else {
                    v = hc;
                    if (ix >= M - HALF || ix < HALF) v += a.nux_f[ix] * (hx - hc);
                    v += nuy * (hy - hc);
                }
                hs[r * M + ix] = v;
                R += v;
                if constexpr (DP) jx += xix * v;
                else X += xix * v;
            }
            rho += R;
            if constexpr (!DP) jx += X;
            jy += pick<TC>(a.xi, a.xi_f, iy) * R;
        }
    };
    if (!walls) transport(std::false_type{}, std::false_type{});
    else if (__any_sync(__activemask(), wb || wt)) transport(std::true_type{}, std::true_type{});
    else transport(std::true_type{}, std::false_type{});   // no y ghosts at a side wall
    if (NS > 1) {
        s_mom[0][g][cl] = rho;
        s_mom[1][g][cl] = jx;
        s_mom[2][g][cl] = jy;
        __syncthreads();
        if constexpr (TWO) {
            if (g < 3) {
                TC t = 0;
#pragma unroll
                for (int q = 0; q < NS; ++q) t += s_mom[g][q][cl];
                s_tot[g][cl] = t;
            }
            __syncthreads();
            rho = s_tot[0][cl];
            jx = s_tot[1][cl];
            jy = s_tot[2][cl];
        } else {
            rho = jx = jy = 0;
#pragma unroll
            for (int q = 0; q < NS; ++q) {
                rho += s_mom[0][q][cl];
                jx += s_mom[1][q][cl];
                jy += s_mom[2][q][cl];
            }
        }
    }

    // ---- relaxation, store, residual ----
    TC psd = 0, psn = 0;
    if (DP && !a.fold)
#pragma unroll
        for (int k = 0; k < RPL * M; ++k) hs[k] *= (TC)a.b;
    TS *hn = reinterpret_cast<TS *>(a.hn) + (long)(g * RPL * M) * ncells + c;
#pragma unroll
    for (int r = 0; r < RPL; ++r) {
        const int iy = g * RPL + r;
        const TC wom = DP ? (TC)a.omw[iy] : (TC)(a.omega_f * a.w1_f[iy]);
        const TC q = wom * (rho + pick<TC>(a.xi, a.xi_f, iy) * jy);
        const TC jj = wom * jx;
        auto put = [&](int ix, TC v) {
            const long off = (long)(r * M + ix) * ncells;
            if constexpr (SOURCE) v += sv[r * M + ix];
            if (ACC) {
                const TC d = v - (TC)hp[off];
                psd += d * d;
                psn += v * v;
                if (DEFECT) v = d;
            }
            if (valid) hn[off] = (TS)v;
        };
        if constexpr (DP) {
#pragma unroll
            for (int ix = 0; ix < M; ++ix) {
                TC v = a.w1[ix] * q + hs[r * M + ix];
                if (2 * ix + 1 != M) v += a.wxi[ix] * jj;      // xi = 0 in the middle of an odd set
                put(ix, v);
            }
        } else {
#pragma unroll
            for (int ix = 0; ix < M; ++ix) put(ix, a.b_f * hs[r * M + ix] + a.w1_f[ix] * (q + a.xi_f[ix] * jj));
        }
    }

    if (ACC) {
        // fixed order: the lanes of each warp by a butterfly, then the warps (one FP64 operation
        // of one lane costs the pipe as much as a warp's)
        const int T = W * NS * blockDim.z, t = threadIdx.x + W * (g + NS * threadIdx.z);
        const int lanes = T - (t & ~31) < 32 ? T - (t & ~31) : 32;
        const unsigned mask = lanes == 32 ? 0xffffffffu : (1u << lanes) - 1;
        double d = valid ? (double)psd : 0.0, n = valid ? (double)psn : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double dd = __shfl_down_sync(mask, d, o), dnn = __shfl_down_sync(mask, n, o);
            if (o < lanes) {
                const bool in = (t & 31) + o < lanes;
                d += in ? dd : 0.0;
                n += in ? dnn : 0.0;
            }
        }
        if ((t & 31) == 0) {
            s_red[0][t >> 5] = d;
            s_red[1][t >> 5] = n;
        }
        __syncthreads();
        if (t == 0) {
            for (int k = 1; 32 * k < T; ++k) {
                d += s_red[0][k];
                n += s_red[1][k];
            }
            a.partials[2 * (long)blockIdx.x] = d;
            a.partials[2 * (long)blockIdx.x + 1] = n;
        }
    }
}

// One step, launched so that the next step's blocks may be set up while this one runs (they
// wait for it before reading the state).
template <typename TS, typename TC, int M, int NS, bool RESID, bool SOURCE, bool DEFECT>
cudaError_t launch_tile(const StepArgs &a, cudaStream_t s)
{
    const int W = a.tile_w, R = a.tile_r;
    if (W < 1 || R < 1 || W * R > tile_cells<NS>()) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)tile_blocks(a.nx, a.ny, W, R));
    cfg.blockDim = dim3(W, NS, R);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = s != nullptr ? 1 : 0;
    // 32 places a block: a large grid (tile_plan)
    constexpr bool HAS = sizeof(TC) == 4 && !SOURCE && ((M == 4 && NS == 1) || (M == 6 && NS == 2) || (M == 8 && NS == 4));
    if (HAS && W == 32) return cudaLaunchKernelEx(&cfg, step_tile_kernel<TS, TC, M, NS, RESID, SOURCE, DEFECT, HAS>, a);
    return cudaLaunchKernelEx(&cfg, step_tile_kernel<TS, TC, M, NS, RESID, SOURCE, DEFECT>, a);
}

}  // namespace lbmk
