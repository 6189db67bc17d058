// Kernels of the single-cavity path: the fused collide-and-stream step, the
// observables pass with its FP64 reductions and the Nusselt number, the state
// export, and the porosity conversion.
#include <algorithm>

#include "lbm_internal.h"

namespace lbm {

// ---- fused step -------------------------------------------------------------------

// One time step for every node, pull form: each thread gathers the post-
// collision populations that stream into its node (Eq. 18, 35), applies the
// wall rule on perimeter nodes (Section 4), collides (Eq. 17, 34) and writes
// the node's post-collision populations to the other buffer.  The buffer
// pair alternates, so dst holds B_{n+1} when src holds B_n.
//
// Launched as a programmatic dependent of the previous step (back-to-back
// steps of small lattices), a block starts while that step drains and waits
// here until it has completed and its writes are visible: the step reads the
// whole previous lattice and rewrites the buffer the previous step read.
// Without that launch attribute the wait returns at once.
__device__ __forceinline__ void wait_for_previous_step() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// OBS: an observing step, which also stores the temperatures of the node
// columns next to the vertical walls into obs (obs_put) for the Nusselt
// number of the new state; otherwise obs is unused.
//
// FP32 and FP64 storage (Core<T>): the blocks from column `cols` of the grid on
// take the border's nodes one per thread, the others rows of fluid nodes only
// (see border_node).  Measured against rows that hold the walls too, us per
// step: FP64 257^2 31 -> 26, 512^2 92 -> 75, FP32 601 x 397 4.8 -> 4.3.  FP16 flow storage: no such
// columns, every block takes what it meets.
//
// On a lattice far larger than the cache (cols < 0; FP32) a row of blocks takes
// the border nodes of its own rows, and the first and last rows of blocks the
// y walls: a border node shares 32-byte sectors with its row, which otherwise
// reach memory twice.  One step per launch, us: 2048^2 74.9 -> 72.0, 4096^2 282.7 -> 275.1.
template <class T, bool FIELD, bool OBS, bool PAIRS>
__device__ __forceinline__ void step_border(const Src<T>& src, const Dst<T>& dst, const typename T::P* __restrict__ phi,
                                            const Geom& gm, const CoefOf<T>& c, int* __restrict__ status,
                                            double* __restrict__ obs, int cols) {
    const int threads = blockDim.x * blockDim.y, t = threadIdx.y * blockDim.x + threadIdx.x;
    int x, y;
    if (PAIRS && cols < 0) {
        const int nbc = border_columns<PAIRS>(gm.nx), own = nbc * (int)blockDim.y, j = blockIdx.y;
        if (t < own) {
            const int r = t / nbc, col = t - r * nbc;
            y = 1 + j * (int)blockDim.y + r;
            if (y >= gm.ny - 1) return;
            x = col < 2 ? col : gm.nx - nbc + col;
        } else {
            const int m = threads - own, last = (int)gridDim.y - (gm.nx + m - 1) / m;
            if (j >= last) {
                x = (j - last) * m + t - own;
                y = gm.ny - 1;
            } else {
                x = j * m + t - own;
                y = 0;
            }
            if (x >= gm.nx) return;
        }
    } else {
        const int b = ((blockIdx.x - cols) * gridDim.y + blockIdx.y) * threads + t;
        if (b >= border_count<PAIRS>(gm.nx, gm.ny)) return;
        border_node<PAIRS>(b, gm.nx, gm.ny, x, y);
    }
    update_node<T, FIELD, OBS>(c, gm, src, dst, phi, x, y, status, obs);
}

template <class T, bool FIELD, bool OBS>
__global__ void __launch_bounds__(256) k_step(Src<T> src, Dst<T> dst, const typename T::P* __restrict__ phi,
                                              Geom gm, CoefOf<T> c, int* __restrict__ status,
                                              double* __restrict__ obs, int cols) {
    wait_for_previous_step();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if constexpr (Core<T>::value) {
        if ((int)blockIdx.x >= cols) {
            step_border<T, FIELD, OBS, false>(src, dst, phi, gm, c, status, obs, cols);
            return;
        }
        const int y = 1 + blockIdx.y * blockDim.y + threadIdx.y;
        if (x == 0 || x >= gm.nx - 1 || y >= gm.ny - 1) return;
        update_fluid<T, FIELD, OBS>(c, gm, src, dst, phi, x, y, status, obs);
    } else {
        const int y = blockIdx.y * blockDim.y + threadIdx.y;
        if (x >= gm.nx || y >= gm.ny) return;
        update_node<T, FIELD, OBS>(c, gm, src, dst, phi, x, y, status, obs);
    }
}

// Blocks of 256 threads per SM that the two-node kernels are compiled for (see k_step2).
template <class T> constexpr int step_blocks() {
    return sizeof(typename T::R) == 8 ? 1 : sizeof(typename T::SF) == 4 ? 3 : 4;
}

// Two nodes per thread, (x, y) and (x, y + blockDim.y): all 28 loads are issued
// before any arithmetic, doubling the bytes in flight per thread (the FP16-flow
// variant moves 38 B per node, too few to cover HBM latency with one node per
// thread).
// FP32 storage: at most 80 registers (3 blocks of 256 threads, 6 of 128 per
// SM), where the paired collision spills nothing (140 bytes under 64).  Measured
// at 4096^2 / 1024^2 / 512^2 / 200^2: 273.7 / 17.7 / 5.5 / 3.1 us per step, under
// 64 registers 310.7 / 22.8 / 7.3 / 3.7, with the collision before this form 274.7 /
// 20.1 / 7.2 / 4.4.  FP16 flow: at most 64 (4 blocks), which its direct form fits.
// FP64 would spill under either limit.
template <class T, bool FIELD, bool OBS>
__global__ void __launch_bounds__(256, step_blocks<T>())
    k_step2(Src<T> src, Dst<T> dst, const typename T::P* __restrict__ phi, Geom gm, CoefOf<T> c,
            int* __restrict__ status, double* __restrict__ obs, int cols) {
    wait_for_previous_step();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if constexpr (Core<T>::value) {
        if ((int)blockIdx.x >= cols) {
            step_border<T, FIELD, OBS, false>(src, dst, phi, gm, c, status, obs, cols);
            return;
        }
        const int y0 = 1 + blockIdx.y * (2 * blockDim.y) + threadIdx.y, y1 = y0 + blockDim.y;
        if (x == 0 || x >= gm.nx - 1 || y0 >= gm.ny - 1) return;
        if (y1 < gm.ny - 1)
            update_pair<T, FIELD, OBS>(c, gm, src, dst, phi, x, y0, true, x, y1, true, status, obs);
        else
            update_fluid<T, FIELD, OBS>(c, gm, src, dst, phi, x, y0, status, obs);
    } else {
        const int y0 = blockIdx.y * (2 * blockDim.y) + threadIdx.y;
        const int y1 = y0 + blockDim.y;
        if (x >= gm.nx || y0 >= gm.ny) return;
        update_pair<T, FIELD, OBS>(c, gm, src, dst, phi, x, y0, true, x, y1, y1 < gm.ny, status, obs);
    }
}

// Two nodes per thread side by side, (x0, y) and (x0 + 1, y) with x0 even:
// the populations with e_x = 0 are loaded, and every population stored, as
// aligned pairs (8-byte FP32, 4-byte FP16 accesses), a third fewer memory
// instructions than two nodes apart along y.  Same register cap.
template <class T, bool FIELD, bool OBS>
__global__ void __launch_bounds__(256, step_blocks<T>())
    k_step2x(Src<T> src, Dst<T> dst, const typename T::P* __restrict__ phi, Geom gm, CoefOf<T> c,
             int* __restrict__ status, double* __restrict__ obs, int cols) {
    wait_for_previous_step();
    const int x0 = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    if constexpr (Core<T>::value) {
        if ((int)blockIdx.x >= abs(cols)) {
            step_border<T, FIELD, OBS, true>(src, dst, phi, gm, c, status, obs, cols);
            return;
        }
        const int y = 1 + blockIdx.y * blockDim.y + threadIdx.y;
        if (x0 == 0 || x0 + 1 >= gm.nx - 1 || y >= gm.ny - 1) return;
        update_fluid_xpair<T, FIELD, OBS>(c, gm, src, dst, phi, x0, y, status, obs);
    } else {
        const int y = blockIdx.y * blockDim.y + threadIdx.y;
        if (x0 >= gm.nx || y >= gm.ny) return;
        update_xpair<T, FIELD, OBS>(c, gm, src, dst, phi, x0, y, status, obs);
    }
}

// ---- observables ------------------------------------------------------------------

// Observables of the post-stream state S_n, rebuilt by pulling from B_{n-1}
// and applying the wall rule: the macroscopic fields, and FP64 max|u|, max|u -
// u_prev|, sum of population deviations, sum of T - T0, and both mean Nusselt
// numbers (Eq. 38): Nu(y) = -L dT/dx / dT, trapezoidal mean over y.
//
// The first `nodes` blocks take the nodes, the others the rows of the Nusselt
// numbers; each leaves four partial results, and the last block to finish folds
// them in a fixed order (the grid depends on the lattice's size alone, so the
// sums are reproducible) and re-arms the counter.
// out[0..6] = nu_hot, nu_cold, max|u|, max|du|, sum d, sum (T - T0), status.
//
// FP64 is scarce (an SM retires two lanes per cycle), so a node spends four FP64
// operations, those of the two sums: maxima are kept as integers, and of |du|
// the square, which is formed in FP64 only where an FP32 estimate does not rule
// it out.  64^2: 17 us, against 27 + 38 in two kernels with an FP64 butterfly in
// every warp and an FP64 root per node; 1024^2: 59 us against 87 + 77.
template <class T, bool FIELD>
__global__ void __launch_bounds__(256)
    k_observe(Src<T> prev, const typename T::P* __restrict__ phi, Geom gm, CoefOf<T> c,
              typename T::R* ux_out, typename T::R* uy_out, typename T::R* T_out, typename T::R* p_out,
              typename T::R* snap, int snap_valid, double* __restrict__ partials, int nodes, double L, double dT,
              const int* __restrict__ status, unsigned* __restrict__ counter, double* __restrict__ out) {
    using R = typename T::R;
    __shared__ double sh[4][256];
    __shared__ bool last;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    if ((int)blockIdx.x < nodes) {
        const unsigned n = (unsigned)gm.nx * (unsigned)gm.ny, stride = (unsigned)nodes * 256u;
        decltype(order_bits(R(0))) umax = 0;
        double du2 = 0.0;  // max |u - u_prev|^2
        float ruled = -1.f;  // FP32 estimates up to this are below it
        for (unsigned k = blockIdx.x * 256u + threadIdx.x; k < n; k += stride) {
            const int y = (int)(k / (unsigned)gm.nx), x = (int)(k - (unsigned)y * (unsigned)gm.nx);
            R d[9], h[5];
            Drag<R> dr;
            const Macro<R> mc = node_state<T, FIELD>(c, gm, prev, phi, x, y, dr, d, h);
            R sd = R(0);
#pragma unroll
            for (int i = 0; i < 9; ++i) sd += d[i];
            if (ux_out) ux_out[k] = mc.ux;
            if (uy_out) uy_out[k] = mc.uy;
            if (T_out) T_out[k] = c.T0 + mc.dT;
            if (p_out) p_out[k] = (R(1.0 / 3.0) + mc.dP) * dr.iphi;
            if (snap) {
                if (snap_valid) {
                    const R bx = snap[2 * (size_t)k], by = snap[2 * (size_t)k + 1];
                    float e2 = 0.f;
                    if constexpr (sizeof(R) == 4) e2 = (mc.ux - bx) * (mc.ux - bx) + (mc.uy - by) * (mc.uy - by);
                    if (!(e2 <= ruled)) {  // (a NaN gets through; FP64 lattices: always)
                        const double ax = (double)mc.ux - (double)bx, ay = (double)mc.uy - (double)by;
                        const double a2 = ax * ax + ay * ay;
                        if (a2 > du2 || a2 != a2) {
                            du2 = a2;
                            if (sizeof(R) == 4 && a2 > 1e-30) ruled = (float)a2 * 0.99999f;
                        }
                    }
                }
                snap[2 * (size_t)k] = mc.ux;
                snap[2 * (size_t)k + 1] = mc.uy;
            }
            umax = max(umax, order_bits(mc.umag));
            v[2] += (double)sd;
            v[3] += (double)mc.dT;
        }
        v[0] = from_order(umax);
        v[1] = du2;
    } else {
        const int blocks = gridDim.x - nodes;
        for (int y = (blockIdx.x - nodes) * 256 + threadIdx.x; y < gm.ny; y += blocks * 256) {
            double tl[5], tr[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                tl[k] = (double)node_dT<T>(c, gm, prev, k, y);
                tr[k] = (double)node_dT<T>(c, gm, prev, gm.nx - 1 - k, y);
            }
            const double wt = (y == 0 || y == gm.ny - 1) ? 0.5 : 1.0;
            v[2] += wt * slope_hot(tl);
            v[3] += wt * slope_cold(tr);
        }
    }
    fold_block(v, sh);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < 4; ++k) partials[blockIdx.x * 4 + k] = v[k];
        __threadfence();
        last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double w[4] = {0.0, 0.0, 0.0, 0.0}, nu[4] = {0.0, 0.0, 0.0, 0.0};
    for (unsigned b = threadIdx.x; b < gridDim.x; b += 256) {
        const double p0 = __ldcg(partials + 4 * b), p1 = __ldcg(partials + 4 * b + 1);
        const double p2 = __ldcg(partials + 4 * b + 2), p3 = __ldcg(partials + 4 * b + 3);
        if (b < (unsigned)nodes) {
            w[0] = order_bits(p0) > order_bits(w[0]) ? p0 : w[0];
            w[1] = order_bits(p1) > order_bits(w[1]) ? p1 : w[1];
            w[2] += p2;
            w[3] += p3;
        } else {
            nu[2] += p2;
            nu[3] += p3;
        }
    }
    fold_block(w, sh);
    __syncthreads();
    fold_block(nu, sh);
    if (threadIdx.x == 0) {
        const double scale = -L / (12.0 * dT) / (double)(gm.ny - 1);
        out[0] = nu[2] * scale;
        out[1] = nu[3] * scale;
        out[2] = w[0];
        out[3] = sqrt(w[1]);
        out[4] = w[2];
        out[5] = w[3];
        out[6] = (double)(*status);
        *counter = 0u;
    }
}

// Row-parallel mean Nusselt numbers (Eq. 38): one thread per wall row in
// one-warp blocks (so the rows' scattered loads spread over many SMs), warp
// sums into partials; the last block to finish folds the partials in a fixed
// order (deterministic), writes out[0..1] and re-arms the counter.  OBS: the
// temperatures come from the wall columns the step before stored (obs_dT),
// else they are pulled from B_{n-1} (node_dT); both give the same values.
template <class T, bool OBS>
__global__ void __launch_bounds__(32) k_nusselt_rows(Src<T> prev, const double* __restrict__ obs, Geom gm,
                                                     CoefOf<T> c, double L, double dT,
                                                     double* __restrict__ partials, unsigned* __restrict__ counter,
                                                     double* __restrict__ out) {
    __shared__ bool last;
    double a = 0.0, b = 0.0;
    const int y = blockIdx.x * blockDim.x + threadIdx.x;
    if (y < gm.ny) {
        double tl[5], tr[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            if constexpr (OBS) {
                tl[k] = obs_dT<T>(c, gm, obs, k, y);
                tr[k] = obs_dT<T>(c, gm, obs, 5 + k, y);
            } else {
                tl[k] = (double)node_dT<T>(c, gm, prev, k, y);
                tr[k] = (double)node_dT<T>(c, gm, prev, gm.nx - 1 - k, y);
            }
        }
        const double wt = (y == 0 || y == gm.ny - 1) ? 0.5 : 1.0;
        a = wt * slope_hot(tl);
        b = wt * slope_cold(tr);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = a;
        partials[2 * blockIdx.x + 1] = b;
        __threadfence();
        last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    a = 0.0;
    b = 0.0;
    for (unsigned k = threadIdx.x; k < gridDim.x; k += 32) {
        a += __ldcg(partials + 2 * k);
        b += __ldcg(partials + 2 * k + 1);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if (threadIdx.x == 0) {
        // -L / dT once for all rows, not a quotient per row
        const double scale = -L / (12.0 * dT) / (double)(gm.ny - 1);
        out[0] = a * scale;
        out[1] = b * scale;
        *counter = 0u;
    }
}

// Full FP64 populations of the post-stream state, dense [q][ny][nx].
template <class T, bool FIELD>
__global__ void __launch_bounds__(256) k_read_state(Src<T> prev, const typename T::P* __restrict__ phi, Geom gm,
                                                    CoefOf<T> c, double* __restrict__ f,
                                                    double* __restrict__ g) {
    using R = typename T::R;
    const long n = (long)gm.nx * gm.ny;
    // rest weights in FP64 (Eq. 37 first occurrence), independent of the arithmetic type
    const double varpi = (double)c.varpi, T0 = (double)c.T0;
    const double wt0 = (1.0 - varpi) / 5.0, wt1 = (4.0 + varpi) / 20.0;
    for (long k = blockIdx.x * (long)blockDim.x + threadIdx.x; k < n; k += (long)gridDim.x * blockDim.x) {
        const int y = (int)(k / gm.nx), x = (int)(k - (long)y * gm.nx);
        R d[9], h[5];
        // framed storage: h is relative to T0 + F (F = 0 otherwise)
        const R F = node_populations<T, FIELD>(c, gm, prev, phi, x, y, d, h);
        const double Tr = Framed<T>::value ? T0 + (double)F : T0;
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i * n + k] = w9(i) + (double)d[i];
        g[k] = wt0 * Tr + (double)h[0];
#pragma unroll
        for (int j = 1; j < 5; ++j) g[j * n + k] = wt1 * Tr + (double)h[j];
    }
}

// Counts the cells of a porosity field outside the open interval (0, 1)
// (NaN included) into *bad.
template <class In>
__global__ void k_count_bad_phi(const In* __restrict__ in, long n, unsigned long long* __restrict__ bad) {
    unsigned long long c = 0;
    for (long k = blockIdx.x * (long)blockDim.x + threadIdx.x; k < n; k += (long)gridDim.x * blockDim.x) {
        const In v = in[k];
        c += (v > In(0) && v < In(1)) ? 0ull : 1ull;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(bad, c);
}

template <class In, class P>
__global__ void k_convert_phi(const In* __restrict__ in, P* __restrict__ out, Geom gm) {
    const long n = (long)gm.nx * gm.ny;
    for (long k = blockIdx.x * (long)blockDim.x + threadIdx.x; k < n; k += (long)gridDim.x * blockDim.x) {
        const int y = (int)(k / gm.nx), x = (int)(k - (long)y * gm.nx);
        out[y * gm.pitch + x] = (P)in[k];
    }
}

// ---- host launchers ---------------------------------------------------------------

template <class T> static const CoefOf<T>& coef_of(const CoefSet& cs);
template <> const Coef<double>& coef_of<PrecF64>(const CoefSet& cs) { return cs.d; }
template <> const Coef<float>& coef_of<PrecF32Q>(const CoefSet& cs) { return cs.f; }
template <> const Direct& coef_of<PrecF16>(const CoefSet& cs) { return cs.h; }
template <> const Coef<float>& coef_of<PrecF32T>(const CoefSet& cs) { return cs.f; }

// Launches kernel k with the step's arguments, as a programmatic dependent of
// the previous work on the stream when L.pdl is set.  gx, gy: blocks over the
// nodes; PAIRS: which border goes apart.
template <class T, bool PAIRS, class K>
static cudaError_t launch_one_step(K k, int gx, int gy, const StepLaunch& L, const CoefOf<T>& c, bool field) {
    const int per_col = gy * L.bx * L.by;  // border nodes that a column of blocks holds
    int border = Core<T>::value ? (border_count<PAIRS>(L.gm.nx, L.gm.ny) + per_col - 1) / per_col : 0;
    bool spread = false;  // see step_border
    if (PAIRS && border && (long)L.gm.nx * L.gm.ny >= (1L << 21)) {
        const int others = L.bx * L.by - border_columns<PAIRS>(L.gm.nx) * L.by;  // threads left for the y walls
        spread = others > 0 && 2 * ((L.gm.nx + others - 1) / others) <= gy;
        if (spread) border = 1;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(gx + border, gy);
    cfg.blockDim = dim3(L.bx, L.by);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = L.stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = L.pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, src_view<T>(L.src, L.gm.plane), dst_view<T>(L.dst, L.gm.plane),
                              field ? (const typename T::P*)L.phi : nullptr, L.gm, c, L.status, L.obs,
                              spread ? -gx : gx);
}

template <class T, bool FIELD, bool OBS>
static cudaError_t launch_step_k(const StepLaunch& L, const CoefSet& cs) {
    const CoefOf<T>& c = coef_of<T>(cs);
    const int rows = Core<T>::value ? L.gm.ny - 2 : L.gm.ny;  // the rows without the border, or all
    const int per = L.npt == 2 ? 2 * L.by : L.by, wide = L.npt == 3 ? 2 * L.bx : L.bx;
    const int gx = (L.gm.nx + wide - 1) / wide, gy = (rows + per - 1) / per;
    if (L.npt == 2) return launch_one_step<T, false>(k_step2<T, FIELD, OBS>, gx, gy, L, c, FIELD);
    if (L.npt == 3) return launch_one_step<T, true>(k_step2x<T, FIELD, OBS>, gx, gy, L, c, FIELD);
    return launch_one_step<T, false>(k_step<T, FIELD, OBS>, gx, gy, L, c, FIELD);
}

template <class T>
static cudaError_t launch_step_t(const StepLaunch& L, const CoefSet& cs) {
    if (L.obs) return L.phi ? launch_step_k<T, true, true>(L, cs) : launch_step_k<T, false, true>(L, cs);
    return L.phi ? launch_step_k<T, true, false>(L, cs) : launch_step_k<T, false, false>(L, cs);
}

template <class T>
static cudaError_t launch_observe_t(const ObserveLaunch& L, const CoefSet& cs) {
    using R = typename T::R;
    const Src<T> s = src_view<T>(L.prev, L.gm.plane);
    // blocks for the rows of the Nusselt numbers, and for the nodes as many as the
    // lattice fills, up to L.nblocks in all
    const int rows = std::min(64, (L.gm.ny + 255) / 256);
    const long full = ((long)L.gm.nx * L.gm.ny + 255) / 256;
    const int nodes = (int)std::min<long>(L.nblocks - rows, full);
    auto run = [&](auto kernel, const typename T::P* phi) {
        kernel<<<nodes + rows, 256, 0, L.stream>>>(s, phi, L.gm, coef_of<T>(cs), (R*)L.ux, (R*)L.uy, (R*)L.T, (R*)L.p,
                                                   (R*)L.snap, L.snap_valid, L.partials, nodes, L.L, L.dT, L.status,
                                                   L.counter, L.out);
    };
    if (L.phi) run(k_observe<T, true>, (const typename T::P*)L.phi);
    else run(k_observe<T, false>, nullptr);
    return cudaGetLastError();
}

template <class T>
static cudaError_t launch_nusselt_t(const ObserveLaunch& L, const CoefSet& cs) {
    // partials holds 2 doubles per block; counter is zero between launches
    const int nb = (L.gm.ny + 31) / 32;
    const Src<T> s = src_view<T>(L.prev, L.gm.plane);
    if (L.obs)
        k_nusselt_rows<T, true><<<nb, 32, 0, L.stream>>>(s, L.obs, L.gm, coef_of<T>(cs), L.L, L.dT, L.partials,
                                                         L.counter, L.out);
    else
        k_nusselt_rows<T, false><<<nb, 32, 0, L.stream>>>(s, nullptr, L.gm, coef_of<T>(cs), L.L, L.dT, L.partials,
                                                          L.counter, L.out);
    return cudaGetLastError();
}

template <class T>
static cudaError_t launch_read_state_t(const ReadStateLaunch& L, const CoefSet& cs) {
    const Src<T> s = src_view<T>(L.prev, L.gm.plane);
    if (L.phi)
        k_read_state<T, true><<<L.nblocks, 256, 0, L.stream>>>(s, (const typename T::P*)L.phi, L.gm,
                                                               coef_of<T>(cs), L.f, L.g);
    else
        k_read_state<T, false><<<L.nblocks, 256, 0, L.stream>>>(s, nullptr, L.gm, coef_of<T>(cs), L.f, L.g);
    return cudaGetLastError();
}

#define LBM_DISPATCH(prec, fn, ...)                     \
    switch (prec) {                                     \
        case PREC_F64: return fn<PrecF64>(__VA_ARGS__); \
        case PREC_F32: return fn<PrecF32Q>(__VA_ARGS__); \
        case PREC_F32T: return fn<PrecF32T>(__VA_ARGS__); \
        default: return fn<PrecF16>(__VA_ARGS__);       \
    }

cudaError_t launch_step(const StepLaunch& L, const CoefSet& cs) { LBM_DISPATCH(L.precision, launch_step_t, L, cs) }
cudaError_t launch_observe(const ObserveLaunch& L, const CoefSet& cs) {
    LBM_DISPATCH(L.precision, launch_observe_t, L, cs)
}
cudaError_t launch_nusselt(const ObserveLaunch& L, const CoefSet& cs) {
    LBM_DISPATCH(L.precision, launch_nusselt_t, L, cs)
}
cudaError_t launch_read_state(const ReadStateLaunch& L, const CoefSet& cs) {
    LBM_DISPATCH(L.precision, launch_read_state_t, L, cs)
}

size_t state_buffer_bytes(int precision, int plane) {
    switch (precision) {
        case PREC_F64: return buffer_bytes<PrecF64>(plane);
        case PREC_F32: return buffer_bytes<PrecF32Q>(plane);
        case PREC_F32T: return buffer_bytes<PrecF32T>(plane);
        default: return buffer_bytes<PrecF16>(plane);
    }
}

size_t phi_bytes(int precision, int plane) {
    return (size_t)plane * (precision == PREC_F64 ? sizeof(double) : sizeof(float));
}

cudaError_t launch_count_bad_phi(const void* in, int in_is_double, long n, unsigned long long* bad, int nblocks,
                                 cudaStream_t s) {
    if (in_is_double) k_count_bad_phi<double><<<nblocks, 256, 0, s>>>((const double*)in, n, bad);
    else k_count_bad_phi<float><<<nblocks, 256, 0, s>>>((const float*)in, n, bad);
    return cudaGetLastError();
}

cudaError_t launch_convert_phi(const void* in, int in_is_double, void* out, int precision, const Geom& gm,
                               int nblocks, cudaStream_t s) {
    const bool to_double = precision == PREC_F64;
    if (in_is_double) {
        if (to_double) k_convert_phi<double, double><<<nblocks, 256, 0, s>>>((const double*)in, (double*)out, gm);
        else k_convert_phi<double, float><<<nblocks, 256, 0, s>>>((const double*)in, (float*)out, gm);
    } else {
        if (to_double) k_convert_phi<float, double><<<nblocks, 256, 0, s>>>((const float*)in, (double*)out, gm);
        else k_convert_phi<float, float><<<nblocks, 256, 0, s>>>((const float*)in, (float*)out, gm);
    }
    return cudaGetLastError();
}

}  // namespace lbm
