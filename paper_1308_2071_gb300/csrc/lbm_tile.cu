// Several time steps per launch on lattices that fit on chip (FP32 arithmetic
// and storage).
//
// A step of such a lattice takes less time than starting a kernel and waiting
// for its first loads.  Here a block owns a tile of nodes and takes `steps`
// steps of it by itself: the first pulls B_n from memory for the tile and a
// surround of steps - 1 nodes, each further one pulls from shared memory for a
// surround one node narrower, and the last writes the tile of B_{n+steps}.
// Nothing is exchanged between blocks, so no wait is needed; the surround is
// computed by the neighbours as well.  Two copies of the region alternate in
// shared memory, with one barrier per step.  Measured, us per step against one
// step per launch: 64^2 2.2 -> 0.98, 128^2 1.9 -> 1.3, 200^2 2.2 -> 1.7; from 250^2 on the
// repeated surround costs more than the launches (300^2 2.3 -> 2.7).  Bound by the
// latency of a node's chain of operations (0.8 us per step) on small lattices, by
// the FMA pipe on the repeated nodes on the larger: two nodes per thread in paired
// instructions halve the instructions and gain 3 % at 200^2 but lose 5 % at 64^2
// (not kept).
//
// The tile and the number of steps come from a cost model (tile_shape): larger
// tiles repeat less of the surround, smaller ones spread over more SMs, and
// more steps share one launch but need a wider surround.
#include <algorithm>

#include "lbm_internal.h"

namespace lbm {

namespace {

constexpr int kTileThreads = 256;
constexpr int kTileNodes = 944;  // of a region; 2 copies x 15 values: 113,280 bytes, two blocks per SM
constexpr size_t kTileSmem = sizeof(float) * 2 * 15 * kTileNodes;
constexpr int kTileMostSteps = 12;
constexpr double kTileLaunch = 1.6, kTileLatency = 0.72, kTileIssue = 0.065;

// Nodes [xa, xb) x [ya, yb).
struct Rect {
    int xa, ya, xb, yb;
    __host__ __device__ int nodes() const { return (xb - xa) * (yb - ya); }
};

// The region grown by m nodes on every side, within the lattice.  With tiles of
// at least kTileLeast nodes across, one more node on every side holds all that
// a step of r pulls, beside a wall too (whose nodes pull what their inner
// neighbours do: three nodes deep, four with second-order adiabatic walls).
constexpr int kTileLeast = 4;
__host__ __device__ inline Rect grown(const Rect& r, int m, int nx, int ny) {
    Rect p;
    p.xa = r.xa > m ? r.xa - m : 0;
    p.ya = r.ya > m ? r.ya - m : 0;
    p.xb = r.xb + m < nx ? r.xb + m : nx;
    p.yb = r.yb + m < ny ? r.yb + m : ny;
    return p;
}

// A region in shared memory, [population][node], the frame (in its unit) last.
struct RegionSource {
    const float* v;
    const Coll<float>& k;
    int xa, ya, w;
    __device__ __forceinline__ float pulled(int x, int y, float (&d)[9], float (&h)[5]) const {
        const float* o = v + (y - ya) * w + (x - xa);
        const float *s = o - w, *n = o + w;  // the rows that e_y = 1 and e_y = -1 come from
        auto row = [&](int i) { return ey9(i) == 0 ? o : ey9(i) > 0 ? s : n; };
#pragma unroll
        for (int i = 0; i < 9; ++i) d[i] = row(i)[i * kTileNodes - ex9(i)];
        const float F = o[14 * kTileNodes];
        h[0] = o[9 * kTileNodes];
#pragma unroll
        for (int j = 1; j < 5; ++j)
            h[j] = op::fma(k.w1, op::sub(row(j)[14 * kTileNodes - ex9(j)], F), row(j)[(9 + j) * kTileNodes - ex9(j)]);
        return F;
    }
    __device__ __forceinline__ float frame(int x, int y) const { return v[14 * kTileNodes + (y - ya) * w + (x - xa)]; }
    __device__ __forceinline__ float heat_at(int x, int y, float& F) const {
        float d[9], h[5];
        F = op::mul(pulled(x, y, d, h), k.fu);
        return heat(h);
    }
};

}  // namespace

// One step of the nodes r from `from`, into shared memory (to: region r) or,
// last, into the lattice.  The fluid nodes come first and the wall nodes after
// them in warps of their own, so that no warp runs both ways.
template <class T, bool FIELD, bool LAST, class Source>
__device__ __forceinline__ void tile_step(const Source& from, float* to, const Dst<T>& dst,
                                          const typename T::P* __restrict__ phi, const Geom& gm,
                                          const Coll<float>& k, int* __restrict__ status, const Rect& r) {
    const int w = r.xb - r.xa;
    Rect in;  // the fluid nodes
    in.xa = max(r.xa, 1);
    in.ya = max(r.ya, 1);
    in.xb = min(r.xb, gm.nx - 1);
    in.yb = min(r.yb, gm.ny - 1);
    const int wi = in.xb - in.xa, hi = in.yb - in.ya, ni = wi * hi;
    const int walls = r.nodes() - ni;
    const int first_wall = walls ? (ni + 31) & ~31 : ni;
    const int rows = (r.ya == 0) + (r.yb == gm.ny);  // y walls in the region
    const int left = r.xa == 0;
    const float iw = 1.f / (float)wi;
    for (int j = threadIdx.x; j < first_wall + walls; j += kTileThreads) {
        int x, y;
        if (j < first_wall) {
            if (j >= ni) continue;
            const int row = (int)(((float)j + 0.5f) * iw);  // exact: j < 2^12
            x = in.xa + j - row * wi;
            y = in.ya + row;
        } else {
            int i = j - first_wall;
            if (i < rows * w) {
                const bool second = i >= w;
                x = r.xa + (second ? i - w : i);
                y = r.ya == 0 && !second ? 0 : gm.ny - 1;
            } else {
                i -= rows * w;
                const bool second = i >= hi;
                x = left && !second ? 0 : gm.nx - 1;
                y = in.ya + (second ? i - hi : i);
            }
        }
        float d[9], h[5];
        const Post<float> p = core_post<T, FIELD>(k, gm, from, phi, x, y, d, h);
        if (!p.wall && too_fast(p.v)) atomicOr(status, 1);
        typename FrameStore<T>::type code;
        float next;
        const float shift = frame_next<T>(k, p.dT, p.F, next, code);
        core_collide<T, FIELD>(k, p, shift, d, h);
        if constexpr (LAST) {
            const int o = y * gm.pitch + x;
            if (!in_plane(gm, o)) continue;
            dst.t[o] = code;
#pragma unroll
            for (int i = 0; i < 9; ++i) dst.f[(size_t)i * gm.plane + o] = d[i];
#pragma unroll
            for (int i = 0; i < 5; ++i) dst.g[(size_t)i * gm.plane + o] = h[i];
        } else {
            float* v = to + (y - r.ya) * w + (x - r.xa);
#pragma unroll
            for (int i = 0; i < 9; ++i) v[i * kTileNodes] = d[i];
#pragma unroll
            for (int i = 0; i < 5; ++i) v[(9 + i) * kTileNodes] = h[i];
            v[14 * kTileNodes] = next;
        }
    }
}

template <class T, bool FIELD>
__global__ void __launch_bounds__(kTileThreads, 2)
    k_tile(Src<T> src, Dst<T> dst, const typename T::P* __restrict__ phi, const __grid_constant__ Geom gm,
           const __grid_constant__ Coef<float> c, int* __restrict__ status, int steps) {
    extern __shared__ float region[];
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the previous step is complete
    Rect out;  // the lattice shared out evenly
    out.xa = (int)blockIdx.x * gm.nx / (int)gridDim.x;
    out.xb = ((int)blockIdx.x + 1) * gm.nx / (int)gridDim.x;
    out.ya = (int)blockIdx.y * gm.ny / (int)gridDim.y;
    out.yb = ((int)blockIdx.y + 1) * gm.ny / (int)gridDim.y;
    Rect r = grown(out, steps - 1, gm.nx, gm.ny);
    float *to = region, *other = region + 15 * kTileNodes;
    tile_step<T, FIELD, false>(BufferSource<T>{c, gm, src}, to, dst, phi, gm, c.k, status, r);
#pragma unroll 1
    for (int s = 2; s < steps; ++s) {
        __syncthreads();
        const RegionSource from{to, c.k, r.xa, r.ya, r.xb - r.xa};
        r = grown(out, steps - s, gm.nx, gm.ny);
        tile_step<T, FIELD, false>(from, other, dst, phi, gm, c.k, status, r);
        float* swap = to;
        to = other;
        other = swap;
    }
    __syncthreads();
    const RegionSource from{to, c.k, r.xa, r.ya, r.xb - r.xa};
    tile_step<T, FIELD, true>(from, nullptr, dst, phi, gm, c.k, status, out);
}

// Tile and steps per launch for a lattice; steps = 0: this way is not faster.
// The model (microseconds, from timings on GB300): a launch and its first
// loads, then per step the larger of a node's latency times the passes of a
// block and the SM's issue time for all its warps.
TileShape tile_shape(int nx, int ny, int nsm) {
    TileShape best;
    for (int tx = 1; tx <= std::min(64, nx / kTileLeast); ++tx)
        for (int ty = 1; ty <= std::min(64, ny / kTileLeast); ++ty) {
            const int tw = (nx + tx - 1) / tx, th = (ny + ty - 1) / ty, tiles = tx * ty;
            if (tiles > 2 * nsm) break;  // one wave
            const double issue = kTileIssue * (tiles > nsm ? 2 : 1);  // blocks on an SM
            double t = kTileLaunch;
            for (int k = 1; k <= kTileMostSteps; ++k) {
                // the region of the k-th step from the last, of an inner tile
                const int n = (tw + 2 * (k - 1)) * (th + 2 * (k - 1));
                if (n > kTileNodes) break;
                t += std::max(kTileLatency * ((n + kTileThreads - 1) / kTileThreads), issue * ((n + 31) / 32));
                if (k >= 2 && t < best.us * k) {
                    best.us = t / k;
                    best.tx = tx;
                    best.ty = ty;
                    best.steps = k;
                }
            }
        }
    return best;
}

template <class T, bool FIELD> static cudaError_t launch_tile_k(const StepLaunch& L, const CoefSet& cs, const TileShape& s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(s.tx, s.ty);
    cfg.blockDim = dim3(kTileThreads);
    cfg.dynamicSmemBytes = kTileSmem;
    cfg.stream = L.stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = L.pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k_tile<T, FIELD>, src_view<T>(L.src, L.gm.plane), dst_view<T>(L.dst, L.gm.plane),
                              FIELD ? (const float*)L.phi : nullptr, L.gm, cs.f, L.status, s.steps);
}

template <class T> static cudaError_t tile_prepare_t(bool field) {
    return cudaFuncSetAttribute(field ? k_tile<T, true> : k_tile<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kTileSmem);
}

cudaError_t tile_prepare(int precision, bool field) {
    return precision == PREC_F32T ? tile_prepare_t<PrecF32T>(field) : tile_prepare_t<PrecF32Q>(field);
}

cudaError_t launch_tile(const StepLaunch& L, const CoefSet& cs, const TileShape& s) {
    if (L.precision == PREC_F32T)
        return L.phi ? launch_tile_k<PrecF32T, true>(L, cs, s) : launch_tile_k<PrecF32T, false>(L, cs, s);
    return L.phi ? launch_tile_k<PrecF32Q, true>(L, cs, s) : launch_tile_k<PrecF32Q, false>(L, cs, s);
}

}  // namespace lbm
