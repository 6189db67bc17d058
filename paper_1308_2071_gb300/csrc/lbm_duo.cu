// The launch that takes two time steps of one lattice at once (lbm_duo.cuh).
#include <math.h>

#include <algorithm>

#include "lbm_duo.cuh"
#include "lbm_internal.h"

namespace lbm {

// Blocks: the wall tiles, then strips x segments, a strip's neighbours side by
// side, so that the blocks at work together read a band of whole rows.
template <class T, bool FIELD, int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS == 64 ? 8 : 5)
    k_duo(Src<T> src, Dst<T> dst, const typename T::P* __restrict__ phi, const __grid_constant__ Geom gm,
          const __grid_constant__ Coef<float> c, int* __restrict__ status, int strips, int width, int rows) {
    __shared__ float2 sh[kDuoRows * (THREADS + 2)];
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the previous step is complete
    const int b = (int)blockIdx.x - duo_tiles(gm.nx, gm.ny, THREADS);
    if (b >= 0)
        duo_march_block<T, FIELD, THREADS>(b, src, dst, phi, gm, c.k, status, strips, width, rows, sh);
    else
        duo_wall_block<T, FIELD, THREADS>((int)blockIdx.x, src, dst, phi, gm, c, status, (float*)sh);
}

// resident[i]: blocks of 64 + 32 i threads that the GPU holds at a time.  At
// most kMostRows rows, so that the blocks at work together stay within a band
// of rows (few open DRAM and address-translation pages) and even out.
constexpr int kMostRows = 32;
static DuoShape shape_of(const Geom& gm, const int (&resident)[2]) {
    const int npairs = duo_last_pair(gm.nx) - duo_first_pair() + 1, inner = gm.ny - 4;
    DuoShape best;
    double cost = 1e300;
    for (int threads = 64; threads <= 96; threads += 32) {
        DuoShape s;
        s.threads = threads;
        s.strips = (npairs + threads - 3) / (threads - 2);
        s.width = (npairs + s.strips - 1) / s.strips;
        s.strips = (npairs + s.width - 1) / s.width;
        const int slots = resident[threads / 32 - 2];
        s.segs = std::max(1, std::min(slots / s.strips, (inner + 3) / 4));
        s.rows = std::min((inner + s.segs - 1) / s.segs, kMostRows);
        s.segs = (inner + s.rows - 1) / s.rows;
        const double waves = ceil((double)s.strips * s.segs / slots);
        const double cst = waves * threads * slots * (2.0 * s.rows + 2.0);
        if (cst < cost) {
            cost = cst;
            best = s;
        }
    }
    return best;
}

template <class T, bool FIELD> static cudaError_t duo_shape_t(const Geom& gm, int nsm, DuoShape* out) {
    int per[2] = {0, 0};
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per[0], k_duo<T, FIELD, 64>, 64, 0);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per[1], k_duo<T, FIELD, 96>, 96, 0);
    if (e != cudaSuccess) return e;
    const int resident[2] = {nsm * std::max(1, per[0]), nsm * std::max(1, per[1])};
    *out = shape_of(gm, resident);
    return cudaSuccess;
}

// Two steps in one launch need FP32 storage, first-order adiabatic walls (the
// second-order rule reads a node further in) and a few rows and pairs.
cudaError_t duo_shape(int precision, bool field, const Geom& gm, int nsm, DuoShape* out) {
    *out = DuoShape();
    if ((precision != PREC_F32 && precision != PREC_F32T) || gm.adi_order != 1 || gm.nx < 8 || gm.ny < 8)
        return cudaSuccess;
    if (precision == PREC_F32T)
        return field ? duo_shape_t<PrecF32T, true>(gm, nsm, out) : duo_shape_t<PrecF32T, false>(gm, nsm, out);
    return field ? duo_shape_t<PrecF32Q, true>(gm, nsm, out) : duo_shape_t<PrecF32Q, false>(gm, nsm, out);
}

template <class T, bool FIELD> static cudaError_t launch_duo_k(const StepLaunch& L, const CoefSet& cs, const DuoShape& s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(duo_tiles(L.gm.nx, L.gm.ny, s.threads) + s.strips * s.segs);
    cfg.blockDim = dim3(s.threads);
    cfg.stream = L.stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = L.pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, s.threads == 64 ? k_duo<T, FIELD, 64> : k_duo<T, FIELD, 96>,
                              src_view<T>(L.src, L.gm.plane), dst_view<T>(L.dst, L.gm.plane),
                              FIELD ? (const float*)L.phi : nullptr, L.gm, cs.f, L.status, s.strips, s.width, s.rows);
}

cudaError_t launch_duo(const StepLaunch& L, const CoefSet& cs, const DuoShape& s) {
    if (L.precision == PREC_F32T)
        return L.phi ? launch_duo_k<PrecF32T, true>(L, cs, s) : launch_duo_k<PrecF32T, false>(L, cs, s);
    return L.phi ? launch_duo_k<PrecF32Q, true>(L, cs, s) : launch_duo_k<PrecF32Q, false>(L, cs, s);
}

}  // namespace lbm
