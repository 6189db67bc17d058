// Discrete adjoint of the time stepping: gradient of the mean Nusselt number
// of the hot wall (Eq. 38) after N steps with respect to a per-cell porosity
// field, by reverse sweeps with checkpoint-and-recompute.
//
// Notation: B_k is the post-collision lattice after step k (B_{-1} = rest),
// S_N = pull(B_{N-1}) + wall rule, J = Nu_hot(S_N).  The adjoint state
// M^(k)(x) = dJ / d(populations pulled into node x at step k) lives on nodes;
// dJ/dB_k(y)_i = M^(k)_i(y + e_i) is gathered (the reverse of the pull, read
// over reversed directions, so no atomics).  A wall node uses the pulled
// populations of its inner neighbour, so a fluid node also folds in the
// reverse of the wall nodes that extrapolate from it.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <type_traits>
#include <vector>

#include "lbm_adjoint.cuh"
#include "lbm_internal.h"

using namespace lbm;

namespace lbm {

constexpr int kAdjThreads = 128, kAdjBlocks = 5;

// dJ/dS_N as the initial adjoint state: J depends on T at the columns 1..4
// next to the hot wall (the wall column is the imposed T_h); on first-order
// adiabatic walls T(x, 0) = T(x, 1) and T(x, ny-1) = T(x, ny-2).
template <class R>
__global__ void k_adj_seed(R* __restrict__ M, Geom gm, double L, double dT) {
    const int y = blockIdx.x * blockDim.x + threadIdx.x;
    if (y < 1 || y > gm.ny - 2) return;
    const double cx[5] = {-25.0, 48.0, -36.0, 16.0, -3.0};
    double wy = 1.0;
    if (gm.thermal_bc == 0) {
        if (y == 1) wy += 0.5;
        if (y == gm.ny - 2) wy += 0.5;
    }
    for (int x = 1; x <= 4 && x <= gm.nx - 2; ++x) {
        const double a = -L * cx[x] / (12.0 * dT * (double)(gm.ny - 1)) * wy;
        for (int j = 0; j < 5; ++j) M[(9 + j) * gm.plane + y * gm.pitch + x] = (R)a;
    }
}

// Element at a uniform base and a thread's byte offset (as at() above does for a
// node's offset).
template <class S> __device__ __forceinline__ S* at(S* base, unsigned bytes) {
    if constexpr (std::is_const<S>::value) return (S*)((const char*)base + bytes);
    else return (S*)((char*)base + bytes);
}

// lambda and mu of node (x, y): the adjoint of what it sent along each e_i.
// Plain loads, not the read-only path: a launch may start while the one that
// wrote these values is still running (it reads them after its wait).
// EDGE: next to or on a wall, where neighbours may lie outside.
template <class R, bool EDGE>
__device__ __forceinline__ void gather_adjoint(const R* M, const Geom& gm, int x, int y, R (&l)[9], R (&m)[5]) {
    const unsigned off = (unsigned)(y * gm.pitch + x) * (unsigned)sizeof(R);
#pragma unroll
    for (int q = 0; q < NPOP; ++q) {
        const int i = q < 9 ? q : q - 9, xs = x + ex9(i), ys = y + ey9(i);
        const bool in = !EDGE || (xs >= 0 && xs < gm.nx && ys >= 0 && ys < gm.ny);
        const R v = in ? __ldcg(at(M + (q * gm.plane + ey9(i) * gm.pitch + ex9(i)), off)) : R(0);
        if (q < 9) l[q] = v;
        else m[q - 9] = v;
    }
}

// What the transpose needs of the populations pulled into a fluid node (a and b
// only next to a wall).
template <class T>
__device__ __forceinline__ void tape_at(const Coef<typename T::R>& c, const Src<T>& src, const Geom& gm,
                                        const typename T::P* __restrict__ phi, int off, Tape<typename T::R>& t) {
    using R = typename T::R;
    R d[9], h[5];
    d[0] = R(0);
#pragma unroll
    for (int i = 1; i < 9; ++i) {
        const int e = -ey9(i) * gm.pitch - ex9(i);
        d[i] = in_plane(gm, off + e) ? Conv<typename T::SF, R, T::cg>::ld(at(src.f, i * gm.plane + e, off)) : R(0);
    }
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const int e = -ey9(j) * gm.pitch - ex9(j);
        h[j] = in_plane(gm, off + e) ? Conv<typename T::SG, R, T::cg>::ld(at(src.g, j * gm.plane + e, off)) : R(0);
    }
    const R F = op::mul(core_frame_in<T>(c.k, src, gm, off, h), c.k.fu);
    tape_node<R, Framed<T>::value>(c.k, (R)phi[off], sums_of(d, h), F, t);
}

// Two nodes side by side (x0 even): values whose two nodes start at an even x
// come as pairs.
template <class T> struct PairAt {
    using R = typename T::R;
    // plane p's values that e_i carries into the pair at off
    static __device__ __forceinline__ float2 state(const float* p, const Geom& gm, int off, int ex, int ey) {
        const int d = -ey * gm.pitch - ex;
        const unsigned b = 4u * (unsigned)off;
        if (ex == 0)
            return in_plane(gm, off + d, 2) ? Conv2<float, float, T::cg>::ld(at(p + d, b)) : make_float2(0.f, 0.f);
        return make_float2(in_plane(gm, off + d) ? Conv<float, float, T::cg>::ld(at(p + d, b)) : 0.f,
                           in_plane(gm, off + d + 1) ? Conv<float, float, T::cg>::ld(at(p + d, b) + 1) : 0.f);
    }
    static __device__ __forceinline__ void tape(const Coef<float>& c, const Src<T>& src, const Geom& gm,
                                                const float* __restrict__ phi, int off, Tape<F2>& t) {
        float h0[5], h1[5], F0, F1;
        F2 d[9], h[5];
        d[0] = F2(0.f);
#pragma unroll
        for (int i = 1; i < 9; ++i)
            d[i] = F2(state(src.f + i * gm.plane, gm, off, ex9(i), ey9(i)));
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            const float2 v = state(src.g + j * gm.plane, gm, off, ex9(j), ey9(j));
            h0[j] = v.x;
            h1[j] = v.y;
        }
        core_frame_in_x2<T>(c.k, src, gm, off, h0, h1, F0, F1);
#pragma unroll
        for (int j = 0; j < 5; ++j) h[j] = F2(h0[j], h1[j]);
        const float2 ph = __ldg((const float2*)at(phi, 4u * (unsigned)off));
        tape_node<F2, Framed<T>::value>(c.k, F2(ph), sums_of(d, h), op::mul(c.k.fu, F2(F0, F1)), t);
    }
    static __device__ __forceinline__ void gather(const float* M, const Geom& gm, int off, F2 (&l)[9], F2 (&m)[5]) {
#pragma unroll
        for (int q = 0; q < NPOP; ++q) {
            const int i = q < 9 ? q : q - 9;
            const float* p = at(M + (q * gm.plane + ey9(i) * gm.pitch + ex9(i)), 4u * (unsigned)off);
            const F2 v = ex9(i) == 0 ? F2(__ldca((const float2*)p)) : F2(__ldca(p), __ldca(p + 1));
            if (q < 9) l[q] = v;
            else m[q - 9] = v;
        }
    }
};

// n / d for n < 2^31 by a multiplication (d >= 2: m = ceil(2^(31 + l) / d), l = ceil(log2 d))
struct Divider {
    unsigned m = 0, s = 0;
    explicit Divider(unsigned d) {
        if (d < 2) return;
        unsigned l = 1;
        while ((1ull << l) < d) ++l;
        m = (unsigned)(((1ull << (31 + l)) + d - 1) / d);
        s = l - 1;
    }
    __device__ __forceinline__ int quotient(unsigned n) const { return (int)(m ? __umulhi(n, m) >> s : n); }
};

// Reverse of one step at the interior nodes, two or more from every wall, and in
// the first `edge` blocks (their nodes take longer) at the fluid nodes next to a
// wall together with the wall nodes that extrapolate from them: M^(k) from
// M^(k+1) and the forward input B_k, and this step's porosity sensitivity added
// to gphi.  M at the wall nodes stays 0: they read no pulled populations of
// their own.
//
// The state and the tape need nothing of the previous reverse step, so a launch
// starts early, as a programmatic dependent, and waits only then (late start:
// 10.8 ms instead of 10.0 for the call below).
//
// Everything but the forward states stays in L2; a step moves 72 MB through it
// at 512^2 and is bound by that latency and by issue slots (545 instructions per
// pair, some 205 of them arithmetic; 1.35 waves of 20 warps per SM).  512^2 FP32, us
// per reverse step alone: 7.6; 8.3 with an index per access, and 23.4 for the
// direct formulas in one kernel for the interior and one for the ring of nodes
// near the walls on a stream of its own.  The gradient of 600 steps: 19.8 -> 9.8 ms.
template <class T>
__global__ void __launch_bounds__(kAdjThreads, sizeof(typename T::R) == 4 ? kAdjBlocks : 2)
    k_adjoint(Src<T> state, const typename T::R* Mnext, typename T::R* Mcur, const typename T::P* __restrict__ phi,
              double* gphi, Geom gm, Coef<typename T::R> c, int edge, Divider rows_of) {
    using R = typename T::R;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if ((int)blockIdx.x < edge) {
        const int j = blockIdx.x * kAdjThreads + threadIdx.x, rows = 2 * (gm.nx - 2);
        int x = 0, y = 0;
        const bool in = j < rows + 2 * (gm.ny - 4);
        Tape<R> t;
        if (in) {
            if (j < rows) {
                x = 1 + (j >> 1);
                y = j & 1 ? gm.ny - 2 : 1;
            } else {
                x = j & 1 ? gm.nx - 2 : 1;
                y = 2 + ((j - rows) >> 1);
            }
            tape_at<T>(c, state, gm, phi, y * gm.pitch + x, t);
        }
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (!in) return;
        const int off = y * gm.pitch + x;
        R l[9], m[5];
        gather_adjoint<R, true>(Mnext, gm, x, y, l, m);
        Seeds<R> b = {};
        own_seeds(c.k, l[0], sums_of(l, m), b);
        const int sx = x == 1 ? -1 : x == gm.nx - 2 ? 1 : 0, sy = y == 1 ? -1 : y == gm.ny - 2 ? 1 : 0;
#pragma unroll 1
        for (int w = 0; w < 3; ++w) {  // the wall nodes beside, below or above, and across the corner
            if ((w != 1 && sx == 0) || (w != 0 && sy == 0)) continue;
            const int xb = w == 1 ? x : x + sx, yb = w == 0 ? y : y + sy;
            R lb[9], mb[5];
            gather_adjoint<R, true>(Mnext, gm, xb, yb, lb, mb);
            const bool dirichlet = gm.thermal_bc == 1 || w != 1;
            const R dTw = gm.thermal_bc == 0 && xb == 0 ? c.k.dTh : c.k.dTc;
            const R pb = wall_seeds<R>(c.k, t, (R)phi[yb * gm.pitch + xb], dirichlet, dTw, lb[0], mb[0],
                                       sums_of(lb, mb), b);
            gphi[(long)yb * gm.nx + xb] += (double)pb;
#pragma unroll
            for (int i = 0; i < 9; ++i) l[i] = op::add(l[i], lb[i]);
#pragma unroll
            for (int i = 0; i < 5; ++i) m[i] = op::add(m[i], mb[i]);
        }
        const R pb = node_adjoint<R, true>(c.k, t, b, sums_of(l, m), l, m);
#pragma unroll
        for (int q = 0; q < NPOP; ++q) Mcur[q * gm.plane + off] = q < 9 ? l[q] : m[q - 9];
        gphi[(long)y * gm.nx + x] += (double)pb;
        return;
    }
    const int n = (blockIdx.x - edge) * kAdjThreads + threadIdx.x;
    if constexpr (sizeof(R) == 4) {  // FP32: two nodes per thread
        const int w = (gm.nx - 3) / 2, yi = rows_of.quotient(n), x = 2 + 2 * (n - yi * w), y = 2 + yi, off = y * gm.pitch + x;
        const bool in = yi < gm.ny - 4;
        Tape<F2> t;
        if (in) PairAt<T>::tape(c, state, gm, phi, off, t);
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (!in) return;
        double* g = gphi + ((long)y * gm.nx + x);
        const bool two = x + 1 < gm.nx - 2;  // else the second node is next to the wall
        F2 l[9], m[5];
        PairAt<T>::gather(Mnext, gm, off, l, m);
        const double g0 = __ldcg(g), g1 = __ldcg(g + 1);
        const Sums<F2> s = sums_of(l, m);
        Seeds<F2> b;
        own_seeds(c.k, l[0], s, b);
        const F2 pb = node_adjoint<F2, false>(c.k, t, b, s, l, m);
#pragma unroll
        for (int q = 0; q < NPOP; ++q) {
            const F2 v = q < 9 ? l[q] : m[q - 9];
            R* p = at(Mcur + q * gm.plane, 4u * (unsigned)off);
            if (two) *(float2*)p = v.v;
            else *p = v.v.x;
        }
        g[0] = g0 + (double)pb.v.x;
        if (two) g[1] = g1 + (double)pb.v.y;
    } else {
        const int w = gm.nx - 4, yi = rows_of.quotient(n), x = 2 + n - yi * w, y = 2 + yi, off = y * gm.pitch + x;
        const bool in = yi < gm.ny - 4;
        Tape<R> t;
        if (in) tape_at<T>(c, state, gm, phi, off, t);
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (!in) return;
        R l[9], m[5];
        gather_adjoint<R, false>(Mnext, gm, x, y, l, m);
        const Sums<R> s = sums_of(l, m);
        Seeds<R> b;
        own_seeds(c.k, l[0], s, b);
        const R pb = node_adjoint<R, false>(c.k, t, b, s, l, m);
#pragma unroll
        for (int q = 0; q < NPOP; ++q) Mcur[q * gm.plane + off] = q < 9 ? l[q] : m[q - 9];
        gphi[(long)y * gm.nx + x] += (double)pb;
    }
}

template <class Out>
__global__ void k_adj_out(const double* __restrict__ g, Out* __restrict__ out, long n) {
    for (long k = blockIdx.x * (long)blockDim.x + threadIdx.x; k < n; k += (long)gridDim.x * blockDim.x)
        out[k] = (Out)g[k];
}

}  // namespace lbm

namespace {

// Second stream for the recomputation of the next segment, with an event per
// half of the segment storage for "recomputed" and for "read by the reverse
// sweep" (both recorded once at the start, so the first waits pass).
struct RecomputeStream {
    cudaStream_t s3 = nullptr;
    cudaEvent_t ready[2] = {nullptr, nullptr}, free[2] = {nullptr, nullptr}, end = nullptr;
    cudaError_t init(cudaStream_t main) {
        cudaError_t e = cudaStreamCreateWithFlags(&s3, cudaStreamNonBlocking);
        for (int k = 0; k < 2 && e == cudaSuccess; ++k) {
            e = cudaEventCreateWithFlags(&ready[k], cudaEventDisableTiming);
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(&free[k], cudaEventDisableTiming);
            if (e == cudaSuccess) e = cudaEventRecord(free[k], main);  // after the set-up on the main stream
        }
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&end, cudaEventDisableTiming);
        return e;
    }
    // an event behind all recompute work (the main stream waits for it before it returns)
    cudaEvent_t done() {
        return cudaEventRecord(end, s3) == cudaSuccess ? end : ready[0];
    }
    ~RecomputeStream() {
        if (end) cudaEventDestroy(end);
        for (int k = 0; k < 2; ++k) {
            if (ready[k]) cudaEventDestroy(ready[k]);
            if (free[k]) cudaEventDestroy(free[k]);
        }
        if (s3) cudaStreamDestroy(s3);
    }
};

template <class T>
cudaError_t adjoint_sweep(const AdjointJob& J) {
    using R = typename T::R;
    const Geom& gm = J.gm;
    const Coef<R>& c = *(const Coef<R>*)J.coef;
    const int N = (int)J.nsteps, K = (int)J.ckpt_every;
    const size_t buf = J.buf_bytes;
    const size_t mbytes = (size_t)gm.plane * NPOP * sizeof(R);
    cudaStream_t s = J.stream;
    const int wide = sizeof(R) == 4 ? (gm.nx - 3) / 2 : gm.nx - 4;  // threads per interior row
    const long inner = (long)wide * (gm.ny - 4);
    const Divider rows_of((unsigned)wide);
    const long next = 2L * (gm.nx - 2) + 2L * (gm.ny - 4);
    const int edge = (int)((next + kAdjThreads - 1) / kAdjThreads);
    const int nblk = edge + (int)((inner + kAdjThreads - 1) / kAdjThreads);
    const int nseg = (N + K - 1) / K;
    R* M[2] = {(R*)J.madj, (R*)J.madj + (size_t)gm.plane * NPOP};
    cudaError_t e = cudaMemsetAsync(M[0], 0, 2 * mbytes, s);
    if (e != cudaSuccess) return e;
    k_adj_seed<R><<<(gm.ny + 255) / 256, 256, 0, s>>>(M[0], gm, J.L, J.dT);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(J.gphi, 0, sizeof(double) * (size_t)gm.nx * gm.ny, s)) != cudaSuccess) return e;
    // The recomputation of a segment needs only its checkpoint, so it runs on a
    // second stream into the other half of the segment storage while the main
    // stream reverses the segment after it: forward steps and reverse steps overlap.
    RecomputeStream rc;
    if ((e = rc.init(s)) != cudaSuccess) return e;
    CoefSet cs;
    if (sizeof(R) == 8) cs.d = *(const Coef<double>*)J.coef;
    else cs.f = *(const Coef<float>*)J.coef;
    const size_t half = (size_t)(K > 1 ? K - 1 : 0) * buf;  // bytes of one half of the segment storage
    auto seg_len = [&](int sg) { return (N - sg * K) < K ? (N - sg * K) : K; };
    auto slot_of = [&](int sg, int hf, int m) -> const void* {
        return m == 0 ? (const char*)J.ckpt + (size_t)sg * buf : (const char*)J.seg + hf * half + (size_t)(m - 1) * buf;
    };
    // recompute segment sg into half hf on the second stream, once the reverse
    // sweep that last read that half is done
    auto recompute = [&](int sg, int hf) -> cudaError_t {
        cudaError_t er = cudaStreamWaitEvent(rc.s3, rc.free[hf], 0);
        for (int m = 1; m < seg_len(sg) && er == cudaSuccess; ++m) {
            StepLaunch L;
            L.precision = J.precision;
            L.src = slot_of(sg, hf, m - 1);
            L.dst = (void*)slot_of(sg, hf, m);
            L.phi = J.phi;
            L.gm = gm;
            L.bx = J.bx;
            L.by = J.by;
            L.npt = J.npt;
            L.status = J.status;
            L.stream = rc.s3;
            L.pdl = m > 1;  // directly behind the previous recomputing step
            er = launch_step(L, cs);
        }
        if (er == cudaSuccess) er = cudaEventRecord(rc.ready[hf], rc.s3);
        return er;
    };
    int a = 0, hf = 0;
    e = recompute(nseg - 1, 0);
    for (int sg = nseg - 1; sg >= 0 && e == cudaSuccess; --sg, hf ^= 1) {
        const int j0 = sg * K, len = seg_len(sg);
        if (sg > 0 && (e = recompute(sg - 1, hf ^ 1)) != cudaSuccess) break;
        if ((e = cudaStreamWaitEvent(s, rc.ready[hf], 0)) != cudaSuccess) break;
        for (int j = j0 + len - 1; j >= j0; --j) {
            const Src<T> st = src_view<T>(slot_of(sg, hf, j - j0), gm.plane);
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(nblk);
            cfg.blockDim = dim3(kAdjThreads);
            cfg.stream = s;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            at[0].val.programmaticStreamSerializationAllowed = 1;
            cfg.attrs = at;
            cfg.numAttrs = j < j0 + len - 1 ? 1 : 0;  // directly behind a reverse step of the same segment
            e = cudaLaunchKernelEx(&cfg, k_adjoint<T>, st, (const R*)M[a], M[a ^ 1], (const typename T::P*)J.phi,
                                   J.gphi, gm, c, edge, rows_of);
            if (e != cudaSuccess) break;
            a ^= 1;
        }
        // the half is free again once this segment's reverse sweep is done
        if (e == cudaSuccess) e = cudaEventRecord(rc.free[hf], s);
    }
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s, rc.done(), 0);
    if (e != cudaSuccess) return e;
    const long n = (long)gm.nx * gm.ny;
    if (sizeof(R) == 8) k_adj_out<double><<<kReduceBlocks, 256, 0, s>>>(J.gphi, (double*)J.out, n);
    else k_adj_out<float><<<kReduceBlocks, 256, 0, s>>>(J.gphi, (float*)J.out, n);
    return cudaGetLastError();
}

}  // namespace

namespace lbm {
cudaError_t launch_adjoint_sweep(const AdjointJob& J) {
    if (J.precision == PREC_F64) return adjoint_sweep<PrecF64>(J);
    if (J.precision == PREC_F32T) return adjoint_sweep<PrecF32T>(J);
    return adjoint_sweep<PrecF32Q>(J);
}
}  // namespace lbm
