// Two time steps per launch (FP32 arithmetic and storage): the lattice is read
// and written once for both, so a lattice larger than L2 moves half the
// bytes per step, and a smaller one needs half the launches.
//
// Most blocks march: each owns a strip of node pairs along x and moves up the
// rows.  In the iteration of row r it takes the first step at row r (pulling
// B_n from memory) and leaves the result in shared memory; then it takes the
// second step at row r - 1, which pulls the first step's rows r - 2, r - 1 and r
// from there, and writes B_{n+2}.  B_{n+1} never reaches memory.  Shared memory
// keeps a row of a population as long as the second step needs it: what streams
// up two rows back, sideways one, down the current row.
//
// The march meets fluid nodes only: the nodes within two (or, at a wall that
// falls on the first node of a pair, three) of a wall are stepped by small
// tiles of their own, blocks of the same launch that take both steps node by
// node with the wall rule; they start first and run beside the march.
//
// Bound: bytes in flight and latency.  A march moves 114 bytes per node and two
// steps and issues about 2 x 200 instructions for them (two nodes per
// instruction in the paired FP32 forms).  Redundant work: one pair on each
// side of a strip, and two rows of the first step per segment of rows.  Measured,
// us per step against one step per launch: 4096^2 274 -> 170 (DRAM 5.8 TB/s, 1.96
// GB per launch, issue 43 % busy), 1024^2 17.8 -> 14.0, 8192^2 with a porosity
// field 1,270 -> 770.  Not kept: copies into shared memory by the bulk copy engine
// (185 us memory alone against 169 with plain loads), rows prefetched into
// registers (no change), 96 registers and six blocks per SM (190 us: the loads'
// lines leave L1 before their second use), segments of a hundred rows (186
// us), the wall rule inside the march (192 us).
#pragma once

#include "lbm_node.cuh"

namespace lbm {
// Where population q (0..13; 14: the frame, in its unit) of a row of W pairs
// lies in shared memory: `slots` rows are kept.  A row is read in the
// iteration of its own row (age 0: e_y = -1), the next (age 1: e_y = 0, and the
// frames) or the one after (age 2: e_y = 1, own frames).  A neighbour may still
// be reading age a while this thread writes a + 1 rows later (one barrier per
// row), so values that stream along x keep a + 2 rows, the others a + 1.
__host__ __device__ constexpr int duo_slots(int q) {
    const int i = q < 9 ? q : q - 9;
    if (q == 14) return 4;
    const int age = 1 + ey9(i);
    return age + (ex9(i) != 0 ? 2 : 1);
}
__host__ __device__ constexpr int duo_first(int q) {
    int n = 0;
    for (int k = 0; k < q; ++k) n += duo_slots(k);
    return n;
}
constexpr int kDuoRows = duo_first(15);  // rows of W float2 per block

constexpr int kAhead = 2;

// A pair of nodes (x0, x0 + 1), one value per population: pulled populations,
// frames (in their unit) and porosities.
struct Pair {
    F2 d[9], h[5], c, phi;
};

// Re-expresses the pulled thermal values in the pair's own frames; s, n: the
// frames below and above the pair, w, e: of the nodes west and east of it.
__device__ __forceinline__ void pair_frames(const Coll<float>& k, Pair& p, F2 s, F2 n, float w, float e) {
    const float c0 = p.c.v.x, c1 = p.c.v.y;
    p.h[1] = op::fma(k.w1, F2(op::sub(w, c0), op::sub(c0, c1)), p.h[1]);
    p.h[2] = op::fma(k.w1, op::sub(s, p.c), p.h[2]);
    p.h[3] = op::fma(k.w1, F2(op::sub(c1, c0), op::sub(e, c1)), p.h[3]);
    p.h[4] = op::fma(k.w1, op::sub(n, p.c), p.h[4]);
}

// One value or an aligned pair of a plane at a 32-bit byte offset: the plane's
// address stays in uniform registers, so an access costs no address arithmetic.
template <class S> __device__ __forceinline__ S duo_ld(const Geom& gm, const void* plane, uint32_t byte, int size) {
    return in_plane(gm, (int)(byte / (uint32_t)size), (int)(sizeof(S) / size)) ? __ldg((const S*)((const char*)plane + byte))
                                                                            : S{};
}


// First and last pair that marches put out: the pairs clear of the nodes within
// two of an x wall.
__host__ __device__ constexpr int duo_first_pair() { return 1; }
__host__ __device__ inline int duo_last_pair(int nx) { return (nx & 1) ? (nx + 1) / 2 - 3 : nx / 2 - 2; }

// The march of one block over rows s0 <= y < s1 (2 <= y <= ny - 3) of the strip
// of pairs p0 .. p0 + n - 1.
template <class T, bool FIELD, int THREADS>
__device__ __forceinline__ void duo_march(const Src<T>& src, const Dst<T>& dst, const typename T::P* __restrict__ phi,
                                          const Geom& gm, const Coll<float>& k, int* __restrict__ status, int p0,
                                          int n, int s0, int s1, float2* sh) {
    using ST = typename FrameStore<T>::type;
    constexpr int W = THREADS + 2;
    const int t = threadIdx.x;
    // thread t: pair p0 - 1 + t, the first and the last only for the first step
    const bool out = t >= 1 && t <= n;
    if ((t & ~31) > n + 1) return;  // a warp without a pair (the barriers count the others)
    const int x0 = 2 * min(p0 - 1 + t, (gm.nx + 1) / 2 - 1);
    const int xw = max(x0 - 1, 0) - x0, xe = min(x0 + 2, gm.nx - 1) - x0;
    const int pitch = gm.pitch;

    auto porosity = [&](int y) {
        F2 v(1.f, 1.f);
        if constexpr (FIELD) v = F2(duo_ld<float2>(gm, phi, 4u * (uint32_t)(y * pitch + x0), 4));
        return v;
    };
    // both nodes in place; returns the new frames
    auto fluid = [&](Pair& p, ST& q0, ST& q1) {
        const Por<F2> por = por_of<F2, FIELD>(k, p.phi);
        const Sums<F2> s = sums_of(p.d, p.h);
        const Vel<F2> v = velocity<F2, true, FIELD>(k, por, s, op::mul(k.fu, p.c));
        if (out && too_fast(v)) atomicOr(status, 1);
        F2 next;
        const F2 shift = frame_next<T>(k, v.dT, p.c, next, q0, q1);
        collide_fluid<F2, FIELD, true>(k, por, s, v, shift, p.d, p.h);
        return next;
    };

    int m3 = (s0 - 1) % 3;
#pragma unroll 1
    for (int r = s0 - 1; r <= s1; ++r) {
        // rows of the slots: r, r - 1, r - 2 modulo the slots kept
        const int m3b = m3 == 0 ? 2 : m3 - 1, m3c = m3 == 2 ? 0 : m3 + 1;
        auto at = [&](int q, int age) {
            const int ns = duo_slots(q);
            const int sl = ns == 1 ? 0 : ns == 2 ? ((r - age) & 1) : ns == 4 ? ((r - age) & 3) : age == 0 ? m3 : age == 1 ? m3b : m3c;
            return sh + (duo_first(q) + sl) * W + 1 + t;
        };
        {
            // first step at row r, into shared memory
            if (r + kAhead <= s1) {
                // the rows that the first step reads kAhead iterations on, into L2: a
                // line per lane, two of each plane cover the warp's 64 nodes
                const int lane = t & 31, q = lane >> 1, i = q < 9 ? q : q - 9;
                const int up = 0x64 >> i & 1, down = 0x190 >> i & 1;  // e_y of f_i; g_j streams like f_j
                const int y = r + kAhead - up + down;
                const int xl = min(2 * (p0 - 1 + (t & ~31)) + 32 * (lane & 1), pitch - 1);
                if (q < 14) asm volatile("prefetch.global.L2 [%0];" ::"l"(src.f + (size_t)q * gm.plane + (size_t)y * pitch + xl));
            }
            Pair p;
            const uint32_t o = 4u * (uint32_t)(r * pitch + x0), step = 4u * (uint32_t)pitch;
            const uint32_t w = o + 4 * xw, e = o + 4 * xe;
            auto row_of = [&](uint32_t b, int i) { return ey9(i) == 0 ? b : ey9(i) > 0 ? b - step : b + step; };
            auto load = [&](const float* pl, int i) {
                if (ex9(i) == 0) return F2(duo_ld<float2>(gm, pl, row_of(o, i), 4));
                if (ex9(i) > 0) return F2(duo_ld<float>(gm, pl, row_of(w, i), 4), duo_ld<float>(gm, pl, row_of(o, i), 4));
                return F2(duo_ld<float>(gm, pl + 1, row_of(o, i), 4), duo_ld<float>(gm, pl, row_of(e, i), 4));
            };
#pragma unroll
            for (int i = 0; i < 9; ++i) p.d[i] = load(src.f + (size_t)i * gm.plane, i);
#pragma unroll
            for (int j = 0; j < 5; ++j) p.h[j] = load(src.g + (size_t)j * gm.plane, j);
            const uint32_t of = (uint32_t)(r * pitch + x0) * sizeof(ST), sf = (uint32_t)pitch * sizeof(ST);
            auto frame2 = [&](uint32_t b) {
                if constexpr (sizeof(ST) == 1) {
                    const char2 c = duo_ld<char2>(gm, src.t, b, 1);
                    return F2((float)(signed char)c.x, (float)(signed char)c.y);
                } else {
                    return F2(duo_ld<float2>(gm, src.t, b, 4));
                }
            };
            p.c = frame2(of);
            p.phi = porosity(r);
            pair_frames(k, p, frame2(of - sf), frame2(of + sf), (float)duo_ld<ST>(gm, src.t, of + xw * (int)sizeof(ST), sizeof(ST)),
                        (float)duo_ld<ST>(gm, src.t, of + xe * (int)sizeof(ST), sizeof(ST)));
            ST q0, q1;
            const F2 next = fluid(p, q0, q1);
#pragma unroll
            for (int i = 0; i < 9; ++i) *at(i, 0) = p.d[i].v;
#pragma unroll
            for (int j = 0; j < 5; ++j) *at(9 + j, 0) = p.h[j].v;
            *at(14, 0) = next.v;
        }
        __syncthreads();
        if (r > s0) {
            // second step at row r - 1, from the first step's rows r - 2, r - 1 and r
            Pair p;
            auto load = [&](int q, int i) {
                const float2* v = at(q, 1 + ey9(i));
                return ex9(i) == 0 ? F2(*v) : ex9(i) > 0 ? F2(v[-1].y, v->x) : F2(v->y, v[1].x);
            };
#pragma unroll
            for (int i = 0; i < 9; ++i) p.d[i] = load(i, i);
#pragma unroll
            for (int j = 0; j < 5; ++j) p.h[j] = load(9 + j, j);
            const float2* c = at(14, 1);
            p.c = F2(*c);
            p.phi = porosity(r - 1);
            pair_frames(k, p, F2(*at(14, 2)), F2(*at(14, 0)), c[-1].y, c[1].x);
            ST q0, q1;
            fluid(p, q0, q1);
            const int o = (r - 1) * pitch + x0;
            const uint32_t o2 = (uint32_t)o >> 1;
            if (out && in_plane(gm, o, 2)) {
                frame_st2<T>(dst.t + o, q0, q1);
#pragma unroll
                for (int i = 0; i < 9; ++i) ((float2*)(dst.f + (size_t)i * gm.plane))[o2] = p.d[i].v;
#pragma unroll
                for (int j = 0; j < 5; ++j) ((float2*)(dst.g + (size_t)j * gm.plane))[o2] = p.h[j].v;
            }
        }
        m3 = m3c;
    }
}

// A tile of nodes whose populations lie in shared memory, [population][node],
// the frame (in its unit) behind them.
struct TileSource {
    const float* v;
    const Coll<float>& k;
    int xa, ya, w, nodes;  // first node, width, nodes of the tile
    __device__ __forceinline__ float value(int q, int x, int y) const { return v[q * nodes + (y - ya) * w + (x - xa)]; }
    __device__ __forceinline__ float pulled(int x, int y, float (&d)[9], float (&h)[5]) const {
#pragma unroll
        for (int i = 0; i < 9; ++i) d[i] = value(i, x - ex9(i), y - ey9(i));
        const float F = value(14, x, y);
        h[0] = value(9, x, y);
#pragma unroll
        for (int j = 1; j < 5; ++j)
            h[j] = op::fma(k.w1, op::sub(value(14, x - ex9(j), y - ey9(j)), F), value(9 + j, x - ex9(j), y - ey9(j)));
        return F;
    }
    __device__ __forceinline__ float frame(int x, int y) const { return value(14, x, y); }
    __device__ __forceinline__ float heat_at(int x, int y, float& F) const {
        float d[9], h[5];
        F = op::mul(pulled(x, y, d, h), k.fu);
        return heat(h);
    }
};

// Both steps of the nodes [xa, xb) x [ya, yb) beside a wall: the first step of
// these nodes and of those within two along the wall and one across goes to
// shared memory, the second step pulls from it.
template <class T, bool FIELD, int THREADS>
__device__ __forceinline__ void duo_tile(const Src<T>& src, const Dst<T>& dst, const typename T::P* __restrict__ phi,
                                         const Geom& gm, const Coef<float>& c, int* __restrict__ status, int xa, int ya,
                                         int xb, int yb, int reach_x, int reach_y, float* sh) {
    const int xl = max(xa - reach_x, 0), yl = max(ya - reach_y, 0);
    const int w = min(xb + reach_x, gm.nx) - xl, h = min(yb + reach_y, gm.ny) - yl;
    const int t = threadIdx.x;
    const Coll<float>& k = c.k;
    for (int j = t; j < w * h; j += THREADS) {
        const int y = yl + j / w, x = xl + j % w;
        float d[9], g[5];
        const Post<float> p = core_post<T, FIELD>(k, gm, BufferSource<T>{c, gm, src}, phi, x, y, d, g);
        if (!p.wall && too_fast(p.v)) atomicOr(status, 1);
        typename FrameStore<T>::type code;
        float next;
        const float shift = frame_next<T>(k, p.dT, p.F, next, code);
        core_collide<T, FIELD>(k, p, shift, d, g);
#pragma unroll
        for (int i = 0; i < 9; ++i) sh[i * (w * h) + j] = d[i];
#pragma unroll
        for (int i = 0; i < 5; ++i) sh[(9 + i) * (w * h) + j] = g[i];
        sh[14 * (w * h) + j] = next;
    }
    __syncthreads();
    const TileSource tile{sh, k, xl, yl, w, w * h};
    for (int j = t; j < (xb - xa) * (yb - ya); j += THREADS) {
        const int y = ya + j / (xb - xa), x = xa + j % (xb - xa);
        float d[9], g[5];
        const Post<float> p = core_post<T, FIELD>(k, gm, tile, phi, x, y, d, g);
        if (!p.wall && too_fast(p.v)) atomicOr(status, 1);
        typename FrameStore<T>::type code;
        float next;
        const float shift = frame_next<T>(k, p.dT, p.F, next, code);
        core_collide<T, FIELD>(k, p, shift, d, g);
        const int o = y * gm.pitch + x;
        if (in_plane(gm, o)) {
            dst.t[o] = code;
#pragma unroll
            for (int i = 0; i < 9; ++i) dst.f[(size_t)i * gm.plane + o] = d[i];
#pragma unroll
            for (int i = 0; i < 5; ++i) dst.g[(size_t)i * gm.plane + o] = g[i];
        }
    }
}

// The tiles along the walls: rows 0, 1 and ny - 2, ny - 1 in pieces of
// duo_along_x nodes, then the columns beside the x walls of the rows between,
// in pieces of duo_along_y nodes (with the first step's surround a node per
// thread).
__host__ __device__ constexpr int duo_along_x(int threads) { return threads / 3 - 4; }
__host__ __device__ constexpr int duo_along_y(int threads) { return threads / 4 - 2; }
__host__ __device__ inline int duo_tiles_x(int nx, int threads) {
    return (nx + duo_along_x(threads) - 1) / duo_along_x(threads);
}
__host__ __device__ inline int duo_tiles_y(int ny, int threads) {
    return (ny - 4 + duo_along_y(threads) - 1) / duo_along_y(threads);
}
__host__ __device__ inline int duo_tiles(int nx, int ny, int threads) {
    return 2 * duo_tiles_x(nx, threads) + 2 * duo_tiles_y(ny, threads);
}

// Wall tile i of a lattice.
template <class T, bool FIELD, int THREADS>
__device__ __forceinline__ void duo_wall_block(int i, const Src<T>& src, const Dst<T>& dst,
                                               const typename T::P* __restrict__ phi, const Geom& gm,
                                               const Coef<float>& c, int* __restrict__ status, float* sh) {
    const int nx = gm.nx, ny = gm.ny, tx = duo_tiles_x(nx, THREADS), ty = duo_tiles_y(ny, THREADS);
    int xa, xb, ya, yb, rx, ry;
    if (i < 2 * tx) {
        const bool top = i >= tx;
        xa = (top ? i - tx : i) * duo_along_x(THREADS);
        xb = min(xa + duo_along_x(THREADS), nx);
        ya = top ? ny - 2 : 0;
        yb = ya + 2;
        rx = 2;
        ry = 1;
    } else {
        i -= 2 * tx;
        const bool right = i >= ty;
        ya = 2 + (right ? i - ty : i) * duo_along_y(THREADS);
        yb = min(ya + duo_along_y(THREADS), ny - 2);
        xa = right ? 2 * duo_last_pair(nx) + 2 : 0;
        xb = right ? nx : 2;
        rx = ry = 1;
    }
    duo_tile<T, FIELD, THREADS>(src, dst, phi, gm, c, status, xa, ya, xb, yb, rx, ry, sh);
}

// March b of a lattice: strips of `width` pairs, side by side, by segments of
// `rows` rows.
template <class T, bool FIELD, int THREADS>
__device__ __forceinline__ void duo_march_block(int b, const Src<T>& src, const Dst<T>& dst,
                                                const typename T::P* __restrict__ phi, const Geom& gm,
                                                const Coll<float>& k, int* __restrict__ status, int strips, int width,
                                                int rows, float2* sh) {
    const int strip = b % strips, seg = b / strips;
    const int p0 = duo_first_pair() + strip * width, s0 = 2 + seg * rows;
    duo_march<T, FIELD, THREADS>(src, dst, phi, gm, k, status, p0, min(width, duo_last_pair(gm.nx) - p0 + 1), s0,
                                 min(s0 + rows, gm.ny - 2), sh);
}

}  // namespace lbm
