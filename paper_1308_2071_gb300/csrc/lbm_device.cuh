// Device building blocks of the coupled D2Q9 / D2Q5 MRT lattice Boltzmann step
// (Liu, He, Li, Tao, arXiv:1308.2071, Section 3) on the side-heated cavity of
// Section 4.
//
// Populations are held as deviations from the rest state of the initial
// condition: d_i = f_i - w_i rho0 (D2Q9) and h_j = g_j - w~_j T0 (D2Q5).  The
// model is affine in that shift (sum_i e_i w_i = 0, M w rho0 = rho0 (1, -2, 1,
// 0, ...), N w~ T0 = T0 (1, 0, 0, varpi, 0)), so every formula below is the
// paper's formula minus its value at rest, with rho0 = 1 and delta_t = 1
// (Section 4).  Deviations are O(Ma^2) and O(Delta T), which keeps FP32 and
// FP16 storage accurate.
//
// Storage layout (structure of arrays): plane q of a buffer holds population
// q for every node, row-major with x fastest and a row pitch (in elements)
// that makes every row start on a 128-byte boundary; planes 0..8 are f
// (Eq. 8 order: rest, E, N, W, S, NE, NW, SW, SE), planes 9..13 are g (Eq. 26
// order: rest, E, N, W, S).  Flow and thermal planes may use different
// storage types (see PrecF16); both use the same pitch in elements.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

namespace lbm {

// ---- lattice -----------------------------------------------------------------

// D2Q9 velocity components of Eq. 8 (c = 1).
__host__ __device__ constexpr int ex9(int i) {
    return (i == 1 || i == 5 || i == 8) ? 1 : (i == 3 || i == 6 || i == 7) ? -1 : 0;
}
__host__ __device__ constexpr int ey9(int i) {
    return (i == 2 || i == 5 || i == 6) ? 1 : (i == 4 || i == 7 || i == 8) ? -1 : 0;
}
// D2Q9 weights (stated after Eq. 13).
__host__ __device__ constexpr double w9(int i) {
    return i == 0 ? 4.0 / 9.0 : (i <= 4 ? 1.0 / 9.0 : 1.0 / 36.0);
}
// D2Q5 velocities of Eq. 26 are the first five D2Q9 velocities.

constexpr int NPOP = 14;  // 9 flow + 5 thermal planes per buffer

// ---- storage conversions ------------------------------------------------------

// CG = false: read-only (non-coherent) cached loads, for buffers never
// written during the launch.  CG = true: coherent loads (ld.global.ca), for
// kernels that read data other blocks of the same launch wrote (the
// persistent batched kernel): a weak load observes every write that happens
// before it through the kernel's release/acquire synchronisation (the grid
// barrier, or the dataflow schedule's wait), and may hit L1, which the
// neighbouring nodes' shifted pulls and frames reuse; the non-coherent path
// of __ldg gives no such guarantee within a launch.
template <class S, class R, bool CG = false> struct Conv;
template <bool CG> struct Conv<double, double, CG> {
    static __device__ __forceinline__ double ld(const double* p) { return CG ? __ldca(p) : __ldg(p); }
    static __device__ __forceinline__ void st(double* p, double v) { *p = v; }
};
template <bool CG> struct Conv<float, float, CG> {
    static __device__ __forceinline__ float ld(const float* p) { return CG ? __ldca(p) : __ldg(p); }
    static __device__ __forceinline__ void st(float* p, float v) { *p = v; }
};
template <bool CG> struct Conv<__half, float, CG> {
    static __device__ __forceinline__ float ld(const __half* p) { return __half2float(CG ? __ldca(p) : __ldg(p)); }
    static __device__ __forceinline__ void st(__half* p, float v) { *p = __float2half_rn(v); }
};

// Two nodes side by side along x, starting at an even x: every row starts on
// a 128-byte boundary, so the pair is one aligned 2-element access.
template <class S, class R, bool CG = false> struct Conv2;
template <bool CG> struct Conv2<double, double, CG> {
    static __device__ __forceinline__ double2 ld(const double* p) {
        return CG ? __ldca((const double2*)p) : __ldg((const double2*)p);
    }
    static __device__ __forceinline__ void st(double* p, double a, double b) { *(double2*)p = make_double2(a, b); }
};
template <bool CG> struct Conv2<float, float, CG> {
    static __device__ __forceinline__ float2 ld(const float* p) {
        return CG ? __ldca((const float2*)p) : __ldg((const float2*)p);
    }
    static __device__ __forceinline__ void st(float* p, float a, float b) { *(float2*)p = make_float2(a, b); }
};
template <bool CG> struct Conv2<__half, float, CG> {
    static __device__ __forceinline__ float2 ld(const __half* p) {
        return __half22float2(CG ? __ldca((const __half2*)p) : __ldg((const __half2*)p));
    }
    static __device__ __forceinline__ void st(__half* p, float a, float b) { *(__half2*)p = __floats2half2_rn(a, b); }
};

// ---- precision variants -----------------------------------------------------------
// SF: storage of the nine flow planes, SG: storage of the five thermal planes,
// R: arithmetic, P: storage of a per-cell porosity field.
struct PrecF64 {
    using SF = double;
    using SG = double;
    using R = double;
    using P = double;
    static constexpr bool cg = false;
};
struct PrecF32 {
    using SF = float;
    using SG = float;
    using R = float;
    using P = float;
    static constexpr bool cg = false;
};
// Storage with a per-node temperature frame: one more plane holds F(x), the
// node's T - T0 when the node was last written, rounded to the frame's
// storage type ST, and the thermal planes hold g_j - w~_j (T0 + F(x)) instead
// of g_j - w~_j T0.  The stored thermal values are then the small
// non-equilibrium parts, so FP32 resolves the per-step change of T even where
// |T - T0| is near 1/2 (about 1e-8 per step on a 1024^2 lattice, against the
// 3e-8 spacing of FP32 numbers near 0.3, where plain deviations lose it).
//
// PrecF32T: the frame in FP32.  PrecF32Q: the frame as an 8-bit integer k,
// F = k fq with fq a power of two (Coef::fq), so that F(x) - F(x') and the
// frame change of a node are exact in FP32 and the frame costs one byte per
// node each way.  The remainder |T - T0 - F| <= fq / 2 is then small enough
// that FP32 keeps the slow evolution (checked against FP64 over 50,000 steps).
struct PrecF32T : PrecF32 {
    static constexpr bool framed = true;
    using ST = float;
};
struct PrecF32Q : PrecF32 {
    static constexpr bool framed = true;
    using ST = int8_t;
};
// FP16 flow deviations (|d| stays near 1e-2, where half rounds to ~4e-6) with
// FP32 thermal deviations relative to the 8-bit frame of PrecF32Q (thermal
// deviations reach w~_0 (T_h - T0) = 0.3 at the hot wall, where half would
// round to ~1.2e-4 and drift the temperature field).
struct PrecF16 {
    using SF = __half;
    using SG = float;
    using R = float;
    using P = float;
    static constexpr bool cg = false;
    static constexpr bool framed = true;
    using ST = int8_t;
};
// FP32 and FP64 storage run the collision of lbm_core.cuh; FP16 flow storage
// keeps the direct form below, whose dithered rounding (dither_to_half)
// follows the low bits of every value.
template <class T> struct Core {
    static constexpr bool value = !std::is_same<typename T::SF, __half>::value;
};
template <class T, class = void> struct Framed {
    static constexpr bool value = false;
};
template <class T> struct Framed<T, decltype((void)T::framed)> {
    static constexpr bool value = T::framed;
};
// Storage type of the frame plane (the thermal type when there is none).
template <class T, class = void> struct FrameStore {
    using type = typename T::SG;
};
template <class T> struct FrameStore<T, decltype((void)sizeof(typename T::ST))> {
    using type = typename T::ST;
};

// Same arithmetic, L2-only loads (persistent kernels).
struct PrecF64P : PrecF64 {
    static constexpr bool cg = true;
};
struct PrecF32P : PrecF32 {
    static constexpr bool cg = true;
};
struct PrecF32TP : PrecF32P {
    static constexpr bool framed = true;
    using ST = float;
};
struct PrecF32QP : PrecF32P {
    static constexpr bool framed = true;
    using ST = int8_t;
};

// Read-only typed view of one state buffer: 9 flow planes then 5 thermal
// planes (then, for framed storage, the frame plane t).
template <class T> struct Src {
    const typename T::SF* __restrict__ f;
    const typename T::SG* __restrict__ g;
    const typename FrameStore<T>::type* __restrict__ t;
};
template <class T> struct Dst {
    typename T::SF* __restrict__ f;
    typename T::SG* __restrict__ g;
    typename FrameStore<T>::type* __restrict__ t;
};
template <class T> __host__ __device__ inline Src<T> src_view(const void* base, int plane) {
    Src<T> s;
    s.f = (const typename T::SF*)base;
    s.g = (const typename T::SG*)((const char*)base + (size_t)9 * plane * sizeof(typename T::SF));
    s.t = (const typename FrameStore<T>::type*)(s.g + (size_t)5 * plane);
    return s;
}
template <class T> __host__ __device__ inline Dst<T> dst_view(void* base, int plane) {
    Dst<T> d;
    d.f = (typename T::SF*)base;
    d.g = (typename T::SG*)((char*)base + (size_t)9 * plane * sizeof(typename T::SF));
    d.t = (typename FrameStore<T>::type*)(d.g + (size_t)5 * plane);
    return d;
}
template <class T> __host__ __device__ constexpr size_t buffer_bytes(int plane) {
    return (size_t)plane * (9 * sizeof(typename T::SF) + 5 * sizeof(typename T::SG) +
                            (Framed<T>::value ? sizeof(typename FrameStore<T>::type) : 0));
}

// ---- two nodes in one register pair ------------------------------------------------

// FP32 values of two nodes side by side.  Each +, -, * is one paired FP32
// instruction for both nodes (sm_100-class GPUs), rounded to nearest like its
// scalar counterpart; the pair is never fused into an FMA, so a result may
// differ from the scalar path's (which the compiler contracts) by a rounding.
// Division and sqrt are taken per component.  The type and its functions
// live in a namespace of their own, so that sqrt(float) here keeps meaning
// the CUDA function while sqrt(F2) is found by argument-dependent lookup.
namespace x2 {
struct F2 {
    float2 v;
    F2() = default;
    __device__ __forceinline__ F2(float2 a) : v(a) {}
    __device__ __forceinline__ F2(float a, float b) : v(make_float2(a, b)) {}
    __device__ __forceinline__ explicit F2(double c) : v(make_float2((float)c, (float)c)) {}
    __device__ __forceinline__ explicit F2(float c) : v(make_float2(c, c)) {}
    __device__ __forceinline__ explicit F2(int c) : v(make_float2((float)c, (float)c)) {}
};
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return F2(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ F2 operator*(F2 a, F2 b) { return F2(__fmul2_rn(a.v, b.v)); }
// a - b = a + (-1) b: the product is exact, so this rounds once, as a subtraction does
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return F2(__ffma2_rn(b.v, make_float2(-1.f, -1.f), a.v)); }
__device__ __forceinline__ F2 operator-(F2 a) { return F2(-a.v.x, -a.v.y); }
__device__ __forceinline__ F2 operator/(F2 a, F2 b) { return F2(a.v.x / b.v.x, a.v.y / b.v.y); }
__device__ __forceinline__ F2 operator+(float a, F2 b) { return F2(a) + b; }
__device__ __forceinline__ F2 operator+(F2 a, float b) { return a + F2(b); }
__device__ __forceinline__ F2 operator-(float a, F2 b) { return F2(a) - b; }
__device__ __forceinline__ F2 operator-(F2 a, float b) { return a - F2(b); }
__device__ __forceinline__ F2 operator*(float a, F2 b) { return F2(a) * b; }
__device__ __forceinline__ F2 operator*(F2 a, float b) { return a * F2(b); }
__device__ __forceinline__ F2 sqrt(F2 a) { return F2(sqrtf(a.v.x), sqrtf(a.v.y)); }
}  // namespace x2
using x2::F2;

// FP16 flow storage: moves each FP32 flow value onto the half-precision grid
// (13 low mantissa bits cleared) with the rounding threshold taken from the
// low mantissa bits of two other populations of the node, instead of
// rounding to nearest.  Those bits change from step to step and do not
// depend on the value rounded, so the rounding error averages out over the
// steps instead of repeating: rounded to nearest, a slowly changing value
// is rounded the same way step after step, and the slow Darcy relaxation
// integrates that bias into the velocity.  The store's conversion to half
// is then exact (in half's normal range; below 2^-14 it rounds once more).
// The threshold is added to the bit pattern, whose low 31 bits are the
// magnitude for either sign.  NaN passes unchanged (infinities stay
// infinite).
__device__ __forceinline__ void dither_to_half(float (&v)[9]) {
    uint32_t b[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) b[i] = __float_as_uint(v[i]);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const uint32_t r = (b[(i + 1) % 9] ^ b[(i + 5) % 9]) & 0x1fffu;
        const float m = __uint_as_float((b[i] + r) & 0xffffe000u);
        v[i] = v[i] != v[i] ? v[i] : m;
    }
}

// ---- per-launch coefficients ----------------------------------------------------

// The collision's constants as lbm_core.cuh uses them (FP32 and FP64 storage
// variants), derived from the rates and parameters on the host in FP64.
template <class R> struct Coll {
    R hb;                        // phi g beta / 2 (porosity field: g beta / 2)
    R cc, ec, l1;                // c_lin / 4, cc + cc^2, c_quad / 2 (field: a_lin / 4, 0, a_quad / 2)
    R iphi, niphi;               // 1 / phi, -1 / phi of the uniform porosity
    R qhalf;                     // Q / (2 sigma)
    R a0, a1, a2;                // rest population: of m_0, z, E
    R b0, b1, b2;                // axis populations
    R c0, c1, c2;                // diagonal populations
    R k7, f7, k8, f8;            // stress moments: of m - m_eq, of the forcing product
    R s4a, s4d, s6a, s6d;        // energy-flux moments: axis and diagonal part
    R s3, s4, s5, s6, f5, f6;    // wall nodes: rates and force factors of m_3 .. m_6, in sixths
    R is, Tis, nis, nTis;        // 1 / sigma, T_0 / sigma, and their negatives
    R q0, q1;                    // heat source per step of the rest and moving populations
    R t4, h4, t1, h1;            // n_3: of the sum of the moving populations and of the rest population
    R z1, z2, z4, nz4;           // n_1, n_2, n_4
    R fu, ifu;                   // unit of the stored frames (8-bit: the quantum; FP32: 1), its inverse
    R w1, nw0, nw1;              // w~_1 fu, -w~_0 fu, -w~_1 fu
    R wt0, wt1;                  // w~_0, w~_1
    R dTh, dTc, gb;              // wall temperatures minus T0, g beta
};

// Everything a step needs besides the buffers.  Each storage variant's kernels take
// what they use: a launch's time grows with its parameters (FP16, 64^2: 0.2 us per
// step more with both forms' constants in one struct of 408 bytes).
//
// FP32 and FP64 storage, in the arithmetic type R.
template <class R> struct Coef {
    Coll<R> k;
    R dTh, dTc;  // wall temperatures minus T0
    R T0;
    R varpi;     // D2Q5 constant (Eq. 29)
    R qhalf;     // Q / (2 sigma), the source part of Eq. 36
    R phi;       // uniform porosity
};

// FP16 flow storage: the direct form's.
struct Direct {
    float s[9];       // flow relaxation rates (Eq. 20)
    float hs[9];      // 1 - s_k / 2
    float z[5];       // thermal relaxation rates (Eq. 31)
    float hz[5];      // 1 - zeta_k / 2
    float gbeta;      // g beta (buoyancy G = g beta (T - T0) j, Section 2)
    float dTh, dTc;   // wall temperatures minus T0
    float T0;
    float inv_sigma;  // 1 / sigma
    float varpi;      // D2Q5 constant (Eq. 29)
    float inv_csT2;   // 1 / c_sT^2 = 10 / (4 + varpi)
    float wt0, wt1;   // D2Q5 weights w~_0 = (1 - varpi)/5, w~_i = (4 + varpi)/20
    float psi0, psi3; // Psi_0 = Q/sigma, Psi_3 = varpi Q/sigma (Eq. 30)
    float qhalf;      // Q / (2 sigma), the source part of Eq. 36
    float phi;        // uniform porosity
    float c_lin;      // phi nu / K         (uniform porosity)
    float c_quad;     // phi F_phi / sqrt K (uniform porosity)
    float a_lin;      // per-cell: phi nu / K      = a_lin  (1 - phi)^2 / phi^2
    float a_quad;     // per-cell: phi F_phi / sqrt K = a_quad (1 - phi) / phi^2
    float fq, ifq;    // 8-bit temperature frames: quantum (a power of two) and its inverse
    float wt1fq;      // w~_1 fq (exact: fq is a power of two)
};
template <class T> using CoefOf = std::conditional_t<Core<T>::value, Coef<typename T::R>, Direct>;
static_assert(sizeof(Direct) == 48 * sizeof(float), "what a launch of the direct form carries");

// Geometry of one lattice in one pair of buffers.
struct Geom {
    int nx, ny;
    int pitch;        // elements per row
    int plane;        // elements per population plane (pitch * ny)
    int thermal_bc;   // 0 side-heated, 1 cooled
    int adi_order;    // 1 or 2
#ifdef LBM_BOUNDS_CHECK
    int* oob;         // counter of accesses outside their plane (bounds-checked build)
#endif
};

// Bounds-checked build (LBM_BOUNDS_CHECK): every population, frame and
// porosity access of the step's pull, wall rule and stores is checked against
// its plane [0, plane) first; an access outside it is skipped (a load reads 0)
// and counted in *gm.oob.  In the normal build the check is compiled away.
__device__ __forceinline__ bool in_plane(const Geom& gm, int o, int n = 1) {
#ifdef LBM_BOUNDS_CHECK
    if (o >= 0 && o <= gm.plane - n) return true;
    atomicAdd(gm.oob, 1);
    return false;
#else
    (void)gm, (void)o, (void)n;
    return true;
#endif
}

// Porosity-dependent drag coefficients (Eq. 4 and Eq. 5 per cell).
template <class R> struct Drag {
    R phi, iphi, c_lin, c_quad;
};

// Drag coefficients of one cell from its porosity (FIELD) or the uniform ones.
template <class R, bool FIELD>
__device__ __forceinline__ Drag<R> drag_of(const Direct& c, R phi) {
    Drag<R> dr;
    if constexpr (FIELD) {
        R iphi = R(1) / phi;
        R om = R(1) - phi;
        R ip2 = iphi * iphi;
        dr.phi = phi;
        dr.iphi = iphi;
        dr.c_lin = c.a_lin * om * om * ip2;
        dr.c_quad = c.a_quad * om * ip2;
    } else {
        dr.phi = c.phi;
        dr.iphi = R(1) / c.phi;
        dr.c_lin = c.c_lin;
        dr.c_quad = c.c_quad;
    }
    return dr;
}

template <class R, bool FIELD, class P>
__device__ __forceinline__ Drag<R> drag_at(const Direct& c, const P* phi_field, int off) {
    if constexpr (FIELD) return drag_of<R, true>(c, Conv<P, R>::ld(phi_field + off));
    return drag_of<R, false>(c, R(0));
}
template <class R, bool FIELD, class P>
__device__ __forceinline__ Drag<R> drag_at(const Direct& c, const Geom& gm, const P* phi_field, int off) {
    if constexpr (FIELD) return drag_at<R, FIELD, P>(c, phi_field, in_plane(gm, off) ? off : 0);
    return drag_of<R, false>(c, R(0));
}

// Element off + delta of a plane, off (a thread's node) apart from delta (the same
// for all threads): the plane's address with delta stays in uniform registers
// and one 32-bit byte offset serves every access of a node.  (A plane has fewer
// than 2^31 / 14 nodes, so the offset fits.)  For node pairs, where an index per
// access made up a fifth of the instructions: us per step 4.55 -> 4.27 on 601 x
// 397 with a porosity field, 4.25 -> 4.16 on 500^2.  Single nodes keep indices,
// which the on-chip tiles and FP64 run 0.5 % faster with.
template <class S> __device__ __forceinline__ const S* at(const S* plane, int delta, int off) {
    return (const S*)((const char*)(plane + delta) + (uint32_t)off * (uint32_t)sizeof(S));
}
template <class S> __device__ __forceinline__ S* at(S* plane, int delta, int off) {
    return (S*)((char*)(plane + delta) + (uint32_t)off * (uint32_t)sizeof(S));
}

// ---- temperature frames -------------------------------------------------------------

// FP16 flow storage: a frame is an 8-bit integer k with F = k fq.
template <class T> __device__ __forceinline__ float frame_ld(const Direct& c, const int8_t* p) {
    const int8_t k = T::cg ? __ldca((const signed char*)p) : __ldg((const signed char*)p);
    return (float)(int)k * c.fq;
}

// The frame a node takes for temperature deviation v, as it will read back,
// and its stored form.
__device__ __forceinline__ float frame_make(const Direct& c, float v, int8_t& code) {
    // a NaN or an overflowing value saturates (the divergence flag reports it)
    const float k = fminf(fmaxf(rintf(v * c.ifq), -128.f), 127.f);
    code = (int8_t)(int)k;
    return k * c.fq;
}

// The stored code k of an 8-bit frame (F = k fq), and of a node pair.
template <class T>
__device__ __forceinline__ int frame_code(const typename FrameStore<T>::type* p) {
    return (int)(T::cg ? __ldca((const signed char*)p) : __ldg((const signed char*)p));
}
template <class T>
__device__ __forceinline__ char2 frame_pair_code(const typename FrameStore<T>::type* p) {
    return T::cg ? __ldca((const char2*)p) : __ldg((const char2*)p);
}

// Stores the frames of the node pair (x0, x0 + 1), x0 even.
template <class T>
__device__ __forceinline__ void frame_st2(typename FrameStore<T>::type* p, typename FrameStore<T>::type a,
                                          typename FrameStore<T>::type b) {
    if constexpr (sizeof(typename FrameStore<T>::type) == 1)
        *(char2*)p = make_char2((char)a, (char)b);
    else
        Conv2<typename FrameStore<T>::type, typename FrameStore<T>::type, T::cg>::st(p, a, b);
}

// ---- pull of one node ------------------------------------------------------------

// f_i(x, t+1) = f_i^+(x - e_i, t) (Eq. 18) and g_j likewise (Eq. 35).
// off = y * pitch + x of the receiving node.
template <class T>
__device__ __forceinline__ void pull(const Src<T>& src, const Geom& gm, int off,
                                     typename T::R (&d)[9], typename T::R (&h)[5]) {
    using R = typename T::R;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int o = off - ey9(i) * gm.pitch - ex9(i);
        d[i] = in_plane(gm, o) ? Conv<typename T::SF, R, T::cg>::ld(src.f + i * gm.plane + o) : R(0);
    }
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const int o = off - ey9(j) * gm.pitch - ex9(j);
        h[j] = in_plane(gm, o) ? Conv<typename T::SG, R, T::cg>::ld(src.g + j * gm.plane + o) : R(0);
    }
}

// The pull of the node pair off0, off0 + 1 (x0 even): populations with
// e_x = 0 come as one aligned pair access, the others (shifted by one node)
// as two single accesses.
template <class T>
__device__ __forceinline__ void pull_x2(const Src<T>& src, const Geom& gm, int off0, typename T::R (&d0)[9],
                                        typename T::R (&h0)[5], typename T::R (&d1)[9], typename T::R (&h1)[5]) {
    using R = typename T::R;
    using SF = typename T::SF;
    using SG = typename T::SG;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int e = -ey9(i) * gm.pitch - ex9(i), o = off0 + e;
        const SF* p = at(src.f, i * gm.plane + e, off0);
        if (ex9(i) == 0) {
            const auto v = in_plane(gm, o, 2) ? Conv2<SF, R, T::cg>::ld(p) : decltype(Conv2<SF, R, T::cg>::ld(p)){};
            d0[i] = v.x;
            d1[i] = v.y;
        } else {
            d0[i] = in_plane(gm, o) ? Conv<SF, R, T::cg>::ld(p) : R(0);
            d1[i] = in_plane(gm, o + 1) ? Conv<SF, R, T::cg>::ld(p + 1) : R(0);
        }
    }
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const int e = -ey9(j) * gm.pitch - ex9(j), o = off0 + e;
        const SG* p = at(src.g, j * gm.plane + e, off0);
        if (ex9(j) == 0) {
            const auto v = in_plane(gm, o, 2) ? Conv2<SG, R, T::cg>::ld(p) : decltype(Conv2<SG, R, T::cg>::ld(p)){};
            h0[j] = v.x;
            h1[j] = v.y;
        } else {
            h0[j] = in_plane(gm, o) ? Conv<SG, R, T::cg>::ld(p) : R(0);
            h1[j] = in_plane(gm, o + 1) ? Conv<SG, R, T::cg>::ld(p + 1) : R(0);
        }
    }
}

// frame_in for the node pair off0, off0 + 1 (x0 even): the pair's own frames
// and those of the rows above and below come as pairs, the east and west
// neighbours' as single values.
template <class T>
__device__ __forceinline__ void frame_in_x2(const Direct& c, const Src<T>& src, const Geom& gm, int off0, float (&h0)[5],
                                            float (&h1)[5], float& F0, float& F1) {
    using R = float;
    // differences taken on the integers, as in frame_in
    char2 own = make_char2(0, 0), sth = own, nth = own;
    signed char w = 0, e = 0;
    if (in_plane(gm, off0, 2)) own = frame_pair_code<T>(at(src.t, 0, off0));
    if (in_plane(gm, off0 - gm.pitch, 2)) sth = frame_pair_code<T>(at(src.t, -gm.pitch, off0));  // j = 2: y - 1
    if (in_plane(gm, off0 + gm.pitch, 2)) nth = frame_pair_code<T>(at(src.t, gm.pitch, off0));  // j = 4: y + 1
    if (in_plane(gm, off0 - 1)) w = (signed char)frame_code<T>(at(src.t, -1, off0));
    if (in_plane(gm, off0 + 2)) e = (signed char)frame_code<T>(at(src.t, 2, off0));
    const int k0 = (signed char)own.x, k1 = (signed char)own.y;
    h0[1] += c.wt1fq * R((int)w - k0);
    h1[1] += c.wt1fq * R(k0 - k1);
    h0[2] += c.wt1fq * R((int)(signed char)sth.x - k0);
    h1[2] += c.wt1fq * R((int)(signed char)sth.y - k1);
    h0[3] += c.wt1fq * R(k1 - k0);
    h1[3] += c.wt1fq * R((int)e - k1);
    h0[4] += c.wt1fq * R((int)(signed char)nth.x - k0);
    h1[4] += c.wt1fq * R((int)(signed char)nth.y - k1);
    F0 = R(k0) * c.fq;
    F1 = R(k1) * c.fq;
}

// FP16 flow storage: thermal values pulled into node off were stored in the
// frames of the nodes they came from; re-express them in this node's frame F
// (add w~_j (F(x - e_j) - F), j >= 1: w~_1 (F_s - F) = (w~_1 fq) (k_s - k), the
// difference taken on the integers) and return F.
template <class T>
__device__ __forceinline__ float frame_in(const Direct& c, const Src<T>& src, const Geom& gm, int off, float (&h)[5]) {
    const int k = in_plane(gm, off) ? frame_code<T>(src.t + off) : 0;
#pragma unroll
    for (int j = 1; j < 5; ++j) {
        const int o = off - ey9(j) * gm.pitch - ex9(j);
        h[j] += c.wt1fq * (float)((in_plane(gm, o) ? frame_code<T>(src.t + o) : 0) - k);
    }
    return (float)k * c.fq;
}

// ---- macroscopic values -------------------------------------------------------------

template <class R> struct Macro {
    R ux, uy;  // velocity (Eq. 21)
    R dP;      // phi p - rho0 c_s^2 (Eq. 23)
    R dT;      // T - T0 (Eq. 36)
    R Fx, Fy;  // total force (Eq. 4)
    R umag;    // |u|
    R F, dTl;  // the node's frame and T - T0 - F (no frames: 0 and dT)
};

// Eq. 36, Section 2 buoyancy, Eq. 22, Eq. 21, Eq. 23, Eq. 4 at a fluid node (R:
// float, or F2 for a node pair).  The thermal values h are relative to the
// frame F.
template <class R>
__device__ __forceinline__ Macro<R> fluid_macros(const Direct& c, const Drag<R>& dr, const R (&d)[9], const R (&h)[5],
                                                 R F) {
    Macro<R> m;
    const R n0 = h[0] + h[1] + h[2] + h[3] + h[4];
    m.F = F;
    m.dTl = n0 + c.qhalf;
    m.dT = F + m.dTl;
    const R Gy = c.gbeta * m.dT;
    const R jx = (d[1] - d[3]) + (d[5] - d[6]) - (d[7] - d[8]);
    const R jy = (d[2] - d[4]) + (d[5] + d[6]) - (d[7] + d[8]);
    const R by = R(0.5) * dr.phi * Gy;  // half the buoyancy impulse
    const R vx = jx;
    const R vy = jy + by;
    // Eq. 22
    const R l1 = R(0.5) * dr.c_quad;
    const R vm = sqrt(vx * vx + vy * vy);
    const R l0 = R(0.5) + R(0.25) * dr.c_lin;
    const R den = R(1) / (l0 + sqrt(l0 * l0 + l1 * vm));
    m.ux = vx * den;
    m.uy = vy * den;
    m.umag = vm * den;
    const R uu = m.ux * m.ux + m.uy * m.uy;
    const R s18 = (d[1] + d[2] + d[3] + d[4]) + (d[5] + d[6] + d[7] + d[8]);
    // c_s^2 / (1 - w_0) = 3/5 and rho0 s_0(u) = -(2/3) |u|^2 / phi
    m.dP = R(0.6) * s18 - R(0.4) * uu * dr.iphi;
    const R drag = dr.c_lin + dr.c_quad * m.umag;
    m.Fx = -drag * m.ux;
    m.Fy = -drag * m.uy + dr.phi * Gy;
    return m;
}

// ---- collision ------------------------------------------------------------------------

// Eq. 17 with m_eq of Eq. 16 and S of Eq. 19, then f+ = M^-1 m+ (Eq. 18,
// M^-1 = M^T diag(1/9, 1/36, 1/36, 1/6, 1/12, 1/6, 1/12, 1/4, 1/4));
// Eq. 34 with n_eq of Eq. 29 and Psi of Eq. 30, then g+ = N^-1 n+ (Eq. 35,
// N^-1 = N^T diag(1/5, 1/2, 1/2, 1/20, 1/4)).  In place on d and h.  FP16 flow
// storage; the FP32 and FP64 variants run the increments of lbm_core.cuh.
template <class R>
__device__ __forceinline__ void collide(const Direct& c, R iphi, const Macro<R>& mc, R (&d)[9], R (&h)[5]) {
    // m = M d (Eq. 9-11), as a deviation from the rest moments
    const R a = (d[1] + d[2]) + (d[3] + d[4]);
    const R b = (d[5] + d[6]) + (d[7] + d[8]);
    const R ex13 = d[1] - d[3], ey24 = d[2] - d[4];
    const R dx = (d[5] - d[6]) - (d[7] - d[8]);  // diagonal x-momentum
    const R dy = (d[5] + d[6]) - (d[7] + d[8]);  // diagonal y-momentum
    const R m0 = d[0] + a + b;
    const R m1 = R(-4) * d[0] - a + R(2) * b;
    const R m2 = R(4) * d[0] - R(2) * a + b;
    const R m4 = R(-2) * ex13 + dx;
    const R m6 = R(-2) * ey24 + dy;
    const R m7 = (d[1] - d[2]) + (d[3] - d[4]);
    const R m8 = (d[5] - d[6]) + (d[7] - d[8]);

    // m_eq (Eq. 16) minus rest moments
    const R ux = mc.ux, uy = mc.uy;
    const R uu = ux * ux + uy * uy;
    const R q = R(3) * uu * iphi;
    const R eq1 = R(6) * mc.dP + q;
    const R eq2 = R(-9) * mc.dP - q;
    const R eq7 = (ux * ux - uy * uy) * iphi;
    const R eq8 = ux * uy * iphi;
    // S (Eq. 19)
    const R uF = ux * mc.Fx + uy * mc.Fy;
    const R S1 = R(6) * uF * iphi;
    const R S7 = R(2) * (ux * mc.Fx - uy * mc.Fy) * iphi;
    const R S8 = (ux * mc.Fy + uy * mc.Fx) * iphi;

    // Eq. 17, scaled by the diagonal of M^-1
    const R m3 = ex13 + dx, m5 = ey24 + dy;
    const R p0 = (m0 - c.s[0] * m0) * R(1.0 / 9.0);
    const R p1 = (m1 - c.s[1] * (m1 - eq1) + c.hs[1] * S1) * R(1.0 / 36.0);
    const R p2 = (m2 - c.s[2] * (m2 - eq2) - c.hs[2] * S1) * R(1.0 / 36.0);
    const R p3 = (m3 - c.s[3] * (m3 - ux) + c.hs[3] * mc.Fx) * R(1.0 / 6.0);
    const R p4 = (m4 - c.s[4] * (m4 + ux) - c.hs[4] * mc.Fx) * R(1.0 / 12.0);
    const R p5 = (m5 - c.s[5] * (m5 - uy) + c.hs[5] * mc.Fy) * R(1.0 / 6.0);
    const R p6 = (m6 - c.s[6] * (m6 + uy) - c.hs[6] * mc.Fy) * R(1.0 / 12.0);
    const R p7 = (m7 - c.s[7] * (m7 - eq7) + c.hs[7] * S7) * R(0.25);
    const R p8 = (m8 - c.s[8] * (m8 - eq8) + c.hs[8] * S8) * R(0.25);

    // f+ = M^T p (columns of Eq. 11)
    const R r1 = p0 - p1 - R(2) * p2;  // common part of the axis directions
    const R r5 = p0 + R(2) * p1 + p2;  // common part of the diagonals
    const R x34 = p3 - R(2) * p4, y56 = p5 - R(2) * p6;
    const R x34d = p3 + p4, y56d = p5 + p6;
    d[0] = p0 - R(4) * p1 + R(4) * p2;
    d[1] = r1 + x34 + p7;
    d[2] = r1 + y56 - p7;
    d[3] = r1 - x34 + p7;
    d[4] = r1 - y56 - p7;
    d[5] = r5 + x34d + y56d + p8;
    d[6] = r5 - x34d + y56d - p8;
    d[7] = r5 - x34d - y56d + p8;
    d[8] = r5 + x34d - y56d - p8;

    // thermal: n = N h (Eq. 27-28), deviation from T0 (1, 0, 0, varpi, 0)
    const R n0 = (h[0] + h[1]) + (h[2] + h[3]) + h[4];
    const R n1 = h[1] - h[3];
    const R n2 = h[2] - h[4];
    const R n3 = R(-4) * h[0] + (h[1] + h[2]) + (h[3] + h[4]);
    const R n4 = (h[1] - h[2]) + (h[3] - h[4]);
    const R T = c.T0 + mc.dT;
    const R ne1 = ux * T * c.inv_sigma;
    const R ne2 = uy * T * c.inv_sigma;
    // n and the conserved part of n_eq are taken relative to T0 + F, the flux
    // part (u T / sigma) uses the absolute T
    const R dTn = mc.dTl;
    const R ne3 = c.varpi * dTn;
    const R q0 = (n0 - c.z[0] * (n0 - dTn) + c.hz[0] * c.psi0) * R(0.2);
    const R q1 = (n1 - c.z[1] * (n1 - ne1)) * R(0.5);
    const R q2 = (n2 - c.z[2] * (n2 - ne2)) * R(0.5);
    const R q3 = (n3 - c.z[3] * (n3 - ne3) + c.hz[3] * c.psi3) * R(0.05);
    const R q4 = (n4 - c.z[4] * n4) * R(0.25);
    h[0] = q0 - R(4) * q3;
    h[1] = q0 + q1 + q3 + q4;
    h[2] = q0 + q2 + q3 - q4;
    h[3] = q0 - q1 + q3 + q4;
    h[4] = q0 - q2 + q3 - q4;
}

}  // namespace lbm
