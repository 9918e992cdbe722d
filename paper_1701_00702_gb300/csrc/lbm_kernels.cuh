// Device code of the fused three-lattice time step (Liu, He & Li, arXiv
// 1701.00702, Sec. III).  One thread owns one node (fused_step) or two
// neighbouring nodes (fused_step_pair); the whole step is one pass over HBM:
// 9 + 2*Q_T populations and the exchange history are read once (pull
// streaming, Eqs. 15, 33, 44) and written once.
//
// Everything after the pull works in moment space:
//   * m+ = M f+, n_g = M g, n_h = M h with the integer matrices of Eq. 13
//     (D2Q9) and Eq. B1 (D2Q5), hand-unrolled;
//   * flow populations are stored as deviations f_i - w_i from the rest
//     equilibrium f^eq(rho_0 = 1, 0) = w_i (Eq. 27), an exact change of
//     variables that keeps storage resolution proportional to u instead of
//     rho; all flow moments below are deviations from r = M w = (1, -2, 1,
//     0, ..., 0) and delta_rho = rho - 1;
//   * the volumetric blend f = f_l f+ + (1 - f_l) f^eq(rho, 0) (Eq. 20) is
//     linear, and M f^eq(rho, 0) = rho r (Eq. 18 at u = 0), so in deviation
//     form m - r = f_l (m+ - r) + (1 - f_l) delta_rho r;
//   * the wall rule of Eq. 52 is linear too: m+(x_b) = m+(x_f) +
//     m^eq(rho_f, u_b = 0) - m^eq(rho_f, u_f), and likewise for the thermal
//     moments with their own equilibria (Eqs. 34/B2, 45/B4);
//   * the collisions are Eq. 14 (flow, with forcing Eq. 19), Eq. 32 (PCM,
//     source Eqs. 35-36 or App. B) and Eq. 43 (metal, Eqs. 46-47 or App. B),
//     followed by f* = M^-1 m*, with M^-1 = M^T diag(1/|row|^2) for D2Q9;
//   * the PCM enthalpy is bookkept exactly: with FP32 storage the rest
//     population g_0 is kept as an unevaluated float-float sum (hi in the
//     g_0 plane, lo in one extra plane), H = g_0 + sum_{i>=1} g_i is formed
//     as a compensated sum of error-free additions (Knuth's TwoSum, Dekker's
//     Fast2Sum), and the post-collision rest population is the remainder
//     g_0* = n_0* - sum_{i>=1} g_i* of the stored moving populations, so that
//     streaming and collision conserve the enthalpy to ~2^-46 instead of
//     accumulating FP32 rounding in the isothermal mushy zone, where nothing
//     damps it;
//   * every other rest population is a remainder as well (the FP32 metal's
//     takes what its movers give up, without passing through their sum), and the
//     PCM's exchange source is the opposite of the change the metal's n_0
//     actually took (scaled by the heat capacities), so the exchange moves no
//     energy that the metal's rounding dropped;
//   * the state is chunked: [chunk][plane][kChunk] with chunks of kChunk nodes
//     along x, so one pointer per pulled neighbour reaches all its planes;
//   * the arithmetic is written once over a lane type (one node, or a pair of
//     nodes in the packed two-lane FP32 instructions of sm_100 and later), with
//     every rounding named, so that all kernels give a node the same bits.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

namespace lbmk {

// Storage modes.  Arithmetic is FP64 for MODE_F64 and FP32 otherwise.
//   MODE_F64  every population in FP64;
//   MODE_F32  every population in FP32, the PCM rest population as a
//             float-float pair (one extra FP32 plane for the low part);
//   MODE_F16, MODE_BF16  flow deviations (scaled by 2^10 for FP16) and the
//             moving thermal populations in 16 bits, the two thermal rest
//             populations and the exchange history in FP32.  A moving thermal
//             population is stored as its deviation from a reference that any
//             reader rebuilds from the FP32 rest population of the node that
//             sent it: at equilibrium with u = 0 every moving population is
//             w'_i c_ref T and the rest population is g_0 = H - omega c_ref T
//             (Eqs. 40, 49, B3, B5), a monotone map of the node's state, so
//             T (hence the reference) follows from g_0 alone.  The 16-bit
//             values then carry only the flux and non-equilibrium parts, and
//             the sender stores the rest population that closes the balance
//             with the movers as readers decode them.
enum : int { MODE_F64 = 0, MODE_F32 = 1, MODE_F16 = 2, MODE_BF16 = 3 };

template <int M> struct ModeTraits;
template <> struct ModeTraits<MODE_F64> { using R = double; using B = double; };
template <> struct ModeTraits<MODE_F32> { using R = float; using B = float; };
template <> struct ModeTraits<MODE_F16> { using R = float; using B = __half; };
template <> struct ModeTraits<MODE_BF16> { using R = float; using B = __nv_bfloat16; };

template <int M> constexpr bool kSplit = (M == MODE_F16 || M == MODE_BF16);
// FP16 stores the flow deviations times 2^10 (|f_i - w_i| < 1 while |u| < 0.3
// keeps them in the normal range); the other modes store them as they are.
template <int M> constexpr int kFlowScale = (M == MODE_F16) ? 1024 : 1;
template <int M> constexpr bool kComp = (M == MODE_F32);

__device__ __forceinline__ float to_f(__half v) { return __half2float(v); }
__device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ double to_f(double v) { return v; }

template <typename B> __device__ __forceinline__ B from_f(float v);
template <> __device__ __forceinline__ __half from_f<__half>(float v) { return __float2half_rn(v); }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <typename B> __device__ __forceinline__ B from_f(double v) { return v; }

// Plane numbering inside one state copy.  Bulk planes hold type B; the wide
// planes (16-bit modes only) hold the PCM (0) and metal (1) rest populations.
template <int M, int QT, bool FLOW>
struct Planes {
    static constexpr int fb = FLOW ? 9 : 0;
    __host__ __device__ static constexpr int pcm(int q) { return kSplit<M> ? fb + q - 1 : fb + q; }   // q >= 1 when split
    __host__ __device__ static constexpr int met(int q) { return kSplit<M> ? fb + (QT - 1) + q - 1 : fb + QT + q; }
    static constexpr int lo = fb + 2 * QT;                                                  // MODE_F32 only
    static constexpr int bulk = kSplit<M> ? fb + 2 * (QT - 1) : fb + 2 * QT + (kComp<M> ? 1 : 0);
    static constexpr int wide = kSplit<M> ? 2 : 0;
};

// State layout: each row is cut into chunks of kChunk nodes along x, and a
// chunk holds every plane of its nodes, [chunk][plane][kChunk]: the bulk
// planes (the mode's storage type), then the wide planes (FP32).  A node's
// element in plane q lies kChunk * q elements after its element in plane 0,
// so one pointer per pulled neighbour reaches all of that neighbour's planes
// through constant offsets.  Chunk y * cpr + x / kChunk holds node (x, y).
constexpr int kChunk = 128;
constexpr int kChunkShift = 7;

template <int M, int QT, bool FLOW>
struct Chunk {
    using B = typename ModeTraits<M>::B;
    using PL = Planes<M, QT, FLOW>;
    static constexpr int wide_off = PL::bulk * kChunk * (int)sizeof(B);        // bytes to wide plane 0
    static constexpr int bytes = wide_off + PL::wide * kChunk * (int)sizeof(float);
};

// ---------------------------------------------------------------------------
// Lanes
// ---------------------------------------------------------------------------
// The node update is written once, over a lane type T: float or double (one
// node per thread), or W, two neighbouring nodes of a row per thread.  A W
// operation is one packed instruction for both nodes (the .f32x2 add, multiply
// and fused multiply-add of sm_100 and later), which halves the issue slots of
// the arithmetic; scalar constants broadcast, negations and lane swaps cost
// nothing in packed operands.  Every operation names its rounding, and a product
// whose sum with something is a rounding of its own is taken with vmul_alone,
// since a packed one would be contracted all the same; so a node's result is the
// same bit for bit in every kernel and lane type.
template <typename R>
struct alignas(2 * sizeof(R)) V2 {
    R x, y;
};
using W = V2<float>;

struct Mask2 {
    bool x, y;
};

template <typename T> struct Lane { using R = T; using Mask = bool; static constexpr int n = 1; };
template <> struct Lane<W> { using R = float; using Mask = Mask2; static constexpr int n = 2; };

template <typename T> __device__ __forceinline__ T bc(typename Lane<T>::R v) {   // broadcast
    if constexpr (Lane<T>::n == 2) return {v, v};
    else return v;
}

__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double vadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double vsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double vmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float2 f2(W a) { return make_float2(a.x, a.y); }
__device__ __forceinline__ W vadd(W a, W b) {
    const float2 r = __fadd2_rn(f2(a), f2(b));
    return {r.x, r.y};
}
__device__ __forceinline__ W vsub(W a, W b) { return vadd(a, W{-b.x, -b.y}); }
__device__ __forceinline__ W vfma(W a, W b, W c) {
    const float2 r = __ffma2_rn(f2(a), f2(b), f2(c));
    return {r.x, r.y};
}
__device__ __forceinline__ W vmul(W a, W b) {
    const float2 r = __fmul2_rn(f2(a), f2(b));
    return {r.x, r.y};
}
// A product that is then added or subtracted (not an fma's addend, and not one by
// a power of two, which is exact): ptxas 13.0 may fuse a packed multiply with the
// addition of its product although both name their rounding (-fmad=false does not
// stop it), and the pair's sum would be rounded once where a single node's is
// rounded twice; in an error-free sum the error taken would be another number's.
// One scalar multiply per lane is left alone.
__device__ __forceinline__ float vmul_alone(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double vmul_alone(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ W vmul_alone(W a, W b) { return {__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y)}; }
__device__ __forceinline__ float vneg(float a) { return -a; }
__device__ __forceinline__ double vneg(double a) { return -a; }
__device__ __forceinline__ W vneg(W a) { return {-a.x, -a.y}; }

// with a constant factor or term
template <typename T> __device__ __forceinline__ T vmulc(typename Lane<T>::R c, T a) { return vmul(bc<T>(c), a); }
template <typename T> __device__ __forceinline__ T vfmac(typename Lane<T>::R c, T a, T b) { return vfma(bc<T>(c), a, b); }
template <typename T> __device__ __forceinline__ T vaddc(T a, typename Lane<T>::R c) { return vadd(a, bc<T>(c)); }

template <typename R> __device__ __forceinline__ R vsel(bool m, R a, R b) { return m ? a : b; }
__device__ __forceinline__ W vsel(Mask2 m, W a, W b) { return {m.x ? a.x : b.x, m.y ? a.y : b.y}; }

// sat(a c), min(a, c), max(a, 0)
__device__ __forceinline__ float vsatmul(float a, float c) { return __saturatef(__fmul_rn(a, c)); }
__device__ __forceinline__ W vsatmul(W a, float c) { return {vsatmul(a.x, c), vsatmul(a.y, c)}; }
__device__ __forceinline__ float vminc(float a, float c) { return fminf(a, c); }
__device__ __forceinline__ W vminc(W a, float c) { return {fminf(a.x, c), fminf(a.y, c)}; }
__device__ __forceinline__ float vmax0(float a) { return fmaxf(a, 0.0f); }
__device__ __forceinline__ W vmax0(W a) { return {fmaxf(a.x, 0.0f), fmaxf(a.y, 0.0f)}; }

// 1/a (within 1 ulp) and sqrt(a), a >= 0 (within 2^-23), in FP32: one instruction
// each; subnormal speeds, below 1e-19 lattice units, flush to zero.  vsqrt_pos,
// a > 0, is a times 1/sqrt(a) (within 2^-22.4).
__device__ __forceinline__ float vrcp(float a) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ float vsqrt(float a) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ float vsqrt_pos(float a) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return __fmul_rn(a, r);
}
__device__ __forceinline__ W vrcp(W a) { return {vrcp(a.x), vrcp(a.y)}; }
__device__ __forceinline__ W vsqrt(W a) { return {vsqrt(a.x), vsqrt(a.y)}; }
__device__ __forceinline__ W vsqrt_pos(W a) { return {vsqrt_pos(a.x), vsqrt_pos(a.y)}; }
// In FP64, where one warp instruction occupies its scheduler's FP64 unit for 64
// cycles (GB300: two FP64 lanes per SM and clock), 3 and 5 FP64 operations from
// the hardware's seed y (relative error below 2^-20).  1/a by one third-order step
// (Householder, The Numerical Treatment of a Single Nonlinear Equation, 1970):
// with e = 1 - a y, 1/a = y (1 + e + e^2 + ...), the neglected e^3 below 2^-60.
// sqrt(a) by two steps of Newton's method for s^2 = a from s = a y, with y / 2 for
// the 1 / (2 s) of both: the first leaves 3/2 2^-40, the second takes a - s^2 in one
// rounding and leaves less than 2^-59.  Both are so within 0.5 + 2^-6 ulp of the
// exact value (a third-order step for the root, as many operations, keeps half
// the rounding of a y: 0.75 ulp).
// sqrt takes a >= 0, gives 0 below 2^-900 (speeds below 1e-135 lattice units) and
// leaves infinity and NaN what they are; 1/a is for normal numbers below 2^1022
// (zero and infinity give NaN, which the state's check reports).
__device__ __forceinline__ double vrcp(double a) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
    const double e = vfma(-a, y, 1.0);
    return vfma(y, vfma(e, e, e), y);
}
__device__ __forceinline__ double vsqrt(double a) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
    const double h = __hiloint2double(__double2hiint(y) - (1 << 20), __double2loint(y));   // y / 2
    const double s0 = vmul(a, y);
    const double s = vfma(s0, vfma(-s0, h, 0.5), s0);
    const double r = vfma(vfma(-s, s, a), h, s);
    // by the unsigned high word, as which a NaN of either sign is large; infinity's seed is zero
    const unsigned hi = __double2hiint(a);
    return hi < (1023u - 900u) << 20 ? 0.0 : hi == 0x7ff00000u ? a : r;
}
__device__ __forceinline__ double vsqrt_pos(double a) { return vsqrt(a); }

// Per-run constants, passed by value (__grid_constant__).
template <typename R>
struct StepParams {
    const char* src;     // current state copy, [chunk][plane][kChunk]
    char* dst;           // next state copy
    R* dT;               // [ny][pitch] exchange history T_m - T_f of the previous step
    R* dT_out;           // two-step kernel: the history after its second step (another array)
    unsigned int* status;
    int nx, ny, pitch;   // pitch = cpr * kChunk
    int cpr;             // chunks per row
    int per_x, per_y;
    int solid_scheme;    // 0: volumetric blend; 1: bounce-back where f_l <= 0.5 (Sec. V B)
    int prefetch_rows;   // > 0: each block asks L2 for its chunk this many rows ahead
    int wall_kind[4];
    R wall_T[4], wall_T_lo[4], wall_H[4], wall_H_lo[4];
    R fscale, finv;      // flow deviations are stored times fscale (a power of two)
    // 16-bit modes: references of the moving thermal populations
    R w_move[9];         // w'_i: the equilibrium weight of mover i (D2Q9 w_i, D2Q5 varpi/4)
    R wk_move[9];        // w'_i kappa_m: metal mover reference per unit of h_0
    R g0_fs, g0_fl;      // PCM rest population at solidus / liquidus equilibrium
    R cr_solid, cr_liquid;   // c_f,ref dT/dg_0 on the solid and liquid branches
    R cr_fs, cr_dsl;     // c_f,ref T_fs, c_f,ref (T_fl - T_fs)
    R inv_dg0;           // 1 / (g0_fl - g0_fs)
    R kappa_m;           // c_m,ref / (c_pm - omega c_m,ref): mover reference per unit of h_0 / w'_i
    R om_cf;             // omega c_f,ref (omega = sum of the w'_i): g_0 = H - om_cf T(H) at equilibrium
    R rest_m;            // 1 - omega c_m,ref / c_pm: h_0 = rest_m c_pm T_m at equilibrium
    // flow (Eqs. 3, 7, 16, 25)
    R inv_phi, fgb, T0, l0, l0sq, l1;   // fgb = phi gbeta
    R nlin, nforch;      // -phi nu_f / K and -phi F_phi / sqrt(K): the negated drag is nlin + nforch |u|
    R k_uu, k_uf;        // 3 s_e / phi and 6 (1 - s_e / 2) / phi
    R c_v, k_v, k_h, k_2h;   // 1 - s_v, s_v / phi, (1 - s_v / 2) / phi and twice that
    // thermal (Eqs. 38-39, 34, 45, App. B)
    // (c_pl = c_pm = 1 in the lattice units of Eq. 54, so they appear nowhere below)
    R H_fs, H_fl, inv_dH, T_fs, T_off, dT_sl, inv_c_ps;   // T_off = T_fl - H_fl, dT_sl = T_fl - T_fs
    R c_fref, c_mref, varpi;
    R vcf, vcm;          // varpi c_f,ref and varpi c_m,ref (D2Q5 equilibria, Eqs. B2, B4)
    R nz[9], ne[9];      // -zeta_k, -eta_k (D2Q9)
    // D2Q5 relaxation, with the factors 1/2 (j) and 1/4 (n_3, n_4) of M^-1 folded in
    R z_j, z_ju, z_3, z_3T, z_4;   // (1 - z_a)/2, z_a/(2 phi), (1 - z_e)/4, z_e varpi c_f,ref / 4, (1 - z_eps)/4
    R e_j, e_3, e_3T, e_4;         // the metal's
    R quart_varpi;       // varpi / 4
    R x_now, x_prev;     // -1.5 a_m, 0.5 a_m with a_m = h_v/((1 - phi) rho_m): Eq. 47 and Remark III
    R x_pm;              // -a_f/a_m = -(1 - phi) rho_m/(phi rho_l): PCM source per unit of metal source
    // Eq. 9 variant: PCM rates from the node's liquid fraction
    int phase_k;         // 1: k_s != k_l, rates per node
    R ks_c, kd_c;        // k_s and k_l - k_s over (rho_l c_fref c_sT^2)
    R zr_a[9], zr_b[9];  // PCM rate k = zr_a[k] + zr_b[k] zeta_alpha
};

enum : unsigned int { STATUS_UNSTABLE = 1u };

// ---------------------------------------------------------------------------
// Error-free sums
// ---------------------------------------------------------------------------
// The rounding error of s = fl(a + b) (Knuth's TwoSum, the sum already taken).
template <typename T>
__device__ __forceinline__ T sum_err(T a, T b, T s) {
    const T bb = vsub(s, a);
    return vadd(vsub(a, vsub(s, bb)), vsub(b, bb));
}

template <typename T>
struct FF {
    T hi, lo;
};

template <typename T>
__device__ __forceinline__ FF<T> fast_two_sum(T a, T b) {   // Dekker, |a| >= |b|
    const T s = vadd(a, b);
    return {s, vsub(b, vsub(s, a))};
}

// v[1] + ... + v[Q-1] by pairs, opposite directions first (the sums that the
// moments need too).
template <int Q, typename T>
__device__ __forceinline__ T mover_sum(const T* v) {
    const T s = vadd(vadd(v[1], v[3]), vadd(v[2], v[4]));
    if constexpr (Q == 5) return s;
    else return vadd(s, vadd(vadd(v[5], v[7]), vadd(v[6], v[8])));
}

// The same, and the sum of the rounding errors made on the way.
template <int Q, typename T>
__device__ __forceinline__ FF<T> mover_sum_ff(const T* v) {
    const T a = vadd(v[1], v[3]), b = vadd(v[2], v[4]), s = vadd(a, b);
    T e = vadd(vadd(sum_err(v[1], v[3], a), sum_err(v[2], v[4], b)), sum_err(a, b, s));
    if constexpr (Q == 5) {
        return {s, e};
    } else {
        const T c = vadd(v[5], v[7]), d = vadd(v[6], v[8]), r = vadd(c, d), t = vadd(s, r);
        e = vadd(e, vadd(vadd(sum_err(v[5], v[7], c), sum_err(v[6], v[8], d)), sum_err(c, d, r)));
        return {t, vadd(e, sum_err(s, r, t))};
    }
}

// ---------------------------------------------------------------------------
// Transforms
// ---------------------------------------------------------------------------

// Eq. 13: m = M f (rho, e, eps, j_x, q_x, j_y, q_y, p_xx, p_xy).
template <typename T>
__device__ __forceinline__ void m_from_f9(const T* f, T* m) {
    const T a = vadd(f[1], f[3]), b = vadd(f[2], f[4]), c = vadd(f[5], f[7]), d = vadd(f[6], f[8]);
    const T dx = vsub(f[1], f[3]), dy = vsub(f[2], f[4]), ec = vsub(f[5], f[7]), ed = vsub(f[6], f[8]);
    const T s14 = vadd(a, b), s58 = vadd(c, d);
    const T ax = vsub(ec, ed), ay = vadd(ec, ed);
    m[0] = vadd(f[0], vadd(s14, s58));
    m[1] = vfmac<T>(-4, f[0], vfmac<T>(2, s58, vneg(s14)));
    m[2] = vfmac<T>(-2, s14, vfmac<T>(4, f[0], s58));
    m[3] = vadd(dx, ax);
    m[4] = vfmac<T>(-2, dx, ax);
    m[5] = vadd(dy, ay);
    m[6] = vfmac<T>(-2, dy, ay);
    m[7] = vsub(a, b);
    m[8] = vsub(c, d);
}

// f = M^-1 m, every f scaled by SC (a power of two: the 16-bit flow storage
// scale, folded into the row norms).
template <typename T, int SC = 1>
__device__ __forceinline__ void f_from_m9(const T* m, T* f) {
    using R = typename Lane<T>::R;
    constexpr double s = SC;
    const T A = vmulc<T>(R(s / 9.0), m[0]);
    f[0] = vfmac<T>(R(s / 9.0), m[2], vfmac<T>(R(-s / 9.0), m[1], A));
    const T b1 = vfmac<T>(R(-s / 18.0), m[2], vfmac<T>(R(-s / 36.0), m[1], A));
    const T b5 = vfmac<T>(R(s / 36.0), m[2], vfmac<T>(R(s / 18.0), m[1], A));
    const T DX = vmulc<T>(R(s / 6.0), m[3]), DY = vmulc<T>(R(s / 6.0), m[5]);
    const T tx = vfmac<T>(R(-s / 6.0), m[4], DX), ty = vfmac<T>(R(-s / 6.0), m[6], DY);
    const T X = vfmac<T>(R(s / 12.0), m[4], DX), Y = vfmac<T>(R(s / 12.0), m[6], DY);
    const T bp = vfmac<T>(R(s * 0.25), m[7], b1), bm = vfmac<T>(R(-s * 0.25), m[7], b1);
    f[1] = vadd(bp, tx);
    f[3] = vsub(bp, tx);
    f[2] = vadd(bm, ty);
    f[4] = vsub(bm, ty);
    const T gp = vfmac<T>(R(s * 0.25), m[8], b5), gm = vfmac<T>(R(-s * 0.25), m[8], b5);
    const T hp = vadd(X, Y), hm = vsub(Y, X);
    f[5] = vadd(gp, hp);
    f[7] = vsub(gp, hp);
    f[6] = vadd(gm, hm);
    f[8] = vsub(gm, hm);
}

// Eq. B1: n_0 = sum g, n_1 = g_1 - g_3, n_2 = g_2 - g_4,
// n_3 = g_1 + g_2 + g_3 + g_4, n_4 = g_1 - g_2 + g_3 - g_4.
template <typename T, int Q>
__device__ __forceinline__ void thermal_moments(const T* g, T* n) {
    if constexpr (Q == 5) {
        const T a = vadd(g[1], g[3]), b = vadd(g[2], g[4]);
        n[1] = vsub(g[1], g[3]);
        n[2] = vsub(g[2], g[4]);
        n[3] = vadd(a, b);
        n[4] = vsub(a, b);
        n[0] = vadd(g[0], n[3]);
    } else {
        m_from_f9(g, n);
    }
}

// ---------------------------------------------------------------------------
// Equations of state
// ---------------------------------------------------------------------------

// Eqs. 38-39 without branches: f_l = clamp((H - H_s)/(H_l - H_s), 0, 1) and
// T = min(H/c_ps, T_s) + f_l (T_l - T_s) + max(H - H_l, 0)/c_pl, which is
// H/c_ps below the solidus, T_s + f_l (T_l - T_s) in the mushy zone and
// T_l + (H - H_l)/c_pl above the liquidus (c_pl = 1).
template <typename T>
__device__ __forceinline__ void enthalpy_state(const StepParams<float>& P, T H, T& Tf, T& fl) {
    fl = vsatmul(vaddc(H, -P.H_fs), P.inv_dH);
    Tf = vadd(vfmac<T>(P.dT_sl, fl, vminc(vmulc<T>(P.inv_c_ps, H), P.T_fs)), vmax0(vaddc(H, -P.H_fl)));
}

// In FP64 the branch is chosen by comparing bit patterns (order_key keeps the
// order of the numbers it maps), which takes no FP64 operation, and T is one
// multiply-add of the branch's own slope and offset.
__device__ __forceinline__ long long order_key(double v) {
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

__device__ __forceinline__ void enthalpy_state(const StepParams<double>& P, double H, double& Tf, double& fl) {
    const long long k = order_key(H);
    const bool solid = k <= order_key(P.H_fs), liquid = !solid && k >= order_key(P.H_fl);
    const double f = vmul(vsub(H, P.H_fs), P.inv_dH);
    fl = solid ? 0.0 : liquid || __double_as_longlong(f) > __double_as_longlong(1.0) ? 1.0 : f;
    Tf = vfma(solid || liquid ? H : fl, solid ? P.inv_c_ps : liquid ? 1.0 : P.dT_sl,
              solid ? 0.0 : liquid ? P.T_off : P.T_fs);
}

// c_f,ref T at equilibrium as a function of the PCM rest population g_0: the
// inverse of g_0 = H - omega c_f,ref T(H) with T(H) from Eq. 38 (16-bit modes).
// The three branches as in enthalpy_state: solid slope up to g0_fs, a linear
// rise of c_f,ref (T_fl - T_fs) across the mushy zone, liquid slope above g0_fl.
template <typename T>
__device__ __forceinline__ T pcm_ref(const StepParams<float>& P, T g0) {
    const T a = vfmac<T>(P.cr_dsl, vsatmul(vaddc(g0, -P.g0_fs), P.inv_dg0), vminc(vmulc<T>(P.cr_solid, g0), P.cr_fs));
    return vfmac<T>(P.cr_liquid, vmax0(vaddc(g0, -P.g0_fl)), a);
}

// ---------------------------------------------------------------------------
// Node state
// ---------------------------------------------------------------------------

template <int M, int QT, bool FLOW, typename T>
struct NodeState {
    T mp[FLOW ? 9 : 1];  // moments of f+ minus r, times kFlowScale<M> (after the wall rule)
    T n[QT], k[QT];      // PCM and metal moments (after the wall rule); n[0] = H (high part), k[0] = c_pm T_m = T_m
    T Hlo, Elo;          // low parts of H and c_pm T_m (error-free bookkeeping; 0 where unused)
    T h0, hs;            // metal rest population and the sum of its movers: k[0] = h0 + hs before rounding (FP32)
    T Tf, fl, rho, drho, ux, uy, um, G;   // um = |u|, G = phi G_y (Eq. 7)
};

// the lane's type in a mode's one-node kernels
template <int M> using Node1 = typename ModeTraits<M>::R;

// Reads of a state copy.  EV: marked evict-first (ld.global.cs), for grids whose
// two copies and history come near L2's 129 MB or a little above: a step's
// source is dead once its neighbours have read it, until the next step
// overwrites it whole, and gives way to the copy being written, which the next
// step reads (GB300, us per step without / with: FP32 768^2, 97 MB, 11.7 / 9.3,
// 1024^2 one step per launch, 172 MB, 26.3 / 21.5; FP16 1200^2, 127 MB, 25.3 /
// 18.6; at 80 MB 1 % slower, at 276 MB 7 %).
template <bool EV, typename V>
__device__ __forceinline__ V read_state(const V* p) {
    if constexpr (EV) return __ldcs(p);
    else return __ldg(p);
}

template <int M, bool EV = false>
__device__ __forceinline__ typename ModeTraits<M>::R ldb(const typename ModeTraits<M>::B* p) {
    return to_f(read_state<EV>(p));
}

template <int M, typename R>
__device__ __forceinline__ void stb(typename ModeTraits<M>::B* p, R v) {
    using B = typename ModeTraits<M>::B;
    *p = from_f<B>(v);
}

// Two adjacent elements of a plane, as stored (16-bit: one 32-bit access; FP32: 64-bit).
__device__ __forceinline__ W unpack2(__half2 v) {
    const float2 f = __half22float2(v);
    return {f.x, f.y};
}
__device__ __forceinline__ W unpack2(__nv_bfloat162 v) {
    const float2 f = __bfloat1622float2(v);
    return {f.x, f.y};
}
__device__ __forceinline__ W unpack2(float2 v) { return {v.x, v.y}; }
template <typename B> struct Two;
template <> struct Two<__half> { using type = __half2; };
template <> struct Two<__nv_bfloat16> { using type = __nv_bfloat162; };
template <> struct Two<float> { using type = float2; };

// Stores v at p (the lanes adjacent); returns the values as a reader decodes them.
template <int M, typename T>
__device__ __forceinline__ T put(typename ModeTraits<M>::B* p, T v) {
    if constexpr (Lane<T>::n == 1) {
        const typename ModeTraits<M>::B b = from_f<typename ModeTraits<M>::B>(v);
        *p = b;
        return to_f(b);
    } else if constexpr (M == MODE_F16) {
        const __half2 h = __floats2half2_rn(v.x, v.y);
        *reinterpret_cast<__half2*>(p) = h;
        return unpack2(h);
    } else if constexpr (M == MODE_BF16) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
        *reinterpret_cast<__nv_bfloat162*>(p) = h;
        return unpack2(h);
    } else {
        *reinterpret_cast<float2*>(p) = f2(v);
        return v;
    }
}
template <typename R> __device__ __forceinline__ void put_real(R* p, R v) { *p = v; }
__device__ __forceinline__ void put_real(float* p, W v) { *reinterpret_cast<float2*>(p) = f2(v); }
template <typename T, typename R> __device__ __forceinline__ T get_real(const R* p) {
    if constexpr (Lane<T>::n == 2) return unpack2(*reinterpret_cast<const float2*>(p));
    else return *p;
}

// Byte offset, within a state copy, of the chunk holding node (x, y).
template <int M, int QT, bool FLOW, typename R>
__device__ __forceinline__ long long chunk_at(const StepParams<R>& P, int x, int y) {
    return (long long)(y * P.cpr + (x >> kChunkShift)) * Chunk<M, QT, FLOW>::bytes;
}

// Node (x, y)'s element in bulk plane 0 and in wide plane 0 of a copy; plane q
// follows at q * kChunk elements.
template <int M, int QT, bool FLOW, typename R, typename C>
__device__ __forceinline__ auto bulk_at(C* base, const StepParams<R>& P, int x, int y) {
    using B = typename ModeTraits<M>::B;
    using T = std::conditional_t<std::is_const_v<C>, const B, B>;
    return reinterpret_cast<T*>(base + chunk_at<M, QT, FLOW>(P, x, y)) + (x & (kChunk - 1));
}

template <int M, int QT, bool FLOW, typename R, typename C>
__device__ __forceinline__ auto wide_at(C* base, const StepParams<R>& P, int x, int y) {
    using T = std::conditional_t<std::is_const_v<C>, const float, float>;
    return reinterpret_cast<T*>(base + chunk_at<M, QT, FLOW>(P, x, y) + Chunk<M, QT, FLOW>::wide_off) +
           (x & (kChunk - 1));
}

// Byte offset of node x's element in bulk plane 0 (WIDE: wide plane 0) from
// the start of its row of chunks; a row of chunks is cpr * Chunk::bytes long
// (below 2^31 bytes for every admitted grid).
template <int M, int QT, bool FLOW, bool WIDE = false>
__device__ __forceinline__ int col_off(int x) {
    using CH = Chunk<M, QT, FLOW>;
    constexpr int es = WIDE ? (int)sizeof(float) : (int)sizeof(typename ModeTraits<M>::B);
    return (x >> kChunkShift) * CH::bytes + (WIDE ? CH::wide_off : 0) + (x & (kChunk - 1)) * es;
}

// Pull streaming around node (xs, ys): the population along e_i comes from
// xs - e_i.  The index wrap is also correct for interior nodes of a walled
// direction, which never reach the edge.  PullAt holds the addressing (one
// 64-bit row pointer per source row, one 32-bit offset per source column).
// Source column and row (x - e_x, y - e_y) of direction q, D2Q9 order of Eq. 11,
// as 0 (x - 1 or y - 1), 1 (x or y), 2 (x + 1 or y + 1): columns 1 0 1 2 1 0 2 2 0,
// rows 1 1 0 1 2 0 0 2 2, two bits per direction.
__host__ __device__ constexpr int src_col(int q) { return (0xa191 >> (2 * q)) & 3; }
__host__ __device__ constexpr int src_row(int q) { return (0x28245 >> (2 * q)) & 3; }

template <int M, int QT, bool FLOW, bool EV = false>
struct PullAt {
    const char* row[3];
    int dc[3];   // bulk plane 0 of source columns x - 1, x, x + 1, from this node's
    int dw[3];   // wide plane 0 of the same columns (16-bit modes)
    int xm, xs, xp, c0;
    __device__ __forceinline__ PullAt(const StepParams<typename ModeTraits<M>::R>& P, int x, int ys) : xs(x) {
        xm = xs == 0 ? P.nx - 1 : xs - 1;
        xp = xs == P.nx - 1 ? 0 : xs + 1;
        const int ym = ys == 0 ? P.ny - 1 : ys - 1;
        const int yp = ys == P.ny - 1 ? 0 : ys + 1;
        const int rb = P.cpr * Chunk<M, QT, FLOW>::bytes;
        c0 = col_off<M, QT, FLOW>(xs);
        const char* own = P.src + ((long long)ys * rb + c0);
        row[0] = own + (long long)(ym - ys) * rb;
        row[1] = own;
        row[2] = own + (long long)(yp - ys) * rb;
        dc[0] = col_off<M, QT, FLOW>(xm) - c0;
        dc[1] = 0;
        dc[2] = col_off<M, QT, FLOW>(xp) - c0;
        if constexpr (kSplit<M>) {
            dw[0] = col_off<M, QT, FLOW, true>(xm) - c0;
            dw[1] = col_off<M, QT, FLOW, true>(xs) - c0;
            dw[2] = col_off<M, QT, FLOW, true>(xp) - c0;
        }
    }
    // the source node of direction q: its element in bulk plane 0
    __device__ __forceinline__ const typename ModeTraits<M>::B* src(int q) const {
        return reinterpret_cast<const typename ModeTraits<M>::B*>(row[src_row(q)] + dc[src_col(q)]);
    }
    // bulk plane `plane` and wide plane w (16-bit modes) of the source node of direction q
    __device__ __forceinline__ typename ModeTraits<M>::R bulk(int q, int plane) const {
        return ldb<M, EV>(src(q) + plane * kChunk);
    }
    __device__ __forceinline__ float wide(int q, int w) const {
        return read_state<EV>(reinterpret_cast<const float*>(row[src_row(q)] + dw[src_col(q)]) + w * kChunk);
    }
};

// The same around the node pair (x0, x0 + 1), x0 even (both nodes in one
// chunk): own reads the pair's two adjacent elements, west the elements of
// x0 - 1 and x0, east those of x0 + 1 and x0 + 2.
template <int M, int QT, bool EV = false>
struct PairAt {
    using B = typename ModeTraits<M>::B;
    using CH = Chunk<M, QT, true>;
    static constexpr int es = (int)sizeof(B);
    const char* row[3];
    int cm, cp, w0, wm, wp;   // west, east and wide elements, from the pair's bulk plane 0
    __device__ __forceinline__ PairAt(const StepParams<float>& P, int x0, int ys) {
        const int xm = x0 == 0 ? P.nx - 1 : x0 - 1;       // west of x0
        const int xp = x0 + 2 >= P.nx ? 0 : x0 + 2;       // east of x0 + 1
        const int ym = ys == 0 ? P.ny - 1 : ys - 1;
        const int yp = ys == P.ny - 1 ? 0 : ys + 1;
        const int rb = P.cpr * CH::bytes;
        const int c0 = col_off<M, QT, true>(x0);
        const char* own = P.src + ((long long)ys * rb + c0);
        row[0] = own + (long long)(ym - ys) * rb;
        row[1] = own;
        row[2] = own + (long long)(yp - ys) * rb;
        cm = col_off<M, QT, true>(xm) - c0;
        cp = col_off<M, QT, true>(xp) - c0;
        if constexpr (kSplit<M>) {
            w0 = col_off<M, QT, true, true>(x0) - c0;
            wm = col_off<M, QT, true, true>(xm) - c0;
            wp = col_off<M, QT, true, true>(xp) - c0;
        }
    }
    __device__ __forceinline__ static float one(const char* p) { return ldb<M, EV>(reinterpret_cast<const B*>(p)); }
    __device__ __forceinline__ static float onew(const char* p) {
        return read_state<EV>(reinterpret_cast<const float*>(p));
    }
    __device__ __forceinline__ W bulk(int q, int plane) const {
        const char* r = row[src_row(q)] + plane * kChunk * es;
        if (src_col(q) == 0) return {one(r + cm), one(r)};
        if (src_col(q) == 2) return {one(r + es), one(r + cp)};
        return unpack2(read_state<EV>(reinterpret_cast<const typename Two<B>::type*>(r)));
    }
    __device__ __forceinline__ W wide(int q, int w) const {
        const char* r = row[src_row(q)] + w * kChunk * 4;
        if (src_col(q) == 0) return {onew(r + wm), onew(r + w0)};
        if (src_col(q) == 2) return {onew(r + w0 + 4), onew(r + wp)};
        return unpack2(read_state<EV>(reinterpret_cast<const float2*>(r + w0)));
    }
};

// Flow moments of the pulled populations (Eqs. 13, 15), deviation form, as
// stored (times kFlowScale<M>).  A is the accessor of the pulled
// neighbourhood: PullAt or PairAt (the state copy in global memory) or
// PullTile (a staged copy in shared memory).
template <int M, int QT, bool FLOW, typename T, typename A>
__device__ __forceinline__ void pull_flow(const A& a, NodeState<M, QT, FLOW, T>& n) {
    if constexpr (FLOW) {
        T f[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) f[q] = a.bulk(q, q);
        m_from_f9(f, n.mp);
    }
}

// PCM and metal moments of the pulled populations (Eqs. 33, 44, B1).
template <int M, int QT, bool FLOW, typename T, typename A>
__device__ __forceinline__ void pull_thermal(const StepParams<typename ModeTraits<M>::R>& P, const A& a,
                                             NodeState<M, QT, FLOW, T>& n) {
    using PL = Planes<M, QT, FLOW>;
    T g[QT], h[QT];
    if constexpr (kSplit<M>) {
        g[0] = a.wide(0, 0);
        h[0] = a.wide(0, 1);
#pragma unroll
        for (int q = 1; q < QT; ++q) {   // deviation + reference of the sending node
            const int w = QT == 5 ? 1 : q;   // D2Q5: one weight varpi/4 for all movers (App. B)
            g[q] = vfmac<T>(P.w_move[w], pcm_ref(P, a.wide(q, 0)), a.bulk(q, PL::pcm(q)));
            h[q] = vfmac<T>(P.wk_move[w], a.wide(q, 1), a.bulk(q, PL::met(q)));
        }
    } else {
#pragma unroll
        for (int q = 0; q < QT; ++q) {
            g[q] = a.bulk(q, PL::pcm(q));
            h[q] = a.bulk(q, PL::met(q));
        }
    }
    thermal_moments<T, QT>(g, n.n);
    thermal_moments<T, QT>(h, n.k);
    n.Hlo = bc<T>(0);
    n.Elo = bc<T>(0);
    n.h0 = h[0];
    n.hs = QT == 5 ? n.k[3] : mover_sum<QT>(h);
    if constexpr (kComp<M>) {
        // H = (g_0 hi + g_0 lo) + sum of movers, without rounding loss
        const FF<T> s = mover_sum_ff<QT>(g);
        const T t = vadd(g[0], s.hi);
        const FF<T> H = fast_two_sum(t, vadd(vadd(s.lo, sum_err(g[0], s.hi, t)), a.bulk(0, PL::lo)));
        n.n[0] = H.hi;
        n.Hlo = H.lo;
    }
}

// Macroscopic state from the moments (Eqs. 21, 23-25, 37-39, 48, 7): the
// thermal side (H -> T_f, f_l; T_m = k[0]) and the flow side, which needs T_f
// and f_l (buoyancy, Eq. 7; the blended momentum, Eq. 24).
template <int M, int QT, bool FLOW, typename T>
__device__ __forceinline__ void buoyancy(const StepParams<typename ModeTraits<M>::R>& P, NodeState<M, QT, FLOW, T>& n) {
    if constexpr (FLOW) n.G = vmulc<T>(P.fgb, vmul(vaddc(n.Tf, -P.T0), n.fl));
}

template <int M, int QT, bool FLOW, typename T>
__device__ __forceinline__ void macro(const StepParams<typename ModeTraits<M>::R>& P, NodeState<M, QT, FLOW, T>& n) {
    using R = typename Lane<T>::R;
    enthalpy_state(P, n.n[0], n.Tf, n.fl);
    if constexpr (FLOW) {
        constexpr R is = R(1.0 / kFlowScale<M>);
        buoyancy<M, QT, FLOW, T>(P, n);
        n.drho = kFlowScale<M> == 1 ? n.mp[0] : vmulc<T>(is, n.mp[0]);
        n.rho = vaddc(n.drho, R(1));
        // Eq. 24 with sum_i e_i f_i = f_l sum_i e_i f+_i (the equilibrium at rest carries no
        // momentum); without the blend (bounce-back variant) sum_i e_i f_i = sum_i e_i f+_i
        T a = n.fl;
        if constexpr (Lane<T>::n == 1)
            if (P.solid_scheme) a = R(1);
        a = vmul(a, vrcp(n.rho));
        if constexpr (kFlowScale<M> != 1) a = vmulc<T>(is, a);
        const T vx = vmul(a, n.mp[3]);
        const T vy = vfmac<T>(R(0.5), n.G, vmul(a, n.mp[5]));
        const T vm = vsqrt(vfma(vy, vy, vmul(vx, vx)));
        const T den = vrcp(vaddc(vsqrt_pos(vfma(bc<T>(P.l1), vm, bc<T>(P.l0sq))), P.l0));   // Eq. 23
        n.ux = vmul(vx, den);
        n.uy = vmul(vy, den);
        n.um = vmul(vm, den);
        if constexpr (Lane<T>::n == 1)
            if (P.solid_scheme && n.fl <= R(0.5)) n.ux = n.uy = n.um = R(0);
    } else {
        n.drho = bc<T>(0);
        n.rho = bc<T>(1);
        n.ux = n.uy = n.um = n.G = bc<T>(0);
    }
}

// Wall nodes: x_f = x_b + inward normal (diagonal at corners) and the side
// whose temperature rule applies (the left/right wall at corners).  A node
// pair on a left or right wall pulls both nodes at its own columns, and the
// wall node then takes its partner's moments (its x_f).
template <typename T> struct WallAt;
template <typename R>
struct WallAt {
    bool any;            // some lane is a wall node
    bool wall;
    int xs, ys, side;    // where to pull
    template <typename P_>
    __device__ __forceinline__ WallAt(const P_& P, int x, int y) {
        const bool wx = !P.per_x && (x == 0 || x == P.nx - 1);
        const bool wy = !P.per_y && (y == 0 || y == P.ny - 1);
        any = wall = wx || wy;
        xs = wx ? (x == 0 ? 1 : P.nx - 2) : x;
        ys = wy ? (y == 0 ? 1 : P.ny - 2) : y;
        side = wx ? (x == 0 ? 0 : 1) : (y == 0 ? 2 : 3);
    }
    __device__ __forceinline__ void from_inward(R&) const {}
    __device__ __forceinline__ R of_side(const R* v) const { return v[side]; }
    __device__ __forceinline__ bool dirichlet(const int* kind) const { return kind[side] == 0; }
};
template <>
struct WallAt<W> {
    bool any, xa, xb;    // xa, xb: the pair's first (second) node is on the left (right) wall
    Mask2 wall;
    int xs, ys, sa, sb;
    __device__ __forceinline__ WallAt(const StepParams<float>& P, int x0, int y) {
        const bool wy = !P.per_y && (y == 0 || y == P.ny - 1);
        xa = !P.per_x && x0 == 0;
        xb = !P.per_x && x0 + 1 == P.nx - 1;
        wall = {xa || wy, xb || wy};
        any = wy || xa || xb;
        xs = x0;
        ys = wy ? (y == 0 ? 1 : P.ny - 2) : y;
        const int sy = y == 0 ? 2 : 3;
        sa = xa ? 0 : sy;
        sb = xb ? 1 : sy;
    }
    __device__ __forceinline__ void from_inward(W& v) const { v = {xa ? v.y : v.x, xb ? v.x : v.y}; }
    __device__ __forceinline__ W of_side(const float* v) const { return {v[sa], v[sb]}; }
    __device__ __forceinline__ Mask2 dirichlet(const int* kind) const {
        return {wall.x && kind[sa] == 0, wall.y && kind[sb] == 0};
    }
};

// Eq. 52 in moment space at the wall lanes (n holds the state of x_f):
// m+(x_b) = m+(x_f) + m^eq(rho_f, u_b = 0) - m^eq(rho_f, u_f), written out so
// that the rho r parts cancel exactly, and likewise for the thermal moments
// with the wall's temperature (Dirichlet: T_f = T_m = T_w, H = H(T_w);
// adiabatic: those of x_f) and the velocity u_f in the PCM equilibrium.  The
// other lanes of a pair go through with corrections of zero.
template <int M, int QT, bool FLOW, typename T>
__device__ __forceinline__ void apply_wall(const StepParams<typename ModeTraits<M>::R>& P, const WallAt<T>& w,
                                           NodeState<M, QT, FLOW, T>& n) {
    using R = typename Lane<T>::R;
    const T zero = bc<T>(0);
    const T ux = vsel(w.wall, n.ux, zero), uy = vsel(w.wall, n.uy, zero);
    if constexpr (FLOW) {
        constexpr R sc = R(kFlowScale<M>);
        T jx = vmul_alone(n.rho, ux), jy = vmul_alone(n.rho, uy);
        if constexpr (kFlowScale<M> != 1) {
            jx = vmulc<T>(sc, jx);
            jy = vmulc<T>(sc, jy);
        }
        const T a = vmul(jx, ux);
        const T q = vmul_alone(bc<T>(vmul(R(3), P.inv_phi)), vfma(jy, uy, a));
        n.mp[1] = vsub(n.mp[1], q);
        n.mp[2] = vadd(n.mp[2], q);
        n.mp[3] = vsub(n.mp[3], jx);
        n.mp[4] = vadd(n.mp[4], jx);
        n.mp[5] = vsub(n.mp[5], jy);
        n.mp[6] = vadd(n.mp[6], jy);
        n.mp[7] = vfmac<T>(-P.inv_phi, vfma(vneg(jy), uy, a), n.mp[7]);
        n.mp[8] = vfmac<T>(-P.inv_phi, vmul(jx, uy), n.mp[8]);
    }
    const auto dir = w.dirichlet(P.wall_kind);
    const T Tb = w.of_side(P.wall_T), Hb = w.of_side(P.wall_H);
    const T dT = vsel(dir, vsub(Tb, n.Tf), zero), dM = vsel(dir, vsub(Tb, n.k[0]), zero);
    const T t = FLOW ? vmulc<T>(P.inv_phi, n.Tf) : zero, mt = vneg(t);   // c_pl T / phi
    if constexpr (QT == 5) {
        if constexpr (FLOW) {
            n.n[1] = vfma(mt, ux, n.n[1]);
            n.n[2] = vfma(mt, uy, n.n[2]);
        }
        n.n[3] = vfmac<T>(P.vcf, dT, n.n[3]);
        n.k[3] = vfmac<T>(P.vcm, dM, n.k[3]);
    } else {
        const T dH = vsel(dir, vsub(Hb, n.n[0]), zero);
        const T cT = vmulc<T>(P.c_fref, dT), cM = vmulc<T>(P.c_mref, dM);
        n.n[1] = vadd(n.n[1], vfmac<T>(R(-4), dH, vadd(cT, cT)));
        n.n[2] = vadd(n.n[2], vfmac<T>(R(4), dH, vmulc<T>(R(-3), cT)));
        if constexpr (FLOW) {
            n.n[3] = vfma(mt, ux, n.n[3]);
            n.n[4] = vfma(t, ux, n.n[4]);
            n.n[5] = vfma(mt, uy, n.n[5]);
            n.n[6] = vfma(t, uy, n.n[6]);
        }
        n.k[1] = vadd(n.k[1], vfmac<T>(R(-4), dM, vadd(cM, cM)));
        n.k[2] = vadd(n.k[2], vfmac<T>(R(4), dM, vmulc<T>(R(-3), cM)));
    }
    // n_0 = H_b and c_pm T_m = c_pm T_b exactly (adiabatic: those of x_f, unchanged)
    n.n[0] = vsel(dir, Hb, n.n[0]);
    n.Hlo = vsel(dir, w.of_side(P.wall_H_lo), n.Hlo);
    n.k[0] = vsel(dir, Tb, n.k[0]);
    if constexpr (QT == 5) n.hs = n.k[3];
    n.h0 = vsel(dir, vsub(Tb, n.hs), n.h0);
    if constexpr (kSplit<M>) n.Elo = vsel(dir, w.of_side(P.wall_T_lo), n.Elo);
    enthalpy_state(P, n.n[0], n.Tf, n.fl);
    buoyancy<M, QT, FLOW, T>(P, n);
    n.ux = vsel(w.wall, zero, n.ux);
    n.uy = vsel(w.wall, zero, n.uy);
    n.um = vsel(w.wall, zero, n.um);
}

// State of a node (pair) from its pulled neighbourhood a (pulled at x_f on
// walls, then Eq. 52 in moment space).  LATE: the thermal lattices are pulled
// first.
template <int M, int QT, bool FLOW, typename T, bool LATE = kComp<M>, typename A>
__device__ __forceinline__ void node_state(const StepParams<typename ModeTraits<M>::R>& P, const A& a,
                                           const WallAt<T>& w, NodeState<M, QT, FLOW, T>& n) {
    if constexpr (LATE) {
        pull_thermal<M, QT, FLOW, T>(P, a, n);
        pull_flow<M, QT, FLOW, T>(a, n);
    } else {
        pull_flow<M, QT, FLOW, T>(a, n);
        pull_thermal<M, QT, FLOW, T>(P, a, n);
    }
    if constexpr (Lane<T>::n == 2) {
        if (w.xa || w.xb) {
#pragma unroll
            for (int q = 0; q < 9; ++q) w.from_inward(n.mp[q]);
#pragma unroll
            for (int q = 0; q < QT; ++q) {
                w.from_inward(n.n[q]);
                w.from_inward(n.k[q]);
            }
            w.from_inward(n.Hlo);
            w.from_inward(n.h0);
            w.from_inward(n.hs);
        }
    }
    macro<M, QT, FLOW, T>(P, n);
    if (w.any) apply_wall<M, QT, FLOW, T>(P, w, n);
}

// Full state of node (x, y) in a state copy: interior nodes pull at
// themselves, wall nodes at x_f = x_b + inward normal.
template <int M, int QT, bool FLOW>
__device__ __forceinline__ void node_state_at(const StepParams<typename ModeTraits<M>::R>& P, int x, int y,
                                              NodeState<M, QT, FLOW, Node1<M>>& n) {
    const WallAt<Node1<M>> w(P, x, y);
    node_state<M, QT, FLOW, Node1<M>>(P, PullAt<M, QT, FLOW>(P, w.xs, w.ys), w, n);
}

// ---------------------------------------------------------------------------
// Collisions
// ---------------------------------------------------------------------------

// Flow collision and store of one node (pair) (Eqs. 3, 14, 18-20): f* at db,
// the element in flow plane 0 of the next copy, PS elements from one plane to
// the next.
template <int M, int QT, bool FLOW, int PS, typename T>
__device__ __forceinline__ void flow_collide(const StepParams<typename ModeTraits<M>::R>& P,
                                             const NodeState<M, QT, FLOW, T>& n, typename ModeTraits<M>::B* db) {
    using R = typename Lane<T>::R;
    if constexpr (FLOW) {
        constexpr R is = R(1.0 / kFlowScale<M>);   // takes the storage scale off the pulled moments
        T m[9], f[9];
        T fb = n.fl;
        if constexpr (Lane<T>::n == 1) {
            if (P.solid_scheme && n.fl <= R(0.5)) {
                // bounce-back solid node: f*_i = f+_opp(i); reversing every link flips the
                // sign of the odd moments (j, q) and keeps the even ones (deviation form too)
#pragma unroll
                for (int q = 0; q < 9; ++q) m[q] = vmul(q >= 3 && q <= 6 ? -is : is, n.mp[q]);
                f_from_m9<T, kFlowScale<M>>(m, f);
#pragma unroll
                for (int q = 0; q < 9; ++q) put<M>(db + q * PS, f[q]);
                return;
            }
            if (P.solid_scheme) fb = R(1);   // no blend in the bounce-back variant
        }
        const T drag = vfma(bc<T>(P.nforch), n.um, bc<T>(P.nlin));   // Eq. 3, negated
        const T Fx = vmul(drag, n.ux), Fy = vfma(drag, n.uy, n.G);
        const T jx = vmul(n.rho, n.ux), jy = vmul(n.rho, n.uy);
        const T fx = vmul(n.rho, Fx), fy = vmul(n.rho, Fy);
        const T xx = vmul(jx, n.ux), fxx = vmul(jx, Fx);
        const T up = vfma(jy, n.uy, xx), um = vfma(vneg(jy), n.uy, xx);      // j_x u_x +- j_y u_y
        const T fp = vfma(jy, Fy, fxx), fm = vfma(vneg(jy), Fy, fxx);        // j_x F_x +- j_y F_y
        // Eq. 14 on the blended moments (Eq. 20: f_l m+ + (1 - f_l) delta_rho r in deviation
        // form) with the equilibria of Eq. 18 and the forcing moments of Eq. 19.  The rates of
        // Sec. III C are constants (s_rho = s_j = 1, s_e = s_eps = 1.1, s_q = 1.2); only s_v
        // depends on the run.  m - s (m - m^eq) is taken as (1 - s) m + s m^eq, with 1 - s
        // exact; for e and eps the parts along r collect to (-2, 1) (delta_rho + s' f_l
        // delta_rho), s' = s - 1.  Where s = 1 the result is m^eq + S/2 whatever the blend gave.
        constexpr R s1 = R(1.1) - R(1), s2 = R(1.2) - R(1);
        const T b1 = vmulc<T>(-s1 * is, fb), b2 = vmulc<T>(-s2 * is, fb), bv = vmulc<T>(P.c_v * is, fb);
        const T K = vfma(vmulc<T>(s1, fb), n.drho, n.drho);
        const T Q = vfmac<T>(P.k_uf, fp, vmulc<T>(P.k_uu, up));
        m[0] = n.drho;
        m[1] = vfma(b1, n.mp[1], vfmac<T>(R(-2), K, Q));
        m[2] = vfma(b1, n.mp[2], vsub(K, Q));
        m[3] = vfmac<T>(R(0.5), fx, jx);
        m[5] = vfmac<T>(R(0.5), fy, jy);
        m[4] = vfma(b2, n.mp[4], vfmac<T>(R(-0.4), fx, vmulc<T>(R(-1.2), jx)));
        m[6] = vfma(b2, n.mp[6], vfmac<T>(R(-0.4), fy, vmulc<T>(R(-1.2), jy)));
        m[7] = vfma(bv, n.mp[7], vfmac<T>(P.k_v, um, vmulc<T>(P.k_2h, fm)));
        m[8] = vfma(bv, n.mp[8],
                    vfmac<T>(P.k_v, vmul(jx, n.uy), vmulc<T>(P.k_h, vfma(jx, Fy, vmul(jy, Fx)))));
        f_from_m9<T, kFlowScale<M>>(m, f);
#pragma unroll
        for (int q = 0; q < 9; ++q) put<M>(db + q * PS, f[q]);
    }
}

// PCM and metal collisions and stores of one node (pair) (Eqs. 32, 36, 43, 47
// with the backward difference of Remark III): dTp is the exchange history,
// db/dw the element in bulk and wide plane 0 of the next copy; returns the new
// history T_m - T_f.  Each rest population is the remainder n_0 - sum of the
// moving populations as they are stored, so the stored populations carry the
// enthalpy (internal energy) that the collision produced: the FP32 PCM rest
// population to float-float accuracy, the FP32 metal one to one rounding, the
// 16-bit forms to FP32 rounding as readers decode them, FP64 to FP64 rounding.
template <int M, int QT, bool FLOW, bool PH, int PS, typename T>
__device__ __forceinline__ T thermal_collide(const StepParams<typename ModeTraits<M>::R>& P,
                                             const NodeState<M, QT, FLOW, T>& n, T dTp,
                                             typename ModeTraits<M>::B* db, float* dw) {
    using R = typename Lane<T>::R;
    using PL = Planes<M, QT, FLOW>;
    const T dTn = vsub(n.k[0], n.Tf);
    const T S_met = vfmac<T>(P.x_now, dTn, vmulc<T>(P.x_prev, dTp));
    // metal n_0 after its source (n_0 is conserved by the collision, Eq. 43).  The
    // PCM takes the opposite of what the metal's n_0 actually changed by, scaled
    // by the heat capacities (S_PCM = -(a_f/a_m) S_metal, Eqs. 36, 47), so an
    // exchange that the metal's rounding drops moves no energy into the PCM (FP32:
    // n_0 takes what the stored metal took, below)
    const T hm = vadd(n.k[0], S_met);
    const T took = kComp<M> ? S_met : vsub(hm, n.k[0]);
    const T S_pcm = vmulc<T>(P.x_pm, took);
    const T n0 = vfmac<T>(P.x_pm, took, n.n[0]);   // H + S_PCM (n_0 is conserved up to the source, Eq. 32)
    T g[QT], h[QT];   // post-collision populations; g[0], h[0]: provisional rest populations
    if constexpr (QT == 5) {
        // n* = (1 - z) n + z n^eq + S s, the factors of M^-1 folded into the constants:
        // j = n*_{1,2} / 2, a3 = n*_3 / 4, and with z4 n_4 = n*_4 / 4 the movers are a3 +- z4 n_4 +- j
        T jx, jy, a3, z4 = bc<T>(P.z_4);
        if (PH && P.phase_k) {
            // Eq. 9 at the node's liquid fraction -> zeta_alpha (Eq. A19) -> zeta_e (Eq. 53)
            const T za = vrcp(vaddc(vfma(bc<T>(P.kd_c), n.fl, bc<T>(P.ks_c)), R(0.5)));
            T z[5];
#pragma unroll
            for (int k = 1; k < 5; ++k) z[k] = vfma(bc<T>(P.zr_b[k]), za, bc<T>(P.zr_a[k]));
            const T t = vmulc<T>(P.inv_phi, n.Tf);
            const T d1 = vfma(vneg(t), n.ux, n.n[1]), d2 = vfma(vneg(t), n.uy, n.n[2]);
            jx = vmulc<T>(R(0.5), vfma(vneg(z[1]), d1, n.n[1]));
            jy = vmulc<T>(R(0.5), vfma(vneg(z[2]), d2, n.n[2]));
            const T d3 = vfmac<T>(-P.vcf, n.Tf, n.n[3]);
            a3 = vfmac<T>(P.quart_varpi, S_pcm, vmulc<T>(R(0.25), vfma(vneg(z[3]), d3, n.n[3])));
            z4 = vmulc<T>(R(0.25), vaddc(vneg(z[4]), R(1)));
        } else {
            jx = vmulc<T>(P.z_j, n.n[1]);
            jy = vmulc<T>(P.z_j, n.n[2]);
            if constexpr (FLOW) {
                const T t = vmulc<T>(P.z_ju, n.Tf);
                jx = vfma(t, n.ux, jx);
                jy = vfma(t, n.uy, jy);
            }
            a3 = vfmac<T>(P.z_3, n.n[3], vfmac<T>(P.z_3T, n.Tf, vmulc<T>(P.quart_varpi, S_pcm)));
        }
        const T c3 = vfmac<T>(P.e_3, n.k[3], vfmac<T>(P.e_3T, n.k[0], vmulc<T>(P.quart_varpi, S_met)));
        const T gp = vfma(z4, n.n[4], a3), gm = vfma(vneg(z4), n.n[4], a3);
        const T hp = vfmac<T>(P.e_4, n.k[4], c3), hq = vfmac<T>(-P.e_4, n.k[4], c3);
        if (FLOW || (PH && P.phase_k)) {
            g[1] = vadd(gp, jx); g[3] = vsub(gp, jx); g[2] = vadd(gm, jy); g[4] = vsub(gm, jy);
        } else {
            g[1] = vfmac<T>(P.z_j, n.n[1], gp); g[3] = vfmac<T>(-P.z_j, n.n[1], gp);
            g[2] = vfmac<T>(P.z_j, n.n[2], gm); g[4] = vfmac<T>(-P.z_j, n.n[2], gm);
        }
        h[1] = vfmac<T>(P.e_j, n.k[1], hp); h[3] = vfmac<T>(-P.e_j, n.k[1], hp);
        h[2] = vfmac<T>(P.e_j, n.k[2], hq); h[4] = vfmac<T>(-P.e_j, n.k[2], hq);
        g[0] = vfmac<T>(R(-4), a3, n0);
        h[0] = vfmac<T>(R(-4), c3, hm);
    } else {
        T a[9], c[9], z[9];
#pragma unroll
        for (int k = 1; k < 9; ++k) z[k] = bc<T>(P.nz[k]);
        if (PH && P.phase_k) {
            const T za = vrcp(vaddc(vfma(bc<T>(P.kd_c), n.fl, bc<T>(P.ks_c)), R(0.5)));
#pragma unroll
            for (int k = 1; k < 9; ++k) z[k] = vneg(vfma(bc<T>(P.zr_b[k]), za, bc<T>(P.zr_a[k])));
        }
        const T cT = vmulc<T>(P.c_fref, n.Tf), cM = vmulc<T>(P.c_mref, n.k[0]);
        const T t = vmulc<T>(P.inv_phi, n.Tf), mt = vneg(t);
        // distances from the equilibria of Eqs. 34 and 45 (zero for k = 7, 8)
        const T d[9] = {n.n[0], vsub(n.n[1], vfmac<T>(R(-4), n.n[0], vadd(cT, cT))),
                        vsub(n.n[2], vfmac<T>(R(4), n.n[0], vmulc<T>(R(-3), cT))),
                        FLOW ? vfma(mt, n.ux, n.n[3]) : n.n[3], FLOW ? vfma(t, n.ux, n.n[4]) : n.n[4],
                        FLOW ? vfma(mt, n.uy, n.n[5]) : n.n[5], FLOW ? vfma(t, n.uy, n.n[6]) : n.n[6], n.n[7], n.n[8]};
        const T e[9] = {n.k[0], vsub(n.k[1], vfmac<T>(R(-4), n.k[0], vadd(cM, cM))),
                        vsub(n.k[2], vfmac<T>(R(4), n.k[0], vmulc<T>(R(-3), cM))),
                        n.k[3], n.k[4], n.k[5], n.k[6], n.k[7], n.k[8]};
#pragma unroll
        for (int k = 1; k < 9; ++k) {
            a[k] = vfma(z[k], d[k], n.n[k]);
            c[k] = vfma(bc<T>(P.ne[k]), e[k], n.k[k]);
        }
        a[1] = vfmac<T>(R(-2), S_pcm, a[1]);
        a[2] = vadd(a[2], S_pcm);
        c[1] = vfmac<T>(R(-2), S_met, c[1]);
        c[2] = vadd(c[2], S_met);
        a[0] = n0;
        c[0] = hm;
        f_from_m9<T>(a, g);
        f_from_m9<T>(c, h);
    }
    if constexpr (kSplit<M>) {
        // 16-bit deviations from the reference of the provisional rest population,
        // then the rest population readers will see the balance with.  Readers
        // rebuild the reference from the stored rest population g_0; with
        // Y = n_0 - sum of the stored deviations the balance needs
        // g_0 + omega ref(g_0) = Y, and since g_0 = H - omega c_ref T(H) is the
        // equilibrium rest population of an enthalpy H (Eqs. 38, 40, B3; Eqs. 49,
        // B5 for the metal), the solution is that of H = Y: g_0 = Y - omega
        // c_ref T(Y), whose reference is c_ref T(Y).  The stored populations as
        // read then carry n_0 to FP32 rounding.
        const T ref = pcm_ref(P, g[0]);
        T sg, sh;
#pragma unroll
        for (int k = 1; k < QT; ++k) {
            const int w = QT == 5 ? 1 : k;
            const T dg = put<M>(db + PL::pcm(k) * PS, vfmac<T>(-P.w_move[w], ref, g[k]));
            const T dh = put<M>(db + PL::met(k) * PS, vfmac<T>(-P.wk_move[w], h[0], h[k]));
            sg = k == 1 ? dg : vadd(sg, dg);
            sh = k == 1 ? dh : vadd(sh, dh);
        }
        const T Y = vsub(n0, sg);
        T TY, fY;
        enthalpy_state(P, Y, TY, fY);
        put_real(dw, vfmac<T>(-P.om_cf, TY, Y));
        put_real(dw + PS, vmulc<T>(P.rest_m, vsub(hm, sh)));
    } else {
#pragma unroll
        for (int k = 1; k < QT; ++k) {
            put<M>(db + PL::pcm(k) * PS, g[k]);
            put<M>(db + PL::met(k) * PS, h[k]);
        }
        if constexpr (kComp<M>) {
            // the metal's rest population takes what its movers give up, t, and the source,
            // without passing through their sum with the rest population, whose rounding is
            // coarser; what it took of the source after rounding is what the PCM gives
            const T t = vsub(n.hs, mover_sum<QT>(h));
            const T rh = vadd(n.h0, vadd(t, S_met));
            put<M>(db + PL::met(0) * PS, rh);
            const T S = vmul_alone(bc<T>(P.x_pm), vsub(vsub(rh, n.h0), t));
            // (the PCM rest population is a float-float pair)
            const T n0 = vadd(n.n[0], S);
            const FF<T> s = mover_sum_ff<QT>(g);
            const T r = vsub(n0, s.hi);
            const T lo = vadd(vadd(sum_err(n.n[0], S, n0), n.Hlo), vsub(sum_err(n0, vneg(s.hi), r), s.lo));
            const FF<T> rest = fast_two_sum(r, lo);
            put<M>(db + PL::pcm(0) * PS, rest.hi);
            put<M>(db + PL::lo * PS, rest.lo);
        } else {
            put<M>(db + PL::met(0) * PS, vsub(hm, mover_sum<QT>(h)));
            put<M>(db + PL::pcm(0) * PS, vsub(n0, mover_sum<QT>(g)));
        }
    }
    return dTn;
}

// Non-finite or runaway state: raises the sticky flag (no trap).  A NaN
// anywhere fails a comparison; the sum overflows if any term is huge.
template <typename R>
__device__ __forceinline__ bool runaway(R H, R Tm, R rho, R um) {
    if constexpr (sizeof(R) == 8) {   // nothing large (2^97), on the high words: no FP64 operation
        const int big = (1023 + 97) << 20;
        const unsigned h = __double2hiint(rho), u = __double2hiint(um);
        if ((__double2hiint(H) & 0x7fffffff) < big && (__double2hiint(Tm) & 0x7fffffff) < big && h - 1 < big - 1 &&
            u < (unsigned)__double2hiint(0.3))
            return false;
    }
    return !(fabs(H) + fabs(Tm) + rho < R(1e30)) || !(rho > R(0)) || !(um <= R(0.3));
}

template <int M, int QT, bool FLOW, typename T>
__device__ __forceinline__ void check_state(const StepParams<typename ModeTraits<M>::R>& P,
                                            const NodeState<M, QT, FLOW, T>& n) {
    bool bad;
    if constexpr (Lane<T>::n == 2)
        bad = runaway(n.n[0].x, n.k[0].x, n.rho.x, n.um.x) || runaway(n.n[0].y, n.k[0].y, n.rho.y, n.um.y);
    else
        bad = runaway(n.n[0], n.k[0], n.rho, n.um);
    if (bad) atomicOr(P.status, STATUS_UNSTABLE);
}

// Node (x, y)'s element in bulk plane 0 and in wide plane 0 (16-bit modes) of
// the next copy.
template <int M, int QT, bool FLOW>
__device__ __forceinline__ typename ModeTraits<M>::B* next_bulk(const StepParams<typename ModeTraits<M>::R>& P, int x,
                                                                int y) {
    const long long ro = (long long)y * (P.cpr * Chunk<M, QT, FLOW>::bytes);
    return reinterpret_cast<typename ModeTraits<M>::B*>(P.dst + (ro + col_off<M, QT, FLOW>(x)));
}

template <int M, int QT, bool FLOW>
__device__ __forceinline__ float* next_wide(const StepParams<typename ModeTraits<M>::R>& P, int x, int y) {
    if constexpr (kSplit<M>) {
        const long long ro = (long long)y * (P.cpr * Chunk<M, QT, FLOW>::bytes);
        return reinterpret_cast<float*>(P.dst + (ro + col_off<M, QT, FLOW, true>(x)));
    } else {
        return nullptr;
    }
}

// One time step of a node (pair) whose neighbourhood the accessor a reads:
// steps a1-a9 (pull, walls, state, blend, velocity, three collisions, store).
// PH = true compiles the Eq. 9 variant's per-node PCM rates in (taken where
// P.phase_k is set); PH = false leaves them out of the kernel altogether.
// The history is read before any store: the compiler cannot move it above
// stores that may alias it, and a load after them adds a memory round trip to
// the step; LATE (FP32, one node per thread), it is read after the state is known,
// and the thermal lattices are pulled first (one step per launch 330^2 3.17 ->
// 2.98 us, 512^2 4.98 -> 4.84, 1024^2 27.3 -> 26.4).  TF: the thermal lattices
// collide before the flow.  Returns the new history.
template <int M, int QT, bool FLOW, bool PH, int PS, typename T, bool TF = false, bool LATE = kComp<M>, typename A>
__device__ __forceinline__ T advance(const StepParams<typename ModeTraits<M>::R>& P, const A& a, const WallAt<T>& w,
                                     const typename Lane<T>::R* history, typename ModeTraits<M>::B* db, float* dw) {
    NodeState<M, QT, FLOW, T> n;
    T dTp;
    if constexpr (Lane<T>::n == 1 && !LATE) dTp = get_real<T>(history);
    node_state<M, QT, FLOW, T, LATE>(P, a, w, n);
    if constexpr (Lane<T>::n == 1 && LATE) dTp = get_real<T>(history);
    if constexpr (!TF) flow_collide<M, QT, FLOW, PS, T>(P, n, db);
    if constexpr (Lane<T>::n == 2) dTp = get_real<T>(history);
    const T dTn = thermal_collide<M, QT, FLOW, PH, PS, T>(P, n, dTp, db, dw);
    if constexpr (TF) flow_collide<M, QT, FLOW, PS, T>(P, n, db);
    check_state<M, QT, FLOW, T>(P, n);
    return dTn;
}

// One time step of node (x, y) from the state copy to the next.
template <int M, int QT, bool FLOW, bool PH = false, bool EV = false, bool TF = false, bool LATE = kComp<M>>
__device__ __forceinline__ void step_node(const StepParams<typename ModeTraits<M>::R>& P, int x, int y) {
    using T = Node1<M>;
    const WallAt<T> w(P, x, y);
    T* h = P.dT + (y * P.pitch + x);
    *h = advance<M, QT, FLOW, PH, kChunk, T, TF, LATE>(P, PullAt<M, QT, FLOW, EV>(P, w.xs, w.ys), w, h,
                                              next_bulk<M, QT, FLOW>(P, x, y), next_wide<M, QT, FLOW>(P, x, y));
}

// One time step of the node pair (x0, x0 + 1), x0 even, both in the grid.
template <int M, int QT, bool PH = false, bool EV = false>
__device__ __forceinline__ void step_pair(const StepParams<float>& P, int x0, int y) {
    const WallAt<W> w(P, x0, y);
    float* h = P.dT + (y * P.pitch + x0);
    put_real(h, advance<M, QT, true, PH, kChunk, W>(P, PairAt<M, QT, EV>(P, x0, w.ys), w, h,
                                                     next_bulk<M, QT, true>(P, x0, y), next_wide<M, QT, true>(P, x0, y)));
}

// Blocks of 256 threads each SM must hold, which caps the registers per
// thread: five for the FP32 and 16-bit forms of D2Q5 with flow (48 registers,
// where the FP32 step at 2048^2 runs at the copy bandwidth) and four for 16-bit
// D2Q9 (64: at the 72 it takes uncapped, fewer warps stay resident: 512^2 FP16 7.08 /
// 6.80 us per step, 2048^2 BF16 101.4 / 98.1, a batch of 60 runs under map 3 48.9 / 45.9);
// the others take what their registers allow (FP64 and FP32 D2Q9, where four
// blocks cost single runs 1-4 %, are bound by arithmetic).
template <int M, int QT, bool FLOW>
constexpr int kMinBlocks = !FLOW || M == MODE_F64 ? 1 : QT == 5 ? 5 : kSplit<M> ? 4 : 1;

// The same of grouped launches' blocks of 128 threads: the D2Q9 forms, whose many
// runs fill the device, at 64 registers (60 runs under map 4, us per step of all,
// uncapped, FP32 73 and 16-bit 96 registers / 64: FP32 58.0 / 55.3, FP16 55.8 / 47.1,
// BF16 56.4 / 47.1; 12 runs FP32 10.8 / 9.9, FP16 10.9 / 9.2).
template <int M, int QT, bool FLOW>
constexpr int kGroupBlocks = QT == 9 && FLOW && M != MODE_F64 ? 8 : 2 * kMinBlocks<M, QT, FLOW>;

// Programmatic dependent launch (sm_90 and later): the step kernels are
// launched as programmatic dependents of the previous step, so their launch
// overlaps its tail.  griddep_wait blocks until the previous grid in the
// stream has completed and its writes are visible (it returns at once when
// this grid was not launched as a programmatic dependent); no thread touches
// the state before it.  The dependents are released when this grid's blocks
// exit (no early trigger: dependents scheduled while this grid still runs took
// its SM resources, 256^2 went from 2.75 to 3.52 us per step; released at exit,
// 2.50).
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// L2 prefetch ahead of the blocks that will run next (node pairs and two steps
// per launch on large grids): a block's first thread asks L2, by bulk prefetches
// (cp.async.bulk.prefetch.L2), for the chunk of x in `rows` rows starting at
// y0 and for their exchange history, so that the block launched for those
// rows later finds them in L2 instead of waiting for HBM.  No registers or
// shared memory hold the data; rows past the grid are skipped.
__device__ __forceinline__ void l2_prefetch(const void* p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

template <int M, int QT, bool FLOW>
__device__ __forceinline__ void prefetch_rows(const StepParams<typename ModeTraits<M>::R>& P, int x, int y0, int rows) {
    using R = typename ModeTraits<M>::R;
    constexpr uint32_t cb = Chunk<M, QT, FLOW>::bytes;   // a multiple of 16, as is every chunk's offset
    for (int y = y0; y < y0 + rows && y < P.ny; ++y) {
        l2_prefetch(P.src + ((long long)y * P.cpr + (x >> kChunkShift)) * cb, cb);
        l2_prefetch(P.dT + (long long)y * P.pitch + (x & ~(kChunk - 1)), kChunk * (uint32_t)sizeof(R));
    }
}

// One run: one thread per node, in blocks of the launcher's choice (step_block;
// up to 256 threads, the batch's map 3 may take any of its shapes).  FP32 grids
// beyond L2 are bound by HBM (2048^2 100 us per step, 160 B per update at
// 6.7 TB/s); smaller ones by the launch floor, one warp's chain and instruction
// issue (256^2 2.41 us per step before the update was written in named
// multiply-adds and single-instruction reciprocals and roots, 2.21 now).  FP64
// is bound by its two lanes per SM and clock: 252 FP64 operations per node took
// 39.7 us per step at 256^2, 187 take 27.6 (in 64 x 1 blocks).
template <int M, int QT, bool FLOW, bool PH, bool EV = false>
__global__ void __launch_bounds__(256, (kMinBlocks<M, QT, FLOW>)) fused_step(const __grid_constant__ StepParams<typename ModeTraits<M>::R> P) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= P.nx || y >= P.ny) return;
    griddep_wait();
    step_node<M, QT, FLOW, PH, EV>(P, x, y);
}

// FP64 runs without flow on grids that leave most schedulers idle: two lanes
// per node, the even one with the PCM, the odd one with the metal lattice.  One
// warp's chain of FP64 operations, 64 cycles each whatever its lanes do, is the
// step's time there (200 x 4: both lattices in one lane 3.46 us a step, one
// each 2.63, 4.96 before either), and the two lattices take the same operations
// with constants of their own; the temperatures cross by shuffle.  Operation for
// operation step_node's, D2Q5 with constant PCM properties.
template <int M>   // MODE_F64
__global__ void __launch_bounds__(64) conduction_step_lanes(const __grid_constant__ StepParams<double> P) {
    const int xr = blockIdx.x * 32 + (threadIdx.x >> 1), y = blockIdx.y;
    const bool metal = threadIdx.x & 1, live = xr < P.nx;
    // a warp without a node returns: it would read the history that another warp writes, in no order
    if (blockIdx.x * 32 + (threadIdx.x >> 5) * 16 >= P.nx) return;
    const int x = live ? xr : P.nx - 1;   // lanes beyond the grid go along with their own warp and put nothing
    griddep_wait();
    const WallAt<double> w(P, x, y);
    const PullAt<M, 5, false> a(P, w.xs, w.ys);
    double* h = P.dT + (y * P.pitch + x);
    const double dTp = *h;
    const int first = metal ? 5 : 0;   // the lattice's first plane
    double g[5], n[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) g[q] = __ldg(a.src(q) + (first + q) * kChunk);
    thermal_moments<double, 5>(g, n);
    double Tf, fl;
    enthalpy_state(P, n[0], Tf, fl);
    auto exchange = [&]() {   // both temperatures on both lanes
        const double mine = metal ? n[0] : Tf, other = __shfl_xor_sync(0xffffffffu, mine, 1);
        Tf = metal ? other : mine;
        return metal ? mine : other;
    };
    double Tm = exchange();
    if (__any_sync(0xffffffffu, w.wall && P.wall_kind[w.side] == 0)) {
        if (w.wall && P.wall_kind[w.side] == 0) {   // Eq. 52 (an adiabatic wall at rest keeps x_f's moments)
            const double Tb = P.wall_T[w.side];
            n[3] = vfma(metal ? P.vcm : P.vcf, vsub(Tb, metal ? Tm : Tf), n[3]);
            n[0] = metal ? Tb : P.wall_H[w.side];
            enthalpy_state(P, n[0], Tf, fl);
        }
        Tm = exchange();
    }
    const double S_met = vfma(P.x_now, vsub(Tm, Tf), vmul(P.x_prev, dTp));
    const double hm = vadd(Tm, S_met), took = vsub(hm, Tm);
    const double S = metal ? S_met : vmul(P.x_pm, took), n0 = metal ? hm : vfma(P.x_pm, took, n[0]);
    const double zj = metal ? P.e_j : P.z_j;
    const double a3 = vfma(metal ? P.e_3 : P.z_3, n[3],
                           vfma(metal ? P.e_3T : P.z_3T, metal ? Tm : Tf, vmul(P.quart_varpi, S)));
    const double z4 = metal ? P.e_4 : P.z_4;
    const double p = vfma(z4, n[4], a3), q = vfma(-z4, n[4], a3);
    const double v1 = vfma(zj, n[1], p), v3 = vfma(-zj, n[1], p), v2 = vfma(zj, n[2], q), v4 = vfma(-zj, n[2], q);
    __syncwarp();   // both lanes have read the history that one of them writes
    if (!live) return;
    double* db = next_bulk<M, 5, false>(P, x, y) + first * kChunk;
    db[0] = vsub(n0, vadd(vadd(v1, v3), vadd(v2, v4)));
    db[kChunk] = v1;
    db[2 * kChunk] = v2;
    db[3 * kChunk] = v3;
    db[4 * kChunk] = v4;
    if (!metal) {
        *h = vsub(Tm, Tf);
        if (runaway(n[0], Tm, 1.0, 0.0)) atomicOr(P.status, STATUS_UNSTABLE);
    }
}

// ---------------------------------------------------------------------------
// Two time steps per launch
// ---------------------------------------------------------------------------
// On small grids (state resident in L2) a step costs the launch-to-launch floor
// of a dependent launch plus one warp's dependency chain with its L2 loads,
// more than the issue time of the work itself; on grids whose state exceeds
// L2 a step moves the whole state through HBM.  fused_step2 advances two time
// steps per launch.  A block of kT2W x H threads (one node each, 4 <= H <=
// kT2H) owns an inner tile of (kT2W - 2) x (H - 2) nodes and the one-node ring
// around it:
//   1. every thread advances its node one step from the state in global
//      memory (the ring's nodes belong to neighbouring tiles and are advanced
//      there too), storing the result in shared memory in the storage
//      encoding of a state copy, as a global store would;
//   2. after a barrier, the inner nodes advance a second step with their
//      neighbourhood read from shared memory, and store to the next copy.
// Tile origins are clamped to the grid (the last tile along an axis ends at
// the grid's edge, overlapping its neighbour), so that a wall node's x_f and
// the neighbours of x_f lie in the tile (H >= 4).  Nodes of overlapping tiles
// are computed by both blocks with the same inputs and code, and written with
// the same values.  The history is read from P.dT and written to P.dT_out:
// other blocks still read the previous history of their rings.  Flow runs
// only.  The host picks H per grid (t2_block in the launcher).  Three builds of
// the kernel: HM = kT2H (any H up to 15, registers as they come: fastest where
// one or two blocks per SM fit anyway); HM = kT2HTwo (tiles of up to 14 rows,
// two per SM, capped at 64 registers for two resident blocks where the first
// build's registers would leave one: FP16 320^2 3.40 -> 2.62 us per step, 334 x
// 303 3.55 -> 2.90; on smaller tiles the cap costs, 64^2 1.186 -> 1.218); and HM =
// kT2HMany (H = 12 for grids of many tiles per SM, launch bounds that leave
// three FP32 D2Q5 blocks resident: at 52 registers only two fit, 2048^2 FP32
// 104 against 84 us per step; two blocks of the other builds, which would spill
// under the three-block cap).  Small grids are bound by the
// launch floor and two dependency chains (64^2 FP32 1.315 us per step before
// the update was written in named multiply-adds, 1.09 now; 256^2 2.05 and 1.82),
// grids beyond L2 by instruction issue once their rows are prefetched (2048^2
// 79.9 us per step before, 70.6 now; 49.5 at the copy bandwidth).  Two nodes
// per thread in the tile, side by side or one above the other, were slower
// (2048^2 77.0 and 73.3, 64^2 1.37): more registers, fewer warps.
constexpr int kT2W = 34, kT2H = 15, kT2HTwo = 14, kT2HMany = 12;

template <int HM, int M, int QT>
constexpr int kT2Blocks = HM == kT2HMany ? (M == MODE_F32 && QT == 5 ? 3 : 2) : HM == kT2HTwo ? 2 : 1;

// Dynamic shared memory of a two-step block of up to HM rows, planes
// kT2W * HM elements apart: the bulk planes (storage type), the wide planes
// (FP32) and the history.
template <int M, int QT, int HM>
struct Tile2 {
    using PL = Planes<M, QT, true>;
    static constexpr int n = (kT2W * HM + 7) / 8 * 8;
    static constexpr size_t wide_off = (size_t)PL::bulk * n * sizeof(typename ModeTraits<M>::B);
    static constexpr size_t dT_off = wide_off + (size_t)PL::wide * n * sizeof(float);
    static constexpr size_t bytes = dT_off + (size_t)n * sizeof(typename ModeTraits<M>::R);
    static_assert(wide_off % 16 == 0 && dT_off % 16 == 0, "16-byte aligned parts");
};

// Neighbourhood of the node at tile index i (pull node) in the tile, planes
// PS elements apart.
template <int M, int PS>
struct PullTile {
    const typename ModeTraits<M>::B* b;
    const float* wd;
    int i;
    __device__ __forceinline__ int at(int q) const { return i + (src_row(q) - 1) * kT2W + (src_col(q) - 1); }
    __device__ __forceinline__ typename ModeTraits<M>::R bulk(int q, int plane) const {
        return to_f(b[plane * PS + at(q)]);
    }
    __device__ __forceinline__ float wide(int q, int p) const { return wd[p * PS + at(q)]; }
};

// First node of the ring of tile k along an axis of n nodes with inner width w.
__host__ __device__ __forceinline__ int t2_origin(int k, int w, int n) {
    return (n > w ? min(k * w, n - w) : 0) - 1;
}

// Tiles along an axis of n nodes with inner width w.
__host__ __device__ __forceinline__ int t2_count(int n, int w) { return n > w ? (n + w - 1) / w : 1; }

// Both steps of tile (bx, by) of run P, by a block of kT2W x blockDim.y
// threads (blockDim.y <= HM) with Tile2<M, QT, HM>::bytes of dynamic shared
// memory.
template <int M, int QT, bool PH, int HM, bool EV = false, bool TF = false>
__device__ __forceinline__ void step2_tile(const StepParams<typename ModeTraits<M>::R>& P, int bx, int by) {
    using R = typename ModeTraits<M>::R;
    using B = typename ModeTraits<M>::B;
    using TL = Tile2<M, QT, HM>;
    extern __shared__ __align__(16) unsigned char t2_smem[];
    B* sb = reinterpret_cast<B*>(t2_smem);
    float* sw = reinterpret_cast<float*>(t2_smem + TL::wide_off);
    R* sdT = reinterpret_cast<R*>(t2_smem + TL::dT_off);
    const int H = blockDim.y;   // blockDim.x == kT2W, H <= HM
    const int lx = threadIdx.x, ly = threadIdx.y, i = ly * kT2W + lx;
    const int x2 = t2_origin(bx, kT2W - 2, P.nx) + lx, y2 = t2_origin(by, H - 2, P.ny) + ly;
    // step-1 node: coordinates wrapped on periodic sides, none beyond a walled side
    int x = x2, y = y2;
    bool live = true;
    if (x < 0 || x >= P.nx) {
        if (P.per_x) x = ((x % P.nx) + P.nx) % P.nx;
        else live = false;
    }
    if (y < 0 || y >= P.ny) {
        if (P.per_y) y = ((y % P.ny) + P.ny) % P.ny;
        else live = false;
    }
    griddep_wait();
    // the tile's rows, prefetch_rows further on, of the chunk that starts at its first inner
    // column (in the many-tiles build only: the test costs 64^2 0.03 us a step)
    if (HM == kT2HMany && !EV && P.prefetch_rows > 0 && lx == 1 && (x2 & (kChunk - 1)) == 0 && ly >= 1 && ly <= H - 2)
        prefetch_rows<M, QT, true>(P, x2, y2 + P.prefetch_rows, 1);
    if (live) {
        const WallAt<R> w(P, x, y);
        sdT[i] = advance<M, QT, true, PH, TL::n, R, TF>(P, PullAt<M, QT, true, EV>(P, w.xs, w.ys), w, P.dT + (y * P.pitch + x),
                                                     sb + i, sw + i);
    }
    __syncthreads();
    // step 2: the inner nodes of the tile that lie in the grid
    if (lx < 1 || lx > kT2W - 2 || ly < 1 || ly > H - 2 || x2 >= P.nx || y2 >= P.ny) return;
    const WallAt<R> w(P, x2, y2);
    const PullTile<M, TL::n> a{sb, sw, i + (w.ys - y2) * kT2W + (w.xs - x2)};
    P.dT_out[y2 * P.pitch + x2] = advance<M, QT, true, PH, kChunk, R, TF>(
        P, a, w, sdT + i, next_bulk<M, QT, true>(P, x2, y2), next_wide<M, QT, true>(P, x2, y2));
}

template <int M, int QT, bool PH, int HM, bool EV = false, bool TF = false>
__global__ void __launch_bounds__(kT2W * HM, (kT2Blocks<HM, M, QT>)) fused_step2(const __grid_constant__ StepParams<typename ModeTraits<M>::R> P) {
    step2_tile<M, QT, PH, HM, EV, TF>(P, blockIdx.x, blockIdx.y);
}

// ---------------------------------------------------------------------------
// Two nodes per thread
// ---------------------------------------------------------------------------

// Runs of the default configuration (flow, D2Q5 thermal lattices, volumetric
// blend, FP32/FP16/BF16 storage) may advance node pairs (x0, x0 + 1), x0 even,
// one pair per thread: the parameter loads and the index arithmetic serve both
// nodes, and the pair is read and written with one access per plane wherever
// both elements are adjacent (x0 even keeps them inside one chunk, aligned).
// The last node of an odd width, and both nodes of a bounce-back run, step
// one by one.  Bound by instruction issue up to L2's size and by HBM beyond
// (us per step, before / with the update in named multiply-adds and 80
// registers: FP16 512^2 5.52 / 4.77 (before: one node per thread), 1024^2 18.4 /
// 15.2, 2048^2 61.2 / 57.5, BF16 2048^2 61.3 / 57.6).
template <int M, bool PH, bool EV = false>
__device__ __forceinline__ void step_pair_or_nodes(const StepParams<float>& P, int x0, int y) {
    if (!P.solid_scheme && x0 + 1 < P.nx) {
        step_pair<M, 5, PH, EV>(P, x0, y);
    } else {
#pragma unroll 1
        for (int x = x0; x < min(x0 + 2, P.nx); ++x) step_node<M, 5, true, PH, EV>(P, x, y);
    }
}

// Blocks of pairs per SM: six of 128 threads cap the registers at 80.  Seven
// (72 registers) spill some 50 bytes: 2048^2 FP16 59.5 against 58.5 us per
// step, BF16 60.4 against 57.8 (56.9 at the copy bandwidth on the 92 bytes the
// form moves); eight, 78; three blocks of 256 threads, 61.7.
constexpr int kPairBlocks = 6;

// A block of 32 x 4 threads covers 64 x 4 nodes; the first of a chunk's two
// blocks prefetches its rows (2048^2 FP16 61.09 against 61.22 us per step when
// both did).
template <int M, bool PH, bool EV = false>
__global__ void __launch_bounds__(128, kPairBlocks) fused_step_pair(const __grid_constant__ StepParams<float> P) {
    const int x0 = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x0 >= P.nx || y >= P.ny) return;
    griddep_wait();
    if (!EV && P.prefetch_rows > 0 && threadIdx.x == 0 && threadIdx.y == 0 && (x0 & (kChunk - 1)) == 0)
        prefetch_rows<M, 5, true>(P, x0, y + P.prefetch_rows, blockDim.y);   // the chunk's first block
    step_pair_or_nodes<M, PH, EV>(P, x0, y);
}

// Many small runs in one launch per step, each run on the code of the
// single-run kernel (map 4 of a batch).  The parameter blocks of up to
// kGroupRuns runs travel in the kernel's own parameter space (the constant
// bank, up to 32 KB), with the prefix sums of the runs' block counts; block b
// finds its run by a binary search over them (uniform across the block) and
// takes block b - first_block[run] of that run's tiles: w x (128 / w) nodes,
// one node per thread, w = 32 << tile[run] chosen so that the run's width
// leaves the fewest threads idle.  With all small runs in one grid the device
// sees one large launch instead of many small ones, each bound by the latency
// of a few warps.
template <typename R>
constexpr int kGroupRuns = (32000 - 16) / (int)(sizeof(StepParams<R>) + 2 * sizeof(int));

// Groups of up to kGroupFew runs have a build of their own with smaller
// parameters: a launch and a graph node copy all of them, 30 KB at full size
// (12 FP16 cavities in two groups, first 64 steps with the graph's build 1.92
// ms at full size).
constexpr int kGroupFew = 8;

template <typename R, int NR>
struct GroupParams {
    int nruns;
    int first_block[NR + 1];
    int tile[NR];
    StepParams<R> run[NR];
};

// The run of block b: the last one whose first block is <= b.
template <typename R, int NR>
__device__ __forceinline__ int group_run(const GroupParams<R, NR>& G, int b) {
    int lo = 0, hi = G.nruns - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (G.first_block[mid] <= b) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

template <int M, int QT, bool FLOW, bool PH, int NR, bool EV>
__global__ void __launch_bounds__(128, (kGroupBlocks<M, QT, FLOW>)) group_step(
    const __grid_constant__ GroupParams<typename ModeTraits<M>::R, NR> G) {
    const int b = blockIdx.x, lo = group_run(G, b);
    const StepParams<typename ModeTraits<M>::R>& P = G.run[lo];
    const int lb = b - G.first_block[lo];
    const int lw = 5 + G.tile[lo];   // log2 of the tile width
    const int t = (int)threadIdx.x;
    const int gx = (P.nx + (1 << lw) - 1) >> lw;
    const int x = (lb % gx) * (1 << lw) + (t & ((1 << lw) - 1));
    const int y = (lb / gx) * (128 >> lw) + (t >> lw);
    if (x >= P.nx || y >= P.ny) return;
    griddep_wait();
    step_node<M, QT, FLOW, PH, EV>(P, x, y);
}

// The same for runs in 16-bit storage with flow and the D2Q5 thermal lattices,
// a node pair per thread: tiles of w x 256 / w nodes, w = 32 << tile.  Batches
// with nodes enough (group_pairs) are bound by instruction issue, and a pair takes some 650 instructions
// where its nodes one by one take 1,000 (64 cavities of 64-512 nodes a side,
// FP16: 132.7 us per step of all with one node per thread, 123.1 with pairs;
// 12 cavities 22.2 and 17.5 with the groups side by side as well).
template <int M, bool PH, int NR, bool EV>
__global__ void __launch_bounds__(128, kPairBlocks) group_step_pair(const __grid_constant__ GroupParams<float, NR> G) {
    const int b = blockIdx.x, lo = group_run(G, b);
    const StepParams<float>& P = G.run[lo];
    const int lb = b - G.first_block[lo];
    const int lw = 5 + G.tile[lo], lp = lw - 1;   // log2 of the tile width in nodes and in pairs
    const int t = (int)threadIdx.x;
    const int gx = (P.nx + (1 << lw) - 1) >> lw;
    const int x0 = (lb % gx) * (1 << lw) + 2 * (t & ((1 << lp) - 1));
    const int y = (lb / gx) * (128 >> lp) + (t >> lp);
    if (x0 >= P.nx || y >= P.ny) return;
    griddep_wait();
    step_pair_or_nodes<M, PH, EV>(P, x0, y);
}

// Batch map 5: the grouped launch of the two-step form.  Run k owns blocks
// first_block[k] .. first_block[k + 1] - 1, one per two-step tile (blocks of
// kT2W x kT2HMany threads, inner tiles of (kT2W - 2) x (kT2HMany - 2) nodes,
// row-major over the run's tiles); each block advances its tile two steps as
// fused_step2 does, with its run's parameter block.
template <int M, int QT, bool PH, int NR, bool EV>
__global__ void __launch_bounds__(kT2W * kT2HMany, (kT2Blocks<kT2HMany, M, QT>)) group_step2(
    const __grid_constant__ GroupParams<typename ModeTraits<M>::R, NR> G) {
    const int b = blockIdx.x, lo = group_run(G, b);
    const StepParams<typename ModeTraits<M>::R>& P = G.run[lo];
    const int lb = b - G.first_block[lo];
    const int gx = t2_count(P.nx, kT2W - 2);
    step2_tile<M, QT, PH, kT2HMany, EV>(P, lb % gx, lb / gx);
}

// Many runs in one launch.  A tile is w x (256 / w) nodes of one run (w a
// power of two, 32..256); thread t of a block takes node (x0 + t mod w,
// y0 + t div w).  Each run has two parameter blocks in global memory, one per
// ping-pong direction ([run][2]); a run whose current copy differs from the
// batch's parity carries flip = 1 in its tiles.  A block copies the block of
// its current run into shared memory when the run changes.  Map: chunk > 0
// gives block b the tiles [b chunk, (b+1) chunk), chunk = 0 strides over the
// tiles by the grid size.
struct Tile {
    int run, x0, y0, log2w_flip;   // log2 w in bits 0-7, flip in bit 8
};

// The order of a node's reads and collisions and the register bound are what
// measured best with the parameters in shared memory (us per step of all, FP32
// D2Q5 with LATE / without: 12 runs under map 0 10.0 / 9.8, 60 runs 55.6 / 55.0;
// FP16 D2Q5 flow / thermal lattices first: 12 runs 11.3 / 11.1, 60 runs 51.8 / 50.2; FP32
// D2Q9 unbounded / with three blocks per SM: 12 runs 15.7 / 15.2, 60 runs 76.2 / 72.5).
template <int M, int QT, bool FLOW, bool PH>
__global__ void __launch_bounds__(256, (M == MODE_F32 && QT == 9 && FLOW ? 3 : 0)) batch_step(const StepParams<typename ModeTraits<M>::R>* __restrict__ runs,
                                                  const Tile* __restrict__ tiles, int ntiles, int chunk, int parity) {
    using R = typename ModeTraits<M>::R;
    __shared__ StepParams<R> P;
    static_assert(sizeof(StepParams<R>) % 4 == 0, "parameter block copied as words");
    int cached = -1;
    const int t0 = chunk > 0 ? blockIdx.x * chunk : blockIdx.x;
    const int t1 = chunk > 0 ? min(ntiles, t0 + chunk) : ntiles;
    const int dt = chunk > 0 ? 1 : gridDim.x;
    for (int t = t0; t < t1; t += dt) {
        const Tile tl = tiles[t];
        if (tl.run != cached) {   // uniform across the block
            __syncthreads();
            const int dir = parity ^ ((tl.log2w_flip >> 8) & 1);
            const int* src = reinterpret_cast<const int*>(runs + 2 * tl.run + dir);
            int* dst = reinterpret_cast<int*>(&P);
            for (int i = threadIdx.x; i < (int)(sizeof(StepParams<R>) / 4); i += blockDim.x) dst[i] = __ldg(src + i);
            __syncthreads();
            cached = tl.run;
        }
        const int lg = tl.log2w_flip & 0xff;
        const int x = tl.x0 + (threadIdx.x & ((1 << lg) - 1));
        const int y = tl.y0 + (threadIdx.x >> lg);
        if (x < P.nx && y < P.ny)
            step_node<M, QT, FLOW, PH, false, M == MODE_F16 && QT == 5, kComp<M> && QT == 9>(P, x, y);
    }
}

// Fields at the current time level (LBM_FIELD_* order).
template <typename R>
struct FieldOut {
    R* dst[7];
    int mask;
    int ld;   // row stride of the outputs (elements)
};

template <int M, int QT, bool FLOW>
__global__ void __launch_bounds__(256) fields_kernel(const __grid_constant__ StepParams<typename ModeTraits<M>::R> P,
                                                     const __grid_constant__ FieldOut<typename ModeTraits<M>::R> out) {
    using R = typename ModeTraits<M>::R;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= P.nx || y >= P.ny) return;
    NodeState<M, QT, FLOW, R> n;
    node_state_at<M, QT, FLOW>(P, x, y, n);
    const long long o = (long long)y * out.ld + x;
    const R v[7] = {n.Tf, n.k[0], n.fl, n.ux, n.uy, n.rho, n.n[0]};   // H: high part
#pragma unroll
    for (int i = 0; i < 7; ++i)
        if (out.mask & (1 << i)) out.dst[i][o] = v[i];
}

// Diagnostics: FP64 sums of f_l, enthalpy, mass and the left-wall heat flux.
// An FP64 operation occupies a scheduler's FP64 unit for 64 cycles (two lanes
// per SM and clock), so the sums are arranged around their number: the
// conversions from FP32 are integer operations, the enthalpy's weights are
// applied to a thread's sums instead of to each node's terms, a thread takes
// up to eight rows before its block reduces, and the warp reduces its four
// sums in 6 additions instead of 20 (each exchange halves the sums a lane
// keeps).  The wall flux, three node states per row, has blocks of its own
// (the last column of blocks), beside the others instead of in their chains; they
// write their row's flux sum into the first column's partials.  GB300, us per
// lbm_diag call with the copy of the results, before / with this arrangement:
// FP32 64^2 38 / 30, 1024^2 115 / 54, 2048^2 359 / 130.
struct DiagConst {
    double phi, rho_l, rho_m, c_pm, k_f, k_s, k_m;   // k_f: liquid PCM conductivity, k_s: solid (Eq. 9)
    int left_wall;  // 1 when x = 0 is a wall (Nusselt number defined)
    int rows;       // rows of nodes per thread
};

// v as a double, by integer operations for zero and normal numbers.
__device__ __forceinline__ double to_double(double v) { return v; }
__device__ __forceinline__ double to_double(float v) {
    const unsigned u = __float_as_uint(v), m = u & 0x7fffffffu;
    if (m - 0x00800000u >= 0x7f000000u) return m ? (double)v : 0.0;   // subnormal, infinite, NaN; zero
    return __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(u << 29));
}

template <int M, int QT, bool FLOW>
__global__ void __launch_bounds__(256) diag_partial(const __grid_constant__ StepParams<typename ModeTraits<M>::R> P,
                                                    const __grid_constant__ DiagConst C,
                                                    double* __restrict__ scratch) {
    const int x = blockIdx.x * 128 + threadIdx.x;
    double fl = 0.0, H = 0.0, Tm = 0.0, drho = 0.0, flux = 0.0;
    const bool wall = blockIdx.x == gridDim.x - 1;
    if (wall) {   // the left wall's heat flux, a row per thread
        const int rows = blockDim.y * C.rows, y = blockIdx.y * rows + threadIdx.x;
        if (C.left_wall && threadIdx.y == 0 && threadIdx.x < rows && y < P.ny) {
            double tf[3], tm[3], kw = 0.0;
#pragma unroll 1
            for (int k = 0; k < 3; ++k) {
                NodeState<M, QT, FLOW, Node1<M>> n;
                node_state_at<M, QT, FLOW>(P, k, y, n);
                tf[k] = (double)n.Tf;
                tm[k] = (double)n.k[0];
                // PCM conductivity of the wall node's own liquid fraction (Eq. 9)
                if (k == 0) kw = C.k_s == C.k_f ? C.k_f : (double)n.fl * C.k_f + (1.0 - (double)n.fl) * C.k_s;
            }
            const double gf = 0.5 * (3.0 * tf[0] - 4.0 * tf[1] + tf[2]);
            const double gm = 0.5 * (3.0 * tm[0] - 4.0 * tm[1] + tm[2]);
            flux = C.phi * kw * gf + (1.0 - C.phi) * C.k_m * gm;
        }
    } else if (x < P.nx) {
        const int y0 = (blockIdx.y * blockDim.y + threadIdx.y) * C.rows, y1 = min(y0 + C.rows, P.ny);
#pragma unroll 1
        for (int y = y0; y < y1; ++y) {
            NodeState<M, QT, FLOW, Node1<M>> n;
            node_state_at<M, QT, FLOW>(P, x, y, n);
            fl += to_double(n.fl);
            H += to_double(n.n[0]);
            Tm += to_double(n.k[0]);
            if constexpr (M != MODE_F64) H += to_double(n.Hlo);
            if constexpr (kSplit<M>) Tm += to_double(n.Elo);
            if constexpr (FLOW) drho += to_double(n.drho);
        }
    }
    const double E = C.phi * C.rho_l * H + (1.0 - C.phi) * C.rho_m * C.c_pm * Tm;
    // lanes 0-15 take (fl, E), 16-31 (drho, flux); then each eight lanes one of the two
    const int lane = threadIdx.x & 31, warp = threadIdx.y * 4 + (threadIdx.x >> 5);
    const bool h16 = lane & 16, h8 = lane & 8;
    const double a = (h16 ? drho : fl) + __shfl_xor_sync(0xffffffffu, h16 ? fl : drho, 16);
    const double b = (h16 ? flux : E) + __shfl_xor_sync(0xffffffffu, h16 ? E : flux, 16);
    double v = (h8 ? b : a) + __shfl_xor_sync(0xffffffffu, h8 ? a : b, 8);
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    __shared__ double red[8][4];
    if ((lane & 7) == 0) red[warp][lane >> 3] = v;
    __syncthreads();
    const int i = threadIdx.x;
    if (threadIdx.y != 0 || i >= 4) return;
    double t = (red[0][i] + red[1][i]) + (red[2][i] + red[3][i]);
    if (blockDim.y == 2) t += (red[4][i] + red[5][i]) + (red[6][i] + red[7][i]);
    // partial sums [row of blocks][column of nodes' blocks][4]; the flux, slot 3, is the wall block's
    const int columns = gridDim.x - 1;
    double* out = scratch + (long long)blockIdx.y * columns * 4 + i;
    if (wall) {
        if (i == 3) *out = t;
    } else if (i < 3 || blockIdx.x > 0) {
        out[blockIdx.x * 4] = t;
    }
}

// Sums the partials in a fixed order (one block of 512 threads, four sums side
// by side): out[0..3] = sum f_l, sum enthalpy, nodes + sum delta_rho, sum
// left-wall flux.
__global__ void diag_finalize(const double* __restrict__ scratch, int nblocks, double nodes, double* __restrict__ out);

}  // namespace lbmk
