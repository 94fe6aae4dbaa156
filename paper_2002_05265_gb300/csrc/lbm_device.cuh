// Device code of the D2Q9 stream-and-collide kernels: storage conversions, the per-node
// collision of every model of App. B written in non-equilibrium form, the per-segment pull
// step shared by all stepping kernels, and the single-lattice and multi-lattice step kernels.
//
// Layout in HBM (one lattice): nine SoA planes g_i[y][x], row pitch `pitch` elements (rows
// 32-byte aligned or better), plane = ny * pitch elements.  Stored values are shifted
// populations g_i = f_i - s_i in the storage type, where the shift s_i = f^eq_i(rho0, u_ref)
// is the extended equilibrium at a reference state; with u_ref = 0 (the default) it is
// s_i = w_i rho0.  Two such buffers alternate: a step reads buffer A and writes buffer B.
//
// Buffer semantics: A_i(z) holds the post-collision population f*_i(z, t-1) emitted by node z,
// so node x gathers its pre-collision populations as f_i(x, t) = A_i(x - xi_i) (pull form of
// Eq. StreamCollide), collides them, and writes f*_i(x, t) to B_i(x).
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace lbm {

enum Model { BGK = 0, RM = 1, HM = 2, CM = 3, CHM = 4, CUM = 5, PR = 6, RR = 7 };

// D2Q9 velocities in the library's index order.
__host__ __device__ constexpr int ex_of(int i) {
    return (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0);
}
__host__ __device__ constexpr int ey_of(int i) {
    return (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0);
}
// D2Q9 weights w_i = W(ex) W(ey), W(0) = 2/3, W(+-1) = 1/6.
__host__ __device__ constexpr double weight_of(int i) {
    return (i == 0) ? 4.0 / 9.0 : ((i <= 4) ? 1.0 / 9.0 : 1.0 / 36.0);
}
// One-dimensional factor of the extended equilibrium (Eq. extendedFeq, product form):
// phi_0(u) = 2/3 - u^2, phi_+-1(u) = (u^2 +- u + 1/3) / 2.
__host__ __device__ inline double phi1d(int s, double u) {
    return s == 0 ? 2.0 / 3.0 - u * u : 0.5 * (u * u + s * u + 1.0 / 3.0);
}
// Shift s_i = rho0 phi_ex(urx) phi_ey(ury) (= w_i rho0 when u_ref = 0).
__host__ __device__ inline double shift_of(int i, double rho0, double urx, double ury) {
    return rho0 * phi1d(ex_of(i), urx) * phi1d(ey_of(i), ury);
}

// Collision constants, computed once on the host in both precisions (kernels then do no
// FP64 set-up work, which GB300's narrow FP64 pipe would make costly):
//  [0-5]   w_nu, w3, w4, rho0, urx, ury
//  [6-11]  Px0, Px+, Px-, Py0, Py+, Py- (shift factors phi_s(u_ref))
//  [12-13] urx^2 + cs^2, ury^2 + cs^2
//  [14-17] ka, kb, kappa, dkappa/dw_nu -- ka, kb the cumulant model's coefficients
//          cs^2 (c4 - kappa), c4 - kappa^2 (c4 = 1 - w4; kappa = 1 - w_nu, 1 or 0 for the
//          post-collision, pre-collision or equilibrium rebuild of K~22, field `kread`)
//  [18-25] combinations the collision uses: -rho0, w - w3, 2 (w3 - w4), w - 2 w3 + w4,
//          cs^2 (w - w4), w3 - 1, w4 - 1, cs^2 (w - 1); [26-29] -kb, -w, -w3, -w4
constexpr int kNumConsts = 30;

struct StepArgs {
    int nx, ny;          // lattice size
    int pitch;           // row pitch in elements
    int nseg;            // vector segments per row = ceil(nx / VEC)
    long long plane;     // elements per population plane
    double w_nu, w3, w4; // relaxation frequencies of orders 2, 3, 4
    double rho0;         // shift reference density
    double urx, ury;     // shift reference velocity
    int kread;           // cumulant rebuild: 0 post-collision, 1 pre-collision, 2 equilibrium
    double cd[kNumConsts];   // the constants above, FP64 (filled by fill_consts)
    float cf[kNumConsts];    // the same, rounded to FP32
};

// Second-order central moments of the cumulant model's rebuild of K~22, as a multiple kappa
// of the non-equilibrium ones n: post-collision (1 - w_nu) n, pre-collision n, equilibrium 0.
__host__ __device__ inline double cumulant_kappa(int kread, double w_nu) {
    return kread == 1 ? 1.0 : (kread == 2 ? 0.0 : 1.0 - w_nu);
}

// Fills the constant tables of a StepArgs from its rates, rho0 and shift velocity.
__host__ __device__ inline void fill_consts(StepArgs& a) {
    const double kap = cumulant_kappa(a.kread, a.w_nu), c4 = 1.0 - a.w4;
    const double v[kNumConsts] = {a.w_nu, a.w3, a.w4, a.rho0, a.urx, a.ury,
                                  phi1d(0, a.urx), phi1d(1, a.urx), phi1d(-1, a.urx),
                                  phi1d(0, a.ury), phi1d(1, a.ury), phi1d(-1, a.ury),
                                  a.urx * a.urx + 1.0 / 3.0, a.ury * a.ury + 1.0 / 3.0,
                                  (c4 - kap) / 3.0, c4 - kap * kap, kap, a.kread == 0 ? -1.0 : 0.0,
                                  -a.rho0, a.w_nu - a.w3, 2.0 * (a.w3 - a.w4), a.w_nu - 2.0 * a.w3 + a.w4,
                                  (a.w_nu - a.w4) / 3.0, a.w3 - 1.0, a.w4 - 1.0, (a.w_nu - 1.0) / 3.0,
                                  -(c4 - kap * kap), -a.w_nu, -a.w3, -a.w4};
    for (int k = 0; k < kNumConsts; ++k) {
        a.cd[k] = v[k];
        a.cf[k] = (float)v[k];
    }
    // in FP32 the combinations are those of the rounded rates
    const float w = a.cf[0], w3 = a.cf[1], w4 = a.cf[2];
    a.cf[19] = w - w3;
    a.cf[20] = 2.0f * (w3 - w4);
    const float w2 = w - 2.0f * w3;
    a.cf[21] = w2 + w4;
    const float d = w - w4;
    a.cf[22] = (float)(1.0 / 3.0) * d;
    a.cf[23] = w3 - 1.0f;
    a.cf[24] = w4 - 1.0f;
}

// ---------------------------------------------------------------------------------------
// Element conversions between the storage type S and the collision type T.
template <typename S> struct Conv;
template <> struct Conv<double> {
    using T = double;
    __device__ static __forceinline__ T to_T(double s) { return s; }
    __device__ static __forceinline__ double from_T(T v) { return v; }
    __device__ static __forceinline__ double to_double(double s) { return s; }
    __device__ static __forceinline__ double from_double(double d) { return d; }
};
template <> struct Conv<float> {
    using T = float;
    __device__ static __forceinline__ T to_T(float s) { return s; }
    __device__ static __forceinline__ float from_T(T v) { return v; }
    __device__ static __forceinline__ double to_double(float s) { return (double)s; }
    __device__ static __forceinline__ float from_double(double d) { return __double2float_rn(d); }
};
template <> struct Conv<__half> {
    using T = float;
    __device__ static __forceinline__ T to_T(__half s) { return __half2float(s); }
    __device__ static __forceinline__ __half from_T(T v) { return __float2half_rn(v); }
    __device__ static __forceinline__ double to_double(__half s) { return (double)__half2float(s); }
    __device__ static __forceinline__ __half from_double(double d) { return __double2half(d); }
};
template <> struct Conv<__nv_bfloat16> {
    using T = float;
    __device__ static __forceinline__ T to_T(__nv_bfloat16 s) { return __bfloat162float(s); }
    __device__ static __forceinline__ __nv_bfloat16 from_T(T v) { return __float2bfloat16_rn(v); }
    __device__ static __forceinline__ double to_double(__nv_bfloat16 s) { return (double)__bfloat162float(s); }
    __device__ static __forceinline__ __nv_bfloat16 from_double(double d) { return __double2bfloat16(d); }
};

// Default vector width: VEC consecutive x-nodes of one row move as one access of
// VEC * sizeof(S) bytes: 16 bytes for FP64 and FP32; for the 16-bit types LBM_HALF_VEC
// nodes (8 = 16-byte accesses, 4 = 8-byte accesses and about half the registers).
#ifndef LBM_HALF_VEC
#define LBM_HALF_VEC 8
#endif
template <typename S> struct DefaultVec {
    static constexpr int value = (sizeof(S) == 2) ? LBM_HALF_VEC : 16 / (int)sizeof(S);
};

// Nodes per thread of the register-staged step kernels: the default, but one for FP64, where a
// scheduler takes 64 clocks for an instruction of one warp (measured, whatever lanes are active): what
// counts there is that every scheduler has one.  With CTAs to match (spread_block) a step of 128 x 128
// BGK takes 4.0 us instead of 11.0, 67 x 37 CHM 4.3 us instead of 16.4.
template <typename S> struct StepVec {
    static constexpr int value = sizeof(S) == 8 ? 1 : DefaultVec<S>::value;
};

template <int BYTES> struct Raw;
template <> struct Raw<4> { using type = uint32_t; };
template <> struct Raw<8> { using type = uint2; };
template <> struct Raw<16> { using type = uint4; };

// aligned vector load / store of VEC elements (VEC * sizeof(S) in {4, 8, 16} bytes)
template <typename S, int VEC>
__device__ __forceinline__ void vload(const S* p, typename Conv<S>::T (&v)[VEC]) {
    using R = typename Raw<VEC * (int)sizeof(S)>::type;
    const R r = *reinterpret_cast<const R*>(p);
    S e[VEC];
    memcpy(e, &r, sizeof(R));
#pragma unroll
    for (int j = 0; j < VEC; ++j) v[j] = Conv<S>::to_T(e[j]);
}
// pairs of floats rounded to a packed pair of 16-bit values in one conversion
__device__ __forceinline__ uint32_t pack2(__half, float a, float b) {
    const __half2 h = __floats2half2_rn(a, b);
    uint32_t u;
    memcpy(&u, &h, 4);
    return u;
}
__device__ __forceinline__ uint32_t pack2(__nv_bfloat16, float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    uint32_t u;
    memcpy(&u, &h, 4);
    return u;
}
template <typename S, int VEC>
__device__ __forceinline__ void vstore(S* p, const typename Conv<S>::T (&v)[VEC]) {
    using R = typename Raw<VEC * (int)sizeof(S)>::type;
    R r;
    if constexpr (sizeof(S) == 2) {
        uint32_t w[VEC / 2];
#pragma unroll
        for (int k = 0; k < VEC / 2; ++k) w[k] = pack2(S(), v[2 * k], v[2 * k + 1]);
        memcpy(&r, w, sizeof(R));
    } else {
        S e[VEC];
#pragma unroll
        for (int j = 0; j < VEC; ++j) e[j] = Conv<S>::from_T(v[j]);
        memcpy(&r, e, sizeof(R));
    }
    *reinterpret_cast<R*>(p) = r;
}

// ---------------------------------------------------------------------------------------
// Arithmetic of the collision, written with explicit fused multiply-adds: every kernel family
// then rounds alike, whatever the compiler would contract in its own context, and a pair of
// FP32 nodes can be collided by Blackwell's two-wide FP32 instructions (F2: one instruction for
// both nodes; each half rounds as the scalar instruction does).  The two-wide instructions have
// the FLOP rate of the scalar ones (measured 73.6 against 73.7 TFLOP/s) from half the issue slots.
struct F2 {
    unsigned long long v;
};
template <typename P> struct PairOf {
    static constexpr bool value = false;
};
template <> struct PairOf<F2> {
    static constexpr bool value = true;
};
__device__ __forceinline__ F2 f2_make(float lo, float hi) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_split(F2 a, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v));
}
__device__ __forceinline__ float f2_lo(F2 a) {
    float lo, hi;
    f2_split(a, lo, hi);
    return lo;
}
__device__ __forceinline__ float f2_hi(F2 a) {
    float lo, hi;
    f2_split(a, lo, hi);
    return hi;
}

// a literal in the type one instruction works on
template <typename P> __device__ __forceinline__ P lit(double c) { return P(c); }
template <> __device__ __forceinline__ F2 lit<F2>(double c) { return f2_make((float)c, (float)c); }

__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma3(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double fma3(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ F2 fma3(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ F2 add(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 mul(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
// a - b: there is no two-wide subtraction; a + (-1) b rounds the same (adding the negated halves
// instead lets the assembler fuse a product into the sum, which does not)
__device__ __forceinline__ F2 sub(F2 a, F2 b) { return fma3(b, f2_make(-1.0f, -1.0f), a); }

// -s for s = a + b, from -a and b: an operand sign for one node, an instruction for two
__device__ __forceinline__ float negative(float s, float, float) { return -s; }
__device__ __forceinline__ F2 negative(F2, F2 na, F2 b) { return sub(na, b); }

// 1/x.  FP32: the hardware approximation (rcp.approx) refined by one Newton-Raphson step,
// r' = r + r (1 - x r), two FMAs; within an ulp of the rounded quotient and free of any
// data-dependent branch, so a lattice that has blown up (non-finite populations) steps as fast
// as a healthy one.  FP64: the correctly rounded reciprocal intrinsic.
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float recip(float x) {
    const float r = rcp_approx(x);
    return fmaf(r, fmaf(-x, r, 1.0f), r);
}
__device__ __forceinline__ double recip(double x) { return __drcp_rn(x); }
// 1/x from x and -x, bit for bit recip(x) in both halves
__device__ __forceinline__ float recip2(float x, float nx) {
    const float r = rcp_approx(x);
    return __fmaf_rn(r, __fmaf_rn(nx, r, 1.0f), r);
}
__device__ __forceinline__ F2 recip2(F2 x, F2 nx) {
    const F2 r = f2_make(rcp_approx(f2_lo(x)), rcp_approx(f2_hi(x)));
    return fma3(r, fma3(nx, r, f2_make(1.0f, 1.0f)), r);
}

// Per-launch constants of the collision in the type it works on (the entries of the constant
// table; see kNumConsts).
template <typename T> struct Consts {
    T w, w3, w4, rho0, urx, ury;
    T Xr, Yr;                // mu_2(u_ref) = u_ref^2 + c_s^2 per axis
    T ka, kb, nkb;           // cumulant coefficients
    T nrho0;                 // -rho0
    T ww3, rr, qq;           // w - w3, 2 (w3 - w4), w - 2 w3 + w4
    T sw4;                   // c_s^2 (w - w4)
    T nc3, nc4, sw1;         // w3 - 1, w4 - 1, c_s^2 (w - 1)
    T nw, nw3, nw4;          // -w, -w3, -w4
};
template <typename T> __device__ __forceinline__ const T* const_table(const StepArgs& a);
template <> __device__ __forceinline__ const float* const_table<float>(const StepArgs& a) { return a.cf; }
template <> __device__ __forceinline__ const double* const_table<double>(const StepArgs& a) { return a.cd; }

template <typename T>
__device__ __forceinline__ Consts<T> make_consts_table(const T* t) {
    Consts<T> c;
    c.w = t[0]; c.w3 = t[1]; c.w4 = t[2]; c.rho0 = t[3]; c.urx = t[4]; c.ury = t[5];
    c.Xr = t[12]; c.Yr = t[13];
    c.ka = t[14]; c.kb = t[15];
    // (the entries 18, 26-29, as operand signs)
    c.nkb = -c.kb; c.nrho0 = -c.rho0;
    c.nw = -c.w; c.nw3 = -c.w3; c.nw4 = -c.w4;
    c.ww3 = t[19]; c.rr = t[20]; c.qq = t[21];
    c.sw4 = t[22];
    c.nc3 = t[23]; c.nc4 = t[24]; c.sw1 = t[25];
    return c;
}
template <typename T>
__device__ __forceinline__ Consts<T> make_consts(const StepArgs& a) {
    return make_consts_table<T>(const_table<T>(a));
}

// ---------------------------------------------------------------------------------------
// Per-node collision (App. B) on shifted populations g_i = f_i - s_i.  P is the type one
// instruction works on: double, float, or F2 (two FP32 nodes).
//
// Every model of App. B relaxes the moments of f towards those of f^eq with the same rho
// and u, through a transform that is linear in f for the node's u, and keeps the conserved
// moments (order 0 and 1).  So each model is f* = f - T(u)^-1 D with D = n - n*: n the
// non-equilibrium moments M(f) - M^eq(rho, u), n* their post-collision values, and D's
// conserved components exactly zero.  The kernels compute that directly on the stored
// g = f - s: the nine raw moments of g by x-then-y partial sums; n = M(g) - (M^eq - M(s)),
// where M^eq_pq = rho mu_p(u_x) mu_q(u_y) and M_pq(s) = rho0 mu_p(ur_x) mu_q(ur_y) are the
// product-form moments of Eq. extendedFeq (mu_0 = 1, mu_1 = u, mu_2 = u^2 + c_s^2), their
// difference written without cancellation; the model's relaxation of n (raw, Hermite,
// central, central-Hermite, cumulant, recursive); and g* = g - (back-transform of D, Eq.
// Q9postCollVDF_RM with D_00 = D_10 = D_01 = 0).  BGK is the raw-moment relaxation with one
// rate for every order (exact for the D2Q9 moment basis).  Every intermediate is small, which
// is what makes FP32 arithmetic on FP16-stored populations accurate, and the stored mass and
// momentum change only by the rounding of D.  rho, ux, uy of the pre-collision state are
// returned for diagnostics.  SHIFT = false is the default shift s = w rho0 (u_ref = 0), which
// keeps the shift constants out of the arithmetic.
//
// With a21 = 2 ux n11 + uy n20, a12 = 2 uy n11 + ux n02, R = 2 (ux n12 + uy n21) and
// Q = ux a12 + uy a21 = ux^2 n02 + uy^2 n20 + 4 ux uy n11 the models are
//   RM, BGK (Eq. RMcoll)       D21 = w3 n21, D12 = w3 n12, D22 = w4 n22;
//   HM, PR (Hermite moments: A_2 = n_2, A_21 = n_21, A_12 = n_12, A_22 = n_22 - c_s^2 (n_20 + n_02);
//      Eq. HM2RM_Q9)           D22 = w4 A_22 + c_s^2 (D20 + D02); PR: w3 = w4 = 1;
//   RR (Eqs. HMColl_Q9, RRformulas_D2Q9: third- and fourth-order A^neq from the recursion, a21, a12
//      and Q; A* = A^eq + (1 - w) A^neq_rec)
//                              D21 = n21 - (1 - w3) a21, ..., D22 = A_22 - (1 - w4) Q + c_s^2 (D20 + D02);
//   CM, CHM, K: central moments k = S(-u) n of f^neq (binomial shift, first-order parts vanish),
//      relaxed by order (d = rates . k), shifted back D = S(u) d; folded into one expression in n
//      (k21 = n21 - a21, k12 = n12 - a12, k22 = n22 - R + Q)
//                              D21 = w3 n21 + (w - w3) a21,   D12 = w3 n12 + (w - w3) a12,
//                              D22 = w4 n22 + (w3 - w4) R + (w - 2 w3 + w4) Q + (d22 - w4 k22).
//      CHM: the central Hermite A~_22 = K~_22 - c_s^2 (K~_20 + K~_02) relaxes with w4, the second
//      order with w (Eqs. CHpoly, CHMcoll): d22 = w4 k22 + c_s^2 (w - w4) (n20 + n02).
//      K: the cumulant C22 = K22 - (K20 K02 + 2 K11^2)/rho relaxes to 0 and K22* is rebuilt with
//      second-order central moments kappa n (deviations from the equilibrium central moments
//      rho c_s^2, 0, rho c_s^4): kappa = 1 - w for the post-collision values (the paper's K), 1 or 0
//      for the pre-collision / equilibrium readings.  With S = n20 + n02, P = n20 n02 + 2 n11^2 and
//      c4 = 1 - w4: C22 = k22 - c_s^2 S - P / rho, K22* = c4 C22 + c_s^2 kappa S + kappa^2 P / rho, so
//      d22 = k22 - K22* = w4 k22 + ka S + kb P / rho, ka = c_s^2 (c4 - kappa), kb = c4 - kappa^2.
//
// FP64: the FP64 pipe bounds the kernels, so the expressions share what they can and leave no
// negation over: j and 1/rho are formed negated, E = M(s) - M^eq enters n by additions.
// Operations of one node, the reciprocal's aside: BGK 58 .. K 83 (SHIFT 10 more); against the
// expressions of collide_f32 a step of 128 x 128 BGK takes 11.0 us instead of 13.7, 67 x 37 CHM
// 16.4 us instead of 18.5.
template <int MODEL, bool SHIFT>
__device__ __forceinline__ void collide_f64(const double (&g)[9], double (&o)[9], const Consts<double>& c,
                                            double& rho_out, double& ux_out, double& uy_out) {
    using P = double;
    const P cs2 = P(1.0 / 3.0), ncs2 = P(-1.0 / 3.0);
    const P w = c.w;
    // row sums of the velocity set (xi_y = +1, 0, -1): weights 1 (a), xi_x (d), xi_x^2 (s)
    const P s56 = add(g[5], g[6]), d56 = sub(g[5], g[6]);
    const P s78 = add(g[8], g[7]), d87 = sub(g[8], g[7]);
    const P s13 = add(g[1], g[3]), d31 = sub(g[3], g[1]);
    const P a0p = add(g[2], s56), a0m = add(g[4], s78), a0z = add(g[0], s13);
    // raw moments of g (App. B, M_pq = sum xi_x^p xi_y^q g); sum s = rho0, sum xi s = rho0 u_ref
    const P m02 = add(a0p, a0m), njy = sub(a0m, a0p);
    const P drho = add(m02, a0z);
    const P m22 = add(s56, s78), m21 = sub(s56, s78);
    const P m12 = add(d56, d87), m11 = sub(d56, d87);
    const P m20 = add(s13, m22), njx = sub(d31, m12);
    const P rho = add(drho, c.rho0);
    const P nir = -recip(rho);
    P ux, uy, dx, dy;
    if (SHIFT) {
        // u - u_ref = (j - drho u_ref) / rho, j the momentum of g
        dx = mul(fma3(c.urx, drho, njx), nir);
        dy = mul(fma3(c.ury, drho, njy), nir);
        ux = add(dx, c.urx);
        uy = add(dy, c.ury);
    } else {
        ux = mul(njx, nir);
        uy = mul(njy, nir);
    }
    rho_out = rho; ux_out = ux; uy_out = uy;

    // non-equilibrium raw moments n = M(g) + E, E_pq = M_pq(s) - M^eq_pq (Eq. extendedFeq)
    const P e = mul(ncs2, drho);
    P n20, n02, n11, n21, n12, n22;
    if (SHIFT) {
        // E_20 = -(j_x u_x + rho0 ur_x (u_x - ur_x) + cs2 drho), E_22 = E_20 Y + Xr (E_02 + drho Y)
        const P qx = mul(dx, c.nrho0), qy = mul(dy, c.nrho0);
        const P Y = fma3(uy, uy, cs2);
        const P eX = fma3(njx, ux, fma3(c.urx, qx, e)), eY = fma3(njy, uy, fma3(c.ury, qy, e));
        n20 = add(m20, eX);
        n02 = add(m02, eY);
        n11 = fma3(njx, uy, fma3(c.urx, qy, m11));
        n21 = fma3(uy, eX, fma3(c.Xr, qy, m21));
        n12 = fma3(ux, eY, fma3(c.Yr, qx, m12));
        n22 = fma3(Y, fma3(c.Xr, drho, eX), fma3(c.Xr, eY, m22));
    } else {
        // E_20 = -(j_x u_x + cs2 drho), E_21 = -X j_y, E_22 = -(Y j_x u_x + cs2 (j_y u_y + cs2 drho))
        const P X = fma3(ux, ux, cs2), Y = fma3(uy, uy, cs2);
        const P pX = mul(njx, ux), eY = fma3(njy, uy, e);
        n20 = add(m20, add(pX, e));
        n02 = add(m02, eY);
        n11 = fma3(njx, uy, m11);
        n21 = fma3(X, njy, m21);
        n12 = fma3(Y, njx, m12);
        n22 = fma3(Y, pX, fma3(cs2, eY, m22));
    }
    // D = n - n* (the moments the collision removes), per model; BGK's one rate is left to the
    // coefficients of the back-transform (D = n there)
    P D20 = n20, D02 = n02, D11 = n11, D21 = n21, D12 = n12, D22 = n22;
    if (MODEL != BGK) {
        D20 = mul(w, n20); D02 = mul(w, n02); D11 = mul(w, n11);
    }
    if (MODEL == BGK) {
    } else if (MODEL == RM) {
        // Eq. RMcoll
        D21 = mul(c.w3, n21); D12 = mul(c.w3, n12); D22 = mul(c.w4, n22);
    } else if (MODEL == HM) {
        // Hermite moments: A_2 = n_2, A_21 = n_21, A_12 = n_12 (conserved parts vanish),
        // A_22 = n_22 - c_s^2 (n_20 + n_02); relaxed, back with Eq. HM2RM_Q9:
        // D22 = w4 A_22 + c_s^2 (D20 + D02)
        D21 = mul(c.w3, n21); D12 = mul(c.w3, n12);
        D22 = fma3(c.sw4, add(n20, n02), mul(c.w4, n22));
    } else if (MODEL == PR) {
        // HM with omega3 = omega4 = 1
        D22 = fma3(c.sw1, add(n20, n02), n22);
    } else {
        // a21 = 2 ux n11 + uy n20, a12 = 2 uy n11 + ux n02 and
        // Q = ux a12 + uy a21 = ux^2 n02 + uy^2 n20 + 4 ux uy n11
        const P t = add(n11, n11);
        const P a21 = fma3(ux, t, mul(uy, n20)), a12 = fma3(uy, t, mul(ux, n02));
        const P Q = fma3(ux, a12, mul(uy, a21));
        if (MODEL == RR) {
            // Eqs. HMColl_Q9, RRformulas_D2Q9: third/fourth-order A^neq from the recursion
            // (a21, a12, Q), A* = A^eq + (1 - omega) A^neq_rec, so D = A^neq - (1 - omega) A^neq_rec
            D21 = fma3(c.nc3, a21, n21);
            D12 = fma3(c.nc3, a12, n12);
            D22 = fma3(c.sw1, add(n20, n02), fma3(c.nc4, Q, n22));
        } else {
            // central moments k = S(-u) n of f^neq (binomial shift, first-order parts vanish),
            // relaxed by order (d = rates . k), shifted back D = S(u) d.  The three linear steps
            // are folded into one expression in n: with R = 2 (ux n12 + uy n21) one has
            // k21 = n21 - a21, k12 = n12 - a12, k22 = n22 - R + Q, and
            //   D21 = w3 n21 + (w - w3) a21,   D12 = w3 n12 + (w - w3) a12,
            //   D22 = w4 n22 + (w3 - w4) R + (w - 2 w3 + w4) Q + (model terms),
            // the model terms being d22 - w4 k22 (zero for CM).
            D21 = fma3(c.ww3, a21, mul(c.w3, n21));
            D12 = fma3(c.ww3, a12, mul(c.w3, n12));
            const P R = fma3(ux, n12, mul(uy, n21));
            D22 = fma3(c.qq, Q, fma3(c.rr, R, mul(c.w4, n22)));
            if (MODEL == CHM) {
                // central Hermite: A~_22 = K~_22 - c_s^2 (K~_20 + K~_02) relaxed with w4, the
                // second order with w (Eqs. CHpoly, CHMcoll): d22 = w4 A~_22 + c_s^2 (d20 + d02)
                // = w4 k22 + c_s^2 (w - w4) (n20 + n02)
                D22 = fma3(c.sw4, add(n20, n02), D22);
            } else if (MODEL != CM) {
                // cumulants: C22 = K22 - (K20 K02 + 2 K11^2)/rho relaxes to 0 and K22* is rebuilt
                // with second-order central moments kappa n (written for deviations from the
                // equilibrium central moments rho c_s^2, 0, rho c_s^4): kappa = 1 - w for the
                // post-collision values (the paper's K), 1 or 0 for the pre-collision / equilibrium
                // readings.  With S = n20 + n02, P = n20 n02 + 2 n11^2 and c4 = 1 - w4:
                // C22 = k22 - c_s^2 S - P / rho, K22* = c4 C22 + c_s^2 kappa S + kappa^2 P / rho, so
                // d22 = k22 - K22* = w4 k22 + ka S + kb P / rho with the per-launch constants
                // ka = c_s^2 (c4 - kappa), kb = c4 - kappa^2
                const P PP = fma3(n20, n02, mul(t, n11));
                D22 = fma3(mul(c.nkb, nir), PP, fma3(c.ka, add(n20, n02), D22));
            }
        }
    }

    // g* = g - (Eq. Q9postCollVDF_RM applied to D, with D_00 = D_10 = D_01 = 0)
    const P nh = MODEL == BGK ? mul(P(-0.5), w) : P(-0.5);
    const P nq = MODEL == BGK ? mul(P(-0.25), w) : P(-0.25);
    const P A = sub(D20, D22), B = sub(D02, D22);
    o[0] = MODEL == BGK ? fma3(w, add(A, D02), g[0]) : add(g[0], add(A, D02));
    o[1] = fma3(nh, sub(A, D12), g[1]);
    o[3] = fma3(nh, add(A, D12), g[3]);
    o[2] = fma3(nh, sub(B, D21), g[2]);
    o[4] = fma3(nh, add(B, D21), g[4]);
    const P E = add(D22, D11), F = sub(D22, D11), U = add(D21, D12), V = sub(D21, D12);
    o[5] = fma3(nq, add(E, U), g[5]);
    o[7] = fma3(nq, sub(E, U), g[7]);
    o[6] = fma3(nq, add(F, V), g[6]);
    o[8] = fma3(nq, sub(F, V), g[8]);
}


// FP32 (one node: float, two: F2).  The operations, their order and what is fused are fixed here,
// so that every kernel form and both widths give the same bits; 16-bit storage needs that most: one
// population rounded the other way spreads until, after some hundred steps, two BF16 runs differ by
// as much as either does from FP64.  Products that a sum takes up fused are not formed again.
// Operations of one node: BGK 80, K 103 (the expressions of collide_f64 would be 60 and 85, the
// reciprocal's two included, and the time-fused kernel 8-11 % faster, 1042 us against 1157 a step of
// 16384^2 K; they round differently).
template <int MODEL, typename P, bool SHIFT>
__device__ __forceinline__ void collide_f32(const P (&g)[9], P (&o)[9], const Consts<P>& c, P& rho_out, P& ux_out,
                                            P& uy_out) {
    constexpr bool ONE_BY_ONE = MODEL == BGK || MODEL == RM || MODEL == HM;   // D21 = w3 n21, D12 = w3 n12
    const P cs2 = lit<P>(1.0 / 3.0), ncs2 = lit<P>(-1.0 / 3.0);
    const P w = c.w, nw = c.nw;
    const P w3 = MODEL == BGK ? c.w : c.w3, nw3 = MODEL == BGK ? c.nw : c.nw3;
    const P w4 = MODEL == BGK ? c.w : c.w4, nw4 = MODEL == BGK ? c.nw : c.nw4;
    const P a0p = add(add(g[6], g[2]), g[5]), a1p = sub(g[5], g[6]), a2p = add(g[5], g[6]);
    const P a0z = add(add(g[3], g[0]), g[1]), a1z = sub(g[1], g[3]), a2z = add(g[1], g[3]);
    const P a0m = add(add(g[7], g[4]), g[8]), a1m = sub(g[8], g[7]), a2m = add(g[8], g[7]);
    const P drho = add(add(a0p, a0z), a0m);
    P jx = add(add(a1p, a1z), a1m), jy = sub(a0p, a0m);
    const P m20 = add(add(a2p, a2z), a2m), m02 = add(a0p, a0m), m11 = sub(a1p, a1m);
    const P m21 = sub(a2p, a2m), m12 = add(a1p, a1m), m22 = add(a2p, a2m);
    const P rho = add(drho, c.rho0), nrho = negative(rho, c.nrho0, drho);
    if (SHIFT) {
        jx = fma3(c.rho0, c.urx, jx);
        jy = fma3(c.rho0, c.ury, jy);
    }
    const P irho = recip2(rho, nrho);
    const P ux = mul(jx, irho), uy = mul(jy, irho);
    const P uxx = mul(ux, ux), uyy = mul(uy, uy), uxy = mul(ux, uy);
    rho_out = rho; ux_out = ux; uy_out = uy;

    P n20, n02, n11, n21, n12, n22;
    if (SHIFT) {
        constexpr bool SQUARES = MODEL == RR || MODEL == CM || MODEL == CHM || MODEL == CUM;   // uxx, uyy serve twice
        const P X = SQUARES ? add(uxx, cs2) : fma3(ux, ux, cs2), Y = SQUARES ? add(uyy, cs2) : fma3(uy, uy, cs2);
        const P dx = sub(ux, c.urx), dy = sub(uy, c.ury);
        const P dX = mul(dx, add(ux, c.urx)), dY = mul(dy, add(uy, c.ury));
        n20 = sub(m20, fma3(drho, X, mul(c.rho0, dX)));
        n02 = sub(m02, fma3(drho, Y, mul(c.rho0, dY)));
        n11 = sub(m11, fma3(drho, uxy, mul(c.rho0, fma3(dx, uy, mul(c.urx, dy)))));
        n21 = sub(m21, fma3(drho, mul(X, uy), mul(c.rho0, fma3(c.Xr, dy, mul(dX, uy)))));
        n12 = sub(m12, fma3(drho, mul(ux, Y), mul(c.rho0, fma3(dx, Y, mul(c.urx, dY)))));
        n22 = sub(m22, fma3(drho, mul(X, Y), mul(c.rho0, fma3(dX, Y, mul(c.Xr, dY)))));
    } else {
        const P X = add(uxx, cs2), Y = add(uyy, cs2);
        n20 = sub(m20, fma3(cs2, drho, mul(rho, uxx)));
        n02 = sub(m02, fma3(cs2, drho, mul(rho, uyy)));
        n11 = fma3(nrho, uxy, m11);
        n21 = fma3(mul(nrho, X), uy, m21);
        n12 = fma3(mul(nrho, ux), Y, m12);
        n22 = sub(m22, fma3(drho, mul(X, Y), mul(c.rho0, fma3(cs2, uyy, mul(uxx, Y)))));
    }

    const P D02 = mul(w, n02), DS = fma3(w, n20, D02);   // DS = D20 + D02
    P D21, D12, D22;
    if (MODEL == BGK || MODEL == RM) {
        D21 = mul(w3, n21); D22 = mul(w4, n22);
    } else if (MODEL == HM || MODEL == PR) {
        const P a22 = fma3(ncs2, add(n20, n02), n22);
        if (MODEL == HM) {
            D21 = mul(w3, n21);
            D22 = fma3(cs2, DS, mul(w4, a22));
        } else {
            D21 = n21; D12 = n12;
            D22 = fma3(cs2, DS, a22);
        }
    } else {
        const P t = add(n11, n11);
        const P a21 = SHIFT ? fma3(uy, n20, mul(ux, t)) : fma3(ux, t, mul(uy, n20));
        const P a12 = SHIFT ? fma3(ux, n02, mul(uy, t)) : fma3(uy, t, mul(ux, n02));
        if (MODEL == RR) {
            const P a22 = fma3(uxy, add(t, t), fma3(uyy, n20, mul(uxx, n02)));
            D21 = fma3(c.nc3, a21, n21);
            D12 = fma3(c.nc3, a12, n12);
            D22 = fma3(cs2, DS, fma3(c.nc4, a22, fma3(ncs2, add(n20, n02), n22)));
        } else {
            const P R = fma3(ux, n12, mul(uy, n21));
            const P Q = fma3(uxy, add(t, t), fma3(uxx, n02, mul(uyy, n20)));
            D21 = fma3(w3, n21, mul(c.ww3, a21));
            D12 = fma3(w3, n12, mul(c.ww3, a12));
            D22 = fma3(c.qq, Q, fma3(w4, n22, mul(c.rr, R)));
            if (MODEL == CHM) {
                D22 = fma3(c.sw4, add(n20, n02), D22);
            } else if (MODEL != CM) {
                const P PP = fma3(n20, n02, mul(t, n11));
                D22 = add(D22, fma3(c.ka, add(n20, n02), mul(mul(c.kb, irho), PP)));
            }
        }
    }

    const P h = lit<P>(0.5), nh = lit<P>(-0.5), nq = lit<P>(-0.25);
    const P nA = fma3(nw, n20, D22), B = sub(D02, D22);   // -(D20 - D22), D02 - D22
    o[0] = add(g[0], (MODEL == BGK || MODEL == RM) ? fma3(nw4, n22, DS) : sub(DS, D22));
    P U, V;   // D21 + D12, D21 - D12
    if (ONE_BY_ONE) {
        o[1] = fma3(h, fma3(w3, n12, nA), g[1]);
        o[3] = fma3(h, fma3(nw3, n12, nA), g[3]);
        o[2] = fma3(nh, fma3(nw3, n21, B), g[2]);
        o[4] = fma3(nh, fma3(w3, n21, B), g[4]);
        U = fma3(w3, n12, D21);
        V = fma3(nw3, n12, D21);
    } else {
        o[1] = fma3(h, add(nA, D12), g[1]);
        o[3] = fma3(h, sub(nA, D12), g[3]);
        o[2] = fma3(nh, sub(B, D21), g[2]);
        o[4] = fma3(nh, add(B, D21), g[4]);
        U = add(D12, D21);
        V = sub(D21, D12);
    }
    const P E = fma3(w, n11, D22), F = fma3(nw, n11, D22);   // D22 +- D11
    o[5] = fma3(nq, add(E, U), g[5]);
    o[7] = fma3(nq, sub(E, U), g[7]);
    o[6] = fma3(nq, add(F, V), g[6]);
    o[8] = fma3(nq, sub(F, V), g[8]);
}

// BGK with the second-order equilibrium of Sec. 2 (EQ = 2, population space) or the partial
// third-order one of Fig. 4 (EQ = 3: Hermite A^eq_22 = 0, M^eq_22 without its rho u_x^2 u_y^2 term),
// u_ref = 0.
template <int EQ, typename T>
__device__ __forceinline__ void collide_truncated(const T (&g)[9], T (&o)[9], const Consts<T>& c, T& rho_out,
                                                  T& ux_out, T& uy_out) {
    const T cs2 = T(1) / T(3), w = c.w;
    const T a0p = (g[6] + g[2]) + g[5], a1p = g[5] - g[6], a2p = g[5] + g[6];
    const T a0z = (g[3] + g[0]) + g[1], a1z = g[1] - g[3], a2z = g[1] + g[3];
    const T a0m = (g[7] + g[4]) + g[8], a1m = g[8] - g[7], a2m = g[8] + g[7];
    const T drho = (a0p + a0z) + a0m, rho = c.rho0 + drho;
    const T jx = (a1p + a1z) + a1m, jy = a0p - a0m;
    const T irho = recip(rho);
    const T ux = jx * irho, uy = jy * irho;
    const T uxx = ux * ux, uyy = uy * uy;
    rho_out = rho; ux_out = ux; uy_out = uy;
    if (EQ == 2) {
        // second-order equilibrium (Sec. 2, Hermite reading), shift s = w rho0 (u_ref = 0):
        // f^eq_i = w_i rho (1 + 3 xi.u + 4.5 (xi.u)^2 - 1.5 u^2); BGK in population space
        const T usq = T(1.5) * (uxx + uyy);
        const T cc = T(1) - w;
        T fn[9], geq[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const T wi = T(weight_of(i));
            const T eu = T(3) * (T(ex_of(i)) * ux + T(ey_of(i)) * uy);
            geq[i] = wi * drho + wi * rho * (eu + T(0.5) * eu * eu - usq);
            fn[i] = g[i] - geq[i];
        }
        // f^neq carries the rounding of the conserved moments, which (1 - omega) would feed
        // back with a factor ~1 at low viscosity: remove it (populations carrying exactly the
        // residual mass and momentum), the map is unchanged
        const T e0 = ((fn[0] + fn[1]) + (fn[2] + fn[3])) + ((fn[4] + fn[5]) + (fn[6] + fn[7])) + fn[8];
        const T hx = T(0.5) * ((fn[1] - fn[3]) + ((fn[5] - fn[7]) + (fn[8] - fn[6])));
        const T hy = T(0.5) * ((fn[2] - fn[4]) + ((fn[5] - fn[7]) + (fn[6] - fn[8])));
        fn[0] -= e0;
        fn[1] -= hx; fn[3] += hx;
        fn[2] -= hy; fn[4] += hy;
#pragma unroll
        for (int i = 0; i < 9; ++i) o[i] = geq[i] + cc * fn[i];
        return;
    }
    const T m20 = (a2p + a2z) + a2m, m02 = a0p + a0m, m11 = a1p - a1m;
    const T m21 = a2p - a2m, m12 = a1p + a1m, m22 = a2p + a2m;
    const T Y = uyy + cs2;
    const T rX = rho * (uxx + cs2);
    const T n20 = m20 - (cs2 * drho + rho * uxx);
    const T n02 = m02 - (cs2 * drho + rho * uyy);
    const T n11 = m11 - rho * (ux * uy);
    const T n21 = m21 - rX * uy;
    const T n12 = m12 - (rho * ux) * Y;
    const T n22 = m22 - (drho * ((uxx + cs2) * Y) + c.rho0 * (uxx * Y + cs2 * uyy)) + rho * (uxx * uyy);
    const T D20 = w * n20, D02 = w * n02, D11 = w * n11, D21 = w * n21, D12 = w * n12, D22 = w * n22;
    const T h = T(0.5), q = T(0.25);
    o[0] = g[0] - (D22 - (D20 + D02));
    o[1] = g[1] - h * ((D20 - D22) - D12);
    o[3] = g[3] - h * ((D20 - D22) + D12);
    o[2] = g[2] - h * ((D02 - D22) - D21);
    o[4] = g[4] - h * ((D02 - D22) + D21);
    o[5] = g[5] - q * ((D22 + D11) + (D12 + D21));
    o[6] = g[6] - q * ((D22 - D11) + (D21 - D12));
    o[7] = g[7] - q * ((D22 + D11) - (D12 + D21));
    o[8] = g[8] - q * ((D22 - D11) + (D12 - D21));
}

template <int MODEL, int EQ, typename P, bool SHIFT>
__device__ __forceinline__ void collide(const P (&g)[9], P (&o)[9], const Consts<P>& c, P& rho, P& ux, P& uy) {
    if constexpr (EQ != 4) collide_truncated<EQ, P>(g, o, c, rho, ux, uy);
    else if constexpr (sizeof(P) == 8 && !PairOf<P>::value) collide_f64<MODEL, SHIFT>(g, o, c, rho, ux, uy);
    else collide_f32<MODEL, P, SHIFT>(g, o, c, rho, ux, uy);
}

// Per-thread FP64 accumulators of the blow-up diagnostics (used by the batched sweep).
struct Diag {
    double pert;      // sum |u - u_ref|^2
    double ke;        // sum |u|^2
    double rho_min;   // min rho
    double nonfinite; // count of nodes with a non-finite rho or u
};

// ---------------------------------------------------------------------------------------
// Gather of the nine planes of one vector segment (VEC consecutive x-nodes of row y) at the
// periodic offsets -SIGN * xi_i: SIGN = +1 gives the populations that node x collides,
// f_i(x) = A_i(x - xi_i) (pull); SIGN = -1 gives lambda_i(x + xi_i) (reverse streaming of the
// adjoint).  All 32 lanes call it together with consecutive segments; loads are aligned
// vectors, the x-shifted element comes from the neighbouring lane by a warp shuffle, or from
// one scalar load at warp and row edges (where the periodic wrap is applied).
template <typename S, int VEC, int SIGN>
__device__ __forceinline__ void gather_pull(const S* __restrict__ src, int nx, int ny, int pitch, long long plane,
                                            int y, int seg, int nseg, int x0, int nvalid, int lane,
                                            typename Conv<S>::T (&f)[9][VEC]) {
    using T = typename Conv<S>::T;
    const int ym = (y == 0) ? ny - 1 : y - 1;
    const int yp = (y == ny - 1) ? 0 : y + 1;
    const bool left_from_lane = (lane > 0) && (seg > 0);
    const bool right_from_lane = (lane < 31) && (seg < nseg - 1);
    const int xl = (x0 == 0) ? nx - 1 : x0 - 1;           // source of an x-offset of -1 at j = 0
    const int xr = (x0 + nvalid >= nx) ? 0 : x0 + VEC;     // source of an x-offset of +1 at j = nvalid-1
    if constexpr (VEC == 1) {   // a node per lane: its nine sources, straight
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int ex = SIGN * ex_of(i), ey = SIGN * ey_of(i);
            const int row = (ey == 1) ? ym : ((ey == -1) ? yp : y), x = (ex == 1) ? xl : ((ex == -1) ? xr : x0);
            f[i][0] = Conv<S>::to_T(src[(long long)i * plane + (long long)row * pitch + x]);
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int ex = SIGN * ex_of(i), ey = SIGN * ey_of(i);
        const int row = (ey == 1) ? ym : ((ey == -1) ? yp : y);
        const S* p = src + (long long)i * plane + (long long)row * pitch;
        T v[VEC];
        vload<S, VEC>(p + x0, v);
        if (ex == 0) {
#pragma unroll
            for (int j = 0; j < VEC; ++j) f[i][j] = v[j];
        } else if (ex == 1) {
            T left = __shfl_up_sync(0xffffffffu, v[VEC - 1], 1);
            if (!left_from_lane) left = Conv<S>::to_T(p[xl]);
            f[i][0] = left;
#pragma unroll
            for (int j = 1; j < VEC; ++j) f[i][j] = v[j - 1];
        } else {
            T right = __shfl_down_sync(0xffffffffu, v[0], 1);
            if (!right_from_lane) right = Conv<S>::to_T(p[xr]);
#pragma unroll
            for (int j = 0; j < VEC - 1; ++j) f[i][j] = (j + 1 < nvalid) ? v[j + 1] : right;
            f[i][VEC - 1] = right;
        }
    }
}

// ---------------------------------------------------------------------------------------
// One pull step of one vector segment (VEC consecutive x-nodes of one row): gather
// (periodic) -> collide -> store.  All 32 lanes of the warp call it together with
// consecutive segment indices s = base + lane (base a multiple of 32); lanes with s >= total
// take part in the shuffles and store nothing.
template <int MODEL, int EQ, typename S, int VEC, bool DIAG, bool SHIFT>
__device__ __forceinline__ void step_segment(const S* __restrict__ src, S* __restrict__ dst, const StepArgs& a,
                                             const Consts<typename Conv<S>::T>& c, unsigned s, unsigned total,
                                             int lane, Diag& dg) {
    using T = typename Conv<S>::T;
    const bool active = s < total;
    const unsigned sc = active ? s : total - 1;
    const int y = (int)(sc / (unsigned)a.nseg);
    const int seg = (int)(sc - (unsigned)y * (unsigned)a.nseg);
    const int x0 = seg * VEC;
    const int nvalid = min(VEC, a.nx - x0);
    T f[9][VEC];
    gather_pull<S, VEC, 1>(src, a.nx, a.ny, a.pitch, a.plane, y, seg, a.nseg, x0, nvalid, lane, f);

    T out[9][VEC];
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
        T gin[9], gout[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) gin[i] = f[i][j];
        T rho, ux, uy;
        collide<MODEL, EQ, T, SHIFT>(gin, gout, c, rho, ux, uy);
#pragma unroll
        for (int i = 0; i < 9; ++i) out[i][j] = gout[i];
        if (DIAG) {
            if (active && j < nvalid) {
                if (isfinite(rho) && isfinite(ux) && isfinite(uy)) {
                    const T wx = ux - c.urx, wy = uy - c.ury;
                    dg.pert += (double)(wx * wx + wy * wy);
                    dg.ke += (double)(ux * ux + uy * uy);
                    dg.rho_min = fmin(dg.rho_min, (double)rho);
                } else {
                    dg.nonfinite += 1.0;
                }
            }
        }
    }
    if (active) {
#pragma unroll
        for (int i = 0; i < 9; ++i) vstore<S, VEC>(dst + (long long)i * a.plane + (long long)y * a.pitch + x0, out[i]);
    }
}

// ---------------------------------------------------------------------------------------
// Single-lattice step: warps walk the lattice with a grid-stride loop (the grid is sized to
// the resident CTAs of the GPU).
template <int MODEL, int EQ, typename S, bool SHIFT>
__global__ void __launch_bounds__(256) step_kernel(const S* __restrict__ src, S* __restrict__ dst, StepArgs a) {
    // programmatic dependent launch, as in the other step kernels
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    using T = typename Conv<S>::T;
    constexpr int VEC = StepVec<S>::value;
    const int lane = threadIdx.x & 31;
    const unsigned total = (unsigned)a.ny * (unsigned)a.nseg;
    const unsigned stride = gridDim.x * blockDim.x;
    const Consts<T> c = make_consts<T>(a);
    Diag dg;
    for (unsigned base = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); base < total; base += stride)
        step_segment<MODEL, EQ, S, VEC, false, SHIFT>(src, dst, a, c, base + lane, total, lane, dg);
}

// ---------------------------------------------------------------------------------------
// Multi-lattice step: one launch advances every lattice of a group by one time step.  The
// lattices' segment ranges, each padded to a multiple of 32, are concatenated; a warp finds
// its lattice from the warp-aligned base index and runs that lattice's collision model.
// One launch per time step instead of one per lattice removes the per-launch ramp and the
// gaps between graph nodes that dominate small (<= 1024^2) lattices.
constexpr int kGroupMax = 16;

struct GroupEntry {
    const void* src;    // buffers of the storage type of the launch
    void* dst;
    StepArgs a;
    int model;          // lbm::Model
    int eq_order;       // 4, or 2 / 3 (BGK only)
    unsigned begin;     // first padded segment index of this lattice
    unsigned total;     // ny * nseg (unpadded)
};
struct GroupArgs {
    int n;
    unsigned padded_total;
    GroupEntry e[kGroupMax];
};

template <typename S, bool SH>
__device__ __forceinline__ void group_segment(const GroupEntry& e, const Consts<typename Conv<S>::T>& c,
                                              unsigned local, int lane) {
    constexpr int VEC = StepVec<S>::value;
    Diag dg;
    const unsigned s = local + lane;
    const S* src = static_cast<const S*>(e.src);
    S* dst = static_cast<S*>(e.dst);
    switch (e.model) {
        case BGK:
            if (e.eq_order == 2) step_segment<BGK, 2, S, VEC, false, SH>(src, dst, e.a, c, s, e.total, lane, dg);
            else if (e.eq_order == 3) step_segment<BGK, 3, S, VEC, false, SH>(src, dst, e.a, c, s, e.total, lane, dg);
            else step_segment<BGK, 4, S, VEC, false, SH>(src, dst, e.a, c, s, e.total, lane, dg);
            break;
        case RM: step_segment<RM, 4, S, VEC, false, SH>(src, dst, e.a, c, s, e.total, lane, dg); break;
        case HM: step_segment<HM, 4, S, VEC, false, SH>(src, dst, e.a, c, s, e.total, lane, dg); break;
        case CM: step_segment<CM, 4, S, VEC, false, SH>(src, dst, e.a, c, s, e.total, lane, dg); break;
        case CHM: step_segment<CHM, 4, S, VEC, false, SH>(src, dst, e.a, c, s, e.total, lane, dg); break;
        case CUM: step_segment<CUM, 4, S, VEC, false, SH>(src, dst, e.a, c, s, e.total, lane, dg); break;
        case PR: step_segment<PR, 4, S, VEC, false, SH>(src, dst, e.a, c, s, e.total, lane, dg); break;
        default: step_segment<RR, 4, S, VEC, false, SH>(src, dst, e.a, c, s, e.total, lane, dg); break;
    }
}

template <typename S, bool SHIFT>
__global__ void __launch_bounds__(256) group_step_kernel(const __grid_constant__ GroupArgs g) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    using T = typename Conv<S>::T;
    const int lane = threadIdx.x & 31;
    const unsigned stride = gridDim.x * blockDim.x;
    for (unsigned base = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); base < g.padded_total; base += stride) {
        int k = 0;
        while (k + 1 < g.n && base >= g.e[k + 1].begin) ++k;
        group_segment<S, SHIFT>(g.e[k], make_consts<T>(g.e[k].a), base - g.e[k].begin, lane);
    }
}

}  // namespace lbm
