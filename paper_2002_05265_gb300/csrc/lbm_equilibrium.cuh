// The stored populations of an equilibrium node: g_i = f^eq_i(rho, u) - s_i (Eq. extendedFeq in
// product form minus the shift s_i = rho0 P_sx P_sy), exactly as FP64 arithmetic rounds them to the
// storage type, mostly without FP64 arithmetic.
//
// GB300 has 2 FP64 lanes per SM and clock, conversions included; nine populations are about 150
// FP64 operations, and that pipe bounded the initialisation (36.6 ms at 16384^2, 16 GB to move).  So
// g is evaluated in pairs of floats (to 2^-40 of the sum of its terms' sizes, see equilibrium_node)
// and rounded from there when every value within that bound rounds alike (rounding test: Ziv 1991);
// the few others take the FP64 expressions.
#pragma once

#include "lbm_device.cuh"

namespace lbm {

// Value h + l.
struct Wide {
    float h, l;
};
__device__ __forceinline__ Wide wide_mul(Wide a, Wide b) {
    const float p = __fmul_rn(a.h, b.h);
    return Wide{p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p)))};
}
__device__ __forceinline__ Wide wide_add(Wide a, Wide b) {   // two-sum (Knuth) of the heads
    const float s = __fadd_rn(a.h, b.h), t = __fsub_rn(s, a.h);
    const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, t)), __fsub_rn(b.h, t));
    return Wide{s, __fadd_rn(e, __fadd_rn(a.l, b.l))};
}
__device__ __forceinline__ Wide wide_scale(Wide a, float c) { return Wide{a.h * c, a.l * c}; }   // c = +-2^k
// x as the float of its upper 24 bits and the float nearest to the rest, by integer operations;
// false unless x is zero or 2^LO <= |x| < 2^HI.
template <int LO, int HI> __device__ __forceinline__ bool wide_split(double x, Wide& w) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint32_t sign = hi & 0x80000000u, m = hi & 0x7fffffffu, e = m >> 20;
    if ((m | lo) == 0u) {
        w = Wide{0.0f, 0.0f};
        return true;
    }
    w.h = __uint_as_float(sign | ((m - 0x38000000u) << 3) | (lo >> 29));
    // the lower 29 bits, in units of 2^(e - 1023 - 52)
    const float unit = __uint_as_float(sign | ((e - (1023u + 52u - 127u)) << 23));
    w.l = (float)(lo & 0x1fffffffu) * unit;
    return e - (uint32_t)(1023 + LO) < (uint32_t)(HI - LO);
}

// Rounds h + l +- err to the storage type; false if that interval holds values that round apart.
__device__ __forceinline__ bool round_sure(float h, float l, float err, float& out) {
    const float a = __fadd_rn(h, l - err), b = __fadd_rn(h, l + err);
    out = a;
    return a == b;
}
__device__ __forceinline__ bool round_sure(float h, float l, float err, __half& out) {
    const __half a = __float2half_rn(__fadd_rd(h, l - err)), b = __float2half_rn(__fadd_ru(h, l + err));
    out = __float2half_rn(__fadd_rn(h, l));
    return __half2float(a) == __half2float(b);
}
__device__ __forceinline__ bool round_sure(float h, float l, float err, __nv_bfloat16& out) {
    const __nv_bfloat16 a = __float2bfloat16_rn(__fadd_rd(h, l - err)), b = __float2bfloat16_rn(__fadd_ru(h, l + err));
    out = __float2bfloat16_rn(__fadd_rn(h, l));
    return __bfloat162float(a) == __bfloat162float(b);
}

// FP64 expressions: P_s = phi_s(u_ref), D_s = phi_s(u) - phi_s(u_ref) written as differences.
__device__ __forceinline__ double equilibrium_plain(int i, double r, double vx, double vy, double rho0, double urx,
                                                    double ury) {
    const int sx = ex_of(i), sy = ey_of(i);
    const double Px = phi1d(sx, urx), Py = phi1d(sy, ury);
    const double dux = vx - urx, sux = vx + urx, duy = vy - ury, suy = vy + ury;
    const double Dx = sx ? 0.5 * dux * (sux + sx) : -dux * sux;
    const double Dy = sy ? 0.5 * duy * (suy + sy) : -duy * suy;
    return Px * Py * (r - rho0) + r * (Px * Dy + Dx * (Py + Dy));
}

// The shift's factors P_0, P_+, P_- per axis as pairs of floats, and |P_0|, the larger of |P_+-|.
struct EquilibriumConsts {
    float2 px[3], py[3];
    float ax[2], ay[2];
};
__host__ __device__ inline EquilibriumConsts equilibrium_consts(double urx, double ury) {
    EquilibriumConsts c;
    for (int k = 0; k < 3; ++k) {
        const int s = k == 2 ? -1 : k;
        const double x = phi1d(s, urx), y = phi1d(s, ury);
        c.px[k] = make_float2((float)x, (float)(x - (double)(float)x));
        c.py[k] = make_float2((float)y, (float)(y - (double)(float)y));
        // (2^-12 at least: P itself carries 2^-53, whatever is left of it next to its zero)
        const float ax = fmaxf(fabsf(c.px[k].x), 0x1p-12f), ay = fmaxf(fabsf(c.py[k].x), 0x1p-12f);
        c.ax[k != 0] = k == 2 ? fmaxf(c.ax[1], ax) : ax;
        c.ay[k != 0] = k == 2 ? fmaxf(c.ay[1], ay) : ay;
    }
    return c;
}

template <typename S>
__device__ __forceinline__ void equilibrium_node(double r, double vx, double vy, double rho0, double urx, double ury,
                                                 const EquilibriumConsts& c, S (&g)[9]) {
    if constexpr (sizeof(S) == 8) {
#pragma unroll
        for (int i = 0; i < 9; ++i) g[i] = equilibrium_plain(i, r, vx, vy, rho0, urx, ury);
    } else {
        // ranges in which no product below leaves the FP32 range (see the error bound)
        Wide R, dr, dx, dy, sx, sy;
        bool sure = wide_split<-20, 20>(r, R) && wide_split<-60, 20>(r - rho0, dr) &&
                    wide_split<-60, 2>(vx - urx, dx) && wide_split<-60, 2>(vy - ury, dy);
        if (urx == 0.0 && ury == 0.0) {
            sx = dx;
            sy = dy;
        } else {
            sure = sure && wide_split<-60, 2>(vx + urx, sx) && wide_split<-60, 2>(vy + ury, sy);
        }
        // order 0, +, -: D_0 = -d s, D_+- = (d s +- d) / 2
        const Wide X = wide_mul(dx, sx), Y = wide_mul(dy, sy);
        const Wide Dx[3] = {wide_scale(X, -1.0f), wide_scale(wide_add(X, dx), 0.5f),
                            wide_scale(wide_add(X, wide_scale(dx, -1.0f)), 0.5f)};
        const Wide Dy[3] = {wide_scale(Y, -1.0f), wide_scale(wide_add(Y, dy), 0.5f),
                            wide_scale(wide_add(Y, wide_scale(dy, -1.0f)), 0.5f)};
        // Error bound, in u = 2^-24.  Let M be the sum of the sizes of the terms a value is made of.  A
        // split is off by 2 u^2 M with a low part of 2 u M, P by u^2 M and u M; a wide product of (e, l)
        // and (e', l') by e + e' + l + 2 l' + 2 + l l' with a low part of l + l' + 1; a wide sum by
        // max(e) + 2 max(l) + 1 with max(l) + 1.  So d s is off by 16 (low part 5), D by 27 (6), rho D
        // by 57 (9), H and K by 76 (10), P H by 110 (12), D K by 191 (17) and g by 226 (18).  The
        // rounding of l +- err adds 18, FP64's own less than 1: 2^8 u^2 = 2^-40.  M = |P| (|P'| |dr| +
        // |rho| |D'|) + |D| |rho| (|P'| + |D'|) with |d s| and (|d s| + |d|) / 2 for |D_0| and |D_+-|.
        // Underflow: at most 40 operations lose 2^-150 each, times at most 2^20 2^6 after it; below
        // M = 2^-110 nothing but zero is sure.  (With one bound for all nine, |dr| + |rho| (|d_x| + |d_y|)
        // times 2^-43, M was larger by up to 2.4 for |u_ref| near 1.)
        const float mX = fabsf(X.h), mY = fabsf(Y.h), mR = fabsf(R.h), mr = fabsf(dr.h);
        const float mDx[2] = {mX, 0.5f * (mX + fabsf(dx.h))}, mDy[2] = {mY, 0.5f * (mY + fabsf(dy.h))};
        float err[2][2];   // [xi_x != 0][xi_y != 0]
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const float mH = fmaf(c.ay[b], mr, mR * mDy[b]), mK = mR * (c.ay[b] + mDy[b]);
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                const float M = fmaf(c.ax[a], mH, mDx[a] * mK);
                err[a][b] = fmaf(M, 0x1p-40f, fminf(M, 0x1p-110f));
            }
        }
        unsigned open = sure ? 0u : 0x1ffu;   // populations that the bound leaves open
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const Wide Py{c.py[b].x, c.py[b].y};
            const Wide w = wide_mul(R, Dy[b]);
            const Wide H = wide_add(wide_mul(Py, dr), w);   // Py (rho - rho0) + rho Dy
            const Wide K = wide_add(wide_mul(Py, R), w);    // rho (Py + Dy)
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const int ex = a == 2 ? -1 : a, ey = b == 2 ? -1 : b;
                const Wide Px{c.px[a].x, c.px[a].y};
                const Wide v = wide_add(wide_mul(Px, H), wide_mul(Dx[a], K));
                S out;
                const bool known = round_sure(v.h, v.l, err[a != 0][b != 0], out);
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    if (ex_of(i) != ex || ey_of(i) != ey) continue;
                    g[i] = out;
                    open |= known ? 0u : 1u << i;
                }
            }
        }
#pragma unroll 1
        while (open) {
            const int i = __ffs(open) - 1;
            open &= open - 1;
            const S v = Conv<S>::from_double(equilibrium_plain(i, r, vx, vy, rho0, urx, ury));
#pragma unroll
            for (int k = 0; k < 9; ++k)
                if (k == i) g[k] = v;
        }
    }
}

}  // namespace lbm
