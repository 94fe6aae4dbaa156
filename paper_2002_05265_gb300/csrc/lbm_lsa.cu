// Linear stability analysis of the stream-and-collide scheme on the GPU (App. A): the
// perturbed iteration f'(x + xi_i, t + 1) = G f'(x, t), G = d f* / d f the Jacobian of the
// collision map at a uniform equilibrium state, and plane waves f' ~ exp(i(k.x - omega t))
// give the eigenproblem E^D(k) G A = exp(-i omega) A with E^D = diag(exp(-i xi_i . k))
// (Eq. EigenvaluePbDiscrete); the growth rate of a mode is Im(omega) = ln |exp(-i omega)|.
//
// G is exact: row i is the reverse-mode derivative of the kernels' own collision (collide_vjp)
// applied to the unit adjoint e_i.  The eigenvalues of the 9 x 9 complex matrix come from a
// per-thread Householder reduction to upper Hessenberg form and the shifted QR iteration
// (Francis / Wilkinson shift from the trailing 2 x 2 block, Givens rotations, deflation on
// negligible subdiagonal entries), in FP64.
//
// The FP64 pipe bounds the solver: a scheduler takes 64 clocks for an FP64 instruction of a warp, so
// one warp each keeps the pipe busy and what counts is the number of operations.  Only eigenvalues
// are wanted, so rotations stay inside the active block; a rotation takes one reciprocal square root
// instead of four hypot and four divisions; magnitudes in tests are |re| + |im|; the largest |lambda|
// is found squared, with one logarithm at the end; the phases of E^D are products of two.  The
// matrices live in shared memory, 16 bytes an entry and lane (the local arrays of before did not fit
// the L1).  Measured, 16 flows x 64 x 64 wavenumbers of K: 7.7 -> 3.5 ms.
#include <cuda_runtime.h>

#include <cmath>
#include <vector>

#include "lbm.h"
#include "lbm_adjoint.cuh"
#include "lbm_internal.h"

namespace lbm {
namespace {

struct Cx {
    double re, im;
};
__device__ __forceinline__ Cx cx(double r, double i = 0.0) { return Cx{r, i}; }
__device__ __forceinline__ Cx operator+(Cx a, Cx b) { return Cx{a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ Cx operator-(Cx a, Cx b) { return Cx{a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ Cx operator*(Cx a, Cx b) {
    return Cx{a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
__device__ __forceinline__ Cx operator*(double s, Cx a) { return Cx{s * a.re, s * a.im}; }
__device__ __forceinline__ Cx conj(Cx a) { return Cx{a.re, -a.im}; }
__device__ __forceinline__ double norm2(Cx a) { return a.re * a.re + a.im * a.im; }
__device__ __forceinline__ double abs1(Cx a) { return fabs(a.re) + fabs(a.im); }
// principal square root
__device__ __forceinline__ Cx csqrt(Cx a) {
    const double r = sqrt(norm2(a));
    if (r == 0.0) return cx(0.0);
    const double t = sqrt(0.5 * (r + fabs(a.re))), q = a.im / (2.0 * t);
    if (a.re >= 0.0) return Cx{t, q};
    return Cx{fabs(q), a.im >= 0.0 ? t : -t};
}

constexpr int N = 9;
constexpr int kEigLanes = 32;   // matrices of a CTA

// A lane's matrix in shared memory.
struct Matrix {
    double2* p;
    __device__ __forceinline__ Cx get(int r, int c) const {
        const double2 v = p[(r * N + c) * kEigLanes];
        return Cx{v.x, v.y};
    }
    __device__ __forceinline__ void set(int r, int c, Cx v) const { p[(r * N + c) * kEigLanes] = make_double2(v.re, v.im); }
};

// Column C of the Householder reduction to upper Hessenberg form: zeroes a[C + 2 ..][C].
template <int C>
__device__ __forceinline__ void hessenberg_column(const Matrix& a) {
    constexpr int M = N - 1 - C;   // rows C + 1 .. N - 1
    Cx v[M];
    double alpha2 = 0.0;
#pragma unroll
    for (int r = 0; r < M; ++r) {
        v[r] = a.get(C + 1 + r, C);
        alpha2 += norm2(v[r]);
    }
    if (alpha2 == 0.0) return;
    const double alpha = sqrt(alpha2), x2 = norm2(v[0]);
    const double ix = x2 > 0.0 ? rsqrt(x2) : 0.0;
    const Cx ph = x2 > 0.0 ? ix * v[0] : cx(1.0);
    // v = x + ph alpha e_1, H = I - 2 v v^H / (v^H v), v^H v = 2 (alpha^2 + alpha |x_1|)
    const double s = 1.0 / (alpha2 + alpha * (x2 * ix));
    v[0] = v[0] + alpha * ph;
    a.set(C + 1, C, -alpha * ph);
#pragma unroll
    for (int r = 1; r < M; ++r) a.set(C + 1 + r, C, cx(0.0));
#pragma unroll 1
    for (int j = C + 1; j < N; ++j) {   // a <- H a
        Cx x[M], d = cx(0.0);
#pragma unroll
        for (int r = 0; r < M; ++r) {
            x[r] = a.get(C + 1 + r, j);
            d = d + conj(v[r]) * x[r];
        }
        d = s * d;
#pragma unroll
        for (int r = 0; r < M; ++r) a.set(C + 1 + r, j, x[r] - v[r] * d);
    }
#pragma unroll 1
    for (int i = 0; i < N; ++i) {   // a <- a H
        Cx x[M], d = cx(0.0);
#pragma unroll
        for (int r = 0; r < M; ++r) {
            x[r] = a.get(i, C + 1 + r);
            d = d + x[r] * v[r];
        }
        d = s * d;
#pragma unroll
        for (int r = 0; r < M; ++r) a.set(i, C + 1 + r, x[r] - d * conj(v[r]));
    }
}

// Eigenvalues of the complex N x N matrix a (overwritten), each handed to `found` with its index.
// Returns the number of QR sweeps, or -1 if an eigenvalue did not converge within the sweep limit.
template <typename Found>
__device__ int eig9(const Matrix& a, Found found) {
    hessenberg_column<0>(a);
    hessenberg_column<1>(a);
    hessenberg_column<2>(a);
    hessenberg_column<3>(a);
    hessenberg_column<4>(a);
    hessenberg_column<5>(a);
    hessenberg_column<6>(a);
    // shifted QR on the active block [lo, hi]; a subdiagonal entry is negligible against its
    // two diagonal neighbours, or against the matrix norm when both are tiny (zero eigenvalues:
    // with omega_3 = omega_4 = 1 the collision removes whole moments)
    double anorm = 0.0;
#pragma unroll 1
    for (int i = 0; i < N; ++i)
#pragma unroll 1
        for (int j = i > 0 ? i - 1 : 0; j < N; ++j) anorm += norm2(a.get(i, j));
    anorm = sqrt(anorm);
    int hi = N - 1, sweeps = 0;
    while (hi >= 0) {
        // deflation: find the start of the unreduced block ending at hi
        int lo = hi;
        double below = abs1(a.get(hi, hi));
        while (lo > 0) {
            const double above = abs1(a.get(lo - 1, lo - 1));
            if (abs1(a.get(lo, lo - 1)) <= 1e-15 * fmax(below + above, 1e-3 * anorm)) {
                a.set(lo, lo - 1, cx(0.0));
                break;
            }
            below = above;
            --lo;
        }
        if (lo == hi) {
            found(hi, a.get(hi, hi));
            --hi;
            continue;
        }
        if (++sweeps > 60 * N) return -1;
        // Wilkinson shift: eigenvalue of the trailing 2 x 2 block closest to a[hi][hi]
        const Cx p = a.get(hi - 1, hi - 1), q = a.get(hi - 1, hi), r = a.get(hi, hi - 1), t = a.get(hi, hi);
        const Cx half_diff = 0.5 * (p - t), disc = csqrt(half_diff * half_diff + q * r);
        // (e - t) = (p - t) / 2 +- disc, the smaller of the two
        const Cx e1 = half_diff + disc, e2 = half_diff - disc;
        Cx mu = t + (norm2(e1) < norm2(e2) ? e1 : e2);
        if (sweeps % 11 == 10) {   // exceptional shift, rotating in the complex plane
            const double e = 0.75 * (abs1(r) + abs1(a.get(hi - 1, hi - 2 >= 0 ? hi - 2 : 0)));
            double sn, cn;
            sincos(0.7 * sweeps, &sn, &cn);
            mu = t + Cx{e * cn, e * sn};
        }
        // QR step on a[lo..hi] - mu I with Givens rotations, then RQ + mu I.  Rotation k takes rows
        // k, k + 1; the columns k - 1, k take rotation k - 1 right after it, when their rows up to k
        // are those of R.
        double c0 = 1.0;
        Cx s0 = cx(0.0);
        a.set(lo, lo, a.get(lo, lo) - mu);
#pragma unroll 1
        for (int k = lo; k <= hi; ++k) {
            double c = 1.0;
            Cx sn = cx(0.0);
            if (k < hi) {
                a.set(k + 1, k + 1, a.get(k + 1, k + 1) - mu);
                // c = |x| / n, s = (x / |x|) conj(y) / n, n^2 = |x|^2 + |y|^2:
                // [c s; -conj(s) c] [x; y] = [., 0]
                const Cx x = a.get(k, k), y = a.get(k + 1, k);
                const double x2 = norm2(x), n2 = x2 + norm2(y);
                if (x2 * n2 > 1e-290) {
                    const double d = rsqrt(x2 * n2);
                    c = x2 * d;
                    sn = d * (x * conj(y));
                    a.set(k, k, (n2 * d) * x);
                } else if (n2 > 0.0) {   // x vanishes (to 1e-75 at least): swap the rows
                    const double d = rsqrt(n2);
                    c = 0.0;
                    sn = d * conj(y);
                    a.set(k, k, cx(n2 * d));
                }
                a.set(k + 1, k, cx(0.0));
#pragma unroll 1
                for (int j = k + 1; j <= hi; ++j) {
                    const Cx u = a.get(k, j), w = a.get(k + 1, j);
                    a.set(k, j, c * u + sn * w);
                    a.set(k + 1, j, c * w - conj(sn) * u);
                }
            }
            if (k > lo) {
#pragma unroll 1
                for (int i = lo; i <= k; ++i) {
                    const Cx u = a.get(i, k - 1), w = a.get(i, k);
                    a.set(i, k - 1, c0 * u + conj(s0) * w);
                    a.set(i, k, c0 * w - s0 * u);
                }
                a.set(k - 1, k - 1, a.get(k - 1, k - 1) + mu);
            }
            c0 = c;
            s0 = sn;
        }
        a.set(hi, hi, a.get(hi, hi) + mu);
    }
    return sweeps;
}

// G (row-major 9 x 9, FP64) of the collision map at f = f^eq(rho, u) for each base flow.
template <int MODEL>
__global__ void lsa_jacobian_kernel(const double* __restrict__ flows, int nflows, VjpConsts<double> c,
                                    double* __restrict__ G) {
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= nflows) return;
    const double rho = flows[3 * f], ux = flows[3 * f + 1], uy = flows[3 * f + 2];
    double g[9];
#pragma unroll
    for (int i = 0; i < 9; ++i)   // f^eq (Eq. extendedFeq, product form) minus the shift w_i rho0
        g[i] = rho * phi1d(ex_of(i), ux) * phi1d(ey_of(i), uy) - weight_of(i) * c.rho0;
    for (int i = 0; i < 9; ++i) {
        double v[9], gb[9], wb, w3b, w4b;
#pragma unroll
        for (int j = 0; j < 9; ++j) v[j] = (j == i) ? 1.0 : 0.0;
        collide_vjp<MODEL, double>(g, v, gb, c, wb, w3b, w4b);
#pragma unroll
        for (int j = 0; j < 9; ++j) G[(long long)f * 81 + i * 9 + j] = gb[j];
    }
}

// G of BGK with the second-order (eq_order 2) or partial third-order (3) equilibrium, in
// closed form: f*_i = f_i - omega (f_i - rho p_i(u)) with rho = sum f, u = sum xi f / rho, so
// d f*_i / d f_j = (1 - omega) delta_ij + omega (p_i + dp_i/du_x (xi_jx - u_x) + dp_i/du_y (xi_jy - u_y)).
//   order 2: p_i = w_i (1 + 3 xi.u + 9/2 (xi.u)^2 - 3/2 u^2) (Sec. 2, textbook polynomial);
//   order 3: p_i = phi_sx(u_x) phi_sy(u_y) - u_x^2 u_y^2 b(sx) b(sy) (Eq. extendedFeq minus its
//            A_22 term; b(0) = 1, b(+-1) = -1/2).
__global__ void lsa_jacobian_bgk_kernel(const double* __restrict__ flows, int nflows, double omega, int eq_order,
                                        double* __restrict__ G) {
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= nflows) return;
    const double ux = flows[3 * f + 1], uy = flows[3 * f + 2];
    for (int i = 0; i < 9; ++i) {
        const int sx = ex_of(i), sy = ey_of(i);
        double p, px, py;
        if (eq_order == 2) {
            const double w = weight_of(i), eu = sx * ux + sy * uy;
            p = w * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * (ux * ux + uy * uy));
            px = w * (3.0 * sx + 9.0 * eu * sx - 3.0 * ux);
            py = w * (3.0 * sy + 9.0 * eu * sy - 3.0 * uy);
        } else {
            const double fx = phi1d(sx, ux), fy = phi1d(sy, uy);
            const double dfx = sx ? ux + 0.5 * sx : -2.0 * ux, dfy = sy ? uy + 0.5 * sy : -2.0 * uy;
            const double b = (sx ? -0.5 : 1.0) * (sy ? -0.5 : 1.0);
            p = fx * fy - ux * ux * uy * uy * b;
            px = dfx * fy - 2.0 * ux * uy * uy * b;
            py = fx * dfy - 2.0 * ux * ux * uy * b;
        }
        for (int j = 0; j < 9; ++j)
            G[(long long)f * 81 + i * 9 + j] =
                (i == j ? 1.0 - omega : 0.0) + omega * (p + px * (ex_of(j) - ux) + py * (ey_of(j) - uy));
    }
}

// growth[f * nk + k] = max_j ln |lambda_j(E^D(k) G_f)|; eig (optional) the eigenvalues.
__global__ void __launch_bounds__(kEigLanes) lsa_growth_kernel(const double* __restrict__ G, int nflows,
                                                               const double* __restrict__ kvec, int nk,
                                                               double* __restrict__ growth, double* __restrict__ eig,
                                                               int* __restrict__ failed) {
    __shared__ double2 sm[N * N * kEigLanes];
    const long long id = blockIdx.x * (long long)kEigLanes + threadIdx.x;
    if (id >= (long long)nflows * nk) return;
    const int f = (int)(id / nk), k = (int)(id - (long long)f * nk);
    const Matrix a{sm + threadIdx.x};
    // exp(-i k_x), exp(-i k_y) and their products
    Cx ex[3], ey[3];   // index: velocity component + 1
    double sn, cn;
    sincos(kvec[2 * k], &sn, &cn);
    ex[0] = Cx{cn, sn}; ex[1] = cx(1.0); ex[2] = Cx{cn, -sn};
    sincos(kvec[2 * k + 1], &sn, &cn);
    ey[0] = Cx{cn, sn}; ey[1] = cx(1.0); ey[2] = Cx{cn, -sn};
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const Cx e = ex_of(i) == 0 ? ey[ey_of(i) + 1] : (ey_of(i) == 0 ? ex[ex_of(i) + 1] : ex[ex_of(i) + 1] * ey[ey_of(i) + 1]);
#pragma unroll
        for (int j = 0; j < N; ++j) a.set(i, j, G[(long long)f * 81 + i * 9 + j] * e);
    }
    double best = -1.0;
    const int sweeps = eig9(a, [&](int i, Cx lam) {
        const double m = norm2(lam);
        best = m > best ? m : best;
        if (eig) {
            eig[id * 18 + 2 * i] = lam.re;
            eig[id * 18 + 2 * i + 1] = lam.im;
        }
    });
    if (sweeps < 0) {
        atomicExch(failed, 1);
        growth[id] = nan("");
        return;
    }
    growth[id] = best > 0.0 ? 0.5 * log(best) : -1e300;
}

template <int MODEL>
void launch_jacobian(const double* flows, int nflows, const VjpConsts<double>& c, double* G, cudaStream_t s) {
    lsa_jacobian_kernel<MODEL><<<(nflows + 127) / 128, 128, 0, s>>>(flows, nflows, c, G);
}

bool on_device(const void* p) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

}  // namespace
}  // namespace lbm

extern "C" int lbm_lsa_growth(int model, lbm_rates rates, int eq_order, const double* flows, int nflows,
                              const double* k, int nk, double* growth, double* eig, double* jac, void* stream) {
    using namespace lbm;
    if (model < LBM_BGK || model > LBM_K_EQ || !flows || !k || !growth || nflows < 1 || nk < 1 ||
        (long long)nflows * nk > (1LL << 31) || eq_order < 2 || eq_order > 4)
        return LBM_ERR_INVALID_ARG;
    if (eq_order != 4 && model != LBM_BGK) return LBM_ERR_UNSUPPORTED;
    const double r[3] = {rates.omega_nu, rates.omega3, rates.omega4};
    for (double w : r)
        if (!(std::isfinite(w) && w > 0.0 && w < 2.0)) return LBM_ERR_INVALID_ARG;
    for (const double* p : {flows, k, (const double*)growth})
        if (!on_device(p)) return LBM_ERR_INVALID_ARG;
    if ((eig && !on_device(eig)) || (jac && !on_device(jac))) return LBM_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    VjpConsts<double> c;
    c.w = rates.omega_nu;
    c.w3 = model == LBM_PR ? 1.0 : rates.omega3;
    c.w4 = model == LBM_PR ? 1.0 : rates.omega4;
    c.rho0 = 1.0;
    c.urx = c.ury = 0.0;
    c.Xr = c.Yr = 1.0 / 3.0;
    // cumulant readings: LBM_K_PRE / LBM_K_EQ take the K Jacobian with kappa = 1 / 0
    const int kread = model == LBM_K_PRE ? 1 : (model == LBM_K_EQ ? 2 : 0);
    c.kap = cumulant_kappa(kread, rates.omega_nu);
    c.kapw = kread == 0 ? -1.0 : 0.0;
    if (kread) model = LBM_K;
    double* G = jac;
    int* failed = nullptr;
    cudaError_t e = cudaSuccess;
    if (!G) e = cudaMalloc(&G, sizeof(double) * 81 * (size_t)nflows);
    if (e == cudaSuccess) e = cudaMalloc(&failed, sizeof(int));
    if (e == cudaSuccess) e = cudaMemsetAsync(failed, 0, sizeof(int), s);
    if (e == cudaSuccess && eq_order != 4) {
        lsa_jacobian_bgk_kernel<<<(nflows + 127) / 128, 128, 0, s>>>(flows, nflows, rates.omega_nu, eq_order, G);
        e = cudaGetLastError();
    } else if (e == cudaSuccess) {
        switch (model) {
            case LBM_BGK: launch_jacobian<BGK>(flows, nflows, c, G, s); break;
            case LBM_RM: launch_jacobian<RM>(flows, nflows, c, G, s); break;
            case LBM_HM: launch_jacobian<HM>(flows, nflows, c, G, s); break;
            case LBM_CM: launch_jacobian<CM>(flows, nflows, c, G, s); break;
            case LBM_CHM: launch_jacobian<CHM>(flows, nflows, c, G, s); break;
            case LBM_K: launch_jacobian<CUM>(flows, nflows, c, G, s); break;
            case LBM_PR: launch_jacobian<PR>(flows, nflows, c, G, s); break;
            default: launch_jacobian<RR>(flows, nflows, c, G, s); break;
        }
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        const long long n = (long long)nflows * nk;
        lsa_growth_kernel<<<(unsigned)((n + kEigLanes - 1) / kEigLanes), kEigLanes, 0, s>>>(G, nflows, k, nk, growth, eig, failed);
        e = cudaGetLastError();
    }
    int h_failed = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h_failed, failed, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (failed) cudaFree(failed);
    if (G && G != jac) cudaFree(G);
    if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? LBM_ERR_NOMEM : LBM_ERR_CUDA;
    return h_failed ? LBM_ERR_TIMEOUT : LBM_OK;
}
