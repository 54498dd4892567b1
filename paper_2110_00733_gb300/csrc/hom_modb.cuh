// hom_modb.cuh -- point-wise kernels of the MoDBFFT solver (section 2.2):
// the displacement unknown u^ (3 complex components per frequency of the
// half spectrum) is expanded into the strain sym(u^ (x) xi) and the penalty
// vector alpha sym(u^ (x) xi) . xi before the inverse transform, and the
// transformed stress / penalty fields are contracted back, eq. (modbfftfop):
//   A^alpha(u^) = F{ (1-chi_v) C : F^-1{ u^ (x)^s xi } } . xi
//               + F{ chi_v F^-1{ alpha (u^ (x)^s xi) . xi } }.
// Frequencies are the continuous ones of eq. (freq), xi_p = i 2 pi m_p (unit
// cell), with the Nyquist component set to 0; where xi = 0 there is no
// unknown and no equation.  The preconditioner is eq. (precf) with the mean
// stiffness of eq. (avstiff).
#pragma once
#include "hom_sum3.h"
#include "hom_internal.h"

namespace hom {

// frequency index of half-spectrum point f and its continuous xi / (i 2 pi)
template <typename R>
__device__ __forceinline__ void modb_freq(const Geometry &g, int f, R q[3], int &k3) {
    const int hh = g.h;
    k3 = f % hh;
    const int rest = f / hh;
    const int k2 = rest % g.n2, k1 = rest / g.n2;
    const int ks[3] = {k1, k2, k3}, ns[3] = {g.n1, g.n2, g.n3};
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        const int n = ns[p], k = ks[p];
        q[p] = 2 * k == n ? (R)0 : (R)((2 * k < n) ? k : k - n);
    }
}

// out10 = (sym(u (x) xi) Mandel, alpha sym(u (x) xi) . xi, 0), or the first
// six with nc_out = 6 (modb_expand_at)
template <typename R>
__global__ void k_modb_expand(Geometry g, R alpha, int with_penalty, const cpx<R> *__restrict__ u,
                              cpx<R> *__restrict__ out, int nc_out, const MinresState *state) {
    if (state && state->done) return;
    const int hh = g.h;
    for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < (int)g.S; f += gridDim.x * blockDim.x) {
        const int k3 = f % hh, rest = f / hh;
        const int k2 = rest % g.n2, k1 = rest / g.n2;
        modb_expand_at<R>(g, k1, k2, k3, u + 3 * (size_t)f, alpha, with_penalty, nc_out, out + (size_t)f * nc_out);
    }
}

// out3 = tau^ . xi + h^ (10-component input), 0 where xi = 0; with dotv,
// the weighted partial sum <dotv, out3> per CTA
template <typename R>
__global__ void __launch_bounds__(kEwThreads) k_modb_contract(Geometry g, const cpx<R> *__restrict__ in,
                                                              cpx<R> *__restrict__ out,
                                                              const cpx<R> *__restrict__ dotv, double *partials,
                                                              const MinresState *state) {
    if (state && state->done) return;
    const R tp = (R)6.28318530717958647692;
    const R r2 = (R)0.70710678118654752440;
    double acc = 0.0;
    for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < (int)g.S; f += gridDim.x * blockDim.x) {
        R qd[3];
        int k3;
        modb_freq(g, f, qd, k3);
        cpx<R> r[3] = {mk<R>(0, 0), mk<R>(0, 0), mk<R>(0, 0)};
        if (!(qd[0] == 0 && qd[1] == 0 && qd[2] == 0)) {
            const R s[3] = {tp * qd[0], tp * qd[1], tp * qd[2]};
            const cpx<R> *t = in + (size_t)f * 10;
            const cpx<R> T[3][3] = {{t[0], scale<R>(t[5], r2), scale<R>(t[4], r2)},
                                    {scale<R>(t[5], r2), t[1], scale<R>(t[3], r2)},
                                    {scale<R>(t[4], r2), scale<R>(t[3], r2), t[2]}};
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                // (tau xi)_i = i sum_j tau_ij s_j
                const cpx<R> a = add<R>(add<R>(scale<R>(T[i][0], s[0]), scale<R>(T[i][1], s[1])), scale<R>(T[i][2], s[2]));
                r[i] = add<R>(mk<R>(-a.y, a.x), t[6 + i]);
            }
        }
        const double w = (double)pweight(k3, g.n3);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            out[3 * f + i] = r[i];
            if (dotv) {
                const cpx<R> d = dotv[3 * f + i];
                acc += w * ((double)d.x * (double)r[i].x + (double)d.y * (double)r[i].y);
            }
        }
    }
    if (dotv) {
        const double sum = block_sum(acc);
        if (threadIdx.x == 0) partials[blockIdx.x] = sum;
    }
}

// out3 = [xi . Cbar . xi]^-1 in3, Cbar isotropic (lam_b, mu_b).  With xi = i 2 pi q,
// q integers and Q = |q|^2, xi.Cbar.xi = -4 pi^2 ((lam+mu) q q^T + mu Q I), whose
// inverse is A / Q (I - c q q^T / Q), A = -1 / (4 pi^2 mu), c = (lam+mu) / (lam+2 mu).
template <typename R> struct PrecondCoef;
template <> struct PrecondCoef<double> { double A, c; };
// FP32 fields: the coefficients as sums of two floats
template <> struct PrecondCoef<float> { float Ah, Al, ch, cl; };

template <typename R> PrecondCoef<R> precond_coef(double lam_b, double mu_b) {
    const double A = -1.0 / (39.47841760435743447534 * mu_b), c = (lam_b + mu_b) / (lam_b + 2.0 * mu_b);
    if constexpr (sizeof(R) == 8) return PrecondCoef<R>{A, c};
    else {
        const float Ah = (float)A, ch = (float)c;
        return PrecondCoef<R>{Ah, (float)(A - Ah), ch, (float)(c - ch)};
    }
}

__device__ __forceinline__ void modb_precond_point(const PrecondCoef<double> &k, const double q[3], const double2 *v,
                                                   double2 *out) {
    const double Q = q[0] * q[0] + q[1] * q[1] + q[2] * q[2];
    if (Q == 0.0) {
        out[0] = out[1] = out[2] = mk<double>(0, 0);
        return;
    }
    const double iq = 1.0 / Q, a = k.A * iq, b = k.c * iq;
    const double dre = b * (q[0] * v[0].x + q[1] * v[1].x + q[2] * v[2].x),
                 dim = b * (q[0] * v[0].y + q[1] * v[1].y + q[2] * v[2].y);
#pragma unroll
    for (int i = 0; i < 3; ++i) out[i] = mk<double>(a * (v[i].x - q[i] * dre), a * (v[i].y - q[i] * dim));
}

// FP32 fields: the same in sums of two floats (48 bits) rounded to FP32 at the
// end.  FP64 arithmetic gives the same rounding but runs at 1/64 of the rate:
// with its two divisions a point it bound the PCG step (see k_cg_xr).
__device__ __forceinline__ float2 ff_two_sum(float a, float b) {   // (sum, its rounding error)
    const float s = a + b, t = s - a;
    return make_float2(s, (a - (s - t)) + (b - t));
}
// sum_i q_i v_i as (hi, lo)
__device__ __forceinline__ float2 ff_dot3(const float q[3], float v0, float v1, float v2) {
    const float p0 = q[0] * v0, p1 = q[1] * v1, p2 = q[2] * v2;
    const float e0 = fmaf(q[0], v0, -p0), e1 = fmaf(q[1], v1, -p1), e2 = fmaf(q[2], v2, -p2);
    const float2 s1 = ff_two_sum(p0, p1), s2 = ff_two_sum(s1.x, p2);
    const float lo = ((s1.y + s2.y) + (e0 + e1)) + e2, hi = s2.x + lo;   // renormalised
    return make_float2(hi, lo - (hi - s2.x));
}
__device__ __forceinline__ float2 ff_mul(float2 a, float2 b) {
    const float p = a.x * b.x;
    return make_float2(p, fmaf(a.x, b.x, -p) + (a.x * b.y + a.y * b.x));
}
__device__ __forceinline__ void modb_precond_point(const PrecondCoef<float> &k, const float q[3], const float2 *v,
                                                   float2 *out) {
    const float Q = q[0] * q[0] + q[1] * q[1] + q[2] * q[2];   // exact: below 2^24 up to 4096^3
    if (Q == 0.f) {
        out[0] = out[1] = out[2] = mk<float>(0, 0);
        return;
    }
    const float y = 1.0f / Q;
    const float2 iq = make_float2(y, fmaf(-Q, y, 1.0f) * y);
    const float2 a = ff_mul(make_float2(k.Ah, k.Al), iq), b = ff_mul(make_float2(k.ch, k.cl), iq);
    const float2 dre = ff_mul(b, ff_dot3(q, v[0].x, v[1].x, v[2].x)), dim = ff_mul(b, ff_dot3(q, v[0].y, v[1].y, v[2].y));
    auto comp = [&](float x, float qi, float2 d) {   // a (x - q_i d)
        const float p = qi * d.x, e = fmaf(qi, d.x, -p) + qi * d.y;
        const float2 s = ff_two_sum(x, -p);
        const float l = s.y - e;
        const float h = s.x * a.x;
        return h + (fmaf(s.x, a.x, -h) + (s.x * a.y + l * a.x));
    };
#pragma unroll
    for (int i = 0; i < 3; ++i) out[i] = mk<float>(comp(v[i].x, q[i], dre), comp(v[i].y, q[i], dim));
}

template <typename R>
__global__ void k_modb_precond(Geometry g, PrecondCoef<R> pc, const cpx<R> *__restrict__ in, cpx<R> *__restrict__ out) {
    for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < (int)g.S; f += gridDim.x * blockDim.x) {
        R q[3];
        int k3;
        modb_freq(g, f, q, k3);
        modb_precond_point(pc, q, in + 3 * f, out + 3 * f);
    }
}

// PCG step: x += a p; r -= a q; z = M r; partials <r,z> (first half) and
// <r,r> (second half), Parseval-weighted.  Bound by HBM (seven 3-component
// vectors); the sums of a thread's points are kept as three floats (Sum3: as good
// as exact) and added in FP64 over the grid, so that they are as far off as FP64
// sums of the points (1e-16 rms, 24^3 to 256^3); st->sc, a power of two, brings the
// products into the range of FP32.
// In FP64 throughout the pass was bound by the FP64 pipe: 191 us at 128^3.
template <typename R>
__global__ void __launch_bounds__(kEwThreads) k_cg_xr(Geometry g, PrecondCoef<R> pc, cpx<R> *__restrict__ x,
                                                      cpx<R> *__restrict__ r, const cpx<R> *__restrict__ p,
                                                      const cpx<R> *__restrict__ q, cpx<R> *__restrict__ z,
                                                      const CgState *st, double *partials) {
    if (st->done) return;
    const R a = (R)st->a, sc = (R)st->sc;
    const double isc2 = 1.0 / (st->sc * st->sc);
    typename std::conditional<sizeof(R) == 4, Sum3, Acc<R>>::type rz, rr;
    for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < (int)g.S; f += gridDim.x * blockDim.x) {
        R qv[3];
        int k3;
        modb_freq(g, f, qv, k3);
        cpx<R> rv[3], zv[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const cpx<R> pp = p[3 * f + i], qq = q[3 * f + i], xx = x[3 * f + i], rr0 = r[3 * f + i];
            x[3 * f + i] = mk<R>(xx.x + a * pp.x, xx.y + a * pp.y);
            rv[i] = mk<R>(rr0.x - a * qq.x, rr0.y - a * qq.y);
            r[3 * f + i] = rv[i];
        }
        modb_precond_point(pc, qv, rv, zv);
        const R w = (R)pweight(k3, g.n3);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            z[3 * f + i] = zv[i];
            const cpx<R> rs = scale<R>(rv[i], sc), zs = scale<R>(zv[i], sc);
            rz.add_prod(w * rs.x, zs.x);
            rz.add_prod(w * rs.y, zs.y);
            rr.add_prod(w * rs.x, rs.x);
            rr.add_prod(w * rs.y, rs.y);
        }
    }
    const double s1 = block_sum(rz.value());
    if (threadIdx.x == 0) partials[blockIdx.x] = isc2 * s1;
    const double s2 = block_sum(rr.value());
    if (threadIdx.x == 0) partials[gridDim.x + blockIdx.x] = isc2 * s2;
}

// PCG direction: p = z + b p
template <typename R>
__global__ void k_cg_p(int n, cpx<R> *__restrict__ p, const cpx<R> *__restrict__ z, const CgState *st) {
    if (st->done) return;
    const R b = (R)st->b;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const cpx<R> pp = p[i], zz = z[i];
        p[i] = mk<R>(zz.x + b * pp.x, zz.y + b * pp.y);
    }
}

// ----- launchers ------------------------------------------------------------
template <typename R>
void Launch<R>::modb_expand(const Geometry &g, cudaStream_t st, double alpha, int with_penalty, const cpx<R> *u,
                            cpx<R> *out, int nc_out, const MinresState *state) {
    k_modb_expand<R><<<ew_grid(g.S), kEwThreads, 0, st>>>(g, (R)alpha, with_penalty, u, out, nc_out, state);
}
template <typename R>
void Launch<R>::modb_contract(const Geometry &g, cudaStream_t st, const cpx<R> *in10, cpx<R> *out3, const cpx<R> *dotv,
                              double *partials, const MinresState *state) {
    k_modb_contract<R><<<ew_grid(g.S), kEwThreads, 0, st>>>(g, in10, out3, dotv, partials, state);
}
template <typename R>
void Launch<R>::modb_precond(const Geometry &g, cudaStream_t st, double lam_b, double mu_b, const cpx<R> *in,
                             cpx<R> *out) {
    k_modb_precond<R><<<ew_grid(g.S), kEwThreads, 0, st>>>(g, precond_coef<R>(lam_b, mu_b), in, out);
}
template <typename R>
void Launch<R>::cg_xr(const Geometry &g, cudaStream_t st, double lam_b, double mu_b, cpx<R> *x, cpx<R> *r,
                      const cpx<R> *p, const cpx<R> *q, cpx<R> *z, const CgState *state, double *partials) {
    k_cg_xr<R><<<ew_grid(g.S), kEwThreads, 0, st>>>(g, precond_coef<R>(lam_b, mu_b), x, r, p, q, z, state, partials);
}
template <typename R>
void Launch<R>::cg_p(const Geometry &g, cudaStream_t st, cpx<R> *p, const cpx<R> *z, const CgState *state) {
    const int n = (int)(3 * g.S);
    k_cg_p<R><<<ew_grid(n), kEwThreads, 0, st>>>(n, p, z, state);
}

}  // namespace hom
