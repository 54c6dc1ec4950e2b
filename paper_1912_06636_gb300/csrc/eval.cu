// Evaluation phase (Sec. 3.4): basis functions phi_i and their gradients on each batch's
// points, for the functions of the batch's reduced basis nnz(B) (Sec. 3.3.2); and the
// batch-to-atom distances behind nnz(B).
//
// phi_i(r) = R_f(|d|) Y_lm(d/|d|), d = r - R_A, is computed as g(r) S_lm(d) with the real
// solid harmonic S_lm = r^l Y_lm (a polynomial in x, y, z) and g = R / r^l, so that
//   grad phi = g'(r) (d/r) S_lm + g grad S_lm,   g' = (R' - l R / r) / r^l.
// The harmonics of l come from those of l - 1 and l - 2, and their gradients are fixed combinations
// of at most two harmonics of l - 1 (DevSystem::hc, as float-floats hcf), so that no division by sin(theta)
// and no derivative recurrence occurs. R_f is the natural cubic spline in s = ln(r/r0)/Delta, evaluated
// as a per-segment polynomial in t = s - floor(s) (r < r0 uses r0; R = 0 for r >= rc).
#include <cmath>
#include <type_traits>

#include "ff.h"
#include "nao_internal.h"
#include "radial.h"
#include "split_bits.h"

namespace {

// ----------------------------------------------------------------------------------------
// nnz(B): min over each batch's points of |r - R_A|^2 per atom, every operation separately
// rounded (the host then applies r2 < rc*rc per radial function). One warp per atom.
// ----------------------------------------------------------------------------------------
__global__ void minr2_kernel(const double *__restrict__ atom_xyz, const int32_t *__restrict__ bmol,
                             const int32_t *__restrict__ aoff, int max_atoms, const double *__restrict__ px,
                             const double *__restrict__ py, const double *__restrict__ pz,
                             const int32_t *__restrict__ boff, double *__restrict__ minr2) {
    const int b = blockIdx.x, m = bmol[b];
    const int p0 = boff[b], p1 = boff[b + 1];
    const int a0 = aoff[m], na = aoff[m + 1] - a0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    for (int a = warp; a < na; a += nwarp) {
        const double ax = atom_xyz[3 * (a0 + a)], ay = atom_xyz[3 * (a0 + a) + 1], az = atom_xyz[3 * (a0 + a) + 2];
        double mn = __longlong_as_double(0x7ff0000000000000LL);  // +inf
        for (int p = p0 + lane; p < p1; p += 32) {
            const double dx = __dsub_rn(px[p], ax), dy = __dsub_rn(py[p], ay), dz = __dsub_rn(pz[p], az);
            const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
            mn = fmin(mn, r2);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        if (lane == 0) minr2[(size_t)b * max_atoms + a] = mn;
    }
}

// Output addressing of one evaluation launch.
template <typename OutT>
struct EvalOut {
    OutT *phi;    // phi of reduced-basis position j, point q at phi[j*phi_rs + q]
    OutT *grad;   // component c at grad[c*grad_cs + j*grad_rs + q] (nullptr: none)
    int64_t phi_rs, grad_cs, grad_rs;
    int32_t qmax; // points written per row (q >= P_b is written as 0)
};

// Split path (EXPO = 1): per point, the largest biased exponent of phi over the basis, reduced
// while the values are produced (the density slicing's point exponents) into red[q - q0], shared
// memory of the CTA.
struct ExpoIn {
    int *red;
    int q0;
};

// Distance below which the FP32 path evaluates in FP64 (bohr).
constexpr double kNearNucleus = 0.1;

// ---- arithmetics ---------------------------------------------------------------------------
// The solid harmonics and their gradients are computed in H, the radial functions and the products in R.
//   F64: both in FP64.
//   F32: harmonics in float-float, rounded once to FP32 (their recurrences cancel near the nodes of
//        cos(m phi), sin(m phi) and P_l^m(cos theta), where FP32 loses several ulps), the rest in FP32, but
//        ill-conditioned spline segments (DevSystem::seg64) in float-float.
//   FF:  the split path's evaluation, both in float-float (csrc/ff.h), ~48-bit significands on the FP32 pipe.
// The geometry (d, r^2, 1/r) and the radial coordinate t stay in FP64 in all three. Points within
// kNearNucleus of an atom take F64 in all three, and FF takes it for atoms with functions of l >= 5.
struct F64 {
    using H = double;
    using R = double;
};
struct F32 {
    using H = ffa::F;
    using R = float;
};
struct FF {
    using H = ffa::F;
    using R = ffa::F;
};

__device__ __forceinline__ double hmul(double a, double b) { return a * b; }
__device__ __forceinline__ ffa::F hmul(ffa::F a, ffa::F b) { return ffa::mul(a, b); }
__device__ __forceinline__ double hdot(double a, double b, double c, double d) { return fma(a, b, c * d); }
__device__ __forceinline__ ffa::F hdot(ffa::F a, ffa::F b, ffa::F c, ffa::F d) { return ffa::dot2(a, b, c, d); }
__device__ __forceinline__ double hneg(double a) { return -a; }
__device__ __forceinline__ ffa::F hneg(ffa::F a) { return ffa::neg(a); }
template <typename H> __device__ __forceinline__ H from_f64(double x);
template <> __device__ __forceinline__ double from_f64<double>(double x) { return x; }
template <> __device__ __forceinline__ ffa::F from_f64<ffa::F>(double x) { return ffa::from_double_bits(x); }

// Coefficient c of the harmonics' recurrences: in FP64 0 ra, 1 rb, 2 dz, 3 dp, 4 dm, 5 kl at m = 0 (DevSystem::hc), as
// float-floats 0 N, 1 beta, 2 dz, 3 dp, 4 dm (DevSystem::hcf).
template <typename H, int c>
__device__ __forceinline__ H coef(const DevSystem &s, int l, int m) {
    if constexpr (std::is_same<H, double>::value)
        return c == 0 ? s.hc.ra[l][m] : c == 1 ? s.hc.rb[l][m] : c == 2 ? s.hc.dz[l][m] : c == 3 ? s.hc.dp[l][m] : c == 4 ? s.hc.dm[l][m] : s.hc.kl[l];
    else
        return ffa::F{s.hcf[c][l][m][0], s.hcf[c][l][m][1]};
}

// Entry m = mm - l of the harmonics of l from those of l - 1 and l - 2 (S1, S2) and, at m = +-l, from
// A + i B = (x + i y)^l (its rounding at the nodes of cos(l phi) and sin(l phi) is then that of the powers alone).
// FP64: the normalised S_lm. Float-float: T_lm = S_lm / N_lm, whose highest power of z has the coefficient 1 (T_ll =
// A or B), multiplied by N_lm where S_lm is used: with the normalisation in every step the errors of S_3m and S_4m
// were 15 and 7 % larger (5.6e-15 against 4.8e-15 of the norm for l = 3).
template <int l, typename H, int W>
__device__ __forceinline__ H harmonic(const DevSystem &s, const H (&x)[3], H r2, H A, H B, const H (&S1)[W], const H (&S2)[W],
                                      int mm) {
    const int m = mm >= l ? mm - l : l - mm, sg = mm >= l ? 1 : -1;
    if constexpr (std::is_same<H, double>::value) {
        if (m == l) return hmul(coef<H, 5>(s, l, 0), sg > 0 ? A : B);
        if constexpr (l == 1) return hmul(coef<H, 5>(s, 1, 0), x[2]);  // S_1m = kl (x, y, z): one rounding, not two
        const H az = hmul(coef<H, 0>(s, l, m), x[2]);
        if (m > l - 2) return hmul(az, S1[l - 1 + sg * m]);
        return hdot(az, S1[l - 1 + sg * m], hneg(hmul(coef<H, 1>(s, l, m), r2)), S2[l - 2 + sg * m]);
    } else {
        if (m == l) return sg > 0 ? A : B;
        if constexpr (l == 1) return x[2];
        if (m > l - 2) return hmul(x[2], S1[l - 1 + sg * m]);
        return hdot(x[2], S1[l - 1 + sg * m], hneg(hmul(coef<H, 1>(s, l, m), r2)), S2[l - 2 + sg * m]);
    }
}

// d/dx, d/dy or d/dz of S_lm: at most two harmonics of l - 1 (zero: none).
template <int l, typename H, int W>
__device__ __forceinline__ H harmonic_d(const DevSystem &s, const H (&C)[W], int mm, int axis, bool &zero) {
    const int m = mm >= l ? mm - l : l - mm, sg = mm >= l ? 1 : -1;
    constexpr int o = l - 1;
    if constexpr (l == 1) {  // a constant, kl = N_1m (the product of dz or dm and S_00 would be off in every value)
        zero = !(axis == 2 ? m == 0 : m == 1 && (axis == 0) == (sg > 0));
        if constexpr (std::is_same<H, double>::value) return zero ? H{} : coef<H, 5>(s, 1, 0);
        else return zero ? H{} : coef<H, 0>(s, 1, 0);
    }
    zero = false;
    if (axis == 2) {
        zero = m > l - 1;
        return zero ? H{} : hmul(coef<H, 2>(s, l, m), C[o + sg * m]);
    }
    const int t = axis == 0 ? sg : -sg;
    const bool up = m + 1 <= l - 1, down = m >= 1 && !(m == 1 && t < 0);
    H p{}, q{};
    if (up) p = axis == 1 && sg < 0 ? hneg(coef<H, 3>(s, l, m)) : coef<H, 3>(s, l, m);
    if (down) q = axis == 1 && sg > 0 ? hneg(coef<H, 4>(s, l, m)) : coef<H, 4>(s, l, m);
    zero = !up && !down;
    if (up && down) return hdot(p, C[o + t * (m + 1)], q, C[o + t * (m - 1)]);
    if (up) return hmul(p, C[o + t * (m + 1)]);
    return down ? hmul(q, C[o + t * (m - 1)]) : H{};
}

// Biased FP64 exponent of an upper bound of |v| (0: v is taken as zero): the exponent of v.h,
// plus one when v.h's significand is within 2^-15 of 2 (v.l may then carry |v| into the next
// binade). Subnormal v.h (|v| < 2^-126) counts as zero.
__device__ __forceinline__ int ff_bound_eb(ffa::F v) {
    const int b = __float_as_int(v.h) & 0x7FFFFFFF;
    const int e = b >> 23;
    if (e == 0) return 0;
    return e + 896 + ((b & 0x7FFFFF) >= 0x7FFF00 ? 1 : 0);
}

// A point's coordinates relative to one atom and what depends on them alone.
template <typename A>
struct Point {
    typename A::H x[3], r2;
    typename A::R t, xr[3], u, dr;  // xr: x in R; u: 1/r; dr: dR/ds -> dR/dr
    int k;                          // spline segment
    double r;
    ffa::F tf;                      // t as a float-float (F32: for the ill-conditioned segments)
};

// (phi, phi' / r as the factors of S) of one radial function: g and gpu = g'(r) / r.
template <typename A>
__device__ __forceinline__ void radial(const DevSystem &s, const Point<A> &pt, int fn, int l, typename A::R ul,
                                       typename A::R a_dr, typename A::R a_r, typename A::R &g, typename A::R &gpu) {
    const size_t seg = (size_t)fn * (s.n_rgrid - 1) + pt.k;
    if constexpr (std::is_same<A, F64>::value) {
        const double2 *c = reinterpret_cast<const double2 *>(s.coef + seg * 4);
        const double2 c01 = __ldg(c), c23 = __ldg(c + 1);
        // R = c0 + t (c1 + t a), dR/dt = c1 + t (2 a + c3 t), a = c2 + c3 t
        const double a = fma(c23.y, pt.t, c23.x);
        const double R = fma(fma(a, pt.t, c01.y), pt.t, c01.x);
        const double dRds = fma(fma(c23.y, pt.t, a + a), pt.t, c01.y);
        g = R * ul;
        // g'(r) / r = (dR/dr - l R / r) u^l / r
        gpu = l == 0 ? dRds * a_dr : fma(dRds, a_dr, -(R * a_r));
    } else if constexpr (std::is_same<A, F32>::value) {
        const float t = pt.t;
        float R, dRds;
        if (__ldg(s.seg64 + seg)) {
            // ill-conditioned segment: coefficients, t and polynomials as float-floats, rounded once (in FP64
            // they and a log1p per radial function took half of this path's evaluation: 64 atoms, phi and grad phi
            // 2.28 -> 1.19 ms, phi alone 1.78 -> 0.76)
            const float4 ch = __ldg(reinterpret_cast<const float4 *>(s.coef_f32 + seg * 4));
            const float4 cl = __ldg(reinterpret_cast<const float4 *>(s.coef_lo + seg * 4));
            const ffa::F c0{ch.x, cl.x}, c1{ch.y, cl.y}, c2{ch.z, cl.z}, c3{ch.w, cl.w};
            const ffa::F a = ffa::fma(c3, pt.tf, c2);
            R = ffa::fma(ffa::fma(a, pt.tf, c1), pt.tf, c0).h;
            dRds = ffa::fma(ffa::fma(c3, pt.tf, ffa::twice(a)), pt.tf, c1).h;
        } else {
            const float4 c = __ldg(reinterpret_cast<const float4 *>(s.coef_f32 + seg * 4));
            R = fmaf(fmaf(fmaf(c.w, t, c.z), t, c.y), t, c.x);
            dRds = fmaf(fmaf(3.0f * c.w, t, 2.0f * c.z), t, c.y);
        }
        g = R * ul;
        gpu = l == 0 ? dRds * a_dr : fmaf(dRds, a_dr, -(R * a_r));
    } else {
        const float4 ch = __ldg(reinterpret_cast<const float4 *>(s.coef_f32 + seg * 4));
        const float4 cl = __ldg(reinterpret_cast<const float4 *>(s.coef_lo + seg * 4));
        const ffa::F c0{ch.x, cl.x}, c1{ch.y, cl.y}, c2{ch.z, cl.z}, c3{ch.w, cl.w};
        const ffa::F a = ffa::fma(c3, pt.t, c2);
        const ffa::F R = ffa::fma(ffa::fma(a, pt.t, c1), pt.t, c0);
        const ffa::F dRds = ffa::fma(ffa::fma(c3, pt.t, ffa::twice(a)), pt.t, c1);
        g = ffa::mul(R, ul);
        gpu = l == 0 ? ffa::mul(dRds, a_dr) : ffa::dot2(dRds, a_dr, ffa::neg(R), a_r);
    }
}

// g S, and gx S + g G (zero: G is 0).
__device__ __forceinline__ double value(double g, double S) { return g * S; }
__device__ __forceinline__ float value(float g, ffa::F S) { return g * S.h; }
__device__ __forceinline__ ffa::F value(ffa::F g, ffa::F S) { return ffa::mul(g, S); }
__device__ __forceinline__ double slope(double gx, double S, double g, double G, bool zero) { return zero ? gx * S : gx * S + g * G; }
__device__ __forceinline__ float slope(float gx, ffa::F S, float g, ffa::F G, bool zero) {
    return zero ? gx * S.h : gx * S.h + g * G.h;
}
__device__ __forceinline__ ffa::F slope(ffa::F gx, ffa::F S, ffa::F g, ffa::F G, bool zero) {
    return zero ? ffa::mul(gx, S) : ffa::dot2(gx, S, g, G);
}
template <typename OutT, typename R>
__device__ __forceinline__ OutT out(R v) {
    if constexpr (std::is_same<R, ffa::F>::value && !std::is_same<OutT, FF2>::value) return OutT(ffa::to_double(v));
    else return OutT(v);
}
__device__ __forceinline__ int value_eb(FF2 v) { return ff_bound_eb(v.f()); }

__device__ __forceinline__ RfnEntry rfn_entry(const DevSystem &s, int ri) {
    const int4 v = __ldg(reinterpret_cast<const int4 *>(s.rfn + ri));
    return RfnEntry{v.x, v.y, v.z, v.w};
}

// The functions of l = L of one atom at one point, then those of L + 1 .. LMAX. The radial functions of an
// atom are visited in increasing l and share the harmonics; pa + i pb = (x + i y)^L, S1, S2: the harmonics of L - 1,
// L - 2 (in FP64 the normalised ones, as float-floats those divided by N_lm). ul: u^L.
template <int L, int LMAX, typename A, bool GRAD, typename OutT, int EXPO>
__device__ __forceinline__ void eval_level(const DevSystem &s, const AtomGroup &ag, int ri, const Point<A> &pt,
                                           typename A::R ul, typename A::H pa, typename A::H pb,
                                           const typename A::H (&S1)[2 * LMAX + 1],
                                           const typename A::H (&S2)[2 * LMAX + 1], const EvalOut<OutT> &o, int q, int &pt_eb) {
    using H = typename A::H;
    using R = typename A::R;
    H T[2 * LMAX + 1], S[2 * LMAX + 1], G[3][2 * LMAX + 1];
    bool zero[3][2 * LMAX + 1];
    if constexpr (L == 0) {
        if constexpr (std::is_same<H, double>::value) {
            T[0] = S[0] = s.s00;
        } else {
            T[0] = H{1.0f, 0.0f};
            S[0] = coef<H, 0>(s, 0, 0);
        }
        zero[0][0] = zero[1][0] = zero[2][0] = true;
    } else {
#pragma unroll
        for (int mm = 0; mm < 2 * L + 1; mm++) {
            T[mm] = harmonic<L>(s, pt.x, pt.r2, pa, pb, S1, S2, mm);
            if constexpr (std::is_same<H, double>::value) S[mm] = T[mm];
            else S[mm] = hmul(coef<H, 0>(s, L, mm >= L ? mm - L : L - mm), T[mm]);
            if (GRAD)
#pragma unroll
                for (int a = 0; a < 3; a++) G[a][mm] = harmonic_d<L>(s, S1, mm, a, zero[a][mm]);
        }
    }
    const int re = ag.r0 + ag.nr;
    R a_dr, a_r, ulu;
    if constexpr (std::is_same<R, ffa::F>::value) {
        ulu = L == 0 ? pt.u : ffa::mul(ul, pt.u);               // u^(l+1)
        a_dr = ffa::mul(pt.dr, ulu);                            // dR/ds -> g'(r)/r
        a_r = ffa::mulf(ffa::mul(pt.u, ulu), (float)L);         // R -> the l R / r part of g'(r)/r
    } else {
        ulu = ul * pt.u;
        a_dr = pt.dr * ulu;
        a_r = R(L) * pt.u * ulu;
    }
    // the entries and cutoffs by read-only loads, which the stores cannot hold back, one entry ahead
    RfnEntry next = ri < re ? rfn_entry(s, ri) : RfnEntry{0, 0, 0, -1};
    for (; next.l == L;) {
        const RfnEntry e = next;
        const double rc = __ldg(s.fn_rc + e.fn);
        ri++;
        next = ri < re ? rfn_entry(s, ri) : RfnEntry{0, 0, 0, -1};
        OutT *row = o.phi + (int64_t)e.pos * o.phi_rs + q;
        OutT *gr = GRAD ? o.grad + (int64_t)e.pos * o.grad_rs + q : nullptr;
        // r < rc, both non-negative: their bit patterns order alike (the FP64 pipe is the scarce one)
        if (__double_as_longlong(pt.r) < __double_as_longlong(rc)) {
            R g, gpu, gx[3];
            radial<A>(s, pt, e.fn, L, ul, a_dr, a_r, g, gpu);
            if (GRAD)
#pragma unroll
                for (int a = 0; a < 3; a++) {
                    if constexpr (std::is_same<R, ffa::F>::value) gx[a] = ffa::mul(gpu, pt.xr[a]);
                    else gx[a] = gpu * pt.xr[a];
                }
#pragma unroll
            for (int mm = 0; mm < 2 * L + 1; mm++) {
                const OutT f = out<OutT>(value(g, S[mm]));
                if constexpr (EXPO == 1) pt_eb = max(pt_eb, value_eb(f));
                row[mm * o.phi_rs] = f;
                if (GRAD)
#pragma unroll
                    for (int a = 0; a < 3; a++)
                        gr[mm * o.grad_rs + a * o.grad_cs] = out<OutT>(slope(gx[a], S[mm], g, G[a][mm], zero[a][mm]));
            }
        } else {
#pragma unroll
            for (int mm = 0; mm < 2 * L + 1; mm++) {
                row[mm * o.phi_rs] = OutT(0);
                if (GRAD)
#pragma unroll
                    for (int a = 0; a < 3; a++) gr[mm * o.grad_rs + a * o.grad_cs] = OutT(0);
            }
        }
    }
    if constexpr (L < LMAX) {
        if (ri < re) {
            R un;
            if constexpr (std::is_same<R, ffa::F>::value) un = ulu;
            else un = ul * pt.u;
            const H na = L == 0 ? pt.x[0] : hdot(pt.x[0], pa, hneg(pt.x[1]), pb);
            const H nb = L == 0 ? pt.x[1] : hdot(pt.x[0], pb, pt.x[1], pa);
            eval_level<L + 1, LMAX, A, GRAD, OutT, EXPO>(s, ag, ri, pt, un, na, nb, T, S1, o, q, pt_eb);
        }
    }
}

// All relevant radial functions of one atom at one point.
template <int LMAX, typename A, bool GRAD, typename OutT, int EXPO>
__device__ __forceinline__ void eval_group(const DevSystem &s, const AtomGroup &ag, double dx, double dy, double dz, double r2,
                                           double r, double ur, const EvalOut<OutT> &o, int q, const ExpoIn &xi) {
    using H = typename A::H;
    using R = typename A::R;
    Point<A> pt;
    const double rr = fmax(r, s.r0);
    const double dr = s.inv_delta * (r < s.r0 ? __ldg(s.inv_rk) : ur);  // dR/dr = dR/ds * inv_delta / rr
    pt.r = r;
    pt.tf = ffa::F{0.0f, 0.0f};
    if constexpr (std::is_same<A, F32>::value) {
        // FP32 segment, refined as ln(r / r_k)/Delta = log1p(r * (1/r_k) - 1)/Delta with one FP64
        // FMA: t keeps ~1e-7 although a plain FP32 ln(r/r0) carries ~1e-6.
        const float sa = __logf((float)rr * (float)(1.0 / s.r0)) * (float)s.inv_delta;
        int k = (int)floorf(sa);
        k = k < 0 ? 0 : (k > s.n_rgrid - 2 ? s.n_rgrid - 2 : k);
        pt.k = k;
        const double xk = fma(rr, __ldg(s.inv_rk + k), -1.0);
        pt.t = log1pf((float)xk) * (float)s.inv_delta;
        pt.tf = ffa::from_double_bits(log1p_small(xk, s.step_m1) * s.inv_delta);
        pt.u = float(ur);
        pt.dr = float(dr);
    } else {
        const double t = radial_coordinate(s, rr, pt.k);
        pt.t = from_f64<R>(t);
        pt.u = from_f64<R>(ur);
        pt.dr = from_f64<R>(dr);
    }
    pt.x[0] = from_f64<H>(dx);
    pt.x[1] = from_f64<H>(dy);
    pt.x[2] = from_f64<H>(dz);
    pt.r2 = from_f64<H>(r2);
    if constexpr (std::is_same<A, F32>::value) {
#pragma unroll
        for (int a = 0; a < 3; a++) pt.xr[a] = pt.x[a].h;
    } else {
#pragma unroll
        for (int a = 0; a < 3; a++) pt.xr[a] = pt.x[a];
    }
    const H none[2 * LMAX + 1] = {};
    R one;
    if constexpr (std::is_same<R, ffa::F>::value) one = ffa::F{1.0f, 0.0f};
    else one = R(1);
    int pt_eb = 0;  // EXPO 1: largest biased exponent of phi at this point
    eval_level<0, LMAX, A, GRAD, OutT, EXPO>(s, ag, ag.r0, pt, one, H{}, H{}, none, none, o, q, pt_eb);  // (x + i y)^0 is not read
    if constexpr (EXPO == 1) {
        if (pt_eb > 0) atomicMax(xi.red + (q - xi.q0), pt_eb);
    }
}

// The FP64 evaluation of the few points near a nucleus, out of line so that its registers are not the
// others'.
template <int LMAX, bool GRAD, typename OutT, int EXPO>
__device__ __noinline__ void eval_group_near(const DevSystem &s, const AtomGroup &ag, double dx, double dy, double dz, double r2,
                                             double r, double ur, const EvalOut<OutT> &o, int q, const ExpoIn &xi) {
    eval_group<LMAX, F64, GRAD, OutT, EXPO>(s, ag, dx, dy, dz, r2, r, ur, o, q, xi);
}

template <typename A>
struct out_of;
template <>
struct out_of<F64> {
    using type = double;
};
template <>
struct out_of<F32> {
    using type = float;
};
template <>
struct out_of<FF> {
    using type = FF2;
};

constexpr int kEvalPoints = 64, kEvalThreads = 128;  // points and threads of a CTA

// The points [q0, q0 + kEvalPoints) of batch b and all its atoms: a warp takes one atom and 32 points at a
// time, so its lanes share the radial functions' entries and write 32 consecutive values of a row.
// LMAX: at least the largest l of the handle's functions.
template <int LMAX, bool GRAD, typename A, int EXPO, typename OutT>
__device__ __forceinline__ void eval_tile(const DevSystem &s, int b, int q0, const EvalOut<OutT> &o, int *red = nullptr) {
    const int p0 = s.batch_off[b], P = s.batch_off[b + 1] - p0;
    const int g0 = s.agrp_off[b], ng = s.agrp_off[b + 1] - g0;
    const ExpoIn xi{red, q0};
    const int half = o.qmax - q0 > 32 ? 2 : 1;  // sets of 32 points
    for (int idx = threadIdx.x >> 5; idx < half * ng; idx += kEvalThreads / 32) {
        const int gl = idx / half, q = q0 + 32 * (idx - gl * half) + (int)(threadIdx.x & 31);
        if (q >= o.qmax) continue;
        const AtomGroup ag = s.agrp[g0 + gl];
        if (q >= P) {  // padding points: zero rows
            for (int ri = ag.r0; ri < ag.r0 + ag.nr; ri++) {
                const RfnEntry e = s.rfn[ri];
                for (int j = e.pos; j < e.pos + 2 * e.l + 1; j++) {
                    o.phi[(int64_t)j * o.phi_rs + q] = OutT(0);
                    if (GRAD)
                        for (int a = 0; a < 3; a++) o.grad[a * o.grad_cs + (int64_t)j * o.grad_rs + q] = OutT(0);
                }
            }
            continue;
        }
        const int p = p0 + q;
        const double dx = __dsub_rn(s.px[p], s.atom_xyz[3 * ag.atom]);
        const double dy = __dsub_rn(s.py[p], s.atom_xyz[3 * ag.atom + 1]);
        const double dz = __dsub_rn(s.pz[p], s.atom_xyz[3 * ag.atom + 2]);
        const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
        // 1/r from the library's reciprocal square root (about one ulp) and r = r^2 (1/r): one
        // FP64 function instead of a square root and a division
        const double ur = rsqrt(r2);
        const double r = r2 > 0.0 ? r2 * ur : 0.0;
        if constexpr (std::is_same<A, F64>::value) {
            eval_group<LMAX, F64, GRAD, OutT, EXPO>(s, ag, dx, dy, dz, r2, r, ur, o, q, xi);
        } else {
            constexpr int LA = std::is_same<A, FF>::value && LMAX > 4 ? 4 : LMAX;
            if (r < kNearNucleus || ag.lmax > LA)
                eval_group_near<LMAX, GRAD, OutT, EXPO>(s, ag, dx, dy, dz, r2, r, ur, o, q, xi);
            else
                eval_group<LA, A, GRAD, OutT, EXPO>(s, ag, dx, dy, dz, r2, r, ur, o, q, xi);
        }
    }
}

template <bool GRAD, typename T>
__device__ __forceinline__ EvalOut<T> batch_out(const DevSystem &s, int b, int Ppad, T *scratch) {
    EvalOut<T> o;
    o.phi = scratch + s.scr_off[b];
    o.qmax = Ppad;
    if (GRAD) {
        o.phi_rs = 4 * (int64_t)Ppad;
        o.grad = o.phi + Ppad;
        o.grad_cs = Ppad;
        o.grad_rs = 4 * (int64_t)Ppad;
    } else {
        o.phi_rs = Ppad;
        o.grad = nullptr;
        o.grad_cs = o.grad_rs = 0;
    }
    return o;
}

// One CTA per (batch, 64-point tile); the batch's block of scratch holds, per reduced-basis row j,
// [phi | d/dx | d/dy | d/dz] over Ppad points each (GRAD) or phi alone, in A's output type.
// Bound by latency and instruction fetch (dependent float-float or FP64 chains in long unrolled code; 128
// registers, four CTAs per SM). 45-atom slab, float-float: phi and grad phi 5.15 -> 2.96 ms, phi alone 1.75 ->
// 1.21 ms, against one CTA of 256 threads and 255 registers per batch, with the argument block copied to every
// thread's stack and derivative recurrences for the harmonics; a 21-atom molecule (227 batches) 0.59 -> 0.28 ms,
// as the tiles also spread a small system over the SMs.
template <int LMAX, bool GRAD, typename A>
__global__ void __launch_bounds__(kEvalThreads) eval_chunk_kernel(const __grid_constant__ DevSystem s, int32_t b0,
                                                                 typename out_of<A>::type *scratch) {
    using OutT = typename out_of<A>::type;
    const int b = b0 + blockIdx.x, q0 = blockIdx.y * kEvalPoints;
    const int P = s.batch_off[b + 1] - s.batch_off[b];
    const int Ppad = (P + NAO_PPAD - 1) & ~(NAO_PPAD - 1);
    if (q0 < Ppad) eval_tile<LMAX, GRAD, A, 0>(s, b, q0, batch_out<GRAD, OutT>(s, b, Ppad, scratch));
}

// The density's evaluation on the split path (float-float, FF2 values): as eval_chunk_kernel,
// and the point exponents of the slicing: expo[batch_off[b] + q] = the exponent of point q, from
// the binade of an upper bound of max_i |phi_iq| (split_bits::exponent_of_binade); expo_b[b] = 0, where
// slice_nphi_kernel reduces the exponent of P'.
template <int LMAX, bool GRAD>
__global__ void __launch_bounds__(kEvalThreads) eval_split_kernel(const __grid_constant__ DevSystem s, int32_t b0, FF2 *scratch,
                                                                 int32_t *expo, int32_t *expo_b) {
    __shared__ int red[kEvalPoints];
    const int b = b0 + blockIdx.x, q0 = blockIdx.y * kEvalPoints;
    const int p0 = s.batch_off[b], P = s.batch_off[b + 1] - p0;
    const int Ppad = (P + NAO_PPAD - 1) & ~(NAO_PPAD - 1);
    if (blockIdx.y == 0 && threadIdx.x == 0) expo_b[b] = 0;
    if (q0 >= Ppad) return;
    for (int i = threadIdx.x; i < kEvalPoints; i += kEvalThreads) red[i] = 0;
    __syncthreads();
    eval_tile<LMAX, GRAD, FF, 1>(s, b, q0, batch_out<GRAD, FF2>(s, b, Ppad, scratch), red);
    __syncthreads();
    for (int q = q0 + (int)threadIdx.x; q < min(P, q0 + kEvalPoints); q += kEvalThreads)
        expo[p0 + q] = split_bits::exponent_of_binade(red[q - q0]);
}

template <bool GRAD, typename A>
__global__ void __launch_bounds__(kEvalThreads) eval_export_kernel(const __grid_constant__ DevSystem s, int32_t b, double *phi,
                                                                  double *grad) {
    const int P = s.batch_off[b + 1] - s.batch_off[b];
    const int N = s.rel_off[b + 1] - s.rel_off[b];
    EvalOut<double> o;
    o.phi = phi;
    o.phi_rs = P;
    o.grad = grad;
    o.grad_cs = (int64_t)N * P;
    o.grad_rs = P;
    o.qmax = P;
    const int q0 = blockIdx.x * kEvalPoints;
    if (q0 < P) eval_tile<NAO_LMAX, GRAD, A, 0>(s, b, q0, o);
}

// 64-point tiles of the handle's largest batch.
unsigned eval_tiles(const DevSystem &s) { return (unsigned)((s.max_ppad + kEvalPoints - 1) / kEvalPoints); }

}  // namespace

// CALL(LMAX) with the smallest instantiated LMAX >= the handle's largest l.
#define NAO_LMAX_DISPATCH(lmax, CALL) \
    switch (lmax) {                   \
        case 0:                       \
        case 1:                       \
        case 2: CALL(2); break;       \
        case 3: CALL(3); break;       \
        case 4: CALL(4); break;       \
        default: CALL(NAO_LMAX); break; \
    }

cudaError_t launch_relevance_minr2(const double *atom_xyz, const int32_t *bmol, const int32_t *aoff, int32_t max_atoms,
                                   const double *px, const double *py, const double *pz, const int32_t *batch_off,
                                   int64_t n_batches, double *minr2, cudaStream_t st) {
    if (n_batches <= 0) return cudaSuccess;
    minr2_kernel<<<(unsigned)n_batches, 256, 0, st>>>(atom_xyz, bmol, aoff, max_atoms, px, py, pz, batch_off, minr2);
    return cudaGetLastError();
}

template <bool GRAD, typename A>
static cudaError_t launch_eval_t(const DevSystem &s, int32_t b0, int32_t b1, double *scratch, cudaStream_t st) {
    auto *out = reinterpret_cast<typename out_of<A>::type *>(scratch);
#define NAO_EVAL(L) eval_chunk_kernel<L, GRAD, A><<<dim3(b1 - b0, eval_tiles(s)), kEvalThreads, 0, st>>>(s, b0, out)
    NAO_LMAX_DISPATCH(s.lmax, NAO_EVAL)
#undef NAO_EVAL
    return cudaGetLastError();
}

cudaError_t launch_eval(const DevSystem &s, int32_t b0, int32_t b1, nao_precision prec, bool grad, double *scratch,
                        cudaStream_t st) {
    if (b1 <= b0) return cudaSuccess;
    if (prec == NAO_FP32) return grad ? launch_eval_t<true, F32>(s, b0, b1, scratch, st) : launch_eval_t<false, F32>(s, b0, b1, scratch, st);
    if (prec == NAO_SPLIT) return grad ? launch_eval_t<true, FF>(s, b0, b1, scratch, st) : launch_eval_t<false, FF>(s, b0, b1, scratch, st);
    return grad ? launch_eval_t<true, F64>(s, b0, b1, scratch, st) : launch_eval_t<false, F64>(s, b0, b1, scratch, st);
}

cudaError_t launch_eval_split(const DevSystem &s, int32_t b0, int32_t b1, bool grad, double *scratch, int32_t *expo,
                              int32_t *expo_b, cudaStream_t st) {
    if (b1 <= b0) return cudaSuccess;
    const dim3 grid(b1 - b0, eval_tiles(s));
    FF2 *f = reinterpret_cast<FF2 *>(scratch);
#define NAO_EVAL_G(L) eval_split_kernel<L, true><<<grid, kEvalThreads, 0, st>>>(s, b0, f, expo, expo_b)
#define NAO_EVAL_P(L) eval_split_kernel<L, false><<<grid, kEvalThreads, 0, st>>>(s, b0, f, expo, expo_b)
    if (grad) {
        NAO_LMAX_DISPATCH(s.lmax, NAO_EVAL_G)
    } else {
        NAO_LMAX_DISPATCH(s.lmax, NAO_EVAL_P)
    }
#undef NAO_EVAL_G
#undef NAO_EVAL_P
    return cudaGetLastError();
}

cudaError_t launch_eval_one(const DevSystem &s, int32_t b, nao_precision prec, double *phi, double *grad,
                            cudaStream_t st) {
    if (prec == NAO_FP32) {
        if (grad) eval_export_kernel<true, F32><<<eval_tiles(s), kEvalThreads, 0, st>>>(s, b, phi, grad);
        else eval_export_kernel<false, F32><<<eval_tiles(s), kEvalThreads, 0, st>>>(s, b, phi, nullptr);
    } else if (prec == NAO_SPLIT) {
        if (grad) eval_export_kernel<true, FF><<<eval_tiles(s), kEvalThreads, 0, st>>>(s, b, phi, grad);
        else eval_export_kernel<false, FF><<<eval_tiles(s), kEvalThreads, 0, st>>>(s, b, phi, nullptr);
    } else {
        if (grad) eval_export_kernel<true, F64><<<eval_tiles(s), kEvalThreads, 0, st>>>(s, b, phi, grad);
        else eval_export_kernel<false, F64><<<eval_tiles(s), kEvalThreads, 0, st>>>(s, b, phi, nullptr);
    }
    return cudaGetLastError();
}
