// Density Hessian on the FP64 and FP32 paths (Sec. 2: the six second derivatives of Eq. Density
// needed for forces and stresses, each a "straightforward extension" of the density).
//
// For symmetric P, differentiating n = sum_ij phi_i P_ij phi_j twice gives
//   d_a d_b n = 2 sum_ij P_ij (phi_i d_a d_b phi_j + d_a phi_i d_b phi_j),
// so per batch, with T = Phi P and T_a = (d_a Phi) P over the batch's reduced basis,
//   d_a d_b n_q = 2 sum_j (T_qj d_a d_b phi_qj + T_a,qj d_b phi_qj),
// and the same pass gives n_q = sum_j T_qj phi_qj and d_a n_q = 2 sum_j T_qj d_a phi_qj.
//
// Evaluation: four CTAs per batch, one thread per (point, atom); phi = g(r) S_lm with g = R / r^l and
// S_lm the normalised real solid harmonic:
//   d_a phi     = g' (x_a / r) S + g d_a S,
//   d_a d_b phi = (g'' / r^2 - g' / r^3) x_a x_b S + (g' / r)(delta_ab S + x_b d_a S + x_a d_b S)
//                 + g d_a d_b S,
//   g' = R' / r^l - l R / r^(l+1),  g'' = R'' / r^l - 2 l R' / r^(l+1) + l (l+1) R / r^(l+2),
// with R' and R'' from the spline in s = ln(r / r0) / Delta (ds/dr = 1 / (r Delta),
// d^2s/dr^2 = -1 / (r^2 Delta), all at r0 where r < r0). The harmonics of l come from those of l - 1 and
// l - 2, and their derivatives are fixed combinations of at most two harmonics of l - 1 (the second ones
// of the first ones of l - 1), so that an entry takes 3 + 5 + 9 FP64 operations. Every batch's block of scratch holds,
// per reduced-basis row, 10 rows of Ppad points: phi, d/dx, d/dy, d/dz, xx, xy, xz, yy, yz, zz, in the
// path's type T (the values are computed in FP64 on both paths; the FP32 path rounds them once when
// storing). For the Pulay terms (LAP) the fifth row holds the Laplacian instead: S is harmonic and
// homogeneous of degree l, so lap phi = (g'' + (2 l + 2) g' / r) S, and no second derivative is formed.
// Bound by the FP64 pipe, so powers of 1/r replace divisions. Per call, against recurrences for the derivatives
// of Pi(z, r^2) with divisions: 13-atom molecule (76,050 points) 5.28 -> 1.92 ms, with the Laplacian (9 atoms,
// 19,440 points) 3.17 -> 0.43 ms.
//
// Contraction: one CTA per 64-point density tile; for each 64-function tile J the four
// products Phi P, (d_x Phi) P, (d_y Phi) P, (d_z Phi) P over all of K in T (P read from its
// upper triangle, so the matrix used is exactly symmetric), then the epilogue above in T, the
// per-tile sums added in FP64. Every point is written once (no atomics).
#include "nao_internal.h"
#include "radial.h"

namespace {

constexpr int HR = 10;       // rows per basis function in the Hessian scratch
constexpr int TQ = NAO_TILE; // 64 points per density tile
constexpr int TJ = 64;       // functions per tile
constexpr int KC = 8;        // K chunk of the contraction

// (xx, xy, xz, yy, yz, zz)
__device__ __forceinline__ int pair_a(int k) { return k < 3 ? 0 : (k < 5 ? 1 : 2); }
__device__ __forceinline__ int pair_b(int k) { return k == 0 ? 0 : k == 1 ? 1 : k == 2 ? 2 : k == 3 ? 1 : 2; }

// d/dx, d/dy, d/dz of the entry +-m of harmonics l from the entries C of l - 1 (index l - 1 + m), or of
// their gradients where C holds one component of those.
template <int l, int LM>
__device__ __forceinline__ double harmonic_d(const DevSystem &s, const double (&C)[2 * LM + 1], int mm, int axis) {
    // mm: 0 .. 2 l, the entry m = mm - l (m >= 0: the cosine part); a compile-time constant once unrolled
    const int m = mm >= l ? mm - l : l - mm, sg = mm >= l ? 1 : -1;
    constexpr int o = l - 1;
    if (axis == 2) return m <= l - 1 ? s.hc.dz[l][m] * C[o + sg * m] : 0.0;
    // d/dx: the same part of m + 1 and m - 1; d/dy: the other part
    const int t = axis == 0 ? sg : -sg;
    const double p = axis == 0 ? s.hc.dp[l][m] : (sg > 0 ? s.hc.dp[l][m] : -s.hc.dp[l][m]);
    const double q = axis == 0 ? s.hc.dm[l][m] : (sg > 0 ? -s.hc.dm[l][m] : s.hc.dm[l][m]);
    // m = 0 has no sine part: S_l0 has d/dx from +1 and d/dy from -1 with dp alone
    const bool up = m + 1 <= l - 1, down = m >= 1 && !(m == 1 && t < 0);
    if (up && down) return fma(p, C[o + t * (m + 1)], q * C[o + t * (m - 1)]);
    if (up) return p * C[o + t * (m + 1)];
    return down ? q * C[o + t * (m - 1)] : 0.0;
}

// All functions of l = L of one atom at one point, and then of L + 1, .. LMAX. A + i B = (x + i y)^L;
// S1, S2: harmonics of L - 1 and L - 2; G1: their gradients for L - 1.
template <int L, int LMAX, typename OutT, bool LAP>
struct HessLevel {
    static __device__ __forceinline__ void run(const DevSystem &s, const AtomGroup &ag, int &ri, const double (&xa)[3],
                                               double r2, double r, double ur, double ur0, double ul, int k, double t, double ds1,
                                               double A, double B,
                                               const double (&S1)[2 * LMAX + 1], const double (&S2)[2 * LMAX + 1],
                                               const double (&G1)[3][2 * LMAX + 1], OutT *E, int64_t rs, int64_t cs, int q) {
        double S[2 * LMAX + 1], G[3][2 * LMAX + 1], H[6][2 * LMAX + 1];
        if constexpr (L == 0) {
            S[0] = s.s00;
            G[0][0] = G[1][0] = G[2][0] = 0.0;
#pragma unroll
            for (int kk = 0; kk < 6; kk++) H[kk][0] = 0.0;
        } else {
            S[2 * L] = s.hc.kl[L] * A;
            S[0] = s.hc.kl[L] * B;
#pragma unroll
            for (int m = 0; m < L; m++) {
                const double az = s.hc.ra[L][m] * xa[2];
                const double bq = m <= L - 2 ? s.hc.rb[L][m] * r2 : 0.0;
#pragma unroll
                for (int sg = 1; sg >= (m == 0 ? 1 : -1); sg -= 2) {
                    const double v = L == 1 ? s.hc.kl[1] * xa[2] : az * S1[L - 1 + sg * m];  // S_1m = kl (x, y, z)
                    S[L + sg * m] = m <= L - 2 ? fma(-bq, S2[L - 2 + sg * m], v) : v;
                }
            }
#pragma unroll
            for (int mm = 0; mm < 2 * L + 1; mm++) {
#pragma unroll
                for (int a = 0; a < 3; a++)
                    G[a][mm] = L > 1 ? harmonic_d<L, LMAX>(s, S1, mm, a) : mm == (a == 0 ? 2 : a == 1 ? 0 : 1) ? s.hc.kl[1] : 0.0;
                if (!LAP) {
#pragma unroll
                    for (int kk = 0; kk < 6; kk++) H[kk][mm] = harmonic_d<L, LMAX>(s, G1[pair_a(kk)], mm, pair_b(kk));
                }
            }
        }
        for (; ri < ag.r0 + ag.nr; ri++) {
            const RfnEntry e = s.rfn[ri];
            if (e.l != L) break;
            OutT *row = E + (int64_t)e.pos * rs + q;
            double g = 0.0, G1r = 0.0, Q = 0.0, lapr = 0.0;  // g, g'/r, g''/r^2 - g'/r^3, the Laplacian's factor of S
            if (r < s.fn_rc[e.fn]) {
                const double2 *c = reinterpret_cast<const double2 *>(s.coef + ((size_t)e.fn * (s.n_rgrid - 1) + k) * 4);
                const double2 c01 = __ldg(c), c23 = __ldg(c + 1);
                const double a = fma(c23.y, t, c23.x);
                const double R = fma(fma(a, t, c01.y), t, c01.x);
                const double Rs = fma(fma(c23.y, t, a + a), t, c01.y);
                const double Rss = fma(6.0 * c23.y, t, 2.0 * c23.x);
                const double R1 = Rs * ds1, R2 = ds1 * fma(Rss, ds1, -(Rs * ur0));  // d^2s/dr^2 = -ds/dr / max(r, r0)
                g = R * ul;
                const double lr = (double)L * ur;
                const double g1 = fma(-lr, R, R1) * ul;
                const double g2 = fma(-2.0 * lr, R1, fma((double)(L * (L + 1)) * ur * ur, R, R2)) * ul;
                G1r = g1 * ur;
                if (LAP) lapr = fma((double)(2 * L + 2), G1r, g2);
                else Q = (g2 - G1r) * (ur * ur);
            }
            const double gx[3] = {G1r * xa[0], G1r * xa[1], G1r * xa[2]};
            double Qab[6];
            if (!LAP) {
#pragma unroll
                for (int kk = 0; kk < 6; kk++) {
                    const double v = Q * xa[pair_a(kk)];
                    Qab[kk] = pair_a(kk) == pair_b(kk) ? fma(v, xa[pair_b(kk)], G1r) : v * xa[pair_b(kk)];
                }
            }
#pragma unroll
            for (int mm = 0; mm < 2 * L + 1; mm++, row += rs) {
                const double Sv = S[mm];
                row[0] = OutT(g * Sv);
#pragma unroll
                for (int a = 0; a < 3; a++) row[(1 + a) * cs] = OutT(L == 0 ? gx[a] * Sv : fma(gx[a], Sv, g * G[a][mm]));
                if (LAP) {
                    row[4 * cs] = OutT(lapr * Sv);
                } else {
#pragma unroll
                    for (int kk = 0; kk < 6; kk++) {
                        const int a = pair_a(kk), b = pair_b(kk);
                        double v = Qab[kk] * Sv;
                        if (L >= 1) v = fma(gx[b], G[a][mm], fma(gx[a], G[b][mm], v));
                        if (L >= 2) v = fma(g, H[kk][mm], v);
                        row[(4 + kk) * cs] = OutT(v);
                    }
                }
            }
        }
        if constexpr (L < LMAX) {
            if (ri < ag.r0 + ag.nr)
                HessLevel<L + 1, LMAX, OutT, LAP>::run(s, ag, ri, xa, r2, r, ur, ur0, ul * ur, k, t, ds1,
                                                       L == 0 ? xa[0] : fma(xa[0], A, -(xa[1] * B)),
                                                       L == 0 ? xa[1] : fma(xa[0], B, xa[1] * A), S, S1, G, E, rs, cs, q);
        }
    }
};

template <int LMAX, typename OutT, bool LAP>
__device__ __forceinline__ void eval_group_hess(const DevSystem &s, const AtomGroup &ag, double x, double y, double z,
                                                OutT *E, int64_t rs, int64_t cs, int q) {
    const double xa[3] = {x, y, z};
    const double r2 = fma(x, x, fma(y, y, z * z)), ur = rsqrt(r2), r = r2 * ur;
    // for r < r0 R, R' and R'' are those at r0: both factors of d^2s/dr^2 take the clamped 1/r (ur0), while the
    // powers of 1/r of phi = (R / r^l) S are those of r itself (ur)
    const double rr = fmax(r, s.r0);
    int k;
    const double t = radial_coordinate(s, rr, k);
    const double ur0 = r < s.r0 ? 1.0 / s.r0 : ur;
    const double zero[2 * LMAX + 1] = {}, zero3[3][2 * LMAX + 1] = {};
    int ri = ag.r0;
    HessLevel<0, LMAX, OutT, LAP>::run(s, ag, ri, xa, r2, r, ur, ur0, 1.0, k, t, s.inv_delta * ur0, 1.0, 0.0, zero, zero, zero3, E,
                                       rs, cs, q);
}

// LMAX: at least the largest l of the handle's functions.
template <int LMAX, typename OutT, bool LAP>
__global__ void __launch_bounds__(128) eval_hess_kernel(const __grid_constant__ DevSystem s, int32_t b0,
                                                       OutT *__restrict__ scratch, const int64_t *__restrict__ hoff) {
    const int b = b0 + blockIdx.x;
    const int p0 = s.batch_off[b], P = s.batch_off[b + 1] - p0;
    const int Ppad = (P + NAO_PPAD - 1) & ~(NAO_PPAD - 1);
    const int g0 = s.agrp_off[b], ng = s.agrp_off[b + 1] - g0;
    OutT *E = scratch + hoff[b];
    const int64_t rs = (int64_t)HR * Ppad, cs = Ppad;
    for (int idx = blockIdx.y * blockDim.x + threadIdx.x; idx < ng * Ppad; idx += gridDim.y * blockDim.x) {
        const int gl = idx / Ppad, q = idx - gl * Ppad;
        const AtomGroup ag = s.agrp[g0 + gl];
        if (q >= P) {  // padding points: zero rows
            for (int ri = ag.r0; ri < ag.r0 + ag.nr; ri++) {
                const RfnEntry e = s.rfn[ri];
                for (int mm = 0; mm < 2 * e.l + 1; mm++)
                    for (int c = 0; c < (LAP ? 5 : HR); c++) E[(int64_t)(e.pos + mm) * rs + c * cs + q] = OutT(0);
            }
            continue;
        }
        const int p = p0 + q;
        eval_group_hess<LMAX, OutT, LAP>(s, ag, s.px[p] - s.atom_xyz[3 * ag.atom], s.py[p] - s.atom_xyz[3 * ag.atom + 1],
                                         s.pz[p] - s.atom_xyz[3 * ag.atom + 2], E, rs, cs, q);
    }
}

template <typename T>
__global__ void __launch_bounds__(256) density_hess_kernel(DevSystem s, const DWork *__restrict__ work, int32_t w0,
                                                          const T *__restrict__ scratch,
                                                          const int64_t *__restrict__ hoff, double *__restrict__ hess,
                                                          double *__restrict__ ne_part) {
    __shared__ __align__(16) T As[4][KC][TQ];  // phi, d/dx, d/dy, d/dz of rows i, at the tile's points
    __shared__ __align__(16) T Bs[KC][TJ];     // P[rel_i][rel_j]
    __shared__ double acc_n[TQ], acc_g[3][TQ], acc_h[6][TQ];
    __shared__ double red[8];
    const DWork it = work[w0 + blockIdx.x];
    const int b = it.batch, m = s.sys.bmol[b];
    const int p0 = s.batch_off[b], P = s.batch_off[b + 1] - p0;
    const int Ppad = (P + NAO_PPAD - 1) & ~(NAO_PPAD - 1);
    const int N = s.rel_off[b + 1] - s.rel_off[b];
    const int q0 = it.tp * TQ;
    const T *E = scratch + hoff[b];
    const int64_t ld = (int64_t)HR * Ppad;
    const int32_t *rel = s.rel_idx + s.rel_off[b];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    if (tid < TQ) {
        acc_n[tid] = 0.0;
        for (int c = 0; c < 3; c++) acc_g[c][tid] = 0.0;
        for (int c = 0; c < 6; c++) acc_h[c][tid] = 0.0;
    }
    const int nt = (N + TJ - 1) / TJ;
    for (int tj = 0; tj < nt; tj++) {
        T Tm[4][4][4];
#pragma unroll
        for (int c = 0; c < 4; c++)
#pragma unroll
            for (int a = 0; a < 4; a++)
#pragma unroll
                for (int d = 0; d < 4; d++) Tm[c][a][d] = T(0);
        for (int i0 = 0; i0 < N; i0 += KC) {
            __syncthreads();
            for (int u = tid; u < 4 * KC * TQ; u += blockDim.x) {
                const int c = u / (KC * TQ), kk = (u / TQ) % KC, qq = u % TQ;
                const int i = i0 + kk, q = q0 + qq;
                As[c][kk][qq] = (i < N && q < Ppad) ? E[(int64_t)i * ld + (int64_t)c * Ppad + q] : T(0);
            }
            for (int u = tid; u < KC * TJ; u += blockDim.x) {
                const int kk = u / TJ, jj = u % TJ;
                const int i = i0 + kk, j = tj * TJ + jj;
                double pv = 0.0;
                if (i < N && j < N) {
                    int64_t gi = rel[i], gj = rel[j];
                    if (gi > gj) { const int64_t tt = gi; gi = gj; gj = tt; }
                    pv = p_elem(s, m, gi, gj);
                }
                Bs[kk][jj] = T(pv);
            }
            __syncthreads();
#pragma unroll
            for (int kk = 0; kk < KC; kk++) {
                T rb[4];
#pragma unroll
                for (int d = 0; d < 4; d++) rb[d] = Bs[kk][tx * 4 + d];
#pragma unroll
                for (int c = 0; c < 4; c++)
#pragma unroll
                    for (int a = 0; a < 4; a++) {
                        const T ra = As[c][kk][ty * 4 + a];
#pragma unroll
                        for (int d = 0; d < 4; d++) Tm[c][a][d] = fma(ra, rb[d], Tm[c][a][d]);
                    }
            }
        }
        // epilogue: rows q = q0 + ty*4 + a, columns j = tj*64 + tx*4 + d
#pragma unroll
        for (int a = 0; a < 4; a++) {
            const int q = q0 + ty * 4 + a;
            T pn = T(0), pg[3] = {T(0), T(0), T(0)}, ph[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};
#pragma unroll
            for (int d = 0; d < 4; d++) {
                const int j = tj * TJ + tx * 4 + d;
                if (j < N && q < Ppad) {
                    const T *f = E + (int64_t)j * ld + q;
                    T fv[HR];
#pragma unroll
                    for (int c = 0; c < HR; c++) fv[c] = f[(int64_t)c * Ppad];
                    pn = fma(Tm[0][a][d], fv[0], pn);
#pragma unroll
                    for (int c = 0; c < 3; c++) pg[c] = fma(Tm[0][a][d], fv[1 + c], pg[c]);
#pragma unroll
                    for (int kk = 0; kk < 6; kk++)
                        ph[kk] = fma(Tm[1 + pair_a(kk)][a][d], fv[1 + pair_b(kk)], fma(Tm[0][a][d], fv[4 + kk], ph[kk]));
                }
            }
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) {
                pn += __shfl_xor_sync(0xffffffffu, pn, o);
#pragma unroll
                for (int c = 0; c < 3; c++) pg[c] += __shfl_xor_sync(0xffffffffu, pg[c], o);
#pragma unroll
                for (int kk = 0; kk < 6; kk++) ph[kk] += __shfl_xor_sync(0xffffffffu, ph[kk], o);
            }
            if (tx == 0) {
                acc_n[ty * 4 + a] += (double)pn;
#pragma unroll
                for (int c = 0; c < 3; c++) acc_g[c][ty * 4 + a] += 2.0 * (double)pg[c];
#pragma unroll
                for (int kk = 0; kk < 6; kk++) acc_h[kk][ty * 4 + a] += 2.0 * (double)ph[kk];
            }
        }
    }
    __syncthreads();
    double wn = 0.0;
    if (tid < TQ) {
        const int q = q0 + tid;
        if (q < P) {
            const int p = p0 + q;
            *n_at(s, m, p) = acc_n[tid];
            for (int c = 0; c < 3; c++) *gn_at(s, m, p, c) = acc_g[c][tid];
            const int64_t np = s.sys.np[m], o = s.perm[p] - s.sys.poff[m];
            for (int c = 0; c < 6; c++) hess[(int64_t)c * np + o] = acc_h[c][tid];
            wn = s.pw[p] * acc_n[tid];
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) wn += __shfl_xor_sync(0xffffffffu, wn, o);
    if ((tid & 31) == 0) red[tid >> 5] = wn;
    __syncthreads();
    if (tid == 0) {
        double tsum = 0.0;
        for (int w = 0; w < 8; w++) tsum += red[w];
        ne_part[w0 + blockIdx.x] = tsum;
    }
}

}  // namespace

template <typename OutT, bool LAP>
static cudaError_t launch_eval_hess_t(const DevSystem &s, int32_t b0, int32_t b1, OutT *scratch, const int64_t *hoff,
                                      cudaStream_t st) {
    // several CTAs per batch: a batch's (atom, point) pairs are independent, and small systems have
    // fewer batches than the GPU has SMs
    const dim3 grid(b1 - b0, 4);
    switch (s.lmax) {
        case 0:
        case 1: eval_hess_kernel<1, OutT, LAP><<<grid, 128, 0, st>>>(s, b0, scratch, hoff); break;
        case 2: eval_hess_kernel<2, OutT, LAP><<<grid, 128, 0, st>>>(s, b0, scratch, hoff); break;
        case 3: eval_hess_kernel<3, OutT, LAP><<<grid, 128, 0, st>>>(s, b0, scratch, hoff); break;
        case 4: eval_hess_kernel<4, OutT, LAP><<<grid, 128, 0, st>>>(s, b0, scratch, hoff); break;
        default: eval_hess_kernel<NAO_LMAX, OutT, LAP><<<grid, 128, 0, st>>>(s, b0, scratch, hoff); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_eval_hess(const DevSystem &s, int32_t b0, int32_t b1, void *scratch, bool fp32, bool lap,
                             const int64_t *hoff, cudaStream_t st) {
    if (b1 <= b0) return cudaSuccess;
    if (fp32)
        return lap ? launch_eval_hess_t<float, true>(s, b0, b1, static_cast<float *>(scratch), hoff, st)
                   : launch_eval_hess_t<float, false>(s, b0, b1, static_cast<float *>(scratch), hoff, st);
    return lap ? launch_eval_hess_t<double, true>(s, b0, b1, static_cast<double *>(scratch), hoff, st)
               : launch_eval_hess_t<double, false>(s, b0, b1, static_cast<double *>(scratch), hoff, st);
}

cudaError_t launch_density_hess(const DevSystem &s, const DWork *work, int32_t w0, int32_t n_work, const void *scratch,
                                bool fp32, const int64_t *hoff, double *hess, double *ne_part, cudaStream_t st) {
    if (n_work <= 0) return cudaSuccess;
    if (fp32)
        density_hess_kernel<float><<<n_work, 256, 0, st>>>(s, work, w0, static_cast<const float *>(scratch), hoff, hess,
                                                            ne_part);
    else
        density_hess_kernel<double><<<n_work, 256, 0, st>>>(s, work, w0, static_cast<const double *>(scratch), hoff,
                                                             hess, ne_part);
    return cudaGetLastError();
}
