// Split-precision (Ozaki) contractions on the tcgen05 tensor cores.
//
// The batch products of Eq. batch_matrix_mult (Hamiltonian) and of the density (Eq. Density
// restricted to nnz(B)) are dense matrix products whose inputs are FP64. Each input row x
// (one basis function over the batch's points for H; one point over the basis for n; one
// density-matrix row for n) is scaled by a power of two 2^-e so that |x 2^-e| < 1/2, rounded
// to an integer X = round(x 2^(6S-e)) and cut into S balanced base-64 digits
//     X = sum_s d_s 64^(S-1-s),  d_s in [-32, 32],
// (Ozaki, Ogita, Oishi, Rump, "Error-free transformations of matrix multiplication by using
// fast routines of matrix multiplication", Numer. Algorithms 59 (2012): a splitting whose
// slice products are exact in the working precision of the fast product). Every digit is an
// exact bf16 integer, every digit product is at most 2^10, and a K-long sum of the products of
// one slice-order group g = s + t (g + 1 pairs) stays below K (g+1) 2^10 < 2^24, so it is exact
// in the FP32 accumulator. Each group therefore has its own accumulator in tensor memory;
// pairs with s + t >= S are dropped (their weight is below 64^-S). The epilogue recombines the
// groups as integers (three 64-bit parts) and scales once in FP64:
//     x_i . y_j = 2^(e_i + e_j) sum_g M_g 64^-(g+2).
// Tensor memory holds S groups x TN columns: TN = 48 for S <= 10 bf16 slices, else TN = 32.
//
// Hamiltonian: A = F (rows i, K = 4 Ppad: phi | d/dx | d/dy | d/dz weighted by sqrt|d_k|) and
// B = sign(d_k) F (rows j), 128 x TN elements at a time (S groups x TN FP32 columns of tensor memory's 512):
// with TN = 32 any four 32-row blocks against one column tile, so that each pair of blocks is computed once;
// FP64 atomic scatter.
// Density: A = Phi^T (rows = points, K = basis), B = P' (rows j, P'_ij = c_IJ P_ij for groups
// I <= J of functions with c_II = 1, c_IJ = 2, else 0) so that T_qj = sum_i phi_qi P'_ij and
// n_q = sum_j T_qj phi_qj; one per-batch exponent is used for P'.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "ff.h"
#include "nao_internal.h"
#include "split_bits.h"
#include "tc_ptx.h"

namespace {

constexpr long long kWaitCycles = 400000000LL;  // ~0.2 s at 2 GHz: bounded mbarrier waits
constexpr size_t kSmemOptin = 232448;           // shared memory a CTA may opt into on this GPU (227 KB)


// Digits are cut in FP32 arithmetic from a value's FP32 parts (a float-float's two, an FP64's three, taken from its bit
// pattern): on this GPU the FP64 pipe is ~1/60 of the FP32 rate, and a double-to-int64 conversion per element would
// make the slicing kernels FP64-bound.
using split_bits::abs_bits;

// S balanced base-2^B digits (B = 6: base 64, |d| <= 32, bf16; B = 5: base 32, |d| <= 16, e4m3;
// most significant first in dig[0]) of X = round(x 2^(BS-e)), |x 2^-e| < 1/2, as exact
// small-integer floats, for two values at once (.x and .y) in packed FP32x2 arithmetic.
//
// x comes as two or three FP32 parts, each scaled exactly by 2^(BS-e). A part is cut into balanced chunks
// of CB = D B bits (3 x 6 or 4 x 5) from the top: q = rint(R 2^-(c CB)), R <- R - q 2^(c CB), for
// c = 3, 2, 1, then u_0 = rint(R). Every step is exact (R keeps a subset of the part's 24 significand
// bits; |R 2^-(c CB)| < 2^22 keeps the rounding by 1.5 2^23 valid, and an FMA forms the product and
// that rounding at once), so sum_c u_c 2^(c CB) is the part rounded to an integer. The parts' chunks are
// added per chunk, and the digits are peeled off the chunks from the bottom: q = rint(v / 2^B),
// d = v - 2^B q in [-2^(B-1), 2^(B-1)], v <- q, the carry q joining the next chunk. The top digit keeps
// whatever remains, which the bound on |X| keeps in range. The result is within one unit of
// round(|x| 2^(BS-e)).
constexpr float kRint = 12582912.0f;  // 1.5 2^23: y + kRint - kRint = rint(y) for |y| < 2^22

__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }

// u_c += the chunks of part R (|R| < 2^(TOP CB + 22)), c = TOP .. 0.
template <int CB, int TOP>
__device__ __forceinline__ void add_chunks(float2 R, float2 (&u)[4]) {
#pragma unroll
    for (int c = TOP; c >= 1; c--) {
        const float w = c == 3 ? (float)(1ULL << CB) * (float)(1ULL << CB) * (float)(1ULL << CB)
                      : c == 2 ? (float)(1ULL << CB) * (float)(1ULL << CB) : (float)(1ULL << CB);
        const float2 q = __fadd2_rn(__ffma2_rn(R, f2(1.0f / w), f2(kRint)), f2(-kRint));
        R = __ffma2_rn(q, f2(-w), R);
        u[c] = __fadd2_rn(u[c], q);
    }
    u[0] = __fadd2_rn(u[0], __fadd2_rn(__fadd2_rn(R, f2(kRint)), f2(-kRint)));
}

// The digits from the chunks.
template <int S, int B>
__device__ __forceinline__ void peel(const float2 (&u)[4], float2 (&dig)[S]) {
    constexpr int D = B == 6 ? 3 : 4;  // digits per chunk
    const float2 inv = f2(1.0f / (1 << B)), mb = f2(-(float)(1 << B));
    float2 v = u[0];
#pragma unroll
    for (int s = S - 1; s >= 0; s--) {
        const int t = S - 1 - s;  // digits already taken
        if (t > 0 && t % D == 0) v = __fadd2_rn(v, u[t / D]);
        if (s == 0) {
            dig[0] = v;
        } else {
            const float2 q = __fadd2_rn(__ffma2_rn(v, inv, f2(kRint)), f2(-kRint));  // rint(v / 2^B)
            dig[s] = __ffma2_rn(q, mb, v);
            v = q;
        }
    }
}

// 2^(BS-e) as the product of two FP32 powers (the exponent itself may exceed FP32's range); both zero
// for a row that counts as zero (e <= -10000).
template <int S, int B>
struct Scale {
    float2 a, b;
    __device__ __forceinline__ explicit Scale(int e) {
        const int k = B * S - e, k1 = k >> 1;
        a = f2(e <= -10000 ? 0.0f : __int_as_float((127 + k1) << 23));
        b = f2(e <= -10000 ? 0.0f : __int_as_float((127 + k - k1) << 23));
    }
    __device__ __forceinline__ float2 operator()(float2 v) const { return __fmul2_rn(__fmul2_rn(v, a), b); }
};

// Of two float-floats. The low part is below 2^-24 of the high one, so below 2^(2 CB + 22).
template <int S, int B>
__device__ __forceinline__ void digits2(ffa::F x0, ffa::F x1, const Scale<S, B> &sc, float2 (&dig)[S]) {
    constexpr int CB = (B == 6 ? 3 : 4) * B;
    static_assert(B * S - 25 < 2 * CB + 22, "the low part reaches the top chunk");
    float2 u[4] = {f2(0.0f), f2(0.0f), f2(0.0f), f2(0.0f)};
    add_chunks<CB, 3>(sc(make_float2(x0.h, x1.h)), u);
    add_chunks<CB, 2>(sc(make_float2(x0.l, x1.l)), u);
    peel<S, B>(u, dig);
}

// An FP64's 53 bits as three FP32s (24, 23 and 6 bits, all of its sign), scaled by 2^(BS-e) through the exponent
// field: no FP64 instruction (the FP64 pipe has 1/64 of the FP32 rate). FP64s below 2^-900 count as zero.
template <int S, int B>
__device__ __forceinline__ void f64_parts(double x, int e, float &h, float &m, float &l) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const int eb = (int)((hi >> 20) & 0x7FF), ex = eb - 1023 + B * S - e;  // |x| 2^(BS-e) in [2^ex, 2^(ex+1))
    const uint32_t sg = hi & 0x80000000u;
    h = m = l = 0.0f;
    if (eb == 0 || e <= -10000 || ex < -30) return;  // below half a unit
    const uint32_t b1 = sg | (uint32_t)(127 + ex) << 23;
    h = __uint_as_float(b1 | (hi & 0xFFFFFu) << 3 | lo >> 29);
    // the next bits as the fraction of a number of that binade, less its leading one
    const uint32_t b2 = sg | (uint32_t)(127 + ex - 23) << 23;
    m = __fsub_rn(__uint_as_float(b2 | ((lo >> 6) & 0x7FFFFFu)), __uint_as_float(b2));
    const uint32_t b3 = sg | (uint32_t)(127 + ex - 46) << 23;
    l = __fsub_rn(__uint_as_float(b3 | (lo & 0x3Fu) << 17), __uint_as_float(b3));
}
// Of two FP64s.
template <int S, int B>
__device__ __forceinline__ void digits2(double x0, double x1, int e, float2 (&dig)[S]) {
    constexpr int CB = (B == 6 ? 3 : 4) * B;
    float2 p[3], u[4] = {f2(0.0f), f2(0.0f), f2(0.0f), f2(0.0f)};
    f64_parts<S, B>(x0, e, p[0].x, p[1].x, p[2].x);
    f64_parts<S, B>(x1, e, p[0].y, p[1].y, p[2].y);
    add_chunks<CB, 3>(p[0], u);
    add_chunks<CB, 2>(p[1], u);
    add_chunks<CB, 1>(p[2], u);
    peel<S, B>(u, dig);
}

// bf16 bit patterns of two small integers held exactly in floats (their low halves are zero).
__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
    return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
}

// e4m3 bytes of four integers |d| <= 16 held in floats (each exact in e4m3), a at the lowest
// address. cvt...e4m3x2 puts its first source in the upper byte of the pair.
__device__ __forceinline__ uint32_t pack_e4m3x4(float a, float b, float c, float d) {
    unsigned short lo, hi;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(lo) : "f"(b), "f"(a));
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(hi) : "f"(d), "f"(c));
    return (uint32_t)lo | ((uint32_t)hi << 16);
}

// Digits of the 128-byte row segment a lane owns in one K chunk: values x[0..LC-1] of its LC
// columns (2 for bf16, 4 for e4m3; FP64 with the exponent, or float-float with its scale), packed per
// slice into one 32-bit word.
template <int S, int F, typename V, typename E>
__device__ __forceinline__ void lane_digit_words(const V *x, const E &e, uint32_t (&w)[S]) {
    constexpr int B = nao_digit_bits(F);
    float2 d0[S];
    digits2<S, B>(x[0], x[1], e, d0);
    if constexpr (F == NAO_DIGITS_BF16) {
#pragma unroll
        for (int sl = 0; sl < S; sl++) w[sl] = pack_bf16x2(d0[sl].x, d0[sl].y);
    } else {
        float2 d1[S];
        digits2<S, B>(x[2], x[3], e, d1);
#pragma unroll
        for (int sl = 0; sl < S; sl++) w[sl] = pack_e4m3x4(d0[sl].x, d0[sl].y, d1[sl].x, d1[sl].y);
    }
}
// What lane_digit_words takes for a row's exponent, by value type.
template <int S, int F>
__device__ __forceinline__ Scale<S, nao_digit_bits(F)> digit_scale(const ffa::F *, int e) { return Scale<S, nao_digit_bits(F)>(e); }
template <int S, int F>
__device__ __forceinline__ int digit_scale(const double *, int e) { return e; }

// 2^E as an FP64 (0 below the normal range).
__device__ __forceinline__ double pow2(int E) {
    if (E < -1022) return 0.0;
    if (E > 1023) E = 1023;
    return __longlong_as_double((long long)(1023 + E) << 52);
}


// ----------------------------------------------------------------------------------------
// Hamiltonian slicing: one CTA per (batch, tile of `tile` basis functions, 64 or 16). Columns are
// reordered: the negative-weight ones (v < 0 on the potential part) first, padded to a whole
// MMA K step (16 bf16 or 32 e4m3 columns), then the rest, so that B = A and the sign is applied
// per K step.
// One warp per row: the largest magnitude of the row times the column scales sqrt|d_k| (a pass over the row's
// K float-float values), then its digits (a second pass, served from L2: the slices are written with
// evict-first stores so that they do not push the rows out), one 128-byte segment per slice and K chunk.
// Within each K step, lane l of the 8 lanes that write the step's 32 bytes takes the logical columns 2 l,
// 2 l + 1 (, 16 + 2 l, 17 + 2 l): a permutation inside the K step, the same for every row (A and B of H are the
// same digit rows, so every product is unchanged, and each K step keeps its sign), which keeps each load
// instruction of the second pass on a few 64-byte runs of the row.
// Bound by HBM (8 bytes read and 14 or 24 written per value: 5.2 and 5.5 TB/s of the copy's 6.8): 45-atom slab,
// 14 e4m3 slices, 5.89 -> 5.17 ms with the packed digit code; 12 bf16 slices 6.85 -> 6.33 ms. Keeping the scaled
// rows in shared memory between the passes cost more in occupancy than the second read.
// The first pass has eight loads in flight per lane: 5.10 ms with four, 4.82 with eight, 4.73 to 5.14 with 13 to 20
// (whose remainders cost other row lengths more); the next row's prefetch to L2 5.34.
// ----------------------------------------------------------------------------------------
constexpr int kSliceWarps = 8;
// Shared memory of slice_h_kernel for a batch of Ppad padded points: column scales, order, signs.
__host__ __device__ constexpr size_t slice_h_smem(int Ppad, int F) {
    return (size_t)4 * Ppad * (8 + 1) + 32 +
           (size_t)2 * ((4 * Ppad + nao_kstep_cols(F) + nao_chunk_cols(F) - 1) / nao_chunk_cols(F) * nao_chunk_cols(F));
}

template <int S, int F>
__global__ void __launch_bounds__(32 * kSliceWarps, 4) slice_h_kernel(const __grid_constant__ DevSystem s, int32_t b0, int tile,
                                                                  const FF2 *__restrict__ scratch, uint32_t terms,
                                                                  uint8_t *__restrict__ slices,
                                                                  const int64_t *__restrict__ sl_off,
                                                                  int32_t *__restrict__ expo, int32_t *__restrict__ neg16) {
    extern __shared__ __align__(16) unsigned char slice_sh[];
    __shared__ int wsum[kSliceWarps];
    const int b = b0 + blockIdx.x, rt = blockIdx.y, m = s.sys.bmol[b];
    const int p0 = s.batch_off[b], P = s.batch_off[b + 1] - p0;
    const int Ppad = (P + NAO_PPAD - 1) & ~(NAO_PPAD - 1);
    const int N = s.rel_off[b + 1] - s.rel_off[b];
    constexpr int C = nao_chunk_cols(F), KS = nao_kstep_cols(F), LC = C / 32, B = nao_digit_bits(F);  // LC: columns per lane
    const SplitGeom G(P, N, S, 0, F);
    if (N == 0 || rt * tile >= G.R16) return;
    const int K = 4 * Ppad, Kp = C * G.n_kc, T = 32 * kSliceWarps;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float2 *sd = reinterpret_cast<float2 *>(slice_sh);              // [K] column scale sqrt|d| as a float-float
    short *src = reinterpret_cast<short *>(sd + K);                 // [Kp] the column at each logical place (-1: none)
    unsigned char *negf = reinterpret_cast<unsigned char *>(src + Kp);  // [K]
    const FF2 *E = scratch + s.scr_off[b];
    for (int q = threadIdx.x; q < Ppad; q += T) {
        float2 sq[2];
        bool ng[2];
#pragma unroll
        for (int c = 0; c < 2; c++) {  // the potential part, the gradient parts
            const double d = q < P ? split_bits::h_column_weight(s, m, p0 + q, c, terms) : 0.0;
            // sqrt|d| as a float-float: the FP32 square root s0 and one Newton correction
            // (|d| - s0^2) / (2 s0), the residual formed exactly by one FP64 FMA (|d| below the FP32
            // range counts as a zero weight)
            const float a = __double2float_rn(fabs(d));
            sq[c] = make_float2(0.0f, 0.0f);
            if (a >= 1.17549435e-38f) {
                const float s0 = __fsqrt_rn(a);
                const double r = fma(-(double)s0, (double)s0, fabs(d));
                const ffa::F f = ffa::quick(s0, __fmul_rn(__double2float_rn(r), __fdiv_rn(0.5f, s0)));
                sq[c] = make_float2(f.h, f.l);
            }
            ng[c] = d < 0.0;
        }
#pragma unroll
        for (int c = 0; c < 4; c++) {
            sd[c * Ppad + q] = sq[c == 0 ? 0 : 1];
            negf[c * Ppad + q] = ng[c == 0 ? 0 : 1] ? 1 : 0;
        }
    }
    for (int k = threadIdx.x; k < Kp; k += T) src[k] = -1;
    __syncthreads();
    // exclusive scan of the negative flags: thread t owns columns [t*per, t*per + per)
    const int per = (K + T - 1) / T;
    const int kb = min(K, (int)threadIdx.x * per), ke = min(K, kb + per);
    int cnt = 0;
    for (int k = kb; k < ke; k++) cnt += negf[k];
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int before = 0, total = 0;
    for (int w = 0; w < kSliceWarps; w++) {
        if (w < warp) before += wsum[w];
        total += wsum[w];
    }
    before += incl - cnt;
    const int negpad = (total + KS - 1) / KS * KS;  // a whole MMA K step
    for (int k = kb; k < ke; k++) {
        src[negf[k] ? before : negpad + k - before] = (short)k;
        before += negf[k];
    }
    if (rt == 0 && threadIdx.x == 0) neg16[b] = negpad / KS;  // negated K steps
    __syncthreads();
    uint8_t *base = slices + sl_off[b];
    for (int lr = warp; lr < tile; lr += kSliceWarps) {
        const int r = rt * tile + lr;
        if (r >= G.R16) break;
        const float2 *row = reinterpret_cast<const float2 *>(E + (int64_t)(r < N ? r : 0) * K);
        auto scaled = [&](int k) {
            const float2 v = row[k], w = sd[k];
            return ffa::mul(ffa::F{v.x, v.y}, ffa::F{w.x, w.y});
        };
        int mx = 0;
        if (r < N)
#pragma unroll 8
            for (int k = lane; k < K; k += 32) mx = max(mx, __float_as_int(scaled(k).h) & 0x7FFFFFFF);
        mx = __reduce_max_sync(0xffffffffu, mx);
        // |x.h| <= (2 - 2^-23) 2^k and |x.l| <= 2^-24 2^(k+1): |x| < 2^(k+1), and |x 2^-e| < 1/2 with e = k + 2
        const int e = (mx >> 23) != 0 ? (mx >> 23) - 127 + 2 : -10000;
        if (lane == 0 && r < N) expo[s.rel_off[b] + r] = e;
        const Scale<S, B> sc(e);
        for (int kc = 0; kc < G.n_kc; kc++) {
            ffa::F x[LC];
#pragma unroll
            for (int c = 0; c < LC; c += 2) {
                // bf16: columns 2 lane, 2 lane + 1 of the chunk; e4m3: 32 (lane / 8) + 2 (lane % 8) + {0, 1, 16, 17}
                const int at = C * kc + (F == NAO_DIGITS_BF16 ? 2 * lane : KS * (lane >> 3) + 2 * (lane & 7) + 8 * c);
                const short2 kk = *reinterpret_cast<const short2 *>(src + at);
                x[c] = kk.x >= 0 ? scaled(kk.x) : ffa::F{0.0f, 0.0f};
                x[c + 1] = kk.y >= 0 ? scaled(kk.y) : ffa::F{0.0f, 0.0f};
            }
            uint32_t wd[S];
            lane_digit_words<S, F>(x, sc, wd);
            const uint32_t off = tc::sw128_byte((uint32_t)r, (uint32_t)(4 * lane));
#pragma unroll
            for (int sl = 0; sl < S; sl++) __stcs(reinterpret_cast<unsigned int *>(base + G.h_block(sl, kc) + off), wd[sl]);
        }
    }
}

// ----------------------------------------------------------------------------------------
// Density slicing.
// Phi^T: one CTA (4 warps) per (batch, 16-point tile), the point exponents from the evaluation. A K chunk (64 or
// 128 functions) of phi[i][q], read along the points, comes to shared memory while the chunk before it is cut
// into digits; each warp writes its points' rows along K (2 or 4 functions per lane, one 128-byte row segment per
// slice). The first kPexpCtas CTAs of a batch instead reduce its exponent of P' (read along rows of P), as a
// biased exponent.
// Bound by the latency of the loads (a batch has one to four chunks), and with 12 bf16 slices by HBM next (4.8 TB/s):
// against 32 points by 8 warps with one buffer, loads and digits in turn, 64 atoms 1.37 -> 0.92 ms.
// ----------------------------------------------------------------------------------------
// The symmetry c_IJ of P' is taken between groups of GW = nao_split_tn(S, F) functions, whatever width the
// contraction's tiles have: the digits, and so n, do not depend on the tuned width.

constexpr int kPexpCtas = 8;  // CTAs per batch that reduce the exponent of P'
constexpr int kNphiWarps = 4, kNphiPoints = 16;

// Row of function k of a chunk in shared memory: eight more per K step, so that the functions a half-warp reads
// at once (eight each of two K steps) lie in different banks.
template <int F>
__device__ __forceinline__ int stage_row(int k) { return k + 8 * (k / nao_kstep_cols(F)); }
template <int F>
__host__ __device__ constexpr int stage_rows() { return nao_chunk_cols(F) + 8 * (nao_chunk_cols(F) / nao_kstep_cols(F)); }

// 8 bytes global -> shared, zeros where !ok
__device__ __forceinline__ void cp8(void *dst, const void *src, bool ok) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(tc::smem_addr(dst)), "l"(src), "r"(ok ? 8 : 0) : "memory");
}
__device__ __forceinline__ ffa::F stage_value(const FF2 &v) { return v.f(); }
__device__ __forceinline__ double stage_value(double v) { return v; }

// V = FF2: the split path's float-float phi (rows of ld_mult Ppad at scr_off[b]); V = double: the
// density Hessian's FP64 evaluation (rows of 10 Ppad at eoff[b]), component row coff (phi or one
// gradient component). pexp = 0 leaves the P' exponent to another launch.
template <int S, int F, typename V>
__global__ void __launch_bounds__(32 * kNphiWarps) slice_nphi_kernel(const __grid_constant__ DevSystem s, int32_t b0, const V *__restrict__ scratch,
                                                        const int64_t *__restrict__ eoff, int coff,
                                                        uint8_t *__restrict__ slices, const int64_t *__restrict__ sl_off,
                                                        const int32_t *__restrict__ expo_q, int32_t *__restrict__ expo_b,
                                                        int ld_mult, int full, int pexp) {
    constexpr int C = nao_chunk_cols(F), LC = C / 32, GW = nao_split_tn(S, F), W = kNphiWarps, Q = kNphiPoints;
    constexpr int KS = nao_kstep_cols(F);
    __shared__ V t[2][stage_rows<F>()][Q + 1];
    const int b = b0 + blockIdx.x;
    const int p0 = s.batch_off[b], P = s.batch_off[b + 1] - p0;
    const int Ppad = (P + NAO_PPAD - 1) & ~(NAO_PPAD - 1);
    const int N = s.rel_off[b + 1] - s.rel_off[b];
    if (N == 0) return;
    const SplitGeom G(P, N, S, 0, F);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (blockIdx.y < kPexpCtas) {
        if (!pexp) return;
        // max |P'_ij| over i <= j (P' is P on the diagonal groups, 2 P off them, 0 below unless
        // full): the exponent field of |P| plus one off the diagonal groups; each CTA takes every
        // kPexpCtas-th set of W rows (expo_b[b] is zero before: the evaluation clears it)
        const int m = s.sys.bmol[b];
        const int32_t *rel = s.rel_idx + s.rel_off[b];
        int mk = 0;
        for (int i = warp + W * (int)blockIdx.y; i < N; i += W * kPexpCtas) {
            const int64_t gi = rel[i];
#pragma unroll 4
            for (int j = (full ? 0 : i) + lane; j < N; j += 32) {
                const int64_t gj = rel[j];
                const int eb = split_bits::biased_exponent(abs_bits(gi <= gj ? p_elem(s, m, gi, gj) : p_elem(s, m, gj, gi)));
                mk = max(mk, eb + ((eb != 0 && !full && i / GW < j / GW) ? 1 : 0));
            }
        }
        mk = __reduce_max_sync(0xffffffffu, mk);
        if (lane == 0 && mk > 0) atomicMax(expo_b + b, mk);
        return;
    }
    const int q0 = ((int)blockIdx.y - kPexpCtas) * Q;
    if (q0 >= G.P16) return;
    const int64_t ld = (int64_t)ld_mult * Ppad;
    // this thread's point and its first function of a chunk; row i of phi at scratch + eoff[b] + coff Ppad + i ld
    const int lq = threadIdx.x % Q, li = threadIdx.x / Q;
    const bool qin = q0 + lq < P;
    const V *E = scratch + eoff[b] + (int64_t)coff * Ppad + q0 + lq;
    auto load = [&](int kc) {
#pragma unroll
        for (int h = 0; h < C * Q / (32 * W); h++) {
            const int k = li + 32 * W / Q * h, i = kc * C + k;
            const bool ok = i < N && qin;
            cp8(&t[kc & 1][stage_row<F>(k)][lq], ok ? E + (int64_t)i * ld : scratch, ok);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    int eq[Q / W];
#pragma unroll
    for (int h = 0; h < Q / W; h++) {
        const int q = q0 + warp * (Q / W) + h;
        eq[h] = q < P ? expo_q[p0 + q] : -10000;
    }
    uint8_t *base = slices + sl_off[b];
    load(0);
    for (int kc = 0; kc < G.n_kcN; kc++) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();  // this chunk is there, and every warp has left the other buffer
        if (kc + 1 < G.n_kcN) load(kc + 1);
#pragma unroll
        for (int h = 0; h < Q / W; h++) {
            const int ql = warp * (Q / W) + h, q = q0 + ql;  // below P16, a multiple of Q
            // within each K step (KS functions, the words of 8 lanes) lane l packs functions l, l + 8
            // (, l + 16, l + 24): both operands of the density's product (this A and
            // slice_np_kernel's B) order K this way inside each K step, which leaves every slice
            // product unchanged; K steps hold consecutive functions, so that n_tc_kernel can stop
            // at a tile's last one
            decltype(stage_value(V())) x[LC];
#pragma unroll
            for (int c = 0; c < LC; c++) x[c] = stage_value(t[kc & 1][(KS + 8) * (lane >> 3) + (lane & 7) + 8 * c][ql]);
            uint32_t wd[S];
            lane_digit_words<S, F>(x, digit_scale<S, F>(x, eq[h]), wd);
            const uint32_t off = tc::sw128_byte((uint32_t)q, (uint32_t)(4 * lane));
#pragma unroll
            for (int sl = 0; sl < S; sl++) *reinterpret_cast<uint32_t *>(base + G.nA_block(sl, kc) + off) = wd[sl];
        }
    }
}

// P'_ij = c_IJ P[rel_i][rel_j] over GW-function groups I = i/GW <= J = j/GW (c_II = 1,
// c_IJ = 2; every (i, j) with c = 1 when full), read from P's upper triangle, with the batch's
// exponent from slice_nphi_kernel. One CTA per (batch, 16 rows j), one warp per row, 2 or 4
// functions i per lane (slice_nphi_kernel's K order; one 128-byte row segment per slice). Chunks that no
// tile of the contraction reads (n_item_ks: those past the last function of the row's group) are not written.
// Bound by integer and FP32 issue (the digits of FP64 values). Staging P's blocks in shared memory, read along
// its rows, was slower (slab of 45 atoms 2.3 ms against 1.4; with all chunks written 2.0): P is in L2, and
// neighbouring lanes' sectors are used by the next rows' warps.
template <int S, int F>
__global__ void __launch_bounds__(256) slice_np_kernel(const __grid_constant__ DevSystem s, int32_t b0, uint8_t *__restrict__ slices,
                                                      const int64_t *__restrict__ sl_off,
                                                      const int32_t *__restrict__ expo_b, int full) {
    const int b = b0 + blockIdx.x, m = s.sys.bmol[b];
    const int P = s.batch_off[b + 1] - s.batch_off[b];
    const int N = s.rel_off[b + 1] - s.rel_off[b];
    if (N == 0) return;
    constexpr int C = nao_chunk_cols(F), KS = nao_kstep_cols(F), LC = C / 32, GW = nao_split_tn(S, F);
    const SplitGeom G(P, N, S, 0, F);
    const int j0 = blockIdx.y * 16;
    if (j0 >= G.R16) return;
    const int32_t *rel = s.rel_idx + s.rel_off[b];
    const int e = split_bits::exponent_of_binade(expo_b[b]);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint8_t *base = slices + sl_off[b];
    // functions that a 32- or GW-wide tile with these rows multiplies, in K steps
    const int end = full ? N : ((j0 / 32 + 1) * 32 + GW - 1) / GW * GW;
    const int nk = min(G.n_kcN, ((end + KS - 1) / KS + 3) / 4);
#pragma unroll 1
    for (int h = 0; h < 2; h++) {
        const int j = j0 + warp * 2 + h;  // < R16: R16 is a multiple of 16
        const bool jin = j < N;
        const int64_t gj = jin ? rel[j] : 0;
        const int group = j / GW;
        for (int kc = 0; kc < nk; kc++) {
            double xp[LC];
#pragma unroll
            for (int hh = 0; hh < LC; hh++) {
                const int i = C * kc + KS * (lane >> 3) + (lane & 7) + 8 * hh;
                double x = 0.0;
                if (jin && i < N && (full || i / GW <= group)) {
                    const int64_t gi = rel[i];
                    x = gi <= gj ? p_elem(s, m, gi, gj) : p_elem(s, m, gj, gi);
                    // c_IJ = 2 off the diagonal tiles: exact, as one more in the exponent field
                    // (zero and subnormal values, which give no digits, are left as they are)
                    const long long pb = __double_as_longlong(x);
                    if (!full && i / GW < group && split_bits::biased_exponent(pb) != 0)
                        x = __longlong_as_double(pb + (1LL << 52));
                }
                xp[hh] = x;
            }
            uint32_t wd[S];
            lane_digit_words<S, F>(xp, e, wd);
            const uint32_t off = tc::sw128_byte((uint32_t)j, (uint32_t)(4 * lane));
#pragma unroll
            for (int sl = 0; sl < S; sl++) *reinterpret_cast<uint32_t *>(base + G.nB_block(S, sl, kc) + off) = wd[sl];
        }
    }
}

// ----------------------------------------------------------------------------------------
// Slice-product pipeline of the persistent contraction kernels, eighteen warps with TN = 32, fourteen with 48 (sixteen
// or twelve that read the accumulators, the producer, the MMA issuer). Shared memory: a ring of
// ring_slots(S) A-tile buffers (128 rows of 128 B, 16 KB, one slice of one K chunk each) and two sets
// of S B-tile buffers (TN rows, TN x 128 B). Producer (second last warp): for each K chunk, the S B
// slices into B set kc % 2, then the S A slices one by one into the ring, each copy a bulk (TMA)
// transfer completing on a "full" mbarrier. MMA issuer (last warp): for each A slice s, the pairs (s, t)
// with s + t < S as one 128 x TN(S-s) MMA per K step (two where TN(S-s) > 256) into accumulator groups
// s .. S-1 (tensor-memory columns TN s ...); commits release A buffers and B sets back to the producer
// through "empty" mbarriers. The other warps read the accumulators: warp w the rows of quadrant w % 4 and
// part w / 4 of the TN columns. The phases of the ring and of the B sets continue over all the
// accumulations a CTA runs. Every wait is bounded; on a timeout the CTA records NAO_ERR_TIMEOUT and
// skips the rest of its work.
// What bounds them: an earlier form (one issuing thread, four reading warps, 64-bit integer and FP64
// arithmetic) took 18.3 ms for H and 9.2 ms for n on a slab of 45 atoms (14 e4m3 slices); 18.0 and 9.1
// without any copies, 15.0 and 4.4 without the readers' work, 11.8 and 3.5 with the copies alone. So the
// MMA issue and the serial part of the readers (tensor memory holds one accumulator set) decided, not the
// operands' supply: the issuer runs with its whole warp, so that descriptors stay in uniform registers,
// and more warps read, with 32-bit integer and FP32 arithmetic. With the H items of nao_split_h_items and
// the density's K in whole steps: 10.9 and 3.8 ms. Of these 9.8 ms were the H producer's alone (9.4 with a
// quarter of the bytes, 4.8 with one copy per slice): it was one lane of a diverged warp, where every operand of
// a copy costs a loop over lanes. Issued by the converged warp the copies alone take 3.9 ms, H 8.6 and n 3.6 ms
// (12 bf16 slices: H 18.1 -> 13.0); H is now at its MMAs, 8.3 ms without the readers' work.
// ----------------------------------------------------------------------------------------
constexpr int kMaxRing = 8;
constexpr size_t kStaticSmem = 2048;   // room for the CTA's static shared memory (the PPipe barriers)

// A-ring slots: as many 16 KB A tiles as fit beside the two B sets (S tiles of TN rows each),
// at most kMaxRing: 8 for 11-12 bf16 slices (TN = 32), 6 for 10 (TN = 48), 7 for 14 e4m3 slices.
// A deeper ring lets the producer's copies run further ahead of the MMAs that wait for them.
__host__ __device__ constexpr int ring_slots(int S, int F) {
    return (int)((kSmemOptin - kStaticSmem - 1024 - 2 * (size_t)S * nao_split_tn(S, F) * 128) / 16384) < kMaxRing
               ? (int)((kSmemOptin - kStaticSmem - 1024 - 2 * (size_t)S * nao_split_tn(S, F) * 128) / 16384)
               : kMaxRing;
}

__host__ __device__ constexpr size_t pipe_smem_bytes(int S, int F) {
    return (size_t)ring_slots(S, F) * 16384 + 2 * (size_t)S * nao_split_tn(S, F) * 128 + 1024;
}
static_assert(ring_slots(12, 0) >= 4 && ring_slots(10, 0) >= 4 && ring_slots(4, 0) >= 4 && ring_slots(16, 1) >= 4,
              "A ring too shallow");
static_assert(pipe_smem_bytes(12, 0) + kStaticSmem <= kSmemOptin && pipe_smem_bytes(10, 0) + kStaticSmem <= kSmemOptin &&
                  pipe_smem_bytes(16, 1) + kStaticSmem <= kSmemOptin,
              "split pipeline exceeds shared memory");

// The S group accumulators M_g (exact integers, |M_g| < 2^24) of one element, neighbouring groups
// joined in 32-bit integers P = M_g 2^B + M_(g+1) (below 2^30.1):
//   e4m3 (base 32): P_k of groups 2k, 2k + 1, k = 0..7;
//   bf16 (base 64): P_0..P_2 of groups (0, 1), (2, 3), (4, 5), P_3 = M_6, P_4 of (7, 8), P_5 = M_9, P_6 of
//     (10, 11).
// Groups g >= S count as zero.
template <int F>
__host__ __device__ constexpr int n_pairs() { return F == NAO_DIGITS_E4M3 ? 8 : 7; }

// The joined integers of 8 columns of this thread's row. SMALL: every |M_g| <= 2^22, so that adding
// 1.5 2^23 leaves the integer in the significand (one FP32 addition; the conversion instruction has a
// quarter of its rate).
// a += x, b += x as FP32s, in one instruction.
__device__ __forceinline__ void add2(uint32_t &a, uint32_t &b, float x) {
    asm("{\n\t.reg .b64 u, v;\n\t"
        "mov.b64 u, {%0, %1};\n\tmov.b64 v, {%2, %2};\n\t"
        "add.rn.f32x2 u, u, v;\n\t"
        "mov.b64 {%0, %1}, u;\n\t}"
        : "+r"(a), "+r"(b)
        : "r"(__float_as_uint(x)));
}
template <int TN, int F, bool SMALL>
__device__ __forceinline__ void read_pairs8(uint32_t tm_col, int S, int (&p)[n_pairs<F>()][8]) {
    constexpr int B = nao_digit_bits(F), GB = F == NAO_DIGITS_E4M3 ? 4 : 6;  // groups per wait
    constexpr int kMagic = 0x4B400000;  // 1.5 2^23
#pragma unroll
    for (int h = 0; h < (F == NAO_DIGITS_E4M3 ? 4 : 2); h++) {
        uint32_t r[GB][8];
#pragma unroll
        for (int q = 0; q < GB; q++) {
            const int g = h * GB + q;
            if (g < S) {
                tc::tmem_ld8(tm_col + (uint32_t)(g * TN), r[q]);
            } else {
#pragma unroll
                for (int c = 0; c < 8; c++) r[q][c] = 0;
            }
        }
        tc::tmem_ld_wait();
        // in place: the integer of each group, offset by kMagic where SMALL
#pragma unroll
        for (int q = 0; q < GB; q++)
#pragma unroll
            for (int c = 0; c < 8; c += 2) {
                if (SMALL) {
                    add2(r[q][c], r[q][c + 1], 12582912.0f);
                } else {
                    r[q][c] = (uint32_t)__float2int_rn(__uint_as_float(r[q][c]));
                    r[q][c + 1] = (uint32_t)__float2int_rn(__uint_as_float(r[q][c + 1]));
                }
            }
#pragma unroll
        for (int c = 0; c < 8; c++) {
            constexpr uint32_t K1 = SMALL ? (uint32_t)kMagic : 0u, K2 = K1 * ((1u << B) + 1u);
            auto integer = [&](int q) { return (int)(r[q][c] - K1); };
            auto join = [&](int q) { return (int)(r[q][c] * (1u << B) + r[q + 1][c] - K2); };
            if constexpr (F == NAO_DIGITS_E4M3) {
                p[2 * h][c] = join(0);
                p[2 * h + 1][c] = join(2);
            } else if (h == 0) {
                p[0][c] = join(0);
                p[1][c] = join(2);
                p[2][c] = join(4);
            } else {
                p[3][c] = integer(0);
                p[4][c] = join(1);
                p[5][c] = integer(3);
                p[6][c] = join(4);
            }
        }
    }
}
template <int TN, int F>
__device__ __forceinline__ void read_pairs8(uint32_t tm_col, int S, bool small, int (&p)[n_pairs<F>()][8]) {
    if (small) read_pairs8<TN, F, true>(tm_col, S, p);
    else read_pairs8<TN, F, false>(tm_col, S, p);
}
// Whether an accumulation over K columns keeps every |M_g| <= K S 2^(2 B - 2) at or below 2^22.
template <int F>
__device__ __forceinline__ bool small_groups(int K, int S) {
    return (long long)K * S <= (1LL << (24 - 2 * nao_digit_bits(F)));
}

// The parts of one element in units of 2^(e_i + e_j), each exact in 64 bits (below 2^60.1):
//   bf16: hi = sum_{g<=6} M_g 64^(6-g) [units 2^-48], lo = sum_{7<=g<=9} M_g 64^(9-g) [2^-66],
//     lo2 = sum_{g>=10} M_g 64^(12-g) [2^-84] (S = 11, 12 only);
//   e4m3: hi = sum_{g<=7} M_g 32^(7-g) [units 2^-45], lo = sum_{g>=8} M_g 32^(15-g) [2^-85] (S <= 16);
//     lo2 stays 0.
template <int F>
__device__ __forceinline__ void pair_parts(const int (&p)[n_pairs<F>()][8], int c, long long &hi, long long &lo,
                                           long long &lo2) {
    if constexpr (F == NAO_DIGITS_E4M3) {
        hi = (long long)p[0][c] * (1 << 30) + ((long long)p[1][c] * (1 << 20) + ((long long)p[2][c] * (1 << 10) + p[3][c]));
        lo = (long long)p[4][c] * (1 << 30) + ((long long)p[5][c] * (1 << 20) + ((long long)p[6][c] * (1 << 10) + p[7][c]));
        lo2 = 0;
    } else {
        hi = (long long)p[0][c] * (1 << 30) + ((long long)p[1][c] * (1 << 18) + ((long long)p[2][c] * (1 << 6) + p[3][c]));
        lo = (long long)p[4][c] * (1 << 6) + p[5][c];
        lo2 = (long long)p[6][c] * (1 << 6);
    }
}

// An H element from its parts as one 64-bit integer v and a tier t, the value being
// v 2^(e_i + e_j - h_unit<F>(t)):
//   bf16: lo' = lo + round(lo2 / 2^18); t = 0 (|hi| < 2^44): hi 2^18 + lo' exactly (unit 66);
//         t = 1: 4 hi + round(lo' / 2^16) (unit 50; |4 hi| >= 2^46, relative error <= 2^-47);
//   e4m3: t = 0 (|hi| < 2^22): hi 2^40 + lo exactly (unit 85); t = 1 (|hi| < 2^40):
//         hi 2^22 + round(lo / 2^18) (unit 67; relative error <= 2^-45); t = 2:
//         4 hi + round(lo / 2^38) (unit 47; relative error <= 2^-43).
// (hi is in units of 2^-45 and lo of 2^-85 throughout: hi 2^k in units of 2^-(45 + k).)
template <int F>
__device__ __forceinline__ long long h_int(long long hi, long long lo, long long lo2, int &t) {
    if constexpr (F == NAO_DIGITS_BF16) {
        const long long l = lo + ((lo2 + (1LL << 17)) >> 18);
        if (hi > -(1LL << 44) && hi < (1LL << 44)) {
            t = 0;
            return (hi << 18) + l;
        }
        t = 1;
        return (hi << 2) + ((l + (1LL << 15)) >> 16);
    } else {
        if (hi > -(1LL << 22) && hi < (1LL << 22)) {
            t = 0;
            return (hi << 40) + lo;
        }
        if (hi > -(1LL << 40) && hi < (1LL << 40)) {
            t = 1;
            return (hi << 22) + ((lo + (1LL << 17)) >> 18);
        }
        t = 2;
        return (hi << 2) + ((lo + (1LL << 37)) >> 38);
    }
}
template <int F>
__device__ __forceinline__ int h_unit(int t) {
    return F == NAO_DIGITS_BF16 ? (t == 0 ? 66 : 50) : (t == 0 ? 85 : (t == 1 ? 67 : 47));
}
// A density T element from its joined integers, as a float-float in units of 2^(e_q + e_b - kTUnit): v + f / 2^10
// with the 64-bit integer v = floor(4 hi + lo' / 2^16) (bf16; lo' = lo + lo2 / 2^18) or floor(32 hi + lo / 2^35)
// (e4m3), T in units of 2^-50, and the next ten bits f. |T| < K / 4 keeps |v| < 2^61.1 (K <= 8191). v's three 21-bit
// pieces and f become FP32s exactly. kTUnit: 50 bits below, and 21 more because the float-float counts in 2^21. The
// lowest piece and f keep 2^-4 of a unit: with units of 2^-47, where an e4m3 T is about 2^42, that was 2^-46 of T
// (root mean square error of n against the root of its squared terms' sum, 20 functions: 4.1e-15, now 2.8e-15).
constexpr int kTUnit = 50 - 21;
template <int F>
__device__ __forceinline__ ffa::F pair_ff(const int (&p)[n_pairs<F>()][8], int c) {
    long long w;
    int f;
    uint32_t up;
    if constexpr (F == NAO_DIGITS_E4M3) {
        const long long r = (long long)p[4][c] * 32 + (p[5][c] >> 5);  // lo in units of 2^-10 of v's
        w = (long long)p[1][c] * (1 << 25) + ((long long)p[2][c] * (1 << 15) + ((long long)p[3][c] * 32 + (r >> 10)));
        f = (int)r & 1023;
        up = (uint32_t)p[0][c] * 8u;
    } else {
        const int r = p[4][c] + (p[5][c] >> 6) + (p[6][c] >> 18);  // lo', the same
        w = (long long)p[1][c] * (1 << 20) + ((long long)p[2][c] * (1 << 8) + (p[3][c] * 4 + (r >> 10)));
        f = r & 1023;
        up = (uint32_t)p[0][c];
    }
    const uint32_t lo = (uint32_t)w;
    const int hi = (int)((uint32_t)(w >> 32) + up);  // v = hi 2^32 + lo
    auto small = [](uint32_t x) { return __fsub_rn(__uint_as_float(0x4B000000u | x), 8388608.0f); };  // x < 2^23
    const float f2 = __fsub_rn(__int_as_float(0x4B400000 + (hi >> 10)), 12582912.0f);
    const float f1 = small(__funnelshift_r(lo, (uint32_t)hi, 21) & 0x1FFFFFu), f0 = small(lo & 0x1FFFFFu);
    const ffa::F a = ffa::quick(__fmul_rn(f2, 2097152.0f), f1);
    const float low = __fmaf_rn(small((uint32_t)f), 1.0f / 1024.0f, f0);
    return ffa::quick(a.h, __fmaf_rn(low, 1.0f / 2097152.0f, a.l));
}

// A float-float of an FP64, zeros (functions beyond their cutoffs) apart.
__device__ __forceinline__ ffa::F ff_of_bits(double x) {
    return ((uint32_t)__double2hiint(x) & 0x7FF00000u) == 0u ? ffa::F{0.0f, 0.0f} : ffa::from_double_bits(x);
}
// A value that no other thread reads, past L1: shared memory, the same array, is what the MMAs read their operands
// from (27 atoms with grad n: 4.43 -> 4.01 ms).
__device__ __forceinline__ FF2 load_once(const FF2 *p) {
    float h, l;
    asm volatile("ld.global.nc.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(h), "=f"(l) : "l"(p));
    return FF2(ffa::F{h, l});
}
__device__ __forceinline__ double load_once(const double *p) {
    double x;
    asm volatile("ld.global.nc.L1::no_allocate.f64 %0, [%1];" : "=d"(x) : "l"(p));
    return x;
}
__device__ __forceinline__ ffa::F ff_of_value(const FF2 &v) { return v.f(); }
__device__ __forceinline__ ffa::F ff_of_value(double v) { return ff_of_bits(v); }

// p + e = a b (float-floats) to 2^-48
__device__ __forceinline__ float ff_product(ffa::F a, ffa::F b, float &e) {
    const float p = __fmul_rn(a.h, b.h);
    e = __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.h, -p)));
    return p;
}
// acc + rest += a0 b0 + a1 b1 (float-floats), unevaluated. rest collects the rounding of acc.l, which without it is most
// of a density's own error (root mean square against the root of the squared terms' sum, 20 functions, 12 bf16 slices:
// 5.4e-15, with it 2.8e-15; in FP64 with T rounded to 2^-50 of its scale 4.2e-15). Two products at a time: n and
// grad n of 125 atoms, 14 e4m3 slices, 41.8 ms without rest, 44.3 one by one, 42.7 in pairs (12 bf16 slices 52.4,
// 51.3, 50.3).
__device__ __forceinline__ void ff_mac2(ffa::F &acc, float &rest, ffa::F a0, ffa::F b0, ffa::F a1, ffa::F b1) {
    float e0, e1;
    const float p0 = ff_product(a0, b0, e0), p1 = ff_product(a1, b1, e1);
    const ffa::F s = ffa::two_sum(p0, p1), t = ffa::two_sum(acc.h, s.h);
    const ffa::F u = ffa::two_sum(acc.l, __fadd_rn(__fadd_rn(t.l, s.l), __fadd_rn(e0, e1)));
    acc = ffa::F{t.h, u.h};
    rest = __fadd_rn(rest, u.l);
}

__device__ __forceinline__ uint8_t *align1024(uint8_t *p) {
    return reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(p) + 1023) & ~uintptr_t(1023));
}

// Accumulator-reading warps, four (one per quadrant of rows) for each part of the TN columns, 8 of them with
// TN = 32 and 16 with 48; and the CTA's threads with the producer and MMA warps. Tensor memory holds one
// accumulator set, so the MMAs stand still while it is read, and that is bound by latency: eight reading warps
// with 16 and 24 columns took 3.59 ms for n on the slab of 45 atoms where sixteen take 3.19 (27 atoms
// with grad n, 12 bf16 slices: 5.1 -> 4.5 ms; Hessian of a 13-atom molecule 5.4 -> 4.5 ms). More warps would
// leave too few registers for a block of 8 columns.
template <int TN>
__host__ __device__ constexpr int n_parts() { return TN == 48 ? 3 : 4; }
template <int TN>
__host__ __device__ constexpr int n_readers() { return 4 * n_parts<TN>(); }
template <int TN>
__host__ __device__ constexpr int tc_threads() { return 32 * (n_readers<TN>() + 2); }

struct PPipe {
    uint64_t fullA[kMaxRing], emptyA[kMaxRing], fullB[2], emptyB[2];
    uint64_t acc_full, acc_empty, fin;
    uint64_t part_full[4][3], part_empty[4];  // n: the exchange of the column parts' sums, per quadrant
    double part[4][32];
    uint32_t tmem;
    int abort;
};
static_assert(sizeof(PPipe) <= kStaticSmem, "barriers exceed their share of shared memory");

// Barriers, tensor memory; returns its base address. RING: the A ring's slots.
template <int TN>
__device__ __forceinline__ uint32_t pipe_setup(PPipe &pp, int RING, const int32_t *err) {
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        for (int i = 0; i < RING; i++) {
            tc::mbar_init(&pp.fullA[i], 1);
            tc::mbar_init(&pp.emptyA[i], 1);
        }
        for (int i = 0; i < 2; i++) {
            tc::mbar_init(&pp.fullB[i], 1);
            tc::mbar_init(&pp.emptyB[i], 1);
        }
        for (int i = 0; i < 4; i++) {
            for (int x = 0; x < 3; x++) tc::mbar_init(&pp.part_full[i][x], 1);
            tc::mbar_init(&pp.part_empty[i], 1);
        }
        tc::mbar_init(&pp.acc_full, 1);
        tc::mbar_init(&pp.acc_empty, n_readers<TN>());  // one arrival per accumulator-reading warp
        tc::mbar_init(&pp.fin, 1);
        tc::fence_mbar_init();
        pp.abort = *(const volatile int32_t *)err != 0 ? 1 : 0;  // a timeout earlier in this launch
    }
    __syncwarp();
    if (warp == 0) {
        tc::tmem_alloc(&pp.tmem, 512);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    return pp.tmem;
}

// A bounded wait of a whole warp (the outcome is the same on every lane).
__device__ __forceinline__ bool warp_wait(uint64_t *bar, uint32_t parity) {
    return __all_sync(0xffffffffu, tc::mbar_wait(bar, parity, kWaitCycles));
}

// Position in the A ring: slot and the parity of its current use.
struct RingPos {
    int a = 0;
    uint32_t ph = 0;
    __device__ __forceinline__ void next(int RING) {
        if (++a == RING) {
            a = 0;
            ph ^= 1u;
        }
    }
};

// The MMAs of one K chunk: for each A slice sa the pairs (sa, t = 0 .. S-1-sa), one MMA per K step over
// the S - sa B tiles, or, above N = 256, two halves of them (ceil and floor of (S - sa) / 2 tiles: each at
// most 256 columns, starting on a whole tile, so on a swizzle atom), issued K step by K step so that
// consecutive MMAs alternate between the halves' columns: an MMA that accumulates into the columns of the
// one just issued waits for it (about 97 cycles at this size, against about 60 for other columns), and
// equal halves leave no narrow piece whose fixed cost exceeds its work. nks: K steps of this chunk;
// negm: bit ks set: B negated on K step ks; first: the chunk's first MMA overwrites the accumulators.
template <int TN, int F>
__device__ __forceinline__ bool mma_chunk(PPipe &pp, uint32_t lead, uint32_t tm, uint32_t sA, uint32_t bset, int S, int RING,
                                          RingPos &pos, int nks, uint32_t negm, bool first) {
    const uint64_t bd = tc::sdesc_sw128(bset);
    for (int sa = 0; sa < S; sa++) {
        if (!warp_wait(&pp.fullA[pos.a], pos.ph)) return false;
        tc::fence_after_sync();
        const uint64_t ad = tc::sdesc_sw128(sA + (uint32_t)pos.a * 16384u);
        const uint32_t d0 = tm + (uint32_t)(sa * TN);
        const int nb = S - sa;
        if (nb * TN <= 256) {
            const uint32_t id = tc::idesc_digits<F>(128, nb * TN);
#pragma unroll
            for (int ks = 0; ks < 4; ks++)
                if (ks < nks)
                    tc::mma_digits<F>(lead, d0, ad + 2 * ks, bd + 2 * ks, id | ((negm >> ks & 1u) << 14),
                                      (first && sa == 0 && ks == 0) ? 0u : 1u);
        } else {
            const int h = (nb + 1) / 2;
            const uint32_t id0 = tc::idesc_digits<F>(128, h * TN), id1 = tc::idesc_digits<F>(128, (nb - h) * TN);
            const uint32_t d1 = d0 + (uint32_t)(h * TN);
            const uint64_t bd1 = bd + (uint64_t)(h * TN * 128 / 16);
#pragma unroll
            for (int ks = 0; ks < 4; ks++)
                if (ks < nks) {
                    const uint32_t neg = (negm >> ks & 1u) << 14, acc = (first && sa == 0 && ks == 0) ? 0u : 1u;
                    tc::mma_digits<F>(lead, d0, ad + 2 * ks, bd + 2 * ks, id0 | neg, acc);
                    tc::mma_digits<F>(lead, d1, ad + 2 * ks, bd1 + 2 * ks, id1 | neg, acc);
                }
        }
        tc::mma_commit(lead, &pp.emptyA[pos.a]);
        pos.next(RING);
    }
    return true;
}

// The common end: the timeout, and tensor memory back (every issued MMA has completed by then).
__device__ __forceinline__ void pipe_end(PPipe &pp, uint32_t tm, int32_t *err) {
    if (*(volatile int *)&pp.abort && threadIdx.x == 0) atomicExch(err, (int)NAO_ERR_TIMEOUT);
    tc::fence_before_sync();
    __syncthreads();
    if ((threadIdx.x >> 5) == 0) tc::tmem_dealloc(tm, 512);
}

struct HItem {  // geometry of one H work item
    const uint8_t *base, *b0;
    size_t blk;
    uint32_t b_bytes;
    int n_kc, kc0, kc1, neg16, b, m, N, tj, R16;  // K chunks [kc0, kc1) of the item's segment
    HTask task;
};

template <int TN, int F>
__device__ __forceinline__ HItem h_item(const DevSystem &s, const HTask *work, int32_t w, const uint8_t *slices,
                                        const int64_t *sl_off, const int32_t *neg16, int S) {
    HItem h;
    const HTask it = work[w];
    h.task = it;
    h.b = it.batch;
    h.tj = it.tj();
    h.m = s.sys.bmol[h.b];
    const int P = s.batch_off[h.b + 1] - s.batch_off[h.b];
    h.N = s.rel_off[h.b + 1] - s.rel_off[h.b];
    const SplitGeom G(P, h.N, S, TN, F);
    h.R16 = G.R16;
    h.base = slices + sl_off[h.b];
    h.blk = (size_t)G.R16 * 128;
    h.b0 = h.base + (size_t)h.tj * TN * 128;
    h.b_bytes = (uint32_t)min(TN, G.R16 - h.tj * TN) * 128u;
    h.n_kc = G.n_kc;
    nao_split_h_seg_range(G.n_kc, nao_split_h_nseg(P, S, F), it.seg(), S, h.kc0, h.kc1, F);
    h.neg16 = neg16[h.b];
    return h;
}

// Persistent, warp-specialised H contraction: one CTA per SM walks the work items w =
// blockIdx.x, blockIdx.x + gridDim.x, ... The readers take an item's accumulators into registers, hand
// tensor memory back to the MMA warp ("acc_empty") and then scatter into H while the next item's MMAs
// run, so the scatter and the next item's first loads overlap the MMAs. A quadrant of the readers has one
// of the item's four row blocks.
template <int TN, int F>
__global__ void __launch_bounds__(tc_threads<TN>(), 1)
    h_tc_kernel(const __grid_constant__ DevSystem s, const HTask *__restrict__ work, int32_t w0, int32_t n_work,
                const uint8_t *__restrict__ slices, const int64_t *__restrict__ sl_off, const int32_t *__restrict__ expo,
                const int32_t *__restrict__ neg16, int S, int scatter, int32_t *__restrict__ err) {
    constexpr uint32_t B_BLOCK = TN * 128;
    constexpr int HC = TN / n_parts<TN>(), NB8 = HC / 8;  // columns per reader thread, in blocks of 8
    extern __shared__ uint8_t smem_dyn[];
    __shared__ PPipe pp;
    uint8_t *smem = align1024(smem_dyn);
    const int RING = ring_slots(S, F);
    uint8_t *sA = smem, *sB = smem + (size_t)RING * 16384;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const uint32_t tm = pipe_setup<TN>(pp, RING, err);
    volatile int *abort = &pp.abort;

    if (warp == n_readers<TN>()) {
        // ---- producer (the whole warp; one lane's copies take effect) ----
        const uint32_t lead = tc::elect_one(), sA_addr = tc::smem_addr(sA), sB_addr = tc::smem_addr(sB);
        const uint32_t fullA = tc::smem_addr(pp.fullA), fullB = tc::smem_addr(pp.fullB);
        int gk = 0;
        RingPos pos;
        pos.ph = 1u;  // the parity that an unused slot's "empty" barrier passes
        bool ok = __all_sync(0xffffffffu, *abort == 0);
        for (int w = blockIdx.x; w < n_work && ok; w += gridDim.x) {
            const HItem h = h_item<TN, F>(s, work, w0 + w, slices, sl_off, neg16, S);
            // the A tile's row blocks as runs of consecutive ones: tile offset, source offset, bytes
            uint32_t run_to[4], run_at[4], run_n[4], a_bytes = 0;
            int nrun = 0;
#pragma unroll
            for (int x = 0; x < 4; x++) {
                run_to[x] = run_at[x] = run_n[x] = 0;
                const uint32_t r = h.task.row(x);
                if (r == kNoRows) continue;
                const uint32_t at = r * 4096u, n = (uint32_t)min(32, h.R16 - (int)r * 32) * 128u;
                a_bytes += n;
                bool joined = false;
#pragma unroll
                for (int y = 0; y < 4; y++)
                    if (y == nrun - 1 && run_at[y] + run_n[y] == at && run_to[y] + run_n[y] == x * 4096u) {
                        run_n[y] += n;
                        joined = true;
                    }
                if (joined) continue;
#pragma unroll
                for (int y = 0; y < 4; y++)
                    if (y == nrun) {
                        run_to[y] = x * 4096u;
                        run_at[y] = at;
                        run_n[y] = n;
                    }
                nrun++;
            }
            const size_t step = (size_t)h.n_kc * h.blk;  // from one slice to the next
            for (int kc = h.kc0; kc < h.kc1 && ok; kc++, gk++) {
                const int bb = gk & 1, ub = gk >> 1;
                if (ub >= 1) ok = warp_wait(&pp.emptyB[bb], (ub - 1) & 1);
                if (!ok) break;
                tc::mbar_arrive_expect_tx(lead, fullB + 8u * bb, (uint32_t)S * h.b_bytes);
                const uint8_t *src = h.b0 + (size_t)kc * h.blk;
                uint32_t dst = sB_addr + (uint32_t)(bb * S) * B_BLOCK;
                for (int t = 0; t < S; t++, src += step, dst += B_BLOCK)
                    tc::bulk_g2s(lead, dst, src, h.b_bytes, fullB + 8u * bb);
                src = h.base + (size_t)kc * h.blk;
                for (int sa = 0; sa < S; sa++, src += step) {
                    ok = warp_wait(&pp.emptyA[pos.a], pos.ph);
                    if (!ok) break;
                    const uint32_t bar = fullA + 8u * pos.a;
                    dst = sA_addr + (uint32_t)pos.a * 16384u;
                    tc::mbar_arrive_expect_tx(lead, bar, a_bytes);
                    tc::bulk_g2s(lead, dst + run_to[0], src + run_at[0], run_n[0], bar);
                    if (nrun > 1) {
#pragma unroll
                        for (int y = 1; y < 4; y++)
                            if (y < nrun) tc::bulk_g2s(lead, dst + run_to[y], src + run_at[y], run_n[y], bar);
                    }
                    pos.next(RING);
                }
            }
            ok = ok && __all_sync(0xffffffffu, *abort == 0);
        }
        if (!ok && lane == 0) *abort = 1;
        __syncwarp();
    } else if (warp == n_readers<TN>() + 1) {
        // ---- MMA issuer (the whole warp; one lane's tcgen05 instructions take effect) ----
        const uint32_t lead = tc::elect_one();
        const uint32_t sA_addr = tc::smem_addr(sA), sB_addr = tc::smem_addr(sB);
        int gk = 0;
        uint32_t t = 0;
        RingPos pos;
        bool ok = __all_sync(0xffffffffu, *abort == 0);
        for (int w = blockIdx.x; w < n_work && ok; w += gridDim.x, t++) {
            const HItem h = h_item<TN, F>(s, work, w0 + w, slices, sl_off, neg16, S);
            // the accumulators of the previous item have been read
            if (t >= 1) ok = warp_wait(&pp.acc_empty, (t - 1) & 1u);
            tc::fence_after_sync();
            for (int kc = h.kc0; kc < h.kc1 && ok; kc++, gk++) {
                const int bb = gk & 1;
                ok = warp_wait(&pp.fullB[bb], (uint32_t)(gk >> 1) & 1u);
                if (!ok) break;
                const int nn = min(max(h.neg16 - kc * 4, 0), 4);  // negated K steps of this chunk
                ok = mma_chunk<TN, F>(pp, lead, tm, sA_addr, sB_addr + (uint32_t)bb * S * B_BLOCK, S, RING, pos, 4,
                                      (1u << nn) - 1u, kc == h.kc0);
                if (ok) tc::mma_commit(lead, &pp.emptyB[bb]);
            }
            if (ok) tc::mma_commit(lead, &pp.acc_full);  // this item's accumulators are complete
            ok = ok && __all_sync(0xffffffffu, *abort == 0);
        }
        if (!ok && lane == 0) *abort = 1;
        // every issued MMA has completed before tensor memory is released
        tc::mma_commit(lead, &pp.fin);
        if (!warp_wait(&pp.fin, 0) && lane == 0) *abort = 1;
    } else {
        // ---- accumulator readers and scatter ----
        uint32_t t = 0;
        const int quad = warp & 3, part = warp >> 2;
        const uint32_t tm_row = tm + ((uint32_t)(quad * 32) << 16) + (uint32_t)(part * HC);
        for (int w = blockIdx.x; w < n_work; w += gridDim.x, t++) {
            const HItem h = h_item<TN, F>(s, work, w0 + w, slices, sl_off, neg16, S);
            const uint32_t rb = h.task.row(quad);
            const int i = (int)rb * 32 + lane;
            const bool row_ok = rb != kNoRows && i < h.N;
            const int32_t *rel = s.rel_idx + s.rel_off[h.b];
            const int32_t *ex = expo + s.rel_off[h.b];
            const int ei = row_ok ? ex[i] : -10000;
            const int64_t gi = row_ok ? rel[i] : 0;
            if (*abort || !tc::mbar_wait(&pp.acc_full, t & 1u, kWaitCycles)) *abort = 1;
            if (__any_sync(0xffffffffu, *abort != 0)) break;
            tc::fence_after_sync();
            int p[NB8][n_pairs<F>()][8];
            if (rb != kNoRows) {
                const bool small = small_groups<F>((h.kc1 - h.kc0) * nao_chunk_cols(F), S);
#pragma unroll
                for (int c8 = 0; c8 < NB8; c8++) read_pairs8<TN, F>(tm_row + 8 * c8, S, small, p[c8]);
            }
            // tensor memory is free for the next item
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&pp.acc_empty);
            if (scatter && row_ok) {
                // 48-wide tiles lie on or above the diagonal; the 32-wide ones are whole blocks off it
                // (either triangle) and the upper triangle on it
                const bool whole = TN == 32 && (int)rb != h.tj;
#pragma unroll
                for (int c8 = 0; c8 < NB8; c8++)
#pragma unroll
                    for (int c = 0; c < 8; c++) {
                        const int j = h.tj * TN + part * HC + 8 * c8 + c;
                        if (j >= h.N || (!whole && j < i)) continue;
                        const int ej = ex[j];
                        long long hi, lo, lo2;
                        pair_parts<F>(p[c8], c, hi, lo, lo2);
                        int tier;
                        const long long v = h_int<F>(hi, lo, lo2, tier);
                        const double x = (ei > -10000 && ej > -10000) ? (double)v * pow2(ei + ej - h_unit<F>(tier)) : 0.0;
                        const int64_t gj = rel[j];
                        h_add(s, h.m, gi < gj ? gi : gj, gi < gj ? gj : gi, x);
                    }
            }
            __syncwarp();
        }
    }
    pipe_end(pp, tm, err);
}

// Density contraction, persistent and warp-specialised as h_tc_kernel: one CTA per SM walks
// the work items (batch, 128-point tile, nJ TN-function tiles) w = blockIdx.x, blockIdx.x +
// gridDim.x, ...; each item is nJ accumulations T_qJ = Phi_q P'_J (K = the functions up to
// tile J's group, where P' is nonzero, in whole K steps), one after another through the single accumulator set.
// The readers take tile J's accumulators, hand tensor memory back and then add sum_j T_qj phi_qj to
// the point's sums in registers while tile J+1's MMAs run (products and their sums over eight functions
// as float-floats: on the FP64 pipe, two lanes per clock, this took longer than the MMAs); after the last tile the column parts' sums are added and
// stored (no atomics: one item owns each point).
// GRADN (density gradient, Sec. 2): P' = P over all of K, and the epilogue also forms
// grad n_q = 2 sum_j T_qj grad phi_qj from the rows [phi | grad phi] of 4 Ppad.
struct NItem {  // geometry of one density work item
    const uint8_t *a0, *b0;  // A: slice 0, chunk 0 of the point tile; B: slice 0, chunk 0, tile 0
    size_t a_s, a_kc, b_s, b_kc;
    uint32_t a_bytes;
    int nJ, n_ks, R16, b, m, p0, P, Ppad, N, ti;  // n_ks: K steps of all functions
};

template <int TN, int F>
__device__ __forceinline__ NItem n_item(const DevSystem &s, const HWork *work, int32_t w, const uint8_t *slices,
                                        const int64_t *sl_off, int S) {
    NItem h;
    const HWork it = work[w];  // batch, 128-point tile, number of TN-function tiles
    h.b = it.batch;
    h.ti = it.ti;
    h.nJ = it.tj;
    h.m = s.sys.bmol[h.b];
    h.p0 = s.batch_off[h.b];
    h.P = s.batch_off[h.b + 1] - h.p0;
    h.Ppad = (h.P + NAO_PPAD - 1) & ~(NAO_PPAD - 1);
    h.N = s.rel_off[h.b + 1] - s.rel_off[h.b];
    const SplitGeom G(h.P, h.N, S, TN, F);
    const uint8_t *base = slices + sl_off[h.b];
    h.a0 = base + G.nA_block(0, 0) + (size_t)it.ti * 128 * 128;
    h.a_s = (size_t)G.n_kcN * G.P16 * 128;
    h.a_kc = (size_t)G.P16 * 128;
    h.b0 = base + G.nB_block(S, 0, 0);
    h.b_s = (size_t)G.n_kcN * G.R16 * 128;
    h.b_kc = (size_t)G.R16 * 128;
    h.a_bytes = (uint32_t)min(128, G.P16 - it.ti * 128) * 128u;
    constexpr int KS = nao_kstep_cols(F);
    h.n_ks = (h.N + KS - 1) / KS;
    h.R16 = G.R16;
    return h;
}

// K steps of tile J: P' is zero for basis functions beyond the GW-function group of the tile's last one
// (all of K for GRADN)
template <int TN, bool GRADN, int F>
__device__ __forceinline__ int n_item_ks(const NItem &h, int J, int S) {
    constexpr int KS = nao_kstep_cols(F);
    const int GW = nao_split_tn(S, F);
    return GRADN ? h.n_ks : min(h.n_ks, (((J + 1) * TN + GW - 1) / GW * GW + KS - 1) / KS);
}

// MODE 0: n; 1: n and grad n (GRADN); 2: the density Hessian's first pass (A = Phi: n, grad n and
// 2 sum_j T_qj d_a d_b phi_qj into hess); 3: a later pass (A = d_hc Phi: hess_(hc, b) +=
// 2 sum_j T_qj d_b phi_qj for b >= hc). Modes 0, 1 read the float-float evaluation at scr_off,
// modes 2, 3 the Hessian's 10-row FP64 evaluation at eoff.
template <int TN, int MODE, int F>
__global__ void __launch_bounds__(tc_threads<TN>(), 1)
    n_tc_kernel(const __grid_constant__ DevSystem s, const HWork *__restrict__ work, int32_t w0, int32_t n_work,
                const uint8_t *__restrict__ slices, const int64_t *__restrict__ sl_off, const int32_t *__restrict__ expo_q,
                const int32_t *__restrict__ expo_b, const void *__restrict__ scratch_v,
                const int64_t *__restrict__ eoff, int S, int hc, double *__restrict__ hess,
                int32_t *__restrict__ err) {
    constexpr bool GRADN = MODE >= 1;  // P' over all of K
    constexpr int NC = MODE == 0 ? 1 : (MODE == 1 ? 4 : (MODE == 2 ? 10 : 3));  // sums per point
    constexpr int R0 = MODE == 3 ? 1 : 0;  // the first row of the evaluation that they take
    using V = typename std::conditional<(MODE >= 2), double, FF2>::type;
    const V *scratch = static_cast<const V *>(scratch_v);
    constexpr uint32_t B_BLOCK = TN * 128;
    constexpr int PARTS = n_parts<TN>(), HC = TN / PARTS, NB8 = HC / 8;
    extern __shared__ uint8_t smem_dyn[];
    __shared__ PPipe pp;
    uint8_t *smem = align1024(smem_dyn);
    const int RING = ring_slots(S, F);
    uint8_t *sA = smem, *sB = smem + (size_t)RING * 16384;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const uint32_t tm = pipe_setup<TN>(pp, RING, err);
    volatile int *abort = &pp.abort;

    if (warp == n_readers<TN>()) {
        // ---- producer ----
        const uint32_t lead = tc::elect_one(), sA_addr = tc::smem_addr(sA), sB_addr = tc::smem_addr(sB);
        const uint32_t fullA = tc::smem_addr(pp.fullA), fullB = tc::smem_addr(pp.fullB);
        int gk = 0;
        RingPos pos;
        pos.ph = 1u;
        bool ok = __all_sync(0xffffffffu, *abort == 0);
        for (int w = blockIdx.x; w < n_work && ok; w += gridDim.x) {
            const NItem h = n_item<TN, F>(s, work, w0 + w, slices, sl_off, S);
            for (int J = 0; J < h.nJ && ok; J++) {
                const int nk = (n_item_ks<TN, GRADN, F>(h, J, S) + 3) / 4;
                const uint8_t *bJ = h.b0 + (size_t)J * TN * 128;
                const uint32_t b_bytes = (uint32_t)min(TN, h.R16 - J * TN) * 128u;
                for (int kc = 0; kc < nk && ok; kc++, gk++) {
                    const int bb = gk & 1, ub = gk >> 1;
                    if (ub >= 1) ok = warp_wait(&pp.emptyB[bb], (ub - 1) & 1);
                    if (!ok) break;
                    tc::mbar_arrive_expect_tx(lead, fullB + 8u * bb, (uint32_t)S * b_bytes);
                    const uint8_t *src = bJ + kc * h.b_kc;
                    uint32_t dst = sB_addr + (uint32_t)(bb * S) * B_BLOCK;
                    for (int t = 0; t < S; t++, src += h.b_s, dst += B_BLOCK)
                        tc::bulk_g2s(lead, dst, src, b_bytes, fullB + 8u * bb);
                    src = h.a0 + kc * h.a_kc;
                    for (int sa = 0; sa < S; sa++, src += h.a_s) {
                        ok = warp_wait(&pp.emptyA[pos.a], pos.ph);
                        if (!ok) break;
                        const uint32_t bar = fullA + 8u * pos.a;
                        tc::mbar_arrive_expect_tx(lead, bar, h.a_bytes);
                        tc::bulk_g2s(lead, sA_addr + (uint32_t)pos.a * 16384u, src, h.a_bytes, bar);
                        pos.next(RING);
                    }
                }
                ok = ok && __all_sync(0xffffffffu, *abort == 0);
            }
        }
        if (!ok && lane == 0) *abort = 1;
        __syncwarp();
    } else if (warp == n_readers<TN>() + 1) {
        // ---- MMA issuer ----
        const uint32_t lead = tc::elect_one();
        const uint32_t sA_addr = tc::smem_addr(sA), sB_addr = tc::smem_addr(sB);
        int gk = 0;
        uint32_t t = 0;
        RingPos pos;
        bool ok = __all_sync(0xffffffffu, *abort == 0);
        for (int w = blockIdx.x; w < n_work && ok; w += gridDim.x) {
            const NItem h = n_item<TN, F>(s, work, w0 + w, slices, sl_off, S);
            for (int J = 0; J < h.nJ && ok; J++, t++) {
                const int ks = n_item_ks<TN, GRADN, F>(h, J, S);
                // the accumulators of the previous tile have been read
                if (t >= 1) ok = warp_wait(&pp.acc_empty, (t - 1) & 1u);
                tc::fence_after_sync();
                for (int kc = 0; 4 * kc < ks && ok; kc++, gk++) {
                    const int bb = gk & 1;
                    ok = warp_wait(&pp.fullB[bb], (uint32_t)(gk >> 1) & 1u);
                    if (!ok) break;
                    ok = mma_chunk<TN, F>(pp, lead, tm, sA_addr, sB_addr + (uint32_t)bb * S * B_BLOCK, S, RING, pos,
                                          min(4, ks - 4 * kc), 0u, kc == 0);
                    if (ok) tc::mma_commit(lead, &pp.emptyB[bb]);
                }
                if (ok) tc::mma_commit(lead, &pp.acc_full);  // tile J's accumulators are complete
                ok = ok && __all_sync(0xffffffffu, *abort == 0);
            }
        }
        if (!ok && lane == 0) *abort = 1;
        // every issued MMA has completed before tensor memory is released
        tc::mma_commit(lead, &pp.fin);
        if (!warp_wait(&pp.fin, 0) && lane == 0) *abort = 1;
    } else {
        // ---- accumulator readers and the n epilogue ----
        uint32_t t = 0, x = 0;  // accumulations read, exchanges made
        const int quad = warp & 3, part = warp >> 2;
        const uint32_t tm_row = tm + ((uint32_t)(quad * 32) << 16) + (uint32_t)(part * HC);
        bool ok = __all_sync(0xffffffffu, *abort == 0);
        for (int w = blockIdx.x; w < n_work && ok; w += gridDim.x) {
            const NItem h = n_item<TN, F>(s, work, w0 + w, slices, sl_off, S);
            const int q = h.ti * 128 + quad * 32 + lane;
            const bool row_ok = q < h.P;
            const bool any_row = h.ti * 128 + quad * 32 < h.P;
            const int64_t ld = MODE >= 2 ? 10 * (int64_t)h.Ppad : (GRADN ? 4 * (int64_t)h.Ppad : (int64_t)h.Ppad);
            const V *E = scratch + eoff[h.b] + (int64_t)R0 * h.Ppad + (row_ok ? q : 0);
            const bool small = small_groups<F>(h.n_ks * nao_kstep_cols(F), S);
            double tot[NC];
#pragma unroll
            for (int d = 0; d < NC; d++) tot[d] = 0.0;
            for (int J = 0; J < h.nJ && ok; J++, t++) {
                const int j0 = J * TN + part * HC, jn = min(HC, h.N - j0);
                // a single sum's phi arrive while this tile's MMAs run (more sums' values would not fit in
                // registers, and prefetching them to L2 costs more than it gives)
                V f0[MODE == 0 ? HC : 1];
                if constexpr (MODE == 0)
#pragma unroll
                    for (int c = 0; c < HC; c++) f0[c] = row_ok && c < jn ? load_once(E + (j0 + c) * ld) : V(0);
                if (*abort || !tc::mbar_wait(&pp.acc_full, t & 1u, kWaitCycles)) *abort = 1;
                if (__any_sync(0xffffffffu, *abort != 0)) {
                    ok = false;
                    break;
                }
                tc::fence_after_sync();
                // the joined integers of all columns before tensor memory is handed back, the float-floats
                // after; beside several sums, or with 16 columns, the integers do not fit in registers
                // and become float-floats at once
                constexpr bool NOW = NB8 > 1 || NC > 1;
                ffa::F tv[HC];
                int p[NB8][n_pairs<F>()][8];
                if (any_row)
#pragma unroll
                    for (int c8 = 0; c8 < NB8; c8++) {
                        read_pairs8<TN, F>(tm_row + 8 * c8, S, small, p[c8]);
                        if (NOW)
#pragma unroll
                            for (int c = 0; c < 8; c++) tv[8 * c8 + c] = pair_ff<F>(p[c8], c);
                    }
                // tensor memory is free for the next tile
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&pp.acc_empty);
                if (any_row && !NOW)
#pragma unroll
                    for (int c = 0; c < HC; c++) tv[c] = pair_ff<F>(p[c / 8], c % 8);
                if (row_ok) {
                    const V *f = E + (int64_t)j0 * ld;
                    // eight columns' products are summed as float-floats, and these in FP64
                    constexpr int CB = NC == 1 ? 8 : (NC <= 4 ? 4 : 2);  // columns whose loads are in flight together
#pragma unroll
                    for (int c8 = 0; c8 < HC; c8 += 8) {
                        ffa::F sum[NC];
                        float rest[NC];
#pragma unroll
                        for (int d = 0; d < NC; d++) {
                            sum[d] = ffa::F{0.0f, 0.0f};
                            rest[d] = 0.0f;
                        }
#pragma unroll
                        for (int c = c8; c < c8 + 8; c += CB) {
                            V fv[CB][NC];
#pragma unroll
                            for (int y = 0; y < CB; y++)
#pragma unroll
                                for (int d = 0; d < NC; d++) fv[y][d] = MODE == 0 ? f0[MODE == 0 ? c + y : 0] : (c + y < jn ? load_once(f + (c + y) * ld + d * h.Ppad) : V(0));
#pragma unroll
                            for (int y = 0; y < CB; y += 2) {
                                // (of an odd last column's neighbour the value is zero and T, whatever integers it
                                // came from, finite)
                                if (c + y < jn)
#pragma unroll
                                    for (int d = 0; d < NC; d++)
                                        ff_mac2(sum[d], rest[d], tv[c + y], ff_of_value(fv[y][d]), tv[c + y + 1],
                                                ff_of_value(fv[y + 1][d]));
                            }
                        }
#pragma unroll
                        for (int d = 0; d < NC; d++)
                            tot[d] += __dadd_rn(ffa::widen(sum[d].h), __dadd_rn(ffa::widen(sum[d].l), ffa::widen(rest[d])));
                    }
                }
                __syncwarp();
            }
            if (!ok) break;
            // the parts' sums from the last part's warp of the quadrant to the first's, each adding its own
#pragma unroll
            for (int d = 0; d < NC; d++, x++) {
                if (part < PARTS - 1) {
                    if (!tc::mbar_wait(&pp.part_full[quad][part], x & 1u, kWaitCycles)) *abort = 1;
                    tot[d] += pp.part[quad][lane];
                } else if (!tc::mbar_wait(&pp.part_empty[quad], (x & 1u) ^ 1u, kWaitCycles)) {
                    *abort = 1;
                }
                if (part > 0) pp.part[quad][lane] = tot[d];
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(part > 0 ? &pp.part_full[quad][part - 1] : &pp.part_empty[quad]);
            }
            if (__any_sync(0xffffffffu, *abort != 0)) break;
            if (part == 0 && row_ok) {
                const int eq = expo_q[h.p0 + q], eb = split_bits::exponent_of_binade(expo_b[h.b]);
                const bool live = eq > -10000 && eb > -10000;
                const double sc = pow2(eq + eb - kTUnit);
                if (MODE <= 2) *n_at(s, h.m, h.p0 + q) = live ? tot[0] * sc : 0.0;
                if (MODE == 1 || MODE == 2)
#pragma unroll
                    for (int d = 0; d < 3; d++) *gn_at(s, h.m, h.p0 + q, d) = live ? 2.0 * tot[NC > 3 ? 1 + d : 0] * sc : 0.0;
                if (MODE >= 2) {
                    // hess: component-major (xx, xy, xz, yy, yz, zz), the system's original point order
                    const int64_t np = s.sys.np[h.m], o = s.perm[h.p0 + q] - s.sys.poff[h.m];
                    if (MODE == 2) {
#pragma unroll
                        for (int k = 0; k < 6; k++) hess[k * np + o] = live ? 2.0 * tot[NC > 9 ? 4 + k : 0] * sc : 0.0;
                    } else {
                        // pair (hc, b) of components 1..3 -> 0, 1, 2 (x.), 3, 4 (y.), 5 (zz)
                        const int kb = (hc - 1) * 3 - ((hc - 1) * (hc - 2)) / 2 - hc;
#pragma unroll
                        for (int d = 0; d < 3; d++)
                            if (d + 1 >= hc && live) hess[(kb + d + 1) * np + o] += 2.0 * tot[NC > 2 ? d : 0] * sc;
                    }
                }
            }
        }
    }
    pipe_end(pp, tm, err);
}

// sum over each density tile of 64 points of w n (then the deterministic final reduction), a warp per tile
// (a CTA per tile: 78 us for 64 atoms, 1.2 million points; now 20)
constexpr int kWnWarps = 8;
__global__ void __launch_bounds__(32 * kWnWarps) wn_partial_kernel(const __grid_constant__ DevSystem s, const DWork *__restrict__ work,
                                                                   int32_t w0, int32_t n_work, double *__restrict__ ne_part) {
    const int w = blockIdx.x * kWnWarps + (threadIdx.x >> 5);
    if (w >= n_work) return;
    const DWork it = work[w0 + w];
    const int p0 = s.batch_off[it.batch], P = s.batch_off[it.batch + 1] - p0, m = s.sys.bmol[it.batch];
    double wn[2];
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const int q = it.tp * NAO_TILE + 32 * h + (int)(threadIdx.x & 31);
        wn[h] = q < P ? s.pw[p0 + q] * *n_at(s, m, p0 + q) : 0.0;
    }
#pragma unroll
    for (int h = 0; h < 2; h++)
        for (int o = 16; o > 0; o >>= 1) wn[h] += __shfl_xor_sync(0xffffffffu, wn[h], o);
    if ((threadIdx.x & 31) == 0) ne_part[w0 + w] = wn[0] + wn[1];
}

// The timeout path of the bounded waits, exercised without a stuck pipeline: one thread waits on
// an mbarrier that expects one arrival which never comes (no copy or MMA is in flight, so giving
// up leaves nothing behind), then records the timeout the way the contraction kernels do.
__global__ void wait_timeout_probe_kernel(long long max_cycles, int32_t *__restrict__ err) {
    __shared__ uint64_t bar;
    tc::mbar_init(&bar, 1);
    tc::fence_mbar_init();
    if (!tc::mbar_wait(&bar, 0, max_cycles)) {
        atomicExch(err + 1, 1);
        atomicExch(err, (int)NAO_ERR_TIMEOUT);
    }
}

// Point exponents of the Hessian's four A operands (phi and the three gradient components, rows
// c = 0..3 of the 10-row FP64 evaluation): expo4[c n_points + batch_off[b] + q] from the binade
// of max_i |row c of function i at point q|. Clears the batch's exponent of P' for slice_nphi_kernel.
__global__ void __launch_bounds__(256) hess_point_expo_kernel(const __grid_constant__ DevSystem s, int32_t b0,
                                                             const double *__restrict__ scratch,
                                                             const int64_t *__restrict__ hoff, int32_t *__restrict__ expo4,
                                                             int64_t n_points, int32_t *__restrict__ expo_b) {
    const int b = b0 + blockIdx.x;
    const int p0 = s.batch_off[b], P = s.batch_off[b + 1] - p0;
    const int Ppad = (P + NAO_PPAD - 1) & ~(NAO_PPAD - 1);
    const int N = s.rel_off[b + 1] - s.rel_off[b];
    const double *E = scratch + hoff[b];
    const int64_t ld = 10 * (int64_t)Ppad;
    // blockIdx.y: component and 32-point tile; the eight warps share the rows, a lane per point
    __shared__ int red[8][32];
    const int c = blockIdx.y & 3, q = 32 * (blockIdx.y >> 2) + (threadIdx.x & 31), warp = threadIdx.x >> 5;
    if (blockIdx.y == 0 && threadIdx.x == 0) expo_b[b] = 0;
    if (32 * (int)(blockIdx.y >> 2) >= P) return;
    int mx = 0;
    if (q < P) {
        const double *col = E + (int64_t)c * Ppad + q;
#pragma unroll 8
        for (int i = warp; i < N; i += 8) mx = max(mx, split_bits::biased_exponent(abs_bits(__ldg(col + i * ld))));
    }
    red[warp][threadIdx.x & 31] = mx;
    __syncthreads();
    if (warp == 0 && q < P) {
#pragma unroll
        for (int w = 1; w < 8; w++) mx = max(mx, red[w][threadIdx.x]);
        expo4[c * n_points + p0 + q] = split_bits::exponent_of_binade(mx);
    }
}

}  // namespace

size_t split_smem_bytes(int S, int F) { return pipe_smem_bytes(S, F); }

cudaError_t launch_wait_timeout_probe(long long max_cycles, int32_t *err, cudaStream_t st) {
    wait_timeout_probe_kernel<<<1, 1, 0, st>>>(max_cycles, err);
    return cudaGetLastError();
}

cudaError_t split_configure() {
    size_t bytes = 0;
    for (int S = 4; S <= NAO_SPLIT_MAX_SLICES; S++) bytes = std::max(bytes, split_smem_bytes(S, NAO_DIGITS_BF16));
    for (int S = 8; S <= NAO_SPLIT_MAX_SLICES_E4M3; S++) bytes = std::max(bytes, split_smem_bytes(S, NAO_DIGITS_E4M3));
    const void *fns[] = {(const void *)h_tc_kernel<48, 0>,    (const void *)h_tc_kernel<32, 0>,
                         (const void *)h_tc_kernel<32, 1>,    (const void *)n_tc_kernel<48, 0, 0>,
                         (const void *)n_tc_kernel<48, 1, 0>, (const void *)n_tc_kernel<48, 2, 0>,
                         (const void *)n_tc_kernel<48, 3, 0>, (const void *)n_tc_kernel<32, 0, 0>,
                         (const void *)n_tc_kernel<32, 1, 0>, (const void *)n_tc_kernel<32, 2, 0>,
                         (const void *)n_tc_kernel<32, 3, 0>, (const void *)n_tc_kernel<32, 0, 1>,
                         (const void *)n_tc_kernel<32, 1, 1>, (const void *)n_tc_kernel<32, 2, 1>,
                         (const void *)n_tc_kernel<32, 3, 1>};
    for (const void *f : fns) {
        const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Slice counts with compiled slicers: 4..12 with bf16 digits, 8..16 with e4m3 digits.
#define NAO_SPLIT_DISPATCH(S, F, CALL)                                                                 \
    if (F == NAO_DIGITS_E4M3) {                                                                        \
        switch (S) {                                                                                   \
            case 8: CALL(8, 1); break;                                                                 \
            case 9: CALL(9, 1); break;                                                                 \
            case 10: CALL(10, 1); break;                                                               \
            case 11: CALL(11, 1); break;                                                               \
            case 12: CALL(12, 1); break;                                                               \
            case 13: CALL(13, 1); break;                                                               \
            case 14: CALL(14, 1); break;                                                               \
            case 15: CALL(15, 1); break;                                                               \
            default: CALL(16, 1); break;                                                               \
        }                                                                                              \
    } else {                                                                                           \
        switch (S) {                                                                                   \
            case 4: CALL(4, 0); break;                                                                 \
            case 5: CALL(5, 0); break;                                                                 \
            case 6: CALL(6, 0); break;                                                                 \
            case 7: CALL(7, 0); break;                                                                 \
            case 8: CALL(8, 0); break;                                                                 \
            case 9: CALL(9, 0); break;                                                                 \
            case 10: CALL(10, 0); break;                                                               \
            case 11: CALL(11, 0); break;                                                               \
            default: CALL(12, 0); break;                                                               \
        }                                                                                              \
    }

cudaError_t launch_slice_h(const DevSystem &s, int32_t b0, int32_t b1, int32_t max_rt, const double *scratch, uint32_t terms, uint8_t *slices, const int64_t *sl_off, int32_t *expo,
                           int32_t *neg16, int S, int F, cudaStream_t st) {
    if (b1 <= b0 || max_rt <= 0) return cudaSuccess;
    const FF2 *ev = reinterpret_cast<const FF2 *>(scratch);  // the split path's evaluation: float-float values
    const size_t sm = slice_h_smem(s.max_ppad, F);
    // 64 rows per CTA (max_rt such tiles cover the largest batch), 16 where that gives fewer than two CTAs per
    // SM: a small system's launch is as long as one CTA (3-atom molecule, 66 batches: 41 -> 26 us)
    const int tile = (int64_t)(b1 - b0) * max_rt < 2 * s.n_sm ? 16 : 64;
    const dim3 grid(b1 - b0, max_rt * (64 / tile));
    static_assert(slice_h_smem(NAO_SPLIT_MAX_PPAD, 0) <= 47 * 1024 && slice_h_smem(NAO_SPLIT_MAX_PPAD, 1) <= 47 * 1024,
                  "the H slicer's columns exceed the shared memory of a plain launch");
#define NAO_SLICE_H(SS, FF) \
    slice_h_kernel<SS, FF><<<grid, 32 * kSliceWarps, sm, st>>>(s, b0, tile, ev, terms, slices, sl_off, expo, neg16)
    NAO_SPLIT_DISPATCH(S, F, NAO_SLICE_H)
#undef NAO_SLICE_H
    return cudaGetLastError();
}

cudaError_t launch_h_tc(const DevSystem &s, const HTask *work, int32_t w0, int32_t n_work, const uint8_t *slices,
                        const int64_t *sl_off, const int32_t *expo, const int32_t *neg16, int S, int F, int tn,
                        int scatter, int32_t *err, cudaStream_t st) {
    if (n_work <= 0) return cudaSuccess;
    const int grid = n_work < s.n_sm ? n_work : s.n_sm;  // persistent: one CTA per SM
    const size_t sm = split_smem_bytes(S, F);
    if (F == NAO_DIGITS_E4M3 && tn == 32)
        h_tc_kernel<32, 1><<<grid, tc_threads<32>(), sm, st>>>(s, work, w0, n_work, slices, sl_off, expo, neg16, S, scatter, err);
    else if (F == NAO_DIGITS_BF16 && tn == 48 && S <= 10)
        h_tc_kernel<48, 0><<<grid, tc_threads<48>(), sm, st>>>(s, work, w0, n_work, slices, sl_off, expo, neg16, S, scatter, err);
    else if (F == NAO_DIGITS_BF16 && tn == 32)
        h_tc_kernel<32, 0><<<grid, tc_threads<32>(), sm, st>>>(s, work, w0, n_work, slices, sl_off, expo, neg16, S, scatter, err);
    else
        return cudaErrorInvalidValue;
    return cudaGetLastError();
}

cudaError_t launch_slice_n(const DevSystem &s, int32_t b0, int32_t b1, int32_t max_qt, int32_t max_rt,
                           const double *scratch, uint8_t *slices, const int64_t *sl_off, const int32_t *expo_q,
                           int32_t *expo_b, int S, int F, bool grad, cudaStream_t st) {
    if (b1 <= b0) return cudaSuccess;
    const FF2 *ev = reinterpret_cast<const FF2 *>(scratch);
    // y < kPexpCtas: the exponent of P'; above: tiles of kNphiPoints points (128 max_qt >= P16)
#define NAO_SLICE_NPHI(SS, FF)                                                                            \
    slice_nphi_kernel<SS, FF, FF2><<<dim3(b1 - b0, 128 / kNphiPoints * max_qt + kPexpCtas), 32 * kNphiWarps, 0, st>>>(                        \
        s, b0, ev, s.scr_off, 0, slices, sl_off, expo_q, expo_b, grad ? 4 : 1, grad ? 1 : 0, 1)
    NAO_SPLIT_DISPATCH(S, F, NAO_SLICE_NPHI)
#undef NAO_SLICE_NPHI
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || max_rt <= 0) return e;
    // 16 rows per CTA (64 max_rt >= R16)
#define NAO_SLICE_NP(SS, FF) \
    slice_np_kernel<SS, FF><<<dim3(b1 - b0, 4 * max_rt), 256, 0, st>>>(s, b0, slices, sl_off, expo_b, grad ? 1 : 0)
    NAO_SPLIT_DISPATCH(S, F, NAO_SLICE_NP)
#undef NAO_SLICE_NP
    return cudaGetLastError();
}

cudaError_t launch_slice_n_hess(const DevSystem &s, int32_t b0, int32_t b1, int32_t max_qt, int32_t max_rt,
                                const double *scratch, const int64_t *hoff, int comp, uint8_t *slices,
                                const int64_t *sl_off, const int32_t *expo_q, int32_t *expo_b, int S, int F, cudaStream_t st) {
    if (b1 <= b0) return cudaSuccess;
    const int first = comp == 0 ? 1 : 0;  // P' (its exponent and its slices) once, with the first pass
#define NAO_SLICE_NPHI(SS, FF)                                                                                   \
    slice_nphi_kernel<SS, FF, double><<<dim3(b1 - b0, 128 / kNphiPoints * max_qt + kPexpCtas), 32 * kNphiWarps, 0, st>>>(                            \
        s, b0, scratch, hoff, comp, slices, sl_off, expo_q, expo_b, 10, 1, first)
    NAO_SPLIT_DISPATCH(S, F, NAO_SLICE_NPHI)
#undef NAO_SLICE_NPHI
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !first || max_rt <= 0) return e;
#define NAO_SLICE_NP(SS, FF) \
    slice_np_kernel<SS, FF><<<dim3(b1 - b0, 4 * max_rt), 256, 0, st>>>(s, b0, slices, sl_off, expo_b, 1)
    NAO_SPLIT_DISPATCH(S, F, NAO_SLICE_NP)
#undef NAO_SLICE_NP
    return cudaGetLastError();
}

cudaError_t launch_hess_point_expo(const DevSystem &s, int32_t b0, int32_t b1, const double *scratch, const int64_t *hoff,
                                   int32_t *expo4, int64_t n_points, int32_t *expo_b, cudaStream_t st) {
    if (b1 <= b0) return cudaSuccess;
    hess_point_expo_kernel<<<dim3(b1 - b0, 4 * ((s.max_ppad + 31) / 32)), 256, 0, st>>>(s, b0, scratch, hoff, expo4, n_points,
                                                                                      expo_b);
    return cudaGetLastError();
}

// One launch of n_tc_kernel<TN, MODE, F> for the width and digit format at hand.
static cudaError_t launch_n_tc_mode(const DevSystem &s, const HWork *work, int32_t w0, int32_t n_work,
                                    const uint8_t *slices, const int64_t *sl_off, const int32_t *expo_q,
                                    const int32_t *expo_b, const void *ev, const int64_t *eoff, int S, int F, int tn,
                                    int mode, int hc, double *hess, int32_t *err, cudaStream_t st) {
    if (n_work <= 0) return cudaSuccess;
    if (F == NAO_DIGITS_E4M3 ? tn != 32 : (tn != 32 && !(tn == 48 && S <= 10))) return cudaErrorInvalidValue;
    const size_t sm = split_smem_bytes(S, F);
    const int grid = n_work < s.n_sm ? n_work : s.n_sm;  // persistent: one CTA per SM
#define NAO_N_TC(TNV, M, FF)                                                                                  \
    n_tc_kernel<TNV, M, FF><<<grid, tc_threads<TNV>(), sm, st>>>(s, work, w0, n_work, slices, sl_off, expo_q, expo_b, ev, eoff, S, hc, \
                                                   hess, err)
#define NAO_N_TC_MODES(TNV, FF)             \
    switch (mode) {                         \
        case 0: NAO_N_TC(TNV, 0, FF); break; \
        case 1: NAO_N_TC(TNV, 1, FF); break; \
        case 2: NAO_N_TC(TNV, 2, FF); break; \
        default: NAO_N_TC(TNV, 3, FF); break; \
    }
    if (F == NAO_DIGITS_E4M3) NAO_N_TC_MODES(32, 1)
    else if (tn == 48) NAO_N_TC_MODES(48, 0)
    else NAO_N_TC_MODES(32, 0)
#undef NAO_N_TC_MODES
#undef NAO_N_TC
    return cudaGetLastError();
}

cudaError_t launch_n_tc(const DevSystem &s, const HWork *work, int32_t w0, int32_t n_work, const uint8_t *slices,
                        const int64_t *sl_off, const int32_t *expo_q, const int32_t *expo_b, const double *scratch, int S,
                        int F, int tn, bool grad, int32_t *err, cudaStream_t st) {
    return launch_n_tc_mode(s, work, w0, n_work, slices, sl_off, expo_q, expo_b, scratch, s.scr_off, S, F, tn, grad ? 1 : 0,
                            0, nullptr, err, st);
}

cudaError_t launch_n_tc_hess(const DevSystem &s, const HWork *work, int32_t w0, int32_t n_work, const uint8_t *slices,
                             const int64_t *sl_off, const int32_t *expo_q, const int32_t *expo_b, const double *scratch,
                             const int64_t *hoff, int comp, double *hess, int S, int F, int tn, int32_t *err,
                             cudaStream_t st) {
    return launch_n_tc_mode(s, work, w0, n_work, slices, sl_off, expo_q, expo_b, scratch, hoff, S, F, tn,
                            comp == 0 ? 2 : 3, comp, hess, err, st);
}

cudaError_t launch_wn_partial(const DevSystem &s, const DWork *work, int32_t w0, int32_t n_work, double *ne_part,
                              cudaStream_t st) {
    if (n_work <= 0) return cudaSuccess;
    wn_partial_kernel<<<(n_work + kWnWarps - 1) / kWnWarps, 32 * kWnWarps, 0, st>>>(s, work, w0, n_work, ne_part);
    return cudaGetLastError();
}
