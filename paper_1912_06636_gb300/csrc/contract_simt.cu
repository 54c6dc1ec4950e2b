// Batch contractions on the CUDA cores, in FP64 or FP32 (T).
//
// Hamiltonian (Eq. batch_matrix_mult with K and L stacked over the potential and the three
// gradient components): for batch B with reduced basis of size N and points padded to Ppad,
// the evaluated block E (N rows x 4 Ppad columns: phi | d/dx | d/dy | d/dz) gives
//   h[B]_ij = sum_k E_ik d_k E_jk,  d_k = w_q v_q (phi part) or w_q / 2 (gradient parts),
// computed for upper-triangular 64 x 64 tile pairs (I <= J) only and added into the global
// H[rel_i][rel_j] with FP64 atomics (the indexing step of Sec. 3.4 (ii)); a final pass
// copies the upper triangle onto the lower one, so H is exactly symmetric.
//
// Density (Eq. Density restricted to nnz(B)): n_q = sum_ij phi_iq P_ij phi_jq, evaluated per
// 64-point tile as the sum over tile pairs I <= J of c_IJ sum_{i in I, j in J} phi_iq P_ij phi_jq
// with c_II = 1 and c_IJ = 2 (I < J), which reads only P's upper triangle; I and J are groups of 64 functions in FP32
// and of 8 in FP64.
//
// FP32: products accumulate in FP32 over chunks of 32 terms; each chunk sum is folded into an
// FP32 (hi, lo) pair with Knuth's TwoSum, and hi + lo is widened to FP64 for the scatter.
//
// What bounds them: the FP64 pipe (two lanes per clock and SM, 1/64 of the FP32 rate), which FP64
// products use by definition and which every conversion between FP64 and a 32-bit type uses as
// well. So (1) a CTA's 64 x 64 tile is cut into small subtiles, up to eight per warp, and a warp
// leaves out the subtiles that lie below the diagonal, beyond the batch's functions or beyond its
// points: in FP64 8 x 8 (H) and 16 x 16 (density), in FP32 32 x 16 (with smaller ones the operands' loads
// would be too many for the FP32 rate). Which warp takes which subtile turns with the CTA's index, so that the idle ones
// spread over the SM's four schedulers. (2) The FP32 kernels convert with integer instructions and
// keep their sums over functions as float-float pairs.
#include "ff.h"
#include "nao_internal.h"

namespace {

constexpr int T_ = NAO_TILE;  // 64

// Subtile of a warp: 8 x 4 lanes of MR rows x 4 columns, SR = 8 MR rows x 16 columns; KC: K chunk
// (128 bytes of an operand row).
template <typename T> struct Cfg;
template <> struct Cfg<double> { static constexpr int KC = 16, MR = 2, SR = 16, NU = 2; };
template <> struct Cfg<float> { static constexpr int KC = 32, MR = 4, SR = 32, NU = 1; };
// The H kernel's: MR rows x MC columns per lane. In FP64 8 x 8 subtiles: the FP64 pipe is the limit, shared memory
// far from it, and they compute 1.15 times the wanted triangle of the 8-atom cluster's batches where 16 x 16 ones
// compute 1.30.
template <typename T> struct HCfg : Cfg<T> { static constexpr int MC = 4; };
template <> struct HCfg<double> { static constexpr int KC = 16, MR = 1, MC = 2, SR = 8, NU = 8; };

template <typename T> struct Vec16;  // 16 bytes of T
template <> struct Vec16<double> { using type = double2; };
template <> struct Vec16<float> { using type = float4; };
__device__ __forceinline__ double vget(const double2 &v, int e) { return e == 0 ? v.x : v.y; }
__device__ __forceinline__ float vget(const float4 &v, int e) { return e == 0 ? v.x : e == 1 ? v.y : e == 2 ? v.z : v.w; }
__device__ __forceinline__ double2 vmul(double2 v, double2 w) { return make_double2(v.x * w.x, v.y * w.y); }
__device__ __forceinline__ float4 vmul(float4 v, float4 w) { return make_float4(v.x * w.x, v.y * w.y, v.z * w.z, v.w * w.w); }

// 16 bytes global -> shared, asynchronously; zeros when !ok (nothing is read then).
__device__ __forceinline__ void cp16(void *dst, const void *src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(ok ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// FP64 -> FP32, round to nearest even, with integer instructions (the conversion instruction runs on
// the FP64 pipe). Values outside FP32's normal range take the conversion.
__device__ __forceinline__ float to_f32(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint32_t e = (hi >> 20) & 0x7FFu;
    if (e - 897u > 253u) return __double2float_rn(x);
    const uint32_t m = (hi << 12) | (lo >> 20);  // the 32 leading bits of the fraction
    const uint32_t tail = (m & 0x1FFu) << 1 | ((lo & 0xFFFFFu) != 0u ? 1u : 0u);  // the 29 dropped bits, the last one sticky
    const uint32_t f = (hi & 0x80000000u) | ((e - 896u) << 23) | (m >> 9);
    return __uint_as_float(f + (tail + 0x1FFu + (f & 1u) >= 0x400u ? 1u : 0u));
}
// (hi, lo) += x with Knuth's TwoSum (exact transformation of hi + x).
__device__ __forceinline__ void two_sum_acc(float &hi, float &lo, float x) {
    const float s = __fadd_rn(hi, x);
    const float bb = __fsub_rn(s, hi);
    const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(x, bb));
    hi = s;
    lo = __fadd_rn(lo, err);
}

// The lane's accumulators of one subtile: FP64 accumulates directly; FP32 keeps a chunk sum and a
// (hi, lo) pair.
template <typename T, int MR = Cfg<T>::MR, int MC = 4> struct Block;
template <int MR, int MC> struct Block<double, MR, MC> {
    double c[MR][MC];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int a = 0; a < MR; a++)
#pragma unroll
            for (int b = 0; b < MC; b++) c[a][b] = 0.0;
    }
    __device__ __forceinline__ void fold() {}
    __device__ __forceinline__ double value(int a, int b) const { return c[a][b]; }
};
template <int MR, int MC> struct Block<float, MR, MC> {
    float c[MR][MC], hi[MR][MC], lo[MR][MC];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int a = 0; a < MR; a++)
#pragma unroll
            for (int b = 0; b < MC; b++) c[a][b] = hi[a][b] = lo[a][b] = 0.0f;
    }
    __device__ __forceinline__ void fold() {
#pragma unroll
        for (int a = 0; a < MR; a++)
#pragma unroll
            for (int b = 0; b < MC; b++) {
                two_sum_acc(hi[a][b], lo[a][b], c[a][b]);
                c[a][b] = 0.0f;
            }
    }
    __device__ __forceinline__ double value(int a, int b) const { return __dadd_rn(ffa::widen(hi[a][b]), ffa::widen(lo[a][b])); }
};

// Shared-memory row of one K chunk: 128 bytes and 16 more, so that the eight rows that a warp reads at
// once (one per lane group) lie in different banks.
template <typename T> struct HTile {
    static constexpr int LD = 144 / sizeof(T);
    T a[2][T_][LD], b[2][T_][LD];
};

// One CTA per tile pair. Per K chunk of 128 bytes the rows of tile I come by cp.async and those of
// tile J through registers, where they take their weights; two buffers, one barrier per chunk. The
// chunks stay row-major (K along the row): a lane reads 16 bytes, 2 or 4 terms, of each of its rows
// (ly + 8 a) and columns (lx + 4 b).
// Whole 64 x 64 tiles computed 2.5 times the wanted triangle on the 8-atom cluster (batches of 75
// functions on average) and 1.9 times on the 64-atom one, 16 x 16 and 32 x 16 subtiles 1.3 times. Measured
// with the density below, H + n: 8 atoms FP64 13.7 -> 8.9 ms, 64 atoms FP32 15.7 -> 12.0 ms (H 6.7 -> 4.2, n
// 3.7 -> 2.4). In FP64 (the FP64 pipe 98 % busy) 8 x 8 subtiles then took H from 5.33 to 4.75 ms.
template <typename T>
__global__ void __launch_bounds__(256, sizeof(T) == 8 ? 3 : 2)
    h_simt_kernel(const __grid_constant__ DevSystem s, const HWork *__restrict__ work, const T *__restrict__ scratch,
                  uint32_t terms) {
    using V = typename Vec16<T>::type;
    constexpr int KC = HCfg<T>::KC, MR = HCfg<T>::MR, MC = HCfg<T>::MC, SR = HCfg<T>::SR, NU = HCfg<T>::NU, VK = 16 / sizeof(T);
    constexpr int SC = 4 * MC, NSC = T_ / SC, NS = (T_ / SR) * NSC;  // a subtile's columns, subtiles across, of the tile
    __shared__ __align__(16) HTile<T> sm;
    extern __shared__ __align__(16) unsigned char dyn[];
    const HWork it = work[blockIdx.x];
    const int b = it.batch, m = s.sys.bmol[b];
    const int p0 = s.batch_off[b], P = s.batch_off[b + 1] - p0;
    const int Ppad = (P + NAO_PPAD - 1) & ~(NAO_PPAD - 1);
    const int N = s.rel_off[b + 1] - s.rel_off[b];
    T *wt = reinterpret_cast<T *>(dyn);  // [2][Ppad]: weights of the potential part, of the gradient parts
    const int64_t ld = 4 * (int64_t)Ppad;
    const T *E = scratch + s.scr_off[b];
    const int tid = threadIdx.x, lane = tid & 31, lx = lane & 3, ly = lane >> 2;

    for (int q = tid; q < Ppad; q += blockDim.x) {
        const double w = q < P ? s.pw[p0 + q] : 0.0;
        const double vv = q < P ? v_at(s, m, p0 + q) : 1.0;
        wt[q] = T((terms & NAO_TERM_POTENTIAL) ? w * vv : 0.0);
        const double kin = (terms & NAO_TERM_KINETIC) ? 1.0 : 0.0;
        wt[Ppad + q] = T(0.5 * w * ((terms & NAO_TERM_TAU) && q < P ? kin + vt_at(s, m, p0 + q) : kin));
    }

    const int i0 = it.ti * T_, j0 = it.tj * T_;
    const bool diag = it.ti == it.tj;
    // this warp's subtiles: every eighth of the active ones (-1: none)
    int sub[NU];
    {
        int k = 0;
        const int w = ((tid >> 5) + blockIdx.x) & 7;
#pragma unroll
        for (int u = 0; u < NU; u++) sub[u] = -1;
        for (int x = 0; x < NS; x++) {
            const int r = x / NSC, c = x % NSC;
            if (i0 + r * SR >= N || j0 + c * SC >= N || (diag && c * SC + SC - 1 < r * SR)) continue;
#pragma unroll
            for (int u = 0; u < NU; u++)
                if (k == w + 8 * u) sub[u] = x;
            k++;
        }
    }
    Block<T, MR, MC> acc[NU];
#pragma unroll
    for (int u = 0; u < NU; u++) acc[u].zero();

    const int lv = tid & 7, lr = tid >> 3;  // loader: 16-byte vector lv of rows lr and lr + 32
    const T *Ar[2], *Br[2];
    bool aok[2], bok[2];
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const int r = lr + 32 * h;
        aok[h] = i0 + r < N;
        bok[h] = j0 + r < N;
        Ar[h] = E + (int64_t)(aok[h] ? i0 + r : 0) * ld;
        Br[h] = E + (int64_t)(bok[h] ? j0 + r : 0) * ld;
    }
    V bv[2];
    // this CTA's points [qa, qa + Ps) (see the launcher) and, of the next chunk's column of this vector, the
    // point after qa and the component (phi, d/dx, d/dy, d/dz)
    const int per = (Ppad / NAO_PPAD + (int)gridDim.y - 1) / (int)gridDim.y * NAO_PPAD;
    const int qa = (int)blockIdx.y * per, Ps = min(Ppad - qa, per), nk = 4 * Ps / KC;
    if (Ps <= 0) return;
    int wq = lv * VK, comp = 0;
    auto wrap = [&]() {
        while (wq >= Ps) {
            wq -= Ps;
            comp++;
        }
    };
    auto load = [&](int buf) {
        const int k = comp * Ppad + qa + wq;
#pragma unroll
        for (int h = 0; h < 2; h++) {
            cp16(&sm.a[buf][lr + 32 * h][lv * VK], Ar[h] + k, aok[h]);
            if (bok[h]) bv[h] = *reinterpret_cast<const V *>(Br[h] + k);
        }
    };
    auto store = [&](int buf) {
        const V w = *reinterpret_cast<const V *>(wt + (comp == 0 ? 0 : Ppad) + qa + wq);
#pragma unroll
        for (int h = 0; h < 2; h++) {
            V x{};
            if (bok[h]) x = vmul(bv[h], w);
            *reinterpret_cast<V *>(&sm.b[buf][lr + 32 * h][lv * VK]) = x;
        }
        wq += KC;
        wrap();
    };
    wrap();
    load(0);
    __syncthreads();  // the weights are written
    store(0);
    for (int kc = 0; kc < nk; kc++) {
        const int buf = kc & 1;
        cp_wait_all();
        __syncthreads();  // this chunk is complete, and every warp has left the other buffer
        if (kc + 1 < nk) load(buf ^ 1);
#pragma unroll
        for (int u = 0; u < NU; u++) {
            if (sub[u] < 0) continue;
            const T *a = &sm.a[buf][(sub[u] / NSC) * SR + ly][0], *bb = &sm.b[buf][(sub[u] % NSC) * SC + lx][0];
#pragma unroll
            for (int kv = 0; kv < KC; kv += VK) {
                V ra[MR], rb[MC];
#pragma unroll
                for (int x = 0; x < MR; x++) ra[x] = *reinterpret_cast<const V *>(a + 8 * x * HTile<T>::LD + kv);
#pragma unroll
                for (int y = 0; y < MC; y++) rb[y] = *reinterpret_cast<const V *>(bb + 4 * y * HTile<T>::LD + kv);
#pragma unroll
                for (int e = 0; e < VK; e++)
#pragma unroll
                    for (int x = 0; x < MR; x++)
#pragma unroll
                        for (int y = 0; y < MC; y++) acc[u].c[x][y] = fma(vget(ra[x], e), vget(rb[y], e), acc[u].c[x][y]);
            }
            acc[u].fold();
        }
        if (kc + 1 < nk) store(buf ^ 1);
    }

    const int32_t *rel = s.rel_idx + s.rel_off[b];
#pragma unroll
    for (int u = 0; u < NU; u++) {
        if (sub[u] < 0) continue;
#pragma unroll
        for (int x = 0; x < MR; x++) {
            const int i = i0 + (sub[u] / NSC) * SR + ly + 8 * x;
            if (i >= N) continue;
            const int64_t gi = rel[i];
#pragma unroll
            for (int y = 0; y < MC; y++) {
                const int j = j0 + (sub[u] % NSC) * SC + lx + 4 * y;
                if (j >= N || (diag && j < i)) continue;
                h_add(s, m, gi, rel[j], acc[u].value(x, y));
            }
        }
    }
}

// Copy the upper triangle of each system's H onto its lower one, through 32 x 32 tiles; one
// CTA per task (system, column tile bx, row tile by) with by <= bx.
// In the deterministic mode the upper triangle comes from the fixed-point accumulators, converted
// once here (and written to both triangles).
__global__ void mirror_kernel(DevSystem s, const int4 *__restrict__ tasks) {
    __shared__ double tile[32][33];
    const int4 tk = tasks[blockIdx.x];
    const int m = tk.x, bx = tk.y, by = tk.z;
    double *H = s.sys.H[m];
    const unsigned long long *acc = s.sys.Hacc[m];
    const int64_t nb = s.sys.nbm[m];
    const int tx = threadIdx.x, ty = threadIdx.y;
    for (int r = ty; r < 32; r += blockDim.y) {
        const int64_t row = (int64_t)by * 32 + r, col = (int64_t)bx * 32 + tx;
        double h = 0.0;
        if (row < nb && col < nb) {
            if (acc) {
                if (row <= col) {
                    h = det_value(acc + 2 * (row * nb + col));
                    H[row * nb + col] = h;
                }
            } else {
                h = H[row * nb + col];
            }
        }
        tile[r][tx] = h;
    }
    __syncthreads();
    for (int r = ty; r < 32; r += blockDim.y) {
        const int64_t row = (int64_t)bx * 32 + r, col = (int64_t)by * 32 + tx;  // destination, lower part
        if (row < nb && col < nb && row > col) H[row * nb + col] = tile[tx][r];
    }
}

// H = 0 for each task (system, first element, count); in the deterministic mode its fixed-point
// accumulators instead (H itself is then written whole by the mirror pass).
__global__ void __launch_bounds__(256) zero_h_kernel(DevSystem s, const int4 *__restrict__ tasks) {
    const int4 tk = tasks[blockIdx.x];
    unsigned long long *acc = s.sys.Hacc[tk.x];
    if (acc) {
        acc += 2 * ((int64_t)tk.y * 65536);
        for (int i = threadIdx.x; i < 2 * tk.z; i += blockDim.x) acc[i] = 0ULL;
        return;
    }
    double *H = s.sys.H[tk.x] + (int64_t)tk.y * 65536;
    for (int i = threadIdx.x; i < tk.z; i += blockDim.x) H[i] = 0.0;
}

// Sums over functions of T_qj f_qj: in FP64, or as a float-float on the FP32 path (T there is a
// (hi, lo) pair and f an FP32; the products are exact but for the 2^-48 terms).
template <typename T> struct PointSum;
template <> struct PointSum<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(const Block<double> &t, int a, int b, double f) { s += t.c[a][b] * f; }
    __device__ __forceinline__ double value() const { return s; }
};
template <> struct PointSum<float> {
    float h = 0.0f, l = 0.0f;
    __device__ __forceinline__ void add(const Block<float> &t, int a, int b, float f) {
        const float p = __fmul_rn(t.hi[a][b], f);
        const float e = __fmaf_rn(t.lo[a][b], f, __fmaf_rn(t.hi[a][b], f, -p));
        two_sum_acc(h, l, p);
        l = __fadd_rn(l, e);
    }
    __device__ __forceinline__ double value() const { return __dadd_rn(ffa::widen(h), ffa::widen(l)); }
};

// GRADN: the density gradient too (Sec. 2; grad n = 2 sum_ij grad phi_i P_ij phi_j): with
// T_qj = sum_i phi_qi P_ij over all of P (no tile-pair symmetry), n_q = sum_j T_qj phi_qj and
// grad n_q = 2 sum_j T_qj grad phi_qj; the scratch rows then hold [phi | d/dx | d/dy | d/dz].
// One CTA per 64-point tile; per 64-function tile J the K chunks of rows i are staged K-major (phi by
// cp.async, P' through registers), two buffers and one barrier per chunk. A warp keeps one
// 16-function column group and one or two groups of points for the whole tile loop, so that a point's
// sums over functions stay in registers until the end. In FP64 the symmetry c_IJ is taken in blocks of
// 8 functions instead of 64 (a warp leaves out the chunks below its column group's diagonal block, and on it a
// quarter: 8 atoms 1.54 ms, with blocks of 16 1.68).
// Three CTAs per SM without GRADN: with two the FP32 form had too few warps for its shared-memory latency (64 atoms
// 2.44 -> 2.17 ms, in spite of some spills; the H kernel above is faster with two, 4.2 against 4.4).
template <typename T, bool GRADN>
__global__ void __launch_bounds__(256, GRADN ? 2 : 3)
    density_simt_kernel(const __grid_constant__ DevSystem s, const DWork *__restrict__ work, int32_t w0,
                        const T *__restrict__ scratch, double *__restrict__ ne_part) {
    using V = typename Vec16<T>::type;
    constexpr int KC = Cfg<T>::KC, MR = Cfg<T>::MR, SR = Cfg<T>::SR, NU = Cfg<T>::NU, VK = 16 / sizeof(T);
    constexpr bool FP = std::is_same<T, double>::value;
    constexpr int NC = GRADN ? 4 : 1;          // sums per point: n, grad n
    constexpr int VR = T_ / VK;                // vectors per row of phi
    constexpr int BR = KC / 8;                 // rows of P' per warp and chunk
    __shared__ __align__(16) T As[2][KC][T_];  // phi[i][q]
    __shared__ __align__(16) T Bs[2][KC][T_];  // c_IJ P[rel_i][rel_j]
    __shared__ double part[4][NC][T_];
    __shared__ double red[8];
    const DWork it = work[w0 + blockIdx.x];
    const int b = it.batch, m = s.sys.bmol[b];
    const int p0 = s.batch_off[b], P = s.batch_off[b + 1] - p0;
    const int Ppad = (P + NAO_PPAD - 1) & ~(NAO_PPAD - 1);
    const int N = s.rel_off[b + 1] - s.rel_off[b];
    const int q0 = it.tp * T_;
    const T *E = scratch + s.scr_off[b];  // row stride Ppad (phi only) or 4 Ppad (GRADN)
    const int64_t ld = GRADN ? 4 * (int64_t)Ppad : (int64_t)Ppad;
    const int32_t *rel = s.rel_idx + s.rel_off[b];
    const int32_t bo = s.sys.boff[m];
    const int64_t nbm = s.sys.nbm[m];
    const double *Pm = s.sys.P[m];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, lx = lane & 3, ly = lane >> 2;
    const int role = (warp + blockIdx.x) & 7, cg = role & 3;  // column group
    // column y of the lane in the group: in FP64 two in each half, so that on the diagonal block the warp leaves out
    // the products of its second eight rows with the first half
    auto col = [&](int y) { return FP && !GRADN ? 2 * lx + (y & 1) + 8 * (y >> 1) : 4 * lx + y; };
    const int nt = (N + T_ - 1) / T_;
    int row[NU];  // first point (of the tile) of each of the warp's point groups, -1: beyond the batch
#pragma unroll
    for (int u = 0; u < NU; u++) {
        row[u] = SR * ((role >> 2) + 2 * u);
        if (q0 + row[u] >= P) row[u] = -1;
    }
    PointSum<T> sum[NU][MR][NC];

    for (int tj = 0; tj < nt; tj++) {
        Block<T> acc[NU];
#pragma unroll
        for (int u = 0; u < NU; u++) acc[u].zero();
        const int kend = GRADN ? N : min(N, (tj + 1) * T_);
        const int nk = (kend + KC - 1) / KC;
        const bool live = row[0] >= 0 && tj * T_ + cg * 16 < N;
        int64_t gj[2];  // the columns of P' that this lane loads: lane and lane + 32
        bool jok[2];
#pragma unroll
        for (int c = 0; c < 2; c++) {
            const int j = tj * T_ + lane + 32 * c;
            jok[c] = j < N;
            gj[c] = jok[c] ? rel[j] - bo : 0;
        }
        double pv[BR][2];
        auto load = [&](int kc, int buf) {
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int x = tid + 256 * h, kk = x / VR, v = (x % VR) * VK, i = kc * KC + kk;
                const bool ok = i < N && q0 + v < Ppad;
                cp16(&As[buf][kk][v], ok ? E + (int64_t)i * ld + q0 + v : E, ok);
            }
#pragma unroll
            for (int r = 0; r < BR; r++) {
                const int i = kc * KC + warp * BR + r;
                const int64_t gi = i < N ? rel[i] - bo : 0;
#pragma unroll
                for (int c = 0; c < 2; c++)
                    if (i < N && jok[c]) pv[r][c] = gi <= gj[c] ? Pm[gi * nbm + gj[c]] : Pm[gj[c] * nbm + gi];
            }
        };
        auto store = [&](int kc, int buf) {
#pragma unroll
            for (int r = 0; r < BR; r++) {
                const int i = kc * KC + warp * BR + r;
#pragma unroll
                for (int c = 0; c < 2; c++) {
                    const int j = tj * T_ + lane + 32 * c;
                    // c_IJ = 2 above the diagonal blocks, 1 on them (those below are not used); FP64
                    // blocks of 8 functions, FP32 blocks of 64
                    const bool two = !GRADN && (FP ? (i >> 3) < (j >> 3) : (i >> 6) < tj);
                    T x = T(0);
                    if (i < N && jok[c]) {
                        if constexpr (FP) x = pv[r][c];
                        else x = to_f32(pv[r][c]);
                        if (two) x += x;
                    }
                    Bs[buf][warp * BR + r][lane + 32 * c] = x;
                }
            }
        };
        load(0, 0);
        store(0, 0);
        for (int kc = 0; kc < nk; kc++) {
            const int buf = kc & 1;
            cp_wait_all();
            __syncthreads();  // this chunk is complete, and every warp has left the other buffer
            if (kc + 1 < nk) load(kc + 1, buf ^ 1);
            if (live && !(FP && !GRADN && kc > tj * 4 + cg)) {
#pragma unroll
                for (int u = 0; u < NU; u++) {
                    if (row[u] < 0) continue;
                    const T *a = &As[buf][0][row[u] + ly * MR], *bb = &Bs[buf][0][cg * 16];
                    auto products = [&](int kk, int y0) {  // with the columns from y0 on
                        T ra[MR], rb[4];
#pragma unroll
                        for (int x = 0; x < MR; x += VK) {
                            const V v = *reinterpret_cast<const V *>(a + kk * T_ + x);
#pragma unroll
                            for (int e = 0; e < VK; e++) ra[x + e] = vget(v, e);
                        }
#pragma unroll
                        for (int y = 0; y < 4; y += VK) {
                            if (y < y0) continue;
                            const V v = *reinterpret_cast<const V *>(bb + kk * T_ + col(y));
#pragma unroll
                            for (int e = 0; e < VK; e++) rb[y + e] = vget(v, e);
                        }
#pragma unroll
                        for (int x = 0; x < MR; x++)
#pragma unroll
                            for (int y = 0; y < 4; y++)
                                if (y >= y0) acc[u].c[x][y] = fma(ra[x], rb[y], acc[u].c[x][y]);
                    };
                    const bool half = FP && !GRADN && kc == tj * 4 + cg;
                    const int k1 = half ? KC / 2 : KC;
#pragma unroll 8
                    for (int kk = 0; kk < k1; kk++) products(kk, 0);
                    if (half)
#pragma unroll
                        for (int kk = KC / 2; kk < KC; kk++) products(kk, 2);
                    acc[u].fold();
                }
            }
            if (kc + 1 < nk) store(kc + 1, buf ^ 1);
        }
        // n_q += sum_{j in J} T_qj phi_jq (and grad n): this lane's points and four columns
#pragma unroll
        for (int u = 0; u < NU; u++) {
            const int q = q0 + row[u] + ly * MR;
            if (row[u] < 0 || q >= Ppad) continue;
#pragma unroll
            for (int y = 0; y < 4; y++) {
                const int j = tj * T_ + cg * 16 + col(y);
                if (j >= N) continue;
#pragma unroll
                for (int d = 0; d < NC; d++)
#pragma unroll
                    for (int x = 0; x < MR; x += VK) {
                        const V f = *reinterpret_cast<const V *>(E + (int64_t)j * ld + d * Ppad + q + x);
#pragma unroll
                        for (int e = 0; e < VK; e++) sum[u][x + e][d].add(acc[u], x + e, y, vget(f, e));
                    }
            }
        }
        __syncthreads();  // the next tile's first chunk goes into buffer 0
    }
    for (int x = tid; x < 4 * NC * T_; x += blockDim.x) (&part[0][0][0])[x] = 0.0;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < NU; u++)
#pragma unroll
        for (int x = 0; x < MR; x++)
#pragma unroll
            for (int d = 0; d < NC; d++) {
                double t = sum[u][x][d].value();
                t += __shfl_xor_sync(0xffffffffu, t, 1);
                t += __shfl_xor_sync(0xffffffffu, t, 2);
                if (lx == 0 && row[u] >= 0) part[cg][d][row[u] + ly * MR + x] = t;
            }
    __syncthreads();
    double wn = 0.0;
    if (tid < T_) {
        const int q = q0 + tid;
        if (q < P) {
            auto total = [&](int d) { return (part[0][d][tid] + part[1][d][tid]) + (part[2][d][tid] + part[3][d][tid]); };
            const double nv = total(0);
            *n_at(s, m, p0 + q) = nv;
            if (GRADN)
#pragma unroll
                for (int d = 0; d < 3; d++) *gn_at(s, m, p0 + q, d) = 2.0 * total(GRADN ? 1 + d : 0);
            wn = s.pw[p0 + q] * nv;
        }
    }
    // fixed-order block sum of w n over the tile
    for (int o = 16; o > 0; o >>= 1) wn += __shfl_xor_sync(0xffffffffu, wn, o);
    if (lane == 0) red[warp] = wn;
    __syncthreads();
    if (tid == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; w++) t += red[w];
        ne_part[w0 + blockIdx.x] = t;
    }
}

// N_e of each system: one CTA per system sums its density work items' partial sums in a fixed
// assignment and tree order (deterministic).
__global__ void __launch_bounds__(1024) reduce_ne_kernel(DevSystem s, const double *__restrict__ part,
                                                        const int32_t *__restrict__ sys_dw0) {
    __shared__ double red[32];
    const int m = blockIdx.x;
    double *out = s.sys.ne[m];
    if (!out) return;
    double t = 0.0;
    for (int64_t i = sys_dw0[m] + threadIdx.x; i < sys_dw0[m + 1]; i += blockDim.x) t += part[i];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x < 32) {
        t = red[threadIdx.x];
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) out[0] = t;
    }
}

// Pointer-table entries passed by value in the kernel's arguments.
constexpr int kPtrBatch = 480;
struct PtrBatch {
    void *p[kPtrBatch];
};
__global__ void set_pointers_kernel(double **__restrict__ dst, PtrBatch src, int32_t n) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = static_cast<double *>(src.p[i]);
}

// n = 0 (and grad n = 0) at the points of each density work item: the tensor-core density
// writes only the points of batches that have basis functions.
__global__ void __launch_bounds__(64) zero_n_kernel(DevSystem s, const DWork *__restrict__ work, int grad) {
    const DWork it = work[blockIdx.x];
    const int p0 = s.batch_off[it.batch], P = s.batch_off[it.batch + 1] - p0;
    const int q = it.tp * NAO_TILE + threadIdx.x;
    if (q >= P) return;
    const int m = s.sys.bmol[it.batch];
    *n_at(s, m, p0 + q) = 0.0;
    if (grad)
        for (int d = 0; d < 3; d++) *gn_at(s, m, p0 + q, d) = 0.0;
}

}  // namespace

template <typename T>
static cudaError_t launch_h_simt_t(const DevSystem &s, const HWork *work, int32_t n_work, const T *scratch, uint32_t terms,
                                   cudaStream_t st) {
    const size_t dyn = 2 * (size_t)s.max_ppad * sizeof(T);  // the weights
    if (dyn + sizeof(HTile<T>) > 48 * 1024) {
        const cudaError_t e =
            cudaFuncSetAttribute(h_simt_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * NAO_MAX_BATCH * (int)sizeof(T));
        if (e != cudaSuccess) return e;
    }
    // A tile pair of a few hundred points keeps an SM's FP64 pipe busy for most of a millisecond: with fewer than
    // 20 FP64 items per SM their points are cut into up to four segments, or the last ones leave most SMs idle.
    // Segments of points, not of K: a point's four components may cancel in phi_i phi_j d and the gradients'
    // product, and a sum over points of h's terms has no larger partial sums than the magnitudes it is measured
    // against. 8-atom cluster (490 batches): H 6.60 -> 5.33 ms.
    const int kseg = sizeof(T) == 4 || n_work >= 20 * s.n_sm ? 1 : (n_work >= 10 * s.n_sm ? 2 : 4);
    h_simt_kernel<T><<<dim3(n_work, kseg), 256, dyn, st>>>(s, work, scratch, terms);
    return cudaGetLastError();
}

cudaError_t launch_h_simt(const DevSystem &s, nao_precision prec, const HWork *work, int32_t n_work,
                          const double *scratch, uint32_t terms, cudaStream_t st) {
    if (n_work <= 0) return cudaSuccess;
    if (prec == NAO_FP32) return launch_h_simt_t(s, work, n_work, reinterpret_cast<const float *>(scratch), terms, st);
    return launch_h_simt_t(s, work, n_work, scratch, terms, st);
}

cudaError_t launch_zero_h(const DevSystem &s, const int4 *tasks, int32_t n_tasks, cudaStream_t st) {
    if (n_tasks <= 0) return cudaSuccess;
    zero_h_kernel<<<n_tasks, 256, 0, st>>>(s, tasks);
    return cudaGetLastError();
}

cudaError_t launch_mirror(const DevSystem &s, const int4 *tasks, int32_t n_tasks, cudaStream_t st) {
    if (n_tasks <= 0) return cudaSuccess;
    mirror_kernel<<<n_tasks, dim3(32, 8), 0, st>>>(s, tasks);
    return cudaGetLastError();
}

cudaError_t launch_density_simt(const DevSystem &s, nao_precision prec, const DWork *work, int32_t w0, int32_t n_work,
                                const double *scratch, double *ne_part, bool grad, cudaStream_t st) {
    if (n_work <= 0) return cudaSuccess;
    const float *sf = reinterpret_cast<const float *>(scratch);
    if (prec == NAO_FP32 && grad) density_simt_kernel<float, true><<<n_work, 256, 0, st>>>(s, work, w0, sf, ne_part);
    else if (prec == NAO_FP32) density_simt_kernel<float, false><<<n_work, 256, 0, st>>>(s, work, w0, sf, ne_part);
    else if (grad) density_simt_kernel<double, true><<<n_work, 256, 0, st>>>(s, work, w0, scratch, ne_part);
    else density_simt_kernel<double, false><<<n_work, 256, 0, st>>>(s, work, w0, scratch, ne_part);
    return cudaGetLastError();
}

cudaError_t launch_reduce_ne(const DevSystem &s, const double *part, const int32_t *sys_dw0, int32_t n_sys,
                             cudaStream_t st) {
    if (n_sys <= 0) return cudaSuccess;
    reduce_ne_kernel<<<n_sys, 1024, 0, st>>>(s, part, sys_dw0);
    return cudaGetLastError();
}

cudaError_t launch_set_pointers(double **dst, void *const *src, int32_t n, cudaStream_t st) {
    for (int32_t i0 = 0; i0 < n; i0 += kPtrBatch) {
        const int32_t c = n - i0 < kPtrBatch ? n - i0 : kPtrBatch;
        PtrBatch b;
        for (int32_t i = 0; i < c; i++) b.p[i] = src[i0 + i];
        set_pointers_kernel<<<1, 128, 0, st>>>(dst + i0, b, c);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_zero_n(const DevSystem &s, const DWork *work, int32_t n_work, bool grad, cudaStream_t st) {
    if (n_work <= 0) return cudaSuccess;
    zero_n_kernel<<<n_work, 64, 0, st>>>(s, work, grad ? 1 : 0);
    return cudaGetLastError();
}
