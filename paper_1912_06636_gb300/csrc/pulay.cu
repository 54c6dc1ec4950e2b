// Local Pulay force terms on the FP64 and FP32 paths (Sec. 2, the local parts of the Pulay forces,
//     F_at = -2 sum_ij int [grad_at phi_i] n_ij h_KS phi_j + 2 sum_ij int [grad_at phi_i] q_ij phi_j,
// q the energy-weighted density matrix), assembled, as the paper describes for forces, from
// matrix elements with basis-function indices first (Sec. "Density and Density Derivatives"):
//     M^c_ij = sum_p w_p d_c phi_i (h phi_j),  h phi_j = -1/2 lap phi_j + v phi_j,
//     S^c_ij = sum_p w_p d_c phi_i phi_j,                       c = x, y, z,
// then, since grad_at phi_i = -grad phi_i for a function on atom at,
//     F_at,c = 2 sum_{i on at} sum_j (n_ij M^c_ij - q_ij S^c_ij).
// The batches' basis functions come from the density Hessian's evaluation (10 rows per function:
// phi, grad phi and, in place of the six second derivatives, the Laplacian).
// Work items are the 64 x 64 tile pairs (I, J) of a batch (all pairs: the matrices are not symmetric);
// FP64 atomics add each tile into the global matrices.
// FP64: bound by the FP64 pipe (two lanes per clock and SM), 6 N^2 P products per batch. One CTA takes half
// an item, 64 x 32, and each warp up to four 8 x 8 subtiles of it with all six products; subtiles beyond the
// batch's functions are left out. The rows d_c phi_i come by cp.async as they lie, the weights go into the
// columns: w phi_j and w h phi_j. 9 atoms, 19,440 points: 11.3 -> 9.5 ms, with
// the points of an item in up to four CTAs 8.3, with 8 x 8 subtiles instead of 16 x 16 7.96 (floor 7.2).
// FP32: per 8-point chunk w d_c phi_i (three components) and h phi_j or phi_j, each chunk's sums added
// into compensated (hi, lo) pairs, in two passes of three products.
#include "nao_internal.h"

namespace {

constexpr int HR = 10;  // rows per basis function in the Hessian evaluation
constexpr int TT = 64;  // tile edge (functions)
constexpr int KC = 8;   // points per K chunk (FP32)

constexpr int KP = 16;      // points per K chunk (FP64): 128 bytes of a row
constexpr int LDP = 18;     // and 16 bytes more: the eight rows a warp reads at once in different banks

__device__ __forceinline__ void cp16(void *dst, const void *src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(ok ? 16 : 0)
                 : "memory");
}

__global__ void __launch_bounds__(256, 2)
    pulay_fp64_kernel(const __grid_constant__ DevSystem s, const HWork *__restrict__ work, int32_t w0,
                      const double *__restrict__ scratch, const int64_t *__restrict__ hoff, double *__restrict__ M,
                      double *__restrict__ Sm, int64_t nb) {
    __shared__ __align__(16) double As[3][TT][LDP];      // d_c phi_i
    __shared__ __align__(16) double Bs[2][TT / 2][LDP];  // w h phi_j, w phi_j
    extern __shared__ __align__(16) double wt[];         // [2][Ppad]: w, w v
    const HWork it = work[w0 + blockIdx.x];
    const int b = it.batch, m = s.sys.bmol[b];
    const int p0 = s.batch_off[b], P = s.batch_off[b + 1] - p0;
    const int Ppad = (P + NAO_PPAD - 1) & ~(NAO_PPAD - 1);
    const int N = s.rel_off[b + 1] - s.rel_off[b];
    const int i0 = it.ti * TT, j0 = it.tj * TT + (int)blockIdx.y * (TT / 2);
    if (j0 >= N) return;
    const double *E = scratch + hoff[b];
    const int64_t ld = (int64_t)HR * Ppad;
    const int tid = threadIdx.x, lane = tid & 31, lx = lane & 3, ly = lane >> 2;
    for (int q = tid; q < Ppad; q += 256) {
        const double w = q < P ? s.pw[p0 + q] : 0.0;
        wt[q] = w;
        wt[Ppad + q] = q < P ? w * v_at(s, m, p0 + q) : 0.0;
    }
    // this warp's 8 x 8 subtiles: every eighth of those within the batch's functions (the first nr x nc of 8 x 4), the
    // first of which turns with the CTA; subtile k at row k / nc, column k % nc, -1: none
    const int nr = min(8, (N - i0 + 7) / 8), nc = min(4, (N - j0 + 7) / 8);
    int sub[4];
#pragma unroll
    for (int t = 0; t < 4; t++) {
        const int k = (((tid >> 5) + (int)blockIdx.x) & 7) + 8 * t;
        sub[t] = k < nr * nc ? 8 * (k / nc) | 8 * (k % nc) << 8 : -1;  // first row | first column << 8
    }
    double acc[4][3][2][2];
#pragma unroll
    for (int x = 0; x < 48; x++) (&acc[0][0][0][0])[x] = 0.0;
    const int lv = tid & 7, lr = tid >> 3;  // loader: vector lv (two points), rows lr and lr + 32
    // this CTA's points (see the launcher)
    const int chunks = Ppad / KP, per = (chunks + (int)gridDim.z - 1) / (int)gridDim.z;
    const int qa = (int)blockIdx.z * per * KP, qb = min(Ppad, qa + per * KP);
    if (qa >= qb) return;
    for (int q0 = qa; q0 < qb; q0 += KP) {
        __syncthreads();  // the weights are written; every warp has left the last chunk
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int i = i0 + lr + 32 * h;
            const double *row = E + (int64_t)(i < N ? i : 0) * ld + q0 + 2 * lv;
#pragma unroll
            for (int c = 0; c < 3; c++) cp16(&As[c][lr + 32 * h][2 * lv], row + (int64_t)(1 + c) * Ppad, i < N);
        }
        double2 wh = make_double2(0.0, 0.0), wf = wh;
        if (j0 + lr < N) {
            const double *row = E + (int64_t)(j0 + lr) * ld + q0 + 2 * lv;
            const double2 f = *reinterpret_cast<const double2 *>(row);
            const double2 lap = *reinterpret_cast<const double2 *>(row + 4 * (int64_t)Ppad);
            const double2 w = *reinterpret_cast<const double2 *>(wt + q0 + 2 * lv);
            const double2 wv = *reinterpret_cast<const double2 *>(wt + Ppad + q0 + 2 * lv);
            wf = make_double2(w.x * f.x, w.y * f.y);
            wh = make_double2(fma(wv.x, f.x, -0.5 * w.x * lap.x), fma(wv.y, f.y, -0.5 * w.y * lap.y));
        }
        *reinterpret_cast<double2 *>(&Bs[0][lr][2 * lv]) = wh;
        *reinterpret_cast<double2 *>(&Bs[1][lr][2 * lv]) = wf;
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
#pragma unroll
        for (int t = 0; t < 4; t++) {
            if (sub[t] < 0) continue;
            const double *a = &As[0][(sub[t] & 255) + ly][0], *bb = &Bs[0][(sub[t] >> 8) + lx][0];
#pragma unroll 1
            for (int kv = 0; kv < KP; kv += 2) {
                double2 ra[3], rb[2][2];
#pragma unroll
                for (int c = 0; c < 3; c++) ra[c] = *reinterpret_cast<const double2 *>(a + c * TT * LDP + kv);
#pragma unroll
                for (int u = 0; u < 2; u++)
#pragma unroll
                    for (int y = 0; y < 2; y++) rb[u][y] = *reinterpret_cast<const double2 *>(bb + (u * (TT / 2) + 4 * y) * LDP + kv);
#pragma unroll
                for (int c = 0; c < 3; c++)
#pragma unroll
                    for (int u = 0; u < 2; u++)
#pragma unroll
                        for (int y = 0; y < 2; y++)
                            acc[t][c][u][y] = fma(ra[c].y, rb[u][y].y, fma(ra[c].x, rb[u][y].x, acc[t][c][u][y]));
            }
        }
    }
    const int32_t *rel = s.rel_idx + s.rel_off[b];
    const int64_t nn = nb * nb;
#pragma unroll
    for (int t = 0; t < 4; t++) {
        const int i = i0 + (sub[t] & 255) + ly;
        if (sub[t] < 0 || i >= N) continue;
        const int64_t gi = rel[i];
#pragma unroll
        for (int y = 0; y < 2; y++) {
            const int j = j0 + (sub[t] >> 8) + lx + 4 * y;
            if (j >= N) continue;
            const int64_t e = gi * nb + rel[j];
#pragma unroll
            for (int c = 0; c < 3; c++) {
                atomicAdd(M + c * nn + e, acc[t][c][0][y]);
                atomicAdd(Sm + c * nn + e, acc[t][c][1][y]);
            }
        }
    }
}

// (hi, lo) += x with Knuth's TwoSum (exact transformation of hi + x): the FP32 path's running
// sums over the chunks, so that only each 8-point chunk is summed in plain FP32.
__device__ __forceinline__ void two_sum_acc(float &hi, float &lo, float x) {
    const float t = __fadd_rn(hi, x);
    const float bb = __fsub_rn(t, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, bb)), __fsub_rn(x, bb)));
    hi = t;
}

// One of the two products: u0 = 0 (h phi_j, into M) or 1 (phi_j, into S), which leaves registers for the
// compensated sums.
__global__ void __launch_bounds__(256) pulay_fp32_kernel(const __grid_constant__ DevSystem s, const HWork *__restrict__ work,
                                                        int32_t w0, const float *__restrict__ scratch,
                                                        const int64_t *__restrict__ hoff, double *__restrict__ out, int64_t nb,
                                                        int u0) {
    __shared__ __align__(16) float As[3][KC][TT];  // w_q d_c phi_i(q)
    __shared__ __align__(16) float Bs[KC][TT];     // h phi_j(q) or phi_j(q)
    const HWork it = work[w0 + blockIdx.x];
    const int b = it.batch, m = s.sys.bmol[b];
    const int p0 = s.batch_off[b], P = s.batch_off[b + 1] - p0;
    const int Ppad = (P + NAO_PPAD - 1) & ~(NAO_PPAD - 1);
    const int N = s.rel_off[b + 1] - s.rel_off[b];
    const float *E = scratch + hoff[b];
    const int64_t ld = (int64_t)HR * Ppad;
    const int32_t *rel = s.rel_idx + s.rel_off[b];
    const int i0 = it.ti * TT, j0 = it.tj * TT;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    float acc[3][4][4], hi[3][4][4], lo[3][4][4];
#pragma unroll
    for (int c = 0; c < 3; c++)
#pragma unroll
        for (int a = 0; a < 4; a++)
#pragma unroll
            for (int d = 0; d < 4; d++) acc[c][a][d] = hi[c][a][d] = lo[c][a][d] = 0.0f;
    for (int q0 = 0; q0 < P; q0 += KC) {
        __syncthreads();
        for (int u = tid; u < 3 * KC * TT; u += blockDim.x) {
            const int c = u / (KC * TT), kk = (u / TT) % KC, ii = u % TT;
            const int i = i0 + ii, q = q0 + kk;
            As[c][kk][ii] =
                (i < N && q < P) ? float(s.pw[p0 + q] * (double)E[(int64_t)i * ld + (int64_t)(1 + c) * Ppad + q]) : 0.0f;
        }
        for (int u = tid; u < KC * TT; u += blockDim.x) {
            const int kk = u / TT, jj = u % TT;
            const int j = j0 + jj, q = q0 + kk;
            float f = 0.0f;
            if (j < N && q < P) {
                const float *row = E + (int64_t)j * ld + q;
                f = row[0];
                if (u0 == 0) {
                    const double lap = (double)row[4 * (int64_t)Ppad];  // the evaluation's Laplacian row
                    f = float(-0.5 * lap + v_at(s, m, p0 + q) * (double)f);
                }
            }
            Bs[kk][jj] = f;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < KC; kk++) {
            float rb[4];
#pragma unroll
            for (int d = 0; d < 4; d++) rb[d] = Bs[kk][tx * 4 + d];
#pragma unroll
            for (int c = 0; c < 3; c++)
#pragma unroll
                for (int a = 0; a < 4; a++) {
                    const float ra = As[c][kk][ty * 4 + a];
#pragma unroll
                    for (int d = 0; d < 4; d++) acc[c][a][d] = fmaf(ra, rb[d], acc[c][a][d]);
                }
        }
#pragma unroll
        for (int c = 0; c < 3; c++)
#pragma unroll
            for (int a = 0; a < 4; a++)
#pragma unroll
                for (int d = 0; d < 4; d++) {
                    two_sum_acc(hi[c][a][d], lo[c][a][d], acc[c][a][d]);
                    acc[c][a][d] = 0.0f;
                }
    }
    const int64_t nn = nb * nb;
#pragma unroll
    for (int a = 0; a < 4; a++) {
        const int i = i0 + ty * 4 + a;
        if (i >= N) continue;
        const int64_t gi = rel[i];
#pragma unroll
        for (int d = 0; d < 4; d++) {
            const int j = j0 + tx * 4 + d;
            if (j >= N) continue;
            const int64_t e = gi * nb + rel[j];
#pragma unroll
            for (int c = 0; c < 3; c++) atomicAdd(out + c * nn + e, (double)hi[c][a][d] + (double)lo[c][a][d]);
        }
    }
}

// One CTA per atom: F[3 a + c] = 2 sum_{i on a} sum_j (n_ij M^c_ij - q_ij S^c_ij).
__global__ void __launch_bounds__(256) pulay_force_kernel(const double *__restrict__ nmat, const double *__restrict__ qmat,
                                                         const double *__restrict__ M, const double *__restrict__ Sm,
                                                         const int64_t *__restrict__ atom_basis, int64_t nb,
                                                         double *__restrict__ F) {
    __shared__ double red[3][8];
    const int a = blockIdx.x;
    const int64_t i0 = atom_basis[a], i1 = atom_basis[a + 1], nn = nb * nb;
    double part[3] = {0.0, 0.0, 0.0};
    for (int64_t e = i0 * nb + threadIdx.x; e < i1 * nb; e += blockDim.x) {
        const double n = nmat[e], q = qmat[e];
#pragma unroll
        for (int c = 0; c < 3; c++) part[c] = fma(n, M[c * nn + e], fma(-q, Sm[c * nn + e], part[c]));
    }
#pragma unroll
    for (int c = 0; c < 3; c++) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) part[c] += __shfl_xor_sync(0xffffffffu, part[c], o);
        if ((threadIdx.x & 31) == 0) red[c][threadIdx.x >> 5] = part[c];
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double t = 0.0;
        for (int w = 0; w < 8; w++) t += red[threadIdx.x][w];
        F[3 * a + threadIdx.x] = 2.0 * t;
    }
}

}  // namespace

cudaError_t launch_pulay(const DevSystem &s, const HWork *work, int32_t w0, int32_t n_work, const void *scratch, bool fp32,
                         const int64_t *hoff, double *M, double *S, int64_t nb, cudaStream_t st) {
    if (n_work <= 0) return cudaSuccess;
    if (fp32) {
        for (int u0 = 0; u0 < 2; u0++) {
            pulay_fp32_kernel<<<n_work, 256, 0, st>>>(s, work, w0, static_cast<const float *>(scratch), hoff, u0 == 0 ? M : S,
                                                      nb, u0);
            const cudaError_t e = cudaGetLastError();
            if (e != cudaSuccess) return e;
        }
    } else {
        const size_t dyn = 2 * (size_t)s.max_ppad * sizeof(double);  // the weights
        if (dyn > 11 * 1024) {  // beyond 48 KB with the 36.9 KB of operands
            const cudaError_t e = cudaFuncSetAttribute(pulay_fp64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       2 * NAO_MAX_BATCH * (int)sizeof(double));
            if (e != cudaSuccess) return e;
        }
        // few items: their points are cut into up to four segments, whose partial sums simply add (an item
        // keeps an SM's FP64 pipe busy for most of a millisecond; at 900 items two segments took 8.44 ms, four 8.30)
        const int seg = n_work >= 20 * s.n_sm ? 1 : (n_work >= 10 * s.n_sm ? 2 : 4);
        pulay_fp64_kernel<<<dim3(n_work, 2, seg), 256, dyn, st>>>(s, work, w0, static_cast<const double *>(scratch), hoff, M, S, nb);
    }
    return cudaGetLastError();
}

cudaError_t launch_pulay_forces(const double *nmat, const double *qmat, const double *M, const double *S,
                                const int64_t *atom_basis, int32_t n_atoms, int64_t nb, double *F, cudaStream_t st) {
    if (n_atoms <= 0) return cudaSuccess;
    pulay_force_kernel<<<n_atoms, 256, 0, st>>>(nmat, qmat, M, S, atom_basis, nb, F);
    return cudaGetLastError();
}
