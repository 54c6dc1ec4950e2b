// Periodic systems (Eq. HamPeriodic, Eq. RealSpaceHamPeriodic, Eq. Bloch-basis).
//
// The real-space matrix h^uc is integrated over the unit cell's points with the same code as a
// finite system: the system's atoms are the periodic images R_A + T (T = n1 a1 + n2 a2 + n3 a3)
// whose functions can be non-zero in the cell, so its basis is the N_rs real-space functions of
// the paper. nao_periodic_images lists those images (host), nao_periodic_basis_map relates every
// image function to its unit-cell function and image, and nao_bloch_sum forms on the GPU
//     h_ij(k) = sum_{i' -> i, j' -> j} h^uc_{i'j'} e^{i k.(T_j' - T_i')},
// which is Eq. Bloch-basis, chi_ik = sum_T e^{i k.T} phi_i(r - T), inserted into Eq. HamPeriodic
// (conj(chi_i) on the left). The overlap s(k) follows from h^uc = S^uc (NAO_TERM_POTENTIAL, v = 1).
#include <cmath>
#include <string>
#include <vector>

#include "nao_internal.h"

namespace {

struct Lattice {
    double a[9];  // rows a1, a2, a3
};

constexpr int kBlochThreads = 256;
// Dynamic shared memory that the row form of the sum may take: 227 KB less its static part, of which the parts' sums
// (cells of at most 128 functions) are 4 KB.
constexpr size_t bloch_smem_limit(bool parts) { return (parts ? 222 : 226) * 1024; }

// e^{i k.T} of image (c0, c1, c2).
__device__ __forceinline__ double2 image_phase(const Lattice &L, const int32_t *c, const double *k) {
    double ph = 0.0;
#pragma unroll
    for (int d = 0; d < 3; d++)
        ph = fma(k[d], (double)c[0] * L.a[d] + (double)c[1] * L.a[3 + d] + (double)c[2] * L.a[6 + d], ph);
    double sn, cs;
    sincos(ph, &sn, &cs);
    return make_double2(cs, sn);
}

// (h, l) += a b as an unevaluated sum: the product's and the addition's rounding errors go into l.
__device__ __forceinline__ void add_product(double2 &s, double a, double b) {
    const double p = __dmul_rn(a, b), e = fma(a, b, -p), t = __dadd_rn(s.x, p), bb = __dsub_rn(t, s.x);
    s.y += (__dsub_rn(s.x, __dsub_rn(t, bb)) + __dsub_rn(p, bb)) + e;
    s.x = t;
}
// k.a_c of one lattice vector.
__device__ __forceinline__ double2 k_dot(const Lattice &L, int c, const double *k) {
    double2 s = make_double2(0.0, 0.0);
#pragma unroll
    for (int d = 0; d < 3; d++) add_product(s, k[d], L.a[3 * c + d]);
    return s;
}
// e^{i k.T} of image (c0, c1, c2) with the argument in twice the precision (ka: k.a_c): the row form multiplies the
// phases of two images, whose arguments may be far larger than their difference, the only one the general form takes
// (cells 1000 lattice vectors from the origin: h(k) to 4e-13 with the argument in FP64 as well, 5e-16 in both forms).
__device__ __forceinline__ double2 image_phase2(const double2 *ka, const int32_t *c) {
    double2 s = make_double2(0.0, 0.0);
#pragma unroll
    for (int x = 0; x < 3; x++) {
        add_product(s, (double)c[x], ka[x].x);
        s.y = fma((double)c[x], ka[x].y, s.y);
    }
    const double ph = __dadd_rn(s.x, s.y), lo = __dsub_rn(s.y, __dsub_rn(ph, s.x));
    double sn, cs;
    sincos(ph, &sn, &cs);
    return make_double2(fma(-sn, lo, cs), fma(cs, lo, sn));
}

// The sum by rows of h(k): one CTA takes `rows` unit-cell functions i and KQ k points (blockIdx.y).
// It lists the real-space functions of every unit-cell function (a stable counting sort of fn_map in shared
// memory) and the phases of every image, once. Then for each real-space function i' of i
//     G_j = sum_{j' -> j} h^uc_{i'j'} e^{i k.T_j'}      (thread j; two FMAs per element and k point)
// is multiplied by e^{-i k.T_i'} and added to h_ij(k) in registers: no atomics, every h(k) element is
// written once, and its terms are added in the same order on every call. Bound by the FP64 pipe (two lanes per clock
// and SM); elements that are zero for the whole warp are left out. Periodic silicon, N_rs = 2350, 64 k points:
// 0.79 ms, against 6.2 ms with one sincos and two atomics per element and k point (bloch_kernel).
// With at most 128 unit-cell functions a thread takes every parts-th i' only, parts = 256 / nb, and the parts' sums
// are added in order: a small cell has long lists (N_rs / nb entries each) and few functions. One thread per j, as
// with more functions, walked all (N_rs / nb)^2 elements by itself:
//     nb = 4, N_rs = 1600, 1 / 8 k points     44.3 / 113 -> 1.01 / 3.16 ms (bloch_kernel 2.70 / 19.9)
//     nb = 13, N_rs = 1300, 1 / 8 k points    3.00 / 7.38 -> 0.33 / 0.81 ms (0.48 / 2.63)
//     nb = 25, N_rs = 2500, 1 / 8 k points    3.07 / 7.40 -> 0.47 / 1.31 ms (0.63 / 4.07)
//     nb = 50, N_rs = 2500, 1 / 8 k points    0.90 / 1.99 -> 0.33 / 0.76 ms (0.63 / 4.06)
// (whole calls through the Python binding, about 0.15 ms of them on the host).
template <int KQ, bool PARTS>
__global__ void __launch_bounds__(kBlochThreads) bloch_rows_kernel(const double *__restrict__ huc, int32_t n_rs,
                                                                  const int32_t *__restrict__ fn_map,
                                                                  const int32_t *__restrict__ fn_image,
                                                                  const int32_t *__restrict__ img_cell, int32_t n_images,
                                                                  const __grid_constant__ Lattice L,
                                                                  const double *__restrict__ kpts, int32_t n_k, int32_t nb,
                                                                  int32_t rows, double *__restrict__ hk) {
    extern __shared__ __align__(16) unsigned char dyn[];
    double2 *ph = reinterpret_cast<double2 *>(dyn);          // [n_images][KQ]
    int *off = reinterpret_cast<int *>(ph + (size_t)n_images * KQ);  // [nb + 1] first entry of each function
    int *cur = off + nb + 1;                                 // [nb] fill position
    int2 *ent = reinterpret_cast<int2 *>(cur + nb + ((2 * nb + 1) & 1));  // [n_rs] (real-space function, image)
    __shared__ int wsum[kBlochThreads / 32];
    __shared__ double2 ka[KQ][3];             // k.a_c
    __shared__ double2 red[PARTS ? kBlochThreads : 1];  // the parts' sums
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int k0 = blockIdx.y * KQ;
    auto valid = [&](int r, int &i, int &t) {
        i = fn_map[r];
        t = fn_image[r];
        return i >= 0 && i < nb && t >= 0 && t < n_images;
    };
    if (tid < 3 * KQ) {
        const int q = tid / 3, c = tid % 3;
        ka[q][c] = k0 + q < n_k ? k_dot(L, c, kpts + 3 * (int64_t)(k0 + q)) : make_double2(0.0, 0.0);
    }
    for (int i = tid; i < nb; i += kBlochThreads) cur[i] = 0;
    __syncthreads();
    for (int x = tid; x < n_images * KQ; x += kBlochThreads)
        ph[x] = image_phase2(ka[x % KQ], img_cell + 3 * (int64_t)(x / KQ));
    int i, t;
    for (int r = tid; r < n_rs; r += kBlochThreads)
        if (valid(r, i, t)) atomicAdd(cur + i, 1);
    __syncthreads();
    // exclusive prefix sum of the counts: thread t owns `per` consecutive functions
    const int per = (nb + kBlochThreads - 1) / kBlochThreads, lo = min(nb, tid * per), hi = min(nb, lo + per);
    int cnt = 0;
    for (int x = lo; x < hi; x++) cnt += cur[x];
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int at = incl - cnt;
    for (int w = 0; w < warp; w++) at += wsum[w];
    for (int x = lo; x < hi; x++) {
        const int c = cur[x];
        off[x] = cur[x] = at;
        at += c;
    }
    if (tid == kBlochThreads - 1) off[nb] = at;
    __syncthreads();
    // the entries of every function by increasing r
    if constexpr (!PARTS) {
        for (int r = tid; r < n_rs; r += kBlochThreads)
            if (valid(r, i, t)) ent[atomicAdd(cur + i, 1)] = make_int2(r, t);
        __syncthreads();
        for (int x = tid; x < nb; x += kBlochThreads)  // a fixed order whatever the atomics' (with so many functions the lists are short)
            for (int p = off[x] + 1; p < off[x + 1]; p++) {
                const int2 e = ent[p];
                int q = p;
                for (; q > off[x] && ent[q - 1].x > e.x; q--) ent[q] = ent[q - 1];
                ent[q] = e;
            }
        __syncthreads();
    } else {
        // 256 at a time, the warps one after the other, a warp's lanes by rank: lists may hold thousands
        for (int r0 = 0; r0 < n_rs; r0 += kBlochThreads) {
            const int r = r0 + tid;
            if (r >= n_rs || !valid(r, i, t)) i = -1;
            const unsigned same = __match_any_sync(0xffffffffu, i);
            const int rank = __popc(same & ((1u << lane) - 1u));
#pragma unroll 1
            for (int w = 0; w < kBlochThreads / 32 && r0 + 32 * w < n_rs; w++) {
                if (w == warp && i >= 0) {
                    const int p = cur[i];
                    ent[p + rank] = make_int2(r, t);
                    __syncwarp(same);
                    if (rank == 0) cur[i] = p + __popc(same);
                }
                __syncthreads();
            }
        }
    }

    const int parts = PARTS ? kBlochThreads / nb : 1;
    const int part = PARTS ? tid / nb : 0, jt = PARTS ? tid - part * nb : tid;
    const int r1 = min(nb, (int)(blockIdx.x + 1) * rows);
    for (int row = blockIdx.x * rows; row < r1; row++)
        for (int j0 = 0; j0 < nb; j0 += kBlochThreads) {  // once where PARTS
            const int j = j0 + jt;
            const int s0 = j < nb ? off[j] : 0, s1 = j < nb ? off[j + 1] : 0;
            double2 acc[KQ];
#pragma unroll
            for (int q = 0; q < KQ; q++) acc[q] = make_double2(0.0, 0.0);
            for (int a = part < parts ? off[row] + part : off[row + 1]; a < off[row + 1]; a += parts) {
                const double *h = huc + (int64_t)ent[a].x * n_rs;
                double2 G[KQ];
#pragma unroll
                for (int q = 0; q < KQ; q++) G[q] = make_double2(0.0, 0.0);
                bool any = false;
                for (int x = s0; x < s1; x++) {
                    const int2 e = ent[x];
                    const double hv = h[e.x];
                    if (hv == 0.0) continue;
                    any = true;
                    const double2 *p = ph + e.y * KQ;
#pragma unroll
                    for (int q = 0; q < KQ; q++) {
                        const double2 w = p[q];
                        G[q].x = fma(hv, w.x, G[q].x);
                        G[q].y = fma(hv, w.y, G[q].y);
                    }
                }
                if (!any) continue;
                const double2 *p = ph + ent[a].y * KQ;
#pragma unroll
                for (int q = 0; q < KQ; q++) {  // += G conj(phase)
                    const double2 w = p[q];
                    acc[q].x = fma(w.x, G[q].x, fma(w.y, G[q].y, acc[q].x));
                    acc[q].y = fma(w.x, G[q].y, fma(-w.y, G[q].x, acc[q].y));
                }
            }
#pragma unroll
            for (int q = 0; q < KQ; q++) {
                if (PARTS) {
                    __syncthreads();
                    red[tid] = acc[q];
                    __syncthreads();
                    if (part == 0)
                        for (int x = 1; x < parts; x++) {
                            const double2 y = red[x * nb + jt];
                            acc[q].x += y.x;
                            acc[q].y += y.y;
                        }
                }
                if (part == 0 && j < nb && k0 + q < n_k) {  // as two doubles: hk need not lie on a 16-byte boundary
                    double *out = hk + 2 * (((int64_t)(k0 + q) * nb + row) * nb + j);
                    out[0] = acc[q].x;
                    out[1] = acc[q].y;
                }
            }
        }
}

// Counts the non-zero elements of h^uc whose row or column has an out-of-range map entry.
__global__ void __launch_bounds__(256) bloch_check_kernel(const double *__restrict__ huc, int64_t n_rs,
                                                         const int32_t *__restrict__ fn_map,
                                                         const int32_t *__restrict__ fn_image, int32_t n_images, int64_t nb,
                                                         int32_t *__restrict__ err) {
    const int64_t r = blockIdx.x;
    auto bad = [&](int64_t x) { return fn_map[x] < 0 || fn_map[x] >= nb || fn_image[x] < 0 || fn_image[x] >= n_images; };
    const bool row = bad(r);
    int c = 0;
    for (int64_t x = threadIdx.x; x < n_rs; x += blockDim.x)
        if ((row || bad(x)) && huc[r * n_rs + x] != 0.0) c++;
    if (c) atomicAdd(err, c);
}

// The general form: one thread per element (i', j') of h^uc for one k point (blockIdx.y); both the
// real and the imaginary part of e^{i k.(T_j' - T_i')} h^uc_{i'j'} are added into h(k)[fn(i')][fn(j')].
// It runs where the tables of bloch_rows_kernel do not fit in shared memory.
// The maps come from the caller: an element whose fn_map entry lies outside [0, nb) or whose
// fn_image entry lies outside [0, n_images) is skipped (and counted by bloch_check_kernel), so that no
// map value can move a read or an atomic outside its array.
__global__ void __launch_bounds__(256) bloch_kernel(const double *__restrict__ huc, int64_t n_rs,
                                                   const int32_t *__restrict__ fn_map,
                                                   const int32_t *__restrict__ fn_image,
                                                   const int32_t *__restrict__ img_cell, int32_t n_images, Lattice L,
                                                   const double *__restrict__ kpts, int64_t nb, double *__restrict__ hk) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n_rs * n_rs) return;
    const double hv = huc[e];
    if (hv == 0.0) return;
    const int64_t i = e / n_rs, j = e - i * n_rs;
    const int32_t mi = fn_map[i], mj = fn_map[j], ti = fn_image[i], tj = fn_image[j];
    if (mi < 0 || mi >= nb || mj < 0 || mj >= nb || ti < 0 || ti >= n_images || tj < 0 || tj >= n_images) return;
    const int32_t *ci = img_cell + 3 * (int64_t)ti, *cj = img_cell + 3 * (int64_t)tj;
    const int32_t d[3] = {cj[0] - ci[0], cj[1] - ci[1], cj[2] - ci[2]};
    const double2 w = image_phase(L, d, kpts + 3 * (int64_t)blockIdx.y);
    double *out = hk + 2 * (((int64_t)blockIdx.y * nb + mi) * nb + mj);
    atomicAdd(out, w.x * hv);
    atomicAdd(out + 1, w.y * hv);
}

// Shared memory of bloch_rows_kernel<KQ>, in bytes.
size_t bloch_rows_smem(int64_t n_rs, int64_t n_images, int64_t nb, int KQ) {
    return (size_t)n_images * KQ * 16 + 4 * (size_t)(2 * nb + 2) + 8 * (size_t)n_rs;
}

template <int KQ, bool PARTS>
cudaError_t launch_bloch_rows(const double *huc, int32_t n_rs, const int32_t *fn_map, const int32_t *fn_image,
                              const int32_t *img_cell, int32_t n_images, const Lattice &L, const double *k, int32_t n_k,
                              int32_t nb, double *hk, cudaStream_t st) {
    const size_t smem = bloch_rows_smem(n_rs, n_images, nb, KQ);
    cudaError_t e = cudaSuccess;
    if (smem > 40 * 1024) {
        e = cudaFuncSetAttribute(bloch_rows_kernel<KQ, PARTS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)bloch_smem_limit(PARTS));
        if (e != cudaSuccess) return e;
    }
    // about four CTAs per SM: more would repeat the lists and phases, fewer leave a tail
    int dev = 0, n_sm = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int nq = (n_k + KQ - 1) / KQ, want = (4 * n_sm + nq - 1) / nq, rows = (nb + want - 1) / want;
    bloch_rows_kernel<KQ, PARTS><<<dim3((nb + rows - 1) / rows, nq), kBlochThreads, smem, st>>>(
        huc, n_rs, fn_map, fn_image, img_cell, n_images, L, k, n_k, nb, rows, hk);
    return cudaGetLastError();
}

bool inv3(const double *A, double *R) {
    const double det = A[0] * (A[4] * A[8] - A[5] * A[7]) - A[1] * (A[3] * A[8] - A[5] * A[6]) +
                       A[2] * (A[3] * A[7] - A[4] * A[6]);
    if (!(std::fabs(det) > 0.0) || !std::isfinite(det)) return false;
    R[0] = (A[4] * A[8] - A[5] * A[7]) / det;
    R[1] = (A[2] * A[7] - A[1] * A[8]) / det;
    R[2] = (A[1] * A[5] - A[2] * A[4]) / det;
    R[3] = (A[5] * A[6] - A[3] * A[8]) / det;
    R[4] = (A[0] * A[8] - A[2] * A[6]) / det;
    R[5] = (A[2] * A[3] - A[0] * A[5]) / det;
    R[6] = (A[3] * A[7] - A[4] * A[6]) / det;
    R[7] = (A[1] * A[6] - A[0] * A[7]) / det;
    R[8] = (A[0] * A[4] - A[1] * A[3]) / det;
    return true;
}

nao_status bad(nao_status s, const std::string &msg) {
    nao_set_last_error(msg);
    return s;
}

}  // namespace

extern "C" {

nao_status nao_periodic_images(const double *atom_xyz, int32_t n_atoms, const double *lattice, double reach,
                               int32_t max_images, double *img_xyz, int32_t *img_atom, int32_t *img_cell,
                               int32_t *n_images) {
    if (!atom_xyz || !lattice || !n_images || n_atoms <= 0 || !(reach >= 0.0) || max_images < 0)
        return bad(NAO_ERR_INVALID_ARG, "nao_periodic_images: bad argument");
    double Ainv[9];
    if (!inv3(lattice, Ainv)) return bad(NAO_ERR_INVALID_ARG, "nao_periodic_images: singular lattice");
    // fractional coordinates f = x Ainv (x = f A, rows of A are a1, a2, a3); the planes f_c =
    // const are 1 / |column c of Ainv| apart, so reach is m_c = reach |column c| in f_c
    double m[3];
    for (int c = 0; c < 3; c++)
        m[c] = reach * std::sqrt(Ainv[c] * Ainv[c] + Ainv[3 + c] * Ainv[3 + c] + Ainv[6 + c] * Ainv[6 + c]);
    const double eps = 1e-12;
    std::vector<double> xyz;
    std::vector<int32_t> atom, cell;
    for (int pass = 0; pass < 2; pass++)  // the atoms themselves (T = 0) first, then the other images
        for (int32_t a = 0; a < n_atoms; a++) {
            const double *x = atom_xyz + 3 * (int64_t)a;
            double f[3];
            for (int c = 0; c < 3; c++) f[c] = x[0] * Ainv[c] + x[1] * Ainv[3 + c] + x[2] * Ainv[6 + c];
            int lo[3], hi[3];
            for (int c = 0; c < 3; c++) {
                lo[c] = (int)std::floor(-m[c] - f[c]) - 1;
                hi[c] = (int)std::ceil(1.0 + m[c] - f[c]) + 1;
                if (hi[c] - lo[c] > 2000) return bad(NAO_ERR_INVALID_ARG, "nao_periodic_images: reach too large for the cell");
            }
            for (int n0 = lo[0]; n0 <= hi[0]; n0++)
                for (int n1 = lo[1]; n1 <= hi[1]; n1++)
                    for (int n2 = lo[2]; n2 <= hi[2]; n2++) {
                        const bool home = n0 == 0 && n1 == 0 && n2 == 0;
                        if ((pass == 0) != home) continue;
                        const int n[3] = {n0, n1, n2};
                        bool keep = true;
                        for (int c = 0; c < 3 && keep; c++) {
                            const double g = f[c] + n[c];
                            keep = g > -m[c] - eps && g < 1.0 + m[c] + eps;
                        }
                        if (!keep && !home) continue;
                        for (int c = 0; c < 3; c++)
                            xyz.push_back(x[c] + n0 * lattice[c] + n1 * lattice[3 + c] + n2 * lattice[6 + c]);
                        atom.push_back(a);
                        cell.push_back(n0);
                        cell.push_back(n1);
                        cell.push_back(n2);
                    }
        }
    *n_images = (int32_t)atom.size();
    if ((int64_t)atom.size() > max_images)
        return bad(NAO_ERR_INVALID_ARG, "nao_periodic_images: " + std::to_string(atom.size()) +
                                            " images exceed max_images (n_images holds the count)");
    if (!img_xyz || !img_atom || !img_cell) return bad(NAO_ERR_INVALID_ARG, "nao_periodic_images: NULL output");
    std::copy(xyz.begin(), xyz.end(), img_xyz);
    std::copy(atom.begin(), atom.end(), img_atom);
    std::copy(cell.begin(), cell.end(), img_cell);
    return NAO_OK;
}

nao_status nao_periodic_basis_map(const int32_t *atom_species, int32_t n_atoms, const int32_t *species_fn_offset,
                                  int32_t n_species, const int32_t *fn_l, const int32_t *img_atom, int32_t n_images,
                                  int64_t max_rs, int32_t *fn_map, int32_t *fn_image, int64_t *n_rs) {
    if (!atom_species || !species_fn_offset || !fn_l || !img_atom || !n_rs || n_atoms <= 0 || n_species <= 0 ||
        n_images < 0)
        return bad(NAO_ERR_INVALID_ARG, "nao_periodic_basis_map: bad argument");
    std::vector<int64_t> first(n_atoms + 1, 0);
    std::vector<int32_t> count(n_atoms, 0);
    for (int32_t a = 0; a < n_atoms; a++) {
        const int32_t sp = atom_species[a];
        if (sp < 0 || sp >= n_species) return bad(NAO_ERR_INVALID_ARG, "nao_periodic_basis_map: bad species");
        int32_t c = 0;
        for (int32_t f = species_fn_offset[sp]; f < species_fn_offset[sp + 1]; f++) c += 2 * fn_l[f] + 1;
        count[a] = c;
        first[a + 1] = first[a] + c;
    }
    int64_t total = 0;
    for (int32_t k = 0; k < n_images; k++) {
        if (img_atom[k] < 0 || img_atom[k] >= n_atoms) return bad(NAO_ERR_INVALID_ARG, "nao_periodic_basis_map: bad image atom");
        total += count[img_atom[k]];
    }
    *n_rs = total;
    if (total > max_rs) return bad(NAO_ERR_INVALID_ARG, "nao_periodic_basis_map: n_rs exceeds max_rs (n_rs holds the count)");
    if (!fn_map || !fn_image) return bad(NAO_ERR_INVALID_ARG, "nao_periodic_basis_map: NULL output");
    int64_t pos = 0;
    for (int32_t k = 0; k < n_images; k++) {
        const int32_t a = img_atom[k];
        for (int32_t t = 0; t < count[a]; t++, pos++) {
            fn_map[pos] = (int32_t)(first[a] + t);
            fn_image[pos] = k;
        }
    }
    return NAO_OK;
}

nao_status nao_bloch_sum(const double *h_uc_dev, int64_t n_rs, const int32_t *fn_map_dev, const int32_t *fn_image_dev,
                         const int32_t *img_cell_dev, int32_t n_images, const double *lattice, const double *k_dev,
                         int32_t n_k, int64_t nb, double *hk_dev, int32_t *err_dev, void *cuda_stream) {
    if (!h_uc_dev || !fn_map_dev || !fn_image_dev || !img_cell_dev || !lattice || !k_dev || !hk_dev || n_rs <= 0 ||
        n_k <= 0 || nb <= 0 || n_k > 65535 || n_images <= 0)
        return bad(NAO_ERR_INVALID_ARG, "nao_bloch_sum: bad argument");
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    Lattice L;
    for (int c = 0; c < 9; c++) L.a[c] = lattice[c];
    const int64_t blocks = (n_rs * n_rs + 255) / 256;
    if (blocks > 0x7FFFFFFF) return bad(NAO_ERR_INVALID_ARG, "nao_bloch_sum: h^uc too large");
    cudaError_t e = err_dev ? cudaMemsetAsync(err_dev, 0, sizeof(int32_t), st) : cudaSuccess;
    if (e == cudaSuccess && err_dev) {
        bloch_check_kernel<<<(unsigned)n_rs, 256, 0, st>>>(h_uc_dev, n_rs, fn_map_dev, fn_image_dev, n_images, nb, err_dev);
        e = cudaGetLastError();
    }
    // the row form where its tables fit, with as many k points per CTA as there are, up to 8
    const int KQ = n_k >= 8 ? 8 : (n_k >= 4 ? 4 : (n_k >= 2 ? 2 : 1));
    if (e != cudaSuccess) {
    } else if (nb < (1 << 20) && bloch_rows_smem(n_rs, n_images, nb, KQ) <= bloch_smem_limit(nb <= kBlochThreads / 2)) {
#define NAO_BLOCH(K)                                                                             \
    (nb <= kBlochThreads / 2 ? launch_bloch_rows<K, true> : launch_bloch_rows<K, false>)(        \
        h_uc_dev, (int32_t)n_rs, fn_map_dev, fn_image_dev, img_cell_dev, n_images, L, k_dev, n_k, \
        (int32_t)nb, hk_dev, st)
        e = KQ == 8 ? NAO_BLOCH(8) : KQ == 4 ? NAO_BLOCH(4) : KQ == 2 ? NAO_BLOCH(2) : NAO_BLOCH(1);
#undef NAO_BLOCH
    } else {
        e = cudaMemsetAsync(hk_dev, 0, 2 * (size_t)n_k * (size_t)nb * (size_t)nb * sizeof(double), st);
        if (e == cudaSuccess) {
            bloch_kernel<<<dim3((unsigned)blocks, (unsigned)n_k), 256, 0, st>>>(h_uc_dev, n_rs, fn_map_dev, fn_image_dev,
                                                                                img_cell_dev, n_images, L, k_dev, nb, hk_dev);
            e = cudaGetLastError();
        }
    }
    if (e != cudaSuccess) return bad(NAO_ERR_CUDA, std::string("nao_bloch_sum: ") + cudaGetErrorString(e));
    return NAO_OK;
}

}  // extern "C"
