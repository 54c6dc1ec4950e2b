// Bit-pattern helpers of the split (Ozaki) path, shared by the density's evaluation kernel
// (which reduces the point exponents while it produces the values) and the slicing kernels
// (which turn the values into digits).
//
// On this GPU the FP64 pipe is ~1/60 of the FP32 rate, so exponents are taken from FP64 bit
// patterns with integer and FP32 instructions rather than from FP64 products.
#pragma once

#ifdef __CUDACC__
#include "nao_internal.h"

namespace split_bits {

// |x| as an ordered integer: for non-negative doubles the bit patterns order like the values.
__device__ __forceinline__ long long abs_bits(double x) { return __double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFLL; }

// The biased exponent field of the FP64 with bit pattern xb.
__device__ __forceinline__ int biased_exponent(long long xb) { return (int)((xb >> 52) & 0x7FF); }

// Exponent e with max * 2^-e in [0.25, 0.5), from the biased exponent eb of max; rows whose
// magnitude is below 2^-900 (or zero, eb = 0) are taken as zero (flag -10000).
__device__ __forceinline__ int exponent_of_binade(int eb) {
    if (eb <= 0) return -10000;
    const int ex = eb - 1022;  // max = f 2^ex, f in [0.5, 1)
    return ex < -900 ? -10000 : ex + 1;
}

// d_k of the Hamiltonian's column k = (component c, batch-ordered point p): w v on the potential
// part (c = 0), w (kappa + v_tau) / 2 on the three gradient parts (Eq. H_decomp; kappa = 1 with
// the kinetic term, v_tau with the meta-GGA term), 0 for a term that is off; the column's scale
// is sqrt|d_k| (formed in the H slicer).
__device__ __forceinline__ double h_column_weight(const DevSystem &s, int m, int p, int c, uint32_t terms) {
    const double w = s.pw[p];
    if (c == 0) return (terms & NAO_TERM_POTENTIAL) ? w * v_at(s, m, p) : 0.0;
    const double kin = (terms & NAO_TERM_KINETIC) ? 1.0 : 0.0;
    return 0.5 * w * ((terms & NAO_TERM_TAU) ? kin + vt_at(s, m, p) : kin);
}

}  // namespace split_bits
#endif
