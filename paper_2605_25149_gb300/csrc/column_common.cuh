// Index arithmetic of the kernels that keep one column's levels in shared memory
// (k_vcoarse.cu, k_pcg_small.cu).
#pragma once

namespace hq {

constexpr int VC_THREADS = 1024;
constexpr int VT4 = 4;   // restriction taps in use: mc = mf / 2 gives at most four

// a / d for 0 <= a < 2^22 and 1 <= d < 2^12: the quotient through the FP32
// reciprocal (relative error below 2^-23, so at most one off) and one
// correction step; a few instructions instead of an integer division's
// sequence, which dominated this kernel's index set-up per pass
__device__ __forceinline__ int fdiv(int a, int d) {
    int q = __float2int_rz(__int2float_rn(a) * __frcp_rn(__int2float_rn(d)));
    const int r = a - q * d;
    q += r < 0 ? -1 : (r >= d ? 1 : 0);
    return q;
}

__device__ __forceinline__ void decomp(int p, int m, int &i, int &j, int &k) {
    const int q = fdiv(p, m);
    i = p - q * m;
    k = fdiv(q, m);
    j = q - k * m;
}

}  // namespace hq
