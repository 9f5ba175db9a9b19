// Column vectors and the six-neighbour sum shared by the grid kernels.
#pragma once
#include <cuda_runtime.h>

namespace hq {

template <typename T, int V>
struct alignas(sizeof(T) * V) VT {
    T v[V];
};

template <typename T, int V>
__device__ __forceinline__ VT<T, V> ldv(const T *p) {
    return *reinterpret_cast<const VT<T, V> *>(p);
}
template <typename T, int V>
__device__ __forceinline__ void stv(T *p, const VT<T, V> &x) {
    *reinterpret_cast<VT<T, V> *>(p) = x;
}

// sum of six neighbours in the order west, east, south, north, below, above;
// in[k] false: outside the grid (the value loaded for it counts as zero)
__device__ __forceinline__ float sum6(const float (&x)[6], const bool (&in)[6]) {
    float a[6];
#pragma unroll
    for (int k = 0; k < 6; k++) a[k] = in[k] ? x[k] : 0.f;
    return ((a[0] + a[1]) + (a[2] + a[3])) + (a[4] + a[5]);
}

// Six FP64 values summed on the integer pipes.  GB300 retires 0.5 FP64 lanes
// per clock and scheduler, so the five additions of a 7-point sum hold the
// FP64 pipe for 280 clocks per warp (measured), more than half of every FP64
// sweep; the same sum takes about 100 integer-ALU instructions (200 clocks) on
// another pipe than the products around it.  Measured: the operator at 64^3,
// 64 columns 272 -> 130 us (FP64 pipe 68%, integer ALU 75% busy), an FP64
// block PCG at 64^3, 32 columns 10.9 -> 8.1 ms.  Moving the shifts and
// additions to the FMA pipe as wide multiply-adds was slower (240 against 198
// clocks per sum).  The terms are aligned to the largest
// exponent E of the six as 60-bit magnitudes (7 guard bits below the 53 of
// the largest term), added in 64 bits and rounded once: the error is at most
// 6 truncations of 2^-59 2^E and one rounding of the result.  That is an absolute
// bound, relative to the largest term: where larger terms cancel exactly, what lies 59
// binades below them is lost, which additions in a lucky order would have kept.  The
// sum is an odd, order-independent function of its terms.  Terms with E outside [64, 2040]
// (subnormal or near overflow) are scaled by a power of two first; an infinity
// or a NaN among them takes the plain additions.
// hi, lo, ex: the words and biased exponents of the six values, E: the largest
// exponent.
__device__ __forceinline__ double sum6_aligned(const unsigned (&hi)[6], const unsigned (&lo)[6],
                                               const unsigned (&ex)[6], unsigned E) {
    long long s = 0;
    int neg = 0;   // number of negative terms
#pragma unroll
    for (int k = 0; k < 6; k++) {
        const int sg = (int)hi[k] >> 31;   // all ones for a negative term
        unsigned mh;   // (hi & 0x000fffff) | 0x00100000 in one instruction
        asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(mh) : "r"(hi[k]), "r"(0x000fffffu), "r"(0x00100000u));
        const int vh = (int)__funnelshift_l(lo[k], mh, 7) ^ sg;
        const unsigned vl = (lo[k] << 7) ^ (unsigned)sg;
        const long long v = ((long long)vh << 32) | vl;
        long long w;
        // one's complement: ~(|v| >> d), one short of -(|v| >> d); shr clamps
        // shifts of 64 and more (a zero or far smaller term: 0)
        asm("shr.s64 %0, %1, %2;" : "=l"(w) : "l"(v), "r"(E - ex[k]));
        s += w;
        neg -= sg;
    }
    s += neg;
    const int sm = (int)(s >> 32) >> 31;
    const unsigned long long u = (unsigned long long)((s ^ sm) - sm);
    // the magnitude's leading bit to bit 62, rounded to the 53 bits 62 .. 10
    const int lz = __clzll((long long)u);
    const unsigned long long t = (u << (lz - 1)) + 512ull;
    const unsigned th = (unsigned)(t >> 32);
    const unsigned rh = ((th >> 10) + ((E + 3u - (unsigned)lz) << 20)) | ((unsigned)sm & 0x80000000u);
    return u == 0 ? 0.0 : __hiloint2double((int)rh, (int)__funnelshift_r((unsigned)t, th, 10));
}
// a[k] or zero: the terms of the rare exponents
static __device__ __noinline__ double sum6_scaled(double a0, double a1, double a2, double a3, double a4,
                                           double a5) {
    double a[6] = {a0, a1, a2, a3, a4, a5};
    unsigned hi[6], lo[6], ex[6], E = 0, any = 0;
#pragma unroll
    for (int k = 0; k < 6; k++) {
        E = max(E, ((unsigned)__double2hiint(a[k]) << 1) >> 21);
        any |= ((unsigned)__double2hiint(a[k]) << 1) | (unsigned)__double2loint(a[k]);
    }
    // six zeros, the first residual of a solve from zero: the scaling's products on
    // the FP64 pipe made it the slowest case of all (64^3, 64 columns 478 us)
    if (any == 0) return 0.0;
    if (E == 2047u) return ((a0 + a1) + (a2 + a3)) + (a4 + a5);
    const bool low = E < 64u;
    E = 0;
#pragma unroll
    for (int k = 0; k < 6; k++) {
        a[k] *= low ? 0x1p128 : 0x1p-128;
        hi[k] = (unsigned)__double2hiint(a[k]);
        lo[k] = (unsigned)__double2loint(a[k]);
        ex[k] = (hi[k] << 1) >> 21;
        E = max(E, ex[k]);
    }
    return sum6_aligned(hi, lo, ex, E) * (low ? 0x1p-128 : 0x1p128);
}
__device__ __forceinline__ double sum6(const double (&a)[6], const bool (&in)[6]) {
    unsigned hi[6], lo[6], ex[6], E = 0;
#pragma unroll
    for (int k = 0; k < 6; k++) {
        // a term outside the grid gets exponent 0: shifted out whatever its low word
        hi[k] = in[k] ? (unsigned)__double2hiint(a[k]) : 0u;
        lo[k] = (unsigned)__double2loint(a[k]);
        ex[k] = (hi[k] << 1) >> 21;
        E = max(E, ex[k]);
    }
    if (E - 64u > 2040u - 64u)
        return sum6_scaled(in[0] ? a[0] : 0.0, in[1] ? a[1] : 0.0, in[2] ? a[2] : 0.0,
                           in[3] ? a[3] : 0.0, in[4] ? a[4] : 0.0, in[5] ? a[5] : 0.0);
    return sum6_aligned(hi, lo, ex, E);
}

// (A x)_p and (b - A x)_p of a point from its neighbour sum, with the roundings
// spelled out where kernels have to agree bit for bit
__device__ __forceinline__ double op_value(double d, double x, double c, double s) {
    return fma(d, x, -(c * s));
}
__device__ __forceinline__ float op_value(float d, float x, float c, float s) { return d * x - c * s; }
__device__ __forceinline__ double resid_value(double b, double d, double x, double c, double s) {
    return fma(c, s, fma(-d, x, b));
}
__device__ __forceinline__ float resid_value(float b, float d, float x, float c, float s) {
    return (b - d * x) + c * s;
}

// groups in which the thread rows of a CTA are summed (block_col_reduce): the
// rows of a group in order, then the groups in order
__host__ __device__ __forceinline__ int row_groups(int ty) { return ty >= 16 ? 8 : 1; }

// (double) f through integers: a conversion is an FP64-pipe instruction (56
// clocks per warp, as an FMA), the bit form seven of the integer ALU.  Zeros,
// subnormals, infinities and NaN take the conversion.
__device__ __forceinline__ double widen(float f) {
    const unsigned u = __float_as_uint(f), e = u & 0x7f800000u;
    if (e - 0x00800000u >= 0x7f000000u) return (double)f;
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)),
                            (int)(u << 29));
}

}  // namespace hq
