// FP64 block x small-matrix products on the tcgen05 tensor cores by exact
// integer slicing (the splitting idea of Ozaki, Ogita, Oishi and Rump, 2012).
//
//   Out (n x ncol) = [A1 A2] (n x K) [M1; M2] (K x ncol) (+ Cin), all FP64.
//
// GB300 retires about two FP64 lane operations per clock per SM, so the FP64
// SIMT form of these products is bound by the FP64 pipe.  Here every value is
// written as a scaled sum of 7 balanced base-256 digits,
//   A[p][k] = 2^(e_p + 1) sum_{i=1..7} a_i 2^(-8i)   (+- 2^-55 |row max|, rounded),
// with e_p taken from the largest exponent of row p (points) of [A1 A2], 2^(e_p - 1) <=
// |row max| < 2^e_p, and likewise for each column c of [M1; M2].  Digits are integers
// -128..128, exact in fp16.  Products of digit pairs with the same i + j = t share the
// scale 2^(-8t) and are accumulated by kind::f16 MMAs into one FP32 TMEM accumulator D_t; every partial sum is an integer of at most
// 7 * K * 128^2 < 2^24 for K <= 128, so the accumulation is exact.  Pairs with
// t <= 8 are kept (the dropped ones, six of t = 9 first, are below 2^-51 of |row max|
// |column max| per term: 6 128^2 2^-72 2^(e_p + f_c + 2); digits 65, -128, .., -128 on both
// sides come to 2^-51.4).  The epilogue combines D_2..D_8 in 64-bit fixed point, converts
// once to FP64, applies 2^(e_p + f_c), adds Cin and optionally sums squares.
// (Eight 7-bit sign-magnitude digits in bf16 have the same bounds but 36 digit
// products instead of 28, and took 3.5 instead of 1.3 instructions per digit
// to extract, where these kernels are bound by the integer pipe.)
//
// CTA = 128 points x 64 output columns, all K; per 64-wide K chunk the 512
// threads (256 hid less of the latencies: 355 against 321 us at 64^3, K = 64)
// convert the FP64 rows into 7 digit planes (K-major, 128-byte
// swizzle) while bulk copies bring the 7 digit planes of the small matrix
// (prepared once per call by k_oz_split); one thread issues the 28 digit
// products of a K step of 16 as 10 MMAs.  TMEM: 7 accumulators x 64 columns.  The output
// tile is staged in the freed digit planes for whole-row Cin reads and Out
// writes.  Every wait is bounded.
#include "hq_internal.cuh"
#include "tc_common.cuh"

#include <algorithm>

namespace hq {

namespace {

constexpr int OZ_M = 128;                 // points per CTA (TMEM lanes)
constexpr int OZ_NT = 64;                 // output columns per CTA
constexpr int OZ_KC = 64;                 // K per chunk: 128 bytes of fp16 per row
constexpr int OZ_S = 7;                   // digits per value
constexpr int OZ_BITS = 8;                // bits per digit
constexpr int OZ_THREADS = 512;           // 16 warps: warp w reads TMEM lanes 32 (w % 4)..
constexpr int OZ_EC = OZ_NT / (OZ_THREADS / 128);   // output columns per thread (16)
constexpr int OZ_APLANE = OZ_M * 128;     // one digit plane of the point rows: 16 KB
constexpr int OZ_BPLANE = OZ_NT * 128;    // one digit plane of the small matrix: 8 KB
constexpr int OZ_SMEM = OZ_S * (OZ_APLANE + OZ_BPLANE) + 1024;
constexpr int OZ_EBAD = 0x7FF;            // biased exponent of Inf / NaN
constexpr int OZ_FRAC = 40;               // fraction bits of the fixed-point combination
constexpr int OZ_SLD = OZ_NT + 1;         // row stride (doubles) of the staged output tile
static_assert(OZ_M * OZ_SLD * 8 <= OZ_S * OZ_APLANE, "output tile fits the digit planes");

// byte offset of 16-bit element (row r, k) in a K-major tile of 64-element
// rows with the 128-byte swizzle (16-byte chunk c of row r at c ^ (r & 7))
__device__ __forceinline__ uint32_t sw128_offset16(int r, int k) {
    return (uint32_t)((r >> 3) * 1024 + (r & 7) * 128 + ((((k >> 3) ^ (r & 7)) & 7) << 4) +
                      ((k & 7) << 1));
}

// instruction descriptor: D f32, A/B fp16, both K-major
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N) {
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_f16(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(da), "l"(db), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ int biased_exp(double x) {
    return (int)((__double_as_longlong(x) >> 52) & 0x7FF);
}

// F + 0x4040404040404040 with F = x / 2^(emax - 1022) in 62-bit fixed point (0 for
// zero and subnormals; unspecified for Inf and NaN, whose rows and columns the
// exponent marks).  Digit i has its unit at bit 63 - 8i; the constant adds 128
// units to each and half a unit of the last, so the digits are the bytes above
// bit 6 less 128 (the first, of F up to 2^62, can reach 256 - 128).
__device__ __forceinline__ unsigned long long oz_word(double x, int emax) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const int ex = (int)((hi >> 20) & 0x7FF), sg = (int)hi >> 31;
    const uint32_t fh = (__funnelshift_l(lo, hi, 9) & 0x1FFFFFFFu) | 0x20000000u;
    const int d = ex ? emax - ex : 64;   // >= 0; shifts of 64 and more give 0
    unsigned long long f;
    asm("shr.u64 %0, %1, %2;" : "=l"(f) : "l"(((unsigned long long)fh << 32) | (lo << 9)), "r"(d));
    const long long s = sg;
    return (f ^ (unsigned long long)s) + (0x4040404040404040ull - (unsigned long long)s);
}

// the 7 digits of two values of one row / column relative to the biased
// exponent emax as fp16 integers, packed in pairs plane by plane (x0 in the low
// half): a byte b behind 0x64 is 1024 + b, less 1152
__device__ __forceinline__ void oz_digits2(double x0, double x1, int emax, uint32_t (&pk)[OZ_S]) {
    const unsigned long long w0 = oz_word(x0, emax), w1 = oz_word(x1, emax);
    const uint32_t h0 = (uint32_t)(w0 >> 31), h1 = (uint32_t)(w1 >> 31);
    const uint32_t l0 = (uint32_t)w0 << 1, l1 = (uint32_t)w1 << 1;
    const uint32_t y23 = __byte_perm(h0, h1, 0x5612), y67 = __byte_perm(l0, l1, 0x5612);
    pk[0] = __byte_perm((uint32_t)(w0 >> 55), (uint32_t)(w1 >> 55), 0x5410) | 0x64006400u;
    pk[1] = __byte_perm(y23, 0x64u, 0x4240);
    pk[2] = __byte_perm(y23, 0x64u, 0x4341);
    pk[3] = (__byte_perm(h0, h1, 0x4400) & 0x00FF00FFu) | 0x64006400u;
    pk[4] = (__byte_perm(l0, l1, 0x7733) & 0x00FF00FFu) | 0x64006400u;
    pk[5] = __byte_perm(y67, 0x64u, 0x4240);
    pk[6] = __byte_perm(y67, 0x64u, 0x4341);
#pragma unroll
    for (int i = 0; i < OZ_S; i++) asm("sub.f16x2 %0, %0, %1;" : "+r"(pk[i]) : "r"(0x64806480u));
}

// sum_t D_t 2^(-8(t-2)), t = 2 .. 8, of 16 columns as 64-bit fixed point with FRAC
// fraction bits (32 <= FRAC <= 48).  |D_t| <= (t - 1) 2^21: D_2 and D_3 join in 32
// bits, the rest by wide multiply-adds; D_7 and D_8 are truncated once (below
// 2^-FRAC).  tm: the thread's lane and first column.
template <int FRAC>
__device__ __forceinline__ void oz_combine(uint32_t tm, long long (&acc)[16], bool add) {
    static_assert(OZ_S == 7 && OZ_BITS == 8 && FRAC >= 32 && FRAC <= 48, "");
#pragma unroll
    for (int g = 0; g < 16; g += 8) {
        const uint32_t c = tm + (uint32_t)g;
        float a[8], b[8];
        long long q[8];
        int d[8];
        tmem_ld8x2(c, c + OZ_NT, a, b);
#pragma unroll
        for (int j = 0; j < 8; j++) d[j] = __float2int_rn(a[j]) * 256 + __float2int_rn(b[j]);
        tmem_ld8x2(c + 2 * OZ_NT, c + 3 * OZ_NT, a, b);
#pragma unroll
        for (int j = 0; j < 8; j++) {
            q[j] = ((long long)d[j] * 256 + __float2int_rn(a[j])) * 65536;   // units 2^-32
            d[j] = __float2int_rn(b[j]);
        }
        tmem_ld8x2(c + 4 * OZ_NT, c + 5 * OZ_NT, a, b);
#pragma unroll
        for (int j = 0; j < 8; j++) {
            q[j] += (long long)d[j] * 256 + __float2int_rn(a[j]);
            d[j] = __float2int_rn(b[j]);
        }
        tmem_ld8(c + 6 * OZ_NT, a);
#pragma unroll
        for (int j = 0; j < 8; j++)
            acc[g + j] = (add ? acc[g + j] : 0ll) + (q[j] << (FRAC - 32)) +
                         (((long long)d[j] * 256 + __float2int_rn(a[j])) >> (48 - FRAC));
    }
}

__device__ __forceinline__ double pow2(int e) {
    // 2^e for |e| <= 2000 as a product of two normal powers of two
    const int e1 = e / 2, e2 = e - e1;
    return __longlong_as_double((long long)(e1 + 1023) << 52) *
           __longlong_as_double((long long)(e2 + 1023) << 52);
}

// Digit planes of the small matrix [M1; M2] (K x ncol) in the layout the MMA
// reads: image[((ct * kchunks + ch) * 7 + j) * 8 KB] holds digit j of rows =
// output columns ct*64 .. +63 and K = ch*64 .. +63; fexp[c] = the column's
// largest biased exponent.  CTA = one column tile; thread (kg, cl) takes
// column cl and the pairs k = 2 (kg + SPL_G i), 2 (kg + SPL_G i) + 1 (the
// column maxima are reduced over the SPL_G groups in shared memory first).
constexpr int SPL_G = 16;

__global__ void __launch_bounds__(OZ_NT * SPL_G) k_oz_split(int K, int k1, int ncol, int kchunks,
                                                            const double *M1, const double *M2,
                                                            unsigned char *image, int *fexp) {
    __shared__ int emx[SPL_G][OZ_NT];
    const int ct = blockIdx.x, cl = threadIdx.x % OZ_NT, kg = threadIdx.x / OZ_NT;
    const int c = ct * OZ_NT + cl;
    auto val = [&](int k) -> double {
        if (c >= ncol || k >= K) return 0.0;
        return k < k1 ? M1[(size_t)k * ncol + c] : M2[(size_t)(k - k1) * ncol + c];
    };
    const int npairs = kchunks * OZ_KC / 2;
    int em = 0;
    for (int q = kg; q < npairs; q += SPL_G)
        em = max(em, max(biased_exp(val(2 * q)), biased_exp(val(2 * q + 1))));
    emx[kg][cl] = em;
    __syncthreads();
    em = 0;
#pragma unroll
    for (int g = 0; g < SPL_G; g++) em = max(em, emx[g][cl]);
    if (kg == 0 && c < ncol) fexp[c] = em;
    for (int q = kg; q < npairs; q += SPL_G) {
        const int k = 2 * q, ch = k / OZ_KC, kl = k % OZ_KC;
        unsigned char *base = image + (size_t)(ct * kchunks + ch) * OZ_S * OZ_BPLANE;
        uint32_t pk[OZ_S];
        oz_digits2(val(k), val(k + 1), em, pk);
        const uint32_t off = sw128_offset16(cl, kl);
#pragma unroll
        for (int j = 0; j < OZ_S; j++)
            *reinterpret_cast<uint32_t *>(base + (size_t)j * OZ_BPLANE + off) = pk[j];
    }
}

// largest biased exponent of every point row of [A1 A2] (one warp per row)
__global__ void __launch_bounds__(256) k_oz_rowexp(long n, int k1, int k2, const double *A1,
                                                   const double *A2, int *erow) {
    const int lane = threadIdx.x & 31;
    const long p = (long)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (p >= n) return;
    int em = 0;
    for (int k = lane; k < k1; k += 32) em = max(em, biased_exp(A1[(size_t)p * k1 + k]));
    for (int k = lane; k < k2; k += 32) em = max(em, biased_exp(A2[(size_t)p * k2 + k]));
    for (int o = 16; o > 0; o >>= 1) em = max(em, __shfl_xor_sync(0xffffffffu, em, o));
    if (lane == 0) erow[p] = em;
}

// acc 2^es, rounded to FP64: the leading bit to the implicit one by integer
// shifts (the conversion of a 64-bit integer is three FP64-pipe instructions,
// which held that pipe for 10,000 of a tile's 37,000 clocks)
__device__ __forceinline__ double oz_scaled(long long acc, int es) {
    const long long sm = acc >> 63;
    const unsigned long long u = (unsigned long long)((acc ^ sm) - sm);   // < 2^63
    if (u == 0) return 0.0;
    const int lz = __clzll((long long)u), ex = 1086 - lz + es;
    if (ex < 1 || ex > 2045) {   // subnormal or overflowing result
        if (es < -1200) return 0.0;
        const double v = (double)acc;
        return es >= -1022 && es <= 1023 ? v * __longlong_as_double((long long)(es + 1023) << 52) : v * pow2(es);
    }
    const unsigned long long t = (u << (lz - 1)) + 512ull;
    const unsigned long long bits = (t >> 10) + ((unsigned long long)(ex - 1) << 52);
    return __longlong_as_double((long long)(bits | ((unsigned long long)sm << 63)));
}

// Persistent: one CTA per SM strides the tiles (point blocks x column tiles, the
// column tiles of a point block next to each other); an item's start, its TMEM
// allocation and its end cost a third of the one-tile-per-CTA form.  Per 64-wide
// K chunk the digit planes are written in two halves of 32, and the MMAs of the
// first run while the second is converted.  Measured at 64^3 points, K = 64, 64
// columns, with Cin: 375 -> 269 us, and 240 with the base-256 digits; of the
// 35,000 clocks per tile before these the conversion took 6,000, the exposed MMAs
// 7,000, the epilogue 14,000 (removing its arithmetic saved 6,000) and the output
// rows 3,200.
__global__ void __launch_bounds__(OZ_THREADS, 1)
    k_tall_oz(long n, int k1, int k2, int ncol, int kchunks, int ctiles, const double *__restrict__ A1,
              const double *__restrict__ A2, const unsigned char *__restrict__ image,
              const int *__restrict__ fexp, const int *__restrict__ erow_g,
              const double *Cin, double *Out, double *part_sq, int *status) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char *planesA = smem;
    unsigned char *planesB = smem + OZ_S * OZ_APLANE;
    __shared__ uint64_t mbar, bbar;
    __shared__ uint32_t tmem_base_sh;
    __shared__ int erow[OZ_M];
    __shared__ __align__(16) int fexp_sh[OZ_NT];   // largest exponents of the tile's columns
    __shared__ int abort_sh, tmem_free_sh;
    __shared__ double red[OZ_THREADS / 32];
    constexpr uint32_t TCOLS = 512;   // OZ_S accumulators of 64, a power of two

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int K = k1 + k2;
    if (tid == 0) {
        mbar_init(&mbar, 1);
        mbar_init(&bbar, 1);
        abort_sh = 0;
        tmem_free_sh = 1;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tmem_base_sh)),
                     "r"(TCOLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base_sh;
    const long pblocks = (n + OZ_M - 1) / OZ_M, tiles = pblocks * ctiles;
    unsigned commits = 0, bulks = 0;   // thread 0: completed phases of mbar, bbar
    int resident = -1;                 // thread 0: (column tile, chunk) in planesB
    bool copying = false;              // thread 0: a wait for the bulk copies gave up

    // A values of chunk ch of point block pb: half-warp hw takes rows
    // warp 8 + 2 q + hw, lane kk of it the pairs k = 32 h + 2 kk, + 1
    constexpr int RPW = OZ_M / (OZ_THREADS / 32);   // rows per warp (8)
    const int hw = lane >> 4, kk = lane & 15;
    double xv[2][RPW / 2][2];
    auto load = [&](long pb, int ch) {
#pragma unroll
        for (int h = 0; h < 2; h++)
#pragma unroll
            for (int q = 0; q < RPW / 2; q++) {
                const long p = pb * OZ_M + warp * RPW + 2 * q + hw;
#pragma unroll
                for (int e = 0; e < 2; e++) {
                    const int k = ch * OZ_KC + 32 * h + 2 * kk + e;
                    double v = 0.0;
                    if (p < n && k < K) v = k < k1 ? A1[(size_t)p * k1 + k] : A2[(size_t)p * k2 + (k - k1)];
                    xv[h][q][e] = v;
                }
            }
    };
    if ((long)blockIdx.x < tiles) load((long)blockIdx.x / ctiles, 0);

    for (long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const long pb = tile / ctiles, r0 = pb * OZ_M;
        const int ct = (int)(tile % ctiles);
        // row exponents: from k_oz_rowexp when K spans several chunks, else
        // formed below from the chunk's values (erow_g null)
        if (erow_g)
            for (int r = tid; r < OZ_M; r += OZ_THREADS) erow[r] = (r0 + r < n) ? erow_g[r0 + r] : 0;
        if (tid < OZ_NT) fexp_sh[tid] = ct * OZ_NT + tid < ncol ? fexp[ct * OZ_NT + tid] : 0;
        for (int ch = 0; ch < kchunks; ch++) {
            // the planes are free: the MMAs of the previous chunk or tile were
            // waited for
            if (ch > 0 && tid == 0 && !mbar_wait(&mbar, (commits++) & 1u)) abort_sh = 1;
            if (tid == 0 && !abort_sh && resident != ct * kchunks + ch) {
                // the chunk's digit planes of the small matrix arrive by bulk
                // copies while the threads convert A
                const unsigned char *src = image + (size_t)(ct * kchunks + ch) * OZ_S * OZ_BPLANE;
                mbar_expect_tx(&bbar, (uint32_t)(OZ_S * OZ_BPLANE));
#pragma unroll
                for (int j = 0; j < OZ_S; j++)
                    bulk_g2s(planesB + j * OZ_BPLANE, src + j * OZ_BPLANE, OZ_BPLANE, &bbar);
            }
            __syncthreads();
            if (abort_sh) break;
            int em[RPW / 2];
#pragma unroll
            for (int q = 0; q < RPW / 2; q++) {
                const int r = warp * RPW + 2 * q + hw;
                if (erow_g) {
                    em[q] = erow[r];
                } else {
                    em[q] = max(max(biased_exp(xv[0][q][0]), biased_exp(xv[0][q][1])),
                                max(biased_exp(xv[1][q][0]), biased_exp(xv[1][q][1])));
#pragma unroll
                    for (int o = 8; o > 0; o >>= 1)   // over the row's 16 lanes
                        em[q] = max(em[q], __shfl_xor_sync(0xffffffffu, em[q], o));
                    if (kk == 0) erow[r] = em[q];
                }
            }
#pragma unroll
            for (int h = 0; h < 2; h++) {
#pragma unroll
                for (int q = 0; q < RPW / 2; q++) {
                    const int r = warp * RPW + 2 * q + hw;
                    uint32_t pk[OZ_S];
                    oz_digits2(xv[h][q][0], xv[h][q][1], em[q], pk);
                    const uint32_t off = sw128_offset16(r, 32 * h + 2 * kk);
#pragma unroll
                    for (int i = 0; i < OZ_S; i++)
                        *reinterpret_cast<uint32_t *>(planesA + i * OZ_APLANE + off) = pk[i];
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncthreads();
                if (tid == 0 && !abort_sh) {
                    if (h == 0 && resident != ct * kchunks + ch) {
                        if (mbar_wait(&bbar, bulks & 1u)) {
                            resident = ct * kchunks + ch;
                            bulks++;
                        } else {
                            abort_sh = 1;   // no MMA of this chunk is issued
                            copying = true;
                        }
                    }
                    if (!abort_sh) {
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                        for (int ks = 2 * h; ks < 2 * h + 2; ks++) {
                            // digit i of A times digits j = 1 .. 8 - i of the small
                            // matrix: their planes follow each other as 64-row
                            // blocks of one B operand and so do the accumulators
                            // D_{i+1} .. D_8, so up to four digits make one MMA of
                            // 256 columns (10 MMAs in place of 28 of 64 columns,
                            // each of which took 80 clocks, the time A's rows take)
                            const uint32_t ko = ks * 32;
#pragma unroll
                            for (int i = 1; i <= OZ_S; i++) {
                                const uint64_t da = make_desc_sw128(smem_u32(planesA + (i - 1) * OZ_APLANE) + ko);
#pragma unroll
                                for (int j = 1; j <= OZ_S + 1 - i; j += 4) {
                                    const int cnt = OZ_S + 2 - i - j < 4 ? OZ_S + 2 - i - j : 4;
                                    const uint64_t db =
                                        make_desc_sw128(smem_u32(planesB + (j - 1) * OZ_BPLANE) + ko);
                                    mma_f16(tmem + (uint32_t)((i + j - 2) * OZ_NT), da, db,
                                             idesc_f16(OZ_M, cnt * OZ_NT), (ch > 0 || ks > 0 || i > 1) ? 1u : 0u);
                                }
                            }
                        }
                        if (h == 1) mma_commit(&mbar);
                    }
                }
            }
            if (abort_sh) break;   // (set before the barrier of the second half)
            if (ch + 1 < kchunks) load(pb, ch + 1);
        }
        if (abort_sh) break;
        // the tile's rows and columns; the next tile's first values and Cin's
        // tile (coalesced: a warp reads 32 consecutive columns of one row) are
        // loaded while the last MMAs run
        if (tile + gridDim.x < tiles) load((tile + gridDim.x) / ctiles, 0);
        const int ncl = min(OZ_NT, ncol - ct * OZ_NT);
        const long nrw = min((long)OZ_M, n - r0);
        constexpr int EPT = OZ_M * OZ_NT / OZ_THREADS;   // tile elements per thread
        double cpre[EPT];
        if (Cin) {
#pragma unroll
            for (int u = 0; u < EPT; u++) {
                const int idx = tid + u * OZ_THREADS, rr = idx / OZ_NT, jj = idx % OZ_NT;
                cpre[u] = (rr < nrw && jj < ncl) ? Cin[(size_t)(r0 + rr) * ncol + ct * OZ_NT + jj] : 0.0;
            }
        }
        if (tid == 0 && !mbar_wait(&mbar, (commits++) & 1u)) abort_sh = 1;
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (abort_sh) break;
        // the digit planes are free once the MMAs are done: the output tile is
        // staged there (row stride OZ_SLD doubles: a half-warp's 8-byte
        // accesses to one column of 16 rows, or to 16 columns of one row, fall
        // in distinct banks), so Cin is read and Out written in whole rows
        double *stg = reinterpret_cast<double *>(planesA);
        double sq = 0.0;
        if (Cin) {
#pragma unroll
            for (int u = 0; u < EPT; u++) {
                const int idx = tid + u * OZ_THREADS;
                stg[(idx / OZ_NT) * OZ_SLD + idx % OZ_NT] = cpre[u];
            }
            __syncthreads();
        }
        {
            // epilogue: thread = one point row (TMEM lane 32 (warp % 4) + lane)
            // and OZ_EC of the 64 output columns (warp / 4)
            const int r = (warp & 3) * 32 + lane, cb = (warp >> 2) * OZ_EC;
            const int em = erow[r];
            // a 64-bit fixed-point integer with 40 fraction bits (|D_2| < 2^21:
            // no overflow)
            long long acc[OZ_EC];
            oz_combine<OZ_FRAC>(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)cb, acc, false);
            // the columns' exponents, ahead of the outputs
            int fc[OZ_EC];
#pragma unroll
            for (int j = 0; j < OZ_EC; j += 4) {
                const int4 f = *reinterpret_cast<const int4 *>(fexp_sh + cb + j);
                fc[j] = f.x;
                fc[j + 1] = f.y;
                fc[j + 2] = f.z;
                fc[j + 3] = f.w;
            }
            double *sl = stg + r * OZ_SLD + cb;
#pragma unroll
            for (int j = 0; j < OZ_EC; j++) {
                const int es = (em - 1021) + (fc[j] - 1021) - 2 * OZ_BITS - OZ_FRAC;
                double o = em == OZ_EBAD || fc[j] == OZ_EBAD ? __longlong_as_double(0x7FF8000000000000ll)
                                                             : oz_scaled(acc[j], es);
                if (Cin) o += sl[j];
                sl[j] = o;
                // points and columns beyond the block: zero digits, o = 0 (+ Cin's 0)
                if (part_sq) sq = fma(o, o, sq);
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        if (part_sq) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
            if (lane == 0) red[warp] = sq;
        }
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (part_sq && tid == 0) {
            double v = 0.0;
            for (int w = 0; w < OZ_THREADS / 32; w++) v += red[w];
            part_sq[(size_t)pb * ctiles + ct] = v;
        }
        if (Out) {
#pragma unroll
            for (int u = 0; u < EPT; u++) {
                const int idx = tid + u * OZ_THREADS, rr = idx / OZ_NT, jj = idx % OZ_NT;
                if (rr < nrw && jj < ncl)
                    Out[(size_t)(r0 + rr) * ncol + ct * OZ_NT + jj] = stg[rr * OZ_SLD + jj];
            }
        }
        __syncthreads();   // the staged tile and erow are read: the next tile may write them
    }
    __syncthreads();
    if (abort_sh && tid == 0) {
        atomicOr(status, ST_TC_TIMEOUT);
        // the MMAs of the last commit may still be writing TMEM, the bulk copies
        // shared memory: one more bounded wait for them before the columns are
        // released; if the MMAs are still running, the columns stay allocated
        // (only the status word is meaningful after a timeout)
        if (copying) mbar_wait(&bbar, bulks & 1u);
        if (commits > 0) tmem_free_sh = mbar_wait(&mbar, (commits - 1) & 1u) ? 1 : 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0 && tmem_free_sh)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TCOLS)
                     : "memory");
}

// ---------------------------------------------------------------------------
// FP64 Grams by the same digit slicing, with per-column exponents over all
// points (k_oz_colexp): <X, X> = w X^T X of X = [X1 X2] (n x na, na <= 128), or,
// with a third block, <X, Y> = w X^T Y (Y: n x ny).
// CTA = all na rows x 64 output columns over a chunk of points.  A slice of 32
// points has the digit planes of the na rows (operand A) and, contiguously,
// those of the tile's 64 columns (operand B: a second copy of the A rows
// ct*64.., or Y's); 64-byte rows, 64-byte swizzle.  Contiguous planes make four
// digits of B one MMA of up to 256 columns: 10 MMAs per 16 points (28 of 64
// columns would take 80 clocks each).  Two slices are in flight: slice
// s is converted while the MMAs of slice s - 1 run; 512 threads, of which one
// issues the MMAs (a 17th warp for that cost every thread a fifth of its
// registers: spills).  Bound by the integer instructions of the conversion and
// the read-out: 64^3 points, 64 x 64 columns, X and Y separate: 219 -> 180 us
// (36 products of 7-bit digits as MMAs of 64 columns; the same digits with this
// schedule: 215).  The exact-sum bound holds for 128 points, so every four
// slices the seven accumulators are read and added into 64-bit fixed-point
// registers (OZ_GFRAC fraction bits, the rest truncated: below 2^-44 of |x max| |y max|
// per read-out); the chunk's FP64 partial tile is
// summed over chunks in a fixed order by k_oz_gram_reduce.  D_t(i,j) and
// D_t(j,i) are the same integers, so <X, X> is exactly symmetric.
// ---------------------------------------------------------------------------
constexpr int OZ_GFRAC = 32;
constexpr int OZ_GKC = 32;                       // points per slice: 64-byte rows
constexpr int OZ_GPLANE = OZ_M * 64;             // one digit plane of a slice's rows: 8 KB
constexpr int OZ_GBPLANE = OZ_NT * 64;           // and of its columns: 4 KB
constexpr int OZ_GSTAGE = OZ_S * (OZ_GPLANE + OZ_GBPLANE);   // the planes of a slice: 84 KB
constexpr int OZ_GST = 2;                        // slices in flight
constexpr int OZ_GFLUSH = 128 / OZ_GKC;          // slices per exact accumulation
constexpr int OZ_GSMEM = OZ_GST * OZ_GSTAGE + 2048;   // + alignment slack

// byte offset of 16-bit element (row r, k) in a K-major tile of 32-element
// rows with the 64-byte swizzle (16-byte chunk c of row r at c ^ ((r >> 1) & 3))
__device__ __forceinline__ uint32_t sw64_offset16(int r, int k) {
    return (uint32_t)((r >> 3) * 512 + (r & 7) * 64 + ((((k >> 3) ^ (r >> 1)) & 3) << 4) +
                      ((k & 7) << 1));
}

// shared-memory matrix descriptor: K-major, 64-byte swizzle, SBO = 512 B
__device__ __forceinline__ uint64_t make_desc_sw64(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFF) >> 4);   // start address
    d |= (uint64_t)(1) << 16;                  // leading byte offset (unused, swizzled K-major)
    d |= (uint64_t)(512 >> 4) << 32;           // stride byte offset: 8 rows x 64 B
    d |= (uint64_t)1 << 46;                    // descriptor version (sm_100 family)
    d |= (uint64_t)4 << 61;                    // swizzle mode: 64 B
    return d;
}

// colexp[c] = the largest biased exponent of column c of [X1 X2] (zeroed before)
__global__ void __launch_bounds__(256) k_oz_colexp(long n, int n1, int n2, const double *X1,
                                                   const double *X2, int *colexp) {
    const int na = n1 + n2, per = 256 / na;   // rows per pass of the CTA
    const int c = threadIdx.x % na, g = threadIdx.x / na;
    if (g >= per) return;
    const double *src = c < n1 ? X1 + c : X2 + (c - n1);
    const size_t ld = c < n1 ? n1 : n2;
    const long step = (long)gridDim.x * per;
    int em = 0;
    for (long p = (long)blockIdx.x * per + g; p < n; p += 4 * step) {
        int e[4];
#pragma unroll
        for (int u = 0; u < 4; u++) e[u] = p + u * step < n ? biased_exp(src[(size_t)(p + u * step) * ld]) : 0;
        em = max(em, max(max(e[0], e[1]), max(e[2], e[3])));
    }
    atomicMax(&colexp[c], em);
}

// 512 threads convert; they meet at mbarriers: full[st] (the planes of a slice
// are written; OZ_GISSUE issues its MMAs), done[st] (these completed, the stage is
// free) and tfree (the accumulators were read out at a flush)
constexpr int OZ_GTHREADS = 512;
constexpr int OZ_GISSUE = OZ_GTHREADS - 32;   // of the warp with the fewest units

template <bool HASY>
__global__ void __launch_bounds__(OZ_GTHREADS, 1)
    k_gram_oz(long n, int n1, int n2, int ny, long chunk_rows, const double *__restrict__ X1,
              const double *__restrict__ X2, const double *__restrict__ Y, const int *__restrict__ colexp,
              const int *__restrict__ yexp, double *__restrict__ partials, int *status) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *planes = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ uint64_t full[OZ_GST], done[OZ_GST], tfree;
    __shared__ uint32_t tmem_base_sh;
    __shared__ int cexp[OZ_M], bexp[OZ_NT];   // exponents of the rows, of the tile's columns
    __shared__ volatile int abort_sh;
    __shared__ int last_sh, tmem_free_sh;
    constexpr uint32_t TCOLS = 512;   // OZ_S accumulators of 64, a power of two
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int na = n1 + n2, ct = blockIdx.x;   // output column tile
    const int nb = HASY ? ny : na;                   // output columns
    const long p0 = (long)blockIdx.y * chunk_rows;
    const long p1 = (n < p0 + chunk_rows) ? n : p0 + chunk_rows;
    const int nslices = p1 > p0 ? (int)((p1 - p0 + OZ_GKC - 1) / OZ_GKC) : 0;
    if (tid == 0) {
        for (int i = 0; i < OZ_GST; i++) {
            mbar_init(&full[i], OZ_GTHREADS);
            mbar_init(&done[i], 1);
        }
        mbar_init(&tfree, OZ_GTHREADS);
        abort_sh = 0;
        last_sh = -1;   // last slice whose MMAs were committed
        tmem_free_sh = 1;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < OZ_M) cexp[tid] = tid < na ? colexp[tid] : 0;
    if (tid < OZ_NT) bexp[tid] = ct * OZ_NT + tid < nb ? (HASY ? yexp : colexp)[ct * OZ_NT + tid] : 0;
    // rows and columns beyond the blocks keep these zero digits
    if (na < OZ_M || nb < (ct + 1) * OZ_NT)
        for (int t = tid; t < OZ_GST * OZ_GSTAGE / 16; t += OZ_GTHREADS)
            reinterpret_cast<uint4 *>(planes)[t] = make_uint4(0, 0, 0, 0);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tmem_base_sh)),
                     "r"(TCOLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base_sh;
    // completion of the MMAs of slice q: the (q / OZ_GST)-th commit on
    // done[q % OZ_GST].  No thread can run a phase ahead of the one another
    // waits for (each next arrival needs the awaited phase), so every
    // parity below is unambiguous.
    auto wait_done = [&](int q) -> bool {
        return mbar_wait(&done[q % OZ_GST], (unsigned)((q / OZ_GST) & 1));
    };
    // TMEM is read by whole converged warps (tcgen05.ld.sync.aligned), so every
    // exit from the slice loop is a decision of the warp, and the lanes that went
    // their own ways (units without values, the issuing thread) meet again first.
    auto warp_aborted = [&]() -> bool { return __any_sync(0xffffffffu, abort_sh); };
    auto warp_done = [&](int q) -> bool { return __all_sync(0xffffffffu, wait_done(q)); };
    // fixed-point sums: thread = TMEM lane 32 (warp % 4) + lane (Gram row), 16
    // output columns (warp / 4)
    const int grow = (warp & 3) * 32 + lane, gcb = (warp >> 2) * 16;
    long long facc[16];
#pragma unroll
    for (int j = 0; j < 16; j++) facc[j] = 0;
    auto flush = [&]() {
        __syncwarp();
        oz_combine<OZ_GFRAC>(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)gcb, facc, true);
    };
    // the MMAs of slice sl (one thread): digit i of the rows times up to four
    // digits j of the columns, j <= 8 - i, into D_{i + j}..; i = 1 reaches all
    // seven accumulators, so it comes first and starts a fresh sum
    auto issue = [&](int sl, bool fresh) {
        const uint32_t stage = smem_u32(planes + (sl % OZ_GST) * OZ_GSTAGE);
#pragma unroll
        for (int ks = 0; ks < OZ_GKC / 16; ks++) {
            const uint32_t ko = ks * 32;
#pragma unroll
            for (int i = 1; i <= OZ_S; i++) {
                const uint64_t da = make_desc_sw64(stage + (i - 1) * OZ_GPLANE + ko);
#pragma unroll
                for (int j = 1; j <= OZ_S + 1 - i; j += 4) {
                    const int nd = OZ_S + 2 - i - j < 4 ? OZ_S + 2 - i - j : 4;
                    const uint64_t db = make_desc_sw64(stage + OZ_S * OZ_GPLANE + (j - 1) * OZ_GBPLANE + ko);
                    mma_f16(tmem + (uint32_t)((i + j - 2) * OZ_NT), da, db, idesc_f16(OZ_M, nd * OZ_NT),
                             fresh && ks == 0 && i == 1 ? 0u : 1u);
                }
            }
        }
        mma_commit(&done[sl % OZ_GST]);
        last_sh = sl;
    };
    // Conversion units: 16 columns (of X, then of Y, each padded to 16) x 8 points
    // per warp; lane = column lane >> 1, points 4 (lane & 1) .. + 3, so that the
    // lanes of a column fill one 16-byte chunk of each digit plane (no bank
    // conflicts) and loads are 128-byte rows.  A unit's values of the next slice
    // are loaded as soon as it is converted, under the conversion of the others.
    constexpr int U = HASY ? 3 : 2;
    const int ga = (na + 15) / 16, ng = ga + (HASY ? (min(ny - ct * OZ_NT, OZ_NT) + 15) / 16 : 0);
    const double *src[U];   // the unit's first point of slice 0 (null: none)
    int ld[U], ue[U], pt[U];
    uint32_t off[U], offb[U];   // first plane of the values, and of their copy (offb != 0)
#pragma unroll
    for (int k = 0; k < U; k++) {
        const int wu = warp + k * (OZ_GTHREADS / 32), grp = wu % ng, oct = wu / ng;
        const bool isy = HASY && grp >= ga;
        const int c = (isy ? grp - ga : grp) * 16 + (lane >> 1);   // row of the planes
        const int col = isy ? ct * OZ_NT + c : c;
        src[k] = nullptr;
        ld[k] = ue[k] = 0;
        off[k] = offb[k] = 0;
        pt[k] = 8 * oct + 4 * (lane & 1);
        if (oct >= OZ_GKC / 8 || col >= (isy ? ny : na)) continue;
        ld[k] = isy ? ny : (col < n1 ? n1 : n2);
        src[k] = (isy ? Y + col : (col < n1 ? X1 + col : X2 + (col - n1))) + (size_t)(p0 + pt[k]) * ld[k];
        ue[k] = isy ? bexp[c] : cexp[c];
        off[k] = (isy ? OZ_S * OZ_GPLANE : 0) + sw64_offset16(c, pt[k]);
        const int bc = c - ct * OZ_NT;
        if (!HASY && bc >= 0 && bc < OZ_NT) offb[k] = OZ_S * OZ_GPLANE + sw64_offset16(bc, pt[k]);
    }
    double xv[U][4];
    auto load = [&](int sl, int k) {
        const long left = src[k] ? p1 - p0 - (long)sl * OZ_GKC - pt[k] : 0;   // points there are
        const double *q = src[k] + (size_t)sl * OZ_GKC * ld[k];
#pragma unroll
        for (int j = 0; j < 4; j++) xv[k][j] = j < left ? q[(size_t)j * ld[k]] : 0.0;
    };
    if (nslices > 0)
#pragma unroll
        for (int k = 0; k < U; k++) load(0, k);
    for (int sl = 0; sl < nslices; sl++) {
        if (warp_aborted()) break;
        const int st = sl % OZ_GST;
        const bool fresh = sl % OZ_GFLUSH == 0;
        // the stage's previous slice is consumed
        if (sl >= OZ_GST && !warp_done(sl - OZ_GST)) {
            abort_sh = 1;
            break;
        }
        unsigned char *stage = planes + st * OZ_GSTAGE;
#pragma unroll
        for (int k = 0; k < U; k++) {
            if (!src[k]) continue;
            uint32_t lo[OZ_S], hi[OZ_S];
            oz_digits2(xv[k][0], xv[k][1], ue[k], lo);
            oz_digits2(xv[k][2], xv[k][3], ue[k], hi);
            if (sl + 1 < nslices) load(sl + 1, k);
            const uint32_t ps = HASY && off[k] >= OZ_S * OZ_GPLANE ? OZ_GBPLANE : OZ_GPLANE;
#pragma unroll
            for (int i = 0; i < OZ_S; i++)
                *reinterpret_cast<uint2 *>(stage + off[k] + i * ps) = make_uint2(lo[i], hi[i]);
            if (!HASY && offb[k])
#pragma unroll
                for (int i = 0; i < OZ_S; i++)
                    *reinterpret_cast<uint2 *>(stage + offb[k] + i * OZ_GBPLANE) = make_uint2(lo[i], hi[i]);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive(&full[st]);
        if (fresh && sl > 0) {
            // 128 points accumulated: every MMA so far is complete
            if (!warp_done(sl - 1)) {
                abort_sh = 1;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            flush();
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mbar_arrive(&tfree);
        }
        if (tid == OZ_GISSUE) {
            if (!mbar_wait(&full[st], (unsigned)((sl / OZ_GST) & 1)) ||
                (fresh && sl > 0 && !mbar_wait(&tfree, (unsigned)((sl / OZ_GFLUSH - 1) & 1)))) {
                abort_sh = 1;
            } else {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                issue(sl, fresh);
            }
        }
        __syncwarp();
    }
    if (!abort_sh && nslices > 0 && !wait_done(nslices - 1)) abort_sh = 1;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // after a wait that gave up, one more bounded wait for the last commit
    // before the columns are released (if it fails too they stay allocated,
    // and only the status word is meaningful)
    if (tid == OZ_GISSUE && abort_sh && last_sh >= 0) tmem_free_sh = wait_done(last_sh) ? 1 : 0;
    __syncthreads();
    if (abort_sh) {
        if (tid == 0) atomicOr(status, ST_TC_TIMEOUT);
    } else {
        if (nslices > 0) flush();
        double *dst = partials + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * OZ_M * OZ_NT;
        const int ea = cexp[grow];
#pragma unroll
        for (int j = 0; j < 16; j++) {
            double o = 0.0;
            if (grow < na && ct * OZ_NT + gcb + j < nb) {
                const int eb = bexp[gcb + j];
                const int es = (ea - 1021) + (eb - 1021) - 2 * OZ_BITS - OZ_GFRAC;
                o = ea == OZ_EBAD || eb == OZ_EBAD ? __longlong_as_double(0x7FF8000000000000ll)
                                                   : oz_scaled(facc[j], es);
            }
            dst[(size_t)grow * OZ_NT + gcb + j] = o;
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0 && tmem_free_sh)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TCOLS)
                     : "memory");
}

// out[i][j] = w * sum over chunks of the chunk partials (na x nb, row-major).
// CTA = 32 entries x 8 threads, each summing an eighth of the chunks in order,
// then the eighths in order (one thread per entry waited for 152 dependent
// loads: 42 us at na = 128; see k_gram_reduce)
__global__ void __launch_bounds__(256) k_oz_gram_reduce(int na, int nb, int ctiles, int chunks,
                                                        const double *partials, double w, double *out) {
    __shared__ double red[8][33];
    const int e = blockIdx.x * 32 + threadIdx.x, g = threadIdx.y;
    const int i = e / nb, j = e % nb, ct = j / OZ_NT, jl = j % OZ_NT;
    const bool ok = e < na * nb;
    const int per = (chunks + 7) / 8, c0 = min(chunks, g * per), c1 = min(chunks, c0 + per);
    const size_t stride = (size_t)ctiles * OZ_M * OZ_NT;
    red[g][threadIdx.x] =
        ok ? ordered_sum(partials + ((size_t)ct * OZ_M + i) * OZ_NT + jl + c0 * stride, c1 - c0, stride) : 0.0;
    __syncthreads();
    if (g != 0 || !ok) return;
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < 8; k++) s += red[k][threadIdx.x];
    out[e] = w * s;
}

}  // namespace

bool tall_oz_supported(int k1, int k2) { return k1 + k2 >= 1 && k1 + k2 <= 128; }

size_t tall_oz_image_bytes(long n, int K, int ncol) {
    const int kchunks = (K + OZ_KC - 1) / OZ_KC;
    const int ctiles = (ncol + OZ_NT - 1) / OZ_NT;
    return (size_t)ctiles * kchunks * OZ_S * OZ_BPLANE + sizeof(int) * (size_t)(ncol + 64 + n);
}

int tall_oz_partials(long n, int ncol) {
    return (int)(((n + OZ_M - 1) / OZ_M) * ((ncol + OZ_NT - 1) / OZ_NT));
}

void oz_prepare() {
    static bool done = false;
    if (done) return;
    cudaFuncSetAttribute(k_tall_oz, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_SMEM);
    cudaFuncSetAttribute(k_gram_oz<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_GSMEM);
    cudaFuncSetAttribute(k_gram_oz<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_GSMEM);
    done = true;
}

bool gram_oz_supported(int na) { return na >= 1 && na <= OZ_M; }

namespace {
struct OzGramPlan {
    int ctiles, chunks;
    long chunk_rows;
};
// nb output columns
OzGramPlan make_oz_gram_plan(long n, int nb) {
    OzGramPlan g;
    g.ctiles = (nb + OZ_NT - 1) / OZ_NT;
    // one CTA per SM; at most 16384 points per chunk: the 64-bit fixed-point
    // sums then stay below 2^60 (2^53 per 128-point flush)
    long chunks = std::max((long)152 / g.ctiles, (n + 16383) / 16384);
    chunks = std::max(1L, std::min(chunks, (n + OZ_KC - 1) / OZ_KC));
    long rows = (n + chunks - 1) / chunks;
    rows = (rows + OZ_KC - 1) / OZ_KC * OZ_KC;
    g.chunk_rows = rows;
    g.chunks = (int)((n + rows - 1) / rows);
    return g;
}
size_t oz_gram_tiles(long n, int nb) {
    const OzGramPlan g = make_oz_gram_plan(n, nb);
    return (size_t)g.chunks * g.ctiles;
}
int *oz_exponents(double *scratch, long n, int na) {
    return reinterpret_cast<int *>(scratch + std::max(oz_gram_tiles(n, na), oz_gram_tiles(n, OZ_NT)) * OZ_M * OZ_NT);
}
void oz_colexp(long n, const double *X1, int n1, const double *X2, int n2, int *colexp, cudaStream_t s) {
    cudaMemsetAsync(colexp, 0, sizeof(int) * OZ_M, s);
    HQ_LAUNCH(HQ_K_GRAM, k_oz_colexp<<<1024, 256, 0, s>>>(n, n1, n2, X1, X2, colexp));
}
}  // namespace

// the exponents of the rows and of a separate block's columns follow the partials
// of na or OZ_NT output columns, whichever are more
size_t gram_oz_scratch_bytes(long n, int na) {
    return sizeof(double) * std::max(oz_gram_tiles(n, na), oz_gram_tiles(n, OZ_NT)) * OZ_M * OZ_NT +
           sizeof(int) * 2 * OZ_M;
}

void launch_gram_oz(long n, const double *X1, int n1, const double *X2, int n2, double w,
                    double *scratch, double *out, int *status, cudaStream_t s) {
    if (!X2) n2 = 0;
    const int na = n1 + n2;
    const OzGramPlan g = make_oz_gram_plan(n, na);
    int *colexp = oz_exponents(scratch, n, na);
    oz_colexp(n, X1, n1, X2, n2, colexp, s);
    HQ_LAUNCH(HQ_K_GRAM, k_gram_oz<false><<<dim3(g.ctiles, g.chunks), OZ_GTHREADS, OZ_GSMEM, s>>>(
                             n, n1, n2, 0, g.chunk_rows, X1, X2, nullptr, colexp, nullptr, scratch, status));
    HQ_LAUNCH(HQ_K_GRAM, k_oz_gram_reduce<<<(na * na + 31) / 32, dim3(32, 8), 0, s>>>(na, na, g.ctiles, g.chunks,
                                                                                      scratch, w, out));
}

void launch_gram_oz_xy(long n, const double *X1, int n1, const double *X2, int n2, const double *Y, int ny,
                       int na_scratch, bool have_xexp, double w, double *scratch, double *out, int *status,
                       cudaStream_t s) {
    if (!X2) n2 = 0;
    const int na = n1 + n2;
    const OzGramPlan g = make_oz_gram_plan(n, ny);
    int *xexp = oz_exponents(scratch, n, na_scratch), *yexp = xexp + OZ_M;
    if (!have_xexp) oz_colexp(n, X1, n1, X2, n2, xexp, s);
    oz_colexp(n, Y, ny, nullptr, 0, yexp, s);
    HQ_LAUNCH(HQ_K_GRAM, k_gram_oz<true><<<dim3(g.ctiles, g.chunks), OZ_GTHREADS, OZ_GSMEM, s>>>(
                             n, n1, n2, ny, g.chunk_rows, X1, X2, Y, xexp, yexp, scratch, status));
    HQ_LAUNCH(HQ_K_GRAM, k_oz_gram_reduce<<<(na * ny + 31) / 32, dim3(32, 8), 0, s>>>(na, ny, g.ctiles, g.chunks,
                                                                                      scratch, w, out));
}

void launch_tall_oz(long n, const double *A1, int k1, const double *M1, const double *A2, int k2,
                    const double *M2, int ncol, const double *Cin, double *Out, double *part_sq,
                    unsigned char *image, int *status, cudaStream_t s) {
    if (!A2) k2 = 0;
    const int K = k1 + k2;
    const int kchunks = (K + OZ_KC - 1) / OZ_KC;
    const int ctiles = (ncol + OZ_NT - 1) / OZ_NT;
    int *fexp = reinterpret_cast<int *>(image + (size_t)ctiles * kchunks * OZ_S * OZ_BPLANE);
    int *erow = fexp + ncol + 64;
    HQ_LAUNCH(HQ_K_BLOCKGEMM, k_oz_split<<<ctiles, OZ_NT * SPL_G, 0, s>>>(K, k1, ncol, kchunks, M1,
                                                                   k2 ? M2 : nullptr, image, fexp));
    // one K chunk: the product kernel forms the row exponents from the values
    // it converts; more: a pass over the rows first
    if (kchunks > 1)
        HQ_LAUNCH(HQ_K_BLOCKGEMM, k_oz_rowexp<<<(unsigned)((n + 7) / 8), 256, 0, s>>>(
                                      n, k1, k2, A1, k2 ? A2 : nullptr, erow));
    const unsigned gx = (unsigned)((n + OZ_M - 1) / OZ_M);
    HQ_LAUNCH(HQ_K_BLOCKGEMM,
              k_tall_oz<<<(unsigned)std::min(152L, (long)gx * ctiles), OZ_THREADS, OZ_SMEM, s>>>(
                  n, k1, k2, ncol, kchunks, ctiles, A1, k2 ? A2 : nullptr, image, fexp,
                  kchunks > 1 ? erow : nullptr, Cin, Out,
                  part_sq, status));
}

}  // namespace hq
