// The block PCG of a small FP64 problem with the FP32 preconditioner in one launch.
//
// One CTA carries one column (the columns' recurrences are independent) through the
// whole solve: the direction in shared memory, r and q in registers, and the FP32
// V-cycle on levels that lie in shared memory with a zero halo around each iterate,
// loaded once per solve.  Every operation repeats the expression of its separate
// kernel (k_grid.cu, k_rows.cu, k_vcoarse.cu), so the solve is theirs bit for bit.
#include "column_common.cuh"
#include "grid_common.cuh"
#include "hq_internal.cuh"

#include <algorithm>

namespace hq {

namespace {

constexpr int VT4 = 4;   // restriction taps in use: mc = mf / 2 gives at most four
constexpr int PS_MAX_SMEM = 226 * 1024;

// offset of point (i, j, k) in an iterate with its zero halo
__device__ __forceinline__ int padded(int m, int i, int j, int k) {
    return (i + 1) + (m + 2) * ((j + 1) + (m + 2) * (k + 1));
}

// A thread's points on an m^3 level: the z-column segment (i, j, k0 .. k1 - 1).
// The iterates are stored with a zero halo, (m + 2)^3, so that a stencil reads its
// neighbours unmasked and carries those below and above in registers; r, D, wD
// and the transfer temporary have none.  (Points strided over the threads with
// masked neighbours: 49,000 clocks per V-cycle of a 16^3 column with the tables
// in place, against 43,000.)
struct Seg {
    int k0, k1;      // k0 >= k1: no points
    int m, i, j;
    int p, q;        // offsets of (i, j, k0) in an unpadded and a padded vector
    __device__ __forceinline__ explicit Seg(int m_) : m(m_) {
        const int mm = m * m, nseg = max(1, fdiv(VC_THREADS, mm)), len = fdiv(m + nseg - 1, nseg);
        const int t = threadIdx.x, sg = fdiv(t, mm), c = t - sg * mm;
        j = fdiv(c, m);
        i = c - j * m;
        k0 = sg * len;
        k1 = sg < nseg ? min(m, k0 + len) : 0;
        p = i + m * (j + m * k0);
        q = padded(m, i, j, k0);
    }
};

// zout = (1 - omega) zin + wD (r + c nbrsum(zin)), the sum grouped as nbr_sum
// groups it
__device__ void sm_jacobi(const Seg &g, const float *wD, float c, float omw, const float *r,
                          const float *zin, float *zout) {
    if (g.k0 >= g.k1) return;
    const int mm = g.m * g.m, sy = g.m + 2, sz = sy * sy;
    int p = g.p, q = g.q;
    float below = zin[q - sz], zc = zin[q];
    for (int k = g.k0; k < g.k1; k++, p += mm, q += sz) {
        const float above = zin[q + sz];
        const float s = ((zin[q - 1] + zin[q + 1]) + (zin[q - sy] + zin[q + sy])) + (below + above);
        zout[q] = omw * zc + wD[p] * (r[p] + c * s);
        below = zc;
        zc = above;
    }
}

// y = (b - D x) + c nbrsum(x)
__device__ void sm_resid(const Seg &g, const float *D, float c, const float *x, const float *b,
                         float *y) {
    if (g.k0 >= g.k1) return;
    const int mm = g.m * g.m, sy = g.m + 2, sz = sy * sy;
    int p = g.p, q = g.q;
    float below = x[q - sz], xc = x[q];
    for (int k = g.k0; k < g.k1; k++, p += mm, q += sz) {
        const float above = x[q + sz];
        const float s = ((x[q - 1] + x[q + 1]) + (x[q - sy] + x[q + sy])) + (below + above);
        y[q] = (b[p] - D[p] * xc) + c * s;
        below = xc;
        xc = above;
    }
}

// x pass of the restriction: out[k][j][ic] = sum of the taps over the padded res
__device__ void sm_restrict_x(int m, int mc, const int *ri, const float *rw, const float *res, float *out) {
    const int nout = m * m * mc;
    for (int t = threadIdx.x; t < nout; t += VC_THREADS) {
        const int jk = fdiv(t, mc), ic = t - jk * mc, k = fdiv(jk, m), j = jk - k * m;
        const float *row = res + padded(m, 0, j, k);
        float acc = 0.f;
#pragma unroll
        for (int u = 0; u < VT4; u++) {
            const int ii = ri[ic * XFER_RTAPS + u];
            if (ii >= 0) acc += rw[ic * XFER_RTAPS + u] * row[ii];
        }
        out[t] = acc;
    }
}

// y and z passes: the coarse right-hand side rc = scale sum_z w sum_y w in, and the
// coarse level's first sweep from zero, z = wD rc (padded)
__device__ void sm_restrict_yz(int m, int mc, const int *ri, const float *rw, float scale, const float *in,
                               const float *wD, float *rc, float *z) {
    const int nout = mc * mc * mc;
    for (int t = threadIdx.x; t < nout; t += VC_THREADS) {
        int ic, jc, kc;
        decomp(t, mc, ic, jc, kc);
        float acc = 0.f;
#pragma unroll
        for (int u = 0; u < VT4; u++) {
            const int kk = ri[kc * XFER_RTAPS + u];
            if (kk < 0) continue;
            float v = 0.f;
#pragma unroll
            for (int w = 0; w < VT4; w++) {
                const int jj = ri[jc * XFER_RTAPS + w];
                if (jj >= 0) v += rw[jc * XFER_RTAPS + w] * in[(kk * m + jj) * mc + ic];
            }
            acc += rw[kc * XFER_RTAPS + u] * v;
        }
        const float o = scale * acc;
        rc[t] = o;
        z[padded(mc, ic, jc, kc)] = wD[t] * o;
    }
}

// zout = zin + P ec (padded), the passes nested z, y, x: a thread keeps the four
// coarse columns around its (i, j) at the two coarse planes around k
__device__ void sm_prolong(const Seg &g, int mc, const int *pi, const float *pw, const float *ec,
                           const float *zin, float *zout) {
    if (g.k0 >= g.k1) return;
    const int m = g.m, sz = (m + 2) * (m + 2), cy = mc + 2, cz = cy * cy;
    const int x0 = pi[2 * g.i], x1 = pi[2 * g.i + 1], y0 = pi[2 * g.j], y1 = pi[2 * g.j + 1];
    const float wx0 = pw[2 * g.i], wx1 = pw[2 * g.i + 1], wy0 = pw[2 * g.j], wy1 = pw[2 * g.j + 1];
    // columns (x, y): 00, 10, 01, 11; an absent tap (-1) reads the halo and is skipped
    const int o0 = (x0 + 1) + cy * (y0 + 1), o1 = (x1 + 1) + cy * (y0 + 1);
    const int o2 = (x0 + 1) + cy * (y1 + 1), o3 = (x1 + 1) + cy * (y1 + 1);
    int q = g.q, at = -2;   // lo, hi: coarse planes at, at + 1 (plane -1: the halo)
    float lo[4] = {0.f, 0.f, 0.f, 0.f}, hi[4] = {0.f, 0.f, 0.f, 0.f};
    for (int k = g.k0; k < g.k1; k++, q += sz) {
        const int z0 = pi[2 * k], z1 = pi[2 * k + 1];
        const float wz0 = pw[2 * k], wz1 = pw[2 * k + 1];
        const int want = z0 >= 0 ? z0 : z1 - 1;   // coarse plane at or below k
        if (want != at) {
            const float *a = ec + cz * (want + 1), *b = a + cz;   // want + 2 <= mc + 1
            lo[0] = a[o0];
            lo[1] = a[o1];
            lo[2] = a[o2];
            lo[3] = a[o3];
            hi[0] = b[o0];
            hi[1] = b[o1];
            hi[2] = b[o2];
            hi[3] = b[o3];
            at = want;
        }
        float t[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            t[u] = 0.f;
            if (z0 >= 0) t[u] += wz0 * lo[u];
            if (z1 >= 0) t[u] += wz1 * hi[u];
        }
        float u0 = 0.f, u1 = 0.f;
        if (y0 >= 0) {
            u0 += wy0 * t[0];
            u1 += wy0 * t[1];
        }
        if (y1 >= 0) {
            u0 += wy1 * t[2];
            u1 += wy1 * t[3];
        }
        float acc = zin[q];
        if (x0 >= 0) acc += wx0 * u0;
        if (x1 >= 0) acc += wx1 * u1;
        zout[q] = acc;
    }
}

// z = Ainv r on the coarsest level: per point, eight FP64 partial sums over
// the terms qq = y, y + 8, ... (y = 0..7; one thread each), added in y order
// (the grouping of k_coarse_solve), rounded to FP32 into the padded z; part:
// 8 nc doubles
__device__ void sm_coarse(int m, int nc, const double *__restrict__ Ainv, const float *r, float *z,
                          double *part) {
    for (int t = threadIdx.x; t < 8 * nc; t += VC_THREADS) {
        const int p = t >> 3, y = t & 7;
        // nc <= 64: at most eight terms, their loads issued together
        double a[8], rv[8];
#pragma unroll
        for (int u = 0; u < 8; u++) {
            const int qq = y + 8 * u;
            a[u] = qq < nc ? __ldg(Ainv + (size_t)p * nc + qq) : 0.0;
            rv[u] = qq < nc ? widen(r[qq]) : 0.0;
        }
        double acc = 0.0;
#pragma unroll
        for (int u = 0; u < 8; u++)
            if (y + 8 * u < nc) acc += a[u] * rv[u];
        part[t] = acc;
    }
    __syncthreads();
    for (int p = threadIdx.x; p < nc; p += VC_THREADS) {
        double s = 0.0;
        for (int y = 0; y < 8; y++) s += part[p * 8 + y];
        int i, j, k;
        decomp(p, m, i, j, k);
        z[padded(m, i, j, k)] = (float)s;
    }
}

// shared-memory layout of one column (floats unless stated): per level l the
// two iterates a, b (2 (m_l + 2)^3, zero halo), then r, D, wD (3 n_l), then the
// x-restricted residual (m0^2 m1), per level pair the restriction taps (ridx:
// 6 m_{l+1} ints, rw: 6 m_{l+1}) and prolongation taps (pidx: 2 m_l ints, pw:
// 2 m_l), padding to 8 bytes, and 8 nc doubles of coarse-solve partials.
// Offsets are computed where they are used, so that every pointer is visibly
// derived from the shared array.
__host__ __device__ inline int vc_n(const VCoarse &v, int l) { return v.m[l] * v.m[l] * v.m[l]; }
__host__ __device__ inline int vc_np(const VCoarse &v, int l) {
    return (v.m[l] + 2) * (v.m[l] + 2) * (v.m[l] + 2);
}
__host__ __device__ inline int vc_lev(const VCoarse &v, int l) {   // a of level l; b, r, D, wD follow
    int s = 0;
    for (int i = 0; i < l; i++) s += 2 * vc_np(v, i) + 3 * vc_n(v, i);
    return s;
}
__host__ __device__ inline int vc_taps(const VCoarse &v, int l) {   // taps of level pair l -> l + 1
    int s = vc_lev(v, v.levels) + (v.levels > 1 ? v.m[0] * v.m[0] * v.m[1] : 0);
    for (int i = 0; i < l; i++) s += 2 * XFER_RTAPS * v.m[i + 1] + 4 * v.m[i];
    return s;
}
__host__ __device__ inline size_t vc_floats(const VCoarse &v) {
    return ((size_t)vc_taps(v, v.levels - 1) + 1) & ~(size_t)1;
}

// zero halos and the level tables: D and omega / D of every level, the transfer
// taps
__device__ void vc_load_tables(const VCoarse &v, float *vsm) {
    const int Lf = v.levels;
    int *const vsi = reinterpret_cast<int *>(vsm);
    for (int l = 0; l < Lf; l++) {
        const int n = vc_n(v, l), np = vc_np(v, l);
        float *a = vsm + vc_lev(v, l), *d = a + 2 * np + n, *w = d + n;
        // four points per thread in flight: loads first, then the stores
        for (int p0 = threadIdx.x; p0 < n; p0 += 4 * VC_THREADS) {
            float dv[4], wv[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int p = p0 + u * VC_THREADS;
                dv[u] = p < n ? __ldg(v.D[l] + p) : 0.f;
                wv[u] = p < n ? __ldg(v.wD[l] + p) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int p = p0 + u * VC_THREADS;
                if (p < n) {
                    d[p] = dv[u];
                    w[p] = wv[u];
                }
            }
        }
        for (int p = threadIdx.x; p < 2 * np; p += VC_THREADS) a[p] = 0.f;
    }
    for (int l = 0; l + 1 < Lf; l++) {
        const int mf = v.m[l], mc = v.m[l + 1], o = vc_taps(v, l);
        int *ri = vsi + o;
        float *rw = vsm + o + XFER_RTAPS * mc;
        int *pi = vsi + o + 2 * XFER_RTAPS * mc;
        float *pw = vsm + o + 2 * XFER_RTAPS * mc + 2 * mf;
        for (int t = threadIdx.x; t < XFER_RTAPS * mc; t += VC_THREADS) {
            ri[t] = __ldg(v.ridx[l] + t);
            rw[t] = __ldg(v.rw[l] + t);
        }
        for (int t = threadIdx.x; t < 2 * mf; t += VC_THREADS) {
            pi[t] = __ldg(v.pidx[l] + t);
            pw[t] = __ldg(v.pw[l] + t);
        }
    }
}

// one V-cycle: the right-hand side r of level l0 and its first sweep a = wD r are
// in shared memory (complete behind a barrier, as the tables are); returns the
// iterate, with its halo (complete behind a barrier)
__device__ float *vc_cycle(const VCoarse &v, float *vsm, double *cpart) {
    const int Lf = v.levels;   // levels: l0 .. l0 + Lf - 1 (last = coarsest)
    int *const vsi = reinterpret_cast<int *>(vsm);
    float *const tmp = vsm + vc_lev(v, Lf);
    // down: the remaining pre-smoothing sweeps, residual, restriction.  in_b:
    // bit l set when level l's pre-smoothed iterate ended in b (else in a)
    unsigned in_b = 0;
    for (int l = 0; l + 1 < Lf; l++) {
        const int m = v.m[l], mc = v.m[l + 1], n = vc_n(v, l), np = vc_np(v, l), ot = vc_taps(v, l);
        float *c0 = vsm + vc_lev(v, l), *o0 = c0 + np;
        const float *r = o0 + np, *D = r + n, *wD = D + n;
        const Seg g(m);
        bool cb = false;
        for (int s = 1; s < v.nu1; s++) {
            sm_jacobi(g, wD, v.c[l], v.omw, r, c0, o0);
            __syncthreads();
            float *t = c0;
            c0 = o0;
            o0 = t;
            cb = !cb;
        }
        sm_resid(g, D, v.c[l], c0, r, o0);
        __syncthreads();
        const int *ri = vsi + ot;
        const float *rw = vsm + ot + XFER_RTAPS * mc;
        sm_restrict_x(m, mc, ri, rw, o0, tmp);
        __syncthreads();
        float *ca = vsm + vc_lev(v, l + 1), *cr = ca + 2 * vc_np(v, l + 1);
        sm_restrict_yz(m, mc, ri, rw, v.rscale[l], tmp, cr + 2 * vc_n(v, l + 1), cr, ca);
        __syncthreads();
        if (cb) in_b |= 1u << l;
    }
    // coarsest solve into b (a holds the unused first sweep)
    float *zc;
    {
        const int np = vc_np(v, Lf - 1);
        zc = vsm + vc_lev(v, Lf - 1) + np;
        sm_coarse(v.m[Lf - 1], v.nc, v.Ainv, zc + np, zc, cpart);
    }
    __syncthreads();
    // up: prolongation added to the pre-smoothed iterate, post-smoothing; zc:
    // the finished correction of the level below
    for (int l = Lf - 2; l >= 0; l--) {
        const int m = v.m[l], mc = v.m[l + 1], n = vc_n(v, l), np = vc_np(v, l), ot = vc_taps(v, l);
        float *a = vsm + vc_lev(v, l), *b = a + np;
        const float *r = b + np, *wD = r + 2 * n;
        float *c0 = ((in_b >> l) & 1u) ? b : a;
        float *o0 = ((in_b >> l) & 1u) ? a : b;
        const int *pi = vsi + ot + 2 * XFER_RTAPS * mc;
        const float *pw = vsm + ot + 2 * XFER_RTAPS * mc + 2 * m;
        const Seg g(m);
        sm_prolong(g, mc, pi, pw, zc, c0, o0);
        __syncthreads();
        {
            float *t = c0;
            c0 = o0;
            o0 = t;
        }
        for (int s = 0; s < v.nu2; s++) {
            sm_jacobi(g, wD, v.c[l], v.omw, r, c0, o0);
            __syncthreads();
            float *t = c0;
            c0 = o0;
            o0 = t;
        }
        zc = c0;
    }
    return zc;
}

// ---------------------------------------------------------------------------
// The whole block PCG of a small FP64 problem with the FP32 preconditioner, one
// CTA per column (the columns' recurrences are independent): r, q and the
// direction never leave the SM, the V-cycle's tables are loaded once per solve,
// and an iteration is one pass of barriers instead of seven launches.  Where the
// whole V-cycle fits one CTA (about 17^3 points) those launches were bound by
// their latencies: 75 us per iteration at 16^3, 8 columns; 56 us here, of which the
// V-cycle takes 21.  One thread forms alpha, beta and the norms: the divisions and
// roots of all 1024 threads cost 7 us per iteration.
//
// Same recurrence, roundings and orders as pcg_half / pcg_body with the kernels
// of the geometry g64 (launch_apply, k_pcg_xr, k_vcoarse<true>, k_pcg_p and
// k_finalize's sums), so the solve is theirs bit for bit.
// ---------------------------------------------------------------------------
constexpr int PS_U = 5;   // points per thread: n <= 5 x 1024 (17^3)

// sum over the column of a(p) b(p) (b: shared; a: any accessor of FP64 values) in
// the order of block_col_reduce and k_finalize: chains of ppt points per (row,
// thread row), thread rows in groups, then rows in chunks of 128 by eight
// warps.  chain: gy TY doubles (may be b: every product is formed before the
// first store); rows: gy; st: 8 R.  Thread 0 calls finish(sum), behind whose
// stores all threads return (divisions and square roots of all 1024 threads
// would each hold the FP64 pipe for thousands of clocks).
template <typename A, typename F>
__device__ __forceinline__ void ps_dot(int n, int TY, int ppt, int gy, A a, const double *b, double *chain,
                                       double *rows, double *st, F finish) {
    const int tid = threadIdx.x, nt = gy * TY;
    double acc[PS_U];
#pragma unroll
    for (int u = 0; u < PS_U; u++) {
        const int t = tid + u * VC_THREADS;
        acc[u] = 0.0;
        if (t >= nt) continue;
        const int row = fdiv(t, TY), y = t - row * TY;
        for (int k = 0; k < ppt; k++) {
            const int p = (row * ppt + k) * TY + y;
            if (p < n) acc[u] = fma(a(p), b[p], acc[u]);
        }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < PS_U; u++)
        if (tid + u * VC_THREADS < nt) chain[tid + u * VC_THREADS] = acc[u];
    __syncthreads();
    // thread rows: (row, group) partials, then the groups of a row in order
    const int G = row_groups(TY), gr = (TY + G - 1) / G;
#pragma unroll
    for (int u = 0; u < PS_U; u++) {
        const int t = tid + u * VC_THREADS;
        if (u > 0 && u * VC_THREADS >= gy * G) break;   // uniform
        acc[u] = 0.0;
        if (t >= gy * G) continue;
        const int row = fdiv(t, G), g = t - row * G;
        for (int y = g * gr; y < min(TY, (g + 1) * gr); y++) acc[u] += chain[row * TY + y];
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < PS_U; u++)
        if (tid + u * VC_THREADS < gy * G) chain[tid + u * VC_THREADS] = acc[u];
    __syncthreads();
    for (int row = tid; row < gy; row += VC_THREADS) {
        double s = 0.0;
        for (int g = 0; g < G; g++) s += chain[row * G + g];
        rows[row] = s;
    }
    __syncthreads();
    // k_finalize: chunks of 128 rows, warp w of a chunk takes rows w, w + 8, ...
    const int R = (gy + 127) / 128;
    if (tid < 8 * R) {
        const int c = tid >> 3, w = tid & 7, y1 = min(gy, (c + 1) * 128);
        double s = 0.0;
        for (int y = c * 128 + w; y < y1; y += 8) s += rows[y];
        st[tid] = s;
    }
    __syncthreads();
    if (tid == 0) {
        double s = 0.0;
        for (int c = 0; c < R; c++) {
            double t = 0.0;
            for (int w = 0; w < 8; w++) t += st[c * 8 + w];
            s += t;
        }
        finish(s);
    }
    __syncthreads();
}

__global__ void __launch_bounds__(VC_THREADS)
    k_pcg_small(const __grid_constant__ VCoarse v, int N, int TY, int ppt, int gy,
                const double *__restrict__ D64, double c64, const double *__restrict__ B,
                double *__restrict__ X, PcgScalars sc, double rtol, int maxit) {
    extern __shared__ __align__(16) float vsm[];
    const int col = blockIdx.x, tid = threadIdx.x;
    const int m = v.m[0], n = m * m * m;
    double *const cpart = reinterpret_cast<double *>(vsm + vc_floats(v));
    double *const pv = cpart + 8 * v.nc;   // the direction (first: x), n
    double *const w = pv + n;              // operand of the dot products, then chains
    double *const rows = w + max(n, gy * TY), *const st = rows + gy;
    float *const a32 = vsm, *const r32 = a32 + 2 * vc_np(v, 0), *const wD32 = r32 + 2 * n;
    __shared__ double rz, bn, rn, step;   // r . z, |b|, |r|, beta or alpha (thread 0)
    __shared__ int go;                    // the column is active
    vc_load_tables(v, vsm);
    double r[PS_U], q[PS_U];
#pragma unroll
    for (int u = 0; u < PS_U; u++) {
        const int p = tid + u * VC_THREADS;
        r[u] = q[u] = 0.0;
        if (p < n) pv[p] = X[(size_t)p * N + col];
    }
    __syncthreads();
    // neighbour sum of pv at p
    auto nbr = [&](int p) {
        int i, j, k;
        decomp(p, m, i, j, k);
        const bool in[6] = {i > 0, i < m - 1, j > 0, j < m - 1, k > 0, k < m - 1};
        const int mm = m * m;
        const double a[6] = {pv[in[0] ? p - 1 : p], pv[in[1] ? p + 1 : p], pv[in[2] ? p - m : p],
                             pv[in[3] ? p + m : p], pv[in[4] ? p - mm : p], pv[in[5] ? p + mm : p]};
        return sum6(a, in);
    };
    auto at_w = [&](int p) { return w[p]; };
    auto at_p = [&](int p) { return pv[p]; };
    // r = b - A x, |b|, |r|
#pragma unroll
    for (int u = 0; u < PS_U; u++) {
        const int p = tid + u * VC_THREADS;
        if (p >= n) continue;
        q[u] = B[(size_t)p * N + col];
        r[u] = resid_value(q[u], D64[p], pv[p], c64, nbr(p));
        w[p] = q[u];
    }
    __syncthreads();
    ps_dot(n, TY, ppt, gy, at_w, w, w, rows, st, [&](double s) { bn = sqrt(s); });
#pragma unroll
    for (int u = 0; u < PS_U; u++)
        if (tid + u * VC_THREADS < n) w[tid + u * VC_THREADS] = r[u];
    __syncthreads();
    ps_dot(n, TY, ppt, gy, at_w, w, w, rows, st, [&](double s) {
        rn = sqrt(s);
        go = rn > rtol * bn;
        if (!isfinite(rn) || !isfinite(bn)) atomicOr(sc.status, ST_NONFINITE);
    });
    int its = 0;
    while (go && its < maxit) {
        // z = M r; r . z; p = z + beta p
#pragma unroll
        for (int u = 0; u < PS_U; u++) {
            const int p = tid + u * VC_THREADS;
            if (p >= n) continue;
            int i, j, k;
            decomp(p, m, i, j, k);
            const float rf = (float)r[u];
            r32[p] = rf;
            a32[padded(m, i, j, k)] = wD32[p] * rf;
            w[p] = r[u];
        }
        __syncthreads();
        const float *zc = vc_cycle(v, vsm, cpart);
        auto zat = [&](int p) {
            int i, j, k;
            decomp(p, m, i, j, k);
            return widen(zc[padded(m, i, j, k)]);
        };
        ps_dot(n, TY, ppt, gy, zat, w, w, rows, st, [&](double s) {
            step = its > 0 ? s / rz : 0.0;
            rz = s;
        });
        const double beta = step;
#pragma unroll
        for (int u = 0; u < PS_U; u++) {
            const int p = tid + u * VC_THREADS;
            if (p < n) pv[p] = its > 0 ? fma(beta, pv[p], zat(p)) : zat(p);
        }
        __syncthreads();
        // q = A p; alpha = rz / p . q
#pragma unroll
        for (int u = 0; u < PS_U; u++) {
            const int p = tid + u * VC_THREADS;
            if (p >= n) continue;
            q[u] = op_value(D64[p], pv[p], c64, nbr(p));
            w[p] = q[u];
        }
        __syncthreads();
        ps_dot(n, TY, ppt, gy, at_p, w, w, rows, st, [&](double s) {
            if (!(s > 0.0) || !isfinite(s)) {
                atomicOr(sc.status, ST_BREAKDOWN);
                go = -1;
            } else {
                step = rz / s;
            }
        });
        if (go < 0) break;
        const double alpha = step;
        // x += alpha p, r -= alpha q, |r|
#pragma unroll
        for (int u = 0; u < PS_U; u++) {
            const int p = tid + u * VC_THREADS;
            if (p >= n) continue;
            double *x = X + (size_t)p * N + col;
            *x = fma(alpha, pv[p], *x);
            r[u] = fma(-alpha, q[u], r[u]);
            w[p] = r[u];
        }
        __syncthreads();
        its++;
        ps_dot(n, TY, ppt, gy, at_w, w, w, rows, st, [&](double s) {
            rn = sqrt(s);
            if (!isfinite(rn)) atomicOr(sc.status, ST_NONFINITE);
            if (rn <= rtol * bn || !isfinite(rn)) go = 0;
        });
    }
    if (tid == 0) {
        sc.bnorm[col] = bn;
        sc.rnorm[col] = rn;
        sc.iters[col] = its;
        sc.active[col] = go;
    }
}

// after k_pcg_small: num_active[0] = columns still active, num_active[1] =
// iterations of the slowest column (with the one a column broke down in: active
// < 0, cleared here); counters (nullable) += those iterations;
// ST_PCG_MAXIT for columns that reached the cap (check)
__global__ void __launch_bounds__(256) k_pcg_small_end(int N, PcgScalars sc, long long *counters, int check) {
    __shared__ int act_sh[8], it_sh[8];
    int act = 0, it = 0;
    for (int c = threadIdx.x; c < N; c += 256) {
        const int a = sc.active[c];
        act += a > 0;
        it = max(it, sc.iters[c] + (a < 0));
        if (a < 0) sc.active[c] = 0;
    }
    act = __reduce_add_sync(0xffffffffu, act);
    it = __reduce_max_sync(0xffffffffu, it);
    if ((threadIdx.x & 31) == 0) {
        act_sh[threadIdx.x >> 5] = act;
        it_sh[threadIdx.x >> 5] = it;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int w = 1; w < 8; w++) {
        act += act_sh[w];
        it = max(it, it_sh[w]);
    }
    sc.num_active[0] = act;
    sc.num_active[1] = it;
    if (counters) counters[0] += it;
    if (act > 0 && check) atomicOr(sc.status, ST_PCG_MAXIT);
}

size_t ps_smem_bytes(const VCoarse &v, const GridGeom &g) {
    const size_t n = (size_t)v.m[0] * v.m[0] * v.m[0], R = (g.gy + 127) / 128;
    const size_t chains = std::max(n, (size_t)g.gy * g.ty);
    return vc_floats(v) * sizeof(float) + sizeof(double) * (8 * (size_t)v.nc + n + chains + g.gy + 8 * R);
}

}  // namespace

// One CTA per column and SM: a second wave of columns still beats the separate
// kernels up to 16^3 (to rounding there), a third nowhere.  15 iterations, one launch
// against separate kernels: 160 columns 8^3 870, 994 us, 13^3 1474, 1514, 16^3 1920, 1915, 17^3
// 2205, 2055; 320 columns 8^3 1280, 1108, 13^3 2186, 1916, 16^3 2636, 2441.
bool pcg_small_fits(const VCoarse &v, const GridGeom &g) {
    const long n = (long)v.m[0] * v.m[0] * v.m[0];
    if (g.N > (n <= 4096 ? 2 : 1) * 152) return false;
    return v.levels >= 2 && n <= (long)PS_U * VC_THREADS && (long)g.gy * g.ty <= (long)PS_U * VC_THREADS &&
           (g.gy + 127) / 128 <= VC_THREADS / 8 && ps_smem_bytes(v, g) <= (size_t)PS_MAX_SMEM;
}

void launch_pcg_small(const VCoarse &v, const GridGeom &g, const double *D64, double c64, const double *B,
                      double *X, const PcgScalars &sc, double rtol, int maxit, long long *counters,
                      int check_maxit, cudaStream_t s) {
    HQ_LAUNCH_W(HQ_K_COARSE, (double)g.n * g.N,
                k_pcg_small<<<g.N, VC_THREADS, ps_smem_bytes(v, g), s>>>(v, g.N, g.ty, g.ppt, g.gy, D64, c64,
                                                                        B, X, sc, rtol, maxit));
    HQ_LAUNCH(HQ_K_REDUCE, k_pcg_small_end<<<1, 256, 0, s>>>(g.N, sc, counters, check_maxit));
}

void pcg_small_prepare() {
    cudaFuncSetAttribute(k_pcg_small, cudaFuncAttributeMaxDynamicSharedMemorySize, PS_MAX_SMEM);
}

}  // namespace hq
