// Grid passes fused along whole x-rows.
//
// The multigrid passes of a level that does not fit one CTA are bound by
// memory traffic (FP32) or launches, and passes that look only along x, or at
// the point itself, need no halo when a CTA owns whole x-rows: a row of
// m points x up to 64 FP32 (32 FP64) columns lies in shared memory between
// the two passes.
//
//   residual + x-restriction   reads z, r, writes half a block (was: a block
//                              written, read again, half a block written)
//   first + second sweep       reads r, writes z (was: z1 written and read)
//   y- and z-restriction       one pass over the half block
//   prolongation               one pass: z and y interpolated in registers,
//                              x from the shared row, added to the iterate
//
// Measured (GB300; before, as separate kernels): FP32 V-cycle at 64^3, 64 columns
// 389 -> 299 us, 128^3, 256 columns 9.49 -> 7.04 ms (there: residual and
// x-restriction 1.95 -> 1.28 ms for 2.5 words, 0.62 of the copy bandwidth; first two
// sweeps 1.56 -> 1.09 ms; y/z-restriction and prolongation 1.75 -> 1.18 ms);
// FP64 at 64^3, 64 columns 1.64 -> 1.06 ms (with the integer neighbour sums).
//
// Every value is formed by the expression of the separate kernels (k_grid.cu)
// in the same order, so the results are theirs bit for bit.
//
// Tried and slower: two stencil passes per kernel on 20 x 16 point tiles with
// a halo of two (r to the second sweep and the residual; prolongation and two
// sweeps).  They move 60% of the words, but the halo (1.7 times the points)
// and the in-plane exchange hold the L1 data pipe for twice the DRAM time.
#include "grid_common.cuh"
#include "hq_internal.cuh"

#include <algorithm>
#include <type_traits>

namespace hq {

namespace {

constexpr int ROW_THREADS = 512;
constexpr int ROW_MAXQ = 2;   // points of a row per thread
constexpr int RT = 4;         // restriction taps in use: mc = mf / 2 gives at most four
constexpr size_t ROW_MAX_SMEM = 100 * 1024;

enum { ROW_RESID = 0, ROW_SWEEP2 = 1 };

// CTA = one x-row (y = blockIdx.y mod m) x blockDim.x column vectors, marching
// a range of z-planes; a thread owns the points ty + q blockDim.y of the row
// and keeps their z - 1, z, z + 1 values in registers.  y-neighbours are read
// from memory (L2: the neighbouring rows' CTAs march beside this one),
// x-neighbours from the row in shared memory.
// ROW_RESID:  out[k][j][ic] = sum of restriction taps over the row of
//             (b - D x) + c nbrsum(x); the taps of plane k - 1 are taken while
//             plane k's residual is formed (two row buffers of each)
// ROW_SWEEP2: out = (1 - omega) z1 + wD (r + c nbrsum(z1)), z1 = wD r
//             (x = r, D = wD, c2 = 1 - omega)
// One barrier per plane; the plane's loads are issued ahead of it.  What
// bounds the kernel is their latency, so the shape is chosen for two CTAs of
// 512 threads and 64 registers per SM: three of 40 registers spilled and took
// 1.4 times as long, one of four points a thread and 126 registers 1.6 times.
template <typename T, int V, int Q, int MODE>
__global__ void __launch_bounds__(ROW_THREADS, Q == 1 ? 2 : 1)
    k_row(int m, int mc, int N, int mz, const T *__restrict__ D, T c, T c2, const T *__restrict__ x,
          const T *__restrict__ b, const int *__restrict__ ridx, const T *__restrict__ rw,
          T *__restrict__ out) {
    using W = VT<T, V>;
    extern __shared__ __align__(16) unsigned char row_smem[];
    const int LX = blockDim.x, TY = blockDim.y, lane = threadIdx.x, ty = threadIdx.y;
    const int RS = m * LX;   // a row buffer
    W *cur = reinterpret_cast<W *>(row_smem), *res = cur + 2 * RS;
    T *tw = reinterpret_cast<T *>(res + 2 * RS);
    int *ti = reinterpret_cast<int *>(tw + RT * mc);
    const int col = (blockIdx.x * LX + lane) * V;
    const bool cv = col < N;
    const int j = blockIdx.y % m, k0 = (blockIdx.y / m) * mz, k1 = min(m, k0 + mz);
    const size_t sy = (size_t)m * N, sz = (size_t)m * m * N;
    const int mm = m * m;
    if (MODE == ROW_RESID)
        for (int t = ty * LX + lane; t < RT * mc; t += LX * TY) {
            const int g = (t / RT) * XFER_RTAPS + t % RT;
            ti[t] = ridx[g];
            tw[t] = rw[g];
        }
    const bool bs = j > 0, bn = j < m - 1;
    W zero;
#pragma unroll
    for (int v = 0; v < V; v++) zero.v[v] = T(0);
    auto scaled = [&](const W &r, T w) {   // z1 = wD r
        W o;
#pragma unroll
        for (int v = 0; v < V; v++) o.v[v] = w * r.v[v];
        return o;
    };
    W xp[Q], xc[Q], rc[Q];
    T wc[Q];
#pragma unroll
    for (int q = 0; q < Q; q++) {
        const int i = ty + TY * q;
        const bool ok = cv && i < m;
        const int p = (k0 * m + j) * m + i;
        const size_t e = (size_t)p * N + col;
        xc[q] = ok ? ldv<T, V>(x + e) : zero;
        xp[q] = ok && k0 > 0 ? ldv<T, V>(x + e - sz) : zero;
        if (MODE == ROW_SWEEP2) {
            rc[q] = xc[q];
            wc[q] = ok ? D[p] : T(0);
            xc[q] = scaled(xc[q], wc[q]);
            xp[q] = scaled(xp[q], ok && k0 > 0 ? D[p - mm] : T(0));
        }
    }
    // the x-taps of the residual row of plane k
    auto taps_x = [&](int k) {
        const W *row = res + (k & 1) * RS;
        if (!cv) return;
        for (int ic = ty; ic < mc; ic += TY) {
            T acc[V];
#pragma unroll
            for (int v = 0; v < V; v++) acc[v] = T(0);
#pragma unroll
            for (int t = 0; t < RT; t++) {
                const int ii = ti[ic * RT + t];
                if (ii < 0) break;   // the valid taps come first
                const T w = tw[ic * RT + t];
                const W a = row[ii * LX + lane];
#pragma unroll
                for (int v = 0; v < V; v++) acc[v] += w * a.v[v];
            }
            W o;
#pragma unroll
            for (int v = 0; v < V; v++) o.v[v] = acc[v];
            stv<T, V>(out + (size_t)((k * m + j) * mc + ic) * N + col, o);
        }
    };
    for (int k = k0; k < k1; k++) {
        // this plane's loads, ahead of the barrier
        W xn[Q], as[Q], an[Q], bb[Q];
        T dn[Q], ds[Q], db[Q];
        const bool top = k + 1 < m;
        W *row = cur + (k & 1) * RS;
#pragma unroll
        for (int q = 0; q < Q; q++) {
            const int i = ty + TY * q;
            if (!(cv && i < m)) continue;
            const int p = (k * m + j) * m + i;
            const size_t e = (size_t)p * N + col;
            row[i * LX + lane] = xc[q];
            xn[q] = top ? ldv<T, V>(x + e + sz) : zero;
            as[q] = ldv<T, V>(x + (bs ? e - sy : e));
            an[q] = ldv<T, V>(x + (bn ? e + sy : e));
            if (MODE == ROW_RESID) {
                bb[q] = ldv<T, V>(b + e);
                dn[q] = D[p];
            } else {
                ds[q] = D[bs ? p - m : p];
                db[q] = D[bn ? p + m : p];
                dn[q] = top ? D[p + mm] : T(0);
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < Q; q++) {
            const int i = ty + TY * q;
            if (!(cv && i < m)) continue;
            const bool in[6] = {i > 0, i < m - 1, bs, bn, true, true};
            const W aw = row[(in[0] ? i - 1 : i) * LX + lane], ae = row[(in[1] ? i + 1 : i) * LX + lane];
            const W up = MODE == ROW_SWEEP2 ? scaled(xn[q], dn[q]) : xn[q];
            if (MODE == ROW_SWEEP2) {
                as[q] = scaled(as[q], ds[q]);
                an[q] = scaled(an[q], db[q]);
            }
            W o;
#pragma unroll
            for (int v = 0; v < V; v++) {
                const T a[6] = {aw.v[v], ae.v[v], as[q].v[v], an[q].v[v], xp[q].v[v], up.v[v]};
                const T s = sum6(a, in);
                if (MODE == ROW_RESID) o.v[v] = (bb[q].v[v] - dn[q] * xc[q].v[v]) + c * s;
                else o.v[v] = c2 * xc[q].v[v] + wc[q] * (rc[q].v[v] + c * s);
            }
            if (MODE == ROW_RESID) res[(k & 1) * RS + i * LX + lane] = o;
            else stv<T, V>(out + (size_t)((k * m + j) * m + i) * N + col, o);
            xp[q] = xc[q];
            xc[q] = up;
            if (MODE == ROW_SWEEP2) {
                rc[q] = xn[q];
                wc[q] = dn[q];
            }
        }
        if (MODE == ROW_RESID && k > k0) taps_x(k - 1);
    }
    if (MODE == ROW_RESID) {
        __syncthreads();
        taps_x(k1 - 1);
    }
}

// y- and z-restriction of an mf x mf x mc block (z, y, x): a thread marches the
// fine planes of its coarse (ic, jc), forms the y-taps of a plane and adds
// them to the two coarse planes around it (each fine plane belongs to at most
// two), so a fine row is read once per coarse row that uses it.
template <typename T, int V>
__global__ void __launch_bounds__(256)
    k_restrict_yz(int mf, int mc, int N, int cz, const int *__restrict__ ridx, const T *__restrict__ rw,
                  const T *__restrict__ pw, T scale, const T *__restrict__ in, T *__restrict__ out) {
    using W = VT<T, V>;
    const int col = (blockIdx.x * blockDim.x + threadIdx.x) * V;
    const int p2 = blockIdx.y * blockDim.y + threadIdx.y;
    if (col >= N || p2 >= mc * mc) return;
    const int ic = p2 % mc, jc = p2 / mc;
    const int c0 = blockIdx.z * cz, c1 = min(mc, c0 + cz);
    int yi[RT];
    T yw[RT];
#pragma unroll
    for (int t = 0; t < RT; t++) {
        yi[t] = ridx[jc * XFER_RTAPS + t];
        yw[t] = rw[jc * XFER_RTAPS + t];
    }
    const int f0 = ridx[c0 * XFER_RTAPS];
    int f1 = f0;   // last fine plane of the chunk's last coarse plane
#pragma unroll
    for (int t = 0; t < RT; t++) f1 = max(f1, ridx[(c1 - 1) * XFER_RTAPS + t]);
    const size_t srow = (size_t)mc * N, spl = (size_t)mf * mc * N;
    const T *src = in + (size_t)ic * N + col + (size_t)f0 * spl;
    T *dst = out + ((size_t)jc * mc + ic) * N + col;
    const size_t sout = (size_t)mc * mc * N;
    W lo, hi;   // sums of the coarse planes cl and cl + 1
#pragma unroll
    for (int v = 0; v < V; v++) lo.v[v] = hi.v[v] = T(0);
    auto emit = [&](int c, const W &a) {
        if (c < c0 || c >= c1) return;
        W o;
#pragma unroll
        for (int v = 0; v < V; v++) o.v[v] = scale * a.v[v];
        stv<T, V>(dst + (size_t)c * sout, o);
    };
    int cl = ((f0 + 1) * (mc + 1)) / (mf + 1) - 1;
    W a[RT], an[RT];
    auto load = [&](const T *p, W (&d)[RT]) {
#pragma unroll
        for (int t = 0; t < RT; t++)
            if (yi[t] >= 0) d[t] = ldv<T, V>(p + (size_t)yi[t] * srow);
    };
    load(src, an);
    for (int f = f0; f <= f1; f++) {
#pragma unroll
        for (int t = 0; t < RT; t++) a[t] = an[t];
        src += spl;
        if (f < f1) load(src, an);   // ahead of this plane's sums
        const T w0 = pw[2 * f], w1 = pw[2 * f + 1];
        T y[V];
#pragma unroll
        for (int v = 0; v < V; v++) y[v] = T(0);
#pragma unroll
        for (int t = 0; t < RT; t++) {
            if (yi[t] < 0) continue;
#pragma unroll
            for (int v = 0; v < V; v++) y[v] += yw[t] * a[t].v[v];
        }
        const int c = ((f + 1) * (mc + 1)) / (mf + 1) - 1;
        if (c > cl) {
            emit(cl, lo);
            lo = hi;
#pragma unroll
            for (int v = 0; v < V; v++) hi.v[v] = T(0);
            cl = c;
        }
        if (w0 != T(0)) {
#pragma unroll
            for (int v = 0; v < V; v++) lo.v[v] += w0 * y[v];
        }
        if (w1 != T(0)) {
#pragma unroll
            for (int v = 0; v < V; v++) hi.v[v] += w1 * y[v];
        }
    }
    emit(cl, lo);
    emit(cl + 1, hi);
}

// Prolongation added to an iterate.  CTA = the x-rows j of a range in one fine
// plane k: the coarse rows around j, interpolated in z, stay in registers
// (a thread owns coarse points ty + q blockDim.y) and move on every second
// fine row; their y-interpolation goes through the shared row to the
// x-interpolation.  One barrier per row (two row buffers).
template <typename T, int V, int Q>
__global__ void __launch_bounds__(ROW_THREADS, Q == 1 ? 2 : 1)
    k_prolong_rows(int mf, int mc, int N, int nj, const int *__restrict__ pidx, const T *__restrict__ pw,
                   const T *__restrict__ ec, const T *efin, T *efout) {
    using W = VT<T, V>;
    extern __shared__ __align__(16) unsigned char row_smem[];
    const int LX = blockDim.x, TY = blockDim.y, lane = threadIdx.x, ty = threadIdx.y;
    W *rows = reinterpret_cast<W *>(row_smem);
    const int col = (blockIdx.x * LX + lane) * V;
    const bool cv = col < N;
    const int k = blockIdx.y % mf, j0 = (blockIdx.y / mf) * nj, j1 = min(mf, j0 + nj);
    const int z0 = pidx[2 * k], z1 = pidx[2 * k + 1];
    const T wz0 = pw[2 * k], wz1 = pw[2 * k + 1];
    const size_t spl = (size_t)mc * mc * N;
    W zero;
#pragma unroll
    for (int v = 0; v < V; v++) zero.v[v] = T(0);
    // row jc of the correction interpolated in z (nothing outside the grid)
    auto zrow = [&](int jc, W (&t)[Q]) {
#pragma unroll
        for (int q = 0; q < Q; q++) {
            const int ic = ty + TY * q;
            t[q] = zero;
            if (!(cv && ic < mc) || jc < 0 || jc >= mc) continue;
            const T *src = ec + ((size_t)jc * mc + ic) * N + col;
            W a, b;
            if (z0 >= 0) a = ldv<T, V>(src + (size_t)z0 * spl);
            if (z1 >= 0) b = ldv<T, V>(src + (size_t)z1 * spl);
#pragma unroll
            for (int v = 0; v < V; v++) {
                if (z0 >= 0) t[q].v[v] += wz0 * a.v[v];
                if (z1 >= 0) t[q].v[v] += wz1 * b.v[v];
            }
        }
    };
    auto lower = [&](int f) { return ((f + 1) * (mc + 1)) / (mf + 1) - 1; };
    W ta[Q], tb[Q];
    int jl = lower(j0);
    zrow(jl, ta);
    zrow(jl + 1, tb);
    for (int j = j0; j < j1; j++) {
        W *row = rows + (size_t)(j & 1) * mc * LX;
        if (lower(j) > jl) {
            jl++;
#pragma unroll
            for (int q = 0; q < Q; q++) ta[q] = tb[q];
            zrow(jl + 1, tb);
        }
        const int y0 = pidx[2 * j], y1 = pidx[2 * j + 1];
        const T wy0 = pw[2 * j], wy1 = pw[2 * j + 1];
#pragma unroll
        for (int q = 0; q < Q; q++) {
            const int ic = ty + TY * q;
            if (!(cv && ic < mc)) continue;
            W t = zero;
#pragma unroll
            for (int v = 0; v < V; v++) {
                if (y0 >= 0) t.v[v] += wy0 * ta[q].v[v];
                if (y1 >= 0) t.v[v] += wy1 * tb[q].v[v];
            }
            row[ic * LX + lane] = t;
        }
        const size_t er = (size_t)(k * mf + j) * mf;
        W e[2 * Q + 1];
#pragma unroll
        for (int q = 0; q < 2 * Q + 1; q++) {
            const int i = ty + TY * q;
            if (cv && i < mf) e[q] = ldv<T, V>(efin + (er + i) * N + col);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 2 * Q + 1; q++) {
            const int i = ty + TY * q;
            if (!(cv && i < mf)) continue;
            const int x0 = pidx[2 * i], x1 = pidx[2 * i + 1];
            const T wx0 = pw[2 * i], wx1 = pw[2 * i + 1];
            W o = e[q];
            if (x0 >= 0) {
                const W a = row[x0 * LX + lane];
#pragma unroll
                for (int v = 0; v < V; v++) o.v[v] += wx0 * a.v[v];
            }
            if (x1 >= 0) {
                const W a = row[x1 * LX + lane];
#pragma unroll
                for (int v = 0; v < V; v++) o.v[v] += wx1 * a.v[v];
            }
            stv<T, V>(efout + (er + i) * N + col, o);
        }
    }
}

// launch shape of the row kernels: lx column vectors x ty row points, one point
// per thread while 512 threads hold the row (16 vectors up to 32 points, 8 up
// to 64, 4 up to 128), then q of them
struct RowShape {
    int vec, lx, ty, gx, q;
};
template <typename T>
RowShape row_shape(int len, int N) {
    RowShape s;
    s.vec = sizeof(T) == 8 ? (N % 2 == 0 ? 2 : 1) : (N % 4 == 0 ? 4 : (N % 2 == 0 ? 2 : 1));
    const int vecs = N / s.vec, most = len <= 32 ? 16 : (len <= 64 ? 8 : 4);
    s.gx = (vecs + most - 1) / most;
    s.lx = (vecs + s.gx - 1) / s.gx;
    s.ty = std::min(ROW_THREADS / s.lx, len);
    s.q = (len + s.ty - 1) / s.ty;
    return s;
}
// steps per CTA of a march of `len` steps: about 16 CTAs per SM (2 to 16 per SM
// measured: 64^3, 64 columns 320, 301, 294, 299 us per V-cycle, 96^3 925, 871, 854,
// 834 us, 128^3 within 2%) but at least four steps; fewer where even so the CTAs
// do not fill `few` per SM (a step waits for its loads, so on small levels the
// march itself was the time: y/z-restriction of 16^3, 32 columns 16 us).  Four,
// but two for the FP64 y/z-restriction: a chunk forms the y-taps of the fine planes it
// shares with the next one again, on the FP64 pipe (restriction from 20^3, 256 columns
// 39.6 -> 33.6 us, 64^3, 8 columns 38.8 -> 33.6; 35.7 and 35.7 as three passes).
int march_chunk(long ctas, int len, long few = 4) {
    auto chunk = [&](long target) {
        const long ch = std::max(1L, std::min((long)len, (target + ctas - 1) / ctas));
        return (int)((len + ch - 1) / ch);
    };
    return std::max(chunk(152L * 16), std::min(4, chunk(152L * few)));
}
template <typename T>
size_t row_smem_bytes(const RowShape &s, int m, int mc) {
    return 4 * sizeof(T) * (size_t)m * s.lx * s.vec + (sizeof(T) + sizeof(int)) * RT * (size_t)mc;
}

template <typename T>
const T *taps(const double *d, const float *f);
template <>
const double *taps<double>(const double *d, const float *) { return d; }
template <>
const float *taps<float>(const double *, const float *f) { return f; }

template <typename T, int V, int MODE>
void run_row(int cls, const RowShape &s, int m, int mc, int N, const T *D, T c, T c2, const T *x,
             const T *b, const int *ridx, const T *rw, T *out, cudaStream_t st) {
    const int mz = march_chunk((long)s.gx * m, m);
    const dim3 grid(s.gx, m * ((m + mz - 1) / mz)), blk(s.lx, s.ty);
    const size_t sm = row_smem_bytes<T>(s, m, mc);
    auto go = [&](auto kernel) {
        HQ_LAUNCH_W(cls, (double)m * m * m * N,
                    kernel<<<grid, blk, sm, st>>>(m, mc, N, mz, D, c, c2, x, b, ridx, rw, out));
    };
    if (s.q == 1) go(k_row<T, V, 1, MODE>);
    else go(k_row<T, V, 2, MODE>);
}

template <typename T, int V>
void run_restrict_yz(const RowShape &s, int mf, int mc, int N, const XferTab &t, T scale, const T *in,
                     T *out, cudaStream_t st) {
    const int ty = std::max(1, 256 / s.lx), gy = (mc * mc + ty - 1) / ty;
    const int cz = march_chunk((long)s.gx * gy, mc, sizeof(T) == 8 ? 2 : 4);
    HQ_LAUNCH_W(HQ_K_TRANSFER, (double)mc * mc * mc * N,
                k_restrict_yz<T, V><<<dim3(s.gx, gy, (mc + cz - 1) / cz), dim3(s.lx, ty), 0, st>>>(
                    mf, mc, N, cz, t.ridx, taps<T>(t.rw, t.rwf), taps<T>(t.pw, t.pwf), scale, in, out));
}

template <typename T, int V>
void run_prolong(const RowShape &s, int mf, int mc, int N, const XferTab &t, const T *ec, const T *efin,
                 T *efout, cudaStream_t st) {
    const int nj = march_chunk((long)s.gx * mf, mf);
    const dim3 grid(s.gx, mf * ((mf + nj - 1) / nj)), blk(s.lx, s.ty);
    const size_t sm = 2 * sizeof(T) * V * (size_t)mc * s.lx;
    const T *pw = taps<T>(t.pw, t.pwf);
    auto go = [&](auto kernel) {
        HQ_LAUNCH_W(HQ_K_TRANSFER, (double)mf * mf * mf * N,
                    kernel<<<grid, blk, sm, st>>>(mf, mc, N, nj, t.pidx, pw, ec, efin, efout));
    };
    // 2 q + 1 fine points cover twice q coarse ones and the odd last point
    if (s.q == 1) go(k_prolong_rows<T, V, 1>);
    else go(k_prolong_rows<T, V, 2>);
}

template <typename T, typename F>
void vec_dispatch(int vec, F f) {
    if (vec == 4) f(std::integral_constant<int, sizeof(T) == 4 ? 4 : 2>());
    else if (vec == 2) f(std::integral_constant<int, 2>());
    else f(std::integral_constant<int, 1>());
}

}  // namespace

namespace {
template <typename T, int V>
void prepare_v() {
    auto set = [](auto kernel) {
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ROW_MAX_SMEM);
    };
    set(k_row<T, V, 1, ROW_RESID>);
    set(k_row<T, V, 2, ROW_RESID>);
    if constexpr (sizeof(T) == 4) {
        set(k_row<T, V, 1, ROW_SWEEP2>);
        set(k_row<T, V, 2, ROW_SWEEP2>);
    }
    set(k_prolong_rows<T, V, 1>);
    set(k_prolong_rows<T, V, 2>);
}
}  // namespace

void rows_prepare() {
    prepare_v<float, 4>();
    prepare_v<float, 2>();
    prepare_v<float, 1>();
    prepare_v<double, 2>();
    prepare_v<double, 1>();
}

// rows of at most ROW_MAXQ points per thread whose two buffers fit
template <typename T>
bool rows_fit(int m, int mc, int N) {
    const RowShape s = row_shape<T>(m, N);
    return s.q <= ROW_MAXQ && row_smem_bytes<T>(s, m, mc) <= ROW_MAX_SMEM;
}

template <typename T>
void launch_resid_restrict_x(int m, int mc, int N, const XferTab &t, const T *D, T c, const T *x,
                             const T *b, T *out, cudaStream_t st) {
    const RowShape s = row_shape<T>(m, N);
    vec_dispatch<T>(s.vec, [&](auto v) {
        run_row<T, v.value, ROW_RESID>(HQ_K_RESIDUAL, s, m, mc, N, D, c, T(0), x, b, t.ridx,
                                       taps<T>(t.rw, t.rwf), out, st);
    });
}

void launch_sweep2(int m, int N, const float *wD, float c, float omw, const float *r, float *z,
                   cudaStream_t st) {
    const RowShape s = row_shape<float>(m, N);
    vec_dispatch<float>(s.vec, [&](auto v) {
        run_row<float, v.value, ROW_SWEEP2>(HQ_K_SMOOTH, s, m, 0, N, wD, c, omw, r, nullptr, nullptr,
                                            nullptr, z, st);
    });
}

template <typename T>
void launch_restrict_yz(int mf, int mc, int N, const XferTab &t, const T *in, T *out, cudaStream_t st) {
    const double q = (double)(mc + 1) / (double)(mf + 1);
    const RowShape s = row_shape<T>(mc, N);
    vec_dispatch<T>(s.vec, [&](auto v) {
        run_restrict_yz<T, v.value>(s, mf, mc, N, t, (T)(q * q * q), in, out, st);
    });
}

template <typename T>
bool launch_prolong_rows(int mf, int mc, int N, const XferTab &t, const T *ec, const T *efin, T *efout,
                         cudaStream_t st) {
    const RowShape s = row_shape<T>(mc, N);
    // a thread's fine points: 2 q + 1 >= ceil(mf / ty) since mf <= 2 mc + 1
    if (s.q > 2 || 2 * sizeof(T) * s.vec * (size_t)mc * s.lx > ROW_MAX_SMEM) return false;
    vec_dispatch<T>(s.vec, [&](auto v) { run_prolong<T, v.value>(s, mf, mc, N, t, ec, efin, efout, st); });
    return true;
}

#define HQ_ROWS_INST(T)                                                                              \
    template bool rows_fit<T>(int, int, int);                                                        \
    template void launch_resid_restrict_x<T>(int, int, int, const XferTab &, const T *, T, const T *, \
                                             const T *, T *, cudaStream_t);                          \
    template void launch_restrict_yz<T>(int, int, int, const XferTab &, const T *, T *, cudaStream_t); \
    template bool launch_prolong_rows<T>(int, int, int, const XferTab &, const T *, const T *, T *,  \
                                         cudaStream_t);
HQ_ROWS_INST(double)
HQ_ROWS_INST(float)

}  // namespace hq
