// Pseudo-block flexible GMRES building blocks (Section 6: GMRES right-
// preconditioned by ORAS, stopped on the unpreconditioned relative residual;
// Section 6.3: pseudo-block fusion of the operations of several right-hand
// sides).  Every vector is row-major [n][m] (m right-hand sides contiguous), so
// one launch serves all columns, and columns stay independent: each keeps its
// own Hessenberg matrix, Givens rotations and convergence flag.
//
// Orthogonalisation is classical Gram-Schmidt applied twice (CGS2): dots of
// all basis vectors with w in one pass, then one fused update pass.
#include <algorithm>
#include <cstring>
#include <type_traits>

#include "common.h"
#include "df.h"
#include "gmres.h"
#include "kernels.h"
#include "per_device.h"

namespace mwi {

// ---------------------------------------------------------------- SpMM
// Y = A X: a group of G lanes (G = min(32, pow2 >= m)) per row, lanes over columns.
template <typename C, int G>
__global__ void __launch_bounds__(256) spmm_kernel(int64_t n, const int32_t* __restrict__ rp,
                                                   const int32_t* __restrict__ col, const C* __restrict__ val,
                                                   const C* __restrict__ X, C* __restrict__ Y, int m) {
    const int lane = threadIdx.x % G;
    const int64_t row = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / G;
    if (row >= n) return;
    const int b = rp[row], e = rp[row + 1];
    for (int c0 = 0; c0 < m; c0 += G) {
        const int c = c0 + lane;
        if (c >= m) break;
        C acc = czero<C>();
        for (int q = b; q < e; ++q) acc = cfma(val[q], X[(int64_t)col[q] * m + c], acc);
        Y[row * m + c] = acc;
    }
}

template <typename C>
void spmm(int64_t n, const int32_t* row_ptr, const int32_t* col, const C* val, const C* x, C* y, int m,
          cudaStream_t st) {
    const int th = 256;
    if (m >= 32) {
        int64_t blocks = (n * 32 + th - 1) / th;
        spmm_kernel<C, 32><<<(unsigned)blocks, th, 0, st>>>(n, row_ptr, col, val, x, y, m);
    } else if (m >= 8) {
        int64_t blocks = (n * 8 + th - 1) / th;
        spmm_kernel<C, 8><<<(unsigned)blocks, th, 0, st>>>(n, row_ptr, col, val, x, y, m);
    } else {
        int64_t blocks = (n * 4 + th - 1) / th;
        spmm_kernel<C, 4><<<(unsigned)blocks, th, 0, st>>>(n, row_ptr, col, val, x, y, m);
    }
    MWI_CHECK_LAUNCH();
}
template void spmm<double2>(int64_t, const int32_t*, const int32_t*, const double2*, const double2*, double2*, int,
                            cudaStream_t);
template void spmm<float2>(int64_t, const int32_t*, const int32_t*, const float2*, const float2*, float2*, int,
                           cudaStream_t);

// ---------------------------------------------------------------- dots
// partial[b][i][c] = sum over this block's rows of conj(V_i[r][c]) W[r][c].
// Rows are visited four at a time with independent loads, so that enough
// memory requests are in flight to stream V and W at HBM rate.
// With self = 1 the product conj(W) W is appended as vector index nvec.
// A block is (columns) x (8 row lanes) threads, columns the power of two at or
// above m, at most 32: idle lanes would still take their share of the FP64
// pipe (two multiply-adds per clock and SM), which bounds the FP64 form (a
// gradient step of 8 columns on 46,080 tets 152 -> 142 ms).
template <typename C>
__global__ void __launch_bounds__(256) dots_kernel(int64_t n, int m, int nvec_in, const C* __restrict__ V,
                                                   int64_t vstride, const C* __restrict__ W, int self,
                                                   double2* __restrict__ partial) {
    __shared__ double2 red[8][8][33];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int c = blockIdx.y * blockDim.x + tx;
    const int64_t stride = (int64_t)gridDim.x * 8;
    const int nvec = nvec_in + self;
    for (int i0 = 0; i0 < nvec; i0 += 8) {
        const int nq = min(8, nvec - i0);
        C acc[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[q] = czero<C>();
        if (c < m) {
            int64_t r = blockIdx.x * 8 + ty;
            for (; r + 3 * stride < n; r += 4 * stride) {
                C w[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) w[u] = W[(r + u * stride) * m + c];
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (q < nq) {
                        const C* Vq = (i0 + q < nvec_in ? V + (int64_t)(i0 + q) * vstride : W) + c;
                        C v[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) v[u] = Vq[(r + u * stride) * m];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            acc[q].x += v[u].x * w[u].x + v[u].y * w[u].y;
                            acc[q].y += v[u].x * w[u].y - v[u].y * w[u].x;
                        }
                    }
            }
            for (; r < n; r += stride) {
                const C w = W[r * m + c];
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (q < nq) {
                        const C v = (i0 + q < nvec_in ? V + (int64_t)(i0 + q) * vstride : W)[r * m + c];
                        acc[q].x += v.x * w.x + v.y * w.y;
                        acc[q].y += v.x * w.y - v.y * w.x;
                    }
            }
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) red[ty][q][tx] = make_double2((double)acc[q].x, (double)acc[q].y);
        __syncthreads();
        // thread (tx, ty) reduces vector q = ty over the 8 row lanes, in a fixed order
        {
            const int q = ty;
            double sx = 0.0, sy = 0.0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                sx += red[k][q][tx].x;
                sy += red[k][q][tx].y;
            }
            if (c < m && i0 + q < nvec) partial[((int64_t)blockIdx.x * nvec + i0 + q) * m + c] = make_double2(sx, sy);
        }
        __syncthreads();
    }
}

// h[i][c] = sum_b partial[b][i][c] for i < nvec; hacc[i][c] += h[i][c] for i < nacc;
// clear (optional): two counters set to zero on the way.
// One block per vector index i: 32 warps split the blocks b (b = warp, warp +
// 32, ...), lanes over columns, then a fixed-order sum of the 32 partial sums.
// The chain of loads and FP64 additions per warp bounds it (with 8 warps a
// forward solve of 4 columns on 3,072 tets took 6.25 ms, with 32 it takes 5.62).
__global__ void __launch_bounds__(1024) dots_reduce_kernel(int nblk, int nvec, int nacc, int m,
                                                          const double2* __restrict__ partial,
                                                          double2* __restrict__ h, double2* __restrict__ hacc,
                                                          int* __restrict__ clear) {
    __shared__ double2 red[32][33];
    const int i = blockIdx.x;
    if (clear && i == 0 && threadIdx.x < 2) clear[threadIdx.x] = 0;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int c0 = 0; c0 < m; c0 += 32) {
        const int c = c0 + tx;
        double sx = 0.0, sy = 0.0;
        if (c < m) {
#pragma unroll 10
            for (int b = ty; b < nblk; b += 32) {
                const double2 v = partial[((int64_t)b * nvec + i) * m + c];
                sx += v.x;
                sy += v.y;
            }
        }
        red[ty][tx] = make_double2(sx, sy);
#pragma unroll
        for (int w = 16; w > 0; w >>= 1) {
            __syncthreads();
            if (ty < w) red[ty][tx] = cadd(red[ty][tx], red[ty + w][tx]);
        }
        if (ty == 0 && c < m) {
            const double2 s = red[0][tx];
            const int e = i * m + c;
            h[e] = s;
            if (hacc && i < nacc) { hacc[e].x += s.x; hacc[e].y += s.y; }
        }
        __syncthreads();
    }
}

// W[r][c] -= sum_i V_i[r][c] h[i][c]
template <typename C>
__global__ void cgs_update_kernel(int64_t n, int m, int nvec, const C* __restrict__ V, int64_t vstride,
                                  const double2* __restrict__ h, C* __restrict__ W) {
    typedef typename real_of<C>::type R;
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n * m) return;
    const int c = (int)(e % m);
    C w = W[e];
    for (int i = 0; i < nvec; ++i) {
        const double2 hh = h[i * m + c];
        C hc;
        hc.x = (R)hh.x;
        hc.y = (R)hh.y;
        w = cfms(V[(int64_t)i * vstride + e], hc, w);
    }
    W[e] = w;
}

// V[r][c] = W[r][c] * s[c]
template <typename C>
__global__ void scale_kernel(int64_t n, int m, const C* __restrict__ W, const double* __restrict__ s,
                             C* __restrict__ V) {
    typedef typename real_of<C>::type R;
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n * m) return;
    const R f = (R)s[e % m];
    C w = W[e];
    w.x *= f;
    w.y *= f;
    V[e] = w;
}

// X[r][c] += sum_i Z_i[r][c] y[i][c]
template <typename C>
__global__ void lincomb_kernel(int64_t n, int m, int nvec, const C* __restrict__ Z, int64_t zstride,
                               const double2* __restrict__ y, C* __restrict__ X) {
    typedef typename real_of<C>::type R;
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n * m) return;
    const int c = (int)(e % m);
    C x = X[e];
    for (int i = 0; i < nvec; ++i) {
        const double2 yy = y[i * m + c];
        C yc;
        yc.x = (R)yy.x;
        yc.y = (R)yy.y;
        x = cfma(Z[(int64_t)i * zstride + e], yc, x);
    }
    X[e] = x;
}

// R = B - R  (R holds A X on entry)
template <typename C>
__global__ void sub_from_kernel(int64_t nm, const C* __restrict__ B, C* __restrict__ R) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= nm) return;
    R[e] = csub(B[e], R[e]);
}

template <typename A, typename B>
__global__ void convert_kernel(int64_t nm, const A* __restrict__ a, B* __restrict__ b) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= nm) return;
    b[e].x = a[e].x;
    b[e].y = a[e].y;
}

// The small per-column kernels below run one warp per column.  Their chains of
// dependent FP64 operations bound them: with one thread per column and a global
// load in every link a step's kernel took 27 us over 11 steps and the back
// substitution 55 us (24 steps: 55 and 200 us), more than anything else of a
// step on a small problem.  Lanes now hold 32 entries at a time and only the
// recurrences are serial: 15 and 17 us (24 steps: 24 and 33 us).

__device__ __forceinline__ double2 shfl2(double2 v, int lane) {
    return make_double2(__shfl_sync(0xffffffffu, v.x, lane), __shfl_sync(0xffffffffu, v.y, lane));
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double2 warp_sum(double2 v) { return make_double2(warp_sum(v.x), warp_sum(v.y)); }

// Rotations 0..j-1 of column c applied to a Hessenberg column with entries
// entry(0..j) (row i of entry is asked for by lane i % 32); row i < j of the
// rotated column goes to out(i, value), row j is returned to every lane.
template <typename Entry, typename Out>
__device__ __forceinline__ double2 rotate_column(int j, int m, int c, const double2* cs, const double2* sn,
                                                 Entry entry, Out out) {
    const int lane = threadIdx.x & 31;
    double2 t = entry(0);
    for (int base = 0; base < j; base += 32) {
        const int i = base + lane;
        double2 ci = make_double2(1.0, 0.0), si = make_double2(0.0, 0.0), h = si, u = si, mine = si;
        if (i < j) {
            ci = cs[i * m + c];
            si = sn[i * m + c];
            h = entry(i + 1);
            u = cmul(cconj(ci), h);
        }
        const int nq = min(32, j - base);
        for (int q = 0; q < nq; ++q) {
            if (lane == q) mine = t;
            t = csub(shfl2(u, q), cmul(cconj(shfl2(si, q)), t));
        }
        if (i < j) out(i, cadd(cmul(ci, mine), cmul(si, h)));
    }
    return t;
}

// the rotation that clears b against a, rows j and j + 1 of the column's
// factor R and of g (lane 0 writes); returns g's new last entry
__device__ __forceinline__ double2 new_rotation(int j, int m, int c, double2 a, double2 b, double2* Hj, double2* cs,
                                                double2* sn, double2* g) {
    const double den = sqrt(cabs2(a) + cabs2(b));
    double2 cj, sj;
    if (den > 0.0) { cj = cscale(cconj(a), 1.0 / den); sj = cscale(cconj(b), 1.0 / den); }
    else { cj = make_double2(1.0, 0.0); sj = make_double2(0.0, 0.0); }
    const double2 gj = g[j * m + c];
    const double2 gn = cscale(cmul(cconj(sj), gj), -1.0);
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
        cs[j * m + c] = cj;
        sn[j * m + c] = sj;
        Hj[j * m + c] = make_double2(den, 0.0);
        Hj[(j + 1) * m + c] = make_double2(0.0, 0.0);
        g[(j + 1) * m + c] = gn;
        g[j * m + c] = cmul(cj, gj);
    }
    __syncwarp();
    return gn;
}

// Per column c: rotate the Hessenberg column k (h[0..k], hnorm) by the previous
// rotations, form the new one, update g, decide convergence.
__global__ void arnoldi_kernel(int m, int k, int restart, const double2* __restrict__ h,
                               const double* __restrict__ hnorm2, double2* __restrict__ H, double2* cs, double2* sn,
                               double2* g, int* __restrict__ active, int* __restrict__ kcol,
                               const double* __restrict__ tol, double* __restrict__ resid,
                               double* __restrict__ inv_norm, int* __restrict__ n_active) {
    const int c = blockIdx.x, lane = threadIdx.x;
    if (!active[c]) {
        if (lane == 0) inv_norm[c] = 0.0;
        return;
    }
    double2* Hk = H + (int64_t)k * (restart + 1) * m;
    const double hn = sqrt(fmax(hnorm2[c], 0.0));
    const double2 a = rotate_column(
        k, m, c, cs, sn, [&](int i) { return h[i * m + c]; }, [&](int i, double2 v) { Hk[i * m + c] = v; });
    const double2 gn = new_rotation(k, m, c, a, make_double2(hn, 0.0), Hk, cs, sn, g);
    if (lane == 0) {
        kcol[c] = k + 1;
        const double rr = sqrt(cabs2(gn));
        resid[c] = rr;
        inv_norm[c] = hn > 0.0 ? 1.0 / hn : 0.0;
        if (rr <= tol[c] || hn == 0.0 || !(rr == rr)) active[c] = 0;
        else atomicAdd(n_active, 1);
    }
}

// y = R^{-1} g per column (R = rotated Hessenberg, kcol[c] columns), by columns
// of R: the right-hand side sits in shared memory (or, beyond its size, in y)
// ydf (optional) receives y as double-floats (re hi, re lo, im hi, im lo)
__global__ void lsq_kernel(int m, int restart, int in_smem, const double2* __restrict__ H,
                           const double2* __restrict__ g, const int* __restrict__ kcol, double2* y,
                           float4* __restrict__ ydf) {
    extern __shared__ double2 lsq_smem[];
    const int c = blockIdx.x, lane = threadIdx.x;
    double2* w = in_smem ? lsq_smem : y + c;
    const int ws = in_smem ? 1 : m;
    const int kk = kcol[c];
    for (int i = lane; i < restart; i += 32) {
        if (i < kk) w[i * (int64_t)ws] = g[i * m + c];
        else y[i * (int64_t)m + c] = make_double2(0.0, 0.0);
    }
    __syncwarp();
    auto R = [&](int r, int i) { return H[((int64_t)i * (restart + 1) + r) * m + c]; };
    double2 d = kk > 0 ? R(kk - 1, kk - 1) : make_double2(0.0, 0.0);
    double2 r0 = lane < kk - 1 ? R(lane, kk - 1) : make_double2(0.0, 0.0);
    for (int i = kk - 1; i >= 0; --i) {
        // the next column's entries on their way while this one's quotient is formed
        const double2 dn = i > 0 ? R(i - 1, i - 1) : d;
        const double2 rn = lane < i - 1 ? R(lane, i - 1) : r0;
        const double2 s = w[i * (int64_t)ws];
        const double2 yi = (d.x == 0.0 && d.y == 0.0) ? make_double2(0.0, 0.0) : cdiv(s, d);
        __syncwarp();
        for (int r = lane; r < i; r += 32)
            w[r * (int64_t)ws] = csub(w[r * (int64_t)ws], cmul(r == lane ? r0 : R(r, i), yi));
        if (lane == 0) w[i * (int64_t)ws] = yi;
        __syncwarp();
        d = dn;
        r0 = rn;
    }
    for (int i = lane; i < restart; i += 32) {
        const double2 v = i < kk ? w[i * (int64_t)ws] : make_double2(0.0, 0.0);
        if (in_smem && i < kk) y[i * (int64_t)m + c] = v;
        if (ydf) {
            const float2 a = df_split(v.x), b = df_split(v.y);
            ydf[i * (int64_t)m + c] = make_float4(a.x, a.y, b.x, b.y);
        }
    }
}

// start of a cycle: g = (beta, 0, ...), inv = 1/beta, active = beta > tol
__global__ void cycle_start_kernel(int m, const double* __restrict__ beta2, const double* __restrict__ tol,
                                   int* __restrict__ active, int* __restrict__ kcol, double2* __restrict__ g,
                                   double* __restrict__ inv_norm, double* __restrict__ resid,
                                   float2* __restrict__ inv_df) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= m) return;
    const double b = sqrt(fmax(beta2[c], 0.0));
    g[c] = make_double2(b, 0.0);
    kcol[c] = 0;
    resid[c] = b;
    const bool act = b > tol[c];
    active[c] = act ? 1 : 0;
    inv_norm[c] = act ? 1.0 / b : 0.0;
    if (inv_df) inv_df[c] = df_split(inv_norm[c]);
}

__global__ void tol_kernel(int m, const double* __restrict__ b2, double rtol, double* __restrict__ tol,
                           double* __restrict__ bnorm) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= m) return;
    const double b = sqrt(fmax(b2[c], 0.0));
    bnorm[c] = b;
    tol[c] = rtol * b;
}

// extract the real part of the diagonal dots (||w_c||^2)
__global__ void real_part_kernel(int m, const double2* __restrict__ h, double* __restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= m) return;
    out[c] = h[c].x;
}


// ---------------------------------------------------------------- double-float vectors
// A double-float [n][m] complex vector is two float2 planes, hi at p and lo at
// p + n m (value = hi + lo per real component).

// W = A Z (Z exact in FP32, RES = false) or W = B - A X (X and B double-float,
// RES = true), A as double-float planes (Ah, Al); G lanes per row over columns
template <int G, bool RES>
__global__ void __launch_bounds__(256) spmm_df_kernel(int64_t n, const int32_t* __restrict__ rp,
                                                      const int32_t* __restrict__ col, const float2* __restrict__ Ah,
                                                      const float2* __restrict__ Al, const float2* __restrict__ Xh,
                                                      const float2* __restrict__ Xl, const float2* __restrict__ Bh,
                                                      const float2* __restrict__ Bl, float2* __restrict__ Wh,
                                                      float2* __restrict__ Wl, int m) {
    const int lane = threadIdx.x % G;
    const int64_t row = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / G;
    if (row >= n) return;
    const int b = rp[row], e = rp[row + 1];
    for (int c0 = 0; c0 < m; c0 += G) {
        const int c = c0 + lane;
        if (c >= m) break;
        if constexpr (!RES) {
            dfl2 acc = {both(0.f), both(0.f)};
            for (int q = b; q < e; ++q) {
                const float2 ah = Ah[q], al = Al[q];
                const float2 xh = Xh[(int64_t)col[q] * m + c];
                df_mac1_2(acc, xh, both(ah.x), both(-ah.x), both(al.x));
                df_mac1_2(acc, make_float2(-xh.y, xh.x), both(ah.y), both(-ah.y), both(al.y));
            }
            acc = df_norm_2(acc);
            Wh[row * m + c] = acc.h;
            Wl[row * m + c] = acc.l;
            continue;
        }
        dfl re = {0.f, 0.f}, im = {0.f, 0.f};
        if constexpr (RES) {
            const float2 bh = Bh[row * m + c], bl = Bl[row * m + c];
            re = dfl{bh.x, bl.x};
            im = dfl{bh.y, bl.y};
        }
        for (int q = b; q < e; ++q) {
            const float2 ah = Ah[q], al = Al[q];
            const int64_t xi = (int64_t)col[q] * m + c;
            const float2 xh = Xh[xi], xl = Xl[xi];
            df_mac(re, -ah.x, -al.x, xh.x, xl.x);
            df_mac(re, ah.y, al.y, xh.y, xl.y);
            df_mac(im, -ah.x, -al.x, xh.y, xl.y);
            df_mac(im, -ah.y, -al.y, xh.x, xl.x);
        }
        re = df_norm(re);
        im = df_norm(im);
        Wh[row * m + c] = make_float2(re.h, im.h);
        Wl[row * m + c] = make_float2(re.l, im.l);
    }
}

// The same product for an even m with two adjacent columns per lane (16-byte
// loads of the right-hand sides; G lanes per row, the power of two at or above
// m / 2, at least 2, at most 16): four independent accumulation chains per thread instead of
// two.  Entries are applied in the same ascending order, so the results are the
// same bit for bit.
// w = A z (RES = false): the error-free products and sums bound it; they run on
// (re, im) pairs, two operations per instruction.  458,220 rows, 7.35 M entries,
// ms per product: 32 columns 0.48 -> 0.45, with two entries' loads in flight
// 0.41; 31 columns (one per lane, 32 lanes a row instead of four passes of 8)
// 0.57 -> 0.46; 6 columns 0.156 -> 0.115.
template <int G, bool RES>
__global__ void __launch_bounds__(256) spmm_df2_kernel(int64_t n, const int32_t* __restrict__ rp,
                                                       const int32_t* __restrict__ col, const float2* __restrict__ Ah,
                                                       const float2* __restrict__ Al, const float4* __restrict__ Xh,
                                                       const float4* __restrict__ Xl, const float4* __restrict__ Bh,
                                                       const float4* __restrict__ Bl, float4* __restrict__ Wh,
                                                       float4* __restrict__ Wl, int m) {
    const int lane = threadIdx.x % G;
    const int64_t row = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / G;
    if (row >= n) return;
    const int h = m >> 1;  // column pairs per row
    const int b = rp[row], e = rp[row + 1];
    for (int c0 = 0; c0 < h; c0 += G) {
        const int c = c0 + lane;
        if (c >= h) break;
        if constexpr (!RES) {
            dfl2 a0 = {both(0.f), both(0.f)}, a1 = a0;
            auto mac = [&](float2 ah, float2 al, float4 xh) {
                const float2 rh = both(ah.x), nrh = both(-ah.x), rl = both(al.x);
                const float2 ih = both(ah.y), nih = both(-ah.y), il = both(al.y);
                df_mac1_2(a0, make_float2(xh.x, xh.y), rh, nrh, rl);
                df_mac1_2(a1, make_float2(xh.z, xh.w), rh, nrh, rl);
                df_mac1_2(a0, make_float2(-xh.y, xh.x), ih, nih, il);
                df_mac1_2(a1, make_float2(-xh.w, xh.z), ih, nih, il);
            };
            int q = b;
            for (; q + 1 < e; q += 2) {  // two entries' loads in flight together
                const float2 ah0 = Ah[q], al0 = Al[q], ah1 = Ah[q + 1], al1 = Al[q + 1];
                const float4 x0 = Xh[(int64_t)col[q] * h + c], x1 = Xh[(int64_t)col[q + 1] * h + c];
                mac(ah0, al0, x0);
                mac(ah1, al1, x1);
            }
            if (q < e) mac(Ah[q], Al[q], Xh[(int64_t)col[q] * h + c]);
            a0 = df_norm_2(a0);
            a1 = df_norm_2(a1);
            Wh[row * h + c] = make_float4(a0.h.x, a0.h.y, a1.h.x, a1.h.y);
            Wl[row * h + c] = make_float4(a0.l.x, a0.l.y, a1.l.x, a1.l.y);
            continue;
        }
        dfl re0 = {0.f, 0.f}, im0 = {0.f, 0.f}, re1 = {0.f, 0.f}, im1 = {0.f, 0.f};
        if constexpr (RES) {
            const float4 bh = Bh[row * h + c], bl = Bl[row * h + c];
            re0 = dfl{bh.x, bl.x};
            im0 = dfl{bh.y, bl.y};
            re1 = dfl{bh.z, bl.z};
            im1 = dfl{bh.w, bl.w};
        }
        for (int q = b; q < e; ++q) {
            const float2 ah = Ah[q], al = Al[q];
            const int64_t xi = (int64_t)col[q] * h + c;
            const float4 xh = Xh[xi], xl = Xl[xi];
            df_mac(re0, -ah.x, -al.x, xh.x, xl.x);
            df_mac(re0, ah.y, al.y, xh.y, xl.y);
            df_mac(im0, -ah.x, -al.x, xh.y, xl.y);
            df_mac(im0, -ah.y, -al.y, xh.x, xl.x);
            df_mac(re1, -ah.x, -al.x, xh.z, xl.z);
            df_mac(re1, ah.y, al.y, xh.w, xl.w);
            df_mac(im1, -ah.x, -al.x, xh.w, xl.w);
            df_mac(im1, -ah.y, -al.y, xh.z, xl.z);
        }
        re0 = df_norm(re0);
        im0 = df_norm(im0);
        re1 = df_norm(re1);
        im1 = df_norm(im1);
        Wh[row * h + c] = make_float4(re0.h, im0.h, re1.h, im1.h);
        Wl[row * h + c] = make_float4(re0.l, im0.l, re1.l, im1.l);
    }
}

// V = W s per column (W, V double-float, s double-float [m])
__global__ void scale_df_kernel(int64_t nm, int m, const float2* __restrict__ W, const float2* __restrict__ s,
                                float2* __restrict__ V) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= nm) return;
    const float2 f = s[e % m];
    const float2 wh = W[e], wl = W[nm + e];
    const dfl re = df_mul(wh.x, wl.x, f.x, f.y), im = df_mul(wh.y, wl.y, f.x, f.y);
    V[e] = make_float2(re.h, im.h);
    V[nm + e] = make_float2(re.l, im.l);
}

// X += sum_i Z_i y_i per column (Z_i exact in FP32, X double-float, y
// double-float [nvec][m])
__global__ void __launch_bounds__(256) lincomb_df_kernel(int64_t nm, int m, int nvec, const float2* __restrict__ Z,
                                                         int64_t zstride, const float4* __restrict__ ydf,
                                                         float2* __restrict__ X) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= nm) return;
    const int c = (int)(e % m);
    const float2 xh = X[e], xl = X[nm + e];
    dfl re = {xh.x, xl.x}, im = {xh.y, xl.y};
    for (int i = 0; i < nvec; ++i) {
        const float2 z = Z[(int64_t)i * zstride + e];
        const float4 y = ydf[i * m + c];
        df_mac1(re, z.x, y.x, y.y);
        df_mac1(re, -z.y, y.z, y.w);
        df_mac1(im, z.x, y.z, y.w);
        df_mac1(im, z.y, y.x, y.y);
    }
    re = df_norm(re);
    im = df_norm(im);
    X[e] = make_float2(re.h, im.h);
    X[nm + e] = make_float2(re.l, im.l);
}

// double-float planes of a c128 array of count entries, and back
__global__ void split_c128_kernel(int64_t count, const double2* __restrict__ a, float2* __restrict__ out) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= count) return;
    const double2 v = a[e];
    const float2 x = df_split(v.x), y = df_split(v.y);
    out[e] = make_float2(x.x, y.x);
    out[count + e] = make_float2(x.y, y.y);
}

__global__ void join_c128_kernel(int64_t count, const float2* __restrict__ in, double2* __restrict__ a) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= count) return;
    const float2 h = in[e], l = in[count + e];
    a[e] = make_double2(df_join(h.x, l.x), df_join(h.y, l.y));
}


// ---------------------------------------------------------------- DCGS2 Arnoldi (double-float basis)
// Classical Gram-Schmidt with delayed reorthogonalisation (the one-reduction
// DCGS2 Arnoldi of Swirydowicz, Langou, Ananthan, Yang and Thomas, "Low
// synchronization Gram-Schmidt and generalized minimal residual algorithms",
// 2021): step k makes one pass of dot products over the basis for both the
// new vector w = A z_k and the once-orthogonalised v_k, then one fused update
// pass that reorthogonalises v_k into q_k and projects w into the next v_{k+1}.

// partial[b][j][c], j < nq: conj(Q_j) x; nq + j: conj(Q_j) y; 2 nq: conj(x) x;
// 2 nq + 1: conj(x) y; 2 nq + 2: conj(y) y (FP32 heads, FP32 sums per thread,
// FP64 across threads); eight basis vectors per pass over the rows
__global__ void __launch_bounds__(256) dots2_kernel(int64_t n, int m, int nq, const float2* __restrict__ V,
                                                    int64_t vstride, const float2* __restrict__ X,
                                                    const float2* __restrict__ Yv, double2* __restrict__ partial) {
    __shared__ double2 red[8][8][33];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int c = blockIdx.y * 32 + tx;
    const int64_t stride = (int64_t)gridDim.x * 8;
    const int nout = 2 * nq + 3;
    // fixed-order sum over the eight row lanes of the values in red[.][q][tx]
    auto flush = [&](int nv, int j0, int jstride) {
        __syncthreads();
        if (ty < nv && c < m) {
            double sx = 0.0, sy = 0.0;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                sx += red[r][ty][tx].x;
                sy += red[r][ty][tx].y;
            }
            partial[((int64_t)blockIdx.x * nout + j0 + ty * jstride) * m + c] = make_double2(sx, sy);
        }
        __syncthreads();
    };
    for (int q0 = 0; q0 < (nq > 0 ? nq : 1); q0 += 8) {
        const int nqc = nq > 0 ? min(8, nq - q0) : 0;
        const bool self = q0 == 0;
        float2 A[8], B[8], G = make_float2(0.f, 0.f), D = G, O = G;
#pragma unroll
        for (int q = 0; q < 8; ++q) A[q] = B[q] = make_float2(0.f, 0.f);
        if (c < m) {
            // two rows per iteration, their loads issued together
            for (int64_t r = blockIdx.x * 8 + ty; r < n; r += 2 * stride) {
                const bool two = r + stride < n;
                const int64_t r2 = two ? r + stride : r;
                const float2 x0 = X[r * m + c], y0 = Yv[r * m + c];
                const float2 x1 = two ? X[r2 * m + c] : make_float2(0.f, 0.f);
                const float2 y1 = two ? Yv[r2 * m + c] : make_float2(0.f, 0.f);
                float2 v0[8], v1[8];
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (q < nqc) {
                        const float2* Vq = V + (int64_t)(q0 + q) * vstride + c;
                        v0[q] = Vq[r * m];
                        v1[q] = two ? Vq[r2 * m] : make_float2(0.f, 0.f);
                    }
                if (self) {
                    G.x += x0.x * x0.x + x0.y * x0.y + x1.x * x1.x + x1.y * x1.y;
                    D.x += x0.x * y0.x + x0.y * y0.y + x1.x * y1.x + x1.y * y1.y;
                    D.y += x0.x * y0.y - x0.y * y0.x + x1.x * y1.y - x1.y * y1.x;
                    O.x += y0.x * y0.x + y0.y * y0.y + y1.x * y1.x + y1.y * y1.y;
                }
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (q < nqc) {
                        A[q].x += v0[q].x * x0.x + v0[q].y * x0.y + v1[q].x * x1.x + v1[q].y * x1.y;
                        A[q].y += v0[q].x * x0.y - v0[q].y * x0.x + v1[q].x * x1.y - v1[q].y * x1.x;
                        B[q].x += v0[q].x * y0.x + v0[q].y * y0.y + v1[q].x * y1.x + v1[q].y * y1.y;
                        B[q].y += v0[q].x * y0.y - v0[q].y * y0.x + v1[q].x * y1.y - v1[q].y * y1.x;
                    }
            }
        }
        if (nqc > 0) {
#pragma unroll
            for (int q = 0; q < 8; ++q) red[ty][q][tx] = make_double2(A[q].x, A[q].y);
            flush(nqc, q0, 1);
#pragma unroll
            for (int q = 0; q < 8; ++q) red[ty][q][tx] = make_double2(B[q].x, B[q].y);
            flush(nqc, nq + q0, 1);
        }
        if (self) {
            red[ty][0][tx] = make_double2(G.x, 0.0);
            red[ty][1][tx] = make_double2(D.x, D.y);
            red[ty][2][tx] = make_double2(O.x, 0.0);
            flush(3, 2 * nq, 1);
        }
    }
}

// Per column: finalise column k-1 of the Hessenberg matrix with v_k's
// reorthogonalisation (coefficients a, norm nu), form column k from w's
// projections (provisional: its last entry rho_k is the Pythagorean norm of
// the projected w, made exact by the next step's correction), test the
// residual estimate with a provisional rotation of column k, and emit the
// double-float coefficients of the fused update.  A column that converges (or
// the last step) keeps column k as it stands: v_{k+1} then closes the basis
// without reorthogonalisation, which leaves the Arnoldi relation exact.
__device__ __forceinline__ double2 conjmul(double2 a, double2 b) { return cmul(cconj(a), b); }

__device__ __forceinline__ float4 df4(double2 v) {
    const float2 a = df_split(v.x), b = df_split(v.y);
    return make_float4(a.x, a.y, b.x, b.y);
}

__global__ void arnoldi_dcgs_kernel(int m, int k, int restart, int last, const double2* __restrict__ dots,
                                    double2* H, double2* Hp, double2* cs, double2* sn, double2* g,
                                    int* __restrict__ active, int* __restrict__ kcol, const double* __restrict__ tol,
                                    double* __restrict__ resid, double* __restrict__ rho,
                                    int* __restrict__ n_active, float4* __restrict__ coefQ,
                                    float4* __restrict__ coefW, float4* __restrict__ scal) {
    // n_active[0]: columns still active; n_active[1]: the largest of their residuals
    // over their tolerances, as the bits of a float (non-negative, so ordered alike)
    const int c = blockIdx.x, lane = threadIdx.x;
    const int nq = k;
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!active[c]) {
        for (int i = lane; i < nq; i += 32) coefQ[i * m + c] = coefW[i * m + c] = z4;
        if (lane == 0) scal[c] = scal[m + c] = z4;
        return;
    }
    const double2* a = dots + c;           // a_i = conj(q_i) v_k
    const double2* b = dots + nq * m + c;  // b_i = conj(q_i) w
    const double gam = dots[(2 * nq) * m + c].x;
    const double2 del = dots[(2 * nq + 1) * m + c];
    const double om = dots[(2 * nq + 2) * m + c].x;
    // |a|^2, |b|^2 and q_k^H w's a^H b
    double a2 = 0.0, b2 = 0.0;
    double2 ab = make_double2(0.0, 0.0);
    for (int i = lane; i < nq; i += 32) {
        const double2 ai = a[i * m], bi = b[i * m];
        a2 += cabs2(ai);
        b2 += cabs2(bi);
        ab = cadd(ab, conjmul(ai, bi));
    }
    a2 = warp_sum(a2);
    b2 = warp_sum(b2);
    ab = warp_sum(ab);
    double nu = 1.0;
    if (k > 0) {
        nu = sqrt(fmax(gam - a2, 1e-30 * fmax(gam, 1e-300)));
        // column k-1: v_k = Q a + nu q_k, so h(i, k-1) += rho_{k-1} a_i and h(k, k-1) = rho_{k-1} nu
        const double r1 = rho[c];
        double2* Hc = H + (int64_t)(k - 1) * (restart + 1) * m;
        const double2 t = rotate_column(
            k - 1, m, c, cs, sn, [&](int i) { return cadd(Hp[i * m + c], cscale(a[i * m], r1)); },
            [&](int i, double2 v) { Hc[i * m + c] = v; });
        new_rotation(k - 1, m, c, t, make_double2(r1 * nu, 0.0), Hc, cs, sn, g);
    }
    // q_k^H w and the projected w's norm
    const double2 ck = cscale(csub(del, ab), 1.0 / nu);
    const double rk = sqrt(fmax(om - b2 - cabs2(ck), 1e-14 * om));
    // provisional column k: (b_0 .. b_{k-1}, c_k, rho_k); its rotated entry k (rotations
    // 0..k-1), then the provisional residual
    auto col = [&](int i) { return i < k ? b[i * m] : ck; };
    const double2 t = rotate_column(k, m, c, cs, sn, col, [](int, double2) {});
    const double den = sqrt(cabs2(t) + rk * rk);
    const double rr = den > 0.0 ? rk / den * sqrt(cabs2(g[k * m + c])) : 0.0;
    for (int i = lane; i <= k; i += 32) Hp[i * m + c] = col(i);
    const bool stop = rr <= tol[c] || !(rr == rr) || rk == 0.0 || last;
    if (stop) {
        double2* Hc = H + (int64_t)k * (restart + 1) * m;
        rotate_column(k, m, c, cs, sn, col, [&](int i, double2 v) { Hc[i * m + c] = v; });
        new_rotation(k, m, c, t, make_double2(rk, 0.0), Hc, cs, sn, g);
    }
    if (lane == 0) {
        Hp[(k + 1) * m + c] = make_double2(rk, 0.0);
        resid[c] = rr;
        rho[c] = rk;
        kcol[c] = stop ? k + 1 : k;
        if (stop && !last) {
            active[c] = 0;
        } else if (!stop || !(rr <= tol[c])) {
            atomicAdd(n_active, 1);
            atomicMax(n_active + 1, __float_as_int(fminf((float)(rr / tol[c]), 3e38f)));
        }
    }
    // fused update: q_k = v_k / nu - sum_i q_i a_i / nu;
    // v_{k+1} = w / rho_k - sum_i q_i (b_i - a_i c_k / nu) / rho_k - v_k c_k / (nu rho_k)
    const double inu = 1.0 / nu, irk = 1.0 / rk;
    for (int i = lane; i < nq; i += 32) {
        const double2 ai = a[i * m];
        coefQ[i * m + c] = df4(cscale(ai, -inu));
        coefW[i * m + c] = df4(cscale(csub(b[i * m], cscale(cmul(ai, ck), inu)), -irk));
    }
    if (lane == 0) {
        scal[c] = df4(make_double2(k > 0 ? inu : 1.0, irk));  // (1 / nu, 1 / rho_k) as reals
        scal[m + c] = df4(cscale(ck, -inu * irk));            // -c_k / (nu rho_k)
    }
}

// q_k (into V slot k, when k > 0) and v_{k+1} (into V slot k + 1) in one pass
// over the basis: per element, two double-float accumulators over the k basis
// vectors, v_k and w
__global__ void __launch_bounds__(256) dcgs_update_df_kernel(int64_t nm, int m, int k, float2* __restrict__ V,
                                                             int64_t vstride, const float2* __restrict__ W,
                                                             const float4* __restrict__ coefQ,
                                                             const float4* __restrict__ coefW,
                                                             const float4* __restrict__ scal, int write_next) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= nm) return;
    const int c = (int)(e % m);
    const float4 s1 = scal[c], s2 = scal[m + c];
    float2* vk = V + (int64_t)k * vstride;
    const float2 vh = vk[e], vl = vk[nm + e];
    // q accumulator: v_k / nu; x accumulator: w / rho_k + v_k (-c_k / (nu rho_k));
    // (re, im) pairs, the operations in the order of the even-m form
    dfl2 q = df_mul_2(vh, vl, both(s1.x), both(s1.y)), x = df_mul_2(W[e], W[nm + e], both(s1.z), both(s1.w));
    df_mac_2(x, vh, vl, both(s2.x), both(-s2.x), both(s2.y));
    df_mac_2(x, make_float2(-vh.y, vh.x), make_float2(-vl.y, vl.x), both(s2.z), both(-s2.z), both(s2.w));
#pragma unroll 2
    for (int i = 0; i < k; ++i) {
        const float2 uh = V[(int64_t)i * vstride + e], ul = V[(int64_t)i * vstride + nm + e];
        const float2 th = make_float2(-uh.y, uh.x), tl = make_float2(-ul.y, ul.x);
        const float4 a = coefQ[i * m + c], b = coefW[i * m + c];
        df_mac_2(q, uh, ul, both(a.x), both(-a.x), both(a.y));
        df_mac_2(q, th, tl, both(a.z), both(-a.z), both(a.w));
        df_mac_2(x, uh, ul, both(b.x), both(-b.x), both(b.y));
        df_mac_2(x, th, tl, both(b.z), both(-b.z), both(b.w));
    }
    if (k > 0) {
        q = df_norm_2(q);
        vk[e] = q.h;
        vk[nm + e] = q.l;
    }
    if (write_next) {
        x = df_norm_2(x);
        float2* vn = V + (int64_t)(k + 1) * vstride;
        vn[e] = x.h;
        vn[nm + e] = x.l;
    }
}

constexpr int kUpdRing = 4;
constexpr int kUpdSmem = kUpdRing * 4 * 256 * 16;

__device__ __forceinline__ void copy16(float4* dst, const float4* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// The same pass for an even m, bound by memory (16 k + 64 bytes per element): a
// thread takes two adjacent columns (16-byte accesses) of two rows, so that the
// coefficients and their packed forms serve both, and has the next three basis
// vectors on their way into shared memory (its own places, no barrier) while it
// works on one: registers for as many bytes in flight would leave too few
// threads.  A block is (column pairs) x (rows), rows contiguous in memory.  With
// one column of one row per thread the Arnoldi steps of a solve (458,220 rows, 32
// columns, 24 steps, dot products included) took 25.8 ms; two by two with the
// next vector in registers 24.0; now 22.8.
__global__ void __launch_bounds__(256) dcgs_update_df2_kernel(int64_t n, int h, int k, float4* __restrict__ V,
                                                              int64_t vstride, const float4* __restrict__ W,
                                                              const float4* __restrict__ coefQ,
                                                              const float4* __restrict__ coefW,
                                                              const float4* __restrict__ scal, int write_next) {
    const int cp = blockIdx.y * blockDim.x + threadIdx.x;
    if (cp >= h) return;
    const int64_t r0 = blockIdx.x * (int64_t)(2 * blockDim.y) + threadIdx.y;
    if (r0 >= n) return;
    const int64_t nh = n * h;
    const bool two = r0 + blockDim.y < n;
    const int64_t e0 = r0 * h + cp, e1 = two ? e0 + (int64_t)blockDim.y * h : e0;
    const int m = 2 * h;
    float4* const vk = V + (int64_t)k * vstride;
    struct Pair { float4 h[2], l[2]; };  // two columns of the two rows
    auto load = [&](const float4* p) { return Pair{{p[e0], p[e1]}, {p[nh + e0], p[nh + e1]}}; };
    extern __shared__ __align__(16) float4 ring[];  // [kUpdRing][4][256]
    float4* const mine = ring + threadIdx.y * blockDim.x + threadIdx.x;
    auto fetch = [&](int i) {
        if (i < k) {
            const float4* p = V + (int64_t)i * vstride;
            float4* d = mine + (i % kUpdRing) * 4 * 256;
            copy16(d, p + e0);
            copy16(d + 256, p + e1);
            copy16(d + 512, p + nh + e0);
            copy16(d + 768, p + nh + e1);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int i = 0; i < kUpdRing - 1; ++i) fetch(i);
    auto lo2 = [](float4 v, int c) { return c ? make_float2(v.z, v.w) : make_float2(v.x, v.y); };
    const Pair v = load(vk), w = load(W);
    dfl2 q[2][2], x[2][2];  // [column][row]: q_k and v_{k+1}
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const float4 s1 = scal[2 * cp + c], s2 = scal[m + 2 * cp + c];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const float2 vh = lo2(v.h[r], c), vl = lo2(v.l[r], c);
            q[c][r] = df_mul_2(vh, vl, both(s1.x), both(s1.y));
            x[c][r] = df_mul_2(lo2(w.h[r], c), lo2(w.l[r], c), both(s1.z), both(s1.w));
            df_mac_2(x[c][r], vh, vl, both(s2.x), both(-s2.x), both(s2.y));
            df_mac_2(x[c][r], make_float2(-vh.y, vh.x), make_float2(-vl.y, vl.x), both(s2.z), both(-s2.z),
                     both(s2.w));
        }
    }
    for (int i = 0; i < k; ++i) {
        fetch(i + kUpdRing - 1);
        asm volatile("cp.async.wait_group %0;" ::"n"(kUpdRing - 1) : "memory");
        const float4* const d = mine + (i % kUpdRing) * 4 * 256;
        const Pair u = {{d[0], d[256]}, {d[512], d[768]}};
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const float4 a = coefQ[i * m + 2 * cp + c], b = coefW[i * m + 2 * cp + c];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const float2 uh = lo2(u.h[r], c), ul = lo2(u.l[r], c);
                const float2 th = make_float2(-uh.y, uh.x), tl = make_float2(-ul.y, ul.x);
                df_mac_2(q[c][r], uh, ul, both(a.x), both(-a.x), both(a.y));
                df_mac_2(q[c][r], th, tl, both(a.z), both(-a.z), both(a.w));
                df_mac_2(x[c][r], uh, ul, both(b.x), both(-b.x), both(b.y));
                df_mac_2(x[c][r], th, tl, both(b.z), both(-b.z), both(b.w));
            }
        }
    }
    auto put = [&](float4* p, dfl2 (&a)[2][2]) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if (r == 1 && !two) continue;
            const int64_t e = r ? e1 : e0;
            const dfl2 c0 = df_norm_2(a[0][r]), c1 = df_norm_2(a[1][r]);
            p[e] = make_float4(c0.h.x, c0.h.y, c1.h.x, c1.h.y);
            p[nh + e] = make_float4(c0.l.x, c0.l.y, c1.l.x, c1.l.y);
        }
    };
    if (k > 0) put(vk, q);
    if (write_next) put(vk + vstride, x);
}

// ----------------------------------------------------------------------------
static inline unsigned nblocks(int64_t n, int th) { return (unsigned)((n + th - 1) / th); }

static void launch_lsq(int m, int restart, const double2* H, const double2* g, const int* kcol, double2* y,
                       float4* ydf, cudaStream_t st) {
    const size_t sm = (size_t)restart * sizeof(double2);
    const bool fits = sm <= 48 * 1024;
    lsq_kernel<<<m, 32, fits ? sm : 0, st>>>(m, restart, fits ? 1 : 0, H, g, kcol, y, ydf);
    MWI_CHECK_LAUNCH();
}

template <typename C>
void Gmres<C>::reserve(int64_t n_, int m_, int restart_) {
    n = n_;
    m = m_;
    restart = restart_;
    V.ensure((size_t)(restart + 1) * n * m);
    Z.ensure((size_t)restart * n * m);
    W.ensure((size_t)n * m);
    H.ensure((size_t)restart * (restart + 1) * m);
    cs.ensure((size_t)restart * m);
    sn.ensure((size_t)restart * m);
    g.ensure((size_t)(restart + 1) * m);
    y.ensure((size_t)restart * m);
    h.ensure((size_t)(restart + 2) * m);
    hacc.ensure((size_t)(restart + 1) * m);
    partial.ensure((size_t)kDotBlocks * (restart + 2) * m);
    dvec.ensure((size_t)8 * m);
    ivec.ensure((size_t)4 * m + 4);
}

// out[i][c] = conj(V_i)^T w for i < nvec (+ conj(w)^T w at nvec when self = 1),
// acc[i] += out[i] for i < nvec (optional)
template <typename C>
static void dots_launch(int64_t n, int m, const C* Vb, int nvec, int64_t vstride, const C* w, double2* partial,
                        double2* out, double2* acc, cudaStream_t st, int self) {
    int mx = 1;
    while (mx < std::min(m, 32)) mx *= 2;
    dim3 blk(mx, 8), grd(kDotBlocks, (m + mx - 1) / mx);
    dots_kernel<C><<<grd, blk, 0, st>>>(n, m, nvec, Vb, vstride, w, self, partial);
    MWI_CHECK_LAUNCH();
    const int nt = nvec + self;
    dots_reduce_kernel<<<nt, 1024, 0, st>>>(kDotBlocks, nt, nvec, m, partial, out, acc, nullptr);
    MWI_CHECK_LAUNCH();
}

template <typename C>
void Gmres<C>::dots(const C* Vb, int nvec, int64_t vstride, const C* w, double2* out, double2* acc,
                    cudaStream_t st, int self) {
    dots_launch<C>(n, m, Vb, nvec, vstride, w, partial.p, out, acc, st, self);
}

template <typename C>
void Gmres<C>::column_norms2(const C* x, double* out, cudaStream_t st) {
    column_norms2_into(x, out, h.p, st);
}

// ||x_c||^2 with tmp [m] double2 scratch
template <typename C>
void Gmres<C>::column_norms2_into(const C* x, double* out, double2* tmp, cudaStream_t st) {
    dots(x, 0, 0, x, tmp, nullptr, st, 1);
    real_part_kernel<<<nblocks(m, 128), 128, 0, st>>>(m, tmp, out);
    MWI_CHECK_LAUNCH();
}

template <typename C>
int Gmres<C>::cycle(const OpFn& A, const OpFn& M, const C* r0, C* x, const double* tol, int max_steps,
                    cudaStream_t st, double* resid_host, int* iters_used) {
    const int64_t nm = n * m;
    const int64_t vs = nm;
    double* beta2 = dvec.p;            // [m]
    double* inv = dvec.p + m;          // [m]
    double* resid = dvec.p + 2 * m;    // [m]
    double* hn2 = dvec.p + 3 * m;      // [m]
    int* active = ivec.p;
    int* kcol = ivec.p + m;
    int* nact = ivec.p + 4 * m;
    column_norms2(r0, beta2, st);
    cycle_start_kernel<<<nblocks(m, 128), 128, 0, st>>>(m, beta2, tol, active, kcol, g.p, inv, resid, nullptr);
    MWI_CHECK_LAUNCH();
    scale_kernel<C><<<nblocks(nm, 256), 256, 0, st>>>(n, m, r0, inv, V.p);
    MWI_CHECK_LAUNCH();
    int k = 0;
    int n_active_host = 1;
    for (; k < max_steps; ++k) {
        C* vk = V.p + (int64_t)k * vs;
        C* zk = Z.p + (int64_t)k * vs;
        M(vk, zk);
        A(zk, W.p);
        // classical Gram-Schmidt applied twice (CGS2)
        auto ortho = [&] {
            MWI_CUDA(cudaMemsetAsync(hacc.p, 0, (size_t)(k + 1) * m * sizeof(double2), st));
            for (int pass = 0; pass < 2; ++pass) {
                dots(V.p, k + 1, vs, W.p, h.p, hacc.p, st, 0);
                cgs_update_kernel<C><<<nblocks(nm, 256), 256, 0, st>>>(n, m, k + 1, V.p, vs, h.p, W.p);
                MWI_CHECK_LAUNCH();
            }
            column_norms2(W.p, hn2, st);
        };
        if (timer) timer(2, ortho);
        else ortho();
        MWI_CUDA(cudaMemsetAsync(nact, 0, sizeof(int), st));
        arnoldi_kernel<<<m, 32, 0, st>>>(m, k, restart, hacc.p, hn2, H.p, cs.p, sn.p, g.p, active, kcol, tol, resid,
                                         inv, nact);
        MWI_CHECK_LAUNCH();
        if (k + 1 < max_steps) {
            scale_kernel<C><<<nblocks(nm, 256), 256, 0, st>>>(n, m, W.p, inv, V.p + (int64_t)(k + 1) * vs);
            MWI_CHECK_LAUNCH();
        }
        MWI_CUDA(cudaMemcpyAsync(&n_active_host, nact, sizeof(int), cudaMemcpyDeviceToHost, st));
        MWI_CUDA(cudaStreamSynchronize(st));
        if (n_active_host == 0) { ++k; break; }
    }
    launch_lsq(m, restart, H.p, g.p, kcol, y.p, nullptr, st);
    lincomb_kernel<C><<<nblocks(nm, 256), 256, 0, st>>>(n, m, k, Z.p, vs, y.p, x);
    MWI_CHECK_LAUNCH();
    if (resid_host) {
        MWI_CUDA(cudaMemcpyAsync(resid_host, resid, m * sizeof(double), cudaMemcpyDeviceToHost, st));
        MWI_CUDA(cudaStreamSynchronize(st));
    }
    if (iters_used) *iters_used = k;
    return k;
}

template struct Gmres<double2>;
template struct Gmres<float2>;

// ---------------------------------------------------------------- double-float FGMRES
void GmresDF::reserve(int64_t n_, int m_, int restart_) {
    n = n_;
    m = m_;
    restart = restart_;
    V.ensure((size_t)(restart + 1) * 2 * n * m);
    Z.ensure((size_t)restart * n * m);
    W.ensure((size_t)2 * n * m);
    H.ensure((size_t)restart * (restart + 1) * m);
    cs.ensure((size_t)restart * m);
    sn.ensure((size_t)restart * m);
    g.ensure((size_t)(restart + 1) * m);
    y.ensure((size_t)restart * m);
    h.ensure((size_t)(2 * restart + 3) * m);
    partial.ensure((size_t)kDotBlocks * (2 * restart + 3) * m);
    hdf.ensure((size_t)(restart + 1) * m);
    hdf2.ensure((size_t)(restart + 1) * m);
    scal.ensure((size_t)2 * m);
    Hp.ensure((size_t)(restart + 2) * m);
    ydf.ensure((size_t)restart * m);
    invdf.ensure((size_t)m);
    dvec.ensure((size_t)8 * m);
    ivec.ensure((size_t)4 * m + 4);
}

void GmresDF::norms2(const float2* xh, double* out, cudaStream_t st) {
    dots_launch<float2>(n, m, xh, 0, 0, xh, partial.p, h.p, nullptr, st, 1);
    real_part_kernel<<<nblocks(m, 128), 128, 0, st>>>(m, h.p, out);
    MWI_CHECK_LAUNCH();
}

static void allow_update_smem() {
    static PerDevice<bool> set;
    set.get(current_device(), [] {
        MWI_CUDA(cudaFuncSetAttribute(dcgs_update_df2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kUpdSmem));
        return true;
    });
}

int GmresDF::cycle(const OpA& A, const OpM& M, const float2* r0, float2* x, const double* tol, int max_steps,
                   cudaStream_t st, int* iters_used) {
    const int64_t nm = n * m;
    const int64_t vs = 2 * nm;  // stride of the double-float basis vectors
    double* beta2 = dvec.p;
    double* inv = dvec.p + m;
    double* resid = dvec.p + 2 * m;
    double* rho = dvec.p + 3 * m;
    int* active = ivec.p;
    int* kcol = ivec.p + m;
    int* nact = ivec.p + 4 * m;
    norms2(r0, beta2, st);
    cycle_start_kernel<<<nblocks(m, 128), 128, 0, st>>>(m, beta2, tol, active, kcol, g.p, inv, resid, invdf.p);
    MWI_CHECK_LAUNCH();
    // v_0 = r0 / beta exactly (q_0 = v_0: no reorthogonalisation at step 0)
    scale_df_kernel<<<nblocks(nm, 256), 256, 0, st>>>(nm, m, r0, invdf.p, V.p);
    MWI_CHECK_LAUNCH();
    status.create();
    int k = 0;
    bool ahead = false;   // z_k has been launched with the step before
    float left = 0.f, left_before = 0.f;  // largest residual over tolerance after this step and the one before
    for (; k < max_steps; ++k) {
        float2* vk = V.p + (int64_t)k * vs;
        float2* zk = Z.p + (int64_t)k * nm;
        // the preconditioner sees the FP32 head of v_k (once orthogonalised);
        // z_k is stored exactly
        if (!ahead) M(vk, zk);
        A(zk, W.p);
        const int last = k + 1 == max_steps ? 1 : 0;
        auto ortho = [&] {
            // one wave: two resident blocks per SM at this kernel's register use
            const int nblk = kDotBlocks / 2;
            dim3 blk(32, 8), grd(nblk, (m + 31) / 32);
            dots2_kernel<<<grd, blk, 0, st>>>(n, m, k, V.p, vs, vk, W.p, partial.p);
            MWI_CHECK_LAUNCH();
            const int nout = 2 * k + 3;
            dots_reduce_kernel<<<nout, 1024, 0, st>>>(nblk, nout, 0, m, partial.p, h.p, nullptr, nact);
            MWI_CHECK_LAUNCH();
            arnoldi_dcgs_kernel<<<m, 32, 0, st>>>(m, k, restart, last, h.p, H.p, Hp.p, cs.p, sn.p, g.p, active, kcol,
                                                  tol, resid, rho, nact, hdf.p, hdf2.p, scal.p);
            MWI_CHECK_LAUNCH();
            MWI_CUDA(cudaMemcpyAsync(status.host, nact, 2 * sizeof(int), cudaMemcpyDeviceToHost, st));
            MWI_CUDA(cudaEventRecord(status.ready, st));
            if (m % 2 == 0) {
                const int h = m / 2, hx = std::min(h, 256), hy = 256 / hx;
                allow_update_smem();
                dcgs_update_df2_kernel<<<dim3(nblocks(n, 2 * hy), (h + hx - 1) / hx), dim3(hx, hy), kUpdSmem, st>>>(
                    n, h, k, reinterpret_cast<float4*>(V.p), vs / 2, reinterpret_cast<const float4*>(W.p), hdf.p,
                    hdf2.p, scal.p, last ? 0 : 1);
            } else {
                dcgs_update_df_kernel<<<nblocks(nm, 256), 256, 0, st>>>(nm, m, k, V.p, vs, W.p, hdf.p, hdf2.p,
                                                                        scal.p, last ? 0 : 1);
            }
            MWI_CHECK_LAUNCH();
        };
        if (timer) timer(2, ortho);
        else ortho();
        // The next preconditioner application is launched before this step's status
        // has come back if the last step's reduction of the residual, twice over,
        // would still leave it above the tolerance: the GPU then has work while the
        // host waits and launches (12 us a step).  A wrong guess costs one application.
        ahead = !last && k > 0 && left_before > 0.f && left * (left / left_before) * (left / left_before) > 1.f;
        if (ahead) M(V.p + (int64_t)(k + 1) * vs, Z.p + (int64_t)(k + 1) * nm);
        MWI_CUDA(cudaEventSynchronize(status.ready));
        left_before = left;
        std::memcpy(&left, status.host + 1, sizeof(float));
        if (status.host[0] == 0) { ++k; break; }
    }
    launch_lsq(m, restart, H.p, g.p, kcol, y.p, ydf.p, st);
    lincomb_df_kernel<<<nblocks(nm, 256), 256, 0, st>>>(nm, m, k, Z.p, nm, ydf.p, x);
    MWI_CHECK_LAUNCH();
    if (iters_used) *iters_used = k;
    return k;
}

template <bool RES>
static void launch_spmm_df(int64_t n, const int32_t* row_ptr, const int32_t* col, const float2* A, int64_t nnz,
                           const float2* x, const float2* b, float2* w, int m, cudaStream_t st) {
    const int th = 256;
    const int64_t nm = n * m;
    auto f4 = [](const float2* p) { return reinterpret_cast<const float4*>(p); };
    auto pairs = [&](auto g) {
        constexpr int G = decltype(g)::value;
        spmm_df2_kernel<G, RES><<<(unsigned)((n * G + th - 1) / th), th, 0, st>>>(
            n, row_ptr, col, A, A + nnz, f4(x), RES ? f4(x + nm) : nullptr, RES ? f4(b) : nullptr,
            RES ? f4(b + nm) : nullptr, reinterpret_cast<float4*>(w), reinterpret_cast<float4*>(w + nm), m);
    };
    auto singles = [&](auto g) {
        constexpr int G = decltype(g)::value;
        spmm_df_kernel<G, RES><<<(unsigned)((n * G + th - 1) / th), th, 0, st>>>(
            n, row_ptr, col, A, A + nnz, x, RES ? x + nm : nullptr, b, RES ? b + nm : nullptr, w, w + nm, m);
    };
    if ((m & 1) == 0) {
        if (m > 16) pairs(std::integral_constant<int, 16>());
        else if (m > 8) pairs(std::integral_constant<int, 8>());
        else if (m > 4) pairs(std::integral_constant<int, 4>());
        else pairs(std::integral_constant<int, 2>());
    } else {
        if (m > 16) singles(std::integral_constant<int, 32>());
        else if (m > 8) singles(std::integral_constant<int, 16>());
        else if (m > 4) singles(std::integral_constant<int, 8>());
        else singles(std::integral_constant<int, 4>());
    }
    MWI_CHECK_LAUNCH();
}

void spmm_df(int64_t n, const int32_t* row_ptr, const int32_t* col, const float2* A, int64_t nnz, const float2* x,
             float2* w, int m, cudaStream_t st) {
    launch_spmm_df<false>(n, row_ptr, col, A, nnz, x, nullptr, w, m, st);
}

void residual_df(int64_t n, const int32_t* row_ptr, const int32_t* col, const float2* A, int64_t nnz, const float2* b,
                 const float2* x, float2* r, int m, cudaStream_t st) {
    launch_spmm_df<true>(n, row_ptr, col, A, nnz, x, b, r, m, st);
}

void split_c128(int64_t count, const double2* a, float2* out, cudaStream_t st) {
    split_c128_kernel<<<nblocks(count, 256), 256, 0, st>>>(count, a, out);
    MWI_CHECK_LAUNCH();
}

void join_c128(int64_t count, const float2* in, double2* a, cudaStream_t st) {
    join_c128_kernel<<<nblocks(count, 256), 256, 0, st>>>(count, in, a);
    MWI_CHECK_LAUNCH();
}

void convert_c128_to_c64(int64_t nm, const double2* a, float2* b, cudaStream_t st) {
    convert_kernel<double2, float2><<<nblocks(nm, 256), 256, 0, st>>>(nm, a, b);
    MWI_CHECK_LAUNCH();
}
void convert_c64_to_c128(int64_t nm, const float2* a, double2* b, cudaStream_t st) {
    convert_kernel<float2, double2><<<nblocks(nm, 256), 256, 0, st>>>(nm, a, b);
    MWI_CHECK_LAUNCH();
}
void residual_c128(int64_t nm, const double2* b, double2* r, cudaStream_t st) {
    sub_from_kernel<double2><<<nblocks(nm, 256), 256, 0, st>>>(nm, b, r);
    MWI_CHECK_LAUNCH();
}
__global__ void copy_columns_kernel(int64_t n, int ms, int sc0, int mc, const double2* __restrict__ src, int md,
                                    int dc0, double2* __restrict__ dst) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n * mc) return;
    const int64_t r = e / mc;
    const int c = (int)(e - r * mc);
    dst[r * md + dc0 + c] = src[r * ms + sc0 + c];
}

void copy_columns(int64_t n, int ms, int sc0, int mc, const double2* src, int md, int dc0, double2* dst,
                  cudaStream_t st) {
    copy_columns_kernel<<<nblocks(n * mc, 256), 256, 0, st>>>(n, ms, sc0, mc, src, md, dc0, dst);
    MWI_CHECK_LAUNCH();
}

void tolerances(int m, const double* b2, double rtol, double* tol, double* bnorm, cudaStream_t st) {
    tol_kernel<<<nblocks(m, 128), 128, 0, st>>>(m, b2, rtol, tol, bnorm);
    MWI_CHECK_LAUNCH();
}

}  // namespace mwi
