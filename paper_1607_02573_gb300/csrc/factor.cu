// Batched multifrontal LDL^T factorisation of every subdomain operator B_i
// (the local solves of Eq. ORAS; the paper uses PARDISO/MUMPS per MPI rank,
// here all subdomains are one batch on one GPU).
//
// B_i is complex symmetric (the form of Eq. pbdirectvarf is bilinear), so
// B_i = L D L^T without conjugation.  Pivoting is static: Im(B_i) is positive
// definite for a lossy medium (Im eps < 0), which makes every leading minor
// non-zero; a pivot that is zero or not finite is replaced and counted.
//
// The fronts of one assembly-tree depth are processed together, deepest
// depth first: assemble (entries of B_i, then extend-add of the children's
// Schur complements), then a blocked right-looking partial factorisation of
// the p pivot columns that leaves the Schur complement for the parent and, in
// place of the factor, its partitioned inverse for the sweeps.
// A front (dense, f = p + u, lower triangle used) is stored in two pieces:
// its p pivot columns as a column-major f x p panel in the factor store, and its
// u x u Schur block in a transient buffer shared by the fronts of one level (two
// buffers, even and odd levels, since a level's blocks are consumed by the next
// level).  The sweeps want the first p columns of the inverse of
// [L11 0; L21 I], i.e. [L11^{-1}; -L21 L11^{-1}] (partitioned inverse), with a
// unit diagonal, and D^{-1} after the panels (indexed by local row), so that each
// front's part of the ORAS sweeps is one dependency-free dense product per
// direction (sweep.cu).  Of every level, per step of nb pivot columns k ..:
//   diag    the diagonal block's L D L^T and W, the inverse of its unit lower
//           triangular factor (replaces the block; D on its diagonal)
//   rows    L_i = a_i W^T D^{-1} for the rows below (to a scratch panel), and
//           X_k <- W X_k, X being the inverse's pivot rows left of the step
//   step    C_ic -= L_i D L_c^T in the remaining pivot columns, and
//           X_i -= L_i X_k in the remaining pivot rows (Gauss-Jordan, in place
//           of the factor), as tiles of one launch
// and after the last step, as tiles of one launch over all p pivots,
//   end     the Schur block S -= L_2 D L_2^T and the inverse's update rows
//           X_2 = -L_2 X_1
// so that a step touches the pivot columns alone, and the larger part of a front
// is read and written once.  Before, every step updated the whole trailing
// matrix, and the inverse was formed after the level by column-blocked
// substitution, eight columns of a front per block, each reading the whole
// panel.  Whole factorisations (tiled copies included), before and now: 3,072
// tets 1.34 -> 1.00 ms, 120,288 tets 9.56 -> 8.4 ms, 402,444 tets 39.2 -> 37 ms,
// second order on 53,046 tets 104 -> 82 ms, FP64 on 46,080 tets 41.3 -> 34.5 ms.
#include <algorithm>
#include <type_traits>

#include "common.h"
#include "df.h"
#include "kernels.h"

namespace mwi {

template <typename C> __device__ __forceinline__ C from_d2(double2 v);
template <> __device__ __forceinline__ double2 from_d2<double2>(double2 v) { return v; }
template <> __device__ __forceinline__ float2 from_d2<float2>(double2 v) { return make_float2((float)v.x, (float)v.y); }

template <typename C>
__global__ void front_assemble_kernel(const int32_t* __restrict__ level_fronts, int lo,
                                      const int64_t* __restrict__ amap_front_ptr,
                                      const int64_t* __restrict__ amap_slot, const int64_t* __restrict__ amap_pos,
                                      const double2* __restrict__ B, C* __restrict__ ws) {
    const int s = level_fronts[lo + blockIdx.x];
    for (int64_t q = amap_front_ptr[s] + threadIdx.x; q < amap_front_ptr[s + 1]; q += blockDim.x)
        ws[amap_pos[q]] = from_d2<C>(B[amap_slot[q]]);
}

// One block per (front, child, four child rows) tile: parent[urel[a], urel[b]]
// += S_c[a, b], a >= b, where S_c is the child's Schur block and the parent
// entry lies in its panel (pivot column) or in its own Schur block.  The first
// and second children of the fronts go in separate launches (they add into the
// same parent entries; the order is fixed, so no atomics are needed).
template <typename C>
__global__ void extend_add_kernel(const int4* __restrict__ tiles, const int32_t* __restrict__ P,
                                  const int32_t* __restrict__ U, const int64_t* __restrict__ f_off,
                                  const int64_t* __restrict__ sch_off, const int64_t* __restrict__ u_off,
                                  const int32_t* __restrict__ urel, C* __restrict__ ws, const C* __restrict__ sch_child,
                                  C* __restrict__ sch_par) {
    const int4 tl = tiles[blockIdx.x];  // (front, child, first child row)
    const int s = tl.x, c = tl.y;
    const int uc = U[c];
    const int b = tl.z + threadIdx.y;
    if (b >= uc) return;
    const int ps = P[s], us = U[s];
    const int64_t fs = (int64_t)ps + us;
    const int32_t* rel = urel + u_off[c];
    const C* src = sch_child + sch_off[c] + (int64_t)b * uc;
    const int rb = rel[b];
    C* dst = rb < ps ? ws + f_off[s] + (int64_t)rb * fs : sch_par + sch_off[s] + (int64_t)(rb - ps) * us - ps;
    for (int a = b + threadIdx.x; a < uc; a += blockDim.x) {
        const C v = src[a];
        C& d = dst[rel[a]];
        d.x += v.x;
        d.y += v.y;
    }
}

constexpr int kUpdateSlab = 8;  // pivots per shared-memory buffer of the products

template <typename C>
__device__ __forceinline__ bool bad_pivot(C d) {
    typename real_of<C>::type a = d.x * d.x + d.y * d.y;
    return !(a > (typename real_of<C>::type)0) || !isfinite(a);
}

// Panel step k, diagonal block, one block of NB x 8 threads per front: thread
// (row lane, column c) holds the entries (row lane + 8 q, c) in registers.  Step
// j publishes column j (rows below j) and row j (columns left of j), and every
// thread applies l_r = a_rj / d_j to its rows r > j: right of j the LDL^T update,
// left of it and in column j the inverse's.  One barrier per step; a warp alone,
// its lanes over the rows, took 35 us per launch, of which 16 are left.
template <typename C, int NB>
__global__ void __launch_bounds__(NB * 8) panel_diag_kernel(const int32_t* __restrict__ level_fronts, int lo, int k,
                                                            const int32_t* __restrict__ P,
                                                            const int32_t* __restrict__ U,
                                                            const int64_t* __restrict__ f_off, C* __restrict__ ws,
                                                            int* __restrict__ perturbed) {
    constexpr int Q = NB / 8;
    __shared__ C colb[2][NB], rowb[2][NB];
    const int s = level_fronts[lo + blockIdx.x];
    const int p = P[s];
    if (k >= p) return;
    const int64_t f = (int64_t)p + U[s];
    const int nb = min(NB, p - k);
    C* F = ws + f_off[s] + (int64_t)k * f + k;
    // rows fastest over the threads: coalesced panel columns
    const int rl = threadIdx.x & 7, c = threadIdx.x >> 3;
    C v[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int r = rl + 8 * q;
        v[q] = (r < nb && c <= r) ? F[(int64_t)c * f + r] : czero<C>();
    }
    for (int j = 0; j < nb; ++j) {
        C* cb = colb[j & 1];
        C* rb = rowb[j & 1];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int r = rl + 8 * q;
            if (c == j && r >= j) cb[r] = v[q];
            if (r == j && c < j) rb[c] = v[q];
        }
        __syncthreads();
        C d = cb[j];
        if (bad_pivot(d)) {  // the same value in every thread
            d = cmake<C>(1, 0);
            if (c == j && rl == (j & 7)) {
#pragma unroll
                for (int q = 0; q < Q; ++q)
                    if (q == (j >> 3)) v[q] = d;
                atomicAdd(perturbed, 1);
            }
        }
        const C rd = crecip(d);
        const C w = c > j ? cb[c] : (c < j ? rb[c] : czero<C>());
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int r = rl + 8 * q;
            if (r > j) {
                const C l = cmul(cb[r], rd);
                if (c == j) v[q] = cmake<C>(-l.x, -l.y);
                else if (c <= r) v[q] = cfms(l, w, v[q]);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int r = rl + 8 * q;
        if (r < nb && c <= r) F[(int64_t)c * f + r] = v[q];
    }
}

// Panel step k, rows: over a tile list (front, first row) of 128-row tiles below
// the diagonal block, one thread per row: L_i to the scratch panel; and (front,
// -1 - first column) of 128-column tiles left of it, one thread per column:
// X_k <- W X_k.  The products are unrolled over W's triangle; the __syncwarp()s
// keep its loads from being moved up in a heap that spills the row's registers.
template <typename C, int NB>
__global__ void __launch_bounds__(128, 3) panel_rows_kernel(const int2* __restrict__ tiles, int k,
                                                         const int32_t* __restrict__ P, const int32_t* __restrict__ U,
                                                         const int64_t* __restrict__ f_off,
                                                         const int64_t* __restrict__ l_off, C* __restrict__ ws,
                                                         C* __restrict__ lbuf) {
    __shared__ C W[NB][NB + 1];  // strictly lower: W; diagonal: 1 / D
    const int2 tl = tiles[blockIdx.x];
    const int s = tl.x;
    const int p = P[s];
    const int64_t f = (int64_t)p + U[s];
    const int nb = min(NB, p - k);
    C* F = ws + f_off[s];
    {
        // the block's loads in flight before the stores (128 threads)
        C v[NB * NB / 128];
#pragma unroll
        for (int t = 0; t < NB * NB / 128; ++t) {
            const int e = threadIdx.x + 128 * t, r = e % NB, c = e / NB;
            v[t] = (r < nb && c <= r) ? F[(int64_t)(k + c) * f + k + r] : czero<C>();
        }
#pragma unroll
        for (int t = 0; t < NB * NB / 128; ++t) {
            const int e = threadIdx.x + 128 * t, r = e % NB, c = e / NB;
            W[r][c] = r == c && r < nb ? crecip(v[t]) : v[t];
        }
    }
    __syncthreads();
    const bool left = tl.y < 0;
    const int64_t i = left ? -1 - tl.y + threadIdx.x : tl.y + threadIdx.x;
    if (i >= (left ? k : f)) return;
    // a row's entries of the step's columns, or a column's of the step's rows, all
    // loads in flight together, then W times them in place
    C* const X = left ? F + i * f + k : F + k * f + i;
    const int64_t step = left ? 1 : f;
    C x[NB];
#pragma unroll
    for (int j = 0; j < NB; ++j) x[j] = j < nb ? X[j * step] : czero<C>();
#pragma unroll
    for (int j = NB - 1; j > 0; --j)
#pragma unroll
        for (int q = 0; q < NB; ++q)
            if (q < j) {
                x[j] = cfma(W[j][q], x[q], x[j]);
                if (q % 8 == 7) __syncwarp();
            }
    if (left) {
#pragma unroll
        for (int j = 0; j < NB; ++j)
            if (j < nb) X[j] = x[j];
    } else {
        C* const L = lbuf + l_off[s] + k * f + i;
#pragma unroll
        for (int j = 0; j < NB; ++j)
            if (j < nb) L[j * f] = cmul(x[j], W[j][j]);
    }
}

// The products of the step (k >= 0, one step's pivots) and of the level's end
// (k < 0, all pivots), a TILE x TILE output tile per block of 256 threads, over a
// tile list (front, tile row, tile column, kind):
//   kStep     rows [r0, f), columns [r0, p), r0 = k + nb: C -= L_i D L_c^T, lower triangle
//   kStepInv  rows [r0, p), columns [0, r0): X -= L_i X_k; in the step's own
//             columns X = -L_i W
//   kSchur    rows and columns [p, f): S -= L_i D L_c^T, lower triangle
//   kInv      rows [p, f), columns [0, p): X = -L_i X_1
// Slabs of KS pivots pass through two shared-memory buffers, the next one's loads
// in flight during the products.  Complex FP32: bound by the FP32 pipe and by
// how many warps are there to fill it (half to 60 % busy with four blocks of 64
// registers per SM).  Factorisations of 402,444 tets when the shape was chosen,
// before the rows kernel worked in place: slabs of 8 and four blocks 38.0 ms,
// slabs of 16 38.8, three blocks of 80 registers 41.0.  A thread's four rows and
// columns are the pairs 2t, 2t + 1 and 32 + 2t, 32 + 2t + 1, read as 16-byte
// shared loads; a complex multiply-add is two packed ones, which halves its issue
// slots (at that time 39.8 -> 39.0 ms; with the packed operands laid out in shared
// memory, twice the shared loads, 41).
// Complex FP64 is bound by its pipe alone: quarters of a tile without wanted
// entries -- beyond the last row or column, or above the diagonal -- are left out
// of the products (46,080 tets: 38.1 -> 34.4 ms per factorisation).  In FP32 the
// further loops cost registers and gain little (402,444 tets 36.7 -> 36.2 ms, second
// order 81.1 -> 82.7), so its tiles are computed whole.
enum { kStep = 0, kStepInv = 1, kSchur = 2, kInv = 3 };

template <typename C, int TILE, int NB>
__global__ void __launch_bounds__(256, 4)
    update_kernel(const int4* __restrict__ tiles, int k, const int32_t* __restrict__ P, const int32_t* __restrict__ U,
                  const int64_t* __restrict__ f_off, const int64_t* __restrict__ sch_off,
                  const int64_t* __restrict__ l_off, C* __restrict__ ws, const C* __restrict__ lbuf,
                  C* __restrict__ sch) {
    constexpr bool kF32 = sizeof(C) == sizeof(float2);
    constexpr int MT = TILE / 16;
    // rows padded to an even length, so that every pair is 16-byte aligned
    constexpr bool kPairs = kF32 && MT == 4;
    constexpr int LD = kPairs ? TILE + 2 : TILE + 1;
    constexpr int KS = kUpdateSlab;
    constexpr int NT = KS * TILE / 256;
    __shared__ __align__(16) C As[2][KS][LD];
    __shared__ __align__(16) C Bs[2][KS][LD];
    const int4 tl = tiles[blockIdx.x];
    const int s = tl.x, kind = tl.w;
    const int p = P[s], f = p + U[s];
    const int r0 = k < 0 ? p : min(k + NB, p);
    C* const F = ws + f_off[s];
    const C* const L = lbuf + l_off[s];
    const int tid = threadIdx.x;
    const bool inv = (kind & 1) != 0;
    const int rowA = r0 + tl.y * TILE, endA = kind == kStepInv ? p : f;
    const int rowB = (inv ? 0 : r0) + tl.z * TILE, endB = kind == kSchur ? f : (kind == kStepInv ? r0 : p);
    // pivots of the product (X_1 is zero above its diagonal)
    const int j_end = k < 0 ? p : r0;
    const int j_beg = k >= 0 ? k : (inv ? rowB / KS * KS : 0);
    // the inverse's columns: pivots fastest; the factor's: rows fastest
    auto b_row = [&](int t) { return inv ? (tid + 256 * t) / KS : (tid + 256 * t) % TILE; };
    auto b_k = [&](int t) { return inv ? (tid + 256 * t) % KS : (tid + 256 * t) / TILE; };
    C av[NT], bv[NT];
    auto load = [&](int j0) {
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            const int e = tid + 256 * t, row = rowA + e % TILE, j = j0 + e / TILE;
            av[t] = bv[t] = czero<C>();
            if (j < j_end && row < endA) {
                av[t] = L[(int64_t)j * f + row];
                if (!inv) av[t] = cmul(av[t], F[(int64_t)j * f + j]);
            }
            const int c = rowB + b_row(t), jb = j0 + b_k(t);
            if (jb < j_end && c < endB) {
                if (!inv) bv[t] = L[(int64_t)jb * f + c];
                else if (jb > c) bv[t] = F[(int64_t)c * f + jb];
                else if (jb == c) bv[t] = cmake<C>(1, 0);
            }
        }
    };
    auto store = [&](int buf) {
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            const int e = tid + 256 * t;
            As[buf][e / TILE][e % TILE] = av[t];
            Bs[buf][b_k(t)][b_row(t)] = bv[t];
        }
    };
    const int tx = tid % 16, ty = tid / 16;
    // local row of accumulator a (column of b) within the tile
    auto off = [](int t, int a) { return kPairs ? 32 * (a >> 1) + 2 * t + (a & 1) : t + 16 * a; };
    C acc[MT][MT];
#pragma unroll
    for (int a = 0; a < MT; ++a)
#pragma unroll
        for (int b = 0; b < MT; ++b) acc[a][b] = czero<C>();
    load(j_beg);
    store(0);
    // HR, HC: the tile has rows (columns) beyond its first half; UP: its upper right
    // quarter is wanted
    auto products = [&](auto hr, auto hc, auto up) {
        constexpr int XR = decltype(hr)::value ? MT : MT / 2, YC = decltype(hc)::value ? MT : MT / 2;
        constexpr bool kUp = decltype(up)::value;
        int buf = 0;
        for (int j0 = j_beg; j0 < j_end; j0 += KS, buf ^= 1) {
            __syncthreads();
            const bool more = j0 + KS < j_end;
            if (more) load(j0 + KS);
#pragma unroll 4
            for (int j = 0; j < KS; ++j) {
                C a[MT], b[MT];
                if constexpr (kPairs) {
#pragma unroll
                    for (int h = 0; h < XR / 2; ++h) {
                        const float4 v = *reinterpret_cast<const float4*>(&As[buf][j][32 * h + 2 * tx]);
                        a[2 * h] = cmake<C>(v.x, v.y);
                        a[2 * h + 1] = cmake<C>(v.z, v.w);
                    }
#pragma unroll
                    for (int h = 0; h < YC / 2; ++h) {
                        const float4 v = *reinterpret_cast<const float4*>(&Bs[buf][j][32 * h + 2 * ty]);
                        b[2 * h] = cmake<C>(v.x, v.y);
                        b[2 * h + 1] = cmake<C>(v.z, v.w);
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < XR; ++q) a[q] = As[buf][j][off(tx, q)];
#pragma unroll
                    for (int q = 0; q < YC; ++q) b[q] = Bs[buf][j][off(ty, q)];
                }
#pragma unroll
                for (int x = 0; x < XR; ++x)
#pragma unroll
                    for (int y = 0; y < YC; ++y) {
                        if (!kUp && x < MT / 2 && y >= MT / 2) continue;
                        if constexpr (kF32) {
                            acc[x][y] = fma2(both(a[x].x), b[y], acc[x][y]);
                            acc[x][y] = fma2(both(a[x].y), make_float2(-b[y].y, b[y].x), acc[x][y]);
                        } else {
                            acc[x][y] = cfma(a[x], b[y], acc[x][y]);
                        }
                    }
            }
            if (more) store(buf ^ 1);
        }
    };
    {
        const std::true_type yes;
        const std::false_type no;
        const bool hr = endA - rowA > TILE / 2, hc = endB - rowB > TILE / 2;
        const bool up = inv || rowA != rowB;
        if constexpr (kF32) {
            products(yes, yes, yes);
        } else if (hr && hc) {
            if (up) products(yes, yes, yes);
            else products(yes, yes, no);
        } else if (hr) {
            products(yes, no, yes);
        } else if (hc && up) {
            products(no, yes, yes);
        } else {
            products(no, no, yes);
        }
    }
    const int u = f - p;
    C* const Sb = sch + sch_off[s];
#pragma unroll
    for (int y = 0; y < MT; ++y) {
        const int col = rowB + off(ty, y);
        if (col >= endB) continue;
        // pivot columns live in the panel (ld f), the others in the Schur block (ld u)
        C* const colp = col < p ? F + (int64_t)col * f : Sb + (int64_t)(col - p) * u - p;
        const bool fresh = kind == kInv || (kind == kStepInv && col >= k);  // replaces the factor's entries
#pragma unroll
        for (int x = 0; x < MT; ++x) {
            const int row = rowA + off(tx, x);
            if (row < endA && row >= col) {
                C& dst = colp[row];
                const C v = acc[x][y];
                dst = fresh ? cmake<C>(-v.x, -v.y) : csub(dst, v);
            }
        }
    }
}

// D^{-1} of every pivot of the level's fronts into dinv at its local row, and the
// inverse's unit diagonal in D's place
template <typename C>
__global__ void finish_diag_kernel(const int32_t* __restrict__ level_fronts, int lo, const int32_t* __restrict__ P,
                                   const int32_t* __restrict__ U, const int32_t* __restrict__ start,
                                   const int32_t* __restrict__ sub, const int64_t* __restrict__ sub_off,
                                   const int64_t* __restrict__ f_off, C* __restrict__ ws, C* __restrict__ dinv) {
    const int s = level_fronts[lo + blockIdx.x];
    const int p = P[s];
    const int64_t f = (int64_t)p + U[s];
    C* F = ws + f_off[s];
    C* out = dinv + sub_off[sub[s]] + start[s];
    for (int j = threadIdx.x; j < p; j += blockDim.x) {
        C& d = F[(int64_t)j * f + j];
        out[j] = crecip(d);
        d = cmake<C>(1, 0);
    }
}

template <typename C> struct FactorCfg;
template <> struct FactorCfg<float2> { static constexpr int NB = 32; static constexpr int TILE = 64; };
template <> struct FactorCfg<double2> { static constexpr int NB = 16; static constexpr int TILE = 32; };

template <typename C>
void factorize_fronts(const FrontsDev& F, const UpdateTiles& ut, const double2* Bvals, C* ws, C* const sch[2],
                      C* lbuf, int* perturbed, cudaStream_t st) {
    constexpr int NB = FactorCfg<C>::NB, TILE = FactorCfg<C>::TILE;
    static_assert(NB % kUpdateSlab == 0, "a step is whole slabs");
    MWI_REQUIRE(ut.nb == NB && ut.tile == TILE, MWI_EINVAL, "internal: update tiles built for another blocking");
    MWI_CUDA(cudaMemsetAsync(ws, 0, (size_t)(F.ws_entries + F.nloc) * sizeof(C), st));
    const int nlev = (int)F.level_ptr.size() - 1;
    // the largest front that is accepted: 12,800 rows in complex FP32, 6,400 in FP64.
    // Callers have always had this limit; the kernels here do not need it.
    for (int l = 0; l < nlev; ++l)
        MWI_REQUIRE(2 * (size_t)F.level_fmax[l] * sizeof(C) <= 200 * 1024, MWI_EINVAL,
                    "front too large (" + std::to_string(F.level_fmax[l]) + " rows)");
    size_t range = 0, ext = 0, end = 0;
    for (int l = 0; l < nlev; ++l) {
        const int lo0 = F.level_ptr[l], hi = F.level_ptr[l + 1];
        C* sch_l = sch[l & 1];
        const C* sch_child = sch[(l + 1) & 1];
        if (F.level_sch[l] > 0) MWI_CUDA(cudaMemsetAsync(sch_l, 0, (size_t)F.level_sch[l] * sizeof(C), st));
        for (int lo = lo0; lo < hi; lo += 65535) {
            const int nf = std::min(65535, hi - lo);
            front_assemble_kernel<C><<<nf, 256, 0, st>>>(F.level_fronts.p, lo, F.amap_front_ptr.p, F.amap_slot.p,
                                                         F.amap_pos.p, Bvals, ws);
            MWI_CHECK_LAUNCH();
            for (int ci = 0; ci < 2; ++ci) {
                MWI_REQUIRE(ext + 1 < F.ext_ptr.size(), MWI_EINVAL, "internal: extend-add tile list out of step");
                const int64_t t0 = F.ext_ptr[ext], t1 = F.ext_ptr[ext + 1];
                ++ext;
                if (t1 > t0) {
                    extend_add_kernel<C><<<(unsigned)(t1 - t0), dim3(64, 4), 0, st>>>(
                        F.ext_tiles.p + t0, F.p.p, F.u.p, F.f_off.p, F.sch_off.p, F.u_off.p, F.urel.p, ws, sch_child,
                        sch_l);
                    MWI_CHECK_LAUNCH();
                }
            }
            const int pmax = F.level_pmax[l];
            for (int k = 0; k < pmax; k += NB) {
                panel_diag_kernel<C, NB><<<nf, NB * 8, 0, st>>>(F.level_fronts.p, lo, k, F.p.p, F.u.p, F.f_off.p, ws,
                                                                perturbed);
                MWI_CHECK_LAUNCH();
                {
                    const int64_t r0 = ut.rptr[range], r1 = ut.rptr[range + 1];
                    if (r1 > r0) {
                        panel_rows_kernel<C, NB><<<(unsigned)(r1 - r0), 128, 0, st>>>(
                            ut.rtiles.p + r0, k, F.p.p, F.u.p, F.f_off.p, F.l_off.p, ws, lbuf);
                        MWI_CHECK_LAUNCH();
                    }
                }
                MWI_REQUIRE(range + 1 < ut.ptr.size() && range + 1 < ut.rptr.size(), MWI_EINVAL,
                            "internal: update tile list out of step");
                const int64_t t0 = ut.ptr[range], t1 = ut.ptr[range + 1];
                ++range;
                if (t1 > t0) {
                    update_kernel<C, TILE, NB><<<(unsigned)(t1 - t0), 256, 0, st>>>(
                        ut.tiles.p + t0, k, F.p.p, F.u.p, F.f_off.p, F.sch_off.p, F.l_off.p, ws, lbuf, sch_l);
                    MWI_CHECK_LAUNCH();
                }
            }
            {
                MWI_REQUIRE(end + 1 < ut.eptr.size(), MWI_EINVAL, "internal: update tile list out of step");
                const int64_t t0 = ut.eptr[end], t1 = ut.eptr[end + 1];
                ++end;
                if (t1 > t0) {
                    update_kernel<C, TILE, NB><<<(unsigned)(t1 - t0), 256, 0, st>>>(
                        ut.etiles.p + t0, -1, F.p.p, F.u.p, F.f_off.p, F.sch_off.p, F.l_off.p, ws, lbuf, sch_l);
                    MWI_CHECK_LAUNCH();
                }
            }
            finish_diag_kernel<C><<<nf, 128, 0, st>>>(F.level_fronts.p, lo, F.p.p, F.u.p, F.start.p, F.sub.p,
                                                      F.sub_off.p, F.f_off.p, ws, ws + F.ws_entries);
            MWI_CHECK_LAUNCH();
        }
    }
}

template void factorize_fronts<float2>(const FrontsDev&, const UpdateTiles&, const double2*, float2*,
                                       float2* const[2], float2*, int*, cudaStream_t);
template void factorize_fronts<double2>(const FrontsDev&, const UpdateTiles&, const double2*, double2*,
                                        double2* const[2], double2*, int*, cudaStream_t);

int factor_block_cols(bool fp32) { return fp32 ? FactorCfg<float2>::NB : FactorCfg<double2>::NB; }
int factor_tile_rows(bool fp32) { return fp32 ? FactorCfg<float2>::TILE : FactorCfg<double2>::TILE; }

}  // namespace mwi
