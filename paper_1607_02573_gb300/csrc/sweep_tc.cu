// ORAS sweeps on the fifth-generation tensor cores (tcgen05, sm_103a): the
// multifrontal forward and backward products of sweep.cu (the B_i^{-1} of
// Eq. ORAS applied to m right-hand sides at once, Section 3), with the factor
// panels streamed by bulk asynchronous copies into shared memory and the
// products accumulated in tensor memory.
//
// Factor layout ("tiled panels", written once per factorisation by
// pack_tiled_kernel).  The A operand is K-major (K contiguous in a line), and the
// two sweeps contract a front's
// f x p partitioned-inverse panel [L11^{-1}; -L21 L11^{-1}] over different
// indices -- the forward product over pivots, the backward one over rows --
// so the panel is stored twice, cut into 8 x 8 blocks (rows and pivots padded
// to multiples of 8 with zeros).  A block is two 256-byte planes (real parts,
// then imaginary parts), each 8 lines of 32 bytes in the 32-byte swizzled
// order of the tensor cores (16-byte chunk j of line r at chunk
// j ^ ((r >> 2) & 1)):
//   - forward copy: line = front row, 8 floats = pivots; blocks ordered
//     [pivot chunk][row group][plane], so one 8-pivot K step of a 128-row
//     tile is 16 consecutive blocks (row groups at the stride-byte offset);
//   - backward copy: line = pivot, 8 floats = front rows; blocks ordered
//     [row chunk][pivot group][plane].
// A stage of kKS K steps is at most kKS contiguous byte ranges, copied with
// cp.async.bulk.  The right-hand sides are the B operand as they lie in memory,
// N contiguous (MN-major): the TF32 form takes that in one layout only, the
// 128-byte swizzle of 32-byte atoms -- 128 bytes (32 real columns) per K row,
// 4 K rows per 512-byte atom, 32-byte chunk j of K row k at chunk j ^ (k & 3).
// A gathered row is two such 128-byte pieces, its 16-byte units copied straight
// to their places.
//
// Complex product as two real products.  With A = Ar + i Ai (the two planes)
// and the right-hand sides B stored as reals [k][2c + (0 re, 1 im)], the MMA
// computes Dr = Ar B and Di = Ai B (N = 64 real columns for 32 complex
// columns, TF32 inputs -- the tensor core reads the FP32 bits and drops the
// low 13 mantissa bits, see Rounding below -- FP32 accumulation); then
//   Re C(i, c) = Dr[i][2c] - Di[i][2c+1],  Im C(i, c) = Dr[i][2c+1] + Di[i][2c].
//
// Rounding.  The panels are rounded to the nearest TF32 value when they are
// packed.  The rows that the backward sweep reads are FP32 words biased by half a
// TF32 unit (tf32.h), so that the truncation rounds them to nearest as well: Z,
// which nothing else reads, and the pivot rows of Y that the backward tiles
// write, which come back biased and whose reader takes the bias off again
// (oras.cu).  The forward sweep's rows are truncated.
//
// Kernel: one launch for both sweeps over the whole tree, two CTAs per SM.
// Every CTA draws tiles (front, 128-row tile, 32-column chunk) from one list by
// an atomic counter: the forward tiles, deepest level first, then the backward
// ones, root level first, a level's tiles by subdomain and front, first
// children before second ones.  What a tile waits for comes earlier in the
// list, so it is done or being done by a running CTA whatever the number of
// CTAs that run at the same time:
//   - forward tile of a front: all forward tiles of its children, counted per
//     front by the epilogues (release) and polled by the gather warps (acquire),
//     which hand the order on to their other lanes and to the tile's epilogue;
//   - backward tile: all backward tiles of the parent (of the root: its own
//     forward tiles), which closes the chain over everything else it reads.
// The children add their update rows straight into the parent's pivot rows in
// Y, the first child, then the second (whose epilogue waits for the first
// child's count), so the sum has a fixed order; update rows that meet the
// parent's update rows go through upd.  (With the two children next to each
// other in the list the waits formed chains from CTA to CTA: 6.8 ms per
// application of 32 columns on 402,444 tets.)
// Why one launch: with a launch per level and direction (and one more for the
// extend-add of the pivot rows) every level ended in a partly filled last wave
// and began with the set-up of all CTAs; subdomains, whose levels are
// independent of each other, now overlap across levels.  Per application of 32
// columns on 402,444 tets, gather and scatter included: 1.87 -> 1.38 ms.
// Warp roles:
//   warp 0      streams the panel blocks by bulk copies, which depend on no
//               other tile
//   warp 1      owns the tensor memory (2 x 128 columns: accumulators double
//               buffered across tiles); one lane issues tcgen05.mma and commits
//   warps 2-3   wait for a tile's dependencies and gather the right-hand-side
//               rows into the B operand by 16-byte asynchronous copies (16 lanes
//               a row).  The chain of a stage -- free, gathered, multiplied --
//               sets its rate: with a K-major B, which took a transposition
//               through shared memory between the two, an application took
//               2.10 ms where this one took 1.82 (conversions to FP64 included)
//   warps 4-7   epilogue: tcgen05.ld, complex combine, D^{-1} scaling or
//               extend-add, global stores, the front's count
//   warp 8      draws the tiles, one ahead of warp 0 (a long tile does not hold
//               back one that others wait for): descriptor into the ring,
//               update-row indices into shared memory.  (Fetching the first part
//               of the tile's panel into L2 as well cost 1.75 against 1.55 ms.)
// Stages (per CTA, two CTAs per SM) form a ring shared by all tiles of the CTA,
// so loads of the next tile overlap the products and the epilogue of the
// current one.  The rows are copied in units of 16 bytes, so the engine needs an
// even number of columns.
// Every wait is bounded: on expiry the kernel records an error code, the other
// roles stop at their next wait, other CTAs at their next dependency wait, and
// the CTA lets its copies and products in flight land, frees its tensor memory
// and returns.
#include <algorithm>

#include "common.h"
#include "kernels.h"
#include "per_device.h"
#include "tf32.h"

namespace mwi {
namespace {

constexpr int kCtasPerSm = 2;
constexpr int kStages = 2;                  // stage ring per CTA
constexpr int kKS = 4;                      // K steps of 8 per stage
constexpr int kKRows = 8 * kKS;
constexpr int kAStage = kKS * 8192;         // K steps x 16 groups of 8 M lines x 2 planes x 256 B
constexpr int kBStage = kKRows * 256;       // two column groups x K rows x 128 B
constexpr int kStage = kAStage + kBStage;
constexpr int kUrCache = 1024;              // update-row indices of a backward tile kept in shared memory
// tiles that can be under way in one CTA, each of one stage at least: index
// buffers and descriptors (power of two) come round again after them
constexpr int kSurBufs = kStages + 1;
constexpr int kRing = 8;
static_assert(kRing >= kStages + 3, "descriptor ring");
constexpr int kThreads = 288;
constexpr int kTmemCols = 256;
constexpr int kSmemBytes =
    kStages * kStage + 1024 /* barriers */ + kRing * 128 + kSurBufs * kUrCache * 4 + 1024 /* alignment */;
static_assert((3 * kStages + 4 + 2 * kRing + kSurBufs + 1) * 8 + 8 <= 1024, "barriers");
static_assert(kSmemBytes * kCtasPerSm <= 228 * 1024 - 2048, "shared memory per SM");
constexpr int kWaitLimit = 1 << 24;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait on a phase; false if the CTA aborts or the limit expires
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* err,
                                          int code) {
    for (int it = 0; it < kWaitLimit; ++it) {
        if (mbar_try(bar, parity)) return true;  // try_wait suspends in hardware for a while
        if (*abort_flag) return false;
        if (it > (1 << 20)) __nanosleep(256);
    }
    *abort_flag = 1;
    atomicExch(err, code);
    return false;
}

// The same for a whole warp, which has to leave its loop as one, since its
// warp-wide instructions need all lanes, while lanes may see the abort at
// different times: they look together and take the decision by votes.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* err,
                                               int code) {
    for (int it = 0; it < kWaitLimit; ++it) {
        if (__all_sync(0xffffffffu, mbar_try(bar, parity))) return true;
        if (__any_sync(0xffffffffu, *abort_flag)) return false;
        if (it > (1 << 20)) __nanosleep(256);
    }
    *abort_flag = 1;
    atomicExch(err, code);
    return false;
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// shared-memory matrix descriptor: start, leading and stride byte offsets (>> 4),
// version 1 (bit 46), layout type at bits 61-63 (1 = 128-byte swizzle of 32-byte
// atoms, 6 = 32-byte swizzle).  K-major: stride offset between groups of 8
// lines, leading offset unused; MN-major: leading offset between groups of 32
// columns, stride offset between groups of 4 K rows
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo, uint32_t layout) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFF);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)layout << 61;
    return d;
}
constexpr uint32_t kSw128Base32 = 1, kSw32 = 6;

// instruction descriptor of kind::tf32: D FP32 (bits 4-5 = 1), A and B TF32
// (bits 7-9, 10-12 = 2), A K-major (bit 15 = 0), B MN-major (bit 16 = 1),
// N >> 3 at bits 17-22, M >> 4 at bits 24-28
__host__ __device__ constexpr uint32_t idesc_tf32(int M, int N) {
    return (1u << 4) | (2u << 7) | (2u << 10) | (1u << 16) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_tf32(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

// 32 consecutive accumulator columns of this warp's 32 lanes
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// 16 bytes global -> shared past L1, asynchronously (bytes = 0: zeros, nothing
// is read); copies_arrive: this thread's arrival on the barrier once its copies
// so far have landed
__device__ __forceinline__ void copy16(uint32_t dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void copies_arrive(uint32_t bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
// 32 bytes per access (sm_100 and later), 32-byte aligned; loads past L1
__device__ __forceinline__ void store32(float2* p, const float* v) {
    asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
                 "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                 : "memory");
}
__device__ __forceinline__ void load32(const float2* p, float* v) {
    asm volatile("ld.global.cg.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "l"(p)
                 : "memory");
}
__device__ __forceinline__ int ld_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release(int* p) {
    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(p) : "memory");
}
// bounded wait without the abort: for what is in flight when the CTA ends
__device__ __forceinline__ void mbar_drain(uint32_t bar, uint32_t parity) {
    for (int it = 0; it < (1 << 12); ++it)
        if (mbar_try(bar, parity)) break;
}

// bounded wait until *cnt >= target (one lane; dep_wait_warp for all), at most
// `polls` looks; false if the CTA aborts, another CTA has reported an error or the
// limit expires
__device__ __forceinline__ bool dep_wait(const int* cnt, int target, int polls, volatile int* abort_flag, int* err,
                                         int code) {
    for (int it = 0; it < polls; ++it) {
        if (ld_acquire(cnt) >= target) return true;
        if (*abort_flag) return false;
        if ((it & 63) == 63) {
            if (ld_acquire(err)) {
                *abort_flag = 1;
                return false;
            }
        }
        if (it > 64) __nanosleep(64);
    }
    *abort_flag = 1;
    atomicExch(err, code);
    return false;
}
// The same for a whole warp: each lane polls its own count (cnt = nullptr: none).
// A vote does not order memory; the __syncwarp() is what orders the other lanes'
// reads after a lane's acquire.
__device__ __forceinline__ bool dep_wait_warp(const int* cnt, int target, int polls, volatile int* abort_flag,
                                              int* err, int code) {
    const bool ok = !cnt || dep_wait(cnt, target, polls, abort_flag, err, code);
    const bool all = __all_sync(0xffffffffu, ok);
    __syncwarp();
    return all;
}

// Tile geometry shared by every role.  Forward: M = front rows row0..
// (row groups g0.., ng of them), K = pivots [0, min(p, row0 + 128)) in chunks
// of 8.  Backward: M = pivots row0.. (pivot groups g0..), K = front rows from
// row0 (the panel is zero above its diagonal) to f, in chunks of 8.  The
// chunks of a front's copy are cstride blocks apart.
struct TcGeom {
    int p, f, row0, g0, ng, k0, nk, nst, cstride;
    bool bwd;
};

__device__ __forceinline__ TcGeom tc_geom(int p, int f, int row0, bool bwd) {
    TcGeom g;
    g.p = p;
    g.f = f;
    g.row0 = row0;
    g.bwd = bwd;
    const int F8 = (f + 7) >> 3, P8 = (p + 7) >> 3;
    g.g0 = row0 >> 3;
    if (!bwd) {
        g.ng = min(16, F8 - g.g0);
        g.k0 = 0;
        g.nk = (min(p, row0 + 128) + 7) >> 3;
        g.cstride = F8;
    } else {
        g.ng = min(16, P8 - g.g0);
        g.k0 = row0 >> 3;
        g.nk = F8 - g.k0;
        g.cstride = P8;
    }
    g.nst = (g.nk + kKS - 1) / kKS;
    return g;
}

// number of the stage's K rows that hold data (the rest of its last K step is zero)
__device__ __forceinline__ int stage_rows(const TcGeom& G, int st) {
    const int lim = !G.bwd ? min(G.p, G.row0 + 128) - st * kKRows : G.f - (G.row0 + st * kKRows);
    return min(kKRows, lim);
}

// backward tiles keep their update-row indices in shared memory, if they fit
// beside the up to three that the copy's alignment brings along
__device__ __forceinline__ bool indices_cached(const TcGeom& G) {
    return G.bwd && G.f > G.p && G.f - G.p <= kUrCache - 3;
}

// a tile as the roles read it from the ring: the descriptor's words, then the
// chunk's first column and whether there is a tile
struct RingSlot {
    TcTile d;
    int c0, valid;
    int pad[32 - sizeof(TcTile) / 4 - 2];
};
static_assert(sizeof(RingSlot) == 128 && sizeof(TcTile) % 4 == 0, "one descriptor per 128 bytes");
constexpr int kTileWords = sizeof(TcTile) / 4;

__global__ void __launch_bounds__(kThreads, kCtasPerSm) sweep_tc_kernel(
    const TcTile* __restrict__ tiles, int ntiles, int nchunks, int* __restrict__ cnt,
    const int32_t* __restrict__ urows, const int2* __restrict__ asm2, const int32_t* __restrict__ pdst,
    const float* __restrict__ wt, const float2* __restrict__ dinv, float2* Y, float2* Z, float2* upd, int m,
    int polls, int* err) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                           ~(uintptr_t)1023);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * kStage);
    // bars: raw[kStages] (panel blocks landed), rows[kStages] (right-hand-side rows
    // landed), empty[kStages] (stage consumed), tfull[2], tempty[2], tile[kRing]
    // (descriptor written), sur[kSurBufs], begun (tile begun), deps[kRing] (the tile's
    // dependencies are met)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 3 * kStages + 4 + 2 * kRing + kSurBufs + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    RingSlot* ring = reinterpret_cast<RingSlot*>(smem + kStages * kStage + 1024);
    int32_t* sur = reinterpret_cast<int32_t*>(smem + kStages * kStage + 1024 + kRing * 128);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t sbase = smem_u32(smem);
    auto raw_bar = [&](int s) { return smem_u32(bars + s); };
    auto rows_bar = [&](int s) { return smem_u32(bars + kStages + s); };
    auto empty_bar = [&](int s) { return smem_u32(bars + 2 * kStages + s); };
    auto tfull_bar = [&](int b) { return smem_u32(bars + 3 * kStages + b); };
    auto tempty_bar = [&](int b) { return smem_u32(bars + 3 * kStages + 2 + b); };
    auto tile_bar = [&](int it) { return smem_u32(bars + 3 * kStages + 4 + (it & (kRing - 1))); };
    auto tile_par = [&](int it) { return (uint32_t)(it / kRing) & 1; };
    auto sur_bar = [&](int b) { return smem_u32(bars + 3 * kStages + 4 + kRing + b); };
    const uint32_t begun_bar = smem_u32(bars + 3 * kStages + 4 + kRing + kSurBufs);
    auto deps_bar = [&](int it) {
        return smem_u32(bars + 3 * kStages + 4 + kRing + kSurBufs + 1 + (it & (kRing - 1)));
    };

    // stale shared memory must be finite: the MMA reads whole 128-row groups of
    // panel blocks, and the columns and rows without data go nowhere
    for (int i = threadIdx.x; i < kStages * kStage / 16; i += kThreads)
        reinterpret_cast<uint4*>(smem)[i] = make_uint4(0, 0, 0, 0);
    fence_proxy_async();
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(raw_bar(s), 1);       // the copy lane, with the stage's transaction bytes
            mbar_init(rows_bar(s), 64);     // the lanes of the gather warps
            mbar_init(empty_bar(s), 1);     // tcgen05.commit
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(tfull_bar(b), 1);
            mbar_init(tempty_bar(b), 4);    // the 4 epilogue warps
        }
        for (int b = 0; b < kSurBufs; ++b) mbar_init(sur_bar(b), 1);
        for (int b = 0; b < kRing; ++b) mbar_init(tile_bar(b), 1);
        for (int b = 0; b < kRing; ++b) mbar_init(deps_bar(b), 1);
        mbar_init(begun_bar, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const int total = ntiles * nchunks;

    // what a role has under way, for the end of a CTA that gives up: stages copied or
    // multiplied, tiles multiplied, index buffers filled
    long long g = 0;
    int done = 0, nsur = 0;
    bool ok = true;

    if (warp == 0) {
        // ---------------- panel blocks
        for (int it = 0; ok; ++it) {
            if (!mbar_wait_warp(tile_bar(it), tile_par(it), abort_flag, err, 8)) break;
            const RingSlot* slot = ring + (it & (kRing - 1));
            if (!slot->valid) break;
            const TcGeom G = tc_geom(slot->d.p, slot->d.f, slot->d.row0, slot->d.bwd != 0);
            const float* P = wt + slot->d.a_off;
            const uint32_t a_bytes = (uint32_t)G.ng * 512u;
            for (int st = 0; st < G.nst; ++st, ++g) {
                const int s = (int)(g % kStages);
                const uint32_t ph = (uint32_t)((g / kStages) & 1);
                if (!(ok = mbar_wait_warp(empty_bar(s), ph ^ 1, abort_flag, err, 1))) break;
                // the barrier's one arrival keeps the phase open, whichever comes first, the
                // count of the expected bytes or another lane's copy
                const int k0 = G.k0 + st * kKS, nk = min(kKS, G.k0 + G.nk - k0);
                if (lane == 0) mbar_arrive_tx(raw_bar(s), a_bytes * nk);
                if (lane < nk)
                    bulk_g2s(sbase + s * kStage + lane * 8192, P + ((int64_t)(k0 + lane) * G.cstride + G.g0) * 128,
                             a_bytes, raw_bar(s));
                if (st == 0 && lane == 0) mbar_arrive(begun_bar);
            }
        }
    } else if (warp == 1) {
        // ---------------- tensor-core products
        if (lane == 0) {
            constexpr uint32_t kIdesc = idesc_tf32(128, 64);
            for (int it = 0; ok; ++it) {
                if (!mbar_wait(tile_bar(it), tile_par(it), abort_flag, err, 8)) break;
                const RingSlot* slot = ring + (it & (kRing - 1));
                if (!slot->valid) break;
                const TcGeom G = tc_geom(slot->d.p, slot->d.f, slot->d.row0, slot->d.bwd != 0);
                const int buf = it & 1;
                if (!(ok = mbar_wait(tempty_bar(buf), ((it >> 1) & 1) ^ 1, abort_flag, err, 2))) break;
                tc_fence_after();
                const uint32_t dr = tmem + buf * 128, di = dr + 64;
                for (int st = 0; st < G.nst; ++st, ++g) {
                    const int s = (int)(g % kStages);
                    const uint32_t ph = (uint32_t)((g / kStages) & 1);
                    if (!(ok = mbar_wait(raw_bar(s), ph, abort_flag, err, 3))) break;
                    if (!(ok = mbar_wait(rows_bar(s), ph, abort_flag, err, 4))) break;
                    fence_proxy_async();
                    tc_fence_after();
                    const uint32_t a0 = sbase + s * kStage, b0 = a0 + kAStage;
                    const int nk = min(kKS, G.nk - st * kKS);
                    for (int c = 0; c < nk; ++c) {
                        // B: K step c = two 512-byte atoms in each of the two column groups
                        const uint64_t bd = smem_desc(b0 + c * 1024, kKRows * 128, 512, kSw128Base32);
                        const uint32_t acc = (st > 0 || c > 0) ? 1u : 0u;
                        mma_tf32(dr, smem_desc(a0 + c * 8192, 16, 512, kSw32), bd, kIdesc, acc);
                        mma_tf32(di, smem_desc(a0 + c * 8192 + 256, 16, 512, kSw32), bd, kIdesc, acc);
                    }
                    mma_commit(empty_bar(s));
                }
                if (!ok) break;
                mma_commit(tfull_bar(buf));
                ++done;
            }
        }
    } else if (warp < 4) {
        // ---------------- right-hand-side rows into the B operand: this warp's half
        // of the stage's K rows
        constexpr int kMine = kKRows / 4;  // row pairs of a stage per warp
        const int seg = lane & 15, half = lane >> 4, first = (warp - 2) * (kKRows / 2) + half;
        for (int it = 0; ok; ++it) {
            if (!mbar_wait_warp(tile_bar(it), tile_par(it), abort_flag, err, 8)) break;
            const RingSlot* slot = ring + (it & (kRing - 1));
            if (!slot->valid) break;
            const TcGeom G = tc_geom(slot->d.p, slot->d.f, slot->d.row0, slot->d.bwd != 0);
            const int c0 = slot->c0, nc = min(32, m - c0);
            // rows in units of 16 bytes from the first of this lane
            const uint32_t ld = (uint32_t)m >> 1;
            const float4* own = reinterpret_cast<const float4*>((G.bwd ? Z : Y) + slot->d.rowbase * m + c0) + seg;
            const float4* anc = reinterpret_cast<const float4*>(Y + slot->d.sbase * m + c0) + seg;
            const int32_t* iu = urows + slot->d.u_off;
            const int kfirst = G.bwd ? G.row0 : 0;
            if (indices_cached(G)) {
                if (!mbar_wait_warp(sur_bar(nsur % kSurBufs), (uint32_t)(nsur / kSurBufs) & 1, abort_flag, err, 6))
                    break;
                iu = sur + (nsur % kSurBufs) * kUrCache + (slot->d.u_off & 3);
                ++nsur;
            }
            // the rows are other tiles' results; the epilogue, which reads such rows
            // as well, learns from warp 2 that they are there
            const int dep = lane == 0 ? slot->d.dep0 : (lane == 1 ? slot->d.dep1 : -1);
            const int need = lane == 0 ? slot->d.need0 : slot->d.need1;
            if (!dep_wait_warp(dep >= 0 ? cnt + dep : nullptr, need * nchunks, polls, abort_flag, err, 7)) break;
            if (warp == 2 && lane == 0) mbar_arrive(deps_bar(it));
            for (int st = 0; st < G.nst; ++st, ++g) {
                const int s = (int)(g % kStages);
                const uint32_t ph = (uint32_t)((g / kStages) & 1);
                const int nv = stage_rows(G, st);
                const int nz = min(kKRows, (nv + 7) & ~7);  // rows that the products read
                const uint32_t R = sbase + s * kStage + kAStage + (seg >> 3) * (kKRows * 128) + (seg & 1) * 16;
                if (!(ok = mbar_wait_warp(empty_bar(s), ph ^ 1, abort_flag, err, 1))) break;
                if (seg < (nc >> 1)) {
                    // all addresses before the copies, which the compiler keeps in order
                    // with the index loads
                    const float4* src[kMine];
#pragma unroll
                    for (int j = 0; j < kMine; ++j) {
                        const int r = min(first + 2 * j, nv - 1);  // row of the stage
                        const int k = kfirst + st * kKRows + r;
                        const bool piv = !G.bwd || k < G.p;
                        const uint32_t row = piv ? k : iu[k - G.p];
                        src[j] = (piv ? own : anc) + (uint64_t)row * ld;
                    }
#pragma unroll
                    for (int j = 0; j < kMine; ++j) {
                        const int r = first + 2 * j;
                        if (r < nz)
                            copy16(R + r * 128 + ((((seg & 7) >> 1) ^ (r & 3)) << 5), src[j], r < nv ? 16u : 0u);
                    }
                }
                copies_arrive(rows_bar(s));
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else if (warp == 8) {
        // ---------------- tiles.  A ring slot or an index buffer is free when it
        // comes round again: tile i is drawn after the first panel blocks of tile
        // i - 1 are under way, i.e. after the products of the stage kStages before,
        // which is of tile i - 1 - kStages or later: that tile's rows are gathered,
        // and its accumulator waited for the epilogue of the tile two before.
        for (int it = 0;; ++it) {
            if (it > 0 && !mbar_wait_warp(begun_bar, (uint32_t)(it - 1) & 1, abort_flag, err, 10)) break;
            const int tk = __shfl_sync(0xffffffffu, lane == 0 ? atomicAdd(cnt, 1) : 0, 0);
            const int ti = tk / nchunks;
            RingSlot* slot = ring + (it & (kRing - 1));
            uint32_t w = 0;
            if (lane < kTileWords) w = tk < total ? reinterpret_cast<const uint32_t*>(tiles + ti)[lane] : 0u;
            else if (lane == kTileWords) w = (uint32_t)((tk - ti * nchunks) * 32);
            else if (lane == kTileWords + 1) w = tk < total ? 1u : 0u;
            reinterpret_cast<uint32_t*>(slot)[lane] = w;
            __syncwarp();
            if (lane == 0) mbar_arrive(tile_bar(it));
            if (tk >= total) break;
            const TcGeom G = tc_geom(slot->d.p, slot->d.f, slot->d.row0, slot->d.bwd != 0);
            if (indices_cached(G) && lane == 0) {
                // one bulk copy, the start rounded down to 16 bytes (the list is padded at its end)
                const int off = (int)(slot->d.u_off & 3);
                const uint32_t bar = sur_bar(nsur % kSurBufs), bytes = (uint32_t)((G.f - G.p + off + 3) / 4) * 16u;
                fence_proxy_async();
                mbar_arrive_tx(bar, bytes);
                bulk_g2s(smem_u32(sur + (nsur % kSurBufs) * kUrCache), urows + (slot->d.u_off - off), bytes, bar);
            }
            nsur += indices_cached(G) ? 1 : 0;
        }
    } else {
        // ---------------- epilogue
        const int lg = warp & 3;  // tensor-memory lane group of this warp
        const int i = lg * 32 + lane;
        for (int it = 0;; ++it) {
            if (!mbar_wait_warp(tile_bar(it), tile_par(it), abort_flag, err, 8)) break;
            const RingSlot* slot = ring + (it & (kRing - 1));
            if (!slot->valid) break;
            const TcTile d = slot->d;
            const bool bwd = d.bwd != 0;
            const int c0 = slot->c0, nc = min(32, m - c0);
            const int buf = it & 1;
            // loads that do not depend on the product, issued before waiting for it
            const int gi = d.row0 + i;
            float2 dv = make_float2(0.f, 0.f);
            int2 src = make_int2(-1, -1);
            float2* dst = nullptr;
            bool add = false;  // dst holds rows to add to: a pivot row of the parent
            if (gi < d.p) {
                if (!bwd) dv = dinv[d.rowbase + gi];
                dst = (bwd ? Y : Z) + (d.rowbase + gi) * m + c0;
            } else if (!bwd && gi < d.f) {
                src = asm2[d.asm_base + gi];
                const int pd = pdst[d.upd_row + gi - d.p];
                add = pd >= 0;
                dst = add ? Y + (int64_t)pd * m + c0 : upd + (d.upd_row + gi - d.p) * m + c0;
            }
            if (d.sib >= 0 && __any_sync(0xffffffffu, add)) {
                // the second child adds to the parent's rows after the first
                if (!dep_wait_warp(lane == 0 ? cnt + d.sib : nullptr, d.needs * nchunks, polls, abort_flag, err,
                                   9))
                    break;
            }
            // the second is past already (the product came after it): it orders this lane's
            // reads of the children's rows after the gather warp's acquire
            if (!mbar_wait_warp(tfull_bar(buf), (it >> 1) & 1, abort_flag, err, 5)) break;
            if (!mbar_wait_warp(deps_bar(it), tile_par(it), abort_flag, err, 11)) break;
            tc_fence_after();
            const uint32_t t0 = tmem + ((uint32_t)(lg * 32) << 16) + buf * 128;
            // whole 32-byte accesses: a lane's row is a line of its own, so an access
            // of the warp takes 32 passes whatever its width (32 columns, 402,444 tets:
            // 1.82 -> 1.75 ms; 64 columns 2.93 -> 2.72 ms)
            const bool wide = nc == 32 && (m & 3) == 0;
            // one or two halves of 16 complex columns: tensor-memory loads, combine,
            // D^{-1} or the rows to add, stores; the accumulator is released once
            // the last half is in registers.  Rows that other tiles of this launch
            // have written are read past L1.  The two halves share one copy of the
            // body: two in a row are more than the instruction cache takes beside the
            // other roles (32 columns, 402,444 tets: 1.65 ms per application, 1.54
            // with one).  At most 16 columns get a copy of their own, without the
            // loop (14 columns, 19k tets: 202 -> 174 us; one column, 7,392 tets:
            // 125 -> 120 us).
            auto half = [&](int h) {
                __syncwarp();  // lanes without a row left the first half early
                float o[32];
                {
                    float dr[32], di[32];
                    tmem_ld32(t0 + h * 32, dr);
                    tmem_ld32(t0 + 64 + h * 32, di);
                    tmem_ld_wait();
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        o[2 * q] = dr[2 * q] - di[2 * q + 1];
                        o[2 * q + 1] = dr[2 * q + 1] + di[2 * q];
                    }
                }
                if (16 * (h + 1) >= nc) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(tempty_bar(buf));
                }
                const int cb = 16 * h;  // first complex column of the half
                if (!dst) return;
                if (gi < d.p && !bwd) {
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        const float re = o[2 * q], im = o[2 * q + 1];
                        o[2 * q] = re * dv.x - im * dv.y;
                        o[2 * q + 1] = re * dv.y + im * dv.x;
                    }
                }
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const float2* a = k == 2 ? (add ? dst + cb : nullptr)
                                             : ((k ? src.y : src.x) >= 0
                                                    ? upd + (int64_t)(k ? src.y : src.x) * m + c0 + cb
                                                    : nullptr);
                    if (!a) continue;
                    if (wide) {
                        float v[32];
#pragma unroll
                        for (int q = 0; q < 4; ++q) load32(a + 4 * q, v + 8 * q);
#pragma unroll
                        for (int q = 0; q < 32; ++q) o[q] += v[q];
                        continue;
                    }
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        if (cb + 2 * q < nc) {
                            const float4 v = __ldcg(reinterpret_cast<const float4*>(a) + q);
                            o[4 * q] += v.x;
                            o[4 * q + 1] += v.y;
                            o[4 * q + 2] += v.z;
                            o[4 * q + 3] += v.w;
                        }
                }
                if (gi < d.p) {  // operands of the backward sweep, Z or Y
#pragma unroll
                    for (int q = 0; q < 32; ++q) o[q] = tf32_bias(o[q]);
                }
                if (wide) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) store32(dst + cb + 4 * q, o + 8 * q);
                    return;
                }
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (cb + 2 * q < nc)
                        reinterpret_cast<float4*>(dst + cb)[q] =
                            make_float4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
                        };
            if (nc <= 16) {
                half(0);
            } else {
#pragma unroll 1
                for (int h = 0; h < 2; ++h) half(h);
            }
            __syncwarp();
            if (lane == 0) red_release(cnt + d.cnt);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        // copies still on their way land before the CTA gives its shared memory back,
        // products before it frees the tensor memory (every role has stopped; the flag
        // is the same for all threads)
        if (lane == 0) {
            for (long long q = g > kStages ? g - kStages : 0; q < g; ++q) {
                const uint32_t ph = (uint32_t)((q / kStages) & 1);
                if (warp == 0) mbar_drain(raw_bar((int)(q % kStages)), ph);
                if (warp == 1) mbar_drain(empty_bar((int)(q % kStages)), ph);
            }
            for (int q = max(0, done - 2); q < done; ++q) mbar_drain(tfull_bar(q & 1), (uint32_t)(q >> 1) & 1);
            if (warp == 8)
                for (int q = max(0, nsur - kSurBufs); q < nsur; ++q)
                    mbar_drain(sur_bar(q % kSurBufs), (uint32_t)(q / kSurBufs) & 1);
        }
        __syncthreads();
    }
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
    }
}

// One block per (front, 32-row block): the block's panel rows, for every
// 8-pivot chunk, into both tiled copies (layout in the header comment).
__device__ __forceinline__ int swz32(int line, int e) { return line * 8 + ((((e >> 2) ^ ((line >> 2) & 1)) << 2) | (e & 3)); }

__global__ void __launch_bounds__(256) pack_tiled_kernel(const int2* __restrict__ blocks,
                                                         const int64_t* __restrict__ f_off,
                                                         const int64_t* __restrict__ t_off,
                                                         const int32_t* __restrict__ P, const int32_t* __restrict__ U,
                                                         const float2* __restrict__ ws, float* __restrict__ wt,
                                                         int64_t bwd_base) {
    const int2 bl = blocks[blockIdx.x];  // (front, 32-row block)
    const int s = bl.x;
    const int p = P[s], f = p + U[s];
    const int F8 = (f + 7) >> 3, P8 = (p + 7) >> 3;
    const float2* L = ws + f_off[s];
    float* Tf = wt + t_off[s];
    float* Tb = wt + bwd_base + t_off[s];
    const int e = threadIdx.x >> 5, rr = threadIdx.x & 31;  // pivot in its chunk, row in the block
    const int row = bl.y * 32 + rr;
    if ((row >> 3) >= F8) return;
    const int rg = row >> 3, rl = row & 7;
    for (int kc = 0; kc < P8; ++kc) {
        const int k = kc * 8 + e;
        float2 v = (k < p && row < f) ? L[(int64_t)k * f + row] : make_float2(0.f, 0.f);
        v = make_float2(tf32_round(v.x), tf32_round(v.y));
        float* bf = Tf + ((int64_t)kc * F8 + rg) * 128;   // forward: line = row, element = pivot
        bf[swz32(rl, e)] = v.x;
        bf[64 + swz32(rl, e)] = v.y;
        float* bb = Tb + ((int64_t)rg * P8 + kc) * 128;   // backward: line = pivot, element = row
        bb[swz32(e, rl)] = v.x;
        bb[64 + swz32(e, rl)] = v.y;
    }
}

}  // namespace

// floats of one tiled copy of a front (8 x 8 blocks, two planes)
int64_t tiled_panel_floats(int p, int f) { return (int64_t)((f + 7) / 8) * ((p + 7) / 8) * 128; }

void pack_tiled(const int2* blocks, int64_t nblocks, const int64_t* f_off, const int64_t* t_off, const int32_t* P,
                const int32_t* U, const float2* ws, float* wt, int64_t bwd_base, cudaStream_t st) {
    for (int64_t b = 0; b < nblocks; b += 65535 * 64) {
        const int64_t n = std::min<int64_t>(nblocks - b, 65535 * 64);
        pack_tiled_kernel<<<(unsigned)n, 256, 0, st>>>(blocks + b, f_off, t_off, P, U, ws, wt, bwd_base);
        MWI_CHECK_LAUNCH();
    }
}

// CTAs of a launch on the current device, and the kernel's shared memory allowed there
static int sweep_tc_ctas() {
    static PerDevice<int> ctas;
    const int dev = current_device();
    return ctas.get(dev, [dev] {
        int sms = 0;
        MWI_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        MWI_CUDA(cudaFuncSetAttribute(sweep_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes));
        return std::max(1, sms * kCtasPerSm);
    });
}

// both sweeps; cnt holds F.tc_counts() zeros; the rows of Y come back biased (tf32.h)
void sweep_tc_solve(const FrontsDev& F, int m, const float* wt, const float2* dinv, float2* Y, float2* Z,
                    float2* upd, int* cnt, int polls, int* err, cudaStream_t st) {
    const int ctas = sweep_tc_ctas();
    const int nchunks = (m + 31) / 32;
    const int64_t total = F.tc_ntiles * nchunks;
    MWI_REQUIRE(total + 2 * ctas < ((int64_t)1 << 31), MWI_EINVAL, "too many sweep tiles");
    if (total <= 0) return;
    const int grid = (int)std::min<int64_t>(total, ctas);
    sweep_tc_kernel<<<grid, kThreads, kSmemBytes, st>>>(F.tc_tiles.p, (int)F.tc_ntiles, nchunks, cnt, F.urows.p,
                                                        F.asm2.p, F.pdst.p, wt, dinv, Y, Z, upd, m, polls, err);
    MWI_CHECK_LAUNCH();
}

}  // namespace mwi
