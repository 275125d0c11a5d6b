// k_trsv.cu -- z = M^{-1} r for the RAS/ILU(k) preconditioner (Sections
// 2.5-2.6): for every RAS block, gather r on V_b, solve L_b y = r_b level by
// level (Eq. 11, Algorithm 3), solve U_b z = y level by level, write z on the
// rows the block owns.
//
// Design for sm_103a.  Each RAS block is solved by one CTA, or by a chain of
// P CTAs of one thread-block cluster ("parts": contiguous ranges of the
// block's rows, see trsv_layout.cpp).  A CTA walks its "program": its rows of
// every level of L_b, then of U_b, packed level-major into chunks (a chunk
// holds rows of one level only; rows inside a level are independent).  A
// chunk is one contiguous byte range in HBM holding, for its rows, the factor
// entries (value, dependency slot), the source index of the right-hand side,
// for U the destination row and the inverted diagonal, and for rows a
// neighbouring part reads, the slot they go to there.  Two chunk formats:
//   - fixed-slot (every row padded to one width FW <= 8): each thread's data
//     sits at a compile-time offset from the stage, and one set of solving
//     warps copies its rows of the next chunk into registers while the other
//     set solves the current one -- a level's critical path is then the ring
//     loads, the chain and the barrier;
//   - generic (wider rows): per-warp widths, rows solved from shared memory.
// Nothing on a level's critical path waits for HBM:
//   - an issuer warp streams chunks into a ring of shared-memory stages with
//     cp.async.bulk (the TMA bulk-copy engine, evict-first in L2) completing
//     on mbarriers, S chunks ahead of the solving warps;
//   - three gatherer warps, taking chunks in turn, gather each landed chunk's
//     right-hand sides (L pass: from r; U pass: from the L results, once the
//     L pass is complete) with 4- or 8-byte cp.async, ahead of the solving
//     warps, and hand the chunk over (an mbarrier per stage) once the copies
//     have completed and the neighbouring parts have completed the chunks its
//     thresholds name;
//   - solved values of the last few levels live in a shared-memory ring
//     indexed by level-major position (the setup checks that every
//     dependency of a chunk lies within the ring's window; passes whose
//     window does not fit read dependencies from the global scratch); values
//     a neighbouring part reads are also stored straight into that part's
//     import ring (distributed shared memory);
//   - a signaller warp forwards the completed-chunk count to the neighbouring
//     parts (a release at cluster scope, then the count stored into their
//     shared memory), off the solving warps' path.
// Levels are separated by a barrier of the solving warps only -- no
// grid-wide synchronisation.  Every wait is bounded: a wait that runs out
// sets the device error word, one thread waits (bounded) for the copies still
// in flight, and the CTA returns.
#include <type_traits>

#include "per_device.h"
#include "ptx.cuh"
#include "reduce.cuh"

namespace hec {

// Shared memory of one CTA: S stages, S right-hand-side slots of kThreads
// values, the ring (own and import slots: ring_slots in all), 2 S + 1
// mbarriers and two progress counters.  vbytes: 8 (FP64) or 4 (FP32).
size_t trsv_smem_bytes(int stage_bytes, int nstages, int ring_slots, int vbytes)
{
    const size_t ring = ((size_t)ring_slots * vbytes + 7) & ~(size_t)7;
    return (size_t)stage_bytes * nstages + (size_t)nstages * kThreads * vbytes + ring +
           (size_t)(2 * nstages + 1) * sizeof(uint64_t) + 2 * sizeof(uint32_t);
}

// Gatherer warps of a CTA: they take the chunks in turn and keep up to
// kGatherDepth chunks' right-hand-side gathers in flight each.  Two, three and
// four of them, FP64 / FP32 apply in us: 128^3 ILU(1) 325 / 290, 318 / 231,
// 320 / 234; 96^3 ILU(0) 171 / 178, 151 / 150, 153 / 150; 40^3 ILU(0) in 4
// blocks 84 / 96, 72 / 82, 72 / 82.
constexpr int kGatherers = 3;
constexpr int kGatherDepth = 2;

constexpr int kMaxStages = 16; // of the streamed kernel
// Shared memory that the stages leave: with all but 1 KB in stages, copies run
// further ahead than the solving warps need and the FP64 applies are slower
// (101^3 ILU(1) 461 us, 437 so; 82^3 ILU(0) 257 and 237; FP32 within 2% but for
// 101^3, 229 and 213).
constexpr int kLeaveFree = 24 * 1024;

int trsv_stages_for(int stage_bytes, int ring_slots, int vbytes)
{
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        optin = 227 * 1024;
    optin -= kLeaveFree; // and its own static shared memory
    int S = kMaxStages;
    while (S > 3 && trsv_smem_bytes(stage_bytes, S, ring_slots, vbytes) > (size_t)optin)
        --S;
    return S;
}

// ------------------------------------------------------------------ debug build
// Compiled with HEC_DEBUG, the kernel checks what it reads before it uses it:
// every chunk's header against the position the program has reached, every
// gathered index against the array it indexes, every dependency slot against
// the ring.  A failed check records the first violation (code, program,
// chunk, thread, value, bound), sets the error word to HEC_ERR_DEBUG and
// skips the access; nothing traps.
__device__ int g_trsv_debug[8];

#ifdef HEC_DEBUG
__device__ __noinline__ void debug_fail(int *err, int code, int c, int val, int bound)
{
    if (atomicCAS(&g_trsv_debug[0], 0, code) == 0) {
        g_trsv_debug[1] = (int)blockIdx.x;
        g_trsv_debug[2] = c;
        g_trsv_debug[3] = (int)threadIdx.x;
        g_trsv_debug[4] = val;
        g_trsv_debug[5] = bound;
    }
    atomicExch(err, HEC_ERR_DEBUG);
}
#define HEC_CHECK(cond, code, c, val, bound)                                                     \
    ((cond) ? true : (debug_fail(a.err, (code), (c), (int)(val), (int)(bound)), false))
#else
#define HEC_CHECK(cond, code, c, val, bound) true
#endif

// Drain bound for copies already issued when a wait ran out: copies complete
// in microseconds, this only guarantees that the CTA never waits forever.
constexpr long long kDrainPolls = 1ll << 24;

// A wait ran out: the handle's error word, and the end of the solve that this
// apply is part of -- its loop would otherwise go on to its budget of steps,
// each with the same wait.
__device__ __forceinline__ void report_timeout(const TrsvArgs &a)
{
    atomicExch(a.err, HEC_ERR_TIMEOUT);
    if (a.st) {
        a.st->err = HEC_ERR_TIMEOUT;
        a.st->done = 1;
    }
}

// Polls (with a pause between them) until the progress counter of a neighbouring
// part reaches `need`; `seen` is the value seen last.
__device__ __forceinline__ bool progress_wait(const uint32_t *ctr, int &seen, int need,
                                              long long limit)
{
    if (seen >= need || (seen = (int)ld_acquire_cluster_u32(ctr)) >= need)
        return true;
    const long long t0 = clock64();
    for (long long it = 1; it < limit && clock64() - t0 < kWaitCycles; ++it) {
        __nanosleep(32);
        if ((seen = (int)ld_acquire_cluster_u32(ctr)) >= need)
            return true;
    }
    return false;
}

// A chunk in shared memory (layout written by trsv_layout.cpp; T is the
// value type, double or float):
//   [0, 16)   nrows, nwarps, first position, flags (bit 0: U pass, bit 1: exports)
//   [16, 48)  width of every warp's segment
//   [48, 80)  byte offset of every warp's segment
//   [80, 96)  byte offsets of src, dst, dinv, exp
//   [96, 112) need_prev, need_next: completed chunks of part p - 1 / p + 1 to wait for
//   per warp w < nwarps: val[width_w][stride_w] (T), dep[width_w][stride_w] (int32),
//     stride_w = 32 for a full warp, the row count rounded up to 4 for the last one
//   src[r32(nrows)] (int32); for U: dst[r32(nrows)] (int32), dinv[r32(nrows)] (T);
//   with exports: exp[r32(nrows)] (int32), the row's slot in the neighbour's ring
// A dependency is a slot of the ring in ring mode (own values below R,
// imported ones from R on), else a position in the block's global scratch.
constexpr int kWarpRows = 32;
constexpr int kMaxWarps = kThreads / kWarpRows;
constexpr int kFeedThreads = 32 * (kGatherers + 2); // issuer, gatherers and the signaller

__device__ __forceinline__ int seg_stride(int w, int nrows)
{
    const int left = nrows - w * kWarpRows;
    return left >= kWarpRows ? kWarpRows : (left + 3) & ~3;
}

template <class T> struct ChunkView {
    int nrows, nwarps, base;
    bool upass, exports;
    const int *src, *dst, *exp;
    const T *dinv;
};

template <class T> __device__ __forceinline__ ChunkView<T> view_chunk(const unsigned char *ch)
{
    ChunkView<T> v;
    const int4 hdr = *reinterpret_cast<const int4 *>(ch);
    const int4 off = *reinterpret_cast<const int4 *>(ch + 16 + 8 * kMaxWarps);
    v.nrows = hdr.x;
    v.nwarps = hdr.y;
    v.base = hdr.z;
    v.upass = (hdr.w & 1) != 0;
    v.exports = (hdr.w & 2) != 0;
    v.src = reinterpret_cast<const int *>(ch + off.x);
    v.dst = reinterpret_cast<const int *>(ch + off.y);
    v.dinv = reinterpret_cast<const T *>(ch + off.z);
    v.exp = reinterpret_cast<const int *>(ch + off.w);
    return v;
}

// The segment of warp w: entry k of lane l at val[k * stride + l], dep[k * stride + l].
template <class T> struct Segment {
    int width, stride;
    const T *val;
    const int *dep;
};

template <class T>
__device__ __forceinline__ Segment<T> warp_segment(const unsigned char *ch, int nrows, int w)
{
    const int *hdr = reinterpret_cast<const int *>(ch);
    Segment<T> g;
    g.width = hdr[4 + w];
    g.stride = seg_stride(w, nrows);
    g.val = reinterpret_cast<const T *>(ch + hdr[4 + kMaxWarps + w]);
    g.dep = reinterpret_cast<const int *>(g.val + (size_t)g.width * g.stride);
    return g;
}

// s - sum_k val[k] * y[dep[k]] for one row in ascending column order (y: the
// ring slot dep[k], or the global-scratch position dep[k]), width W
// known at compile time: every shared-memory load of the row is issued before
// the first multiply.  One accumulator: in FP64 the pipe's throughput, not
// the 64-cycle latency of a dependent DFMA, bounds a level once several warps
// are busy, and a second accumulator would cost one more FP64 add per row.
template <int W, bool RING, class T>
__device__ __forceinline__ T row_solve(const Segment<T> &g, int lane, const T *ring, const T *gdep,
                                       T s)
{
    if constexpr (W == 0) {
        return s;
    } else {
        T l[W], y[W];
        int d[W];
#pragma unroll
        for (int k = 0; k < W; ++k) {
            l[k] = g.val[k * g.stride + lane];
            d[k] = g.dep[k * g.stride + lane];
        }
#pragma unroll
        for (int k = 0; k < W; ++k)
            y[k] = RING ? ring[d[k]] : gdep[d[k]];
#pragma unroll
        for (int k = 0; k < W; ++k)
            s = fma(-l[k], y[k], s);
        return s;
    }
}

template <bool RING, class T>
__device__ __forceinline__ T row_solve_any(const Segment<T> &g, int lane, const T *ring,
                                           const T *gdep, T s)
{
    switch (g.width) {
    case 0: return s;
    case 1: return row_solve<1, RING>(g, lane, ring, gdep, s);
    case 2: return row_solve<2, RING>(g, lane, ring, gdep, s);
    case 3: return row_solve<3, RING>(g, lane, ring, gdep, s);
    case 4: return row_solve<4, RING>(g, lane, ring, gdep, s);
    case 5: return row_solve<5, RING>(g, lane, ring, gdep, s);
    case 6: return row_solve<6, RING>(g, lane, ring, gdep, s);
    case 7: return row_solve<7, RING>(g, lane, ring, gdep, s);
    case 8: return row_solve<8, RING>(g, lane, ring, gdep, s);
    default: {
        // wide rows: loads in blocks of 8 entries
        int k = 0;
        for (; k + 8 <= g.width; k += 8) {
            T l[8], y[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                l[q] = g.val[(k + q) * g.stride + lane];
                const int d = g.dep[(k + q) * g.stride + lane];
                y[q] = RING ? ring[d] : gdep[d];
            }
#pragma unroll
            for (int q = 0; q < 8; ++q)
                s = fma(-l[q], y[q], s);
        }
        for (; k < g.width; ++k) {
            const int d = g.dep[k * g.stride + lane];
            s = fma(-g.val[k * g.stride + lane], RING ? ring[d] : gdep[d], s);
        }
        return s;
    }
    }
}

// Barrier of the NT solving threads only (named barrier 1), AND-reducing a flag.
template <int NT> __device__ __forceinline__ int solvers_sync_and(int flag)
{
    int all;
    asm volatile("{\n\t.reg .pred p, q;\n\t"
                 "setp.ne.s32 p, %1, 0;\n\t"
                 "barrier.cta.red.and.pred q, 1, %2, p;\n\t"
                 "selp.s32 %0, 1, 0, q;\n\t}"
                 : "=r"(all)
                 : "r"(flag), "n"(NT)
                 : "memory");
    return all;
}

#ifdef HEC_DEBUG
// Barrier of one set of solving warps (named barriers 2 and 3).
__device__ __forceinline__ void solvers_set_sync(int set)
{
    asm volatile("bar.sync %0, %1;" ::"r"(2 + set), "n"(kThreads) : "memory");
}
#endif

// Plain barrier of the NT solving threads (named barrier 1).  Measured on
// GB300: 19 cycles for 4 warps, the AND-reducing form 60; so the two-set loops
// use this one.  They do not leave early on a failed wait: it sets a shared
// word, and from then on a set loads nothing more, so the remaining levels
// are barriers only.  bar.sync is an aligned barrier, counted by the warp: a
// warp that reached it in two parts would be counted twice, and the set would
// be out of step from then on, with no bound on its last barrier.  The waits
// before it poll lane by lane, so the warp converges first (128^3 FP64 apply
// 327.7 us without, 327.9 with).
template <int NT> __device__ __forceinline__ void solvers_sync_converged()
{
    asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
}
template <int NT> __device__ __forceinline__ void solvers_sync()
{
    __syncwarp();
    solvers_sync_converged<NT>();
}

// ------------------------------------------------------------------ generic format
// The row of a chunk solved from shared memory: s - sum_k l_k y_dep(k), times
// dinv in the U pass.
template <class T>
__device__ __forceinline__ T solve_row_smem(const unsigned char *ch, const ChunkView<T> &v, int t,
                                            bool rm, const T *ring, const T *gdep, T sacc)
{
    const Segment<T> g = warp_segment<T>(ch, v.nrows, t / kWarpRows);
    const int lane = t % kWarpRows;
    sacc = rm ? row_solve_any<true, T>(g, lane, ring, gdep, sacc)
              : row_solve_any<false, T>(g, lane, ring, gdep, sacc);
    if (v.upass)
        sacc *= v.dinv[t];
    return sacc;
}

// ------------------------------------------------------------------ fixed-slot format
// (written by trsv_layout.cpp; every row padded to FW entries)
//   [0, 16)   nrows, nwarps, first position, flags (bit 0: U pass, bit 1: exports)
//   [16, 32)  need_prev, need_next, FW, xend (exports of the pass so far)
//   per warp w < nwarps a block, lane l = row 32w + l: val (ceil(FW / VW)
//   vectors of 32 lanes x 16 bytes, VW = 16 / sizeof(T)), dep (ceil(FW / 4)
//   vectors of 32 lanes x 4 int32), U: dinv[32] (T), src[32] (int32), U:
//   dst[32] (int32), exp[32] (int32 export positions, -1: none) in launches
//   with exp_arrays
constexpr int kFixedHeader = 32;

template <class T> struct Vec16;
template <> struct Vec16<double> {
    using type = double2;
    __device__ static double get(const double2 &v, int j) { return j == 0 ? v.x : v.y; }
};
template <> struct Vec16<float> {
    using type = float4;
    __device__ static float get(const float4 &v, int j)
    {
        return j == 0 ? v.x : j == 1 ? v.y : j == 2 ? v.z : v.w;
    }
};
__device__ __forceinline__ int get4(const int4 &v, int j)
{
    return j == 0 ? v.x : j == 1 ? v.y : j == 2 ? v.z : v.w;
}

template <class T, int FW> struct Fixed {
    static constexpr int VW = 16 / (int)sizeof(T);
    static constexpr int NV = (FW + VW - 1) / VW; // value vectors per lane
    static constexpr int ND = (FW + 3) / 4;       // dependency vectors per lane
    __device__ static constexpr int dep() { return NV * 512; }
    __device__ static constexpr int dinv() { return (NV + ND) * 512; }
    __device__ static constexpr int src(bool u) { return dinv() + (u ? 32 * (int)sizeof(T) : 0); }
    __device__ static constexpr int dst(bool u) { return src(u) + 128; }
    __device__ static constexpr int exp(bool u) { return src(u) + 128 + (u ? 128 : 0); }
    __device__ static constexpr int block(bool u, bool e) { return exp(u) + (e ? 128 : 0); }
};

// A solving thread's copy of its row of one fixed-slot chunk, with the
// chunk's header fields.
template <class T, int FW> struct RowRegs {
    int nrows, nwarps, base, flags;
    typename Vec16<T>::type lv[Fixed<T, FW>::NV];
    int4 dv[Fixed<T, FW>::ND];
    T rhs, dinv;
    int dst, exp;
    __device__ T l(int k) const { return Vec16<T>::get(lv[k / Fixed<T, FW>::VW], k % Fixed<T, FW>::VW); }
    __device__ int d(int k) const { return get4(dv[k / 4], k % 4); }
};

// Row t = 32 w + lane of a chunk (header hdr).  Every address depends on the
// stage, the thread and the pass alone: all loads issue back to back, 16
// bytes each for the row's entries.
template <class T, int FW>
__device__ __forceinline__ void load_fixed(const unsigned char *ch, const int4 &hdr, const T *rslot,
                                           int w, int lane, bool upass, bool exps,
                                           RowRegs<T, FW> &R)
{
    using F = Fixed<T, FW>;
    R.nrows = hdr.x;
    R.nwarps = hdr.y;
    R.base = hdr.z;
    R.flags = hdr.w;
    const unsigned char *blk = ch + kFixedHeader + (size_t)w * F::block(upass, exps);
    const typename Vec16<T>::type *val = reinterpret_cast<const typename Vec16<T>::type *>(blk) + lane;
#pragma unroll
    for (int v = 0; v < F::NV; ++v)
        R.lv[v] = val[v * 32];
    const int4 *dep = reinterpret_cast<const int4 *>(blk + F::dep()) + lane;
#pragma unroll
    for (int v = 0; v < F::ND; ++v)
        R.dv[v] = dep[v * 32];
    R.rhs = rslot[w * kWarpRows + lane];
    if (upass) {
        R.dinv = reinterpret_cast<const T *>(blk + F::dinv())[lane];
        R.dst = reinterpret_cast<const int *>(blk + F::dst(true))[lane];
    }
    R.exp = exps ? reinterpret_cast<const int *>(blk + F::exp(upass))[lane] : -1;
}

// The issuer warp of both kernels: streams chunk c of the program into stage
// c mod S once the consumers released chunk c - S.  The factor layout is read
// once per apply, so its lines are marked first to leave L2, which keeps the
// gathered right-hand sides and the y scratch there (measured on the 128^3
// case: FP32 apply 0.321 -> 0.286 ms, FP64 unchanged).  (Copying a chunk with
// lane-parallel 16-byte cp.async instead of one cp.async.bulk was measured
// there too: 1.3x slower in FP64, 2x in FP32.)  Returns false when a wait ran
// out.
__device__ __forceinline__ bool issue_chunks(const uint2 *chunks, int nch, int S, int stage_bytes,
                                             const unsigned char *pack, unsigned char *stages,
                                             uint64_t *full, uint64_t *empty, long long limit,
                                             int lane, int *s_issued)
{
    uint2 win = make_uint2(0, 0);
    int wbase = -64;
    int s = 0;
    uint32_t par = 1; // parity of the release of the stage's previous chunk
    const uint64_t pol = l2_evict_first_policy();
    for (int c = 0; c < nch; ++c) {
        if (c >= wbase + 32) { // 32 descriptors per warp-wide load
            wbase = c;
            win = (c + lane < nch) ? chunks[c + lane] : make_uint2(0, 0);
        }
        const unsigned off16 = __shfl_sync(0xffffffffu, win.x, c - wbase);
        const unsigned bytes = __shfl_sync(0xffffffffu, win.y, c - wbase);
        // every wait decision is a warp vote: the lanes must stay converged
        if (c >= S && __any_sync(0xffffffffu, !bounded_wait(&empty[s], par, limit)))
            return false;
        if (lane == 0) {
            mbar_arrive_expect_tx(&full[s], bytes);
            bulk_g2s_hint(stages + (size_t)s * stage_bytes, pack + (size_t)off16 * 16, bytes,
                          &full[s], pol);
            *s_issued = c + 1;
        }
        if (++s == S) {
            s = 0;
            par ^= 1u;
        }
    }
    return true;
}

// Warp-specialised CTA: 8 warps (fixed-slot chunks: two sets of 8) solve rows,
// one row per thread per chunk; the last five warps feed them.  Per chunk c
// in stage s = c mod S:
//   issuer: wait empty[s] (chunk c - S released) -> arm full[s] with
//             the chunk's byte count -> cp.async.bulk the chunk;
//   gatherers (three warps, chunks in turn): wait full[s] -> gather
//             the chunk's right-hand sides into slot s with cp.async, one
//             commit group per chunk (a U chunk waits for ldone first: its
//             right-hand side is the L pass's output) -> once the group has
//             completed (waited for while the warp's next chunks are gathered)
//             and lane 0 has seen the neighbouring parts' progress counters
//             reach the chunk's thresholds, lane 0 arrives on the stage's
//             handover mbarrier (40 cycles; a release-add to a shared counter
//             takes 90);
//   solvers, fixed-slot chunks: two sets of 8 warps take the chunks in turn,
//             and a barrier of both ends every level.  While one set solves
//             chunk c -- ring loads, the row's multiply-add chain, the result
//             into the ring (for exports also into the neighbour's import
//             ring) -- the other copies chunk c + 1's rows into registers and
//             forms every address its level will need.  So a level's
//             critical path holds none of that: with one set doing all of it,
//             the next chunk's copy and address arithmetic were the longer
//             half of a level.  128^3, ILU(1), 64 blocks in two parts: FP64
//             apply 427 -> 323 us; 101^3: 557 -> 457; 32^3, 8 blocks: 109 ->
//             78 (FP32 72 -> 52).
//             Three sets of 4 warps, with the addresses formed in a level of
//             their own, were no faster (335 us), and adding the older
//             levels' entries ahead of the barrier slower (410): the FP64
//             unit is shared by the SM (16 cycles a warp-wide multiply-add,
//             one in flight per warp), so the two sets then queue for it;
//   solvers, generic chunks: one set, rows solved from shared memory;
//   signaller: for a split block, forwards the completed count to
//             the neighbouring parts (a release at cluster scope, then the
//             count stored into their shared memory) as often as the fence
//             allows -- the count may jump several chunks at once.
// T = double: the FP64 path; T = float: the FP32 inner solves of the
// mixed-precision mode (FP32 factors, products and accumulation).
// Solving threads of a CTA: two sets of 8 warps for fixed-slot chunks.
template <int FW> constexpr int kSolvers = FW > 0 ? 2 * kThreads : kThreads;

template <class T, int FW>
__global__ void __launch_bounds__(kSolvers<FW> + kFeedThreads, 1) k_trsv_ras(TrsvArgs a)
{
    constexpr int NT = kSolvers<FW>; // solving threads; the feeding warps follow
    extern __shared__ __align__(128) unsigned char smem[];
    count_launch(a.st);
    if (a.st && a.st->skip)
        return; // uniform over the grid: no CTA of a cluster reaches a cluster barrier
    const T *r = reinterpret_cast<const T *>(a.r);
    if (a.r_from_j)
        r += (int64_t)a.st->j * a.ldv;

    const bool clustered = a.parts > 1;
    const int part = clustered ? (int)cluster_ctarank() : 0;
    const TrsvBlock blk = a.blocks[blockIdx.x];
    const int S = a.nstages;
    unsigned char *stages = smem;
    T *rhs = reinterpret_cast<T *>(smem + (size_t)S * a.stage_bytes);
    T *ring = rhs + (size_t)S * kThreads;
    const int nown = a.ring_mask + 1;
    const int RI = a.import_slots;
    const int nring = nown + RI; // own values, then values imported from a neighbour
    uint64_t *full = reinterpret_cast<uint64_t *>(reinterpret_cast<unsigned char *>(ring) +
                                                  (((size_t)nring * sizeof(T) + 7) & ~(size_t)7));
    uint64_t *empty = full + S;
    uint64_t *ldone = empty + S;
    uint32_t *ctr = reinterpret_cast<uint32_t *>(ldone + 1); // [0]: from part p - 1, [1]: from p + 1
    const int nch = blk.chunk_end - blk.chunk_begin;
    const int nL = blk.chunk_mid - blk.chunk_begin; // chunks of the L pass
    const bool has_prev = (blk.links & 1) != 0, has_next = (blk.links & 2) != 0;
    const bool signal = has_prev || has_next;
    const bool exps = FW > 0 && a.exp_arrays != 0;
    const bool stall_test = a.spin_limit < 0;       // fault injection: nothing is issued
    const long long limit = stall_test ? -a.spin_limit : a.spin_limit;
    const uint2 *chunks = a.chunks + blk.chunk_begin;
    T *ysc_w = reinterpret_cast<T *>(a.ysc) + blk.yoff;
    const T *ysc = ysc_w;
    T *zsc = a.zsc ? reinterpret_cast<T *>(a.zsc) + blk.zoff : nullptr;
    T *z = reinterpret_cast<T *>(a.z);
    const int t = threadIdx.x;
    // shared state of the roles (written before the final barrier)
    __shared__ int s_issued, s_err;
    __shared__ uint32_t s_done;             // chunks the consumers have completed
    __shared__ uint64_t s_hand[kMaxStages]; // handover mbarrier of every stage: a phase per chunk

    if (t == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
            mbar_init(&s_hand[s], 1);
        }
        mbar_init(ldone, 1);
        ctr[0] = ctr[1] = 0;
        s_issued = 0;
        s_err = 0;
        s_done = 0;
        fence_mbar_init();
    }
    for (int i = t; i < nown; i += blockDim.x)
        ring[i] = T(0);
    __syncthreads();
    // the neighbours store into this CTA's ring and counters only after they
    // are initialised
    if (clustered)
        cluster_sync_all();
    int failed = 0;

    if (t >= NT && t < NT + 32 && !stall_test) {
        // ------------------------------------------------------------ issuer warp
        if (!issue_chunks(chunks, nch, S, a.stage_bytes, a.pack, stages, full, empty, limit,
                          t - NT, &s_issued))
            failed = 1;
    } else if (t >= NT + 32 && t < NT + 32 * (1 + kGatherers) && !stall_test) {
        // ------------------------------------------------------------ gatherer warps
        // follow the chunks as they land, in turn:
        // gather each one's right-hand sides as one cp.async group, and hand
        // the chunk over once its group has completed and the neighbours'
        // progress allows it.  Every lane waits for its own copies before the
        // warp's vote and lane 0's release (an arrive-on-completion of the
        // copies, measured on this GPU, did not make them visible to the
        // solving warps in time).
        const int gw = (t - NT - 32) / 32;
        const int lane = t % 32;
        bool ldone_seen = false;
        // with 3 stages two of them work: the phase tests below tell a stage's
        // uses apart when a chunk that this warp saw land was issued after the
        // stage's last use but one was released (S >= NG; one more to spare)
        const int NG = S > kGatherers ? kGatherers : 2;
        int sg = gw; // gw < NG <= S: chunk gw lies in stage gw, phase 0
        uint32_t par = 0;
        int seen0 = 0, seen1 = 0; // lane 0: the neighbours' progress seen last
        int sh = sg, pend = 0; // stage of the oldest chunk in flight; chunks in flight
        constexpr int depth = FW > 0 ? kGatherDepth : 1; // (generic chunks: 0.5% faster so)
        // hand the oldest chunk over: its copies have landed, and lane 0 waits
        // for the neighbours' progress
        auto finish = [&]() -> bool {
            switch (pend) { // groups committed after it (kGatherDepth = 2)
            case 1: cp_async_wait_group<0>(); break;
            default: cp_async_wait_group<kGatherDepth - 1>(); break;
            }
            int late = 0;
            if (lane == 0 && clustered) {
                // the values this chunk imports are in the ring, and the
                // import slots its exports overwrite have been read
                const unsigned char *ch = stages + (size_t)sh * a.stage_bytes;
                const int2 need = *reinterpret_cast<const int2 *>(ch + (FW > 0 ? 16 : 96));
                // polls back off, leaving the issue slots to the solving warps;
                // none where the progress seen last covers the chunk
                late = !progress_wait(&ctr[0], seen0, need.x, limit) ||
                       !progress_wait(&ctr[1], seen1, need.y, limit);
            }
            // (the vote also orders every lane's landed copies before the release)
            if (__any_sync(0xffffffffu, late))
                return false;
            __syncwarp();
            if (lane == 0)
                mbar_arrive(&s_hand[sh]);
            sh += NG;
            if (sh >= S)
                sh -= S;
            --pend;
            return true;
        };
        for (int g = gw; gw < NG && g < nch;) {
            // chunks in flight are handed over first when the next one has not
            // landed, or needs the whole L pass
            const bool wait_l = g >= nL && !ldone_seen;
            // (the stage's previous chunk has been released, then its next landed)
            if (pend > 0 &&
                (pend == depth || wait_l ||
                 !__all_sync(0xffffffffu, (g < S || mbar_test_wait(&empty[sg], par ^ 1u)) &&
                                              mbar_test_wait(&full[sg], par)))) {
                if (!finish()) {
                    failed = 1;
                    break;
                }
                continue;
            }
            if ((g >= S && __any_sync(0xffffffffu, !bounded_wait(&empty[sg], par ^ 1u, limit))) ||
                __any_sync(0xffffffffu, !bounded_wait(&full[sg], par, limit)) ||
                (wait_l && __any_sync(0xffffffffu, !bounded_wait(ldone, 0u, limit)))) {
                failed = 1;
                break;
            }
            ldone_seen |= wait_l;
            const unsigned char *ch = stages + (size_t)sg * a.stage_bytes;
            int4 hdr = *reinterpret_cast<const int4 *>(ch);
            const bool upass = (hdr.w & 1) != 0;
            if (!HEC_CHECK(upass == (g >= nL), 1, g, hdr.w, nL) ||
                !HEC_CHECK(hdr.x >= 1 && hdr.x <= kThreads, 2, g, hdr.x, kThreads))
                hdr.x = 0; // nothing gathered from a chunk that is not the expected one
            T *slot = rhs + (size_t)sg * kThreads;
            const T *from = upass ? ysc : r;
            if constexpr (FW > 0) {
                const int blkb = Fixed<T, FW>::block(upass, exps);
                const unsigned char *src = ch + kFixedHeader + Fixed<T, FW>::src(upass) + 4 * lane;
                for (int i0 = 0; i0 < hdr.x; i0 += 128) { // four rows' sources read at once
                    int si[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (i0 + 32 * q + lane < hdr.x)
                            si[q] = *reinterpret_cast<const int *>(
                                src + (size_t)(i0 / 32 + q) * blkb);
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (i0 + 32 * q + lane < hdr.x &&
                            HEC_CHECK(si[q] >= 0 && (upass || si[q] < a.n), 3, g, si[q], a.n))
                            cp_async_v<sizeof(T)>(&slot[i0 + 32 * q + lane], from + si[q]);
                }
            } else {
                const ChunkView<T> v = view_chunk<T>(ch);
                for (int i = lane; i < hdr.x; i += 32)
                    if (HEC_CHECK(v.src[i] >= 0 && (upass || v.src[i] < a.n), 3, g, v.src[i], a.n))
                        cp_async_v<sizeof(T)>(&slot[i], from + v.src[i]);
            }
            cp_async_commit();
            ++pend;
            g += NG;
            sg += NG;
            if (sg >= S) {
                sg -= S;
                par ^= 1u;
            }
        }
        while (!failed && pend > 0)
            if (!finish())
                failed = 1;
        cp_async_wait_all();
    } else if (t >= NT + 32 * (1 + kGatherers)) {
        // ------------------------------------------------------------ signaller warp
        // publishes the completed-chunk count to the neighbours: the release
        // at cluster scope covers the consumers' stores into the neighbours'
        // import rings, ordered before the count by the consumer barrier
        if (signal && t == NT + 32 * (1 + kGatherers)) {
            const uint32_t to_prev = has_prev ? mapa_shared(smem_u32(&ctr[1]), part - 1) : 0;
            const uint32_t to_next = has_next ? mapa_shared(smem_u32(&ctr[0]), part + 1) : 0;
            uint32_t pub = 0;
            long long it = 0, t0 = clock64(); // since the last change of the count
            while (pub < (uint32_t)nch) {
                const uint32_t v = ld_acquire_cta_u32(&s_done);
                if (v > pub) {
                    fence_acq_rel_cluster();
                    if (has_prev)
                        st_relaxed_cluster_u32(to_prev, v);
                    if (has_next)
                        st_relaxed_cluster_u32(to_next, v);
                    pub = v;
                    it = 0;
                    t0 = clock64();
                } else if (*reinterpret_cast<volatile int *>(&s_err) || ++it >= limit ||
                           clock64() - t0 >= kWaitCycles) {
                    failed = 1;
                    break;
                } else {
                    __nanosleep(64);
                }
            }
        }
    } else if (t < NT) {
    // ---------------------------------------------------------------- consumer warps
    volatile int *verr = &s_err;
    // the neighbours' import rings: L values go to part p + 1, U values to p - 1
    const uint32_t imp_next =
        has_next ? mapa_shared(smem_u32(ring + nown), part + 1) : 0;
    const uint32_t imp_prev =
        has_prev ? mapa_shared(smem_u32(ring + nown), part - 1) : 0;
    int s = 0;         // stage of chunk c
    uint32_t hpar = 0; // the parity of that stage's handover of chunk c
    int err = 0;
    // wait (bounded) until the chunk in stage st has been handed over
    auto handed = [&](int st, uint32_t par) { return bounded_wait(&s_hand[st], par, limit); };
    // a solved row leaves: ring or scratch, neighbour's import ring; returns
    // where its global copy goes (written after the level's barrier)
    auto put = [&](bool upass, bool rm, int pos, int dst, int e, T acc) -> T * {
        T *gout = nullptr;
        if (upass) {
            if (rm)
                ring[pos & a.ring_mask] = acc;
            else
                zsc[pos] = acc; // read by later levels of this pass
            if (dst >= 0)
                gout = z + dst;
        } else if (rm) {
            ring[pos & a.ring_mask] = acc;
            gout = ysc_w + pos;
        } else {
            ysc_w[pos] = acc; // read by later levels of this pass
        }
        if (e >= 0)
            st_cluster((upass ? imp_prev : imp_next) + (uint32_t)((e & (RI - 1)) * sizeof(T)),
                       acc);
        return gout;
    };
    // after the level's barrier: global copies, end of the L pass, progress
    auto close = [&](int c, T *gout, T out) {
        if (gout)
            *gout = out;
        if (c == nL - 1) {
            // every y of the L pass is written before the gatherers read
            // the U pass's right-hand sides from them
            solvers_sync_and<NT>(1);
            if (t == kThreads - 1)
                mbar_arrive(ldone);
        }
        if (t == kThreads - 1 && signal)
            st_release_cta_u32(&s_done, (uint32_t)(c + 1));
    };
    if constexpr (FW > 0) {
        const int set = t / kThreads, lane = t % kWarpRows;
        const int w = (t / kWarpRows) % kMaxWarps;
        const int row = w * kWarpRows + lane;
        volatile int *vfail = &s_err;
#ifdef HEC_DEBUG
        __shared__ int s_base; // position the program has reached in its pass
        volatile int *vbase = &s_base;
#endif
        // One pass: chunks [c0, c1), U: the upper-triangular pass, RM: the
        // dependencies are in the ring (else in the global scratch).  Set
        // (c - c0) mod 2 solves chunk c.
        auto run = [&](auto Ucst, auto RMcst, int c0, int c1) {
            constexpr bool U = decltype(Ucst)::value, RM = decltype(RMcst)::value;
            const T *gdep = U ? zsc : ysc;
            T *scr = U ? zsc : ysc_w;
            const uint32_t imp = U ? imp_prev : imp_next;
            const uint32_t ring_a = smem_u32(ring);
            RowRegs<T, FW> R;
            uint32_t ya[FW]; // RM: shared addresses of the row's dependencies
            uint32_t own_a = 0, exp_to = 0;
            T *own = nullptr, *gout = nullptr;
            T acc = T(0);
            bool rows = false, mine = false, exports = false;
            bool landed = false; // the chunk copied last had been handed over
            // FP32, unsplit blocks: the set's last warp (with the shortest or
            // no rows) confirms a chunk's handover a level before the set
            // that copies it, so that the copy starts right after the barrier
            // with the header in the first load, and the last result's global
            // copy is written while the loads are under way: there the copy,
            // not the chain, paces a level (128^3 280 -> 262 us, 101^3 242 ->
            // 234).  In FP64 the chain does, and the same order costs (128^3
            // 327 -> 340, 101^3 463 -> 471); in split blocks, asking a level
            // early ties the parts closer together.
            constexpr bool kAhead = sizeof(T) == 4;
            const bool ahead = kAhead && !clustered;
            const bool confirmer = ahead && w == kMaxWarps - 1;
            auto confirm = [&](int st, uint32_t par) -> bool {
                if (*vfail)
                    return false;
                if (handed(st, par))
                    return true;
                *vfail = 1;
                return false;
            };
            // copies this set's next chunk, c, in stage s, and forms every
            // address the chunk's level will need
            auto fetch = [&](int c) {
                const unsigned char *ch = stages + (size_t)s * a.stage_bytes;
                if (ahead) {
                    landed = !*vfail;
                    const int4 hdr = *reinterpret_cast<const int4 *>(ch);
                    rows = landed && w < hdr.y; // warps past the chunk's last one hold no rows
                    if (rows)
                        load_fixed<T, FW>(ch, hdr, rhs + (size_t)s * kThreads, w, lane, U, exps,
                                          R);
                    if (gout)
                        *gout = acc;
                } else {
                    if (gout)
                        *gout = acc;
                    rows = landed = confirm(s, hpar);
                    if (rows) {
                        const int4 hdr = *reinterpret_cast<const int4 *>(ch);
                        rows = w < hdr.y;
                        if (rows)
                            load_fixed<T, FW>(ch, hdr, rhs + (size_t)s * kThreads, w, lane, U,
                                              exps, R);
                    }
                }
                mine = exports = false;
                gout = nullptr;
                if (!rows)
                    return;
#ifdef HEC_DEBUG
                rows = rows && HEC_CHECK((R.flags & 1) == (U ? 1 : 0), 1, c, R.flags, nL) &&
                       HEC_CHECK(R.nrows >= 1 && R.nrows <= kThreads &&
                                     R.nwarps == (R.nrows + 31) / 32,
                                 2, c, R.nrows, R.nwarps);
                if (rows)
                    for (int k = 0; k < FW; ++k)
                        rows &= RM ? HEC_CHECK(R.d(k) >= 0 && R.d(k) < nring, 5, c, R.d(k), nring)
                                   : HEC_CHECK(R.l(k) == T(0) ||
                                                   (R.d(k) >= 0 && R.d(k) < R.base),
                                               6, c, R.d(k), R.base);
                if (rows && row < R.nrows && U)
                    rows &= HEC_CHECK(R.dst < a.n, 7, c, R.dst, a.n);
#else
                (void)c;
#endif
                // padding lanes of the last warp carry valid slots
#pragma unroll
                for (int k = 0; k < FW; ++k)
                    ya[k] = ring_a + (uint32_t)(R.d(k) * sizeof(T));
                mine = rows && row < R.nrows;
                const int pos = R.base + row;
                own_a = ring_a + (uint32_t)((pos & a.ring_mask) * sizeof(T));
                own = scr + pos; // !RM: read by later levels
                if (mine && U)
                    gout = R.dst >= 0 ? z + R.dst : nullptr;
                else if (mine && RM)
                    gout = ysc_w + pos;
                exports = mine && R.exp >= 0; // -1 without export slots
                exp_to = imp + (uint32_t)((R.exp & (RI - 1)) * sizeof(T));
                acc = R.rhs;
            };
            // solves chunk c: the previous level's barrier has passed
            auto solve = [&]() {
                if (!rows)
                    return;
                T y[FW];
#pragma unroll
                for (int k = 0; k < FW; ++k) {
                    // global scratch: padding of a dependency-free row
                    // points at a position this apply has not written (it
                    // may hold NaN); entries of value 0 are not read
                    if constexpr (RM)
                        lds(ya[k], y[k]);
                    else
                        y[k] = R.l(k) != T(0) ? gdep[R.d(k)] : T(0);
                }
#pragma unroll
                for (int k = 0; k < FW; ++k)
                    acc = fma(-R.l(k), y[k], acc);
                if (U)
                    acc *= R.dinv;
                if (mine) {
                    if constexpr (RM)
                        sts(own_a, acc);
                    else
                        *own = acc;
                }
                if (exports)
                    st_cluster(exp_to, acc);
            };
            // the next chunk's stage and handover parity
            auto advance = [&]() {
                if (++s == S) {
                    s = 0;
                    hpar ^= 1u;
                }
            };
            // the confirmation of chunk n, the one after that in stage s
            auto confirm_next = [&](int n) {
                if (confirmer && n < c1) {
                    const bool wrap = s + 1 == S;
                    confirm(wrap ? 0 : s + 1, wrap ? hpar ^ 1u : hpar);
                }
            };
            // the stage of a chunk copied before the last barrier is free (not
            // that of one whose wait ran out: its copy may be in flight, and the
            // issuer, finding no free stage, gives up too)
            auto free_stage = [&](int c) {
                if (row == 0 && c < c1 && landed)
                    mbar_arrive(&empty[s]);
            };
#ifdef HEC_DEBUG
            if (t == 0)
                s_base = 0;
#endif
            int c = c0 + set; // the chunk this set solves next, in stage s
            if (set == 1)
                advance();
            if (confirmer && c < c1)
                confirm(s, hpar);
            solvers_sync<NT>();
            if (set == 0)
                fetch(c);
            solvers_sync<NT>();
            if (set == 0) {
                free_stage(c);
                advance();
            } else { // level c0 belongs to set 0
                if (c < c1) {
                    fetch(c);
                    confirm_next(c + 1);
                }
                solvers_sync<NT>();
                free_stage(c);
                advance();
            }
            while (c < c1) {
                // ---- level c: this set solves
#ifdef HEC_DEBUG
                if (rows && lane == 0)
                    HEC_CHECK(R.base == *vbase, 4, c, R.base, *vbase);
                solvers_set_sync(set);
                if (rows && row == 0)
                    *vbase = R.base + R.nrows;
#endif
                solve();
                solvers_sync<NT>();
                // ---- level c + 1: the other set solves, this one fetches
                if (signal && row == 0)
                    st_release_cta_u32(&s_done, (uint32_t)(c + 1));
                if (c + 1 >= c1)
                    break;
                advance();
                if (c + 2 < c1) {
                    fetch(c + 2);
                    confirm_next(c + 3);
                }
                solvers_sync<NT>();
                free_stage(c + 2);
                advance();
                c += 2;
            }
            if (gout) // the last result's global copy
                *gout = acc;
        };
        auto pass = [&](auto Ucst, int c0, int c1) {
            constexpr bool U = decltype(Ucst)::value;
            const int s0 = s;
            const uint32_t h0 = hpar;
            if (c0 < c1) {
                if (U ? blk.ring_U : blk.ring_L)
                    run(Ucst, std::true_type(), c0, c1);
                else
                    run(Ucst, std::false_type(), c0, c1);
            }
            // both sets go on from the stage after the pass's last chunk
            const int n = s0 + (c1 - c0);
            s = n % S;
            hpar = h0 ^ ((uint32_t)(n / S) & 1u);
        };
        pass(std::false_type(), 0, nL);
        if (nL > 0) {
            // every y of the L pass is written before the gatherers read
            // the U pass's right-hand sides from them
            solvers_sync<NT>();
            if (t == 0)
                mbar_arrive(ldone);
        }
        pass(std::true_type(), nL, nch);
        solvers_sync<NT>();
        failed = *vfail;

    } else {
        // The last warp, whose rows are the shortest, sees that chunk c + 1 has been
        // handed over before chunk c's barrier (at the L pass's end after it: the
        // U pass's right-hand sides need the whole L pass); the barrier tells the
        // other warps.  (Every thread asking for its own chunk: 32^3 ILU(2), one
        // block, 769 us, 753 so.)
        const bool asks = t >= kThreads - kWarpRows;
        auto ask = [&](int st, uint32_t par) {
            if (asks && !handed(st, par)) {
                err = 1;
                *verr = 1;
            }
        };
        if (nch > 0)
            ask(s, hpar);
        if (!solvers_sync_and<NT>(!err))
            failed = 1;
        for (int c = 0; c < nch && !failed; ++c) {
            T out = T(0);
            T *gout = nullptr;
            const unsigned char *ch = stages + (size_t)s * a.stage_bytes;
            const ChunkView<T> v = view_chunk<T>(ch);
            if (t < v.nrows) {
                const bool rm = v.upass ? blk.ring_U : blk.ring_L;
                const T acc = solve_row_smem<T>(ch, v, t, rm, ring, v.upass ? zsc : ysc,
                                                rhs[(size_t)s * kThreads + t]);
                gout = put(v.upass, rm, v.base + t, v.upass ? v.dst[t] : -1,
                           v.exports ? v.exp[t] : -1, acc);
                out = acc;
            }
            const int s0 = s;
            if (++s == S) {
                s = 0;
                hpar ^= 1u;
            }
            if (c + 1 < nch && c + 1 != nL)
                ask(s, hpar);
            if (!solvers_sync_and<NT>(!err)) {
                failed = 1; // the feeding warps' own waits run out
                break;
            }
            if (t == kThreads - 1)
                mbar_arrive(&empty[s0]); // the stage and its right-hand-side slot are free
            close(c, gout, out);
            if (c + 1 < nch && c + 1 == nL) {
                ask(s, hpar);
                if (!solvers_sync_and<NT>(!err))
                    failed = 1;
            }
        }
    }
    }
    // every role has left its loop: drain the copies still in flight, report
    __syncthreads();
    if (t == NT) {
        const int issued = s_issued;
        const int first = issued - S > 0 ? issued - S : 0;
        for (int c = first; c < issued; ++c)
            bounded_wait(&full[c % S], (uint32_t)(c / S) & 1u, kDrainPolls);
    }
    if (failed)
        report_timeout(a);
    // no CTA leaves while a neighbour may still store into its shared memory
    if (clustered)
        cluster_sync_all();
}

// ------------------------------------------------------------------ resident-vector kernel
// A RAS block whose right-hand side fits in shared memory next to the chunk
// stages is solved in place, by one CTA, with nothing on a level's critical
// path but shared memory: xs[i] starts as r[V_b[i]] (all local rows, gathered
// once at launch), the L pass overwrites it with y_i, the U pass with z_i, and
// the owned rows are written to z at the end.  A row's right-hand side is its
// own slot and its dependencies are the slots of its columns (local row
// indices), so there are no gatherer warps, no global scratch and no handover
// counters: one issuer warp streams the chunks (rows of one level) into the
// stages S chunks ahead with cp.async.bulk, and three sets of solving warps
// take the chunks in turn:
//   level c: one set reads the dependencies and the right-hand side of chunk
//            c's rows from xs, runs the multiply-add chain and stores the
//            results into xs; the set whose chunk is c + 1 unpacks its slots
//            into shared addresses; the set whose chunk is c + 2 confirms that
//            its group has landed and copies its rows into registers; barrier
//            of all sets.
// (One set that did all of it spent 278 cycles a level solving and 680 on the
// next chunk.  64^2, ILU(0), one block, FP64 apply: 88.7 -> 47.1 us.)
// The per-level critical path is a shared-memory load, the row's dependent
// multiply-adds (for U, the multiply by 1/u_ii) and a barrier of the solving
// warps.  This is the latency-first form for small systems (a single ILU block
// of a few thousand rows has hundreds of levels of a few dozen rows each).
//
// Chunk format (trsv_layout.cpp, flag bits 3 and 5): [0, 16) nrows, nwarps,
// first position, flags (bit 0: U pass); [16, 32) 0, 0, FW, 0; then per warp
// w < nwarps a block: val (ceil(FW / VW) 16-byte vectors of 32 lanes), idx
// (ceil((FW + 1) / 8) 16-byte vectors of 32 lanes x 8 uint16: the FW
// dependency slots, then the row's own slot), for U dinv[32].  Padding
// entries have value 0 and slot nv (a slot that holds 0); padding rows have
// row slot nv and are not stored.
template <class T, int FW> struct Res {
    static constexpr int VW = 16 / (int)sizeof(T);
    static constexpr int NV = (FW + VW - 1) / VW; // value vectors per lane
    static constexpr int NI = (FW + 1 + 7) / 8;   // index vectors per lane
    __device__ static constexpr int idx() { return NV * 512; }
    __device__ static constexpr int dinv() { return (NV + NI) * 512; }
    __device__ static constexpr int block() { return dinv() + 32 * (int)sizeof(T); }
};

// Three sets of NW solving warps (chunks of at most 32 NW rows, NW sized at
// setup to the widest level) and one issuer warp.
constexpr int kResSets = 3;
template <int NW> constexpr int kResSolvers = kResSets * NW * 32;
template <class T, int FW, int NW>
__global__ void __launch_bounds__(kResSolvers<NW> + 32, 1) k_trsv_res(TrsvArgs a)
{
    constexpr int NT = kResSolvers<NW>; // solving threads
    extern __shared__ __align__(128) unsigned char smem[];
    count_launch(a.st);
    if (a.st && a.st->skip)
        return; // uniform over the grid
    const T *r = reinterpret_cast<const T *>(a.r);
    if (a.r_from_j)
        r += (int64_t)a.st->j * a.ldv;
    T *z = reinterpret_cast<T *>(a.z);
    const TrsvBlock blk = a.blocks[blockIdx.x];
    const int S = a.nstages;
    unsigned char *stages = smem;
    T *xs = reinterpret_cast<T *>(smem + (size_t)S * a.stage_bytes);
    uint64_t *full = reinterpret_cast<uint64_t *>(reinterpret_cast<unsigned char *>(xs) +
                                                  (((size_t)a.res_slots * sizeof(T) + 7) & ~(size_t)7));
    uint64_t *empty = full + S;
    const int nch = blk.chunk_end - blk.chunk_begin;
    const int nL = blk.chunk_mid - blk.chunk_begin;
    const int *vrows = a.vrows + blk.yoff; // V_b: the global row of every local slot
    const bool stall_test = a.spin_limit < 0; // fault injection: nothing is issued
    const long long limit = stall_test ? -a.spin_limit : a.spin_limit;
    const int t = threadIdx.x;
    __shared__ int s_issued, s_fail;
    if (t == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        s_issued = 0;
        s_fail = 0;
        fence_mbar_init();
    }
    __syncthreads();
    int failed = 0;
    if (t >= NT) {
        // ------------------------------------------------------------ issuer warp
        if (!stall_test &&
            !issue_chunks(a.groups + blk.zoff, blk.ngroups, S, a.stage_bytes, a.pack, stages,
                          full, empty, limit, t - NT, &s_issued))
            failed = 1;
    } else {
        // ------------------------------------------------------------ solving warps
        // r on V_b into the resident vector; slot nv holds 0 (padding)
        // (kBatch rows' loads in flight)
        constexpr int kBatch = 8;
        for (int i0 = t; i0 < blk.nv; i0 += kBatch * NT) {
            int g[kBatch];
            T v[kBatch];
#pragma unroll
            for (int q = 0; q < kBatch; ++q)
                g[q] = i0 + q * NT < blk.nv ? vrows[i0 + q * NT] : -1;
#pragma unroll
            for (int q = 0; q < kBatch; ++q)
                v[q] = i0 + q * NT < blk.nv && HEC_CHECK(g[q] >= 0 && g[q] < a.n, 3, 0, g[q], a.n)
                           ? r[g[q]]
                           : T(0);
#pragma unroll
            for (int q = 0; q < kBatch; ++q)
                if (i0 + q * NT < blk.nv)
                    xs[i0 + q * NT] = v[q];
        }
        if (t == 0)
            xs[blk.nv] = T(0);
        // each set's warps are turned by one more, so that the sets' chunks of
        // few warps use other sub-partitions of the SM
        const int set = t / (NW * 32), lane = t % kWarpRows;
        const int w = (t / kWarpRows + set) % NW;
        const int row = w * kWarpRows + lane;
        // Chunks arrive in groups of G (one bulk copy each) in stage order, all
        // of one size CB: chunk k of a group sits at k CB in its group's stage.
        // A chunk's place is that stage ls, the stage's phase parity lph and lk.
        constexpr int CB = kFixedHeader + NW * Res<T, FW>::block();
        const int G = a.res_group;
        const uint32_t xs_a = smem_u32(xs);
        volatile int *vfail = &s_fail;
        int ls = 0, lk = 0; // the place of this set's next chunk
        uint32_t lph = 0;
        auto advance = [&](int n) {
            for (lk += n; lk >= G; lk -= G)
                if (++ls == S) {
                    ls = 0;
                    lph ^= 1u;
                }
        };
        using F = Res<T, FW>;
        typename Vec16<T>::type lv[F::NV];
        uint4 iv[F::NI];
        T dinv = T(0);
        int nrows = 0;
        uint32_t xa[FW + 1]; // shared addresses of the dependencies and the own slot
        bool rows = false, mine = false, upper = false;
        bool landed = false; // the chunk copied last lies in a group that landed
        // copies this set's next chunk, at (ls, lph, lk), once its group has
        // landed (after the first barrier, only the chunk that opens a group
        // asks: the other sets copy from it in later levels)
        auto fetch = [&](bool ask) {
            rows = landed = false;
            if (*vfail) // a group that never landed: nothing is read from it
                return;
            // a vote: the warp stays converged for the barriers (a __syncwarp at
            // every barrier instead: 64^2 ILU(0) 49.1 us, 46.4 so)
            if (ask && __any_sync(0xffffffffu, !bounded_wait(&full[ls], lph, limit))) {
                *vfail = 1;
                return;
            }
            const unsigned char *ch = stages + (size_t)ls * a.stage_bytes + (size_t)lk * CB;
            const int2 hdr = *reinterpret_cast<const int2 *>(ch); // rows, warps
            const unsigned char *blkp = ch + kFixedHeader + (size_t)w * F::block();
#pragma unroll
            for (int v = 0; v < F::NV; ++v)
                lv[v] = (reinterpret_cast<const typename Vec16<T>::type *>(blkp) + lane)[v * 32];
#pragma unroll
            for (int v = 0; v < F::NI; ++v)
                iv[v] = (reinterpret_cast<const uint4 *>(blkp + F::idx()) + lane)[v * 32];
            dinv = reinterpret_cast<const T *>(blkp + F::dinv())[lane];
            nrows = hdr.x;
            landed = true;
            rows = w < hdr.y; // warps past the chunk's last one idle
        };
        // chunk c's slots as shared addresses; the chunk that opens a group
        // frees the stage of the one before (its last chunk was copied at least
        // a barrier ago; after a wait that ran out nothing is freed: a copy may
        // be in flight, and the issuer, finding no free stage, gives up too)
        auto prepare = [&](int c) {
            if (row == 0 && lk == 0 && c > 0 && landed)
                mbar_arrive(&empty[ls == 0 ? S - 1 : ls - 1]);
#pragma unroll
            for (int k = 0; k <= FW; ++k) { // vectors of 8 uint16
                const uint4 v = iv[k / 8];
                const uint32_t word = (k % 8) / 2 == 0 ? v.x : (k % 8) / 2 == 1 ? v.y
                                      : (k % 8) / 2 == 2 ? v.z : v.w;
                uint32_t sl = (word >> (16 * (k % 2))) & 0xffffu;
#ifdef HEC_DEBUG
                if (rows && !HEC_CHECK(sl <= (uint32_t)blk.nv, k < FW ? 5 : 7, c, sl, blk.nv))
                    sl = blk.nv;
#endif
                xa[k] = xs_a + sl * (uint32_t)sizeof(T);
            }
            mine = rows && row < nrows && xa[FW] < xs_a + blk.nv * (uint32_t)sizeof(T);
            upper = c >= nL;
        };
        int c = set; // the chunk this set solves next
        advance(set);
        // before level 0: its chunk is ready, the next one copied
        if (set < 2 && c < nch)
            fetch(true);
        if (set == 0)
            prepare(c);
        // the gather above is complete too
        solvers_sync_converged<NT>();
        for (int l = 0; l < c && l < nch; ++l) { // the levels before this set's first
            if (l == c - 1)
                prepare(c);
            else if (c < nch)
                fetch(lk == 0);
            solvers_sync_converged<NT>();
        }
        while (c < nch) {
            // ---- level c
            if (rows) {
                T y[FW], acc;
#pragma unroll
                for (int k = 0; k < FW; ++k)
                    lds(xa[k], y[k]);
                lds(xa[FW], acc);
#pragma unroll
                for (int k = 0; k < FW; ++k)
                    acc = fma(-Vec16<T>::get(lv[k / F::VW], k % F::VW), y[k], acc);
                if (upper)
                    acc *= dinv;
                if (mine)
                    sts(xa[FW], acc);
            }
            solvers_sync_converged<NT>();
            // ---- level c + 1
            if (c + 1 >= nch)
                break;
            advance(kResSets);
            if (c + kResSets < nch)
                fetch(lk == 0);
            else
                rows = landed = false;
            solvers_sync_converged<NT>();
            // ---- level c + 2
            if (c + 2 >= nch)
                break;
            prepare(c + kResSets);
            solvers_sync_converged<NT>();
            c += kResSets;
        }
        solvers_sync_converged<NT>();
        failed = *vfail;
        if (!failed)
            for (int i0 = blk.own0 + t; i0 < blk.own1; i0 += kBatch * NT) {
                int g[kBatch];
#pragma unroll
                for (int q = 0; q < kBatch; ++q)
                    g[q] = i0 + q * NT < blk.own1 ? vrows[i0 + q * NT] : -1;
#pragma unroll
                for (int q = 0; q < kBatch; ++q)
                    if (i0 + q * NT < blk.own1)
                        z[g[q]] = xs[i0 + q * NT];
            }
    }
    // every role has left its loop: drain the copies still in flight, report
    __syncthreads();
    if (t == NT) {
        const int issued = s_issued;
        const int first = issued - S > 0 ? issued - S : 0;
        for (int c = first; c < issued; ++c)
            bounded_wait(&full[c % S], (uint32_t)(c / S) & 1u, kDrainPolls);
    }
    if (failed)
        report_timeout(a);
}

// ------------------------------------------------------------------ long-row kernel
// Blocks whose rows are too long for the resident kernel but whose FP32 vector
// fits in shared memory: the vector is solved in place as there, and a row's
// entries are spread over a group of lanes (4 a lane), summed by shuffles.  One
// thread per row leaves a level of such a block with a handful of active lanes
// and one long chain: the 27-point matrix with irregular rows has 17 rows in
// the median level, 13 entries a row (up to 117), and its dependencies reach
// further back than any ring, so the streamed kernel also read them from
// global memory: 72^3, ILU(0), 64 blocks 1,806 -> 295 us.
// A warp's work in a level is a unit (kernels.cuh); kLongWarps units, one per
// warp, travel in one bulk copy.  A warp copies its next unit into registers,
// forms its addresses and waits until the units of the earlier levels are
// solved: every warp publishes how many units it has solved, and the lanes read
// all warps' counts.  So a warp without a unit in a level takes no part in it,
// and every wait between warps has its limit.
// (A barrier of all warps per level as bar.sync, 305 us on the case above, is
// not sound here: on a served stream of eight lanes a solve's steps changed from
// run to run and some applies never ended, three of five runs, while the same
// kernel with counted waits gave the same steps in every run.  As an mbarrier of
// all warps: 553 us.  This form: 350; with 16 warps 3% more.)
constexpr int kLongThreads = 32 * kLongWarps;
constexpr int kLongPolls = 64; // polls between two readings of the clock
__global__ void __launch_bounds__(kLongThreads + 32, 1) k_trsv_long(TrsvArgs a)
{
    constexpr int NT = kLongThreads;
    extern __shared__ __align__(128) unsigned char smem[];
    count_launch(a.st);
    if (a.st && a.st->skip)
        return; // uniform over the grid
    const float *r = reinterpret_cast<const float *>(a.r);
    if (a.r_from_j)
        r += (int64_t)a.st->j * a.ldv;
    float *z = reinterpret_cast<float *>(a.z);
    const TrsvBlock blk = a.blocks[blockIdx.x];
    const int S = a.nstages;
    unsigned char *stages = smem;
    float *xs = reinterpret_cast<float *>(smem + (size_t)S * a.stage_bytes);
    uint64_t *full = reinterpret_cast<uint64_t *>(
        reinterpret_cast<unsigned char *>(xs) + (((size_t)a.res_slots * sizeof(float) + 7) & ~(size_t)7));
    uint64_t *empty = full + S;
    const int ng = blk.ngroups;
    const int *vrows = a.vrows + blk.yoff;
    const bool stall_test = a.spin_limit < 0; // fault injection: nothing is issued
    const long long limit = stall_test ? -a.spin_limit : a.spin_limit;
    const int t = threadIdx.x;
    __shared__ int s_issued, s_fail;
    __shared__ uint32_t s_solved[kLongWarps]; // per warp: 1 + its solved units (0: not gathered yet)
    if (t < kLongWarps)
        s_solved[t] = 0;
    if (t == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], kLongWarps);
        }
        s_issued = 0;
        s_fail = 0;
        fence_mbar_init();
    }
    __syncthreads();
    int failed = 0;
    if (t >= NT) {
        // ------------------------------------------------------------ issuer warp
        if (!stall_test &&
            !issue_chunks(a.groups + blk.zoff, ng, S, a.stage_bytes, a.pack, stages, full, empty,
                          limit, t - NT, &s_issued))
            failed = 1;
    } else {
        // ------------------------------------------------------------ solving warps
        constexpr int kBatch = 8;
        for (int i0 = t; i0 < blk.nv; i0 += kBatch * NT) {
            int g[kBatch];
            float v[kBatch];
#pragma unroll
            for (int q = 0; q < kBatch; ++q)
                g[q] = i0 + q * NT < blk.nv ? vrows[i0 + q * NT] : -1;
#pragma unroll
            for (int q = 0; q < kBatch; ++q)
                v[q] = i0 + q * NT < blk.nv && HEC_CHECK(g[q] >= 0 && g[q] < a.n, 3, 0, g[q], a.n)
                           ? r[g[q]]
                           : 0.0f;
#pragma unroll
            for (int q = 0; q < kBatch; ++q)
                if (i0 + q * NT < blk.nv)
                    xs[i0 + q * NT] = v[q];
        }
        if (t == 0)
            xs[blk.nv] = 0.0f; // padding
        const int w = t / 32, lane = t % 32;
        const uint32_t xs_a = smem_u32(xs);
        volatile int *vfail = &s_fail;
        int s = 0; // the stage of the warp's next unit and its phase
        uint32_t par = 0;
        float4 val;
        float mul = 1.0f;
        uint32_t xa[kLongPerLane + 1]; // shared addresses of the dependencies and the own slot
        int flags = 0;
        // copies the unit of group g and forms its addresses; the stage is
        // free once every warp has its unit
        auto fetch = [&](int g) -> bool {
            // a vote: what follows (the unit's waits and shuffles) is the whole warp's
            if (__any_sync(0xffffffffu, !bounded_wait(&full[s], par, limit))) {
                *vfail = 1;
                return false;
            }
            const unsigned char *u = stages + (size_t)s * a.stage_bytes + w * kLongUnit;
            val = reinterpret_cast<const float4 *>(u)[lane];
            const uint4 rec = reinterpret_cast<const uint4 *>(u + 512)[lane];
            uint32_t sl[kLongPerLane + 1] = {rec.x & 0xffffu, rec.x >> 16, rec.y & 0xffffu,
                                             rec.y >> 16, rec.z & 0xffffu};
            flags = (int)(rec.z >> 16);
            mul = __uint_as_float(rec.w);
#pragma unroll
            for (int k = 0; k <= kLongPerLane; ++k) {
#ifdef HEC_DEBUG
                if (!HEC_CHECK(sl[k] <= (uint32_t)blk.nv, k < kLongPerLane ? 5 : 7, g, sl[k], blk.nv))
                    sl[k] = blk.nv;
#endif
                xa[k] = xs_a + sl[k] * 4u;
            }
            (void)g;
            __syncwarp();
            if (lane == 0)
                mbar_arrive(&empty[s]);
            if (++s == S) {
                s = 0;
                par ^= 1u;
            }
            return true;
        };
        // this warp's count, after its stores
        auto publish = [&](uint32_t solved) {
            __syncwarp();
            if (lane == 0)
                st_release_cta_u32(&s_solved[w], 1u + solved);
        };
        // waits until the units below index `first` are solved (and every warp
        // has gathered): lane l reads warp l mod kLongWarps's count
        auto wait_for = [&](int first) -> bool {
            const uint32_t need = 1u + (uint32_t)(first + kLongWarps - 1 - lane % kLongWarps) / kLongWarps;
            const uint32_t *p = &s_solved[lane % kLongWarps];
            bool ok = __all_sync(0xffffffffu, ld_relaxed_cta_u32(p) >= need);
            long long t0 = 0;
            for (long long left = limit - 1; !ok && left > 0; left -= kLongPolls) {
#pragma unroll 1
                for (int k = 0; k < kLongPolls; ++k)
                    if ((ok = __all_sync(0xffffffffu, ld_relaxed_cta_u32(p) >= need)))
                        break;
                if (ok)
                    break;
                const long long now = clock64(); // (read once in kLongPolls polls)
                if (t0 == 0)
                    t0 = now;
                if (__any_sync(0xffffffffu, now - t0 >= kWaitCycles))
                    break;
            }
            fence_acq_rel_cta();
            __syncwarp(); // every lane's reads come after every count
            if (!ok)
                *vfail = 1;
            return ok;
        };
        publish(0);
        bool have = true;
        for (int g = 0; g < ng && have; ++g) {
            have = fetch(g);
            if (!have)
                break;
            have = wait_for(g * kLongWarps + w - (flags >> 7));
            if (!have)
                break;
            float y[kLongPerLane], acc, x;
#pragma unroll
            for (int k = 0; k < kLongPerLane; ++k)
                lds(xa[k], y[k]);
            lds(xa[kLongPerLane], x);
            acc = (flags & 64) ? x : 0.0f; // the row's first lane holds its right-hand side
            acc = fmaf(-val.x, y[0], acc);
            acc = fmaf(-val.y, y[1], acc);
            acc = fmaf(-val.z, y[2], acc);
            acc = fmaf(-val.w, y[3], acc);
            const int lg = flags & 7, maxlg = (flags >> 3) & 7;
            for (int q = 0; q < maxlg; ++q) {
                const float o = __shfl_xor_sync(0xffffffffu, acc, 1 << q);
                acc += q < lg ? o : 0.0f;
            }
            if (flags & 64)
                sts(xa[kLongPerLane], acc * mul);
            publish((uint32_t)g + 1u);
        }
        // the block is solved
        failed = !have || !wait_for(ng * kLongWarps) || *vfail;
        if (!failed)
            for (int i0 = blk.own0 + t; i0 < blk.own1; i0 += kBatch * NT) {
                int g[kBatch];
#pragma unroll
                for (int q = 0; q < kBatch; ++q)
                    g[q] = i0 + q * NT < blk.own1 ? vrows[i0 + q * NT] : -1;
#pragma unroll
                for (int q = 0; q < kBatch; ++q)
                    if (i0 + q * NT < blk.own1)
                        z[g[q]] = xs[i0 + q * NT];
            }
    }
    // every role has left its loop: drain the copies still in flight, report
    __syncthreads();
    if (t == NT) {
        const int issued = s_issued;
        const int first = issued - S > 0 ? issued - S : 0;
        for (int c = first; c < issued; ++c)
            bounded_wait(&full[c % S], (uint32_t)(c / S) & 1u, kDrainPolls);
    }
    if (failed)
        report_timeout(a);
}

// The dynamic shared memory limit is an attribute of the kernel on a device:
// raised once to the device's opt-in maximum, which covers static and dynamic
// shared memory, so that launches of different sizes from several host threads
// never race on it.
template <class K> static cudaError_t prepare_trsv(PerDevice<cudaError_t> &once, K kernel)
{
    int dev = 0;
    cudaGetDevice(&dev);
    return once.get(dev, [&]() {
        int optin = 0;
        cudaFuncAttributes fa{};
        cudaError_t e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        if (e == cudaSuccess)
            e = cudaFuncGetAttributes(&fa, kernel);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     optin - (int)fa.sharedSizeBytes);
        return e;
    });
}

template <class T, int FW> static int launch_t(const TrsvArgs &a, cudaStream_t s)
{
    const size_t smem =
        trsv_smem_bytes(a.stage_bytes, a.nstages, a.ring_mask + 1 + a.import_slots, sizeof(T));
    static PerDevice<cudaError_t> once;
    if (prepare_trsv(once, k_trsv_ras<T, FW>) != cudaSuccess)
        return -1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)a.nblocks);
    cfg.blockDim = dim3(kSolvers<FW> + kFeedThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)a.parts;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = a.parts > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k_trsv_ras<T, FW>, a) == cudaSuccess ? 0 : -1;
}

template <class T, int FW, int NW> static int launch_res(const TrsvArgs &a, cudaStream_t s)
{
    const size_t smem = trsv_res_smem_bytes(a.stage_bytes, a.nstages, a.res_slots, sizeof(T));
    static PerDevice<cudaError_t> once;
    if (prepare_trsv(once, k_trsv_res<T, FW, NW>) != cudaSuccess)
        return -1;
    k_trsv_res<T, FW, NW><<<a.nblocks, kResSolvers<NW> + 32, smem, s>>>(a);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

static int launch_long(const TrsvArgs &a, cudaStream_t s)
{
    static PerDevice<cudaError_t> once;
    if (prepare_trsv(once, k_trsv_long) != cudaSuccess)
        return -1;
    const size_t smem = trsv_res_smem_bytes(a.stage_bytes, a.nstages, a.res_slots, sizeof(float));
    k_trsv_long<<<a.nblocks, kLongThreads + 32, smem, s>>>(a);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

template <class T, int FW> static int launch_res_w(const TrsvArgs &a, cudaStream_t s)
{
    switch (a.res_warps) {
    case 2: return launch_res<T, FW, 2>(a, s);
    case 4: return launch_res<T, FW, 4>(a, s);
    case 8: return launch_res<T, FW, 8>(a, s);
    default: return -1;
    }
}

size_t trsv_res_smem_bytes(int stage_bytes, int nstages, int res_slots, int vbytes)
{
    return (size_t)stage_bytes * nstages + (((size_t)res_slots * vbytes + 7) & ~(size_t)7) +
           (size_t)2 * nstages * sizeof(uint64_t);
}

int trsv_res_stages_for(int stage_bytes, int res_slots, int vbytes)
{
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        optin = 227 * 1024;
    optin -= 1024; // static shared memory of the kernel
    for (int S = 8; S >= 3; --S)
        if (trsv_res_smem_bytes(stage_bytes, S, res_slots, vbytes) <= (size_t)optin)
            return S;
    return 0;
}

int trsv_debug_read(int *out, bool clear)
{
    if (cudaMemcpyFromSymbol(out, g_trsv_debug, sizeof(g_trsv_debug)) != cudaSuccess)
        return -1;
    if (clear) {
        static const int zero[8] = {};
        if (cudaMemcpyToSymbol(g_trsv_debug, zero, sizeof(zero)) != cudaSuccess)
            return -1;
    }
    return 0;
}

bool trsv_debug_build()
{
#ifdef HEC_DEBUG
    return true;
#else
    return false;
#endif
}

int launch_trsv(const TrsvArgs &a, cudaStream_t s, bool fp32)
{
    if (a.resident == 2)
        return fp32 ? launch_long(a, s) : -1;
    if (a.resident) {
#define HEC_RES_CASE(W)                                                                          \
    case W: return fp32 ? launch_res_w<float, W>(a, s) : launch_res_w<double, W>(a, s);
        switch (a.fixed_width) {
            HEC_RES_CASE(2)
            HEC_RES_CASE(3)
            HEC_RES_CASE(4)
            HEC_RES_CASE(6)
            HEC_RES_CASE(8)
        default: return -1;
        }
#undef HEC_RES_CASE
    }
    // fixed-slot layouts by their uniform width; generic layouts
    if (!fp32) {
        switch (a.fixed_width) {
        case 4: return launch_t<double, 4>(a, s);
        case 6: return launch_t<double, 6>(a, s);
        case 8: return launch_t<double, 8>(a, s);
        default: return launch_t<double, 0>(a, s);
        }
    }
    switch (a.fixed_width) {
    case 4: return launch_t<float, 4>(a, s);
    case 6: return launch_t<float, 6>(a, s);
    case 8: return launch_t<float, 8>(a, s);
    default: return launch_t<float, 0>(a, s);
    }
}

int trsv_uniform_width(int longest_row)
{
    return longest_row <= 4 ? 4 : longest_row <= 6 ? 6 : longest_row <= 8 ? 8 : 0;
}

} // namespace hec
