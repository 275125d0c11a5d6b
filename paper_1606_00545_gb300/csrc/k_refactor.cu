// k_refactor.cu -- numeric refactorisation on the GPU: a matrix with the same
// sparsity pattern and new values replaces the old one without a host round
// trip.  The HEC slab and tail take the new values (Section 2.1), every RAS
// block's ILU(k) factor is recomputed on its existing fill pattern by the
// IKJ elimination of Algorithm 2 (the pattern -- Eqs. 9-10 -- does not depend
// on the values), scheduled by the L level sets of Eq. 11 (a row's
// elimination reads only rows of lower levels), and the triangular-solve
// layouts get the new factor values.
//
// The elimination performs exactly the host's operations in the host's
// order -- per row, pivots p ascending; l_ip = a_ip / u_pp; a_ij -= l_ip u_pj
// for the j of row p's U part that row i holds -- with separately rounded
// multiply and subtract (no contraction, as the host code is compiled), so
// the factors are bit-identical to a host factorisation of the new matrix.
#include "per_device.h"
#include "ptx.cuh"
#include "reduce.cuh"

namespace hec {

// New CSR values -> slab / tail slots: slot >= 0 is an ELL slot, slot < 0 the
// tail entry -slot - 1.
__global__ void k_scatter_hec(int64_t nnz, const double *val, const int64_t *slot, double *ell,
                              double *tail)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t s = slot[e];
        if (s >= 0)
            ell[s] = val[e];
        else
            tail[-s - 1] = val[e];
    }
}

__global__ void k_cast_f32(int64_t n, const double *x, float *y)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        y[i] = (float)x[i];
}

// Factor entries start from A's values on the original pattern, 0 on fill.
__global__ void k_gather_factor(int64_t nent, const double *val, const int *src, double *f)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nent;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int s = src[e];
        f[e] = s >= 0 ? val[s] : 0.0;
    }
}

// Rows of at most kLocalRow entries are eliminated in per-thread arrays:
// the row is read once and written once, and its merges against the pivot
// rows read only the pivot rows from memory.  Longer rows run the same steps
// on global memory.
constexpr int kLocalRow = 48;

__device__ __forceinline__ bool eliminate_row_local(const RefactorArgs &a, int row0, int r)
{
    const int b0 = a.rp[r], len = a.rp[r + 1] - b0, nl = a.dg[r] - b0;
    int ci[kLocalRow];
    double f[kLocalRow];
    for (int q = 0; q < len; ++q) {
        ci[q] = a.ci[b0 + q];
        f[q] = a.f[b0 + q];
    }
    bool ok = true;
    for (int k = 0; k < nl; ++k) {
        const int p = row0 + ci[k]; // pivot row
        const int dp = a.dg[p], ep = a.rp[p + 1];
        const double upp = a.f[dp];
        if (upp == 0.0) {
            ok = false;
            break;
        }
        const double lip = __ddiv_rn(f[k], upp);
        f[k] = lip;
        // row i's entries right of p against row p's U part (both ascending)
        int x = k + 1, y = dp + 1;
        int cy = y < ep ? a.ci[y] : 0x7fffffff;
        double fy = y < ep ? a.f[y] : 0.0;
        while (x < len && y < ep) {
            const int cx = ci[x];
            if (cx == cy) {
                f[x] = __dsub_rn(f[x], __dmul_rn(lip, fy));
                ++x;
                ++y;
                if (y < ep) {
                    cy = a.ci[y];
                    fy = a.f[y];
                }
            } else if (cx < cy) {
                ++x;
            } else {
                ++y;
                if (y < ep) {
                    cy = a.ci[y];
                    fy = a.f[y];
                }
            }
        }
    }
    for (int q = 0; q < len; ++q)
        a.f[b0 + q] = f[q];
    return ok && f[nl] != 0.0;
}

__device__ __forceinline__ bool eliminate_row_global(const RefactorArgs &a, int row0, int r)
{
    double *f = a.f;
    const int end_i = a.rp[r + 1];
    for (int e = a.rp[r]; e < a.dg[r]; ++e) {
        const int p = row0 + a.ci[e]; // pivot row
        const double upp = f[a.dg[p]];
        if (upp == 0.0)
            return false;
        const double lip = __ddiv_rn(f[e], upp);
        f[e] = lip;
        int x = e + 1, y = a.dg[p] + 1;
        const int end_p = a.rp[p + 1];
        while (x < end_i && y < end_p) {
            const int cx = a.ci[x], cy = a.ci[y];
            if (cx == cy) {
                f[x] = __dsub_rn(f[x], __dmul_rn(lip, f[y]));
                ++x;
                ++y;
            } else if (cx < cy) {
                ++x;
            } else {
                ++y;
            }
        }
    }
    return f[a.dg[r]] != 0.0;
}

// One CTA per RAS block, one thread per row of the current L level, a CTA
// barrier between levels.  Row data is global-entry indexed: row r (global
// over all blocks) holds entries [rp[r], rp[r+1]), local columns ci, its
// diagonal at dg[r].  Within a row the pivots are taken in ascending order
// and each update is a separately rounded multiply and subtract: the host's
// operations in the host's order.
__global__ void __launch_bounds__(kThreads) k_iluk_numeric(RefactorArgs a)
{
    const int b = blockIdx.x;
    const int row0 = a.blk_row0[b];
    const int *lptr = a.lptr + a.blk_lev0[b];
    const int nlev = a.blk_lev0[b + 1] - a.blk_lev0[b] - 1;
    const int *lrows = a.lrows + row0;
    for (int l = 0; l < nlev; ++l) {
        for (int q = lptr[l] + threadIdx.x; q < lptr[l + 1]; q += blockDim.x) {
            const int r = row0 + lrows[q];
            const bool ok = (a.rp[r + 1] - a.rp[r] <= kLocalRow)
                                ? eliminate_row_local(a, row0, r)
                                : eliminate_row_global(a, row0, r);
            if (!ok)
                atomicExch(a.err, HEC_ERR_ZERO_PIVOT);
        }
        __syncthreads();
    }
}

// The same elimination for blocks whose rows hold at most LEN entries.  The
// merges of k_iluk_numeric chase one pivot entry at a time through memory,
// and that latency, not the arithmetic, is its time (23 us a level on the
// 101^3 ILU(1) case).  Here a row's values are in shared memory, a pivot's U
// part comes in with independent loads, up to kAhead entries at once and one
// pivot ahead of their use (the pivot's place in memory two ahead), and where
// an entry goes is known from a plan made once per pattern (k_iluk_plan: 4
// bits for each of those entries, 0 for none -- an update never hits position
// 0); rows of 17 to 32 entries compare columns instead, which costs 2,000
// instructions a row (4.8 ms on that case instead of 3.7).  What is left is the chain
// of one division and a few updates per pivot.  A block's rows go to C CTAs
// of a cluster, warp by warp, with a cluster barrier between levels: 64 blocks
// alone leave most SMs idle.  101^3, ILU(1), 64 blocks: 7.08 -> 3.7 ms (of
// hec_refactor's 8.2 -> 4.8 with an SpMV and an apply behind it).
constexpr int kAhead = 8;

// The position among the row's columns of column c, -1 if it holds none.
template <int LEN> __device__ __forceinline__ int find_col(const int (&col)[LEN], int c)
{
    int x = -1;
#pragma unroll
    for (int j = 0; j < LEN; ++j)
        x = col[j] == c ? j : x;
    return x;
}

template <int LEN> __global__ void __launch_bounds__(kThreads) k_iluk_plan(RefactorArgs a)
{
    static_assert(LEN <= 16 && kAhead * 4 <= 32, "4 bits per entry");
    const int row0 = a.blk_row0[blockIdx.x], nv = a.blk_row0[blockIdx.x + 1] - row0;
    for (int i = blockIdx.y * kThreads + threadIdx.x; i < nv; i += gridDim.y * kThreads) {
        const int r = row0 + i, b0 = a.rp[r], len = a.rp[r + 1] - b0, nl = a.dg[r] - b0;
        int col[LEN];
#pragma unroll
        for (int x = 0; x < LEN; ++x)
            col[x] = x < len ? a.ci[b0 + x] : 0x7fffffff;
        for (int k = 0; k < nl; ++k) {
            const int p = row0 + a.ci[b0 + k], y0 = a.dg[p] + 1, ep = a.rp[p + 1];
            uint32_t plan = 0;
#pragma unroll
            for (int y = 0; y < kAhead; ++y)
                if (y0 + y < ep) {
                    const int x = find_col<LEN>(col, a.ci[y0 + y]);
                    plan |= x > 0 ? (uint32_t)x << (4 * y) : 0u;
                }
            a.plan[b0 + k] = plan;
        }
    }
}

template <int LEN, bool PLAN>
__global__ void __launch_bounds__(kThreads) k_iluk_rows(RefactorArgs a, int C)
{
    extern __shared__ __align__(16) unsigned char smem[];
    double *fs = reinterpret_cast<double *>(smem);            // [LEN][kThreads]
    int *cs = reinterpret_cast<int *>(fs + LEN * kThreads);    // [LEN][kThreads]
    const int t = threadIdx.x;
    const int b = blockIdx.x / C, rank = blockIdx.x % C;
    const int row0 = a.blk_row0[b];
    const int *lptr = a.lptr + a.blk_lev0[b];
    const int nlev = a.blk_lev0[b + 1] - a.blk_lev0[b] - 1;
    const int *lrows = a.lrows + row0;
    const int vt = ((t / 32) * C + rank) * 32 + t % 32; // warps in turn over the CTAs
    for (int l = 0; l < nlev; ++l) {
        const int q1 = lptr[l + 1];
        for (int q = lptr[l] + vt; q < q1; q += kThreads * C) {
            const int r = row0 + __ldg(&lrows[q]);
            const int b0 = __ldg(&a.rp[r]), len = __ldg(&a.rp[r + 1]) - b0,
                      nl = __ldg(&a.dg[r]) - b0;
            int col[LEN];
#pragma unroll
            for (int x = 0; x < LEN; ++x)
                col[x] = x < len ? __ldg(&a.ci[b0 + x]) : 0x7fffffff;
#pragma unroll
            for (int x = 0; x < LEN; ++x) {
                cs[x * kThreads + t] = col[x];
                if (x < len)
                    fs[x * kThreads + t] = __ldcg(&a.f[b0 + x]);
            }
            // pivot k: its diagonal's and its row's end in memory and its plan;
            // its U part
            struct Place {
                int dp, ep;
                uint32_t plan;
            };
            struct Pivot {
                double upp, u[kAhead];
                int c[PLAN ? 1 : kAhead];
            };
            auto place = [&](int k) -> Place {
                if (k >= nl)
                    return Place{0, 0, 0u};
                const int p = row0 + cs[k * kThreads + t];
                return Place{__ldg(&a.dg[p]), __ldg(&a.rp[p + 1]),
                             PLAN ? __ldg(&a.plan[b0 + k]) : 0u};
            };
            auto load = [&](const Place &pl, int k, Pivot &P) {
                if (k >= nl)
                    return;
                P.upp = __ldcg(&a.f[pl.dp]);
#pragma unroll
                for (int y = 0; y < kAhead; ++y)
                    if (PLAN ? (pl.plan >> (4 * y) & 15u) != 0u : pl.dp + 1 + y < pl.ep) {
                        if constexpr (!PLAN)
                            P.c[y] = __ldg(&a.ci[pl.dp + 1 + y]);
                        P.u[y] = __ldcg(&a.f[pl.dp + 1 + y]);
                    }
            };
            Place p0 = place(0), p1 = place(1);
            Pivot P0, P1;
            load(p0, 0, P0);
            bool ok = true;
            for (int k = 0; k < nl; ++k) {
                const Place p2 = place(k + 2);
                load(p1, k + 1, P1);
                if (P0.upp == 0.0) {
                    ok = false;
                    break;
                }
                const double lip = __ddiv_rn(fs[k * kThreads + t], P0.upp);
                fs[k * kThreads + t] = lip;
                // the entries' columns differ, so their positions do: every
                // load comes before the first store
                int at[kAhead];
                double g[kAhead];
#pragma unroll
                for (int y = 0; y < kAhead; ++y) {
                    if constexpr (PLAN)
                        at[y] = (int)(p0.plan >> (4 * y) & 15u);
                    else
                        at[y] = p0.dp + 1 + y < p0.ep ? find_col<LEN>(col, P0.c[y]) : -1;
                }
#pragma unroll
                for (int y = 0; y < kAhead; ++y)
                    if (at[y] > 0)
                        g[y] = fs[at[y] * kThreads + t];
#pragma unroll
                for (int y = 0; y < kAhead; ++y)
                    if (at[y] > 0)
                        fs[at[y] * kThreads + t] = __dsub_rn(g[y], __dmul_rn(lip, P0.u[y]));
                for (int e = p0.dp + 1 + kAhead; e < p0.ep; ++e) {
                    const int x = find_col<LEN>(col, __ldg(&a.ci[e]));
                    if (x > 0)
                        fs[x * kThreads + t] =
                            __dsub_rn(fs[x * kThreads + t], __dmul_rn(lip, __ldcg(&a.f[e])));
                }
                p0 = p1;
                p1 = p2;
                P0 = P1;
            }
#pragma unroll
            for (int x = 0; x < LEN; ++x)
                if (x < len)
                    a.f[b0 + x] = fs[x * kThreads + t];
            if (!ok || fs[nl * kThreads + t] == 0.0)
                atomicExch(a.err, HEC_ERR_ZERO_PIVOT);
        }
        __syncwarp();
        if (C > 1)
            cluster_sync_all();
        else
            __syncthreads();
    }
}

// The triangular-solve layout's value slots from the new factor values: one
// CTA per chunk, thread t on row t.  Row t of chunk c takes the factor
// entries [start, start + len) of its pass (L: the multipliers; U: the
// entries right of the diagonal) and, for U, 1 / u_tt.  The chunk formats
// of trsv_layout.cpp: fixed-slot (flag bit 3: every row padded to FW entries,
// 16-byte vectors per lane in per-warp blocks; bit 5: the resident kernel's
// blocks, with 16-bit slots) and generic (per-warp widths).
template <class T> __global__ void __launch_bounds__(kThreads) k_fill_pack(FillArgs a)
{
    const int c = blockIdx.x;
    unsigned char *ch = a.pack + (size_t)a.chunks[c].x * 16;
    const int *hdr = reinterpret_cast<const int *>(ch);
    const int nrows = hdr[0];
    const bool upass = (hdr[3] & 1) != 0;
    const int t = threadIdx.x;
    if (t >= nrows)
        return;
    const int w = t / 32, lane = t % 32;
    const int64_t q = a.chunk_row0[c] + t;
    const int start = a.rm_start[q], len = a.rm_len[q];
    if (hdr[3] & 8) { // fixed-slot: 16-byte vectors of VW values per lane
        const int FW = hdr[6];
        constexpr int vb = (int)sizeof(T), VW = 16 / vb;
        const int NV = (FW + VW - 1) / VW;
        int blk, dinv_off;
        if (hdr[3] & 32) { // resident format: index vectors of 8 uint16, every block with dinv
            const int NI = (FW + 1 + 7) / 8;
            dinv_off = (NV + NI) * 512;
            blk = dinv_off + 32 * vb;
        } else {
            const bool exps = (hdr[3] & 16) != 0;
            const int ND = (FW + 3) / 4;
            dinv_off = (NV + ND) * 512;
            blk = dinv_off + 128 + (upass ? 32 * vb + 128 : 0) + (exps ? 128 : 0);
        }
        T *val = reinterpret_cast<T *>(ch + 32 + (size_t)w * blk);
        for (int k = 0; k < NV * VW; ++k)
            val[(k / VW) * 32 * VW + lane * VW + k % VW] = k < len ? T(a.f[start + k]) : T(0);
        if (upass)
            reinterpret_cast<T *>(ch + 32 + (size_t)w * blk + dinv_off)[lane] =
                T(__ddiv_rn(1.0, a.f[a.rm_diag[q]]));
        return;
    }
    const int left = nrows - w * 32;
    const int stride = left >= 32 ? 32 : (left + 3) & ~3;
    const int width = hdr[4 + w];
    T *val = reinterpret_cast<T *>(ch + hdr[4 + 8 + w]);
    for (int k = 0; k < width; ++k)
        val[k * stride + lane] = k < len ? T(a.f[start + k]) : T(0);
    if (upass) {
        T *dinv = reinterpret_cast<T *>(ch + hdr[4 + 16 + 2]);
        dinv[t] = T(__ddiv_rn(1.0, a.f[a.rm_diag[q]]));
    }
}

// The same for the long-row kernel's units (kernels.cuh): a warp per unit.
__global__ void __launch_bounds__(kThreads) k_fill_long(FillArgs a, int nunits)
{
    const int u = blockIdx.x * (kThreads / 32) + threadIdx.x / 32, lane = threadIdx.x % 32;
    if (u >= nunits)
        return;
    unsigned char *ch = a.pack + (size_t)a.chunks[u].x * 16;
    const int64_t q = a.chunk_row0[u] + lane;
    const int start = a.rm_start[q], cnt = a.rm_len[q] & 0xff, G = a.rm_len[q] >> 8;
    const int dg = a.rm_diag[q];
    float v[kLongPerLane];
#pragma unroll
    for (int k = 0; k < kLongPerLane; ++k)
        v[k] = k < cnt ? (float)a.f[start + k * G] : 0.0f;
    reinterpret_cast<float4 *>(ch)[lane] = make_float4(v[0], v[1], v[2], v[3]);
    if (dg >= 0)
        reinterpret_cast<float *>(ch + 512 + 16 * lane)[3] = (float)__ddiv_rn(1.0, a.f[dg]);
}

__global__ void k_jacobi_dinv(int n, const double *val, const int64_t *diag, double omega,
                              double *dinv, float *dinv32, int *err)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double d = val[diag[i]];
        if (d == 0.0)
            atomicExch(err, HEC_ERR_ZERO_PIVOT);
        const double v = __ddiv_rn(omega, d);
        dinv[i] = v;
        if (dinv32)
            dinv32[i] = (float)v;
    }
}

static int grid_of(int64_t n) { return (int)std::min<int64_t>(std::max<int64_t>(1, (n + 255) / 256), 4096); }

int launch_scatter_hec(int64_t nnz, const double *val, const int64_t *slot, double *ell,
                       double *tail, cudaStream_t s)
{
    k_scatter_hec<<<grid_of(nnz), 256, 0, s>>>(nnz, val, slot, ell, tail);
    return 0;
}

int launch_cast_f32(int64_t n, const double *x, float *y, cudaStream_t s)
{
    if (n > 0)
        k_cast_f32<<<grid_of(n), 256, 0, s>>>(n, x, y);
    return 0;
}

template <int LEN, bool PLAN>
static int launch_rows(const RefactorArgs &a, int nblocks, int C, cudaStream_t s)
{
    constexpr int smem = LEN * kThreads * (int)(sizeof(double) + sizeof(int));
    static PerDevice<cudaError_t> once;
    int dev = 0;
    cudaGetDevice(&dev);
    if (once.get(dev, []() {
            return cudaFuncSetAttribute(k_iluk_rows<LEN, PLAN>,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        }) != cudaSuccess)
        return -1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(nblocks * C));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = C > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k_iluk_rows<LEN, PLAN>, a, C) == cudaSuccess ? 0 : -1;
}

int launch_refactor_plan(const RefactorArgs &a, int nblocks, cudaStream_t s)
{
    // a thread per row, up to 8,192 CTAs
    const int rows = (a.largest_block + kThreads - 1) / kThreads;
    const int per = std::max(1, std::min(rows, 8192 / nblocks));
    k_iluk_plan<kPlannedRow><<<dim3(nblocks, per), kThreads, 0, s>>>(a);
    return 0;
}

int launch_refactor(const RefactorArgs &a, int nblocks, int sms, cudaStream_t s)
{
    k_gather_factor<<<grid_of(a.nent), 256, 0, s>>>(a.nent, a.val, a.src, a.f);
    // Short rows in narrow levels have few pivots to look ahead to, and what the
    // planned form sets up per row costs more than the merges (hec_refactor in
    // us, merges / planned): 2D 5-point (5 entries) 200^2 in 4 blocks, 40 rows a
    // level, 945 / 1,170; 900^2 in 4 blocks, 180 rows, 7,010 / 7,850; 500^2,
    // 250 rows, 7,150 / 5,450; 3D 7-point (7 entries) 64^3 in 64 blocks, 95
    // rows, 1,190 / 1,255; 40^3 in 8, 131 rows, 700 / 640; 20^3, 137 rows, 515 / 425.
    const int narrow = a.longest_row <= 5 ? 192 : a.longest_row <= 8 ? 96 : 0;
    // rows of more than 32 entries do not fit the registers and shared memory
    if (a.longest_row > 32 || a.level_rows <= narrow) {
        k_iluk_numeric<<<nblocks, kThreads, 0, s>>>(a);
        return 0;
    }
    // CTAs per block: while the SMs allow it and a level keeps every CTA at
    // least a warp of rows
    int C = 1;
    while (C < 8 && 2 * C * nblocks <= sms && a.level_rows >= 2 * C * 32)
        C *= 2;
    return a.longest_row <= kPlannedRow ? launch_rows<kPlannedRow, true>(a, nblocks, C, s)
                                        : launch_rows<32, false>(a, nblocks, C, s);
}

int launch_fill_pack(const FillArgs &a, int nchunks, bool fp32, cudaStream_t s)
{
    if (nchunks <= 0)
        return 0;
    if (a.long_rows) {
        const int per = kThreads / 32;
        k_fill_long<<<(nchunks + per - 1) / per, kThreads, 0, s>>>(a, nchunks);
        return 0;
    }
    if (fp32)
        k_fill_pack<float><<<nchunks, kThreads, 0, s>>>(a);
    else
        k_fill_pack<double><<<nchunks, kThreads, 0, s>>>(a);
    return 0;
}

int launch_jacobi_dinv(int n, const double *val, const int64_t *diag, double omega, double *dinv,
                       float *dinv32, int *err, cudaStream_t s)
{
    k_jacobi_dinv<<<grid_of(n), 256, 0, s>>>(n, val, diag, omega, dinv, dinv32, err);
    return 0;
}

} // namespace hec
