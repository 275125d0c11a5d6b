// k_vec.cu -- vector operations (Section 2.3, Eqs. 3-6) and the fused vector
// updates of the Krylov loops (Algorithm 4 and GMRES), each with its dot
// products reduced in the same launch.
#include "per_device.h"
#include "ptx.cuh"
#include "reduce.cuh"

namespace hec {

template <int OP>
__global__ void __launch_bounds__(kThreads) k_vec(VecArgs a)
{
    count_launch(a.st);
    SolverState *st = a.st;
    constexpr int ND = (OP == V_DOT || OP == V_NRM2SQ || OP == V_BICG_S || OP == V_CG_XR) ? 1
                       : (OP == V_BICG_XR || OP == V_CG_XRZ)                                ? 2
                                                                                            : 0;
    if (OP == V_BICG_S && st->skip)
        return;
    if ((OP == V_CG_P || OP == V_CG_PZ) && st->done)
        return;
    if (OP == V_ZERO_IF_ST && !st->zero_x)
        return;
    if ((a.guard == 1 && st->cycle_end) || (a.guard == 2 && st->done))
        return;
    const double *x = a.x;
    double *z = a.z;
    if (a.x_from_j)
        x += (int64_t)st->j * a.ldv;
    if (a.z_from_j)
        z += (int64_t)st->j * a.ldv;
    double acc[ND > 0 ? ND : 1];
#pragma unroll
    for (int d = 0; d < (ND > 0 ? ND : 1); ++d)
        acc[d] = 0.0;

    // per-launch scalars
    double c0 = a.a, c1 = a.b;
    int mode = 0;
    if (OP == V_SCALE_ST)
        c0 = st->scale;
    if (OP == V_BICG_P) {
        if (st->iters == 0) {
            mode = 1; // first pass: p = r
        } else {
            c0 = (st->rho / st->rho_prev) * (st->alpha / st->omega); // beta
            c1 = st->omega;
        }
    }
    if (OP == V_BICG_S)
        c0 = st->alpha;
    if (OP == V_CG_XR || OP == V_CG_XRZ) {
        c0 = st->alpha;
        mode = st->skip; // breakdown in alpha: no update (the sum still runs)
    }
    if (OP == V_CG_P || OP == V_CG_PZ) {
        mode = st->iters == 0; // first pass: p = z
        c0 = st->cg_beta;
    }
    if (OP == V_BICG_XR) {
        c0 = st->alpha;
        c1 = st->omega;
        mode = st->s_conv ? 1 : (st->skip ? 2 : 0);
    }

    // kUnroll elements per thread and pass, all their loads issued before the
    // first store, so that enough bytes are in flight to stream from HBM
    struct Elem {
        double p0, p1, p2, p3, p4;
    };
    auto load = [&](int i) -> Elem {
        Elem e{};
        if (OP == V_AXPBY)
            e = {x[i], z[i], 0, 0, 0};
        else if (OP == V_WAXPBY || OP == V_DOT || OP == V_BICG_S)
            e = {x[i], a.y[i], 0, 0, 0};
        else if (OP == V_NRM2SQ || OP == V_COPY || OP == V_SCALE_ST)
            e.p0 = x[i];
        else if (OP == V_BICG_P) {
            e.p0 = x[i];
            if (!mode) {
                e.p1 = a.y[i];
                e.p2 = z[i];
            }
        } else if (OP == V_BICG_XR) {
            if (mode == 0)
                e = {a.w[i], a.u[i], a.v[i], a.q[i], x[i]};
            else if (mode == 1)
                e = {a.w[i], a.u[i], 0, 0, 0};
        } else if (OP == V_CG_XR) {
            if (!mode)
                e = {a.w[i], a.u[i], a.q[i], z[i], 0};
        } else if (OP == V_CG_XRZ) {
            if (!mode)
                e = {a.w[i], a.u[i], a.q[i], z[i], a.v ? a.v[i] : 1.0};
        } else if (OP == V_CG_P || OP == V_CG_PZ) {
            e.p0 = x[i];
            if (OP == V_CG_PZ && a.v)
                e.p0 *= a.v[i];
            if (!mode)
                e.p1 = z[i];
        } else if (OP == V_AXPY_ST1)
            e = {x[i], z[i], 0, 0, 0};
        return e;
    };
    auto store = [&](int i, const Elem &e) {
        if (OP == V_AXPBY || OP == V_WAXPBY) {
            z[i] = c0 * e.p0 + c1 * e.p1;
        } else if (OP == V_DOT) {
            acc[0] = fma(e.p0, e.p1, acc[0]);
        } else if (OP == V_NRM2SQ) {
            acc[0] = fma(e.p0, e.p0, acc[0]);
        } else if (OP == V_COPY) {
            z[i] = e.p0;
        } else if (OP == V_SCALE_ST) {
            z[i] = c0 * e.p0;
        } else if (OP == V_BICG_P) {
            // x = r, y = v, z = p
            z[i] = mode ? e.p0 : fma(c0, e.p2 - c1 * e.p1, e.p0);
        } else if (OP == V_BICG_S) {
            // x = r, y = v, z = s
            const double s = fma(-c0, e.p1, e.p0);
            z[i] = s;
            acc[0] = fma(s, s, acc[0]);
        } else if (OP == V_BICG_XR) {
            // w = x (solution), u = p*, v = s*, q = t, x = s, y = r0, z = r
            if (mode == 0) {
                a.w[i] = fma(c1, e.p2, fma(c0, e.p1, e.p0));
                const double r = fma(-c1, e.p3, e.p4);
                z[i] = r;
                acc[0] = fma(r, r, acc[0]);
                acc[ND - 1] = fma(a.y[i], r, acc[ND - 1]);
            } else if (mode == 1) {
                a.w[i] = fma(c0, e.p1, e.p0);
            }
        } else if (OP == V_CG_XR) {
            // w = x (solution), u = p, q = A p, z = r
            if (!mode) {
                a.w[i] = fma(c0, e.p1, e.p0);
                const double r = fma(-c0, e.p2, e.p3);
                z[i] = r;
                acc[0] = fma(r, r, acc[0]);
            }
        } else if (OP == V_CG_XRZ) {
            // as V_CG_XR; v = d (null: ones), (r, d .* r) in the same pass
            if (!mode) {
                a.w[i] = fma(c0, e.p1, e.p0);
                const double r = fma(-c0, e.p2, e.p3);
                z[i] = r;
                acc[0] = fma(r, r, acc[0]);
                acc[ND - 1] = fma(r, __dmul_rn(e.p4, r), acc[ND - 1]);
            }
        } else if (OP == V_CG_P || OP == V_CG_PZ) {
            // x = z (preconditioned residual; V_CG_PZ: r, scaled by v), z = p
            z[i] = mode ? e.p0 : fma(c0, e.p1, e.p0);
        } else if (OP == V_AXPY_ST1) {
            z[i] = e.p1 + e.p0;
        } else if (OP == V_ZERO_IF_ST) {
            z[i] = 0.0;
        }
    };
    constexpr int kUnroll = OP == V_BICG_XR ? 2 : 4;
    const int stride = gridDim.x * kThreads;
    int i = blockIdx.x * kThreads + threadIdx.x;
    for (; i < a.n - (kUnroll - 1) * stride; i += kUnroll * stride) {
        Elem e[kUnroll];
#pragma unroll
        for (int q = 0; q < kUnroll; ++q)
            e[q] = load(i + q * stride);
#pragma unroll
        for (int q = 0; q < kUnroll; ++q)
            store(i + q * stride, e[q]);
    }
    for (; i < a.n; i += stride)
        store(i, load(i));
    if constexpr (ND > 0) {
        double v[ND];
#pragma unroll
        for (int d = 0; d < ND; ++d)
            v[d] = acc[d];
        reduce_and_finalize<ND>(v, a.red, a.op, a.result, st);
    }
}

int launch_vec(VecOp vop, const VecArgs &a, int grid, cudaStream_t s)
{
    switch (vop) {
#define HEC_VEC_CASE(OPV)                                                                        \
    case OPV:                                                                                    \
        k_vec<OPV><<<grid, kThreads, 0, s>>>(a);                                                 \
        return 0;
        HEC_VEC_CASE(V_AXPBY)
        HEC_VEC_CASE(V_WAXPBY)
        HEC_VEC_CASE(V_DOT)
        HEC_VEC_CASE(V_NRM2SQ)
        HEC_VEC_CASE(V_COPY)
        HEC_VEC_CASE(V_SCALE_ST)
        HEC_VEC_CASE(V_BICG_P)
        HEC_VEC_CASE(V_BICG_S)
        HEC_VEC_CASE(V_BICG_XR)
        HEC_VEC_CASE(V_AXPY_ST1)
        HEC_VEC_CASE(V_ZERO_IF_ST)
        HEC_VEC_CASE(V_CG_XR)
        HEC_VEC_CASE(V_CG_P)
        HEC_VEC_CASE(V_CG_XRZ)
        HEC_VEC_CASE(V_CG_PZ)
#undef HEC_VEC_CASE
    }
    return -1;
}

// ------------------------------------------------------------------ typed vector kernels

// V_COPY, V_SCALE_ST, V_AXPY_ST1, V_JACOBI with element types TX (x) and TZ (z).
template <int OP, class TX, class TZ> __global__ void __launch_bounds__(kThreads) k_vec_typed(VecArgs a)
{
    count_launch(a.st);
    SolverState *st = a.st;
    if ((a.guard == 1 && st->cycle_end) || (a.guard == 2 && st->done))
        return;
    if (OP == V_JACOBI && st && st->skip) // as the triangular solves: a skipped apply
        return;
    const TZ *d = reinterpret_cast<const TZ *>(a.dv);
    const TX *x = reinterpret_cast<const TX *>(a.xv);
    TZ *z = reinterpret_cast<TZ *>(a.zv);
    if (a.x_from_j)
        x += (int64_t)st->j * a.ldv;
    if (a.z_from_j)
        z += (int64_t)st->j * a.ldv;
    const double sc = (OP == V_SCALE_ST) ? st->scale : 1.0;
    const int stride = gridDim.x * kThreads;
    for (int i = blockIdx.x * kThreads + threadIdx.x; i < a.n; i += stride) {
        if (OP == V_COPY)
            z[i] = TZ(x[i]);
        else if (OP == V_SCALE_ST)
            z[i] = TZ(sc * double(x[i]));
        else if (OP == V_AXPY_ST1)
            z[i] = z[i] + TZ(x[i]);
        else if (OP == V_JACOBI)
            z[i] = d[i] * TZ(x[i]);
    }
}

template <int OP> static int launch_typed_op(const VecArgs &a, bool x32, bool z32, int grid, cudaStream_t s)
{
    if (x32 && z32)
        k_vec_typed<OP, float, float><<<grid, kThreads, 0, s>>>(a);
    else if (x32)
        k_vec_typed<OP, float, double><<<grid, kThreads, 0, s>>>(a);
    else if (z32)
        k_vec_typed<OP, double, float><<<grid, kThreads, 0, s>>>(a);
    else
        k_vec_typed<OP, double, double><<<grid, kThreads, 0, s>>>(a);
    return 0;
}

int launch_vec_typed(VecOp vop, const VecArgs &a, bool x32, bool z32, int grid, cudaStream_t s)
{
    switch (vop) {
    case V_COPY: return launch_typed_op<V_COPY>(a, x32, z32, grid, s);
    case V_SCALE_ST: return launch_typed_op<V_SCALE_ST>(a, x32, z32, grid, s);
    case V_AXPY_ST1: return launch_typed_op<V_AXPY_ST1>(a, x32, z32, grid, s);
    case V_JACOBI: return launch_typed_op<V_JACOBI>(a, x32, z32, grid, s);
    default: return -1;
    }
}

// ------------------------------------------------------------------ GMRES basis kernels
// The basis (m + 1 vectors of n) is streamed by every projection and update
// pass and is larger than L2 for large n; it is read under an evict-first L2
// policy so that w, which every vector group re-reads, stays in L2.
// (Measured on the 128^3 case: the mixed-precision GMRES(30) solve 5% faster,
// the FP64 one unchanged.)
__device__ __forceinline__ uint64_t basis_policy()
{
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ double ld_basis(const double *p, uint64_t pol)
{
    double v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.f64 %0, [%1], %2;"
                 : "=d"(v) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ float ld_basis(const float *p, uint64_t pol)
{
    float v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.f32 %0, [%1], %2;"
                 : "=f"(v) : "l"(p), "l"(pol));
    return v;
}


constexpr int kGroup = 8; // basis vectors per CTA in a projection

// Sums of kGroup per-thread values over a warp: the lane whose bits 4..2 are
// q ends with the warp's sum of value (bit 4: value bit 2, bit 3: value bit
// 1, bit 2: value bit 0).  Each halving step adds half as many values as the
// one before, so a warp takes 4 + 2 + 1 + 1 + 1 = 9 FP64 adds for 8 values
// where 8 separate shuffle sums take 40: on this part's FP64 pipe those sums
// cost as much as the projection itself (n = 2,097,152, k = 30 in 4,864 CTAs).
__device__ __forceinline__ double warp_sum_group(double (&v)[kGroup], int lane)
{
#pragma unroll
    for (int h = kGroup / 2, o = 16; h >= 1; h >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int q = 0; q < h; ++q) {
            const double keep = up ? v[q + h] : v[q];
            const double send = up ? v[q] : v[q + h];
            v[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    double t = v[0];
    t += __shfl_xor_sync(0xffffffffu, t, 2);
    t += __shfl_xor_sync(0xffffffffu, t, 1);
    return t;
}

// h[i] = (V_i, w), i < k.  A CTA takes one row block of one group of kGroup
// vectors, keeps kGroup running sums per thread (in T) and reduces them once at
// the end (in FP64, fixed order).  In FP64 the multiply-adds bound it: k n of
// them at two per cycle and SM (2,097,152 x 30: 101 us at 2.07 GHz, the HBM
// stream 78), so the grid holds only as many CTAs as run at once and each pays
// one reduction for many rows, and two rows' loads are in flight per thread:
// 166 -> 121 us (k = 8: 74 -> 43).  Inside a GMRES step the launch is sized
// for a whole cycle and k is the step's: the CTAs are split over the groups
// that k has, so that the first steps of a cycle use every SM as well (by the
// cycle's groups, restart 128 left 17 CTAs reading the first eight vectors:
// 128^3, 8 steps of GMRES(128) 6.4 ms, 1.9 so; 30 steps of GMRES(30) 12.9 and
// 11.0).
template <class T> __global__ void __launch_bounds__(kThreads) k_multidot(BasisArgs a)
{
    count_launch(a.st);
    int k = a.k;
    if (a.k_from_st == 1)
        k = a.st->j + 1;
    else if (a.k_from_st == 2)
        k = a.st->jend;
    const T *V = reinterpret_cast<const T *>(a.V);
    const T *w = reinterpret_cast<const T *>(a.w);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __shared__ double sh[kThreads / 32][kGroup];
    __shared__ int s_last;
    // row blocks per group: as many as there are rows or CTAs for
    const int rb = a.row_ctas ? a.row_ctas
                              : min((a.n - 1) / kThreads + 1,
                                    (int)gridDim.x / ((k + kGroup - 1) / kGroup));
    const int g0 = (int)blockIdx.x / rb * kGroup, rblk = (int)blockIdx.x % rb;
    if (g0 < k) {
        T acc[kGroup];
#pragma unroll
        for (int q = 0; q < kGroup; ++q)
            acc[q] = T(0);
        const uint64_t pol = basis_policy();
        const int stride = rb * kThreads;
        const T *Vg = V + (int64_t)g0 * a.ldv;
        const int cnt = min(kGroup, k - g0); // vectors of this group
        int i = rblk * kThreads + threadIdx.x;
        for (; i < a.n - stride; i += 2 * stride) { // two rows' loads in flight
            T v0[kGroup], v1[kGroup];
#pragma unroll
            for (int q = 0; q < kGroup; ++q)
                if (q < cnt) {
                    v0[q] = ld_basis(&Vg[q * a.ldv + i], pol);
                    v1[q] = ld_basis(&Vg[q * a.ldv + i + stride], pol);
                }
            const T w0 = w[i], w1 = w[i + stride];
#pragma unroll
            for (int q = 0; q < kGroup; ++q)
                if (q < cnt)
                    acc[q] = fma(v1[q], w1, fma(v0[q], w0, acc[q]));
        }
        if (i < a.n) {
            const T wi = w[i];
#pragma unroll
            for (int q = 0; q < kGroup; ++q)
                if (q < cnt)
                    acc[q] = fma(ld_basis(&Vg[q * a.ldv + i], pol), wi, acc[q]);
        }
        double v[kGroup];
#pragma unroll
        for (int q = 0; q < kGroup; ++q)
            v[q] = double(acc[q]);
        const double t = warp_sum_group(v, lane);
        if ((lane & 3) == 0)
            sh[wid][(lane >> 2) & 7] = t; // lane bits 4..2 = value bits 2..0
    }
    __syncthreads();
    if (g0 < k && threadIdx.x < kGroup) {
        double t = 0.0;
#pragma unroll
        for (int ww = 0; ww < kThreads / 32; ++ww)
            t += sh[ww][threadIdx.x];
        // partials layout: [vector][row block]
        const int q = g0 + threadIdx.x;
        if (q < k)
            a.red.partials[(size_t)q * rb + rblk] = t;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        unsigned tk = atomicAdd(a.red.ticket, 1u);
        s_last = (tk == gridDim.x - 1);
    }
    __syncthreads();
    if (!s_last)
        return;
    __threadfence();
    // the last CTA: eight lanes per vector, each over every eighth partial
    for (int q0 = 0; q0 < k; q0 += kThreads / 8) {
        const int q = q0 + threadIdx.x / 8, part = threadIdx.x % 8;
        double t = 0.0;
        if (q < k) {
            const double *pq = &a.red.partials[(size_t)q * rb];
#pragma unroll 4
            for (int c = part; c < rb; c += 8)
                t += __ldcg(&pq[c]);
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1)
            t += __shfl_xor_sync(0xffffffffu, t, o);
        if (q < k && part == 0) {
            if (a.op == FIN_GMRES_H1)
                a.st->h1[q] = t;
            else if (a.op == FIN_GMRES_H2)
                a.st->h2[q] = t;
            else
                a.result[q] = t;
        }
    }
    if (threadIdx.x == 0)
        *a.red.ticket = 0u;
}

int launch_multidot(BasisArgs a, int sms, cudaStream_t s, bool fp32)
{
    // a.k is the number of vectors, or an upper bound of it when k_from_st.
    // Row blocks: FP64, at most kMultidotCtas CTAs per SM over all groups;
    // FP32, two per SM and group -- more rows per thread would lengthen its
    // FP32 running sums.
    const int groups = (a.k + kGroup - 1) / kGroup;
    const int need = (int)(((int64_t)a.n + kThreads - 1) / kThreads);
    if (fp32) {
        a.row_ctas = min(need, 2 * sms);
        k_multidot<float><<<a.row_ctas * groups, kThreads, 0, s>>>(a);
        return 0;
    }
    a.row_ctas = 0; // split on the device
    const int64_t most = max(sms * kMultidotCtas, groups);
    k_multidot<double><<<(int)min((int64_t)need * groups, most), kThreads, 0, s>>>(a);
    return 0;
}

// wout = w - sum_{i<k} coef[i] V_i, optionally with (wout, wout) reduced.
template <bool NORM, class T> __global__ void __launch_bounds__(kThreads) k_basis_update(BasisArgs a)
{
    count_launch(a.st);
    int k = a.k;
    if (a.k_from_st == 1)
        k = a.st->j + 1;
    else if (a.k_from_st == 2)
        k = a.st->jend;
    const T *V = reinterpret_cast<const T *>(a.V);
    const T *w = reinterpret_cast<const T *>(a.w);
    T *wout = reinterpret_cast<T *>(a.wout);
    __shared__ T sc[kMaxRestart + 1];
    for (int q = threadIdx.x; q < k; q += kThreads)
        sc[q] = T(a.coef[q]);
    __syncthreads();
    T acc = T(0);
    const uint64_t pol = basis_policy();
    const int stride = gridDim.x * kThreads;
    for (int i = blockIdx.x * kThreads + threadIdx.x; i < a.n; i += stride) {
        T t = w[i];
        int q = 0;
        for (; q + kGroup <= k; q += kGroup) { // a group's loads first
            T v[kGroup];
#pragma unroll
            for (int g = 0; g < kGroup; ++g)
                v[g] = ld_basis(&V[(int64_t)(q + g) * a.ldv + i], pol);
#pragma unroll
            for (int g = 0; g < kGroup; ++g)
                t = fma(-sc[q + g], v[g], t);
        }
        for (; q < k; ++q)
            t = fma(-sc[q], ld_basis(&V[(int64_t)q * a.ldv + i], pol), t);
        wout[i] = t;
        if (NORM)
            acc = fma(t, t, acc);
    }
    if (NORM) {
        double v[1] = {double(acc)};
        reduce_and_finalize<1>(v, a.red, a.op, a.result, a.st);
    }
}

int launch_basis_update(const BasisArgs &a, bool with_norm, int grid, cudaStream_t s, bool fp32)
{
    if (with_norm) {
        if (fp32)
            k_basis_update<true, float><<<grid, kThreads, 0, s>>>(a);
        else
            k_basis_update<true, double><<<grid, kThreads, 0, s>>>(a);
    } else {
        if (fp32)
            k_basis_update<false, float><<<grid, kThreads, 0, s>>>(a);
        else
            k_basis_update<false, double><<<grid, kThreads, 0, s>>>(a);
    }
    return 0;
}

// wout = sum_{i<k} coef[i] V_i
template <class T> __global__ void __launch_bounds__(kThreads) k_basis_combine(BasisArgs a)
{
    count_launch(a.st);
    int k = a.k;
    if (a.k_from_st == 1)
        k = a.st->j + 1;
    else if (a.k_from_st == 2)
        k = a.st->jend;
    const T *V = reinterpret_cast<const T *>(a.V);
    T *wout = reinterpret_cast<T *>(a.wout);
    __shared__ T sc[kMaxRestart + 1];
    for (int q = threadIdx.x; q < k; q += kThreads)
        sc[q] = T(a.coef[q]);
    __syncthreads();
    const uint64_t pol = basis_policy();
    const int stride = gridDim.x * kThreads;
    for (int i = blockIdx.x * kThreads + threadIdx.x; i < a.n; i += stride) {
        T t = T(0);
        int q = 0;
        for (; q + kGroup <= k; q += kGroup) { // a group's loads first
            T v[kGroup];
#pragma unroll
            for (int g = 0; g < kGroup; ++g)
                v[g] = ld_basis(&V[(int64_t)(q + g) * a.ldv + i], pol);
#pragma unroll
            for (int g = 0; g < kGroup; ++g)
                t = fma(sc[q + g], v[g], t);
        }
        for (; q < k; ++q)
            t = fma(sc[q], ld_basis(&V[(int64_t)q * a.ldv + i], pol), t);
        wout[i] = t;
    }
}

int launch_basis_combine(const BasisArgs &a, int grid, cudaStream_t s, bool fp32)
{
    if (fp32)
        k_basis_combine<float><<<grid, kThreads, 0, s>>>(a);
    else
        k_basis_combine<double><<<grid, kThreads, 0, s>>>(a);
    return 0;
}

// ------------------------------------------------------------------ small systems
// The Arnoldi step of a small system is bound by its launches and by the
// reduction at the end of each, not by the vectors.  Here one cluster of kArnoldiCtas CTAs keeps w
// in registers (a thread owns up to kArnoldiPerThread rows), and a reduction is
// one exchange of per-CTA sums through distributed shared memory: every CTA
// stores its sums into every other's, a cluster barrier, and all add them in
// the same order.  16 CTAs: the FP64 unit is the SM's, so 8 would take the
// multiply-adds twice as long.  The basis is read four times, the last three
// from L1.  64^2 GMRES(30) solve: 11.8 -> 11.2 ms; what bounds it now is the
// chain of FP64 adds (65 cycles each, one in flight per warp) of three
// reductions and the Givens step.
struct ArnoldiShared {
    double part[3][kArnoldiCtas][kArnoldiRestart + 1]; // per exchange: each CTA's sums
    double warp[kThreads / 32][kArnoldiRestart + 2];
    double h[kArnoldiRestart + 1];
};

// Sums over the cluster of the cnt values that warp w of this CTA left in
// S.warp[w][0 .. cnt), into S.h; exchange x of the launch.
__device__ __forceinline__ void cluster_sums(ArnoldiShared &S, int x, int cnt, int rank)
{
    const int t = threadIdx.x;
    __syncthreads();
    if (t < cnt) {
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < kThreads / 32; ++w)
            s += S.warp[w][t];
        const uint32_t to = smem_u32(&S.part[x][rank][t]);
        for (int c = 0; c < kArnoldiCtas; ++c)
            st_cluster(mapa_shared(to, c), s);
    }
    cluster_sync_all();
    for (int q0 = 0; q0 < cnt; q0 += kThreads / 8) { // eight lanes per value
        const int q = q0 + t / 8, l = t % 8;
        double s = q < cnt ? S.part[x][l][q] + S.part[x][l + 8][q] : 0.0;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1)
            s += __shfl_xor_sync(0xffffffffu, s, o);
        if (q < cnt && l == 0)
            S.h[q] = s;
    }
    __syncthreads();
}

template <class T> __global__ void __launch_bounds__(kThreads) k_arnoldi(BasisArgs a)
{
    static_assert(kArnoldiCtas == 16, "cluster_sums adds two CTAs per lane");
    __shared__ ArnoldiShared S;
    count_launch(a.st);
    SolverState *st = a.st;
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const int rank = (int)cluster_ctarank();
    cluster_sync_all(); // every CTA runs before another one stores into it
    const int j = st->j, k = j + 1;
    const T *__restrict__ V = reinterpret_cast<const T *>(a.V);
    const T *w_in = reinterpret_cast<const T *>(a.w);
    constexpr int Q = kArnoldiPerThread, stride = kArnoldiCtas * kThreads;
    const int i0 = rank * kThreads + t;
    T w[Q];
    T ww = T(0);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        w[q] = i0 + q * stride < a.n ? w_in[i0 + q * stride] : T(0);
        ww = fma(w[q], w[q], ww);
    }
    // warp sums of (V_g, w), g < k, into S.warp[wid]
    auto project = [&]() {
        for (int g0 = 0; g0 < k; g0 += kGroup) {
            T acc[kGroup];
#pragma unroll
            for (int g = 0; g < kGroup; ++g)
                acc[g] = T(0);
#pragma unroll
            for (int q = 0; q < Q; ++q)
                if (i0 + q * stride < a.n) {
#pragma unroll
                    for (int g = 0; g < kGroup; ++g)
                        if (g0 + g < k)
                            acc[g] = fma(__ldg(&V[(int64_t)(g0 + g) * a.ldv + i0 + q * stride]),
                                         w[q], acc[g]);
                }
            double v[kGroup];
#pragma unroll
            for (int g = 0; g < kGroup; ++g)
                v[g] = double(acc[g]);
            const double s = warp_sum_group(v, lane);
            const int g = g0 + ((lane >> 2) & 7);
            if ((lane & 3) == 0 && g < k)
                S.warp[wid][g] = s;
        }
    };
    // w -= V h
    auto subtract = [&]() {
        for (int g0 = 0; g0 < k; g0 += kGroup)
#pragma unroll
            for (int q = 0; q < Q; ++q)
                if (i0 + q * stride < a.n) {
                    T v[kGroup];
#pragma unroll
                    for (int g = 0; g < kGroup; ++g)
                        if (g0 + g < k)
                            v[g] = __ldg(&V[(int64_t)(g0 + g) * a.ldv + i0 + q * stride]);
#pragma unroll
                    for (int g = 0; g < kGroup; ++g)
                        if (g0 + g < k)
                            w[q] = fma(-T(S.h[g0 + g]), v[g], w[q]);
                }
    };
    auto norm2 = [&]() {
        T s = T(0);
#pragma unroll
        for (int q = 0; q < Q; ++q)
            s = fma(w[q], w[q], s);
        return s;
    };
    project();
    const double ws = warp_sum(double(ww));
    if (lane == 0)
        S.warp[wid][k] = ws;
    cluster_sums(S, 0, k + 1, rank); // h1, ||w||^2
    if (rank == 0) {
        if (t < k)
            st->h1[t] = S.h[t];
        if (t == 0)
            st->w0norm = sqrt(S.h[k]);
    }
    subtract();
    project();
    cluster_sums(S, 1, k, rank); // h2
    if (rank == 0 && t < k)
        st->h2[t] = S.h[t];
    subtract();
    const double ns = warp_sum(double(norm2()));
    __syncthreads(); // S.h and S.warp have been read
    if (lane == 0)
        S.warp[wid][0] = ns;
    cluster_sums(S, 2, 1, rank);
    const double nn = S.h[0];
    // v_{j+1} (not read when the cycle ends here)
    const double sc = 1.0 / sqrt(nn);
    T *vn = reinterpret_cast<T *>(a.wout) + (int64_t)k * a.ldv;
#pragma unroll
    for (int q = 0; q < Q; ++q)
        if (i0 + q * stride < a.n)
            vn[i0 + q * stride] = T(sc * double(w[q]));
    if (rank == 0)
        finalize_gmres_step(&nn, st);
}

static cudaLaunchConfig_t arnoldi_config(cudaLaunchAttribute *attr, cudaStream_t s)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(kArnoldiCtas);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = s;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = kArnoldiCtas;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

template <class T> static bool arnoldi_ready()
{
    // a cluster of 16 is above the portable size: allowed once per device
    static PerDevice<bool> once;
    int dev = 0;
    cudaGetDevice(&dev);
    return once.get(dev, []() {
        cudaLaunchAttribute attr;
        const cudaLaunchConfig_t cfg = arnoldi_config(&attr, nullptr);
        int clusters = 0;
        const bool ok =
            cudaFuncSetAttribute(k_arnoldi<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
                cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&clusters, k_arnoldi<T>, &cfg) == cudaSuccess &&
            clusters > 0;
        if (!ok)
            cudaGetLastError(); // the several-launch form runs instead
        return ok;
    });
}

bool arnoldi_available(bool fp32) { return fp32 ? arnoldi_ready<float>() : arnoldi_ready<double>(); }

int launch_arnoldi(const BasisArgs &a, cudaStream_t s, bool fp32)
{
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = arnoldi_config(&attr, s);
    const cudaError_t e = fp32 ? cudaLaunchKernelEx(&cfg, k_arnoldi<float>, a)
                               : cudaLaunchKernelEx(&cfg, k_arnoldi<double>, a);
    return e == cudaSuccess ? 0 : -1;
}

// ------------------------------------------------------------------ small kernels

// Back substitution R y = g of the Givens-reduced Hessenberg matrix (one thread).
__global__ void k_gmres_lsq(SolverState *st)
{
    count_launch(st);
    if (threadIdx.x != 0)
        return;
    const int je = st->jend, ld = kMaxRestart;
    for (int i = je - 1; i >= 0; --i) {
        double s = st->g[i];
        for (int l = i + 1; l < je; ++l)
            s -= st->H[i * ld + l] * st->y[l];
        st->y[i] = s / st->H[i * ld + i];
    }
}

int launch_gmres_lsq(SolverState *st, cudaStream_t s)
{
    k_gmres_lsq<<<1, 32, 0, s>>>(st);
    return 0;
}

// Loop condition of the solve graph's while node.
__global__ void k_loopcond(SolverState *st)
{
    count_launch(st);
    if (threadIdx.x == 0)
        set_cond(st, st->h_while, !st->done);
}

int launch_loopcond(SolverState *st, cudaStream_t s)
{
    k_loopcond<<<1, 32, 0, s>>>(st);
    return 0;
}

} // namespace hec
