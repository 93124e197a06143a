// Pair passes of the tangent-point library: the O(|E|^2) loops over ordered pairs of edges that
// share no vertex.  Every pass is a gather: one thread owns TPT target edges I and loops over all
// source edges J staged through shared memory, so each output row is written by exactly one thread
// (no atomics, deterministic).  A persistent grid pulls (target block, source chunk) items from a
// queue; chunk results land in partial slots that a second kernel sums per row and gathers to the
// vertices through the vertex->edge incidence lists.
//
//   energy  : E_I   = sum_J E_IJ,  E_IJ = (1/4) l_I l_J sum_{a,b} k(g_ia, g_jb, T_I)   (Eqs. 3, 17-18)
//   diff    : d/d(g_i1, g_i2) of sum_J (E_IJ + E_JI)                                 (Sec. 5.1)
//   apply   : h_I = sum_J 2 w_IJ (du_I - <T_I,T_J> du_J),  l_I = sum_J (w0_IJ + w0_JI)(ub_I - ub_J)
//             (A u)_{i1,i2} = -/+ h_I / l_I + l_I / 2                                 (Secs. 5.2.2-5.2.3)
//   diag    : diag(A)_v = sum_{I ni v} [2 sum_J w_IJ / l_I^2 + sum_J (w0_IJ + w0_JI) / 4]
//
// w_IJ = (1/4) l_I l_J sum_ab |d|^-p and w0_IJ = (1/4) l_I l_J sum_ab |T_I x d|^2 |d|^-(4+p) with
// d = g_ia - g_jb and p = 2 sigma + 1.  The quadratic forms of Eq. 21 and Sec. 5.2.3 reduce to these
// row sums because w_IJ is symmetric in (I, J) and only w0_IJ + w0_JI enters the low-order form.
//
// Precision (template PREC): P64 all FP64; P32 FP32 pair arithmetic with the partial sums of every
// tile folded into FP64 accumulators; PMIX as P32 but positions are double-float (hi + lo) so that
// d = g_ia - g_jb keeps full FP32 relative accuracy, and pairs with |g_i1 - g_j1| below the near
// cutoff are evaluated in FP64 from the FP64 inputs instead.
//
// |T x d|^2 is formed as |d - (T.d) T|^2 (never as |d|^2 - (T.d)^2, which cancels for the nearly
// parallel pairs along the curve).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "tpe_internal.cuh"

namespace tpe {

#define TPE_CHECK(x)                          \
    do {                                      \
        cudaError_t e_ = (x);                 \
        if (e_ != cudaSuccess) return e_;     \
    } while (0)

// ---------------------------------------------------------------------------------- K0: edge records

// isfinite without an FP64 comparison
__device__ __forceinline__ bool finite64(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

// a / b from ib = 1 / b with one residual correction: within an ulp of the quotient, three FP64 instructions after
// the shared reciprocal.  An infinite or zero quotient has no residual and stays as it is.
__device__ __forceinline__ double div_by(double a, double b, double ib)
{
    const double q = a * ib, r = fma(-q, b, a);
    return finite64(r) ? fma(r, ib, q) : q;
}

// The per-edge kernels run in blocks of 64: FP64 instructions bound them (2 per clock and SM), so what counts is
// that a short graph spreads over many SMs (256 edges in one block of 256 took 10 us).
constexpr int kRecThreads = 64;

__global__ void k_records(int nE, const double *__restrict__ g, const int *__restrict__ E, RecF *__restrict__ recF,
                          RecLo *__restrict__ recLo, RecD *__restrict__ recD, double *__restrict__ ell,
                          double *__restrict__ T, double *__restrict__ x, int *__restrict__ err,
                          float *__restrict__ ell_lo)
{
    int I = blockIdx.x * blockDim.x + threadIdx.x;
    if (I >= nE) return;
    int i1 = E[2 * I], i2 = E[2 * I + 1];
    double p1[3], p2[3], e[3];
    for (int k = 0; k < 3; ++k) {
        p1[k] = g[3 * i1 + k];
        p2[k] = g[3 * i2 + k];
        e[k] = p2[k] - p1[k];
    }
    double l = sqrt(e[0] * e[0] + e[1] * e[1] + e[2] * e[2]);
    const bool fin = finite64(l) && finite64(p1[0] + p1[1] + p1[2]) && finite64(p2[0] + p2[1] + p2[2]);
    if (!fin) {
        atomicCAS(err, 0, (int)TP_ERR_NONFINITE);
        l = 1.0;
    } else if (!(l > 0.0)) {
        atomicCAS(err, 0, (int)TP_ERR_DEGENERATE_EDGE);
        l = 1.0;
    }
    const double li = 1.0 / l;
    double t[3] = {div_by(e[0], l, li), div_by(e[1], l, li), div_by(e[2], l, li)};
    ell[I] = l;
    if (ell_lo) ell_lo[I] = (float)(l - (double)(float)l);
    for (int k = 0; k < 3; ++k) {
        T[3 * I + k] = t[k];
        x[3 * I + k] = 0.5 * (p1[k] + p2[k]);
    }
    if (recF) {
        float h1[3], h2[3];
        for (int k = 0; k < 3; ++k) {
            h1[k] = (float)p1[k];
            h2[k] = (float)p2[k];
        }
        RecF r;
        r.a = make_float4(h1[0], h1[1], h1[2], (float)l);
        r.b = make_float4(h2[0], h2[1], h2[2], (float)t[0]);
        r.c = make_float4((float)t[1], (float)t[2], __int_as_float(i1), __int_as_float(i2));
        recF[I] = r;
        if (recLo) {
            RecLo q;
            q.lo = make_float4((float)(p1[0] - (double)h1[0]), (float)(p1[1] - (double)h1[1]),
                               (float)(p1[2] - (double)h1[2]), (float)(p2[0] - (double)h2[0]));
            float th[3] = {(float)t[0], (float)t[1], (float)t[2]};
            q.lo2 = make_float4((float)(p2[1] - (double)h2[1]), (float)(p2[2] - (double)h2[2]),
                                (float)(t[0] - (double)th[0]), (float)(t[1] - (double)th[1]));
            q.lo3 = make_float4((float)(t[2] - (double)th[2]), (float)e[0], (float)e[1], (float)e[2]);
            recLo[I] = q;
        }
    }
    if (recD) {
        RecD r;
        r.a0 = make_double2(p1[0], p1[1]);
        r.a1 = make_double2(p1[2], l);
        r.b0 = make_double2(p2[0], p2[1]);
        r.b1 = make_double2(p2[2], t[0]);
        r.c0 = make_double2(t[1], t[2]);
        r.i1 = i1;
        r.i2 = i2;
        r.pad0 = r.pad1 = 0;
        recD[I] = r;
    }
}

// Per-edge data of u for an apply: du = (u_j2 - u_j1)/l_J, ub = (u_j1 + u_j2)/2 (3 components).
__global__ void k_urecs(int nE, const double *__restrict__ u, const int *__restrict__ E,
                        const double *__restrict__ ell, URecF *__restrict__ uf, URecD *__restrict__ ud)
{
    int I = blockIdx.x * blockDim.x + threadIdx.x;
    if (I >= nE) return;
    int i1 = E[2 * I], i2 = E[2 * I + 1];
    const double l = ell[I], li = 1.0 / l;
    double du[3], ub[3];
    for (int k = 0; k < 3; ++k) {
        double a = u[3 * i1 + k], b = u[3 * i2 + k];
        du[k] = div_by(b - a, l, li);
        ub[k] = 0.5 * (a + b);
    }
    if (uf) {
        float dh[3], uh[3], dl[3], ul[3];
        for (int k = 0; k < 3; ++k) {
            dh[k] = (float)du[k];
            uh[k] = (float)ub[k];
            dl[k] = (float)(du[k] - (double)dh[k]);
            ul[k] = (float)(ub[k] - (double)uh[k]);
        }
        URecF r;
        r.a = make_float4(dh[0], dh[1], dh[2], uh[0]);
        r.b = make_float4(uh[1], uh[2], dl[0], dl[1]);
        r.c = make_float4(dl[2], ul[0], ul[1], ul[2]);
        uf[I] = r;
    }
    if (ud) {
        URecD r;
        r.du0 = make_double2(du[0], du[1]);
        r.du1 = make_double2(du[2], 0.0);
        r.ub0 = make_double2(ub[0], ub[1]);
        r.ub1 = make_double2(ub[2], 0.0);
        ud[I] = r;
    }
}

}  // namespace tpe

#include "pair_device.cuh"

namespace tpe {

// Resident CTAs per SM the register allocation is sized for: the differential and the 4-target
// apply / diag need more than the 170 registers per thread that 3 CTAs allow, so they get 2.  The FP64 energy is held to
// six (80 registers; with 84 it has five, and 3,000 edges take 2,450 us instead of 2,040).
template <int PREC, int OP, int TPT>
__host__ __device__ constexpr int pair_min_blocks()
{
    return PREC == P64 ? (OP == OP_ENERGY ? 6 : 1) : ((OP == OP_DIFF || (TPT >= 4 && OP != OP_ENERGY)) ? 2 : 3);
}

template <int PREC, int OP, int TPT, bool FAST>
__global__ void __launch_bounds__(kThreads, (pair_min_blocks<PREC, OP, TPT>())) k_pairs(const PairArgs pa)
{
    using R = typename RealOf<PREC>::type;
    constexpr bool NEEDU = (OP == OP_APPLY);
    __shared__ Tile<PREC, NEEDU> tl;
    __shared__ int s_item;
    __shared__ float s_box[2][kThreads / 32][6];
    constexpr int S = part_stride<OP>();
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(pa.counter, 1);
        __syncthreads();
        const int it = s_item;
        __syncthreads();
        if (it >= pa.n_items) {
            queue_done(it, pa.n_items, pa.counter);
            break;
        }
        const WorkItem w = pa.items[it];
        if (pa.skip && pa.skip[w.pad]) continue;  // problem already converged: its output is not used
        Tgt<R> tg[TPT];
        UVal<R> tu[TPT];
        int tI[TPT];
#pragma unroll
        for (int k = 0; k < TPT; ++k) {
            int loc = threadIdx.x + k * kThreads;
            tI[k] = w.tgt0 + min(loc, w.ntgt - 1);
            load_target<PREC>(tg[k], tI[k], pa.recF, pa.recLo, pa.recD);
            if constexpr (NEEDU) load_uval<PREC>(tu[k], pa.urecF, pa.urecD, tI[k]);
        }
        Acc64<OP> A[TPT];
        Acc32<PREC, OP> a[TPT];
#pragma unroll
        for (int k = 0; k < TPT; ++k) acc64_zero<OP>(A[k]);
        float tbox[6];  // bounding box of this warp's targets (mixed path): min xyz, max xyz
        if constexpr (PREC == PMIX) {
            float b[6] = {1e30f, 1e30f, 1e30f, -1e30f, -1e30f, -1e30f};
#pragma unroll
            for (int k = 0; k < TPT; ++k) box_add(b, tg[k].p1, tg[k].p2);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                for (int q = 0; q < 6; ++q) {
                    float v = __shfl_xor_sync(0xffffffffu, b[q], o);
                    b[q] = q < 3 ? fminf(b[q], v) : fmaxf(b[q], v);
                }
            for (int q = 0; q < 6; ++q) tbox[q] = b[q];
        }
        int tiles_since_fold = 0;
        for (int s0 = w.src0; s0 < w.src1; s0 += kTile) {
            const int cnt = min(kTile, w.src1 - s0);
            __syncthreads();
            float sb[6] = {1e30f, 1e30f, 1e30f, -1e30f, -1e30f, -1e30f};
            if (threadIdx.x < cnt) {
                int J = s0 + threadIdx.x;
                if constexpr (PREC == P64) {
                    tl.r[threadIdx.x] = pa.recD[J];
                    if constexpr (NEEDU) tl.u[threadIdx.x] = pa.urecD[J];
                } else {
                    RecF r = pa.recF[J];
                    tl.r[threadIdx.x] = r;
                    if constexpr (PREC == PMIX) {
                        tl.lo[threadIdx.x] = pa.recLo[J];
                        box_add(sb, V3<float>{r.a.x, r.a.y, r.a.z}, V3<float>{r.b.x, r.b.y, r.b.z});
                    }
                    if constexpr (NEEDU) tl.u[threadIdx.x] = pa.urecF[J];
                }
            }
            if constexpr (PREC == PMIX) block_box(sb, s_box[1]);  // contains the barriers
            else __syncthreads();
            if (tiles_since_fold == 0) {
#pragma unroll
                for (int k = 0; k < TPT; ++k) acc_zero<PREC, OP>(a[k]);
            }
            const bool check = !(s0 + cnt - 1 < w.nb_lo || s0 > w.nb_hi);
            int mode = 2;
            if constexpr (PREC == PMIX) {
                // squared distance between the two boxes decides the arithmetic of the whole tile
                float g2 = 0.f;
                for (int q = 0; q < 3; ++q) {
                    float gap = fmaxf(fmaxf(sb[q] - tbox[3 + q], tbox[q] - sb[3 + q]), 0.f);
                    g2 += gap * gap;
                }
                const float nr2 = (OP == OP_DIFF) ? pa.kp.near2f_diff : pa.kp.near2f;
                mode = (g2 < nr2) ? 2 : (g2 < pa.kp.mid2f ? 1 : 0);
                // In the Gram weights |T x d|^2 enters only the low-order weight w0, whose near-pair
                // entries are ~(kappa l)^2 / 4 of the high-order ones, so FP32 double-float accuracy
                // suffices there: no FP64 near path for apply / diag.
                if constexpr (OP == OP_APPLY || OP == OP_DIAG) mode = min(mode, 1);
            }
            if (check || mode == 2) {
                if (check && (OP == OP_APPLY || OP == OP_DIAG) && PREC == PMIX)
                    tile_loop<PREC, OP, TPT, FAST, true, 1>(tg, tI, tu, tl, cnt, s0, a, A, pa);
                else if (check)
                    tile_loop<PREC, OP, TPT, FAST, true, 2>(tg, tI, tu, tl, cnt, s0, a, A, pa);
                else
                    tile_loop<PREC, OP, TPT, FAST, false, 2>(tg, tI, tu, tl, cnt, s0, a, A, pa);
            } else if (mode == 1) {
                tile_loop<PREC, OP, TPT, FAST, false, 1>(tg, tI, tu, tl, cnt, s0, a, A, pa);
            } else {
                tile_loop<PREC, OP, TPT, FAST, false, 0>(tg, tI, tu, tl, cnt, s0, a, A, pa);
            }
            // fold the tile accumulators into FP64 every 4 tiles and at the end of the item
            if (++tiles_since_fold == 4 || s0 + kTile >= w.src1) {
#pragma unroll
                for (int k = 0; k < TPT; ++k) acc_add(A[k], a[k]);
                tiles_since_fold = 0;
            }
        }
        // write this item's partial results for the valid targets
#pragma unroll
        for (int k = 0; k < TPT; ++k) {
            int loc = threadIdx.x + k * kThreads;
            if (loc >= w.ntgt) continue;
            int I = w.tgt0 + loc;
            double *o = pa.part + ((size_t)w.slot * pa.nE + I) * S;
            if constexpr (OP == OP_ENERGY) {
                o[0] = A[k].s;
            } else if constexpr (OP == OP_DIFF) {
                // G_i1 = (1/4)[-T S + l_I G1 - (Id - T T^t) GT],  G_i2 = (1/4)[T S + l_I G2 + (Id - T T^t) GT]
                const double *T = pa.na.T + 3 * I;
                double l = pa.na.ell[I];
                double tg3[3] = {T[0], T[1], T[2]};
                const double quarter = PREC == PMIX ? 0.25 / (double)pa.kp.sum_scale : 0.25;
                double gt = tg3[0] * A[k].GT[0] + tg3[1] * A[k].GT[1] + tg3[2] * A[k].GT[2];
                for (int c = 0; c < 3; ++c) {
                    double pgt = A[k].GT[c] - gt * tg3[c];
                    o[c] = quarter * (-tg3[c] * A[k].S + l * A[k].G1[c] - pgt);
                    o[3 + c] = quarter * (tg3[c] * A[k].S + l * A[k].G2[c] + pgt);
                }
            } else if constexpr (OP == OP_APPLY) {
                // h_I / l_I = A1 / 2 (to +i2, -i1) and l_I / 2 = l_I A2 / 8 (to both endpoints)
                double l = pa.na.ell[I];
                for (int c = 0; c < 3; ++c) {
                    o[c] = 0.5 * A[k].A1[c];
                    o[3 + c] = 0.125 * l * A[k].A2[c];
                }
            } else {
                double l = pa.na.ell[I];
                o[0] = A[k].Sw / (2.0 * l) + l * A[k].Sw0 / 16.0;
            }
        }
    }
}

// ---------------------------------------------------------------------------------- reductions / gathers

// Sum of the ns slots of value i (slot stride `step`) by the eight warps of a 256-thread block, 32 values a
// block: warp w adds slots w, w + 8, ... and the partial sums are added in warp order.  Valid in warp 0.  One
// thread per value waits for 64 slots in turn (12 us at 256 edges).
__device__ __forceinline__ double slot_sum(const double *part, size_t step, size_t i, int ns, double (*sh)[32])
{
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double s = 0.0;
#pragma unroll 4
    for (int k = w; k < ns; k += 8) s += part[k * step + i];
    sh[w][lane] = s;
    __syncthreads();
    if (w == 0)
        for (int k = 1; k < 8; ++k) s += sh[k][lane];
    return s;
}

// rows[I] = (l_I / 4) sum_slots part[slot][I]; 32 rows per block
__global__ void __launch_bounds__(256) k_energy_rows(int nE, const int *__restrict__ eslots, const double *__restrict__ part,
                                                     const double *__restrict__ ell, double *__restrict__ rows)
{
    __shared__ double sh[8][32];
    const int I = blockIdx.x * 32 + (threadIdx.x & 31);
    const double s = slot_sum(part, nE, min(I, nE - 1), I < nE ? eslots[I] : 0, sh);
    if (threadIdx.x < 32 && I < nE) rows[I] = 0.25 * ell[I] * s;
}

// Per-problem sums of a per-edge array (deterministic: one block per problem, fixed order).  One block reads
// the whole of a problem, so its loads in flight set the time: 1,024 threads with eight loads each take
// 32,768 rows in 8 us where 256 threads with one took 65.
constexpr int kSegThreads = 1024;
__global__ void __launch_bounds__(kSegThreads) k_segment_sum(const int *__restrict__ off, const double *__restrict__ x,
                                                             double *__restrict__ out)
{
    const int q = blockIdx.x, b = off[q], e = off[q + 1];
    double s = 0.0;
#pragma unroll 8
    for (int i = b + threadIdx.x; i < e; i += kSegThreads) s += x[i];
    __shared__ double sh[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x >= 32) return;
    s = sh[threadIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) out[q] = s;
}

// out_v = sum_{(I, slot) in inc(v)} sum_k part[k][I][slot*3 + c] (diff: slot selects G_i1 / G_i2;
// apply: -/+ first triple plus the second triple).
template <int OP>
__global__ void k_vertex_gather(int nV, int nE, const int *__restrict__ inc_ptr, const int *__restrict__ inc,
                                const int *__restrict__ eslots, const double *__restrict__ part,
                                double *__restrict__ out)
{
    int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= nV) return;
    double o[3] = {0, 0, 0};
    for (int k = inc_ptr[v]; k < inc_ptr[v + 1]; ++k) {
        int I = inc[k] >> 1, sl = inc[k] & 1;
        int ns = eslots[I];
        for (int q = 0; q < ns; ++q) {
            const double *p = part + ((size_t)q * nE + I) * (OP == OP_DIAG ? 1 : 6);
            if constexpr (OP == OP_DIFF) {
                for (int c = 0; c < 3; ++c) o[c] += p[3 * sl + c];
            } else if constexpr (OP == OP_APPLY) {
                double sg = sl ? 1.0 : -1.0;
                for (int c = 0; c < 3; ++c) o[c] += sg * p[c] + p[3 + c];
            } else {
                o[0] += p[0];
            }
        }
    }
    if constexpr (OP == OP_DIAG) {
        out[v] = o[0];
    } else {
        for (int c = 0; c < 3; ++c) out[3 * v + c] = o[c];
    }
}

// Two-stage gather for many slots: each edge's slots are summed once (k_edge_slots), then every vertex
// combines its edges' sums (k_vertex_from_edges).  The one-stage gather reads an edge's slots once per
// endpoint, twice the traffic when an edge has tens of slots (the symmetric passes on long curves).
template <int OP>
__global__ void __launch_bounds__(256) k_edge_slots(int nE, const int *__restrict__ eslots, const double *__restrict__ part,
                                                    double *__restrict__ esum)
{
    constexpr int W = OP == OP_DIAG ? 1 : 6;
    __shared__ double sh[8][32];
    const int i = blockIdx.x * 32 + (threadIdx.x & 31), n = nE * W;
    const double s = slot_sum(part, n, min(i, n - 1), i < n ? eslots[i / W] : 0, sh);
    if (threadIdx.x < 32 && i < n) esum[i] = s;
}

template <int OP>
__global__ void k_vertex_from_edges(int nV, const int *__restrict__ inc_ptr, const int *__restrict__ inc,
                                    const double *__restrict__ esum, double *__restrict__ out)
{
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= nV) return;
    double o[3] = {0, 0, 0};
    for (int k = inc_ptr[v]; k < inc_ptr[v + 1]; ++k) {
        const int I = inc[k] >> 1, sl = inc[k] & 1;
        if constexpr (OP == OP_DIAG) {
            o[0] += esum[I];
        } else {
            const double *p = esum + 6 * (size_t)I;
            if constexpr (OP == OP_DIFF) {
                for (int c = 0; c < 3; ++c) o[c] += p[3 * sl + c];
            } else {
                const double sg = sl ? 1.0 : -1.0;
                for (int c = 0; c < 3; ++c) o[c] += sg * p[c] + p[3 + c];
            }
        }
    }
    if constexpr (OP == OP_DIAG) {
        out[v] = o[0];
    } else {
        for (int c = 0; c < 3; ++c) out[3 * v + c] = o[c];
    }
}

// out from per-edge sums
template <int OP>
static cudaError_t vertices_from_edges(Ctx &c, const double *esum, double *out, cudaStream_t s)
{
    if (c.nV == 0) return cudaSuccess;
    k_vertex_from_edges<OP><<<(c.nV + 255) / 256, 256, 0, s>>>(c.nV, c.d_inc_ptr, c.d_inc, esum, out);
    c.launches++;
    return cudaGetLastError();
}

// Sum the partial slots of a pass into the per-vertex output, in one or two stages by slot count.
template <int OP>
static cudaError_t gather_slots(Ctx &c, const Ctx::Plan &pl, double *out, cudaStream_t s)
{
    if (c.nV == 0) return cudaSuccess;
    if (pl.max_slots > 2 && c.d_esum) {
        const int values = c.nE * (OP == OP_DIAG ? 1 : 6);
        k_edge_slots<OP><<<(values + 31) / 32, 256, 0, s>>>(c.nE, pl.d_eslots, c.d_part, c.d_esum);
        c.launches++;
        return vertices_from_edges<OP>(c, c.d_esum, out, s);
    } else {
        k_vertex_gather<OP><<<(c.nV + 255) / 256, 256, 0, s>>>(c.nV, c.nE, c.d_inc_ptr, c.d_inc, pl.d_eslots, c.d_part,
                                                              out);
        c.launches++;
    }
    return cudaGetLastError();
}

cudaError_t gather_apply(Ctx &c, const Ctx::Plan &pl, double *Au, cudaStream_t s)
{
    return gather_slots<OP_APPLY>(c, pl, Au, s);
}

cudaError_t vertices_apply(Ctx &c, const double *esum, double *Au, cudaStream_t s)
{
    return vertices_from_edges<OP_APPLY>(c, esum, Au, s);
}

// ---------------------------------------------------------------------------------- planning

// Resize the buffer of partial sums.  The old one is freed first (on the longest curves both would not fit), so a
// failed allocation takes the old size back, or holds nothing where even that is gone: part_elems is always
// what d_part holds, and every pass reserves what it writes before it launches.
cudaError_t part_resize(Ctx &c, size_t elems)
{
    if (c.capturing) return cudaErrorStreamCaptureUnsupported;  // a captured pass reserved its part before
    graphs_reset(c);  // captured blocks hold the old buffer
    TPE_CHECK(cudaFree(c.d_part));
    const size_t old = c.part_elems;
    c.d_part = nullptr;
    c.part_elems = 0;
    cudaError_t e = cudaMalloc(&c.d_part, sizeof(double) * elems);
    if (e == cudaSuccess) {
        c.part_elems = elems;
        return e;
    }
    cudaGetLastError();  // reported by the return value
    c.d_part = nullptr;
    if (old && old < elems && cudaMalloc(&c.d_part, sizeof(double) * old) == cudaSuccess) {
        c.part_elems = old;
    } else {
        c.d_part = nullptr;
        cudaGetLastError();
    }
    return e;
}

cudaError_t part_reserve(Ctx &c, size_t elems) { return elems <= c.part_elems ? cudaSuccess : part_resize(c, elems); }

// Whether partial sums of this size may be taken for a faster form of a pass that has another: at most 32 GB, and
// half of the free memory on top of what the buffer already holds.
bool part_fits(const Ctx &c, size_t elems)
{
    const size_t bytes = sizeof(double) * elems;
    if (bytes > (size_t)32 << 30) return false;
    if (elems <= c.part_elems) return true;
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) free_b = 0;
    return bytes <= sizeof(double) * c.part_elems + free_b / 2;
}

void plan_free(Ctx::Plan &pl)
{
    if (pl.d_items) cudaFree(pl.d_items);
    if (pl.d_eslots) cudaFree(pl.d_eslots);
    pl = Ctx::Plan{};
}

// Copy a work list to the device; on failure the plan is empty (d_items NULL).
cudaError_t plan_upload(Ctx::Plan &pl, const std::vector<WorkItem> &items, const std::vector<int> &eslots)
{
    const size_t ni = items.size(), ns = eslots.size();
    cudaError_t e = cudaMalloc(&pl.d_items, sizeof(WorkItem) * std::max<size_t>(1, ni));
    if (e == cudaSuccess) e = cudaMalloc(&pl.d_eslots, sizeof(int) * std::max<size_t>(1, ns));
    if (e == cudaSuccess) e = cudaMemcpy(pl.d_items, items.data(), sizeof(WorkItem) * ni, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(pl.d_eslots, eslots.data(), sizeof(int) * ns, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        cudaGetLastError();
        plan_free(pl);
    }
    return e;
}

constexpr int kMinChunk = 4;  // sources of the shortest item

// Source chunks of the gather passes.  Items of at least eight source tiles amortise their targets; where those would
// leave resident CTAs without an item, one wave of short items is faster: a pass over 256 edges was two CTAs, each
// walking all 256 sources in turn (energy 284 us, FP64 differential 2,117 us), and is 64 to 128 of them.
struct Chunking {
    int tb;              // targets per item
    long long resident;  // resident CTAs
    double total;        // squared edges, summed over problems
    bool small = false;  // the short items

    int blocks(int n) const { return (n + tb - 1) / tb; }
    int chunks(int n) const
    {
        const double share = total > 0 ? (double)n * n / total : 1.0;
        const double want = std::ceil(share * (double)(small ? resident : 3 * resident) / blocks(n));
        const int most = std::min(64, small ? n / kMinChunk : n / (8 * kTile));
        return (int)std::max(1.0, std::min(want, (double)most));
    }
    int length(int n) const
    {
        const int nch = chunks(n), len = (n + nch - 1) / nch;
        return small ? len : (len + kTile - 1) / kTile * kTile;
    }
};

// Build the (target block, source chunk) queue of one pass.  Items of big problems come first
// so the persistent grid ends with the small ones.
cudaError_t plan_pass(Ctx &c, Ctx::Plan &pl, int tpt, int occupancy)
{
    const int tb = kThreads * tpt;
    std::vector<WorkItem> items;
    // neighbour spans per target block: min/max edge index sharing a vertex with the block
    std::vector<int> vmin(c.nV, INT32_MAX), vmax(c.nV, -1);
    for (int I = 0; I < c.nE; ++I)
        for (int s = 0; s < 2; ++s) {
            int v = c.h_edges[2 * I + s];
            vmin[v] = std::min(vmin[v], I);
            vmax[v] = std::max(vmax[v], I);
        }
    // total work estimate to size chunks
    double total = 0.0;
    for (int q = 0; q < c.nProb; ++q) {
        double n = c.h_prob_e[q + 1] - c.h_prob_e[q];
        total += n * n;
    }
    Chunking ck{tb, (long long)c.sm_count * std::max(1, occupancy), total};
    long long whole = 0;
    for (int q = 0; q < c.nProb; ++q) {
        const int n = c.h_prob_e[q + 1] - c.h_prob_e[q];
        if (n > 0) whole += (long long)ck.blocks(n) * ck.chunks(n);
    }
    ck.small = whole < ck.resident;
    int max_slots = 1;
    std::vector<int> eslots(c.nE, 1);
    struct Tmp {
        WorkItem w;
        double cost;
    };
    std::vector<Tmp> tmp;
    for (int q = 0; q < c.nProb; ++q) {
        int e0 = c.h_prob_e[q], e1 = c.h_prob_e[q + 1], n = e1 - e0;
        if (n <= 0) continue;
        const int nblk = ck.blocks(n), clen = ck.length(n), nch = (n + clen - 1) / clen;
        max_slots = std::max(max_slots, nch);
        for (int b = 0; b < nblk; ++b) {
            int t0 = e0 + b * tb, nt = std::min(tb, e1 - t0);
            int lo = INT32_MAX, hi = -1;
            for (int I = t0; I < t0 + nt; ++I)
                for (int s = 0; s < 2; ++s) {
                    int v = c.h_edges[2 * I + s];
                    lo = std::min(lo, vmin[v]);
                    hi = std::max(hi, vmax[v]);
                }
            for (int k = 0; k < nch; ++k) {
                int s0 = e0 + k * clen, s1 = std::min(e1, s0 + clen);
                WorkItem w{t0, nt, s0, s1, k, lo, hi, q};
                tmp.push_back({w, (double)nt * (s1 - s0)});
            }
        }
        for (int I = e0; I < e1; ++I) eslots[I] = nch;
    }
    std::stable_sort(tmp.begin(), tmp.end(), [](const Tmp &a, const Tmp &b) { return a.cost > b.cost; });
    for (auto &t : tmp) items.push_back(t.w);
    pl.n_items = (int)items.size();
    pl.max_slots = max_slots;
    pl.tpt = tpt;
    pl.grid = std::max(1, std::min(pl.n_items, c.sm_count * std::max(1, occupancy)));
    return plan_upload(pl, items, eslots);
}

constexpr int kTptEnergy = 4, kTptDiff = 2, kTptApply = 2;

// Targets per thread: one on short graphs (see small_graph), the default of the op class otherwise, and for
// the mixed-precision passes with the specialised powers ((alpha, beta) = (2, 4.5)) the value the autotuner
// chose; only those are instantiated for every candidate.
static int op_class(int op) { return op == OP_ENERGY ? 0 : (op == OP_DIFF ? 1 : 2); }

int tpt_default(const Ctx &c, int cls)
{
    if (c.prm.precision == TP_FP64) return 1;
    return cls == 0 ? kTptEnergy : (cls == 1 ? kTptDiff : kTptApply);
}

static bool tunable(const Ctx &c) { return c.prm.precision == TP_MIXED && c.kp.fast; }

int tpt_candidates(const Ctx &c, int cls, int *out)
{
    if (!tunable(c)) {
        out[0] = tpt_default(c, cls);
        return 1;
    }
    if (cls == 1) {
        out[0] = 1;
        out[1] = 2;
        return 2;
    }
    out[0] = 1;
    out[1] = 2;
    out[2] = 4;
    return 3;
}

// Too few edges to give every SM two items of tpt targets per thread and eight source tiles: one target
// per thread then doubles or quadruples the items (256 edges: energy with four targets 16 items, with one 64).
static long long long_items(long long n, int tpt)
{
    return ((n + kThreads * tpt - 1) / (kThreads * tpt)) * std::max(1LL, n / (8 * kTile));
}
static bool small_graph(const Ctx &c, int tpt)
{
    long long items = 0;
    for (int q = 0; q < c.nProb; ++q) items += long_items(c.h_prob_e[q + 1] - c.h_prob_e[q], tpt);
    return items < 2LL * c.sm_count;
}

static int tpt_for(const Ctx &c, int cls)
{
    if (tunable(c) && c.tpt[cls]) return c.tpt[cls];
    const int t = tpt_default(c, cls);
    return small_graph(c, t) ? 1 : t;
}

// f(kernel) of one pass at tpt targets per thread (the values instantiated for it; the op's default otherwise)
template <int PREC, int OP, bool FAST, class F>
static void with_pair_kernel(int tpt, F f)
{
    constexpr int D = PREC == P64 ? 1 : (OP == OP_ENERGY ? kTptEnergy : (OP == OP_DIFF ? kTptDiff : kTptApply));
    if constexpr (D != 1)
        if (tpt == 1) return f(k_pairs<PREC, OP, 1, FAST>);
    if constexpr (PREC == PMIX && FAST && D == 4)
        if (tpt == 2) return f(k_pairs<PREC, OP, 2, FAST>);
    if constexpr (PREC == PMIX && FAST && D == 2 && OP != OP_DIFF)
        if (tpt == 4) return f(k_pairs<PREC, OP, 4, FAST>);
    f(k_pairs<PREC, OP, D, FAST>);
}

template <int OP, class F>
static void with_pair_kernel(const Ctx &c, int tpt, F f)
{
    const bool fast = c.kp.fast != 0;
    if (c.prm.precision == TP_FP64)
        fast ? with_pair_kernel<P64, OP, true>(tpt, f) : with_pair_kernel<P64, OP, false>(tpt, f);
    else if (c.prm.precision == TP_MIXED)
        fast ? with_pair_kernel<PMIX, OP, true>(tpt, f) : with_pair_kernel<PMIX, OP, false>(tpt, f);
    else
        fast ? with_pair_kernel<P32, OP, true>(tpt, f) : with_pair_kernel<P32, OP, false>(tpt, f);
}

// ---------------------------------------------------------------------------------- profiling

constexpr int kProfSlots = 1024;

int prof_begin(Ctx &c, int op, cudaStream_t s)
{
    if (c.capturing) {  // inside a captured CG block: external event nodes on events the graph owns
        CgGraph &g = *c.capturing;
        const int k = (int)g.prof_op.size();
        if (2 * k + 1 >= (int)g.ev.size()) return -1;  // events are created before the capture
        g.prof_op.push_back(op);
        cudaEventRecordWithFlags(g.ev[2 * k], s, cudaEventRecordExternal);
        return -2 - k;
    }
    if (c.prof_pool.empty()) {
        c.prof_pool.resize(2 * kProfSlots);
        for (auto &e : c.prof_pool) cudaEventCreate(&e);
    }
    if ((int)c.prof_pending.size() == kProfSlots) prof_harvest(c);
    int slot = (int)c.prof_pending.size();
    c.prof_pending.push_back({op, slot});
    cudaEventRecord(c.prof_pool[2 * slot], s);
    return slot;
}

void prof_end(Ctx &c, int slot, cudaStream_t s)
{
    if (slot <= -2) {
        cudaEventRecordWithFlags(c.capturing->ev[2 * (-2 - slot) + 1], s, cudaEventRecordExternal);
        return;
    }
    cudaEventRecord(c.prof_pool[2 * slot + 1], s);
}

void prof_harvest(Ctx &c)
{
    for (auto &pe : c.prof_pending) {
        cudaEventSynchronize(c.prof_pool[2 * pe.second + 1]);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, c.prof_pool[2 * pe.second], c.prof_pool[2 * pe.second + 1]);
        c.prof_ms[pe.first] += ms;
        c.prof_n[pe.first] += 1;
    }
    c.prof_pending.clear();
}

static int occupancy_cls(const Ctx &c, int cls, int tpt)
{
    int occ = 0;
    auto ask = [&](auto kern) { cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kThreads, 0); };
    if (cls == 0)
        with_pair_kernel<OP_ENERGY>(c, tpt, ask);
    else if (cls == 1)
        with_pair_kernel<OP_DIFF>(c, tpt, ask);
    else
        with_pair_kernel<OP_APPLY>(c, tpt, ask);
    return occ;
}

static Ctx::Plan &plan_of(Ctx &c, int cls) { return cls == 0 ? c.plan_energy : (cls == 1 ? c.plan_diff : c.plan_apply); }

cudaError_t make_plans(Ctx &c)
{
    // Every slot of an op class shares one layout, so all passes of an op class use the same
    // targets-per-thread (the plan records it and the launch follows the plan).
    for (int cls = 0; cls < 3; ++cls) {
        const int t = tpt_for(c, cls);
        TPE_CHECK(plan_pass(c, plan_of(c, cls), t, occupancy_cls(c, cls, t)));
    }
    return cudaSuccess;
}

cudaError_t replan(Ctx &c, int cls)
{
    graphs_reset(c);
    Ctx::Plan pl;
    const int t = tpt_for(c, cls);
    TPE_CHECK(plan_pass(c, pl, t, occupancy_cls(c, cls, t)));  // the old plan stays on failure
    plan_free(plan_of(c, cls));
    plan_of(c, cls) = pl;
    const int ms = std::max(std::max(c.plan_energy.max_slots, c.plan_diff.max_slots), c.plan_apply.max_slots);
    TPE_CHECK(part_reserve(c, (size_t)ms * std::max(1, c.nE) * 6));
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------- no-allocation energy

// Items of one problem spanning all edges (target blocks x source chunks); every tile checks
// disjointness (the neighbour span is the whole range) because no incidence lists are built.
__global__ void k_static_items(int nE, int tb, int clen, int nch, WorkItem *items, int *eslots, int *off)
{
    int it = blockIdx.x * blockDim.x + threadIdx.x;
    int nblk = (nE + tb - 1) / tb;
    if (it < nblk * nch) {
        int b = it / nch, k = it % nch;
        int t0 = b * tb, s0 = k * clen;
        items[it] = WorkItem{t0, min(tb, nE - t0), s0, min(nE, s0 + clen), k, 0, nE - 1, 0};
    }
    if (it < nE) eslots[it] = nch;
    if (it == 0) {
        off[0] = 0;
        off[1] = nE;
    }
}

__global__ void k_static_stats(int nV, int nE, const double *__restrict__ g, const double *__restrict__ ell,
                               double *__restrict__ out)
{
    __shared__ double sh[7][256];
    double b[7] = {1e300, 1e300, 1e300, -1e300, -1e300, -1e300, 0.0};
    for (int i = threadIdx.x; i < nV; i += blockDim.x)
        for (int k = 0; k < 3; ++k) {
            b[k] = fmin(b[k], g[3 * i + k]);
            b[3 + k] = fmax(b[3 + k], g[3 * i + k]);
        }
    for (int I = threadIdx.x; I < nE; I += blockDim.x) b[6] += ell[I];
    for (int k = 0; k < 7; ++k) sh[k][threadIdx.x] = b[k];
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w)
            for (int k = 0; k < 7; ++k)
                sh[k][threadIdx.x] = k < 3 ? fmin(sh[k][threadIdx.x], sh[k][threadIdx.x + w])
                                           : (k < 6 ? fmax(sh[k][threadIdx.x], sh[k][threadIdx.x + w])
                                                    : sh[k][threadIdx.x] + sh[k][threadIdx.x + w]);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int k = 0; k < 3; ++k) s += (sh[3 + k][0] - sh[k][0]) * (sh[3 + k][0] - sh[k][0]);
        out[0] = sh[6][0] / (nE > 0 ? nE : 1);  // mean edge length
        out[1] = sqrt(s);                       // bounding-box diagonal
    }
}

cudaError_t static_energy_launch(const double *gamma, const int *edges, int nV, int nE, double alpha, double beta,
                                 double near_cutoff, RecF *recF, RecLo *recLo, double *ell, double *T, double *x,
                                 WorkItem *items, int *eslots, double *part, double *rows, int *counter, int *err,
                                 double *scal, int *off, int max_items, long long max_part, double *E, cudaStream_t s,
                                 int *status)
{
    *status = 0;
    if (nE == 0) return cudaMemsetAsync(E, 0, sizeof(double), s);
    TPE_CHECK(cudaMemsetAsync(err, 0, sizeof(int), s));
    k_records<<<(nE + kRecThreads - 1) / kRecThreads, kRecThreads, 0, s>>>(nE, gamma, edges, recF, recLo, nullptr, ell, T, x, err, nullptr);
    k_static_stats<<<1, 256, 0, s>>>(nV, nE, gamma, ell, scal);
    TPE_CHECK(cudaGetLastError());
    // the cutoffs are kernel arguments: read the two statistics and the error word (synchronises)
    double st[2] = {0.0, 0.0};
    int e = 0;
    TPE_CHECK(cudaMemcpyAsync(st, scal, sizeof(st), cudaMemcpyDeviceToHost, s));
    TPE_CHECK(cudaMemcpyAsync(&e, err, sizeof(int), cudaMemcpyDeviceToHost, s));
    TPE_CHECK(cudaStreamSynchronize(s));
    if (e) {
        *status = e;
        return cudaSuccess;
    }
    KernelParams kp{};
    kp.alpha = alpha;
    kp.beta = beta;
    kp.p = 2.0 * ((beta - 1.0) / alpha - 1.0) + 1.0;
    kp.fast = (alpha == 2.0 && beta == 4.5) ? 1 : 0;
    double rn = near_cutoff * st[0];
    kp.near2 = rn * rn;
    kp.near2f = (float)(rn * rn);
    kp.near2f_diff = (float)(16.0 * rn * rn);
    kp.mid2f = 3.0e38f;  // double-float positions in every tile (the context's default)
    // the blocking of a context's gather pass over the same graph, so that the sums are the same to the bit wherever the
    // scratch holds as many slots
    int dev = 0, sms = 0, occ = 0;
    TPE_CHECK(cudaGetDevice(&dev));
    TPE_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int tpt = long_items(nE, kTptEnergy) < 2LL * sms ? 1 : kTptEnergy;
    auto with_kernel = [&](auto f) {
        if (kp.fast)
            with_pair_kernel<PMIX, OP_ENERGY, true>(tpt, f);
        else
            with_pair_kernel<PMIX, OP_ENERGY, false>(tpt, f);
    };
    with_kernel([&](auto kern) { cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kThreads, 0); });
    Chunking ck{kThreads * tpt, (long long)sms * std::max(1, occ), (double)nE * nE};
    ck.small = (long long)ck.blocks(nE) * ck.chunks(nE) < ck.resident;
    int clen = ck.length(nE), nch = (nE + clen - 1) / clen;
    if ((long long)nch * nE > max_part) {  // longer chunks, as many as the scratch holds partial sums for
        clen = (nE + (int)(max_part / nE) - 1) / (int)(max_part / nE);
        clen = (clen + kTile - 1) / kTile * kTile;
        nch = (nE + clen - 1) / clen;
    }
    const int nit = ck.blocks(nE) * nch;
    if (nit > max_items) return cudaErrorInvalidValue;
    k_static_items<<<(std::max(nit, nE) + 255) / 256, 256, 0, s>>>(nE, ck.tb, clen, nch, items, eslots, off);
    TPE_CHECK(cudaMemsetAsync(counter, 0, sizeof(int), s));
    PairArgs pa;
    pa.items = items;
    pa.n_items = nit;
    pa.counter = counter;
    pa.recF = recF;
    pa.recLo = recLo;
    pa.recD = nullptr;
    pa.urecF = nullptr;
    pa.urecD = nullptr;
    pa.na = NearArgs{gamma, edges, ell, T, nullptr};
    pa.part = part;
    pa.nE = nE;
    pa.kp = kp;
    pa.skip = nullptr;
    const int grid = std::max(1, std::min(nit, sms * std::max(1, occ)));
    with_kernel([&](auto kern) { kern<<<grid, kThreads, 0, s>>>(pa); });
    k_energy_rows<<<(nE + 31) / 32, 256, 0, s>>>(nE, eslots, part, ell, rows);
    k_segment_sum<<<1, kSegThreads, 0, s>>>(off, rows, E);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------- launchers

cudaError_t build_records(Ctx &c, const double *gamma, int which, cudaStream_t s)
{
    int nb = (c.nE + kRecThreads - 1) / kRecThreads;
    const bool p64 = c.prm.precision == TP_FP64;
    RecF *rf = p64 ? nullptr : (which ? c.d_recF2 : c.d_recF);
    // the low parts serve the mixed pair passes and, in FP32 contexts too, the double-float apply
    RecLo *rl = p64 ? nullptr : (which ? c.d_recLo2 : c.d_recLo);
    RecD *rd = p64 ? (which ? c.d_recD2 : c.d_recD) : nullptr;
    if (c.nE == 0) return cudaSuccess;
    k_records<<<nb, kRecThreads, 0, s>>>(c.nE, gamma, c.d_edges, rf, rl, rd, c.d_ellw[which], c.d_Tw[which], c.d_xw[which], c.d_err,
                                 p64 ? nullptr : c.d_ell_lo[which]);
    c.launches++;
    return cudaGetLastError();
}

cudaError_t build_urecs(Ctx &c, const double *u, int which, cudaStream_t s)
{
    if (c.nE == 0) return cudaSuccess;
    int nb = (c.nE + kRecThreads - 1) / kRecThreads;
    const bool p64 = c.prm.precision == TP_FP64;
    k_urecs<<<nb, kRecThreads, 0, s>>>(c.nE, u, c.d_edges, c.d_ellw[which], p64 ? nullptr : c.d_urecF, p64 ? c.d_urecD : nullptr);
    c.launches++;
    return cudaGetLastError();
}

cudaError_t segment_sum(Ctx &c, const double *rows, double *E, cudaStream_t s)
{
    k_segment_sum<<<c.nProb, kSegThreads, 0, s>>>(c.d_prob_e, rows, E);
    c.launches++;
    return cudaGetLastError();
}

cudaError_t build_urecs_into(Ctx &c, const double *u, int which, URecF *uf, URecD *ud, cudaStream_t s)
{
    if (c.nE == 0) return cudaSuccess;
    k_urecs<<<(c.nE + kRecThreads - 1) / kRecThreads, kRecThreads, 0, s>>>(c.nE, u, c.d_edges, c.d_ellw[which], uf, ud);
    c.launches++;
    return cudaGetLastError();
}

template <int OP>
static cudaError_t run_pairs(Ctx &c, int which, const double *gamma, const double *u, cudaStream_t s)
{
    Ctx::Plan &pl = (OP == OP_ENERGY) ? c.plan_energy : (OP == OP_DIFF ? c.plan_diff : c.plan_apply);
    if (pl.n_items == 0) return cudaSuccess;
    TPE_CHECK(part_reserve(c, (size_t)pl.max_slots * c.nE * 6));
    if (!tunable(c) && pl.tpt != 1 && pl.tpt != tpt_default(c, op_class(OP))) return cudaErrorInvalidValue;  // no such kernel
    constexpr int ctr = OP;
    PairArgs pa;
    pa.items = pl.d_items;
    pa.n_items = pl.n_items;
    pa.counter = c.d_counter + ctr;
    pa.recF = which ? c.d_recF2 : c.d_recF;
    pa.recLo = which ? c.d_recLo2 : c.d_recLo;
    pa.recD = which ? c.d_recD2 : c.d_recD;
    pa.urecF = c.d_urecF;
    pa.urecD = c.d_urecD;
    pa.na = NearArgs{gamma, c.d_edges, c.d_ellw[which], c.d_Tw[which], u};
    pa.part = c.d_part;
    pa.nE = c.nE;
    pa.kp = c.kp;
    pa.skip = (OP == OP_APPLY) ? c.d_skip : nullptr;
    // profiling: applies that skip converged problems are recorded apart (op 4), so op 2 always
    // times full passes of pairs_per_pass pairs
    const int slot = c.profile ? prof_begin(c, (OP == OP_APPLY && c.d_skip) ? 4 : OP, s) : -1;
    with_pair_kernel<OP>(c, pl.tpt, [&](auto kern) { kern<<<pl.grid, kThreads, 0, s>>>(pa); });  // the plan's targets per thread
    if (slot >= 0 || slot <= -2) prof_end(c, slot, s);
    c.launches++;
    return cudaGetLastError();
}

cudaError_t pair_energy(Ctx &c, const double *gamma, int which, double *rows_out, double *E_out, cudaStream_t s)
{
    double *rows = rows_out ? rows_out : c.d_rows;
    if (c.energy_sym > 0) {
        TPE_CHECK(sym_energy_pass(c, which, rows, s));
    } else {
        TPE_CHECK(run_pairs<OP_ENERGY>(c, which, gamma, nullptr, s));
        if (c.nE > 0) {
            k_energy_rows<<<(c.nE + 31) / 32, 256, 0, s>>>(c.nE, c.plan_energy.d_eslots, c.d_part, c.d_ellw[which], rows);
            c.launches++;
        }
    }
    if (E_out) TPE_CHECK(segment_sum(c, rows, E_out, s));
    return cudaGetLastError();
}

cudaError_t pair_diff(Ctx &c, const double *gamma, int which, double *dE, cudaStream_t s)
{
    if (c.diff_sym > 0) {
        TPE_CHECK(sym_diff_pass(c, which, s));
        return vertices_from_edges<OP_DIFF>(c, c.d_esum, dE, s);
    }
    TPE_CHECK(run_pairs<OP_DIFF>(c, which, gamma, nullptr, s));
    return gather_slots<OP_DIFF>(c, c.plan_diff, dE, s);
}

cudaError_t pair_apply(Ctx &c, const double *gamma_geom, int which, const double *u, double *Au, cudaStream_t s)
{
    TPE_CHECK(build_urecs(c, u, which, s));
    if (c.apply_sym > 0) {
        TPE_CHECK(sym_apply_pass(c, which, s));
        return vertices_from_edges<OP_APPLY>(c, c.d_esum, Au, s);
    }
    TPE_CHECK(run_pairs<OP_APPLY>(c, which, gamma_geom, u, s));
    return gather_slots<OP_APPLY>(c, c.plan_apply, Au, s);
}

cudaError_t pair_diag(Ctx &c, const double *gamma_geom, int which, double *diag, cudaStream_t s)
{
    TPE_CHECK(run_pairs<OP_DIAG>(c, which, gamma_geom, nullptr, s));
    return gather_slots<OP_DIAG>(c, c.plan_apply, diag, s);
}

}  // namespace tpe
