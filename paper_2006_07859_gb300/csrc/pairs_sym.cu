// Symmetric pair passes: every unordered pair of disjoint edges {I, J} evaluated once, both rows fed.
//
//   apply: the Gram weights are symmetric (w_IJ = w_JI, and the low-order weight enters as w0_IJ + w0_JI,
//     Secs. 5.2.2-5.2.3), so one evaluation yields what row I receives from J and what row J receives from I:
//       row I: h += l_J sw ((du_I - du_J) + (|T_I - T_J|^2 / 2) du_J),   l += l_J sw0 (ub_I - ub_J)
//       row J: h += l_I sw ((du_J - du_I) + (|T_I - T_J|^2 / 2) du_I),   l += l_I sw0 (ub_J - ub_I)
//     with sw = sum_ab |d_ab|^-p and sw0 = sum_ab (|T_I x d_ab|^2 + |T_J x d_ab|^2) |d_ab|^-(4+p);
//   energy: row I receives l_J sum_ab |T_I x d_ab|^2 |d_ab|^-4.5, row J l_I sum_ab |T_J x d_ab|^2 |d_ab|^-4.5;
//   differential: row I accumulates (scaled by l_J) S = sum (f_I + f_J), G_a += v_ab, GT += -a_I (T_I . d_ab)
//     d_ab with v_ab = d(f_I + f_J)/dd at d_ab = g_ia - g_jb; row J sees d' = -d and accumulates (scaled by
//     l_I) the same S, H_b -= v_ab (its endpoint b) and HT += -a_J (T_J . d_ab) d_ab.
//
// What bounds the passes and the layout that follows from it.  A pair of the apply costs about 195
// operations of the FP32 pipe and 8 MUFU; as scalar instructions these, the shared-memory accesses and the
// denormal fix-ups of rsqrtf filled ~299 issue slots of a sub-partition per 32 pairs.  Every thread
// therefore owns TWO target edges and evaluates both pairs with one source in packed f32x2 instructions
// (pair_lanes.cuh), half the issue slots for the same FP32 work, and one load of a source serves two pairs.
// (One target a thread would load 7 LDS.128 a pair, 112 of the ~200 cycles the shared-memory port has
// for it; four targets do not fit in registers.)
//
// Blocks.  A problem's edges are cut into super-blocks of 256 target rows (128 threads x 2 adjacent rows) and
// tiles of 128 source rows.  A work item is one super-block X against half a tile to four tiles beyond it,
// or against itself.  Lane l of a warp takes source (step + 2 l) mod P at step `step`: the 32 lanes touch 32
// distinct sources and add what those receive into the warp's own Kahan-compensated shared-memory
// accumulators (no atomics), and along a curve all lanes are equally far from their sources, so near pairs
// (evaluated in double-float) come in the same steps.  Inside its own super-block a warp takes its own 64
// rows and whole 64-row sections of the others, every pair once (a plain gather there would add 12% of
// the pairs at 4,096 edges).
//
// Partial sums are (sum, low part) float pairs, one slot per writer: a row of super-block X gets slot B from
// every super-block B < X (as a source), slots X to X + 2 from its own super-block (source side, and target
// side of its two tiles) and one slot from every item it is a target of; k_sym_sum adds a row's slots in index order in
// double-float arithmetic, so the passes are deterministic, and no FP64 instruction (2 per clock and SM) is
// left in the pair kernels.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "df.cuh"
#include "pair_device.cuh"

namespace tpe {

#define TPE_CHECK(x)                      \
    do {                                  \
        cudaError_t e_ = (x);             \
        if (e_ != cudaSuccess) return e_; \
    } while (0)

constexpr int kSymWarps = kThreads / 32;
constexpr int kSuper = 2 * kThreads;  // target rows of an item
constexpr int kSection = 64;          // rows of one warp
constexpr int kQueue = 128;           // near pairs a warp holds back: a batch of 64 and one step's worth
constexpr int kSymMaxTiles = 4;       // source tiles of an item: a Kahan sum spans at most 512 sources

struct SymArgs {
    const WorkItem *items;  // slot: (super-block << 16) | target slot; nb_lo: bit t = tile t needs the disjointness test
    int n_items;
    int *counter;
    const RecF *recF;
    const RecLo *recLo;
    const URecF *urecF;
    const float *ell_lo;  // PDF
    float2 *part;  // [slot][nE][W]
    int nE;
    float near2f, mid2f;
    int sum_exp;  // OP_DIFF: the sums are kept at 2^sum_exp of their value
    float sum_scale;
    const int *skip;
};

template <int OP>
__host__ __device__ constexpr int sym_width()
{
    return OP == OP_ENERGY ? 1 : (OP == OP_DIFF ? 10 : (OP == OP_APPLY2 ? 12 : 6));
}
// vector fields of the pass
template <int OP>
__host__ __device__ constexpr int sym_fields()
{
    return OP == OP_APPLY ? 1 : (OP == OP_APPLY2 ? 2 : 0);
}

// Source tile (struct of arrays, 16-byte elements) and the warps' source accumulators.
template <int PREC, int OP>
struct SymSmem {
    static constexpr bool MIX = PREC != P32;
    static constexpr int F = sym_fields<OP>() ? sym_fields<OP>() : 1, U = sym_fields<OP>() ? kTile : 1;
    float4 t0[kTile], t1[kTile], t2[kTile];  // (q1, l), (e, T.x), (T.y, T.z, q1.x lo, q1.y lo)
    float4 t3[MIX ? kTile : 1];              // (q1.z lo, T lo)
    float4 t4[PREC == PDF ? kTile : 1];      // (e lo, l lo)
    float4 u0[F][U], u1[F][U], u2[F][MIX ? U : 1];  // u records
    int2 id[kTile];
    float2 sac[kSymWarps][sym_width<OP>()][kTile];  // (sum, Kahan compensation)
    // differential: the warps' queues of near pairs (row << 8 | slot) and the target sums of those pairs
    float2 tac[OP == OP_DIFF ? kSymWarps : 1][OP == OP_DIFF ? 10 : 1][OP == OP_DIFF ? kSection : 1];
    unsigned short queue[OP == OP_DIFF ? kSymWarps : 1][OP == OP_DIFF ? kQueue : 1];
    float box[kSymWarps][6];
    int item;
};

struct SymSrc {
    float q[3], m[3], e[3], T[3], Tm[3], ell;  // PDF: em the low part of e
    float em[3], ell_lo;
    int j1, j2;
};

template <int PREC, int OP, bool CHECK>
__device__ __forceinline__ void sym_load(SymSrc &s, const SymSmem<PREC, OP> &tl, int j)
{
    const float4 a = tl.t0[j], b = tl.t1[j], c = tl.t2[j];
    s.q[0] = a.x, s.q[1] = a.y, s.q[2] = a.z, s.ell = a.w;
    s.e[0] = b.x, s.e[1] = b.y, s.e[2] = b.z, s.T[0] = b.w;
    s.T[1] = c.x, s.T[2] = c.y;
    if constexpr (PREC == PDF) {
        const float4 d = tl.t4[j];
        s.em[0] = d.x, s.em[1] = d.y, s.em[2] = d.z, s.ell_lo = d.w;
    }
    if constexpr (PREC != P32) {
        const float4 d = tl.t3[j];
        s.m[0] = c.z, s.m[1] = c.w, s.m[2] = d.x;
        s.Tm[0] = d.y, s.Tm[1] = d.z, s.Tm[2] = d.w;
    } else {
        s.m[0] = s.m[1] = s.m[2] = s.Tm[0] = s.Tm[1] = s.Tm[2] = 0.f;
    }
    if constexpr (CHECK) {
        const int2 v = tl.id[j];
        s.j1 = v.x, s.j2 = v.y;
    }
}

using L2 = float2;

// Two target rows of a thread (rows of invalid lanes repeat the last one with length 0, so that they feed
// nothing into the sources, at a place where no power overflows: 0 x inf would reach the sources as NaN).
struct SymTgt {
    LV<L2> p, pl, e, T, Tl;  // PDF: el the low part of e
    LV<L2> el;
    L2 ell, ell_lo;
    int i1[2], i2[2], row[2];
};

// u data of the two rows (apply)
struct SymTgtU {
    LV<L2> dh, uh, dl, ul;
};

// ---------------------------------------------------------------------------------- per-pair bodies

template <int PREC, int OP>
struct SymAcc;
template <int PREC>
struct SymAcc<PREC, OP_ENERGY> {
    L2 s[1], c[1];
};
template <int PREC>
struct SymAcc<PREC, OP_DIFF> {
    L2 s[10], c[10];
};
template <int PREC>
struct SymAcc<PREC, OP_APPLY> {
    L2 s[6], c[6];
};
template <int PREC>
struct SymAcc<PREC, OP_APPLY2> {
    L2 s[12], c[12];
};

// source accumulator += wx vx + wy vy, both compensated
__device__ __forceinline__ void src_add(float2 &ac, L2 w, L2 v)
{
    l_kahan_fma(ac.x, ac.y, w.x, v.x);
    l_kahan_fma(ac.x, ac.y, w.y, v.y);
}

__device__ __forceinline__ void src_add_pos(float2 &ac, L2 w, L2 v)
{
    l_kahan_fma_pos(ac.x, ac.y, w.x, v.x);
    l_kahan_fma_pos(ac.x, ac.y, w.y, v.y);
}

template <int PREC, bool CHECK, int MODE>
__device__ __forceinline__ void sym_pair(const SymTgt &t, const SymTgtU *, const SymSmem<PREC, OP_ENERGY> &, const SymSrc &s,
                                         int, int Jg, bool k0, bool k1, SymAcc<PREC, OP_ENERGY> &a, float2 *sac,
                                         const SymArgs &pa, bool &, bool &)
{
    LV<L2> d[4];
    l_chords<(MODE >= 1 && PREC == PMIX)>(t.p, t.pl, t.e, l_bc3<L2>(s.q[0], s.q[1], s.q[2]),
                                          l_bc3<L2>(s.m[0], s.m[1], s.m[2]), l_bc3<L2>(s.e[0], s.e[1], s.e[2]), d);
    const LV<L2> TJ = l_bc3<L2>(s.T[0], s.T[1], s.T[2]);
    L2 cI[2] = {l_perp2(d[0], t.T), l_perp2(d[1], t.T)};
    L2 cJ[2] = {l_perp2(d[0], TJ), l_perp2(d[2], TJ)};
    L2 r[4], d11;
#pragma unroll
    for (int ab = 0; ab < 4; ++ab) {
        const L2 d2 = l_dot(d[ab], d[ab]);
        if (ab == 0) d11 = d2;
        L2 r2;
        r[ab] = l_pow45(d2, r2);
    }
    if constexpr (MODE == 2) {
        const bool n0 = k0 && d11.x < pa.near2f, n1 = k1 && d11.y < pa.near2f;
        if (n0 || n1) {
            L2 c[4];
            near_energy<L2, true>(pa.recF, pa.recLo, t.row[0], t.row[1], Jg, c);
            cI[0] = make_float2(n0 ? c[0].x : cI[0].x, n1 ? c[0].y : cI[0].y);
            cI[1] = make_float2(n0 ? c[1].x : cI[1].x, n1 ? c[1].y : cI[1].y);
            cJ[0] = make_float2(n0 ? c[2].x : cJ[0].x, n1 ? c[2].y : cJ[0].y);
            cJ[1] = make_float2(n0 ? c[3].x : cJ[1].x, n1 ? c[3].y : cJ[1].y);
        }
    }
    L2 fI = l_energy_sum(cI[0], cI[1], r[0], r[1], r[2], r[3]);
    if constexpr (CHECK) fI = l_keep(k0, k1, fI);
    l_kahan_fma_pos(a.s[0], a.c[0], l_bc<L2>(s.ell), fI);
    L2 fJ = l_energy_sum(cJ[0], cJ[1], r[0], r[2], r[1], r[3]);
    if constexpr (CHECK) fJ = l_keep(k0, k1, fJ);
    float2 ac = *sac;
    src_add_pos(ac, t.ell, fJ);
    *sac = ac;
}

// F = |d|^-2.5 and G = |d|^-6.5 in double-float from |d|^2: r0 = rsqrt(d2.hi) after a Newton step, its residual rho =
// 1 - d2 r0^2 formed through fma, |d|^-1 = r0 (1 + eps) with eps = rho / 2 + 3 rho^2 / 8, and sqrt(r0) = q0 +
// (r0 - q0^2) / (2 q0).  The step makes eps, and with it the low parts whose products l_dfmul drops, four times smaller.
__device__ __forceinline__ void sym_df_powers(dfl<L2> d2, dfl<L2> &F, dfl<L2> &G)
{
    L2 r0 = l_rsqrt(d2.hi);
    r0 = l_fma(r0, l_mul(l_bc<L2>(0.5f), l_fma(l_neg(l_mul(d2.hi, r0)), r0, l_bc<L2>(1.f))), r0);
    const L2 a = l_mul(r0, r0), b = l_fma(r0, r0, l_neg(a));
    L2 rho = l_fma(l_neg(d2.hi), a, l_bc<L2>(1.f));
    rho = l_fma(l_neg(d2.hi), b, rho);
    rho = l_fma(l_neg(d2.lo), a, rho);
    const L2 eps = l_mul(rho, l_fma(l_bc<L2>(0.375f), rho, l_bc<L2>(0.5f)));
    const L2 iq = l_mul(l_bc<L2>(0.5f), l_rsqrt(r0));
    L2 q0 = l_mul(r0, l_add(iq, iq));
    q0 = l_fma(l_fma(l_neg(q0), q0, r0), iq, q0);  // to half an ulp: dq leaves out (r0 - q0^2)^2 / (8 q0^3)
    const L2 dq = l_mul(l_fma(l_neg(q0), q0, r0), iq);
    const dfl<L2> R = {a, b};
    F = l_dfscale(l_dfmul(R, dfl<L2>{q0, dq}), l_mul(eps, l_fma(l_bc<L2>(1.875f), eps, l_bc<L2>(2.5f))));
    const dfl<L2> R2 = l_dfscale(R, l_mul(eps, l_add(l_bc<L2>(2.f), eps)));  // |d|^-2
    G = l_dfmul(F, l_dfsqr(R2));
}

// a - b with both parts' differences exact: rounding al - bl leaves 2^-49 |a|, which for neighbouring edges (|a - b|
// ~ 1e-3 |a|) is a thousand times the rounding of everything else (5.6e-13 against 1.5e-13 in A u at 500 edges).
template <class L>
__device__ __forceinline__ dfl<L> l_dfdiff(L ah, L al, L bh, L bl)
{
    const dfl<L> s = l_two_sum(ah, l_neg(bh)), t = l_two_sum(al, l_neg(bl));
    const dfl<L> r = l_dfnorm(dfl<L>{s.hi, l_add(s.lo, t.hi)});
    return l_dfnorm(dfl<L>{r.hi, l_add(r.lo, t.lo)});
}

// A compensated sum acc - c with c at most half an ulp of acc.  Left to itself c takes up the rounding of every
// addition and the low part of every term, and rounds at its own size each time.
template <class L>
__device__ __forceinline__ void l_kahan_norm(L &acc, L &c)
{
    const dfl<L> s = l_dfnorm(dfl<L>{acc, l_neg(c)});
    acc = s.hi;
    c = l_neg(s.lo);
}

// source sum += both lanes' double-float terms
__device__ __forceinline__ void src_add_df(float2 &ac, dfl<L2> v)
{
    l_kahan_df(ac.x, ac.y, v.hi.x, v.lo.x);
    l_kahan_df(ac.x, ac.y, v.hi.y, v.lo.y);
    l_kahan_norm(ac.x, ac.y);
}

// The accurate apply: every quantity of the pair a double-float, about 1,100 operations against the mixed
// apply's 195; FP32 operand reads bound it (8 x 4,096 edges 2.81 ms; one target per thread in scalar double-float
// arithmetic took 4.75).  Its error against 64 bits stays that of fully renormalised arithmetic (9.6e-15 on trefoils of
// 150 edges, 2.7e-14 of 500, 9.0e-13 on knots of 4,096, random u) as long as the differences are exact, d2 and t are
// renormalised before they are used, and the sums at least every eight terms (1.7e-14 at 150 edges without).
// Sums are (sum, minus low part) like the compensated ones.
template <bool CHECK>
__device__ __forceinline__ void sym_pair_df(const SymTgt &t, const SymTgtU &tu, const SymSmem<PDF, OP_APPLY> &tl,
                                            const SymSrc &s, int j, bool k0, bool k1, SymAcc<PDF, OP_APPLY> &a,
                                            float2 *sac)
{
    const dfv<L2> TI = {{t.T.x, t.Tl.x}, {t.T.y, t.Tl.y}, {t.T.z, t.Tl.z}};
    const dfv<L2> TJ = {{l_bc<L2>(s.T[0]), l_bc<L2>(s.Tm[0])}, {l_bc<L2>(s.T[1]), l_bc<L2>(s.Tm[1])},
                        {l_bc<L2>(s.T[2]), l_bc<L2>(s.Tm[2])}};
    const dfv<L2> eI = {{t.e.x, t.el.x}, {t.e.y, t.el.y}, {t.e.z, t.el.z}};
    const dfv<L2> eJ = {{l_bc<L2>(-s.e[0]), l_bc<L2>(-s.em[0])}, {l_bc<L2>(-s.e[1]), l_bc<L2>(-s.em[1])},
                        {l_bc<L2>(-s.e[2]), l_bc<L2>(-s.em[2])}};
    const auto add3 = [](const dfv<L2> &x, const dfv<L2> &y) {
        return dfv<L2>{l_dfnorm(l_dfadd(x.x, y.x)), l_dfnorm(l_dfadd(x.y, y.y)), l_dfnorm(l_dfadd(x.z, y.z))};
    };
    dfv<L2> dd4[4];
    dd4[0] = {l_dfdiff(t.p.x, t.pl.x, l_bc<L2>(s.q[0]), l_bc<L2>(s.m[0])),
              l_dfdiff(t.p.y, t.pl.y, l_bc<L2>(s.q[1]), l_bc<L2>(s.m[1])),
              l_dfdiff(t.p.z, t.pl.z, l_bc<L2>(s.q[2]), l_bc<L2>(s.m[2]))};
    dd4[1] = add3(dd4[0], eJ);
    dd4[2] = add3(dd4[0], eI);
    dd4[3] = add3(dd4[1], eI);
    dfl<L2> d2[4], F[4], G[4], cI[2], cJ[2];
#pragma unroll
    for (int ab = 0; ab < 4; ++ab) {
        const dfv<L2> &d = dd4[ab];
        d2[ab] = l_dfnorm(l_dfnorm2(d));
        sym_df_powers(d2[ab], F[ab], G[ab]);
        // |T_I x d_ab|^2 depends on b only, |T_J x d_ab|^2 on a only (g_i2 = g_i1 + l_I T_I)
        if (ab < 2) cI[ab] = l_dfnorm(l_dfadd(d2[ab], l_dfneg(l_dfsqr(l_dfnorm(l_dfdot(TI, d))))));
        if (!(ab & 1)) cJ[ab >> 1] = l_dfnorm(l_dfadd(d2[ab], l_dfneg(l_dfsqr(l_dfnorm(l_dfdot(TJ, d))))));
    }
    dfl<L2> sw = l_dfadd(l_dfadd(F[0], F[3]), l_dfadd(F[1], F[2]));
    dfl<L2> sw0 = l_dfadd(l_dfadd(l_dfmul(l_dfadd(cI[0], cJ[0]), G[0]), l_dfmul(l_dfadd(cI[1], cJ[1]), G[3])),
                          l_dfadd(l_dfmul(l_dfadd(cI[1], cJ[0]), G[1]), l_dfmul(l_dfadd(cI[0], cJ[1]), G[2])));
    if constexpr (CHECK) {
        sw = {l_keep(k0, k1, sw.hi), l_keep(k0, k1, sw.lo)};
        sw0 = {l_keep(k0, k1, sw0.hi), l_keep(k0, k1, sw0.lo)};
    }
    const dfl<L2> ls = {l_bc<L2>(s.ell), l_bc<L2>(s.ell_lo)}, lt = {t.ell, t.ell_lo};
    const dfl<L2> Wt = l_dfmul(ls, sw), W0t = l_dfmul(ls, sw0), Ws = l_dfmul(lt, sw), W0s = l_dfneg(l_dfmul(lt, sw0));
    const dfv<L2> dT = {l_dfdiff(TI.x.hi, TI.x.lo, TJ.x.hi, TJ.x.lo), l_dfdiff(TI.y.hi, TI.y.lo, TJ.y.hi, TJ.y.lo),
                        l_dfdiff(TI.z.hi, TI.z.lo, TJ.z.hi, TJ.z.lo)};
    const dfl<L2> n2 = l_dfnorm2(dT), omt = {l_mul(l_bc<L2>(0.5f), n2.hi), l_mul(l_bc<L2>(0.5f), n2.lo)};
    const float4 x = tl.u0[0][j], y = tl.u1[0][j], z = tl.u2[0][j];
    const L2 sd[3] = {l_bc<L2>(x.x), l_bc<L2>(x.y), l_bc<L2>(x.z)}, sdl[3] = {l_bc<L2>(y.z), l_bc<L2>(y.w), l_bc<L2>(z.x)};
    const L2 sb[3] = {l_bc<L2>(x.w), l_bc<L2>(y.x), l_bc<L2>(y.y)}, sbl[3] = {l_bc<L2>(z.y), l_bc<L2>(z.z), l_bc<L2>(z.w)};
    const L2 td[3] = {tu.dh.x, tu.dh.y, tu.dh.z}, tdl[3] = {tu.dl.x, tu.dl.y, tu.dl.z};
    const L2 tb[3] = {tu.uh.x, tu.uh.y, tu.uh.z}, tbl[3] = {tu.ul.x, tu.ul.y, tu.ul.z};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const dfl<L2> dd = l_dfdiff(td[k], tdl[k], sd[k], sdl[k]), db = l_dfdiff(tb[k], tbl[k], sb[k], sbl[k]);
        // row I: (du_I - du_J) + omt du_J;  row J: (du_J - du_I) + omt du_I
        const dfl<L2> h = l_dfmul(Wt, l_dfadd(dd, l_dfmul(omt, dfl<L2>{sd[k], sdl[k]}))), m = l_dfmul(W0t, db);
        l_kahan_df(a.s[k], a.c[k], h.hi, h.lo);
        l_kahan_df(a.s[3 + k], a.c[3 + k], m.hi, m.lo);
        float2 ac = sac[k * kTile], bc = sac[(3 + k) * kTile];
        src_add_df(ac, l_dfmul(Ws, l_dfadd(l_dfmul(omt, dfl<L2>{td[k], tdl[k]}), l_dfneg(dd))));
        src_add_df(bc, l_dfmul(W0s, db));
        sac[k * kTile] = ac;
        sac[(3 + k) * kTile] = bc;
    }
}

template <int PREC, int OP, bool CHECK, int MODE>
__device__ __forceinline__ void sym_pair_apply(const SymTgt &t, const SymTgtU *tus, const SymSmem<PREC, OP> &tl, const SymSrc &s,
                                               int j, bool k0, bool k1, SymAcc<PREC, OP> &a, float2 *sac)
{
    constexpr bool MIX = PREC == PMIX;
    LV<L2> d[4];
    l_chords<(MODE >= 1 && MIX)>(t.p, t.pl, t.e, l_bc3<L2>(s.q[0], s.q[1], s.q[2]), l_bc3<L2>(s.m[0], s.m[1], s.m[2]),
                                 l_bc3<L2>(s.e[0], s.e[1], s.e[2]), d);
    const LV<L2> TJ = l_bc3<L2>(s.T[0], s.T[1], s.T[2]);
    const L2 cI1 = l_perp2(d[0], t.T), cI2 = l_perp2(d[1], t.T);
    const L2 cJ1 = l_perp2(d[0], TJ), cJ2 = l_perp2(d[2], TJ);
    L2 f[4], g[4];
#pragma unroll
    for (int ab = 0; ab < 4; ++ab) f[ab] = l_pow25(l_dot(d[ab], d[ab]), g[ab]);
    // (11 + 22) + (12 + 21): bitwise the same from row I and from row J
    L2 sw = l_add(l_add(f[0], f[3]), l_add(f[1], f[2]));
    L2 sw0 = l_add(l_fma(l_add(cI2, cJ2), g[3], l_mul(l_add(cI1, cJ1), g[0])),
                   l_add(l_mul(l_add(cI2, cJ1), g[1]), l_mul(l_add(cI1, cJ2), g[2])));
    if constexpr (CHECK) sw = l_keep(k0, k1, sw), sw0 = l_keep(k0, k1, sw0);
    LV<L2> dT = l_sub3(t.T, TJ);
    if constexpr (MIX) dT = l_add3(dT, l_sub3(t.Tl, l_bc3<L2>(s.Tm[0], s.Tm[1], s.Tm[2])));
    const L2 omt = l_mul(l_bc<L2>(0.5f), l_dot(dT, dT));  // |T_I - T_J|^2 / 2
    const L2 Wt = l_mul(l_bc<L2>(s.ell), sw), W0t = l_mul(l_bc<L2>(s.ell), sw0);
    const L2 Ws = l_mul(t.ell, sw), W0s = l_neg(l_mul(t.ell, sw0));
#pragma unroll
    for (int f = 0; f < sym_fields<OP>(); ++f) {
        const SymTgtU &tu = tus[f];
        const float4 x = tl.u0[f][j], y = tl.u1[f][j];
        const LV<L2> sdh = l_bc3<L2>(x.x, x.y, x.z);
        LV<L2> dd = l_sub3(tu.dh, sdh), db = l_sub3(tu.uh, l_bc3<L2>(x.w, y.x, y.y));
        if constexpr (MIX) {  // differences of the double-float u records
            const float4 z = tl.u2[f][j];
            dd = l_add3(dd, l_sub3(tu.dl, l_bc3<L2>(y.z, y.w, z.x)));
            db = l_add3(db, l_sub3(tu.ul, l_bc3<L2>(z.y, z.z, z.w)));
        }
        L2 *as = a.s + 6 * f, *ac = a.c + 6 * f;
        l_kahan_fma(as[0], ac[0], Wt, l_fma(omt, sdh.x, dd.x));
        l_kahan_fma(as[1], ac[1], Wt, l_fma(omt, sdh.y, dd.y));
        l_kahan_fma(as[2], ac[2], Wt, l_fma(omt, sdh.z, dd.z));
        l_kahan_fma(as[3], ac[3], W0t, db.x);
        l_kahan_fma(as[4], ac[4], W0t, db.y);
        l_kahan_fma(as[5], ac[5], W0t, db.z);
        const L2 v[6] = {l_fma(omt, tu.dh.x, l_neg(dd.x)), l_fma(omt, tu.dh.y, l_neg(dd.y)),
                         l_fma(omt, tu.dh.z, l_neg(dd.z)), db.x, db.y, db.z};
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            float2 *p = sac + (6 * f + q) * kTile, x2 = *p;
            src_add(x2, q < 3 ? Ws : W0s, v[q]);
            *p = x2;
        }
    }
}

template <int PREC, bool CHECK, int MODE>
__device__ __forceinline__ void sym_pair(const SymTgt &t, const SymTgtU *tu, const SymSmem<PREC, OP_APPLY> &tl, const SymSrc &s,
                                         int j, int, bool k0, bool k1, SymAcc<PREC, OP_APPLY> &a, float2 *sac, const SymArgs &,
                                         bool &, bool &)
{
    if constexpr (PREC == PDF)
        sym_pair_df<CHECK>(t, tu[0], tl, s, j, k0, k1, a, sac);
    else
        sym_pair_apply<PREC, OP_APPLY, CHECK, MODE>(t, tu, tl, s, j, k0, k1, a, sac);
}
template <int PREC, bool CHECK, int MODE>
__device__ __forceinline__ void sym_pair(const SymTgt &t, const SymTgtU *tu, const SymSmem<PREC, OP_APPLY2> &tl, const SymSrc &s,
                                         int j, int, bool k0, bool k1, SymAcc<PREC, OP_APPLY2> &a, float2 *sac, const SymArgs &,
                                         bool &, bool &)
{
    sym_pair_apply<PREC, OP_APPLY2, CHECK, MODE>(t, tu, tl, s, j, k0, k1, a, sac);
}

template <int PREC, bool CHECK, int MODE>
__device__ __forceinline__ void sym_pair(const SymTgt &t, const SymTgtU *, const SymSmem<PREC, OP_DIFF> &, const SymSrc &s,
                                         int, int, bool k0, bool k1, SymAcc<PREC, OP_DIFF> &a, float2 *sac,
                                         const SymArgs &pa, bool &n0, bool &n1)
{
    LV<L2> d[4];
    l_chords<(MODE >= 1)>(t.p, t.pl, t.e, l_bc3<L2>(s.q[0], s.q[1], s.q[2]), l_bc3<L2>(s.m[0], s.m[1], s.m[2]),
                          l_bc3<L2>(s.e[0], s.e[1], s.e[2]), d);
    const LV<L2> TJ = l_bc3<L2>(s.T[0], s.T[1], s.T[2]), TJl = l_bc3<L2>(s.Tm[0], s.Tm[1], s.Tm[2]);
    // both tangents double-float: each is the target tangent of one of the two rows
    L2 tI[2], tJ[2], cI[2], cJ[2];
    LV<L2> pI[2], pJ[2];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        cI[b] = l_perp2_df(d[b], t.T, t.Tl, tI[b], pI[b]);
        cJ[b] = l_perp2_df(d[2 * b], TJ, TJl, tJ[b], pJ[b]);
    }
    const L2 d11 = l_dot(d[0], d[0]);
    if constexpr (MODE == 2) {
        n0 = k0 && d11.x < pa.near2f;
        n1 = k1 && d11.y < pa.near2f;
    }
    const bool m0 = k0 && !n0, m1 = k1 && !n1;  // pairs of the FP32 sums
    L2 S, G[2][3], H[2][3], GT[3], HT[3];
#pragma unroll
    for (int ab = 0; ab < 4; ++ab) {
        const int ia = ab >> 1, jb = ab & 1;
        L2 d2 = ab == 0 ? d11 : l_dot(d[ab], d[ab]);
        if constexpr (CHECK || MODE == 2) d2 = make_float2(m0 ? d2.x : 1.f, m1 ? d2.y : 1.f);
        L2 r2;
        L2 rb = l_pow45(d2, r2);
        if constexpr (CHECK || MODE == 2) rb = l_keep(m0, m1, rb);
        const L2 fs = l_fma(cJ[ia], rb, l_mul(cI[jb], rb));
        const L2 al = l_add(rb, rb);  // alpha |d|^-beta
        const L2 cb = l_neg(l_mul(l_mul(l_bc<L2>(4.5f), fs), r2));
        const L2 mI = l_neg(l_mul(al, ia ? l_add(tI[jb], t.ell) : tI[jb]));
        const L2 mJ = l_neg(l_mul(al, jb ? l_sub(tJ[ia], l_bc<L2>(s.ell)) : tJ[ia]));
        const L2 dv[3] = {d[ab].x, d[ab].y, d[ab].z};
        const LV<L2> ps = l_add3(pI[jb], pJ[ia]);
        const L2 pv[3] = {ps.x, ps.y, ps.z};
        S = ab == 0 ? fs : l_add(S, fs);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const L2 v = l_fma(al, pv[k], l_mul(cb, dv[k]));
            G[ia][k] = jb ? l_add(G[ia][k], v) : v;
            H[jb][k] = ia ? l_sub(H[jb][k], v) : l_neg(v);
            GT[k] = ab == 0 ? l_mul(mI, dv[k]) : l_fma(mI, dv[k], GT[k]);
            HT[k] = ab == 0 ? l_mul(mJ, dv[k]) : l_fma(mJ, dv[k], HT[k]);
        }
    }
    const L2 L = l_bc<L2>(l_mul(s.ell, pa.sum_scale)), tL = l_mul(t.ell, l_bc<L2>(pa.sum_scale));
    l_kahan_fma(a.s[0], a.c[0], L, S);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        l_kahan_fma(a.s[1 + k], a.c[1 + k], L, G[0][k]);
        l_kahan_fma(a.s[4 + k], a.c[4 + k], L, G[1][k]);
        l_kahan_fma(a.s[7 + k], a.c[7 + k], L, GT[k]);
    }
#pragma unroll
    for (int q = 0; q < 10; ++q) {
        float2 ac = sac[q * kTile];
        src_add(ac, tL, q == 0 ? S : (q < 4 ? H[0][(q + 2) % 3] : (q < 7 ? H[1][(q + 2) % 3] : HT[(q + 2) % 3])));
        sac[q * kTile] = ac;
    }
}

// Place of tile row j in the shared arrays: even rows first, so that the rows step + 2 lane of a warp are
// consecutive.
__device__ __forceinline__ int sym_slot(int j) { return ((j & 1) << 6) | (j >> 1); }

// Evaluate `count` near pairs of the differential from a warp's queue, 32 at a time, into the warp's target and
// source sums.  Near pairs held back this way fill all lanes: on short curves every step has a few lanes
// near another strand, and evaluated in place each of them cost the warp a whole double-float pair.  Pairs of
// one round that share a row add in queue order, one at a time.
static __device__ __noinline__ void sym_near_flush(SymSmem<PMIX, OP_DIFF> &sm, int wid, int first, int count, int tgt0, int ntgt,
                                                   int s0, const SymArgs &pa)
{
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int base = 0; base < count; base += 32) {
        bool on = base + lane < count;
        const int v = sm.queue[wid][first + (on ? base + lane : 0)];
        const int row = v >> 8, at = v & 0xff, loc = kSection * wid + row;
        on = on && loc < ntgt;
        dfl<float> x[10], y[10];
        near_diff(pa.recF, pa.recLo, tgt0 + min(loc, ntgt - 1), s0 + (((at & 63) << 1) | (at >> 6)), pa.sum_exp, x, y);
        const unsigned live = __ballot_sync(0xffffffffu, on);
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            const int key = on ? (side ? at : row) : 256 + lane;
            const unsigned same = __match_any_sync(0xffffffffu, key) & live;
            const int rank = __popc(same & ((1u << lane) - 1));
            const int rounds = __reduce_max_sync(0xffffffffu, on ? rank + 1 : 0);
            for (int r = 0; r < rounds; ++r) {
                if (on && rank == r) {
                    float2 *ac = side ? &sm.sac[wid][0][at] : &sm.tac[wid][0][row];
#pragma unroll
                    for (int q = 0; q < 10; ++q, ac += side ? kTile : kSection) {
                        const dfl<float> v = side ? y[q] : x[q];
                        float2 t = *ac;
                        l_kahan_df(t.x, t.y, v.hi, v.lo);
                        *ac = t;
                    }
                }
                __syncwarp();
            }
        }
    }
}

// Staggered loop of one warp over sources [j0, j0 + cnt) of the staged tile (global rows s0 + j).
// CHECK: some pair may share a vertex; MODE 2: near pairs possible, 1: double-float chords, 0: single-float
// chords (far tiles).  OWN: the sources are the warp's own 64 rows; each unordered pair once, by the row that
// sees the other at most half the circle of 64 ahead.  Otherwise steps [first, last) of the circle (last < 0: all).
template <int PREC, int OP, bool CHECK, int MODE, bool OWN>
__device__ __forceinline__ void sym_section(const SymTgt &t, const SymTgtU *tu, SymSmem<PREC, OP> &sm, int wid, int s0,
                                            int j0, int cnt, SymAcc<PREC, OP> &a, int &queued, const WorkItem &w,
                                            const SymArgs &pa, int first = 0, int last = -1)
{
    constexpr bool QUEUE = OP == OP_DIFF && MODE == 2;
    const int lane = threadIdx.x & 31;
    const int P = OWN ? kSection : max((cnt + 1) & ~1, kSection), n = OWN ? kSection / 2 + 2 : (last < 0 ? P : last);
    for (int step = OWN ? 1 : first; step < n; ++step) {
        int j = step + 2 * lane;
        if (j >= P) j -= P;
        const int at = sym_slot(j + j0);
        bool n0 = false, n1 = false;
        if (j < cnt) {
            j += j0;
            SymSrc s;
            sym_load<PREC, OP, CHECK>(s, sm, at);
            bool k0 = true, k1 = true;
            if constexpr (CHECK) {
                k0 = (s.j1 != t.i1[0]) & (s.j1 != t.i2[0]) & (s.j2 != t.i1[0]) & (s.j2 != t.i2[0]);
                k1 = (s.j1 != t.i1[1]) & (s.j1 != t.i2[1]) & (s.j2 != t.i1[1]) & (s.j2 != t.i2[1]);
            }
            if constexpr (OWN) {  // row 2 lane is `step` behind the source, row 2 lane + 1 is step - 1 behind
                k0 = k0 & (step < 32 || (step == 32 && lane < 16));
                k1 = k1 & (step > 1) & (step < 33 || lane < 16);
            }
            sym_pair<PREC, CHECK, MODE>(t, tu, sm, s, at, s0 + j, k0, k1, a, &sm.sac[wid][0][at], pa, n0, n1);
        }
        if constexpr (PREC == PDF)
            if ((step & 3) == 3)
#pragma unroll
                for (int q = 0; q < 6; ++q) l_kahan_norm(a.s[q], a.c[q]);
        __syncwarp();  // the next step hands this lane's source on
        if constexpr (QUEUE) {
            const unsigned b0 = __ballot_sync(0xffffffffu, n0), b1 = __ballot_sync(0xffffffffu, n1);
            if (b0 | b1) {
                const unsigned lt = (1u << lane) - 1;
                if (n0) sm.queue[wid][queued + __popc(b0 & lt)] = (unsigned short)((2 * lane) << 8 | at);
                if (n1) sm.queue[wid][queued + __popc(b0) + __popc(b1 & lt)] = (unsigned short)((2 * lane + 1) << 8 | at);
                queued += __popc(b0) + __popc(b1);
                __syncwarp();
                if (queued >= 64) {  // the last 64; the rest stays queued
                    queued -= 64;
                    sym_near_flush(sm, wid, queued, 64, w.tgt0, w.ntgt, s0, pa);
                }
            }
        }
    }
}

template <int PREC, int OP, int MB>
__global__ void __launch_bounds__(kThreads, MB) k_sym(const SymArgs pa)
{
    constexpr int W = sym_width<OP>();
    constexpr bool MIX = PREC != P32, DF = PREC == PDF, NEAR = PREC == PMIX && (OP == OP_ENERGY || OP == OP_DIFF);
    constexpr int F = sym_fields<OP>();
    extern __shared__ __align__(16) unsigned char dyn[];
    SymSmem<PREC, OP> &sm = *reinterpret_cast<SymSmem<PREC, OP> *>(dyn);
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (;;) {
        if (threadIdx.x == 0) sm.item = atomicAdd(pa.counter, 1);
        __syncthreads();
        const int it = sm.item;
        __syncthreads();
        if (it >= pa.n_items) {
            queue_done(it, pa.n_items, pa.counter);
            break;
        }
        const WorkItem w = pa.items[it];
        if (pa.skip && pa.skip[w.pad]) continue;  // problem already converged
        const int X = w.slot >> 16, tslot = w.slot & 0xffff;
        const bool diag = w.src0 < w.tgt0 + w.ntgt;  // a tile of its own super-block
        SymTgt t;
        SymTgtU tu[F ? F : 1];
        float tbox[6] = {1e30f, 1e30f, 1e30f, -1e30f, -1e30f, -1e30f};
        {
            RecF r[2];
            RecLo q[2];
            bool valid[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int loc = kSection * wid + 2 * lane + k;
                valid[k] = loc < w.ntgt;
                const int I = w.tgt0 + min(loc, w.ntgt - 1);
                t.row[k] = I;
                r[k] = pa.recF[I];
                if constexpr (MIX) q[k] = pa.recLo[I];
                t.i1[k] = __float_as_int(r[k].c.z);
                t.i2[k] = __float_as_int(r[k].c.w);
                if constexpr (MIX)
                    box_add(tbox, V3<float>{r[k].a.x, r[k].a.y, r[k].a.z}, V3<float>{r[k].b.x, r[k].b.y, r[k].b.z});
            }
#define TPE_L2(field) make_float2(r[0].field, r[1].field)
#define TPE_Q2(field) make_float2(q[0].field, q[1].field)
#define TPE_U2(field) make_float2(u[0].field, u[1].field)
            t.p = {TPE_L2(a.x), TPE_L2(a.y), TPE_L2(a.z)};
            t.T = {TPE_L2(b.w), TPE_L2(c.x), TPE_L2(c.y)};
            t.ell = make_float2(valid[0] ? r[0].a.w : 0.f, valid[1] ? r[1].a.w : 0.f);
            if constexpr (MIX) {
                t.pl = {TPE_Q2(lo.x), TPE_Q2(lo.y), TPE_Q2(lo.z)};
                t.Tl = {TPE_Q2(lo2.z), TPE_Q2(lo2.w), TPE_Q2(lo3.x)};
                if constexpr (DF) {
                    const dfl<L2> ex = l_dfdiff(TPE_L2(b.x), TPE_Q2(lo.w), t.p.x, t.pl.x),
                                  ey = l_dfdiff(TPE_L2(b.y), TPE_Q2(lo2.x), t.p.y, t.pl.y),
                                  ez = l_dfdiff(TPE_L2(b.z), TPE_Q2(lo2.y), t.p.z, t.pl.z);
                    t.e = {ex.hi, ey.hi, ez.hi};
                    t.el = {ex.lo, ey.lo, ez.lo};
                    t.ell_lo = make_float2(valid[0] ? pa.ell_lo[t.row[0]] : 0.f, valid[1] ? pa.ell_lo[t.row[1]] : 0.f);
                } else {
                    t.e = {TPE_Q2(lo3.y), TPE_Q2(lo3.z), TPE_Q2(lo3.w)};
                }
            } else {
                t.e = l_sub3(LV<L2>{TPE_L2(b.x), TPE_L2(b.y), TPE_L2(b.z)}, t.p);
            }
#pragma unroll
            for (int f = 0; f < F; ++f) {
                const URecF u[2] = {pa.urecF[(size_t)f * pa.nE + t.row[0]], pa.urecF[(size_t)f * pa.nE + t.row[1]]};
                tu[f].dh = {TPE_U2(a.x), TPE_U2(a.y), TPE_U2(a.z)};
                tu[f].uh = {TPE_U2(a.w), TPE_U2(b.x), TPE_U2(b.y)};
                if constexpr (MIX) {
                    tu[f].dl = {TPE_U2(b.z), TPE_U2(b.w), TPE_U2(c.x)};
                    tu[f].ul = {TPE_U2(c.y), TPE_U2(c.z), TPE_U2(c.w)};
                }
            }
#undef TPE_L2
#undef TPE_Q2
#undef TPE_U2
            if (!valid[0]) t.p.x.x = 1e18f;
            if (!valid[1]) t.p.x.y = 1e18f;
        }
        if constexpr (MIX) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                for (int k = 0; k < 6; ++k) {
                    const float v = __shfl_xor_sync(0xffffffffu, tbox[k], o);
                    tbox[k] = k < 3 ? fminf(tbox[k], v) : fmaxf(tbox[k], v);
                }
        }
        SymAcc<PREC, OP> a;
#pragma unroll
        for (int k = 0; k < W; ++k) a.s[k] = a.c[k] = make_float2(0.f, 0.f);
        const bool have = kSection * wid < w.ntgt;  // this warp has target rows
        int queued = 0;                             // near pairs held back
        if constexpr (OP == OP_DIFF)
            for (int q = 0; q < W; ++q)
                for (int j = lane; j < kSection; j += 32) sm.tac[wid][q][j] = make_float2(0.f, 0.f);
        for (int s0 = w.src0, tile = 0; s0 < w.src1; s0 += kTile, ++tile) {
            const int cnt = min(kTile, w.src1 - s0);
            __syncthreads();  // the previous tile's readers are done
            float sb[6] = {1e30f, 1e30f, 1e30f, -1e30f, -1e30f, -1e30f};
            if (threadIdx.x < cnt) {
                const int J = s0 + threadIdx.x, j = sym_slot(threadIdx.x);
                const RecF r = pa.recF[J];
                sm.t0[j] = r.a;
                sm.id[j] = make_int2(__float_as_int(r.c.z), __float_as_int(r.c.w));
                if constexpr (MIX) {
                    const RecLo q = pa.recLo[J];
                    if constexpr (DF) {
                        const dfl<float> ex = l_dfdiff(r.b.x, q.lo.w, r.a.x, q.lo.x), ey = l_dfdiff(r.b.y, q.lo2.x, r.a.y, q.lo.y),
                                         ez = l_dfdiff(r.b.z, q.lo2.y, r.a.z, q.lo.z);
                        sm.t1[j] = make_float4(ex.hi, ey.hi, ez.hi, r.b.w);
                        sm.t4[j] = make_float4(ex.lo, ey.lo, ez.lo, pa.ell_lo[J]);
                    } else {
                        sm.t1[j] = make_float4(q.lo3.y, q.lo3.z, q.lo3.w, r.b.w);
                    }
                    sm.t2[j] = make_float4(r.c.x, r.c.y, q.lo.x, q.lo.y);
                    sm.t3[j] = make_float4(q.lo.z, q.lo2.z, q.lo2.w, q.lo3.x);
                    box_add(sb, V3<float>{r.a.x, r.a.y, r.a.z}, V3<float>{r.b.x, r.b.y, r.b.z});
                } else {
                    sm.t1[j] = make_float4(r.b.x - r.a.x, r.b.y - r.a.y, r.b.z - r.a.z, r.b.w);
                    sm.t2[j] = make_float4(r.c.x, r.c.y, 0.f, 0.f);
                }
#pragma unroll
                for (int f = 0; f < F; ++f) {
                    const URecF u = pa.urecF[(size_t)f * pa.nE + J];
                    sm.u0[f][j] = u.a;
                    sm.u1[f][j] = u.b;
                    if constexpr (MIX) sm.u2[f][j] = u.c;
                }
            }
            for (int q = 0; q < W; ++q)
                for (int j = lane; j < kTile; j += 32) sm.sac[wid][q][j] = make_float2(0.f, 0.f);
            if constexpr (MIX)
                block_box(sb, sm.box);  // contains the barrier that publishes the tile
            else
                __syncthreads();
            int mode = 1;
            if constexpr (MIX) {
                float g2 = 0.f;
                for (int q = 0; q < 3; ++q) {
                    const float gap = fmaxf(fmaxf(sb[q] - tbox[3 + q], tbox[q] - sb[3 + q]), 0.f);
                    g2 += gap * gap;
                }
                mode = (NEAR && g2 < pa.near2f) ? 2 : (DF || g2 < pa.mid2f ? 1 : 0);
            }
            constexpr int MN = NEAR ? 2 : 1;
            if (diag) {
                // the super-block's 64-row sections: in the tile of its own a warp takes those rows and half of the
                // pairs with the tile's other section, in the other tile one whole section: 65 or 64 steps.  The pair
                // of sections (even, odd) is cut where the even row 2 l sees sources 2 l to 2 l + 31 of the circle;
                // the rest is steps 2 to 33 of the odd section against the even one.
                if (have) {
                    const int sec = (s0 - w.tgt0) / kSection;
                    if ((wid & 2) == sec) {
                        sym_section<PREC, OP, true, MN, true>(t, tu, sm, wid, s0, kSection * (wid & 1),
                                                              min(kSection, w.ntgt - kSection * wid), a, queued, w, pa);
                        const int o = (wid & 1) ^ 1, oc = min(kSection, w.ntgt - kSection * (wid ^ 1));
                        if (oc > 0)
                            sym_section<PREC, OP, true, MN, false>(t, tu, sm, wid, s0, kSection * o, oc, a, queued, w, pa,
                                                                   o ? 0 : 2, o ? kSection / 2 : kSection / 2 + 2);
                    } else {
                        const int g = wid >= 2 ? wid - 2 : 3 - wid, gc = min(kSection, w.ntgt - kSection * g);
                        if (gc > 0)
                            sym_section<PREC, OP, true, MN, false>(t, tu, sm, wid, s0, kSection * (g - sec), gc, a, queued, w,
                                                                   pa);
                    }
                }
            } else if (have) {
                if (((w.nb_lo >> tile) & 1) || mode == 2)
                    sym_section<PREC, OP, true, MN, false>(t, tu, sm, wid, s0, 0, cnt, a, queued, w, pa);
                else if (mode == 1 || !MIX)
                    sym_section<PREC, OP, false, 1, false>(t, tu, sm, wid, s0, 0, cnt, a, queued, w, pa);
                else if constexpr (PREC == PMIX)
                    sym_section<PREC, OP, false, 0, false>(t, tu, sm, wid, s0, 0, cnt, a, queued, w, pa);
            }
            if constexpr (OP == OP_DIFF) {
                if (queued) sym_near_flush(sm, wid, 0, queued, w.tgt0, w.ntgt, s0, pa);
                queued = 0;
            }
            __syncthreads();  // every warp's source accumulators are complete
            if (threadIdx.x < cnt) {
                float2 *o = pa.part + ((size_t)X * pa.nE + s0 + threadIdx.x) * W;
#pragma unroll
                for (int q = 0; q < W; ++q) {
                    const int at = sym_slot(threadIdx.x);
                    float2 x = sm.sac[0][q][at];
                    float lo = -x.y;
#pragma unroll
                    for (int wv = 1; wv < kSymWarps; ++wv) {
                        const float2 y = sm.sac[wv][q][at];
                        const df s = two_sum(x.x, y.x);
                        x.x = s.hi;
                        lo = __fadd_rn(lo, __fsub_rn(s.lo, y.y));
                    }
                    o[q] = make_float2(x.x, lo);
                }
            }
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int loc = kSection * wid + 2 * lane + k;
            if (loc >= w.ntgt) continue;
            float2 *o = pa.part + ((size_t)tslot * pa.nE + w.tgt0 + loc) * W;
            if constexpr (OP == OP_DIFF) {
#pragma unroll
                for (int q = 0; q < W; ++q) {
                    const float2 v = sm.tac[wid][q][2 * lane + k];
                    if (k)
                        l_kahan_df(a.s[q].y, a.c[q].y, v.x, -v.y);
                    else
                        l_kahan_df(a.s[q].x, a.c[q].x, v.x, -v.y);
                }
            }
#pragma unroll
            for (int q = 0; q < W; ++q)
                o[q] = k ? make_float2(a.s[q].y, -a.c[q].y) : make_float2(a.s[q].x, -a.c[q].x);
        }
    }
}

// Row output of the differential from its accumulators (Sec. 5.1 by the chain rule through l_I and T_I):
// G_i1 = (1/4)[-T S + l G1 - (Id - T T^t) GT],  G_i2 = (1/4)[T S + l G2 + (Id - T T^t) GT]; quarter: 1/4 over the scale of
// the sums
__device__ __forceinline__ void diff_row_out(const double *T, double l, double quarter, const double *v, double *o)
{
    const double *G1 = v + 1, *G2 = v + 4, *GT = v + 7;
    const double gt = T[0] * GT[0] + T[1] * GT[1] + T[2] * GT[2];
    for (int c = 0; c < 3; ++c) {
        const double pgt = GT[c] - gt * T[c];
        o[c] = quarter * (-T[c] * v[0] + l * G1[c] - pgt);
        o[3 + c] = quarter * (T[c] * v[0] + l * G2[c] + pgt);
    }
}

// Sum the slots of every row (one thread per value, so that a slot's values are read coalesced) and form the
// row's outputs: energy rows (l_I / 4) sum, or the six endpoint values of an edge into esum.
// D64: in FP64 (the accurate apply), else in double-float.
template <int OP, bool D64 = false>
__global__ void __launch_bounds__(OP == OP_ENERGY ? 256 : 32 * sym_width<OP>())
k_sym_sum(int nE, const int *__restrict__ eslots, const float2 *__restrict__ part, const double *__restrict__ ell,
          const double *__restrict__ T, double quarter, double *__restrict__ out)
{
    constexpr int W = sym_width<OP>(), R = OP == OP_ENERGY ? 256 : 32;  // rows per block
    __shared__ double sh[OP == OP_ENERGY ? 1 : R * W];
    const int row = blockIdx.x * R + threadIdx.x / W;
    double x = 0.0;
    if (row < nE) {
        const size_t step = (size_t)nE * W;
        const float2 *p = part + (size_t)blockIdx.x * R * W + threadIdx.x;
        const int ns = eslots[row];
        float s = 0.f, lo = 0.f;
        int q = 0;
        for (; q + 8 <= ns; q += 8) {
            float2 v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = __ldcs(p + (size_t)(q + k) * step);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if constexpr (D64) {
                    x += (double)v[k].x + (double)v[k].y;
                    continue;
                }
                const df r = two_sum(s, v[k].x);
                s = r.hi;
                lo = __fadd_rn(lo, __fadd_rn(r.lo, v[k].y));
            }
        }
        for (; q < ns; ++q) {
            const float2 v = __ldcs(p + (size_t)q * step);
            if constexpr (D64) {
                x += (double)v.x + (double)v.y;
                continue;
            }
            const df r = two_sum(s, v.x);
            s = r.hi;
            lo = __fadd_rn(lo, __fadd_rn(r.lo, v.y));
        }
        if constexpr (!D64) x = OP == OP_ENERGY && isinf(s) ? (double)s : (double)s + (double)lo;
    }
    if constexpr (OP == OP_ENERGY) {
        if (row < nE) out[row] = quarter * ell[row] * x;
    } else {
        sh[threadIdx.x] = x;
        __syncthreads();
        const int I = blockIdx.x * R + threadIdx.x;
        if (threadIdx.x >= R || I >= nE) return;
        const double *v = sh + W * threadIdx.x;
        const double l = ell[I];
        for (int f = 0; f < (OP == OP_APPLY2 ? 2 : 1); ++f, v += 6, out += 6 * (size_t)nE) {
            double o[6];
            if constexpr (OP == OP_DIFF) {
                diff_row_out(T + 3 * (size_t)I, l, quarter, v, o);
            } else {
                for (int c = 0; c < 3; ++c) {
                    o[c] = 0.5 * v[c];
                    o[3 + c] = 0.125 * l * v[3 + c];
                }
            }
            for (int c = 0; c < 6; ++c) out[6 * (size_t)I + c] = o[c];
        }
    }
}

// ---------------------------------------------------------------------------------- host side

// Source rows per item beyond the own super-block: four tiles (fewer partial slots, longer runs per target load) once
// every resident CTA gets about six items that way, fewer on smaller graphs so that the last wave stays short, and
// half a tile where even whole tiles would be fewer: an item among near pairs takes many times the others' time
// (mixed, half / whole tiles: one knot of 4,096 edges differential 393 / 556 us, apply 103 / 107; 4 x 4,096 610 / 728 and
// 282 / 319; 8 x 1,500 425 / 507 and 105 / 142; 96 x 500, where the super-blocks themselves hold the near pairs, 826 / 792
// and 151 / 175).
static int sym_item_span(const Ctx &c, int resident)
{
    long long tiles = 0;
    for (int q = 0; q < c.nProb; ++q) {
        const long long n = c.h_prob_e[q + 1] - c.h_prob_e[q], nb = (n + kTile - 1) / kTile, ns = (n + kSuper - 1) / kSuper;
        for (long long X = 0; X < ns; ++X) tiles += std::max(0LL, nb - 2 * X - 2);
    }
    const long long per = tiles / (6LL * std::max(1, resident));
    return per ? kTile * (int)std::min<long long>(kSymMaxTiles, per) : kTile / 2;
}

// Slots a row of super-block X of a problem with n rows has at `span` source rows per item.
static int sym_row_slots(int X, int n, int span)
{
    const int nb = (n + kTile - 1) / kTile, m = std::max(0, n - (X + 1) * kSuper);
    return X + std::min(3, nb - 2 * X + 1) + (m + span - 1) / span;
}

static int sym_max_slots(const Ctx &c, int span)
{
    int ms = 1;
    for (int q = 0; q < c.nProb; ++q) {
        const int n = c.h_prob_e[q + 1] - c.h_prob_e[q], ns = (n + kSuper - 1) / kSuper;
        for (int X = 0; X < ns; ++X) ms = std::max(ms, sym_row_slots(X, n, span));
    }
    return ms;
}

static cudaError_t sym_plan(Ctx &c, Ctx::Plan &pl, int occupancy)
{
    const int resident = c.sm_count * std::max(1, occupancy);
    const int span = sym_item_span(c, resident);
    const std::vector<int> &ptr = c.h_inc_ptr, &inc = c.h_inc;  // (edge, end) pairs at every vertex
    struct Tmp {
        WorkItem w;
        int cost;
    };
    std::vector<Tmp> tmp;
    std::vector<int> eslots(std::max(1, c.nE), 0);
    std::vector<char> touch;
    for (int q = 0; q < c.nProb; ++q) {
        const int e0 = c.h_prob_e[q], e1 = c.h_prob_e[q + 1], n = e1 - e0;
        if (n <= 0) continue;
        const int nb = (n + kTile - 1) / kTile, ns = (n + kSuper - 1) / kSuper;
        for (int X = 0; X < ns; ++X) {
            const int t0 = e0 + X * kSuper, nt = std::min(kSuper, e1 - t0);
            touch.assign(nb, 0);
            for (int I = t0; I < t0 + nt; ++I)
                for (int s = 0; s < 2; ++s) {
                    const int v = c.h_edges[2 * I + s];
                    for (int k = ptr[v]; k < ptr[v + 1]; ++k) {
                        const int J = inc[k] >> 1;
                        if (J >= e0 && J < e1) touch[(J - e0) / kTile] = 1;
                    }
                }
            // tiles with near pairs take longer: they and the super-block itself go first
            int slot = X + 1;
            for (int h = t0; h < t0 + nt; h += kTile, ++slot)
                tmp.push_back({WorkItem{t0, nt, h, std::min(h + kTile, t0 + nt), (X << 16) | slot, 3, 0, q}, 1 + kSymMaxTiles});
            for (int s0 = (X + 1) * kSuper; s0 < n; s0 += span, ++slot) {  // whole tiles, or half a tile
                const int s1 = std::min(n, s0 + span);
                int mask = 0;
                for (int k = s0; k < s1; k += kTile) mask |= touch[k / kTile] << ((k - s0) / kTile);
                tmp.push_back({WorkItem{t0, nt, e0 + s0, e0 + s1, (X << 16) | slot, mask, 0, q},
                               (s1 - s0 + kTile - 1) / kTile + (mask ? kSymMaxTiles : 0)});
            }
            std::fill_n(eslots.begin() + t0, nt, sym_row_slots(X, n, span));
        }
    }
    std::stable_sort(tmp.begin(), tmp.end(), [](const Tmp &a, const Tmp &b) { return a.cost > b.cost; });
    std::vector<WorkItem> items;
    items.reserve(tmp.size());
    for (auto &t : tmp) items.push_back(t.w);
    pl.n_items = (int)items.size();
    pl.max_slots = sym_max_slots(c, span);
    pl.grid = std::max(1, std::min(pl.n_items, resident));
    return plan_upload(pl, items, eslots);
}

constexpr int kSymAccurate = 100;  // the apply in double-float

// Variants differ in the CTAs per SM that the register allocation is held to.
template <class F>
static void with_sym_kernel(int prec, int op, int variant, F f)
{
    if (op == OP_ENERGY) {
        if (prec == TP_FP32)
            f(k_sym<P32, OP_ENERGY, 4>, sizeof(SymSmem<P32, OP_ENERGY>));
        else if (variant == 2)
            f(k_sym<PMIX, OP_ENERGY, 4>, sizeof(SymSmem<PMIX, OP_ENERGY>));
        else
            f(k_sym<PMIX, OP_ENERGY, 3>, sizeof(SymSmem<PMIX, OP_ENERGY>));
    } else if (op == OP_DIFF) {
        if (variant >= 3)
            f(k_sym<PMIX, OP_DIFF, 3>, sizeof(SymSmem<PMIX, OP_DIFF>));
        else
            f(k_sym<PMIX, OP_DIFF, 2>, sizeof(SymSmem<PMIX, OP_DIFF>));
    } else if (op == OP_APPLY2) {
        f(k_sym<PMIX, OP_APPLY2, 2>, sizeof(SymSmem<PMIX, OP_APPLY2>));
    } else {
        if (variant == kSymAccurate)
            f(k_sym<PDF, OP_APPLY, 2>, sizeof(SymSmem<PDF, OP_APPLY>));
        else if (prec == TP_FP32)
            f(k_sym<P32, OP_APPLY, 3>, sizeof(SymSmem<P32, OP_APPLY>));
        else if (variant == 2)
            f(k_sym<PMIX, OP_APPLY, 2>, sizeof(SymSmem<PMIX, OP_APPLY>));
        else
            f(k_sym<PMIX, OP_APPLY, 3>, sizeof(SymSmem<PMIX, OP_APPLY>));
    }
}

static int sym_occupancy(const Ctx &c, int op, int variant)
{
    int occ = 0;
    with_sym_kernel(c.prm.precision, op, variant, [&](auto kern, size_t smem) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kThreads, smem);
    });
    return occ;
}

static int sym_op_width(int op) { return op == OP_ENERGY ? 1 : (op == OP_DIFF ? 10 : (op == OP_APPLY2 ? 12 : 6)); }

// Doubles of the partial buffer the symmetric pass of `op` needs.
size_t sym_part_elems(const Ctx &c, int op, int variant)
{
    const int span = sym_item_span(c, c.sm_count * std::max(1, sym_occupancy(c, op, variant)));
    return (size_t)sym_max_slots(c, span) * std::max(1, c.nE) * sym_op_width(op);
}

// Doubles of partial sums the pass of a built plan writes.
static size_t plan_elems(const Ctx &c, const Ctx::Plan &pl, int op)
{
    return (size_t)pl.max_slots * std::max(1, c.nE) * sym_op_width(op);
}

// Switch one pass to its symmetric form (variant > 0) or back to the gather form; grows the partial buffer.  On
// failure the pass runs in gather form.
static cudaError_t select_pass(Ctx &c, int op, int variant, int max_variant, Ctx::Plan &pl, int &flag)
{
    graphs_reset(c);
    plan_free(pl);
    flag = 0;
    if (variant <= 0) return cudaSuccess;
    if (!c.kp.fast || variant > max_variant) return cudaErrorInvalidValue;
    if (c.prm.precision != TP_MIXED && !(c.prm.precision == TP_FP32 && op != OP_DIFF)) return cudaErrorInvalidValue;
    TPE_CHECK(sym_plan(c, pl, sym_occupancy(c, op, variant)));
    pl.tpt = variant;
    const cudaError_t e = part_reserve(c, plan_elems(c, pl, op));
    if (e != cudaSuccess) {
        plan_free(pl);
        return e;
    }
    flag = variant;
    return cudaGetLastError();
}

cudaError_t sym_select(Ctx &c, int v) { return select_pass(c, OP_APPLY, v, 2, c.plan_sym, c.apply_sym); }
cudaError_t sym_select_energy(Ctx &c, int v) { return select_pass(c, OP_ENERGY, v, 2, c.plan_sym_e, c.energy_sym); }
cudaError_t sym_select_diff(Ctx &c, int v) { return select_pass(c, OP_DIFF, v, 4, c.plan_sym_d, c.diff_sym); }

// Whether a context runs the pass of `op` in symmetric form by itself: where a work list of whole tiles gives every
// resident CTA an item, or (mixed precision) where the unordered pairs per SM reach 22,000, for the energy
// 50,000 (sym_default_elems limits the partial sums).  On smaller graphs the gather pass's short chunks spread the work better
// and the symmetric pass waits for its longest item.  Gather / symmetric in us:
//   edges      pairs/SM   differential    apply      energy
//   2,000        13,000     268 / 320     50 / 55    47 / 64
//   2,500        20,500     368 / 456     74 / 72    58 / 80
//   3,000        29,600     448 / 414     96 / 72    67 / 81
//   3,500        40,300     659 / 479    116 / 90    84 / 80
//   4,096        55,200     589 / 402    123 / 104   96 / 90
//   20 x 500     16,400     439 / 353     67 / 73    57 / 73
//   12 x 1,000   39,400     550 / 398    114 / 91    89 / 100
//   120 x 256    25,800     816 / 524     88 / 76    85 / 93
// The rule separates single curves.  A batch of short ones just below it stays on the gather differential although the
// symmetric one is faster there (20 x 500).
static bool sym_pays(const Ctx &c, int op)
{
    if (c.sym_choice[op] >= 0) return false;
    if (!c.kp.fast || c.prm.precision == TP_FP64 || (op == OP_DIFF && c.prm.precision != TP_MIXED)) return false;
    long long items = 0;
    double pairs = 0.0;
    for (int q = 0; q < c.nProb; ++q) {
        const long long n = c.h_prob_e[q + 1] - c.h_prob_e[q], nb = (n + kTile - 1) / kTile, ns = (n + kSuper - 1) / kSuper;
        for (long long X = 0; X < ns; ++X) items += nb - 2 * X;
        pairs += 0.5 * (double)n * (double)n;
    }
    const bool enough = c.prm.precision == TP_MIXED && pairs >= (op == OP_ENERGY ? 50e3 : 22e3) * c.sm_count;
    if (!enough && items < c.sm_count) return false;  // no need to load the kernel for its occupancy
    return enough || items >= (long long)c.sm_count * std::max(1, sym_occupancy(c, op, 1));
}

// Doubles of partial sums the passes that pay may take unasked: 1 GiB a context, and a 64th of the free memory where that
// is less (a program with many contexts, or one whose other pools hold most of the device, gets the gather passes,
// which need tens of MB).  Up to 64 MiB the free memory is not looked up.
size_t sym_default_elems(const Ctx &c)
{
    size_t need = 0, limit = (size_t)1 << 30;
    bool looked_up = false;
    for (int op : {OP_ENERGY, OP_DIFF, OP_APPLY}) {
        if (!sym_pays(c, op)) continue;
        const size_t elems = sym_part_elems(c, op, 1), bytes = sizeof(double) * elems;
        size_t free_b = 0, total_b = 0;
        if (bytes > (size_t)64 << 20 && !looked_up) {
            looked_up = true;
            if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) free_b = 0;
            limit = std::min(limit, std::max((size_t)64 << 20, free_b / 64));
        }
        if (bytes <= limit) need = std::max(need, elems);
    }
    return need;
}

// Select the passes that pay and whose partial sums fit in the buffer.
cudaError_t sym_defaults(Ctx &c)
{
    auto takes = [&](int op) { return sym_pays(c, op) && sym_part_elems(c, op, 1) <= c.part_elems; };
    if (takes(OP_ENERGY)) TPE_CHECK(sym_select_energy(c, 1));
    if (takes(OP_DIFF)) TPE_CHECK(sym_select_diff(c, 1));
    if (takes(OP_APPLY)) TPE_CHECK(sym_select(c, 1));
    return cudaSuccess;
}

// Run the symmetric pass of `op` and sum its slots: energy rows into out [nE], else the edges' endpoint
// values into c.d_esum.
static cudaError_t sym_pass(Ctx &c, int op, Ctx::Plan &pl, int counter, int prof_op, int which, const int *skip, double *out,
                            cudaStream_t s)
{
    if (pl.n_items == 0) return cudaSuccess;  // no edges: nothing reads the sums
    // the buffer is shared with the other passes and may have been resized since the last call
    TPE_CHECK(part_reserve(c, plan_elems(c, pl, op)));
    SymArgs pa;
    pa.items = pl.d_items;
    pa.n_items = pl.n_items;
    pa.counter = c.d_counter + counter;
    pa.recF = which ? c.d_recF2 : c.d_recF;
    pa.recLo = which ? c.d_recLo2 : c.d_recLo;
    pa.urecF = op == OP_APPLY2 ? c.d_urecMF : c.d_urecF;
    pa.ell_lo = c.d_ell_lo[which];
    pa.part = reinterpret_cast<float2 *>(c.d_part);
    pa.nE = c.nE;
    pa.near2f = op == OP_DIFF ? c.kp.near2f_diff : c.kp.near2f;
    pa.mid2f = c.kp.mid2f;
    pa.sum_exp = c.kp.sum_exp;
    pa.sum_scale = c.kp.sum_scale;
    pa.skip = skip;
    const int slot = c.profile ? prof_begin(c, prof_op, s) : -1;
    with_sym_kernel(c.prm.precision, op, pl.tpt, [&](auto kern, size_t smem) { kern<<<pl.grid, kThreads, smem, s>>>(pa); });
    if (slot >= 0 || slot <= -2) prof_end(c, slot, s);
    const double *ell = c.d_ellw[which], *T = c.d_Tw[which], quarter = op == OP_DIFF ? 0.25 / c.kp.sum_scale : 0.25;
    if (op == OP_ENERGY)
        k_sym_sum<OP_ENERGY><<<(c.nE + 255) / 256, 256, 0, s>>>(c.nE, pl.d_eslots, pa.part, ell, T, quarter, out);
    else if (op == OP_DIFF)
        k_sym_sum<OP_DIFF><<<(c.nE + 31) / 32, 320, 0, s>>>(c.nE, pl.d_eslots, pa.part, ell, T, quarter, out);
    else if (op == OP_APPLY2)
        k_sym_sum<OP_APPLY2><<<(c.nE + 31) / 32, 384, 0, s>>>(c.nE, pl.d_eslots, pa.part, ell, T, quarter, out);
    else if (pl.tpt == kSymAccurate)
        k_sym_sum<OP_APPLY, true><<<(c.nE + 31) / 32, 192, 0, s>>>(c.nE, pl.d_eslots, pa.part, ell, T, quarter, out);
    else
        k_sym_sum<OP_APPLY><<<(c.nE + 31) / 32, 192, 0, s>>>(c.nE, pl.d_eslots, pa.part, ell, T, quarter, out);
    c.launches += 2;
    return cudaGetLastError();
}

cudaError_t sym_energy_pass(Ctx &c, int which, double *rows, cudaStream_t s)
{
    return sym_pass(c, OP_ENERGY, c.plan_sym_e, 5, OP_ENERGY, which, nullptr, rows, s);
}

cudaError_t sym_diff_pass(Ctx &c, int which, cudaStream_t s)
{
    return sym_pass(c, OP_DIFF, c.plan_sym_d, 6, OP_DIFF, which, nullptr, c.d_esum, s);
}

cudaError_t sym_apply_pass(Ctx &c, int which, cudaStream_t s)
{
    return sym_pass(c, OP_APPLY, c.plan_sym, 4, c.d_skip ? 4 : 2, which, c.d_skip, c.d_esum, s);
}

// Passes whose plan is built at the first call.
static cudaError_t lazy_plan(Ctx &c, int op, Ctx::Plan &pl, int variant)
{
    if (pl.d_items) return cudaSuccess;
    TPE_CHECK(sym_plan(c, pl, sym_occupancy(c, op, variant)));
    pl.tpt = variant;
    return cudaSuccess;
}

// The accurate apply: edges' endpoint values into c.d_esum.
cudaError_t sym_apply_accurate_pass(Ctx &c, int which, cudaStream_t s)
{
    TPE_CHECK(lazy_plan(c, OP_APPLY, c.plan_df, kSymAccurate));
    return sym_pass(c, OP_APPLY, c.plan_df, 7, 5, which, c.d_skip, c.d_esum, s);
}

bool sym_apply2_ready(Ctx &c)
{
    Ctx::Plan &pl = c.plan_sym2;
    const size_t need = pl.d_items ? plan_elems(c, pl, OP_APPLY2) : sym_part_elems(c, OP_APPLY2, 1);
    return part_fits(c, need) && lazy_plan(c, OP_APPLY2, pl, 1) == cudaSuccess && part_reserve(c, need) == cudaSuccess;
}

// Two vector fields, the weights once per pair.
cudaError_t sym_apply2_pass(Ctx &c, int which, cudaStream_t s)
{
    return sym_pass(c, OP_APPLY2, c.plan_sym2, 10, 7, which, nullptr, c.d_esum2, s);
}

}  // namespace tpe
