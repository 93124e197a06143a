// Lane arithmetic of the FP32 pair passes: the same pair formulas on one target (float) or on two targets
// of a thread at once (float2, the packed f32x2 instructions).
//
// An FFMA2 holds the FP32 pipe for two cycles, as two FFMA do, but takes one issue slot (measured: 0.49
// f32x2 instructions per clock and SM sub-partition against 0.95 scalar ones; a negated operand is
// free).  The scalar passes were bound by issue slots (MUFU, shared-memory and integer instructions
// compete with the FMAs), the packed ones by the FP32 pipe itself.
//
// Every operation is an explicitly rounded multiply, add or fma, so a pair's terms are bitwise the same
// on either lane type and from either of its two rows.
#pragma once

#include <cuda_runtime.h>

#include "tpe_internal.cuh"

namespace tpe {

__device__ __forceinline__ float l_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float l_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float l_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float l_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float l_neg(float a) { return -a; }

__device__ __forceinline__ float2 l_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 l_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 l_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 l_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 l_sub(float2 a, float2 b) { return __fadd2_rn(a, l_neg(b)); }

// rsqrt without the denormal fix-up of rsqrtf (about three instructions a call): a squared distance or its
// inverse root that is subnormal leaves |d|^-2.5 and |d|^-4.5 infinite either way.
__device__ __forceinline__ float l_rsqrt(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float2 l_rsqrt(float2 x) { return make_float2(l_rsqrt(x.x), l_rsqrt(x.y)); }

template <class L>
__device__ __forceinline__ L l_bc(float s);
template <>
__device__ __forceinline__ float l_bc<float>(float s)
{
    return s;
}
template <>
__device__ __forceinline__ float2 l_bc<float2>(float s)
{
    return make_float2(s, s);
}

__device__ __forceinline__ float l_keep(bool k, float a) { return k ? a : 0.f; }
__device__ __forceinline__ float2 l_keep(bool k0, bool k1, float2 a) { return make_float2(k0 ? a.x : 0.f, k1 ? a.y : 0.f); }

template <class L>
struct LV {
    L x, y, z;
};

template <class L>
__device__ __forceinline__ LV<L> l_bc3(float x, float y, float z)
{
    return {l_bc<L>(x), l_bc<L>(y), l_bc<L>(z)};
}

template <class L>
__device__ __forceinline__ LV<L> l_sub3(const LV<L> &a, const LV<L> &b)
{
    return {l_sub(a.x, b.x), l_sub(a.y, b.y), l_sub(a.z, b.z)};
}
template <class L>
__device__ __forceinline__ LV<L> l_add3(const LV<L> &a, const LV<L> &b)
{
    return {l_add(a.x, b.x), l_add(a.y, b.y), l_add(a.z, b.z)};
}
template <class L>
__device__ __forceinline__ L l_dot(const LV<L> &a, const LV<L> &b)
{
    return l_fma(a.z, b.z, l_fma(a.y, b.y, l_mul(a.x, b.x)));
}

// The four chords d_ab = g_ia - g_jb (index 2 (a - 1) + (b - 1)) from d11 and the two edge vectors: d12 = d11 -
// e_J, d21 = d11 + e_I, d22 = d11 + (e_I - e_J).  From row J each is bitwise the negated chord of row I.
// DF: double-float positions (hi difference plus lo difference).
template <bool DF, class L>
__device__ __forceinline__ void l_chords(const LV<L> &p, const LV<L> &pl, const LV<L> &eI, const LV<L> &q,
                                         const LV<L> &ql, const LV<L> &eJ, LV<L> (&d)[4])
{
    d[0] = l_sub3(p, q);
    if constexpr (DF) d[0] = l_add3(d[0], l_sub3(pl, ql));
    d[1] = l_sub3(d[0], eJ);
    d[2] = l_add3(d[0], eI);
    d[3] = l_add3(d[0], l_sub3(eI, eJ));
}

// |d - (T.d) T|^2 = |T x d|^2
template <class L>
__device__ __forceinline__ L l_perp2(const LV<L> &d, const LV<L> &T)
{
    const L t = l_neg(l_dot(T, d));
    const LV<L> dp = {l_fma(t, T.x, d.x), l_fma(t, T.y, d.y), l_fma(t, T.z, d.z)};
    return l_dot(dp, dp);
}

// The same with the double-float tangent T + Tl; also t = T.d and dp = d - t T.
template <class L>
__device__ __forceinline__ L l_perp2_df(const LV<L> &d, const LV<L> &T, const LV<L> &Tl, L &t, LV<L> &dp)
{
    t = l_fma(T.x, d.x, l_fma(T.y, d.y, l_fma(T.z, d.z, l_dot(Tl, d))));
    const L nt = l_neg(t);
    dp = {l_fma(nt, T.x, l_fma(nt, Tl.x, d.x)), l_fma(nt, T.y, l_fma(nt, Tl.y, d.y)),
          l_fma(nt, T.z, l_fma(nt, Tl.z, d.z))};
    return l_dot(dp, dp);
}

// |d|^-4.5 from |d|^2; r2 = |d|^-2
template <class L>
__device__ __forceinline__ L l_pow45(L d2, L &r2)
{
    const L r = l_rsqrt(d2);
    const L sr = l_mul(r, l_rsqrt(r));
    r2 = l_mul(r, r);
    return l_mul(l_mul(r2, r2), sr);
}

// |d|^-2.5; g = |d|^-6.5
template <class L>
__device__ __forceinline__ L l_pow25(L d2, L &g)
{
    const L r = l_rsqrt(d2);
    const L sr = l_mul(r, l_rsqrt(r));
    const L r2 = l_mul(r, r);
    const L f = l_mul(r2, sr);
    g = l_mul(f, l_mul(r2, r2));
    return f;
}

// Kahan-compensated acc += a * b (c: the lost low-order part, to be subtracted).
template <class L>
__device__ __forceinline__ void l_kahan_fma(L &acc, L &c, L a, L b)
{
    const L y = l_fma(a, b, l_neg(c));
    const L t = l_add(acc, y);
    c = l_sub(l_sub(t, acc), y);
    acc = t;
}

// The same for the energy, whose terms are positive and overflow below 2.7e-9: an infinite sum stays infinite.  Its
// compensation would be inf - inf, and the sum NaN with the next term; the smaller of NaN and a number is the number.
__device__ __forceinline__ float l_at_most_max(float a) { return fminf(a, 3.40282347e38f); }
__device__ __forceinline__ float2 l_at_most_max(float2 a) { return make_float2(l_at_most_max(a.x), l_at_most_max(a.y)); }
template <class L>
__device__ __forceinline__ void l_kahan_fma_pos(L &acc, L &c, L a, L b)
{
    l_kahan_fma(acc, c, a, b);
    c = l_at_most_max(c);
}

// The energy's four-term sums of row I (and of row J): f = sum_ab |T x d_ab|^2 |d_ab|^-4.5 from the two
// |T x d|^2 that the row needs (they depend on the other edge's endpoint only), each row in its own order
// of the endpoints.
template <class L>
__device__ __forceinline__ L l_energy_sum(L c0, L c1, L r11, L r12, L r21, L r22)
{
    return l_fma(c1, r22, l_fma(c0, r21, l_fma(c1, r12, l_mul(c0, r11))));
}

// ---------------------------------------------------------------------------------- near pairs
//
// Pairs close along the curve have nearly parallel chord and tangent, so |T x d|^2 and the differential's
// terms (which cancel between a vertex's two edges) need more than FP32.  They are evaluated in
// double-float arithmetic on the FP32 pipe (about 2^-44): an FP64 instruction of a warp holds its
// sub-partition's FP64 pipe for 64 cycles, and one near pair of the differential takes ~500 of them
// (33,000 cycles) against ~2,000 FP32 instructions here.  The pairs are renormalised only where a difference
// cancels (elsewhere lo stays within a few ulp of hi, its own rounding at 2^-47).  The functions load the records themselves
// and are not inlined.  The instruction cache bounds the differential's: unrolled over both endpoints, 48 KB of
// straight-line code took 23,000 cycles a call, and unrolled over one (22 KB) it still left the warps waiting for
// instructions 30% of the time.  It is rolled over both endpoints (13 KB) and takes one pair a lane: packed
// pairs do the same work of the FP32 pipe in half the instructions, but two rounds of the short code hit in
// the cache (differential of 96 x 500 edges: packed, one endpoint unrolled 1,052 us, packed, rolled 1,060, single,
// one unrolled 975, single, rolled 827; 841 with exact chord differences and the scaled power).

template <class L>
struct dfl {
    L hi, lo;
};

template <class L>
__device__ __forceinline__ dfl<L> l_two_sum(L a, L b)
{
    const L s = l_add(a, b), bb = l_sub(s, a);
    return {s, l_add(l_sub(a, l_sub(s, bb)), l_sub(b, bb))};
}
template <class L>
__device__ __forceinline__ dfl<L> l_dfneg(dfl<L> x) { return {l_neg(x.hi), l_neg(x.lo)}; }
// hi and lo of x with |lo| <= ulp(hi) / 2: needed after a difference that cancels, where lo would be left as large
// as hi (products drop lo lo)
template <class L>
__device__ __forceinline__ dfl<L> l_dfnorm(dfl<L> x)
{
    const L s = l_add(x.hi, x.lo);
    return {s, l_sub(x.lo, l_sub(s, x.hi))};
}
// error 2^-47 (|x| + |y|)
template <class L>
__device__ __forceinline__ dfl<L> l_dfadd(dfl<L> x, dfl<L> y)
{
    const dfl<L> s = l_two_sum(x.hi, y.hi);
    return {s.hi, l_add(s.lo, l_add(x.lo, y.lo))};
}
template <class L>
__device__ __forceinline__ dfl<L> l_dfmul(dfl<L> x, dfl<L> y)
{
    const L p = l_mul(x.hi, y.hi);
    return {p, l_fma(x.lo, y.hi, l_fma(x.hi, y.lo, l_fma(x.hi, y.hi, l_neg(p))))};
}
template <class L>
__device__ __forceinline__ dfl<L> l_dfmulf(dfl<L> x, L f)
{
    const L p = l_mul(x.hi, f);
    return {p, l_fma(x.lo, f, l_fma(x.hi, f, l_neg(p)))};
}
template <class L>
__device__ __forceinline__ dfl<L> l_dfsqr(dfl<L> x)
{
    const L p = l_mul(x.hi, x.hi);
    return {p, l_fma(l_add(x.hi, x.hi), x.lo, l_fma(x.hi, x.hi, l_neg(p)))};
}
// x (1 + f) for a small f
template <class L>
__device__ __forceinline__ dfl<L> l_dfscale(dfl<L> x, L f) { return {x.hi, l_fma(x.hi, f, x.lo)}; }

template <class L>
struct dfv {
    dfl<L> x, y, z;
};
template <class L>
__device__ __forceinline__ dfl<L> l_dfdot(const dfv<L> &a, const dfv<L> &b)
{
    return l_dfadd(l_dfadd(l_dfmul(a.x, b.x), l_dfmul(a.y, b.y)), l_dfmul(a.z, b.z));
}
template <class L>
__device__ __forceinline__ dfl<L> l_dfnorm2(const dfv<L> &a)
{
    return l_dfadd(l_dfadd(l_dfsqr(a.x), l_dfsqr(a.y)), l_dfsqr(a.z));
}
// d - t T
template <class L>
__device__ __forceinline__ dfv<L> l_dfperp(const dfv<L> &d, dfl<L> t, const dfv<L> &T)
{
    const dfl<L> n = l_dfneg(t);
    return {l_dfnorm(l_dfadd(d.x, l_dfmul(n, T.x))), l_dfnorm(l_dfadd(d.y, l_dfmul(n, T.y))),
            l_dfnorm(l_dfadd(d.z, l_dfmul(n, T.z)))};
}

// The edges of a lane as the near paths see them: endpoints (hi, lo), tangent (hi, lo), length.
template <class L>
struct NearEdge {
    L p[2][3], l[2][3], T[3], Tl[3], ell;
};

__device__ __forceinline__ float near_2(float a, float, float) { return a; }
__device__ __forceinline__ float2 near_2(float a, float b, float2) { return make_float2(a, b); }

// I0 (and on the second lane I1)
template <class L>
__device__ __forceinline__ void near_load(NearEdge<L> &e, const RecF *recF, const RecLo *recLo, int I0, int I1)
{
    const RecF r = recF[I0], s = recF[I1];
    const RecLo q = recLo[I0], v = recLo[I1];
#define TPE_2(A, B, f) near_2(A.f, B.f, L())
    e.p[0][0] = TPE_2(r, s, a.x), e.p[0][1] = TPE_2(r, s, a.y), e.p[0][2] = TPE_2(r, s, a.z);
    e.p[1][0] = TPE_2(r, s, b.x), e.p[1][1] = TPE_2(r, s, b.y), e.p[1][2] = TPE_2(r, s, b.z);
    e.T[0] = TPE_2(r, s, b.w), e.T[1] = TPE_2(r, s, c.x), e.T[2] = TPE_2(r, s, c.y);
    e.l[0][0] = TPE_2(q, v, lo.x), e.l[0][1] = TPE_2(q, v, lo.y), e.l[0][2] = TPE_2(q, v, lo.z);
    e.l[1][0] = TPE_2(q, v, lo.w), e.l[1][1] = TPE_2(q, v, lo2.x), e.l[1][2] = TPE_2(q, v, lo2.y);
    e.Tl[0] = TPE_2(q, v, lo2.z), e.Tl[1] = TPE_2(q, v, lo2.w), e.Tl[2] = TPE_2(q, v, lo3.x);
    e.ell = TPE_2(r, s, a.w);
#undef TPE_2
}

template <class L>
__device__ __forceinline__ dfv<L> near_tangent(const NearEdge<L> &e)
{
    return {{e.T[0], e.Tl[0]}, {e.T[1], e.Tl[1]}, {e.T[2], e.Tl[2]}};
}
// p - q of double-float coordinates.  The difference of the high parts rounds wherever they differ by more than a factor
// of two (strands on either side of an axis plane), and 2^-25 of the chord is 2^-15 and more of |T x d|: rounded, it
// was the largest error of the differential (4,096 edges: 4.0e-7 of its norm rounded, 1.5e-7 exact).
template <class L>
__device__ __forceinline__ dfl<L> near_diff1(L p, L pl, L q, L ql)
{
    const dfl<L> s = l_two_sum(p, l_neg(q));
    return l_dfnorm(dfl<L>{s.hi, l_add(s.lo, l_sub(pl, ql))});
}
template <class L>
__device__ __forceinline__ dfv<L> near_chord(const NearEdge<L> &I, int a, const NearEdge<L> &J, int b)
{
    return {near_diff1(I.p[a][0], I.l[a][0], J.p[b][0], J.l[b][0]),
            near_diff1(I.p[a][1], I.l[a][1], J.p[b][1], J.l[b][1]),
            near_diff1(I.p[a][2], I.l[a][2], J.p[b][2], J.l[b][2])};
}

// the same with the endpoints chosen in a rolled loop
template <class L>
__device__ __forceinline__ dfv<L> near_chord_k(const NearEdge<L> &I, const NearEdge<L> &J, int a, int b)
{
#define TPE_C(q)                                                   \
    near_diff1(a ? I.p[1][q] : I.p[0][q], a ? I.l[1][q] : I.l[0][q], \
               b ? J.p[1][q] : J.p[0][q], b ? J.l[1][q] : J.l[0][q])
    return {TPE_C(0), TPE_C(1), TPE_C(2)};
#undef TPE_C
}

// |T x d|^2 of a near pair, rounded to FP32
template <class L>
__device__ __forceinline__ L near_perp2(const dfv<L> &d, const dfv<L> &T)
{
    const dfv<L> p = l_dfperp(d, l_dfdot(T, d), T);
    return l_fma(p.z.hi, p.z.hi, l_fma(p.y.hi, p.y.hi, l_mul(p.x.hi, p.x.hi)));
}

// c[0], c[1] = |T_I x d_1b|^2 and, with BOTH, c[2], c[3] = |T_J x d_a1|^2 of a near pair (rows I0, I1 against J)
template <class L, bool BOTH>
static __device__ __noinline__ void near_energy(const RecF *recF, const RecLo *recLo, int I0, int I1, int J0, L (&c)[4])
{
    NearEdge<L> I, J;
    near_load(I, recF, recLo, I0, I1);
    near_load(J, recF, recLo, J0, J0);
    const dfv<L> TI = near_tangent(I), TJ = near_tangent(J);
    const dfv<L> d11 = near_chord(I, 0, J, 0);
    c[0] = near_perp2(d11, TI);
    c[1] = near_perp2(near_chord(I, 0, J, 1), TI);
    if constexpr (BOTH) {
        c[2] = near_perp2(d11, TJ);
        c[3] = near_perp2(near_chord(I, 1, J, 0), TJ);
    }
}

// 2^e, as far as a normal float goes
__device__ __forceinline__ float near_pow2(int e) { return __int_as_float(min(max(e + 127, 1), 254) << 23); }

// |d|^-4.5 2^sum_exp and |d|^-2 in double-float: r0 = rsqrt(d2.hi) with its residual rho = 1 - d2 r0^2 formed through
// fma gives |d|^-1 = r0 (1 + eps), and q0 ~ sqrt(r0) from rsqrt(r0) is corrected by (r0 - q0^2) / (2 q0).
//
// FP32 exponents hold |d|^-4.5 from 2.7e-9 up only, and the low parts of its double-float up to about 1e7.  So the power
// is formed at 4^m times the chord's length, between 1 and 4 (a power of four leaves |d|^-4.5 a power of two, so the
// scaling is exact), and the differential's sums are kept at 2^sum_exp of their value: 2^-56 for the gradient of a pair
// one mean edge apart, so that they hold pairs down to 1e-12 of an edge, about the resolution of double-float positions.
__device__ __forceinline__ dfl<float> near_pow45(dfl<float> d2, int sum_exp, dfl<float> &R2)
{
    using L = float;
    const int m = -((__float_as_int(d2.hi) - (127 << 23)) >> 25);
    const float up = near_pow2(4 * m), back = near_pow2(9 * m + sum_exp);
    d2 = {l_mul(d2.hi, up), l_mul(d2.lo, up)};
    const L r0 = l_rsqrt(d2.hi);
    const L a = l_mul(r0, r0), b = l_fma(r0, r0, l_neg(a));
    L rho = l_fma(l_neg(d2.hi), a, l_bc<L>(1.f));
    rho = l_fma(l_neg(d2.hi), b, rho);
    rho = l_fma(l_neg(d2.lo), a, rho);
    const L eps = l_mul(rho, l_fma(l_bc<L>(0.375f), rho, l_bc<L>(0.5f)));
    const L iq = l_rsqrt(r0), q0 = l_mul(r0, iq);
    const L dq = l_mul(l_fma(l_neg(q0), q0, r0), l_mul(l_bc<L>(0.5f), iq));
    const dfl<L> R = {a, b};  // r0^2
    R2 = l_dfscale(R, l_mul(eps, l_add(l_bc<L>(2.f), eps)));
    R2 = {l_mul(R2.hi, up), l_mul(R2.lo, up)};
    dfl<L> F = l_dfmul(l_dfsqr(R), dfl<L>{q0, dq});  // r0^4.5
    F = l_dfscale(F, l_mul(eps, l_fma(l_bc<L>(7.875f), eps, l_bc<L>(4.5f))));
    return {l_mul(F.hi, back), l_mul(F.lo, back)};
}

// The differential's terms of one near pair, scaled by the other row's length and 2^sum_exp: row I's (S, G1, G2, GT)
// into x and row J's (S, H1, H2, HT) into y, see pairs_sym.cu.
static __device__ __noinline__ void near_diff(const RecF *recF, const RecLo *recLo, int I0, int J0, int sum_exp,
                                              dfl<float> (&x)[10], dfl<float> (&y)[10])
{
    using L = float;
    NearEdge<L> I, J;
    near_load(I, recF, recLo, I0, I0);
    near_load(J, recF, recLo, J0, J0);
    const dfl<L> zero = {0.f, 0.f};
    const dfv<L> TI = near_tangent(I), TJ = near_tangent(J);
    // |T_I x d_ab| and its perpendicular depend on b only, |T_J x d_ab| and its on a only
    dfv<L> pI[2] = {}, pJ[2] = {};
    dfl<L> cI[2] = {}, cJ[2] = {};
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
        const dfv<L> dI = near_chord_k(I, J, 0, k), dJ = near_chord_k(I, J, k, 0);
        pI[0] = pI[1];
        pJ[0] = pJ[1];
        cI[0] = cI[1];
        cJ[0] = cJ[1];
        pI[1] = l_dfperp(dI, l_dfdot(TI, dI), TI);
        pJ[1] = l_dfperp(dJ, l_dfdot(TJ, dJ), TJ);
        cI[1] = l_dfnorm2(pI[1]);
        cJ[1] = l_dfnorm2(pJ[1]);
    }
    dfl<L> S = zero, H[2][3], GT[3] = {zero, zero, zero}, HT[3] = {zero, zero, zero};
#pragma unroll
    for (int k = 0; k < 3; ++k) H[0][k] = H[1][k] = x[4 + k] = zero;
#pragma unroll 1
    for (int a = 0; a < 2; ++a) {
        dfl<L> G[3] = {zero, zero, zero};
#pragma unroll 1
        for (int b = 0; b < 2; ++b) {
            const dfv<L> d = near_chord(I, 0, J, 0);
            dfl<L> r2;
            const dfl<L> rb = near_pow45(l_dfnorm2(d), sum_exp, r2);
            const dfl<L> fs = l_dfmul(l_dfadd(cI[0], cJ[0]), rb);
            const dfl<L> al = {l_add(rb.hi, rb.hi), l_add(rb.lo, rb.lo)};  // alpha |d|^-beta
            const dfl<L> cb = l_dfneg(l_dfmul(l_dfmulf(fs, 4.5f), r2));
            const dfl<L> mI = l_dfneg(l_dfmul(al, l_dfdot(TI, d))), mJ = l_dfneg(l_dfmul(al, l_dfdot(TJ, d)));
            const dfl<L> dk[3] = {d.x, d.y, d.z}, pi[3] = {pI[0].x, pI[0].y, pI[0].z}, pj[3] = {pJ[0].x, pJ[0].y, pJ[0].z};
            S = l_dfadd(S, fs);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const dfl<L> v = l_dfadd(l_dfmul(al, l_dfadd(pi[k], pj[k])), l_dfmul(cb, dk[k]));
                G[k] = l_dfadd(G[k], v);
                const dfl<L> h = l_dfadd(H[0][k], l_dfneg(v));
                GT[k] = l_dfadd(GT[k], l_dfmul(mI, dk[k]));
                HT[k] = l_dfadd(HT[k], l_dfmul(mJ, dk[k]));
                // the other endpoint of J next
                H[0][k] = H[1][k];
                H[1][k] = h;
                const L q = J.p[0][k], ql = J.l[0][k];
                J.p[0][k] = J.p[1][k];
                J.p[1][k] = q;
                J.l[0][k] = J.l[1][k];
                J.l[1][k] = ql;
            }
            const dfv<L> pt = pI[0];
            const dfl<L> ct = cI[0];
            pI[0] = pI[1];
            pI[1] = pt;
            cI[0] = cI[1];
            cI[1] = ct;
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const dfl<L> xo = l_dfmulf(G[k], J.ell);
            x[1 + k] = x[4 + k];
            x[4 + k] = xo;
            // the second endpoint of I for the next round
            I.p[0][k] = I.p[1][k];
            I.l[0][k] = I.l[1][k];
        }
        pJ[0] = pJ[1];
        cJ[0] = cJ[1];
    }
    x[0] = l_dfmulf(S, J.ell);
    y[0] = l_dfmulf(S, I.ell);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        x[7 + k] = l_dfmulf(GT[k], J.ell);
        y[1 + k] = l_dfmulf(H[0][k], I.ell);
        y[4 + k] = l_dfmulf(H[1][k], I.ell);
        y[7 + k] = l_dfmulf(HT[k], I.ell);
    }
}

// (acc, c) += x for a compensated sum acc - c and a double-float x of any size
template <class L>
__device__ __forceinline__ void l_kahan_df(L &acc, L &c, L hi, L lo)
{
    const dfl<L> s = l_two_sum(acc, hi);
    acc = s.hi;
    c = l_sub(c, l_add(s.lo, lo));
}

}  // namespace tpe
