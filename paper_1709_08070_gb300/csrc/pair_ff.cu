// Float-float ("double-single") pair sums of the IBIM operator (Sec. 2.2
// discrete system, Sec. 2.2.1 regularisation) on the FP32 pipe, sm_103a.
//
// Purpose: an operator as accurate as the plain FP64 path (it is held to the
// same 1e-10 element bar against the FP64 oracle) that runs on the GB300's
// FP32 pipe instead of its FP64 pipe, which has a small fraction of the FP32
// rate.  The certification of an FP32 solve (one residual g - A p with an
// FP64-accurate operator) uses it.
//
// Every quantity is an unevaluated sum h + l of two floats (about 48
// significant bits), built from error-free transformations: Knuth's two-sum
// (s + e == a + b exactly) and the FMA two-product (p + e == a b exactly);
// products drop the l l' term (relative 2^-48) and sums renormalise with
// Dekker's fast two-sum where the result is accumulated.
//
//   * Positions.  Node coordinates relative to the molecule centroid are
//     split as x = xh + xl with xh on a power-of-two grid 2^-q fine enough
//     that |x| 2^q < 2^23; the difference of two hi parts is then exact, and
//     r = (xh - yh) + (xl - yl) carries about 2^-41 of the box size.
//   * 1/rho: the MUFU estimate y0 of rsqrt(|r|^2) refined by one Newton step
//     in float-float, y0 (1 - d/2 + 3 d^2/8) with 1 + d = |r|^2 y0^2.
//   * E = exp(-kappa rho): Tang's table-driven method (ACM TOMS 15, 1989):
//     z = -kappa rho log2(e) = k/256 + f with |f| <= 1/512, 2^(k/256) from a
//     256-entry float-float table (2^(i/256), i = 0..255, computed with FP64
//     exp2 on the device), e^(f ln 2) from its Taylor series (the terms past
//     the linear one in FP32), and the power 2^floor(k/256) put into the
//     exponent bits.  z is clamped at -120 (E < 1e-36 there).
//   * Kernels (times 4 pi), with g = 1 - A = (1 - E) - E x, 3 - B = 3 g - E x^2:
//       y1 += s_y (1 - th1 A) a / rho^3 - (1 - E) b / rho
//       y2 += [(g c - (3 - B) s_x s_y / rho^2) a + s_x (1 - th2 A) b] / rho^3
//     and inside the tube (near chunks only) y1 -= K12_tube b.
//   * Tube test (Sec. 2.2.1) in float-float; a pair within 1e-9 (relative)
//     of a threshold is decided again in FP64 with the oracle's operation
//     order, so ties fall as they do in FP64.
//   * Sums: float-float per target over a source tile (renormalised per
//     pair), FP64 across tiles, FP64 partials per (CTA, target tile) summed by
//     the FP32 path's fixup kernel in a fixed order.
//
// Schedule: the one-directional stream-K walk of pair_f32.cu (persistent
// CTAs, source tiles in the golden-ratio order of each row), one target per
// thread, 256-source tiles through two shared-memory stages filled by bulk
// async copies; chunk pairs whose bounding spheres are at least the far
// distance apart skip the tube test, as in the FP32 kernel.
#include "pair_sym_core.cuh"

namespace ibim {

constexpr int kFFThreads = 256;  // one target per thread
constexpr int kFFTTile = kFFThreads;
constexpr int kFFSTile = 256;    // sources per stage
constexpr int kFFStages = 2;
constexpr int kFFChunk = 32;
constexpr int kFFChunksPerTile = kFFSTile / kFFChunk;
constexpr int kFFTab = 256;      // table of 2^(i/256)
constexpr uint64_t kFFWaitNs = 2000000000ull;  // 2 s
static_assert(kPadNodes % kFFSTile == 0 && kPadNodes % kFFTTile == 0, "padding");
// Payload: the nodes p and p + 16 of an aligned 32-node chunk form a pair whose
// values lie side by side, as the packed FP32 instructions take them.  A pair
// has eight float4:
//   0 (xh0 xh0' xh1 xh1')  1 (xh2 xh2' ah ah')  2, 3 the same of xl, al
//   4 (nh0 nh0' nh1 nh1')  5 (nh2 nh2' bh bh')  6, 7 the same of nl, bl
// stored per chunk component by component (the chunk's 16 first float4, then
// its 16 second ones, ...), so that 16 lanes reading the 16 pairs of a chunk
// touch 256 contiguous bytes.
constexpr int kFFNodeF4 = 4;
constexpr int kFFPairs = kFFChunk / 2;
// Float offset of value c of field f of node j: fields (xh, ah), (xl, al), (nh,
// bh), (nl, bl), values 0..2 the components and 3 the scalar.
__host__ __device__ __forceinline__ int64_t ff_off(int64_t j, int f, int c)
{
    const int64_t f4 = (j >> 5) * (32 * kFFNodeF4) + (2 * f + (c >> 1)) * kFFPairs + (j & (kFFPairs - 1));
    return 4 * f4 + 2 * (c & 1) + ((j >> 4) & 1);
}
constexpr uint32_t kFFStageBytes = kFFSTile * kFFNodeF4 * sizeof(float4);
constexpr uint32_t kFFFrameBytes = 2 * kFFChunksPerTile * sizeof(float4);
constexpr float kFFPad = 1.0e4f;  // placeholder coordinate (sources +, targets -)

// ------------------------------------------------------ float-float arithmetic

// Two pairs of nodes per lane in the packed FP32 instructions (add, mul and fma
// of two values; negating an operand costs nothing, measured).  One pair per
// lane took 444 instructions a pair and stood at 0.84 of the issue slots and 0.75
// of the FMA pipe; packed it is 252 (209 of them FMA-pipe instructions of two
// cycles each), so the FMA pipe bounds it (39,406 nodes 10.9 -> 9.8 ms with the
// finer segments below).
__device__ __forceinline__ float2 vneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return __fadd2_rn(a, vneg(b)); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 vset(float a) { return make_float2(a, a); }

struct ff {
    float h, l;
};
struct ff2 {
    float2 h, l;
};

// Constant (h, h, l, l): one 64-bit operand each.
__device__ __forceinline__ ff2 ff_of(const float4& v) { return ff2{make_float2(v.x, v.y), make_float2(v.z, v.w)}; }

__device__ __forceinline__ ff2 ff_wide(ff v) { return ff2{vset(v.h), vset(v.l)}; }
__device__ __forceinline__ ff ff_half(ff2 v, int q) { return q ? ff{v.h.y, v.l.y} : ff{v.h.x, v.l.x}; }

// Knuth's two-sum: s + e == a + b exactly.
__device__ __forceinline__ ff2 two_sum(float2 a, float2 b)
{
    const float2 s = vadd(a, b);
    const float2 bb = vsub(s, a);
    const float2 e = vadd(vsub(a, vsub(s, bb)), vsub(b, bb));
    return ff2{s, e};
}

// Dekker's fast two-sum (exact when |a| >= |b|, or a == 0).
__device__ __forceinline__ ff2 fast_two_sum(float2 a, float2 b)
{
    const float2 s = vadd(a, b);
    return ff2{s, vsub(b, vsub(s, a))};
}

__device__ __forceinline__ ff2 ff_norm(ff2 a) { return fast_two_sum(a.h, a.l); }

// a b with the l l' term dropped (result nearly normalised).
__device__ __forceinline__ ff2 ff_mul(ff2 a, ff2 b)
{
    const float2 p = vmul(a.h, b.h);
    float2 e = vfma(a.h, b.h, vneg(p));
    e = vfma(a.h, b.l, e);
    e = vfma(a.l, b.h, e);
    return ff2{p, e};
}

// a b for a plain number b.
__device__ __forceinline__ ff2 ff_mulf(ff2 a, float2 b)
{
    const float2 p = vmul(a.h, b);
    float2 e = vfma(a.h, b, vneg(p));
    e = vfma(a.l, b, e);
    return ff2{p, e};
}

__device__ __forceinline__ ff2 ff_neg(ff2 a) { return ff2{vneg(a.h), vneg(a.l)}; }

// a + b without the final renormalisation: l may reach a few ulps of max(|a.h|,
// |b.h|), which the products and sums that take it keep (they drop only l l').
// A sum whose parts cancel, or that meets another unnormalised factor, is
// normalised (s_x, s_y, |r|^2, 1/rho, rho, E, g and the running sums: without
// these the error against FP64 grows, up to thirtyfold where g takes an
// unnormalised E).  Against normalising every sum but not E and 1/rho: 432 -> 408
// operations a pair, and the error against FP64 falls by a fifth to a half with
// screening (20,000 nodes, kappa 0.1257: 5.6e-13 -> 4.5e-13) and stays without.
__device__ __forceinline__ ff2 ff_add_u(ff2 a, ff2 b)
{
    const ff2 s = two_sum(a.h, b.h);
    return ff2{s.h, vadd(s.l, vadd(a.l, b.l))};
}

// a + b, renormalised (absolute error about 2^-47 max(|a|, |b|)).
__device__ __forceinline__ ff2 ff_add(ff2 a, ff2 b) { return ff_norm(ff_add_u(a, b)); }

__device__ __forceinline__ ff2 ff_sub(ff2 a, ff2 b) { return ff_add(a, ff_neg(b)); }

// a b + c d without the final renormalisation.
__device__ __forceinline__ ff2 ff_dot2_u(ff2 a, ff2 b, ff2 c, ff2 d)
{
    return ff_add_u(ff_mul(a, b), ff_mul(c, d));
}

// a0 b0 + a1 b1 + a2 b2 (the l l' terms dropped; not renormalised).
__device__ __forceinline__ ff2 ff_dot3(const ff2 (&a)[3], const ff2 (&b)[3])
{
    const ff2 p0 = ff_mul(a[0], b[0]);
    const ff2 p1 = ff_mul(a[1], b[1]);
    const ff2 p2 = ff_mul(a[2], b[2]);
    const ff2 s = two_sum(p0.h, p1.h);
    const ff2 t = two_sum(s.h, p2.h);
    return ff2{t.h, vadd(vadd(s.l, t.l), vadd(vadd(p0.l, p1.l), p2.l))};
}

// (h + l)^2 summed over three components (not renormalised).
__device__ __forceinline__ ff2 ff_norm2(const ff2 (&r)[3])
{
    float2 p[3], e[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        // (h + l)^2 - h h rounded = fma error of h h + (2 h + l) l
        p[q] = vmul(r[q].h, r[q].h);
        e[q] = vfma(vfma(vset(2.0f), r[q].h, r[q].l), r[q].l, vfma(r[q].h, r[q].h, vneg(p[q])));
    }
    const ff2 s = two_sum(p[0], p[1]);
    const ff2 t = two_sum(s.h, p[2]);
    return ff2{t.h, vadd(vadd(s.l, t.l), vadd(vadd(e[0], e[1]), e[2]))};
}

__device__ __forceinline__ float2 vrsqrt(float2 a)
{
    return make_float2(ptx::rsqrt_approx(a.x), ptx::rsqrt_approx(a.y));
}
__device__ __forceinline__ float2 vmax(float2 a, float b) { return make_float2(fmaxf(a.x, b), fmaxf(a.y, b)); }

// Table entry 2^((ki mod 256)/256) and the power 2^floor(ki/256) of ki, the
// integer in the low mantissa bits of t (ki >= -30720).
__device__ __forceinline__ void ff_exp2_parts(float t, const float2* __restrict__ tab, float& Th, float& Tl, float& sc)
{
    const int ki = __float_as_int(t) - 0x4B400000;
    const float2 T = tab[ki & (kFFTab - 1)];
    Th = T.x;
    Tl = T.y;
    sc = __int_as_float(((ki >> 8) + 127) << 23);
}
__device__ __forceinline__ void ff_exp2_parts(float2 t, const float2* __restrict__ tab, float2& Th, float2& Tl,
                                              float2& sc)
{
    ff_exp2_parts(t.x, tab, Th.x, Tl.x, sc.x);
    ff_exp2_parts(t.y, tab, Th.y, Tl.y, sc.y);
}

// 2^z for z <= 0 (float-float), Tang's table-driven reduction; tab[i] = 2^(i/256).
// Normalised: the polynomial leaves a low part of 2^-20, which a product with
// another low part must not drop.
__device__ __forceinline__ ff2 ff_exp2(ff2 z, const float2* __restrict__ tab)
{
    const float2 zh = vmax(z.h, -120.0f);
    // round(zh 256) sits in the low mantissa bits of zh 256 + 1.5 2^23
    const float2 t = vfma(zh, vset(256.0f), vset(12582912.0f));
    const float2 kf = vsub(t, vset(12582912.0f));
    const float2 fh = vfma(kf, vset(-0.00390625f), zh);  // zh - k/256, exact, |fh| <= 1/512
    // u = (fh + zl) ln 2, |u| <= 0.00136
    const float2 L2h = vset(0.693147182464599609375f), L2l = vset(-1.904654323148236e-09f);
    const float2 uh = vmul(fh, L2h);
    float2 ul = vfma(fh, L2h, vneg(uh));
    ul = vfma(fh, L2l, ul);
    ul = vfma(z.l, L2h, ul);
    // e^u = 1 + u + u^2 (1/2 + u/6 + u^2/24) + O(u^5)
    float2 q = vfma(uh, vset(1.0f / 24.0f), vset(1.0f / 6.0f));
    q = vfma(uh, q, vset(0.5f));
    const float2 P = vmul(vmul(uh, uh), q);
    const float2 s = vadd(vset(1.0f), uh);
    const float2 el = vsub(uh, vsub(s, vset(1.0f)));
    const float2 lo = vadd(el, vadd(ul, P));
    float2 Th, Tl, sc;
    ff_exp2_parts(t, tab, Th, Tl, sc);
    const ff2 m = ff_mul(ff2{Th, Tl}, ff2{s, lo});
    return ff_norm(ff2{vmul(m.h, sc), vmul(m.l, sc)});
}

// ---------------------------------------------------------------- constants

struct FFConsts {
    float4 kap, cz;          // kappa and -kappa log2(e)   (h, h, l, l)
    float4 th1, th2;         // eps_E/eps_I, eps_I/eps_E
    float4 om1, om2;         // 1 - th1, 1 - th2
    float4 nk12t;            // -(4 pi x tube value of K12)
    float2 tau2, four_tau2;  // tube thresholds
    double tau2_d, four_tau2_d;
    float far_dist;          // minimum bounding-sphere gap of a far chunk pair (A)
    int rule0;
};

static float2 split(double v)
{
    const float h = (float)v;
    return make_float2(h, (float)(v - (double)h));
}

static float4 split2(double v)
{
    const float2 s = split(v);
    return make_float4(s.x, s.x, s.y, s.y);
}

static FFConsts ff_consts(const PairConsts& k)
{
    FFConsts c;
    c.kap = split2(k.kappa);
    c.cz = split2(-k.kappa * 1.4426950408889634074);
    c.th1 = split2(k.th1);
    c.th2 = split2(k.th2);
    c.om1 = split2(1.0 - k.th1);
    c.om2 = split2(1.0 - k.th2);
    c.nk12t = split2(-k.k12_tube);
    c.rule0 = (k.four_tau2 < 3.0e38) ? 1 : 0;
    c.tau2 = split(k.tau2);
    c.four_tau2 = c.rule0 ? split(k.four_tau2) : make_float2(__builtin_huge_valf(), 0.0f);
    c.tau2_d = k.tau2;
    c.four_tau2_d = k.four_tau2;
    const double two_tau = 2.0 * sqrt(k.tau2);
    c.far_dist = (float)((two_tau > 1.5 ? two_tau : 1.5) * 1.001 + 1e-3);
    return c;
}

// Tube test of one pair in FP64 with the oracle's operations in its order
// (no contraction): used for pairs within rounding of a threshold.
static __device__ __noinline__ bool tube_f64_ordered(const double* __restrict__ geo, int64_t N, int64_t i, int64_t j,
                                                     double tau2, double four_tau2)
{
    const double r0 = __dsub_rn(geo[i], geo[j]);
    const double r1 = __dsub_rn(geo[N + i], geo[N + j]);
    const double r2 = __dsub_rn(geo[2 * N + i], geo[2 * N + j]);
    const double rho2 = __dadd_rn(__dadd_rn(__dmul_rn(r0, r0), __dmul_rn(r1, r1)), __dmul_rn(r2, r2));
    const double sx = __dadd_rn(__dadd_rn(__dmul_rn(r0, geo[3 * N + i]), __dmul_rn(r1, geo[4 * N + i])),
                                __dmul_rn(r2, geo[5 * N + i]));
    const double rp2 = __dsub_rn(rho2, __dmul_rn(sx, sx));
    return (rp2 < tau2) && (rho2 < four_tau2);
}

// ---------------------------------------------------------------- pair

// A target and a pair of sources: position, normal, a = w psi, b = w psin.
struct FFNode {
    ff x[3], n[3], a, b;
};
struct FFPair {
    ff2 x[3], n[3], a, b;
};

// pair pr of the chunk at cb
__device__ __forceinline__ FFPair ff_load(const float4* __restrict__ cb, int pr)
{
    float4 v[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = cb[c * kFFPairs + pr];
    const auto lo = [](const float4& f) { return make_float2(f.x, f.y); };
    const auto hi = [](const float4& f) { return make_float2(f.z, f.w); };
    FFPair s;
#pragma unroll
    for (int f = 0; f < 2; ++f) {  // x, a then n, b
        ff2* d = f ? s.n : s.x;
        d[0] = ff2{lo(v[4 * f]), lo(v[4 * f + 2])};
        d[1] = ff2{hi(v[4 * f]), hi(v[4 * f + 2])};
        d[2] = ff2{lo(v[4 * f + 1]), lo(v[4 * f + 3])};
        (f ? s.b : s.a) = ff2{hi(v[4 * f + 1]), hi(v[4 * f + 3])};
    }
    return s;
}

// Geometry of the (target T <- source s) pairs.
struct FFGeo {
    ff2 rr, sx, sy;
};

__device__ __forceinline__ FFGeo ff_geo(const FFNode& T, const FFPair& s)
{
    ff2 r[3], n[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        // r = x - y: the hi parts share the grid, so their difference is exact
        r[c].h = vsub(vset(T.x[c].h), s.x[c].h);
        r[c].l = vsub(vset(T.x[c].l), s.x[c].l);
        n[c] = ff_wide(T.n[c]);
    }
    FFGeo g;
    g.rr = ff_norm(ff_norm2(r));
    g.sx = ff_norm(ff_dot3(r, n));
    g.sy = ff_norm(ff_dot3(r, s.n));
    return g;
}

// Factors of the two directions: y1 takes P1 s_y a - Q b, y2 takes B3 a + P2 s_x b.
struct FFFactors {
    ff2 P1, Q, P2, B3;
};

__device__ __forceinline__ FFFactors ff_factors(const FFGeo& G, const FFNode& T, const FFPair& s,
                                                   const FFConsts& k, const float2* __restrict__ tab)
{
    const ff2 nt[3] = {ff_wide(T.n[0]), ff_wide(T.n[1]), ff_wide(T.n[2])};
    const ff2 cc = ff_dot3(nt, s.n);
    // 1/rho: MUFU estimate, one Newton step in float-float
    const float2 y0 = vrsqrt(G.rr.h);
    const float2 yy = vmul(y0, y0);  // d = |r|^2 y0^2 - 1, about 2^-21
    const float2 d = vfma(G.rr.h, vfma(y0, y0, vneg(yy)), vfma(G.rr.l, yy, vfma(G.rr.h, yy, vset(-1.0f))));
    const ff2 inv = fast_two_sum(y0, vmul(vmul(y0, d), vfma(vset(0.375f), d, vset(-0.5f))));
    const ff2 rho = ff_norm(ff_mul(G.rr, inv));
    const ff2 x = ff_mul(ff_of(k.kap), rho);
    const ff2 E = ff_exp2(ff_mul(ff_of(k.cz), rho), tab);
    const ff2 Ex = ff_mul(E, x);
    // f = 1 - E (0 < E <= 1: fast two-sum of 1 and -E.h)
    const float2 one = vset(1.0f);
    const float2 fh = vsub(one, E.h);
    const ff2 f{fh, vsub(vsub(vsub(one, fh), E.h), E.l)};
    const ff2 g = ff_sub(f, Ex);                                         // 1 - A
    const ff2 u1 = ff_add_u(ff_of(k.om1), ff_mul(ff_of(k.th1), g));  // 1 - th1 A
    const ff2 u2 = ff_add_u(ff_of(k.om2), ff_mul(ff_of(k.th2), g));  // 1 - th2 A
    const ff2 hb = ff_add_u(ff_mulf(g, vset(3.0f)), ff_neg(ff_mul(Ex, x)));  // 3 - B
    const ff2 inv2 = ff_mul(inv, inv);
    const ff2 inv3 = ff_mul(inv2, inv);
    const ff2 br = ff_dot2_u(g, cc, ff_neg(hb), ff_mul(ff_mul(G.sx, G.sy), inv2));
    return FFFactors{ff_mul(u1, inv3), ff_mul(f, inv), ff_mul(u2, inv3), ff_mul(br, inv3)};
}

// Forward contributions of the pairs.
__device__ __forceinline__ void ff_forward(const FFGeo& G, const FFFactors& F, const FFPair& s, ff2& c1, ff2& c2)
{
    c1 = ff_dot2_u(F.P1, ff_mul(G.sy, s.a), ff_neg(F.Q), s.b);
    c2 = ff_dot2_u(F.B3, s.a, ff_mul(F.P2, G.sx), s.b);
}

// Reverse contributions (s_x' = -s_y, s_y' = -s_x).
__device__ __forceinline__ void ff_reverse(const FFGeo& G, const FFFactors& F, const FFNode& T, ff2& c1, ff2& c2)
{
    const ff2 ai = ff_wide(T.a), bi = ff_wide(T.b);
    c1 = ff_neg(ff_dot2_u(F.P1, ff_mul(G.sx, ai), F.Q, bi));
    c2 = ff_dot2_u(F.B3, ai, ff_neg(ff_mul(F.P2, G.sy)), bi);
}

// Tube tests of the pairs i <- j and i <- j + 16 (reverse: j <- i and j + 16 <- i);
// sn = r . n with the target's normal.
__device__ __forceinline__ void ff_tube(const ff2& rr, const ff2& sn, const FFConsts& k, const double* __restrict__ geo,
                                        int64_t i, int64_t j, int64_t N, bool reverse, bool (&tube)[2])
{
    // rho_P^2 = |r|^2 - s_n^2 < tau^2 and |r|^2 < 4 tau^2 (tube rule 0)
    const ff2 rp2 = ff_sub(rr, ff_mul(sn, sn));
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const ff p = ff_half(rp2, q), d = ff_half(rr, q);
        const float d1 = __fadd_rn(__fsub_rn(p.h, k.tau2.x), __fsub_rn(p.l, k.tau2.y));
        const float d2 = __fadd_rn(__fsub_rn(d.h, k.four_tau2.x), __fsub_rn(d.l, k.four_tau2.y));
        tube[q] = (d1 < 0.0f) && (d2 < 0.0f);
        if ((fabsf(d1) < 1e-9f * k.tau2.x) || (fabsf(d2) < 1e-9f * k.four_tau2.x)) {  // tie
            const int64_t jq = j + q * kFFPairs;
            if (i < N && jq < N)
                tube[q] = reverse ? tube_f64_ordered(geo, N, jq, i, k.tau2_d, k.four_tau2_d)
                                  : tube_f64_ordered(geo, N, i, jq, k.tau2_d, k.four_tau2_d);
        }
    }
}

// Contributions inside the tube: y1 -= K12_tube b, nothing to y2.
__device__ __forceinline__ void ff_tube_select(const bool (&tube)[2], const ff2& b, const FFConsts& k, ff2& c1, ff2& c2)
{
    const ff2 t = ff_mul(ff_of(k.nk12t), b);
    c1.h = make_float2(tube[0] ? t.h.x : c1.h.x, tube[1] ? t.h.y : c1.h.y);
    c1.l = make_float2(tube[0] ? t.l.x : c1.l.x, tube[1] ? t.l.y : c1.l.y);
    c2.h = make_float2(tube[0] ? 0.0f : c2.h.x, tube[1] ? 0.0f : c2.h.y);
    c2.l = make_float2(tube[0] ? 0.0f : c2.l.x, tube[1] ? 0.0f : c2.l.y);
}

// Two pairs: forward into (S1, S2) and, when rev, reverse into (R1, R2).  NEAR:
// they may lie in the regularisation tube (nodes i <- j, j + 16; both sides are
// evaluated and selected, the self pair among the regularised ones).
template <bool NEAR>
__device__ __forceinline__ void ff_pairs2(const FFNode& T, const FFPair& m, const FFConsts& k,
                                          const float2* __restrict__ tab, bool rev, ff2& S1, ff2& S2, ff2& R1, ff2& R2,
                                          const double* __restrict__ geo, int64_t i, int64_t j, int64_t N)
{
    const FFGeo G = ff_geo(T, m);
    bool tf[2], tr[2];
    if (NEAR) {
        ff_tube(G.rr, G.sx, k, geo, i, j, N, false, tf);
        if (rev) ff_tube(G.rr, G.sy, k, geo, i, j, N, true, tr);
    }
    const FFFactors F = ff_factors(G, T, m, k, tab);
    ff2 c1, c2;
    ff_forward(G, F, m, c1, c2);
    if (NEAR) ff_tube_select(tf, m.b, k, c1, c2);
    S1 = ff_add(S1, c1);
    S2 = ff_add(S2, c2);
    if (rev) {
        ff_reverse(G, F, T, c1, c2);
        if (NEAR) ff_tube_select(tr, ff_wide(T.b), k, c1, c2);
        R1 = ff_add(R1, c1);
        R2 = ff_add(R2, c2);
    }
}

// Target i (placeholders from N on lie away from placeholder sources).
__device__ __forceinline__ FFNode ff_target(const float* __restrict__ src, int64_t i, int64_t N)
{
    FFNode T;
    const bool pad = i >= N;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        T.x[c] = pad ? ff{-kFFPad, 0.0f} : ff{src[ff_off(i, 0, c)], src[ff_off(i, 1, c)]};
        T.n[c] = ff{src[ff_off(i, 2, c)], src[ff_off(i, 3, c)]};
    }
    T.a = ff{src[ff_off(i, 0, 3)], src[ff_off(i, 1, 3)]};
    T.b = ff{src[ff_off(i, 2, 3)], src[ff_off(i, 3, 3)]};
    return T;
}

__device__ __forceinline__ double ff_value(ff2 v) { return ((double)v.h.x + (double)v.l.x) + ((double)v.h.y + (double)v.l.y); }

// ---------------------------------------------------------------- kernels

__global__ void __launch_bounds__(kFFThreads, 2)
    pair_ff_kernel(const float4* __restrict__ src, const float4* __restrict__ frames, const float2* __restrict__ tab_g,
                   const double* __restrict__ geo, int64_t N, PairSchedule s, FFConsts k, double* __restrict__ part,
                   unsigned* __restrict__ err, const int* __restrict__ skip)
{
    if (skip != nullptr && *skip) return;
    __shared__ __align__(128) float4 sbuf[kFFStages][kFFSTile * kFFNodeF4];
    __shared__ __align__(16) float4 sfrm[kFFStages][2 * kFFChunksPerTile];
    __shared__ float2 tab[kFFTab];
    __shared__ __align__(8) uint64_t bars[kFFStages];
    __shared__ int abort_flag;

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int64_t s0 = (int64_t)blockIdx.x * s.per_cta;
    const int64_t s1 = (s0 + s.per_cta < s.total) ? s0 + s.per_cta : s.total;
    if (s0 >= s1) return;
    for (int q = tid; q < kFFTab; q += kFFThreads) tab[q] = tab_g[q];
    if (tid == 0) {
        for (int q = 0; q < kFFStages; ++q) ptx::mbar_init(&bars[q], 1);
        ptx::fence_mbar_init();
        abort_flag = 0;
    }
    __syncthreads();

    auto issue = [&](int64_t u) {
        const int64_t st = ((u % s.n_stiles) * s.sperm) % s.n_stiles;
        const int stage = (int)((u - s0) % kFFStages);
        ptx::mbar_arrive_expect_tx(&bars[stage], kFFStageBytes + kFFFrameBytes);
        ptx::bulk_g2s(&sbuf[stage][0], src + st * kFFSTile * kFFNodeF4, kFFStageBytes, &bars[stage]);
        ptx::bulk_g2s(&sfrm[stage][0], frames + st * 2 * kFFChunksPerTile, kFFFrameBytes, &bars[stage]);
    };
    if (tid == 0)
        for (int q = 0; q < kFFStages && s0 + q < s1; ++q) issue(s0 + q);

    const int64_t t_first = s0 / s.n_stiles;
    int64_t t = t_first;
    FFNode T;
    float4 tfh, tfl;  // frame of the warp's target block
    int64_t gi = 0;
    bool idle = false;
    double D1 = 0.0, D2 = 0.0;
    auto load_target = [&](int64_t tile) {
        gi = tile * kFFTTile + tid;
        idle = tile * kFFTTile + warp * kFFChunk >= N;
        T = ff_target(reinterpret_cast<const float*>(src), gi, N);
        const int64_t blk = (tile * kFFTTile + warp * kFFChunk) / kFFChunk;
        tfh = frames[2 * blk];
        tfl = frames[2 * blk + 1];
        D1 = D2 = 0.0;
    };
    load_target(t);

    for (int64_t u = s0; u < s1; ++u) {
        const int stage = (int)((u - s0) % kFFStages);
        const uint32_t parity = (uint32_t)(((u - s0) / kFFStages) & 1);
        if (!ptx::mbar_wait_bounded(&bars[stage], parity, kFFWaitNs)) {
            abort_flag = 1;
            atomicOr(err, kDevErrTimeout);
        }
        __syncthreads();
        if (abort_flag) return;
        const int64_t sp = u % s.n_stiles;
        const int64_t st = (sp * s.sperm) % s.n_stiles;
        if (!idle) {
            ff2 S1{}, S2{}, R1{}, R2{};  // the reverse sums stay zero
            const float4* sb = &sbuf[stage][0];
#pragma unroll 1
            for (int c = 0; c < kFFChunksPerTile; ++c) {
                // far chunk pair: the two blocks' bounding spheres are apart by more than the tube reaches
                const float4 mh = sfrm[stage][2 * c], ml = sfrm[stage][2 * c + 1];
                const float dx = (tfh.x - mh.x) + (tfl.x - ml.x);
                const float dy = (tfh.y - mh.y) + (tfl.y - ml.y);
                const float dz = (tfh.z - mh.z) + (tfl.z - ml.z);
                const float lim = k.far_dist + tfh.w + mh.w;
                const bool far = k.rule0 && (fmaf(dx, dx, fmaf(dy, dy, dz * dz)) >= lim * lim);
                const float4* cb = sb + c * kFFChunk * kFFNodeF4;
                const int64_t j0 = st * kFFSTile + c * kFFChunk;
                if (far) {
#pragma unroll 1
                    for (int p = 0; p < kFFPairs; ++p)
                        ff_pairs2<false>(T, ff_load(cb, p), k, tab, false, S1, S2, R1, R2, geo, gi, j0 + p, N);
                } else {
#pragma unroll 1
                    for (int p = 0; p < kFFPairs; ++p)
                        ff_pairs2<true>(T, ff_load(cb, p), k, tab, false, S1, S2, R1, R2, geo, gi, j0 + p, N);
                }
            }
            D1 += ff_value(S1);
            D2 += ff_value(S2);
        }
        __syncthreads();
        if (tid == 0 && u + kFFStages < s1) {
            ptx::fence_proxy_async_smem();
            issue(u + kFFStages);
        }
        if (sp == s.n_stiles - 1 || u + 1 == s1) {
            const int seg = (int)(t - t_first);
            double* dst = part + ((int64_t)blockIdx.x * s.max_segs + seg) * 2 * kFFTTile;
            dst[tid] = D1;
            dst[kFFTTile + tid] = D2;
            if (sp == s.n_stiles - 1 && u + 1 < s1) {
                ++t;
                load_target(t);
            }
        }
    }
}

// ---------------------------------------------------------------- symmetric
//
// The same operator with each unordered node pair evaluated once for both
// directions (as the symmetric FP32 kernel of pair_sym.cu does): the shared
// float-float work (r, |r|^2, s_x, s_y, n . m, 1/rho, E, g, 1 - th A, 3 - B,
// the combination g c - (3 - B) s_x s_y / rho^2 and the powers of 1/rho) is
// done once, and the reverse direction (target j <- source i) is formed from
// it with r' = -r, s_x' = -s_y, s_y' = -s_x, c' = c:
//   forward   y1_i += u1 s_y a_j / rho^3 - (1 - E) b_j / rho
//             y2_i += [br a_j + u2 s_x b_j] / rho^3
//   reverse   y1_j += -u1 s_x a_i / rho^3 - (1 - E) b_i / rho
//             y2_j += [br a_i - u2 s_y b_i] / rho^3
// with br = g c - (3 - B) s_x s_y / rho^2.  Each direction takes its own tube
// test (the reverse one on the source's normal, rho_P'^2 = |r|^2 - s_y^2).
// 408 FP32 operations per unordered pair against 2 x 346.
//
// Per warp and source chunk the 32 lanes hold 32 targets; each half-warp walks
// the chunk's 16 pairs of sources in a staggered order (lane l takes pair
// (l + k) mod 16 at step k); the float-float reverse sums of a pair ride along
// with it from lane to lane (four shuffles a node pair), so after 16 steps lane l
// holds pair l mod 16's reverse sums over its half's targets; the halves are
// added and go, as doubles, to the reverse vector with FP64 atomics.  Forward
// sums and the schedule (upper triangle, large and small segments, partials per
// (segment, row)) are those of the symmetric FP32 kernel, and its fixup adds
// everything up.
__device__ __forceinline__ ff2 ff_rotate(ff2 v, int lane)
{
    ff2 o;
    o.h.x = __shfl_sync(0xffffffffu, v.h.x, lane + 1, kFFPairs);
    o.h.y = __shfl_sync(0xffffffffu, v.h.y, lane + 1, kFFPairs);
    o.l.x = __shfl_sync(0xffffffffu, v.l.x, lane + 1, kFFPairs);
    o.l.y = __shfl_sync(0xffffffffu, v.l.y, lane + 1, kFFPairs);
    return o;
}

// After 16 rotations lane l holds the pair l mod 16 summed over its half-warp's
// targets: the sum over both halves of node l (first halves' lanes keep .x).
__device__ __forceinline__ double ff_halves_sum(ff2 v, int lane)
{
    const bool low = lane < kFFPairs;
    const ff keep = ff_half(v, low ? 0 : 1), give = ff_half(v, low ? 1 : 0);
    const float gh = __shfl_xor_sync(0xffffffffu, give.h, kFFPairs);
    const float gl = __shfl_xor_sync(0xffffffffu, give.l, kFFPairs);
    return ((double)keep.h + (double)keep.l) + ((double)gh + (double)gl);
}

// THREADS targets (one per thread) and STILE sources per step.  Small steps, as
// a launch on a small molecule has few: 128 x 32 against 256 x 256 takes 38 us
// for 216 at 862 nodes, 105 for 214 at 3,214, 207 for 343 at 5,014.  The CTAs of
// an SM do not advance alike (the scheduler favours the older warps), so most of
// the work is in small segments: at 80,358 nodes 43.1 ms with nine tenths of an
// even share per CTA in large ones, 41.5 with half, 39.9 with one tenth.
template <int THREADS, int STILE>
__global__ void __launch_bounds__(THREADS, 512 / THREADS)
    pair_ffs_kernel(const float4* __restrict__ src, const float4* __restrict__ frames,
                    const float2* __restrict__ tab_g, const double* __restrict__ geo, int64_t N, int64_t n_pad,
                    SymSchedule s, FFConsts k, double* __restrict__ part, double* __restrict__ yrev,
                    unsigned* __restrict__ err, const int* __restrict__ skip)
{
    constexpr int TTILE = THREADS;
    constexpr int CHUNKS = STILE / kFFChunk;
    constexpr uint32_t STAGE_BYTES = STILE * kFFNodeF4 * sizeof(float4);
    constexpr uint32_t FRAME_BYTES = 2 * CHUNKS * sizeof(float4);
    if (skip != nullptr && *skip) return;
    __shared__ __align__(128) float4 sbuf[kFFStages][STILE * kFFNodeF4];
    __shared__ __align__(16) float4 sfrm[kFFStages][2 * CHUNKS];
    __shared__ float2 tab[kFFTab];
    __shared__ __align__(8) uint64_t bars[kFFStages];
    __shared__ int abort_flag;
    __shared__ int64_t seg_next;

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;
    unsigned long long* seg_ctr = reinterpret_cast<unsigned long long*>(yrev + 2 * n_pad);
    for (int q = tid; q < kFFTab; q += THREADS) tab[q] = tab_g[q];
    if (tid == 0) {
        for (int q = 0; q < kFFStages; ++q) ptx::mbar_init(&bars[q], 1);
        ptx::fence_mbar_init();
        abort_flag = 0;
    }
    __syncthreads();

    // ring position: this CTA's n-th step uses stage n mod kFFStages, phase (n / kFFStages) mod 2
    int64_t n_done = 0;
    auto issue = [&](int64_t u, int64_t n) {
        int64_t t, rho, pos;
        sym_locate(s, u, t, rho, pos);
        const int64_t st = s.R * t + pos;
        const int stage = (int)(n % kFFStages);
        ptx::mbar_arrive_expect_tx(&bars[stage], STAGE_BYTES + FRAME_BYTES);
        ptx::bulk_g2s(&sbuf[stage][0], src + st * STILE * kFFNodeF4, STAGE_BYTES, &bars[stage]);
        ptx::bulk_g2s(&sfrm[stage][0], frames + st * 2 * CHUNKS, FRAME_BYTES, &bars[stage]);
    };

    FFNode T;
    float4 tfh, tfl;
    int64_t gi = 0;
    int Ablk = 0;
    bool idle = false;
    double D1 = 0.0, D2 = 0.0;
    auto load_target = [&](int64_t tile) {
        gi = tile * TTILE + tid;
        idle = tile * TTILE + warp * kFFChunk >= N;
        T = ff_target(reinterpret_cast<const float*>(src), gi, N);
        Ablk = (int)((tile * TTILE + warp * kFFChunk) / kFFChunk);
        const int64_t blk = Ablk;
        tfh = frames[2 * blk];
        tfl = frames[2 * blk + 1];
        D1 = D2 = 0.0;
    };

    int64_t seg = blockIdx.x;
    while (seg < s.nseg) {
        const int64_t s0 = sym_seg_start(s, seg), s1 = sym_seg_start(s, seg + 1);
        if (tid == 0)
            for (int q = 0; q < kFFStages && s0 + q < s1; ++q) issue(s0 + q, n_done + q);
        int64_t t, rho, pos;
        sym_locate(s, s0, t, rho, pos);
        load_target(t);
        for (int64_t u = s0; u < s1; ++u) {
            const int64_t n = n_done + (u - s0);
            const int stage = (int)(n % kFFStages);
            if (!ptx::mbar_wait_bounded(&bars[stage], (uint32_t)((n / kFFStages) & 1), kFFWaitNs)) {
                abort_flag = 1;
                atomicOr(err, kDevErrTimeout);
            }
            __syncthreads();
            if (abort_flag) return;
            const int64_t st = s.R * t + pos;
            if (!idle) {
                ff2 S1{}, S2{};
                const float4* sb = &sbuf[stage][0];
#pragma unroll 1
                for (int c = 0; c < CHUNKS; ++c) {
                    const int64_t Bc = st * CHUNKS + c;
                    if (Bc < Ablk) continue;  // the warp holding block Bc covers this block pair
                    const bool rev = Bc > Ablk;
                    const float4 mh = sfrm[stage][2 * c], ml = sfrm[stage][2 * c + 1];
                    const float dx = (tfh.x - mh.x) + (tfl.x - ml.x);
                    const float dy = (tfh.y - mh.y) + (tfl.y - ml.y);
                    const float dz = (tfh.z - mh.z) + (tfl.z - ml.z);
                    const float lim = k.far_dist + tfh.w + mh.w;
                    const bool far = rev && k.rule0 && (fmaf(dx, dx, fmaf(dy, dy, dz * dz)) >= lim * lim);
                    const float4* cb = sb + c * kFFChunk * kFFNodeF4;
                    const int64_t j0 = Bc * kFFChunk;
                    // each half-warp walks the 16 pairs of sources, lane l taking pair
                    // (l + step) mod 16; a pair's reverse sums go to lane - 1 of the half
                    ff2 R1{}, R2{};
                    if (far) {
#pragma unroll 1
                        for (int step = 0; step < kFFPairs; ++step) {
                            const int p = (lane + step) & (kFFPairs - 1);
                            ff_pairs2<false>(T, ff_load(cb, p), k, tab, true, S1, S2, R1, R2, geo, gi, j0 + p, N);
                            R1 = ff_rotate(R1, lane);
                            R2 = ff_rotate(R2, lane);
                        }
                    } else {
#pragma unroll 1
                        for (int step = 0; step < kFFPairs; ++step) {
                            const int p = (lane + step) & (kFFPairs - 1);
                            ff_pairs2<true>(T, ff_load(cb, p), k, tab, rev, S1, S2, R1, R2, geo, gi, j0 + p, N);
                            R1 = ff_rotate(R1, lane);
                            R2 = ff_rotate(R2, lane);
                        }
                    }
                    if (rev) {
                        // source j0 + lane's reverse sums over the warp's targets
                        atomicAdd(yrev + j0 + lane, ff_halves_sum(R1, lane));
                        atomicAdd(yrev + n_pad + j0 + lane, ff_halves_sum(R2, lane));
                    }
                }
                D1 += ff_value(S1);
                D2 += ff_value(S2);
            }
            __syncthreads();
            if (tid == 0 && u + kFFStages < s1) {
                ptx::fence_proxy_async_smem();
                issue(u + kFFStages, n + kFFStages);
            }
            if (pos == sym_row_len(s, t) - 1 || u + 1 == s1) {
                double* dst = part + (seg + rho) * 2 * TTILE;
                dst[tid] = D1;
                dst[TTILE + tid] = D2;
                if (u + 1 < s1) {
                    sym_locate(s, u + 1, t, rho, pos);
                    load_target(t);
                }
            } else {
                ++pos;
            }
        }
        n_done += s1 - s0;
        if (tid == 0) seg_next = s.nbig + (int64_t)atomicAdd(seg_ctr, 1ull);
        __syncthreads();
        seg = seg_next;
        __syncthreads();
    }
}

// 2^(i/256) as float-float pairs, i = 0..255 (FP64 exp2 of the CUDA math library).
__global__ void ff_table_kernel(float2* __restrict__ tab)
{
    const int i = threadIdx.x;
    if (i >= kFFTab) return;
    const double v = exp2((double)i / (double)kFFTab);
    const float h = (float)v;
    tab[i] = make_float2(h, (float)(v - (double)h));
}

// Largest |x* - centroid| component (one CTA; fixed order).
__global__ void ff_extent_kernel(const double* __restrict__ geo, int64_t N, double c0, double c1, double c2,
                                 double* __restrict__ out)
{
    __shared__ double red[256];
    double m = 0.0;
    for (int64_t j = threadIdx.x; j < N; j += blockDim.x)
        m = fmax(m, fmax(fabs(geo[j] - c0), fmax(fabs(geo[N + j] - c1), fabs(geo[2 * N + j] - c2))));
    red[threadIdx.x] = m;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + o]);
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = red[0];
}

// Float-float payload of the padded node range for input `in` (one thread
// per node): coordinates relative to the centroid split on the 2^-q grid,
// normals, a = w psi and b = w psin split into hi + lo.
__global__ void ff_pack_kernel(const double* __restrict__ geo, int64_t N, int64_t n_pad, double c0, double c1,
                               double c2, double grid_scale, VecRef in, float4* __restrict__ src,
                               double* __restrict__ yrev, const int* __restrict__ skip)
{
    if (skip != nullptr && *skip) return;
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n_pad) return;
    if (yrev != nullptr) {  // symmetric kernel: clear its reverse sums and its segment counter
        yrev[j] = 0.0;
        yrev[n_pad + j] = 0.0;
        if (j == 0) *reinterpret_cast<unsigned long long*>(yrev + 2 * n_pad) = 0ull;
    }
    float* dst = reinterpret_cast<float*>(src);
    if (j >= N) {
        for (int c = 0; c < 4; ++c) {
            dst[ff_off(j, 0, c)] = c < 3 ? kFFPad : 0.0f;
            dst[ff_off(j, 1, c)] = 0.0f;
            dst[ff_off(j, 2, c)] = c == 2 ? 1.0f : 0.0f;
            dst[ff_off(j, 3, c)] = 0.0f;
        }
        return;
    }
    const double* p = in.base + (in.kidx ? (int64_t)(*in.kidx + in.koff) * in.stride : 0);
    const double cen[3] = {c0, c1, c2};
    const double w = geo[6 * N + j];
    for (int a = 0; a < 4; ++a) {
        // position and normal components, then a and b
        const double x = a < 3 ? geo[a * N + j] - cen[a] : w * p[j];
        const double n = a < 3 ? geo[(3 + a) * N + j] : w * p[N + j];
        // positions: on the grid, exact as a float
        const float xh = a < 3 ? (float)(rint(x * grid_scale) / grid_scale) : (float)x;
        const float nh = (float)n;
        dst[ff_off(j, 0, a)] = xh;
        dst[ff_off(j, 1, a)] = (float)(x - (double)xh);
        dst[ff_off(j, 2, a)] = nh;
        dst[ff_off(j, 3, a)] = (float)(n - (double)nh);
    }
}

// ------------------------------------------------------------------ host side

int ff_grid_cap(ibim_ctx* c)
{
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, pair_ff_kernel, kFFThreads, 0);
    return (occ < 1 ? 1 : occ) * c->num_sms;
}

PairSchedule ff_schedule(ibim_ctx* c) { return make_schedule(c->N, kFFTTile, c->N, kFFSTile, ff_grid_cap(c)); }

size_t ffs_part_doubles(ibim_ctx* c);

size_t ff_part_doubles(ibim_ctx* c)
{
    const PairSchedule s = ff_schedule(c);
    return std::max((size_t)s.grid * s.max_segs * 2 * kFFTTile, ffs_part_doubles(c));
}

size_t ff_src_bytes(int64_t N) { return (size_t)padded_nodes(N) * kFFNodeF4 * sizeof(float4); }

// Table and grid of the context (once): the 2^(i/256) table and the
// power-of-two grid 2^-q of the hi parts, with |x - centroid| 2^q < 2^23.
static ibim_status ff_prepare(ibim_ctx* c)
{
    if (c->d_fftab != nullptr) return IBIM_OK;
    IBIM_TRY(ensure(c, (void**)&c->d_red, &c->red_bytes, std::max(c->red_bytes, (size_t)4096)));
    ff_extent_kernel<<<1, 256, 0, c->stream>>>(c->d_geo64, c->N, c->centroid[0], c->centroid[1], c->centroid[2],
                                              c->d_red);
    count_launch(c);
    IBIM_CUDA(cudaGetLastError());
    double ext = 0.0;
    IBIM_CUDA(cudaMemcpyAsync(&ext, c->d_red, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    IBIM_CUDA(cudaStreamSynchronize(c->stream));
    int e = 0;
    frexp(ext > 1e-3 ? ext : 1e-3, &e);  // ext < 2^e
    c->ff_grid_scale = ldexp(1.0, 23 - e);
    IBIM_CUDA(cudaMalloc((void**)&c->d_fftab, sizeof(float2) * kFFTab));
    ff_table_kernel<<<1, kFFTab, 0, c->stream>>>(c->d_fftab);
    count_launch(c);
    IBIM_CUDA(cudaGetLastError());
    return IBIM_OK;
}

ibim_status ff_prepare_context(ibim_ctx* c) { return ff_prepare(c); }

constexpr int kFFSThreads = 128, kFFSSTile = 32, kFFSBigShare = 1;
static const auto ffs_kernel = pair_ffs_kernel<kFFSThreads, kFFSSTile>;

int ffs_grid_cap(ibim_ctx* c)
{
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, ffs_kernel, kFFSThreads, 0);
    return (occ < 1 ? 1 : occ) * c->num_sms;
}

size_t ffs_part_doubles(ibim_ctx* c) { return sym_part_doubles(c->N, kFFSThreads, kFFSSTile, ffs_grid_cap(c), kFFSBigShare); }

ibim_status ff_pack(ibim_ctx* c, VecRef in, const int* d_skip)
{
    IBIM_TRY(ff_prepare(c));
    const int64_t N = c->N, n_pad = padded_nodes(N);
    const int bs = 256;
    ff_pack_kernel<<<(unsigned)((n_pad + bs - 1) / bs), bs, 0, c->stream>>>(
        c->d_geo64, N, n_pad, c->centroid[0], c->centroid[1], c->centroid[2], c->ff_grid_scale, in,
        (float4*)c->d_src, c->ff_symmetric ? c->d_yrev : nullptr, d_skip);
    count_launch(c);
    IBIM_CUDA(cudaGetLastError());
    return IBIM_OK;
}

ibim_status ff_pairs(ibim_ctx* c, const PairConsts& k, const PairSchedule& s, const int* d_skip)
{
    if (c->ff_symmetric) {
        const SymSchedule ss = make_sym_schedule(c->N, kFFSThreads, kFFSSTile, ffs_grid_cap(c), kFFSBigShare);
        ffs_kernel<<<ss.grid, kFFSThreads, 0, c->stream>>>(
            (const float4*)c->d_src, c->d_frames, c->d_fftab, c->d_geo64, c->N, padded_nodes(c->N), ss, ff_consts(k),
            c->d_part, c->d_yrev, c->d_err, d_skip);
    } else {
        pair_ff_kernel<<<s.grid, kFFThreads, 0, c->stream>>>((const float4*)c->d_src, c->d_frames, c->d_fftab,
                                                              c->d_geo64, c->N, s, ff_consts(k), c->d_part, c->d_err,
                                                              d_skip);
    }
    count_launch(c);
    IBIM_CUDA(cudaGetLastError());
    return IBIM_OK;
}

ibim_status ff_fixup(ibim_ctx* c, const PairConsts& k, const PairSchedule& s, VecRef in, OutRef out,
                     const int* d_skip)
{
    if (c->ff_symmetric) return sym_fixup_tiles(c, kFFSThreads, kFFSSTile, ffs_grid_cap(c), k, in, out, d_skip, kFFSBigShare);
    return fixup_launch(c, k, s, kFFTTile, in, out, d_skip);
}

}  // namespace ibim
