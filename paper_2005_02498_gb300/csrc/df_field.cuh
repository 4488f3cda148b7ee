// df_field.cuh -- the field of seg_field.cuh in double-float arithmetic: every
// number is an unevaluated sum h + l of two FP32 values (about 48 bits), so
// the work runs on the FP32 pipe, which on this GPU has 64 times the FP64
// pipe's rate.  Used by the FP64 pair kernels for pairs that are not close;
// close pairs stay in FP64 (pair_tile.cuh).
//
// Products are exact through the fused multiply-add's residual, sums through
// Knuth's two-sum, or Dekker's fast two-sum where the larger operand is known;
// a result's low part stays unnormalised where the next operation does not
// need it.  Everything is packed: the two lanes of a float2 are two Gauss
// points, or (for what a pair's four points share) the vectors R and D.
//
// The formula is written in the source's own frame t (tangent), e, n = t x e,
// with e along the part of b normal to t, so b = bt t + be e and q = b x t = -be n.
// With R = x_a - x1 (start node to start node) and D = x_b - x_a the point is
// R_q = R + xi D, and its components y = R_q.t, al = R_q.e, be = R_q.n are affine
// in xi: three packed dot products per pair give all four points.  Then d^2 =
// al^2 + be^2 + a^2, rho1^2 = d^2 + y^2, rho2^2 = d^2 + (L - y)^2 without
// cancellation, Rp.b' and b'.(Rp x b) follow from b'.t, b'.e, b'.n, and the
// stress is assembled from three vectors instead of five:
//   (sigma b')/c2 = S_t t + S_e e + S_n n + c_b b'.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

namespace ptadd {

// Everything here also compiles for the host, where the arithmetic is checked against
// 80-bit numbers pair by pair; DF_HOST_SEED stands in for the error of the hardware's
// reciprocal approximations there.
#define DF_FN __host__ __device__ __forceinline__
#ifndef DF_HOST_SEED
#define DF_HOST_SEED(y) (y)
#endif

// Packed FP32 operations, each rounded once and never contracted.
DF_FN float2 p_add(float2 a, float2 b)
{
#ifdef __CUDA_ARCH__
    return __fadd2_rn(a, b);
#else
    return make_float2(a.x + b.x, a.y + b.y);
#endif
}
DF_FN float2 p_neg(float2 a) { return make_float2(-a.x, -a.y); }
DF_FN float2 p_sub(float2 a, float2 b) { return p_add(a, p_neg(b)); }
DF_FN float2 p_mul(float2 a, float2 b)
{
#ifdef __CUDA_ARCH__
    return __fmul2_rn(a, b);
#else
    return make_float2(a.x * b.x, a.y * b.y);
#endif
}
DF_FN float2 p_fma(float2 a, float2 b, float2 c)
{
#ifdef __CUDA_ARCH__
    return __ffma2_rn(a, b, c);
#else
    return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
#endif
}
DF_FN float2 p_all(float s) { return make_float2(s, s); }
// the hardware's approximations on the device
DF_FN float2 p_rsqrt_seed(float2 x)
{
#ifdef __CUDA_ARCH__
    float2 y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.x) : "f"(x.x));
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.y) : "f"(x.y));
    return y;
#else
    return make_float2(DF_HOST_SEED(1.0f / sqrtf(x.x)), DF_HOST_SEED(1.0f / sqrtf(x.y)));
#endif
}
DF_FN float2 p_rcp_seed(float2 x)
{
#ifdef __CUDA_ARCH__
    float2 y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y.x) : "f"(x.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y.y) : "f"(x.y));
    return y;
#else
    return make_float2(DF_HOST_SEED(1.0f / x.x), DF_HOST_SEED(1.0f / x.y));
#endif
}

// Gauss-Legendre rule on [0,1]: the textbook 4-point abscissae z and
// weights W on [-1,1] mapped by xi = (1 + z)/2, w = W/2.
DF_FN constexpr double gl4_xi(int qp)
{
    constexpr double z0 = 0.8611363115940526, z1 = 0.3399810435848563;
    return qp == 0 ? 0.5 * (1.0 - z0) : qp == 1 ? 0.5 * (1.0 - z1) : qp == 2 ? 0.5 * (1.0 + z1) : 0.5 * (1.0 + z0);
}
DF_FN constexpr double gl4_w(int qp)
{
    constexpr double W0 = 0.3478548451374538, W1 = 0.6521451548625461;
    return (qp == 0 || qp == 3) ? 0.5 * W0 : 0.5 * W1;
}

// ---------------------------------------------------------- double-float
struct DF2 {
    float2 h, l;
};
struct DF1 {  // one value
    float h, l;
};

// An FP64 value to the nearest FP32 one (0 below FP32's normal range, which the
// callers can leave out; infinite above it; NaN stays NaN) on the integer pipe: the hardware
// conversions and every FP64 operation run on the 1/64-rate FP64 pipe.
DF_FN float df_round(double x)
{
#ifdef __CUDA_ARCH__
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
#else
    uint64_t u;
    memcpy(&u, &x, sizeof(u));
    const uint32_t hi = (uint32_t)(u >> 32), lo = (uint32_t)u;
#endif
    const uint32_t e = (hi >> 20) & 0x7FFu, v = (hi << 3) | (lo >> 29);
    // exponents 897 .. 1150: the field moved by 896, plus the first dropped bit, carrying upwards
    uint32_t f = v - (896u << 23) + ((lo >> 28) & 1u);
    if (e < 897u) f = 0u;
    if (e > 1150u) f = e == 0x7FFu && (v & 0x7FFFFFu) ? 0x7FFFFFFFu : 0x7F800000u;
    f |= hi & 0x80000000u;
#ifdef __CUDA_ARCH__
    return __uint_as_float(f);
#else
    float r;
    memcpy(&r, &f, sizeof(r));
    return r;
#endif
}
// FP32 to FP64, exact for 0, the normal range and infinities (2^128 stands for these)
DF_FN double df_widen(float x)
{
#ifdef __CUDA_ARCH__
    const uint32_t u = __float_as_uint(x);
    const uint32_t hi = (u & 0x80000000u) | ((((u >> 23) & 0xFFu) + 896u) << 20) | ((u & 0x7FFFFFu) >> 3);
    return x != 0.0f ? __hiloint2double((int)hi, (int)(u << 29)) : 0.0;
#else
    return (double)x;
#endif
}
// The two FP32 parts of an FP64 value, each to nearest: h + l is within 2^-48 |x| of x, on
// either side alike.  (Truncated parts, one integer operation fewer each, were within 2^-46 and
// always short, and their error in the frames of the sources added up along a loop:
// far-field part of Lp of two loops of 21 segments 3.5e-15 against 1.2e-14.)
DF_FN DF1 df_split(double x)
{
    const float h = df_round(x);
    return DF1{h, df_round(x - df_widen(h))};
}
// the same for a constant
DF_FN constexpr DF1 df_from(double x) { return DF1{(float)x, (float)(x - (double)(float)x)}; }
DF_FN DF2 df_all(DF1 a) { return DF2{p_all(a.h), p_all(a.l)}; }
DF_FN DF2 df_pair2(DF1 a, DF1 b) { return DF2{make_float2(a.h, b.h), make_float2(a.l, b.l)}; }
DF_FN DF2 df_lane_x(DF2 a) { return DF2{p_all(a.h.x), p_all(a.l.x)}; }
DF_FN DF2 df_lane_y(DF2 a) { return DF2{p_all(a.h.y), p_all(a.l.y)}; }
DF_FN DF2 df_neg(DF2 a) { return DF2{p_neg(a.h), p_neg(a.l)}; }
DF_FN float2 two_sum(float2 a, float2 b, float2& e)
{
    const float2 s = p_add(a, b), t = p_sub(s, a);
    e = p_add(p_sub(a, p_sub(s, t)), p_sub(b, t));
    return s;
}
// |a| >= |b| or a = 0
DF_FN float2 fast_two_sum(float2 a, float2 b, float2& e)
{
    const float2 s = p_add(a, b);
    e = p_sub(b, p_sub(s, a));
    return s;
}
DF_FN DF2 df_norm(DF2 a)
{
    DF2 r;
    r.h = fast_two_sum(a.h, a.l, r.l);
    return r;
}
DF_FN DF2 df_add(DF2 a, DF2 b)
{
    float2 e;
    const float2 s = two_sum(a.h, b.h, e);
    return DF2{s, p_add(e, p_add(a.l, b.l))};
}
DF_FN DF2 df_sub(DF2 a, DF2 b) { return df_add(a, df_neg(b)); }
// |a.h| >= |b.h|
DF_FN DF2 df_add_big(DF2 a, DF2 b)
{
    float2 e;
    const float2 s = fast_two_sum(a.h, b.h, e);
    return DF2{s, p_add(e, p_add(a.l, b.l))};
}
DF_FN DF2 df_mul(DF2 a, DF2 b)
{
    const float2 p = p_mul(a.h, b.h);
    return DF2{p, p_fma(a.l, b.h, p_fma(a.h, b.l, p_fma(a.h, b.h, p_neg(p))))};
}
DF_FN DF2 df_sqr(DF2 a)
{
    const float2 p = p_mul(a.h, a.h);
    return DF2{p, p_fma(p_add(a.h, a.h), a.l, p_fma(a.h, a.h, p_neg(p)))};
}
// a b + c: the product's residual, both low parts and the two-sum's error in one chain
DF_FN DF2 df_fma(DF2 a, DF2 b, DF2 c)
{
    const float2 p = p_mul(a.h, b.h);
    float2 e;
    const float2 s = two_sum(c.h, p, e);
    const float2 lo = p_fma(a.l, b.h, p_fma(a.h, b.l, p_add(c.l, p_fma(a.h, b.h, p_neg(p)))));
    return DF2{s, p_add(e, lo)};
}
// the same for |c.h| >= |a b|
DF_FN DF2 df_fma_big(DF2 a, DF2 b, DF2 c)
{
    const float2 p = p_mul(a.h, b.h);
    float2 e;
    const float2 s = fast_two_sum(c.h, p, e);
    const float2 lo = p_fma(a.l, b.h, p_fma(a.h, b.l, p_add(c.l, p_fma(a.h, b.h, p_neg(p)))));
    return DF2{s, p_add(e, lo)};
}
DF_FN DF2 df_dot(const DF2 a[3], const DF2 b[3])
{
    return df_norm(df_fma(a[2], b[2], df_fma(a[1], b[1], df_mul(a[0], b[0]))));
}
struct Lanes {
    bool x, y;
};
DF_FN float2 p_sel(Lanes c, float2 a, float2 b) { return make_float2(c.x ? a.x : b.x, c.y ? a.y : b.y); }
DF_FN DF2 df_sel(Lanes c, DF2 a, DF2 b) { return DF2{p_sel(c, a.h, b.h), p_sel(c, a.l, b.l)}; }

// 1/sqrt(x): the FP32 seed y and one third-order correction y (1 + e/2 + 3 e^2/8)
// of e = 1 - x y^2, y^2 and x y^2 formed to twice FP32
DF_FN DF2 df_rsqrt(DF2 x)
{
    const float2 y = p_rsqrt_seed(x.h);
    const float2 p = p_mul(y, y), pe = p_fma(y, y, p_neg(p));
    const float2 nx = p_neg(x.h);
    const float2 e = p_fma(p_neg(x.l), p, p_fma(nx, pe, p_fma(nx, p, p_all(1.0f))));
    return df_norm(DF2{y, p_mul(p_mul(y, e), p_fma(e, p_all(0.375f), p_all(0.5f)))});
}
// 1/x: y (1 + e + e^2), e = 1 - x y
DF_FN DF2 df_rcp(DF2 x)
{
    const float2 y = p_rcp_seed(x.h);
    const float2 e = p_fma(p_neg(x.l), y, p_fma(p_neg(x.h), y, p_all(1.0f)));
    return DF2{y, p_mul(y, p_fma(e, e, e))};
}

// ------------------------------------------------------------- the field
// Lengths of the double-float path are in units of 2^-DF_SCALE of the
// kernels' unit, so that fourth and sixth powers of distances up to the
// far limit stay inside FP32's range.
constexpr int DF_SCALE = -10;

// Constants of the material: a^2 (scaled), r = -c1/c2, r a^2 (scaled), 1 + 2 r.
struct DFConst {
    DF1 a2, nr, nra2, kn;
};

// What a pair's four Gauss points share.
struct DFPair {
    DF2 y, al, be;          // lanes: the value for R, and for D
    DF1 tb, eb, nb;         // b'.t, b'.e, b'.n
};

// x - x1 of one coordinate, each given as an integer, a multiple of 2^-23 below
// 1/2 and a rest (scaled): the first two subtract exactly
DF_FN DF1 df_diff(const float a[3], const float b[3])
{
#ifdef __CUDA_ARCH__
    const float h = __fsub_rn(a[0], b[0]), m = __fsub_rn(a[1], b[1]), l = __fsub_rn(a[2], b[2]);
    const float s = __fadd_rn(h, m);
    const float lo = __fadd_rn(__fsub_rn(m, __fsub_rn(s, h)), l);
    const float r = __fadd_rn(s, lo);
    return DF1{r, __fsub_rn(lo, __fsub_rn(r, s))};
#else
    const float h = a[0] - b[0], m = a[1] - b[1], l = a[2] - b[2];
    const float s = h + m, lo = (m - (s - h)) + l, r = s + lo;
    return DF1{r, lo - (r - s)};
#endif
}

// Geometry of two Gauss points.
struct DFGeo {
    DF2 y, u2, al, be, d2, r1s, r2s;
};

DF_FN void df_geo(const DFPair& P, DF2 xi, DF2 L, const DFConst& K, DFGeo& G)
{
    G.y = df_fma(xi, df_lane_y(P.y), df_lane_x(P.y));
    G.al = df_fma(xi, df_lane_y(P.al), df_lane_x(P.al));
    G.be = df_fma(xi, df_lane_y(P.be), df_lane_x(P.be));
    G.d2 = df_fma(G.al, G.al, df_fma(G.be, G.be, df_all(K.a2)));
    G.r1s = df_fma(G.y, G.y, G.d2);
    G.u2 = df_sub(L, G.y);
    G.r2s = df_fma(G.u2, G.u2, G.d2);
}

// (sigma b') / c2 of the pair at the two points in the source's frame (St, Se,
// Sn, and cb along b'); far = false gives exactly 0.  One-sided (u1 u2 >= 0) and
// straddling pairs share one reciprocal rr = 1 / (den isum): J0 = num rr Ts,
// J1 = Li rr den, K2 = F V, with (den, num, Ts, F, V) =
// ((p + m)(1 + pm), Li, (1 + pm) isum, Li rr, Z) or (d^2, p - m, isum, J0 rr,
// (3 - S) isum); J0, J1, K2, Z and the coefficients as in seg_sigma_b_geo.
DF_FN void df_field(const DFGeo& G, const DFPair& P, DF2 L, DF2 LL, DF2 bt, DF2 be, const DFConst& K, Lanes far,
                    DF2& St, DF2& Se, DF2& Sn, DF2& cb)
{
    const Lanes one = {(G.y.h.x <= 0.0f) || (G.u2.h.x <= 0.0f), (G.y.h.y <= 0.0f) || (G.u2.h.y <= 0.0f)};
    const DF2 i1 = df_rsqrt(G.r1s), i2 = df_rsqrt(G.r2s);
    const DF2 m = df_mul(df_neg(G.y), i1), p = df_mul(G.u2, i2);
    const DF2 g12 = df_mul(i1, i2), i12 = df_sqr(g12);
    const DF2 ssum = df_add(df_sqr(i1), df_sqr(i2));
    const DF2 isum = df_add(i1, i2);
    const DF2 pm = df_mul(p, m);
    const DF2 pps = df_add(p, m);
    const DF2 S2 = df_add(df_sqr(pps), df_neg(pm));
    const DF2 opm = df_add_big(df_all(DF1{1.0f, 0.0f}), pm);
    const DF2 y2 = DF2{p_add(G.y.h, G.y.h), p_add(G.y.l, G.y.l)};
    const DF2 Li = df_mul(df_fma(df_neg(L), y2, LL), i12);  // L (u1 + u2) / (rho1^2 rho2^2)
    const DF2 E3 = df_add_big(ssum, g12);
    const DF2 Tt = df_mul(opm, isum);
    const DF2 den = df_sel(one, df_mul(pps, opm), G.d2);
    DF2 rr = df_rcp(df_mul(den, isum));
    rr = df_norm(df_sel(far, rr, DF2{p_all(0.0f), p_all(0.0f)}));
    const DF2 Aw = df_add_big(ssum, df_neg(df_mul(G.d2, i12)));
    const DF2 Z = df_fma_big(isum, Aw, df_mul(Tt, ssum));
    const DF2 Q = df_mul(Li, rr);
    const DF2 n0 = df_sel(one, Q, df_mul(df_sub(p, m), rr));
    const DF2 J0 = df_mul(n0, df_sel(one, Tt, isum));
    const DF2 J1 = df_mul(Q, den);
    const DF2 V = df_sel(one, Z, df_mul(df_add_big(df_all(DF1{3.0f, 0.0f}), df_neg(S2)), isum));
    const DF2 K2 = df_mul(df_sel(one, Q, df_mul(J0, rr)), V);
    const DF2 K3 = df_mul(J1, E3), K4 = df_mul(J0, S2);
    const DF2 B0 = df_fma_big(df_all(K.a2), K2, J0);
    const DF2 A0 = df_add_big(B0, J0);
    const DF2 C1 = df_fma(df_all(K.nra2), K3, df_mul(df_all(K.kn), J1));
    const DF2 rA0 = df_mul(df_all(K.nr), A0);
    const DF2 tb = df_all(P.tb), eb = df_all(P.eb), nb = df_all(P.nb);
    const DF2 Rb = df_fma(G.be, nb, df_mul(G.al, eb));           // Rp.b'
    const DF2 M = df_fma(df_neg(G.al), nb, df_mul(G.be, eb));
    const DF2 ga = df_mul(be, G.be);                             // -q.Rp
    const DF2 nqb = df_mul(be, nb);                              // -q.b'
    const DF2 K3n = df_neg(K3);
    const DF2 in1 = df_fma(K2, Rb, df_mul(K3n, tb));
    const DF2 cR = df_fma(df_neg(ga), in1, df_mul(J0, nqb));
    const DF2 Gx = df_mul(df_mul(rA0, tb), bt);         // bt c_Rxb
    const DF2 cq = df_fma(C1, tb, df_mul(df_neg(J0), Rb));
    const DF2 in3 = df_fma(K4, tb, df_mul(K3n, Rb));
    const DF2 ga2 = DF2{p_add(ga.h, ga.h), p_add(ga.l, ga.l)};
    const DF2 Mt = df_fma(df_neg(ga2), tb, df_mul(bt, M));       // Rw - be (Rp.n) t.b'
    Se = df_fma(Gx, G.be, df_mul(cR, G.al));
    Sn = df_fma(df_neg(cq), be, df_fma(df_neg(Gx), G.al, df_mul(cR, G.be)));
    St = df_fma(df_neg(ga), in3, df_fma(df_neg(C1), nqb, df_mul(rA0, Mt)));
    cb = df_mul(df_neg(ga), B0);
}

// The nodal force parts sum_q w_q (s_q x D) of a group of sources, from the group's sums s and
// b (the coefficient along b') at the Gauss points of chain ch (its two points are the
// lanes): F = start node's 3, end node's 3; chain 0 sets them, chain 1 adds.
DF_FN void df_group_forces(int ch, DF2 s[3], DF2 b, const DF2 bt[3], const DF1 D[3], DF2 F[6])
{
    const double x0 = gl4_xi(2 * ch), x1 = gl4_xi(2 * ch + 1), w0 = gl4_w(2 * ch), w1 = gl4_w(2 * ch + 1);
    const DF2 we = df_pair2(df_from(w0 * x0), df_from(w1 * x1));
    const DF2 ws = df_pair2(df_from(w0 * (1.0 - x0)), df_from(w1 * (1.0 - x1)));
#pragma unroll
    for (int e = 0; e < 3; ++e) s[e] = df_fma(b, bt[e], s[e]);
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const int i = (e + 1) % 3, j = (e + 2) % 3;
        const DF2 f = df_fma(s[i], df_all(D[j]), df_neg(df_mul(s[j], df_all(D[i]))));
        F[e] = ch ? df_fma(f, ws, F[e]) : df_mul(f, ws);
        F[3 + e] = ch ? df_fma(f, we, F[3 + e]) : df_mul(f, we);
    }
}

}  // namespace ptadd
