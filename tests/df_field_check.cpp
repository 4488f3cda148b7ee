// Accuracy of df_field.cuh on the host, against the same field in 80-bit numbers.
// Built and read by test_df_field.py.  Prints, one per line,
//   split <largest error relative to the value> <mean signed error>
//   pair <kind> <median> <99 %> <largest error> of (sigma b') relative to |b||b'| int rho^-2 du
//   forces <loops> <error of the far pairs' nodal force parts relative to the largest>
// The reciprocal seeds carry an error of up to 1.5 units of their last bit, as
// the hardware's approximations do.
#include <cstdint>
static uint64_t g_state = 2005;
static uint64_t next_u64()
{
    uint64_t z = (g_state += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
static double uniform(double a, double b) { return a + (b - a) * (double)(next_u64() >> 11) * 0x1p-53; }
static float seed_error(float y) { return (float)(y * (1.0 + uniform(-1.0, 1.0) * 1.5 * 0x1p-23)); }
#define DF_HOST_SEED(y) seed_error(y)
#include "df_field.cuh"

#include <algorithm>
#include <cstdio>
#include <vector>

using namespace ptadd;
typedef long double ld;

static const double A2 = 1.0, NU = 0.34, SC = 1.0 / (1 << -DF_SCALE);
static const double NEAR = 32.0;  // in core widths, as the kernel's rule

struct Seg {
    double x1[3], x2[3], b[3], D[3], L, t[3];
    float x[9];
    DF1 T[3], E[3], N[3], l, ll, bt, be, d[3], bd[3];
    float near2;
};

// x in three parts: integer, multiple of 2^-23, rest
static void parts(double x, float* f)
{
    const double h = rint(x), r = x - h, m = rint(r * 0x1p23) * 0x1p-23;
    f[0] = (float)(h * SC);
    f[1] = (float)(m * SC);
    f[2] = (float)((r - m) * SC);
}

static Seg make_seg(const double x1[3], const double x2[3], const double b[3])
{
    Seg s;
    double LL = 0, e[3], n[3], bt = 0, vv = 0;
    for (int k = 0; k < 3; ++k) {
        s.x1[k] = x1[k], s.x2[k] = x2[k], s.b[k] = b[k], s.D[k] = x2[k] - x1[k];
        LL += s.D[k] * s.D[k];
        parts(x1[k], s.x + 3 * k);
    }
    s.L = sqrt(LL);
    for (int k = 0; k < 3; ++k) s.t[k] = s.D[k] / s.L, bt += b[k] * s.t[k];
    // e along the part of b normal to t (any normal if there is none), in long double
    ld v[3], tl[3], w = 0;
    for (int k = 0; k < 3; ++k) tl[k] = s.t[k];
    for (int k = 0; k < 3; ++k) v[k] = b[k] - bt * tl[k], vv += (double)(v[k] * v[k]);
    const double be = sqrt(vv) > 1e-17 ? sqrt(vv) : 0.0;
    if (be == 0.0) {
        const int m = fabs(s.t[0]) < 0.6 ? 0 : 1;
        for (int k = 0; k < 3; ++k) v[k] = (k == m) - tl[m] * tl[k];
    }
    for (int pass = 0; pass < 2; ++pass) {
        ld c = 0;
        for (int k = 0; k < 3; ++k) c += v[k] * tl[k];
        for (int k = 0; k < 3; ++k) v[k] -= c * tl[k];
    }
    for (int k = 0; k < 3; ++k) w += v[k] * v[k];
    for (int k = 0; k < 3; ++k) e[k] = (double)(v[k] / sqrtl(w));
    for (int k = 0; k < 3; ++k) n[k] = s.t[(k + 1) % 3] * e[(k + 2) % 3] - s.t[(k + 2) % 3] * e[(k + 1) % 3];
    for (int k = 0; k < 3; ++k) {
        s.T[k] = df_split(s.t[k]), s.E[k] = df_split(e[k]), s.N[k] = df_split(n[k]);
        s.d[k] = df_split(s.D[k] * SC), s.bd[k] = df_split(b[k]);
    }
    s.l = df_split(s.L * SC), s.ll = df_split(LL * SC * SC), s.bt = df_split(bt), s.be = df_split(be);
    s.near2 = std::max((float)(NEAR * NEAR * SC * SC * A2), s.ll.h / 256.0f);
    return s;
}

// (sigma b') / c2 at Gauss point q of T from S in 80 bits; its scale; squared distance to the source
static void field80(const Seg& T, int q, const Seg& S, ld s[3], ld& scale)
{
    ld t[3], L = 0, R[3], Rp[3], y = 0, d2 = A2, tb = 0, qb = 0, Rb = 0, qR = 0, Rw = 0, bb = 0, bp = 0;
    for (int k = 0; k < 3; ++k) t[k] = (ld)S.x2[k] - S.x1[k], L += t[k] * t[k];
    L = sqrtl(L);
    for (int k = 0; k < 3; ++k) t[k] /= L;
    for (int k = 0; k < 3; ++k) R[k] = T.x1[k] + (ld)gl4_xi(q) * ((ld)T.x2[k] - T.x1[k]) - S.x1[k], y += R[k] * t[k];
    for (int k = 0; k < 3; ++k) Rp[k] = R[k] - y * t[k], d2 += Rp[k] * Rp[k];
    const ld u2 = L - y, r1 = y * y + d2, r2 = u2 * u2 + d2, i1 = 1 / sqrtl(r1), i2 = 1 / sqrtl(r2);
    const ld m = -y * i1, p = u2 * i2, i12 = i1 * i1 * i2 * i2, ss = i1 * i1 + i2 * i2, S2 = p * p + m * m + p * m;
    const ld Li = L * (u2 - y) * i12, J1 = Li / (i1 + i2);
    const bool one = y <= 0 || y >= L;
    const ld J0 = one ? Li / (p + m) : (p - m) / d2;
    const ld K2 = J0 * (one ? (y * y + u2 * u2 + d2) * i12 / (1 + p * m) + ss : (3 - S2) / d2);
    const ld K3 = J1 * (i1 * i2 + ss), K4 = J0 * S2, r = -(1 - (ld)NU) / 2;
    const ld B0 = A2 * K2 + J0, A0 = B0 + J0, C1 = r * (A2 * K3 + 2 * J1) + J1;
    ld Q[3], X[3];
    for (int k = 0; k < 3; ++k) {
        const int i = (k + 1) % 3, j = (k + 2) % 3;
        Q[k] = S.b[i] * t[j] - S.b[j] * t[i];
        X[k] = Rp[i] * S.b[j] - Rp[j] * S.b[i];
    }
    for (int k = 0; k < 3; ++k) {
        tb += t[k] * T.b[k], qb += Q[k] * T.b[k], Rb += Rp[k] * T.b[k], qR += Rp[k] * Q[k], Rw += X[k] * T.b[k];
        bb += (ld)S.b[k] * S.b[k], bp += (ld)T.b[k] * T.b[k];
    }
    const ld cX = r * tb * A0, cq = C1 * tb - J0 * Rb, cR = qR * (K2 * Rb - K3 * tb) - J0 * qb;
    const ld ct = r * A0 * Rw + C1 * qb + qR * (K4 * tb - K3 * Rb), cb = qR * B0;
    for (int k = 0; k < 3; ++k) s[k] = cX * X[k] + cq * Q[k] + cR * Rp[k] + ct * t[k] + cb * T.b[k];
    const ld d = sqrtl(d2);
    scale = sqrtl(bb * bp) * (atanl(u2 / d) + atanl(y / d)) / d;
}

static DFConst constants()
{
    const double r = -(1 - NU) / 2;
    return DFConst{df_from(A2 * SC * SC), df_from(r), df_from(r * A2 * SC * SC), df_from(1 + 2 * r)};
}

// chain ch of the pair: frame components of (sigma b') / c2 and the lanes that are far
struct Chain {
    DF2 St, Se, Sn, cb;
    Lanes far;
};
static Chain chain(const Seg& T, const Seg& S, int ch)
{
    const DFConst K = constants();
    DF2 RD[3], t[3], e[3], n[3], bt[3];
    for (int k = 0; k < 3; ++k) {
        RD[k] = df_pair2(df_diff(T.x + 3 * k, S.x + 3 * k), T.d[k]);
        t[k] = df_all(S.T[k]), e[k] = df_all(S.E[k]), n[k] = df_all(S.N[k]), bt[k] = df_all(T.bd[k]);
    }
    DFPair P;
    P.y = df_dot(RD, t), P.al = df_dot(RD, e), P.be = df_dot(RD, n);
    const DF2 tb = df_dot(t, bt), eb = df_dot(e, bt), nb = df_dot(n, bt);
    P.tb = DF1{tb.h.x, tb.l.x}, P.eb = DF1{eb.h.x, eb.l.x}, P.nb = DF1{nb.h.x, nb.l.x};
    DFGeo G;
    df_geo(P, df_pair2(df_from(gl4_xi(2 * ch)), df_from(gl4_xi(2 * ch + 1))), df_all(S.l), K, G);
    const float near2 = std::max(T.near2, S.near2);
    const float dx = G.y.h.x < 0 ? G.r1s.h.x : G.u2.h.x < 0 ? G.r2s.h.x : G.d2.h.x;
    const float dy = G.y.h.y < 0 ? G.r1s.h.y : G.u2.h.y < 0 ? G.r2s.h.y : G.d2.h.y;
    Chain c;
    c.far = Lanes{!(dx < near2), !(dy < near2)};
    df_field(G, P, df_all(S.l), df_all(S.ll), df_all(S.bt), df_all(S.be), K, c.far, c.St, c.Se, c.Sn, c.cb);
    return c;
}

static double lane(DF2 a, int q) { return q ? (double)a.h.y + a.l.y : (double)a.h.x + a.l.x; }

static void direction(double v[3])
{
    double s;
    do {
        for (int k = 0; k < 3; ++k) v[k] = uniform(-1, 1);
        s = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
    } while (s < 0.05 || s > 1);
    for (int k = 0; k < 3; ++k) v[k] /= sqrt(s);
}

static void pairs(const char* kind, double d_lo, double d_hi, double l_lo, double l_hi, int screw, int edge)
{
    std::vector<double> err;
    while (err.size() < 40000) {
        double t[3], w[3], u[3], b[3], bp[3], x1[3], x2[3], y1[3], y2[3], c = 0;
        direction(t), direction(w), direction(u), direction(b), direction(bp);
        for (int k = 0; k < 3; ++k) c += w[k] * t[k];
        for (int k = 0; k < 3; ++k) w[k] -= c * t[k];  // normal to the source
        c = sqrt(w[0] * w[0] + w[1] * w[1] + w[2] * w[2]);
        const double L = exp(uniform(log(l_lo), log(l_hi))), Lt = exp(uniform(log(l_lo), log(l_hi)));
        const double d = exp(uniform(log(d_lo), log(d_hi)));
        // foot of the perpendicular: anywhere within two lengths, or at an end to 1e-4 of the length
        const double at = edge ? (next_u64() & 1 ? L : 0.0) + uniform(-1e-4, 1e-4) * L : uniform(-2.0, 3.0) * L;
        for (int k = 0; k < 3; ++k) {
            x1[k] = uniform(-2000, 2000);
            x2[k] = x1[k] + L * t[k];
            y1[k] = x1[k] + at * t[k] + d * w[k] / c;
            y2[k] = y1[k] + Lt * u[k];
            if (screw) b[k] = t[k] + (screw > 1 ? 1e-9 * w[k] : 0.0);
        }
        const Seg S = make_seg(x1, x2, b), T = make_seg(y1, y2, bp);
        for (int ch = 0; ch < 2; ++ch) {
            const Chain r = chain(T, S, ch);
            for (int h = 0; h < 2; ++h) {
                const bool far = h ? r.far.y : r.far.x;
                ld s[3], scale, e = 0;
                field80(T, 2 * ch + h, S, s, scale);
                for (int k = 0; k < 3; ++k) {
                    DF2 v = df_mul(r.St, df_all(S.T[k]));
                    v = df_fma(r.Se, df_all(S.E[k]), v);
                    v = df_fma(r.Sn, df_all(S.N[k]), v);
                    v = df_fma(r.cb, df_all(T.bd[k]), v);
                    const ld x = far ? lane(v, h) * SC - s[k] : (ld)lane(v, h);  // a near lane gives exactly 0
                    e += x * x;
                }
                if (far)
                    err.push_back((double)(sqrtl(e) / scale));
                else if (e != 0)
                    err.push_back(1.0);
            }
        }
    }
    std::sort(err.begin(), err.end());
    printf("pair %s %.3e %.3e %.3e\n", kind, err[err.size() / 2], err[err.size() * 99 / 100], err.back());
}

// nodal force parts of every segment from its far sources, in groups of 60 as the kernel sums them
static void forces(int loops, double edge)
{
    std::vector<Seg> g;
    for (int l = 0; l < loops; ++l) {
        double n[3], e1[3], e2[3], c[3], dot = 0;
        direction(n), direction(e1);
        for (int k = 0; k < 3; ++k) dot += n[k] * e1[k], c[k] = uniform(0, edge);
        double m = 0;
        for (int k = 0; k < 3; ++k) e1[k] -= dot * n[k], m += e1[k] * e1[k];
        for (int k = 0; k < 3; ++k) e1[k] /= sqrt(m);
        for (int k = 0; k < 3; ++k) e2[k] = n[(k + 1) % 3] * e1[(k + 2) % 3] - n[(k + 2) % 3] * e1[(k + 1) % 3];
        const int N = 24;
        const double R = uniform(200, 800), ph = uniform(0, 6);
        double x[N][3];
        for (int i = 0; i < N; ++i)
            for (int k = 0; k < 3; ++k)
                x[i][k] = c[k] + R * (cos(ph + 2 * M_PI * i / N) * e1[k] + sin(ph + 2 * M_PI * i / N) * e2[k]);
        for (int i = 0; i < N; ++i) g.push_back(make_seg(x[i], x[(i + 1) % N], e1));
    }
    ld off = 0, most = 0;
    for (const Seg& T : g) {
        DF2 sum[2][4] = {}, bt[3];
        double F[6] = {};
        ld E[6] = {};
        for (int k = 0; k < 3; ++k) bt[k] = df_all(T.bd[k]);
        for (size_t j = 0; j < g.size(); ++j) {
            const Seg& S = g[j];
            for (int ch = 0; ch < 2; ++ch) {
                const Chain r = chain(T, S, ch);
                for (int k = 0; k < 3; ++k) {
                    DF2& s = sum[ch][k];
                    s = df_fma(r.St, df_all(S.T[k]), s);
                    s = df_fma(r.Se, df_all(S.E[k]), s);
                    s = df_fma(r.Sn, df_all(S.N[k]), s);
                }
                sum[ch][3] = df_add(sum[ch][3], r.cb);
                for (int h = 0; h < 2; ++h) {
                    if (!(h ? r.far.y : r.far.x)) continue;
                    const int q = 2 * ch + h;
                    ld s[3], scale;
                    field80(T, q, S, s, scale);
                    for (int e = 0; e < 3; ++e) {
                        const int i = (e + 1) % 3, k = (e + 2) % 3;
                        const ld f = s[i] * T.D[k] - s[k] * T.D[i];
                        E[e] += (ld)gl4_w(q) * (1 - (ld)gl4_xi(q)) * f;
                        E[3 + e] += (ld)gl4_w(q) * gl4_xi(q) * f;
                    }
                }
            }
            if ((j + 1) % 60 == 0 || j + 1 == g.size()) {
                DF2 G[6];
                for (int ch = 0; ch < 2; ++ch) {
                    DF2 s[3] = {sum[ch][0], sum[ch][1], sum[ch][2]};
                    df_group_forces(ch, s, sum[ch][3], bt, T.d, G);
                    for (int k = 0; k < 4; ++k) sum[ch][k] = DF2{p_all(0.0f), p_all(0.0f)};
                }
                for (int k = 0; k < 6; ++k) F[k] += lane(G[k], 0) + lane(G[k], 1);  // c2 = 1; SC of the field and 1/SC of D cancel
            }
        }
        for (int k = 0; k < 6; ++k) off = std::max(off, fabsl(F[k] - E[k])), most = std::max(most, fabsl(E[k]));
    }
    printf("forces %d %.3e\n", loops, (double)(off / most));
}

int main()
{
    double worst = 0, mean = 0;
    const int n = 1000000;
    for (int i = 0; i < n; ++i) {
        const double x = uniform(1, 2) * ldexp(1.0, (int)(next_u64() % 40) - 20) * (next_u64() & 1 ? 1 : -1);
        const DF1 s = df_split(x);
        const double e = (((ld)s.h + s.l) - x) / x;
        worst = std::max(worst, fabs(e)), mean += e / n;
    }
    printf("split %.3e %.3e\n", worst, fabs(mean));
    const double odd[] = {0.0, 1e-300, 1e300, -1e300, INFINITY, -INFINITY};
    const float want[] = {0.0f, 0.0f, INFINITY, -INFINITY, INFINITY, -INFINITY};
    int bad = 0;
    for (int i = 0; i < 6; ++i) bad += df_round(odd[i]) != want[i];
    uint64_t nan_bits[] = {0x7FF8000000000000ull, 0xFFF8000000000000ull, 0x7FFFFFFFFFFFFFFFull, 0x7FF0000000000001ull};
    for (uint64_t u : nan_bits) {
        double x;
        memcpy(&x, &u, 8);
        bad += !(df_round(x) != df_round(x)) && u != 0x7FF0000000000001ull;  // (a payload below FP32's bits is lost)
    }
    bad += df_round(1.0 + 0x1p-24) != 1.0f + 0x1p-23f && df_round(1.0 + 0x1p-24) != 1.0f;
    bad += df_round(0x1.ffffffp0) != 2.0f;
    printf("round %d\n", bad);
    pairs("near_limit", 33, 64, 20, 300, 0, 0);
    pairs("middle", 64, 4000, 20, 1000, 0, 0);
    pairs("ends", 40, 4000, 20, 300, 0, 1);
    pairs("screw", 33, 4000, 20, 300, 1, 0);
    pairs("almost_screw", 33, 4000, 20, 300, 2, 0);
    pairs("long_source", 3000, 6000, 10000, 20000, 0, 0);
    pairs("range_limit", 4e5, 1.5e6, 100, 3000, 0, 0);
    forces(2, 1500);
    forces(16, 4000);
    return 0;
}
