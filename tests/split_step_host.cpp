// Host build of the split RK4 step (iod_ff.cuh) and residuals (iod_ff_cost.cuh).  Prints, for
// groups of arguments (moon, mu, r, h, T), the root mean square position error over that of a
// plain FP64 RK4 (circular orbits about a primary, RK4 in long double as reference); the
// number of state components that words change; and the residuals' root mean square and
// largest error in rad, below 0.1 rad and over the circle.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

// stand for the hardware's estimates: x^(-1/2) and 1/x with relative errors up to 2^-23
static double off()
{
    static unsigned int state = 12345;
    state = state * 1664525u + 1013904223u;
    return 1.0 + ((state >> 8) / 8388608.0 - 1.0) * 0x1p-23;
}
static float rsqrt_estimate(float x) { return (float)(1.0 / std::sqrt((double)x) * off()); }
static float rcp_estimate(float x) { return (float)(1.0 / (double)x * off()); }
#define IOD_RSQRT_EST(x) rsqrt_estimate(x)
#define IOD_RCP_EST(x) rcp_estimate(x)
#include "iod_ff_cost.cuh"

using namespace iod::ff;
typedef long double Ref;

template <class T>
static void rhs(T mu, T omu, const T s[6], T d[6])
{
    const T d1 = s[0] + mu, d2 = s[0] - omu, yz = s[1] * s[1] + s[2] * s[2];
    const T r1 = d1 * d1 + yz, r2 = d2 * d2 + yz;
    const T g1 = omu / (r1 * std::sqrt(r1)), g2 = mu / (r2 * std::sqrt(r2)), gs = g1 + g2;
    d[0] = s[3];
    d[1] = s[4];
    d[2] = s[5];
    d[3] = s[0] + 2 * s[4] - g1 * d1 - g2 * d2;
    d[4] = s[1] - 2 * s[3] - gs * s[1];
    d[5] = -gs * s[2];
}

template <class T>
static void plain_step(T mu, T omu, T h, T s[6])
{
    T k1[6], k2[6], k3[6], k4[6], t[6];
    rhs(mu, omu, s, k1);
    for (int i = 0; i < 6; ++i) t[i] = s[i] + h / 2 * k1[i];
    rhs(mu, omu, t, k2);
    for (int i = 0; i < 6; ++i) t[i] = s[i] + h / 2 * k2[i];
    rhs(mu, omu, t, k3);
    for (int i = 0; i < 6; ++i) t[i] = s[i] + h * k3[i];
    rhs(mu, omu, t, k4);
    for (int i = 0; i < 6; ++i) s[i] += h / 6 * (k1[i] + 2 * (k2[i] + k3[i]) + k4[i]);
}

static void words(double omu, const State &S, Ref s[3])
{
    if (holds_fp64(S)) {
        double d[6];
        held_fp64(S, d);
        for (int i = 0; i < 3; ++i) s[i] = d[i];
        return;
    }
    s[0] = (Ref)S.ph.x + omu + S.pl.x + S.pc.x;
    s[1] = (Ref)S.ph.y + S.pl.y + S.pc.y;
    s[2] = (Ref)S.zh + S.zl + S.zc;
}

static double ratio(int moon, double mu, double r, double h, double T)
{
    const double omu = 1.0 - mu, mass = moon ? mu : omu;
    const int n = (int)std::lround(T / h), part = std::max(1, n / 10);
    const Mass M = make_mass(mu, omu);
    const float hf = (float)h, hl = (float)(h - (double)hf);
    const Step C = make_step(M, hf, hl);
    double e64 = 0, es = 0;
    for (int p = 0; p < 24; ++p) {
        std::mt19937_64 rng(100 + p);
        auto u = [&]() { return (double)(rng() >> 11) * 0x1p-52 - 1.0; };
        double a[3], b[3], q = 0, dot = 0, w = 0;
        for (double &x : a) q += (x = u()) * x;
        for (double &x : a) x /= std::sqrt(q);
        for (int i = 0; i < 3; ++i) dot += a[i] * (b[i] = u());
        for (int i = 0; i < 3; ++i) w += (b[i] -= dot * a[i]) * b[i];
        const double rr = r * (1 + 0.02 * u()), v = std::sqrt(mass / (rr * w));
        double s[6] = {rr * a[0] + (moon ? omu : -mu), rr * a[1], rr * a[2], v * b[0] + rr * a[1], v * b[1] - rr * a[0],
                       v * b[2]};
        Ref x[6];
        for (int i = 0; i < 6; ++i) x[i] = s[i];
        State S = to_state(omu, s);
        Grav G;
        float2 r2;
        bool anew = true;
        int taken = 0;
        for (int j = 1; j <= n; ++j) {
            plain_step<Ref>(mu, omu, h, x);
            plain_step<double>(mu, omu, h, s);
            if (anew && !holds_fp64(S)) attraction(M, S.ph, S.pl, S.zh, S.zl, G, r2);
            if (!holds_fp64(S) && split_ok(C.rmin, S, r2)) {
                rk4_step(M, C, S, G, r2);
                anew = carry_fails(C, r2);
                ++taken;
            } else {
                double d[6];
                from_state(omu, S, d);
                plain_step<double>(mu, omu, h, d);
                S = to_state(omu, d);
                anew = true;
            }
            if (j % part) continue;
            State Q = S;
            if (taken && !holds_fp64(S)) make_up(M, Q, G, (float)taken * (float)((h - (double)hf) - (double)hl));
            Ref y[3];
            words(omu, Q, y);
            for (int i = 0; i < 3; ++i) {
                e64 += (double)((s[i] - x[i]) * (s[i] - x[i]));
                es += (double)((y[i] - x[i]) * (y[i] - x[i]));
            }
        }
    }
    return std::sqrt(es / e64);
}

// to_state and back over random states: how many do not come back as they were
static int changed()
{
    std::mt19937_64 rng(1);
    int bad = 0;
    for (int k = 0; k < 200000; ++k) {
        double s[6], t[6];
        for (double &x : s) {
            x = (double)(rng() >> 11) * 0x1p-52 - 1.0;
            const int kind = (int)(rng() % 8);
            if (kind == 0) x = std::ldexp(x, -(int)(rng() % 160));
            if (kind == 1) x = std::ldexp(x, (int)(rng() % 160));
            if (kind == 2 && rng() % 8 == 0) x = 0.0;
        }
        const double omu = 1.0 - 0.5 * ((double)(rng() >> 11) * 0x1p-53);
        from_state(omu, to_state(omu, s), t);
        for (int i = 0; i < 6; ++i) bad += s[i] != t[i];
    }
    return bad;
}

// residuals of lines of sight within `width` of the observed angles, elevations up to 1.4
static void residual_errors(double width, double &rms, double &most)
{
    const Ref pi = 3.14159265358979323846264338327950288L;
    std::mt19937_64 rng(2);
    auto u = [&]() { return (double)(rng() >> 11) * 0x1p-52 - 1.0; };
    int n = 0;
    rms = most = 0;
    for (int i = 0; i < 200000; ++i) {
        const double ra = 3.1 * u(), dec = 1.3 * u(), a = ra + width * u(), el = dec + width * u();
        if (std::fabs(el) > 1.4) continue;
        const double ca = std::cos(ra), sa = std::sin(ra), cb = std::cos(dec), sb = std::sin(dec);
        Epoch E{};
        E.ok = 1;
        E.far2 = 1.0f;
        E.ka = mk2((float)ca, (float)sa);
        E.kal = mk2((float)(ca - (double)E.ka.x), (float)(sa - (double)E.ka.y));
        E.kb = mk2((float)cb, (float)sb);
        E.kbl = mk2((float)(cb - (double)E.kb.x), (float)(sb - (double)E.kb.y));
        const double x = 0.01 * std::cos(el) * std::cos(a), y = 0.01 * std::cos(el) * std::sin(a), z = 0.01 * std::sin(el);
        const float2 h = mk2((float)x, (float)y), l = mk2((float)(x - (double)h.x), (float)(y - (double)h.y));
        float2 bh, bl;
        float rh, rl;
        if (!residuals(E, h, l, (float)z, (float)(z - (double)(float)z), bh, bl, rh, rl)) continue;
        const Ref A = std::fabs(std::remainder((Ref)ra - std::atan2((Ref)y, (Ref)x), 2 * pi));
        const Ref B = std::fabs((Ref)dec - std::asin((Ref)z / std::sqrt((Ref)x * x + (Ref)y * y + (Ref)z * z)));
        const double e = (double)((Ref)bh.x + bl.x - A), f = (double)((Ref)bh.y + bl.y - B);
        rms += e * e + f * f;
        most = std::max(most, std::max(std::fabs(e), std::fabs(f)));
        n += 2;
    }
    rms = std::sqrt(rms / n);
}

int main(int argc, char **argv)
{
    for (int i = 1; i + 4 < argc; i += 5)
        std::printf("%.4f\n", ratio(std::atoi(argv[i]), std::atof(argv[i + 1]), std::atof(argv[i + 2]),
                                    std::atof(argv[i + 3]), std::atof(argv[i + 4])));
    std::printf("%d\n", changed());
    for (double width : {0.1, 3.1}) {
        double rms, most;
        residual_errors(width, rms, most);
        std::printf("%.3e\n%.3e\n", rms, most);
    }
    return 0;
}
