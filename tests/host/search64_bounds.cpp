// The error bounds of the FP32 model of FP64 angle searches (dp_search64.cuh)
// against extended precision: how much of its bound each error takes.
//
//   search64_bounds <seed> <count> <angles> <polar>
//
// Nodes whose one-step map and corner values let one term after another
// dominate (each coefficient and each mixed difference of the corners is 0,
// small or large at random).  Prints the largest ratio of error to bound of
// the mean slopes, of the values over the table, of the fractions and of the
// FP64 evaluations themselves, and the angles looked at.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "cuda_on_host.h"

#include "dp_search64.cuh"

using namespace dpk;
typedef long double ld;

namespace {

unsigned long long g_state;
double uniform(double a, double b)
{
    g_state += 0x9e3779b97f4a7c15ull;   // SplitMix64 (Steele, Lea, Flood)
    unsigned long long z = g_state;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    z ^= z >> 31;
    return a + (b - a) * ((double)(z >> 11) / 9007199254740992.0);
}
int below(int n) { return std::min(n - 1, (int)uniform(0.0, n)); }
double term() { return uniform(-1.0, 1.0) * (below(3) == 0 ? 0.0 : exp(uniform(-9.0, 0.0))); }

template <int DYN>
void run(long long count, int angles)
{
    constexpr bool kPolar = DYN == kDynPolar;
    typedef CachedEval<double, double, false, DYN, double, false, false> Eval;
    Geo<double> g;
    memset(&g, 0, sizeof g);
    std::vector<double2> hi(256), lo(256);
    for (int k = 0; k < 256; ++k) {
        const ld x = 2.0L * M_PIl * k / 256.0L, y = 2.0L * M_PIl * k / 65536.0L;
        hi[k] = make_double2((double)sinl(x), (double)cosl(x));
        lo[k] = make_double2((double)sinl(y), (double)cosl(y));
    }
    g.tab_hi = hi.data();
    g.tab_lo = lo.data();
    g.M64 = 20.0;
    g.K = angles;
    std::vector<int> code(angles + 1);
    std::vector<double2> sc(angles);
    std::vector<float2> scf(angles);
    build_table(g, code.data(), sc.data(), scf.data());
    Table<double> T{code.data(), sc.data(), angles, 0, scf.data()};
    for (int d = 0; d < 4; ++d) g.n[d] = 4;
    g.n_m = 4;
    g.stride[3] = 1;
    for (int d = 2; d >= 0; --d) g.stride[d] = g.stride[d + 1] * 4;
    g.n_nodes = 256;
    std::vector<double> V(256);

    double worst[4] = {0.0, 0.0, 0.0, 0.0};
    long long looked = 0;
    for (long long it = 0; it < count; ++it) {
        Eval ev;
        ev.g = &g;
        ev.V = V.data();
        ev.vj = below(2) ? 0.0 : uniform(-2.0, 2.0);
        // corners: a multilinear form with coefficients of every size
        double coef[16];
        for (double& c : coef) c = term();
        if (below(2))
            for (int m = 1; m < 16; ++m)
                if (m & (m - 1)) coef[m] = 0.0;   // a linear field: nothing but rounding is left out
        for (int x = 0; x < 16; ++x) {
            double v = 0.0;
            for (int m = 0; m < 16; ++m)
                if ((m & x) == m) v += coef[m];
            V[(1 + (x & 1)) * g.stride[0] + (1 + (x >> 1 & 1)) * g.stride[1] + (1 + (x >> 2 & 1)) * g.stride[2] + 1 + (x >> 3)] = v;
        }
        NodeDyn<double>& nd = ev.nd;
        memset(&nd, 0, sizeof nd);
        const double size = exp(uniform(-9.0, 0.0));
        nd.b0 = size * term();
        nd.b1 = size * term();
        nd.g1 = size * term();
        nd.d1 = size * term();
        nd.b2 = size * term();
        nd.g2 = size * term();
        nd.e2 = size * term();
        if (kPolar) nd.g3 = size * term();
        const double far = exp(uniform(-2.0, 6.0));
        double* a[4] = {&nd.a0, &nd.a1, &nd.a2, &nd.a3};
        for (int d = 0; d < 4; ++d) {
            const double whole = floor(uniform(-far, far));
            ev.i[d] = 1 - (int)whole;
            ev.u0[d] = 0.0;
            *a[d] = whole + uniform(0.05, 0.95);
        }
        ev.sp.um = uniform(0.0, 1.0);
        if (!kPolar) ev.i[3] = 1;
        g.um_c = 0;
        g.um_t = ev.sp.um;
        ev.reset();

        Search64<Eval, false, DYN> S(ev);
        const int k0 = below(angles);
        if (S.start(T.sc[k0].x, T.sc[k0].y, 0.0f) != kSearchCell || !isfinite(S.eps)) continue;
        // exact fractions and D of a lattice code
        auto exact_t = [&](int c, ld t[4]) {
            const ld th = 2.0L * M_PIl * wrap_code(c) / 65536.0L, s = sinl(th), co = cosl(th);
            t[0] = (ld)nd.a0 + nd.b0 * s - (ld)ev.co[0];
            t[1] = (ld)nd.a1 + nd.b1 * s + co * (nd.g1 + nd.d1 * co) - (ld)ev.co[1];
            t[2] = (ld)nd.a2 + nd.b2 * s + co * (nd.g2 + nd.e2 * s) - (ld)ev.co[2];
            t[3] = kPolar ? (ld)nd.a3 + nd.g3 * co - (ld)S.co3 : 0.0L;
        };
        auto exact = [&](int c) {
            ld t[4], e[8];
            exact_t(c, t);
            for (int x = 0; x < 8; ++x) e[x] = kPolar ? (ld)ev.K.e0[x] + t[3] * ev.K.de[x] : (ld)ev.K.e0[x];
            for (int x = 0; x < 4; ++x) e[x] = e[2 * x] + t[2] * (e[2 * x + 1] - e[2 * x]);
            for (int x = 0; x < 2; ++x) e[x] = e[2 * x] + t[1] * (e[2 * x + 1] - e[2 * x]);
            return e[0] + t[0] * (e[1] - e[0]);
        };
        auto note = [&](int what, ld error, double bound) {
            const double r = (double)(fabsl(error) / (ld)bound);
            if (!(r <= worst[what])) worst[what] = r;
        };
        const int k = below(3) ? below(angles) : (k0 + below(5) - 2 + angles) % angles;
        const float s = T.scf[k].x, c = T.scf[k].y;
        if (!S.inside(s, c)) continue;
        ++looked;
        note(1, (ld)S.around(s, c) - ((ld)S.at_sc(T.sc[k].x, T.sc[k].y) - S.D0), S.eps);
        ld t[4];
        exact_t(T.code[k], t);
        // the fractions that inside() tests
        const float f[4] = {fmaf(S.b0, s, S.mid[0]), fmaf(S.b1, s, fmaf(c, fmaf(S.d1, c, S.g1), S.mid[1])),
                            fmaf(S.b2, s, fmaf(c, fmaf(S.e2, s, S.g2), S.mid[2])), fmaf(S.g3, c, S.mid[3])};
        for (int d = 0; d < (kPolar ? 4 : 3); ++d) note(2, (ld)f[d] - t[d], S.face);
        if (angles < kModelMinAngles) continue;
        const int xk = T.code[k], a0 = (k == 0 ? T.code[angles - 1] - kCodes : T.code[k - 1]) - xk, end = T.code[k + 1] - xk;
        if (!S.inside(s, c, kCodeAngle * (float)std::max(end, -a0) * 1.001f)) continue;
        const SlopeModel M = S.slopes(T, k);
        for (int q = 0; q < 6; ++q) {
            const int xa = q < 3 ? 0 : a0 + 1 + below(end - a0 - 1);
            int xb = a0 + 1 + below(end - a0 - 1);
            if (q % 3 == 2) xb = xa + 1 + below(4);
            if (xa == xb || xb >= end) continue;
            const ld diff = exact(xk + xb) - exact(xk + xa), got = (ld)S.at_code(xk + xb) - S.at_code(xk + xa);
            float err;
            const float mu = M.mean(xa, xb, err);
            note(0, (ld)mu - got / ((xb - xa) * (2.0L * M_PIl / 65536.0L)), err);
            note(3, got - diff, 2.0 * M.noise);
        }
    }
    printf("%.4f %.4f %.4f %.4f %lld\n", worst[0], worst[1], worst[2], worst[3], looked);
}

}  // namespace

int main(int argc, char** argv)
{
    if (argc != 5) return 2;
    g_state = strtoull(argv[1], nullptr, 10);
    const long long count = atoll(argv[2]);
    if (atoi(argv[4])) run<kDynPolar>(count, atoi(argv[3]));
    else run<kDynOrbit>(count, atoi(argv[3]));
    return 0;
}
