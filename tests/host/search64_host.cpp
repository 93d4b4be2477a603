// FP64 angle searches decided by the FP32 model (dp_search64.cuh) against the
// searches that evaluate every angle, node by node on the CPU: the same code,
// the same bits of the value at it and the same frozen foot are asked for.
//
//   search64_host <seed> <count> <cells> <thrust> <angles> <polar> <reduced> <near>
//
// cells: largest displacement; thrust: its part that the angle moves (log
// uniform over a factor of 100 up to it); near: feet at a random table angle
// lie within this of a cell face (0: anywhere).  Prints the searches, those the
// model decided, and the mismatches.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "cuda_on_host.h"

#include "dp_search64.cuh"

using namespace dpk;

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

struct Args {
    long long count;
    double cells, thrust, near;
};

template <int DYN, bool REDUCED>
void run(const Args& a, int angles)
{
    constexpr bool kPolar = DYN == kDynPolar;
    typedef CachedEval<double, double, REDUCED, DYN, double, false, false> Eval;
    // one long dimension after another
    static const int kShapes[4][4] = {{1024, 6, 7, 5}, {6, 1024, 7, 5}, {7, 6, 1024, 4}, {6, 7, 5, 1024}};
    Geo<double> g;
    memset(&g, 0, sizeof g);
    std::vector<double2> hi(256), lo(256);
    for (int k = 0; k < 256; ++k) {
        const double x = 2.0 * M_PI * k / 256.0, y = 2.0 * M_PI * k / 65536.0;
        hi[k] = make_double2(sin(x), cos(x));
        lo[k] = make_double2(sin(y), cos(y));
    }
    g.tab_hi = hi.data();
    g.tab_lo = lo.data();
    g.M64 = 20.0;
    g.K = angles;
    g.refine = 1;
    std::vector<int> code(angles + 1);
    std::vector<double2> sc(angles);
    std::vector<float2> scf(angles);
    build_table(g, code.data(), sc.data(), scf.data());
    Table<double> T{code.data(), sc.data(), angles, 0, scf.data()};
    int shortest = 65536;
    for (int k = 0; k < angles; ++k)
        shortest = std::min(shortest, code[k + 1] - (k == 0 ? code[angles - 1] - kCodes : code[k - 1]));
    g.fib_n0 = 4;
    while (g.fib_n0 + 1 < kMaxFib && kFib[g.fib_n0 + 1] <= shortest) ++g.fib_n0;
    g.fib_stop = 3;

    long long model = 0, wrong = 0;
    std::vector<double> V;
    std::vector<int4> rows;
    for (long long it = 0; it < a.count; ++it) {
        if (it % std::max(1LL, a.count / 16) == 0) {
            const int* n = kShapes[kPolar ? below(4) : below(3)];
            for (int d = 0; d < 4; ++d) g.n[d] = n[d];
            g.n_m = n[3];
            g.stride[3] = 1;
            for (int d = 2; d >= 0; --d) g.stride[d] = g.stride[d + 1] * n[d + 1];
            g.n_nodes = g.stride[0] * n[0];
            rows.clear();
            if (REDUCED) {
                int at = 0;
                for (int r = 0; r < n[0] * n[1]; ++r) {
                    const int first = below(2), len = n[2] - first - below(2);
                    rows.push_back(make_int4(at, first, len, 0));
                    at += len * n[3];
                }
                g.n_nodes = at;
            }
            g.rows = rows.data();
            V.resize(g.n_nodes);
            for (double& v : V) v = uniform(0.0, g.M64);
        }
        Eval ev, plain;
        ev.g = &g;
        ev.V = V.data();
        ev.sp.um = 0.0;
        int long_dim = 0;
        for (int d = 0; d < 4; ++d) {
            if (g.n[d] == 1024) long_dim = d;
            ev.i[d] = below(g.n[d]);
            ev.u0[d] = 0.0;
        }
        const double um = uniform(-0.9, 0.0);
        ev.sp.um = um;
        g.um_c = (int)floor(um);
        g.um_t = um - floor(um);
        if (!kPolar) ev.i[3] = 1 + below(g.n[3] - 1);
        const double size = a.thrust * exp(uniform(-4.6, 0.0));
        NodeDyn<double>& nd = ev.nd;
        memset(&nd, 0, sizeof nd);
        nd.b0 = size * uniform(-1, 1);
        nd.b1 = size * uniform(-1, 1);
        nd.g1 = size * uniform(-1, 1);
        nd.d1 = size * size * uniform(-1, 1);
        nd.b2 = size * uniform(-1, 1) * 0.1;
        nd.g2 = size * uniform(-1, 1);
        nd.e2 = size * size * uniform(-1, 1);
        nd.g3 = kPolar ? size * uniform(-1, 1) : 0.0;
        // the displacement: long in the long dimension, to a cell of the box
        double u[4], want[4];
        const int at = below(angles);
        for (int d = 0; d < 4; ++d) {
            double whole;
            if (d == long_dim) whole = floor(uniform(-a.cells, a.cells));
            else whole = below(g.n[d] - 1) - ev.i[d];
            if (d == long_dim && !(kPolar && d == 3)) {
                whole = std::max(whole, (double)-ev.i[d]);
                whole = std::min(whole, (double)(g.n[d] - 2 - ev.i[d]));
            }
            const bool face = a.near > 0.0 && below(2) == 0;
            want[d] = whole + (face ? (below(2) ? 1.0 : 0.0) + a.near * uniform(-1, 1) : uniform(0.05, 0.95));
        }
        heun_cells<double, DYN>(g, ev.sp, nd, sc[at].x, sc[at].y, u);
        nd.a0 = want[0] - u[0];
        nd.a1 = want[1] - u[1];
        nd.a2 = want[2] - u[2];
        if (kPolar) nd.a3 = want[3] - u[3];
        ev.vj = uniform(0.0, g.M64);
        ev.reset();
        plain = ev;

        const int refine = below(4) != 0, walk = below(2), k0 = walk ? below(angles) : 0;
        double D = 0.0, Dp = 0.0;
        int got;
        FootHint fh;
        if (walk) got = search64<REDUCED, DYN, true>(ev, T, g, k0, refine != 0, D, fh);
        else got = search64<REDUCED, DYN, false>(ev, T, g, 0, refine != 0, D, fh);
        const int k = walk ? walk_table(plain, T, k0, Dp) : enumerate_table(plain, T, Dp);
        const int want_code = refine ? fibonacci_refine(plain, T, g.fib_n0, g.fib_stop, k, Dp, Dp) : T.code[k] & (kCodes - 1);
        model += fh.known;
        bool same = got == want_code && bits_as<long long>(D) == bits_as<long long>(Dp);
        if (fh.known) {
            double s, c, t[4];
            code_sincos(g, want_code, s, c);
            const unsigned long long w = plain.foot64_of(s, c, t);
            same = same && w == fh.w && ((w >> 32) != kFootInside || !memcmp(t, fh.t, sizeof t));
        }
        wrong += !same;
    }
    printf("%lld %lld %lld\n", a.count, model, wrong);
}

}  // namespace

int main(int argc, char** argv)
{
    if (argc != 9) return 2;
    g_state = strtoull(argv[1], nullptr, 10);
    Args a;
    a.count = atoll(argv[2]);
    a.cells = atof(argv[3]);
    a.thrust = atof(argv[4]);
    const int angles = atoi(argv[5]), polar = atoi(argv[6]), reduced = atoi(argv[7]);
    a.near = atof(argv[8]);
    if (polar) run<kDynPolar, false>(a, angles);
    else if (reduced) run<kDynOrbit, true>(a, angles);
    else run<kDynOrbit, false>(a, angles);
    return 0;
}
