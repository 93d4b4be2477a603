// dp_loop.cu -- approximate optimal feedback (§3 Eq. (15)) and its closed
// loop (§3 "Computation of the approximate optimal solution").
//
// One warp per state or trajectory.  The feedback at a state y minimises
// tau + beta_tau I[V](y + tau Phi(y, alpha)): the lanes split the tabulated
// angles, a warp argmin (lowest index on ties) picks the tabulated minimiser,
// and the whole warp then takes the same golden-section (Fibonacci) refinement
// as the improvement sweep, several of its steps at a time.  The closed loop
// holds that angle over one classical RK4 step of the dynamics (FP64 state)
// and repeats until the state enters the target or the step budget ends.
//
// What bounds it: the serial chain of a step, not throughput (about seven
// warps an SM at 1,024 states).  1,024 trajectories of 100 steps on a 61^4 FP32
// grid: 2.23 ms with the refinement one evaluation after another and every
// lane doing all of the state's FP64 work (four divisions a right-hand side),
// 1.20 ms with the refinement in three rounds of the whole warp and each lane
// a component of the state.
#include "dp_host.h"
#include "dp_sweep.cuh"

namespace dpk {

// Component d = lane mod 4 of the dynamics at the state whose component d
// each lane holds in yd (the eight groups of four lanes repeat one another).
// The four quotients of a right-hand side are one division of the warp, each
// lane its own; all lanes dividing all four took the FP64 pipe (two lanes a
// clock) four times as long.
template <int DYN>
__device__ __forceinline__ double dyn64_lane(double yd, int d, double s, double c, double mu, double accel,
                                             double mdot, double drag)
{
    constexpr unsigned kAll = 0xffffffffu;
    if (DYN == kDynUnitSpeed) return d == 0 ? (fabs(c) < 1e-12 ? 0.0 : c) : d == 1 ? (fabs(s) < 1e-12 ? 0.0 : s) : 0.0;
    const double y0 = __shfl_sync(kAll, yd, 0, 4), y1 = __shfl_sync(kAll, yd, 1, 4), y2 = __shfl_sync(kAll, yd, 2, 4);
    // lane 0: mu / r^2, 1: v_t^2 / r, 2: -v_r v_t / r, 3: a / m (polar: v_t / r)
    const double num = d == 0 ? mu : d == 1 ? y2 * y2 : d == 2 ? -y1 * y2 : (DYN == kDynOrbit ? accel : y2);
    const double den = d == 0 ? y0 * y0 : (DYN == kDynOrbit && d == 3) ? yd : y0;
    const double q = num / den;
    const double grav = __shfl_sync(kAll, q, 0, 4);
    if (DYN == kDynOrbit) {
        const double am = __shfl_sync(kAll, q, 3, 4);
        return d == 0 ? y1 : d == 1 ? q - grav + am * s : d == 2 ? q + am * c : mdot;
    }
    // thrust off: s = c = 0; drag of the simulated system (Example 2 of §4)
    // with the printed components -C v_rho^2 and -C v_theta^2
    return d == 0 ? y1 : d == 1 ? q - grav + accel * s - drag * y1 * y1 : d == 2 ? q + accel * c - drag * y2 * y2 : q;
}

// fibonacci_refine() of one state by a whole warp, with the same result.  The
// sequential search evaluates one point a step, and which one depends on the
// values before it; here the lanes evaluate every point that the next steps
// can ask for (a binary tree of decisions: both first points and four steps in
// the first round, five steps in each later one), and the decisions then
// follow from the lanes' values: three rounds instead of sixteen evaluations
// in a row at K = 64.  Every lane holds the same state and returns the same.
template <class E, typename G>
__device__ __forceinline__ int fibonacci_refine_warp(E& ev, const Table<G>& T, int n0, int fib_stop, int k,
                                                     typename E::R Dk, typename E::R& Dbest)
{
    typedef typename E::R R;
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int ck = T.code[k];
    const int cl = (k == 0) ? T.code[T.K - 1] - kCodes : T.code[k - 1];
    const int hi_off = T.code[k + 1] - ck, L = hi_off - (cl - ck);
    int n = n0;
    while (kFib[n] < L) ++n;
    int a = cl - ck, kk = n, best = ck;
    R qb = Dk, f1 = ginf<R>(), f2 = ginf<R>();
    // The point a lane evaluates: its index below the leading one is a string
    // of `depth` decisions (0: keep the left part) of the steps from kk on.
    const int depth = 31 - __clz(lane | 1);
    bool first = true;
    bool pend = false;      // later rounds: the decision of step kk is known, its point is not evaluated
    while (first || pend) {
        int x, aa = a, q = kk;
        if (first) {
            x = lane == 0 ? a + kFib[n - 2] : a + kFib[n - 1];
        } else {
            const bool left = f1 <= f2;
            if (left) {
                x = aa + kFib[q - 3];
            } else {
                aa += kFib[q - 2];
                x = aa + kFib[q - 2];
            }
            --q;
        }
        for (int i = depth - 1; i >= 0 && q > 4 && kFib[q] > fib_stop; --i, --q) {
            if ((lane >> i) & 1) {
                aa += kFib[q - 2];
                x = aa + kFib[q - 2];
            } else {
                x = aa + kFib[q - 3];
            }
        }
        const bool skip = x >= hi_off || (E::kMayOff && T.off && wrap_code(ck + x) == kCodeOff);
        const R f = skip ? ginf<R>() : ev.at_code(ck + x);
        int node = 1, levels = first ? 4 : 5;
        if (first) {
            f1 = __shfl_sync(kAll, f, 0);
            f2 = __shfl_sync(kAll, f, 1);
            const int x1 = __shfl_sync(kAll, x, 0), x2 = __shfl_sync(kAll, x, 1);
            if (f1 < qb) { qb = f1; best = ck + x1; }
            if (f2 < qb) { qb = f2; best = ck + x2; }
        }
        for (int l = 0; l < levels && kk > 4 && kFib[kk] > fib_stop; ++l, --kk) {
            const bool left = f1 <= f2;
            if (first || l > 0) node = 2 * node + (left ? 0 : 1);
            const R fn = __shfl_sync(kAll, f, node);
            const int xn = __shfl_sync(kAll, x, node);
            if (left) {
                f2 = f1;
                f1 = fn;
            } else {
                a += kFib[kk - 2];
                f1 = f2;
                f2 = fn;
            }
            if (fn < qb) { qb = fn; best = ck + xn; }
        }
        first = false;
        pend = kk > 4 && kFib[kk] > fib_stop;
    }
    Dbest = qb;
    return wrap_code(best);
}

template <typename G, typename S>
__device__ __forceinline__ bool better(G a, int ka, G b, int kb)
{
    return a < b || (a == b && ka < kb);
}

template <typename G, typename S, bool REDUCED, int DYN>
__global__ void __launch_bounds__(128)
loop_kernel(const __grid_constant__ Geo<G> g, const __grid_constant__ LoopLaunch<G, S> a)
{
    __shared__ int s_code[kMaxAngles + 1];
    __shared__ typename V2<G>::type s_sc[kMaxAngles];
    build_table(g, s_code, s_sc);
    __syncthreads();
    const Table<G> T{s_code, s_sc, g.K, g.off};

    const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (w >= a.n) return;

    // lane d mod 4 = d holds component d of the state and of what belongs to it
    const int dl = lane & 3;
    auto pick4 = [&](auto v0, auto v1, auto v2, auto v3) { return dl == 0 ? v0 : dl == 1 ? v1 : dl == 2 ? v2 : v3; };
    double yd = a.x0[4 * w + dl];
    const double lo_d = pick4((double)g.lo[0], (double)g.lo[1], (double)g.lo[2], (double)g.lo[3]);
    const double h_d = pick4((double)g.h[0], (double)g.h[1], (double)g.h[2], (double)g.h[3]);
    const int n_d = pick4(g.n[0], g.n[1], g.n[2], g.n[3]);
    const double tc_d = pick4(a.tgt_c[0], a.tgt_c[1], a.tgt_c[2], a.tgt_c[3]);
    const double tw_d = pick4(a.tgt_w[0], a.tgt_w[1], a.tgt_w[2], a.tgt_w[3]);

    CachedEval<G, S, REDUCED, DYN> ev;
    ev.g = &g;
    ev.V = a.V;
    ev.sp.dt = (G)a.tau;
    ev.sp.hdt = (G)(0.5 * a.tau);
    ev.sp.um = (G)(a.tau * a.mdot / (double)g.h[3]);

    const long long steps = a.steps > 0 ? a.steps : 1;
    double t_arr = -1.0;
    for (long long step = 0; step < steps; ++step) {
        // --- feedback at y (Eq. (15)) ---
        constexpr unsigned kAll = 0xffffffffu;
        G x[4];
        double yw = yd;
        if (DYN == kDynPolar && dl == 3) {
            // the orbital angle keeps growing along a trajectory: wrap it
            const double per = h_d * n_d;
            yw = lo_d + (yd - lo_d) - per * floor((yd - lo_d) / per);
        }
        const double sd = (yw - lo_d) / h_d;
        double fl = floor(sd);
        fl = fmin(fmax(fl, -4.0), (double)n_d + 4.0);   // keep the index finite
        const int il = (int)fl;
        const G ul = (G)(sd - fl), xl = (G)yw;
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            x[d] = __shfl_sync(kAll, xl, d, 4);
            ev.i[d] = __shfl_sync(kAll, il, d, 4);
            ev.u0[d] = __shfl_sync(kAll, ul, d, 4);
        }
        ev.nd = node_dyn<G, DYN>(g, ev.sp, x);
        // compensation reference: the plain interpolated value at angle 0
        ev.vj = (S)0;
        ev.reset();
        ev.vj = (S)ev.at_code(0);
        ev.reset();          // cached corners are differences to the old vj

        typedef typename CachedEval<G, S, REDUCED, DYN>::R R;
        R Db = ginf<R>();
        int kb = 0x7fffffff;
        for (int k = lane; k < g.K; k += 32) {
            R D = ev.at_sc(T.sc[k].x, T.sc[k].y);
            if (better<R, S>(D, k, Db, kb)) { Db = D; kb = k; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            R Do = __shfl_xor_sync(0xffffffffu, Db, o);
            int ko = __shfl_xor_sync(0xffffffffu, kb, o);
            if (better<R, S>(Do, ko, Db, kb)) { Db = Do; kb = ko; }
        }
        int code = T.code[kb] & (kCodes - 1);
        if (g.refine) code = fibonacci_refine_warp(ev, T, g.fib_n0, g.fib_stop, kb, Db, Db);
        // running cost over tau (polar: Eq. (11); otherwise minimum time) and
        // the thrust-off control, which wins a tie
        double cost = a.tau, q = 0.0;
        if (DYN == kDynPolar) {
            double y4[4];
#pragma unroll
            for (int d = 0; d < 4; ++d) y4[d] = __shfl_sync(kAll, yw, d, 4);
            const double lx = a.tau * state_cost_x(g, y4);
            cost = lx + a.tau * (g.thrust_cost / g.dt64);
            q = cost + a.beta_tau * ((double)ev.vj + (double)Db);
            if (g.off) {
                const double q_off = lx + a.beta_tau * ((double)ev.vj + (double)ev.at_sc((G)0, (G)0));
                if (q_off <= q) {
                    q = q_off;
                    code = kCodeOff;
                }
            }
        } else {
            q = cost + a.beta_tau * ((double)ev.vj + (double)Db);
        }
        const bool off = g.off && code == kCodeOff;

        double2 hi = a.tab_hi64[code >> 8], lo = a.tab_lo64[code & 255];
        double s = off ? 0.0 : hi.x * lo.y + hi.y * lo.x;
        double c = off ? 0.0 : hi.y * lo.y - hi.x * lo.x;

        if (a.steps == 0) {
            if (lane == 0) {
                a.alpha[w] = off ? CUDART_NAN : 6.283185307179586476925286766559 * (double)code / (double)kCodes;
                if (a.q) a.q[w] = q;
            }
            return;
        }

        // --- one RK4 step of the dynamics with the angle held, each lane its component ---
        const double k1 = dyn64_lane<DYN>(yd, dl, s, c, a.mu, a.accel, a.mdot, a.drag);
        const double k2 = dyn64_lane<DYN>(yd + 0.5 * a.h * k1, dl, s, c, a.mu, a.accel, a.mdot, a.drag);
        const double k3 = dyn64_lane<DYN>(yd + 0.5 * a.h * k2, dl, s, c, a.mu, a.accel, a.mdot, a.drag);
        const double k4 = dyn64_lane<DYN>(yd + a.h * k3, dl, s, c, a.mu, a.accel, a.mdot, a.drag);
        yd = yd + a.h / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + k4);

        const bool in = !(tw_d > 0.0) || fabs(yd - tc_d) < tw_d;
        if (__all_sync(kAll, in)) { t_arr = (double)(step + 1) * a.h; break; }
    }
    if (lane == 0) a.t_arrive[w] = t_arr;
    if (lane < 4) a.x_final[4 * w + lane] = yd;
}

template <typename G, typename S>
static cudaError_t launch_loop_t(const LoopLaunch<G, S>& L)
{
    int threads = 128;
    long long blocks = ((long long)L.n * 32 + threads - 1) / threads;
    if (blocks < 1) return cudaSuccess;
    if (L.dyn == kDynUnitSpeed) {
        if (L.reduced) return cudaErrorInvalidValue;
        loop_kernel<G, S, false, kDynUnitSpeed><<<(unsigned)blocks, threads, 0, L.stream>>>(L.g, L);
    } else if (L.dyn == kDynPolar) {
        if (L.reduced || !std::is_same<G, double>::value) return cudaErrorInvalidValue;
        loop_kernel<G, S, false, kDynPolar><<<(unsigned)blocks, threads, 0, L.stream>>>(L.g, L);
    } else if (L.reduced) {
        loop_kernel<G, S, true, kDynOrbit><<<(unsigned)blocks, threads, 0, L.stream>>>(L.g, L);
    } else {
        loop_kernel<G, S, false, kDynOrbit><<<(unsigned)blocks, threads, 0, L.stream>>>(L.g, L);
    }
    return cudaGetLastError();
}

cudaError_t launch_loop(const LoopLaunch<double, double>& L) { return launch_loop_t(L); }
cudaError_t launch_loop(const LoopLaunch<float, float>& L) { return launch_loop_t(L); }
cudaError_t launch_loop(const LoopLaunch<float, double>& L) { return launch_loop_t(L); }

}  // namespace dpk
