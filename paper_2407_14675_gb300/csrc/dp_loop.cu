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
// A block takes a state per warp, up to kLoopWarps, and a warp the decision of
// each.  The FP64 work of a step (the state in grid units, the Runge-Kutta step,
// the polar running cost) is done for all of them by the block's first warp,
// four lanes a state.
//
// What bounds it: the serial chain of a step.  The FP64 pipe takes 16 clocks an
// instruction of a warp whatever lanes are in it, and at 1,024 states an SM has
// about seven: with a warp's FP64 for its own state only, the pipe took most of
// a step.  1,024 trajectories of 100 steps on a 61^4 FP32 grid: 2.23 ms with the
// refinement one evaluation after another and every lane doing all of the
// state's FP64 work (four divisions a right-hand side), 1.00 ms with the
// refinement in three rounds of the whole warp and each lane a component of its
// warp's state, 0.85 ms with eight states' components in one warp (5,000 of 60
// steps on 31^4: 2.21 and 1.61 ms; a single one, all latency, 7.9 us a step in
// either).
#include <climits>

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

constexpr int kLoopWarps = 8, kFeedbackWarps = 4;

template <typename G, typename S, bool REDUCED, int DYN>
__global__ void __launch_bounds__(32 * kLoopWarps, 1)
loop_kernel(const __grid_constant__ Geo<G> g, const __grid_constant__ LoopLaunch<G, S> a)
{
    static_assert(kLoopWarps * 4 == 32, "four lanes of the first warp a state");
    __shared__ int s_code[kMaxAngles + 1];
    __shared__ typename V2<G>::type s_sc[kMaxAngles];
    // per state: the node below it, its offset and coordinates (the decision's
    // inputs; kArrived in place of the index: none to take), the polar running
    // cost, the decided code
    constexpr int kArrived = INT_MIN;
    __shared__ int s_i[kLoopWarps][4], s_pick[kLoopWarps];
    __shared__ G s_u[kLoopWarps][4], s_x[kLoopWarps][4];
    __shared__ double s_cost[kLoopWarps];
    build_table(g, s_code, s_sc);
    __syncthreads();
    const Table<G> T{s_code, s_sc, g.K, g.off};

    constexpr unsigned kAll = 0xffffffffu;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, states = blockDim.x >> 5;
    const int w = blockIdx.x * states + warp;                      // the state this warp decides for
    const int own = blockIdx.x * states + (lane >> 2);             // first warp: the state of this lane

    // lane d mod 4 = d holds component d of the state and of what belongs to it
    const int dl = lane & 3;
    auto pick4 = [&](auto v0, auto v1, auto v2, auto v3) { return dl == 0 ? v0 : dl == 1 ? v1 : dl == 2 ? v2 : v3; };
    double yd = 0.0, lo_d = 0.0, h_d = 1.0, tc_d = 0.0, tw_d = 0.0;
    int n_d = 0;
    const bool mine = (lane >> 2) < states && own < a.n;
    bool live = mine;                                              // first warp: still flying
    if (warp == 0) {
        yd = a.x0[4 * (mine ? own : (int)blockIdx.x * states) + dl];
        lo_d = pick4((double)g.lo[0], (double)g.lo[1], (double)g.lo[2], (double)g.lo[3]);
        h_d = pick4((double)g.h[0], (double)g.h[1], (double)g.h[2], (double)g.h[3]);
        n_d = pick4(g.n[0], g.n[1], g.n[2], g.n[3]);
        tc_d = pick4(a.tgt_c[0], a.tgt_c[1], a.tgt_c[2], a.tgt_c[3]);
        tw_d = pick4(a.tgt_w[0], a.tgt_w[1], a.tgt_w[2], a.tgt_w[3]);
    }

    CachedEval<G, S, REDUCED, DYN> ev;
    ev.g = &g;
    ev.V = a.V;
    ev.sp.dt = (G)a.tau;
    ev.sp.hdt = (G)(0.5 * a.tau);
    ev.sp.um = (G)(a.tau * a.mdot / (double)g.h[3]);

    const long long steps = a.steps > 0 ? a.steps : 1;
    double t_arr = -1.0;
    for (long long step = 0; step < steps; ++step) {
        if (warp == 0) {
            double yw = yd;
            if (DYN == kDynPolar && dl == 3) {
                // the orbital angle keeps growing along a trajectory: wrap it
                const double per = h_d * n_d;
                yw = lo_d + (yd - lo_d) - per * floor((yd - lo_d) / per);
            }
            const double sd = (yw - lo_d) / h_d;
            double fl = floor(sd);
            fl = fmin(fmax(fl, -4.0), (double)n_d + 4.0);   // keep the index finite
            s_i[lane >> 2][dl] = live ? (int)fl : kArrived;
            s_u[lane >> 2][dl] = (G)(sd - fl);
            s_x[lane >> 2][dl] = (G)yw;
            if (DYN == kDynPolar) {
                // running cost over tau, Eq. (11)
                double y4[4];
#pragma unroll
                for (int d = 0; d < 4; ++d) y4[d] = __shfl_sync(kAll, yw, d, 4);
                const double lx = a.tau * state_cost_x(g, y4);
                if (dl == 0) s_cost[lane >> 2] = lx;
            }
        }
        // the states of this step; over once none of the block's flies
        if (!__syncthreads_or(warp == 0 && live)) break;

        // --- feedback at y (Eq. (15)); the warp of a state that has arrived waits:
        // on an FP64 grid its decision would take the pipe from the others' (200
        // steps of eight states an SM of which one flies on, 17^4: 3.9 ms, 8.9 with
        // the others deciding to the end) ---
        if (s_i[warp][0] != kArrived) {
            G x[4];
#pragma unroll
            for (int d = 0; d < 4; ++d) {
                x[d] = s_x[warp][d];
                ev.i[d] = s_i[warp][d];
                ev.u0[d] = s_u[warp][d];
            }
            ev.nd = node_dyn<G, DYN>(g, ev.sp, x);
            // compensation reference: the plain interpolated value at angle 0
            ev.vj = (S)0;
            ev.reset();
            ev.vj = (S)ev.at_code(0);
            ev.reset();          // cached corners are differences to the old vj

            typedef typename CachedEval<G, S, REDUCED, DYN>::R R;
            // (a lane without a better angle names its own index: where no angle
            // compares, as with values that a diverged sweep left NaN, index 0 wins)
            R Db = ginf<R>();
            int kb = lane;
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
            double q = 0.0;
            if (DYN == kDynPolar) {
                const double lx = s_cost[warp];
                const double cost = lx + a.tau * (g.thrust_cost / g.dt64);
                q = cost + a.beta_tau * ((double)ev.vj + (double)Db);
                if (g.off) {
                    const double q_off = lx + a.beta_tau * ((double)ev.vj + (double)ev.at_sc((G)0, (G)0));
                    if (q_off <= q) {
                        q = q_off;
                        code = kCodeOff;
                    }
                }
            } else if (a.steps == 0) {
                q = a.tau + a.beta_tau * ((double)ev.vj + (double)Db);
            }
            if (lane == 0) {
                if (a.steps == 0) {
                    a.alpha[w] = g.off && code == kCodeOff ? CUDART_NAN
                                                           : 6.283185307179586476925286766559 * (double)code / (double)kCodes;
                    if (a.q) a.q[w] = q;
                }
                s_pick[warp] = code;
            }
        }
        if (a.steps == 0) return;
        __syncthreads();   // the codes; the decisions have read their states

        // --- one RK4 step of the dynamics with the angle held, each lane its component ---
        if (warp == 0) {
            const int code = live ? s_pick[lane >> 2] : 0;
            const bool off = g.off && code == kCodeOff;
            const double2 hi = a.tab_hi64[code >> 8], lo = a.tab_lo64[code & 255];
            const double s = off ? 0.0 : hi.x * lo.y + hi.y * lo.x;
            const double c = off ? 0.0 : hi.y * lo.y - hi.x * lo.x;
            const double k1 = dyn64_lane<DYN>(yd, dl, s, c, a.mu, a.accel, a.mdot, a.drag);
            const double k2 = dyn64_lane<DYN>(yd + 0.5 * a.h * k1, dl, s, c, a.mu, a.accel, a.mdot, a.drag);
            const double k3 = dyn64_lane<DYN>(yd + 0.5 * a.h * k2, dl, s, c, a.mu, a.accel, a.mdot, a.drag);
            const double k4 = dyn64_lane<DYN>(yd + a.h * k3, dl, s, c, a.mu, a.accel, a.mdot, a.drag);
            const double yn = yd + a.h / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + k4);
            const bool in = !(tw_d > 0.0) || fabs(yn - tc_d) < tw_d;
            const unsigned at = __ballot_sync(kAll, in) >> (lane & ~3) & 15u;
            if (live) {
                yd = yn;
                if (at == 15u) {
                    t_arr = (double)(step + 1) * a.h;
                    live = false;
                }
            }
        }
    }
    if (warp == 0 && mine) {
        if (dl == 0) a.t_arrive[own] = t_arr;
        a.x_final[4 * own + dl] = yd;
    }
}

template <typename G, typename S>
static cudaError_t launch_loop_t(const LoopLaunch<G, S>& L)
{
    // States per block: as many as spread the states over the SMs (a decision on
    // an FP64 grid takes the SM's FP64 pipe, and 300 steps of 9 states there took
    // 5.4 ms in two blocks, 3.5 in nine), at most kLoopWarps, and for a decision
    // alone, whose shared FP64 work is a division, kFeedbackWarps
    const int most = L.steps > 0 ? kLoopWarps : kFeedbackWarps;
    int states = 1;
    while (states < most && (long long)states * L.sm_count < L.n) states *= 2;
    const int threads = 32 * states;
    const long long blocks = ((long long)L.n + states - 1) / states;
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
