// dp_search64.cuh -- the angle searches of FP64 grids, with FP64 only where it
// decides.
//
// The FP64 pipe of this GPU runs two lanes a clock and SM, a 64th of the FP32
// rate, and a search over angles evaluates about twenty of them at a node.
// What a search needs from most of them is one bit: which of two angles is
// the better one.  Inside one cell the interpolated value along the control
// circle has a closed form, so that bit comes from an FP32 model of it with a
// bound on everything the model and the FP64 evaluations themselves leave
// out; where the difference is not clear of the bound the two angles are
// evaluated in FP64 as before.  Every decision is the one FP64 gives, so the
// chosen code, and the value at it (always evaluated in FP64), are the same
// bits.
//
// The model.  With s, c = sin, cos of the angle the foot's fractions are
//   t_d = mid_d + B_d s + C_d c + F_d s c + Q_d c^2       (dp_device.cuh)
// and D is multilinear in them: around the angle theta_0 with fractions t0,
//   D = D0 + sum_d G_d Dt_d + sum_{d<e} H_de Dt_d Dt_e + H_012 Dt_0 Dt_1 Dt_2.
// G (formed in FP64) gives f = S s + C c + F s c + Q c^2 along the circle; the
// H terms (smaller by the thrust's step in cells, about 1e-3) enter as a
// quadratic form in s - s0 and c - c0.  Table angles, at least two table steps
// of slope apart, are compared by the values this gives (around()).  The points
// of a refinement come as close as 1e-4 rad; they are compared by the mean
// slope between them, which for f over [m - h, m + h] (angles from the
// tabulated minimiser theta_k) is
//   sinc(h) (p cos m - q sin m) + sinc(2 h) (v cos 2m - w sin 2m),
//   p = S c_k - C s_k, q = S s_k + C c_k (FP64, then rounded),
//   v = F cos 2 theta_k - Q sin 2 theta_k, w = F sin 2 theta_k + Q cos 2 theta_k.
// A point counts only where its fractions are clear of the cell's faces.
//
// The bounds, with e = 6e-8 (2^-24) for an FP32 rounding and L_d = |B_d| + |C_d|
// + |F_d| + 2 |Q_d|, so that L_d times the distance |ds| + |dc| bounds a
// fraction's change, and X = |F| + 2 |Q| the part of it that is not linear:
//   f at table angles: S (ds) is S's rounding, the two sines' (e / 2 each, ds
//     up to 2), the product's and two sums': below 10 e |S|, 1e-6 is 16; F and
//     Q with three roundings each and differences of products up to 1: below
//     20 e, 4e-6 is 67;
//   slopes: p, cos m, the product, k1 and two sums, 8 e |p| (6e-7 is 10); q with
//     sin m of |m| <= 0.22 and m's own rounding, 12 e |m| |q| (8e-7 is 13); v and
//     w: F and Q 3 e each, the sine and cosine of 2 theta_k 2.5 e, which with
//     their own rounding leaves 13 e hypot(v, w), the evaluation 5 e, and sinc(2 h)
//     cut off after h^4, 64 h^6 / 5040 = 8e-7 of it for h = 0.2 (1.5e-6 is 25);
//   the H terms: their F and Q parts, sum H (2 L X + X^2) <= 3 Hs Ls X over the
//     circle (chords up to 2: twice 9 here) and, as a slope per radian, 6 Hs Ls X
//     of the distance along s and c, which is up to sqrt 2 of the arc (9); their
//     rounding, ten e of sum H L L (8e-6 Hs Ls), and that of ds and us at a
//     distance of nothing, 5 e of the form's coefficients (4e-7); the slope's
//     variation over [m - h, m + h], a third derivative of at most six times
//     those, h^2 / 6 of it (2 h^2); H_012: 8 L0 L1 L2 of the value (9), 3 L0 L1 L2
//     times the distance squared of the slope;
//   noise, the rounding of one FP64 evaluation (2^-53 = 1.1e-16): a displacement
//     is two roundings of itself and three of L_d, its angle's sine and cosine
//     3.5e-16 of L_d, a slope in a fraction at most 2 E0, so in three or four
//     fractions 1.8e-15 E0 um + 1.8e-15 E0 Ls + 0.9e-15 E0, and the blend 15 to 20
//     roundings of E0 (2.5e-15 E0 (um + 5 + Ls)).  E0 bounds the corners on both
//     sides of the angle coordinate, which an angle's evaluation blends anew.
// tests/host/search64_bounds.cpp measures how much of them the errors take: at
// most 0.97 (the H terms, whose bounds are attained), 0.74 by rounding and the
// series, 0.15 of the noise.
//
// Measured (GB300, with one-round blocks of 64): a value-iteration sweep of
// 17^4, 16 angles, 56 us (60 in a call of 50 sweeps, with its start and end),
// evaluating every angle 166; a walk sweep of a 31x41x25x17 box 0.33 against
// 1.17 ms, of the paper's 110x30^3 1.9 against 9.9 ms.  Before the one-step map's
// shared parts came from tables (node_dyn_table()) 78 us, 0.48 and 6.1 ms.
#pragma once

#include "dp_device.cuh"

namespace dpk {

constexpr float kCodeAngle = 9.5873799242852575e-05f;   // 2 pi / 65536
constexpr int kModelMinAngles = 30;   // refinements of tables at least this fine: brackets within 0.22 rad

// Mean slopes of D near a table angle theta_k.
struct SlopeModel {
    float p, q, v, w, sk, ck, ds, dc;   // ds, dc: sine and cosine of theta_k less those of theta_0
    float ass, asc, acc;                // quadratic form of the H terms, around theta_0
    float e0, e1, e2, noise;            // bound: e0 + e1 am + e2 h^2 + noise / h, am = |m| + h

    // Mean slope of D between the codes x_k + xa and x_k + xb, x_k the code of
    // theta_k, and its bound.
    __device__ __forceinline__ float mean(int xa, int xb, float& err) const
    {
        const float m = 0.5f * kCodeAngle * (float)(xa + xb), h = 0.5f * kCodeAngle * fabsf((float)(xb - xa));
        const float m2 = m * m, h2 = h * h;
        const float sn = m * fmaf(m2, fmaf(m2, 1.0f / 120.0f, -1.0f / 6.0f), 1.0f);
        const float c1 = m2 * fmaf(m2, fmaf(m2, -1.0f / 720.0f, 1.0f / 24.0f), -0.5f);   // cos m - 1
        const float cs = 1.0f + c1, s2 = 2.0f * sn * cs, c2 = fmaf(-2.0f * sn, sn, 1.0f);
        const float us = fmaf(sk, c1, ck * sn), uc = fmaf(ck, c1, -sk * sn);
        const float k1 = fmaf(h2, fmaf(h2, 1.0f / 120.0f, -1.0f / 6.0f), 1.0f);
        const float k2 = fmaf(h2, fmaf(h2, 16.0f / 120.0f, -4.0f / 6.0f), 1.0f);
        const float as = ds + us, ac = dc + uc;
        const float hq = fmaf(2.0f * ass, as, asc * ac) * (ck + uc) - fmaf(asc, as, 2.0f * acc * ac) * (sk + us);
        err = fmaf(fabsf(m) + h, e1, e0) + fmaf(e2, h2, __fdividef(noise, h));
        return fmaf(k1, fmaf(p, cs, -q * sn), fmaf(k2, fmaf(v, c2, -w * s2), hq));
    }
    // Sign of D(x_k + xb) - D(x_k + xa); 0: not decided.
    __device__ __forceinline__ int order(int xa, int xb) const
    {
        float err;
        const float mu = mean(xa, xb, err);
        if (!(fabsf(mu) > err)) return 0;
        return (mu > 0.0f) == (xb > xa) ? 1 : -1;
    }
};

enum { kSearchCell = 0,      // the foot is in a cell of the node set: the model holds there
       kSearchConst = 1,     // every foot near is outside: D is the penalty
       kSearchOpen = 2 };    // neither is certain: evaluate as usual

// The search at one node, on top of its FP64 evaluator E (CachedEval of a
// grid node).
template <class E, bool REDUCED, int DYN>
struct Search64 {
    static constexpr bool kPolar = DYN == kDynPolar;
    static constexpr int kDims = kPolar ? 4 : 3;    // fractions that move with the control
    E& ev;
    double co3;               // polar: offset of the angle coordinate's cell
    double D0, Sd, Cd;        // D at theta_0; S, C
    float s0, c0, S, C, F, Q;
    float b0, b1, g1, d1, b2, g2, e2, g3;
    float mid[4], face;       // constant part of the fractions; how near a face is too near
    float ass, asc, acc;
    float eps;                // bound of around() and the FP64 rounding of a difference
    float eh, et, noise;      // parts of the slopes' bound

    __device__ __forceinline__ Search64(E& e) : ev(e) {}

    // A bound of the largest magnitude, from the exponents and leading bits.
    static __device__ __forceinline__ float top(const double* v, int n)
    {
        unsigned b = 0;
#pragma unroll
        for (int x = 0; x < n; ++x) b = max(b, (unsigned)__double2hiint(v[x]) & 0x7fffffffu);
        return (float)__hiloint2double((int)(b + 1u), 0);
    }

    // Evaluates the angle (s0, c0).  kSearchConst: for every angle within
    // `reach` radians of it.
    __device__ __forceinline__ int start(double sd, double cd, float reach)
    {
        const Geo<double>& g = *ev.g;
        const NodeDyn<double>& nd = ev.nd;
        double u[4], t[4], fl[4];
        int cl[4];
        float tf[4], uf[4];
        heun_cells<double, DYN>(g, ev.sp, nd, sd, cd, u);
        b0 = (float)nd.b0, b1 = (float)nd.b1, g1 = (float)nd.g1, d1 = (float)nd.d1;
        b2 = (float)nd.b2, g2 = (float)nd.g2, e2 = (float)nd.e2, g3 = kPolar ? (float)nd.g3 : 0.0f;
        const float L[4] = {fabsf(b0), fabsf(b1) + fabsf(g1) + 2.0f * fabsf(d1), fabsf(b2) + fabsf(g2) + fabsf(e2), fabsf(g3)};
        // How near a face is too near.  The fractions come from the FP32
        // displacement, off by up to 6e-8 of it (2^-24): 3.1e-5 of a cell at 512
        // cells.  It enters every angle's fractions through mid[], so it is in
        // the margin of all of them, not of the first angle alone.  The rest: a
        // fraction is at most nine FP32 roundings of terms up to L[d] and five
        // of sums up to 1 + L[d], 6e-8 each.
        float um = 0.0f;
#pragma unroll
        for (int d = 0; d < kDims; ++d) {
            uf[d] = (float)u[d];
            um = fmaxf(um, fabsf(uf[d]));
        }
        face = fmaf(3e-7f, um, 4e-6f * (1.0f + L[0] + L[1] + L[2] + L[3]));
        // cell and fractions: the cell from the FP32 displacement, which decides
        // it wherever the fraction is clear of a face
        bool in = true, in_all = true, box = !ev.outm, far = ev.outm;
#pragma unroll
        for (int d = 0; d < kDims; ++d) {
            const float fi = floorf(uf[d]), r = fmaf(1.001f * reach, L[d], face);
            fl[d] = (double)fi;
            t[d] = u[d] - fl[d];
            tf[d] = uf[d] - fi;
            cl[d] = ev.i[d] + (int)fi;
            in = in && tf[d] > face && tf[d] < 1.0f - face;
            in_all = in_all && tf[d] > r && tf[d] < 1.0f - r;
            if (d < 3) {
                box = box && (unsigned)cl[d] <= (unsigned)(g.n[d] - 2);
                const float pos = (float)ev.i[d] + uf[d], rp = r + 1e-3f;
                far = far || pos < -rp || pos > (float)(g.n[d] - 1) + rp;
            } else {
                cl[d] = cl[d] % g.n[d];   // the periodic angle
                if (cl[d] < 0) cl[d] += g.n[d];
            }
        }
        if (!kPolar) {
            cl[3] = ev.cm;
            t[3] = ev.tm;
            tf[3] = 0.5f;
        }
        if (far) return kSearchConst;
        if (!in || !box) return kSearchOpen;
        s0 = (float)sd;
        c0 = (float)cd;
        mid[0] = tf[0] - b0 * s0;
        mid[1] = tf[1] - fmaf(b1, s0, c0 * fmaf(d1, c0, g1));
        mid[2] = tf[2] - fmaf(b2, s0, c0 * fmaf(e2, s0, g2));
        mid[3] = kPolar ? tf[3] - g3 * c0 : 0.0f;
        ev.cout = load_corners<double, double, double, REDUCED, kPolar>(g, ev.V, cl, ev.vj, ev.K);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            ev.cc[d] = cl[d];
            ev.co[d] = fl[d];
        }
        if (kPolar) {
            ev.cm = cl[3];
            co3 = fl[3];
        } else {
            ev.K.fold_m(ev.tm);
        }
        if (ev.cout) return in_all ? kSearchConst : kSearchOpen;

        // D0 with the blend's operations, and the derivatives in the fractions
        double e[8], w[4], f[4];
#pragma unroll
        for (int x = 0; x < 8; ++x) e[x] = kPolar ? ev.K.e0[x] + t[3] * ev.K.de[x] : ev.K.e0[x];
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            w[y] = e[2 * y + 1] - e[2 * y];
            f[y] = e[2 * y] + t[2] * w[y];
        }
        const double v0 = f[1] - f[0], v1 = f[3] - f[2];
        const double h0 = f[0] + t[1] * v0, h1 = f[2] + t[1] * v1, G0 = h1 - h0;
        D0 = h0 + t[0] * G0;
        const double H01 = v1 - v0, G1 = v0 + t[0] * H01;
        const double wa = w[1] - w[0], wb = w[3] - w[2];
        const double x0 = w[0] + t[1] * wa, x1 = w[2] + t[1] * wb, H02 = x1 - x0, G2 = x0 + t[0] * H02;
        const double H012 = wb - wa, H12 = wa + t[0] * H012;
        float E3 = 0.0f;
        Sd = G0 * nd.b0 + G1 * nd.b1 + G2 * nd.b2;
        Cd = G1 * nd.g1 + G2 * nd.g2;
        if (kPolar) {
            // the angle coordinate: its derivative, the blend of the steps along it
            double df[4];
#pragma unroll
            for (int y = 0; y < 4; ++y)
                df[y] = ev.K.de[2 * y] + t[2] * (ev.K.de[2 * y + 1] - ev.K.de[2 * y]);
            const double a0 = df[0] + t[1] * (df[1] - df[0]), a1 = df[2] + t[1] * (df[3] - df[2]);
            Cd += (a0 + t[0] * (a1 - a0)) * nd.g3;
            // and what is left out: how that derivative varies over the cell
            double de[8];
#pragma unroll
            for (int x = 0; x < 8; ++x) de[x] = ev.K.de[x] - ev.K.de[0];
            E3 = top(de, 8);
        }
        S = (float)Sd;
        C = (float)Cd;
        F = (float)G2 * e2;
        Q = (float)G1 * d1;
        const float h01 = (float)H01, h02 = (float)H02, h12 = (float)H12, h012 = fabsf((float)H012);
        ass = h01 * b0 * b1 + h02 * b0 * b2 + h12 * b1 * b2;
        asc = h01 * b0 * g1 + h02 * b0 * g2 + h12 * (b1 * g2 + g1 * b2);
        acc = h12 * g1 * g2;
        // largest corner difference, from the exponents and leading bits (the
        // angle coordinate is blended for every angle: its corners on both sides,
        // which may cancel at this fraction)
        const float E0 = top(e, 8) + (kPolar ? top(ev.K.de, 8) : 0.0f);
        const float Hs = fabsf(h01) + fabsf(h02) + fabsf(h12), Ls = L[0] + L[1] + L[2], X = 2.0f * fabsf(d1) + fabsf(e2);
        // below FP32's range the bounds would not hold (a flat value: all ties)
        if (!(E0 * Ls > 1e-20f)) return kSearchOpen;
        const float hh = Hs * Ls;
        // slopes, per radian from theta_0: the H terms' rounding and F, Q parts, the angle coordinate's cross terms
        eh = fmaf(8e-6f * hh, Ls, 9.0f * hh * X) + 16.0f * E3 * L[3] * Ls;
        et = 3.0f * h012 * L[0] * L[1] * L[2];   // and H_012, per radian squared
        noise = 2.5e-15f * E0 * (um + 5.0f + Ls);   // half the rounding of a difference: slopes are at most 2 E0
        eps = fmaf(1e-6f, fabsf(S) + fabsf(C), 4e-6f * (fabsf(F) + fabsf(Q))) + 2.0f * eh + 3.0f * et + 2.0f * noise;
        return kSearchCell;
    }

    // D(s, c) - D0 within eps, where inside(s, c).
    __device__ __forceinline__ float around(float s, float c) const
    {
        const float ds = s - s0, dc = c - c0;
        const float fq = fmaf(F, fmaf(s, c, -s0 * c0), Q * dc * (c + c0));
        return fmaf(S, ds, fmaf(C, dc, fq)) + fmaf(fmaf(ass, ds, asc * dc), ds, acc * dc * dc);
    }
    // The foot keeps `face` from the cell's faces, and all that is within
    // `reach` radians of it does.
    __device__ __forceinline__ bool inside(float s, float c, float reach = 0.0f) const
    {
        const float t0 = fmaf(b0, s, mid[0]), t1 = fmaf(b1, s, fmaf(c, fmaf(d1, c, g1), mid[1]));
        const float t2 = fmaf(b2, s, fmaf(c, fmaf(e2, s, g2), mid[2]));
        const float r0 = fmaf(reach, fabsf(b0), face), r1 = fmaf(reach, fabsf(b1) + fabsf(g1) + fabsf(d1), face);
        const float r2 = fmaf(reach, fabsf(b2) + fabsf(g2) + fabsf(e2), face);
        bool in = t0 > r0 && t0 < 1.0f - r0 && t1 > r1 && t1 < 1.0f - r1 && t2 > r2 && t2 < 1.0f - r2;
        if (kPolar) {
            const float t3 = fmaf(g3, c, mid[3]), r3 = fmaf(reach, fabsf(g3), face);
            in = in && t3 > r3 && t3 < 1.0f - r3;
        }
        return in;
    }

    // D in FP64 at an angle or code inside the cell: the evaluator's fast path.
    __device__ __forceinline__ double at_sc(double s, double c) const
    {
        double t[4];
        fractions(s, c, t);
        return blend(t);
    }
    __device__ __forceinline__ double blend(const double t[4]) const
    {
        return kPolar ? ev.K.blend(t) : ev.K.blend_m_folded(t);
    }
    // Word of a frozen foot in this cell, as CachedEval::foot64_of() forms it.
    __device__ __forceinline__ unsigned long long foot_word() const
    {
        unsigned long long w = (unsigned long long)kFootInside << 32;
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            const int off = (d < 3 ? ev.cc[d] : ev.cm) - ev.i[d];
            if (off < -128 || off > 127) return (unsigned long long)kFootRecompute << 32;
            w |= (unsigned long long)(unsigned char)(signed char)off << (8 * d);
        }
        return w;
    }
    __device__ __forceinline__ double at_code(int code) const
    {
        double s, c;
        code_sincos(*ev.g, code, s, c);
        return at_sc(s, c);
    }
    __device__ __forceinline__ void fractions(double s, double c, double t[4]) const
    {
        double u[4];
        heun_cells<double, DYN>(*ev.g, ev.sp, ev.nd, s, c, u);
#pragma unroll
        for (int d = 0; d < 3; ++d) t[d] = u[d] - ev.co[d];
        t[3] = kPolar ? u[3] - co3 : ev.tm;
    }

    // enumerate_table() after start(T.sc[0]): only the angles that may be the
    // lowest are evaluated in FP64.  False where some angle leaves the cell.
    __device__ __forceinline__ bool enumerate(const Table<double>& T, int& kb, double& D) const
    {
        float lo = 0.0f;                 // around(angle 0)
        bool in = isfinite(eps);
        for (int k = 1; k < T.K; ++k) {
            const float s = T.scf[k].x, c = T.scf[k].y;
            in = in && inside(s, c);
            lo = fminf(lo, around(s, c));
        }
        if (!in) return false;
        const float lim = lo + 2.0f * eps;
        double Db = CUDART_INF;
        kb = 0;
        for (int k = 0; k < T.K; ++k) {
            while (k < T.K && !((k == 0 ? 0.0f : around(T.scf[k].x, T.scf[k].y)) <= lim)) ++k;
            if (k >= T.K) break;
            const double Dk = at_sc(T.sc[k].x, T.sc[k].y);
            if (Dk < Db) { Db = Dk; kb = k; }
        }
        D = Db;
        return true;
    }

    // walk_table() after start() at its first angle k, with its result.  False
    // where the walk leaves the cell.
    __device__ __forceinline__ bool walk(const Table<double>& T, int& k) const
    {
        const int K = T.K;
        auto value = [&](int kk, bool& in) {
            const float s = T.scf[kk].x, c = T.scf[kk].y;
            in = in && inside(s, c);
            return around(s, c);
        };
        // D(a) < D(b) (or <=) given around()'s values
        auto lower = [&](int a, float va, int b, float vb, bool or_equal) {
            if (fabsf(va - vb) > 2.0f * eps) return va < vb;
            double D[2];
#pragma unroll 1
            for (int r = 0; r < 2; ++r) {
                const int kk = r ? b : a;
                const double x = at_sc(T.sc[kk].x, T.sc[kk].y);
                if (r) D[1] = x;
                else D[0] = x;
            }
            return or_equal ? D[0] <= D[1] : D[0] < D[1];
        };
        bool in = isfinite(eps);
        int kl = k == 0 ? K - 1 : k - 1, kr = k == K - 1 ? 0 : k + 1;
        float vk = 0.0f, vl = value(kl, in), vr = value(kr, in);
        for (int step = 0; in && step < K; ++step) {
            const bool lo_l = lower(kl, vl, k, vk, false), lo_r = lower(kr, vr, k, vk, false);
            if (!lo_l && !lo_r) break;
            // left wins a tie between neighbours
            if (lo_l && (!lo_r || lower(kl, vl, kr, vr, true))) {
                kr = k; vr = vk;
                k = kl; vk = vl;
                kl = k == 0 ? K - 1 : k - 1;
                vl = value(kl, in);
            } else {
                kl = k; vl = vk;
                k = kr; vk = vr;
                kr = k == K - 1 ? 0 : k + 1;
                vr = value(kr, in);
            }
        }
        return in;
    }

    // The slopes around table angle k.
    __device__ __forceinline__ SlopeModel slopes(const Table<double>& T, int k) const
    {
        SlopeModel M;
        const double sd = T.sc[k].x, cd = T.sc[k].y;
        M.sk = T.scf[k].x;
        M.ck = T.scf[k].y;
        M.p = (float)(Sd * cd - Cd * sd);
        M.q = (float)(Sd * sd + Cd * cd);
        const float c2 = fmaf(-2.0f * M.sk, M.sk, 1.0f), s2 = 2.0f * M.sk * M.ck;
        M.v = fmaf(F, c2, -Q * s2);
        M.w = fmaf(F, s2, Q * c2);
        M.ds = M.sk - s0;
        M.dc = M.ck - c0;
        M.ass = ass; M.asc = asc; M.acc = acc;
        const float far = fabsf(M.ds) + fabsf(M.dc);   // at least the distance along s and c
        const float vw = fabsf(M.v) + fabsf(M.w);
        M.e1 = fmaf(8e-7f, fabsf(M.q), eh) + et * (far + 0.5f) * 3.0f;
        const float A = fabsf(ass) + fabsf(asc) + fabsf(acc);
        M.e0 = fmaf(1.5e-6f, vw, fmaf(6e-7f, fabsf(M.p), 4e-7f * A)) + far * fmaf(et, far, eh);
        M.e2 = 2.0f * A;
        M.noise = noise;
        return M;
    }

    // fibonacci_refine() from table angle k, with its result: the chosen code.
    // False where the bracket reaches out of the cell.
    __device__ __forceinline__ bool refine(const Table<double>& T, int n0, int fib_stop, int k, int& code) const
    {
        const int xk = T.code[k];
        const int a0 = (k == 0 ? T.code[T.K - 1] - kCodes : T.code[k - 1]) - xk, hi = T.code[k + 1] - xk, L = hi - a0;
        if (!inside(T.scf[k].x, T.scf[k].y, kCodeAngle * (float)max(hi, -a0) * 1.001f)) return false;
        const SlopeModel M = slopes(T, k);
        // D(xk + xb) < D(xk + xa) (or <=)
        auto better = [&](int xb, int xa, bool or_equal) {
            const int o = M.order(xa, xb);
            if (o != 0) return o < 0;
            double D[2];
#pragma unroll 1
            for (int r = 0; r < 2; ++r) {
                const double x = at_code(xk + (r ? xb : xa));
                if (r) D[1] = x;
                else D[0] = x;
            }
            return or_equal ? D[1] <= D[0] : D[1] < D[0];
        };
        auto inf = [&](int x) { return x >= hi || (E::kMayOff && T.off && wrap_code(xk + x) == kCodeOff); };
        int n = n0;
        while (kFib[n] < L) ++n;
        int best = 0, a = a0, x1 = a + kFib[n - 2], x2 = a + kFib[n - 1];
        bool i1 = inf(x1), i2 = inf(x2);
        if (!i1 && better(x1, best, false)) best = x1;
        if (!i2 && better(x2, best, false)) best = x2;
        for (int kk = n; kk > 4 && kFib[kk] > fib_stop; --kk) {
            const bool left = i2 || (!i1 && better(x1, x2, true));   // f1 <= f2
            int xn;
            if (left) {
                x2 = x1;
                i2 = i1;
                xn = x1 = a + kFib[kk - 3];
            } else {
                a = x1;
                x1 = x2;
                i1 = i2;
                xn = x2 = a + kFib[kk - 2];
            }
            const bool in = inf(xn);
            if (left) i1 = in;
            else i2 = in;
            if (!in && better(xn, best, false)) best = xn;
        }
        code = wrap_code(xk + best);
        return true;
    }
};

// The frozen foot of the chosen code, where the search has it.
struct FootHint {
    bool known = false;
    unsigned long long w;
    double t[4];
};

// The search of a node of an FP64 grid: the chosen code and D at it, as
// walk_table() from k0 (WALK) or enumerate_table() and then, with refine,
// fibonacci_refine() give them.
template <bool REDUCED, int DYN, bool WALK, class E>
__device__ __forceinline__ int search64(E& ev, const Table<double>& T, const Geo<double>& g, int k0, bool refine,
                                        double& D, FootHint& fh)
{
    int k = WALK ? k0 : 0;
    const bool fine = !refine || T.K >= kModelMinAngles;
    if (fine) {
        Search64<E, REDUCED, DYN> S(ev);
        // the walk and the refinement look one table step to either side, the table all round
        const float step = WALK || refine ? 6.2831855f / (float)T.K + 2.0f * kCodeAngle : 0.0f;
        const int how = S.start(T.sc[k].x, T.sc[k].y, WALK ? step : 2.0f);
        if (how == kSearchConst) {
            D = ev.pen;   // nothing is lower than anything
            fh.known = true;
            fh.w = (unsigned long long)kFootOut << 32;
            fh.t[0] = fh.t[1] = fh.t[2] = fh.t[3] = 0.0;
            return T.code[k] & (kCodes - 1);
        }
        if (how == kSearchCell) {
            int code;
            bool ok;
            if (WALK) ok = S.walk(T, k);
            else ok = S.enumerate(T, k, D);
            if (ok && !refine) {
                if (WALK) D = k == k0 ? S.D0 : S.at_sc(T.sc[k].x, T.sc[k].y);
                return T.code[k] & (kCodes - 1);
            }
            if (ok && S.refine(T, g.fib_n0, g.fib_stop, k, code)) {
                double s, c;
                code_sincos(g, code, s, c);
                S.fractions(s, c, fh.t);
                D = S.blend(fh.t);
                fh.known = true;
                fh.w = S.foot_word();
                return code;
            }
        }
    }
    k = WALK ? walk_table(ev, T, k0, D) : enumerate_table(ev, T, D);
    if (!refine) return T.code[k] & (kCodes - 1);
    return fibonacci_refine(ev, T, g.fib_n0, g.fib_stop, k, D, D);
}

}  // namespace dpk
