// dp_gmres.cu -- policy evaluation by restarted GMRES.
//
// §3, after Eq. (14): with the control frozen, the evaluation step of policy
// iteration (Eq. (13)) is a linear system whose row j holds the Q1 weights of
// node j's foot, and the paper solves it with GMRES.  A = I - beta W_f is
// never assembled: a product A x is one gather-and-blend pass over the nodes,
// the work of one evaluation sweep (FP32 grids read the frozen feet that the
// improvement sweep stored, FP64 grids recompute the foot from the policy
// code).  The penalty M and the running cost are the constant part b of the
// affine map T_f(V) = b + beta W_f V, so they never enter a product.
//
// One cycle corrects a value V whose image T_f(V) is already known:
//   r0 = T_f(V) - V, Arnoldi on A from r0 (m steps, classical Gram-Schmidt,
//   optionally twice), y = argmin ||beta0 e1 - H y||, V <- V + Q y.
// The basis vectors are stored unnormalised, with scale[i] = 1 / ||Q_i||.
// An Arnoldi step is three launches: the product (gather-bound, one node per
// thread at the evaluation sweep's occupancy), the projections, and the update
// with the norm.  The streaming launches give every block an equal contiguous
// share of the vectors in 16-byte loads, eight vectors at a time.  A launch
// sums its dot products per block into a partial row, and the last block to
// finish adds the rows in a fixed order (the result does not depend on block
// scheduling) and does the Hessenberg and Givens work from shared memory.  No
// block waits for another.
//
// Element-wise work runs in the basis precision VT (FP32 on FP32 grids: the
// FP64 pipe of this GPU is a small fraction of its FP32 pipe).  A thread sums
// its share of a dot product as a pair of floats (TwoSum, so that long shares
// lose nothing) and the warp's lanes are combined the same way; the warps'
// totals are widened to FP64 for the block and grid sums and the Hessenberg
// problem.
#include <algorithm>

#include "dp_sweep.cuh"

namespace dpk {
namespace {

constexpr int kGmBlock = 256;
constexpr int kGmWarps = kGmBlock / 32;
constexpr int kGmCols = 8;                  // vectors read at a time by the streaming kernels
constexpr int kGmStreamBlocks = 4;          // blocks per SM of the streaming kernels, at most

// A running sum: FP32 terms as an unevaluated pair of floats (Knuth's TwoSum
// keeps what each addition rounds off), FP64 terms plainly.
template <typename T> struct Acc;
template <> struct Acc<float> {
    float hi = 0.0f, lo = 0.0f;
    __device__ __forceinline__ void add(float x)
    {
        const float s = __fadd_rn(hi, x), b = __fadd_rn(s, -hi);
        lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(hi, -__fadd_rn(s, -b)), __fadd_rn(x, -b)));
        hi = s;
    }
    __device__ __forceinline__ double warp_total()
    {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float h = __shfl_xor_sync(0xffffffffu, hi, o), l = __shfl_xor_sync(0xffffffffu, lo, o);
            add(h);
            lo = __fadd_rn(lo, l);
        }
        return (double)hi + (double)lo;
    }
};
template <> struct Acc<double> {
    double v = 0.0;
    __device__ __forceinline__ void add(double x) { v += x; }
    __device__ __forceinline__ double warp_total()
    {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    }
};

// Per-block sums: a row per warp.
struct BlockSums {
    double acc[kGmWarps][kGmLd];
};

// The warp's total of a thread's sum into its row's column c.  Every lane of
// the warp calls it, once per column.
template <typename T>
__device__ __forceinline__ void sums_put(BlockSums& S, int c, Acc<T> a)
{
    const double v = a.warp_total();
    if ((threadIdx.x & 31) == 0) S.acc[threadIdx.x >> 5][c] = v;
}

// Stores the block's columns [0, ncol) among the partial sums (column by column).  Returns true in
// every thread of the last block to finish, with red[c] = the sum over all
// blocks (lane-strided over blocks, then a fixed shuffle tree).
__device__ bool sums_finish(BlockSums& S, int ncol, double* __restrict__ partial, GmCtl* gc, double* red)
{
    __shared__ int s_last;
    __syncthreads();
    for (int c = threadIdx.x; c < ncol; c += kGmBlock) {
        double v = 0.0;
#pragma unroll
        for (int w = 0; w < kGmWarps; ++w) v += S.acc[w][c];
        partial[(size_t)c * gridDim.x + blockIdx.x] = v;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&gc->counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return false;
    __threadfence();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int c = warp; c < ncol; c += kGmWarps) {
        Acc<double> a;
#pragma unroll 8
        for (int b = lane; b < (int)gridDim.x; b += 32) a.add(__ldcg(&partial[(size_t)c * gridDim.x + b]));
        const double v = a.warp_total();
        if (lane == 0) red[c] = v;
    }
    __syncthreads();
    if (threadIdx.x == 0) gc->counter = 0;
    return true;
}

// This block's share [first, last) of the vectors' 4-entry groups.
__device__ __forceinline__ void share(int n, int& first, int& last)
{
    const int n4 = (n >> 2) + ((n & 3) != 0), per = n4 / (int)gridDim.x, more = n4 % (int)gridDim.x;
    first = (int)blockIdx.x * per + min((int)blockIdx.x, more);
    last = first + per + ((int)blockIdx.x < more ? 1 : 0);
}

// Four consecutive entries j4..j4+3 of a vector (j4 a multiple of 4 and the
// vector 16-byte aligned: one or two 16-byte accesses); entries at or past n
// read as 0 and are not written.
__device__ __forceinline__ void ld4(const float* p, float v[4])
{
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void ld4(const double* p, double v[4])
{
    const double2 a = *reinterpret_cast<const double2*>(p);
    const double2 b = *reinterpret_cast<const double2*>(p + 2);
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void st4(float* p, const float v[4])
{
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void st4(double* p, const double v[4])
{
    *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
    *reinterpret_cast<double2*>(p + 2) = make_double2(v[2], v[3]);
}
template <typename T>
__device__ __forceinline__ void load4(const T* p, int j4, int n, T v[4])
{
    if (j4 + 3 < n) {
        ld4(p + j4, v);
    } else {
#pragma unroll
        for (int s = 0; s < 4; ++s) v[s] = j4 + s < n ? p[j4 + s] : (T)0;
    }
}
template <typename T>
__device__ __forceinline__ void store4(T* p, int j4, int n, const T v[4])
{
    if (j4 + 3 < n) {
        st4(p + j4, v);
    } else {
#pragma unroll
        for (int s = 0; s < 4; ++s)
            if (j4 + s < n) p[j4 + s] = v[s];
    }
}

// (A x)_j = x_j - beta (W_f x)_j from node j's frozen foot (FP32 geometry).
// A foot outside the box or the node set, and a target node, have no W row.
template <bool REDUCED, int DYN, typename W>
__device__ __forceinline__ float apply_a_feet(const Geo<float>& g, const float* __restrict__ x, int j, W w,
                                              const uint16_t* __restrict__ code)
{
    const float xj = x[j];
    const int kind = foot_kind(w);
    float D = 0.0f;
    if (kind == kFootInside) D = eval_foot<REDUCED>(g, x, j, w, 0.0f);
    else if (kind == kFootRecompute) D = incr_recompute<REDUCED, DYN>(g, x, j, code[j]);
    return xj - fmaf(g.beta_hi, D, g.beta_lo * D);
}

// The same product with the foot recomputed from the policy code (FP64).  The
// geometry carries M = 0, so a foot outside the box blends to 0.
template <bool REDUCED, int DYN>
__device__ __forceinline__ double apply_a_node(const Geo<double>& g, const double* __restrict__ x, int j,
                                               const uint16_t* __restrict__ code)
{
    const double xj = x[j];
    NodeEval<double, double, REDUCED, DYN> ev;
    decode_node(g, j, ev.i);
    if (in_target(g, ev.i)) return xj;
    setup_node<double, double, DYN>(ev, g, x, xj);
    const int c = code[j];
    double D;
    if (DYN == kDynPolar && g.off && c == kCodeOff) D = ev.at_sc(0.0, 0.0);
    else D = ev.at_code(c);
    return xj - g.beta64 * (xj + D);
}

// The same from an FP64 frozen foot (offsets word and fractions).
template <bool REDUCED, int DYN>
__device__ __forceinline__ double apply_a_feet64(const Geo<double>& g, const double* __restrict__ x, int j,
                                                 const Feet64& f64, const uint16_t* __restrict__ code)
{
    constexpr bool kPer = DYN == kDynPolar;
    const double xj = x[j];
    const unsigned long long w = __ldcs(&f64.w[j]);
    const int kind = (int)((w >> 32) & 3u);
    if (kind == kFootInside) {
        int i[4], cl[4];
        decode_node(g, j, i);
#pragma unroll
        for (int d = 0; d < 4; ++d) cl[d] = i[d] + (int)(signed char)((w >> (8 * d)) & 0xffu);
        if (kPer) cl[3] = cl[3] < 0 ? cl[3] + g.n[3] : (cl[3] >= g.n[3] ? cl[3] - g.n[3] : cl[3]);
        const double2 ta = __ldcs(&f64.t[2 * (size_t)j]), tb = __ldcs(&f64.t[2 * (size_t)j + 1]);
        const double t[4] = {ta.x, ta.y, tb.x, tb.y};
        Corners<double> K;
        load_corners<double, double, double, REDUCED, kPer>(g, x, cl, 0.0, K);
        return xj - g.beta64 * K.blend(t);
    }
    if (kind == kFootRecompute) return apply_a_node<REDUCED, DYN>(g, x, j, code);
    return xj;   // outside or target: no W row
}

// A pair of floats ends at FP32's range.  Columns [0, ncol) whose sum over the
// warp's part of the block's share left it (entries of 1e17 and more; one tile
// of 128 products at a time went to 1e18) are summed again in FP64: column c is
// the product of w with vector(c).  Every warp calls it after its sums_put()s.
template <typename VT, class F>
__device__ __forceinline__ void sums_repair(BlockSums& S, int ncol, const VT* w, F vector, int first, int last, int n)
{
    if constexpr (std::is_same<VT, float>::value) {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        __syncwarp();
        for (int c0 = 0; c0 < ncol; c0 += 32) {
            unsigned bad = __ballot_sync(0xffffffffu, c0 + lane < ncol && !isfinite(S.acc[warp][min(c0 + lane, ncol - 1)]));
            for (; bad; bad &= bad - 1) {
                const int c = c0 + __ffs((int)bad) - 1;
                const VT* q = vector(c);
                Acc<double> a;
#pragma unroll 1
                for (int e = first + (int)threadIdx.x; e < last; e += kGmBlock) {
                    VT x[4], y[4];
                    load4(w, 4 * e, n, x);
                    load4(q, 4 * e, n, y);
#pragma unroll
                    for (int s = 0; s < 4; ++s) a.add((double)x[s] * (double)y[s]);
                }
                const double v = a.warp_total();
                if (lane == 0) S.acc[warp][c] = v;
            }
        }
    }
}

// r0 = V_next - V_in into Q_0, and ||r0||.
template <typename VV, typename VT>
__global__ void __launch_bounds__(kGmBlock)
gm_start_kernel(const VV* Vin, const VV* Vnext, VT* q0, int n, double* __restrict__ partial, GmCtl* gc)
{
    let_next_start();
    wait_for_previous();
    __shared__ BlockSums S;
    __shared__ double red[kGmLd];
    Acc<VT> nrm;
    int first, last;
    share(n, first, last);
#pragma unroll 2
    for (int e = first + (int)threadIdx.x; e < last; e += kGmBlock) {
        const int j4 = 4 * e;
        VV a[4], b[4];
        VT r[4];
        load4(Vin, j4, n, a);
        load4(Vnext, j4, n, b);
        VT d = (VT)0;
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            r[s] = (VT)(b[s] - a[s]);
            d += r[s] * r[s];
        }
        store4(q0, j4, n, r);
        nrm.add(d);
    }
    sums_put(S, 0, nrm);
    sums_repair(S, 1, q0, [&](int) { return q0; }, first, last, n);
    if (!sums_finish(S, 1, partial, gc, red)) return;
    if (threadIdx.x == 0) {
        const double b = sqrt(red[0]);
        const bool ok = b > 0.0 && isfinite(b);
        gc->beta0 = b;
        gc->gv[0] = b;
        gc->rel = ok ? 1.0 : 0.0;
        gc->k = 0;
        gc->scale[0] = ok ? 1.0 / b : 0.0;
        gc->done = ok ? 0 : 1;
    }
}

// Arnoldi step k, the product: Q_{k+1} = A q_k (q_k = scale[k] Q_k).  One
// node per thread, nodes of a warp adjacent, the next node's foot and value
// fetched while this node's corners are in flight (as in the evaluation
// sweep); compiled for the sweep's occupancy on FP32 grids.
template <typename G>
constexpr int matvec_min_blocks() { return std::is_same<G, float>::value ? 6 : 2; }

template <typename G, typename VT, bool REDUCED, int DYN>
__global__ void __launch_bounds__(kGmBlock, matvec_min_blocks<G>())
gm_matvec_kernel(const __grid_constant__ Geo<G> g, VT* __restrict__ Q, long long ldq, int k,
                 const uint16_t* __restrict__ code, const unsigned long long* __restrict__ feet_lo,
                 const unsigned* __restrict__ feet_hi, const Feet64 f64, GmCtl* gc)
{
    let_next_start();
    wait_for_previous();
    if (*(const volatile int*)&gc->done) return;
    const VT* x = Q + (size_t)k * ldq;
    VT* w = Q + (size_t)(k + 1) * ldq;
    const VT sk = (VT)gc->scale[k];
    // without a sign: a node and the stride after it may pass 2^31 together
    const unsigned n = (unsigned)g.n_nodes, stride = gridDim.x * kGmBlock;
    if constexpr (std::is_same<G, float>::value) {
        unsigned j = blockIdx.x * kGmBlock + threadIdx.x;
        if (feet_hi) {
            // the word pair of the FP64-value phase
            FootWord next{0ull, 0u};
            if (j < n) next = FootWord{__ldcs(&feet_lo[j]), __ldcs(&feet_hi[j])};
            for (; j < n; j += stride) {
                const FootWord fw = next;
                if (j + stride < n) next = FootWord{__ldcs(&feet_lo[j + stride]), __ldcs(&feet_hi[j + stride])};
                w[j] = sk * apply_a_feet<REDUCED, DYN>(g, x, (int)j, fw, code);
            }
        } else {
            // 8-byte feet of the FP32-value phase
            unsigned long long next = 0ull;
            if (j < n) next = __ldcs(&feet_lo[j]);
            for (; j < n; j += stride) {
                const unsigned long long fw = next;
                if (j + stride < n) next = __ldcs(&feet_lo[j + stride]);
                w[j] = sk * apply_a_feet<REDUCED, DYN>(g, x, (int)j, fw, code);
            }
        }
    } else if (f64.w) {
        for (unsigned j = blockIdx.x * kGmBlock + threadIdx.x; j < n; j += stride)
            w[j] = sk * apply_a_feet64<REDUCED, DYN>(g, x, (int)j, f64, code);
    } else {
        for (unsigned j = blockIdx.x * kGmBlock + threadIdx.x; j < n; j += stride)
            w[j] = sk * apply_a_node<REDUCED, DYN>(g, x, (int)j, code);
    }
}

// Closes column k once ||Q_{k+1}||^2 is known: rotations, residual estimate,
// and, when the cycle ends, the back substitution R y = g into coef (as
// coefficients of the raw Q_i).  A whole block: what the recurrences read is
// copied to shared memory first, in parallel (read from memory step by step by
// one thread, the column's loads alone took several microseconds, and the
// k^2 / 2 of the substitution tens of them).
__device__ void finalize_column(GmCtl* gc, int k, int m, double rtol, double nrm2, double* sR, double* sh)
{
    double* hc = sh;                               // column k
    double* cs = sh + kGmMaxRestart + 1;
    double* sn = cs + kGmMaxRestart;
    __shared__ int s_kk, s_stop;
    const int tid = threadIdx.x;
    for (int i = tid; i <= k; i += kGmBlock) hc[i] = gc->H[i][k];
    for (int i = tid; i < k; i += kGmBlock) {
        cs[i] = gc->cs[i];
        sn[i] = gc->sn[i];
    }
    __syncthreads();
    if (tid == 0) {
        const double nu = sqrt(fmax(nrm2, 0.0));
        for (int i = 0; i < k; ++i) {
            const double a = hc[i], b = hc[i + 1];
            hc[i] = cs[i] * a + sn[i] * b;
            hc[i + 1] = -sn[i] * a + cs[i] * b;
        }
        const double a = hc[k];
        const double r = hypot(a, nu);
        int kk = k + 1;
        bool stop = kk >= m;
        if (!(r > 0.0) || !isfinite(r)) {
            kk = k;             // no usable column: solve with the previous ones
            stop = true;
        } else {
            const double c = a / r, s = nu / r;
            gc->cs[k] = c;
            gc->sn[k] = s;
            hc[k] = r;
            gc->H[k + 1][k] = 0.0;
            const double g = gc->gv[k], g1 = -s * g;
            gc->gv[k + 1] = g1;
            gc->gv[k] = c * g;
            gc->scale[k + 1] = nu > 0.0 ? 1.0 / nu : 0.0;
            gc->rel = fabs(g1) / gc->beta0;
            // converged, or the Krylov space is (numerically) invariant
            if (fabs(g1) / gc->beta0 <= rtol || !(nu > 1e-14 * r)) stop = true;
        }
        gc->k = kk;
        s_kk = kk;
        s_stop = stop;
    }
    __syncthreads();
    for (int i = tid; i <= k; i += kGmBlock) gc->H[i][k] = hc[i];
    if (!s_stop) return;
    // R (upper triangle, kk x kk) and g to shared memory, then column by column
    const int kk = s_kk;
    __syncthreads();
    for (int e = tid; e < kk * kk; e += kGmBlock) {
        const int i = e / kk, l = e % kk;
        if (l >= i) sR[i * kGmMaxRestart + l] = l == k ? hc[i] : gc->H[i][l];
    }
    double* y = hc;   // hc is stored
    __syncthreads();
    for (int i = tid; i < kk; i += kGmBlock) y[i] = gc->gv[i];
    __syncthreads();
    if (tid < 32) {
        for (int i = kk - 1; i >= 0; --i) {
            const double c = y[i] / sR[i * kGmMaxRestart + i];
            __syncwarp();
            if (tid == 0) y[i] = c;
            for (int l = tid; l < i; l += 32) y[l] -= sR[l * kGmMaxRestart + i] * c;
            __syncwarp();
        }
        for (int i = tid; i < kk; i += 32) gc->coef[i] = y[i] * gc->scale[i];
        if (tid == 0) gc->done = 1;
    }
}

// Vectors are read in equal groups of at most kGmCols: 9 as 5 and 4, not 8 and
// 1, so that every pass keeps enough loads in flight.
__host__ __device__ constexpr int group_width(int count)
{
    const int groups = (count + kGmCols - 1) / kGmCols;
    return (count + groups - 1) / groups;
}

// Runs f with a compile-time width.
template <int N> struct Width { static constexpr int n = N; };
template <class F>
__device__ __forceinline__ void with_width(int w, F f)
{
    switch (w) {
    case 1: f(Width<1>()); break;
    case 2: f(Width<2>()); break;
    case 3: f(Width<3>()); break;
    case 4: f(Width<4>()); break;
    case 5: f(Width<5>()); break;
    case 6: f(Width<6>()); break;
    case 7: f(Width<7>()); break;
    default: f(Width<8>()); break;
    }
}

// Arnoldi step k, the projections h_ik = <q_i, Q_{k+1}>: they set column k of
// H (SECOND: correct it, the second pass of Gram-Schmidt) and become the next
// coefficients.  A thread reads up to eight vectors at a time and keeps their
// sums in registers; the vector itself is read again for the next group.  41^4
// in FP32 (11.3 MB a vector), ten vectors on average: 33 us cold; one tile of
// 1,024 nodes at a time with a widened shared-memory addition per warp, vector
// and tile, which the FP64 pipe bounded at 45 %, 55 us; groups of eight and a
// remainder read one vector after another 40.
template <typename VT, bool SECOND>
__global__ void __launch_bounds__(kGmBlock, sizeof(VT) == 4 ? kGmStreamBlocks : 2)
gm_dots_kernel(const VT* __restrict__ Q, long long ldq, int n, int k, double* __restrict__ partial,
               GmCtl* gc)
{
    let_next_start();
    wait_for_previous();
    if (*(volatile int*)&gc->done) return;
    __shared__ BlockSums S;
    __shared__ double red[kGmLd];
    const VT* w = Q + (size_t)(k + 1) * ldq;
    int first, last;
    share(n, first, last);
    const int width = group_width(k + 1);
    for (int i0 = 0; i0 <= k; i0 += width) {
        const VT* q0 = Q + (size_t)i0 * ldq;
        with_width(min(width, k + 1 - i0), [&](auto wt) {
            constexpr int W = decltype(wt)::n;
            Acc<VT> acc[W];
            for (int e = first + (int)threadIdx.x; e < last; e += kGmBlock) {
                VT wv[4], q[W][4];
                load4(w, 4 * e, n, wv);
#pragma unroll
                for (int c = 0; c < W; ++c) load4(q0 + (size_t)c * ldq, 4 * e, n, q[c]);
#pragma unroll
                for (int c = 0; c < W; ++c) {
                    VT d = (VT)0;
#pragma unroll
                    for (int s = 0; s < 4; ++s) d += q[c][s] * wv[s];
                    acc[c].add(d);
                }
            }
#pragma unroll
            for (int c = 0; c < W; ++c) sums_put(S, i0 + c, acc[c]);
        });
    }
    sums_repair(S, k + 1, w, [&](int c) { return Q + (size_t)c * ldq; }, first, last, n);
    if (!sums_finish(S, k + 1, partial, gc, red)) return;
    for (int i = threadIdx.x; i <= k; i += kGmBlock) {
        const double h = gc->scale[i] * red[i];
        gc->H[i][k] = SECOND ? gc->H[i][k] + h : h;
        gc->coef[i] = h * gc->scale[i];
    }
}

// v += sum over i < count of coef_i Q_i at the 4-entry group e, the vectors in
// groups of W; coefficients past the last are 0 (their loads repeat it).
template <int W, typename VT>
__device__ __forceinline__ void combine(const VT* __restrict__ Q, long long ldq, int n, int e, int count,
                                        const VT* coef, VT v[4])
{
    for (int i = 0; i < count; i += W) {
        VT q[W][4];
#pragma unroll
        for (int c = 0; c < W; ++c) load4(Q + (size_t)min(i + c, count - 1) * ldq, 4 * e, n, q[c]);
#pragma unroll
        for (int c = 0; c < W; ++c) {
            const VT x = coef[i + c];
#pragma unroll
            for (int s = 0; s < 4; ++s) v[s] += x * q[c][s];
        }
    }
}

// Q_{k+1} -= sum_i coef_i Q_i, and (NORM) the norm that closes the column.
// Groups of vectors as the projections read them; each block walks its share
// backwards, from the end that the projections read last and L2 still holds.
// 34 us cold at ten vectors of 41^4; 47 with tiles of 1,024 nodes, four loads
// in flight and the column closed by one thread from memory.
template <typename VT, bool NORM>
__global__ void __launch_bounds__(kGmBlock, sizeof(VT) == 4 ? kGmStreamBlocks : 2)
gm_update_kernel(VT* __restrict__ Q, long long ldq, int n, int k, int m, double rtol, double* __restrict__ partial,
                 GmCtl* gc)
{
    let_next_start();
    wait_for_previous();
    if (*(volatile int*)&gc->done) return;
    // the sums of the norm, then the last block's copy of R
    __shared__ union { BlockSums S; double R[kGmMaxRestart * kGmMaxRestart]; } U;
    __shared__ double red[kGmLd], sh[3 * kGmMaxRestart + 1];
    __shared__ VT s_coef[kGmMaxRestart + 1 + kGmCols];
    for (int i = threadIdx.x; i <= k + kGmCols; i += kGmBlock) s_coef[i] = i <= k ? -(VT)gc->coef[i] : (VT)0;
    __syncthreads();
    VT* w = Q + (size_t)(k + 1) * ldq;
    Acc<VT> nrm;
    int first, last;
    share(n, first, last);
    with_width(group_width(k + 1), [&](auto wt) {
        constexpr int W = decltype(wt)::n;
        for (int e = last - 1 - (int)threadIdx.x; e >= first; e -= kGmBlock) {
            VT wv[4];
            load4(w, 4 * e, n, wv);
            combine<W>(Q, ldq, n, e, k + 1, s_coef, wv);
            store4(w, 4 * e, n, wv);
            if constexpr (NORM) {
                VT d = (VT)0;
#pragma unroll
                for (int s = 0; s < 4; ++s) d += wv[s] * wv[s];
                nrm.add(d);
            }
        }
    });
    if constexpr (NORM) {
        sums_put(U.S, 0, nrm);
        sums_repair(U.S, 1, w, [&](int) { return w; }, first, last, n);
        if (!sums_finish(U.S, 1, partial, gc, red)) return;
        finalize_column(gc, k, m, rtol, red[0], U.R, sh);
    }
}

// V_next = V_in + sum_i coef_i Q_i over the cycle's k columns; the
// correction is summed in the basis precision and added once to V_in.
template <typename VV, typename VT>
__global__ void __launch_bounds__(kGmBlock)
gm_apply_kernel(const VV* Vin, VV* Vnext, const VT* Q, long long ldq, int n, GmCtl* gc, Ctl* ctl)
{
    let_next_start();
    wait_for_previous();
    __shared__ VT s_coef[kGmMaxRestart + kGmCols];
    const int kk = gc->k;
    for (int i = threadIdx.x; i < kk + kGmCols; i += kGmBlock) s_coef[i] = i < kk ? (VT)gc->coef[i] : (VT)0;
    __syncthreads();
    bool bad = false;
    int first, last;
    share(n, first, last);
    with_width(kk > 0 ? group_width(kk) : 1, [&](auto wt) {
        constexpr int W = decltype(wt)::n;
        for (int e = first + (int)threadIdx.x; e < last; e += kGmBlock) {
            VT x[4] = {(VT)0, (VT)0, (VT)0, (VT)0};
            VV v[4];
            load4(Vin, 4 * e, n, v);
            combine<W>(Q, ldq, n, e, kk, s_coef, x);
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                v[s] += (VV)x[s];
                bad = bad || (4 * e + s < n && !isfinite(v[s]));
            }
            store4(Vnext, 4 * e, n, v);
        }
    });
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(&ctl->nonfinite, 1);
}

// Frozen feet of the resident policy, the words an improvement sweep stores:
// the word pair when feet_hi is given (FP64-value phase), else the 8-byte
// word (FP32-value phase).
template <bool REDUCED, int DYN>
__global__ void __launch_bounds__(kGmBlock)
feet_kernel(const __grid_constant__ Geo<float> g, const uint16_t* __restrict__ code,
            unsigned long long* __restrict__ feet_lo, unsigned* __restrict__ feet_hi)
{
    for (unsigned ju = blockIdx.x * kGmBlock + threadIdx.x; ju < (unsigned)g.n_nodes; ju += gridDim.x * kGmBlock) {
        const int j = (int)ju;
        CachedEval<float, float, REDUCED, DYN, float, false> ev;
        decode_node(g, j, ev.i);
        const bool target = in_target(g, ev.i);
        float sn = 0.0f, cs = 0.0f;
        if (!target) {
            setup_node<float, float, DYN>(ev, g, (const float*)nullptr, 0.0f);
            ev.reset();
            code_sincos(g, code[j], sn, cs);
        }
        if (feet_hi) {
            const FootWord w = target ? foot_word_kind(kFootTarget) : ev.foot_of(sn, cs);
            feet_lo[j] = w.lo;
            feet_hi[j] = w.hi;
        } else {
            feet_lo[j] = target ? foot8_kind(kFootTarget) : ev.foot8_of(sn, cs);
        }
    }
}

// Blocks of a streaming launch: the resident ones of every SM, at most
// max_blocks (rows of the partial-sum buffer) and one per 256 4-entry groups.
template <typename K>
int stream_blocks(K kern, int n, int sm_count, int max_blocks, int& per_sm)
{
    if (per_sm == 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kGmBlock, 0) != cudaSuccess) per_sm = 1;
        if (per_sm < 1) per_sm = 1;
    }
    const long long groups = ((long long)n + 4 * kGmBlock - 1) / (4 * kGmBlock);
    long long b = (long long)std::min(per_sm, kGmStreamBlocks) * sm_count;
    if (b > max_blocks) b = max_blocks;
    if (b > groups) b = groups;
    return b < 1 ? 1 : (int)b;
}

template <typename G, typename VT, bool REDUCED, int DYN>
cudaError_t launch_arnoldi(const GmArgs<G, VT>& a, int k)
{
    auto kern = gm_matvec_kernel<G, VT, REDUCED, DYN>;
    static int per_sm = 0;
    if (per_sm == 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kGmBlock, 0) != cudaSuccess) per_sm = 1;
        if (per_sm < 1) per_sm = 1;
    }
    const long long need = ((long long)a.g.n_nodes + kGmBlock - 1) / kGmBlock;
    const long long cap = (long long)per_sm * a.sm_count;
    const int b = (int)(need < cap ? (need < 1 ? 1 : need) : cap);
    return launch_after(kern, b, kGmBlock, 0, a.stream, a.g, a.Q, a.ldq, k, a.code, a.feet_lo, a.feet_hi, a.f64, a.gctl);
}

template <bool SECOND, typename G, typename VT>
cudaError_t launch_dots(const GmArgs<G, VT>& a, int n, int k)
{
    auto kern = gm_dots_kernel<VT, SECOND>;
    static int per_sm = 0;
    const int b = stream_blocks(kern, n, a.sm_count, a.max_blocks, per_sm);
    return launch_after(kern, b, kGmBlock, 0, a.stream, a.Q, a.ldq, n, k, a.partial, a.gctl);
}

template <bool NORM, typename G, typename VT>
cudaError_t launch_update(const GmArgs<G, VT>& a, int n, int k)
{
    auto kern = gm_update_kernel<VT, NORM>;
    static int per_sm = 0;
    const int b = stream_blocks(kern, n, a.sm_count, a.max_blocks, per_sm);
    return launch_after(kern, b, kGmBlock, 0, a.stream, a.Q, a.ldq, n, k, a.m, a.rtol, a.partial, a.gctl);
}

cudaError_t dispatch_arnoldi(const GmArgs<float, float>& a, int k)
{
    if (a.dyn == kDynUnitSpeed && !a.reduced) return launch_arnoldi<float, float, false, kDynUnitSpeed>(a, k);
    if (a.dyn == kDynOrbit) {
        if (a.reduced) return launch_arnoldi<float, float, true, kDynOrbit>(a, k);
        return launch_arnoldi<float, float, false, kDynOrbit>(a, k);
    }
    return cudaErrorInvalidValue;
}

cudaError_t dispatch_arnoldi(const GmArgs<double, double>& a, int k)
{
    if (a.dyn == kDynUnitSpeed && !a.reduced) return launch_arnoldi<double, double, false, kDynUnitSpeed>(a, k);
    if (a.dyn == kDynPolar && !a.reduced) return launch_arnoldi<double, double, false, kDynPolar>(a, k);
    if (a.dyn == kDynOrbit) {
        if (a.reduced) return launch_arnoldi<double, double, true, kDynOrbit>(a, k);
        return launch_arnoldi<double, double, false, kDynOrbit>(a, k);
    }
    return cudaErrorInvalidValue;
}

template <typename G, typename VT, typename VV>
cudaError_t cycle(const GmArgs<G, VT>& a, const VV* Vin, VV* Vnext)
{
    if (a.m < 1 || a.m > kGmMaxRestart || !a.Q || !a.partial || !a.gctl) return cudaErrorInvalidValue;
    if (std::is_same<G, float>::value && !a.feet_lo) return cudaErrorInvalidValue;
    const int n = a.g.n_nodes;
    cudaError_t e;
    {
        auto kern = gm_start_kernel<VV, VT>;
        static int per_sm = 0;
        const int b = stream_blocks(kern, n, a.sm_count, a.max_blocks, per_sm);
        e = launch_after(kern, b, kGmBlock, 0, a.stream, Vin, Vnext, a.Q, n, a.partial, a.gctl);
        if (e != cudaSuccess) return e;
    }
    for (int k = 0; k < a.m; ++k) {
        if ((e = dispatch_arnoldi(a, k)) != cudaSuccess) return e;
        if ((e = launch_dots<false>(a, n, k)) != cudaSuccess) return e;
        if (a.reorth && ((e = launch_update<false>(a, n, k)) != cudaSuccess || (e = launch_dots<true>(a, n, k)) != cudaSuccess))
            return e;
        if ((e = launch_update<true>(a, n, k)) != cudaSuccess) return e;
    }
    auto kern = gm_apply_kernel<VV, VT>;
    static int per_sm = 0;
    const int b = stream_blocks(kern, n, a.sm_count, a.max_blocks, per_sm);
    return launch_after(kern, b, kGmBlock, 0, a.stream, Vin, Vnext, a.Q, a.ldq, n, a.gctl, a.ctl);
}

}  // namespace

cudaError_t gm_cycle(const GmArgs<float, float>& a, const float* Vin, float* Vnext) { return cycle(a, Vin, Vnext); }
cudaError_t gm_cycle(const GmArgs<float, float>& a, const double* Vin, double* Vnext) { return cycle(a, Vin, Vnext); }
cudaError_t gm_cycle(const GmArgs<double, double>& a, const double* Vin, double* Vnext)
{
    return cycle(a, Vin, Vnext);
}

cudaError_t launch_feet(const Geo<float>& g, const uint16_t* code, unsigned long long* feet_lo, unsigned* feet_hi,
                        int dyn, int reduced, int sm_count, cudaStream_t st)
{
    const long long need = ((long long)g.n_nodes + kGmBlock - 1) / kGmBlock;
    const int blocks = (int)(need < 8LL * sm_count ? need : 8LL * sm_count);
    if (blocks < 1) return cudaSuccess;
    if (dyn == kDynUnitSpeed && !reduced)
        feet_kernel<false, kDynUnitSpeed><<<blocks, kGmBlock, 0, st>>>(g, code, feet_lo, feet_hi);
    else if (dyn == kDynOrbit && reduced)
        feet_kernel<true, kDynOrbit><<<blocks, kGmBlock, 0, st>>>(g, code, feet_lo, feet_hi);
    else if (dyn == kDynOrbit)
        feet_kernel<false, kDynOrbit><<<blocks, kGmBlock, 0, st>>>(g, code, feet_lo, feet_hi);
    else
        return cudaErrorInvalidValue;
    return cudaGetLastError();
}

}  // namespace dpk
