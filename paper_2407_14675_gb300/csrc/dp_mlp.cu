// dp_mlp.cu -- the learned warm start: a 4 -> 256 -> 256 -> 256 -> 3 BF16 MLP
// (exact-erf GELU, FP32 accumulation) trained on the GPU on (state, V / M,
// cos alpha*, sin alpha*) samples of a solved grid, then evaluated on every
// node of another grid to initialise V and the policy of policy iteration.
// Not part of the paper: the network only supplies the starting point, and
// the Bellman sweeps alone decide the result.
//
// The two 256 x 256 layers (98.6 % of the FLOPs) run on the fifth-generation
// tensor cores: tcgen05.mma kind::f16, BF16 operands staged in shared memory,
// FP32 accumulators in TMEM, fused epilogues (bias + GELU forward, GELU'
// backward, split-K partial tiles for weight gradients).  The 4-wide input
// layer, the 3-wide output layer, the reductions and Adam run on the CUDA
// cores.  Inference over a grid is one kernel for all layers.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include <cuda_bf16.h>

#include "dp.h"
#include "dp_host.h"
#include "dp_umma.cuh"

namespace dpk {
int record_error(int code, const char* msg);

// View of a grid's resident state (defined in dp_api.cu).
struct GridView {
    Geo<double> g64;
    int fp32;
    const void* V;       // storage precision (FP32 or FP64), compact order
    double* V64;         // FP64 value when the grid holds one (else NULL)
    uint16_t* code;
    long long n;
    double M;
    double lo[4], hi[4];
    cudaStream_t st;
    const double2* tab_hi64;
    const double2* tab_lo64;
};
int grid_view(dp_grid* g, GridView* v);
void grid_after_warm_start(dp_grid* g);
}  // namespace dpk

using namespace dpk;
typedef __nv_bfloat16 bf16;

namespace {

constexpr int kH = 256;                       // hidden width
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kH * 4, kOffW2 = kOffB1 + kH, kOffB2 = kOffW2 + kH * kH;
constexpr int kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kH * kH, kOffW4 = kOffB3 + kH, kOffB4 = kOffW4 + 3 * kH;
constexpr int kParams = kOffB4 + 3;           // 133,635
constexpr int kTileM = 128, kTileN = 128, kKC = 256;
constexpr int kGemmSmem = (kTileM + kTileN) * kKC * 2;   // A and B of a tile, 128 KB
constexpr int kWaitPolls = 1 << 22;
constexpr float kInvSqrt2 = 0.70710678118654752f, kInvSqrt2Pi = 0.39894228040143268f;

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * kInvSqrt2)); }
__device__ __forceinline__ float gelu_grad(float z)
{
    return 0.5f * (1.0f + erff(z * kInvSqrt2)) + z * kInvSqrt2Pi * expf(-0.5f * z * z);
}

// 8 consecutive BF16 values (one 16-byte load) as floats.
__device__ __forceinline__ void row8(const uint4& v, float a[8])
{
    const unsigned u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const __nv_bfloat162 h2 = *reinterpret_cast<const __nv_bfloat162*>(&u[q]);
        a[2 * q] = __low2float(h2);
        a[2 * q + 1] = __high2float(h2);
    }
}

enum { kEpiFwd = 0, kEpiBwd = 1 };

// Four doubles by value (the network's input box corners).
struct Box4 {
    double x, y, z, w;
};

// 16-byte asynchronous copy global -> shared (both 16-byte aligned), and the
// wait for all of this thread's copies.
__device__ __forceinline__ void cp_async16(void* dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// all but the N groups committed last
template <int N>
__device__ __forceinline__ void cp_async_wait_pending()
{
    asm volatile("cp.async.wait_group %0;" :: "n"(N) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
}

// The 128 x 256 operand of 128 rows from r0 of a row-major matrix into shared
// memory (64 KB): four blocks of 64 columns, 128-byte swizzled, K-major.  A warp
// copies one whole row, every 16-byte piece straight to shared memory
// (cp.async).  Taking 64 bytes of eight rows each, as the layout without a
// swizzle wants, a warp's copy touched eight lines per eight lanes and fetched
// every sector twice.
constexpr int kOpBlock = kTileM * 128;    // bytes of a block of 64 columns

template <int THREADS>
__device__ __forceinline__ void stage_rows(unsigned char* dst, const bf16* src, size_t ld, size_t r0)
{
#pragma unroll 8
    for (int q = 0; q < kTileM * kKC / 8 / THREADS; ++q) {
        const int v = (int)threadIdx.x + THREADS * q, row = v >> 5, c = v & 31;
        cp_async16(dst + (c >> 3) * kOpBlock + sw128(row, c & 7), src + (r0 + row) * ld + c * 8);
    }
}

// The 16 MMAs of such a pair of operands; one thread.
__device__ __forceinline__ void mma_rows(unsigned tmem, const unsigned char* sA, const unsigned char* sB)
{
    constexpr unsigned idesc = umma_idesc_bf16(kTileM, kTileN);
#pragma unroll
    for (int s = 0; s < kKC / 16; ++s) {
        const unsigned at = (s >> 2) * kOpBlock + (s & 3) * 32;
        umma_bf16(tmem, umma_desc_sw128(smem_u32(sA) + at, 16, 1024), umma_desc_sw128(smem_u32(sB) + at, 16, 1024), idesc,
                  s > 0 ? 1u : 0u);
    }
}

// C[128 x 128 tile] = A[rows, 256] * B[256, 256]^T on tcgen05, for batches
// below kManyRows rows.
//   A: bf16 [*, lda] row-major (K contiguous); B: bf16 [256, ldb] row-major.
//   Tile rows start at 128 blockIdx.x, columns at 128 blockIdx.y: every thread
//   issues its 16-byte asynchronous copies of both operands at once, then one
//   thread issues the 16 MMAs (K = 16 each) and commits them to an mbarrier.
//   kEpiFwd:    z = acc + bias -> zout (FP32), h = GELU(z) -> hout (bf16)
//   kEpiBwd:    dz = acc * GELU'(zin) -> hout (bf16)
template <int EPI>
__global__ void __launch_bounds__(128)
mlp_gemm_kernel(const bf16* __restrict__ A, int lda, const bf16* __restrict__ B, int ldb, const float* __restrict__ bias,
                float* __restrict__ zout, const float* __restrict__ zin, bf16* __restrict__ hout, int* __restrict__ err,
                int polls)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char* sA = smem;                        // 128 x 256 bf16
    unsigned char* sB = smem + kTileM * kKC * 2;     // 128 x 256 bf16
    __shared__ unsigned tmem_slot;
    __shared__ __align__(8) unsigned long long mbar;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 0) tmem_alloc(&tmem_slot, kTileN);
    if (tid == 0) mbar_init(&mbar);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const unsigned tmem = tmem_slot;
    const size_t row0 = (size_t)blockIdx.x * kTileM;
    const int n0 = blockIdx.y * kTileN;

    stage_rows<128>(sA, A, (size_t)lda, row0);
    stage_rows<128>(sB, B, (size_t)ldb, (size_t)n0);
    cp_async_wait_all();
    fence_async_smem();
    __syncthreads();
    if (tid == 0) {
        fence_after_sync();
        mma_rows(tmem, sA, sB);
        umma_commit(&mbar);
    }
    bool ok = true;
    if (!mbar_wait(&mbar, 0, polls)) {
        // give up (error flag), but let the committed MMAs finish before
        // the accumulator is freed and the staging buffers are released
        ok = false;
        if (lane == 0) atomicOr(err, 1);
        mbar_wait(&mbar, 0, kWaitPolls);
    }
    ok = __syncthreads_and(ok);
    fence_after_sync();
    if (ok) {
        const size_t r = row0 + warp * 32 + lane;   // TMEM lane = tile row
        for (int c0 = 0; c0 < kTileN; c0 += 16) {
            float v[16];
            tmem_ld16(tmem + ((unsigned)(warp * 32) << 16) + c0, v);
            const size_t off = r * kH + n0 + c0;     // 16 consecutive columns, 64-byte aligned
            float z[16];
            if (EPI == kEpiFwd) {
#pragma unroll
                for (int q = 0; q < 16; q += 4) {
                    const float4 b = *(const float4*)(bias + n0 + c0 + q);
                    z[q] = v[q] + b.x; z[q + 1] = v[q + 1] + b.y; z[q + 2] = v[q + 2] + b.z; z[q + 3] = v[q + 3] + b.w;
                    *(float4*)(zout + off + q) = make_float4(z[q], z[q + 1], z[q + 2], z[q + 3]);
                }
#pragma unroll
                for (int q = 0; q < 16; ++q) z[q] = gelu(z[q]);
            } else {
#pragma unroll
                for (int q = 0; q < 16; q += 4) {
                    const float4 zi = *(const float4*)(zin + off + q);
                    z[q] = v[q] * gelu_grad(zi.x); z[q + 1] = v[q + 1] * gelu_grad(zi.y);
                    z[q + 2] = v[q + 2] * gelu_grad(zi.z); z[q + 3] = v[q + 3] * gelu_grad(zi.w);
                }
            }
            unsigned pk[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const __nv_bfloat162 h2 = __floats2bfloat162_rn(z[2 * q], z[2 * q + 1]);
                pk[q] = *(const unsigned*)&h2;
            }
            *(uint4*)(hout + off) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            *(uint4*)(hout + off + 8) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
        }
    }
    fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kTileN);
}

// Weight gradients dz^T h of both hidden layers, split along the batch: the tile
// C[128 blockIdx.x.., 128 blockIdx.y..] over the k_per_cta rows (a multiple of
// kWgRows) from k_per_cta (blockIdx.z mod splits) of A = dz and B = h, both rows
// x 256, read as they are (both operands MN-major, no transposed copies); the
// first `splits` z of the grid are one layer, the others the next.  The tile is
// stored at split blockIdx.z of out (256 x 256 floats per split), for a
// reduction in a fixed order.
//
// What bounds it: 256 KB of operands per CTA from L2 (two slabs of 512 rows at a
// batch of 16,384, 256 CTAs), and the latency of the first of them and of the
// epilogue.  Rows pass through a ring of three 32 KB chunks of 64 rows, two
// ahead of the MMAs, and two CTAs share an SM: 13.4 us for both layers.
// A launch per layer (128 CTAs) with a ring of six took 8.2 us each, 14.0 while
// a warp's copies took 64 bytes of eight rows, and 15.3 with 256 rows staged at a
// time and nothing in flight during their MMAs.
constexpr int kWgRows = 64, kWgSlots = 3, kWgThreads = 256;
constexpr int kWgChunk = kWgRows * kTileM * 2;                     // bytes of one operand's chunk
constexpr int kWgSmem = kWgSlots * 2 * kWgChunk;                   // 96 KB

struct WgPair {
    const bf16 *A[2], *B[2];
};

__global__ void __launch_bounds__(kWgThreads, 2)
mlp_wgrad_kernel(const __grid_constant__ WgPair p, int splits, int k_per_cta, float* __restrict__ out,
                 int* __restrict__ err, int polls)
{
    const bool second = (int)blockIdx.z >= splits;
    const bf16* __restrict__ A = second ? p.A[1] : p.A[0];
    const bf16* __restrict__ B = second ? p.B[1] : p.B[0];
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ unsigned tmem_slot;
    __shared__ __align__(8) unsigned long long done[kWgSlots];     // the slot's MMAs have completed
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.x * kTileM, n0 = blockIdx.y * kTileN;
    const int kbeg = ((int)blockIdx.z - (second ? splits : 0)) * k_per_cta;
    const int chunks = k_per_cta / kWgRows;
    // a chunk is two halves of 64 columns, 128-byte swizzled; a warp copies two
    // rows of 128 columns
    auto stage = [&](int c) {
        unsigned char* dst = smem + (c % kWgSlots) * 2 * kWgChunk;
        const size_t k0 = (size_t)kbeg + (size_t)c * kWgRows;
#pragma unroll
        for (int q = 0; q < 2 * kWgChunk / 16 / kWgThreads; ++q) {
            const int v = tid + kWgThreads * (q % (kWgChunk / 16 / kWgThreads)), kr = v >> 4, c = v & 15;
            const unsigned at = (c >> 3) * (kWgChunk / 2) + sw128(kr, c & 7);
            if (q < kWgChunk / 16 / kWgThreads) cp_async16(dst + at, A + (k0 + kr) * kH + m0 + c * 8);
            else cp_async16(dst + kWgChunk + at, B + (k0 + kr) * kH + n0 + c * 8);
        }
    };
    // one group of copies per chunk and turn, empty ones included, so that the
    // groups left pending count the chunks
#pragma unroll
    for (int c = 0; c < kWgSlots - 1; ++c) {
        if (c < chunks) stage(c);
        cp_async_commit();
    }
    if (warp == 0) tmem_alloc(&tmem_slot, kTileN);
    if (tid == 0) {
        for (int b = 0; b < kWgSlots; ++b) mbar_init(&done[b]);
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const unsigned tmem = tmem_slot;
    constexpr unsigned idesc = umma_idesc_bf16(kTileM, kTileN) | (1u << 15) | (1u << 16);   // both MN-major
    bool ok = true;
    for (int c = 0; c < chunks; ++c) {
        cp_async_wait_pending<kWgSlots - 2>();
        fence_async_smem();
        __syncthreads();
        if (tid == 0) {
            fence_after_sync();
            const unsigned sa = smem_u32(smem + (c % kWgSlots) * 2 * kWgChunk);
#pragma unroll
            for (int s = 0; s < kWgRows / 16; ++s)   // K step s: two atoms of 8 rows
                umma_bf16(tmem, umma_desc_sw128(sa + s * 2048, kWgChunk / 2, 1024),
                          umma_desc_sw128(sa + kWgChunk + s * 2048, kWgChunk / 2, 1024), idesc, c > 0 || s > 0 ? 1u : 0u);
            umma_commit(&done[c % kWgSlots]);
        }
        // the slot of the chunk before takes the next chunk to come once its MMAs are done
        const int next = c + kWgSlots - 1;
        if (next < chunks) {
            if (c > 0 && !mbar_wait(&done[(c - 1) % kWgSlots], ((c - 1) / kWgSlots) & 1, kWaitPolls)) ok = false;
            if (ok) stage(next);
        }
        cp_async_commit();
    }
    cp_async_wait_pending<0>();   // none is left after a full run; after a wait that gave up, no copy may outlive the CTA
    if (!mbar_wait(&done[(chunks - 1) % kWgSlots], ((chunks - 1) / kWgSlots) & 1, polls)) {
        ok = false;
        mbar_wait(&done[(chunks - 1) % kWgSlots], ((chunks - 1) / kWgSlots) & 1, kWaitPolls);   // the committed MMAs finish first
    }
    if (!ok && lane == 0) atomicOr(err, 1);
    ok = __syncthreads_and(ok);
    fence_after_sync();
    if (ok) {
        const int row = (warp & 3) * 32 + lane, c0 = (warp >> 2) * (kTileN / 2);   // TMEM lane = tile row
        float* dst = out + (size_t)blockIdx.z * kH * kH + (size_t)(m0 + row) * kH + n0 + c0;
#pragma unroll
        for (int h = 0; h < kTileN / 2; h += 32) {
            float v[32];
            tmem_ld32(tmem + ((unsigned)((warp & 3) * 32) << 16) + c0 + h, v);
#pragma unroll
            for (int q = 0; q < 32; q += 4)
                *reinterpret_cast<float4*>(dst + h + q) = make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]);
        }
    }
    fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kTileN);
}

// GEMM of a large batch's hidden layer in a training step, persistent: each CTA takes one 128-column half of the
// layer (its 128 x 256 slice of the weights stays in shared memory, 64 KB)
// and walks row tiles blockIdx.x, blockIdx.x + gridDim.x, ...  The next
// tile's 128 x 256 activations are copied (cp.async) into the second of two
// 64 KB buffers while the MMAs and the epilogue of the current tile run.
// Same staging layout, MMAs and epilogue arithmetic as mlp_gemm_kernel<EPI>
// (kEpiFwd or kEpiBwd).
// Thirty-two warps: eight per quarter of the TMEM lanes, each taking 16 of
// the tile's 128 columns in the epilogue (with 16 warps of 32 columns each,
// fewer warps hide the activation's latency: about 1 % slower training).
constexpr int kPersistSmem = (kTileN + 2 * kTileM) * kKC * 2;   // 192 KB
constexpr int kPersistThreads = 1024;
constexpr int kPersistParts = kPersistThreads / 128;            // column parts per TMEM lane quarter

// RED (backward only) adds the sums over each row tile that the next
// gradients need, so that no separate pass re-reads dz: RED = 1 the column
// sums of dz (a bias gradient), RED = 5 also the sums of dz times each of the
// four inputs xin (rows x 4, the first layer's weight gradient), both from
// the FP32 values before dz is rounded to BF16.  Tile t's sums go to
// red[t * RED * 256 ..]: for RED = 5 the 4 x 256 weight-gradient entries
// (feature-major) then the 256 bias-gradient entries, the layout of W1, b1
// in the parameter vector.  Each lane sums its rows in order, a fixed
// shuffle tree combines the lanes of a warp, the CTA adds its four row
// quarters in order, and the tiles are summed afterwards in a fixed order.
template <int EPI, int RED = 0>
__global__ void __launch_bounds__(kPersistThreads)
mlp_persistent_kernel(const bf16* __restrict__ A, int lda, const bf16* __restrict__ B, int ldb, int tiles,
                      const float* __restrict__ bias, float* __restrict__ zout, const float* __restrict__ zin,
                      bf16* __restrict__ hout, const float* __restrict__ xin, float* __restrict__ red,
                      int* __restrict__ err, int polls)
{
    static_assert(RED == 0 || (EPI == kEpiBwd && (RED == 1 || RED == 5)), "tile sums of the backward pass");
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char* sB = smem;                                  // 128 x 256
    unsigned char* sA[2] = {smem + kTileN * kKC * 2, smem + (kTileN + kTileM) * kKC * 2};
    __shared__ unsigned tmem_slot;
    __shared__ __align__(8) unsigned long long mbar;
    __shared__ float sBias[kTileN];                              // this CTA's 128 biases
    __shared__ float sRed[4][RED > 0 ? RED * kTileN : 1];        // per row quarter: the tile sums
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n0 = blockIdx.y * kTileN;
    if (EPI == kEpiFwd && tid < kTileN) sBias[tid] = bias[n0 + tid];
    if (warp == 0) tmem_alloc(&tmem_slot, kTileN);
    if (tid == 0) mbar_init(&mbar);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const unsigned tmem = tmem_slot;
    stage_rows<kPersistThreads>(sB, B, (size_t)ldb, (size_t)n0);
    int t = blockIdx.x;
    if (t < tiles) stage_rows<kPersistThreads>(sA[0], A, (size_t)lda, (size_t)t * kTileM);
    cp_async_wait_all();
    fence_async_smem();
    __syncthreads();

    int phase = 0, buf = 0;
    bool ok = true;
    for (; t < tiles; t += gridDim.x, buf ^= 1) {
        if (tid == 0) {
            fence_after_sync();
            mma_rows(tmem, sA[buf], sB);
            umma_commit(&mbar);
        }
        // the next tile's activations, into the other buffer (its last
        // reader, the previous tile's MMAs, has completed)
        const int tn = t + gridDim.x;
        if (tn < tiles) stage_rows<kPersistThreads>(sA[buf ^ 1], A, (size_t)lda, (size_t)tn * kTileM);
        if (!mbar_wait(&mbar, phase, polls)) {
            ok = false;
            if (lane == 0) atomicOr(err, 1);
            mbar_wait(&mbar, phase, kWaitPolls);   // the committed MMAs finish first
        }
        phase ^= 1;
        fence_after_sync();
        if (!__syncthreads_and(ok)) {
            cp_async_wait_all();   // no copy may outlive the CTA
            break;
        }
        // Each warp takes a 32-row x kCols-column block of the accumulator
        // (TMEM lane = tile row, so the load gives lane l row l).  The block
        // passes through shared memory -- the current tile's activation
        // buffer, whose last reader, the MMAs, has completed -- so that in
        // step k lane l holds row kRps k + l / kLpr and the four columns from
        // 4 (l % kLpr): the global loads and stores then cover whole row
        // segments instead of one 16-byte piece of 32 rows.  The 16-byte
        // chunks of a row are XOR-swizzled so that both passes are free of
        // bank conflicts.
        const int quarter = warp & 3, part = warp >> 2;
        constexpr int kCols = kTileN / kPersistParts;   // columns per warp: one TMEM load, one wait
        constexpr int kLpr = kCols / 4;                 // lanes per row (16-byte chunks of a row)
        constexpr int kRps = 32 / kLpr;                 // rows per step
        static_assert(kCols == 16 || kCols == 32, "one 16- or 32-column TMEM load per thread");
        static_assert(kPersistThreads / 32 * 32 * kCols * 4 <= kTileM * kKC * 2, "scratch fits the A buffer");
        const int c0 = part * kCols, rr = lane / kLpr, cc = lane % kLpr;
        float* S = (float*)sA[buf] + warp * 32 * kCols;
        const size_t g0 = ((size_t)t * kTileM + quarter * 32 + rr) * kH + n0 + c0 + 4 * cc;
        auto goff = [&](int k) { return g0 + (size_t)(kRps * k) * kH; };
        auto sw = [](int row, int c) { return row * kCols + ((c ^ ((row / (8 / kLpr)) % kLpr)) << 2); };
        float cs[4] = {0.0f, 0.0f, 0.0f, 0.0f}, cw[4][4] = {};   // RED: column sums, times x
        float4 zi[kLpr];
        if (EPI == kEpiBwd) {
            // the pre-activations are loaded before the accumulator's wait
#pragma unroll
            for (int k = 0; k < kLpr; ++k) zi[k] = *(const float4*)(zin + goff(k));
        }
        {
            float v[kCols];
            const unsigned ta = tmem + ((unsigned)(quarter * 32) << 16) + c0;
            if constexpr (kCols == 32) tmem_ld32(ta, v);
            else tmem_ld16(ta, v);
#pragma unroll
            for (int c = 0; c < kLpr; ++c)
                *(float4*)(S + sw(lane, c)) = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < kLpr; ++k) {
            const float4 a = *(const float4*)(S + sw(kRps * k + rr, cc));
            float y[4];
            if (EPI == kEpiFwd) {
                const float4 z = make_float4(a.x + sBias[c0 + 4 * cc], a.y + sBias[c0 + 4 * cc + 1],
                                             a.z + sBias[c0 + 4 * cc + 2], a.w + sBias[c0 + 4 * cc + 3]);
                *(float4*)(zout + goff(k)) = z;
                y[0] = gelu(z.x); y[1] = gelu(z.y); y[2] = gelu(z.z); y[3] = gelu(z.w);
            } else {
                y[0] = a.x * gelu_grad(zi[k].x); y[1] = a.y * gelu_grad(zi[k].y);
                y[2] = a.z * gelu_grad(zi[k].z); y[3] = a.w * gelu_grad(zi[k].w);
                if (RED > 0) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) cs[i] += y[i];
                }
                if (RED == 5) {
                    const float4 xk = *(const float4*)(xin + 4 * ((size_t)t * kTileM + quarter * 32 + kRps * k + rr));
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        cw[i][0] += y[i] * xk.x; cw[i][1] += y[i] * xk.y;
                        cw[i][2] += y[i] * xk.z; cw[i][3] += y[i] * xk.w;
                    }
                }
            }
            if (RED != 5) {
                const __nv_bfloat162 p0 = __floats2bfloat162_rn(y[0], y[1]), p1 = __floats2bfloat162_rn(y[2], y[3]);
                *(uint2*)(hout + goff(k)) = make_uint2(*(const unsigned*)&p0, *(const unsigned*)&p1);
            }
        }
        if (RED > 0) {
            // lanes with the same columns (equal lane % kLpr) hold the other rows
#pragma unroll
            for (int o = kLpr; o < 32; o <<= 1) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    cs[i] += __shfl_xor_sync(0xffffffffu, cs[i], o);
                    if (RED == 5) {
#pragma unroll
                        for (int d = 0; d < 4; ++d) cw[i][d] += __shfl_xor_sync(0xffffffffu, cw[i][d], o);
                    }
                }
            }
            if (rr == 0) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int col = c0 + 4 * cc + i;
                    if (RED == 5) {
#pragma unroll
                        for (int d = 0; d < 4; ++d) sRed[quarter][col * 4 + d] = cw[i][d];
                        sRed[quarter][4 * kTileN + col] = cs[i];
                    } else {
                        sRed[quarter][col] = cs[i];
                    }
                }
            }
        }
        // the epilogue's TMEM reads finish before the next tile's MMAs
        // overwrite the accumulator; the next activations must have landed
        cp_async_wait_all();
        fence_async_smem();
        fence_before_sync();
        __syncthreads();
        if (RED > 0) {
            // the four row quarters in order (read before the next tile's
            // epilogue, which follows the next block-wide barrier, writes sRed)
            float* rt = red + (size_t)t * (RED * kH);
            for (int i = tid; i < RED * kTileN; i += kPersistThreads) {
                const float v = ((sRed[0][i] + sRed[1][i]) + sRed[2][i]) + sRed[3][i];
                const size_t gi = RED == 5 ? (i < 4 * kTileN ? (size_t)n0 * 4 + i : (size_t)4 * kH + n0 + (i - 4 * kTileN))
                                           : (size_t)n0 + i;
                rt[gi] = v;
            }
        }
    }
    fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kTileN);
}

// The network's inference in one kernel: a CTA takes 128 rows at a time
// through all four layers, so that no activation leaves the SM.  The 128 x 256
// activations sit in shared memory (64 KB, the MMAs' core-matrix layout), the
// accumulators in TMEM (256 columns), and the 256 x 256 weights of the two
// hidden layers pass through a ring of four 8 KB slots, one K step of 16 each,
// by bulk copies that one thread issues three steps ahead (128 KB a layer and
// tile from L2, about 2.5 TB/s over the chip).  109 KB a CTA, so that two share
// an SM and one's activations cover the other's MMAs.
//
// What bounds it: the exact-erf GELU, 768 a row and 33 instructions each with
// its bias, rounding and store (9.4 ms of issue slots over the 13.8M nodes of
// 61^4); 62 % of the issue slots are busy, the rest is both CTAs waiting for
// MMAs at once.  14.9 ms over 61^4, where separate kernels for the inputs, the
// first layer, each hidden layer, the output layer and the write, passing the
// activations through memory, took 28.0 ms.  With a 32 KB slice of 64 columns
// at a time copied by every thread and a block barrier per slice 17.9 ms; with
// the ring's addresses formed in the issuing thread's loop 16.3 ms.
//
// Same arithmetic as the training step's kernels, in the same order: the
// first layer's FMA chain, K accumulated in steps of 16 from 0, the output
// layer's sums over groups of eight features combined by the tree a warp
// shuffle gives (features 8 g .. 8 g + 7 are group g; groups g and g + 16, then
// g and g + 8, ... are added).
//
// GRID: rows are the stored nodes of a grid, whose normalised coordinates
// come from the table coord (4 x kCoordStride, per dimension), and the outputs
// become the node's value M clamp(y_0, 0, 1) (0 on target nodes) and the code
// of atan2(y_2, y_1); otherwise rows are x (rows x 4) and the outputs go to y
// (rows x 3).
constexpr int kInferThreads = 512;
constexpr int kInferSlots = 4;                                     // ring of weight K steps
constexpr int kInferStep = kH * 16 * 2;                            // bytes of one: 256 rows x 16 columns
constexpr int kInferSteps = kH / 16;                               // per layer
constexpr int kInferSmemA = kTileM * kKC * 2, kInferSmemW = kInferSlots * kInferStep;
constexpr int kInferSmemF = 4 * kH + kH + kH + kH + 3 * kH + 4;    // W1 (by input), b1, b2, b3, W4, b4
constexpr int kInferSmem = kInferSmemA + kInferSmemW + (kInferSmemF + 9 * kTileM) * 4;

struct InferGrid {
    const float* coord;
    double M;
    void* V;
    uint16_t* code;
    int fp32;
};

// Weights of both hidden layers as the ring's steps: step s of a layer holds
// columns 16 s .. 16 s + 15 as core matrices (8 rows x 16 bytes), row block rb
// and K block kb at (rb * 2 + kb) * 128.  One thread per 16 bytes.
__global__ void infer_weights_kernel(const bf16* __restrict__ W2, const bf16* __restrict__ W3,
                                     uint4* __restrict__ out)
{
    const int v = blockIdx.x * blockDim.x + threadIdx.x;           // 2 x 16 x 512
    const int layer = v >> 13, s = (v >> 9) & 15, rb = (v >> 4) & 31, kb = (v >> 3) & 1, row = rb * 8 + (v & 7);
    out[v] = *reinterpret_cast<const uint4*>((layer ? W3 : W2) + (size_t)row * kH + s * 16 + kb * 8);
}

__global__ void coord_table_kernel(const Geo<double> g, Box4 nlo, Box4 nhi, float* __restrict__ coord)
{
    const int d = blockIdx.x, i = threadIdx.x;
    if (i >= g.n[d]) return;
    const double lo[4] = {nlo.x, nlo.y, nlo.z, nlo.w}, hi[4] = {nhi.x, nhi.y, nhi.z, nhi.w};
    const double xd = g.lo[d] + (double)i * g.h[d];
    coord[d * kCoordStride + i] = (float)(2.0 * (xd - lo[d]) / (hi[d] - lo[d]) - 1.0);
}

// GELU of a pair: gelu() of each, the plain multiplications and the addition
// two at a time.
__device__ __forceinline__ unsigned long long gelu2(unsigned long long z)
{
    float a, b;
    unpack2(mul2(z, pack2(kInvSqrt2, kInvSqrt2)), a, b);
    return mul2(mul2(z, pack2(0.5f, 0.5f)), add2(pack2(1.0f, 1.0f), pack2(erff(a), erff(b))));
}

// Eight consecutive floats of shared memory (16-byte aligned) as four pairs.
__device__ __forceinline__ void lds8(const float* p, unsigned long long q[4])
{
    const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(p), b = *reinterpret_cast<const ulonglong2*>(p + 4);
    q[0] = a.x; q[1] = a.y; q[2] = b.x; q[3] = b.y;
}

template <bool GRID>
__global__ void __launch_bounds__(kInferThreads, 2)
mlp_infer_kernel(const __grid_constant__ Geo<double> g, const __grid_constant__ InferGrid ig,
                 const float* __restrict__ x, const float* __restrict__ P, const unsigned char* __restrict__ Wsteps,
                 int count, float* __restrict__ y, int* __restrict__ err, int polls)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char* sA = smem;
    unsigned char* sW = smem + kInferSmemA;
    float* sW1 = reinterpret_cast<float*>(smem + kInferSmemA + kInferSmemW);     // 4 x 256, by input
    float* sB1 = sW1 + 4 * kH;
    float* sB2 = sB1 + kH;
    float* sB3 = sB2 + kH;
    float* sW4 = sB3 + kH;                                                       // 3 x 256, then b4
    float* sT = sW4 + 3 * kH + 4;                                                // 3 outputs x parts 1..3 x 128
    __shared__ unsigned tmem_slot;
    __shared__ int s_fail;
    __shared__ __align__(8) unsigned long long mbar, full[kInferSlots], empty[kInferSlots];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int r = tid & (kTileM - 1), part = tid >> 7;             // row (TMEM lane), column part 0..3

    for (int i = tid; i < 4 * kH; i += kInferThreads) sW1[(i & 3) * kH + (i >> 2)] = P[kOffW1 + i];
    for (int i = tid; i < kH; i += kInferThreads) {
        sB1[i] = P[kOffB1 + i];
        sB2[i] = P[kOffB2 + i];
        sB3[i] = P[kOffB3 + i];
    }
    for (int i = tid; i < 3 * kH + 3; i += kInferThreads) sW4[i] = P[kOffW4 + i];
    if (warp == 0) tmem_alloc(&tmem_slot, kH);
    if (tid == 0) {
        s_fail = 0;
        mbar_init(&mbar);
        for (int b = 0; b < kInferSlots; ++b) {
            mbar_init(&full[b]);
            mbar_init(&empty[b]);
        }
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const unsigned tmem = tmem_slot;
    constexpr unsigned idesc = umma_idesc_bf16(kTileM, kTileN);
    const int tiles = (int)(((long long)count + kTileM - 1) / kTileM);

    // The ring: step s of either layer sits in slot s mod 4 (a layer has 16
    // steps, so slots and phase parities repeat layer by layer and are
    // constants of the unrolled loop).  Thread 0 issues the copies and the
    // MMAs; `left` counts the steps of this CTA not yet requested, `next` is
    // the next one's address.
    const int my_tiles = (tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    long long left = 2LL * kInferSteps * my_tiles;
    const unsigned char* next = Wsteps;
    auto load = [&](int b) {
        mbar_expect_bytes(&full[b], kInferStep);
        bulk_copy(sW + b * kInferStep, next, kInferStep, &full[b]);
        next += kInferStep;
        if (next == Wsteps + 2 * kInferSteps * kInferStep) next = Wsteps;
        --left;
    };
    if (tid == 0) {
#pragma unroll
        for (int b = 0; b < kInferSlots; ++b) load(b);   // a layer has more steps than the ring
    }
    const unsigned long long adesc = umma_desc(smem_u32(sA), 128, kKC / 8 * 128);
    const unsigned long long bdesc = umma_desc(smem_u32(sW), 128, 256);

    int phase = 0;
    bool first = true;
    // One hidden layer: acc = sA W^T.  False after a wait that gave up.
    auto layer = [&]() -> bool {
        fence_async_smem();
        fence_before_sync();
        __syncthreads();
        if (tid == 0) {
            fence_after_sync();
            bool fine = true;
#pragma unroll
            for (int s = 0; s < kInferSteps; ++s) {
                const int b = s % kInferSlots, p = (s + kInferSteps - 1) % kInferSteps;   // p: the step before
                fine = fine && mbar_wait(&full[b], (s / kInferSlots) & 1, kWaitPolls);
                if (fine) {
#pragma unroll
                    for (int h = 0; h < kH / kTileN; ++h)
                        umma_bf16(tmem + h * kTileN, adesc + s * (256 / 16),
                                  bdesc + (b * kInferStep + h * kTileN * 32) / 16, idesc, s > 0 ? 1u : 0u);
                    umma_commit(&empty[b]);
                    // the slot before this one takes its next step once its MMAs are done
                    if (!(first && s == 0) && left > 0) {
                        fine = mbar_wait(&empty[p % kInferSlots], (p / kInferSlots) & 1, kWaitPolls);
                        if (fine) load(p % kInferSlots);
                    }
                }
            }
            if (!fine) s_fail = 1;
            umma_commit(&mbar);
        }
        first = false;
        bool ok = true;
        if (!mbar_wait(&mbar, phase, polls)) {
            ok = false;
            if (lane == 0) atomicOr(err, 1);
            mbar_wait(&mbar, phase, kWaitPolls);   // the committed MMAs finish first
        }
        phase ^= 1;
        fence_after_sync();
        ok = __syncthreads_and(ok);
        if (s_fail) {
            if (tid == 0) atomicOr(err, 1);
            ok = false;
        }
        return ok;
    };
    // 16 bytes (eight features from 8 kb) of this row's activations
    auto store8 = [&](int kb, const unsigned long long h[4]) {
        unsigned u[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float a, b;
            unpack2(h[q], a, b);
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(a, b);
            u[q] = *reinterpret_cast<const unsigned*>(&h2);
        }
        *reinterpret_cast<uint4*>(sA + (size_t)((r >> 3) * (kKC / 8) + kb) * 128 + (r & 7) * 16) =
            make_uint4(u[0], u[1], u[2], u[3]);
    };
    // pre-activations of eight features: accumulator plus bias
    const unsigned trow = tmem + ((unsigned)((warp & 3) * 32) << 16);
    auto pre8 = [&](int kb, const float* bias, unsigned long long z[4]) {
        float v[8];
        unsigned long long b[4];
        tmem_ld8(trow + kb * 8, v);
        lds8(bias + kb * 8, b);
#pragma unroll
        for (int q = 0; q < 4; ++q) z[q] = add2(pack2(v[2 * q], v[2 * q + 1]), b[q]);
    };
#pragma unroll 1
    for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
        const long long s = (long long)t * kTileM + r;
        const bool live = s < count;
        int id[4] = {0, 0, 0, 0};
        float4 xs = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (live) {
            if constexpr (GRID) {
                decode_node(g, (int)s, id);
                xs = make_float4(__ldg(ig.coord + id[0]), __ldg(ig.coord + kCoordStride + id[1]),
                                 __ldg(ig.coord + 2 * kCoordStride + id[2]), __ldg(ig.coord + 3 * kCoordStride + id[3]));
            } else {
                xs = *reinterpret_cast<const float4*>(x + 4 * s);
            }
        }
        {
            const unsigned long long xx[4] = {pack2(xs.x, xs.x), pack2(xs.y, xs.y), pack2(xs.z, xs.z),
                                              pack2(xs.w, xs.w)};
#pragma unroll 1
            for (int k = 0; k < kH / 32; ++k) {
                const int kb = part * (kH / 32) + k;
                unsigned long long z[4], w[4];
                lds8(sB1 + kb * 8, z);
#pragma unroll
                for (int d = 0; d < 4; ++d) {
                    lds8(sW1 + d * kH + kb * 8, w);
#pragma unroll
                    for (int q = 0; q < 4; ++q) z[q] = fma2(w[q], xx[d], z[q]);
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) z[q] = gelu2(z[q]);
                store8(kb, z);
            }
        }
        if (!layer()) break;
#pragma unroll 1
        for (int k = 0; k < kH / 32; ++k) {
            const int kb = part * (kH / 32) + k;
            unsigned long long z[4];
            pre8(kb, sB2, z);
#pragma unroll
            for (int q = 0; q < 4; ++q) z[q] = gelu2(z[q]);
            store8(kb, z);
        }
        if (!layer()) break;
        // output layer: this thread's groups are part, part + 4, ..., taken in
        // the order that leaves the tree's partial sums fewest
        float T[3] = {0.0f, 0.0f, 0.0f};
        {
            float a4[3] = {}, a8[3] = {}, p16[3] = {};
#pragma unroll 1
            for (int k = 0; k < 8; ++k) {
                const int i = ((k & 1) << 2) | (k & 2) | (k >> 2);
                const int kb = part + 4 * i;
                unsigned long long z[4], w[3][4];
                pre8(kb, sB3, z);
#pragma unroll
                for (int o = 0; o < 3; ++o) lds8(sW4 + o * kH + kb * 8, w[o]);
                float p[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float h0, h1;
                    unpack2(gelu2(z[q]), h0, h1);
                    h0 = __bfloat162float(__float2bfloat16(h0));
                    h1 = __bfloat162float(__float2bfloat16(h1));
#pragma unroll
                    for (int o = 0; o < 3; ++o) {
                        float w0, w1;
                        unpack2(w[o][q], w0, w1);
                        p[o] = fmaf(w1, h1, fmaf(w0, h0, p[o]));
                    }
                }
#pragma unroll
                for (int o = 0; o < 3; ++o) {
                    if (!(k & 1)) {
                        p16[o] = p[o];
                    } else {
                        const float q16 = p16[o] + p[o];          // groups g, g + 16
                        if (!(k & 2)) {
                            a8[o] = q16;
                        } else {
                            const float q8 = a8[o] + q16;         // and g + 8, g + 24
                            if (!(k & 4)) a4[o] = q8;
                            else T[o] = a4[o] + q8;               // and g + 4, ...
                        }
                    }
                }
            }
        }
        // the four parts of a row meet in part 0; the others go on to the next tile
        if (part > 0) {
#pragma unroll
            for (int o = 0; o < 3; ++o) sT[(o * 3 + part - 1) * kTileM + r] = T[o];
        }
        __syncthreads();
        if (part == 0 && live) {
            float out[3];
#pragma unroll
            for (int o = 0; o < 3; ++o) {
                const float* q = sT + o * 3 * kTileM + r;
                out[o] = ((T[o] + q[kTileM]) + (q[0] + q[2 * kTileM])) + sW4[3 * kH + o];
            }
            if constexpr (GRID) {
                const double v = fmin(fmax((double)out[0], 0.0), 1.0) * ig.M;
                const bool tgt = in_target(g, id);
                if (ig.fp32) ((float*)ig.V)[s] = tgt ? 0.0f : (float)v;
                else ((double*)ig.V)[s] = tgt ? 0.0 : v;
                const double a = atan2((double)out[2], (double)out[1]);   // (-pi, pi]
                const long long c = llrint(a * (65536.0 / 6.283185307179586476925286766559));
                ig.code[s] = (uint16_t)(c & 65535);
            } else {
#pragma unroll
                for (int o = 0; o < 3; ++o) y[3 * s + o] = out[o];
            }
        }
    }
    if (tid == 0 && left > 0) {
        // a wait gave up: no copy may outlive the CTA.  The slots' last copies
        // were those of the layer's last four steps, or of the next layer's
        // first three and the last: every slot's copy of the current phase
#pragma unroll
        for (int b = 0; b < kInferSlots; ++b) mbar_wait(&full[b], b < kInferSlots - 1 ? 0 : 1, kWaitPolls);
    }
    fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kH);
}

// Training-step state in device memory, so that one captured step can be
// replayed: the epoch's permutation (mult, offset), the first sample of the
// step, and the Adam step count.
struct TrainState {
    long long mult, offset, start;
    int t;
    float lr;        // > 0: the epoch's Adam step size (replaces the kernel argument)
};

// Arbitrary states (device, n x 4 double) normalised to [-1, 1]^4.
__global__ void states_in_kernel(const double* __restrict__ s, int count, Box4 lo, Box4 hi,
                                 float* __restrict__ x)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    x[4 * i + 0] = (float)(2.0 * (s[4 * i + 0] - lo.x) / (hi.x - lo.x) - 1.0);
    x[4 * i + 1] = (float)(2.0 * (s[4 * i + 1] - lo.y) / (hi.y - lo.y) - 1.0);
    x[4 * i + 2] = (float)(2.0 * (s[4 * i + 2] - lo.z) / (hi.z - lo.z) - 1.0);
    x[4 * i + 3] = (float)(2.0 * (s[4 * i + 3] - lo.w) / (hi.w - lo.w) - 1.0);
}

// The nodes a training step's batch is drawn from.
struct TrainGrid {
    const void* V;
    const uint16_t* code;
    const double2 *tab_hi, *tab_lo;
    const float* coord;    // normalised node coordinates (coord_table_kernel)
    long long n;
    double invM;
    const TrainState* ts;
};

// Layer 1 (4 -> 256) with GELU of a training step, z1 and h1 stored, and with
// GRID the batch itself: inputs (normalised to the network's box) and targets
// (V / M, cos, sin) of nodes idx = (mult * (start + i) + offset) mod n of the
// grid (a seeded permutation; S: the values' type), kept in x and t for the
// backward pass; otherwise x is read.  A block takes kL1Rows rows: a thread a
// row for the batch, then two features of half the rows, whose weights stay in
// its registers, so that a warp stores whole row segments.
// The separate batch kernel took 11.1 us for 16,384 rows, bound by its four
// FP64 divisions a row on the 64 SMs it filled; the coordinates now come from a
// table, and with a warp per row the first layer took another 10.3 us.  Both
// in one: 9.6 us.
constexpr int kL1Rows = 16;

template <bool GRID, typename S>
__global__ void __launch_bounds__(256) first_layer_kernel(const __grid_constant__ Geo<double> g, const TrainGrid tg,
                                                          const float* __restrict__ P, float4* __restrict__ x,
                                                          float* __restrict__ t, float* __restrict__ z1,
                                                          bf16* __restrict__ h1)
{
    __shared__ float4 sx[kL1Rows];
    const int tid = threadIdx.x, o = 2 * (tid & 127);
    const size_t s0 = (size_t)blockIdx.x * kL1Rows;
    const float4 w0 = *reinterpret_cast<const float4*>(P + kOffW1 + 4 * o);
    const float4 w1 = *reinterpret_cast<const float4*>(P + kOffW1 + 4 * o + 4);
    const float2 b = *reinterpret_cast<const float2*>(P + kOffB1 + o);
    if (GRID) {
        // one warp the inputs, another the targets
        const int w = tid >> 5, i = tid & 31;
        if (w < 2 && i < kL1Rows) {
            const size_t row = s0 + i;
            const long long j = (long long)(((unsigned long long)tg.ts->mult * (unsigned long long)(tg.ts->start + (long long)row) +
                                             (unsigned long long)tg.ts->offset) % (unsigned long long)tg.n);
            if (w == 0) {
                int id[4];
                decode_node(g, (int)j, id);
                const float4 v = make_float4(__ldg(tg.coord + id[0]), __ldg(tg.coord + kCoordStride + id[1]),
                                             __ldg(tg.coord + 2 * kCoordStride + id[2]), __ldg(tg.coord + 3 * kCoordStride + id[3]));
                sx[i] = v;
                x[row] = v;
            } else {
                const double vj = (double)((const S*)tg.V)[j];
                const int c = tg.code[j];
                const double2 hi = tg.tab_hi[c >> 8], lo = tg.tab_lo[c & 255];
                t[3 * row + 0] = (float)(vj * tg.invM);
                t[3 * row + 1] = (float)(hi.y * lo.y - hi.x * lo.x);   // cos
                t[3 * row + 2] = (float)(hi.x * lo.y + hi.y * lo.x);   // sin
            }
        }
    } else if (tid < kL1Rows) {
        sx[tid] = x[s0 + tid];
    }
    __syncthreads();
#pragma unroll 2
    for (int k = tid >> 7; k < kL1Rows; k += 2) {
        const float4 v = sx[k];
        const size_t at = (s0 + k) * kH + o;
        const float za = fmaf(w0.w, v.w, fmaf(w0.z, v.z, fmaf(w0.y, v.y, fmaf(w0.x, v.x, b.x))));
        const float zb = fmaf(w1.w, v.w, fmaf(w1.z, v.z, fmaf(w1.y, v.y, fmaf(w1.x, v.x, b.y))));
        *reinterpret_cast<float2*>(z1 + at) = make_float2(za, zb);
        *reinterpret_cast<__nv_bfloat162*>(h1 + at) = __floats2bfloat162_rn(gelu(za), gelu(zb));
    }
}

// The output layer of a training step with the first part of its backward
// pass, one warp per sample (grid-stride over the samples): y = W4 h3 + b4,
// the loss gradient dy = 2 (y - t) / (3 B), the loss sum, the output layer's
// gradients dW4 = dy h3^T and db4 = sum dy, and dz3 = (dy W4) * GELU'(z3) for
// the lane's 8 features with its sum db3 (FP32, before the BF16 rounding of
// dz3).  Each lane sums its samples in order, the block sums its warps in
// order, and the block's sums go to part[blockIdx.x] for a reduction in a
// fixed order: db3, dW4, db4 (laid out as b3, W4, b4 are in the parameter
// vector), then the loss.
constexpr int kOutPart = 4 * kH + 4;
__global__ void __launch_bounds__(256) out_train_kernel(const bf16* __restrict__ h3, const float* __restrict__ P,
                                                        const float* __restrict__ t, const float* __restrict__ z3,
                                                        int count, float inv_n, bf16* __restrict__ dz3,
                                                        float* __restrict__ part)
{
    __shared__ float sW[3 * kH + 3];
    __shared__ float sP[8][kOutPart];   // per warp: db3, dW4, db4, loss
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int warps = (int)((gridDim.x * (size_t)blockDim.x) >> 5);
    int s = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5);
    // a sample's h3, z3 and targets, loaded while the one before is worked on
    // (a warp takes about seven at a batch of 16,384, each a chain of loads,
    // sums and shuffles: 14.9 us, 16.6 without)
    uint4 hn = make_uint4(0, 0, 0, 0);
    float4 za = make_float4(0.0f, 0.0f, 0.0f, 0.0f), zb = za;
    float tn[3] = {};
    auto fetch = [&](int q) {
        if (q >= count) return;
        hn = *reinterpret_cast<const uint4*>(h3 + (size_t)q * kH + lane * 8);
        const float4* zp = reinterpret_cast<const float4*>(z3 + (size_t)q * kH + lane * 8);
        za = zp[0];
        zb = zp[1];
#pragma unroll
        for (int k = 0; k < 3; ++k) tn[k] = t[3 * (size_t)q + k];
    };
    fetch(s);
    for (int i = threadIdx.x; i < 3 * kH + 3; i += blockDim.x) sW[i] = P[kOffW4 + i];
    __syncthreads();
    float w[3][8] = {}, b[3] = {}, d3[8] = {}, l = 0.0f;
    for (; s < count; s += warps) {
        float a[8];
        row8(hn, a);
        const float z[8] = {za.x, za.y, za.z, za.w, zb.x, zb.y, zb.z, zb.w}, ts[3] = {tn[0], tn[1], tn[2]};
        fetch(s + warps);
        float dy[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            float sum = 0.0f;
#pragma unroll
            for (int q = 0; q < 8; ++q) sum += sW[k * kH + lane * 8 + q] * a[q];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            const float r = (sum + sW[3 * kH + k]) - ts[k];
            l += r * r;
            dy[k] = 2.0f * r * inv_n;
            b[k] += dy[k];
#pragma unroll
            for (int q = 0; q < 8; ++q) w[k][q] += dy[k] * a[q];
        }
        unsigned u[4];
#pragma unroll
        for (int q = 0; q < 8; q += 2) {
            const int i = lane * 8 + q;
            const float g0 = dy[0] * sW[i] + dy[1] * sW[kH + i] + dy[2] * sW[2 * kH + i];
            const float g1 = dy[0] * sW[i + 1] + dy[1] * sW[kH + i + 1] + dy[2] * sW[2 * kH + i + 1];
            const float e0 = g0 * gelu_grad(z[q]), e1 = g1 * gelu_grad(z[q + 1]);
            d3[q] += e0;
            d3[q + 1] += e1;
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(e0, e1);
            u[q / 2] = *reinterpret_cast<const unsigned*>(&h2);
        }
        *reinterpret_cast<uint4*>(dz3 + (size_t)s * kH + lane * 8) = make_uint4(u[0], u[1], u[2], u[3]);
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) sP[warp][lane * 8 + q] = d3[q];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
#pragma unroll
        for (int q = 0; q < 8; ++q) sP[warp][kH + k * kH + lane * 8 + q] = w[k][q];
    }
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < 3; ++k) sP[warp][4 * kH + k] = b[k];
        sP[warp][4 * kH + 3] = l;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kOutPart; i += blockDim.x) {
        float acc = 0.0f;
#pragma unroll
        for (int k = 0; k < 8; ++k) acc += sP[k][i];
        part[(size_t)blockIdx.x * kOutPart + i] = acc;
    }
}

// Per-feature reductions over a chunk of samples (thread = feature), for
// batches below kManyRows rows (larger ones are summed per tile in the
// persistent backward GEMM's epilogue), in
// sample order:  db[o] = sum_s dz[s][o];  with X = 4 also
// dW[o][d] = sum_s dz[s][o] x[s][d].  Block b writes its sums to
// part[b][0 .. 4 X + ... ): dW (256 X values, feature-major) then db (256),
// for a reduction in a fixed order.  X (0 or 4) is a template argument so
// that the accumulators stay in registers; the inputs x of each 256-sample
// slice of the chunk are staged in shared memory.
template <int X>
__global__ void feat_reduce_kernel(const bf16* __restrict__ dz, const float* __restrict__ x, int rows, int chunk,
                                   float* __restrict__ part)
{
    __shared__ float4 sx[X == 4 ? 256 : 1];
    const int o = threadIdx.x;   // 256 threads
    const int s0 = blockIdx.x * chunk, s1 = min(rows, s0 + chunk);
    float b = 0.0f, w[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (int sb = s0; sb < s1; sb += 256) {
        const int se = min(s1, sb + 256);
        if constexpr (X == 4) {
            __syncthreads();
            if (sb + o < se) sx[o] = reinterpret_cast<const float4*>(x)[sb + o];
            __syncthreads();
        }
#pragma unroll 8
        for (int s = sb; s < se; ++s) {
            const float g = __bfloat162float(dz[(size_t)s * kH + o]);
            b += g;
            if constexpr (X == 4) {
                const float4 xs = sx[s - sb];
                w[0] += g * xs.x;
                w[1] += g * xs.y;
                w[2] += g * xs.z;
                w[3] += g * xs.w;
            }
        }
    }
    float* pb = part + (size_t)blockIdx.x * (kH * X + kH);
    if constexpr (X == 4) {
#pragma unroll
        for (int d = 0; d < 4; ++d) pb[o * 4 + d] = w[d];
    }
    pb[kH * X + o] = b;
}

// Adam (Kingma and Ba) on the FP32 master parameters, writing the BF16 copies of
// W2, W3 and their transposes used by the tensor-core GEMMs as it goes.  The
// step count t (1 for the first step) comes from device memory; the bias
// corrections are 1 - beta^t.
struct AdamArgs {
    float *P, *m, *v;
    float lr, b1, b2, eps;
    TrainState* ts;
    bf16 *W2, *W3, *W2T, *W3T;
    unsigned* arrive;
    int advance;
};

__device__ __forceinline__ void adam_update(const AdamArgs& a, int i, float g)
{
    const float tf = (float)a.ts->t;
    const float lr = a.ts->lr > 0.0f ? a.ts->lr : a.lr;
    const float bc1 = 1.0f - powf(a.b1, tf), bc2 = 1.0f - powf(a.b2, tf);
    // rounded explicitly: the update is compiled into two kernels
    const float mi = fmaf(1.0f - a.b1, g, __fmul_rn(a.b1, a.m[i]));
    const float vi = fmaf(__fmul_rn(1.0f - a.b2, g), g, __fmul_rn(a.b2, a.v[i]));
    a.m[i] = mi;
    a.v[i] = vi;
    const float p = a.P[i] - lr * (mi / bc1) / (sqrtf(vi / bc2) + a.eps);
    a.P[i] = p;
    const bool w2 = i >= kOffW2 && i < kOffW2 + kH * kH, w3 = i >= kOffW3 && i < kOffW3 + kH * kH;
    if (w2 || w3) {
        const int e = i - (w2 ? kOffW2 : kOffW3), o = e / kH, c = e % kH;
        (w2 ? a.W2 : a.W3)[e] = __float2bfloat16(p);
        (w2 ? a.W2T : a.W3T)[c * kH + o] = __float2bfloat16(p);
    }
}

// A replayed training step: the last block to finish moves the step on -- the
// next step's first sample start += advance and t += 1 -- once every block has
// read t and the step size; *arrive counts the finished blocks and is back at 0
// afterwards.  Every thread of the block calls it.
__device__ __forceinline__ void adam_advance(const AdamArgs& a)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(a.arrive, 1u) == gridDim.x - 1) {
            a.ts->start += a.advance;
            a.ts->t += 1;
            *a.arrive = 0u;
        }
    }
}

__global__ void adam_kernel(const __grid_constant__ AdamArgs a, const float* __restrict__ G, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) adam_update(a, i, G[i]);
}

// Fixed-order reductions of per-block partial sums: the gradient of parameter
// at + i, i < len, is the sum over k of part[k * stride + i] (at < 0: the loss,
// which is added to *loss).  Long segments take a thread per output, which sums
// k in order; short ones with many partials a warp per output, lane l summing
// partials l, l + 32, ... in order before a fixed shuffle tree combines the
// lanes.  All of a step's reductions run in one launch, each segment in blocks
// of its own, and ADAM applies the gradients as they come (otherwise they go to
// G): in three launches of their own and Adam after them the sums took 12.3 us
// and Adam 6.1, all of it here 9.2.
struct RedSeg {
    const float* part;
    int n_part, stride, len, at;
    int end;      // blocks of this segment and the ones before it
};
constexpr int kRedSegs = 6, kRedLong = 8192;   // longer segments: a thread per output

struct RedSegs {
    RedSeg s[kRedSegs];
};

template <bool ADAM>
__global__ void __launch_bounds__(256)
reduce_kernel(const __grid_constant__ RedSegs segs, const __grid_constant__ AdamArgs a, float* __restrict__ G,
              float* __restrict__ loss)
{
    int q = 0;
#pragma unroll
    for (int k = 0; k < kRedSegs - 1; ++k) q += (int)blockIdx.x >= segs.s[k].end;
    const RedSeg r = segs.s[q];
    const int blk = (int)blockIdx.x - (q > 0 ? segs.s[q - 1].end : 0);
    auto put = [&](int i, float g) {
        if (r.at < 0) *loss += g;
        else if (ADAM) adam_update(a, r.at + i, g);
        else G[r.at + i] = g;
    };
    if (r.len > kRedLong) {
        const int i = blk * 256 + threadIdx.x;
        if (i < r.len) {
            float acc = 0.0f;
#pragma unroll 8
            for (int k = 0; k < r.n_part; ++k) acc += r.part[(size_t)k * r.stride + i];
            put(i, acc);
        }
    } else {
        const int i = (blk * 256 + (int)threadIdx.x) >> 5, lane = threadIdx.x & 31;
        if (i < r.len) {
            float acc = 0.0f;
            for (int k = lane; k < r.n_part; k += 32) acc += r.part[(size_t)k * r.stride + i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == 0) put(i, acc);
        }
    }
    if (ADAM) adam_advance(a);
}

// Sets the Adam step count (eager steps outside a replayed graph).
__global__ void set_step_kernel(TrainState* ts, int t)
{
    ts->t = t;
    ts->lr = 0.0f;   // the step size of the call
}

__global__ void bf16_weights_kernel(const float* __restrict__ P, bf16* __restrict__ W2, bf16* __restrict__ W3,
                                    bf16* __restrict__ W2T, bf16* __restrict__ W3T)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;   // kH * kH threads
    if (e >= kH * kH) return;
    const int o = e / kH, i = e % kH;
    W2[e] = __float2bfloat16(P[kOffW2 + e]);
    W3[e] = __float2bfloat16(P[kOffW3 + e]);
    W2T[i * kH + o] = __float2bfloat16(P[kOffW2 + e]);
    W3T[i * kH + o] = __float2bfloat16(P[kOffW3 + e]);
}

int fail_cuda(const char* what, cudaError_t e)
{
    char buf[256];
    snprintf(buf, sizeof buf, "%s: %s", what, cudaGetErrorString(e));
    return record_error(DP_ECUDA, buf);
}

#define MCK(call)                                                 \
    do {                                                          \
        cudaError_t e_ = (call);                                  \
        if (e_ != cudaSuccess) return fail_cuda(#call, e_);       \
    } while (0)

}  // namespace

struct dp_mlp {
    int device = 0;
    int sm_count = 1;
    cudaStream_t st = nullptr;
    int cap = 0;                       // activation rows (multiple of 512)
    double lo[4], hi[4];               // input box (normalisation)
    long long step = 0;
    float *P = nullptr, *G = nullptr, *Am = nullptr, *Av = nullptr;
    bf16 *W2b = nullptr, *W3b = nullptr, *W2T = nullptr, *W3T = nullptr;
    float *x = nullptr, *t = nullptr, *z1 = nullptr, *z2 = nullptr, *z3 = nullptr, *y = nullptr;
    bf16 *h1 = nullptr, *h2 = nullptr, *h3 = nullptr, *dz1 = nullptr, *dz2 = nullptr, *dz3 = nullptr;
    double* states = nullptr;
    unsigned char* Wsteps = nullptr;   // hidden weights as the inference kernel's K steps
    float* coord = nullptr;            // normalised node coordinates per dimension (4 x kCoordStride)
    float* loss = nullptr;
    // partial sums of the backward pass: the weight gradients' splits (W3, then
    // W2), the output layer's blocks, and the bias and first-layer gradients'
    // row tiles or blocks (1 and 5 x 256 floats each)
    float *part = nullptr, *out_part = nullptr, *red1 = nullptr, *red5 = nullptr;
    unsigned* arrive = nullptr;        // blocks of the Adam kernel that have finished (0 between launches)
    int* err = nullptr;
    float* h_loss = nullptr;           // pinned
    int* h_err = nullptr;
    int wait_polls = kWaitPolls;       // polls of the first wait for the MMAs (test hook)
    TrainState* ts = nullptr;          // training-step state (device)
    TrainState* h_ts = nullptr;        // pinned staging of its per-epoch values
    cudaStream_t cst = nullptr;        // private stream: training steps are captured and replayed there
    cudaEvent_t ev_in = nullptr, ev_out = nullptr;
};

namespace {

void free_mlp(dp_mlp* m)
{
    if (!m) return;
    cudaSetDevice(m->device);
    if (m->st) cudaStreamSynchronize(m->st);
    void* ps[] = {m->P, m->G, m->Am, m->Av, m->W2b, m->W3b, m->W2T, m->W3T, m->x, m->t, m->z1, m->z2, m->z3, m->y,
                  m->h1, m->h2, m->h3, m->dz1, m->dz2, m->dz3, m->states, m->Wsteps, m->coord, m->loss, m->part,
                  m->out_part, m->red1, m->red5, m->arrive, m->err};
    for (void* p : ps)
        if (p) cudaFree(p);
    if (m->h_loss) cudaFreeHost(m->h_loss);
    if (m->h_err) cudaFreeHost(m->h_err);
    if (m->ts) cudaFree(m->ts);
    if (m->h_ts) cudaFreeHost(m->h_ts);
    if (m->ev_in) cudaEventDestroy(m->ev_in);
    if (m->ev_out) cudaEventDestroy(m->ev_out);
    if (m->cst) cudaStreamDestroy(m->cst);
    delete m;
}

template <typename T>
cudaError_t malloc_n(T** p, size_t n)
{
    return cudaMalloc((void**)p, n * sizeof(T));
}

int refresh_bf16(dp_mlp* m)
{
    bf16_weights_kernel<<<kH * kH / 256, 256, 0, m->st>>>(m->P, m->W2b, m->W3b, m->W2T, m->W3T);
    MCK(cudaGetLastError());
    return DP_OK;
}

// A kernel's dynamic shared-memory limit, raised once per device (function
// attributes hold per device, so a process that drives several GPUs raises
// it on each).
constexpr int kMaxDevices = 64;

template <typename K>
cudaError_t raise_smem_limit(K kernel, int bytes, std::atomic<bool> (&done)[kMaxDevices])
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    if (done[dev].load(std::memory_order_acquire)) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done[dev].store(true, std::memory_order_release);
    return e;
}

// Batches from this size on run the persistent GEMMs.
constexpr int kManyRows = 16384;

// Most splits of the weight gradients (fewer serialise the K loop of each CTA,
// more write more partial tiles), blocks of the output layer, and blocks of the
// feature reductions below kManyRows rows (the persistent backward GEMMs sum
// per row tile instead).
constexpr int kSplitMax = 32, kOutBlocks = 1024, kRedBlocks = 256;

// The persistent kernel over rows (a multiple of 128, at least kManyRows) with
// K = 256; RED > 0 (backward): the per-tile sums into red.
template <int EPI, int RED = 0>
cudaError_t persistent(dp_mlp* m, const bf16* A, int lda, const bf16* B, int ldb, int rows, const float* bias,
                       float* zout, const float* zin, bf16* hout, const float* xin = nullptr, float* red = nullptr)
{
    static std::atomic<bool> attr[kMaxDevices];
    cudaError_t e = raise_smem_limit(mlp_persistent_kernel<EPI, RED>, kPersistSmem, attr);
    if (e != cudaSuccess) return e;
    const int tiles = rows / kTileM;
    const int per_half = std::max(1, std::min(tiles, m->sm_count / 2));
    dim3 grid(per_half, kH / kTileN);
    mlp_persistent_kernel<EPI, RED><<<grid, kPersistThreads, kPersistSmem, m->st>>>(
        A, lda, B, ldb, tiles, bias, zout, zin, hout, xin, red, m->err, m->wait_polls);
    return cudaGetLastError();
}

// A hidden layer (kEpiFwd) or its backward product (kEpiBwd), K = 256.
template <int EPI>
cudaError_t gemm(dp_mlp* m, const bf16* A, int lda, const bf16* B, int ldb, int rows, const float* bias, float* zout,
                 const float* zin, bf16* hout)
{
    if (rows >= kManyRows) return persistent<EPI>(m, A, lda, B, ldb, rows, bias, zout, zin, hout);
    static std::atomic<bool> attr[kMaxDevices];
    cudaError_t e = raise_smem_limit(mlp_gemm_kernel<EPI>, kGemmSmem, attr);
    if (e != cudaSuccess) return e;
    mlp_gemm_kernel<EPI><<<dim3(rows / kTileM, kH / kTileN), 128, kGemmSmem, m->st>>>(A, lda, B, ldb, bias, zout, zin, hout,
                                                                                  m->err, m->wait_polls);
    return cudaGetLastError();
}

// dW3 and dW2 over `rows` rows (a multiple of 256) as `splits` partial tiles each in m->part
cudaError_t weight_gradients(dp_mlp* m, int rows, int splits)
{
    static std::atomic<bool> attr[kMaxDevices];
    cudaError_t e = raise_smem_limit(mlp_wgrad_kernel, kWgSmem, attr);
    if (e != cudaSuccess) return e;
    const WgPair p{{m->dz3, m->dz2}, {m->h2, m->h1}};
    mlp_wgrad_kernel<<<dim3(kH / kTileM, kH / kTileN, 2 * splits), kWgThreads, kWgSmem, m->st>>>(p, splits, rows / splits, m->part,
                                                                                              m->err, m->wait_polls);
    return cudaGetLastError();
}

// Hidden layers of a training step's forward pass of `rows` rows (a multiple of
// 512), held in m->x or, with a grid, its next batch, through h3, keeping
// z1..z3 for the backward pass.
int forward_hidden(dp_mlp* m, int rows, const GridView* gv)
{
    const int b1 = rows / kL1Rows;
    float4* x = reinterpret_cast<float4*>(m->x);
    if (!gv) {
        first_layer_kernel<false, float><<<b1, 256, 0, m->st>>>(Geo<double>(), TrainGrid(), m->P, x, m->t, m->z1, m->h1);
    } else {
        const bool f32 = gv->fp32 && !gv->V64;
        const TrainGrid tg{gv->V64 ? (const void*)gv->V64 : gv->V, gv->code, gv->tab_hi64, gv->tab_lo64, m->coord, gv->n,
                           1.0 / gv->M, m->ts};
        if (f32) first_layer_kernel<true, float><<<b1, 256, 0, m->st>>>(gv->g64, tg, m->P, x, m->t, m->z1, m->h1);
        else first_layer_kernel<true, double><<<b1, 256, 0, m->st>>>(gv->g64, tg, m->P, x, m->t, m->z1, m->h1);
    }
    MCK(cudaGetLastError());
    MCK(gemm<kEpiFwd>(m, m->h1, kH, m->W2b, kH, rows, m->P + kOffB2, m->z2, nullptr, m->h2));
    MCK(gemm<kEpiFwd>(m, m->h2, kH, m->W3b, kH, rows, m->P + kOffB3, m->z3, nullptr, m->h3));
    return DP_OK;
}

// Inference of `count` rows: of m->x into m->y, or (GRID) of a grid's stored
// nodes into its value and policy.
template <bool GRID>
int infer(dp_mlp* m, int count, const Geo<double>& g, const InferGrid& ig)
{
    static std::atomic<bool> attr[kMaxDevices];
    MCK(raise_smem_limit(mlp_infer_kernel<GRID>, kInferSmem, attr));
    infer_weights_kernel<<<2 * kInferSteps * kInferStep / 16 / 256, 256, 0, m->st>>>(m->W2b, m->W3b, (uint4*)m->Wsteps);
    MCK(cudaGetLastError());
    const int tiles = (int)(((long long)count + kTileM - 1) / kTileM);
    mlp_infer_kernel<GRID><<<std::min(tiles, 2 * m->sm_count), kInferThreads, kInferSmem, m->st>>>(
        g, ig, m->x, m->P, m->Wsteps, count, m->y, m->err, m->wait_polls);
    MCK(cudaGetLastError());
    return DP_OK;
}

// Adam (beta1 0.9, beta2 0.999, eps 1e-8) with the step count in m->ts
AdamArgs adam_args(dp_mlp* m, double lr, int advance)
{
    return AdamArgs{m->P, m->Am, m->Av, (float)lr, 0.9f, 0.999f, 1e-8f, m->ts, m->W2b, m->W3b, m->W2T, m->W3T, m->arrive,
                    advance};
}

// Gradients of the mean squared error over a batch of `count` rows (count a
// multiple of 512; m->x / m->t hold the batch, or gv gives it), the loss sum
// added to m->loss.  The output layer and its backward pass run in one kernel.
// The gradients go to m->G, or with adam straight into a step of it.
int forward_backward(dp_mlp* m, int count, float inv_n, const GridView* gv = nullptr, const AdamArgs* adam = nullptr)
{
    const int rows = count;
    int rc;
    if ((rc = forward_hidden(m, rows, gv))) return rc;
    // every gradient sum goes through per-block partial sums and a reduction
    // in a fixed order, so that a training run is reproducible bit for bit
    const int ob = (int)std::min<long long>(std::min<long long>((count + 7) / 8, 2LL * m->sm_count), kOutBlocks);
    out_train_kernel<<<ob, 256, 0, m->st>>>(m->h3, m->P, m->t, m->z3, count, inv_n, m->dz3, m->out_part);
    MCK(cudaGetLastError());
    int nb;   // partial sums of the bias and first-layer gradients
    if (rows >= kManyRows) {
        // persistent backward GEMMs with the bias and first-layer gradients
        // summed per row tile in their epilogues (dz1 is never stored):
        // layer 3, dz2 = (dz3 W3) * GELU'(z2) with db2; layer 2,
        // dz1 = (dz2 W2) * GELU'(z1) summed into dW1 = dz1^T x and db1
        nb = rows / kTileM;
        MCK((persistent<kEpiBwd, 1>(m, m->dz3, kH, m->W3T, kH, rows, nullptr, nullptr, m->z2, m->dz2, nullptr,
                                    m->red1)));
        MCK((persistent<kEpiBwd, 5>(m, m->dz2, kH, m->W2T, kH, rows, nullptr, nullptr, m->z1, nullptr, m->x,
                                    m->red5)));
    } else {
        // the same with dz1 stored, db2 = sum dz2 and dW1, db1 in passes of
        // their own of at most kRedBlocks blocks
        const int chunk = std::max(64, (rows + kRedBlocks - 1) / kRedBlocks);
        nb = (rows + chunk - 1) / chunk;
        MCK(gemm<kEpiBwd>(m, m->dz3, kH, m->W3T, kH, rows, nullptr, nullptr, m->z2, m->dz2));
        MCK(gemm<kEpiBwd>(m, m->dz2, kH, m->W2T, kH, rows, nullptr, nullptr, m->z1, m->dz1));
        feat_reduce_kernel<0><<<nb, 256, 0, m->st>>>(m->dz2, nullptr, rows, chunk, m->red1);
        MCK(cudaGetLastError());
        feat_reduce_kernel<4><<<nb, 256, 0, m->st>>>(m->dz1, m->x, rows, chunk, m->red5);
        MCK(cudaGetLastError());
    }
    // dW3 = dz3^T h2 and dW2 = dz2^T h1; splits: a divisor of rows / 256
    int ks = std::min(rows / kKC, kSplitMax);
    while ((rows / kKC) % ks) --ks;
    MCK(weight_gradients(m, rows, ks));
    RedSegs r{};
    int blocks = 0, q = 0;
    auto seg = [&](const float* part, int n_part, int stride, int len, int at) {
        blocks += len > kRedLong ? (len + 255) / 256 : (len + 7) / 8;
        r.s[q++] = RedSeg{part, n_part, stride, len, at, blocks};
    };
    seg(m->part, ks, kH * kH, kH * kH, kOffW3);
    seg(m->part + (size_t)ks * kH * kH, ks, kH * kH, kH * kH, kOffW2);
    seg(m->out_part, ob, kOutPart, 4 * kH + 3, kOffB3);          // db3, dW4, db4
    seg(m->red1, nb, kH, kH, kOffB2);
    seg(m->red5, nb, 5 * kH, 5 * kH, kOffW1);                    // dW1, db1
    seg(m->out_part + 4 * kH + 3, ob, kOutPart, 1, -1);          // the loss
    if (adam) reduce_kernel<true><<<blocks, 256, 0, m->st>>>(r, *adam, nullptr, m->loss);
    else reduce_kernel<false><<<blocks, 256, 0, m->st>>>(r, AdamArgs(), m->G, m->loss);
    MCK(cudaGetLastError());
    return DP_OK;
}

// One Adam step with the gradient in m->G (the next step count), then the BF16
// copies of the weights.
int adam_step(dp_mlp* m, double lr)
{
    ++m->step;
    set_step_kernel<<<1, 1, 0, m->st>>>(m->ts, (int)m->step);
    MCK(cudaGetLastError());
    adam_kernel<<<(kParams + 255) / 256, 256, 0, m->st>>>(adam_args(m, lr, 0), m->G, kParams);
    MCK(cudaGetLastError());
    return DP_OK;
}

int check_err(dp_mlp* m)
{
    MCK(cudaMemcpyAsync(m->h_err, m->err, sizeof(int), cudaMemcpyDeviceToHost, m->st));
    MCK(cudaStreamSynchronize(m->st));
    if (*m->h_err) {
        // the kernels that gave up drained their MMAs and freed their TMEM:
        // clear the flag so that the next call starts clean
        *m->h_err = 0;
        MCK(cudaMemsetAsync(m->err, 0, sizeof(int), m->st));
        MCK(cudaStreamSynchronize(m->st));
        return record_error(DP_ETIMEOUT, "a tensor-core GEMM gave up waiting for its MMAs");
    }
    return DP_OK;
}

}  // namespace

namespace {

// One training step on a batch of the grid's nodes, everything on m->st:
// the batch of samples start .. start + B - 1 of the epoch's permutation (from
// m->ts), forward, backward, Adam with step count m->ts->t, then the next
// step's start and count.  Replayable: no argument changes between steps.
int train_step(dp_mlp* m, const GridView& gv, int B, double lr)
{
    const AdamArgs adam = adam_args(m, lr, B);   // with the next step's start and count
    return forward_backward(m, B, 1.0f / (3.0f * B), &gv, &adam);
}

// The epochs of dp_mlp_train_grid.  The first step runs as launched (it also
// sets the kernels' attributes); the next one is captured as a CUDA graph
// and every later step replays it, which removes the host's launches
// per step.
int train_grid_steps(dp_mlp* m, const GridView& gv, const dp_mlp_train_opts* o, dp_mlp_train_stats* stats)
{
    const long long n = gv.n;
    const int B = o->batch;
    const long long steps_per_epoch = n / B;
    const Box4 nlo{m->lo[0], m->lo[1], m->lo[2], m->lo[3]};
    const Box4 nhi{m->hi[0], m->hi[1], m->hi[2], m->hi[3]};
    double last_loss = 0.0, first_loss = -1.0;
    unsigned long long rng = o->seed ? o->seed : 14675ull;
    auto next = [&]() {   // splitmix64: seeds of the per-epoch permutation
        rng += 0x9E3779B97F4A7C15ull;
        unsigned long long z = rng;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return z ^ (z >> 31);
    };
    auto gcd = [](unsigned long long a, unsigned long long b) { while (b) { unsigned long long t = a % b; a = b; b = t; } return a; };
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    auto done = [&](int rc) {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
        if (e0) cudaEventDestroy(e0);
        if (e1) cudaEventDestroy(e1);
        return rc;
    };
    int rc;
    cudaError_t e;
    if ((e = cudaEventCreate(&e0)) != cudaSuccess || (e = cudaEventCreate(&e1)) != cudaSuccess ||
        (e = cudaEventRecord(e0, m->st)) != cudaSuccess)
        return done(fail_cuda("training events", e));
    coord_table_kernel<<<4, kCoordStride, 0, m->st>>>(gv.g64, nlo, nhi, m->coord);
    if ((e = cudaGetLastError()) != cudaSuccess) return done(fail_cuda("coordinate table", e));
    for (int ep = 0; ep < o->epochs; ++ep) {
        unsigned long long mult = (next() % (unsigned long long)n) | 1ull;
        while (gcd(mult, (unsigned long long)n) != 1) mult = (mult + 2) % (unsigned long long)n;
        const unsigned long long off = next() % (unsigned long long)n;
        // the previous epoch's copy from h_ts has completed (check_err synchronised)
        // the epoch's step size: geometric from lr to lr_final over the epochs
        double lr_ep = o->lr;
        if (o->lr_final > 0 && o->epochs > 1) lr_ep = o->lr * pow(o->lr_final / o->lr, (double)ep / (o->epochs - 1));
        *m->h_ts = TrainState{(long long)mult, (long long)off, 0, (int)(m->step + 1), (float)lr_ep};
        if ((e = cudaMemcpyAsync(m->ts, m->h_ts, sizeof(TrainState), cudaMemcpyHostToDevice, m->st)) != cudaSuccess ||
            (e = cudaMemsetAsync(m->loss, 0, sizeof(float), m->st)) != cudaSuccess)
            return done(fail_cuda("training state", e));
        for (long long s = 0; s < steps_per_epoch; ++s) {
            if (exec) {
                if ((e = cudaGraphLaunch(exec, m->st)) != cudaSuccess) return done(fail_cuda("graph launch", e));
            } else if (ep == 0 && s == 0) {
                if ((rc = train_step(m, gv, B, o->lr))) return done(rc);
            } else {
                if ((e = cudaStreamBeginCapture(m->st, cudaStreamCaptureModeThreadLocal)) != cudaSuccess)
                    return done(fail_cuda("stream capture", e));
                const int rs = train_step(m, gv, B, o->lr);
                e = cudaStreamEndCapture(m->st, &graph);
                if (rs) return done(rs);
                if (e != cudaSuccess) return done(fail_cuda("stream capture", e));
                if ((e = cudaGraphInstantiate(&exec, graph, 0)) != cudaSuccess ||
                    (e = cudaGraphLaunch(exec, m->st)) != cudaSuccess)
                    return done(fail_cuda("training graph", e));
            }
        }
        m->step += steps_per_epoch;
        if ((e = cudaMemcpyAsync(m->h_loss, m->loss, sizeof(float), cudaMemcpyDeviceToHost, m->st)) != cudaSuccess)
            return done(fail_cuda("loss read-back", e));
        if ((rc = check_err(m))) return done(rc);
        last_loss = *m->h_loss / (3.0 * B * (double)steps_per_epoch);
        if (first_loss < 0) first_loss = last_loss;
    }
    if ((e = cudaEventRecord(e1, m->st)) != cudaSuccess || (e = cudaEventSynchronize(e1)) != cudaSuccess)
        return done(fail_cuda("training events", e));
    float ms = 0;
    cudaEventElapsedTime(&ms, e0, e1);
    if (stats) {
        stats->epochs = o->epochs;
        stats->steps = steps_per_epoch * o->epochs;
        stats->samples = (int64_t)B * steps_per_epoch * o->epochs;
        stats->first_epoch_loss = first_loss;
        stats->last_epoch_loss = last_loss;
        stats->ms = ms;
        stats->flops = 3.0 * 2.0 * 132864.0 * (double)stats->samples;   // forward + 2x backward
    }
    return done(DP_OK);
}

}  // namespace

extern "C" {

int64_t dp_mlp_param_count(void) { return kParams; }

int dp_mlp_create(const double* lo, const double* hi, int32_t batch_capacity, void* stream, dp_mlp** out)
{
    if (!out || !lo || !hi) return record_error(DP_EINVAL, "NULL argument");
    *out = nullptr;
    if (batch_capacity < 512 || batch_capacity % 512 != 0 || batch_capacity > (1 << 20))
        return record_error(DP_EINVAL, "batch_capacity must be a multiple of 512 in [512, 2^20]");
    for (int d = 0; d < 4; ++d)
        if (!(lo[d] < hi[d])) return record_error(DP_EINVAL, "input box needs lo < hi");
    dp_mlp* m = new (std::nothrow) dp_mlp();
    if (!m) return record_error(DP_ENOMEM, "host allocation failed");
    m->st = (cudaStream_t)stream;
    m->cap = batch_capacity;
    for (int d = 0; d < 4; ++d) { m->lo[d] = lo[d]; m->hi[d] = hi[d]; }
    cudaGetDevice(&m->device);
    cudaDeviceGetAttribute(&m->sm_count, cudaDevAttrMultiProcessorCount, m->device);
    const size_t C = (size_t)m->cap, CH = C * kH;
    cudaError_t e = cudaSuccess;
    auto A = [&](auto** p, size_t n) { if (e == cudaSuccess) e = malloc_n(p, n); };
    A(&m->P, kParams); A(&m->G, kParams); A(&m->Am, kParams); A(&m->Av, kParams);
    A(&m->W2b, kH * kH); A(&m->W3b, kH * kH); A(&m->W2T, kH * kH); A(&m->W3T, kH * kH);
    A(&m->x, C * 4); A(&m->t, C * 3); A(&m->y, C * 3);
    A(&m->z1, CH); A(&m->z2, CH); A(&m->z3, CH);
    A(&m->h1, CH); A(&m->h2, CH); A(&m->h3, CH); A(&m->dz1, CH); A(&m->dz2, CH); A(&m->dz3, CH);
    A(&m->states, C * 4); A(&m->Wsteps, 2 * kInferSteps * kInferStep); A(&m->coord, 4 * kCoordStride); A(&m->loss, 1); A(&m->err, 1);
    const size_t R = std::max<size_t>(C / kTileM, kRedBlocks) * kH;
    A(&m->part, 2 * (size_t)kSplitMax * kH * kH); A(&m->out_part, (size_t)kOutBlocks * kOutPart); A(&m->red1, R); A(&m->red5, 5 * R);
    A(&m->arrive, 1);
    A(&m->ts, 1);
    if (e == cudaSuccess) e = cudaMallocHost(&m->h_loss, sizeof(float));
    if (e == cudaSuccess) e = cudaMallocHost(&m->h_err, sizeof(int));
    if (e == cudaSuccess) e = cudaMallocHost(&m->h_ts, sizeof(TrainState));
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&m->cst, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&m->ev_in, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&m->ev_out, cudaEventDisableTiming);
    if (e != cudaSuccess) {
        cudaGetLastError();
        free_mlp(m);
        return record_error(DP_ENOMEM, "device allocation of the network failed");
    }
    cudaMemsetAsync(m->Am, 0, sizeof(float) * kParams, m->st);
    cudaMemsetAsync(m->Av, 0, sizeof(float) * kParams, m->st);
    cudaMemsetAsync(m->err, 0, sizeof(int), m->st);
    cudaMemsetAsync(m->arrive, 0, sizeof(unsigned), m->st);
    *out = m;
    return DP_OK;
}

int dp_mlp_destroy(dp_mlp* m)
{
    free_mlp(m);
    return DP_OK;
}

int dp_mlp_set_params(dp_mlp* m, const float* params, int64_t count)
{
    if (!m || !params) return record_error(DP_EINVAL, "NULL argument");
    if (count != kParams) return record_error(DP_EINVAL, "parameter count mismatch");
    MCK(cudaMemcpyAsync(m->P, params, sizeof(float) * kParams, cudaMemcpyHostToDevice, m->st));
    MCK(cudaMemsetAsync(m->Am, 0, sizeof(float) * kParams, m->st));
    MCK(cudaMemsetAsync(m->Av, 0, sizeof(float) * kParams, m->st));
    m->step = 0;
    int rc = refresh_bf16(m);
    if (rc) return rc;
    MCK(cudaStreamSynchronize(m->st));
    return DP_OK;
}

int dp_mlp_get_params(const dp_mlp* m, float* params, int64_t count)
{
    if (!m || !params) return record_error(DP_EINVAL, "NULL argument");
    if (count != kParams) return record_error(DP_EINVAL, "parameter count mismatch");
    MCK(cudaMemcpyAsync(params, m->P, sizeof(float) * kParams, cudaMemcpyDeviceToHost, m->st));
    MCK(cudaStreamSynchronize(m->st));
    return DP_OK;
}

int dp_mlp_forward(dp_mlp* m, const double* states, int32_t n, float* out)
{
    if (!m || (n > 0 && (!states || !out))) return record_error(DP_EINVAL, "NULL argument");
    if (n < 0) return record_error(DP_EINVAL, "n < 0");
    const Box4 lo{m->lo[0], m->lo[1], m->lo[2], m->lo[3]};
    const Box4 hi{m->hi[0], m->hi[1], m->hi[2], m->hi[3]};
    for (int s0 = 0; s0 < n; s0 += m->cap) {
        const int cnt = std::min(m->cap, n - s0);
        MCK(cudaMemcpyAsync(m->states, states + 4 * (size_t)s0, sizeof(double) * 4 * cnt, cudaMemcpyHostToDevice,
                            m->st));
        states_in_kernel<<<(cnt + 255) / 256, 256, 0, m->st>>>(m->states, cnt, lo, hi, m->x);
        MCK(cudaGetLastError());
        int rc = infer<false>(m, cnt, Geo<double>(), InferGrid());
        if (rc) return rc;
        MCK(cudaMemcpyAsync(out + 3 * (size_t)s0, m->y, sizeof(float) * 3 * cnt, cudaMemcpyDeviceToHost, m->st));
    }
    return check_err(m);
}

int dp_mlp_gradients(dp_mlp* m, const double* states, const float* targets, int32_t n, float* grads, float* loss)
{
    if (!m || !states || !targets || !grads) return record_error(DP_EINVAL, "NULL argument");
    if (n < 512 || n % 512 != 0 || n > m->cap) return record_error(DP_EINVAL, "n must be a multiple of 512 <= capacity");
    const Box4 lo{m->lo[0], m->lo[1], m->lo[2], m->lo[3]};
    const Box4 hi{m->hi[0], m->hi[1], m->hi[2], m->hi[3]};
    MCK(cudaMemcpyAsync(m->states, states, sizeof(double) * 4 * n, cudaMemcpyHostToDevice, m->st));
    MCK(cudaMemcpyAsync(m->t, targets, sizeof(float) * 3 * n, cudaMemcpyHostToDevice, m->st));
    states_in_kernel<<<(n + 255) / 256, 256, 0, m->st>>>(m->states, n, lo, hi, m->x);
    MCK(cudaMemsetAsync(m->loss, 0, sizeof(float), m->st));
    int rc = forward_backward(m, n, 1.0f / (3.0f * n));
    if (rc) return rc;
    MCK(cudaMemcpyAsync(grads, m->G, sizeof(float) * kParams, cudaMemcpyDeviceToHost, m->st));
    MCK(cudaMemcpyAsync(m->h_loss, m->loss, sizeof(float), cudaMemcpyDeviceToHost, m->st));
    if ((rc = check_err(m))) return rc;
    if (loss) *loss = *m->h_loss / (3.0f * n);
    return DP_OK;
}

int dp_mlp_apply_gradients(dp_mlp* m, const float* grads, int64_t count, double lr)
{
    if (!m || !grads) return record_error(DP_EINVAL, "NULL argument");
    if (count != kParams) return record_error(DP_EINVAL, "parameter count mismatch");
    if (!(lr > 0)) return record_error(DP_EINVAL, "lr must be positive");
    MCK(cudaMemcpyAsync(m->G, grads, sizeof(float) * kParams, cudaMemcpyHostToDevice, m->st));
    int rc = adam_step(m, lr);
    if (rc) return rc;
    MCK(cudaStreamSynchronize(m->st));
    return DP_OK;
}

int dp_mlp_set_wait_limit(dp_mlp* m, int32_t polls)
{
    if (!m || polls < -1) return record_error(DP_EINVAL, "bad argument");
    m->wait_polls = polls >= 0 ? polls : kWaitPolls;
    return DP_OK;
}

int dp_mlp_train_grid(dp_mlp* m, dp_grid* grid, const dp_mlp_train_opts* o, dp_mlp_train_stats* stats)
{
    if (!m || !grid || !o) return record_error(DP_EINVAL, "NULL argument");
    if (o->batch < 512 || o->batch % 512 != 0 || o->batch > m->cap || o->epochs < 0 || !(o->lr > 0) ||
        !(o->lr_final >= 0))
        return record_error(DP_EINVAL, "bad training options");
    GridView gv;
    int rc = grid_view(grid, &gv);
    if (rc) return rc;
    if (gv.n < o->batch) return record_error(DP_EINVAL, "grid smaller than one batch");
    // the steps run on the network's private stream, ordered after the
    // caller's stream and before its later work
    cudaStream_t user = m->st;
    MCK(cudaEventRecord(m->ev_in, user));
    MCK(cudaStreamWaitEvent(m->cst, m->ev_in, 0));
    m->st = m->cst;
    rc = train_grid_steps(m, gv, o, stats);
    m->st = user;
    cudaError_t e = cudaEventRecord(m->ev_out, m->cst);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(user, m->ev_out, 0);
    if (rc) return rc;
    MCK(e);
    return DP_OK;
}

int dp_warm_start(dp_mlp* m, dp_grid* grid, double* ms_out)
{
    if (!m || !grid) return record_error(DP_EINVAL, "NULL argument");
    GridView gv;
    int rc = grid_view(grid, &gv);
    if (rc) return rc;
    cudaEvent_t e0, e1;
    MCK(cudaEventCreate(&e0));
    MCK(cudaEventCreate(&e1));
    MCK(cudaEventRecord(e0, m->st));
    // node coordinates of this grid, normalised to the network's own box
    Geo<double> g = gv.g64;
    const Box4 nlo{m->lo[0], m->lo[1], m->lo[2], m->lo[3]};
    const Box4 nhi{m->hi[0], m->hi[1], m->hi[2], m->hi[3]};
    coord_table_kernel<<<4, kCoordStride, 0, m->st>>>(g, nlo, nhi, m->coord);
    MCK(cudaGetLastError());
    // the value goes to the storage-precision buffer (an FP32 grid holding
    // FP64 values after a polish returns to its FP32 values)
    const InferGrid ig{m->coord, gv.M, const_cast<void*>(gv.V), gv.code, gv.fp32};
    if ((rc = infer<true>(m, (int)gv.n, g, ig))) return rc;
    MCK(cudaEventRecord(e1, m->st));
    if ((rc = check_err(m))) return rc;
    float ms = 0;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (ms_out) *ms_out = ms;
    grid_after_warm_start(grid);
    return DP_OK;
}

}  // extern "C"
