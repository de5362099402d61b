// train.cu -- training of the learned a0 proposal on the GPU: forward and
// backward passes of the MLP + rational-quadratic spline negative
// log-likelihood, with the two hidden-layer contractions of each pass on the
// 5th-generation tensor cores (BF16 operands, FP32 accumulation in tensor
// memory), and an Adam update.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <vector>

#include "su2_device.cuh"
#include "su2_internal.h"
#include "tc05.cuh"

namespace su2 {

constexpr uint32_t kMbarPolls = 1u << 26;

__device__ __forceinline__ void mbar_init_fence()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Self-test: D (128 x 32, FP32) = A (128 x K, BF16) * B (32 x K, BF16)^T on the
// tensor cores, K = 16 or 32, for comparison with a host reference.
__global__ void __launch_bounds__(128) mma_selftest_kernel(const uint16_t *__restrict__ A,
                                                           const uint16_t *__restrict__ B, int K,
                                                           float *__restrict__ D, unsigned int *__restrict__ err)
{
    __shared__ __align__(128) unsigned char sA[128 * 32 * 2];
    __shared__ __align__(128) unsigned char sB[32 * 32 * 2];
    __shared__ __align__(8) uint64_t mbar;
    __shared__ uint32_t tmem_base;
    const int t = threadIdx.x, warp = t >> 5;
    for (int k = 0; k < K; ++k) *(uint16_t *)(sA + tc::tile_offset(t, k, K)) = A[t * K + k];
    if (t < 32)
        for (int k = 0; k < K; ++k) *(uint16_t *)(sB + tc::tile_offset(t, k, K)) = B[t * K + k];
    tc::fence_smem_to_async();
    if (warp == 0) tc::tmem_alloc(&tmem_base, 32);
    if (t == 0) {
        tc::mbar_init(&mbar, 1);
        mbar_init_fence();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t taddr = tmem_base;
    if (t == 0) {
        const uint32_t idesc = tc::idesc_bf16_f32(128, 32);
        const uint32_t sbo = (uint32_t)(K / 8) * 128u;
        for (int j = 0; j < K / 16; ++j) {
            const uint64_t ad = tc::smem_desc(tc::smem_addr(sA) + 256u * j, 128u, sbo);
            const uint64_t bd = tc::smem_desc(tc::smem_addr(sB) + 256u * j, 128u, sbo);
            tc::mma_bf16(taddr, ad, bd, idesc, j > 0 ? 1u : 0u);
        }
        tc::mma_commit(&mbar);
    }
    bool ok = tc::mbar_wait(&mbar, 0, kMbarPolls);
    if (!ok) ok = tc::mbar_wait(&mbar, 0, kMbarPolls);  // second bounded wait before giving up
    tc::fence_after_sync();
    if (ok) {
        float v[32];
        tc::tmem_load32(taddr + ((uint32_t)(warp * 32) << 16), v);
#pragma unroll
        for (int n = 0; n < 32; ++n) D[t * 32 + n] = v[n];
    } else if ((t & 31) == 0) {
        atomicAdd(err, 1u);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(taddr, 32);
}

}  // namespace su2

using namespace su2;

extern "C" su2_status su2_selftest_mma(const uint16_t *A, const uint16_t *B, int K, float *D)
{
    if (!A || !B || !D || (K != 16 && K != 32)) return SU2_E_INVAL;
    int dev = 0;
    SU2_CUDA(cudaGetDevice(&dev));
    const size_t bytesA = 128 * (size_t)K * 2, bytesB = 32 * (size_t)K * 2, bytesD = 128 * 32 * 4;
    char *buf = (char *)device_alloc(bytesA + bytesB + bytesD + 512, dev, nullptr);
    if (!buf) return SU2_E_NOMEM;
    uint16_t *dA = (uint16_t *)buf;
    uint16_t *dB = (uint16_t *)(buf + ((bytesA + 255) & ~(size_t)255));
    float *dD = (float *)((char *)dB + ((bytesB + 255) & ~(size_t)255));
    unsigned int *dErr = (unsigned int *)((char *)dD + bytesD);
    su2_status st = SU2_OK;
    cudaError_t e = cudaMemcpy(dA, A, bytesA, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(dB, B, bytesB, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(dErr, 0, sizeof(unsigned int));
    if (e == cudaSuccess) {
        mma_selftest_kernel<<<1, 128>>>(dA, dB, K, dD, dErr);
        e = cudaGetLastError();
    }
    unsigned int err = 0;
    if (e == cudaSuccess) e = cudaMemcpy(D, dD, bytesD, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(&err, dErr, sizeof err, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) st = cuda_fail(e, "su2_selftest_mma");
    else if (err) {
        set_last_error("tensor-core self-test: completion wait gave up");
        st = SU2_E_DEVICE_TIMEOUT;
    }
    device_free(buf, bytesA + bytesB + bytesD + 512, dev, nullptr);
    cudaDeviceSynchronize();
    return st;
}

// ============================================================== training
#include "learned.cuh"
#include "observables.cuh"

namespace su2 {
namespace train {

// A step works on 128 samples per CTA (the MMA M dimension) with four threads
// per sample: thread (row, part) holds columns 8 part .. 8 part + 7 of the
// sample's 32-wide rows, the split in which tensor memory hands the
// accumulator to four warps per 32 rows, and in which the network's outputs
// fall apart (bin widths, bin heights, knot derivatives 0..7, derivative 8),
// so the softmax and softplus work of a sample runs on four warps at once.
// The gradient sums over the 128 rows (rows in order, binary32) take all 16
// warps, four outputs per thread: one 16-byte broadcast and one conflict-free
// load per four multiply-adds.  Batches of 4096 fill 32 SMs with one CTA each,
// so a step is latency, not throughput.  One thread per sample
// took 39.6 us under ncu, this 12.9; a step with its Adam update 33 -> 12 us
// in a fit.
constexpr int kRows = 128;                   // samples per CTA
constexpr int kParts = 4;                    // threads per sample
constexpr int kTrainThreads = kRows * kParts;
constexpr int kPitch = 36;                   // row pitch of the binary32 stashes: 16-byte rows, conflict-free columns
constexpr int kGradSlots = learned::kTrainable + 1;  // 1945 gradients + loss sum

struct StepParams {
    const float *w;            // 1947 master weights (fp32)
    const uint4 *images;       // their BF16 operand tiles (put_images)
    int split;                 // CTAs per 128 samples: 1, 2 or 4
    const float2 *pairs;       // (beta k, a0)
    long long n_pairs;
    int explicit_rows;         // 1: row r of CTA b is pair b*128 + r; 0: random pairs
    uint32_t step, k0, k1;     // Philox key and counter for random pairs
    float *partials;           // [gridDim.x / split][kGradSlots]
    unsigned int *err;
};

__device__ __forceinline__ uint32_t to_bf16(float f)
{
    const uint32_t u = __float_as_uint(f);
    return (u + 0x7FFFu + ((u >> 16) & 1u)) >> 16;
}

// The B operands as the tensor cores take them (BF16, core-matrix layout): W2
// (n = output j, k = input i), W3 (n = output o, padded to 32), W3^T (n = j,
// k = o padded), W2^T (n = i, k = j), 2 KB each.  Kept beside the master
// weights (the Adam kernel writes both), so a CTA fetches them as one 16-byte
// load per thread instead of converting and scattering 1824 weights.
constexpr uint32_t kTileBytes = 32 * 32 * 2;
constexpr uint32_t kImageBytes = 4 * kTileBytes;
static_assert(kImageBytes == 16 * kTrainThreads, "one 16-byte load per thread");

__device__ __forceinline__ void put_images(unsigned char *images, int i, float w)
{
    const bool w2 = i >= learned::kOffW2 && i < learned::kOffB2;
    if (!w2 && !(i >= learned::kOffW3 && i < learned::kOffB3)) return;
    const int q = i - (w2 ? learned::kOffW2 : learned::kOffW3);
    const int r = q >> 5, c = q & 31;
    const uint16_t h = (uint16_t)to_bf16(w);
    *(uint16_t *)(images + (w2 ? 0 : kTileBytes) + tc::tile_offset(r, c, 32)) = h;
    *(uint16_t *)(images + (w2 ? 3 * kTileBytes : 2 * kTileBytes) + tc::tile_offset(c, r, 32)) = h;
}

__global__ void put_images_kernel(const float *__restrict__ w, unsigned char *__restrict__ images)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < learned::kTrainable) put_images(images, i, w[i]);
}

struct Smem {
    unsigned char A[kRows * 32 * 2];     // activation tile (A operand)
    unsigned char W2[kTileBytes], W3[kTileBytes], W3T[kTileBytes], W2T[kTileBytes];  // B operands
    float h1[kRows][kPitch], h2[kRows][kPitch], go[kRows][kPitch], dz2[kRows][kPitch], dz1[kRows][kPitch];
    float w1[32], b1[32], b2[32], b3[32];
    float knot[2][learned::kBins + 1][kRows];  // x_0 .. x_8, y_0 .. y_8 of each sample
    float der[learned::kBins + 1][kRows];
    float g_knot[2][2][kRows];           // gradient at knots k, k + 1 of x and y
    float g_der[2][kRows];               // gradient at derivatives k, k + 1
    float handed_o[3][kRows], handed_q[3][kRows];  // derivatives 5 .. 7: outputs to part 3, sigmoids back
    int bin[kRows];
    float s_in[kRows];
    float loss[kRows];
    uint64_t mbar;
    uint32_t tmem_base;
};

// Dependent launches (the step and the Adam kernel alternate): let the next
// grid of the stream start its independent prologue, and wait until the
// previous grid has finished and its writes are visible.  A grid is resident
// while earlier ones still write what it reads after the wait (operand tiles,
// weights, Adam state, partial sums), so that is not data that stays constant
// for the grid's lifetime: no such pointer is const __restrict__, which would
// allow loads by the non-coherent path.  The partial sums and the Adam state, which
// a thread of the grid before may have read on the same SM, are read from L2
// (__ldcg); the state's loads stand before the sums, as without __restrict__
// they no longer move there (709 against 668 us for 50 steps of 4096).
__device__ __forceinline__ void release_next_grid() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_previous_grid() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// One MMA pass: D (tmem) = A (smem tile, 128 x 32) * B^T (32 x 32), then this
// thread's eight columns of its row of D into v.  Every thread must call it
// (barriers inside).
__device__ bool mma_pass(Smem &sm, const unsigned char *B, uint32_t taddr, uint32_t &phase, float (&v)[8])
{
    tc::fence_smem_to_async();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (threadIdx.x == 0) {
        const uint32_t idesc = tc::idesc_bf16_f32(128, 32);
        for (int j = 0; j < 2; ++j) {
            const uint64_t ad = tc::smem_desc(tc::smem_addr(sm.A) + 256u * j, 128u, 512u);
            const uint64_t bd = tc::smem_desc(tc::smem_addr(B) + 256u * j, 128u, 512u);
            tc::mma_bf16(taddr, ad, bd, idesc, j > 0 ? 1u : 0u);
        }
        tc::mma_commit(&sm.mbar);
    }
    bool ok = tc::mbar_wait(&sm.mbar, phase, kMbarPolls);
    if (!ok) ok = tc::mbar_wait(&sm.mbar, phase, kMbarPolls);
    phase ^= 1u;
    tc::fence_after_sync();
    // a warp reads the 32 lanes of its place in its group of four
    const uint32_t warp = threadIdx.x >> 5;
    if (ok) {
        tc::tmem_load8(taddr + ((warp & 3u) * 32u << 16) + (warp >> 2) * 8u, v);
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = 0.0f;
    }
    tc::fence_before_sync();
    __syncthreads();  // every thread has read D and A before either is overwritten
    return ok;
}

// This thread's eight columns: binary32 into the stash, BF16 into the A tile
// (one row of one core matrix).
__device__ __forceinline__ void stash_row(float (&stash)[kRows][kPitch], int row, int part, const float (&v)[8])
{
    float4 *const to = (float4 *)&stash[row][8 * part];
    to[0] = make_float4(v[0], v[1], v[2], v[3]);
    to[1] = make_float4(v[4], v[5], v[6], v[7]);
}

__device__ __forceinline__ void put_row_bf16(Smem &sm, int row, int part, const float (&v)[8])
{
    uint4 q;
    q.x = to_bf16(v[0]) | (to_bf16(v[1]) << 16);
    q.y = to_bf16(v[2]) | (to_bf16(v[3]) << 16);
    q.z = to_bf16(v[4]) | (to_bf16(v[5]) << 16);
    q.w = to_bf16(v[6]) | (to_bf16(v[7]) << 16);
    *(uint4 *)(sm.A + tc::tile_offset(row, 8 * part, 32)) = q;
}

// -log q(a | o) = log 2 + log f'(f^{-1}(a)) for the spline whose knots and
// derivatives are in sm, and its gradient at the bin's knots and derivatives:
// implicit differentiation of f(z) = a at fixed a (binary32; the same formulas
// as the binary64 reference).
__device__ __forceinline__ void nll_at_knots(Smem &sm, int row, float a)
{
    constexpr int K = learned::kBins;
    int k = 0;
#pragma unroll
    for (int j = 1; j < K; ++j)
        if (sm.knot[1][j][row] <= a) k = j;
    const float xk = sm.knot[0][k][row], yk = sm.knot[1][k][row];
    const float W = sm.knot[0][k + 1][row] - xk, H = sm.knot[1][k + 1][row] - yk;
    const float D0 = sm.der[k][row], D1 = sm.der[k + 1][row];
    const float s = H / W, dy = a - yk, sig = D1 + D0 - 2.0f * s;
    const float al = H * (s - D0) + dy * sig, be = H * D0 - dy * sig, c = -s * dy;
    const float disc = fmaxf(be * be - 4.0f * al * c, 0.0f);
    const float den_q = -be - sqrtf(disc);
    float xi = den_q != 0.0f ? 2.0f * c / den_q : 0.0f;
    xi = fminf(fmaxf(xi, 0.0f), 1.0f);
    const float t = xi * (1.0f - xi);
    const float N = s * xi * xi + D0 * t, Dn = s + sig * t;
    const float M = D1 * xi * xi + 2.0f * s * t + D0 * (1.0f - xi) * (1.0f - xi);
    const float L = 2.0f * log_series(s) + log_series(M) - 2.0f * log_series(Dn);
    const float Np = 2.0f * s * xi + D0 * (1.0f - 2.0f * xi), Dnp = sig * (1.0f - 2.0f * xi);
    const float Mp = 2.0f * D1 * xi + 2.0f * s * (1.0f - 2.0f * xi) - 2.0f * D0 * (1.0f - xi);
    const float F_xi = H * (Np * Dn - N * Dnp) / (Dn * Dn);
    const float L_xi = Mp / M - 2.0f * Dnp / Dn;
    const float r = L_xi / F_xi;
    const float F_s = H * (xi * xi * Dn - N * (1.0f - 2.0f * t)) / (Dn * Dn);
    const float F_D0 = H * t * (Dn - N) / (Dn * Dn);
    const float F_D1 = -H * N * t / (Dn * Dn);
    const float dY = -r;
    const float dHd = -r * (N / Dn);
    const float ds = (2.0f / s + 2.0f * t / M - 2.0f * (1.0f - 2.0f * t) / Dn) - r * F_s;
    sm.g_der[0][row] = ((1.0f - xi) * (1.0f - xi) / M - 2.0f * t / Dn) - r * F_D0;
    sm.g_der[1][row] = (xi * xi / M - 2.0f * t / Dn) - r * F_D1;
    const float dH = dHd + ds / W, dW = -ds * H / (W * W);
    sm.g_knot[0][0][row] = 0.0f - dW;
    sm.g_knot[0][1][row] = dW;
    sm.g_knot[1][0][row] = dY - dH;
    sm.g_knot[1][1][row] = dH;
    sm.bin[row] = k;
    sm.loss[row] = 0.69314718f + L;
}

// The likelihood of the sample and its gradient with respect to this thread's
// network outputs o (part 0: log widths, 1: log heights, 2 and 3: the
// unconstrained derivatives), through the knot sums and the softmax or the
// softplus.  Every thread calls it (barriers inside).
__device__ __forceinline__ void nll_and_grad(Smem &sm, int row, int part, float a, const float (&o)[8], float (&g)[8])
{
    constexpr int K = learned::kBins;
    float q[8];  // parts 0, 1: softmax probabilities; 2, 3: the derivatives' sigmoids
    if (part == 2) {
#pragma unroll
        for (int i = 0; i < 3; ++i) sm.handed_o[i][row] = o[5 + i];
    }
    __syncthreads();
    if (part < 2) {
        float mx = o[0];
#pragma unroll
        for (int i = 1; i < K; ++i) mx = fmaxf(mx, o[i]);
        float sum = 0.0f;
#pragma unroll
        for (int i = 0; i < K; ++i) {
            q[i] = learned::exp_neg(o[i] - mx);
            sum += q[i];
        }
        float kn = -1.0f;
        sm.knot[part][0][row] = kn;
#pragma unroll
        for (int i = 0; i < K; ++i) {
            q[i] = q[i] / sum;
            kn = kn + 2.0f * (learned::kMinBin + (1.0f - K * learned::kMinBin) * q[i]);
            sm.knot[part][i + 1][row] = kn;
        }
    } else {
        // five derivatives in part 2, four in part 3 (three of them handed over)
        const int n = part == 2 ? 5 : 4;  // warp-uniform
        float od[5] = {o[0], o[1], o[2], o[3], o[4]};
        if (part == 3) {
#pragma unroll
            for (int i = 0; i < 3; ++i) od[i] = sm.handed_o[i][row];
            od[3] = o[0];
        }
        float sg[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            sg[i] = 0.0f;
            if (i < n) {
                const float e = learned::exp_neg(od[i] < 0.0f ? od[i] : -od[i]);
                const float one_e = 1.0f + e;
                sm.der[5 * (part - 2) + i][row] =
                    learned::kMinDer + ((od[i] > 0.0f ? od[i] : 0.0f) + log_series(one_e));
                sg[i] = od[i] >= 0.0f ? 1.0f / one_e : e / one_e;
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) q[i] = part == 2 && i < 5 ? sg[i] : 0.0f;
        if (part == 3) {
#pragma unroll
            for (int i = 0; i < 3; ++i) sm.handed_q[i][row] = sg[i];
            q[0] = sg[3];
        }
    }
    __syncthreads();
    if (part == 0) nll_at_knots(sm, row, a);
    __syncthreads();
    const int k = sm.bin[row];
    if (part < 2) {
        // sums of the knots' gradients above each bin: none, k + 1's, both
        const float g1 = 0.0f + sm.g_knot[part][1][row], g01 = g1 + sm.g_knot[part][0][row];
        float dot = 0.0f;
#pragma unroll
        for (int i = 0; i < K; ++i) {
            g[i] = (i > k ? 0.0f : (i == k ? g1 : g01)) * 2.0f * (1.0f - K * learned::kMinBin);
            dot += g[i] * q[i];
        }
#pragma unroll
        for (int i = 0; i < K; ++i) g[i] = q[i] * (g[i] - dot);
    } else {
        if (part == 2) {
#pragma unroll
            for (int i = 0; i < 3; ++i) q[5 + i] = sm.handed_q[i][row];
        }
        const float d0 = sm.g_der[0][row], d1 = sm.g_der[1][row];
        const int first = 8 * (part - 2);
#pragma unroll
        for (int i = 0; i < 8; ++i) g[i] = (first + i == k ? d0 : (first + i == k + 1 ? d1 : 0.0f)) * q[i];
    }
}

// Sum over the rows, in order, of f(r): four products at a time.
__device__ __forceinline__ float4 row_products(const float (&lhs)[kRows][kPitch], int j4, const float (&rhs)[kRows][kPitch],
                                               int col)
{
    float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 8
    for (int r = 0; r < kRows; ++r) {
        const float4 d = *(const float4 *)&lhs[r][j4];
        const float x = rhs[r][col];
        acc.x += d.x * x;
        acc.y += d.y * x;
        acc.z += d.z * x;
        acc.w += d.w * x;
    }
    return acc;
}

// Forward + backward of kRows samples; their sums of the 1945 gradients and of
// the loss go to partials[block].  `split` CTAs run the same samples, each
// adding its share of the gradients: where the batch leaves SMs idle, the
// sums (the longest stage, 7.8 of 28 thousand cycles in one CTA) shrink with
// the split while the repeated forward pass costs nothing.
__global__ void __launch_bounds__(kTrainThreads) train_step_kernel(const StepParams p)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int row = t & (kRows - 1), part = t >> 7;
    const float *w = p.w;

    // what does not depend on the weights: tensor memory, the barrier, the sample
    release_next_grid();
    if (warp == 0) tc::tmem_alloc(&sm.tmem_base, 32);
    if (t == 0) {
        tc::mbar_init(&sm.mbar, 1);
        mbar_init_fence();
    }
    const int block = (int)blockIdx.x / p.split;
    long long idx;
    if (p.explicit_rows) {
        idx = (long long)block * kRows + row;
    } else {
        const uint4 r = philox_key(make_uint4((uint32_t)(block * kRows + row), p.step, 5u << 3, 0u), p.k0, p.k1);
        idx = (long long)(((unsigned long long)r.x * (unsigned long long)p.n_pairs) >> 32);
    }
    const float2 pr = p.pairs[idx];
    wait_previous_grid();

    ((uint4 *)sm.W2)[t] = p.images[t];
    if (warp == 0) sm.w1[lane] = w[learned::kOffW1 + lane];
    if (warp == 1) sm.b1[lane] = w[learned::kOffB1 + lane];
    if (warp == 2) sm.b2[lane] = w[learned::kOffB2 + lane];
    if (warp == 3) sm.b3[lane] = lane < learned::kOut ? w[learned::kOffB3 + lane] : 0.0f;
    const float s = (pr.x - w[learned::kOffMean]) * w[learned::kOffScale];
    const float a = fminf(fmaxf(pr.y, -1.0f), 1.0f);
    if (part == 0) sm.s_in[row] = s;
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t taddr = sm.tmem_base;
    uint32_t phase = 0;
    bool ok = true;

    // layer 1 (fp32), layer 2 (tensor cores)
    const int c0 = 8 * part;
    float v[8], h1[8], h2[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) h1[j] = learned::relu(sm.w1[c0 + j] * s + sm.b1[c0 + j]);
    stash_row(sm.h1, row, part, h1);
    put_row_bf16(sm, row, part, h1);
    ok &= mma_pass(sm, sm.W2, taddr, phase, v);
#pragma unroll
    for (int j = 0; j < 8; ++j) h2[j] = learned::relu(v[j] + sm.b2[c0 + j]);
    stash_row(sm.h2, row, part, h2);
    put_row_bf16(sm, row, part, h2);
    // layer 3 (tensor cores)
    ok &= mma_pass(sm, sm.W3, taddr, phase, v);
    float go[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = v[j] + sm.b3[c0 + j];
    nll_and_grad(sm, row, part, a, v, go);
    stash_row(sm.go, row, part, go);
    put_row_bf16(sm, row, part, go);
    // dh2 = go W3 (tensor cores), through the ReLU
    ok &= mma_pass(sm, sm.W3T, taddr, phase, v);
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = h2[j] > 0.0f ? v[j] : 0.0f;
    stash_row(sm.dz2, row, part, v);
    put_row_bf16(sm, row, part, v);
    // dh1 = dz2 W2 (tensor cores), through the ReLU
    ok &= mma_pass(sm, sm.W2T, taddr, phase, v);
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = h1[j] > 0.0f ? v[j] : 0.0f;
    stash_row(sm.dz1, row, part, v);
    if (!ok && t == 0) atomicAdd(p.err, 1u);
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(taddr, 32);

    // gradient sums (fp32, rows in order), a warp per task: 0..7 four rows of
    // W2 each, 8..14 four rows of W3, 15 the vectors
    const int tasks = 16 / p.split;
    if (warp >= tasks) return;
    const int task = ((int)blockIdx.x - block * p.split) * tasks + warp;
    float *out = p.partials + (size_t)block * kGradSlots;
    if (task < 8) {
        const float4 g = row_products(sm.dz2, 4 * task, sm.h1, lane);
        float *const to = out + learned::kOffW2 + 128 * task + lane;
        to[0] = g.x;
        to[32] = g.y;
        to[64] = g.z;
        to[96] = g.w;
    } else if (task < 15) {
        const int o0 = 4 * (task - 8);
        const float4 g = row_products(sm.go, o0, sm.h2, lane);
        float *const to = out + learned::kOffW3 + 32 * o0 + lane;
        to[0] = g.x;
        if (o0 + 1 < learned::kOut) {
            to[32] = g.y;
            to[64] = g.z;
            to[96] = g.w;
        }
    } else {
        float w1 = 0.0f, b1 = 0.0f, b2 = 0.0f, b3 = 0.0f, loss = 0.0f;
#pragma unroll 8
        for (int r = 0; r < kRows; ++r) {
            const float d = sm.dz1[r][lane];
            w1 += d * sm.s_in[r];
            b1 += d;
            b2 += sm.dz2[r][lane];
            b3 += sm.go[r][lane];
            loss += sm.loss[r];
        }
        out[learned::kOffW1 + lane] = w1;
        out[learned::kOffB1 + lane] = b1;
        out[learned::kOffB2 + lane] = b2;
        if (lane < learned::kOut) out[learned::kOffB3 + lane] = b3;
        if (lane == 0) out[learned::kTrainable] = loss;
    }
}

// Sums the per-CTA partials (in CTA order) into the mean gradient and loss;
// with lr > 0 also applies one Adam step to the master weights.
__global__ void adam_kernel(float *w, float *m, float *v, const float *partials, int nblocks, float inv_batch,
                            float lr, float b1, float b2, float eps, float bias1, float bias2, float *grad_out,
                            float *loss_out, unsigned char *images)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    release_next_grid();
    wait_previous_grid();
    if (i >= kGradSlots) return;
    // the state's loads beside those of the sums, not behind the stores below
    float m0 = 0.0f, v0 = 0.0f, w0 = 0.0f;
    if (lr > 0.0f && i < learned::kTrainable) {
        m0 = __ldcg(m + i);
        v0 = __ldcg(v + i);
        w0 = __ldcg(w + i);
    }
    float gsum = 0.0f;
#pragma unroll 16
    for (int b = 0; b < nblocks; ++b) gsum += __ldcg(partials + (size_t)b * kGradSlots + i);
    const float g = gsum * inv_batch;
    if (i == learned::kTrainable) {
        if (loss_out) *loss_out = g;
        return;
    }
    if (grad_out) grad_out[i] = g;
    if (lr > 0.0f) {
        const float mi = b1 * m0 + (1.0f - b1) * g;
        const float vi = b2 * v0 + (1.0f - b2) * g * g;
        m[i] = mi;
        v[i] = vi;
        const float wi = w0 - lr * (mi / bias1) / (sqrtf(vi / bias2) + eps);
        w[i] = wi;
        put_images(images, i, wi);
    }
}

// mean and 1 / standard deviation of beta k over the pairs -> w[1945],
// w[1946]: block sums in binary64, added in block order by the block that
// finishes last (the ticket returns to 0).  One block for all pairs waited
// for its loads 780 times over 200,000 pairs (255 us under ncu); with a block
// per 2048 pairs, up to one per SM, 13 us.  Up to kScalingOneBlock pairs one
// block is as fast or faster, as it needs no ticket: us per call, one block for
// all pairs / the ticket always / this, 2 pairs 13.0 / 15.4 / 13.1, 2048 15.2 / 18.1 / 15.4,
// 4096 18.0 / 18.0 / 18.0, 10,000 25.5 / 18.6 / 18.3.
constexpr int kScalingThreads = 256;
constexpr size_t kScalingOneBlock = 4096;

__global__ void __launch_bounds__(kScalingThreads)
    input_scaling_kernel(const float2 *__restrict__ pairs, long long n, double *__restrict__ sums,
                         unsigned int *__restrict__ ticket, float *__restrict__ w)
{
    double a = 0.0, b = 0.0;
#pragma unroll 4
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double x = (double)pairs[i].x;
        a += x;
        b += x * x;
    }
    block_sum2(a, b);
    if (gridDim.x > 1) {
        __shared__ bool last;
        if (threadIdx.x == 0) {
            sums[2 * blockIdx.x] = a;
            sums[2 * blockIdx.x + 1] = b;
            __threadfence();
            last = atomicAdd(ticket, 1u) == gridDim.x - 1;
        }
        __syncthreads();
        if (!last) return;
        __threadfence();
        a = b = 0.0;
        for (unsigned int i = threadIdx.x; i < gridDim.x; i += blockDim.x) {
            a += ((volatile double *)sums)[2 * i];
            b += ((volatile double *)sums)[2 * i + 1];
        }
        block_sum2(a, b);
        if (threadIdx.x == 0) *ticket = 0u;
    }
    if (threadIdx.x == 0) {
        const double mean = a / (double)n;
        const double var = b / (double)n - mean * mean;
        w[learned::kOffMean] = (float)mean;
        w[learned::kOffScale] = (float)(1.0 / sqrt(var > 1e-12 ? var : 1e-12));
    }
}

}  // namespace train
}  // namespace su2

struct su2_trainer {
    int device = 0;
    int sms = 0;
    cudaStream_t stream = nullptr;
    uint64_t seed = 0;
    uint32_t step = 0;  // Adam steps taken
    void *block = nullptr;
    size_t block_bytes = 0;
    float *w = nullptr, *m = nullptr, *v = nullptr, *grad = nullptr, *loss = nullptr;
    unsigned int *err = nullptr;  // [0] waits given up, [16] ticket of the input scaling
    unsigned char *images = nullptr;  // BF16 operand tiles of w
    float *partials = nullptr;
    int partial_blocks = 0;
    float *losses = nullptr;  // per step of the last fit
    int losses_cap = 0;
};

namespace su2 {
namespace {

constexpr int kMaxBatch = 65536;

// Launches a kernel whose prologue may overlap the tail of the previous kernel
// of the stream (it waits with griddepcontrol.wait before it touches anything
// that one writes).
template <typename... Args>
cudaError_t launch_dependent(void (*kernel)(Args...), int grid, int threads, size_t smem, cudaStream_t stream,
                             Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

su2_status trainer_launch(su2_trainer *tr, const float *pairs, long long n, int batch, int explicit_rows, float lr,
                          float *loss_dst)
{
    const int nblocks = batch / train::kRows;
    train::StepParams p;
    p.w = tr->w;
    p.images = (const uint4 *)tr->images;
    // CTAs per 128 samples: as many as keep the grid within one CTA per SM
    p.split = 4 * nblocks <= tr->sms ? 4 : (2 * nblocks <= tr->sms ? 2 : 1);
    p.pairs = (const float2 *)pairs;
    p.n_pairs = n;
    p.explicit_rows = explicit_rows;
    p.step = tr->step;
    p.k0 = (uint32_t)tr->seed;
    p.k1 = (uint32_t)(tr->seed >> 32);
    p.partials = tr->partials;
    p.err = tr->err;
    SU2_CUDA(launch_dependent(train::train_step_kernel, nblocks * p.split, train::kTrainThreads, sizeof(train::Smem), tr->stream,
                              p));
    float bias1 = 1.0f, bias2 = 1.0f;
    if (lr > 0.0f) {
        tr->step += 1;
        bias1 = 1.0f - powf(0.9f, (float)tr->step);
        bias2 = 1.0f - powf(0.999f, (float)tr->step);
    }
    SU2_CUDA(launch_dependent(train::adam_kernel, (train::kGradSlots + 63) / 64, 64, 0, tr->stream, tr->w, tr->m, tr->v,
                              (const float *)tr->partials, nblocks, 1.0f / (float)batch, lr, 0.9f, 0.999f, 1e-8f, bias1,
                              bias2, tr->grad, loss_dst, tr->images));
    return SU2_OK;
}

su2_status trainer_check(su2_trainer *tr)
{
    unsigned int err = 0;
    SU2_CUDA(cudaMemcpyAsync(&err, tr->err, sizeof err, cudaMemcpyDeviceToHost, tr->stream));
    SU2_CUDA(cudaStreamSynchronize(tr->stream));
    if (err) {
        set_last_error("training: a tensor-core completion wait gave up");
        return SU2_E_DEVICE_TIMEOUT;
    }
    return SU2_OK;
}

}  // namespace
}  // namespace su2

extern "C" {

su2_status su2_trainer_create(const float *init_weights, uint64_t seed, void *cuda_stream, su2_trainer **out)
{
    if (!init_weights || !out) return SU2_E_INVAL;
    *out = nullptr;
    int dev = 0;
    SU2_CUDA(cudaGetDevice(&dev));
    static bool attr_set[64] = {};
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        SU2_CUDA(cudaFuncSetAttribute(train::train_step_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)sizeof(train::Smem)));
        attr_set[dev] = true;
    }
    su2_trainer *tr = new (std::nothrow) su2_trainer();
    if (!tr) return SU2_E_NOMEM;
    tr->device = dev;
    tr->stream = (cudaStream_t)cuda_stream;
    tr->seed = seed;
    tr->partial_blocks = kMaxBatch / train::kRows;
    const size_t wb = 2048 * sizeof(float);
    tr->block_bytes = 5 * wb + 256 + train::kImageBytes + sizeof(float) * (size_t)tr->partial_blocks * train::kGradSlots;
    tr->block = device_alloc(tr->block_bytes, dev, tr->stream);
    if (!tr->block) {
        delete tr;
        return SU2_E_NOMEM;
    }
    char *q = (char *)tr->block;
    tr->w = (float *)q;
    tr->m = (float *)(q + wb);
    tr->v = (float *)(q + 2 * wb);
    tr->grad = (float *)(q + 3 * wb);
    tr->loss = (float *)(q + 4 * wb);
    tr->err = (unsigned int *)(q + 5 * wb);
    tr->images = (unsigned char *)(q + 5 * wb + 256);
    tr->partials = (float *)(q + 5 * wb + 256 + train::kImageBytes);
    su2_status st = SU2_OK;
    cudaError_t e = cudaDeviceGetAttribute(&tr->sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaMemsetAsync(tr->block, 0, 5 * wb + 256 + train::kImageBytes, tr->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(tr->w, init_weights, sizeof(float) * learned::kWeights, cudaMemcpyHostToDevice, tr->stream);
    if (e == cudaSuccess) {
        train::put_images_kernel<<<(learned::kTrainable + 255) / 256, 256, 0, tr->stream>>>(tr->w, tr->images);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(tr->stream);
    if (e != cudaSuccess) st = cuda_fail(e, "su2_trainer_create");
    if (st != SU2_OK) {
        su2_trainer_destroy(tr);
        return st;
    }
    *out = tr;
    return SU2_OK;
}

su2_status su2_trainer_destroy(su2_trainer *tr)
{
    if (!tr) return SU2_OK;
    DeviceGuard guard(tr->device);
    device_free(tr->losses, sizeof(float) * (size_t)tr->losses_cap, tr->device, tr->stream);
    device_free(tr->block, tr->block_bytes, tr->device, tr->stream);
    const cudaError_t e = cudaStreamSynchronize(tr->stream);
    delete tr;
    return e == cudaSuccess ? SU2_OK : cuda_fail(e, "su2_trainer_destroy");
}

su2_status su2_trainer_set_input_scaling(su2_trainer *tr, const float *dev_pairs, size_t n)
{
    if (!tr || !dev_pairs || n < 2) return SU2_E_INVAL;
    DeviceGuard guard(tr->device);
    // the block sums take the head of the step partials, idle between calls
    const int grid =
        n <= train::kScalingOneBlock ? 1 : (int)std::min<size_t>((n + 2047) / 2048, (size_t)tr->sms);
    train::input_scaling_kernel<<<grid, train::kScalingThreads, 0, tr->stream>>>(
        (const float2 *)dev_pairs, (long long)n, (double *)tr->partials, tr->err + 16, tr->w);
    SU2_CUDA(cudaGetLastError());
    SU2_CUDA(cudaStreamSynchronize(tr->stream));
    return SU2_OK;
}

su2_status su2_trainer_gradient(su2_trainer *tr, const float *dev_pairs, size_t n, double *loss, float *grad)
{
    if (!tr || !dev_pairs || n == 0 || n % train::kRows != 0 || n > (size_t)kMaxBatch) {
        set_last_error("su2_trainer_gradient: n must be a positive multiple of 128, at most 65536");
        return SU2_E_INVAL;
    }
    DeviceGuard guard(tr->device);
    SU2_CUDA(cudaMemsetAsync(tr->err, 0, sizeof(unsigned int), tr->stream));
    su2_status st = trainer_launch(tr, dev_pairs, (long long)n, (int)n, 1, 0.0f, tr->loss);
    if (st != SU2_OK) return st;
    float l = 0.0f;
    if (grad)
        SU2_CUDA(cudaMemcpyAsync(grad, tr->grad, sizeof(float) * learned::kTrainable, cudaMemcpyDeviceToHost,
                                 tr->stream));
    SU2_CUDA(cudaMemcpyAsync(&l, tr->loss, sizeof l, cudaMemcpyDeviceToHost, tr->stream));
    st = trainer_check(tr);
    if (loss) *loss = l;
    return st;
}

su2_status su2_trainer_fit(su2_trainer *tr, const float *dev_pairs, size_t n, int steps, int batch, double lr,
                           float *loss_per_step)
{
    if (!tr || !dev_pairs || n == 0 || steps < 0 || batch < train::kRows || batch % train::kRows != 0 ||
        batch > kMaxBatch || !(lr > 0.0)) {
        set_last_error("su2_trainer_fit: batch must be a multiple of 128 in [128, 65536], lr > 0");
        return SU2_E_INVAL;
    }
    DeviceGuard guard(tr->device);
    if (steps > tr->losses_cap) {
        device_free(tr->losses, sizeof(float) * (size_t)tr->losses_cap, tr->device, tr->stream);
        tr->losses = (float *)device_alloc(sizeof(float) * (size_t)steps, tr->device, tr->stream);
        tr->losses_cap = tr->losses ? steps : 0;
        if (!tr->losses) return SU2_E_NOMEM;
    }
    SU2_CUDA(cudaMemsetAsync(tr->err, 0, sizeof(unsigned int), tr->stream));
    for (int s = 0; s < steps; ++s) {
        su2_status st = trainer_launch(tr, dev_pairs, (long long)n, batch, 0, (float)lr, tr->losses + s);
        if (st != SU2_OK) return st;
    }
    if (loss_per_step && steps > 0)
        SU2_CUDA(cudaMemcpyAsync(loss_per_step, tr->losses, sizeof(float) * steps, cudaMemcpyDeviceToHost,
                                 tr->stream));
    return trainer_check(tr);
}

su2_status su2_trainer_get_weights(su2_trainer *tr, float *host)
{
    if (!tr || !host) return SU2_E_INVAL;
    DeviceGuard guard(tr->device);
    SU2_CUDA(cudaMemcpyAsync(host, tr->w, sizeof(float) * learned::kWeights, cudaMemcpyDeviceToHost, tr->stream));
    SU2_CUDA(cudaStreamSynchronize(tr->stream));
    return SU2_OK;
}

}  // extern "C"
