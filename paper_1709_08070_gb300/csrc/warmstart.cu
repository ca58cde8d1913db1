// Learned warm start for GMRES (not part of the paper's method): a small
// per-node network maps local, size-free features of the right-hand side,
// the geometry and the physical constants to an initial [psi; psin].  GMRES
// from the zero start remains the reference; the network only shortens it.
//
// Features of node i (all O(1) and independent of the molecule's size):
//   S1 = sqrt(sum w g1^2 / sum w), S2 = same for g2 (w = quadrature weights),
//   L = S1/S2 (a length), f0 = g1/S1, f1 = g2/S2, f2 = d/eps (offset in the
//   band), f3 = clamp(H L, -10, 10)/10 (H = Laplacian of the distance),
//   f4 = kappa L/(1 + kappa L), f5 = ln(eps_E/eps_I)/5,
//   f6 = (eps_I/eps_E)/(1 + kappa L), f7 = r1/S1, f8 = r2/S2 with
//   r = g - A Lambda^-1 g = -K Lambda^-1 g, the residual of the Lambda^-1 g
//   start (one application of the FP32 operator): the only non-local input,
//   it carries the reaction field of the first Neumann step to every node.
// Network: 9 -> 64 -> 64 -> 2, tanh hidden layers; BF16 weights, FP32
// arithmetic and accumulation; FP32 master weights and Adam moments.
// Outputs: psi_i = S1 o0 / lambda1, psin_i = S2 o1 / lambda2 (Lambda the
// diagonal of the system, Sec. 3.3).
// Training loss: sum over sampled nodes of (w_i / mean w) |o - t|^2 / batch,
// t = (lambda1 psi/S1, lambda2 psin/S2) of solutions the method computed.
// Scaling the targets by Lambda weights the two blocks by their share of
// the initial residual g - A p0 (A = Lambda + K), which is what GMRES sees:
// unscaled, the psi block (lambda1 = (1 + eps_E/eps_I)/2, 40.5 for
// water/protein) would be under-weighted by lambda1^2.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "ibim_internal.cuh"
#include "ptx.cuh"

namespace ibim {

constexpr int kWsIn = 9, kWsH = 64, kWsOut = 2;
constexpr int kOffW1 = 0;
constexpr int kOffB1 = kOffW1 + kWsH * kWsIn;
constexpr int kOffW2 = kOffB1 + kWsH;
constexpr int kOffB2 = kOffW2 + kWsH * kWsH;
constexpr int kOffW3 = kOffB2 + kWsH;
constexpr int kOffB3 = kOffW3 + kWsOut * kWsH;
constexpr int kWsParams = kOffB3 + kWsOut;  // 4930
constexpr int kWsThreads = 128;             // prediction: nodes per block
constexpr int kHPad = kWsH + 1;             // padded smem row (bank conflicts)
constexpr int kTrainThreads = 256;
constexpr int kTrainBlock = 128;            // training: nodes per block (a pair of CTAs)
constexpr int kTrainNodes = kTrainBlock / 2;  // a CTA's half of it
constexpr int kTrainRow = kTrainNodes + 4;  // row of a transposed half (16-byte aligned, rows four banks apart)
constexpr int kTrainOwn = 20;               // a thread's parameters in the training kernel
constexpr int kPartStride = kWsParams + 2;  // a CTA's gradient, 16-byte aligned

static_assert(kWsParams == IBIM_WS_NPARAMS, "parameter count");

}  // namespace ibim

struct ibim_wsnet {
    int device = 0;
    cudaStream_t stream = nullptr;
    float* d_w = nullptr;           // FP32 master parameters
    __nv_bfloat16* d_wb = nullptr;  // BF16 parameters used by the kernels
    float* d_m = nullptr;           // Adam first moment
    float* d_v = nullptr;           // Adam second moment
    float* d_g = nullptr;           // gradient, then the training CTAs' partial gradients
    double* d_loss = nullptr;       // loss, then the training CTAs' partial losses
    int num_sms = 0;
    double* d_scal = nullptr;       // S1, S2 scratch
    float* d_feat = nullptr;        // training features (n_ex x 8)
    float* d_tgt = nullptr;         // training targets (n_ex x 2)
    float* d_wt = nullptr;          // training node weights (n_ex)
    int64_t n_ex = 0, cap_ex = 0;
    int64_t step = 0;
    uint64_t seed = 0;
};

namespace ibim {

namespace cg = cooperative_groups;

// ---------------------------------------------------------------- features

// S1, S2 (one CTA, fixed summation order).
__global__ void ws_scales_kernel(const double* __restrict__ g, const double* __restrict__ w, int64_t N,
                                 double* __restrict__ scal)
{
    __shared__ double r[3][256];
    double a = 0.0, b = 0.0, c = 0.0;
    for (int64_t i = threadIdx.x; i < N; i += blockDim.x) {
        a += w[i] * g[i] * g[i];
        b += w[i] * g[N + i] * g[N + i];
        c += w[i];
    }
    r[0][threadIdx.x] = a;
    r[1][threadIdx.x] = b;
    r[2][threadIdx.x] = c;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o)
            for (int q = 0; q < 3; ++q) r[q][threadIdx.x] += r[q][threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double sw = r[2][0] > 0.0 ? r[2][0] : 1.0;
        const double s1 = sqrt(r[0][0] / sw), s2 = sqrt(r[1][0] / sw);
        scal[0] = s1 > 0.0 ? s1 : 1.0;
        scal[1] = s2 > 0.0 ? s2 : 1.0;
        scal[2] = sw / (double)(N > 0 ? N : 1);  // mean weight
    }
}

struct WsPhys {
    double kappa, eps_ratio_log, inv_ratio, band_eps;
};

__global__ void ws_features_kernel(const double* __restrict__ g, const double* __restrict__ Ax0,
                                   const double* __restrict__ dist, const double* __restrict__ curv, int64_t N,
                                   const double* __restrict__ scal, WsPhys ph, float* __restrict__ feat)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double S1 = scal[0], S2 = scal[1];
    const double L = S1 / S2;
    const double kL = ph.kappa * L;
    double hl = curv[i] * L;
    hl = hl > 10.0 ? 10.0 : (hl < -10.0 ? -10.0 : hl);
    float* f = feat + i * kWsIn;
    f[0] = (float)(g[i] / S1);
    f[1] = (float)(g[N + i] / S2);
    f[2] = (float)(ph.band_eps > 0.0 ? dist[i] / ph.band_eps : 0.0);
    f[3] = (float)(hl / 10.0);
    f[4] = (float)(kL / (1.0 + kL));
    f[5] = (float)(ph.eps_ratio_log / 5.0);
    f[6] = (float)(ph.inv_ratio / (1.0 + kL));
    f[7] = (float)((g[i] - Ax0[i]) / S1);
    f[8] = (float)((g[N + i] - Ax0[N + i]) / S2);
}

// x0 = Lambda^-1 g (the start of Sec. 3.3).
__global__ void ws_start_kernel(const double* __restrict__ g, int64_t N, double lambda1, double lambda2,
                                double* __restrict__ x0)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    x0[i] = g[i] / lambda1;
    x0[N + i] = g[N + i] / lambda2;
}

__global__ void ws_targets_kernel(const double* __restrict__ p, const double* __restrict__ w, int64_t N,
                                  const double* __restrict__ scal, double lambda1, double lambda2,
                                  float* __restrict__ tgt, float* __restrict__ wt)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    tgt[2 * i] = (float)(lambda1 * p[i] / scal[0]);
    tgt[2 * i + 1] = (float)(lambda2 * p[N + i] / scal[1]);
    wt[i] = (float)(w[i] / scal[2]);
}

// ----------------------------------------------------------------- network

__device__ __forceinline__ void load_params(const __nv_bfloat16* __restrict__ wb, float* sp)
{
    for (int q = threadIdx.x; q < kWsParams; q += blockDim.x) sp[q] = __bfloat162float(wb[q]);
}

// Forward pass of one node from its features (params in shared memory).
__device__ __forceinline__ void ws_forward(const float* sp, const float* x, float* h1, float* h2, float* o)
{
    for (int a = 0; a < kWsH; ++a) {
        float s = sp[kOffB1 + a];
#pragma unroll
        for (int b = 0; b < kWsIn; ++b) s = fmaf(sp[kOffW1 + a * kWsIn + b], x[b], s);
        h1[a] = tanhf(s);
    }
    for (int a = 0; a < kWsH; ++a) {
        float s = sp[kOffB2 + a];
        for (int b = 0; b < kWsH; ++b) s = fmaf(sp[kOffW2 + a * kWsH + b], h1[b], s);
        h2[a] = tanhf(s);
    }
    for (int c = 0; c < kWsOut; ++c) {
        float s = sp[kOffB3 + c];
        for (int a = 0; a < kWsH; ++a) s = fmaf(sp[kOffW3 + c * kWsH + a], h2[a], s);
        o[c] = s;
    }
}

__global__ void __launch_bounds__(kWsThreads)
    ws_predict_kernel(const float* __restrict__ feat, int64_t N, const __nv_bfloat16* __restrict__ wb,
                      const double* __restrict__ scal, double lambda1, double lambda2, double* __restrict__ p0)
{
    extern __shared__ float smem[];
    float* sp = smem;
    float* rows = smem + kWsParams;  // per thread: h1, h2 (2 x kHPad)
    load_params(wb, sp);
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    float x[kWsIn];
#pragma unroll
    for (int b = 0; b < kWsIn; ++b) x[b] = feat[i * kWsIn + b];
    float* h1 = rows + threadIdx.x * 2 * kHPad;
    float* h2 = h1 + kHPad;
    float o[kWsOut];
    ws_forward(sp, x, h1, h2, o);
    p0[i] = scal[0] * (double)o[0] / lambda1;
    p0[N + i] = scal[1] * (double)o[1] / lambda2;
}

// splitmix64 (Steele, Lea, Flood 2014) for minibatch sampling.
__device__ __forceinline__ uint64_t mix64(uint64_t z)
{
    z += 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

// Shared memory of the training kernel (floats).
struct TrainSmem {
    float W1T[kWsIn][kWsH];          // [input][unit]
    float W2[kWsH][kWsH];            // [unit 2][unit 1]
    float W2T[kWsH][kWsH];           // [unit 1][unit 2]
    float W3[kWsOut][kWsH];
    float b1[kWsH], b2[kWsH], b3[kWsOut + 2];
    float X[kWsIn][kTrainRow];       // activations transposed: [unit][node]
    float H1[kWsH][kTrainRow];
    float H2[kWsH][kTrainRow];
    float D1[kWsH][kTrainRow];
    float D2[kWsH][kTrainRow];
    float dO[kWsOut][kTrainRow];
    float e[kWsOut][kTrainRow];
    float wt[kTrainNodes], tgt[kWsOut][kTrainNodes];
    float carry[kTrainOwn][kTrainThreads];  // second CTA of a pair: the first one's sums
    double loss[kTrainNodes];
};

// acc[i][j] = sum_k A[k][4 ty + i] B[k][4 tx + j] on top of acc's start values, k ascending.
template <int K, int LDA, int LDB>
__device__ __forceinline__ void tile_product(const float (*A)[LDA], const float (*B)[LDB], int ty, int tx,
                                             float (&acc)[4][4])
{
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
        const float4 a = *reinterpret_cast<const float4*>(&A[k][4 * ty]);
        const float4 b = *reinterpret_cast<const float4*>(&B[k][4 * tx]);
        const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(bv[j], av[i], acc[i][j]);
    }
}

__device__ __forceinline__ float dot4(const float4& a, const float4& b, float s)
{
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, s))));
}

// s + e == a + b exactly (Knuth's two-sum); e is added to lo.
__device__ __forceinline__ void add_exact(float& hi, float& lo, float x)
{
    const float s = hi + x, b = s - hi;
    lo += (hi - (s - b)) + (x - b);
    hi = s;
}

// Loss and gradient over a batch: node of slot s is either consecutive (first +
// s, full-batch mode) or drawn at random.  The gradient is a sum over blocks of
// 128 nodes: within a block every parameter's products are added node by node in
// FP32, across blocks the sum is exact to float-float (add_exact here, then
// ws_update_kernel) and rounded once.  The BF16 weights of the next step turn a
// difference of one rounding into one of 2^-9 where a weight lies near a
// boundary, so this order is part of the result (64-node tiles, summed in FP32,
// left the results of the former one-thread-per-node kernel, FP32 atomics over
// the same blocks in a varying order, in 4 of 16 runs of 50 steps).
// A pair of CTAs takes a block: each its half of the nodes through the network and
// back; the first then forms its sums and hands them over in the second's shared
// memory, and the second goes on from them.  The products (layer 2 forward, its
// backward, its weight gradient) run as register tiles of 4 x 4 per thread from
// shared memory, activations stored transposed so that every operand is a float4.
// A pair takes blocks p, p + pairs, ... and writes one partial gradient.
// 242 MFLOP at 8,192 nodes: 3 us of the FP32 pipe; bound by the latency of its
// phases.  Measured 24 us a step with the Adam kernel, launches overlapped (92 us
// with one thread per node, FP32 atomics and two memsets; 20 us with 64-node tiles
// summed apart; 30 us with a whole block on one CTA of 512 threads).
__global__ void __cluster_dims__(2) __launch_bounds__(kTrainThreads, 1)
    ws_grad_kernel(const float* __restrict__ feat, const float* __restrict__ tgt, const float* __restrict__ wt,
                   int64_t n_ex, int64_t first, int64_t count, int random, uint64_t seed, double inv_batch,
                   const __nv_bfloat16* __restrict__ wb, float* __restrict__ part, double* __restrict__ part_loss)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TrainSmem& S = *reinterpret_cast<TrainSmem*>(smem_raw);
    const cg::cluster_group pair = cg::this_cluster();
    const int second = (int)pair.block_rank();
    const int64_t npairs = gridDim.x / 2, first_block = blockIdx.x / 2;
    const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
    // four threads per node fetch its features, target and weight (zeros past the batch)
    auto fetch = [&](int64_t block) {
        const int n = t & (kTrainNodes - 1), part4 = t / kTrainNodes;
        const int64_t slot = block * kTrainBlock + second * kTrainNodes + n;
        const bool live = slot < count;
        int64_t i = 0;
        if (live) i = random ? (int64_t)(mix64(seed ^ (uint64_t)slot) % (uint64_t)n_ex) : first + slot;
        for (int b = part4; b < kWsIn; b += 4) S.X[b][n] = live ? feat[i * kWsIn + b] : 0.0f;
        if (part4 == 0) S.wt[n] = live ? wt[i] : 0.0f;
        if (part4 >= 1 && part4 <= kWsOut) S.tgt[part4 - 1][n] = live ? tgt[kWsOut * i + part4 - 1] : 0.0f;
    };
    ptx::grid_dep_launch();  // the Adam kernel may be set up; it waits for this grid
    // this step's first features while the previous Adam step finishes
    fetch(first_block);
    ptx::grid_dep_wait();
    const __nv_bfloat162* w2 = reinterpret_cast<const __nv_bfloat162*>(wb + kOffW2);
#pragma unroll 4
    for (int q = t; q < kWsH * kWsH / 2; q += kTrainThreads) {
        // once along the rows, once across them, so that neither copy stores with bank conflicts
        const int r = q / (kWsH / 2), c = q % (kWsH / 2);
        *reinterpret_cast<float2*>(&S.W2[r][2 * c]) = __bfloat1622float2(w2[q]);
        const int a = q % kWsH, p = q / kWsH;
        const float2 v = __bfloat1622float2(w2[a * (kWsH / 2) + p]);
        S.W2T[2 * p][a] = v.x;
        S.W2T[2 * p + 1][a] = v.y;
    }
    for (int q = t; q < kWsH * kWsIn; q += kTrainThreads) S.W1T[q / kWsH][q % kWsH] = __bfloat162float(wb[kOffW1 + (q % kWsH) * kWsIn + q / kWsH]);
    for (int q = t; q < kWsOut * kWsH; q += kTrainThreads) S.W3[q / kWsH][q % kWsH] = __bfloat162float(wb[kOffW3 + q]);
    if (t < kWsH) {
        S.b1[t] = __bfloat162float(wb[kOffB1 + t]);
        S.b2[t] = __bfloat162float(wb[kOffB2 + t]);
    }
    if (t < kWsOut) S.b3[t] = __bfloat162float(wb[kOffB3 + t]);

    // a thread's parameters: W2, units ty + 16 i (layer 2) x tx + 16 j (layer 1); W1, unit t % 64 and inputs
    // t / 64 + 4 i, the bias in the last; W3[t / 64][t % 64] (t < 128), b2 (t - 128 < 64) or b3 (t - 192 < 2)
    constexpr int kW1 = 16, kRest = 19;
    const bool ownW3 = t < 128, ownB2 = t >= 128 && t < 192, ownB3 = t >= 192 && t < 192 + kWsOut;
    float hi[kTrainOwn], lo[kTrainOwn];  // sums over the pair's blocks
    double l = 0.0;                      // t < 64: loss of the half's nodes t
#pragma unroll
    for (int q = 0; q < kTrainOwn; ++q) hi[q] = lo[q] = 0.0f;

    for (int64_t block = first_block; block * kTrainBlock < count; block += npairs) {
        if (block != first_block) {
            __syncthreads();
            fetch(block);
        }
        pair.barrier_arrive();  // the second CTA's hand-over buffer is free
        __syncthreads();
        float acc[4][4];  // nodes 4 ty + i, units 4 tx + j
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = S.b1[4 * tx + j];
        tile_product<kWsIn>(S.X, S.W1T, ty, tx, acc);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            *reinterpret_cast<float4*>(&S.H1[4 * tx + j][4 * ty]) =
                make_float4(tanhf(acc[0][j]), tanhf(acc[1][j]), tanhf(acc[2][j]), tanhf(acc[3][j]));
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = S.b2[4 * tx + j];
        tile_product<kWsH>(S.H1, S.W2T, ty, tx, acc);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            *reinterpret_cast<float4*>(&S.H2[4 * tx + j][4 * ty]) =
                make_float4(tanhf(acc[0][j]), tanhf(acc[1][j]), tanhf(acc[2][j]), tanhf(acc[3][j]));
        __syncthreads();
        if (t < kWsOut * kTrainNodes) {  // outputs
            const int c = t / kTrainNodes, n = t % kTrainNodes;
            float s = S.b3[c];
#pragma unroll 8
            for (int a = 0; a < kWsH; ++a) s = fmaf(S.W3[c][a], S.H2[a][n], s);
            const float e = block * kTrainBlock + second * kTrainNodes + n < count ? s - S.tgt[c][n] : 0.0f;
            S.e[c][n] = e;
            S.dO[c][n] = (float)(2.0 * inv_batch) * S.wt[n] * e;
        }
        __syncthreads();
        if (t < kTrainNodes) {
            const float w = S.wt[t], e0 = S.e[0][t], e1 = S.e[1][t];
            l += (double)w * ((double)e0 * e0 + (double)e1 * e1) * inv_batch;
        }
        for (int q = t; q < kWsH * kTrainNodes; q += kTrainThreads) {
            const int a = q / kTrainNodes, n = q % kTrainNodes;
            const float h = S.H2[a][n];
            float s = fmaf(S.W3[0][a], S.dO[0][n], 0.0f);
            s = fmaf(S.W3[1][a], S.dO[1][n], s);
            S.D2[a][n] = s * (1.0f - h * h);
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
        tile_product<kWsH>(S.D2, S.W2, ty, tx, acc);  // d1 before the derivative of tanh
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 h = *reinterpret_cast<const float4*>(&S.H1[4 * tx + j][4 * ty]);
            *reinterpret_cast<float4*>(&S.D1[4 * tx + j][4 * ty]) =
                make_float4(acc[0][j] * (1.0f - h.x * h.x), acc[1][j] * (1.0f - h.y * h.y),
                            acc[2][j] * (1.0f - h.z * h.z), acc[3][j] * (1.0f - h.w * h.w));
        }
        __syncthreads();
        pair.barrier_wait();
        // the block's sums, node by node: the first CTA's from zero, the second's from the first's
        float g[kTrainOwn];
        auto sums = [&]() {
#pragma unroll 2
            for (int n = 0; n < kTrainNodes; n += 4) {  // dW2[a][b] = sum_n d2[n][a] h1[n][b]
                float4 d[4], h[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    d[i] = *reinterpret_cast<const float4*>(&S.D2[ty + 16 * i][n]);
                    h[i] = *reinterpret_cast<const float4*>(&S.H1[tx + 16 * i][n]);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) g[4 * i + j] = dot4(d[i], h[j], g[4 * i + j]);
            }
#pragma unroll 4
            for (int n = 0; n < kTrainNodes; n += 4) {  // dW1[a][b] = sum_n d1[n][a] x[n][b], the bias as one more input
                const float4 d = *reinterpret_cast<const float4*>(&S.D1[t % kWsH][n]);
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const int b = t / kWsH + 4 * i;
                    if (b < kWsIn) g[kW1 + i] = dot4(d, *reinterpret_cast<const float4*>(&S.X[b][n]), g[kW1 + i]);
                    else if (b == kWsIn) g[kW1 + i] = (((g[kW1 + i] + d.x) + d.y) + d.z) + d.w;
                }
            }
            if (ownW3)  // dW3[c][a] = sum_n dO[n][c] h2[n][a]
#pragma unroll 4
                for (int n = 0; n < kTrainNodes; n += 4)
                    g[kRest] = dot4(*reinterpret_cast<const float4*>(&S.dO[t / kWsH][n]),
                                    *reinterpret_cast<const float4*>(&S.H2[t % kWsH][n]), g[kRest]);
            else if (ownB2 || ownB3) {
                const float* row = ownB2 ? S.D2[t - 128] : S.dO[t - 192];
#pragma unroll 8
                for (int n = 0; n < kTrainNodes; ++n) g[kRest] += row[n];
            }
        };
        if (!second) {
#pragma unroll
            for (int q = 0; q < kTrainOwn; ++q) g[q] = 0.0f;
            sums();
            float* carry = pair.map_shared_rank(&S.carry[0][0], 1);
#pragma unroll
            for (int q = 0; q < kTrainOwn; ++q) carry[q * kTrainThreads + t] = g[q];
        }
        pair.sync();
        if (second) {
#pragma unroll
            for (int q = 0; q < kTrainOwn; ++q) g[q] = S.carry[q][t];
            sums();
#pragma unroll
            for (int q = 0; q < kTrainOwn; ++q) add_exact(hi[q], lo[q], g[q]);
        }
    }

    // the pair's partial gradient; with several blocks the low parts as a second one
    auto store = [&](float* p, const float (&v)[kTrainOwn]) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) p[kOffW2 + (ty + 16 * i) * kWsH + tx + 16 * j] = v[4 * i + j];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int a = t % kWsH, b = t / kWsH + 4 * i;
            if (b < kWsIn) p[kOffW1 + a * kWsIn + b] = v[kW1 + i];
            else if (b == kWsIn) p[kOffB1 + a] = v[kW1 + i];
        }
        if (ownW3) p[kOffW3 + t] = v[kRest];
        if (ownB2) p[kOffB2 + t - 128] = v[kRest];
        if (ownB3) p[kOffB3 + t - 192] = v[kRest];
    };
    if (second) {
        store(part + first_block * kPartStride, hi);
        if (count > npairs * kTrainBlock) store(part + (npairs + first_block) * kPartStride, lo);
    }
    if (t < kTrainNodes) S.loss[t] = l;
    for (int o = kTrainNodes / 2; o > 0; o >>= 1) {
        __syncthreads();
        if (t < o) S.loss[t] += S.loss[t + o];
    }
    if (t == 0) part_loss[blockIdx.x] = S.loss[0];
}

// Sums the partial gradients (kSumParts threads per parameter over fixed shares,
// exact to float-float) and the CTAs' losses; with adam, one Adam step (Kingma and Ba 2015) on the FP32
// master weights, which refreshes the BF16 copy; else the gradient goes to grad.
constexpr int kSumParts = 8, kSumParams = 32;
__global__ void __launch_bounds__(kSumParts * kSumParams)
    ws_update_kernel(const float* __restrict__ part, const double* __restrict__ part_loss, int nparts, int ctas, int adam,
                     float* __restrict__ w, float* __restrict__ m, float* __restrict__ v, __nv_bfloat16* __restrict__ wb,
                     float lr, float b1, float b2, float c1, float c2, float* __restrict__ grad,
                     double* __restrict__ loss)
{
    __shared__ double sh[kSumParts][kSumParams];
    ptx::grid_dep_launch();  // the next step's gradient may be set up; it waits for this grid
    ptx::grid_dep_wait();
    const int ql = threadIdx.x % kSumParams, pr = threadIdx.x / kSumParams;
    const int q = blockIdx.x * kSumParams + ql;
    float hi = 0.0f, lo = 0.0f;
    if (q < kWsParams) {
#pragma unroll 8
        for (int p = pr; p < nparts; p += kSumParts) add_exact(hi, lo, part[(int64_t)p * kPartStride + q]);
    }
    double d = (double)hi + (double)lo;
    sh[pr][ql] = d;
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        double v = 0.0;
        for (int p = threadIdx.x; p < ctas; p += 32) v += part_loss[p];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (threadIdx.x == 0) *loss = v;
    }
    __syncthreads();
    if (pr != 0 || q >= kWsParams) return;
    for (int p = 1; p < kSumParts; ++p) d += sh[p][ql];
    const float s = (float)d;
    if (!adam) {
        grad[q] = s;
        return;
    }
    const float mq = b1 * m[q] + (1.0f - b1) * s;
    const float vq = b2 * v[q] + (1.0f - b2) * s * s;
    m[q] = mq;
    v[q] = vq;
    const float wq = w[q] - lr * (mq / c1) / (sqrtf(vq / c2) + 1e-8f);
    w[q] = wq;
    wb[q] = __float2bfloat16_rn(wq);
}

__global__ void ws_to_bf16_kernel(const float* __restrict__ w, __nv_bfloat16* __restrict__ wb)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q < kWsParams) wb[q] = __float2bfloat16_rn(w[q]);
}

static size_t grad_smem() { return sizeof(TrainSmem); }
// CTAs of a training launch: a pair for each block, at most one CTA per SM
static unsigned grad_ctas(const ibim_wsnet* n, int64_t count)
{
    return 2u * (unsigned)std::min<int64_t>(std::max(1, n->num_sms / 2), (count + kTrainBlock - 1) / kTrainBlock);
}
// partial gradients of such a launch (see ws_grad_kernel)
static int grad_nparts(unsigned ctas, int64_t count) { return (int)ctas / 2 * (count > (int64_t)ctas * kTrainNodes ? 2 : 1); }
// the partial gradients behind the gradient, the partial losses behind the loss
static float* grad_parts(const ibim_wsnet* n) { return n->d_g + kPartStride; }
static double* loss_parts(const ibim_wsnet* n) { return n->d_loss + 2; }
static size_t predict_smem() { return sizeof(float) * (kWsParams + kWsThreads * 2 * kHPad); }

// Features (into c->d_io as floats after the RHS) and scales of one context.
static ibim_status ws_prepare(ibim_wsnet* net, ibim_ctx* c, const ibim_phys& p, float** feat_out)
{
    const int64_t N = c->N;
    // d_io: 2N doubles RHS g, 2N doubles x0 = Lambda^-1 g, 2N doubles A x0,
    // then N x kWsIn floats features
    IBIM_TRY(ensure(c, (void**)&c->d_io, &c->io_bytes, sizeof(double) * 6 * N + sizeof(float) * kWsIn * N + 64));
    double* g = c->d_io;
    double* x0 = c->d_io + 2 * N;
    double* ax0 = c->d_io + 4 * N;
    float* feat = (float*)(c->d_io + 6 * N);
    IBIM_TRY(rhs_launch(c, p.eps_in, g));
    const PairConsts k = make_consts(p);
    ws_start_kernel<<<(unsigned)((N + 255) / 256), 256, 0, c->stream>>>(g, N, k.lambda1, k.lambda2, x0);
    count_launch(c);
    IBIM_CUDA(cudaGetLastError());
    IBIM_TRY(apply_operator(c, k, IBIM_F32C, VecRef{x0, nullptr, 0, 0}, OutRef{ax0, nullptr, 0, 0}, nullptr));
    ws_scales_kernel<<<1, 256, 0, c->stream>>>(g, c->d_geo64 + 6 * N, N, net->d_scal);
    WsPhys ph;
    ph.kappa = p.kappa;
    ph.eps_ratio_log = log(p.eps_out / p.eps_in);
    ph.inv_ratio = p.eps_in / p.eps_out;
    ph.band_eps = c->band_eps;
    ws_features_kernel<<<(unsigned)((N + 255) / 256), 256, 0, c->stream>>>(g, ax0, c->d_dist, c->d_curv, N,
                                                                          net->d_scal, ph, feat);
    count_launch(c, 2);
    IBIM_CUDA(cudaGetLastError());
    *feat_out = feat;
    return IBIM_OK;
}

// Splitmix-driven uniform initialisation, Glorot bounds per layer.
static void init_params(uint64_t seed, std::vector<float>& w)
{
    w.assign(kWsParams, 0.0f);
    uint64_t s = seed;
    auto next = [&]() {
        s += 0x9e3779b97f4a7c15ull;
        uint64_t z = s;
        z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
        z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
        z ^= z >> 31;
        return (double)(z >> 11) * (1.0 / 9007199254740992.0);
    };
    auto fill = [&](int off, int fan_in, int fan_out) {
        const double a = sqrt(6.0 / (fan_in + fan_out));
        for (int q = 0; q < fan_in * fan_out; ++q) w[off + q] = (float)((2.0 * next() - 1.0) * a);
    };
    fill(kOffW1, kWsIn, kWsH);
    fill(kOffW2, kWsH, kWsH);
    fill(kOffW3, kWsH, kWsOut);
}

}  // namespace ibim

using namespace ibim;

extern "C" {

void ibim_wsnet_destroy(ibim_wsnet* n)
{
    if (n == nullptr) return;
    cudaStreamSynchronize(n->stream);
    cudaFree(n->d_w);
    cudaFree(n->d_wb);
    cudaFree(n->d_m);
    cudaFree(n->d_v);
    cudaFree(n->d_g);
    cudaFree(n->d_loss);
    cudaFree(n->d_scal);
    cudaFree(n->d_feat);
    cudaFree(n->d_tgt);
    cudaFree(n->d_wt);
    delete n;
}

ibim_status ibim_wsnet_create(uint64_t seed, void* stream, ibim_wsnet** out)
{
    if (out == nullptr) {
        set_error("out is NULL");
        return IBIM_ERR_ARG;
    }
    *out = nullptr;
    ibim_wsnet* n = new ibim_wsnet();
    n->stream = (cudaStream_t)stream;
    n->seed = seed;
    std::vector<float> w;
    init_params(seed, w);
    cudaError_t e = cudaGetDevice(&n->device);
    if (e == cudaSuccess) e = cudaMalloc((void**)&n->d_w, sizeof(float) * kWsParams);
    if (e == cudaSuccess) e = cudaMalloc((void**)&n->d_wb, sizeof(__nv_bfloat16) * kWsParams);
    if (e == cudaSuccess) e = cudaMalloc((void**)&n->d_m, sizeof(float) * kWsParams);
    if (e == cudaSuccess) e = cudaMalloc((void**)&n->d_v, sizeof(float) * kWsParams);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n->num_sms, cudaDevAttrMultiProcessorCount, n->device);
    if (e == cudaSuccess) e = cudaMalloc((void**)&n->d_g, sizeof(float) * kPartStride * (2 + (size_t)n->num_sms));
    if (e == cudaSuccess) e = cudaMalloc((void**)&n->d_loss, sizeof(double) * (3 + (size_t)n->num_sms));
    if (e == cudaSuccess) e = cudaMalloc((void**)&n->d_scal, sizeof(double) * 4);
    if (e == cudaSuccess) e = cudaMemcpyAsync(n->d_w, w.data(), sizeof(float) * kWsParams, cudaMemcpyHostToDevice, n->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(n->d_m, 0, sizeof(float) * kWsParams, n->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(n->d_v, 0, sizeof(float) * kWsParams, n->stream);
    if (e == cudaSuccess) {
        ws_to_bf16_kernel<<<(kWsParams + 255) / 256, 256, 0, n->stream>>>(n->d_w, n->d_wb);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(ws_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)grad_smem());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(ws_predict_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)predict_smem());
    if (e == cudaSuccess) e = cudaStreamSynchronize(n->stream);
    if (e != cudaSuccess) {
        ibim_wsnet_destroy(n);
        return cuda_fail(e, "wsnet create", __FILE__, __LINE__);
    }
    *out = n;
    return IBIM_OK;
}

ibim_status ibim_wsnet_get_params(const ibim_wsnet* n, float* h_params)
{
    if (n == nullptr || h_params == nullptr) {
        set_error("NULL argument");
        return IBIM_ERR_ARG;
    }
    IBIM_CUDA(cudaMemcpyAsync(h_params, n->d_w, sizeof(float) * kWsParams, cudaMemcpyDeviceToHost, n->stream));
    IBIM_CUDA(cudaStreamSynchronize(n->stream));
    return IBIM_OK;
}

ibim_status ibim_wsnet_set_params(ibim_wsnet* n, const float* h_params)
{
    if (n == nullptr || h_params == nullptr) {
        set_error("NULL argument");
        return IBIM_ERR_ARG;
    }
    for (int q = 0; q < kWsParams; ++q)
        if (!isfinite(h_params[q])) {
            set_error("non-finite parameter");
            return IBIM_ERR_NONFINITE;
        }
    IBIM_CUDA(cudaMemcpyAsync(n->d_w, h_params, sizeof(float) * kWsParams, cudaMemcpyHostToDevice, n->stream));
    ws_to_bf16_kernel<<<(kWsParams + 255) / 256, 256, 0, n->stream>>>(n->d_w, n->d_wb);
    IBIM_CUDA(cudaGetLastError());
    IBIM_CUDA(cudaMemsetAsync(n->d_m, 0, sizeof(float) * kWsParams, n->stream));
    IBIM_CUDA(cudaMemsetAsync(n->d_v, 0, sizeof(float) * kWsParams, n->stream));
    IBIM_CUDA(cudaStreamSynchronize(n->stream));
    n->step = 0;
    return IBIM_OK;
}

ibim_status ibim_wsnet_features(ibim_wsnet* n, ibim_ctx* c, const ibim_phys* p, float* h_feat, double* h_scales)
{
    if (n == nullptr || c == nullptr) {
        set_error("NULL argument");
        return IBIM_ERR_ARG;
    }
    IBIM_TRY(check_phys(p));
    if (c->Nc <= 0) {
        set_error("no charges set");
        return IBIM_ERR_STATE;
    }
    float* feat = nullptr;
    IBIM_TRY(ws_prepare(n, c, *p, &feat));
    if (h_feat) IBIM_CUDA(cudaMemcpyAsync(h_feat, feat, sizeof(float) * kWsIn * c->N, cudaMemcpyDeviceToHost, c->stream));
    if (h_scales) IBIM_CUDA(cudaMemcpyAsync(h_scales, n->d_scal, sizeof(double) * 3, cudaMemcpyDeviceToHost, c->stream));
    IBIM_CUDA(cudaStreamSynchronize(c->stream));
    return IBIM_OK;
}

ibim_status ibim_wsnet_add_example(ibim_wsnet* n, ibim_ctx* c, const ibim_phys* p, const double* d_p)
{
    if (n == nullptr || c == nullptr || d_p == nullptr) {
        set_error("NULL argument");
        return IBIM_ERR_ARG;
    }
    IBIM_TRY(check_phys(p));
    if (c->Nc <= 0) {
        set_error("no charges set");
        return IBIM_ERR_STATE;
    }
    const int64_t N = c->N;
    if (n->n_ex + N > n->cap_ex) {
        int64_t cap = std::max<int64_t>(2 * n->cap_ex, n->n_ex + N);
        float *f = nullptr, *t = nullptr, *w = nullptr;
        IBIM_CUDA(cudaStreamSynchronize(n->stream));
        IBIM_CUDA(cudaMalloc((void**)&f, sizeof(float) * kWsIn * cap));
        IBIM_CUDA(cudaMalloc((void**)&t, sizeof(float) * kWsOut * cap));
        IBIM_CUDA(cudaMalloc((void**)&w, sizeof(float) * cap));
        if (n->n_ex > 0) {
            IBIM_CUDA(cudaMemcpy(f, n->d_feat, sizeof(float) * kWsIn * n->n_ex, cudaMemcpyDeviceToDevice));
            IBIM_CUDA(cudaMemcpy(t, n->d_tgt, sizeof(float) * kWsOut * n->n_ex, cudaMemcpyDeviceToDevice));
            IBIM_CUDA(cudaMemcpy(w, n->d_wt, sizeof(float) * n->n_ex, cudaMemcpyDeviceToDevice));
        }
        cudaFree(n->d_feat);
        cudaFree(n->d_tgt);
        cudaFree(n->d_wt);
        n->d_feat = f;
        n->d_tgt = t;
        n->d_wt = w;
        n->cap_ex = cap;
    }
    float* feat = nullptr;
    IBIM_TRY(ws_prepare(n, c, *p, &feat));
    IBIM_CUDA(cudaMemcpyAsync(n->d_feat + kWsIn * n->n_ex, feat, sizeof(float) * kWsIn * N, cudaMemcpyDeviceToDevice,
                              c->stream));
    const PairConsts k = make_consts(*p);
    ws_targets_kernel<<<(unsigned)((N + 255) / 256), 256, 0, c->stream>>>(
        d_p, c->d_geo64 + 6 * N, N, n->d_scal, k.lambda1, k.lambda2, n->d_tgt + kWsOut * n->n_ex, n->d_wt + n->n_ex);
    count_launch(c);
    IBIM_CUDA(cudaGetLastError());
    IBIM_CUDA(cudaStreamSynchronize(c->stream));
    n->n_ex += N;
    return IBIM_OK;
}

ibim_status ibim_wsnet_num_examples(const ibim_wsnet* n, int64_t* count)
{
    if (n == nullptr || count == nullptr) {
        set_error("NULL argument");
        return IBIM_ERR_ARG;
    }
    *count = n->n_ex;
    return IBIM_OK;
}

ibim_status ibim_wsnet_gradient(ibim_wsnet* n, int64_t first, int64_t count, double* loss, float* h_grad)
{
    if (n == nullptr || loss == nullptr || h_grad == nullptr || first < 0 || count < 1 || first + count > n->n_ex) {
        set_error("need a net and 0 <= first, first + count <= number of examples, count >= 1");
        return IBIM_ERR_ARG;
    }
    const unsigned ctas = grad_ctas(n, count);
    ws_grad_kernel<<<ctas, kTrainThreads, grad_smem(), n->stream>>>(n->d_feat, n->d_tgt, n->d_wt, n->n_ex, first, count,
                                                                    0, 0, 1.0 / (double)count, n->d_wb, grad_parts(n),
                                                                    loss_parts(n));
    ws_update_kernel<<<(kWsParams + kSumParams - 1) / kSumParams, kSumParts * kSumParams, 0, n->stream>>>(
        grad_parts(n), loss_parts(n), grad_nparts(ctas, count), (int)ctas, 0, n->d_w, n->d_m, n->d_v, n->d_wb, 0.0f, 0.0f, 0.0f, 1.0f, 1.0f,
        n->d_g, n->d_loss);
    IBIM_CUDA(cudaGetLastError());
    IBIM_CUDA(cudaMemcpyAsync(h_grad, n->d_g, sizeof(float) * kWsParams, cudaMemcpyDeviceToHost, n->stream));
    IBIM_CUDA(cudaMemcpyAsync(loss, n->d_loss, sizeof(double), cudaMemcpyDeviceToHost, n->stream));
    IBIM_CUDA(cudaStreamSynchronize(n->stream));
    return IBIM_OK;
}

ibim_status ibim_wsnet_train(ibim_wsnet* n, int steps, int batch_nodes, double lr, double* last_loss)
{
    if (n == nullptr || steps < 1 || batch_nodes < 1 || !(lr > 0.0)) {
        set_error("need a net, steps >= 1, batch_nodes >= 1, lr > 0");
        return IBIM_ERR_ARG;
    }
    if (n->n_ex < 1) {
        set_error("no training examples");
        return IBIM_ERR_STATE;
    }
    const unsigned ctas = grad_ctas(n, batch_nodes);
    const double b1 = 0.9, b2 = 0.999;
    // Each launch may begin while the one before it ends (programmatic dependent
    // launch): the kernels wait for it themselves before they touch what it wrote.
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t grad_cfg = {}, sum_cfg = {};
    grad_cfg.gridDim = dim3(ctas);
    grad_cfg.blockDim = dim3(kTrainThreads);
    grad_cfg.dynamicSmemBytes = grad_smem();
    sum_cfg.gridDim = dim3((kWsParams + kSumParams - 1) / kSumParams);
    sum_cfg.blockDim = dim3(kSumParts * kSumParams);
    grad_cfg.stream = sum_cfg.stream = n->stream;
    grad_cfg.attrs = sum_cfg.attrs = &attr;
    grad_cfg.numAttrs = sum_cfg.numAttrs = 1;
    for (int s = 0; s < steps; ++s) {
        ++n->step;
        const uint64_t sd = n->seed * 0x9e3779b97f4a7c15ull + (uint64_t)n->step * 0xd1b54a32d192ed03ull;
        // (the first launch of a call follows whatever the stream holds in full)
        grad_cfg.numAttrs = s > 0 ? 1 : 0;
        IBIM_CUDA(cudaLaunchKernelEx(&grad_cfg, ws_grad_kernel, (const float*)n->d_feat, (const float*)n->d_tgt,
                                     (const float*)n->d_wt, n->n_ex, (int64_t)0, (int64_t)batch_nodes, 1, sd,
                                     1.0 / (double)batch_nodes, (const __nv_bfloat16*)n->d_wb, grad_parts(n),
                                     loss_parts(n)));
        const float c1 = (float)(1.0 - pow(b1, (double)n->step)), c2 = (float)(1.0 - pow(b2, (double)n->step));
        IBIM_CUDA(cudaLaunchKernelEx(&sum_cfg, ws_update_kernel, (const float*)grad_parts(n),
                                     (const double*)loss_parts(n), grad_nparts(ctas, batch_nodes), (int)ctas, 1, n->d_w, n->d_m, n->d_v, n->d_wb,
                                     (float)lr, (float)b1, (float)b2, c1, c2, n->d_g, n->d_loss));
    }
    if (last_loss) {
        IBIM_CUDA(cudaMemcpyAsync(last_loss, n->d_loss, sizeof(double), cudaMemcpyDeviceToHost, n->stream));
        IBIM_CUDA(cudaStreamSynchronize(n->stream));
    }
    return IBIM_OK;
}

ibim_status ibim_wsnet_predict(ibim_wsnet* n, ibim_ctx* c, const ibim_phys* p, double* d_p0)
{
    if (n == nullptr || c == nullptr || d_p0 == nullptr) {
        set_error("NULL argument");
        return IBIM_ERR_ARG;
    }
    IBIM_TRY(check_phys(p));
    if (c->Nc <= 0) {
        set_error("no charges set");
        return IBIM_ERR_STATE;
    }
    // order the net's own work (training) before the context's stream
    cudaEvent_t ev;
    IBIM_CUDA(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
    IBIM_CUDA(cudaEventRecord(ev, n->stream));
    IBIM_CUDA(cudaStreamWaitEvent(c->stream, ev, 0));
    IBIM_CUDA(cudaEventDestroy(ev));
    float* feat = nullptr;
    IBIM_TRY(ws_prepare(n, c, *p, &feat));
    const unsigned blocks = (unsigned)((c->N + kWsThreads - 1) / kWsThreads);
    const PairConsts k = make_consts(*p);
    ws_predict_kernel<<<blocks, kWsThreads, predict_smem(), c->stream>>>(feat, c->N, n->d_wb, n->d_scal, k.lambda1,
                                                                         k.lambda2, d_p0);
    count_launch(c);
    IBIM_CUDA(cudaGetLastError());
    IBIM_CUDA(cudaStreamSynchronize(c->stream));
    return IBIM_OK;
}

}  // extern "C"
