// Restarted GMRES for (Lambda + K W) p = g (Sec. 3.3), all vector work in FP64
// on the device.
//
// One Arnoldi step is a fixed sequence of launches that reads the step index
// k from a device-resident state, so two steps can be captured once into a CUDA
// graph and replayed for every pair of steps:
//   pack/pairs/fixup        w = A v_k                       (operator of the chosen precision)
//   gs_kernel<0>            dots h = V^T w                  (classical Gram-Schmidt,
//   gs_kernel<1>            w -= V h, dots again             twice: CGS2)
//   gs_kernel<2>            w -= V h, ||w||, then Givens: rotate column k of H, update
//                           the residual estimate, set `done` on convergence / end of cycle
//   scale                   v_{k+1} = w / ||w||
// Every launch first reads `done` and returns at once when it is set, so the
// host can replay a few steps ahead and poll the flag only occasionally.
//
// Outer loop: r = g - A_out x, one GMRES cycle on A_in d = r from d = 0,
// x += d.  Without certification A_out = A_in (plain restarted GMRES).  With
// certification A_out is an FP64-accurate operator: restarted GMRES with A_in
// runs to half the tolerance, then the residual is recomputed with A_out; if
// it misses the tolerance, the correction equation A e = r_out is solved the
// same way with A_in from e = 0 (its restart residuals r_out - A_in e) and
// x += e (iterative refinement).  The reported residual is the FP64-accurate
// one.
#include <math.h>
#include <string.h>

#include <atomic>
#include <vector>

#include "gmres_internal.cuh"

namespace ibim {

// ------------------------------------------------------------ vector kernels

// The finished cycle's outcome into pinned host memory, `done` last.
__device__ void publish_outcome(const GmState* __restrict__ st)
{
    volatile GmOutcome* out = st->out;
    if (out == nullptr) return;
    out->k = st->k;
    out->conv = st->conv;
    __threadfence_system();
    out->done = 1;
}

// Column k of H by one block: earlier rotations (one serial chain, from shared
// memory), new rotation, residual estimate |e_{k+1}|, end-of-cycle flags.
__device__ void givens_column(GmState* __restrict__ st, double hn)
{
    __shared__ double h[kMaxRestart + 1], cs[kMaxRestart], sn[kMaxRestart];
    const int k = st->k, m = st->m;
    __syncthreads();
    for (int j = threadIdx.x; j <= k; j += blockDim.x) h[j] = __ldcg(st->hcol + j);
    for (int j = threadIdx.x; j < k; j += blockDim.x) {
        cs[j] = st->cs[j];
        sn[j] = st->sn[j];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = h[0];
        for (int j = 0; j < k; ++j) {
            const double b = h[j + 1];
            h[j] = cs[j] * a + sn[j] * b;
            a = -sn[j] * a + cs[j] * b;
        }
        const double rr = hypot(a, hn);
        const double c = (rr > 0.0) ? a / rr : 1.0;
        const double s = (rr > 0.0) ? hn / rr : 0.0;
        h[k] = rr;
        st->hn = hn;
        st->cs[k] = c;
        st->sn[k] = s;
        const double e = st->e[k];
        st->e[k + 1] = -s * e;
        st->e[k] = c * e;
        const double resid = fabs(s * e);
        st->resid = resid;
        st->k = k + 1;
        const bool conv = resid <= st->target;
        if (conv) st->conv = 1;
        if (conv || k + 1 >= st->kmax || !(hn > 0.0)) {
            st->done = 1;
            publish_outcome(st);
        }
    }
    __syncthreads();
    for (int j = threadIdx.x; j <= k; j += blockDim.x) st->H[j * m + k] = h[j];
    if (threadIdx.x == 0) st->H[(k + 1) * m + k] = 0.0;
}

constexpr int kUpdateLoads = 4;  // element pairs a thread of the update has in flight
constexpr int kWarps = kVecThreads / 32;

// A pair of basis elements; volatile keeps a batch of these loads together
// ahead of the arithmetic (left to itself the compiler holds two or three).
__device__ __forceinline__ double2 load_pair(const double* p)
{
    double2 v;
    asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
    return v;
}

__device__ __forceinline__ double load_one(const double* p)
{
    double v;
    asm volatile("ld.global.nc.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
}

// One pass of the orthogonalisation of w = V_{k+1} against V_0..V_k.
//   PASS 0: h = V^T w;  1: w -= V h, then h2 = V^T w (hcol = h + h2);
//   2: w -= V h2, ||w||, then the Givens step (givens_column).
// A block owns C consecutive elements of every vector (vectors have even
// length, so they are read in pairs).  Update: one pair per thread; when C/2 is
// below the block size, the threads of a pair share the basis vectors.  Dots:
// a warp takes kDotGroup basis vectors over a slice of the block's elements and
// reduces their sums together, 9 adds instead of 40 (an FP64 add is as dear as
// a multiply: the FP64 pipe, 2 lanes per clock and SM, bounds these kernels
// once the vectors are long, L2 latency before that); while there are fewer
// groups than warps, the warps of a group share the elements.  The last block
// to finish a group adds the blocks' partials in a fixed order, so no reduction
// launch lies between the passes.  gridDim.y systems at once (batched solves).
// Measured per Arnoldi step (dots twice, updates twice, norm, Givens, scaling):
// 58 us at 75k elements and 32 vectors on average (117 us as nine launches with
// one block-wide reduction per dot product and one thread for the Givens
// column), 28 us at 10k elements (41 us), 56 us at 160k and 8 vectors (58 us),
// and 106 us for eight molecules of 27k to 46k elements together (456 us as nine
// launches per molecule).  Sixteen-byte loads in the dots (128 registers, half
// the warps) were 8 % faster for one system and 14 % slower for eight.
template <int PASS>
__global__ void __launch_bounds__(kVecThreads, 4) gs_kernel(GmSys one, const GmSys* __restrict__ many)
{
    const GmSys S = many != nullptr ? many[blockIdx.y] : one;
    GmState* st = S.st;
    if ((int)blockIdx.x >= S.nblk || st->done) return;
    constexpr int STRIDE = kMaxRestart + 1;
    extern __shared__ double2 sw[];  // the block's elements of w
    __shared__ double coef[kMaxRestart + 1 + kUpdateLoads];
    __shared__ double2 share[kVecThreads];
    __shared__ double dsum[kWarps][kMaxRestart + kDotGroup];
    __shared__ double red[kWarps];
    __shared__ int last;
    const int k = st->k, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t base = (int64_t)blockIdx.x * S.C, len = S.len;
    const int pairs = (int)(len - base < S.C ? len - base : S.C) / 2;
    const double* V = S.V + base;
    double2* w = reinterpret_cast<double2*>(S.V + (int64_t)(k + 1) * len + base);
    double nn = 0.0;
    if (PASS == 0) {
        for (int i = tid; i < pairs; i += kVecThreads) sw[i] = w[i];
    } else {
        for (int j = tid; j <= k + kUpdateLoads; j += kVecThreads) coef[j] = j <= k ? st->coef[j] : 0.0;
        __syncthreads();
        // nh threads per pair, thread h of a pair takes the vectors h, h + nh, ... in batches
        const int P = S.C / 2, nh = P < kVecThreads ? kVecThreads / P : 1;
        const int h = nh > 1 ? tid / P : 0, i0 = nh > 1 ? tid - h * P : tid;
        for (int i = i0; i < P; i += kVecThreads) {  // (one round when nh > 1)
            double sx = 0.0, sy = 0.0;
            if (h < nh && i < pairs)
                for (int j0 = h * kUpdateLoads; j0 <= k; j0 += nh * kUpdateLoads) {
                    double2 v[kUpdateLoads];  // past k: the last vector again, with weight 0
#pragma unroll
                    for (int q = 0; q < kUpdateLoads; ++q) v[q] = load_pair(V + (int64_t)min(j0 + q, k) * len + 2 * i);
#pragma unroll
                    for (int q = 0; q < kUpdateLoads; ++q) {
                        sx = fma(coef[j0 + q], v[q].x, sx);
                        sy = fma(coef[j0 + q], v[q].y, sy);
                    }
                }
            if (nh > 1) {
                share[tid] = make_double2(sx, sy);
                __syncthreads();
                if (h == 0)
                    for (int q = 1; q < nh; ++q) {
                        sx += share[q * P + i].x;
                        sy += share[q * P + i].y;
                    }
            }
            if (h == 0 && i < pairs) {
                double2 x = w[i];
                x.x -= sx;
                x.y -= sy;
                w[i] = x;
                if (PASS == 2) nn = fma(x.x, x.x, fma(x.y, x.y, nn));
                else sw[i] = x;
            }
        }
    }
    if (PASS < 2) {
        __syncthreads();
        const int ng = k / kDotGroup + 1;
        const int ns = ng >= kWarps ? 1 : ng > kWarps / 2 ? 1 : ng > kWarps / 4 ? 2 : ng > 1 ? 4 : 8;
        const int slice = warp % ns;
        const int i0 = pairs * slice / ns, i1 = pairs * (slice + 1) / ns;
        for (int g = warp / ns; g < ng; g += kWarps / ns) {
            double acc[kDotGroup];
            const double* row[kDotGroup];
#pragma unroll
            for (int q = 0; q < kDotGroup; ++q) {
                acc[q] = 0.0;
                row[q] = V + (int64_t)min(g * kDotGroup + q, k) * len;  // past k: repeats, not used
            }
            const double* ws = reinterpret_cast<const double*>(sw);
            for (int i = 2 * i0 + lane; i < 2 * i1; i += 32) {
                double v[kDotGroup];
#pragma unroll
                for (int q = 0; q < kDotGroup; ++q) v[q] = load_one(row[q] + i);
                const double x = ws[i];
#pragma unroll
                for (int q = 0; q < kDotGroup; ++q) acc[q] = fma(v[q], x, acc[q]);
            }
            // eight sums over 32 lanes: halve the values with the lanes, 4 + 2 + 1 adds, then two more
#pragma unroll
            for (int h = kDotGroup / 2, o = 16; h > 0; h >>= 1, o >>= 1) {
                const bool up = lane & o;
#pragma unroll
                for (int q = 0; q < kDotGroup / 2; ++q)
                    if (q < h) {
                        const double give = up ? acc[q] : acc[q + h], keep = up ? acc[q + h] : acc[q];
                        acc[q] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                    }
            }
            double v = acc[0];
            v += __shfl_xor_sync(0xffffffffu, v, 2);
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            if ((lane & 3) == 0) dsum[slice][g * kDotGroup + (lane >> 2)] = v;
        }
        __syncthreads();
        for (int g = warp; g < ng; g += kWarps) {
            const int j = g * kDotGroup + (lane >> 2);  // four lanes per dot product
            if ((lane & 3) == 0 && j <= k) {
                double v = dsum[0][j];
                for (int q = 1; q < ns; ++q) v += dsum[q][j];
                S.part[(int64_t)blockIdx.x * STRIDE + j] = v;
            }
            __threadfence();
            __syncwarp();
            int t = 0;
            if (lane == 0) t = atomicAdd(&st->dot_ticket[g], 1);
            if (__shfl_sync(0xffffffffu, t, 0) != S.nblk - 1) continue;
            __threadfence();
            double s = 0.0;
            if (j <= k) {
                for (int b = lane & 3; b < S.nblk; b += 64) {
                    double p[16];
#pragma unroll
                    for (int q = 0; q < 16; ++q)
                        p[q] = b + 4 * q < S.nblk ? __ldcg(S.part + (int64_t)(b + 4 * q) * STRIDE + j) : 0.0;
#pragma unroll
                    for (int q = 0; q < 16; ++q) s += p[q];
                }
            }
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            if ((lane & 3) == 0 && j <= k) {
                st->coef[j] = s;
                st->hcol[j] = PASS == 0 ? s : st->hcol[j] + s;
            }
            if (lane == 0) st->dot_ticket[g] = 0;
        }
        return;
    }
    for (int o = 16; o > 0; o >>= 1) nn += __shfl_down_sync(0xffffffffu, nn, o);
    if (lane == 0) red[warp] = nn;
    __syncthreads();
    if (tid == 0) {
        double s = 0.0;
        for (int q = 0; q < kWarps; ++q) s += red[q];
        S.part[(int64_t)blockIdx.x * STRIDE] = s;
        __threadfence();
        last = atomicAdd(&st->norm_ticket, 1) == S.nblk - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double s = 0.0;
    for (int b = tid; b < S.nblk; b += kVecThreads) s += __ldcg(S.part + (int64_t)b * STRIDE);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    __syncthreads();
    if (lane == 0) red[warp] = s;
    __syncthreads();
    s = 0.0;
    for (int q = 0; q < kWarps; ++q) s += red[q];
    if (tid == 0) st->norm_ticket = 0;
    givens_column(st, sqrt(s));
}

// v_{k+1} = w / ||w|| (after the Givens step: st->k is the new vector's index)
__global__ void __launch_bounds__(kVecThreads) scale_kernel(GmSys one, const GmSys* __restrict__ many)
{
    const GmSys S = many != nullptr ? many[blockIdx.y] : one;
    if ((int)blockIdx.x >= S.nblk || S.st->done) return;
    const double hn = S.st->hn;
    if (!(hn > 0.0)) return;
    const double inv = 1.0 / hn;
    const int64_t base = (int64_t)blockIdx.x * S.C;
    const int cnt = (int)(S.len - base < S.C ? S.len - base : S.C);
    double* w = S.V + (int64_t)S.st->k * S.len + base;
    for (int i = threadIdx.x; i < cnt; i += kVecThreads) w[i] *= inv;
}

// Back substitution H y = e (k x k upper triangular) by one block, column by
// column: the thread of row i forms y_i, the rows above subtract its column.
// The columns are staged in shared memory, so a step costs a division and a
// barrier (k = 64: 32 us; 177 us by one thread reading H from global memory).
__global__ void __launch_bounds__(kMaxRestart) trisolve_kernel(GmState* __restrict__ st)
{
    extern __shared__ double U[];  // column i at i (i + 1) / 2
    __shared__ double y;
    const int k = st->k, m = st->m, t = threadIdx.x;
#pragma unroll 8
    for (int i = 0; i < k; ++i)
        if (t <= i) U[i * (i + 1) / 2 + t] = st->H[t * m + i];
    double e = t < k ? st->e[t] : 0.0;
    __syncthreads();
    for (int i = k - 1; i >= 0; --i) {
        if (t == i) {
            y = e / U[i * (i + 1) / 2 + i];
            st->y[i] = y;
        }
        __syncthreads();
        if (t < i) e -= U[i * (i + 1) / 2 + t] * y;
        __syncthreads();
    }
}

constexpr size_t kTriSmem = sizeof(double) * kMaxRestart * (kMaxRestart + 1) / 2;

static ibim_status trisolve_launch(GmState* st, cudaStream_t stream)
{
    IBIM_CUDA(cudaFuncSetAttribute(trisolve_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTriSmem));
    trisolve_kernel<<<1, kMaxRestart, kTriSmem, stream>>>(st);
    return IBIM_OK;
}

// x += sum_{j<k} y_j V_j
__global__ void xupdate_kernel(double* __restrict__ x, const double* __restrict__ V, int64_t len,
                               const GmState* __restrict__ st)
{
    __shared__ double y[kMaxRestart];
    const int k = st->k;
    for (int j = threadIdx.x; j < k; j += blockDim.x) y[j] = st->y[j];
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x) {
        double s = x[i];
#pragma unroll 8
        for (int j = 0; j < k; ++j) s += y[j] * V[(int64_t)j * len + i];
        x[i] = s;
    }
}

// r = g - t and per-block partial of ||r||^2 (part[b * (m+1)])
__global__ void __launch_bounds__(kVecThreads)
    residual_kernel(const double* __restrict__ g, const double* __restrict__ t, double* __restrict__ r, int64_t len,
                    double* __restrict__ part)
{
    __shared__ double red[kVecThreads / 32];
    double nn = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * kVecThreads + threadIdx.x; i < len; i += (int64_t)gridDim.x * kVecThreads) {
        const double v = g[i] - (t ? t[i] : 0.0);
        r[i] = v;
        nn += v * v;
    }
    for (int o = 16; o > 0; o >>= 1) nn += __shfl_down_sync(0xffffffffu, nn, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = nn;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int q = 0; q < kVecThreads / 32; ++q) s += red[q];
        part[(int64_t)blockIdx.x * (kMaxRestart + 1)] = s;
    }
}

// New cycle: beta = sqrt(sum part), V_0 = r / beta, state reset with e = (beta, 0, ...).
__global__ void cycle_begin_reduce_kernel(const double* __restrict__ part, int nblk, GmState* __restrict__ st,
                                          double target, int kmax)
{
    __shared__ double red[256];
    double s = 0.0;
    for (int b = threadIdx.x; b < nblk; b += blockDim.x) s += part[(int64_t)b * (kMaxRestart + 1)];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double beta = sqrt(red[0]);
        st->hn = beta;  // carries beta to the scaling kernel
        st->k = 0;
        st->conv = (beta <= target) ? 1 : 0;
        st->done = st->conv;
        if (st->done) publish_outcome(st);
        st->kmax = kmax;
        st->target = target;
        st->resid = beta;
        for (int j = 0; j <= st->m; ++j) st->e[j] = 0.0;
        st->e[0] = beta;
    }
}

__global__ void cycle_begin_scale_kernel(const double* __restrict__ r, double* __restrict__ V0, int64_t len,
                                         const GmState* __restrict__ st)
{
    const double beta = st->hn;
    const double inv = (beta > 0.0) ? 1.0 / beta : 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x)
        V0[i] = r[i] * inv;
}

// x += y
__global__ void add_kernel(double* __restrict__ x, const double* __restrict__ y, int64_t len)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x)
        x[i] += y[i];
}

// x0 = Lambda^{-1} g (Sec. 3.3 initial guess with D = 0)
__global__ void lambda_inv_kernel(const double* __restrict__ g, double* __restrict__ x, int64_t N, double l1,
                                  double l2)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    x[i] = g[i] / l1;
    x[N + i] = g[N + i] / l2;
}

// ------------------------------------------------------------------ host side

void gmres_free(ibim_ctx* c)
{
    GmresWork* w = c->gm;
    if (w == nullptr) return;
    if (w->exec) cudaGraphExecDestroy(w->exec);
    if (w->ev) cudaEventDestroy(w->ev);
    for (cudaEvent_t e : w->poll)
        if (e) cudaEventDestroy(e);
    if (w->gs) cudaStreamDestroy(w->gs);
    cudaFree(w->V);
    cudaFree(w->x);
    cudaFree(w->r);
    cudaFree(w->t);
    cudaFree(w->g);
    cudaFree(w->xb);
    cudaFree(w->gin);
    cudaFree(w->part);
    cudaFree(w->st);
    cudaFreeHost(w->h_st);
    delete w;
    c->gm = nullptr;
}

ibim_status gm_alloc(ibim_ctx* c, int m)
{
    const int64_t len = 2 * c->N;
    if (c->gm && c->gm->m >= m && c->gm->len == len) return IBIM_OK;
    gmres_free(c);
    GmresWork* w = new GmresWork();
    c->gm = w;
    w->m = m;
    w->len = len;
    w->nblk = (int)std::min<int64_t>(2 * c->num_sms, (len + kVecThreads - 1) / kVecThreads);
    if (w->nblk < 1) w->nblk = 1;
    IBIM_CUDA(cudaMalloc((void**)&w->V, sizeof(double) * (size_t)(m + 1) * len));
    IBIM_CUDA(cudaMalloc((void**)&w->x, sizeof(double) * len));
    IBIM_CUDA(cudaMalloc((void**)&w->r, sizeof(double) * len));
    IBIM_CUDA(cudaMalloc((void**)&w->t, sizeof(double) * len));
    IBIM_CUDA(cudaMalloc((void**)&w->g, sizeof(double) * len));
    IBIM_CUDA(cudaMalloc((void**)&w->xb, sizeof(double) * len));
    IBIM_CUDA(cudaMalloc((void**)&w->gin, sizeof(double) * len));
    // blocks of C = 128, 256, ... elements: at most 320 of them (two per SM), so
    // that the last warp of a group adds few partials, until a block's elements
    // of w no longer fit shared memory (2.6 million nodes)
    w->sys.len = len;
    w->sys.C = 128;
    while (w->sys.C < 16384 && len > 320 * (int64_t)w->sys.C) w->sys.C *= 2;
    w->sys.nblk = (int)((len + w->sys.C - 1) / w->sys.C);
    IBIM_CUDA(cudaMalloc((void**)&w->part,
                         sizeof(double) * (size_t)std::max(w->nblk, w->sys.nblk) * (kMaxRestart + 1)));
    IBIM_CUDA(cudaMalloc((void**)&w->st, sizeof(GmState)));
    w->sys.V = w->V;
    w->sys.st = w->st;
    w->sys.part = w->part;
    IBIM_CUDA(cudaMallocHost((void**)&w->h_st, sizeof(GmState) + sizeof(GmOutcome)));
    w->h_out = reinterpret_cast<GmOutcome*>(w->h_st + 1);
    IBIM_CUDA(cudaStreamCreateWithFlags(&w->gs, cudaStreamNonBlocking));
    IBIM_CUDA(cudaEventCreateWithFlags(&w->ev, cudaEventDisableTiming));
    for (cudaEvent_t& e : w->poll) IBIM_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    return IBIM_OK;
}

static ibim_status ortho_launch(const GmSys& one, const GmSys* many, int nsys, int nblk, int C, cudaStream_t stream)
{
    const dim3 grid((unsigned)nblk, (unsigned)nsys);
    const size_t smem = sizeof(double) * C;
    if (smem > 40 * 1024) {
        IBIM_CUDA(cudaFuncSetAttribute(gs_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        IBIM_CUDA(cudaFuncSetAttribute(gs_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    }
    gs_kernel<0><<<grid, kVecThreads, smem, stream>>>(one, many);
    gs_kernel<1><<<grid, kVecThreads, smem, stream>>>(one, many);
    gs_kernel<2><<<grid, kVecThreads, 0, stream>>>(one, many);
    scale_kernel<<<grid, kVecThreads, 0, stream>>>(one, many);
    IBIM_CUDA(cudaGetLastError());
    return IBIM_OK;
}

ibim_status gm_ortho(ibim_ctx* c)
{
    const GmSys& S = c->gm->sys;
    IBIM_TRY(ortho_launch(S, nullptr, 1, S.nblk, S.C, c->stream));
    count_launch(c, kOrthoLaunches);
    return IBIM_OK;
}

ibim_status gm_ortho_batch(const GmSys* d_sys, int nsys, int max_nblk, int max_C, cudaStream_t stream)
{
    return ortho_launch(GmSys{}, d_sys, nsys, max_nblk, max_C, stream);
}

// One Arnoldi step (see the file comment), all launches on c->stream.
static ibim_status arnoldi_step(ibim_ctx* c, const PairConsts& k, int precision)
{
    GmresWork* w = c->gm;
    const int64_t len = w->len;
    const int* skip = &w->st->done;
    VecRef in{w->V, &w->st->k, len, 0};
    OutRef out{w->V, &w->st->k, len, 1};
    IBIM_TRY(apply_operator(c, k, precision, in, out, skip));
    return gm_ortho(c);
}

ibim_status gm_cycle_begin(ibim_ctx* c, bool x_zero, double target, int kmax)
{
    GmresWork* w = c->gm;
    const int64_t len = w->len;
    residual_kernel<<<w->nblk, kVecThreads, 0, c->stream>>>(w->g, x_zero ? nullptr : w->t, w->r, len, w->part);
    cycle_begin_reduce_kernel<<<1, 256, 0, c->stream>>>(w->part, w->nblk, w->st, target, kmax);
    cycle_begin_scale_kernel<<<w->nblk, kVecThreads, 0, c->stream>>>(w->r, w->V, len, w->st);
    count_launch(c, 3);
    IBIM_CUDA(cudaGetLastError());
    return IBIM_OK;
}

ibim_status gm_cycle_end(ibim_ctx* c)
{
    GmresWork* w = c->gm;
    IBIM_TRY(trisolve_launch(w->st, c->stream));
    xupdate_kernel<<<w->nblk, kVecThreads, 0, c->stream>>>(w->x, w->V, w->len, w->st);
    count_launch(c, 2);
    IBIM_CUDA(cudaGetLastError());
    return IBIM_OK;
}

ibim_status gm_fetch_state(ibim_ctx* c)
{
    IBIM_CUDA(cudaMemcpyAsync(c->gm->h_st, c->gm->st, 64, cudaMemcpyDeviceToHost, c->stream));
    return IBIM_OK;
}

ibim_status gm_init(ibim_ctx* c, const ibim_phys& p, int m, double* gnorm)
{
    GmresWork* w = c->gm;
    GmState init;
    memset(&init, 0, sizeof(init));
    init.m = m;
    IBIM_CUDA(cudaMemcpyAsync(w->st, &init, sizeof(GmState), cudaMemcpyHostToDevice, c->stream));
    IBIM_TRY(rhs_launch(c, p.eps_in, w->g));
    residual_kernel<<<w->nblk, kVecThreads, 0, c->stream>>>(w->g, nullptr, w->r, w->len, w->part);
    cycle_begin_reduce_kernel<<<1, 256, 0, c->stream>>>(w->part, w->nblk, w->st, 0.0, 0);
    count_launch(c, 2);
    IBIM_CUDA(cudaMemsetAsync(w->x, 0, sizeof(double) * w->len, c->stream));
    IBIM_CUDA(cudaMemcpyAsync(w->h_st, w->st, 64, cudaMemcpyDeviceToHost, c->stream));
    IBIM_CUDA(cudaStreamSynchronize(c->stream));
    *gnorm = w->h_st->resid;
    return IBIM_OK;
}

// r = rhs - A x with the operator of precision `prec` (or r = rhs when x is
// known to be zero); starts a cycle on r.
static ibim_status begin_cycle(ibim_ctx* c, const PairConsts& k, int prec, const double* rhs, bool x_zero,
                               double target, int kmax, double* beta_host)
{
    GmresWork* w = c->gm;
    const int64_t len = w->len;
    if (!x_zero)
        IBIM_TRY(apply_operator(c, k, prec, VecRef{w->x, nullptr, 0, 0}, OutRef{w->t, nullptr, 0, 0}, nullptr));
    residual_kernel<<<w->nblk, kVecThreads, 0, c->stream>>>(rhs, x_zero ? nullptr : w->t, w->r, len, w->part);
    cycle_begin_reduce_kernel<<<1, 256, 0, c->stream>>>(w->part, w->nblk, w->st, target, kmax);
    cycle_begin_scale_kernel<<<w->nblk, kVecThreads, 0, c->stream>>>(w->r, w->V, len, w->st);
    count_launch(c, 3);
    IBIM_CUDA(cudaGetLastError());
    IBIM_CUDA(cudaMemcpyAsync(w->h_st, w->st, 64, cudaMemcpyDeviceToHost, c->stream));
    IBIM_CUDA(cudaStreamSynchronize(c->stream));
    *beta_host = w->h_st->resid;
    return IBIM_OK;
}

static ibim_status capture_step(ibim_ctx* c, const PairConsts& k, int precision)
{
    GmresWork* w = c->gm;
    // Every workspace the step (or a later operator application of either
    // precision) touches is sized for both precisions before capture, so that
    // no later call reallocates a buffer the graph holds a pointer to.
    IBIM_TRY(ensure_operator_workspaces(c));
    if (precision == IBIM_F64) IBIM_TRY(f64_prepare(c));
    if (w->graph_valid && w->graph_prec == precision && memcmp(&w->graph_k, &k, sizeof(k)) == 0 &&
        w->graph_generation == c->ws_generation && w->graph_variant == c->f32_variant && w->graph_bps == c->f32_bps &&
        w->graph_ff == c->ff_symmetric)
        return IBIM_OK;
    if (w->exec) {
        cudaGraphExecDestroy(w->exec);
        w->exec = nullptr;
    }
    w->graph_valid = false;
    cudaGraph_t graph = nullptr;
    IBIM_CUDA(cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal));
    const int64_t launches_before = c->timing.total_launches;
    ibim_status s = IBIM_OK;
    for (int q = 0; q < kStepsPerGraph && s == IBIM_OK; ++q) s = arnoldi_step(c, k, precision);
    c->timing.total_launches = launches_before;  // capture does not launch
    cudaError_t e = cudaStreamEndCapture(c->stream, &graph);
    if (s != IBIM_OK) {
        if (graph) cudaGraphDestroy(graph);
        return s;
    }
    if (e != cudaSuccess) return cuda_fail(e, "capture of the Arnoldi step", __FILE__, __LINE__);
    e = cudaGraphInstantiate(&w->exec, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) return cuda_fail(e, "graph instantiate", __FILE__, __LINE__);
    w->graph_valid = true;
    w->graph_prec = precision;
    w->graph_k = k;
    w->graph_generation = c->ws_generation;
    w->graph_variant = c->f32_variant;
    w->graph_bps = c->f32_bps;
    w->graph_ff = c->ff_symmetric;
    return IBIM_OK;
}

// Runs steps until the device sets `done`; returns the steps taken.  Steps go
// out in pairs (one captured graph), and the step that sets `done` writes the
// outcome to pinned host memory itself, so nothing but an event lies between two
// pairs.  Captured steps: the next pair is in the stream before the host waits
// for a pair, so the device does not idle over the wait and the launch; the pair
// launched past the end finds the solver done and returns at once.  (With a
// copy of the state behind each pair, two graphs and the wait, 40 us a pair went
// by: certified solve of 5,000 nodes, 20 steps of 70 us, 2.03 -> 1.91 ms.)  Steps timed
// kernel by kernel are waited for pair by pair.
static ibim_status run_cycle(ibim_ctx* c, const PairConsts& k, int precision, bool use_graph, int* steps,
                             int* conv)
{
    GmresWork* w = c->gm;
    volatile GmOutcome* out = w->h_out;
    out->done = 0;  // nothing in flight writes it: steps past the end return first
    auto launch_pair = [&](int slot) -> ibim_status {
        if (use_graph) {
            if (!w->graph_valid || w->graph_generation != c->ws_generation) {
                set_error("captured GMRES step is stale (workspace reallocated)");
                return IBIM_ERR_STATE;
            }
            IBIM_CUDA(cudaGraphLaunch(w->exec, c->stream));
            count_launch(c, kStepsPerGraph * (3 + kOrthoLaunches));  // kernels in the captured steps
        } else {
            for (int q = 0; q < kStepsPerGraph; ++q) IBIM_TRY(arnoldi_step(c, k, precision));
        }
        IBIM_CUDA(cudaEventRecord(w->poll[slot], c->stream));
        return IBIM_OK;
    };
    if (use_graph) IBIM_TRY(launch_pair(0));
    for (int seen = 0;; ++seen) {
        IBIM_TRY(launch_pair(use_graph ? (seen + 1) & 1 : seen & 1));
        IBIM_CUDA(cudaEventSynchronize(w->poll[seen & 1]));
        if (out->done) break;
        if (kStepsPerGraph * (seen + 1) > kMaxRestart + 4) {
            set_error("GMRES cycle did not terminate");
            return IBIM_ERR_CUDA;
        }
    }
    std::atomic_thread_fence(std::memory_order_acquire);  // a later pair than the awaited one may have set it
    *steps = out->k;
    *conv = out->conv;
    return IBIM_OK;
}

ibim_status gmres_solve(ibim_ctx* c, const ibim_phys& p, const ibim_solve_opts& o, double* d_p,
                        ibim_solve_info* info)
{
    const int m = std::min(o.restart, kMaxRestart);
    IBIM_TRY(gm_alloc(c, m));
    GmresWork* w = c->gm;
    const int64_t len = w->len, N = c->N;
    const PairConsts k = make_consts(p);
    const int prec_in = o.precision;
    // The symmetric FP32 kernels add their reverse sums in a varying order, so
    // two applications to the same vector differ by about 1e-8 of |A p|; a
    // restart residual then cannot settle below that.  Uncertified solves asked
    // for a tighter tolerance run the one-directional kernel instead (restored
    // on exit).  Certified solves keep the symmetric kernel: once the first
    // check fails, the inner solves work on the correction equation, whose
    // right-hand side is the current residual, so the noise scales with it.
    struct KeepVariant {
        ibim_ctx* c;
        int v, b;
        ~KeepVariant()
        {
            c->f32_variant = v;
            c->f32_bps = b;
        }
    } keep_variant{c, c->f32_variant, c->f32_bps};
    if (prec_in == IBIM_F32C && o.certify == 0 && o.tol < kSymTolFloor && f32_variant_symmetric(c->f32_variant)) {
        c->f32_variant = f32_deterministic_variant();
        c->f32_bps = 0;
    }
    // certification operator: 1 = float-float pair sums (FP64-accurate on the
    // FP32 pipe), 2 = plain FP64 pair sums
    const int prec_out = o.certify == 2 ? IBIM_F64 : (o.certify ? IBIM_FF : o.precision);

    // Work on the solver's own stream (graph capture needs a non-legacy
    // stream), ordered after everything already queued on the caller's.
    cudaStream_t user = c->stream;
    IBIM_CUDA(cudaEventRecord(w->ev, user));
    IBIM_CUDA(cudaStreamWaitEvent(w->gs, w->ev, 0));
    c->stream = w->gs;
    struct Restore {
        ibim_ctx* c;
        cudaStream_t user;
        ~Restore()
        {
            cudaEventRecord(c->gm->ev, c->stream);
            cudaStreamWaitEvent(user, c->gm->ev, 0);
            c->stream = user;
        }
    } restore{c, user};

    GmState init;
    memset(&init, 0, sizeof(init));
    init.m = m;
    init.out = w->h_out;
    IBIM_CUDA(cudaMemcpyAsync(w->st, &init, sizeof(GmState), cudaMemcpyHostToDevice, c->stream));

    IBIM_TRY(rhs_launch(c, p.eps_in, w->g));
    // ||g||
    residual_kernel<<<w->nblk, kVecThreads, 0, c->stream>>>(w->g, nullptr, w->r, len, w->part);
    cycle_begin_reduce_kernel<<<1, 256, 0, c->stream>>>(w->part, w->nblk, w->st, 0.0, 0);
    count_launch(c, 2);
    IBIM_CUDA(cudaMemcpyAsync(w->h_st, w->st, 64, cudaMemcpyDeviceToHost, c->stream));
    IBIM_CUDA(cudaStreamSynchronize(c->stream));
    const double gnorm = w->h_st->resid;

    bool x_zero = false;
    if (o.start == 0) {
        IBIM_CUDA(cudaMemsetAsync(w->x, 0, sizeof(double) * len, c->stream));
        x_zero = true;
    } else if (o.start == 1) {
        lambda_inv_kernel<<<(unsigned)((N + 255) / 256), 256, 0, c->stream>>>(w->g, w->x, N, k.lambda1, k.lambda2);
        count_launch(c);
    } else {
        IBIM_CUDA(cudaMemcpyAsync(w->x, d_p, sizeof(double) * len, cudaMemcpyDeviceToDevice, c->stream));
    }

    const bool use_graph = !c->timing.enabled;
    const double target_abs = o.tol * gnorm;
    const double inner_target = o.certify ? 0.5 * target_abs : target_abs;
    int iters = 0, cycles = 0;
    double beta = 0.0;
    bool converged = false;
    if (gnorm == 0.0) {
        IBIM_CUDA(cudaMemsetAsync(w->x, 0, sizeof(double) * len, c->stream));
        converged = true;
    }
    // Restart residuals use the iteration's operator; with certification the
    // residual is recomputed with the FP64-accurate operator once the iteration's
    // residual meets the inner target (or the iteration budget is spent).  A
    // failed check starts a solve of the correction equation on that residual:
    // xb keeps the iterate, x the correction from zero, gin the residual, and
    // restarts compute gin - A_in x until the next check adds xb back.  (Restart
    // residuals g - A_in x of the whole system would pull the iterate back to
    // A_in's own solution, which misses the tolerance whenever A_in differs
    // from A_out by more than the inner target, e.g. a treecode operator.)
    // A cycle that meets the inner target by its own estimate is followed by
    // the check at once: a restart residual with A_in could only confirm the
    // estimate (then the check follows) or show A_in's accuracy floor (the
    // FP32 operator is linear only to about 1e-8 of |A x|; further cycles
    // could not go lower, so the check follows as well).
    bool check = false, refining = false;
    while (!converged) {
        const int kmax = std::min(m, o.maxit - iters);
        const int prec_r = (check || kmax <= 0) ? prec_out : prec_in;
        if (prec_r == prec_out && refining) {
            add_kernel<<<w->nblk, kVecThreads, 0, c->stream>>>(w->x, w->xb, len);
            count_launch(c);
            refining = false;
        }
        if (!x_zero) {
            if (prec_r == IBIM_F32C || prec_r == IBIM_F32T) info->matvecs_f32 += 1;
            else info->matvecs_f64 += 1;
        }
        IBIM_TRY(begin_cycle(c, k, prec_r, refining ? w->gin : w->g, x_zero, inner_target, std::max(kmax, 0),
                             &beta));
        x_zero = false;
        if (prec_r == prec_out && beta <= target_abs) {
            converged = true;
            break;
        }
        if (prec_r != prec_out && beta <= inner_target) {
            check = true;
            continue;
        }
        check = false;
        if (kmax <= 0) break;
        if (prec_r != prec_in) {  // failed check: the cycle below starts on r = g - A_out x
            IBIM_CUDA(cudaMemcpyAsync(w->xb, w->x, sizeof(double) * len, cudaMemcpyDeviceToDevice, c->stream));
            IBIM_CUDA(cudaMemcpyAsync(w->gin, w->r, sizeof(double) * len, cudaMemcpyDeviceToDevice, c->stream));
            IBIM_CUDA(cudaMemsetAsync(w->x, 0, sizeof(double) * len, c->stream));
            refining = true;
        }
        if (use_graph) IBIM_TRY(capture_step(c, k, prec_in));
        int steps = 0, conv = 0;
        IBIM_TRY(run_cycle(c, k, prec_in, use_graph, &steps, &conv));
        iters += steps;
        ++cycles;
        check = prec_out != prec_in && conv != 0;
        info->matvecs_f32 += (prec_in == IBIM_F32C || prec_in == IBIM_F32T) ? steps : 0;
        info->matvecs_f64 += (prec_in == IBIM_F64 || prec_in == IBIM_FF) ? steps : 0;
        if (steps > 0) {
            IBIM_TRY(trisolve_launch(w->st, c->stream));
            xupdate_kernel<<<w->nblk, kVecThreads, 0, c->stream>>>(w->x, w->V, len, w->st);
            count_launch(c, 2);
            IBIM_CUDA(cudaGetLastError());
        }
    }
    info->iters = iters;
    info->cycles = cycles;
    info->converged = converged ? 1 : 0;
    info->relres = (gnorm > 0.0) ? beta / gnorm : 0.0;
    IBIM_CUDA(cudaMemcpyAsync(d_p, w->x, sizeof(double) * len, cudaMemcpyDeviceToDevice, c->stream));

    double gpol = 0.0, area = 0.0;
    IBIM_TRY(energy_launch(c, p, w->x, nullptr, &gpol, &area));
    info->gpol = gpol;
    info->gpol_kcal = gpol * kKcalPerE2A;
    info->area = area;
    return converged ? IBIM_OK : IBIM_ERR_NOT_CONVERGED;
}

}  // namespace ibim
