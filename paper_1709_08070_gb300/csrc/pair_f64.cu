// Plain FP64 pair sums of the IBIM operator (Sec. 2.2 discrete system,
// Sec. 2.2.1 regularisation), sm_103a.
//
// The kernels (times 4 pi), with g = 1 - A = (1 - E) - E x and 3 - B = 3 g - E x^2,
// x = kappa rho:
//   K11 = s_y (1 - th1 A)/rho^3, K12 = (1 - E)/rho,
//   K21 = [g c - (3 - B) s_x s_y/rho^2]/rho^3, K22 = -s_x (1 - th2 A)/rho^3.
//
// Bound by the FP64 pipe (2 lanes per clock and SM, 1/64 of the FP32 rate), so
// the one thing that counts is FP64 instructions per interaction.  Each
// unordered pair is evaluated once for both directions (r' = -r, s_x' = -s_y,
// s_y' = -s_x, c' = c), 60 instructions per pair: the symmetric combination
// [g c - (3 - B) s_x s_y/rho^2]/rho^3 serves both directions, 1/rho is a
// hardware estimate with one third-order step, and E comes from a table
// (Tang, ACM TOMS 15, 1989).  Pairs of 32-node chunks whose bounding spheres
// are apart by more than the tube reaches skip the tube tests.
//
// Work: the chunks are grouped into n_b blocks; an item is one unordered block
// pair (I, J), taken by one warp.  A chunk pair is 32 steps: the lanes hold 32
// targets and walk the 32 sources in a staggered order, and the two reverse
// sums of a source travel with it from lane to lane, so that after 32 steps
// lane l holds source l's.  A chunk pair takes the FP64 pipe 17 us, so loads,
// shuffles and partial sums in global memory cost nothing beside it, warps need
// no barriers, and items are small enough to balance themselves.
// Every item owns its partial sums (forward of I, reverse of J) and the fixup
// adds them in a fixed order: results repeat bit for bit, whichever warp took
// which item.
//
// Measured: 20,011-node cloud 22.6 ms (55.1 ms with one target per thread, all
// ordered pairs, the library's exp and rsqrt: 81 instructions per interaction).
#include "ibim_internal.cuh"
#include "math64.cuh"

namespace ibim {

constexpr int kF64Chunk = 32;
constexpr int kF64Head = 2;  // doubles before the partial slots: the item counter
// Blocks per side: 160 give about 12,900 items, ten per resident warp, with
// partial sums of 160 x 16 bytes per node.
constexpr int64_t kF64Blocks = 160;

struct F64Consts {
    double th1, th2, om1, om2, kappa, tau2, four_tau2, k12t;
    float far_dist;
    int rule0;
};

struct F64Plan {
    int64_t n_chunks, m, n_b, items;  // m chunks per block
};

__host__ __device__ __forceinline__ F64Plan f64_plan(int64_t N)
{
    F64Plan p;
    p.n_chunks = (N + kF64Chunk - 1) / kF64Chunk;
    p.m = (p.n_chunks + kF64Blocks - 1) / kF64Blocks;
    p.n_b = (p.n_chunks + p.m - 1) / p.m;
    p.items = p.n_b * (p.n_b + 1) / 2;
    return p;
}

// Items q = d n_b + I, J = I + d modulo n_b, d = 0 .. n_b/2: every unordered
// block pair once (for even n_b the last d has n_b/2 items).  Slot of item q:
// forward sums of block I (two vectors of S nodes), then reverse sums of J.

// Payload of node j: (x, y), (z, a), (nx, ny), (nz, b), a = w psi, b = w psin,
// stored per chunk component by component.
__host__ __device__ __forceinline__ int64_t f64_off(int64_t j, int comp)
{
    return (j / kF64Chunk) * (4 * kF64Chunk) + comp * kF64Chunk + (j % kF64Chunk);
}

struct F64Node {
    double x, y, z, a, nx, ny, nz, b;
};

__device__ __forceinline__ F64Node f64_load(const double2* __restrict__ src, int64_t chunk, int lane)
{
    const double2* p = src + chunk * (4 * kF64Chunk) + lane;
    const double2 v0 = p[0], v1 = p[kF64Chunk], v2 = p[2 * kF64Chunk], v3 = p[3 * kF64Chunk];
    return F64Node{v0.x, v0.y, v1.x, v1.y, v2.x, v2.y, v3.x, v3.y};
}

// One unordered pair: forward (target T <- source s) into f1, f2, reverse
// (target s <- source T, weights ra, rb) into v1, v2.
template <bool NEAR>
__device__ __forceinline__ void f64_pair(const F64Node& T, double ra, double rb, const F64Node& e, const F64Consts& k,
                                         const double* __restrict__ tab, double& f1, double& f2, double& v1,
                                         double& v2)
{
    const double r0 = T.x - e.x, r1 = T.y - e.y, r2 = T.z - e.z;
    const double rr = r0 * r0 + r1 * r1 + r2 * r2;
    const double sx = r0 * T.nx + r1 * T.ny + r2 * T.nz;
    const double sy = r0 * e.nx + r1 * e.ny + r2 * e.nz;
    const double cc = T.nx * e.nx + T.ny * e.ny + T.nz * e.nz;
    bool tf = false, tr = false;
    double q = rr;
    if (NEAR) {
        const double pf = rr - sx * sx, pr = rr - sy * sy;
        tf = pf < k.tau2 && rr < k.four_tau2;
        tr = pr < k.tau2 && rr < k.four_tau2;
        if (tf && tr) q = 1.0;  // coincident nodes are always here
    }
    const double inv = rsqrt64(q);
    const double x = k.kappa * (q * inv);
    const double E = exp_neg64(x, tab);
    const double f = 1.0 - E;
    const double Ex = E * x;
    const double g = f - Ex;
    const double hb = fma(3.0, g, -(Ex * x));
    const double inv2 = inv * inv, inv3 = inv2 * inv;
    const double P1 = fma(k.th1, g, k.om1) * inv3;
    const double P2 = fma(k.th2, g, k.om2) * inv3;
    const double W = fma(-(hb * inv2), sx * sy, g * cc) * inv3;
    const double K12 = f * inv;
    if (NEAR) {  // a regularised direction keeps only K12's tube value
        const double aj = tf ? 0.0 : e.a, bj = tf ? 0.0 : e.b, kf = tf ? k.k12t : K12;
        f1 = fma(-kf, e.b, fma(P1 * sy, aj, f1));
        f2 = fma(P2 * sx, bj, fma(W, aj, f2));
        const double ai = tr ? 0.0 : ra, bi = tr ? 0.0 : rb, kr = tr ? k.k12t : K12;
        v1 = fma(-kr, rb, fma(-(P1 * sx), ai, v1));
        v2 = fma(-(P2 * sy), bi, fma(W, ai, v2));
    } else {
        f1 = fma(-K12, e.b, fma(P1 * sy, e.a, f1));
        f2 = fma(P2 * sx, e.b, fma(W, e.a, f2));
        v1 = fma(-K12, rb, fma(-(P1 * sx), ra, v1));
        v2 = fma(-(P2 * sy), rb, fma(W, ra, v2));
    }
}

template <bool NEAR>
__device__ __forceinline__ void f64_chunk_pair(const F64Node& T, double ra, double rb, const double2* __restrict__ src,
                                               int64_t cs, int lane, const F64Consts& k,
                                               const double* __restrict__ tab, double& f1, double& f2, double& v1,
                                               double& v2)
{
    const int next = (lane + 1) & 31;
    F64Node e = f64_load(src, cs, lane);
#pragma unroll 1
    for (int step = 0; step < kF64Chunk; ++step) {
        const F64Node cur = e;
        e = f64_load(src, cs, (lane + step + 1) & 31);  // the next step's source
        f64_pair<NEAR>(T, ra, rb, cur, k, tab, f1, f2, v1, v2);
        v1 = __shfl_sync(0xffffffffu, v1, next);
        v2 = __shfl_sync(0xffffffffu, v2, next);
    }
}

__global__ void __launch_bounds__(128, 4)
    pair_f64_kernel(const double2* __restrict__ src, const float4* __restrict__ frames, F64Plan p, F64Consts k,
                    const double* __restrict__ exptab, double* __restrict__ part, const int* __restrict__ skip)
{
    if (skip != nullptr && *skip) return;
    __shared__ double tab[kExpTab];
    for (int q = threadIdx.x; q < kExpTab; q += blockDim.x) tab[q] = exptab[q];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int64_t S = p.m * kF64Chunk;
    unsigned long long* ctr = reinterpret_cast<unsigned long long*>(part);

    int64_t q = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    while (q < p.items) {
        const int64_t d = q / p.n_b, I = q - d * p.n_b, J = (I + d) % p.n_b;
        const int64_t t0 = I * p.m, t1 = min(t0 + p.m, p.n_chunks);
        const int64_t c0 = J * p.m, c1 = min(c0 + p.m, p.n_chunks);
        double* fwd = part + kF64Head + q * (4 * S) + lane;
        double* rev = fwd + 2 * S;
        for (int64_t cs = c0; cs < c1; ++cs) {
            const float4 mh = frames[2 * cs], ml = frames[2 * cs + 1];
            double v1 = 0.0, v2 = 0.0;
            const int64_t te = d == 0 ? cs + 1 : t1;  // within a block: targets up to the source's own chunk
            for (int64_t ct = t0; ct < te; ++ct) {
                const F64Node T = f64_load(src, ct, lane);
                const float4 th = frames[2 * ct], tl = frames[2 * ct + 1];
                const float dx = (th.x - mh.x) + (tl.x - ml.x);
                const float dy = (th.y - mh.y) + (tl.y - ml.y);
                const float dz = (th.z - mh.z) + (tl.z - ml.z);
                const float lim = k.far_dist + th.w + mh.w;
                const bool far = k.rule0 != 0 && fmaf(dx, dx, fmaf(dy, dy, dz * dz)) >= lim * lim;
                // a chunk with itself holds both orders of its pairs (and the self pairs) in the forward direction
                const double ra = ct == cs && d == 0 ? 0.0 : T.a, rb = ct == cs && d == 0 ? 0.0 : T.b;
                double f1 = 0.0, f2 = 0.0;
                if (far)
                    f64_chunk_pair<false>(T, ra, rb, src, cs, lane, k, tab, f1, f2, v1, v2);
                else
                    f64_chunk_pair<true>(T, ra, rb, src, cs, lane, k, tab, f1, f2, v1, v2);
                double* o = fwd + (ct - t0) * kF64Chunk;
                const bool first = d == 0 ? ct == cs : cs == c0;
                o[0] = first ? f1 : o[0] + f1;
                o[S] = first ? f2 : o[S] + f2;
            }
            rev[(cs - c0) * kF64Chunk] = v1;
            rev[S + (cs - c0) * kF64Chunk] = v2;
        }
        if (lane == 0) q = warps + (int64_t)atomicAdd(ctr, 1ull);
        q = __shfl_sync(0xffffffffu, q, 0);
    }
}

// Payload of the chunk-padded node range (past N: the last node's position and
// normal with zero weights) and the cleared item counter.
__global__ void pack_f64_kernel(const double* __restrict__ geo, VecRef in, int64_t N, int64_t n_pad,
                                double2* __restrict__ src, double* __restrict__ part, const int* __restrict__ skip)
{
    if (skip != nullptr && *skip) return;
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j == 0) *reinterpret_cast<unsigned long long*>(part) = 0ull;
    if (j >= n_pad) return;
    const double* p = in.base + (in.kidx ? (int64_t)(*in.kidx + in.koff) * in.stride : 0);
    const int64_t i = j < N ? j : N - 1;
    const double w = geo[6 * N + i];
    src[f64_off(j, 0)] = make_double2(geo[i], geo[N + i]);
    src[f64_off(j, 1)] = make_double2(geo[2 * N + i], j < N ? w * p[j] : 0.0);
    src[f64_off(j, 2)] = make_double2(geo[3 * N + i], geo[4 * N + i]);
    src[f64_off(j, 3)] = make_double2(geo[5 * N + i], j < N ? w * p[N + j] : 0.0);
}

// y = Lambda p + (1/(4 pi)) (the node's forward and reverse partials), kF64Parts
// threads per node over fixed shares of d, the shares added in a fixed order.
constexpr int kF64Parts = 8, kF64Nodes = 32;
__global__ void __launch_bounds__(kF64Parts * kF64Nodes)
    fixup_f64_kernel(const double* __restrict__ part, F64Plan p, int64_t N, double lambda1, double lambda2, VecRef in,
                     OutRef out, const int* __restrict__ skip)
{
    if (skip != nullptr && *skip) return;
    __shared__ double sh[2][kF64Parts][kF64Nodes];
    const int tl = threadIdx.x % kF64Nodes, pr = threadIdx.x / kF64Nodes;
    const int64_t i = (int64_t)blockIdx.x * kF64Nodes + tl;
    const int64_t S = p.m * kF64Chunk;
    double a1 = 0.0, a2 = 0.0;
    if (i < N) {
        const int64_t B = i / S, l = i - B * S, nd = p.n_b / 2 + 1;
        const double* base = part + kF64Head + l;
        for (int64_t d = nd * pr / kF64Parts; d < nd * (pr + 1) / kF64Parts; ++d) {
            const int64_t qf = d * p.n_b + B;
            if (qf < p.items) {
                a1 += base[qf * (4 * S)];
                a2 += base[qf * (4 * S) + S];
            }
            const int64_t qr = d * p.n_b + (B >= d ? B - d : B - d + p.n_b);
            if (qr < p.items) {
                a1 += base[qr * (4 * S) + 2 * S];
                a2 += base[qr * (4 * S) + 3 * S];
            }
        }
    }
    sh[0][pr][tl] = a1;
    sh[1][pr][tl] = a2;
    __syncthreads();
    if (pr != 0 || i >= N) return;
    for (int q = 1; q < kF64Parts; ++q) {
        a1 += sh[0][q][tl];
        a2 += sh[1][q][tl];
    }
    const double* v = in.base + (in.kidx ? (int64_t)(*in.kidx + in.koff) * in.stride : 0);
    double* y = out.base + (out.kidx ? (int64_t)(*out.kidx + out.koff) * out.stride : 0);
    y[i] = lambda1 * v[i] + kInv4Pi * a1;
    y[N + i] = lambda2 * v[N + i] + kInv4Pi * a2;
}

size_t f64_src_bytes(int64_t N) { return (size_t)f64_plan(N).n_chunks * kF64Chunk * 8 * sizeof(double); }

// The partial sums of the FP64 path (kept apart from the other paths' buffer:
// they take 2.6 KB per node and are allocated on the first FP64 application, once
// per context).  That application may be one that the caller captures after
// applications of another precision: the relaxed mode lets this thread allocate
// meanwhile, and the buffer is an ordinary one that outlives the graph.
ibim_status f64_prepare(ibim_ctx* c)
{
    if (c->d_part64 != nullptr) return IBIM_OK;
    const F64Plan p = f64_plan(c->N);
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    IBIM_CUDA(cudaThreadExchangeStreamCaptureMode(&mode));
    const ibim_status s = ensure(c, (void**)&c->d_part64, &c->part64_bytes,
                                 sizeof(double) * (kF64Head + (size_t)p.items * 4 * p.m * kF64Chunk));
    IBIM_CUDA(cudaThreadExchangeStreamCaptureMode(&mode));  // the thread's own mode again
    return s;
}

ibim_status f64_apply(ibim_ctx* c, const PairConsts& k, VecRef in, OutRef out, const int* d_skip)
{
    IBIM_TRY(f64_prepare(c));
    const int64_t N = c->N;
    const F64Plan p = f64_plan(N);
    const int64_t n_pad = p.n_chunks * kF64Chunk;
    const int bs = 256;
    pack_f64_kernel<<<(unsigned)((n_pad + bs - 1) / bs), bs, 0, c->stream>>>(
        c->d_geo64, in, N, n_pad, (double2*)c->d_src, c->d_part64, d_skip);
    F64Consts kk;
    kk.th1 = k.th1;
    kk.th2 = k.th2;
    kk.om1 = 1.0 - k.th1;
    kk.om2 = 1.0 - k.th2;
    kk.kappa = k.kappa;
    kk.tau2 = k.tau2;
    kk.four_tau2 = k.four_tau2;
    kk.k12t = k.k12_tube;
    kk.rule0 = (k.four_tau2 < 3.0e38) ? 1 : 0;
    const double two_tau = 2.0 * sqrt(k.tau2);
    kk.far_dist = (float)((two_tau > 1.5 ? two_tau : 1.5) * 1.001 + 1e-3);
    // few items: one warp per CTA, so that they spread over the SMs
    const int threads = p.items >= 4 * (int64_t)c->num_sms ? 128 : 32;
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, pair_f64_kernel, threads, 0);
    const int64_t cap = (int64_t)std::max(1, occ) * c->num_sms, per = threads / 32;
    const unsigned grid = (unsigned)std::min<int64_t>(cap, (p.items + per - 1) / per);
    IBIM_TRY(timing_begin(c));
    pair_f64_kernel<<<grid, threads, 0, c->stream>>>((const double2*)c->d_src, c->d_frames, p, kk, c->d_exptab,
                                                      c->d_part64, d_skip);
    IBIM_TRY(timing_end(c, N * N));
    fixup_f64_kernel<<<(unsigned)((N + kF64Nodes - 1) / kF64Nodes), kF64Parts * kF64Nodes, 0, c->stream>>>(
        c->d_part64, p, N, k.lambda1, k.lambda2, in, out, d_skip);
    count_launch(c, 3);
    IBIM_CUDA(cudaGetLastError());
    return IBIM_OK;
}

}  // namespace ibim
