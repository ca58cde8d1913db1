// Right-hand side (Sec. 2.2), reaction potential and polarization energy
// (Sec. 3.5) and surface area (Sec. 3.4), FP64.  These are N x Nc pair sums
// evaluated once per solve; all reductions are deterministic (per-block
// partials summed in a fixed order).
#include <vector>

#include "ibim_internal.cuh"
#include "math64.cuh"

namespace ibim {

// g1_i = sum_k q_k/eps_I G0(x*_i, z_k);  g2_i = sum_k q_k/eps_I dG0(x*_i, z_k)/dn(x*_i),
// dG0(x, z)/dn(x) = -(x - z).n / (4 pi |x - z|^3).  Bound by the FP64 pipe: 18
// instructions per pair, the field sum_k q_k r / |r|^3 as a vector and its
// product with n once per node, 1/|r| by rsqrt64.  A block holds 32 nodes (the
// lanes) and its eight warps take every eighth charge, so that 32-node blocks
// spread evenly over the SMs and a small molecule still fills them.
// 120,011 nodes x 2,000 charges: 7.85 ms; 10.5 ms with 256-node blocks (three or
// four per SM), the library's rsqrt and a dot product per pair.
constexpr int kRhsNodes = 32, kRhsParts = 8;
constexpr int kRhsAtomTile = 256;

__global__ void __launch_bounds__(kRhsNodes * kRhsParts)
    rhs_kernel(const double* __restrict__ geo, int64_t N, const double* __restrict__ z,
               const double* __restrict__ q, int64_t Nc, double inv_eps_in, double* __restrict__ g)
{
    __shared__ double sz[kRhsAtomTile][4];
    __shared__ double red[kRhsParts][4][kRhsNodes];
    const int lane = threadIdx.x % kRhsNodes, part = threadIdx.x / kRhsNodes;
    const int64_t i = (int64_t)blockIdx.x * kRhsNodes + lane;
    const int64_t n = i < N ? i : N - 1;
    const double x0 = geo[n], x1 = geo[N + n], x2 = geo[2 * N + n];
    double g1 = 0.0, e0 = 0.0, e1 = 0.0, e2 = 0.0;
    for (int64_t k0 = 0; k0 < Nc; k0 += kRhsAtomTile) {
        const int cnt = (int)((Nc - k0 < kRhsAtomTile) ? Nc - k0 : kRhsAtomTile);
        __syncthreads();
        for (int t = threadIdx.x; t < cnt; t += kRhsNodes * kRhsParts) {
            sz[t][0] = z[3 * (k0 + t)];
            sz[t][1] = z[3 * (k0 + t) + 1];
            sz[t][2] = z[3 * (k0 + t) + 2];
            sz[t][3] = q[k0 + t];
        }
        __syncthreads();
#pragma unroll 2
        for (int t = part; t < cnt; t += kRhsParts) {
            const double r0 = x0 - sz[t][0], r1 = x1 - sz[t][1], r2 = x2 - sz[t][2];
            const double rr = r0 * r0 + r1 * r1 + r2 * r2;
            // (a charge on the node or out of range: the library's special cases)
            const bool plain = (unsigned)(__double2hiint(rr) - 0x00200000) < 0x7fc00000u;
            const double inv = plain ? rsqrt64(rr) : rsqrt(rr);
            const double qi = sz[t][3] * inv;
            g1 += qi;
            const double q3 = qi * (inv * inv);
            e0 = fma(q3, r0, e0);
            e1 = fma(q3, r1, e1);
            e2 = fma(q3, r2, e2);
        }
    }
    red[part][0][lane] = g1;
    red[part][1][lane] = e0;
    red[part][2][lane] = e1;
    red[part][3][lane] = e2;
    __syncthreads();
    if (part != 0 || i >= N) return;
    for (int p = 1; p < kRhsParts; ++p) {
        g1 += red[p][0][lane];
        e0 += red[p][1][lane];
        e1 += red[p][2][lane];
        e2 += red[p][3][lane];
    }
    g[i] = kInv4Pi * inv_eps_in * g1;
    g[N + i] = -kInv4Pi * inv_eps_in * (e0 * geo[3 * N + i] + e1 * geo[4 * N + i] + e2 * geo[5 * N + i]);
}

ibim_status rhs_launch(ibim_ctx* c, double eps_in, double* d_g)
{
    const int64_t N = c->N;
    rhs_kernel<<<(unsigned)((N + kRhsNodes - 1) / kRhsNodes), kRhsNodes * kRhsParts, 0, c->stream>>>(
        c->d_geo64, N, c->d_z, c->d_q, c->Nc, 1.0 / eps_in, d_g);
    count_launch(c);
    IBIM_CUDA(cudaGetLastError());
    return IBIM_OK;
}

// psi_rxn(z_k) = sum_j w_j [ (th1 A - 1) s_y / (4 pi rho^3) psi_j + (1 - E)/(4 pi rho) psin_j ],
// r = z_k - y*_j, s_y = r.n(y*_j), E = exp(-kappa rho), A = E (1 + kappa rho).
// Grid: (charge groups of ATOMS) x (node splits); each CTA writes one partial per
// charge.  Bound by the FP64 pipe: 32 instructions per pair,
//   ((th1 A - 1) (r . a m) / rho^2 + (1 - E) b) / rho,
// 1/rho by rsqrt64 and E from the table (120,011 nodes x 2,000 charges: 14.6 ms;
// 20.6 ms with the library's exp and rsqrt).  ATOMS = 4 shares the node's loads;
// fewer than four charges take ATOMS = 1, which evaluates no duplicates.
constexpr int kEnThreads = 128;

template <int ATOMS>
__global__ void __launch_bounds__(kEnThreads)
    energy_partial_kernel(const double* __restrict__ geo, int64_t N, const double* __restrict__ z, int64_t Nc,
                          const double* __restrict__ p, double th1, double kappa, int64_t chunk,
                          const double* __restrict__ exptab, double* __restrict__ part)
{
    __shared__ double red[kEnThreads / 32][ATOMS];
    __shared__ double tab[kExpTab];
    for (int q = threadIdx.x; q < kExpTab; q += kEnThreads) tab[q] = exptab[q];
    const int64_t a0 = (int64_t)blockIdx.x * ATOMS;
    const int64_t j0 = (int64_t)blockIdx.y * chunk;
    const int64_t j1 = (j0 + chunk < N) ? j0 + chunk : N;
    double zx[ATOMS], zy[ATOMS], zz[ATOMS], acc[ATOMS];
#pragma unroll
    for (int a = 0; a < ATOMS; ++a) {
        const int64_t k = (a0 + a < Nc) ? a0 + a : Nc - 1;
        zx[a] = z[3 * k];
        zy[a] = z[3 * k + 1];
        zz[a] = z[3 * k + 2];
        acc[a] = 0.0;
    }
    __syncthreads();
    for (int64_t j = j0 + threadIdx.x; j < j1; j += kEnThreads) {
        const double y0 = geo[j], y1 = geo[N + j], y2 = geo[2 * N + j];
        const double w = geo[6 * N + j];
        const double a = w * p[j], b = w * p[N + j];
        const double m0 = a * geo[3 * N + j], m1 = a * geo[4 * N + j], m2 = a * geo[5 * N + j];
#pragma unroll
        for (int q = 0; q < ATOMS; ++q) {
            const double r0 = zx[q] - y0, r1 = zy[q] - y1, r2 = zz[q] - y2;
            const double rr = r0 * r0 + r1 * r1 + r2 * r2;
            const double inv = rsqrt64(rr);
            const double x = kappa * (rr * inv);
            const double E = exp_neg64(x, tab);
            const double A = fma(E, x, E);
            const double sa = r0 * m0 + r1 * m1 + r2 * m2;
            const double u = fma(th1, A, -1.0) * (inv * inv);
            acc[q] = fma(inv, fma(u, sa, fma(-E, b, b)), acc[q]);
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < ATOMS; ++q) {
        double v = acc[q];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) red[warp][q] = v;
    }
    __syncthreads();
    if (threadIdx.x < ATOMS) {
        double v = 0.0;
        for (int w = 0; w < kEnThreads / 32; ++w) v += red[w][threadIdx.x];
        const int64_t k = a0 + threadIdx.x;
        if (k < Nc) part[(int64_t)blockIdx.y * Nc + k] = v;
    }
}

// psi_rxn[k] = (1/(4 pi)) sum_splits part; out[0] = G_pol = 1/2 sum q_k psi_rxn[k].
// Many splits (few charges): a warp per charge, its lanes over the splits;
// otherwise a thread per charge.  Fixed orders.
__global__ void __launch_bounds__(1024)
    energy_final_kernel(const double* __restrict__ part, int64_t nsplit, int64_t Nc,
                                    const double* __restrict__ q, double* __restrict__ psi, double* __restrict__ out)
{
    __shared__ double red[1024];
    double g = 0.0;
    if (nsplit >= 16) {
        const int lane = threadIdx.x & 31;
        for (int64_t k = threadIdx.x >> 5; k < Nc; k += blockDim.x >> 5) {
            double v = 0.0;
            for (int64_t s = lane; s < nsplit; s += 32) v += part[s * Nc + k];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            v *= kInv4Pi;
            if (lane == 0) {
                if (psi != nullptr) psi[k] = v;
                g += q[k] * v;
            }
        }
    } else {
        for (int64_t k = threadIdx.x; k < Nc; k += blockDim.x) {
            double v = 0.0;
            for (int64_t s = 0; s < nsplit; ++s) v += part[s * Nc + k];
            v *= kInv4Pi;
            if (psi != nullptr) psi[k] = v;
            g += q[k] * v;
        }
    }
    red[threadIdx.x] = g;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = 0.5 * red[0];
}

// Surface area: sum_j w_j (Sec. 3.4), deterministic two-level sum.
__global__ void area_kernel(const double* __restrict__ w, int64_t N, double* __restrict__ out)
{
    __shared__ double red[1024];
    double s = 0.0;
    for (int64_t j = threadIdx.x; j < N; j += blockDim.x) s += w[j];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = red[0];
}

ibim_status energy_launch(ibim_ctx* c, const ibim_phys& p, const double* d_p, double* d_psi, double* gpol_host,
                          double* area_host)
{
    const int64_t N = c->N, Nc = c->Nc;
    const int atoms = Nc < 4 ? 1 : 4;
    const int64_t groups = (Nc + atoms - 1) / atoms;
    // about eight CTAs per SM: five fit at a time, and the rest even out the ends
    int64_t nsplit = (8LL * c->num_sms + groups - 1) / groups;
    const int64_t maxsplit = (N + kEnThreads - 1) / kEnThreads;
    if (nsplit > maxsplit) nsplit = maxsplit;
    if (nsplit < 1) nsplit = 1;
    if (nsplit > 65535) nsplit = 65535;
    const int64_t chunk = (N + nsplit - 1) / nsplit;
    IBIM_TRY(ensure(c, (void**)&c->d_red, &c->red_bytes, sizeof(double) * (nsplit * Nc + 8)));
    double* part = c->d_red + 8;
    dim3 grid((unsigned)groups, (unsigned)nsplit);
    if (atoms == 1)
        energy_partial_kernel<1><<<grid, kEnThreads, 0, c->stream>>>(c->d_geo64, N, c->d_z, Nc, d_p,
                                                                    p.eps_out / p.eps_in, p.kappa, chunk, c->d_exptab,
                                                                    part);
    else
        energy_partial_kernel<4><<<grid, kEnThreads, 0, c->stream>>>(c->d_geo64, N, c->d_z, Nc, d_p,
                                                                    p.eps_out / p.eps_in, p.kappa, chunk, c->d_exptab,
                                                                    part);
    energy_final_kernel<<<1, 1024, 0, c->stream>>>(part, nsplit, Nc, c->d_q, d_psi, c->d_red);
    count_launch(c, 2);
    if (area_host != nullptr) {
        area_kernel<<<1, 1024, 0, c->stream>>>(c->d_geo64 + 6 * N, N, c->d_red + 1);
        count_launch(c);
    }
    IBIM_CUDA(cudaGetLastError());
    double out[2];
    IBIM_CUDA(cudaMemcpyAsync(out, c->d_red, sizeof(double) * (area_host ? 2 : 1), cudaMemcpyDeviceToHost, c->stream));
    IBIM_CUDA(cudaStreamSynchronize(c->stream));
    *gpol_host = out[0];
    if (area_host != nullptr) *area_host = out[1];
    return IBIM_OK;
}

ibim_status area_launch(ibim_ctx* c, double* area_host)
{
    IBIM_TRY(ensure(c, (void**)&c->d_red, &c->red_bytes, sizeof(double) * 8));
    area_kernel<<<1, 1024, 0, c->stream>>>(c->d_geo64 + 6 * c->N, c->N, c->d_red + 1);
    count_launch(c);
    IBIM_CUDA(cudaGetLastError());
    IBIM_CUDA(cudaMemcpyAsync(area_host, c->d_red + 1, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    IBIM_CUDA(cudaStreamSynchronize(c->stream));
    return IBIM_OK;
}

}  // namespace ibim
