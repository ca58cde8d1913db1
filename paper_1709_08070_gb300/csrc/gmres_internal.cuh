// Internal GMRES pieces shared by the single-molecule and batched solvers.
#pragma once
#include "ibim_internal.cuh"

namespace ibim {

constexpr int kMaxRestart = 128;
constexpr int kVecThreads = 256;
constexpr int kDotGroup = 8;  // dot products a warp forms together

// What the host reads of a finished cycle (pinned host memory, written by the
// device; no answer before `done`).
struct GmOutcome {
    int done, k, conv;
};
constexpr int kStepsPerGraph = 2;  // Arnoldi steps in the captured graph and between two waits of the host

struct GmState {
    int k;       // current Arnoldi step within the cycle
    int done;    // stop expanding (converged, cycle full or breakdown)
    int conv;    // residual estimate below target
    int kmax;    // steps allowed in this cycle
    int m;       // restart length (row stride of H)
    int norm_ticket;  // blocks that have written their norm partial (back to 0 by the last one)
    double target;     // absolute residual target of the cycle
    double resid;      // |e_{k}| after the last rotation
    double hn;         // ||w|| of the current step
    double coef[kMaxRestart + 1];  // Gram-Schmidt coefficients of the current pass
    double hcol[kMaxRestart + 1];  // accumulated column k of H
    double cs[kMaxRestart], sn[kMaxRestart];
    double e[kMaxRestart + 1];
    double y[kMaxRestart];
    GmOutcome* out;  // nullptr: not wanted (batched solves read the state itself)
    double H[(kMaxRestart + 1) * kMaxRestart];  // row-major, row stride m
    int dot_ticket[(kMaxRestart + 1 + kDotGroup - 1) / kDotGroup];  // blocks done with a group of dot products
};

// One system's vectors as the orthogonalisation kernels see them: the basis, its
// state and partial sums, and the split of the vector into nblk blocks of C
// elements.
struct GmSys {
    double* V;
    int64_t len;
    GmState* st;
    double* part;  // nblk x (kMaxRestart + 1)
    int C, nblk;
};

struct GmresWork {
    int m = 0;
    int64_t len = 0;
    double* V = nullptr;       // (m + 1) x len
    double* x = nullptr;       // len: current iterate (solution accumulator)
    double* r = nullptr;       // len: residual / scratch
    double* t = nullptr;       // len: operator output scratch
    double* g = nullptr;       // len: right-hand side
    double* xb = nullptr;      // len: refinement base iterate (x holds the correction to it)
    double* gin = nullptr;     // len: refinement right-hand side (residual at xb)
    double* part = nullptr;    // per-block partial sums ((kMaxRestart + 1) x max(nblk, sys.nblk))
    int nblk = 0;
    GmSys sys;                 // the orthogonalisation kernels' view
    GmState* st = nullptr;     // device state
    GmState* h_st = nullptr;   // pinned host mirror (small fields only are read)
    GmOutcome* h_out = nullptr;  // pinned, behind h_st
    cudaStream_t gs = nullptr; // capture-capable stream owned by the solver
    cudaEvent_t ev = nullptr;
    cudaEvent_t poll[2] = {nullptr, nullptr};  // behind the two latest pairs of steps
    cudaGraphExec_t exec = nullptr;
    int graph_prec = 0;
    PairConsts graph_k;
    uint64_t graph_generation = 0;  // workspace generation the graph was captured with
    int graph_variant = -1;         // FP32 pair-kernel variant and CTAs per SM captured in the graph
    int graph_bps = -1;
    int graph_ff = -1;              // float-float kernel captured in the graph
    bool graph_valid = false;
};


// Building blocks (gmres.cu); every launch goes on c->stream.
ibim_status gm_alloc(ibim_ctx* c, int m);
ibim_status gm_init(ibim_ctx* c, const ibim_phys& p, int m, double* gnorm);  // state, g, ||g||, x = 0; syncs
// CGS2, norm, Givens and scaling of one Arnoldi step (after w = A v_k): four
// launches for one system, or for nsys systems at once (device array)
constexpr int kOrthoLaunches = 4;
ibim_status gm_ortho(ibim_ctx* c);
ibim_status gm_ortho_batch(const GmSys* d_sys, int nsys, int max_nblk, int max_C, cudaStream_t stream);
ibim_status gm_cycle_begin(ibim_ctx* c, bool x_zero, double target, int kmax);  // r = g - t (t = A x), V0, e
ibim_status gm_cycle_end(ibim_ctx* c);  // y = H^-1 e, x += V y
ibim_status gm_fetch_state(ibim_ctx* c);  // async copy of the small state fields to the pinned mirror

}  // namespace ibim
