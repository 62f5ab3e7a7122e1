// Fused FP32 MinRes iteration for a batch of right-hand sides (the inner
// solve of the mixed-precision D-MinRes, arXiv:0901.3163 Sec. 2).
//
// Two passes over the vectors per iteration, and a third per block of six:
//   K1 (stencil + epilogue, one block = 128 sites of one right-hand side):
//        v_j   = u_j / beta_j                      (u_j: unnormalised Lanczos vector; the
//                                                   v's are never stored, only the u's)
//        w     = Q v_j - beta_j v_{j-1}            (Q u_j / beta_j: Q is linear)
//        alpha_j partial = Re <v_j, w>
//   K2a: u_{j+1} = w - alpha_j v_j and the block partials of ||u_{j+1}||^2;
//   K1b: alpha_j = sum of K1's block partials (one block per right-hand side);
//   K2b: beta_{j+1}, the Givens rotation of step j and the coefficients of its direction
//        (one block per right-hand side);
//   after the fifth iteration of a block: the deferred update of the directions and the
//        iterate (minres_state.cuh has the scheme, the buffers and the traffic).
// For a single right-hand side K1b and K2b are folded into the last block of K1 and K2a to
// finish.  The partials are summed in a fixed order, so results are deterministic.  A block
// of six iterations is captured once as a CUDA graph and replayed.
// Measured on 16^3 x 32 with 11 right-hand sides, a whole call: 322 ms with the directions in
// every iteration, 280 ms with blocks of six, 247 ms with the stencil of k_minres_k1 below.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "dlz_internal.cuh"
#include "krylov_util.cuh"
#include "reduce.cuh"
#include "solvers.h"
#include "minres_state.cuh"
#include "slab_walk.cuh"
#include "wilson_site.cuh"

namespace dlz {



namespace {

constexpr int kThreads = 128;

// K1.  Bound by the gathers (L1 and L2 each about two thirds busy, FMA about half), so it moves
// as few vectors as it can: u gathered, u_{j-1} read, w written.  16^3 x 32, 11 right-hand
// sides: 214 us with the direction update in it (at the memory rate then), 127 us without, 110
// us with multiplications in place of the integer divisions of a site's coordinates and fewer
// address instructions; 415 MB at the memory rate would take 61 us.
__global__ void __launch_bounds__(kThreads, 7)
k_minres_k1(const float4 *__restrict__ Ub, const float4 *__restrict__ Up, float4 *__restrict__ W,
            const float4 *__restrict__ links, Geom g, SlabWalk w, float kappa, int N,
            FusedState *__restrict__ st, double *__restrict__ partials, unsigned *__restrict__ counters) {
    int q, sb, s0, nb;
    slab_rhs(w, blockIdx.x, q, sb);
    slab_block(w, sb, s0, nb);
    const int s = s0 + threadIdx.x;
    const size_t base = (size_t)q * 6 * g.V;
    float facc = 0.f;
    if ((int)threadIdx.x < nb)
        facc = minres_k1_site(s, g, kappa, Ub + base, Up + base, W + base, links, st[q]);
    // block partials of alpha_q; with counters, the last block of q to finish forms
    // alpha_q (one right-hand side: saves a launch); without, k_minres_alpha does
    const int nbq = w.dN.div(gridDim.x);
    if (!counters) {
        block_partial_store<kThreads>(facc, partials + (size_t)q * nbq + sb);
        return;
    }
    double a;
    if (partial_then_last_sum<kThreads>(facc, partials + (size_t)q * nbq, sb, nbq, counters + q, &a) &&
        threadIdx.x == 0)
        fused_alpha(st[q], a);
}

// K2a: bound by memory (60 us for the same size: 415 MB, 6.9 TB/s)
__global__ void __launch_bounds__(kThreads)
k_minres_k2a(const float4 *W, const float4 *Vc, float4 *Out, float4 *Copy, Geom g, int N, int iter,
             FusedState *__restrict__ st, double *__restrict__ partials, unsigned *__restrict__ counters) {
    // Vc: the unnormalised u_j; alpha_j v_j = (alpha_j / beta_j) u_j
    const int q = blockIdx.x % N;
    const int s = (blockIdx.x / N) * blockDim.x + threadIdx.x;
    const size_t base = (size_t)q * 6 * g.V;
    float facc = 0.f;
    if (s < g.V)
        facc = minres_k2a_site(s, g.V, W + base, Vc + base, Out + base, Copy ? Copy + base : nullptr, st[q]);
    // the last block of q to finish: beta_{j+1} and the Givens rotation of step j
    // (with counters; without, k_minres_k2b does it)
    const int nbq = gridDim.x / N;
    if (!counters) {
        block_partial_store<kThreads>(facc, partials + (size_t)q * nbq + blockIdx.x / N);
        return;
    }
    double r2;
    if (partial_then_last_sum<kThreads>(facc, partials + (size_t)q * nbq, blockIdx.x / N, nbq, counters + q, &r2))
        fused_givens(st[q], r2, iter);
}

// the deferred update of a block (LAST: of the one step left at the end), n float4 per
// right-hand side, blockIdx.y the right-hand side
template <bool LAST>
__global__ void __launch_bounds__(256)
k_minres_directions(MinresVectors b, const FusedState *__restrict__ st, long n) {
    const long j = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const size_t i = (size_t)blockIdx.y * n + j;
    if (LAST) minres_last_direction(b, i, st[blockIdx.y]);
    else minres_directions_elem(b, i, st[blockIdx.y]);
}

// alpha_q = sum of the block partials of right-hand side q (block q of the grid),
// in a fixed order
__global__ void __launch_bounds__(1024)
k_minres_alpha(const double *__restrict__ partials, int nbq, FusedState *__restrict__ st) {
    const int q = blockIdx.x;
    double t = 0.0;
    for (int b = threadIdx.x; b < nbq; b += blockDim.x) t += partials[(size_t)q * nbq + b];
    __shared__ double sm[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0;
        for (int w = 0; w < (int)(blockDim.x / 32); ++w) a += sm[w];
        fused_alpha(st[q], a);
    }
}

// K2b: beta_{j+1} = sqrt(sum of K2a's partials) and the Givens rotation of step j,
// one block per right-hand side
__global__ void __launch_bounds__(1024)
k_minres_k2b(const double *__restrict__ partials, int nbq, int iter, FusedState *__restrict__ st) {
    const int q = blockIdx.x;
    double t = 0.0;
    for (int b = threadIdx.x; b < nbq; b += blockDim.x) t += partials[(size_t)q * nbq + b];
    __shared__ double sm[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = t;
    __syncthreads();
    double r2 = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x / 32); ++w) r2 += sm[w];
    fused_givens(st[q], r2, iter);
}

}  // namespace

// The slab walk of K1 for an N-RHS batch (its weight: slab_walk.cuh)
static SlabWalk minres_slab_walk(const Op &op, int N) {
    const Geom &g = op.g;
    return make_slab_walk(g.L[0] * g.L[1], g.L[2], g.L[3], N, 900.0);
}

long minres_blocks_per_rhs(const Op &op, int N) {
    return std::max(slab_blocks(minres_slab_walk(op, N)), (long)(op.g.V + kThreads - 1) / kThreads);
}

int minres_fused_batch(Op &op, int N, const MinresVectors &b, FusedState *ms, double *partials, const double *d_tol,
                       const dlz_params &p, int &iters, GraphExec &ge, bool e_init) {
    const long n = 6L * op.g.V;
    const float4 *r = b.c[0];
    // beta_1 = ||r_q||, rotations reset
    DLZ_TRY(reduce32<16>(op, n, [=] __device__(long i, float (&acc)[16]) {
#pragma unroll
        for (int q = 0; q < 16; ++q)
            if (q < N) { const float4 v = r[(size_t)q * n + i]; acc[q] += (v.x * v.x + v.y * v.y) + (v.z * v.z + v.w * v.w); }
    }, [=] __device__(const double *res) {
        for (int q = 0; q < N; ++q) {
            fused_init(ms[q], sqrt(res[q]));
        }
    }));
    // u_0 = r is in place; u_{-1} and the directions start at zero
    for (float4 *z : {b.c[6], b.d1, b.d2})
        DLZ_CUDA_TRY(cudaMemsetAsync(z, 0, (size_t)N * n * sizeof(float4), op.stream));
    if (!e_init) DLZ_CUDA_TRY(cudaMemsetAsync(b.e, 0, (size_t)N * n * sizeof(float4), op.stream));
    const Geom g = op.g;
    const float kappa = (float)op.kappa;
    const float4 *links = op.gauge32.as<float4>();
    const SlabWalk w = minres_slab_walk(op, N);
    const unsigned blocks1 = (unsigned)(slab_blocks(w) * N), blocks = (unsigned)(((g.V + kThreads - 1) / kThreads) * N);
    const int st1 = blocks1 / N > 512 ? 1024 : 256, st2 = blocks / N > 512 ? 1024 : 256;
    double *partials2 = partials + minres_blocks_per_rhs(op, N) * N;   // K2a's partials after K1's
    unsigned *counters = nullptr;             // block counter, reset by the last block
    if (N == 1) {
        // one right-hand side: the sums are taken by the kernels' last blocks (latency);
        // several: by one-block-per-RHS kernels (cheaper than a tail in every block)
        counters = reinterpret_cast<unsigned *>(partials2 + minres_blocks_per_rhs(op, N) * N);
        DLZ_CUDA_TRY(cudaMemsetAsync(counters, 0, sizeof(unsigned), op.stream));
    }
    auto iteration = [&](int i) -> int {
        // K1 moves 72 reals per site and right-hand side: u_j gathered, u_{j-1} read and w
        // written (24 each), plus the links once per site
        const float4 *U = b.c[mr_u(i)];
        float4 *W = b.c[mr_w(i)];
        if (i == kMrBlock - 1) {
            k_minres_directions<false><<<dim3((unsigned)((n + 255) / 256), N), 256, 0, op.stream>>>(b, ms, n);
            op.prof.launches++;
        }
        op.prof.stencil_start(op.stream, true, g.V, N, 72, 1);
        k_minres_k1<<<blocks1, kThreads, 0, op.stream>>>(U, b.c[mr_up(i)], W, links, g, w, kappa, N, ms, partials,
                                                        counters);
        op.prof.stencil_stop(op.stream);
        if (!counters) k_minres_alpha<<<N, st1, 0, op.stream>>>(partials, (int)(blocks1 / N), ms);
        op.prof.launches += counters ? 1 : 2;
        DLZ_CUDA_TRY(cudaGetLastError());
        // u_{j+1} = w - alpha v_j ; beta_{j+1} ; Givens rotation of step j
        k_minres_k2a<<<blocks, kThreads, 0, op.stream>>>(W, U, b.c[mr_out(i)], i == kMrBlock - 1 ? b.c[6] : nullptr, g,
                                                        N, i, ms, partials2, counters);
        if (!counters) k_minres_k2b<<<N, st2, 0, op.stream>>>(partials2, (int)(blocks / N), i, ms);
        op.prof.launches += counters ? 1 : 2;
        DLZ_CUDA_TRY(cudaGetLastError());
        return DLZ_OK;
    };
    auto six = [&]() -> int {
        for (int i = 0; i < kMrBlock; ++i) DLZ_TRY(iteration(i));
        return DLZ_OK;
    };
    std::vector<FusedState> h(N);
    std::vector<double> tol(N);
    DLZ_TRY(d2h_sync(op, tol.data(), d_tol, N * sizeof(double)));
    const int check = std::max(6, (p.check_every / 6) * 6);
    int it = 0;
    // DLZ_TRACE=1: time the replays of the 6-iteration group (diagnostics)
    const char *trace_env = std::getenv("DLZ_TRACE");
    const bool trace = trace_env && trace_env[0] == '1';
    Event te0, te1;
    double t_graph = 0.0;
    int n_timed = 0;
    if (trace) {
        DLZ_CUDA_TRY(te0.create());
        DLZ_CUDA_TRY(te1.create());
    }
    while (iters < p.max_iter) {
        const bool timed = trace && ge.exec;      // not the replay that captures the graph
        if (timed) DLZ_CUDA_TRY(cudaEventRecord(te0.e, op.stream));
        DLZ_TRY(run_graph(op, ge, six));
        if (timed) {
            DLZ_CUDA_TRY(cudaEventRecord(te1.e, op.stream));
            DLZ_CUDA_TRY(cudaEventSynchronize(te1.e));
            float ms = 0.f;
            if (cudaEventElapsedTime(&ms, te0.e, te1.e) == cudaSuccess) { t_graph += ms; ++n_timed; }
            else cudaGetLastError();
        }
        iters += 6;
        it += 6;
        if (it % check == 0 || iters >= p.max_iter) {
            DLZ_TRY(d2h_sync(op, h.data(), ms, N * sizeof(FusedState)));
            ge.sample(op.prof);
            bool done = true;
            for (int q = 0; q < N; ++q) {
                if (!std::isfinite(h[q].phibar)) return fail(DLZ_ERR_NONFINITE, "MinRes residual not finite");
                if (!(std::fabs(h[q].phibar) <= tol[q] * h[q].r0 || h[q].beta_next == 0.0)) done = false;
            }
            if (done) break;
        }
    }
    if (trace) {
        std::fprintf(stderr, "[dlz] fused MinRes N=%d: %d iterations, graph replay %.4f ms per iteration (%d timed)\n",
                     N, iters, n_timed ? t_graph / (6.0 * n_timed) : 0.0, n_timed);
    }
    // the direction update of the last step
    k_minres_directions<true><<<dim3((unsigned)((n + 255) / 256), N), 256, 0, op.stream>>>(b, ms, n);
    op.prof.launches++;
    DLZ_CUDA_TRY(cudaGetLastError());
    return DLZ_OK;
}

}  // namespace dlz
