// Fused FP32 CG on the normal equations (CGNR) for a batch of right-hand sides:
// the inner solve of the mixed-precision D-CG (arXiv:0901.3163, Sec. 2: CG on
// D^dag D).  For D e = s0 it iterates, per right-hand side, CG on D^dag D e = D^dag s0:
//   p = r + beta p,  t = D p,  alpha = |r|^2 / |t|^2,
//   e += alpha p,  r -= alpha D^dag t,  beta = |r_new|^2 / |r|^2,
// r being the CG residual (it starts as D^dag s0 and is then updated by the recurrence, as
// in CG on any hermitian matrix).  |s|, the norm of the residual of D e = s0 that the inner
// stopping test needs, is a scalar recurrence: |s_{k+1}|^2 = |s_k|^2 - alpha_k |r_k|^2.
// Since D p = D r + beta D p_old, the image t is carried, so each kernel applies its
// stencil to ONE vector and the direction p is needed by nothing but e:
//   K1:  t = D r + beta t      (the stencil gathers r); block partials of |t|^2,
//   K23: r' = r - alpha D^dag t (the stencil gathers t); block partials of |r'|^2.
// p and e are linear in the residuals, so they are brought up to date once per block of
// kCgBlock = 6 iterations: the block keeps its residuals r_0 .. r_5 (K23 writes r' to the
// next buffer, which costs no traffic), the step-length kernel carries the FP64
// coefficients of p and of the block's sum of alpha p over (r_0 .. r_5, p_old), and
// k_cg_directions makes e += ..., p = ... in one streaming pass.  Per site and right-hand
// side an iteration moves 72 (K1) + 72 (K23) + 40 (240 / 6: six r and p, e read; p, e
// written) = 184 reals, against 240 with p and e updated by K1 in every iteration.
// Measured on 24^3 x 48 with 16 right-hand sides, a whole D-CG call of 348 iterations:
// 913 ms with p and e updated in every iteration, 773 ms with blocks, 741 ms with fewer
// instructions per site in the stencil (K1 716, K23 754, the directions 1371 / 6 us per
// iteration; at the memory rate 577, 577 and 1335 / 6).  K1 and K23 are bound by the gathers:
// L1 and L2 each two thirds busy, FMA 45 %.  On 8^4 with 4 right-hand sides, where launches
// bound the iteration, 6.56, 6.33 and 4.6 ms (the last with the work memory of a call kept
// with the operator).
// Each kernel writes only vectors it does not gather (and only at its own site).
// One-block-per-RHS kernels sum the partials in a fixed order and update the step lengths;
// a block of six iterations is a CUDA graph that is captured once and replayed.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "dlz_internal.cuh"
#include "krylov_util.cuh"
#include "reduce.cuh"
#include "slab_walk.cuh"
#include "solvers.h"
#include "stage_gather.cuh"
#include "wilson_eo_site.cuh"
#include "wilson_site.cuh"

namespace dlz {

constexpr int kCgBlock = kCgResiduals;     // iterations per block (and per CUDA graph)

struct CgFusedState {        // one per right-hand side
    double gam;              // |r|^2
    double alpha, beta;
    double ss;               // |s|^2
    // coefficients over (r_0 .. r_{kCgBlock-1}, p_old) of the current p and of the block's
    // sum of alpha p so far
    double pc[kCgBlock + 1], ec[kCgBlock + 1];
    float f[4];              // f0 alpha, f1 beta (FP32 copies for the element updates)
    float fp[kCgBlock + 1], fe[kCgBlock + 1];   // pc and ec of a finished block
};
size_t cg_state_bytes() { return sizeof(CgFusedState); }

namespace {

constexpr int kT = 128;

// block sum of up to two per-thread values into partials (FP64 across threads)
template <int NV>
__device__ inline void block_partials(float (&v)[NV], double *__restrict__ out, size_t stride) {
    __shared__ double sm[NV][kT / 32];
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        double a = (double)v[j];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
        if ((threadIdx.x & 31) == 0) sm[j][threadIdx.x >> 5] = a;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int j = 0; j < NV; ++j) {
            double t = 0.0;
#pragma unroll
            for (int w = 0; w < kT / 32; ++w) t += sm[j][w];
            out[j * stride] = t;
        }
    }
}

// The element update of both kernels at one site: K1 (DAG = false) O = o + c A (o = D r,
// A = t, c = beta), K23 (DAG = true) O = A - c o (o = D^dag t, A = r, c = alpha).  A and O
// may be the same field.  Returns the site's share of |O|^2.
template <bool DAG>
__device__ inline float step_update(const float4 *A, float4 *O, size_t base, int V, int s, float c,
                                    const float2 (&o)[12]) {
    float4 a[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) a[j] = A[base + (size_t)j * V + s];
    float v = 0.f;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const float2 o0 = o[2 * j], o1 = o[2 * j + 1];
        float4 w;
        if (DAG)
            w = make_float4(fmaf(-c, o0.x, a[j].x), fmaf(-c, o0.y, a[j].y), fmaf(-c, o1.x, a[j].z), fmaf(-c, o1.y, a[j].w));
        else
            w = make_float4(fmaf(c, a[j].x, o0.x), fmaf(c, a[j].y, o0.y), fmaf(c, a[j].z, o1.x), fmaf(c, a[j].w, o1.y));
        O[base + (size_t)j * V + s] = w;
        v += (w.x * w.x + w.y * w.y) + (w.z * w.z + w.w * w.w);
    }
    return v;
}

// One stencil step (step_update's K1 or K23): gathers G, reads A and writes O at its own
// site, block partials of |O|^2.
template <bool STAGED, bool DAG>
__device__ inline void cg_step(const float4 *__restrict__ G, const float4 *A, float4 *O,
                               const float4 *__restrict__ links, const Geom &g, const SlabWalk &w, float kappa, int N,
                               const CgFusedState *__restrict__ st, double *__restrict__ partials,
                               int *__restrict__ err) {
    extern __shared__ __align__(128) float4 stage_sm[];
    __shared__ __align__(8) uint64_t mbar;
    int q, sb, s0, nb;
    slab_rhs(w, blockIdx.x, q, sb);
    slab_block(w, sb, s0, nb);
    const int s = s0 + threadIdx.x;
    const size_t base = (size_t)q * 6 * g.V;
    if (threadIdx.x == 0 && nb > 0) {
        if (!STAGED) prefetch_planes_l2(G + base, 6, g.V, s0, nb);
        prefetch_planes_l2(A + base, 6, g.V, s0, nb);
        if (q == 0) prefetch_planes_l2(links, 12, g.V, s0, nb);
    }
    const bool ok = stage_begin<STAGED>(G + base, g, s0, nb, stage_sm, &mbar, err);
    float v[1] = {0.f};
    if ((int)threadIdx.x < nb && ok) {
        const float c = st[q].f[DAG ? 0 : 1];
        float2 o[12];
        const PackedLinks<float> lk{links, g.V};
        if constexpr (STAGED) {
            const StagedGather32 ga = staged_gather(G + base, g, s0, stage_sm);
            wilson_site_g<float, DAG, DAG>(s, g, kappa, ga, lk, o);
        } else {
            const GlobalGather<float> ga{G + base, g.V};
            wilson_site_g<float, DAG, DAG>(s, g, kappa, ga, lk, o);
        }
        v[0] = step_update<DAG>(A, O, base, g.V, s, c, o);
    }
    block_partials<1>(v, partials + (size_t)q * w.dN.div(gridDim.x) + sb, 0);
}

// K1: t = D r + beta t; partial |t|^2.  Gathers r only.
template <bool STAGED>
__global__ void __launch_bounds__(kT, STAGED ? 3 : 7)
k_cg_k1(const float4 *__restrict__ R, float4 *T, const float4 *__restrict__ links, Geom g, SlabWalk w, float kappa,
        int N, const CgFusedState *__restrict__ st, double *__restrict__ partials, int *__restrict__ err) {
    cg_step<STAGED, false>(R, T, T, links, g, w, kappa, N, st, partials, err);
}

// K23: r' = r - alpha D^dag t; partial |r'|^2.  Gathers t only.
template <bool STAGED>
__global__ void __launch_bounds__(kT, STAGED ? 3 : 7)
k_cg_k23(const float4 *__restrict__ T, const float4 *__restrict__ R, float4 *__restrict__ Rn,
         const float4 *__restrict__ links, Geom g, SlabWalk w, float kappa, int N,
         const CgFusedState *__restrict__ st, double *__restrict__ partials, int *__restrict__ err) {
    cg_step<STAGED, true>(T, R, Rn, links, g, w, kappa, N, st, partials, err);
}

struct CgResiduals {
    float4 *r[kCgBlock];
};

// The block's deferred updates, with the coefficients of k_cg_alpha: e += sum_j fe_j r_j +
// fe_p p, p = sum_j fp_j r_j + fp_p p (n float4 per right-hand side, blockIdx.y the
// right-hand side).  A streaming pass: all eight reads are issued before the arithmetic.
__global__ void __launch_bounds__(256)
k_cg_directions(CgResiduals R, float4 *__restrict__ P, float4 *__restrict__ E, const CgFusedState *__restrict__ st,
                long n) {
    const long j = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const int q = blockIdx.y;
    const size_t i = (size_t)q * n + j;
    float4 r[kCgBlock];
#pragma unroll
    for (int k = 0; k < kCgBlock; ++k) r[k] = R.r[k][i];
    const float4 p = P[i];
    float4 e = E[i];
    const float bp = st[q].fp[kCgBlock], be = st[q].fe[kCgBlock];
    float4 pn = make_float4(bp * p.x, bp * p.y, bp * p.z, bp * p.w);
    e.x = fmaf(be, p.x, e.x); e.y = fmaf(be, p.y, e.y); e.z = fmaf(be, p.z, e.z); e.w = fmaf(be, p.w, e.w);
#pragma unroll
    for (int k = 0; k < kCgBlock; ++k) {
        const float cp = st[q].fp[k], ce = st[q].fe[k];
        pn.x = fmaf(cp, r[k].x, pn.x); pn.y = fmaf(cp, r[k].y, pn.y);
        pn.z = fmaf(cp, r[k].z, pn.z); pn.w = fmaf(cp, r[k].w, pn.w);
        e.x = fmaf(ce, r[k].x, e.x); e.y = fmaf(ce, r[k].y, e.y);
        e.z = fmaf(ce, r[k].z, e.z); e.w = fmaf(ce, r[k].w, e.w);
    }
    P[i] = pn;
    E[i] = e;
}

// Block partials of |r|^2 and |s|^2 at the start of a solve (sites of the slab walk, V the
// field's plane stride)
__global__ void __launch_bounds__(kT)
k_cg_start_norms(const float4 *__restrict__ R, const float4 *__restrict__ S, int V, SlabWalk w, int N,
                 double *__restrict__ partials) {
    int q, sb, s0, nb;
    slab_rhs(w, blockIdx.x, q, sb);
    slab_block(w, sb, s0, nb);
    float v[2] = {0.f, 0.f};
    if ((int)threadIdx.x < nb) {
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const size_t i = (size_t)q * 6 * V + (size_t)c * V + s0 + threadIdx.x;
            const float4 r = R[i], s = S[i];
            v[0] += (r.x * r.x + r.y * r.y) + (r.z * r.z + r.w * r.w);
            v[1] += (s.x * s.x + s.y * s.y) + (s.z * s.z + s.w * s.w);
        }
    }
    const size_t nbq = w.dN.div(gridDim.x);
    block_partials<2>(v, partials + q * nbq + sb, N * nbq);
}

// Even-odd operator (Dhat on the even sites): each stencil is two launches, the odd
// hop (eo_hop32, gathering r or gamma5 t) and this Schur-step kernel at the even sites,
// which gathers the odd field M and makes the update of K1 or K23:
//   K1b  (DAG = false): t = (r - kappa^2 H_eo m) + beta t,                  m = H_oe r,
//   K23b (DAG = true):  r' = r - alpha gamma5 (gamma5 t - kappa^2 H_eo m),  m = H_oe gamma5 t.
template <bool DAG>
__device__ inline void cg_eo_step(const float4 *__restrict__ X, const float4 *__restrict__ M, const float4 *A,
                                  float4 *O, const float4 *__restrict__ links, const Geom &gf, const SlabWalk &w,
                                  float kappa2, int N, const CgFusedState *__restrict__ st,
                                  double *__restrict__ partials) {
    int q, sb, c0, nb;
    slab_rhs(w, blockIdx.x, q, sb);
    slab_block(w, sb, c0, nb);
    const int cb = c0 + threadIdx.x;
    const int Vh = gf.V >> 1;
    const size_t base = (size_t)q * 6 * Vh;
    if (threadIdx.x == 0 && nb > 0) {
        prefetch_planes_l2(X + base, 6, Vh, c0, nb);
        prefetch_planes_l2(A + base, 6, Vh, c0, nb);
    }
    float v[1] = {0.f};
    if ((int)threadIdx.x < nb) {
        const float c = st[q].f[DAG ? 0 : 1];
        float2 o[12];
        wilson_eo_schur_site<float, DAG, DAG>(cb, gf, kappa2, X + base, M + base, links, o);
        v[0] = step_update<DAG>(A, O, base, Vh, cb, c, o);
    }
    block_partials<1>(v, partials + (size_t)q * w.dN.div(gridDim.x) + sb, 0);
}
__global__ void __launch_bounds__(kT, 7)
k_cg_eo_k1b(const float4 *__restrict__ R, const float4 *__restrict__ M, float4 *T, const float4 *__restrict__ links,
            Geom gf, SlabWalk w, float kappa2, int N, const CgFusedState *__restrict__ st,
            double *__restrict__ partials) {
    cg_eo_step<false>(R, M, T, T, links, gf, w, kappa2, N, st, partials);
}
__global__ void __launch_bounds__(kT, 7)
k_cg_eo_k23b(const float4 *__restrict__ T, const float4 *__restrict__ M, const float4 *__restrict__ R,
             float4 *__restrict__ Rn, const float4 *__restrict__ links, Geom gf, SlabWalk w, float kappa2, int N,
             const CgFusedState *__restrict__ st, double *__restrict__ partials) {
    cg_eo_step<true>(T, M, R, Rn, links, gf, w, kappa2, N, st, partials);
}

// Threads of the one-block-per-RHS sums: enough that a thread adds a few partials only
constexpr int kSumMax = 1024;
inline int sum_threads(int nbq) { return nbq > 512 ? kSumMax : 256; }

__device__ inline double block_total(const double *__restrict__ p, int n) {
    double t = 0.0;
    for (int b = threadIdx.x; b < n; b += blockDim.x) t += p[b];
    __shared__ double sm[kSumMax / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = t;
    __syncthreads();
    double a = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x / 32); ++w) a += sm[w];
    __syncthreads();
    return a;     // valid in thread 0
}

// alpha = |r|^2 / |t|^2 (one block per right-hand side), and the block's direction
// coefficients for its iteration `slot`: p = r_slot + beta p over (r_0 .. , p_old), and
// ec += alpha p.  FP64; FP32 copies for k_cg_directions after the block's last iteration.
__global__ void __launch_bounds__(kSumMax)
k_cg_alpha(const double *__restrict__ partials, int nbq, int slot, CgFusedState *st) {
    const int q = blockIdx.x;
    const double tt = block_total(partials + (size_t)q * nbq, nbq);
    if (threadIdx.x == 0) {
        CgFusedState &s = st[q];
        const double al = tt > 0.0 ? s.gam / tt : 0.0, be = s.beta;
        s.alpha = al;
        s.f[0] = (float)al;
#pragma unroll
        for (int j = 0; j <= kCgBlock; ++j) {
            double p = 0.0, e = 0.0;
            if (j == kCgBlock) p = slot == 0 ? be : be * s.pc[j];
            else if (j < slot) p = be * s.pc[j];
            else if (j == slot) p = 1.0;
            if (slot > 0) e = s.ec[j];
            e += al * p;
            s.pc[j] = p;
            s.ec[j] = e;
            if (slot == kCgBlock - 1) {
                s.fp[j] = (float)p;
                s.fe[j] = (float)e;
            }
        }
    }
}

// |r_new|^2, |s_new|^2, beta (init: beta = 0, |s|^2 summed).  After the first step
// |s|^2 follows from the recurrence of CG on the normal equations,
//   |s_{k+1}|^2 = |s_k - alpha_k t_k|^2 = |s_k|^2 - alpha_k |r_k|^2,
// since <s_k, t_k> = <s_k, D p_k> = <r_k, p_k> = |r_k|^2 and alpha_k |t_k|^2 = |r_k|^2; it
// only steers the inner stopping test (the outer loop recomputes the residual in FP64).
__global__ void __launch_bounds__(kSumMax) k_cg_beta(const double *__restrict__ partials, int nbq, int N, int init,
                                                     CgFusedState *st) {
    const int q = blockIdx.x;
    const double rr = block_total(partials + (size_t)q * nbq, nbq);
    const double ss = init ? block_total(partials + (size_t)N * nbq + (size_t)q * nbq, nbq) : 0.0;
    if (threadIdx.x == 0) {
        CgFusedState &s = st[q];
        s.beta = (init || !(s.gam > 0.0)) ? 0.0 : rr / s.gam;
        s.ss = init ? ss : fmax(0.0, s.ss - s.alpha * s.gam);
        s.gam = rr;
        s.f[1] = (float)s.beta;
    }
}

// The slab walk of the fused kernels for an N-RHS batch (its weight: slab_walk.cuh); the
// even-odd kernels walk the even sites
SlabWalk cg_slab_walk(const Op &op, int N) {
    const Geom &g = op.eo ? op.gf : op.g;
    return make_slab_walk(g.L[0] * g.L[1] / (op.eo ? 2 : 1), g.L[2], g.L[3], N, 900.0);
}

// Whether the full-lattice kernels stage the gathered field in shared memory
// (DLZ_CG_STAGE=1, when the block's ranges fit).  Off by default: on 24^3 x 48 with 16
// right-hand sides the staged kernels took 2.17 (K23) and 1.67 ms (K1) per launch against
// 1.54 and 1.04 ms reading the neighbours from global memory (both in slabs of 4
// z-planes, with the p and e updates that K1 made then).  With 66 KB of shared memory per block only 3 blocks fit on an SM (12 warps
// against 24), and a block computes nothing until all of its copies have landed.
bool cg_staged(const Op &op) {
    if (op.eo || stage_bytes(op.g.L[0]) > 200 * 1024) return false;
    const char *env = std::getenv("DLZ_CG_STAGE");
    return env && env[0] == '1';
}

// dynamic shared memory of the staged kernels beyond 48 KB (set once, outside any graph
// capture)
int cg_prepare() {
    static int done = 0;
    if (done) return DLZ_OK;
    const int mx = 200 * 1024;
    DLZ_CUDA_TRY(cudaFuncSetAttribute(k_cg_k1<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx));
    DLZ_CUDA_TRY(cudaFuncSetAttribute(k_cg_k23<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx));
    done = 1;
    return DLZ_OK;
}

}  // namespace

long cgnr_blocks_per_rhs(const Op &op, int N) {
    return slab_blocks(cg_slab_walk(op, N));
}

int cgnr_fused_batch(Op &op, int N, const float4 *S, float4 *e, const CgBuffers &bf, CgFusedState *ms,
                     double *partials, const double *d_tol, const dlz_params &p, int &iters, GraphExec &ge) {
    const long n = 6L * op.g.V;
    const Geom g = op.g;
    const float kappa = (float)op.kappa, kappa2 = (float)(op.kappa * op.kappa);
    const float4 *links = op.gauge32.as<float4>();
    const SlabWalk w = cg_slab_walk(op, N);
    const unsigned blocks = (unsigned)(cgnr_blocks_per_rhs(op, N) * N);
    const int nbq = (int)(blocks / N), st = sum_threads(nbq);
    const bool staged = cg_staged(op);
    const int smem = staged ? stage_bytes(g.L[0]) : 0;
    int *err = op.stage_err.as<int>();
    if (staged) DLZ_TRY(cg_prepare());
    float4 *P = bf.p, *T = bf.t, *M = op.eo_tmp32.as<float4>();
    CgResiduals R;
    for (int k = 0; k < kCgBlock; ++k) R.r[k] = bf.r[k];
    // p = t = 0 so that the first K1 (beta = 0) gives t = D r and the first block p = r
    for (float4 *z : {P, T})
        DLZ_CUDA_TRY(cudaMemsetAsync(z, 0, (size_t)N * n * sizeof(float4), op.stream));
    DLZ_CUDA_TRY(cudaMemsetAsync(ms, 0, (size_t)N * sizeof(CgFusedState), op.stream));
    // r_0 = D^dag s0; gamma = |r_0|^2, |s0|^2.  s0 is not read again: its memory may be one
    // of the later residual buffers.
    DLZ_TRY(wilson32_batch(op, R.r[0], S, DLZ_DDAG, N));
    k_cg_start_norms<<<blocks, kT, 0, op.stream>>>(R.r[0], S, g.V, w, N, partials);
    k_cg_beta<<<N, st, 0, op.stream>>>(partials, nbq, N, 1, ms);
    op.prof.launches += 2;
    DLZ_CUDA_TRY(cudaGetLastError());
    // iteration `slot` of a block
    auto iteration = [&](int slot) -> int {
        const float4 *r = R.r[slot];
        float4 *rn = R.r[(slot + 1) % kCgBlock];
        // K1 moves 72 reals per site and RHS (r gathered, t read and written) + links.
        // Even-odd: the odd hop and K1b, 144 reals per even site and RHS (r gathered by the
        // hop, m written, m gathered, r and t read, t written); the pair reads every link
        // twice (192 reals per even site)
        op.prof.stencil_start(op.stream, true, g.V, N, op.eo ? 144 : 72, 1, op.eo ? 192 : -1);
        if (op.eo) {
            DLZ_TRY(eo_hop32(op, M, r, 1, false, N));
            k_cg_eo_k1b<<<blocks, kT, 0, op.stream>>>(r, M, T, links, op.gf, w, kappa2, N, ms, partials);
        } else if (staged) {
            k_cg_k1<true><<<blocks, kT, smem, op.stream>>>(r, T, links, g, w, kappa, N, ms, partials, err);
        } else {
            k_cg_k1<false><<<blocks, kT, 0, op.stream>>>(r, T, links, g, w, kappa, N, ms, partials, err);
        }
        op.prof.stencil_stop(op.stream);
        k_cg_alpha<<<N, st, 0, op.stream>>>(partials, nbq, slot, ms);
        if (slot == kCgBlock - 1) {           // before K23 writes the next block's r_0
            k_cg_directions<<<dim3((unsigned)((n + 255) / 256), N), 256, 0, op.stream>>>(R, P, e, ms, n);
            op.prof.launches++;
        }
        // K23 moves 72 reals per site and RHS (t gathered, r read, r' written) + links;
        // even-odd: 144 as K1
        op.prof.stencil_start(op.stream, true, g.V, N, op.eo ? 144 : 72, 2, op.eo ? 192 : -1);
        if (op.eo) {
            DLZ_TRY(eo_hop32(op, M, T, 1, true, N));
            k_cg_eo_k23b<<<blocks, kT, 0, op.stream>>>(T, M, r, rn, links, op.gf, w, kappa2, N, ms, partials);
        } else if (staged) {
            k_cg_k23<true><<<blocks, kT, smem, op.stream>>>(T, r, rn, links, g, w, kappa, N, ms, partials, err);
        } else {
            k_cg_k23<false><<<blocks, kT, 0, op.stream>>>(T, r, rn, links, g, w, kappa, N, ms, partials, err);
        }
        op.prof.stencil_stop(op.stream);
        k_cg_beta<<<N, st, 0, op.stream>>>(partials, nbq, N, 0, ms);
        op.prof.launches += 4;
        DLZ_CUDA_TRY(cudaGetLastError());
        return DLZ_OK;
    };
    auto six = [&]() -> int {
        for (int slot = 0; slot < kCgBlock; ++slot) DLZ_TRY(iteration(slot));
        return DLZ_OK;
    };
    std::vector<CgFusedState> hsv(N);
    std::vector<double> tol(N);
    DLZ_TRY(d2h_sync(op, tol.data(), d_tol, N * sizeof(double)));
    int it = 0;
    while (it < p.max_iter - iters) {
        DLZ_TRY(run_graph(op, ge, six));
        it += kCgBlock;
        if (it % 12 == 0 || it >= p.max_iter - iters) {
            DLZ_TRY(d2h_sync(op, hsv.data(), ms, N * sizeof(CgFusedState)));
            if (staged) {
                // a staging wait that gave up leaves its block's sums out: stop at once
                int h_err = 0;
                DLZ_TRY(d2h_sync(op, &h_err, err, sizeof(int)));
                if (h_err) break;
            }
            bool all = true;
            for (int q = 0; q < N; ++q) {
                if (!std::isfinite(hsv[q].ss) || !std::isfinite(hsv[q].gam))
                    return fail(DLZ_ERR_NONFINITE, "inner CG residual not finite");
                all = all && std::sqrt(hsv[q].ss) <= tol[q];
            }
            if (all) break;
        }
    }
    ge.sample(op.prof);
    iters += it;
    if (staged) {
        int h_err = 0;
        DLZ_TRY(d2h_sync(op, &h_err, err, sizeof(int)));
        if (h_err) {
            DLZ_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(int), op.stream));
            return fail(DLZ_ERR_DEVICE_TIMEOUT, "a staging wait of the fused CGNR kernels gave up");
        }
    }
    return DLZ_OK;
}

}  // namespace dlz
