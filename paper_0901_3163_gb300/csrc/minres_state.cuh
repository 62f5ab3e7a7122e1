// State and per-site element updates of the fused FP32 MinRes iteration (the
// inner solve of the mixed-precision D-MinRes, arXiv:0901.3163 Sec. 2), shared by
// the one-lattice kernels (minres_fused.cu) and the multi-lattice kernels
// (minres_multi.cu).
#pragma once

#include "dlz_internal.cuh"
#include "wilson_site.cuh"

namespace dlz {

// The directions d and the iterate e of MinRes,
//   d_j = (v_j - delta d_{j-1} - eps d_{j-2}) / gamma,  e += tau_j d_j,
// are linear in the Lanczos vectors and feed nothing but e, so they are brought up to date
// once per block of kMrBlock iterations (minres_directions_site): the kernel that makes the
// Givens rotation carries the FP64 coefficients of d_j, d_{j-1} and the sum of tau d over
// the block's basis (u_{-1}, u_0 .. u_4, d_A, d_B): the last Lanczos vector of the block
// before, the first five of this one, and the two directions of the last update.  Per site
// and right-hand side an iteration moves 72 (K1) + 72 (K2a) + 4 (the copy of u_5) + 48
// (288 / 6: eight vectors of the basis and e read, d_A, d_B and e written) = 196 reals,
// against 264 with d and e updated by K1 in every iteration.
//
// Buffers of a block: c[0..5] hold u_0 .. u_5, c[6] holds u_{-1}.  Iteration i gathers c[i],
// writes w to c[i + 1] (i < 5) where K2a makes u_{i+1} of it in place; after iteration 4 the
// directions are updated, which frees c[6] and c[0..4]; iteration 5 writes w to c[6], and its
// K2a puts u_6 into c[0] and a copy of u_5 into c[6]: the next block finds its vectors where
// this one did.
constexpr int kMrBlock = 6;
constexpr int kMrBasis = kMrBlock + 2;

struct FusedState {          // one per right-hand side (FP64 scalars)
    double beta, alpha, beta_next, inv_beta;
    double c, s, c_old, s_old, phibar;
    double eps, delta, gamma, tau;
    double r0;               // ||r|| at the start of the inner solve
    double cd1[kMrBasis], cd2[kMrBasis], ce[kMrBasis];   // d_j, d_{j-1}, sum of tau d
    // FP32 copies read by the element updates (no FP64 op or conversion per element):
    // f[0] 1/beta_j, f[1] beta_j, f[2] alpha, f[3] 1/beta_{j-1}
    float f[4];
    float fd1[kMrBasis], fd2[kMrBasis], fe[kMrBasis];    // the coefficients at an update
};

// buffer of iteration i of a block: gathered vector, its predecessor, w, and K2a's outputs
__host__ __device__ inline int mr_u(int i) { return i; }
__host__ __device__ inline int mr_up(int i) { return i > 0 ? i - 1 : 6; }
__host__ __device__ inline int mr_w(int i) { return i < 5 ? i + 1 : 6; }
__host__ __device__ inline int mr_out(int i) { return i < 5 ? i + 1 : 0; }

struct MinresVectors {
    float4 *c[7];            // u ring (above)
    float4 *d1, *d2, *e;     // d_A, d_B and the iterate
};

__host__ __device__ inline float4 f4(float a, float b, float c, float d) { return make_float4(a, b, c, d); }

__device__ inline void set_floats(FusedState &s) {
    s.f[0] = (float)s.inv_beta;
    s.f[1] = (float)s.beta_next;
}

// the coefficients at the start of a block's steps: d_j = d_A, d_{j-1} = d_B, nothing summed
__device__ inline void reset_directions(FusedState &s) {
#pragma unroll
    for (int i = 0; i < kMrBasis; ++i) {
        s.cd1[i] = i == kMrBlock ? 1.0 : 0.0;
        s.cd2[i] = i == kMrBlock + 1 ? 1.0 : 0.0;
        s.ce[i] = 0.0;
    }
}

// beta_1 = ||r||, rotations and directions reset; tolerances
// are relative to the normalised outer residual (norm 1)
__device__ inline void fused_init(FusedState &out, double b) {
    FusedState s0 = {};
    s0.beta_next = b;
    s0.inv_beta = b > 0 ? 1.0 / b : 0.0;
    s0.c = 1.0; s0.c_old = 1.0; s0.phibar = b; s0.gamma = 1.0; s0.r0 = 1.0;
    reset_directions(s0);
    set_floats(s0);
    out = s0;
}

__device__ inline void fused_alpha(FusedState &s, double a) {
    s.beta = s.beta_next;
    s.alpha = a;
    s.f[2] = (float)a;
}

// beta_{j+1} = sqrt(r2), the Givens rotation of step j (iteration i of its block) and the
// coefficients of its direction.  Iteration 5 belongs to the next update: basis vector 0.
// Called by all threads of a block (r2 valid in thread 0): the rotation is one thread's,
// the coefficients are one thread per basis vector (all by one thread: 10.1 us per launch
// against 6.0 before the coefficients were carried).
__device__ inline void fused_givens(FusedState &s, double r2, int i) {
    __shared__ double sh[5];
    if (threadIdx.x == 0) {
        const double bn = sqrt(r2);
        const double so = s.s_old, co = s.c_old, sc = s.s, cc = s.c, be = s.beta, al = s.alpha, ph = s.phibar;
        const double deltabar = co * be;
        const double gammabar = -sc * deltabar + cc * al;
        double gamma = hypot(gammabar, bn);
        double cn = 1.0, sn = 0.0;
        if (gamma > 0.0) { cn = gammabar / gamma; sn = bn / gamma; }
        else gamma = 1.0;            // zero right-hand side: hold a no-op
        s.tau = cn * ph;
        s.phibar = -sn * ph;
        s.eps = so * be; s.delta = cc * deltabar + sc * al; s.gamma = gamma;
        s.c_old = cc; s.s_old = sc; s.c = cn; s.s = sn;
        s.beta_next = bn;
        sh[0] = cc * deltabar + sc * al; sh[1] = so * be; sh[2] = 1.0 / gamma; sh[3] = cn * ph; sh[4] = s.inv_beta;
        s.inv_beta = bn > 0 ? 1.0 / bn : 0.0;
        s.f[3] = s.f[0];             // 1/beta_j, to scale u_j into v_j in the next step
        set_floats(s);
    }
    __syncthreads();
    const int k = threadIdx.x, slot = i < 5 ? i + 1 : 0;
    if (k < kMrBasis) {
        // d_j, d_{j-1} and the sum before this step (iteration 5 starts afresh from d_A, d_B)
        const double d1 = slot == 0 ? (k == kMrBlock ? 1.0 : 0.0) : s.cd1[k];
        const double d2 = slot == 0 ? (k == kMrBlock + 1 ? 1.0 : 0.0) : s.cd2[k];
        const double e = slot == 0 ? 0.0 : s.ce[k];
        const double d = ((k == slot ? sh[4] : 0.0) - sh[0] * d1 - sh[1] * d2) * sh[2], en = e + sh[3] * d;
        s.cd2[k] = d1;
        s.cd1[k] = d;
        s.ce[k] = en;
        s.fd1[k] = (float)d;
        s.fd2[k] = (float)d1;
        s.fe[k] = (float)en;
    }
    __syncthreads();                 // sh may be written again by the next call
}

// K1 at one site of one right-hand side (pointers at that right-hand side's
// vectors): w = Q u_j / beta_j - beta_j v_{j-1}; returns the site's share of Re <v_j, w>.
// (W may be u_{j-2}'s memory, never u_j's or u_{j-1}'s.)
__device__ inline float minres_k1_site(int s, const Geom &g, float kappa, const float4 *__restrict__ Ub,
                                       const float4 *__restrict__ Up, float4 *__restrict__ W,
                                       const float4 *__restrict__ links, const FusedState &st) {
    const float ib = st.f[0], bt = st.f[1], ibp = st.f[3];
    float2 o[12];
    wilson_site<float, false, true>(s, g, kappa, Ub, links, o);   // Q u_j
    float facc = 0.f;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        const size_t i = (size_t)c * g.V + s;
        const float4 u = Ub[i], up = Up[i];
        const float4 vj = f4(u.x * ib, u.y * ib, u.z * ib, u.w * ib);
        const float4 vp = f4(up.x * ibp, up.y * ibp, up.z * ibp, up.w * ibp);
        const float4 w = f4(o[2 * c].x * ib - bt * vp.x, o[2 * c].y * ib - bt * vp.y,
                            o[2 * c + 1].x * ib - bt * vp.z, o[2 * c + 1].y * ib - bt * vp.w);
        W[i] = w;
        facc += (vj.x * w.x + vj.y * w.y) + (vj.z * w.z + vj.w * w.w);
    }
    return facc;
}

// K2a at one site: u_{j+1} = w - (alpha_j / beta_j) u_j to Out (which may be W); returns its
// ||.||^2 share.  Copy (may be null, may be W): receives u_j.  All 6 planes are loaded before
// any store so the loads overlap.
__device__ inline float minres_k2a_site(int s, int V, const float4 *W, const float4 *Uc, float4 *Out, float4 *Copy,
                                        const FusedState &st) {
    const float al = st.f[2] * st.f[0];
    float4 w[6], v[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        w[c] = W[(size_t)c * V + s];
        v[c] = Uc[(size_t)c * V + s];
    }
    float facc = 0.f;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        const float4 t = f4(fmaf(-al, v[c].x, w[c].x), fmaf(-al, v[c].y, w[c].y),
                            fmaf(-al, v[c].z, w[c].z), fmaf(-al, v[c].w, w[c].w));
        Out[(size_t)c * V + s] = t;
        if (Copy) Copy[(size_t)c * V + s] = v[c];
        facc += (t.x * t.x + t.y * t.y) + (t.z * t.z + t.w * t.w);
    }
    return facc;
}

__device__ inline void axpy4(float c, const float4 &x, float4 &y) {
    y.x = fmaf(c, x.x, y.x); y.y = fmaf(c, x.y, y.y); y.z = fmaf(c, x.z, y.z); y.w = fmaf(c, x.w, y.w);
}

// The block's deferred update of one element (offset i of every vector): the new d_A, d_B
// and e from the basis (u_{-1}, u_0 .. u_4, d_A, d_B).  A streaming pass; every load is
// issued before the arithmetic.
__device__ inline void minres_directions_elem(const MinresVectors &b, size_t i, const FusedState &st) {
    float4 x[kMrBasis];
    x[0] = b.c[6][i];
#pragma unroll
    for (int k = 1; k < kMrBlock; ++k) x[k] = b.c[k - 1][i];
    x[kMrBlock] = b.d1[i];
    x[kMrBlock + 1] = b.d2[i];
    float4 e = b.e[i], p = f4(0.f, 0.f, 0.f, 0.f), q = p;
#pragma unroll
    for (int k = 0; k < kMrBasis; ++k) {
        axpy4(st.fd1[k], x[k], p);
        axpy4(st.fd2[k], x[k], q);
        axpy4(st.fe[k], x[k], e);
    }
    b.d1[i] = p;
    b.d2[i] = q;
    b.e[i] = e;
}

// The step that no update has taken yet when the iterations stop at a block's end (iteration
// 5: its Lanczos vector is in c[6]): e += tau d
__device__ inline void minres_last_direction(const MinresVectors &b, size_t i, const FusedState &st) {
    const float4 u = b.c[6][i], p = b.d1[i], q = b.d2[i];
    float4 e = b.e[i];
    axpy4(st.fe[0], u, e);
    axpy4(st.fe[kMrBlock], p, e);
    axpy4(st.fe[kMrBlock + 1], q, e);
    b.e[i] = e;
}

// Block sum (FP64 over the threads) of facc stored at *out by thread 0.
template <int BT>
__device__ inline void block_partial_store(float facc, double *__restrict__ out) {
    __shared__ double sm[BT / 32];
    double acc = (double)facc;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < BT / 32; ++w) t += sm[w];
        *out = t;
    }
}

// Block partials with the sum taken by the last block to finish.  Each block of
// right-hand side q stores its partial (FP64 over its threads) at slot[b], then
// counts itself in counter[q]; the block that brings the count to nbq adds all nbq
// partials of q in a fixed order and resets the counter (so the sum is deterministic
// and needs no second launch).  Returns true, with the sum in *total (thread 0), in
// that block only.  BT: threads per block.
template <int BT, typename A>
__device__ inline bool partial_then_last_sum(A facc, double *__restrict__ slot0, int b, int nbq,
                                             unsigned *__restrict__ counter, double *total) {
    __shared__ double sm[BT / 32];
    __shared__ bool last;
    double acc = (double)facc;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < BT / 32; ++w) t += sm[w];
        slot0[b] = t;
        __threadfence();
        last = (atomicAdd(counter, 1u) == (unsigned)nbq - 1u);
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    double t = 0.0;
#pragma unroll 8
    for (int i = threadIdx.x; i < nbq; i += BT) t += __ldcg(&slot0[i]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0;
#pragma unroll
        for (int w = 0; w < BT / 32; ++w) a += sm[w];
        *total = a;
        *counter = 0u;
    }
    return true;
}

}  // namespace dlz
