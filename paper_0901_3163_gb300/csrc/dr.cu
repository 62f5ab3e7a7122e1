// Lan-DR(m,k) and MinRes-DR(m,k) (arXiv:0901.3163, Sec. 1-2), one code path
// for the FP64 basis (plain form) and the FP32 basis (mixed form).
//
// Per cycle:
//   Lanczos steps j0..m-1 on the device: w = A v_j, the coupling of the
//   restart vector to the kept vectors (first step only), three-term
//   subtraction fused with the alpha_j reduction, alpha subtraction fused with
//   the beta_j reduction, periodic re-orthogonalisation against the kept
//   vectors, v_{j+1} = w / beta_j -- all scalars stay on the device;
//   the small projected problem on the host (FP64): Galerkin solve + regular
//   Ritz vectors (Lan-DR) or least squares + harmonic Ritz vectors
//   (MinRes-DR), and the restart coefficients P;
//   x += V_m y (accumulated in FP64), the true residual ||b - D x|| with the
//   FP64 stencil, and the restart V_{k+1} <- V_{m+1} P.
// The mixed form keeps the basis, the stencil and the element updates in
// FP32 and stops the DR phase once its residual stagnates at the FP32 level
// or meets tol; the caller then finishes the solve by FP64 defect correction
// over the deflation set it produced.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <complex>
#include <cstring>
#include <vector>

#include "dlz_internal.cuh"
#include "krylov_util.cuh"
#include "prec.cuh"
#include "reduce.cuh"
#include "restart_plan.h"
#include "small_dense.h"
#include "solvers.h"
#include "minres_state.cuh"
#include "wilson_site.cuh"

namespace dlz {

namespace {

// x64 += sum_j y_j V_j for an FP32 basis (accumulated in FP64)
__global__ void __launch_bounds__(128)
k_accum_x32(double2 *__restrict__ x, const float4 *__restrict__ Vb, long ld, int nin,
            const double *__restrict__ y, int V) {
    extern __shared__ float ysm[];
    for (int t = threadIdx.x; t < nin; t += blockDim.x) ysm[t] = (float)y[t];
    __syncthreads();
    const long n = 6L * V;
    const long stride = (long)gridDim.x * blockDim.x;
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        // the correction V_m y of one cycle in FP32 (the basis precision); x itself in FP64
        float a0 = 0, a1 = 0, a2 = 0, a3 = 0;
        for (int j = 0; j < nin; ++j) {
            const float4 v = Vb[(size_t)j * ld + i];
            const float c = ysm[j];
            a0 = fmaf(c, v.x, a0); a1 = fmaf(c, v.y, a1);
            a2 = fmaf(c, v.z, a2); a3 = fmaf(c, v.w, a3);
        }
        const int cpl = (int)(i / V), s = (int)(i % V);
        double2 &p = x[(size_t)(2 * cpl) * V + s];
        double2 &q = x[(size_t)(2 * cpl + 1) * V + s];
        p.x += a0; p.y += a1; q.x += a2; q.y += a3;
    }
}

template <class P> int accum_x(Op &op, double2 *x, const typename P::E *Vb, long ld, int nin, const double *dev_y);
template <> int accum_x<P64>(Op &op, double2 *x, const double2 *Vb, long ld, int nin, const double *dev_y) {
    return combine<P64>(op, x, ld, 1, Vb, ld, nin, dev_y, 1, true, true);
}
template <> int accum_x<P32>(Op &op, double2 *x, const float4 *Vb, long ld, int nin, const double *dev_y) {
    const long n = 6L * op.g.V;
    long blocks = std::min((n + 127) / 128, 152L * 8);
    k_accum_x32<<<(int)blocks, 128, nin * sizeof(float), op.stream>>>(x, Vb, ld, nin, dev_y, op.g.V);
    op.prof.launches++;
    DLZ_CUDA_TRY(cudaGetLastError());
    return DLZ_OK;
}

// v (precision P) = scale * src (FP64 internal planes)
template <class P> int from64(Op &op, typename P::E *dst, const double2 *src, double scale);
template <> int from64<P64>(Op &op, double2 *dst, const double2 *src, double scale) {
    return map(op, 12L * op.g.V, [=] __device__(long i) {
        const double2 v = src[i];
        dst[i] = make_double2(v.x * scale, v.y * scale);
    });
}
template <> int from64<P32>(Op &op, float4 *dst, const double2 *src, double scale) {
    // once per solve: the FP64 multiply keeps the scaled values exact before rounding
    const int V = op.g.V;
    return map(op, 6L * V, [=] __device__(long i) {
        const int c = (int)(i / V), s = (int)(i % V);
        const double2 a = src[(size_t)(2 * c) * V + s], b = src[(size_t)(2 * c + 1) * V + s];
        dst[i] = make_float4((float)(scale * a.x), (float)(scale * a.y), (float)(scale * b.x), (float)(scale * b.y));
    });
}

// FP64 copy of k basis vectors (for the deflation set)
template <class P> int basis_to64(Op &op, double2 *dst, const typename P::E *src, int k);
template <> int basis_to64<P64>(Op &op, double2 *dst, const double2 *src, int k) {
    DLZ_CUDA_TRY(cudaMemcpyAsync(dst, src, (size_t)k * 12 * op.g.V * sizeof(double2), cudaMemcpyDeviceToDevice, op.stream));
    return DLZ_OK;
}
template <> int basis_to64<P32>(Op &op, double2 *dst, const float4 *src, int k) {
    const long n64 = 12L * op.g.V, n32 = 6L * op.g.V;
    for (int j = 0; j < k; ++j) DLZ_TRY(convert32to64(op, dst + (size_t)j * n64, src + (size_t)j * n32));
    return DLZ_OK;
}

// ---------------------------------------------------------------- fused FP32 Lanczos step
// K1L: v_j = u_j / beta_{j-1} (written to the basis), w = A v_j - beta_{j-1} v_{j-1},
//      block partial of alpha_j = Re <v_j, w>;  A v_j = Q(in) * sin where in = u_j (A = Q)
//      or Q u_j (A = D^dag D = Q Q), so the normalisation of the previous step is folded
//      into this one instead of costing a pass of its own.
// K2aL: u_{j+1} = w - alpha_j v_j and the block partial of ||u_{j+1}||^2.
// The last block of each kernel to finish sums the partials in a fixed order and writes
// the scalar (FP64 and FP32); the block counter sits after the partials and resets itself.
constexpr int kLz = 128;

__global__ void __launch_bounds__(kLz)
k_lanczos_k1(const float4 *__restrict__ in, const float *__restrict__ sin_, const float4 *__restrict__ U,
             const float4 *__restrict__ Vp, const float *__restrict__ bprev, float4 *__restrict__ Vj,
             float4 *__restrict__ W, const float4 *__restrict__ links, Geom g, float kappa,
             double *__restrict__ partials, unsigned *__restrict__ counter, double *__restrict__ d_a,
             float *__restrict__ s_a) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    float facc = 0.f;
    if (s < g.V) {
        const float ib = *sin_, bt = *bprev;
        float2 o[12];
        wilson_site<float, false, true>(s, g, kappa, in, links, o);
        float4 u[6], vp[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            u[c] = U[(size_t)c * g.V + s];
            vp[c] = Vp[(size_t)c * g.V + s];
        }
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const float4 vj = make_float4(u[c].x * ib, u[c].y * ib, u[c].z * ib, u[c].w * ib);
            const float4 w = make_float4(o[2 * c].x * ib - bt * vp[c].x, o[2 * c].y * ib - bt * vp[c].y,
                                         o[2 * c + 1].x * ib - bt * vp[c].z, o[2 * c + 1].y * ib - bt * vp[c].w);
            Vj[(size_t)c * g.V + s] = vj;
            W[(size_t)c * g.V + s] = w;
            facc += (vj.x * w.x + vj.y * w.y) + (vj.z * w.z + vj.w * w.w);
        }
    }
    // the last block to finish forms alpha_j (FP64 and FP32 copies)
    double a;
    if (partial_then_last_sum<kLz>(facc, partials, blockIdx.x, gridDim.x, counter, &a) && threadIdx.x == 0) {
        *d_a = a;
        *s_a = (float)a;
    }
}

__global__ void __launch_bounds__(kLz)
k_lanczos_k2a(float4 *__restrict__ W, const float4 *__restrict__ Vj, const float *__restrict__ salpha, Geom g,
              double *__restrict__ partials, unsigned *__restrict__ counter, double *__restrict__ d_b,
              float *__restrict__ s_b, float *__restrict__ s_ib) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    float facc = 0.f;
    if (s < g.V) {
        const float al = *salpha;
        float4 w[6], v[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            w[c] = W[(size_t)c * g.V + s];
            v[c] = Vj[(size_t)c * g.V + s];
        }
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const float4 t = make_float4(fmaf(-al, v[c].x, w[c].x), fmaf(-al, v[c].y, w[c].y),
                                         fmaf(-al, v[c].z, w[c].z), fmaf(-al, v[c].w, w[c].w));
            W[(size_t)c * g.V + s] = t;
            facc += (t.x * t.x + t.y * t.y) + (t.z * t.z + t.w * t.w);
        }
    }
    // the last block to finish forms beta_{j+1} = ||u_{j+1}|| (and 1/beta in FP32)
    double r2;
    if (partial_then_last_sum<kLz>(facc, partials, blockIdx.x, gridDim.x, counter, &r2) && threadIdx.x == 0) {
        const double b = sqrt(r2);
        *d_b = b;
        *s_b = (float)b;
        *s_ib = (float)(1.0 / b);
    }
}

// Block partials that the fused kernels of a step write (the counter sits after them): at most
// 6 per chunk of 128 sites (k_reorth_norm has 6 per 256, lanczos_fused_step 2 per 128)
inline long lz_partials(int V) { return 6L * ((V + kLz - 1) / kLz); }

// The stencil of an unfused FP32 step with the three-term subtraction: W = Q in - beta_{j-1}
// v_{j-1} (Vp null: none) and alpha_j = Re <v_j, W> by the last block, which saves a pass over
// three vectors.  Bound by the gathers of a single vector.  With k_reorth_norm, Lan-DR(100, 40)
// and D-CG on 4 right-hand sides of 16^3 x 32 take 385.3 ms in place of 393.1.
__global__ void __launch_bounds__(kLz, 7)
k_lanczos_apply(const float4 *__restrict__ in, const float4 *__restrict__ Vj, const float4 *__restrict__ Vp,
                const float *__restrict__ bprev, float4 *__restrict__ W, const float4 *__restrict__ links, Geom g,
                float kappa, double *__restrict__ partials, unsigned *__restrict__ counter, double *__restrict__ d_a,
                float *__restrict__ s_a) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    float facc = 0.f;
    if (s < g.V) {
        float2 o[12];
        wilson_site<float, false, true>(s, g, kappa, in, links, o);
        const float bt = Vp ? *bprev : 0.f;
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const size_t i = (size_t)c * g.V + s;
            float4 w = make_float4(o[2 * c].x, o[2 * c].y, o[2 * c + 1].x, o[2 * c + 1].y);
            if (Vp) w = P32::axpy(-bt, Vp[i], w);
            W[i] = w;
            facc += P32::rdot(Vj[i], w);
        }
    }
    double a;
    if (partial_then_last_sum<kLz>(facc, partials, blockIdx.x, gridDim.x, counter, &a) && threadIdx.x == 0) {
        *d_a = a;
        *s_a = (float)a;
    }
}

// The end of a re-orthogonalised FP32 step: W += sum_l c_l V_l (complex c_l, l < nv), and
// beta_{j+1} = ||W|| by the last block (the combine kernel and a reduction in one pass).  A
// block has one plane of kRn sites, the planes of a chunk of sites follow one another, and the
// chunks go from the last to the first: the multi-dot before it has just read the last chunks of
// all vectors, and L2 still holds about a fifth of them (40 vectors of 16^3 x 32: multi-dot and
// this kernel 201 us with both in the same order and groups of 8 vectors, 173 us so: 94 + 79;
// Lan-DR(100, 40) and D-CG on 4 right-hand sides 385 -> 358 ms).  Eight
// loads in flight per thread; 16 take registers that cost more blocks (78 -> 104 us).
constexpr int kRn = 256;
static_assert(kMaxM * sizeof(float2) <= 48 * 1024, "the coefficients of the kept vectors in shared memory");
__global__ void __launch_bounds__(kRn)
k_reorth_norm(float4 *__restrict__ W, const float4 *__restrict__ V, long ld, int nv, const double2 *__restrict__ coef,
              int sites, double *__restrict__ partials, unsigned *__restrict__ counter, double *__restrict__ d_b,
              float *__restrict__ s_b, float *__restrict__ s_ib) {
    extern __shared__ float2 cs[];
    for (int t = threadIdx.x; t < nv; t += kRn) cs[t] = make_float2((float)coef[t].x, (float)coef[t].y);
    __syncthreads();
    const int b = gridDim.x - 1 - blockIdx.x, s = b / 6 * kRn + threadIdx.x;
    float facc = 0.f;
    if (s < sites) {
        const long i = (long)(b % 6) * sites + s;
        float4 a = P32::zero();
#pragma unroll 8
        for (int l = 0; l < nv; ++l) P32::cacc(cs[l], V[(size_t)l * ld + i], a);
        const float4 w = P32::add(W[i], a);
        W[i] = w;
        facc = P32::nrm(w);
    }
    double r2;
    if (partial_then_last_sum<kRn>(facc, partials, b, gridDim.x, counter, &r2) && threadIdx.x == 0) {
        const double b = sqrt(r2);
        *d_b = b;
        *s_b = (float)b;
        *s_ib = (float)(1.0 / b);
    }
}

// one fused FP32 Lanczos step (see above)
int lanczos_fused_step(Op &op, bool ddagd, const float4 *u, const float *s_ib_prev, const float4 *vp,
                       const float *s_b_prev, float4 *vj, float4 *w_out, float4 *tmp, double *partials,
                       double *d_a, float *s_a, double *d_b, float *s_b, float *s_ib) {
    const Geom g = op.g;
    const unsigned blocks = (unsigned)((g.V + kLz - 1) / kLz);
    const float4 *in = u;
    if (ddagd) {
        DLZ_TRY(wilson32(op, tmp, u, DLZ_Q));      // first factor of Q Q
        in = tmp;
    }
    op.prof.stencil_start(op.stream, true, g.V, 1, 96, 1);
    unsigned *counter = reinterpret_cast<unsigned *>(partials + lz_partials(g.V));
    k_lanczos_k1<<<blocks, kLz, 0, op.stream>>>(in, s_ib_prev, u, vp, s_b_prev, vj, w_out, op.gauge32.as<float4>(),
                                                g, (float)op.kappa, partials, counter, d_a, s_a);
    op.prof.stencil_stop(op.stream);
    k_lanczos_k2a<<<blocks, kLz, 0, op.stream>>>(w_out, vj, s_a, g, partials + blocks, counter, d_b, s_b, s_ib);
    op.prof.launches += 2;
    DLZ_CUDA_TRY(cudaGetLastError());
    return DLZ_OK;
}

}  // namespace

template <class P>
int dr_solve_t(Op &op, bool harmonic, const double2 *b_in, double2 *x_out, const dlz_params &p,
               dlz_defl_s **defl_out, dlz_stats &st) {
    typedef typename P::E E;
    const int m = p.m, k = p.k;
    const long n = P::nel(op);
    const long n64 = 12L * op.g.V;
    const int which = harmonic ? DLZ_Q : DLZ_DDAGD;
    const int mv_per = harmonic ? 1 : 2;
    DevBuf Va, Vb, w, tmp, bb, bp, x, Dx, scal, coef;
    DLZ_TRY(Va.alloc((size_t)(m + 1) * n * sizeof(E)));
    DLZ_TRY(Vb.alloc((size_t)(m + 1) * n * sizeof(E)));
    DLZ_TRY(w.alloc(n * sizeof(E)));
    DLZ_TRY(tmp.alloc(n * sizeof(E)));
    DevBuf w2, fpart;                          // fused FP32 steps: second work vector, partials
    if (P::kF32) {
        DLZ_TRY(reserve_multidot(op, k));
        DLZ_TRY(w2.alloc(n * sizeof(E)));
        DLZ_TRY(fpart.alloc((lz_partials(op.g.V) + 8) * sizeof(double)));
        DLZ_CUDA_TRY(cudaMemsetAsync(fpart.p, 0, fpart.bytes, op.stream));
    }
    DLZ_TRY(bb.alloc(n64 * sizeof(double2)));
    DLZ_TRY(bp.alloc(n64 * sizeof(double2)));
    DLZ_TRY(x.alloc(n64 * sizeof(double2)));
    DLZ_TRY(Dx.alloc(n64 * sizeof(double2)));
    DLZ_TRY(scal.alloc((size_t)(2 * m + 8) * sizeof(double)));
    DLZ_TRY(coef.alloc((size_t)(m + 1) * (m + 1) * sizeof(double2)));
    DevBuf gcoef;                               // the restart GEMM's coefficient matrix
    DLZ_TRY(gcoef.alloc((size_t)(m + 1) * (k + 1) * sizeof(double)));
    double *d_alpha = scal.as<double>(), *d_beta = d_alpha + m, *d_norm = d_beta + m;
    // the same scalars in the element-update precision (written by the finishers)
    typedef typename P::S S;
    DevBuf sscal;
    DLZ_TRY(sscal.alloc((size_t)(3 * m + 4) * sizeof(S)));
    S *s_alpha = sscal.as<S>(), *s_beta = s_alpha + m, *s_invbeta = s_beta + m, *s_nrm = s_invbeta + m;
    HostScratch hs;
    DLZ_TRY(hs.ensure(3 * m + 8));

    DLZ_TRY(v64::copy(op, bb.as<double2>(), b_in));
    // right-hand side of the hermitian system: gamma5 b (Q) or D^dag b (D^dag D), in FP64
    if (harmonic) DLZ_TRY(v64::gamma5(op, bp.as<double2>(), bb.as<double2>()));
    else DLZ_TRY(wilson64(op, bp.as<double2>(), bb.as<double2>(), DLZ_DDAG));
    if (!harmonic) st.mvps += 1;
    DLZ_TRY(v64::zero(op, x.as<double2>()));
    DLZ_TRY(v64::norm2_diff(op, bb.as<double2>(), nullptr, d_norm));
    DLZ_TRY(v64::norm2_diff(op, bp.as<double2>(), nullptr, d_norm + 1));
    DLZ_TRY(d2h_sync(op, hs.p, d_norm, 2 * sizeof(double)));
    const double bnorm = std::sqrt(hs.p[0]), beta0 = std::sqrt(hs.p[1]);
    if (!std::isfinite(bnorm) || !std::isfinite(beta0)) return fail(DLZ_ERR_NONFINITE, "right-hand side is not finite");
    if (bnorm == 0.0) {
        DLZ_TRY(v64::copy(op, x_out, x.as<double2>()));
        st.converged = 1;
        st.true_residual = 0.0;
        if (defl_out) *defl_out = nullptr;
        return DLZ_OK;
    }
    E *V = Va.as<E>(), *Vn = Vb.as<E>();
    DLZ_TRY(from64<P>(op, V, bp.as<double2>(), 1.0 / beta0));   // v_1 = b' / ||b'||
    std::vector<double> T((size_t)(m + 1) * m, 0.0), c(m + 1, 0.0);
    c[0] = beta0;
    int j0 = 0;
    double Anorm = 0.0;
    long long mvps_at_conv = -1;
    bool converged = false;
    int cycle = 0;
    double *coefr = coef.as<double>();
    std::vector<double> hist;
    GraphExec g_first, g_a, g_b;
    // DLZ_TRACE=1: per-phase wall times on stderr (diagnostics)
    const char *trace_env = std::getenv("DLZ_TRACE");
    const bool trace = trace_env && trace_env[0] == '1';
    // Lan-DR: once kept regular Ritz vectors converge (the over-solve), new Lanczos
    // vectors lose orthogonality to them within a few steps (the loss grows like
    // rounding * ||A|| / Ritz residual), and a period of 10 lets spurious Ritz values
    // (negative ones, for the positive definite D^dag D) into the kept set: seen at
    // 16^4 after 8 cycles in FP64 and after 3 in FP32.  Lan-DR therefore
    // re-orthogonalises against the kept vectors at every step.
    const int rperiod = (!harmonic && p.reorth_period > 0) ? 1 : p.reorth_period;
    double t_lanczos = 0, t_host = 0, t_restart = 0;
    auto now = [] { return std::chrono::steady_clock::now(); };
    auto secs = [](std::chrono::steady_clock::time_point a, std::chrono::steady_clock::time_point b) {
        return std::chrono::duration<double>(b - a).count();
    };
    for (cycle = 0; cycle < p.max_cycles; ++cycle) {
        const auto tc0 = now();
        // ---------------- Lanczos steps j0 .. m-1
        if (j0 > 0) {
            std::vector<double> cp(j0);                 // coupling of v_{k+1} to the kept vectors
            for (int i = 0; i < j0; ++i) cp[i] = -T[(size_t)j0 * m + i];
            DLZ_TRY(h2d(op, coefr, cp.data(), j0 * sizeof(double)));
        }
        auto lanczos_steps = [&]() -> int {
        // FP32: steps other than the first of a cycle and the re-orthogonalisation steps
        // run fused (lanczos_fused_step); `ucur` holds the unnormalised u_j, and V[j] is
        // written lazily (by the next fused step, or by a scaling pass before an unfused one)
        E *ucur = w.as<E>(), *uoth = P::kF32 ? w2.as<E>() : nullptr;
        bool vmat = true;
        for (int j = j0; j < m; ++j) {
            const bool reorth_j = (j0 > 0) && rperiod > 0 && ((j - j0) % rperiod == 0);
            if constexpr (P::kF32) {
                // (an even-odd operator has no fused step: its stencil is two launches)
                if (j > j0 && !reorth_j && !op.eo) {
                    DLZ_TRY(lanczos_fused_step(op, !harmonic, ucur, s_invbeta + (j - 1), V + (size_t)(j - 1) * n,
                                               s_beta + (j - 1), V + (size_t)j * n, uoth, tmp.as<E>(),
                                               fpart.as<double>(), d_alpha + j, s_alpha + j, d_beta + j,
                                               s_beta + j, s_invbeta + j));
                    std::swap(ucur, uoth);
                    vmat = false;
                    continue;
                }
                if (!vmat) {
                    E *vjm = V + (size_t)j * n;
                    const E *uc = ucur;
                    const S *ibp = s_invbeta + (j - 1);
                    DLZ_TRY(map(op, n, [=] __device__(long i) { vjm[i] = P::scal(*ibp, uc[i]); }));
                    vmat = true;
                }
            }
            E *vj = V + (size_t)j * n, *wv = ucur;
            if constexpr (P::kF32) {
                // a re-orthogonalised step (Lan-DR: every step) in five passes
                if (reorth_j && j > j0 && !op.eo) {
                    const float4 *in = vj;
                    if (!harmonic) {
                        DLZ_TRY(wilson32(op, tmp.as<E>(), vj, DLZ_Q));
                        in = tmp.as<E>();
                    }
                    const unsigned nb = (unsigned)((op.g.V + kLz - 1) / kLz), nb2 = 6u * (unsigned)((op.g.V + kRn - 1) / kRn);
                    double *part = fpart.as<double>();
                    unsigned *counter = reinterpret_cast<unsigned *>(part + lz_partials(op.g.V));
                    op.prof.stencil_start(op.stream, true, op.g.V, 1, 96, 1);
                    k_lanczos_apply<<<nb, kLz, 0, op.stream>>>(in, vj, V + (size_t)(j - 1) * n, s_beta + (j - 1), wv,
                                                               op.gauge32.as<float4>(), op.g, (float)op.kappa, part,
                                                               counter, d_alpha + j, s_alpha + j);
                    op.prof.stencil_stop(op.stream);
                    const S *saj = s_alpha + j, *sib = s_invbeta + j;
                    DLZ_TRY(map(op, n, [=] __device__(long i) { wv[i] = P::axpy(-*saj, vj[i], wv[i]); }));
                    double2 *cd = coef.as<double2>() + (m + 1);   // after the coupling block
                    DLZ_TRY(multidot<P>(op, V, n, j0, wv, cd, -1.0));
                    k_reorth_norm<<<nb2, kRn, j0 * sizeof(float2), op.stream>>>(wv, V, n, j0, cd, op.g.V, part, counter,
                                                                               d_beta + j, s_beta + j, s_invbeta + j);
                    op.prof.launches += 2;
                    DLZ_CUDA_TRY(cudaGetLastError());
                    E *vn = V + (size_t)(j + 1) * n;
                    DLZ_TRY(map(op, n, [=] __device__(long i) { vn[i] = P::scal(*sib, wv[i]); }));
                    vmat = true;
                    continue;
                }
            }
            // FP64; FP32: a cycle's first step, and every step of an even-odd operator
            DLZ_TRY(P::apply(op, wv, vj, which, tmp.as<E>()));
            if (j == j0 && j0 > 0) DLZ_TRY(combine<P>(op, wv, n, 1, V, n, j0, coefr, 1, true, true));
            const E *vprev = (j > j0) ? V + (size_t)(j - 1) * n : nullptr;
            const S *bprev = (j > j0) ? s_beta + (j - 1) : nullptr;
            double *aj = d_alpha + j, *bj = d_beta + j;
            S *saj = s_alpha + j, *sbj = s_beta + j, *sib = s_invbeta + j;
            DLZ_TRY(red<P, 1>(op, n, [=] __device__(long i, typename P::Acc (&acc)[1]) {
                E x_ = wv[i];
                if (vprev) {
                    x_ = P::axpy(-*bprev, vprev[i], x_);
                    wv[i] = x_;
                }
                acc[0] += P::rdot(vj[i], x_);
            }, [=] __device__(const double *r) { *aj = r[0]; *saj = (S)r[0]; }));
            const bool reorth = reorth_j;
            if (reorth) {
                DLZ_TRY(map(op, n, [=] __device__(long i) { wv[i] = P::axpy(-*saj, vj[i], wv[i]); }));
                double2 *cd = coef.as<double2>() + (m + 1);   // after the coupling block
                DLZ_TRY(multidot<P>(op, V, n, j0, wv, cd, -1.0));
                DLZ_TRY(combine<P>(op, wv, n, 1, V, n, j0, cd, 1, false, true));
                DLZ_TRY(red<P, 1>(op, n, [=] __device__(long i, typename P::Acc (&acc)[1]) { acc[0] += P::nrm(wv[i]); },
                                  [=] __device__(const double *r) {
                                      const double b = sqrt(r[0]);
                                      *bj = b; *sbj = (S)b; *sib = (S)(1.0 / b);
                                  }));
            } else {
                DLZ_TRY(red<P, 1>(op, n, [=] __device__(long i, typename P::Acc (&acc)[1]) {
                    const E x_ = P::axpy(-*saj, vj[i], wv[i]);
                    wv[i] = x_;
                    acc[0] += P::nrm(x_);
                }, [=] __device__(const double *r) {
                    const double b = sqrt(r[0]);
                    *bj = b; *sbj = (S)b; *sib = (S)(1.0 / b);
                }));
            }
            E *vn = V + (size_t)(j + 1) * n;
            DLZ_TRY(map(op, n, [=] __device__(long i) { vn[i] = P::scal(*sib, wv[i]); }));
            vmat = true;
        }
        if (!vmat) {                           // v_{m+1} after a fused last step
            E *vm = V + (size_t)m * n;
            const E *uc = ucur;
            const S *ibp = s_invbeta + (m - 1);
            DLZ_TRY(map(op, n, [=] __device__(long i) { vm[i] = P::scal(*ibp, uc[i]); }));
        }
        return DLZ_OK;
        };
        // the steps of a cycle are the same kernels with the same arguments from one
        // cycle to the next (per basis buffer): capture them once, replay them
        GraphExec &ge = (j0 == 0) ? g_first : (V == Va.as<E>() ? g_a : g_b);
        DLZ_TRY(run_graph(op, ge, lanczos_steps));
        st.mvps += (long long)(m - j0) * mv_per;
        st.iterations += m - j0;
        // ---------------- small problem on the host
        DLZ_TRY(d2h_sync(op, hs.p, d_alpha, 2 * m * sizeof(double)));
        ge.sample(op.prof);
        double tmax = 0.0;
        for (int j = j0; j < m; ++j) {
            const double a = hs.p[j], bt = hs.p[m + j];
            if (!std::isfinite(a) || !std::isfinite(bt)) return fail(DLZ_ERR_NONFINITE, "Lanczos coefficients not finite");
            T[(size_t)j * m + j] = a;
            T[(size_t)(j + 1) * m + j] = bt;
            if (j + 1 < m) T[(size_t)j * m + j + 1] = bt;
            if (j > j0) T[(size_t)(j - 1) * m + j] = T[(size_t)j * m + j - 1];
            tmax = std::max(tmax, std::fabs(a));
        }
        for (int i = 0; i < j0; ++i) T[(size_t)i * m + j0] = T[(size_t)j0 * m + i];
        for (int j = j0; j < m; ++j)
            if (hs.p[m + j] <= 1e-14 * std::max(tmax, Anorm))
                return fail(DLZ_ERR_BREAKDOWN, "Lanczos breakdown (invariant subspace)");
        const auto tc1 = now();
        RestartPlan pl;
        DLZ_TRY(plan_solve(harmonic, m, T, c, pl));
        // ---------------- x += V_m y ; true residual ||b - D x|| / ||b|| in FP64 (on the
        // GPU while the host solves the eigenproblem)
        std::memcpy(hs.p + 2 * m, pl.y.data(), m * sizeof(double));     // pinned staging
        DLZ_TRY(h2d(op, coefr, hs.p + 2 * m, m * sizeof(double)));
        DLZ_TRY(accum_x<P>(op, x.as<double2>(), V, n, m, coefr));
        DLZ_TRY(wilson64(op, Dx.as<double2>(), x.as<double2>(), DLZ_D));
        st.mvps += 1;
        DLZ_TRY(v64::norm2_diff(op, bb.as<double2>(), Dx.as<double2>(), d_norm + 2));
        DLZ_TRY(plan_finish(harmonic, m, k, T, Anorm, pl));
        const auto tc2 = now();
        // FP32 basis: Ritz residuals below ~1e-5 ||A|| are under its rounding level
        const double tol_eig = p.tol_eig > 0 ? p.tol_eig : (P::kF32 ? 1e-5 : 1e-10) * Anorm;
        // ---------------- restart: V_{k+1} <- V_{m+1} P
        // FP32: the tensor-core product (tc_gemm.cu: tcgen05, 3xTF32, FP32 accuracy);
        // FP64: the combine kernel (FP64-ALU-bound; the plain-form step took 39.1 s with
        // cuBLAS DGEMM against 36.8 s with it)
        if constexpr (P::kF32) {
            DLZ_TRY(tc_combine32(op.tc, op.stream, reinterpret_cast<float *>(Vn), 4 * n, reinterpret_cast<const float *>(V),
                                 4 * n, m + 1, 4 * n, pl.P.data(), k + 1, false, &op.prof.launches));
        } else {
            DLZ_TRY(h2d(op, gcoef.p, pl.P.data(), pl.P.size() * sizeof(double)));
            DLZ_TRY(combine<P>(op, Vn, n, k + 1, V, n, m + 1, gcoef.p, k + 1, true, false));
        }
        if (rperiod > 0) {
            // the vector carried across the restart joins the periodic re-orthogonalisation
            E *vk = Vn + (size_t)k * n;
            double2 *cd = coef.as<double2>() + (size_t)(m + 1) * (k + 1);
            DLZ_TRY(multidot<P>(op, Vn, n, k, vk, cd, -1.0));
            DLZ_TRY(combine<P>(op, vk, n, 1, Vn, n, k, cd, 1, false, true));
            S *nrm = s_nrm;
            DLZ_TRY(red<P, 1>(op, n, [=] __device__(long i, typename P::Acc (&acc)[1]) { acc[0] += P::nrm(vk[i]); },
                              [=] __device__(const double *r) { *nrm = (S)(1.0 / sqrt(r[0])); }));
            DLZ_TRY(map(op, n, [=] __device__(long i) { vk[i] = P::scal(*nrm, vk[i]); }));
        }
        DLZ_TRY(d2h_sync(op, hs.p, d_norm + 2, sizeof(double)));
        const auto tc3 = now();
        t_lanczos += secs(tc0, tc1);
        t_host += secs(tc1, tc2);
        t_restart += secs(tc2, tc3);
        const double rel = std::sqrt(hs.p[0]) / bnorm;
        st.true_residual = rel;
        if (!std::isfinite(rel)) return fail(DLZ_ERR_NONFINITE, "residual is not finite");
        hist.push_back(rel);
        if (trace) {
            double bmin = 1e300, tmin = 1e300, tmax = -1e300, rmax = 0.0;
            for (int j = j0; j < m; ++j) bmin = std::min(bmin, T[(size_t)(j + 1) * m + j]);
            for (int l = 0; l < k; ++l) {
                tmin = std::min(tmin, pl.theta[l]);
                tmax = std::max(tmax, pl.theta[l]);
                rmax = std::max(rmax, pl.res[l]);
            }
            std::fprintf(stderr, "[dlz]   cycle %d rel %.3e beta_min %.3e theta [%.4e, %.4e] ritz_res_max %.3e\n",
                         cycle, rel, bmin, tmin, tmax, rmax);
        }
        bool lin_ok = rel <= p.tol;
        if (P::kF32 && !lin_ok && hist.size() >= 4) {
            // FP32 basis: the residual stalls near eps_32 * cond; stop the DR phase there
            const double prev = hist[hist.size() - 4];
            lin_ok = rel > 0.5 * prev && rel < 1e-3;
        }
        if (lin_ok && mvps_at_conv < 0) mvps_at_conv = st.mvps;
        bool eig_ok = true;
        for (int l = 0; l < k; ++l) eig_ok = eig_ok && pl.res[l] <= tol_eig;
        const bool over = mvps_at_conv >= 0 && (double)(st.mvps - mvps_at_conv) >= p.oversolve * (double)mvps_at_conv;
        std::swap(V, Vn);
        T.swap(pl.Tn);
        c.swap(pl.cn);
        j0 = k;
        // eigensolver use: the kept pairs alone decide
        if (p.eig_only ? eig_ok : (lin_ok && (eig_ok || over))) {
            converged = true;
            ++cycle;
            break;
        }
    }
    st.cycles = cycle;
    st.converged = p.eig_only ? (converged ? 1 : 0) : ((converged && st.true_residual <= p.tol) ? 1 : 0);
    DLZ_TRY(v64::copy(op, x_out, x.as<double2>()));
    const auto td0 = now();
    if (defl_out) {
        DevBuf V64;
        double2 *vk64;
        if (P::kF32) {
            DLZ_TRY(V64.alloc((size_t)k * n64 * sizeof(double2)));
            DLZ_TRY(basis_to64<P>(op, V64.as<double2>(), V, k));
            vk64 = V64.as<double2>();
        } else {
            vk64 = reinterpret_cast<double2 *>(V);
        }
        // FP64 basis: H = V_k^dag A V_k is the k x k block of the restarted T (the
        // Lanczos relation holds to FP64 rounding).  FP32 basis: T carries the FP32
        // rounding of the stencil and the vector updates (~1e-7 ||A||), as large as the
        // smallest eigenvalues of D^dag D near the critical kappa (~1e-6 at
        // sigma_min = 1e-3), so H is formed explicitly in FP64 from the FP64 copy of the
        // kept vectors: the Galerkin projection of D-CG / D-MinRes is then exact for the
        // kept subspace (k FP64 products with A)
        std::vector<double> Hk((size_t)k * k);
        for (int i = 0; i < k; ++i)
            for (int j = 0; j < k; ++j) Hk[(size_t)i * k + j] = T[(size_t)i * m + j];
        DLZ_TRY(build_deflation(op, which, vk64, k, defl_out, P::kF32 ? nullptr : Hk.data()));
    }
    DLZ_CUDA_TRY(cudaStreamSynchronize(op.stream));
    if (trace)
        std::fprintf(stderr, "[dlz] DR(%s, %s) cycles %d steps %d: lanczos %.4f s, small problem %.4f s, "
                     "restart+residual %.4f s, deflation set %.4f s\n", harmonic ? "MinRes" : "Lan",
                     P::kF32 ? "f32" : "f64", cycle, st.iterations, t_lanczos, t_host, t_restart, secs(td0, now()));
    return converged ? DLZ_OK : DLZ_ERR_NOT_CONVERGED;
}

// Kernel attributes that must be set before any graph capture.
int prepare_kernels(Op &op) {
    DLZ_TRY(combine<P64>(op, nullptr, 0, 0, nullptr, 0, 0, nullptr, 0, true, false));
    DLZ_TRY(combine<P32>(op, nullptr, 0, 0, nullptr, 0, 0, nullptr, 0, true, false));
    DLZ_TRY(combine64(op, nullptr, 0, 0, nullptr, 0, 0, nullptr, 0, true, false));
    return DLZ_OK;
}

int dr_solve(Op &op, bool harmonic, const double2 *b, double2 *x, const dlz_params &p,
             dlz_defl_s **defl_out, dlz_stats &st) {
    if (p.eig_only) {
        // eigensolver use: the restart cycles only, no finishing solve
        if (p.precision == DLZ_F64) return dr_solve_t<P64>(op, harmonic, b, x, p, defl_out, st);
        return dr_solve_t<P32>(op, harmonic, b, x, p, defl_out, st);
    }
    if (p.precision == DLZ_F64) {
        if (!p.finish) return dr_solve_t<P64>(op, harmonic, b, x, p, defl_out, st);
        // restart cycles, then (if they ended short of tol) D-MinRes / D-CG from x
        dlz_defl_s *d = nullptr;
        int rc = dr_solve_t<P64>(op, harmonic, b, x, p, &d, st);
        if (rc == DLZ_ERR_NOT_CONVERGED && d && st.true_residual > p.tol) {
            dlz_stats s2;
            std::memset(&s2, 0, sizeof(s2));
            rc = harmonic ? dminres64(op, d, b, x, p, s2, x) : dcg64(op, d, b, x, p, s2, x);
            st.iterations += s2.iterations;
            st.mvps += s2.mvps;
            st.true_residual = s2.true_residual;
            st.converged = s2.converged;
        } else if (rc == DLZ_ERR_NOT_CONVERGED && st.true_residual <= p.tol) {
            st.converged = 1;
            rc = DLZ_OK;
        }
        if (defl_out) *defl_out = d;
        else delete d;
        return rc;
    }
    // mixed form: FP32 DR phase, then FP64 defect correction over its deflation set
    dlz_defl_s *d = nullptr;
    int rc = dr_solve_t<P32>(op, harmonic, b, x, p, &d, st);
    if (rc != DLZ_OK && rc != DLZ_ERR_NOT_CONVERGED) {
        delete d;
        return rc;
    }
    if (st.true_residual > p.tol) {
        dlz_stats s2;
        std::memset(&s2, 0, sizeof(s2));
        rc = dsolve_mixed_batch(op, d, harmonic, b, x, 1, p, &s2, x);
        st.iterations += s2.iterations;
        st.mvps += s2.mvps;
        st.true_residual = s2.true_residual;
        st.converged = s2.converged;
    } else {
        st.converged = 1;
        rc = DLZ_OK;
    }
    if (defl_out) *defl_out = d;
    else delete d;
    return rc;
}

}  // namespace dlz
