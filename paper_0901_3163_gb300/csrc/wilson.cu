// Wilson-Dirac stencil kernels (Sec. 2 of arXiv:0901.3163: the Wilson matrix M,
// used as gamma5 M and M^dagger M) and the layout conversions around them.
//
// One thread per lattice site.  Spinor and link planes are component-major,
// so each load instruction of a warp reads consecutive 16-byte (FP64 double2,
// FP32 float4) or 8-byte (FP32 link float2) words; the eight neighbour
// spinors of a site are re-read from L1/L2 (the time neighbour of site s is
// Lx*Ly*Lz sites away: a window of a few MB that stays in the 129 MB L2), so
// DRAM sees each spinor and link about once per application.
#include <algorithm>
#include <cstdint>

#include "dlz_internal.cuh"
#include "slab_walk.cuh"
#include "wilson_site.cuh"

namespace dlz {

namespace {

constexpr int kStencilThreads32 = 128;

template <typename T, bool G5IN, bool G5OUT>
__global__ void __launch_bounds__(128)
k_wilson(typename Field<T>::vec *__restrict__ out, const typename Field<T>::vec *__restrict__ in,
         const typename Link<T>::vec *__restrict__ U, Geom g, T kappa) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.V) return;
    cx<T> o[12];
    wilson_site<T, G5IN, G5OUT>(s, g, kappa, in, U, o);
    Field<T>::store(out, g.V, s, o);
}

// N right-hand sides stored one after another (each nel elements); consecutive
// blocks take the same sites of different right-hand sides, so the links they
// share are read from L2 (and DRAM) once.
template <typename T, bool G5IN, bool G5OUT>
__device__ inline void wilson_batch_body(typename Field<T>::vec *__restrict__ out,
                                         const typename Field<T>::vec *__restrict__ in,
                                         const typename Link<T>::vec *__restrict__ U, const Geom &g, T kappa,
                                         int nrhs, long nel) {
    const int r = blockIdx.x % nrhs;
    const int s = (blockIdx.x / nrhs) * blockDim.x + threadIdx.x;
    if (s >= g.V) return;
    cx<T> o[12];
    wilson_site<T, G5IN, G5OUT>(s, g, kappa, in + (size_t)r * nel, U, o);
    Field<T>::store(out + (size_t)r * nel, g.V, s, o);
}

template <typename T, bool G5IN, bool G5OUT>
__global__ void __launch_bounds__(128)
k_wilson_batch(typename Field<T>::vec *__restrict__ out, const typename Field<T>::vec *__restrict__ in,
               const typename Link<T>::vec *__restrict__ U, Geom g, T kappa, int nrhs, long nel) {
    wilson_batch_body<T, G5IN, G5OUT>(out, in, U, g, kappa, nrhs, nel);
}

// FP32: at most 80 registers (6 blocks per SM), measured 5% faster at 11-16
// right-hand sides than without the bound.  Blocks of 128 sites in the slab walk
// (slab_walk.cuh).
template <bool G5IN, bool G5OUT>
__global__ void __launch_bounds__(kSlabBlock, 6)
k_wilson_batch32(float4 *__restrict__ out, const float4 *__restrict__ in, const float4 *__restrict__ U, Geom g,
                 SlabWalk w, float kappa, int nrhs, long nel) {
    int r, sb, s0, nb;
    slab_rhs(w, blockIdx.x, r, sb);
    slab_block(w, sb, s0, nb);
    if (threadIdx.x == 0 && nb > 0) {
        prefetch_planes_l2(in + (size_t)r * nel, 6, g.V, s0, nb);
        if (r == 0) prefetch_planes_l2(U, 12, g.V, s0, nb);
    }
    if ((int)threadIdx.x >= nb) return;
    const int s = s0 + threadIdx.x;
    float2 o[12];
    wilson_site<float, G5IN, G5OUT>(s, g, kappa, in + (size_t)r * nel, U, o);
    Field<float>::store(out + (size_t)r * nel, g.V, s, o);
}

template <typename T, bool G5IN, bool G5OUT>
inline void launch_batch_kernel(unsigned blocks, int threads, cudaStream_t st, typename Field<T>::vec *out,
                                const typename Field<T>::vec *in, const typename Link<T>::vec *U, const Geom &g,
                                const SlabWalk &w, T kappa, int nrhs, long nel) {
    if constexpr (sizeof(T) == 4)
        k_wilson_batch32<G5IN, G5OUT><<<blocks, kSlabBlock, 0, st>>>(out, in, U, g, w, kappa, nrhs, nel);
    else
        k_wilson_batch<T, G5IN, G5OUT><<<blocks, threads, 0, st>>>(out, in, U, g, kappa, nrhs, nel);
}

template <typename T>
int launch_wilson_batch(Op &op, typename Field<T>::vec *out, const typename Field<T>::vec *in,
                        const typename Link<T>::vec *U, int which, int nrhs, long nel, int threads) {
    const Geom &g = op.g;
    // FP32: the slab walk for a stencil moving ~200 bytes per site and right-hand side
    const SlabWalk w = make_slab_walk(g.L[0] * g.L[1], g.L[2], g.L[3], nrhs, 200.0);
    const long blocks = sizeof(T) == 4 ? slab_blocks(w) * nrhs : (long)((g.V + threads - 1) / threads) * nrhs;
    const T kappa = (T)op.kappa;
    op.prof.stencil_start(op.stream, sizeof(T) == 4, g.V, nrhs);
    switch (which) {
    case DLZ_D: launch_batch_kernel<T, false, false>((unsigned)blocks, threads, op.stream, out, in, U, g, w, kappa, nrhs, nel); break;
    case DLZ_DDAG: launch_batch_kernel<T, true, true>((unsigned)blocks, threads, op.stream, out, in, U, g, w, kappa, nrhs, nel); break;
    case DLZ_Q: launch_batch_kernel<T, false, true>((unsigned)blocks, threads, op.stream, out, in, U, g, w, kappa, nrhs, nel); break;
    default: return fail(DLZ_ERR_BADARG, "stencil: which must be D, DDAG or Q");
    }
    op.prof.stencil_stop(op.stream);
    op.prof.launches++;
    DLZ_CUDA_TRY(cudaGetLastError());
    return DLZ_OK;
}

template <typename T>
int launch_wilson(Op &op, typename Field<T>::vec *out, const typename Field<T>::vec *in,
                  const typename Link<T>::vec *U, int which, int threads) {
    const Geom &g = op.g;
    const int blocks = (g.V + threads - 1) / threads;
    const T kappa = (T)op.kappa;
    op.prof.stencil_start(op.stream, sizeof(T) == 4, g.V, 1);
    switch (which) {
    case DLZ_D: k_wilson<T, false, false><<<blocks, threads, 0, op.stream>>>(out, in, U, g, kappa); break;
    case DLZ_DDAG: k_wilson<T, true, true><<<blocks, threads, 0, op.stream>>>(out, in, U, g, kappa); break;
    case DLZ_Q: k_wilson<T, false, true><<<blocks, threads, 0, op.stream>>>(out, in, U, g, kappa); break;
    default: return fail(DLZ_ERR_BADARG, "stencil: which must be D, DDAG or Q");
    }
    op.prof.stencil_stop(op.stream);
    op.prof.launches++;
    DLZ_CUDA_TRY(cudaGetLastError());
    return DLZ_OK;
}

// ------------------------------------------------------------------ user layout
// A spinor in the user layout is 12 consecutive complex numbers per site: W words of 16
// bytes.  A block of BT sites is one contiguous range there, moved in coalesced 16-byte
// words through shared memory whose rows are padded by one word (W + 1 words, so the eight
// lanes of a 16-byte access phase hit different banks).
template <typename T> struct UserRow {
    static constexpr int W = Field<T>::vec_per_site, RS = W + 1;
};
template <typename T, int BT>
__device__ inline void user_regs_to_row(typename Field<T>::vec *sm, const cx<T> (&v)[12]) {
    typename Field<T>::vec *row = sm + threadIdx.x * UserRow<T>::RS;
#pragma unroll
    for (int c = 0; c < UserRow<T>::W; ++c) {
        if constexpr (sizeof(T) == 4) row[c] = make_float4(v[2 * c].x, v[2 * c].y, v[2 * c + 1].x, v[2 * c + 1].y);
        else row[c] = v[c];
    }
}
template <typename T, int BT>
__device__ inline void user_store(typename Field<T>::vec *__restrict__ dst, const typename Field<T>::vec *sm, int nb) {
    for (int j = threadIdx.x; j < nb * UserRow<T>::W; j += BT)
        dst[j] = sm[(j / UserRow<T>::W) * UserRow<T>::RS + j % UserRow<T>::W];
}
// neighbours read straight from the user layout (16-byte words at a stride of a site)
template <typename T> struct UserGather {
    const typename Field<T>::vec *__restrict__ in;
    template <int MU, int DIR>
    __device__ inline void get(int n, bool, cx<T> (&p)[12]) const {
#pragma unroll
        for (int c = 0; c < UserRow<T>::W; ++c) {
            const typename Field<T>::vec q = in[(size_t)n * UserRow<T>::W + c];
            if constexpr (sizeof(T) == 4) {
                p[2 * c] = make_float2(q.x, q.y);
                p[2 * c + 1] = make_float2(q.z, q.w);
            } else {
                p[c] = q;
            }
        }
    }
};

// One application of the stencil for a user's vectors, all right-hand sides in one launch:
// UIN / UOUT say whether in / out are in the user layout or internal planes (the middle
// vector of D^dag D).  The neighbours are read straight from the user layout.  FP64 is bound
// by its ALU (888 FP64 instructions per site at 2 per cycle and SM), which hides the strided
// reads; FP32 pays more L1 cycles for them than for planes, but less than a pass that packs
// the vectors first.  FP32 Q, direct and packed first: 8^4, 1 RHS 15.0 and 19.3 us; 16^4, 3
// RHS 33.4 and 35.5 us; 16^3 x 32, 12 RHS 160 and 195 us; 24^3 x 48, 16 RHS 1011 and 1339 us.
// Against a pack, stencil and unpack launch per right-hand side with three temporary device
// allocations: FP32 D on 8^4, 1 RHS 40.0 -> 14.9 us; FP32 Q on 16^3 x 32, 12 RHS 675 -> 160 us
// (floor 48 us); FP64 D^dag D on 12 x 10 x 14 x 18, 3 RHS 768 -> 337 us (FP64-ALU floor 256 us).
template <typename T, bool G5IN, bool G5OUT, bool UIN, bool UOUT, int BT>
__global__ void __launch_bounds__(BT, sizeof(T) == 4 ? 768 / BT : 1)
k_wilson_user(typename Field<T>::vec *__restrict__ out, const typename Field<T>::vec *__restrict__ in,
              const typename Link<T>::vec *__restrict__ U, Geom g, SlabWalk w, T kappa, int nrhs) {
    __shared__ typename Field<T>::vec sm[UOUT ? BT * UserRow<T>::RS : 1];
    int r, sb, s0, nb;
    slab_rhs(w, blockIdx.x, r, sb);
    if (BT == kSlabBlock) {
        slab_block(w, sb, s0, nb);
    } else {
        s0 = sb * BT;
        nb = min(BT, g.V - s0);
    }
    const typename Field<T>::vec *inr = in + (size_t)r * UserRow<T>::W * g.V;
    typename Field<T>::vec *outr = out + (size_t)r * UserRow<T>::W * g.V;
    if ((int)threadIdx.x < nb) {
        const int s = s0 + threadIdx.x;
        cx<T> o[12];
        const PackedLinks<T> lk{U, g.V};
        if constexpr (UIN) {
            const UserGather<T> ga{inr};
            wilson_site_g<T, G5IN, G5OUT>(s, g, kappa, ga, lk, o);
        } else {
            const GlobalGather<T> ga{inr, g.V};
            wilson_site_g<T, G5IN, G5OUT>(s, g, kappa, ga, lk, o);
        }
        if (UOUT) user_regs_to_row<T, BT>(sm, o);
        else Field<T>::store(outr, g.V, s, o);
    }
    if (UOUT) {
        __syncthreads();
        user_store<T, BT>(outr + (size_t)s0 * UserRow<T>::W, sm, nb);
    }
}

}  // namespace

// Threads of a plain-order block (32, 64 or 128) for `total` sites of FP64-ALU-bound work:
// the SM with the most sites ends last, so the size that gives the fullest SMs fewest sites
// (31680 sites on 152 SMs: 256 with 128 threads, 224 with 32).
int balanced_threads(int V, int nrhs) {
    int best = 128;
    long most = 0;
    for (int bt : {128, 64, 32}) {
        const long blocks = (long)((V + bt - 1) / bt) * nrhs, m = (blocks + 151) / 152 * bt;
        if (bt == 128 || m < most) {
            best = bt;
            most = m;
        }
    }
    return best;
}

namespace {

template <typename T, bool UIN, bool UOUT, int BT>
void launch_user_bt(Op &op, typename Field<T>::vec *out, const typename Field<T>::vec *in,
                    const typename Link<T>::vec *U, int which, int nrhs) {
    const Geom &g = op.g;
    const SlabWalk w = sizeof(T) == 4 ? make_slab_walk(g.L[0] * g.L[1], g.L[2], g.L[3], nrhs, 200.0)
                                      : slab_walk_of(g.L[0] * g.L[1], g.L[2], g.L[3], g.L[2], nrhs);
    const unsigned blocks = (unsigned)((BT == kSlabBlock ? slab_blocks(w) : (long)(g.V + BT - 1) / BT) * nrhs);
    const T kappa = (T)op.kappa;
    switch (which) {
    case DLZ_D: k_wilson_user<T, false, false, UIN, UOUT, BT><<<blocks, BT, 0, op.stream>>>(out, in, U, g, w, kappa, nrhs); break;
    case DLZ_DDAG: k_wilson_user<T, true, true, UIN, UOUT, BT><<<blocks, BT, 0, op.stream>>>(out, in, U, g, w, kappa, nrhs); break;
    default: k_wilson_user<T, false, true, UIN, UOUT, BT><<<blocks, BT, 0, op.stream>>>(out, in, U, g, w, kappa, nrhs);
    }
    op.prof.launches++;
}
template <typename T, bool UIN, bool UOUT>
int launch_user(Op &op, void *out, const void *in, int which, int nrhs) {
    typedef typename Field<T>::vec vec;
    const typename Link<T>::vec *U = (const typename Link<T>::vec *)(sizeof(T) == 4 ? op.gauge32.p : op.gauge64.p);
    vec *o = (vec *)out;
    const vec *i = (const vec *)in;
    // FP32: 32 threads spread a short call over the SMs (8^4: 128 blocks)
    const int bt = sizeof(T) == 8 ? balanced_threads(op.g.V, nrhs) : UIN && (long)op.g.V * nrhs <= 152L * 64 ? 32 : 128;
    if (bt == 32) launch_user_bt<T, UIN, UOUT, 32>(op, o, i, U, which, nrhs);
    else if (bt == 64) launch_user_bt<T, UIN, UOUT, 64>(op, o, i, U, which, nrhs);
    else launch_user_bt<T, UIN, UOUT, 128>(op, o, i, U, which, nrhs);
    DLZ_CUDA_TRY(cudaGetLastError());
    return DLZ_OK;
}
// ------------------------------------------------------------------ layout kernels
__global__ void k_pack64(double2 *__restrict__ dst, const double2 *__restrict__ src, int V) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;   // canonical index s*12 + a
    if (i >= 12L * V) return;
    const size_t base = (size_t)blockIdx.y * 12 * V;       // blockIdx.y: the right-hand side
    const int s = (int)(i / 12), a = (int)(i % 12);
    dst[base + (size_t)a * V + s] = src[base + i];
}
__global__ void k_unpack64(double2 *__restrict__ dst, const double2 *__restrict__ src, int V) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 12L * V) return;
    const size_t base = (size_t)blockIdx.y * 12 * V;
    const int s = (int)(i / 12), a = (int)(i % 12);
    dst[base + i] = src[base + (size_t)a * V + s];
}
__global__ void k_pack32(float4 *__restrict__ dst, const float2 *__restrict__ src, int V) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;   // s*6 + c
    if (i >= 6L * V) return;
    const size_t base = (size_t)blockIdx.y * 6 * V;
    const int s = (int)(i / 6), c = (int)(i % 6);
    const float2 a = src[2 * base + (size_t)s * 12 + 2 * c], b = src[2 * base + (size_t)s * 12 + 2 * c + 1];
    dst[base + (size_t)c * V + s] = make_float4(a.x, a.y, b.x, b.y);
}
__global__ void k_unpack32(float2 *__restrict__ dst, const float4 *__restrict__ src, int V) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 6L * V) return;
    const size_t base = (size_t)blockIdx.y * 6 * V;
    const int s = (int)(i / 6), c = (int)(i % 6);
    const float4 q = src[base + (size_t)c * V + s];
    dst[2 * base + (size_t)s * 12 + 2 * c] = make_float2(q.x, q.y);
    dst[2 * base + (size_t)s * 12 + 2 * c + 1] = make_float2(q.z, q.w);
}
// internal FP64 planes <-> internal FP32 planes (plane c of FP32 = planes 2c, 2c+1)
__global__ void k_64to32(float4 *__restrict__ dst, const double2 *__restrict__ src, int V) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;   // c*V + s
    if (i >= 6L * V) return;
    const int c = (int)(i / V), s = (int)(i % V);
    const double2 a = src[(size_t)(2 * c) * V + s], b = src[(size_t)(2 * c + 1) * V + s];
    dst[i] = make_float4((float)a.x, (float)a.y, (float)b.x, (float)b.y);
}
__global__ void k_32to64(double2 *__restrict__ dst, const float4 *__restrict__ src, int V) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 6L * V) return;
    const int c = (int)(i / V), s = (int)(i % V);
    const float4 q = src[i];
    dst[(size_t)(2 * c) * V + s] = make_double2(q.x, q.y);
    dst[(size_t)(2 * c + 1) * V + s] = make_double2(q.z, q.w);
}

inline int grid_for(long n, int threads) { return (int)((n + threads - 1) / threads); }

}  // namespace

// An even-odd operator applies its Schur complement (wilson_eo.cu) wherever a solver
// asks for D, D^dag or Q: the solvers run unchanged on its even-site vectors.
int wilson64(Op &op, double2 *out, const double2 *in, int which) {
    if (op.eo) return eo_apply64(op, out, in, which, 1);
    return launch_wilson<double>(op, out, in, op.gauge64.as<double2>(), which, balanced_threads(op.g.V, 1));
}
int wilson32(Op &op, float4 *out, const float4 *in, int which) {
    if (op.eo) return eo_apply32(op, out, in, which, 1);
    return launch_wilson<float>(op, out, in, op.gauge32.as<float4>(), which, kStencilThreads32);
}

int wilson32_batch(Op &op, float4 *out, const float4 *in, int which, int nrhs) {
    if (op.eo) return eo_apply32(op, out, in, which, nrhs);
    return launch_wilson_batch<float>(op, out, in, op.gauge32.as<float4>(), which, nrhs, 6L * op.g.V,
                                      kStencilThreads32);
}
int wilson64_batch(Op &op, double2 *out, const double2 *in, int which, int nrhs) {
    if (op.eo) return eo_apply64(op, out, in, which, nrhs);
    return launch_wilson_batch<double>(op, out, in, op.gauge64.as<double2>(), which, nrhs, 12L * op.g.V,
                                       balanced_threads(op.g.V, nrhs));
}

int apply64(Op &op, double2 *out, const double2 *in, int which, double2 *tmp) {
    if (which == DLZ_DDAGD) {
        // D^dag D = Q Q (gamma5 D is hermitian, Q^2 = gamma5 D gamma5 D = D^dag D)
        DLZ_TRY(wilson64(op, tmp, in, DLZ_Q));
        return wilson64(op, out, tmp, DLZ_Q);
    }
    return wilson64(op, out, in, which);
}
int apply32(Op &op, float4 *out, const float4 *in, int which, float4 *tmp) {
    if (which == DLZ_DDAGD) {
        DLZ_TRY(wilson32(op, tmp, in, DLZ_Q));
        return wilson32(op, out, tmp, DLZ_Q);
    }
    return wilson32(op, out, in, which);
}

// ------------------------------------------------------------------ a user's call
// FP32 reads 16-byte words of the user's vectors; a vector that is only 8-byte aligned (a
// view at an odd complex element) takes the layout kernels that read single complex numbers.
static bool user_direct(const Op &op, const void *in, const void *out, int dtype) {
    if (op.eo || dtype == DLZ_BF16) return false;
    return dtype == DLZ_F64 || (((uintptr_t)in | (uintptr_t)out) & 15) == 0;
}

size_t apply_user_scratch(const Op &op, int which, const void *in, const void *out, int dtype) {
    const size_t vec = (size_t)12 * op.g.V * (dtype == DLZ_F64 ? 16 : dtype == DLZ_F32 ? 8 : 4);
    return ((user_direct(op, in, out, dtype) ? 0 : 2) + (which == DLZ_DDAGD ? 1 : 0)) * vec;
}

// out = A in on nrhs user vectors, `scratch` of at least apply_user_scratch() bytes; takes as
// many right-hand sides at a time as it holds.  D^dag D = Q Q, the middle vector in planes.
int apply_user(Op &op, int which, const void *in, void *out, int dtype, int nrhs, void *scratch, size_t bytes) {
    const size_t n = (size_t)12 * op.g.V, esz = dtype == DLZ_F64 ? 16 : 8;
    const size_t vec = n * (dtype == DLZ_BF16 ? 4 : esz), per = apply_user_scratch(op, which, in, out, dtype);
    const bool direct = user_direct(op, in, out, dtype);
    // (the launches' grids: at most 65535 right-hand sides in y, 2^31 - 1 blocks in x)
    const long most = std::max(1L, std::min(65535L, (1L << 30) / ((op.g.V + 31) / 32)));
    const int chunk = (int)std::min<size_t>({(size_t)nrhs, (size_t)most, per ? std::max<size_t>(1, bytes / per) : (size_t)nrhs});
    const int first = which == DLZ_DDAGD ? DLZ_Q : which;
    for (int r0 = 0; r0 < nrhs; r0 += chunk) {
        const int nb = std::min(chunk, nrhs - r0);
        const char *src = (const char *)in + (size_t)r0 * n * esz;
        char *dst = (char *)out + (size_t)r0 * n * esz;
        char *a = (char *)scratch, *b = a + vec * nb, *c = b + vec * nb;
        const bool two = which == DLZ_DDAGD;
        if (dtype == DLZ_BF16) {
            DLZ_TRY(pack_bf16(op, (uint2 *)a, (const float2 *)src, nb));
            // D^dag D is rounded to bfloat16 in between
            DLZ_TRY(wilson_bf16_batch(op, (uint2 *)b, (const uint2 *)a, first, nb));
            if (two) DLZ_TRY(wilson_bf16_batch(op, (uint2 *)c, (const uint2 *)b, DLZ_Q, nb));
            DLZ_TRY(unpack_bf16(op, (float2 *)dst, (const uint2 *)(two ? c : b), nb));
        } else if (dtype == DLZ_F64 && op.eo) {
            DLZ_TRY(pack64(op, (double2 *)a, (const double2 *)src, nb));
            DLZ_TRY(eo_apply64(op, (double2 *)b, (const double2 *)a, first, nb));
            if (two) DLZ_TRY(eo_apply64(op, (double2 *)c, (const double2 *)b, DLZ_Q, nb));
            DLZ_TRY(unpack64(op, (double2 *)dst, (const double2 *)(two ? c : b), nb));
        } else if (!direct) {
            DLZ_TRY(pack32(op, (float4 *)a, (const float2 *)src, nb));
            DLZ_TRY(wilson32_batch(op, (float4 *)b, (const float4 *)a, first, nb));
            if (two) DLZ_TRY(wilson32_batch(op, (float4 *)c, (const float4 *)b, DLZ_Q, nb));
            DLZ_TRY(unpack32(op, (float2 *)dst, (const float4 *)(two ? c : b), nb));
        } else if (dtype == DLZ_F64) {
            if (two) DLZ_TRY((launch_user<double, true, false>(op, a, src, DLZ_Q, nb)));
            if (two) DLZ_TRY((launch_user<double, false, true>(op, dst, a, DLZ_Q, nb)));
            else DLZ_TRY((launch_user<double, true, true>(op, dst, src, which, nb)));
        } else {
            if (two) DLZ_TRY((launch_user<float, true, false>(op, a, src, DLZ_Q, nb)));
            if (two) DLZ_TRY((launch_user<float, false, true>(op, dst, a, DLZ_Q, nb)));
            else DLZ_TRY((launch_user<float, true, true>(op, dst, src, which, nb)));
        }
    }
    return DLZ_OK;
}

int pack64(Op &op, double2 *dst, const double2 *src, int nrhs) {
    const long n = 12L * op.g.V;
    k_pack64<<<dim3(grid_for(n, 256), nrhs), 256, 0, op.stream>>>(dst, src, op.g.V);
    op.prof.launches++;
    DLZ_CUDA_TRY(cudaGetLastError());
    return DLZ_OK;
}
int unpack64(Op &op, double2 *dst, const double2 *src, int nrhs) {
    const long n = 12L * op.g.V;
    k_unpack64<<<dim3(grid_for(n, 256), nrhs), 256, 0, op.stream>>>(dst, src, op.g.V);
    op.prof.launches++;
    DLZ_CUDA_TRY(cudaGetLastError());
    return DLZ_OK;
}
int pack32(Op &op, float4 *dst, const float2 *src, int nrhs) {
    const long n = 6L * op.g.V;
    k_pack32<<<dim3(grid_for(n, 256), nrhs), 256, 0, op.stream>>>(dst, src, op.g.V);
    op.prof.launches++;
    DLZ_CUDA_TRY(cudaGetLastError());
    return DLZ_OK;
}
int unpack32(Op &op, float2 *dst, const float4 *src, int nrhs) {
    const long n = 6L * op.g.V;
    k_unpack32<<<dim3(grid_for(n, 256), nrhs), 256, 0, op.stream>>>(dst, src, op.g.V);
    op.prof.launches++;
    DLZ_CUDA_TRY(cudaGetLastError());
    return DLZ_OK;
}
int convert64to32(Op &op, float4 *dst, const double2 *src) {
    const long n = 6L * op.g.V;
    k_64to32<<<grid_for(n, 256), 256, 0, op.stream>>>(dst, src, op.g.V);
    op.prof.launches++;
    DLZ_CUDA_TRY(cudaGetLastError());
    return DLZ_OK;
}
int convert32to64(Op &op, double2 *dst, const float4 *src) {
    const long n = 6L * op.g.V;
    k_32to64<<<grid_for(n, 256), 256, 0, op.stream>>>(dst, src, op.g.V);
    op.prof.launches++;
    DLZ_CUDA_TRY(cudaGetLastError());
    return DLZ_OK;
}

}  // namespace dlz
