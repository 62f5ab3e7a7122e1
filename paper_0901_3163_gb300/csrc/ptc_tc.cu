// Tensor-core (tcgen05) form of a parallel-transport convolution layer: no counterpart in
// arXiv:0901.3163, see ptc.cu for the layer,
//   out[c'](x) = sum_o sum_c W[o][c'][c] (T_o in[c])(x).
//
// For every offset o the layer is a matrix product: a row is a site and colour, K runs over
// the input channels, spins and re/im, N over the output channels, spins and re/im, with the
// real form [[Re W, Im W], [-Im W, Re W]]^T of the complex spin matrices.  The weights are
// bfloat16, exact as they are; a transported FP32 value is the exact sum of three bfloat16
// parts (8 mantissa bits each, rounded off one after another), so every product is exact and only
// the FP32 accumulation rounds.  The tensor cores cut off their sums instead of rounding them
// to nearest (measured as about 2e-8 of the result per MMA step), so an accumulator takes
// kMaxSteps steps of K = 16 at most before it is added, rounding to nearest, to an FP32 sum in
// registers.  Error against 64 bits of three layers 1 -> 12 -> 16 -> 1 on 16^4: 6.5e-7, 8.2e-7
// with FP32 arithmetic on the CUDA cores (27 steps per accumulator: 9.5e-7).
//
// Block: tiles of 42 sites (126 rows) of one vector.  kGroups groups of four filling warps
// (thread = site and a third of the chunk's channels) load a neighbour's spinor, transport it,
// cut the values into parts and store them as the A operands (K-major 8 x 16-byte core
// matrices, no swizzle); one warp issues the MMAs; eight warps add finished accumulators up and
// write the tile.  They meet at mbarriers only.
#include <algorithm>
#include <cstring>

#include "ptc_tc.cuh"
#include "tc_util.cuh"
#include "wilson_site.cuh"

namespace dlz {
namespace {

constexpr int kGroups = 3, kEpi = 8;
constexpr int kThreads = 32 * (kEpi + 1) + 128 * kGroups;
constexpr int kSites = 42;                       // sites of a tile: 126 of the 128 rows
constexpr int kMaxSteps = 9;

// A chunk is an offset and up to 6 input channels (two per filling thread), an even number
__host__ __device__ inline int channel_chunks(int cin) { return (cin + 5) / 6; }
__host__ __device__ inline int chunk_channels(int cin) {
    const int n = channel_chunks(cin);
    return ((cin + n - 1) / n + 1) / 2 * 2;
}
__host__ __device__ inline int npad_of(int cout) { return (8 * cout + 15) / 16 * 16; }

struct FwdArgs {
    float4 *out;
    const float4 *in, *U;
    const __nv_bfloat16 *img;
    Geom g;
    int cin, cout, npad, nvec, nbuf, ncols;
    PtcStatus status;
};

__device__ __forceinline__ void report(const PtcStatus &s, int bit) {
    atomicOr(s.bits, bit);
    *static_cast<volatile int *>(s.host) = 1;
}

struct FwdShared {
    uint64_t full[kGroups], empty[kGroups], acc_full[4], acc_empty[4], drained;
    uint32_t tbase;
    int failed;
};

__device__ __forceinline__ void mma_bf16(uint32_t taddr, uint32_t da, uint32_t db, uint32_t dhi, uint32_t idesc, bool acc) {
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\tmov.b64 a, {%1, %5};\n\tmov.b64 b, {%2, %5};\n\t"
                 "setp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\t}\n" ::"r"(taddr),
                 "r"(da), "r"(db), "r"(idesc), "r"(acc ? 1u : 0u), "r"(dhi));
}

// sum[0 .. 15] += columns addr .. addr + 15 of this warp's lane quarter (the first 8 if !wide)
__device__ __forceinline__ void tmem_add(uint32_t addr, bool wide, float *sum) {
    uint32_t r[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) r[j] = 0u;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(addr));
    if (wide)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                     : "r"(addr + 8));
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]));
#pragma unroll
    for (int j = 0; j < 16; ++j) sum[j] += __uint_as_float(r[j]);
}

// two values rounded to bfloat16 in one word (a in the low half), which are taken off them
__device__ __forceinline__ uint32_t take_part(float &a, float &b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    uint32_t w;
    memcpy(&w, &h, 4);
    a -= __uint_as_float(w << 16);
    b -= __uint_as_float(w & 0xffff0000u);
    return w;
}

// One channel's transported spinor t of the tile's site sl as K octet `oct` of the rows 3 sl +
// colour of the three parts (part h at h * part): 8 values (spin, re/im) = 16 bytes each
__device__ __forceinline__ void store_parts(unsigned char *stage, int part, int sbo, int sl, int oct, const float2 (&t)[12]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int row = 3 * sl + c;
        unsigned char *dst = stage + (row >> 3) * sbo + oct * 128 + (row & 7) * 16;
        float x[8];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            x[2 * s] = t[3 * s + c].x;
            x[2 * s + 1] = t[3 * s + c].y;
        }
#pragma unroll
        for (int h = 0; h < 3; ++h)
            *reinterpret_cast<uint4 *>(dst + h * part) =
                make_uint4(take_part(x[0], x[1]), take_part(x[2], x[3]), take_part(x[4], x[5]), take_part(x[6], x[7]));
    }
}

// Bound by the filling warps (transport, splitting, stores).  16^4, 4 vectors, one GB300,
// against the CUDA-core kernel: 12 -> 16 channels 4.95 -> 1.09 ms, 16 -> 12 (its adjoint) 4.9
// -> 1.48 ms, 1 -> 12 and 1 -> 16 0.57 -> 0.38 ms.  Two filling groups: 1.19 and 1.56 ms; four
// (fewer registers each): 1.41 and 1.54 ms.  Tiles of 128 sites with an accumulator per colour,
// whose partial results do not fit in registers and went through global memory: 2.2 and 2.4 ms.
__global__ void __launch_bounds__(kThreads, 1) k_ptc_tc_fwd(FwdArgs a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) FwdShared sh;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int cc = chunk_channels(a.cin), ncp = channel_chunks(a.cin), sbo = cc * 128;
    const int part = 16 * sbo, b_bytes = (a.npad / 8) * sbo, stage_bytes = 3 * part + b_bytes;
    if (threadIdx.x == 0) {
        sh.failed = 0;
        for (int i = 0; i < kGroups; ++i) {
            mbar_init(&sh.full[i], 4);
            mbar_init(&sh.empty[i], 1);
        }
        for (int i = 0; i < 4; ++i) {
            mbar_init(&sh.acc_full[i], 1);
            mbar_init(&sh.acc_empty[i], kEpi);
        }
        mbar_init(&sh.drained, 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    tmem_alloc(&sh.tbase, a.ncols);
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t taddr = sh.tbase;
    volatile int *failed = &sh.failed;
    const int V = a.g.V, tiles_per_vec = (V + kSites - 1) / kSites, ntiles = tiles_per_vec * a.nvec;
    // a tile's chunks, and the segments of chunks that one accumulator takes
    const int nch = 9 * ncp, per = max(1, kMaxSteps / (3 * cc / 2)), nseg = (nch + per - 1) / per;
    const size_t plane = (size_t)6 * V;
    const int mine = (ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;     // the block's tiles
    const int ft = (int)threadIdx.x - 32 * (kEpi + 1);
    if (ft >= 0) {
        // ---- fill: group grp takes the chunks (tile, offset, channels) grp, grp + kGroups, ...;
        // a thread the channels cg and cg + 3 of its site
        const int grp = ft / 128, tid = ft % 128, sl = tid % kSites, cg = tid / kSites;
        unsigned char *stage = smem + grp * stage_bytes;
        const long total = (long)mine * nch;
        uint32_t round = 0;
        int tile_of = -1, s = 0, vec = 0;
        int c4[4] = {0, 0, 0, 0};
        bool ok = false;
        int ti = 0, r = grp;                       // chunk r of the block's tile ti
        for (long q = grp; q < total; q += kGroups, ++round) {
            while (r >= nch) { r -= nch; ++ti; }
            const int o = r / ncp, p = r % ncp;
            if (ti != tile_of) {
                const int t = (int)blockIdx.x + ti * (int)gridDim.x;
                vec = t / tiles_per_vec;
                s = (t % tiles_per_vec) * kSites + sl;
                ok = s < V;
                int d = ok ? s : 0;
                c4[0] = d % a.g.L[0]; d /= a.g.L[0];
                c4[1] = d % a.g.L[1]; d /= a.g.L[1];
                c4[2] = d % a.g.L[2];
                c4[3] = d / a.g.L[2];
                tile_of = ti;
            }
            int sn = ok ? s : 0;
            float2 u[9];
            if (o > 0 && ok) {
                const int mu = (o - 1) >> 1;
                const bool fwd = ((o - 1) & 1) == 0;
                const int L = a.g.L[mu], c = mu == 0 ? c4[0] : mu == 1 ? c4[1] : mu == 2 ? c4[2] : c4[3];
                const int st = mu == 0 ? 1 : mu == 1 ? a.g.L[0] : mu == 2 ? a.g.L[0] * a.g.L[1]
                                                                          : a.g.L[0] * a.g.L[1] * a.g.L[2];
                sn = fwd ? (c == L - 1 ? s - (L - 1) * st : s + st) : (c == 0 ? s + (L - 1) * st : s - st);
                Link<float>::load(a.U, V, mu, fwd ? s : sn, u);
                if (!fwd) {                       // U^dag
#pragma unroll
                    for (int i = 0; i < 3; ++i)
#pragma unroll
                        for (int j = i; j < 3; ++j) {
                            const float2 x = u[3 * i + j], y = u[3 * j + i];
                            u[3 * i + j] = make_float2(y.x, -y.y);
                            u[3 * j + i] = make_float2(x.x, -x.y);
                        }
                }
            }
            const float4 *src = a.in + ((size_t)vec * a.cin + p * cc) * plane;
            if (round > 0 && !__all_sync(0xffffffffu, mbar_wait(&sh.empty[grp], (round - 1) & 1u, failed))) break;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int ch = cg + 3 * h;
                if (ch < cc && cg < 3) {
                    float2 x[12], t[12];
                    if (ok && p * cc + ch < a.cin) {
                        Field<float>::load(src + ch * plane, V, sn, x);
                        if (o > 0) {
#pragma unroll
                            for (int sp = 0; sp < 4; ++sp)
#pragma unroll
                                for (int i = 0; i < 3; ++i) {
                                    float2 z = make_float2(0.f, 0.f);
#pragma unroll
                                    for (int j = 0; j < 3; ++j) z = cfma(u[3 * i + j], x[3 * sp + j], z);
                                    t[3 * sp + i] = z;
                                }
                        } else {
#pragma unroll
                            for (int j = 0; j < 12; ++j) t[j] = x[j];
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 12; ++j) t[j] = make_float2(0.f, 0.f);
                    }
                    store_parts(stage, part, sbo, sl, ch, t);
                }
            }
            // the chunk's weights in operand order
            const uint4 *w = reinterpret_cast<const uint4 *>(a.img) + (size_t)r * (b_bytes / 16);
            for (int i = tid; i < b_bytes / 16; i += 128) reinterpret_cast<uint4 *>(stage + 3 * part)[i] = w[i];
            asm volatile("fence.proxy.async.shared::cta;");
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.full[grp]);
            r += kGroups;
        }
    } else if (warp == kEpi) {
        // ---- MMA (the warp is uniform; lane 0 issues): parts from the smallest up
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(a.npad >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        const uint32_t d0 = sdesc_lo(su32(smem)), dhi = ((uint32_t)sbo >> 4) | 1u << 14, w_stage = stage_bytes >> 4;
        int st = 0, n = 0;
        uint32_t round = 0;
        bool ok = true, issued = false;
        for (int ti = 0; ti < mine && ok; ++ti)
            for (int sg = 0; sg < nseg && ok; ++sg, ++n) {
                const int acc = n % a.nbuf, use = n / a.nbuf;
                const int chunks = min(nch, (sg + 1) * per) - sg * per;
                if (use > 0 && !__all_sync(0xffffffffu, mbar_wait(&sh.acc_empty[acc], (use - 1) & 1, failed))) { ok = false; break; }
                for (int ch = 0; ch < chunks; ++ch) {
                    ok = __all_sync(0xffffffffu, mbar_wait(&sh.full[st], round & 1u, failed));
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    const uint32_t da = d0 + st * w_stage, db = da + (3 * part >> 4);
                    if (lane == 0) {
                        for (int h = 2; h >= 0; --h)
                            for (int k = 0; k < cc / 2; ++k)
                                mma_bf16(taddr + acc * a.npad, da + (h * part >> 4) + k * 16, db + k * 16, dhi, idesc,
                                         ch > 0 || h < 2 || k > 0);
                        commit_to(&sh.empty[st]);
                        issued = true;
                    }
                    if (++st == kGroups) { st = 0; ++round; }
                }
                if (ok && lane == 0) commit_to(&sh.acc_full[acc]);
            }
        mma_drain(&sh.drained, issued, failed);
    } else {
        // ---- results: warp w has rows 32 (w % 4) .. of a tile and half of the columns; the
        // thread of row 3 sl + c sums colour c of its output channels in registers
        const int lq = warp & 3, half = a.npad / 2, c_lo = (warp >> 2) * half;
        const int row = 32 * lq + lane, sl = row / 3, col = row - 3 * sl;
        int n = 0;
        bool ok = true;
        for (int ti = 0; ti < mine && ok; ++ti) {
            float sum[64];
#pragma unroll
            for (int j = 0; j < 64; ++j) sum[j] = 0.f;
            for (int sg = 0; sg < nseg; ++sg, ++n) {
                const int acc = n % a.nbuf, use = n / a.nbuf;
                ok = __all_sync(0xffffffffu, mbar_wait(&sh.acc_full[acc], use & 1, failed));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
                for (int j = 0; j < 64; j += 16)
                    if (j < half)
                        tmem_add(taddr + ((uint32_t)(32 * lq) << 16) + (uint32_t)(acc * a.npad + c_lo + j), j + 8 < half, sum + j);
                asm volatile("tcgen05.fence::before_thread_sync;");
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.acc_empty[acc]);
            }
            const int t = (int)blockIdx.x + ti * (int)gridDim.x, vec = t / tiles_per_vec;
            const int s = (t % tiles_per_vec) * kSites + sl;
            if (!ok || sl >= kSites || s >= V) continue;
            // column 8 c' + 2 s' + re/im; component 3 s' + colour is half of plane (..) / 2
            float4 *dst = a.out + (size_t)vec * a.cout * plane + s;
            float nan = 0.f;              // 0 times every result: NaN if one is not finite
#pragma unroll
            for (int j = 0; j < 64; j += 2) {
                const int ch = (c_lo + j) / 8, comp = 3 * ((j % 8) / 2) + col;
                if (j < half && ch < a.cout) {
                    reinterpret_cast<float2 *>(dst + (size_t)ch * plane + (size_t)(comp >> 1) * V)[comp & 1] =
                        make_float2(sum[j], sum[j + 1]);
                    nan = fmaf(sum[j], 0.f, fmaf(sum[j + 1], 0.f, nan));
                }
            }
            if (nan != 0.f) report(a.status, kPtcNonfinite);
        }
    }
    __syncthreads();
    if (sh.failed && threadIdx.x == 0) report(a.status, kPtcTimeout);
    tc_teardown(taddr, a.ncols);
}

// ------------------------------------------------------------------ weight gradient
// G(W)[o][c'][c] = sum over sites and colours of G(out) (T_o in)^dag as P[m][n] = sum_k A[m][k]
// B[n][k]: m = 8 c' + 2 s' + re/im of G(out), n = 8 c + 2 s + re/im of the transported input, k
// the sites and colours; re G = P[re][re] + P[im][im], im G = P[im][re] - P[re][im].  Both
// operands are FP32 values in three bfloat16 parts h, m, l, rounded: |m| <= 2^-8 and |l| <= 2^-17 of
// the value's power of two, with either sign.  Of the nine products of parts the six down to 2^-16
// are formed, smallest first, so that only the three steps of h h are cut off at the size of the
// sum.  The others are 2^-24 together at most and of either sign.  (Parts that are cut off have
// the value's sign: what they leave out reaches 2^-21 and adds up in sums of one sign.)
// A block has one offset and every gridDim.x-th tile of 16 sites: a stage is one tile, 48 k (K
// step = colour).  The operands are stored as they come, 16 bytes = the 8 values of a channel at
// one k, i.e. M- and N-major: 8 x 8 core matrices of 8 k x 16 bytes, k groups 128 bytes apart,
// row groups 768.  Each tile's accumulator is added to FP32 sums in registers.
constexpr int kGSites = 16, kGSbo = 3 * kGSites * 16, kGPartA = 16 * kGSbo;

struct GradArgs {
    float2 *partials;
    const float4 *gout, *in, *U;
    Geom g;
    int cin, cout, npad, nvec, nbuf, ncols;
    PtcStatus status;
};

// channel octet `oct` at site sl in the three parts (part p at p * part)
__device__ __forceinline__ void store_parts_k(unsigned char *base, int part, int oct, int sl, const float2 (&t)[12]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        unsigned char *dst = base + oct * kGSbo + (2 * c + (sl >> 3)) * 128 + (sl & 7) * 16;
        float x[8];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            x[2 * s] = t[3 * s + c].x;
            x[2 * s + 1] = t[3 * s + c].y;
        }
#pragma unroll
        for (int h = 0; h < 3; ++h)
            *reinterpret_cast<uint4 *>(dst + h * part) =
                make_uint4(take_part(x[0], x[1]), take_part(x[2], x[3]), take_part(x[4], x[5]), take_part(x[6], x[7]));
    }
}

__global__ void __launch_bounds__(kThreads, 1) k_ptc_tc_wgrad(GradArgs a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) FwdShared sh;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int part_b = (a.npad / 8) * kGSbo, stage_bytes = 3 * (kGPartA + part_b);
    if (threadIdx.x == 0) {
        sh.failed = 0;
        for (int i = 0; i < kGroups; ++i) {
            mbar_init(&sh.full[i], 4);
            mbar_init(&sh.empty[i], 1);
        }
        for (int i = 0; i < 4; ++i) {
            mbar_init(&sh.acc_full[i], 1);
            mbar_init(&sh.acc_empty[i], kEpi);
        }
        mbar_init(&sh.drained, 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    tmem_alloc(&sh.tbase, a.ncols);
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t taddr = sh.tbase;
    volatile int *failed = &sh.failed;
    const int V = a.g.V, tiles_per_vec = (V + kGSites - 1) / kGSites, ntiles = tiles_per_vec * a.nvec;
    const int o = blockIdx.y, rows = 4 * a.cout, cols = 4 * a.cin;
    const size_t plane = (size_t)6 * V;
    const int mine = (int)blockIdx.x < ntiles ? (ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
    const int ft = (int)threadIdx.x - 32 * (kEpi + 1);
    if (ft >= 0) {
        // ---- fill: group grp takes the block's tiles grp, grp + kGroups, ...; a thread its site's
        // channels tid / 16, tid / 16 + 8, ... of G(out) and then of the input
        const int grp = ft / 128, tid = ft % 128, sl = tid % kGSites;
        unsigned char *stage = smem + grp * stage_bytes;
        uint32_t round = 0;
        for (int q = grp; q < mine; q += kGroups, ++round) {
            const int t = (int)blockIdx.x + q * (int)gridDim.x, vec = t / tiles_per_vec;
            const int s = (t % tiles_per_vec) * kGSites + sl;
            const bool ok = s < V;
            int sn = ok ? s : 0;
            float2 u[9];
            if (o > 0 && ok) {
                const int mu = (o - 1) >> 1;
                const bool fwd = ((o - 1) & 1) == 0;
                int d = s, st = 1;
                for (int i = 0; i < mu; ++i) { d /= a.g.L[i]; st *= a.g.L[i]; }
                const int L = a.g.L[mu], c = d % L;
                sn = fwd ? (c == L - 1 ? s - (L - 1) * st : s + st) : (c == 0 ? s + (L - 1) * st : s - st);
                Link<float>::load(a.U, V, mu, fwd ? s : sn, u);
                if (!fwd) {                       // U^dag
#pragma unroll
                    for (int i = 0; i < 3; ++i)
#pragma unroll
                        for (int j = i; j < 3; ++j) {
                            const float2 x = u[3 * i + j], y = u[3 * j + i];
                            u[3 * i + j] = make_float2(y.x, -y.y);
                            u[3 * j + i] = make_float2(x.x, -x.y);
                        }
                }
            }
            if (round > 0 && !__all_sync(0xffffffffu, mbar_wait(&sh.empty[grp], (round - 1) & 1u, failed))) break;
            for (int ch = tid / kGSites; ch < a.cout + a.cin; ch += 128 / kGSites) {
                const bool is_g = ch < a.cout;
                const int c = is_g ? ch : ch - a.cout;
                float2 x[12];
                if (!ok) {
#pragma unroll
                    for (int j = 0; j < 12; ++j) x[j] = make_float2(0.f, 0.f);
                } else if (is_g) {
                    Field<float>::load(a.gout + ((size_t)vec * a.cout + c) * plane, V, s, x);
                } else {
                    Field<float>::load(a.in + ((size_t)vec * a.cin + c) * plane, V, sn, x);
                    if (o > 0) {
#pragma unroll
                        for (int sp = 0; sp < 4; ++sp) {
                            const float2 y0 = x[3 * sp], y1 = x[3 * sp + 1], y2 = x[3 * sp + 2];
#pragma unroll
                            for (int i = 0; i < 3; ++i)
                                x[3 * sp + i] = cfma(u[3 * i + 2], y2, cfma(u[3 * i + 1], y1, cfma(u[3 * i], y0, make_float2(0.f, 0.f))));
                        }
                    }
                }
                store_parts_k(is_g ? stage : stage + 3 * kGPartA, is_g ? kGPartA : part_b, c, sl, x);
            }
            asm volatile("fence.proxy.async.shared::cta;");
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.full[grp]);
        }
    } else if (warp == kEpi) {
        // ---- MMA (the warp is uniform; lane 0 issues); both operands M- / N-major (bits 15, 16)
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                               ((uint32_t)(a.npad >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        const uint32_t d0 = sdesc_lo(su32(smem)), w_stage = stage_bytes >> 4;
        const int pa[6] = {2, 0, 1, 1, 0, 0}, pb[6] = {0, 2, 1, 0, 1, 0};
        int st = 0;
        uint32_t round = 0;
        bool issued = false;
        for (int n = 0; n < mine; ++n) {
            const int acc = n % a.nbuf, use = n / a.nbuf;
            if (use > 0 && !__all_sync(0xffffffffu, mbar_wait(&sh.acc_empty[acc], (use - 1) & 1, failed))) break;
            if (!__all_sync(0xffffffffu, mbar_wait(&sh.full[st], round & 1u, failed))) break;
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint32_t da = d0 + st * w_stage, db = da + (3 * kGPartA >> 4);
            if (lane == 0) {
#pragma unroll
                for (int p = 0; p < 6; ++p)
#pragma unroll
                    for (int k = 0; k < 3; ++k)
                        mma_bf16(taddr + acc * a.npad, da + (pa[p] * kGPartA >> 4) + k * 16, db + (pb[p] * part_b >> 4) + k * 16,
                                 kDescHi<kGSbo>, idesc, p > 0 || k > 0);
                commit_to(&sh.empty[st]);
                commit_to(&sh.acc_full[acc]);
                issued = true;
            }
            if (++st == kGroups) { st = 0; ++round; }
        }
        mma_drain(&sh.drained, issued, failed);
    } else {
        // ---- sums: warp w has rows 32 (w % 4) .. and half of the columns
        const int lq = warp & 3, half = a.npad / 2, c_lo = (warp >> 2) * half;
        float sum[64];
#pragma unroll
        for (int j = 0; j < 64; ++j) sum[j] = 0.f;
        for (int n = 0; n < mine; ++n) {
            const int acc = n % a.nbuf, use = n / a.nbuf;
            if (!__all_sync(0xffffffffu, mbar_wait(&sh.acc_full[acc], use & 1, failed))) break;
            asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
            for (int j = 0; j < 64; j += 16)
                if (j < half)
                    tmem_add(taddr + ((uint32_t)(32 * lq) << 16) + (uint32_t)(acc * a.npad + c_lo + j), j + 8 < half, sum + j);
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.acc_empty[acc]);
        }
        // row 2 r + (0 re, 1 im): the re lane combines its sums with its neighbour's
        const int r = (32 * lq + lane) / 2;
        float2 *pb = a.partials + ((size_t)o * gridDim.x + blockIdx.x) * rows * cols;
        float nan = 0.f;                  // 0 times every result: NaN if one is not finite
#pragma unroll
        for (int j = 0; j < 64; j += 2) {
            const float q0 = __shfl_down_sync(0xffffffffu, sum[j], 1), q1 = __shfl_down_sync(0xffffffffu, sum[j + 1], 1);
            const int c = (c_lo + j) / 2;
            if (j < half && (lane & 1) == 0 && r < rows && c < cols) {
                const float2 v = make_float2(sum[j] + q1, q0 - sum[j + 1]);
                pb[(size_t)r * cols + c] = v;
                nan = fmaf(v.x, 0.f, fmaf(v.y, 0.f, nan));
            }
        }
        if (nan != 0.f) report(a.status, kPtcNonfinite);
    }
    __syncthreads();
    if (sh.failed && threadIdx.x == 0) report(a.status, kPtcTimeout);
    tc_teardown(taddr, a.ncols);
}

int grad_stage_bytes(int cin) { return 3 * (kGPartA + (npad_of(cin) / 8) * kGSbo); }

int tmem_columns(int need) { return need <= 64 ? 64 : need <= 128 ? 128 : need <= 256 ? 256 : 512; }

// the weight image: chunk (o, channels) of npad x 8 cc bf16 (cc channels), element (n, k) of the
// K-major operand at (n / 8) * 64 cc + (k / 8) * 64 + (n % 8) * 8 + k % 8; n = 8 c' + 2 s' +
// (0 re, 1 im), k = 8 (c within the chunk) + 2 s + (0 re, 1 im)
__global__ void k_ptc_tc_image(__nv_bfloat16 *__restrict__ img, const __nv_bfloat162 *__restrict__ w, int cin, int cout,
                               int npad, long total) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int cc = chunk_channels(cin), ncp = channel_chunks(cin), per = npad * 8 * cc;
    const int e = (int)(i % per), chunk = (int)(i / per), o = chunk / ncp, p = chunk % ncp;
    const int n = (e / (64 * cc)) * 8 + (e / 8) % 8, k = ((e / 64) % cc) * 8 + e % 8;
    const int co = n / 8, so = (n % 8) / 2, io = n % 2, ci = p * cc + k / 8, si = (k % 8) / 2, ii = k % 2;
    __nv_bfloat16 v = __float2bfloat16_rn(0.f);
    if (co < cout && ci < cin && k / 8 < cc) {
        const __nv_bfloat162 z = w[(((size_t)o * cout + co) * cin + ci) * 16 + 4 * so + si];
        v = io == ii ? z.x : io == 1 ? z.y : __hneg(z.y);
    }
    img[i] = v;
}

int stage_bytes_of(int cin, int cout) { return chunk_channels(cin) * 128 * (3 * 16 + npad_of(cout) / 8); }

}  // namespace

size_t ptc_tc_image_size(int cin, int cout) {
    return (size_t)9 * channel_chunks(cin) * npad_of(cout) * 8 * chunk_channels(cin);
}

// The tensor-core kernel pads the output channels to N = 16 at least and fills the same operands
// however few there are, so its time hardly depends on C_out, while the CUDA cores' goes with C_in
// C_out.  us on 16^4 with 4 vectors, tensor cores / CUDA cores: 1 -> 4 318 / 144, 1 -> 8 331 /
// 283, 1 -> 9 350 / 449; 2 -> 4 309 / 245, 2 -> 5 315 / 405; 3 -> 4 447 / 346, 3 -> 5 451 / 558; 4
// -> 3 450 / 434, 4 -> 4 450 / 451; 8 -> 3 868 / 805, 8 -> 4 868 / 866; 16 -> 1 1401 / 650.
// Below 4096 sites both are bound by latency: 8^4 with 1 vector 1 -> 4 and 1 -> 8 13 / 17 (with 4
// vectors 27 / 17 and 28 / 22), 4^4 12 / 16.  The rule does not look at the number of vectors: a
// vector's result is the same in every batch.
bool ptc_tc_layer(int cin, int cout, int sites) {
    return cout >= (sites < 4096 ? 4 : cin == 1 ? 9 : cin < 4 ? 5 : 4);
}

int ptc_tc_prepare() {
    static int done = 0;
    if (done) return DLZ_OK;
    DLZ_CUDA_TRY(cudaFuncSetAttribute(k_ptc_tc_fwd, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      kGroups * stage_bytes_of(6, 16)));
    DLZ_CUDA_TRY(cudaFuncSetAttribute(k_ptc_tc_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      kGroups * grad_stage_bytes(16)));
    done = 1;
    return DLZ_OK;
}

int ptc_tc_image(Op &op, __nv_bfloat16 *img, const __nv_bfloat162 *w, int cin, int cout) {
    const long total = (long)ptc_tc_image_size(cin, cout);
    k_ptc_tc_image<<<(unsigned)((total + 255) / 256), 256, 0, op.stream>>>(img, w, cin, cout, npad_of(cout), total);
    op.prof.launches++;
    DLZ_CUDA_TRY(cudaGetLastError());
    return DLZ_OK;
}

int ptc_tc_forward(Op &op, float4 *out, const float4 *in, const __nv_bfloat16 *img, int cin, int cout, int nvec,
                   PtcStatus status) {
    FwdArgs a;
    a.out = out; a.in = in; a.U = op.gauge32.as<float4>(); a.img = img; a.g = op.g;
    a.cin = cin; a.cout = cout; a.npad = npad_of(cout); a.nvec = nvec; a.status = status;
    a.nbuf = 4;
    const int need = a.npad * a.nbuf;
    a.ncols = tmem_columns(need);
    const long tiles = (long)((op.g.V + kSites - 1) / kSites) * nvec;
    int dev = 0, nsm = 0;
    DLZ_CUDA_TRY(cudaGetDevice(&dev));
    DLZ_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    k_ptc_tc_fwd<<<(unsigned)std::min<long>(tiles, nsm), kThreads, kGroups * stage_bytes_of(cin, cout), op.stream>>>(a);
    op.prof.launches++;
    DLZ_CUDA_TRY(cudaGetLastError());
    return DLZ_OK;
}

int ptc_tc_wgrad(Op &op, float2 *partials, const float4 *gout, const float4 *in, int cin, int cout, int nvec, PtcStatus status,
                 int &blocks) {
    GradArgs a;
    a.partials = partials; a.gout = gout; a.in = in; a.U = op.gauge32.as<float4>(); a.g = op.g;
    a.cin = cin; a.cout = cout; a.npad = npad_of(cin); a.nvec = nvec; a.status = status;
    a.nbuf = 4;
    a.ncols = tmem_columns(a.npad * a.nbuf);
    // nine offsets share the SMs
    const long tiles = (long)((op.g.V + kGSites - 1) / kGSites) * nvec;
    int dev = 0, nsm = 0;
    DLZ_CUDA_TRY(cudaGetDevice(&dev));
    DLZ_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    blocks = (int)std::max<long>(1, std::min<long>({tiles, (long)nsm / 9, (long)kPtcMaxGradBlocks}));
    k_ptc_tc_wgrad<<<dim3(blocks, 9), kThreads, kGroups * grad_stage_bytes(cin), op.stream>>>(a);
    op.prof.launches++;
    DLZ_CUDA_TRY(cudaGetLastError());
    return DLZ_OK;
}

}  // namespace dlz
