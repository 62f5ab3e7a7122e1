// Tensor-core (tcgen05) products of the Krylov basis, FP32 data with 3xTF32 splitting:
// the Rayleigh-Ritz restart V_{k+1} = V_{m+1} P of Lan-DR / MinRes-DR (arXiv:0901.3163,
// Sec. 1-2) and the Galerkin projection of D-CG / D-MinRes, C = V_k^dag R and
// E = V_k C' for a batch of right-hand sides (Sec. 2: projection at the start, repeated
// at every defect-correction restart).
//
// Both are dense contractions whose intensity (tens of flops per byte) is above the FP32
// CUDA-core ridge, so they run on the 5th-generation tensor cores: operands staged in
// shared memory, one thread issues tcgen05.mma (kind::tf32, M = 128), the accumulator
// lives in tensor memory and is read back with tcgen05.ld.  FP32 accuracy comes from
// splitting each operand x = hi + lo with hi = tf32(x) and lo = x - hi, and summing
// hi*hi + hi*lo + lo*hi (the lo*lo term is below FP32 rounding), all accumulated in FP32.
//
// Shared-memory operand layout (both operands K-major, no swizzle, 8-row x 16-byte
// core matrices): element (row, k) of a 32-wide K chunk at
//   (row / 8) * 1024 + (k / 4) * 128 + (row % 8) * 16 + (k % 4) * 4 bytes;
// descriptor: leading byte offset 128 (the next 4 k), stride byte offset 1024 (the next
// 8 rows); an MMA's K step of 8 advances the start address by 256 bytes.  The basis
// vectors are contiguous along the rows of the combine's A operand, so its staging
// transposes 4 x 4 blocks in registers.
// Every mbarrier wait is bounded: a wait that gives up sets an error word (reported as
// DLZ_ERR_DEVICE_TIMEOUT) and the kernel still frees its tensor memory.
#include <algorithm>
#include <cstdint>
#include <cstring>
#include <vector>

#include "dlz_internal.cuh"
#include "tc_util.cuh"

namespace dlz {

namespace {

// Warps of a block: the first kEpiWarps read the accumulators (warp w: TMEM lane quarter w % 4)
// and store the results, the next one issues the MMAs, four copy raw FP32 chunks into a ring of
// shared-memory slots, and S groups of four warps split them into the operand stages, group g the chunks
// g, g + S, ... into stage g.  They meet only at mbarriers, so copies, splits, MMAs and stores
// of different chunks overlap.  The restart of 121 vectors of 16^3 x 32 to 61, and the dots
// of 121 with 16 vectors (ncu, one GB300): 1.81 and 0.93 ms with one role for all threads, two
// block barriers per chunk and one chunk loaded ahead; 0.66 and 0.71 ms with roles but the
// splitting warps copying their own chunks; 0.62 and 0.64 ms in this form (3.7 and 2.7 TB/s).
// No single stage bounds it now: without its copies the combine takes 0.61 ms, with a twelfth
// of its MMAs 0.53 ms, without its split stores 0.66 ms.
constexpr int kEpiWarps = 8;
constexpr int kFill = 128;                                   // threads of a group, and of the copying warps
constexpr int tc_threads(int groups) { return 32 * (kEpiWarps + 1) + (groups + 1) * kFill; }
constexpr int kKC = 32;             // K chunk staged per pipeline stage
constexpr int kTcMaxSmem = 226 * 1024;      // dynamic shared memory a block may ask for
constexpr int kABytes = 128 * kKC * 4;      // one part (hi or lo) of an A chunk

// instruction descriptor: D FP32 (bits 4-5), A and B TF32 (7-9, 10-12), both K-major
// (bits 15, 16 zero), N / 8 (17-22), M / 16 (24-28) with M = 128
__device__ __forceinline__ uint32_t idesc_tf32(int n, uint32_t a_mn) {
    return (1u << 4) | (2u << 7) | (2u << 10) | (a_mn << 15) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

template <bool ACC>
__device__ __forceinline__ void mma_tf32(uint32_t taddr, uint32_t da, uint32_t db, uint32_t idesc, bool acc = true) {
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\tmov.b64 a, {%1, %5};\n\tmov.b64 b, {%2, %5};\n\t"
                 "setp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::tf32 [%0], a, b, %3, p;\n\t}\n" ::"r"(taddr),
                 "r"(da), "r"(db), "r"(idesc), "r"(ACC ? 1u : (acc ? 1u : 0u)), "r"(kDescHi<1024>));
}

// Asynchronous 16-byte copy of the raw ring; valid = false fills the slot with zeros.
__device__ __forceinline__ void ring_load(float4 *slot, const float *src, bool valid) {
    asm volatile("cp.async.cg.shared.global.L2::256B [%0], [%1], 16, %2;" ::"r"(su32(slot)), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}
// arrive on mbar once this thread's copies so far have landed
__device__ __forceinline__ void ring_arrive(uint64_t *mbar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(su32(mbar)) : "memory");
}

// x rounded to TF32 (10 mantissa bits, nearest, ties away from zero) by two integer operations
__device__ __forceinline__ float tf32_hi(float x) {
    return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xffffe000u);
}

__device__ __forceinline__ void tmem_wait(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]));
}
// columns addr .. addr + 15, or the first 8 of them
__device__ __forceinline__ void tmem_read(uint32_t addr, bool wide, float (&v)[16]) {
    uint32_t r[16] = {};
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(addr));
    if (wide)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                     : "r"(addr + 8));
    tmem_wait(r);
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

__device__ __forceinline__ void st_split(float *hi, float *lo, int off_floats, float4 v) {
    const float4 h = make_float4(tf32_hi(v.x), tf32_hi(v.y), tf32_hi(v.z), tf32_hi(v.w));
    *reinterpret_cast<float4 *>(hi + off_floats) = h;
    *reinterpret_cast<float4 *>(lo + off_floats) = make_float4(v.x - h.x, v.y - h.y, v.z - h.z, v.w - h.w);
}

// ------------------------------------------------------------------ combine
// Out[j][r] = sum_k A[r][k] Bt[j][k] for r in [0, rows), j in [0, nout), with
//   A[r][k] = V_k[r] (k < nin) and, for complex coefficients (cplx), A[r][nin + i] =
//   (i V_i)[r] (re <- -im, im <- re of each complex pair), so that Bt = [Re C'^T | Im C'^T]
//   gives Out = V C' for complex C'.  Bt (npad x kpad, K contiguous) comes split in hi, lo.
struct CombineArgs {
    const float *V;
    long ldv;          // floats between consecutive input vectors
    int nin;
    long rows;         // floats per vector (a multiple of 4)
    const float *Bhi, *Blo;
    int kpad, npad, nout, cplx;
    float *Out;
    long ldo;
    int *err;
};

// The block's synchronisation.  Ring slot r of R: raw_full[r] completes when every copying
// thread's part has landed, raw_empty[r] when the group that took it has read it.  Operand
// stage s of S: full[s] when every warp of its group has written it, empty[s] when the MMAs
// that read it are done.  Accumulator a of two: acc_full[a] when a tile's MMAs are done,
// acc_empty[a] when it has been read; drained when no MMA is in flight any more.  A wait on a phase's parity is only right while the
// waiter is at most one phase behind: each stage has a group of its own, and R is a multiple
// of S, so that one group takes all chunks of a slot.
template <int S, int R> struct TcShared {
    static_assert(R % S == 0, "ring slots per group");
    uint64_t raw_full[R], raw_empty[R], full[S], empty[S], acc_full[2], acc_empty[2], drained;
    uint32_t tbase;
    int failed;
};

// barriers, and `ncols` columns of tensor memory (warp 0); returns their address
template <int S, int R> __device__ __forceinline__ uint32_t tc_setup(TcShared<S, R> &sh, int ncols) {
    if (threadIdx.x == 0) {
        sh.failed = 0;
        for (int i = 0; i < R; ++i) {
            mbar_init(&sh.raw_full[i], kFill);
            mbar_init(&sh.raw_empty[i], kFill / 32);
        }
        for (int i = 0; i < S; ++i) {
            mbar_init(&sh.full[i], kFill / 32);
            mbar_init(&sh.empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sh.acc_full[i], 1);
            mbar_init(&sh.acc_empty[i], kEpiWarps);
        }
        mbar_init(&sh.drained, 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    tmem_alloc(&sh.tbase, ncols);
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    return sh.tbase;
}

// One chunk's MMAs into the accumulator at `acc`: hi hi + hi lo + lo hi over 32 k, from the
// low words of the operands' descriptors.  (The issuing warp is kept uniform, one lane issuing:
// a lone thread that built every descriptor took longer than the MMAs.)
__device__ __forceinline__ void chunk_mmas(uint32_t acc, uint32_t ah, uint32_t al, uint32_t bh, uint32_t bl,
                                           uint32_t idesc, bool first) {
#pragma unroll
    for (int ks = 0; ks < kKC / 8; ++ks) {
        const uint32_t k = ks * (256 >> 4);
        if (ks == 0) mma_tf32<false>(acc, ah, bh, idesc, !first);
        else mma_tf32<true>(acc, ah + k, bh + k, idesc);
        mma_tf32<true>(acc, ah + k, bl + k, idesc);
        mma_tf32<true>(acc, al + k, bh + k, idesc);
    }
}


// The combine's A operand, item (row quad, k quad kq) of a chunk: vectors 4 kq .. 4 kq + 3 of
// K chunk kc at rows r .. r + 3 (zero beyond the data; for complex coefficients the second
// half of K holds i times the vectors, made by combine_take_a)
__device__ __forceinline__ void combine_load_a(const CombineArgs &a, int kc, int kq, long r, float4 *slot) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int k = kc * kKC + 4 * kq + j;
        const int v = k < a.nin ? k : k - a.nin;
        const bool ok = r < a.rows && (k < a.nin || (a.cplx && k < 2 * a.nin));
        ring_load(slot + j * kFill, ok ? a.V + (size_t)v * a.ldv + r : a.V, ok);
    }
}
__device__ __forceinline__ void combine_take_a(const CombineArgs &a, int kc, int kq, const float4 *slot, float4 (&v)[4]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float4 u = slot[j * kFill];
        v[j] = kc * kKC + 4 * kq + j < a.nin ? u : make_float4(-u.y, u.x, -u.w, u.z);   // i times the complex pairs
    }
}

// Bound by memory: (nin + nout) vectors move.  Shared memory is next: a chunk's 16 KB pass
// it as raw copy, read, two split parts and three MMA operand reads, about 1000 cycles of
// the SM against 740 of its share of the memory bandwidth for the reads alone.  RES: both
// parts of the coefficient matrix stay in shared memory for the whole kernel (when they fit
// beside two stages); otherwise every chunk's part is copied from L2.
template <int S, int R, bool RES>
__global__ void __launch_bounds__(tc_threads(S), 1) k_tc_combine(CombineArgs a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) TcShared<S, R> sh;
    const int b_bytes = a.npad * kKC * 4;
    const int stage_bytes = 2 * kABytes + (RES ? 0 : 2 * b_bytes);
    const int nkc = a.kpad / kKC;
    float4 *ring = reinterpret_cast<float4 *>(smem + S * stage_bytes);             // [R][2 x 4][kFill]
    unsigned char *bres = smem + S * stage_bytes + R * kABytes;                    // RES: [nkc][hi, lo]
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int ncols = tmem_cols(2 * a.npad);
    const long ntiles = (a.rows + 127) / 128;
    // B chunk kc: npad rows (outputs) x 32 k, K-major, from the pre-split global copies
    auto load_b = [&](int kc, unsigned char *dst, int t0, int nt) {
        float *Bhi = reinterpret_cast<float *>(dst), *Blo = reinterpret_cast<float *>(dst + b_bytes);
        for (int w = t0; w < a.npad * (kKC / 4); w += nt) {
            const int j = w % a.npad, q = w / a.npad;                        // k = 4 q .. 4 q + 3
            const size_t gi = (size_t)j * a.kpad + kc * kKC + 4 * q;
            const int off = (j / 8) * 256 + q * 32 + (j % 8) * 4;
            *reinterpret_cast<float4 *>(Bhi + off) = *reinterpret_cast<const float4 *>(a.Bhi + gi);
            *reinterpret_cast<float4 *>(Blo + off) = *reinterpret_cast<const float4 *>(a.Blo + gi);
        }
    };
    if (RES) {
        for (int kc = 0; kc < nkc; ++kc) load_b(kc, bres + (size_t)kc * 2 * b_bytes, threadIdx.x, blockDim.x);
        asm volatile("fence.proxy.async.shared::cta;");
    }
    const uint32_t taddr = tc_setup(sh, ncols);
    volatile int *failed = &sh.failed;
    // A chunk: 128 rows x 32 k.  Item (row quad rq, k quad kq): the four vectors 4 kq .. 4 kq
    // + 3 at rows 4 rq .. 4 rq + 3 (float4 each, 128 contiguous bytes per vector across the 8
    // lanes of equal kq); a thread takes the row quads rq and rq + 16.
    const int ft = threadIdx.x - 32 * (kEpiWarps + 1), tid = ft % kFill;
    const int rq = (tid & 7) + 8 * (tid >> 6), kq = (tid >> 3) & 7;
    float4 *slots = ring + tid;
    const long mine = ((ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x) * nkc;   // the block's chunks
    if (ft >= kFill) {
        // ---- split.  An item is a 4 x 4 block, transposed and stored K-major as one 16-byte
        // k quad per row; a lane stores its rows in the order (c + rot) so that the eight
        // lanes of a store phase (rq = 0 .. 7) hit eight different 16-byte banks.
        const int grp = ft / kFill - 1, rot = (tid >> 1) & 3;
        unsigned char *sbase = smem + grp * stage_bytes;
        float *Ahi = reinterpret_cast<float *>(sbase), *Alo = reinterpret_cast<float *>(sbase + kABytes);
        int kc = grp % nkc, slot = grp;
        uint32_t round = 0, rround = 0;        // uses of the stage and of the slot before this one
        for (long q = grp; q < mine; q += S, ++round) {
            const float4 *raw = slots + (size_t)slot * 8 * kFill;
            if (!__all_sync(0xffffffffu, mbar_wait(&sh.raw_full[slot], rround & 1u, failed))) break;
            if (round > 0 && !__all_sync(0xffffffffu, mbar_wait(&sh.empty[grp], (round - 1) & 1u, failed))) break;
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                float4 v[4];
                combine_take_a(a, kc, kq, raw + half * 4 * kFill, v);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int cc = (c + rot) & 3;                             // the row this lane stores now
                    float4 w4;
                    w4.x = cc == 0 ? v[0].x : cc == 1 ? v[0].y : cc == 2 ? v[0].z : v[0].w;
                    w4.y = cc == 0 ? v[1].x : cc == 1 ? v[1].y : cc == 2 ? v[1].z : v[1].w;
                    w4.z = cc == 0 ? v[2].x : cc == 1 ? v[2].y : cc == 2 ? v[2].z : v[2].w;
                    w4.w = cc == 0 ? v[3].x : cc == 1 ? v[3].y : cc == 2 ? v[3].z : v[3].w;
                    const int row = 4 * rq + 64 * half + cc;
                    st_split(Ahi, Alo, (row >> 3) * 256 + kq * 32 + (row & 7) * 4, w4);
                }
            }
            if (!RES) load_b(kc, sbase + 2 * kABytes, tid, kFill);
            asm volatile("fence.proxy.async.shared::cta;");
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&sh.raw_empty[slot]);
                mbar_arrive(&sh.full[grp]);
            }
            for (kc += S; kc >= nkc;) kc -= nkc;
            if ((slot += S) >= R) { slot = grp; ++rround; }
        }
    } else if (ft >= 0) {
        // ---- copy
        long t = blockIdx.x;
        int kc = 0, slot = 0;
        uint32_t round = 0;
        for (long q = 0; q < mine; ++q) {
            if (round > 0 && !mbar_wait(&sh.raw_empty[slot], (round - 1) & 1u, failed)) break;
            float4 *raw = slots + (size_t)slot * 8 * kFill;
            combine_load_a(a, kc, kq, t * 128 + 4 * rq, raw);
            combine_load_a(a, kc, kq, t * 128 + 4 * rq + 64, raw + 4 * kFill);
            ring_arrive(&sh.raw_full[slot]);
            if (++kc == nkc) { kc = 0; t += gridDim.x; }
            if (++slot == R) { slot = 0; ++round; }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");       // no copy may land after the block has ended
    } else if (warp == kEpiWarps) {
        // ---- MMA (the warp is uniform; lane 0 issues)
        const uint32_t idesc = idesc_tf32(a.npad, 0u);
        const uint32_t d_stage = sdesc_lo(su32(smem)), d_res = RES ? sdesc_lo(su32(bres)) : 0u;
        const uint32_t w_stage = stage_bytes >> 4, w_b = b_bytes >> 4;
        int st = 0, n = 0;
        uint32_t round = 0;
        bool ok = true, issued = false;
        for (long t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++n) {
            const int acc = n & 1;
            if (n >= 2 && !__all_sync(0xffffffffu, mbar_wait(&sh.acc_empty[acc], ((n >> 1) - 1) & 1, failed))) break;
            for (int kc = 0; kc < nkc; ++kc) {
                ok = __all_sync(0xffffffffu, mbar_wait(&sh.full[st], round & 1u, failed));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;");
                const uint32_t da = d_stage + st * w_stage;
                const uint32_t db = RES ? d_res + 2 * kc * w_b : da + (2 * kABytes >> 4);
                if (lane == 0) {
                    chunk_mmas(taddr + acc * a.npad, da, da + (kABytes >> 4), db, db + w_b, idesc, kc == 0);
                    commit_to(&sh.empty[st]);
                    issued = true;
                }
                if (++st == S) { st = 0; ++round; }
            }
            if (ok && lane == 0) commit_to(&sh.acc_full[acc]);
        }
        mma_drain(&sh.drained, issued, failed);
    } else {
        // ---- results: warp w reads rows 32 (w % 4) .. of each tile, half of the columns (with
        // four warps and 8 columns per read the stores, not the loads, set the pace)
        int n = 0;
        const int lq = warp & 3, c_lo = (warp >> 2) * (a.npad / 2), c_hi = min(c_lo + a.npad / 2, a.nout);
        for (long t = blockIdx.x; t < ntiles; t += gridDim.x, ++n) {
            const int acc = n & 1;
            if (!__all_sync(0xffffffffu, mbar_wait(&sh.acc_full[acc], (n >> 1) & 1, failed))) break;
            asm volatile("tcgen05.fence::after_thread_sync;");
            const long r = t * 128 + 32 * lq + lane;
            for (int c0 = c_lo; c0 < c_hi; c0 += 16) {
                float v[16];
                tmem_read(taddr + ((uint32_t)(32 * lq) << 16) + (uint32_t)(acc * a.npad + c0), c0 + 8 < c_lo + a.npad / 2, v);
                float *o = a.Out + (size_t)c0 * a.ldo + r;
                if (r < a.rows) {
#pragma unroll
                    for (int j = 0; j < 16; ++j, o += a.ldo)
                        if (c0 + j < c_hi) *o = v[j];
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.acc_empty[acc]);
        }
    }
    __syncthreads();
    if (sh.failed && threadIdx.x == 0) atomicExch(a.err, 1);
    tc_teardown(taddr, ncols);
}

// ------------------------------------------------------------------ dots
// Cpart[blk][i][c] (FP64) = sum over this block's segments of A[i][k] B[c][k], k running
// over the floats of the vectors: A rows = the nin basis vectors (rows >= nin are zero),
// B rows c < nq = R_c, nq <= c < 2 nq = rot(R_{c-nq}) with (re, im) -> (im, -re), so that
// for complex vectors sum_k A[i][k] B[c][k] = Re <v_i, r_c> and the rotated rows give
// Im <v_i, r_c>.  After each segment of kSegChunks chunks the FP32 accumulator is added into
// FP64 registers and the next segment starts afresh.
struct DotsArgs {
    const float *V;
    long ldv;
    int nin;
    const float *R;
    long ldr;
    int nq, npad;
    long len;          // floats per vector (a multiple of 32)
    double *Cpart;     // [gridDim.x][128][npad]
    int *err;
};
constexpr int kSegChunks = 64;      // 64 chunks of 32 floats per segment

// The dots' operands of one thread of a group for chunk ch: A items w = tid + 128 i (i < 8;
// row 8 (w >> 6) + (w & 7), k quad (w >> 3) & 7), and B items w = tid + 128 i < 8 npad (i < 2;
// rows nq .. 2 nq - 1 are rotated when taken from the ring)
__device__ __forceinline__ void dots_load(const DotsArgs &a, long ch, int tid, float4 *slot) {
    const long k0 = ch * kKC;
#pragma unroll
    for (int q = 0; q < 10; ++q) {
        const int w = tid + kFill * (q < 8 ? q : q - 8);
        if (q >= 8 && w >= a.npad * (kKC / 4)) break;
        const int i = 8 * (w >> 6) + (w & 7), kq = (w >> 3) & 7;
        const float *src = a.V;
        bool ok;
        if (q < 8) {
            ok = i < a.nin;
            if (ok) src = a.V + (size_t)i * a.ldv + k0 + 4 * kq;
        } else {
            ok = i < 2 * a.nq;
            if (ok) src = a.R + (size_t)(i < a.nq ? i : i - a.nq) * a.ldr + k0 + 4 * kq;
        }
        ring_load(slot + q * kFill, src, ok);
    }
}

// Bound by memory: nin + nq vectors are read, 128 x npad partial sums written per block.
// Every block takes consecutive segments, one FP32 accumulation of kSegChunks chunks each.
constexpr int kDotsStages = 2, kDotsRing = 6;
__global__ void __launch_bounds__(tc_threads(kDotsStages), 1) k_tc_dots(DotsArgs a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) TcShared<kDotsStages, kDotsRing> sh;
    const int b_bytes = a.npad * kKC * 4;
    const int stage_bytes = 2 * kABytes + 2 * b_bytes;
    float4 *ring = reinterpret_cast<float4 *>(smem + kDotsStages * stage_bytes);   // [ring][8 A + 2 B][kFill]
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int ncols = tmem_cols(2 * a.npad);
    const long nchunks = a.len / kKC, nseg = (nchunks + kSegChunks - 1) / kSegChunks;
    const long first = nseg * blockIdx.x / gridDim.x * kSegChunks;
    const long last = min(nchunks, nseg * (blockIdx.x + 1) / gridDim.x * kSegChunks);
    const uint32_t taddr = tc_setup(sh, ncols);
    volatile int *failed = &sh.failed;
    const int ft = threadIdx.x - 32 * (kEpiWarps + 1), tid = ft % kFill;
    float4 *slots = ring + tid;
    const long mine = last - first;
    if (ft >= kFill) {
        // ---- split.  A chunk: 128 rows x 32 k, K-major; a warp instruction covers 8 rows x 4
        // k quads
        const int grp = ft / kFill - 1;
        unsigned char *sbase = smem + grp * stage_bytes;
        float *Ahi = reinterpret_cast<float *>(sbase), *Alo = reinterpret_cast<float *>(sbase + kABytes);
        float *Bhi = reinterpret_cast<float *>(sbase + 2 * kABytes);
        float *Blo = reinterpret_cast<float *>(sbase + 2 * kABytes + b_bytes);
        int slot = grp;
        uint32_t round = 0, rround = 0;        // uses of the stage and of the slot before this one
        for (long q = grp; q < mine; q += kDotsStages, ++round) {
            const float4 *raw = slots + (size_t)slot * 10 * kFill;
            if (!__all_sync(0xffffffffu, mbar_wait(&sh.raw_full[slot], rround & 1u, failed))) break;
            if (round > 0 && !__all_sync(0xffffffffu, mbar_wait(&sh.empty[grp], (round - 1) & 1u, failed))) break;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int w = tid + kFill * k;
                st_split(Ahi, Alo, (w >> 6) * 256 + ((w >> 3) & 7) * 32 + (w & 7) * 4, raw[k * kFill]);
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int w = tid + kFill * k;
                if (w < a.npad * (kKC / 4)) {
                    float4 u = raw[(8 + k) * kFill];
                    if (8 * (w >> 6) + (w & 7) >= a.nq) u = make_float4(u.y, -u.x, u.w, -u.z);
                    st_split(Bhi, Blo, (w >> 6) * 256 + ((w >> 3) & 7) * 32 + (w & 7) * 4, u);
                }
            }
            asm volatile("fence.proxy.async.shared::cta;");
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&sh.raw_empty[slot]);
                mbar_arrive(&sh.full[grp]);
            }
            if ((slot += kDotsStages) >= kDotsRing) { slot = grp; ++rround; }
        }
    } else if (ft >= 0) {
        // ---- copy
        int slot = 0;
        uint32_t round = 0;
        for (long q = 0; q < mine; ++q) {
            if (round > 0 && !mbar_wait(&sh.raw_empty[slot], (round - 1) & 1u, failed)) break;
            dots_load(a, first + q, tid, slots + (size_t)slot * 10 * kFill);
            ring_arrive(&sh.raw_full[slot]);
            if (++slot == kDotsRing) { slot = 0; ++round; }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");       // no copy may land after the block has ended
    } else if (warp == kEpiWarps) {
        // ---- MMA: one accumulator per segment (the warp is uniform; lane 0 issues)
        const uint32_t idesc = idesc_tf32(a.npad, 0u);
        const uint32_t d_stage = sdesc_lo(su32(smem)), w_stage = stage_bytes >> 4, w_b = b_bytes >> 4;
        int st = 0, n = 0;
        uint32_t round = 0;
        bool ok = true, issued = false;
        for (long ch0 = first; ch0 < last && ok; ch0 += kSegChunks, ++n) {
            const int acc = n & 1, nch = (int)(min(last, ch0 + kSegChunks) - ch0);
            if (n >= 2 && !__all_sync(0xffffffffu, mbar_wait(&sh.acc_empty[acc], ((n >> 1) - 1) & 1, failed))) break;
            for (int ch = 0; ch < nch; ++ch) {
                ok = __all_sync(0xffffffffu, mbar_wait(&sh.full[st], round & 1u, failed));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;");
                const uint32_t da = d_stage + st * w_stage, db = da + (2 * kABytes >> 4);
                if (lane == 0) {
                    chunk_mmas(taddr + acc * a.npad, da, da + (kABytes >> 4), db, db + w_b, idesc, ch == 0);
                    commit_to(&sh.empty[st]);
                    issued = true;
                }
                if (++st == kDotsStages) { st = 0; ++round; }
            }
            if (ok && lane == 0) commit_to(&sh.acc_full[acc]);
        }
        mma_drain(&sh.drained, issued, failed);
    } else {
        // ---- sums over the segments in FP64: a thread has one row (basis vector) and half of
        // the columns
        double sum[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) sum[j] = 0.0;
        int n = 0;
        const int lq = warp & 3, c_lo = (warp >> 2) * (a.npad / 2);
        for (long ch0 = first; ch0 < last; ch0 += kSegChunks, ++n) {
            const int acc = n & 1;
            if (!__all_sync(0xffffffffu, mbar_wait(&sh.acc_full[acc], (n >> 1) & 1, failed))) break;
            asm volatile("tcgen05.fence::after_thread_sync;");
            float v[16];
            tmem_read(taddr + ((uint32_t)(32 * lq) << 16) + (uint32_t)(acc * a.npad + c_lo), a.npad == 32, v);
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (j < a.npad / 2) sum[j] += (double)v[j];
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.acc_empty[acc]);
        }
        double *out = a.Cpart + ((size_t)blockIdx.x * 128 + 32 * lq + lane) * a.npad + c_lo;
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (j < a.npad / 2) out[j] = sum[j];
    }
    __syncthreads();
    if (sh.failed && threadIdx.x == 0) atomicExch(a.err, 1);
    tc_teardown(taddr, ncols);
}

// C[i][q] (complex) = sum over blocks of Cpart[blk][i][q] + i Cpart[blk][i][nq + q], in a
// fixed order.  One block per basis vector i; its threads are (group of partials, column),
// so a group's reads are one contiguous row (one thread per entry, striding over all blocks'
// partials, took 156 us for 121 x 16 entries).
__global__ void __launch_bounds__(256)
k_tc_dots_sum(const double *__restrict__ Cpart, int nblk, int nin, int nq, int npad, double2 *__restrict__ C) {
    __shared__ double sm[256];
    const int i = blockIdx.x, col = threadIdx.x % npad, grp = threadIdx.x / npad, ngrp = 256 / npad;
    double t = 0.0;
    for (int b = grp; b < nblk; b += ngrp) t += Cpart[((size_t)b * 128 + i) * npad + col];
    sm[threadIdx.x] = t;
    __syncthreads();
    if ((int)threadIdx.x >= nq) return;
    double re = 0.0, im = 0.0;
    for (int k = 0; k < ngrp; ++k) {
        re += sm[k * npad + threadIdx.x];
        im += sm[k * npad + nq + threadIdx.x];
    }
    C[(size_t)threadIdx.x * nin + i] = make_double2(re, im);
}

// round to the 10-bit TF32 mantissa (nearest, ties away), as cvt.rna.tf32.f32 does
inline float tf32_round_host(float x) {
    uint32_t u;
    std::memcpy(&u, &x, 4);
    if ((u & 0x7f800000u) != 0x7f800000u) u = (u + 0x1000u) & 0xffffe000u;
    float r;
    std::memcpy(&r, &u, 4);
    return r;
}

inline int round_up(int v, int m) { return (v + m - 1) / m * m; }

int num_sms() {
    static int n = 0;
    if (!n) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            n = 148;
    }
    return n;
}

constexpr size_t kErrBytes = 256;      // the error word at the start of a call's scratch

// The combine's launch: stages, raw chunks in the ring, and whether the coefficients stay in
// shared memory (with as many raw chunks as fit beside them) or are copied per chunk
typedef void (*CombineKernel)(CombineArgs);
struct CombineForm {
    CombineKernel fn;
    int stages, smem;
};
CombineForm pick_combine(int npad, int kpad) {
    const int b_all = 2 * npad * kpad * 4, b_stage = 2 * npad * kKC * 4;
    // hi and lo of an A chunk per stage, R raw chunks
    if (10 * kABytes + b_all <= kTcMaxSmem) return {k_tc_combine<2, 6, true>, 2, 10 * kABytes + b_all};
    if (8 * kABytes + b_all <= kTcMaxSmem) return {k_tc_combine<2, 4, true>, 2, 8 * kABytes + b_all};
    if (10 * kABytes + 2 * b_stage <= kTcMaxSmem) return {k_tc_combine<2, 6, false>, 2, 10 * kABytes + 2 * b_stage};
    if (8 * kABytes + 2 * b_stage <= kTcMaxSmem) return {k_tc_combine<2, 4, false>, 2, 8 * kABytes + 2 * b_stage};
    return {k_tc_combine<1, 4, false>, 1, 6 * kABytes + b_stage};
}

}  // namespace

int tc_prepare() {
    // dynamic shared memory beyond 48 KB (set once, outside any graph capture); the opt-in
    // limit (227 KB) also covers the kernels' static shared memory
    static int done = 0;
    if (done) return DLZ_OK;
    for (CombineKernel k : {(CombineKernel)k_tc_combine<2, 6, true>, (CombineKernel)k_tc_combine<2, 4, true>,
                            (CombineKernel)k_tc_combine<2, 6, false>, (CombineKernel)k_tc_combine<2, 4, false>,
                            (CombineKernel)k_tc_combine<1, 4, false>})
        DLZ_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcMaxSmem));
    DLZ_CUDA_TRY(cudaFuncSetAttribute(k_tc_dots, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcMaxSmem));
    done = 1;
    return DLZ_OK;
}

// Both calls keep everything they need on the device in one allocation of the scratch (the
// error word first), and read the error word back with the results.
int tc_combine32(TcScratch &sc, cudaStream_t st, float *out, long ldo, const float *in, long ldv, int nin, long len,
                 const double *coef, int nout, bool cplx, long long *launches) {
    if (nin < 1 || nout < 1 || len < 1) return DLZ_OK;
    if (len % 4 || ldv % 4 || ldo % 4 || nout > 256) return fail(DLZ_ERR_BADARG, "tensor-core combine: shape");
    DLZ_TRY(tc_prepare());
    const int K = cplx ? 2 * nin : nin;
    const int kpad = round_up(K, kKC), npad = std::max(16, round_up(nout, 16));
    // the error word (0), then Bt[j][k] (K contiguous) in two parts: real coef[i][j] at
    // k = i; complex: Re at k = i, Im at k = nin + i
    const size_t nb = (size_t)npad * kpad, ne = kErrBytes / sizeof(float);
    std::vector<float> h(ne + 2 * nb, 0.f);
    float *hi = h.data() + ne, *lo = hi + nb;
    for (int j = 0; j < nout; ++j)
        for (int i = 0; i < nin; ++i) {
            const float re = (float)(cplx ? coef[2 * ((size_t)i * nout + j)] : coef[(size_t)i * nout + j]);
            const float hr = tf32_round_host(re);
            hi[(size_t)j * kpad + i] = hr;
            lo[(size_t)j * kpad + i] = re - hr;
            if (cplx) {
                const float im = (float)coef[2 * ((size_t)i * nout + j) + 1];
                const float hm = tf32_round_host(im);
                hi[(size_t)j * kpad + nin + i] = hm;
                lo[(size_t)j * kpad + nin + i] = im - hm;
            }
        }
    DLZ_TRY(sc.buf.reserve(h.size() * sizeof(float)));
    DLZ_CUDA_TRY(cudaMemcpyAsync(sc.buf.ptr(), h.data(), h.size() * sizeof(float), cudaMemcpyHostToDevice, st));
    CombineArgs a;
    a.V = in; a.ldv = ldv; a.nin = nin; a.rows = len; a.Bhi = sc.buf.as<float>() + ne; a.Blo = a.Bhi + nb;
    a.kpad = kpad; a.npad = npad; a.nout = nout; a.cplx = cplx ? 1 : 0; a.Out = out; a.ldo = ldo;
    a.err = sc.buf.as<int>();
    const CombineForm f = pick_combine(npad, kpad);
    const long ntiles = (len + 127) / 128;
    f.fn<<<(int)std::min<long>(ntiles, num_sms()), tc_threads(f.stages), f.smem, st>>>(a);
    if (launches) *launches += 1;
    DLZ_CUDA_TRY(cudaGetLastError());
    int err = 0;
    DLZ_CUDA_TRY(cudaMemcpyAsync(&err, sc.buf.ptr(), sizeof(int), cudaMemcpyDeviceToHost, st));
    DLZ_CUDA_TRY(cudaStreamSynchronize(st));
    if (err) return fail(DLZ_ERR_DEVICE_TIMEOUT, "a tensor-core kernel's mbarrier wait gave up");
    return DLZ_OK;
}

int tc_dots32(TcScratch &sc, cudaStream_t st, double2 *C_host, const float *V, long ldv, int nin, const float *R,
              long ldr, int nq, long len, long long *launches) {
    if (nin < 1 || nq < 1) return DLZ_OK;
    if (nin > 128 || nq > 16 || len % kKC || ldv % 4 || ldr % 4) return fail(DLZ_ERR_BADARG, "tensor-core dots: shape");
    DLZ_TRY(tc_prepare());
    const int npad = std::max(16, round_up(2 * nq, 16));
    const int smem = kDotsStages * (2 * kABytes + 2 * npad * kKC * 4) + kDotsRing * 10 * kFill * (int)sizeof(float4);
    static_assert(kDotsStages * (2 * kABytes + 2 * 32 * kKC * 4) + kDotsRing * 10 * kFill * 16 <= kTcMaxSmem, "ring depth");
    const long nseg = (len / kKC + kSegChunks - 1) / kSegChunks;
    const int grid = (int)std::max<long>(1, std::min<long>(nseg, num_sms()));
    const size_t ne = (size_t)nin * nq, npart = (size_t)grid * 128 * npad;
    DLZ_TRY(sc.buf.reserve(kErrBytes + ne * sizeof(double2) + npart * sizeof(double)));
    double2 *Cd = reinterpret_cast<double2 *>(sc.buf.as<char>() + kErrBytes);
    double *part = reinterpret_cast<double *>(Cd + ne);
    DLZ_CUDA_TRY(cudaMemsetAsync(sc.buf.ptr(), 0, sizeof(int), st));
    DotsArgs a;
    a.V = V; a.ldv = ldv; a.nin = nin; a.R = R; a.ldr = ldr; a.nq = nq; a.npad = npad; a.len = len;
    a.Cpart = part; a.err = sc.buf.as<int>();
    k_tc_dots<<<grid, tc_threads(kDotsStages), smem, st>>>(a);
    k_tc_dots_sum<<<nin, 256, 0, st>>>(part, grid, nin, nq, npad, Cd);
    if (launches) *launches += 2;
    DLZ_CUDA_TRY(cudaGetLastError());
    std::vector<char> h(kErrBytes + ne * sizeof(double2));
    DLZ_CUDA_TRY(cudaMemcpyAsync(h.data(), sc.buf.ptr(), h.size(), cudaMemcpyDeviceToHost, st));
    DLZ_CUDA_TRY(cudaStreamSynchronize(st));
    int err = 0;
    std::memcpy(&err, h.data(), sizeof(int));
    if (err) return fail(DLZ_ERR_DEVICE_TIMEOUT, "a tensor-core kernel's mbarrier wait gave up");
    std::memcpy(C_host, h.data() + kErrBytes, ne * sizeof(double2));
    return DLZ_OK;
}

}  // namespace dlz

// ------------------------------------------------------------------ C ABI (test and measurement)
extern "C" int dlz_basis_combine(const float *V, long long ldv, int nin, long long len, const double *coef, int nout,
                                 int cplx, float *out, long long ldo) {
    if (!V || !coef || !out || nin < 0 || nout < 0 || len < 0) return dlz::fail(DLZ_ERR_BADARG, "basis_combine arguments");
    dlz::TcScratch sc;
    return dlz::tc_combine32(sc, 0, out, (long)ldo, V, (long)ldv, nin, (long)len, coef, nout, cplx != 0, nullptr);
}

extern "C" int dlz_basis_dots(const float *V, long long ldv, int nin, const float *R, long long ldr, int nq,
                              long long len, double *C) {
    if (!V || !R || !C || nin < 0 || nq < 0 || len < 0) return dlz::fail(DLZ_ERR_BADARG, "basis_dots arguments");
    dlz::TcScratch sc;
    return dlz::tc_dots32(sc, 0, reinterpret_cast<double2 *>(C), V, (long)ldv, nin, R, (long)ldr, nq, (long)len, nullptr);
}
