// M2L translations on the 5th-generation tensor cores (tcgen05, TMEM accumulators).
//
// For one offset class c and a chunk of (source, target) pairs, the product
//   Y[pair, rhs][n] = sum_k T_c[n][k] X[src, rhs][k]
// is up to two MMA tiles D_t = A_t B^T with M = 128 rows (pair, rhs) each, N = K = K_c, the
// class's truncated size (p_c^2 rounded up to 16; P rounded up without truncation):
// A_t = gathered multipole rows, B = T_c (row n of T_c is K-contiguous, i.e. K-major). The
// tiles share every staged block of T_c, which divides its traffic; a chunk of a class with
// K_c <= 128 has two tiles (TMEM columns 128 apart), the others one, so the small truncated
// classes amortise a block's set-up and pipeline fill over more rows; a block takes half the SM's
// tensor memory, for two blocks per SM.
//
// Accuracy: both operands are split into three BF16 pieces, x = x0 + x1 + x2 (x0 = bf16(x),
// x1 = bf16(x - x0), x2 = bf16(x - x0 - x1)), and D accumulates in FP32 the six products with
// i + j <= 2: x0 y0 + (x0 y1 + x1 y0) + (x0 y2 + x1 y1 + x2 y0). The dropped terms and the
// rest of x beyond x2 are ~2^-24 of the product, so the translation is as accurate as an FP32
// product. (Translation sums cancel strongly, so a two-piece split leaves noise near 1e-6 in
// the operator, which a GMRES solve to 1e-6 cannot tolerate.) T_c is split once per operator
// build from its FP64 values; the multipoles are split once per product (k_split_x).
//
// Data movement: K advances 16 at a time (one kind::f16 MMA); each 16-wide K step is one
// pipeline stage holding A (tiles x 128 rows) and B (3 pieces x N_pad x 16). B has the canonical
// K-major layout without swizzle (8-row x 16-byte core matrices, K-adjacent core matrices 128 B
// apart, 8-row groups 256 B apart). The split multipoles lie in memory as they are gathered: per box
// and right-hand side, per K step, the three pieces side by side in one 128-byte line (96 bytes
// used); A keeps them so, one 128-byte row per tile row in the 128-byte-swizzled K-major layout (16-byte
// unit u of row r at u ^ (r % 8)), and an MMA takes piece i by starting 32 i bytes into the rows. With
// a plane per piece and no swizzle a copy brought one 32-byte sector of each of 16 rows, whose halves fell
// into the same banks: the target-major kernel at 192600 points wrote 20.6M wavefronts of copies where
// it now writes 13.9M, next to 16.2M of operand reads that fill the same pipe (M2L of 192600 points 144 ->
// 128 us, of 3.21M points 1268 -> 963, of the diagonal product at 963000 points 3303 -> 2908; the pipe is
// still 89 % busy and bounds the kernel). The block is warp-specialised: warps 1-7
// fill the stages with cp.async (16-byte copies; rows past the chunk read as zeros), two
// stages deep (three in the target-major kernel), and let each stage's "full"
// mbarrier count their copies' arrival (cp.async.mbarrier.arrive.noinc); one thread of warp 0
// waits on "full", issues the stage's MMAs and commits them to the stage's "empty" mbarrier,
// which releases the stage for refilling. No block-wide barrier runs inside the K loop. Every
// wait is bounded: one that runs out raises a shared abort flag that stops the other side at
// its next wait, sets the error flag, and the block waits (bounded) for its MMAs in flight
// before it releases its tensor memory. The same kernel serves the 4-RHS diagonal product
// (R = 4, N_pad up to 256).
#include <cuda_bf16.h>

#include "internal.h"
#include "tcgen05.cuh"

#include <algorithm>
#include <vector>

namespace bem {
namespace {

constexpr int TC_M = 128;        // rows per tile
constexpr int TC_MAXT = 2;       // tiles per block at most (same class, shared B stages)
constexpr int TC_SMALL_K = 128;  // classes truncated to at most this size take two tiles per block
constexpr uint32_t TC_AROW = 128;           // bytes of one row of A: the three pieces of a K step
constexpr uint32_t TC_ATILE = TC_M * TC_AROW;
// bytes of one pipeline stage: A and B (3 pieces x K_c x 16), for two tiles with K_c <= 128 or one
// tile with K_c <= 256 (the larger of the two)
constexpr size_t TC_STAGE_BYTES = 2 * TC_ATILE + 3 * 128 * 16 * 2;
static_assert(TC_STAGE_BYTES >= TC_ATILE + 3 * 256 * 16 * 2 && TC_STAGE_BYTES % 1024 == 0, "both forms fit");
constexpr int TC_TMEM = 256;  // TMEM columns of a block: half of the SM's, for two blocks per SM
constexpr int TC_THREADS = 256;  // 8 warps: two warp groups share the loads and the epilogue

// Row-major T_c [P][P] (FP64) -> per class, per 16-wide K step, per piece, an N_pad x 16
// block in the canonical K-major layout, zero-padded (n >= P or k >= P).
__global__ void k_build_tc_table(int P, int Npad, const double *__restrict__ T, __nv_bfloat16 *__restrict__ out) {
    const int cls = blockIdx.y;
    const int nsteps = Npad / TC_K;
    const size_t blk = (size_t)Npad * TC_K;  // one piece of one K step
    const size_t per_cls = blk * 3 * nsteps;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < blk * nsteps;
         e += (size_t)gridDim.x * blockDim.x) {
        const int ks = (int)(e / blk);
        const int rem = (int)(e % blk);
        // inverse of kmajor_off: rem = (n/8)*128 + (kk/8)*64 + (n%8)*8 + kk%8
        const int g = rem >> 7, r2 = rem & 127;
        const int j = r2 >> 6, r3 = r2 & 63;
        const int n = g * 8 + (r3 >> 3), kk = j * 8 + (r3 & 7);
        const int k = ks * TC_K + kk;
        const double v = (n < P && k < P) ? T[((size_t)cls * P + n) * P + k] : 0.0;
        __nv_bfloat16 b0, b1, b2;
        split3_d(v, b0, b1, b2);
        __nv_bfloat16 *o = out + (size_t)cls * per_cls + (size_t)ks * 3 * blk + rem;
        o[0] = b0;
        o[blk] = b1;
        o[2 * blk] = b2;
    }
}

// Multipoles X [rows][P] (FP32, P a multiple of 4) -> Xs [rows][Kp / 16][64]: per K step the three
// BF16 pieces of 16 coefficients each (zero-padded to Kp) and 16 unused elements; one thread per four
// coefficients.
constexpr int XS_STEP = 64;   // elements per row and K step
constexpr int XS_UNITS = 6;   // 16-byte units of it that are used: (piece, 8-coefficient half)
__global__ void k_split_x(int64_t rows, int P, int Kp, const float *__restrict__ X, __nv_bfloat16 *__restrict__ Xs) {
    const int quads = Kp / 4;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < rows * quads; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = e / quads;
        const int k = (int)(e - r * quads) * 4;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k < P) v = *reinterpret_cast<const float4 *>(X + r * P + k);
        const float x[4] = {v.x, v.y, v.z, v.w};
        alignas(8) __nv_bfloat16 b[3][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) split3_f(x[i], b[0][i], b[1][i], b[2][i]);
        __nv_bfloat16 *o = Xs + (r * (Kp / TC_K) + k / TC_K) * XS_STEP + k % TC_K;
#pragma unroll
        for (int c = 0; c < 3; ++c) *reinterpret_cast<uint2 *>(o + c * TC_K) = *reinterpret_cast<const uint2 *>(b[c]);
    }
}

// operand A of one K step and piece: rows of 128 bytes, 128-byte swizzle, K-major (8-row groups 1024 B
// apart); the tile starts on a 1024-byte boundary
__device__ __forceinline__ uint64_t make_desc_a(uint32_t tile, int piece) {
    const uint32_t a = tile + 32u * piece;
    return (uint64_t)((a & 0x3FFFFu) >> 4) | (uint64_t)1 << 16 | (uint64_t)(1024 >> 4) << 32 | (uint64_t)1 << 46 |
           (uint64_t)2 << 61;
}
// byte offset of unit `u` of row `row` within A
__device__ __forceinline__ uint32_t a_unit(int row, int u) { return (uint32_t)row * TC_AROW + (uint32_t)((u ^ (row & 7)) << 4); }

struct TcLayout {
    size_t stage_bytes, total;
};

// Row stride (floats) of the epilogue's tile in shared memory: 4 past a multiple of 16, so that the
// eight rows of a 16-byte store phase fall in different banks (a stride of 256, p = 16, put all of
// them in one: 3.77 against 3.30 ms for the diagonal product at 963000 points)
__host__ __device__ constexpr int epi_stride(int Npad) { return Npad + 4; }

// The pair-major epilogue moves at most this many columns of a tile at a time
constexpr int TC_EPI_COLS = 128;

// ST pipeline stages and three mbarriers per stage (empty, full, bfull); the epilogue reuses
// the stages for 128 columns of one tile of FP32 rows
__host__ __device__ inline TcLayout tc_layout(int ST) {
    TcLayout L;
    L.stage_bytes = TC_STAGE_BYTES;  // two stages or more hold the epilogue's rows
    L.total = ST * L.stage_bytes + 3 * ST * 8 + 16 + 1024;
    return L;
}

// tiles per block and TMEM columns per tile for a class truncated to K_c
__host__ __device__ inline int tc_tiles_for(int Kc) { return Kc <= TC_SMALL_K ? TC_MAXT : 1; }

template <int R, int TC_STAGES>
__global__ void __launch_bounds__(TC_THREADS, 2) k_m2l_tc(int P, int Npad, const __nv_bfloat16 *__restrict__ tcB,
                                                       const XChunk *__restrict__ chunks,
                                                       const int32_t *__restrict__ srcs,
                                                       const __nv_bfloat16 *__restrict__ Xs, float *__restrict__ Ypair,
                                                       const int32_t *__restrict__ cls_K, int *__restrict__ err) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // 1024-byte aligned base for the operand stages
    unsigned char *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const TcLayout Lo = tc_layout(TC_STAGES);
    static_assert(TC_STAGES * TC_STAGE_BYTES >= (size_t)TC_M * epi_stride(TC_EPI_COLS) * 4, "the epilogue's rows fit");
    uint64_t *empty = reinterpret_cast<uint64_t *>(smem + TC_STAGES * Lo.stage_bytes);
    uint64_t *full = empty + TC_STAGES;  // NPROD producer arrivals per use (the gathered A rows)
    uint64_t *bfull = full + TC_STAGES;  // one arrival + the bulk copy's bytes (the block of T_c)
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bfull + TC_STAGES);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    constexpr int NPROD = TC_THREADS - 32;  // warps 1.. fill the stages, warp 0 issues the MMAs
    __shared__ int s_src[TC_MAXT * TC_M];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // once a block has reported a wait that ran out, the rest skip their work
    if (*reinterpret_cast<volatile int *>(err) != 0) return;
    const XChunk ch = chunks[blockIdx.x];
    const int nrows = ch.count * R;
    const int ntiles = (nrows + TC_M - 1) / TC_M;
    // the class's truncated size (a multiple of 16, <= Npad): K steps and output columns; small
    // classes take two tiles per block (TMEM columns 128 apart), the others one
    const int Kc = cls_K ? cls_K[ch.cls] : Npad;
    const int nsteps = Kc / TC_K;
    const int tcap = tc_tiles_for(Kc);
    const uint32_t colstride = Kc <= TC_SMALL_K ? 128u : 256u;
    for (int r = tid; r < TC_MAXT * TC_M; r += TC_THREADS) s_src[r] = (r < nrows) ? srcs[ch.start + r / R] : -1;
    if (tid == 0) {
        for (int s = 0; s < TC_STAGES; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&full[s])), "r"(NPROD));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bfull[s])));
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "n"(TC_TMEM));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = *tmem_slot;
    const uint32_t idesc = make_idesc(TC_M, Kc);
    const int xrow = Npad / TC_K * XS_STEP;  // elements of one row of Xs
    const __nv_bfloat16 *Bc = tcB + (size_t)ch.cls * (Npad / TC_K) * 3 * Npad * TC_K;  // the class's full table
    const uint32_t sbase = smem_u32(smem);
    const uint32_t a_bytes = (uint32_t)tcap * TC_ATILE;
    const uint32_t bpiece = (uint32_t)Kc * TC_K * 2;        // one piece's K_c rows in shared memory
    const size_t bpiece_g = (size_t)Npad * TC_K * 2;        // one piece's block in the table

    // Warp-specialised pipeline. Producers (warps 1..) wait until the MMAs that last read a stage
    // are done (its empty barrier), gather their share of the next K step's A rows into it and let
    // the stage's full barrier count their arrival once those copies have landed
    // (cp.async.mbarrier.arrive.noinc); one producer thread also moves the step's block of T_c
    // (three contiguous pieces) with bulk copies counted on bfull. One thread of warp 0 waits for
    // full and bfull, makes the gathered copies visible to the tensor core (proxy fence), issues
    // the step's MMAs and commits them to empty.
    // No block-wide barrier inside the loop; every wait is bounded and a timeout raises the shared
    // abort flag, which stops the other side at its next wait.
    __shared__ int s_last_ks;
    if (warp == 0) {
        if (lane == 0) {
            int ks = 0;
            for (; ks < nsteps; ++ks) {
                const int st = ks % TC_STAGES;
                const uint32_t ph = (uint32_t)((ks / TC_STAGES) & 1);
                if (!mbar_wait(smem_u32(&full[st]), ph) || !mbar_wait(smem_u32(&bfull[st]), ph) || *abort_flag) {
                    *abort_flag = 1;
                    break;
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("tcgen05.fence::after_thread_sync;");
                const uint32_t sa = sbase + st * (uint32_t)Lo.stage_bytes;
                const uint32_t sb = sa + a_bytes;
                for (int t = 0; t < ntiles; ++t) {
                    const uint32_t d = tmem + (uint32_t)t * colstride;
                    const uint32_t at = sa + t * TC_ATILE;
                    // smallest terms first: (2,0) (1,1) (0,2) (1,0) (0,1) (0,0)
                    mma_bf16(d, make_desc_a(at, 2), make_desc(sb), idesc, ks > 0 ? 1u : 0u);
                    mma_bf16(d, make_desc_a(at, 1), make_desc(sb + bpiece), idesc, 1u);
                    mma_bf16(d, make_desc_a(at, 0), make_desc(sb + 2 * bpiece), idesc, 1u);
                    mma_bf16(d, make_desc_a(at, 1), make_desc(sb), idesc, 1u);
                    mma_bf16(d, make_desc_a(at, 0), make_desc(sb + bpiece), idesc, 1u);
                    mma_bf16(d, make_desc_a(at, 0), make_desc(sb), idesc, 1u);
                }
                mma_commit(smem_u32(&empty[st]));
            }
            s_last_ks = ks - 1;  // last committed step (-1: none)
        }
        __syncwarp();
    } else {
        const int pt = tid - 32;
        // this thread's A copies, fixed for the block: unit pt % 6 = (piece, 8-element half) of the rows
        // pt / 6 + PROWS i of every K step (six neighbouring lanes read one row's line)
        constexpr int PROWS = NPROD / XS_UNITS, AU = (TC_MAXT * TC_M + PROWS - 1) / PROWS;
        const int arows = ntiles * TC_M;
        const int unit = pt % XS_UNITS, row0 = pt < PROWS * XS_UNITS ? pt / XS_UNITS : arows;  // the rest copies nothing
        int a_row[AU];  // row of Xs, -1: a zero row
#pragma unroll
        for (int i = 0; i < AU; ++i) {
            const int row2 = row0 + i * PROWS;
            const int s = row2 < arows ? s_src[row2] : -1;
            a_row[i] = s >= 0 ? s * R + row2 % R : -1;
        }
        const bool bulk = pt == 0;
        int issued = -1;  // last K step whose block of T_c this thread requested
        for (int ks = 0; ks < nsteps; ++ks) {
            const int st = ks % TC_STAGES;
            // the stage's previous use (step ks - ST) must be consumed: completion ks / ST - 1
            if (ks >= TC_STAGES &&
                (!mbar_wait(smem_u32(&empty[st]), (uint32_t)((ks / TC_STAGES - 1) & 1)) || *abort_flag)) {
                *abort_flag = 1;
                break;
            }
            const uint32_t sa = sbase + st * (uint32_t)Lo.stage_bytes;
            if (bulk) {
                // B: the first K_c rows of each piece's pre-tiled block (8-row core-matrix groups are
                // contiguous, so that is a prefix of the block)
                const uint32_t bb = smem_u32(&bfull[st]);
                mbar_expect_tx(bb, 3u * bpiece);
                const unsigned char *bsrc = reinterpret_cast<const unsigned char *>(Bc + (size_t)ks * 3 * Npad * TC_K);
                for (int piece = 0; piece < 3; ++piece)
                    bulk_g2s(sa + a_bytes + piece * bpiece, bsrc + (size_t)piece * bpiece_g, bpiece, bb);
                issued = ks;
            }
            const __nv_bfloat16 *xk = Xs + unit * 8 + ks * XS_STEP;
#pragma unroll
            for (int i = 0; i < AU; ++i)
                if (row0 + i * PROWS < arows)
                    cp_async16(sa + a_unit(row0 + i * PROWS, unit), xk + (int64_t)max(a_row[i], 0) * xrow,
                               a_row[i] >= 0 ? 16u : 0u);
            asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&full[st])) : "memory");
        }
        cp_async_wait<0>();  // nothing of this thread in flight past this point
        // the bulk copies of the last steps (those an abort left unconsumed included) land before
        // the block moves on: each stage's latest bfull phase completes when its copy has landed
        for (int ks = issued; ks >= 0 && ks > issued - TC_STAGES; --ks)
            if (!mbar_wait(smem_u32(&bfull[ks % TC_STAGES]), (uint32_t)((ks / TC_STAGES) & 1))) *abort_flag = 1;
    }
    __syncthreads();
    // tcgen05.commit tracks every earlier MMA of the issuing thread: the last commit covers all
    const int lk = s_last_ks;
    const bool done = lk >= 0 && mbar_wait(smem_u32(&empty[lk % TC_STAGES]), (uint32_t)((lk / TC_STAGES) & 1));
    bool ok = !*abort_flag && lk == nsteps - 1 && done;
    if (!ok && tid == 0) atomicOr(err, 1);
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (ok) {
        // epilogue, at most 128 columns of a tile at a time: warp w holds TMEM lanes 32 (w % 4) ..;
        // each thread moves its part of a row into shared memory, then each warp writes whole rows
        // of Ypair with coalesced 16-byte stores (the first Kc coefficients; the per-target sums
        // read no more)
        constexpr int es = epi_stride(TC_EPI_COLS);
        const int kw = min(Kc, P);
        float *stage = reinterpret_cast<float *>(smem);  // the operand stages are free now
        for (int u = 0; u < ntiles * ((Kc + TC_EPI_COLS - 1) / TC_EPI_COLS); ++u) {
            const int t = u % ntiles, cb = u / ntiles * TC_EPI_COLS;
            const int rows_t = min(TC_M, nrows - t * TC_M);
            // a warp reads its own quarter of the TMEM lanes (warp % 4); the two warp groups take
            // the lower and the upper half of the 16-column groups
            const int q4 = warp & 3, half = warp >> 2;
            const int ngroups = min(Kc - cb, TC_EPI_COLS) / 16, mid = (ngroups + 1) / 2;
            float *srow = stage + (size_t)(q4 * 32 + lane) * es;
            for (int g = half ? mid : 0; g < (half ? ngroups : mid); ++g) {
                const int c0 = g * 16;
                uint32_t v[16];
                const uint32_t taddr =
                    tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)t * colstride + (uint32_t)(cb + c0);
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
                    "[%16];"
                    : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                      "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
                      "=r"(v[15])
                    : "r"(taddr));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int i = 0; i < 16; i += 4)
                    *reinterpret_cast<float4 *>(srow + c0 + i) =
                        make_float4(__uint_as_float(v[i]), __uint_as_float(v[i + 1]), __uint_as_float(v[i + 2]),
                                    __uint_as_float(v[i + 3]));
            }
            __syncthreads();
            const int n4 = (min(kw, cb + TC_EPI_COLS) - cb) / 4;  // P % 4 == 0: whole 16-byte groups, at most 32
            float4 *dst = reinterpret_cast<float4 *>(Ypair + ((size_t)ch.start * R + t * TC_M) * P + cb);
            if (lane < n4)
                for (int row = warp; row < rows_t; row += TC_THREADS / 32)
                    dst[(size_t)row * (P / 4) + lane] = reinterpret_cast<const float4 *>(stage + (size_t)row * es)[lane];
            __syncthreads();
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(TC_TMEM));
}

}  // namespace

bool m2l_tc_supported(int P) { return P % 4 == 0 && P <= 256; }

int m2l_tc_pairs_per_chunk(int R, int Kc) { return tc_tiles_for(Kc) * TC_M / R; }

void build_tc_tables(Context &c, Operators &o) {
    const int P = o.P;
    if (!m2l_tc_supported(P)) return;
    o.tc_Npad = (P + 15) / 16 * 16;
    o.tc_Kpad = o.tc_Npad;
    const size_t per = (size_t)3 * o.tc_Npad * o.tc_Kpad;
    o.m2l_tc.resize(kNumM2LClasses * per);
    dim3 grid(64, kNumM2LClasses);
    k_build_tc_table<<<grid, 256, 0, c.stream>>>(P, o.tc_Npad, o.m2l64.p,
                                                 reinterpret_cast<__nv_bfloat16 *>(o.m2l_tc.p));
    BEM_LAUNCH_CHECK();
}

// the multipoles, split once for all translations of a product
static __nv_bfloat16 *split_multipoles(Context &c, const Operators &o, const float *X, int64_t xrows, cudaStream_t st) {
    const int Npad = o.tc_Npad;
    c.xsplit.resize((size_t)xrows * (Npad / TC_K) * XS_STEP);
    __nv_bfloat16 *xs = reinterpret_cast<__nv_bfloat16 *>(c.xsplit.p);
    const int nb = (int)std::min<int64_t>(div_up(xrows * (Npad / 4), 256), 152 * 16);
    k_split_x<<<nb, 256, 0, st>>>(xrows, o.P, Npad, X, xs);
    BEM_LAUNCH_CHECK();
    return xs;
}

template <int R>
void launch_m2l_tc(Context &c, const Operators &o, const XChunk *chunks, int64_t nchunks, const float *X,
                   int64_t xrows, float *Ypair, int *err, cudaStream_t st) {
    const int Npad = o.tc_Npad;
    __nv_bfloat16 *xs = split_multipoles(c, o, X, xrows, st);
    // pipeline depth: the context's choice (parameter or autotuner), else two stages, with which two
    // blocks fit on an SM and one's set-up and epilogue run under the other's MMAs (one block of three
    // stages and twice the tiles: diagonal product of 963000 points 2.91 against 2.49 ms, product of
    // 192600 points 106 against 81 us)
    const int stages = c.tuned_stages == 3 ? 3 : 2;
    const size_t sm = tc_layout(stages).total;
    auto kern = stages == 2 ? k_m2l_tc<R, 2> : k_m2l_tc<R, 3>;
    // set on every launch: the attribute belongs to the current device (~1 us against a ms kernel)
    BEM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    kern<<<(unsigned)nchunks, TC_THREADS, sm, st>>>(o.P, Npad, reinterpret_cast<const __nv_bfloat16 *>(o.m2l_tc.p),
                                                   chunks, c.tree.m2l_src.p, xs, Ypair,
                                                   o.margin >= 0 ? o.cls_K.p : nullptr, err);
    BEM_LAUNCH_CHECK();
}

template void launch_m2l_tc<1>(Context &, const Operators &, const XChunk *, int64_t, const float *, int64_t, float *,
                               int *, cudaStream_t);
template void launch_m2l_tc<4>(Context &, const Operators &, const XChunk *, int64_t, const float *, int64_t, float *,
                               int *, cudaStream_t);

// ------------------------------------------------------------------------------ target-major form
//
// Instead of one output row per translation (summed per target afterwards), a block
// accumulates, for a tile of 256 rows = 256 / R target boxes x R right-hand sides (two M = 128
// tensor-memory accumulators), the translations of a few offset classes: for class c a row's A is
// the multipole of its target's class-c source for its right-hand side (zero rows where a target
// has none), B = T_c, and the MMAs of all the item's classes accumulate into the same columns
// (N = K_c per class), zeroed first. The pipeline is the pair-major kernel's (gathered A rows by
// cp.async, T_c blocks by bulk copies, one MMA thread, bounded waits), but it runs across the
// item's classes without a break. The FP32 accumulation runs from small terms to large: classes
// by truncated size ascending (the far classes, whose translations are the smallest), and within
// a class the K steps from the highest degrees down. A target's items are summed by k_tm_reduce
// in a fixed order with TwoSum compensation, so the FP32 accumulation in tensor memory spans at
// most an item. Target boxes are grouped by octant (their
// position in the parent), since the 189 classes a box can have depend on it: a tile's classes
// are then about two thirds full. The products use it with one RHS; with four (the diagonal
// product, 64 targets per tile) it was slower than the pair-major kernel.
namespace {

constexpr int TM_ROWS = 2 * TC_M;  // rows per tile: (target, rhs)
// Classes per item at most (an item's cost limits them before): up to 32 small classes add up in an item's FP32
// accumulators, where items of 8 classes of any size did; the largest classes come one or two to an item.
// Products of dense trees against FP64 at p = 14: 0.7e-6 to 1.1e-6, with 8 classes an item 1.2e-6 to 1.7e-6.
constexpr int TM_MAXCLS = 32;
constexpr size_t TM_STAGE_BYTES = 2 * TC_ATILE + 3 * 256 * 16 * 2;  // A (two tiles) + B (K_c <= 256)

// target boxes: the boxes of levels 2.. with at least one M2L translation, key = octant
__global__ void k_tm_flags(int64_t first, int64_t n, const int32_t *__restrict__ tgt_off, int32_t *__restrict__ flag) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) flag[i] = tgt_off[first + i + 1] > tgt_off[first + i] ? 1 : 0;
}
__global__ void k_tm_emit(int64_t first, int64_t n, const int32_t *__restrict__ flag, const int32_t *__restrict__ ex,
                          const uint32_t *__restrict__ bkey, uint32_t *__restrict__ key, int32_t *__restrict__ box) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n && flag[i]) {
        key[ex[i]] = bkey[first + i] & 7u;
        box[ex[i]] = (int32_t)(first + i);
    }
}
__global__ void k_tm_slots(int64_t ntgt, int64_t nslots, const int32_t *__restrict__ sorted,
                           int32_t *__restrict__ tm_box, int32_t *__restrict__ pos) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= nslots) return;
    const int32_t b = i < ntgt ? sorted[i] : -1;
    tm_box[i] = b;
    if (b >= 0) pos[b] = (int32_t)i;
}
// every translation (s -> t, class c) fills its (tile, class, slot) entry; TT targets per tile
__global__ void k_tm_fill(int64_t np, int TT, const int32_t *__restrict__ src, const int32_t *__restrict__ tgt,
                          const uint32_t *__restrict__ cls, const int32_t *__restrict__ pos, int32_t *__restrict__ tab) {
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= np) return;
    const int32_t r = pos[tgt[k]];
    const int64_t tile = r / TT, slot = r % TT;
    tab[(tile * kNumM2LClasses + cls[k]) * TT + slot] = src[k];
}
// Time of one class in an item, in arbitrary units: K_c / 16 K steps, whose shared-memory traffic (the
// MMAs' operand reads and the staged copies: about 576 + 3.75 K_c clocks) bounds a step.
__device__ __forceinline__ int tm_cost(int Kc) { return Kc / TC_K * (Kc + 160); }
// inclusive prefix sum over a block of 512 threads
__device__ __forceinline__ int tm_scan(int v, int *warp_tot) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    __syncthreads();
    if (lane == 31) warp_tot[w] = v;
    __syncthreads();
    for (int i = 0; i < w; ++i) v += warp_tot[i];
    return v;
}
// which classes a tile has: a warp per (tile, class) looks through the class's slots
__global__ void __launch_bounds__(256) k_tm_has(int64_t n, int TT, const int32_t *__restrict__ tab, uint8_t *__restrict__ has) {
    const int64_t e = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (e >= n) return;
    const int lane = threadIdx.x & 31;
    bool f = false;
    for (int r = lane; r < TT; r += 32) f = f || tab[e * TT + r] >= 0;
    const unsigned any = __ballot_sync(0xffffffffu, f);
    if (lane == 0) has[e] = any != 0;
}
// per tile, the classes present, in the order `order` (truncated size ascending), and their cost
__global__ void __launch_bounds__(512) k_tm_classes(const uint8_t *__restrict__ has, const int32_t *__restrict__ order,
                                                    const int32_t *__restrict__ cls_K, int Npad,
                                                    int32_t *__restrict__ tcls, int32_t *__restrict__ ncls,
                                                    int32_t *__restrict__ cost) {
    __shared__ int warp_tot[16];
    const int tile = blockIdx.x, k = threadIdx.x;
    const int f = k < kNumM2LClasses && has[(int64_t)tile * kNumM2LClasses + order[k]];
    const int idx = tm_scan(f, warp_tot);  // inclusive
    if (f) tcls[(int64_t)tile * kNumM2LClasses + idx - 1] = order[k];
    const int c = tm_scan(f ? tm_cost(cls_K ? cls_K[order[k]] : Npad) : 0, warp_tot);
    if (k == 511) {
        ncls[tile] = idx;
        cost[tile] = c;
    }
}
// The tile's classes cut into items of about equal cost, n = cost / target of them (rounded up): a class
// belongs to the item that the middle of its cost falls into, and an item has at most TM_MAXCLS classes.
// Pass 0 counts the items, pass 1 writes them from off[tile] on. One block per tile.
__global__ void __launch_bounds__(512) k_tm_items(int target, const int32_t *__restrict__ ncls,
                                                  const int32_t *__restrict__ tcls, const int32_t *__restrict__ cls_K,
                                                  int Npad, const int32_t *__restrict__ cost, int pass,
                                                  int32_t *__restrict__ cnt, const int32_t *__restrict__ off,
                                                  int4 *__restrict__ items) {
    __shared__ int warp_tot[16];
    __shared__ int part[513], first[513];
    const int tile = blockIdx.x, i = threadIdx.x, n = ncls[tile];
    const int64_t total = cost[tile], parts = max((int64_t)1, (total + target - 1) / target);
    const int Kc = i < n ? (cls_K ? cls_K[tcls[(int64_t)tile * kNumM2LClasses + i]] : Npad) : 0;
    const int mine = i < n ? tm_cost(Kc) : 0;
    const int64_t mid = tm_scan(mine, warp_tot) - (mine + 1) / 2;
    part[i] = i < n ? (int)(mid * parts / total) : -1;
    __syncthreads();
    // the first class of i's part, then a cut every TM_MAXCLS classes from there
    int lo = i;
    if (i < n)
        while (lo > 0 && part[lo - 1] == part[i]) --lo;
    const int f = i < n && (i - lo) % TM_MAXCLS == 0;
    first[i] = f || i >= n;
    const int idx = tm_scan(f, warp_tot) - 1;  // (its barriers also publish `first`)
    if (pass && i < n) {
        const bool last = i + 1 == n || first[i + 1];
        if (last) {
            int c0 = i;
            while (!first[c0]) --c0;
            items[off[tile] + idx] = make_int4(tile, c0, i + 1 - c0, Kc);  // K_c: the largest of the item
        }
    }
    if (!pass && i == 511) cnt[tile] = idx + 1;
}

__device__ __forceinline__ void two_sum_add(float &s, float &c, float v) {
    const float t = s + v, bp = t - s;
    c += (s - (t - bp)) + (v - bp);
    s = t;
}

// lc[box][rhs][col] = sum over the tile's items of the partial row (fixed order, compensated)
// (the loads of four items are issued before their sums, which stay in item order; a row's
// coefficients past an item's size read as zero and leave the TwoSum unchanged)
constexpr int TM_MAXITEMS = kNumM2LClasses;  // items of one tile at most
template <int R>
__global__ void k_tm_reduce(int P, int Npad, const int32_t *__restrict__ tm_box, const int32_t *__restrict__ item_off,
                            const int4 *__restrict__ items, const float *__restrict__ part, float *__restrict__ lc) {
    constexpr int TT = TM_ROWS / R;
    __shared__ int s_kmax[TM_MAXITEMS];
    const int64_t tile = blockIdx.x;
    const int row = blockIdx.y;
    const int32_t box = tm_box[tile * TT + row / R];
    if (box < 0) return;  // uniform in the block
    const int i0 = item_off[tile], i1 = item_off[tile + 1], ni = i1 - i0;
    for (int i = threadIdx.x; i < ni; i += blockDim.x) s_kmax[i] = items[i0 + i].w;
    __syncthreads();
    float *dst = lc + ((int64_t)box * R + row % R) * P;
    const float *src = part + ((int64_t)i0 * TM_ROWS + row) * Npad;
    const int64_t istride = (int64_t)TM_ROWS * Npad;
    for (int col = threadIdx.x; col < P; col += blockDim.x) {
        float s = 0.f, c = 0.f;
        int i = 0;
        for (; i + 4 <= ni; i += 4) {
            float v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = col < s_kmax[i + u] ? src[(i + u) * istride + col] : 0.f;
#pragma unroll
            for (int u = 0; u < 4; ++u) two_sum_add(s, c, v[u]);
        }
        for (; i < ni; ++i)
            if (col < s_kmax[i]) two_sum_add(s, c, src[i * istride + col]);
        dst[col] = s + c;
    }
}

template <int R, int TC_STAGES>
__global__ void __launch_bounds__(TC_THREADS, 1) k_m2l_tm(int P, int Npad, const __nv_bfloat16 *__restrict__ tcB,
                                                       const int4 *__restrict__ items, const int32_t *__restrict__ tab,
                                                       const int32_t *__restrict__ tcls,
                                                       const __nv_bfloat16 *__restrict__ Xs, float *__restrict__ part,
                                                       const int32_t *__restrict__ cls_K, int *__restrict__ err) {
    constexpr int TT = TM_ROWS / R;  // target slots per tile
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const size_t stage_bytes = TM_STAGE_BYTES;
    const size_t epi_bytes = (size_t)TC_M * epi_stride(Npad) * 4;
    uint64_t *empty = reinterpret_cast<uint64_t *>(
        smem + (TC_STAGES * stage_bytes > epi_bytes ? TC_STAGES * stage_bytes : epi_bytes));
    uint64_t *full = empty + TC_STAGES;
    uint64_t *bfull = full + TC_STAGES;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bfull + TC_STAGES);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    constexpr int NPROD = TC_THREADS - 32;
    __shared__ int s_cls[TM_MAXCLS], s_K[TM_MAXCLS];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (*reinterpret_cast<volatile int *>(err) != 0) return;
    const int4 it = items[blockIdx.x];
    const int64_t tile = it.x;
    const int nc = it.z, kmax = it.w;
    if (tid < nc) {
        const int cl = tcls[tile * kNumM2LClasses + it.y + tid];
        s_cls[tid] = cl;
        s_K[tid] = cls_K ? cls_K[cl] : Npad;
    }
    if (tid == 0) {
        for (int s = 0; s < TC_STAGES; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&full[s])), "r"(NPROD));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bfull[s])));
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "n"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = *tmem_slot;
    {
        // zero the accumulators' first kmax columns: warp w writes its lane quarter (w % 4) of
        // tile w / 4; every MMA then accumulates
        const uint32_t zr = 0u;
        const uint32_t tb = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(warp >> 2) * 256u;
        for (int c0 = 0; c0 < kmax; c0 += 16)
            asm volatile(
                "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(
                    tb + (uint32_t)c0),
                "r"(zr)
                : "memory");
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;");
    }
    int nsteps = 0;
    for (int j = 0; j < nc; ++j) nsteps += s_K[j] / TC_K;
    const int xrow = Npad / TC_K * XS_STEP;  // elements of one row of Xs
    const uint32_t sbase = smem_u32(smem);
    const uint32_t a_bytes = 2 * TC_ATILE;
    const size_t bpiece_g = (size_t)Npad * TC_K * 2;
    const size_t cls_stride = (size_t)(Npad / TC_K) * 3 * Npad * TC_K;  // elements of one class's table

    __shared__ int s_last_ks;
    if (warp == 0) {
        if (lane == 0) {
            int ks = 0;
            bool stop = false;
            for (int j = 0; j < nc && !stop; ++j) {
                const int Kj = s_K[j];
                const uint32_t idesc = make_idesc(TC_M, Kj);
                const uint32_t bpiece = (uint32_t)Kj * TC_K * 2;
                for (int s = 0; s < Kj / TC_K; ++s, ++ks) {  // K steps from the highest degrees down
                    const int st = ks % TC_STAGES;
                    const uint32_t ph = (uint32_t)((ks / TC_STAGES) & 1);
                    if (!mbar_wait(smem_u32(&full[st]), ph) || !mbar_wait(smem_u32(&bfull[st]), ph) || *abort_flag) {
                        *abort_flag = 1;
                        stop = true;
                        break;
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    const uint32_t sa = sbase + st * (uint32_t)stage_bytes;
                    const uint32_t sb = sa + a_bytes;
                    for (int t = 0; t < 2; ++t) {
                        const uint32_t d = tmem + (uint32_t)t * 256u;
                        const uint32_t at = sa + t * TC_ATILE;
                        mma_bf16(d, make_desc_a(at, 2), make_desc(sb), idesc, 1u);
                        mma_bf16(d, make_desc_a(at, 1), make_desc(sb + bpiece), idesc, 1u);
                        mma_bf16(d, make_desc_a(at, 0), make_desc(sb + 2 * bpiece), idesc, 1u);
                        mma_bf16(d, make_desc_a(at, 1), make_desc(sb), idesc, 1u);
                        mma_bf16(d, make_desc_a(at, 0), make_desc(sb + bpiece), idesc, 1u);
                        mma_bf16(d, make_desc_a(at, 0), make_desc(sb), idesc, 1u);
                    }
                    mma_commit(smem_u32(&empty[st]));
                }
            }
            s_last_ks = ks - 1;
        }
        __syncwarp();
    } else {
        const int pt = tid - 32;
        // unit pt % 6 = (piece, 8-element half) of the rows pt / 6 + PROWS i, as in k_m2l_tc
        constexpr int PROWS = NPROD / XS_UNITS, AU = (TM_ROWS + PROWS - 1) / PROWS;
        const int unit = pt % XS_UNITS, row0 = pt < PROWS * XS_UNITS ? pt / XS_UNITS : TM_ROWS;
        // rows of Xs of the next class, read while the current one is moved; -1: a target without the
        // class, a zero row
        int nxt[AU];
        auto rows_of = [&](int j) {
#pragma unroll
            for (int i = 0; i < AU; ++i) {
                const int row2 = row0 + i * PROWS;  // (target slot, rhs) = (row2 / R, row2 % R)
                nxt[i] = row2 < TM_ROWS && j < nc ? tab[(tile * kNumM2LClasses + s_cls[j]) * TT + row2 / R] : -1;
            }
        };
        rows_of(0);
        const bool bulk = pt == 0;
        int issued = -1, ks = 0;
        bool stop = false;
        for (int j = 0; j < nc && !stop; ++j) {
            const int Kj = s_K[j];
            const uint32_t bpiece = (uint32_t)Kj * TC_K * 2;
            const __nv_bfloat16 *Bc = tcB + (size_t)s_cls[j] * cls_stride;
            int a_row[AU];
#pragma unroll
            for (int i = 0; i < AU; ++i) a_row[i] = nxt[i] >= 0 ? nxt[i] * R + (row0 + i * PROWS) % R : -1;
            rows_of(j + 1);
            for (int s = 0; s < Kj / TC_K; ++s, ++ks) {
                const int st = ks % TC_STAGES;
                if (ks >= TC_STAGES &&
                    (!mbar_wait(smem_u32(&empty[st]), (uint32_t)((ks / TC_STAGES - 1) & 1)) || *abort_flag)) {
                    *abort_flag = 1;
                    stop = true;
                    break;
                }
                const uint32_t sa = sbase + st * (uint32_t)stage_bytes;
                const int kstep = Kj / TC_K - 1 - s;  // highest degrees first
                if (bulk) {
                    const uint32_t bb = smem_u32(&bfull[st]);
                    mbar_expect_tx(bb, 3u * bpiece);
                    const unsigned char *bsrc =
                        reinterpret_cast<const unsigned char *>(Bc + (size_t)kstep * 3 * Npad * TC_K);
                    for (int piece = 0; piece < 3; ++piece)
                        bulk_g2s(sa + a_bytes + piece * bpiece, bsrc + (size_t)piece * bpiece_g, bpiece, bb);
                    issued = ks;
                }
                const __nv_bfloat16 *xk = Xs + unit * 8 + kstep * XS_STEP;
#pragma unroll
                for (int i = 0; i < AU; ++i)
                    if (row0 + i * PROWS < TM_ROWS)
                        cp_async16(sa + a_unit(row0 + i * PROWS, unit), xk + (int64_t)max(a_row[i], 0) * xrow,
                                   a_row[i] >= 0 ? 16u : 0u);
                asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&full[st])) : "memory");
            }
        }
        cp_async_wait<0>();
        for (int k2 = issued; k2 >= 0 && k2 > issued - TC_STAGES; --k2)
            if (!mbar_wait(smem_u32(&bfull[k2 % TC_STAGES]), (uint32_t)((k2 / TC_STAGES) & 1))) *abort_flag = 1;
    }
    __syncthreads();
    const int lk = s_last_ks;
    const bool done = lk >= 0 && mbar_wait(smem_u32(&empty[lk % TC_STAGES]), (uint32_t)((lk / TC_STAGES) & 1));
    bool ok = !*abort_flag && lk == nsteps - 1 && done;
    if (!ok && tid == 0) atomicOr(err, 1);
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (ok) {
        // epilogue, one tile at a time, as in k_m2l_tc: TMEM -> shared memory -> coalesced rows of
        // the item's partial (the first kmax coefficients; the rest of the row is never read)
        float *stage = reinterpret_cast<float *>(smem);
        float *dst_item = part + (size_t)blockIdx.x * TM_ROWS * Npad;
        const int es = epi_stride(Npad), kw = kmax / 4, n4 = Npad / 4;
        for (int t = 0; t < 2; ++t) {
            const int q4 = warp & 3, half = warp >> 2;
            const int ngroups = kmax / 16, g0 = half ? (ngroups + 1) / 2 : 0, g1 = half ? ngroups : (ngroups + 1) / 2;
            float *srow = stage + (size_t)(q4 * 32 + lane) * es;
            for (int c0 = g0 * 16; c0 < g1 * 16; c0 += 16) {
                uint32_t v[16];
                const uint32_t taddr = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)t * 256u + (uint32_t)c0;
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
                    "[%16];"
                    : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                      "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
                      "=r"(v[15])
                    : "r"(taddr));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int i = 0; i < 16; i += 4)
                    *reinterpret_cast<float4 *>(srow + c0 + i) =
                        make_float4(__uint_as_float(v[i]), __uint_as_float(v[i + 1]), __uint_as_float(v[i + 2]),
                                    __uint_as_float(v[i + 3]));
            }
            __syncthreads();
            float4 *dst = reinterpret_cast<float4 *>(dst_item + (size_t)t * TC_M * Npad);
            for (int row = warp; row < TC_M; row += TC_THREADS / 32) {
                const float4 *src = reinterpret_cast<const float4 *>(stage + (size_t)row * es);
                for (int col = lane; col < kw; col += 32) dst[(size_t)row * n4 + col] = src[col];
            }
            __syncthreads();
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(512));
}

}  // namespace

// Items: whole rounds of the SMs (one block per SM), of equal cost. The rounds are those that 8
// average classes per item would take, rounded up: cutting every tile into items of 8 classes gave
// 307 items at 192600 points, three rounds for the work of two (M2L 191 us, 144 us since), and 80 items for 152
// SMs at 40962 (97 us, 45 us since).
template <int R>
static void build_tm_tables(Context &c, const Operators &o, cudaStream_t st) {
    Context::TmState &S = c.tm[R == 1 ? 0 : 1];
    constexpr int TT = TM_ROWS / R;
    Tree &t = c.tree;
    const int tb = 256;
    const int64_t first = t.base[2], n = (int64_t)t.nbox - first;
    if (n <= 0 || t.n_m2l == 0) {  // no translations: nothing to launch
        S.ntiles = S.nitems = 0;
        S.ok = true;
        S.ops = &o;
        return;
    }
    DevBuf<int32_t> &flag = S.s_i32[0], &ex = S.s_i32[1], &tot = S.s_i32[2];
    flag.resize(std::max<int64_t>(n, 1));
    ex.resize(std::max<int64_t>(n, 1));
    tot.resize(1);
    k_tm_flags<<<div_up(n, tb), tb, 0, st>>>(first, n, t.m2l_tgt_off.p, flag.p);
    BEM_LAUNCH_CHECK();
    exclusive_scan_i32(flag.p, ex.p, n, tot.p, st);
    int32_t ntgt = 0;
    BEM_CUDA(cudaMemcpyAsync(&ntgt, tot.p, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    BEM_CUDA(cudaStreamSynchronize(st));
    DevBuf<uint32_t> &key = S.s_u32[0], &ktmp = S.s_u32[1];
    DevBuf<int32_t> &box = S.s_i32[3], &btmp = S.s_i32[4], &pos = S.s_i32[5];
    key.resize(std::max(ntgt, 1));
    ktmp.resize(std::max(ntgt, 1));
    box.resize(std::max(ntgt, 1));
    btmp.resize(std::max(ntgt, 1));
    pos.resize(t.nbox);
    k_tm_emit<<<div_up(n, tb), tb, 0, st>>>(first, n, flag.p, ex.p, t.bkey.p, key.p, box.p);
    BEM_LAUNCH_CHECK();
    if (ntgt > 0) radix_sort_u32(key.p, box.p, ntgt, 3, ktmp.p, btmp.p, st);  // stable: box order within an octant
    const int64_t ntiles = div_up((int64_t)ntgt, TT);
    S.ntiles = ntiles;
    S.box.resize(std::max<int64_t>(ntiles * TT, 1));
    k_tm_slots<<<div_up(ntiles * TT, tb), tb, 0, st>>>(ntgt, ntiles * TT, box.p, S.box.p, pos.p);
    BEM_LAUNCH_CHECK();
    const size_t ntab = (size_t)ntiles * kNumM2LClasses * TT;
    S.src.resize(std::max<size_t>(ntab, 1));
    BEM_CUDA(cudaMemsetAsync(S.src.p, 0xff, std::max<size_t>(ntab, 1) * sizeof(int32_t), st));
    k_tm_fill<<<div_up(t.n_m2l, tb), tb, 0, st>>>(t.n_m2l, TT, t.m2l_src.p, t.m2l_tgt.p, t.m2l_cls.p, pos.p, S.src.p);
    BEM_LAUNCH_CHECK();
    // class order: truncated size ascending, ties by class index
    const int P16 = o.tc_Npad;
    std::vector<int32_t> order(kNumM2LClasses);
    for (int k = 0; k < kNumM2LClasses; ++k) order[k] = k;
    auto Kof = [&](int k) { return o.margin >= 0 ? o.cls_Kh[k] : P16; };
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return Kof(a) < Kof(b); });
    DevBuf<int32_t> &ncls = S.s_i32[6], &icnt = S.s_i32[7];
    DevBuf<int32_t> dorder;
    dorder.resize(kNumM2LClasses);
    ncls.resize(std::max<int64_t>(ntiles, 1));
    icnt.resize(ntiles + 1);
    BEM_CUDA(cudaMemcpyAsync(dorder.p, order.data(), kNumM2LClasses * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    S.cls.resize(std::max<int64_t>(ntiles * kNumM2LClasses, 1));
    S.item_off.resize(ntiles + 1);
    const int32_t *clsK = o.margin >= 0 ? o.cls_K.p : nullptr;
    DevBuf<int32_t> &cost = S.s_i32[8];
    cost.resize(ntiles);
    const int64_t nhas = ntiles * kNumM2LClasses;
    S.has.resize(std::max<int64_t>(nhas, 1));
    k_tm_has<<<div_up(nhas, 8), 256, 0, st>>>(nhas, TT, S.src.p, S.has.p);
    BEM_LAUNCH_CHECK();
    k_tm_classes<<<(unsigned)ntiles, 512, 0, st>>>(S.has.p, dorder.p, clsK, P16, S.cls.p, ncls.p, cost.p);
    BEM_LAUNCH_CHECK();
    std::vector<int32_t> hcost(ntiles);
    BEM_CUDA(cudaMemcpyAsync(hcost.data(), cost.p, ntiles * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    BEM_CUDA(cudaStreamSynchronize(st));
    int64_t total = 0, mean8 = 0;  // mean8: 8 average classes
    for (int32_t v : hcost) total += v;
    for (int k = 0; k < kNumM2LClasses; ++k) mean8 += 8 * (int64_t)(Kof(k) / TC_K * (Kof(k) + 160));
    mean8 /= kNumM2LClasses;
    const int64_t rounds = std::max<int64_t>(1, div_up(total, c.num_sms * mean8));
    // the smallest target that gives at most rounds x SMs items (a tile's last item is its own)
    auto count = [&](int64_t target) {
        int64_t n = 0;
        for (int32_t v : hcost) n += std::max<int64_t>(1, (v + target - 1) / target);
        return n;
    };
    int64_t lo = 1, hi = std::max<int64_t>(1, total);
    while (lo < hi) {
        const int64_t mid = (lo + hi) / 2;
        if (count(mid) <= rounds * c.num_sms) hi = mid;
        else lo = mid + 1;
    }
    const int target = (int)lo;
    k_tm_items<<<(unsigned)ntiles, 512, 0, st>>>(target, ncls.p, S.cls.p, clsK, P16, cost.p, 0, icnt.p, nullptr, nullptr);
    BEM_LAUNCH_CHECK();
    exclusive_scan_i32(icnt.p, S.item_off.p, ntiles, tot.p, st);
    BEM_CUDA(cudaMemcpyAsync(S.item_off.p + ntiles, tot.p, sizeof(int32_t), cudaMemcpyDeviceToDevice, st));
    int32_t nitems = 0;
    BEM_CUDA(cudaMemcpyAsync(&nitems, tot.p, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    BEM_CUDA(cudaStreamSynchronize(st));
    S.nitems = nitems;
    S.items.resize(std::max(nitems, 1));
    k_tm_items<<<(unsigned)ntiles, 512, 0, st>>>(target, ncls.p, S.cls.p, clsK, P16, cost.p, 1, nullptr, S.item_off.p,
                                                 S.items.p);
    BEM_LAUNCH_CHECK();
    S.part.resize(std::max<size_t>((size_t)nitems * TM_ROWS * P16, 1));
    BEM_CUDA(cudaStreamSynchronize(st));  // dorder is freed on return
    S.ok = true;
    S.ops = &o;
}

template <int R>
void launch_m2l_tm(Context &c, const Operators &o, const float *X, int64_t xrows, int *err, cudaStream_t st) {
    Context::TmState &S = c.tm[R == 1 ? 0 : 1];
    if (!S.ok || S.ops != &o) build_tm_tables<R>(c, o, st);
    const int Npad = o.tc_Npad;
    __nv_bfloat16 *xs = split_multipoles(c, o, X, xrows, st);
    if (S.nitems == 0) return;
    const int stages = 3;
    const size_t epi = (size_t)TC_M * epi_stride(Npad) * 4;
    const size_t sm = (stages * TM_STAGE_BYTES > epi ? stages * TM_STAGE_BYTES : epi) + 3 * stages * 8 + 16 + 1024;
    BEM_CUDA(cudaFuncSetAttribute(k_m2l_tm<R, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    k_m2l_tm<R, 3><<<(unsigned)S.nitems, TC_THREADS, sm, st>>>(
        o.P, Npad, reinterpret_cast<const __nv_bfloat16 *>(o.m2l_tc.p), S.items.p, S.src.p, S.cls.p, xs, S.part.p,
        o.margin >= 0 ? o.cls_K.p : nullptr, err);
    BEM_LAUNCH_CHECK();
}

template <int R>
void launch_m2l_tm_reduce(Context &c, const Operators &o, float *lc, cudaStream_t st) {
    Context::TmState &S = c.tm[R == 1 ? 0 : 1];
    if (S.nitems == 0) return;
    dim3 grid((unsigned)S.ntiles, TM_ROWS);
    k_tm_reduce<R><<<grid, 128, 0, st>>>(o.P, o.tc_Npad, S.box.p, S.item_off.p, S.items.p, S.part.p, lc);
    BEM_LAUNCH_CHECK();
}

template void launch_m2l_tm<1>(Context &, const Operators &, const float *, int64_t, int *, cudaStream_t);
template void launch_m2l_tm_reduce<1>(Context &, const Operators &, float *, cudaStream_t);

}  // namespace bem
