// Learned GMRES initial guess (the paper's method starts from the previous step's q,
// Sections 3.5 and 3.8; that stays the fallback).
//
// Per bubble m, features f_m = [c(phi_m), c(q_prev,m), c(q_prev,m) - c(q_prev2,m)] with
// c(x) = G+ x the least-squares real spherical-harmonic coefficients of degree <= lmax on the
// bubble's initial directions (the projector of the shape filter, Eqs. (3.22)-(3.23)) and
// q_prev2 the start of the solve before. Samples are taken in the Adams-Bashforth phase, where
// consecutive solves are one step apart. A multilayer perceptron
//   h1 = relu(W1 f + b1), h2 = relu(W2 h1 + b2), h3 = relu(W3 h2 + b3), y = W4 h3 + b4
// predicts the change of q's coefficients from the solve's base start q_prev (the extrapolated
// guess when bem_step_params.guess >= 1, else the previous solve's q), and the guess is
// q0_m = q_prev,m + G_m y_m. Features and targets are scaled per column by their root mean
// square over the recorded samples (computed at training); training minimises the mean of
// |y - (c(q) - c(q_prev)) / tscale|^2 / 2 over recorded solves with Adam.
//
// The matrix products run on the tensor cores (tcgen05.mma kind::f16, BF16 operands, FP32
// accumulation in tensor memory); weights keep an FP32 master copy. Every operand exists with its
// summation index contiguous (weights and, in training, activations and errors also transposed,
// written by the kernels that make them), in rows padded to 16 bytes, so all products of the forward
// and the backward pass are filled by 16-byte asynchronous copies. Waits on the MMA barriers are
// bounded.
#include "internal.h"

#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <random>

namespace cg = cooperative_groups;

namespace bem {

struct Mlp {
    bool ready = false;
    int lmax = 10, Psh = 121;
    int dims[5] = {0, 0, 0, 0, 0};
    DevBuf<float> W[4], b[4], mW[4], vW[4], mb[4], vb[4];
    DevBuf<float> grad;           // gradients in parameter order: W1, b1, ..., W4, b4
    DevBuf<__nv_bfloat16> Wb[4], WTb[4];  // BF16 weights [out][ld(in)] and transposed [in][ld(out)]
    float *gW(int i) const { return grad.p + goff[2 * i]; }
    float *gb(int i) const { return grad.p + goff[2 * i + 1]; }
    int64_t goff[9] = {0};        // offsets of W1, b1, ... in the parameter vector
    int64_t adam_t = 0;
    // recorded samples
    DevBuf<float> SF, ST;
    int64_t ns = 0, cap = 0;
    // work space (batch rows)
    int64_t wrows = 0;
    DevBuf<__nv_bfloat16> Hb[5];  // layer inputs in BF16 [rows][ld(dim)] (Hb[0] = features)
    DevBuf<__nv_bfloat16> HT[4];  // ... and transposed [dim][ld(rows)] (training)
    DevBuf<float> Z[4];           // pre-activations
    // gradient w.r.t. a layer's output (two: a layer's is read while the one below is written), in
    // FP32 [rows][dim], BF16 [rows][ld(dim)] and transposed [dim][ld(rows)]
    DevBuf<float> G[2];
    DevBuf<__nv_bfloat16> Gb[2], GT[2];
    DevBuf<float> loss;           // partial sums of the loss
    HostPinned<float> hloss;      // the same on the host, then the error flag
    ShBasis feat;
    DevBuf<double> qprev, cphi, cqp, cq, cqp_last;  // q_prev [N]; coefficients [M][Psh]
    bool have_last = false;
    bool uniform = false;  // the current solve is in the Adams-Bashforth phase
    bool record = false, use = false, compare = false;
    DevBuf<int> err;
    MlpStats stats;
    // input and output scales of the recorded data (per column: the root mean square over the
    // samples at the last training call; 1 before): the network sees features / fscale and is
    // trained on targets / tscale, and its output is multiplied by tscale in the guess
    DevBuf<float> fscale, tscale, Tb;
};

void mlp_free(Mlp *m) { delete m; }

namespace {

constexpr int GM = 128;           // tile rows
constexpr int GN = 64;            // tile columns
constexpr int GK = 64;            // K chunk (bf16): 128 bytes per row = 8 core matrices
constexpr int G_STAGES = 4, G_THREADS = 256;
constexpr int G_STAGE_ELEMS = (GM + GN) * GK;
constexpr int G_RED_PITCH = GN + 1;
constexpr int G_SMEM = G_STAGES * G_STAGE_ELEMS * 2 + 1024;  // aligned to 1024 by the kernel
static_assert(GM * G_RED_PITCH * 4 <= G_STAGES * G_STAGE_ELEMS * 2, "the split sums reuse the stages");
constexpr int G_SPLIT = 8;        // CTAs sharing a long K (one cluster)
constexpr int G_SPLIT_K = 512;    // from this K on
constexpr int LOSS_BLOCKS = 128;
constexpr uint32_t G_LBO = 128, G_SBO = 1024;
constexpr long long kWait = 1ll << 20;  // polls before a wait gives up, as in the other tensor-core kernels

constexpr int64_t ld8(int64_t n) { return (n + 7) / 8 * 8; }  // row length padded to 16 bytes of BF16

__device__ __forceinline__ uint32_t sa(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ uint64_t desc(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((G_LBO >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((G_SBO >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// kind::f16 instruction descriptor: D = F32, A = B = BF16, K-major.
constexpr uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity) {
    for (long long it = 0; it < kWait; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

enum { EPI_STORE = 0, EPI_BIAS_RELU = 1, EPI_BIAS = 2, EPI_RELU_MASK = 3 };

// C[m][n] = sum_k A(m,k) B(n,k), A(m,k) = A[m*lda + k], B(n,k) = B[n*ldb + k], rows 16-byte aligned.
// Epilogues: STORE: C = acc; BIAS: C = acc + bias[n]; BIAS_RELU: C = acc + bias[n] and
// H = bf16(relu(C)); RELU_MASK: C = acc where Zm[m*ldc + n] > 0, else 0, and H = bf16(C). HT (when set):
// H transposed.
//
// One 128 x 64 tile per CTA; K in chunks of 64, four of them in flight. The layers are at most a few
// hundred wide, so a product is a few dozen CTAs and bound by latency: a product of 1000 x 256 with
// K = 363 took 166 us as 8 CTAs that copied each chunk element by element between two barriers. Weight
// gradients (K = the batch, a small result) split K over the 8 CTAs of a cluster, whose sums are
// joined through distributed shared memory in rank order.
struct GemmOut {
    float *C;
    int64_t ldc;
    int epi;
    const float *bias, *Zm;
    __nv_bfloat16 *H, *HT;
    int64_t ldh, ldt;
};
// value of C at (m, n) from the sum a
__device__ __forceinline__ float gemm_epi(const GemmOut &o, int m, int n, float a) {
    if (o.epi == EPI_BIAS || o.epi == EPI_BIAS_RELU) a += o.bias[n];
    if (o.epi == EPI_RELU_MASK) a = o.Zm[(int64_t)m * o.ldc + n] > 0.f ? a : 0.f;
    return a;
}
__device__ __forceinline__ __nv_bfloat16 gemm_h(const GemmOut &o, float c) {
    return __float2bfloat16(o.epi == EPI_BIAS_RELU ? fmaxf(c, 0.f) : c);
}

template <bool SPLIT>
__global__ void __launch_bounds__(G_THREADS) k_gemm_bf16(int M, int N, int K, const __nv_bfloat16 *__restrict__ A,
                                                         int64_t lda, const __nv_bfloat16 *__restrict__ B, int64_t ldb,
                                                         GemmOut out, int *__restrict__ err) {
    extern __shared__ unsigned char g_smem[];
    __shared__ uint64_t bars[G_STAGES];  // a stage's MMAs are done
    __shared__ uint32_t tslot;
    unsigned char *smem = g_smem + ((1024u - (sa(g_smem) & 1023u)) & 1023u);
    __nv_bfloat16 *st0 = reinterpret_cast<__nv_bfloat16 *>(smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int rank = 0, nr = 1, tile_m = blockIdx.x;
    if constexpr (SPLIT) {
        cg::cluster_group cl = cg::this_cluster();
        rank = (int)cl.block_rank();
        nr = (int)cl.num_blocks();
        tile_m = blockIdx.x / nr;
    }
    const int m0 = tile_m * GM, n0 = blockIdx.y * GN;
    if (tid == 0) {
        for (int i = 0; i < G_STAGES; ++i) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sa(&bars[i])));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sa(&tslot)), "n"(GN));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tslot;
    const int nall = (K + GK - 1) / GK;
    const int c0 = rank * nall / nr, nc = (rank + 1) * nall / nr - c0;  // this CTA's chunks
    // 16-byte units (8 consecutive k of one row) into the canonical layout; past the edges zeros
    auto load = [&](int i) {
        if (i < nc) {
            __nv_bfloat16 *As = st0 + (i % G_STAGES) * G_STAGE_ELEMS, *Bs = As + GM * GK;
            const int k0 = (c0 + i) * GK;
#pragma unroll
            for (int v = 0; v < (GM + GN) * (GK / 8) / G_THREADS; ++v) {
                const int u = tid + v * G_THREADS, j = u % (GK / 8), k = k0 + j * 8;
                const bool isA = v < GM * (GK / 8) / G_THREADS;
                const int row = isA ? u / (GK / 8) : u / (GK / 8) - GM, g = (isA ? m0 : n0) + row;
                const bool in = g < (isA ? M : N) && k < K;
                const __nv_bfloat16 *src = isA ? A + (in ? (int64_t)g * lda + k : 0) : B + (in ? (int64_t)g * ldb + k : 0);
                __nv_bfloat16 *dst = (isA ? As : Bs) + (row / 8) * 512 + j * 64 + (row % 8) * 8;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sa(dst)), "l"(src),
                             "r"(in ? min(16, 2 * (K - k)) : 0)
                             : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");  // one group per call, empty past the end
    };
    bool ok = true;
    for (int i = 0; i < G_STAGES; ++i) load(i);
    for (int i = 0; i < nc; ++i) {
        asm volatile("cp.async.wait_group %0;" ::"n"(G_STAGES - 2) : "memory");  // chunk i (this thread's part)
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;");
            const __nv_bfloat16 *As = st0 + (i % G_STAGES) * G_STAGE_ELEMS, *Bs = As + GM * GK;
            const int ksteps = (min(GK, K - (c0 + i) * GK) + 15) / 16;
            for (int s = 0; s < ksteps; ++s) {
                const uint32_t o = s * 2 * G_LBO;
                const uint32_t acc = (i > 0 || s > 0) ? 1u : 0u;
                asm volatile(
                    "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
                    "l"(desc(sa(As) + o)), "l"(desc(sa(Bs) + o)), "r"(idesc_bf16(GM, GN)), "r"(acc));
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             sa(&bars[i % G_STAGES]))
                         : "memory");
        }
        __syncwarp();
        // refill the stage of chunk i - 1, once its MMAs are done
        if (i >= 1 && i - 1 + G_STAGES < nc) {
            ok = ok && wait_bar(sa(&bars[(i - 1) % G_STAGES]), ((i - 1) / G_STAGES) & 1);
            if (ok) load(i - 1 + G_STAGES);
            else asm volatile("cp.async.commit_group;" ::: "memory");
        } else {
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    // the last commit covers every MMA before it
    if (nc > 0) ok = wait_bar(sa(&bars[(nc - 1) % G_STAGES]), ((nc - 1) / G_STAGES) & 1) && ok;
    ok = __syncthreads_and(ok);
    if (!ok && tid == 0) atomicOr(err, 1);
    asm volatile("tcgen05.fence::after_thread_sync;");
    const int row = (warp & 3) * 32 + lane, qh = warp >> 2;  // TMEM lanes of a warp; the halves take half the columns
    // the tile goes through shared memory ([row][G_RED_PITCH], in the free stages), so that every store
    // below is coalesced: 192 scattered stores per thread took most of a product's 32 us
    float *red = reinterpret_cast<float *>(smem);
    if (ok) {
        for (int q = qh * (GN / 2); q < (qh + 1) * (GN / 2); q += 16) {
            uint32_t v[16];
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                  "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
                  "=r"(v[15])
                : "r"(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)q));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int i = 0; i < 16; ++i) red[row * G_RED_PITCH + q + i] = nc > 0 ? __uint_as_float(v[i]) : 0.f;
        }
    }
    if constexpr (SPLIT) {
        cg::cluster_group cl = cg::this_cluster();
        cl.sync();
        // rank r joins the rows r, r + nr, ... of the tile (a CTA whose wait ran out has set the flag)
        for (int e = tid; e < GM / nr * GN; e += G_THREADS) {
            const int rr = rank + e / GN * nr, q = e % GN;
            if (m0 + rr >= M || n0 + q >= N) continue;
            float a = 0.f;
            for (int c = 0; c < nr; ++c) a += cl.map_shared_rank(red, c)[rr * G_RED_PITCH + q];
            out.C[(int64_t)(m0 + rr) * out.ldc + n0 + q] = a;  // a weight gradient: EPI_STORE
        }
        cl.sync();  // no CTA leaves while another still reads its sums
    } else {
        __syncthreads();
        if (ok) {
#pragma unroll 4
            for (int e = tid; e < GM * GN; e += G_THREADS) {
                const int rr = e / GN, q = e % GN, m = m0 + rr, n = n0 + q;
                if (m >= M || n >= N) continue;
                const float a = gemm_epi(out, m, n, red[rr * G_RED_PITCH + q]);
                red[rr * G_RED_PITCH + q] = a;
                out.C[(int64_t)m * out.ldc + n] = a;
                if (out.H) out.H[(int64_t)m * out.ldh + n] = gemm_h(out, a);
            }
            if (out.HT) {
                __syncthreads();
#pragma unroll 4
                for (int e = tid; e < GM * GN; e += G_THREADS) {
                    const int rr = e % GM, q = e / GM, m = m0 + rr, n = n0 + q;
                    if (m < M && n < N) out.HT[(int64_t)n * out.ldt + m] = gemm_h(out, red[rr * G_RED_PITCH + q]);
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(GN));
}

// H[r][c] = bf16(x[r][c] / scale[c]) (scale may be null), rows of ldh; HT (when set) transposed, rows of
// ldt. Tiles of 32 x 32 through shared memory, row of tiles after row of tiles on gridDim.x (the rows may be
// millions, and a column of tiles after another reads 50000 rows 11 us slower).
template <class T>
__global__ void k_to_bf16(int rows, int cols, const T *__restrict__ x, const float *__restrict__ scale,
                          __nv_bfloat16 *__restrict__ H, int64_t ldh, __nv_bfloat16 *__restrict__ HT, int64_t ldt) {
    __shared__ __nv_bfloat16 t[32][34];
    const int tc = (cols + 31) / 32, r0 = (int)(blockIdx.x / tc) * 32, q0 = (int)(blockIdx.x % tc) * 32;
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int r = r0 + i, q = q0 + threadIdx.x;
        if (r < rows && q < cols) {
            const float v = (float)x[(int64_t)r * cols + q];
            const __nv_bfloat16 h = __float2bfloat16(scale ? v / scale[q] : v);
            H[(int64_t)r * ldh + q] = h;
            t[i][threadIdx.x] = h;
        }
    }
    if (!HT) return;
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int q = q0 + i, r = r0 + threadIdx.x;
        if (r < rows && q < cols) HT[(int64_t)q * ldt + r] = t[threadIdx.x][i];
    }
}

template <class S, class D>
__global__ void k_convert(int64_t n, const S *__restrict__ x, D *__restrict__ y) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = (D)x[i];
}

// G = (Y - T) / B (also BF16 and transposed); partial sums of the loss, one per block (LOSS_BLOCKS of
// them, added up in order on the host). Tiles of 32 rows x 32 columns.
__global__ void __launch_bounds__(256) k_loss_grad(int rows, int cols, const float *__restrict__ Y,
                                                   const float *__restrict__ T, float *__restrict__ G,
                                                   __nv_bfloat16 *__restrict__ Gb, int64_t ldh,
                                                   __nv_bfloat16 *__restrict__ GT, int64_t ldt, float *__restrict__ loss) {
    __shared__ float red[256];
    __shared__ __nv_bfloat16 t[32][34];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int tc = (cols + 31) / 32, nt = tc * ((rows + 31) / 32);
    float s = 0.f;
    for (int tile = blockIdx.x; tile < nt; tile += gridDim.x) {
        const int r0 = tile / tc * 32, q0 = tile % tc * 32;
        __syncthreads();
        for (int i = ty; i < 32; i += 8) {
            const int r = r0 + i, q = q0 + tx;
            if (r < rows && q < cols) {
                const int64_t ix = (int64_t)r * cols + q;
                const float d = Y[ix] - T[ix];
                s += d * d;
                const float g = d / (float)rows;
                G[ix] = g;
                const __nv_bfloat16 h = __float2bfloat16(g);
                Gb[(int64_t)r * ldh + q] = h;
                t[i][tx] = h;
            }
        }
        __syncthreads();
        for (int i = ty; i < 32; i += 8) {
            const int q = q0 + i, r = r0 + tx;
            if (r < rows && q < cols) GT[(int64_t)q * ldt + r] = t[tx][i];
        }
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
        if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) loss[blockIdx.x] = 0.5f * red[0] / (float)rows;
}

// db[n] = sum_rows G[row][n]: 32 columns per block, 32 rows at a time, joined in a fixed order
__global__ void __launch_bounds__(1024) k_colsum(int rows, int cols, const float *__restrict__ G, float *__restrict__ db) {
    __shared__ float red[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, n = blockIdx.x * 32 + tx;
    float s = 0.f;
    if (n < cols)
        for (int r = ty; r < rows; r += 32) s += G[(int64_t)r * cols + n];
    red[ty][tx] = s;
    __syncthreads();
    if (ty == 0 && n < cols) {
        float t = 0.f;
#pragma unroll
        for (int k = 0; k < 32; ++k) t += red[k][tx];
        db[n] = t;
    }
}

// pb, pt (when set): the BF16 copies of a weight matrix with `din` columns, [out][ldb] and transposed
__global__ void k_adam(int64_t n, float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, float lr, float b1, float b2, float c1, float c2, float eps, int din,
                       __nv_bfloat16 *__restrict__ pb, int64_t ldb, __nv_bfloat16 *__restrict__ pt, int64_t ldt) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    float mm = b1 * m[i] + (1.f - b1) * g[i];
    float vv = b2 * v[i] + (1.f - b2) * g[i] * g[i];
    m[i] = mm;
    v[i] = vv;
    float x = p[i] - lr * (mm / c1) / (sqrtf(vv / c2) + eps);
    p[i] = x;
    if (pb) {
        const int64_t o = i / din, k = i - o * din;
        const __nv_bfloat16 h = __float2bfloat16(x);
        pb[o * ldb + k] = h;
        pt[k * ldt + o] = h;
    }
}

// out[m][p] = sum_i Gp_m[p][i] x[a_m + i]  (per-bubble SH coefficients; one block per bubble)
__global__ void k_sh_project(int64_t M, const int64_t *__restrict__ voff, const int32_t *__restrict__ shape_of,
                             const int64_t *__restrict__ g_off, int P, const double *__restrict__ Gp,
                             const double *__restrict__ x, double *__restrict__ out) {
    int m = blockIdx.x;
    int64_t a = voff[m];
    int nd = (int)(voff[m + 1] - a);
    const double *G = Gp + g_off[shape_of[m]];
    for (int p = threadIdx.x; p < P; p += blockDim.x) {
        double s = 0.0;
        for (int i = 0; i < nd; ++i) s = fma(G[(size_t)p * nd + i], x[a + i], s);
        out[(size_t)m * P + p] = s;
    }
}

// q[a_m + i] = qprev[a_m + i] + sum_p G_m[i][p] y[m][p]
__global__ void k_sh_synth_add(int64_t M, const int64_t *__restrict__ voff, const int32_t *__restrict__ shape_of,
                               const int64_t *__restrict__ g_off, int P, const double *__restrict__ G,
                               const float *__restrict__ y, const float *__restrict__ yscale,
                               const double *__restrict__ qprev, double *__restrict__ q) {
    int m = blockIdx.x;
    int64_t a = voff[m];
    int nd = (int)(voff[m + 1] - a);
    const double *Gm = G + g_off[shape_of[m]];
    for (int i = threadIdx.x; i < nd; i += blockDim.x) {
        double s = qprev[a + i];
        for (int p = 0; p < P; ++p)
            s = fma(Gm[(size_t)i * P + p], (double)y[(size_t)m * P + p] * (double)yscale[p], s);
        q[a + i] = s;
    }
}

// per column: out[j] = sqrt(mean_r X[r][j]^2) (1 where that is 0); one thread per column
__global__ void k_col_rms(int64_t rows, int cols, const float *__restrict__ X, float *__restrict__ out) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= cols) return;
    double s = 0.0;
    for (int64_t r = 0; r < rows; ++r) {
        const double v = X[r * cols + j];
        s += v * v;
    }
    const double rms = sqrt(s / (double)(rows > 0 ? rows : 1));
    out[j] = rms > 0.0 ? (float)rms : 1.f;
}

// y[r][j] = x[r][j] / scale[j] (training targets)
__global__ void k_div_cols(int64_t n, int cols, const float *__restrict__ x, const float *__restrict__ scale,
                           float *__restrict__ y) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) y[i] = x[i] / scale[i % cols];
}

// features [M][3P] (float): c(phi), c(q_prev), c(q_prev) - c(q_prev2); targets [M][P] = c(q) - c(q_prev)
__global__ void k_pack_features(int64_t M, int P, const double *__restrict__ cphi, const double *__restrict__ cqp,
                                const double *__restrict__ cqp_last, float *__restrict__ F) {
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= M * 3 * P) return;
    int64_t m = e / (3 * P);
    int k = (int)(e % (3 * P));
    double v;
    if (k < P) v = cphi[m * P + k];
    else if (k < 2 * P) v = cqp[m * P + (k - P)];
    else v = cqp_last ? cqp[m * P + (k - 2 * P)] - cqp_last[m * P + (k - 2 * P)] : 0.0;
    F[e] = (float)v;
}

__global__ void k_pack_targets(int64_t M, int P, const double *__restrict__ cq, const double *__restrict__ cqp,
                               float *__restrict__ T) {
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= M * P) return;
    T[e] = (float)(cq[e] - cqp[e]);
}

Mlp &mlp_of(Context &c) {
    if (!c.mlp) c.mlp = new Mlp();
    return *c.mlp;
}

void gemm(Context &c, Mlp &m, int M, int N, int K, const __nv_bfloat16 *A, int64_t lda, const __nv_bfloat16 *B,
          int64_t ldb, const GemmOut &out) {
    // the split form stores plain sums only (weight gradients; the layers' products have K <= 363)
    const bool split = K >= G_SPLIT_K && out.epi == EPI_STORE && !out.H && !out.HT;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(div_up(M, GM) * (split ? G_SPLIT : 1)), (unsigned)div_up(N, GN));
    cfg.blockDim = dim3(G_THREADS);
    cfg.dynamicSmemBytes = G_SMEM;
    cfg.stream = c.stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = G_SPLIT;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = split ? 1 : 0;
    auto kern = split ? k_gemm_bf16<true> : k_gemm_bf16<false>;
    BEM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, G_SMEM));
    BEM_CUDA(cudaLaunchKernelEx(&cfg, kern, M, N, K, A, lda, B, ldb, out, m.err.p));
    BEM_LAUNCH_CHECK();
}

template <class T>
void to_bf16(Context &c, int rows, int cols, const T *x, const float *scale, __nv_bfloat16 *H, __nv_bfloat16 *HT) {
    const unsigned grid = (unsigned)((int64_t)div_up(rows, 32) * div_up(cols, 32));
    k_to_bf16<T><<<grid, dim3(32, 8), 0, c.stream>>>(rows, cols, x, scale, H, ld8(cols), HT, ld8(rows));
    BEM_LAUNCH_CHECK();
}

void ensure_work(Mlp &m, int64_t rows) {
    if (rows <= m.wrows) return;
    m.wrows = rows;
    const int dmax = *std::max_element(m.dims, m.dims + 5);
    for (int i = 0; i <= 4; ++i) m.Hb[i].resize((size_t)(rows * ld8(m.dims[i])));
    for (int i = 0; i < 4; ++i) {
        m.HT[i].resize((size_t)(m.dims[i] * ld8(rows)));
        m.Z[i].resize((size_t)rows * m.dims[i + 1]);
    }
    for (int i = 0; i < 2; ++i) {
        m.G[i].resize((size_t)rows * dmax);
        m.Gb[i].resize((size_t)(rows * ld8(dmax)));
        m.GT[i].resize((size_t)(dmax * ld8(rows)));
    }
    m.loss.resize(LOSS_BLOCKS);
}

// BF16 copies of the weights of layer i, also transposed
void refresh_weights(Context &c, Mlp &m, int i) {
    to_bf16(c, m.dims[i + 1], m.dims[i], m.W[i].p, (const float *)nullptr, m.Wb[i].p, m.WTb[i].p);
}

// Forward pass on Hb[0] (rows x dims[0]); Z[3] holds the output y. train: also the transposed
// activations that the backward pass reads.
void forward(Context &c, Mlp &m, int rows, bool train) {
    for (int i = 0; i < 4; ++i) {
        const bool last = i == 3;
        const int din = m.dims[i], dout = m.dims[i + 1];
        GemmOut o{m.Z[i].p, dout, last ? EPI_BIAS : EPI_BIAS_RELU, m.b[i].p, nullptr, nullptr, nullptr, ld8(dout), ld8(rows)};
        if (!last) {
            o.H = m.Hb[i + 1].p;
            o.HT = train ? m.HT[i + 1].p : nullptr;
        }
        gemm(c, m, rows, dout, din, m.Hb[i].p, ld8(din), m.Wb[i].p, ld8(din), o);
    }
}

// Gradients (into m.grad) and the loss's partial sums for targets T (rows x dims[4], float).
void backward(Context &c, Mlp &m, int rows, const float *T) {
    int cur = 0;
    k_loss_grad<<<LOSS_BLOCKS, 256, 0, c.stream>>>(rows, m.dims[4], m.Z[3].p, T, m.G[0].p, m.Gb[0].p, ld8(m.dims[4]),
                                                   m.GT[0].p, ld8(rows), m.loss.p);
    BEM_LAUNCH_CHECK();
    for (int i = 3; i >= 0; --i, cur ^= 1) {
        const int dout = m.dims[i + 1], din = m.dims[i];
        // dW_i = G^T H_i  [dout x din], summed over the rows
        gemm(c, m, dout, din, rows, m.GT[cur].p, ld8(rows), m.HT[i].p, ld8(rows),
             GemmOut{m.gW(i), din, EPI_STORE, nullptr, nullptr, nullptr, nullptr, 0, 0});
        k_colsum<<<div_up(dout, 32), 1024, 0, c.stream>>>(rows, dout, m.G[cur].p, m.gb(i));
        BEM_LAUNCH_CHECK();
        if (i > 0)  // G_prev = (G W_i) masked by Z_{i-1} > 0
            gemm(c, m, rows, din, dout, m.Gb[cur].p, ld8(dout), m.WTb[i].p, ld8(dout),
                 GemmOut{m.G[cur ^ 1].p, din, EPI_RELU_MASK, nullptr, m.Z[i - 1].p, m.Gb[cur ^ 1].p, m.GT[cur ^ 1].p,
                         ld8(din), ld8(rows)});
    }
}

// The loss of the last backward pass (its partial sums, in order) after everything queued; fails when a
// product's wait ran out.
float read_loss(Context &c, Mlp &m) {
    float *h = m.hloss.get(LOSS_BLOCKS + 1);
    BEM_CUDA(cudaMemcpyAsync(h, m.loss.p, LOSS_BLOCKS * sizeof(float), cudaMemcpyDeviceToHost, c.stream));
    BEM_CUDA(cudaMemcpyAsync(h + LOSS_BLOCKS, m.err.p, sizeof(int), cudaMemcpyDeviceToHost, c.stream));
    BEM_CUDA(cudaStreamSynchronize(c.stream));
    int bad;
    std::memcpy(&bad, h + LOSS_BLOCKS, sizeof(int));
    if (bad) fail(BEM_ERR_TIMEOUT, "tensor-core GEMM wait ran out");
    double s = 0.0;
    for (int i = 0; i < LOSS_BLOCKS; ++i) s += h[i];
    return (float)s;
}

void check_err(Context &c, Mlp &m) {
    int h = 0;
    BEM_CUDA(cudaMemcpyAsync(&h, m.err.p, sizeof(int), cudaMemcpyDeviceToHost, c.stream));
    BEM_CUDA(cudaStreamSynchronize(c.stream));
    if (h) fail(BEM_ERR_TIMEOUT, "tensor-core GEMM wait ran out");
}

}  // namespace

int64_t mlp_num_params(const Mlp &m) {
    int64_t n = 0;
    for (int i = 0; i < 4; ++i) n += (int64_t)m.dims[i + 1] * m.dims[i] + m.dims[i + 1];
    return n;
}

void mlp_init(Context &c, int hidden, int lmax, uint64_t seed, const double *xyz0) {
    if (hidden < 16 || hidden > 256 || hidden % 16) fail(BEM_ERR_ARG, "hidden width must be a multiple of 16 in 16..256");
    if (lmax < 0 || lmax > 10) fail(BEM_ERR_ARG, "lmax must be in 0..10");
    Mlp &m = mlp_of(c);
    m.lmax = lmax;
    m.Psh = (lmax + 1) * (lmax + 1);
    const int dims[5] = {3 * m.Psh, hidden, hidden, hidden, m.Psh};
    std::memcpy(m.dims, dims, sizeof(dims));
    m.err.resize(1);
    m.loss.resize(1);
    BEM_CUDA(cudaMemsetAsync(m.err.p, 0, sizeof(int), c.stream));
    std::mt19937_64 rng(seed);
    std::normal_distribution<double> nd(0.0, 1.0);
    for (int i = 0; i < 4; ++i) {
        const int64_t nw = (int64_t)dims[i + 1] * dims[i];
        std::vector<float> w(nw), bz(dims[i + 1], 0.f);
        const double sc = std::sqrt(2.0 / dims[i]) * (i == 3 ? 0.1 : 1.0);
        for (auto &x : w) x = (float)(nd(rng) * sc);
        for (auto *bf : {&m.W[i], &m.mW[i], &m.vW[i]}) bf->resize(nw);
        for (auto *bf : {&m.b[i], &m.mb[i], &m.vb[i]}) bf->resize(dims[i + 1]);
        m.goff[2 * i + 1] = m.goff[2 * i] + nw;
        m.goff[2 * i + 2] = m.goff[2 * i + 1] + dims[i + 1];
        m.Wb[i].resize(dims[i + 1] * ld8(dims[i]));
        m.WTb[i].resize(dims[i] * ld8(dims[i + 1]));
        BEM_CUDA(cudaMemcpyAsync(m.W[i].p, w.data(), nw * sizeof(float), cudaMemcpyHostToDevice, c.stream));
        BEM_CUDA(cudaMemcpyAsync(m.b[i].p, bz.data(), bz.size() * sizeof(float), cudaMemcpyHostToDevice, c.stream));
        BEM_CUDA(cudaMemsetAsync(m.mW[i].p, 0, nw * sizeof(float), c.stream));
        BEM_CUDA(cudaMemsetAsync(m.vW[i].p, 0, nw * sizeof(float), c.stream));
        BEM_CUDA(cudaMemsetAsync(m.mb[i].p, 0, dims[i + 1] * sizeof(float), c.stream));
        BEM_CUDA(cudaMemsetAsync(m.vb[i].p, 0, dims[i + 1] * sizeof(float), c.stream));
        refresh_weights(c, m, i);
        BEM_CUDA(cudaStreamSynchronize(c.stream));  // host vectors go out of scope
    }
    m.grad.resize(m.goff[8]);
    m.adam_t = 0;
    m.ns = 0;
    m.wrows = 0;
    m.have_last = false;
    {
        std::vector<float> one(std::max(dims[0], dims[4]), 1.f);
        m.fscale.resize(dims[0]);
        m.tscale.resize(dims[4]);
        BEM_CUDA(cudaMemcpyAsync(m.fscale.p, one.data(), dims[0] * sizeof(float), cudaMemcpyHostToDevice, c.stream));
        BEM_CUDA(cudaMemcpyAsync(m.tscale.p, one.data(), dims[4] * sizeof(float), cudaMemcpyHostToDevice, c.stream));
        BEM_CUDA(cudaStreamSynchronize(c.stream));
    }
    // features basis from the initial shapes
    DevBuf<int> bad;
    bad.resize(1);
    BEM_CUDA(cudaMemsetAsync(bad.p, 0, sizeof(int), c.stream));
    build_sh_basis(c, lmax + 1, m.feat, bad.p, xyz0);
    int hb = 0;
    BEM_CUDA(cudaMemcpyAsync(&hb, bad.p, sizeof(int), cudaMemcpyDeviceToHost, c.stream));
    BEM_CUDA(cudaStreamSynchronize(c.stream));
    if (hb) fail(BEM_ERR_MESH, "singular spherical-harmonic basis for the features");
    m.ready = true;
}

void mlp_set_mode(Context &c, int record, int use, int compare) {
    Mlp &m = mlp_of(c);
    if (!m.ready) fail(BEM_ERR_NOT_BUILT, "bem_mlp_init has not been called");
    m.record = record != 0;
    m.use = use != 0;
    m.compare = compare != 0;
}

bool mlp_active(Context &c) { return c.mlp && c.mlp->ready && (c.mlp->record || c.mlp->use); }
bool mlp_compare(Context &c) { return c.mlp && c.mlp->ready && c.mlp->use && c.mlp->compare && c.mlp->uniform; }

// Before a solve with initial guess q (= q_prev): features; when the solve is in the uniform
// (Adams-Bashforth) phase, record them and, with `use`, replace q by q_prev + G y.
void mlp_before_solve(Context &c, const double *phi, double *q, bool uniform) {
    Mlp &m = *c.mlp;
    const int64_t M = c.M, N = c.N;
    const int P = m.Psh;
    m.uniform = uniform;
    m.qprev.resize(N);
    m.cphi.resize((size_t)M * P);
    m.cqp.resize((size_t)M * P);
    m.cq.resize((size_t)M * P);
    m.cqp_last.resize((size_t)M * P);
    BEM_CUDA(cudaMemcpyAsync(m.qprev.p, q, N * sizeof(double), cudaMemcpyDeviceToDevice, c.stream));
    DevBuf<int64_t> &voff = c.voff_d;
    k_sh_project<<<(unsigned)M, 128, 0, c.stream>>>(M, voff.p, m.feat.shape_of.p, m.feat.g_off.p, P, m.feat.Gp.p, phi,
                                                    m.cphi.p);
    k_sh_project<<<(unsigned)M, 128, 0, c.stream>>>(M, voff.p, m.feat.shape_of.p, m.feat.g_off.p, P, m.feat.Gp.p, q,
                                                    m.cqp.p);
    BEM_LAUNCH_CHECK();
    ensure_work(m, M);
    DevBuf<float> F;
    F.resize((size_t)M * 3 * P);
    k_pack_features<<<div_up(M * 3 * P, 256), 256, 0, c.stream>>>(M, P, m.cphi.p, m.cqp.p,
                                                                  m.have_last ? m.cqp_last.p : nullptr, F.p);
    BEM_LAUNCH_CHECK();
    BEM_CUDA(cudaMemcpyAsync(m.cqp_last.p, m.cqp.p, M * P * sizeof(double), cudaMemcpyDeviceToDevice, c.stream));
    m.have_last = true;
    if (m.record && uniform) {
        if (m.ns + M > m.cap) {
            int64_t nc = std::max<int64_t>(2 * m.cap, m.ns + M);
            DevBuf<float> nf, nt;
            nf.resize((size_t)nc * 3 * P);
            nt.resize((size_t)nc * P);
            if (m.ns) {
                BEM_CUDA(cudaMemcpyAsync(nf.p, m.SF.p, m.ns * 3 * P * sizeof(float), cudaMemcpyDeviceToDevice, c.stream));
                BEM_CUDA(cudaMemcpyAsync(nt.p, m.ST.p, m.ns * P * sizeof(float), cudaMemcpyDeviceToDevice, c.stream));
            }
            BEM_CUDA(cudaStreamSynchronize(c.stream));
            std::swap(m.SF.p, nf.p);
            std::swap(m.SF.cap, nf.cap);
            std::swap(m.SF.n, nf.n);
            std::swap(m.ST.p, nt.p);
            std::swap(m.ST.cap, nt.cap);
            std::swap(m.ST.n, nt.n);
            m.cap = nc;
        }
        BEM_CUDA(cudaMemcpyAsync(m.SF.p + m.ns * 3 * P, F.p, M * 3 * P * sizeof(float), cudaMemcpyDeviceToDevice,
                                 c.stream));
    }
    if (m.use && uniform) {
        to_bf16(c, (int)M, 3 * P, F.p, m.fscale.p, m.Hb[0].p, (__nv_bfloat16 *)nullptr);
        forward(c, m, (int)M, false);
        k_sh_synth_add<<<(unsigned)M, 128, 0, c.stream>>>(M, voff.p, m.feat.shape_of.p, m.feat.g_off.p, P, m.feat.G.p,
                                                          m.Z[3].p, m.tscale.p, m.qprev.p, q);
        BEM_LAUNCH_CHECK();
    }
    BEM_CUDA(cudaStreamSynchronize(c.stream));
}

const double *mlp_qprev(Context &c) { return c.mlp->qprev.p; }

// After the solve: with `record`, the target c(q) - c(q_prev) of the sample stored before.
void mlp_after_solve(Context &c, const double *q) {
    Mlp &m = *c.mlp;
    if (!m.record || !m.uniform) return;
    const int64_t M = c.M;
    const int P = m.Psh;
    DevBuf<int64_t> &voff = c.voff_d;
    k_sh_project<<<(unsigned)M, 128, 0, c.stream>>>(M, voff.p, m.feat.shape_of.p, m.feat.g_off.p, P, m.feat.Gp.p, q,
                                                    m.cq.p);
    BEM_LAUNCH_CHECK();
    k_pack_targets<<<div_up(M * P, 256), 256, 0, c.stream>>>(M, P, m.cq.p, m.cqp.p, m.ST.p + m.ns * P);
    BEM_LAUNCH_CHECK();
    m.ns += M;
}

// Adam over the recorded samples in minibatches of `batch` rows, `epochs` passes; returns the
// mean loss of the last epoch.
double mlp_train(Context &c, int epochs, int batch, double lr) {
    Mlp &m = mlp_of(c);
    if (!m.ready) fail(BEM_ERR_NOT_BUILT, "bem_mlp_init has not been called");
    if (m.ns == 0) fail(BEM_ERR_ARG, "no recorded samples");
    batch = (int)std::min<int64_t>(std::max(1, batch), m.ns);
    ensure_work(m, batch);
    const int P = m.Psh;
    // column scales of the recorded features and targets (the network learns the scaled map)
    k_col_rms<<<div_up(3 * P, 128), 128, 0, c.stream>>>(m.ns, 3 * P, m.SF.p, m.fscale.p);
    k_col_rms<<<div_up(P, 128), 128, 0, c.stream>>>(m.ns, P, m.ST.p, m.tscale.p);
    BEM_LAUNCH_CHECK();
    m.Tb.resize((size_t)batch * P);
    double last = 0.0;
    for (int ep = 0; ep < epochs; ++ep) {
        double tot = 0.0;
        int nb = 0;
        for (int64_t r0 = 0; r0 < m.ns; r0 += batch) {
            const int rows = (int)std::min<int64_t>(batch, m.ns - r0);
            to_bf16(c, rows, 3 * P, m.SF.p + r0 * 3 * P, m.fscale.p, m.Hb[0].p, m.HT[0].p);
            k_div_cols<<<div_up((int64_t)rows * P, 256), 256, 0, c.stream>>>((int64_t)rows * P, P, m.ST.p + r0 * P,
                                                                             m.tscale.p, m.Tb.p);
            BEM_LAUNCH_CHECK();
            forward(c, m, rows, true);
            backward(c, m, rows, m.Tb.p);
            m.adam_t += 1;
            const float b1 = 0.9f, b2 = 0.999f;
            const float c1 = 1.f - std::pow(b1, (float)m.adam_t), c2 = 1.f - std::pow(b2, (float)m.adam_t);
            for (int i = 0; i < 4; ++i) {
                int64_t nw = (int64_t)m.dims[i + 1] * m.dims[i];
                k_adam<<<div_up(nw, 256), 256, 0, c.stream>>>(nw, m.W[i].p, m.gW(i), m.mW[i].p, m.vW[i].p, (float)lr,
                                                               b1, b2, c1, c2, 1e-8f, m.dims[i], m.Wb[i].p,
                                                               ld8(m.dims[i]), m.WTb[i].p, ld8(m.dims[i + 1]));
                k_adam<<<div_up(m.dims[i + 1], 256), 256, 0, c.stream>>>(m.dims[i + 1], m.b[i].p, m.gb(i), m.mb[i].p,
                                                                          m.vb[i].p, (float)lr, b1, b2, c1, c2, 1e-8f, 1,
                                                                          nullptr, 0, nullptr, 0);
                BEM_LAUNCH_CHECK();
            }
            tot += read_loss(c, m);
            ++nb;
        }
        last = tot / std::max(1, nb);
    }
    return last;
}

// Loss and flat gradients (W1, b1, ..., W4, b4; W row-major [out][in]) for one batch given in
// FP64 host or device arrays already copied to device (F [B][din], T [B][dout]).
double mlp_loss_grad(Context &c, int B, const double *F, const double *T, double *grads_dev) {
    Mlp &m = mlp_of(c);
    if (!m.ready) fail(BEM_ERR_NOT_BUILT, "bem_mlp_init has not been called");
    ensure_work(m, B);
    const int din = m.dims[0], dout = m.dims[4];
    const int64_t nt = (int64_t)B * dout, np = mlp_num_params(m);
    to_bf16(c, B, din, F, (const float *)nullptr, m.Hb[0].p, m.HT[0].p);
    m.Tb.resize((size_t)nt);
    k_convert<double, float><<<std::min(div_up(nt, 256), 1024), 256, 0, c.stream>>>(nt, T, m.Tb.p);
    BEM_LAUNCH_CHECK();
    forward(c, m, B, true);
    backward(c, m, B, m.Tb.p);
    k_convert<float, double><<<std::min(div_up(np, 256), 1024), 256, 0, c.stream>>>(np, m.grad.p, grads_dev);
    BEM_LAUNCH_CHECK();
    return read_loss(c, m);
}

// Forward only: Y [B][dout] (device FP64) from F [B][din] (device FP64).
void mlp_forward(Context &c, int B, const double *F, double *Y) {
    Mlp &m = mlp_of(c);
    if (!m.ready) fail(BEM_ERR_NOT_BUILT, "bem_mlp_init has not been called");
    ensure_work(m, B);
    const int din = m.dims[0], dout = m.dims[4];
    to_bf16(c, B, din, F, (const float *)nullptr, m.Hb[0].p, (__nv_bfloat16 *)nullptr);
    forward(c, m, B, false);
    const int64_t ny = (int64_t)B * dout;
    k_convert<float, double><<<std::min(div_up(ny, 256), 1024), 256, 0, c.stream>>>(ny, m.Z[3].p, Y);
    BEM_LAUNCH_CHECK();
    check_err(c, m);
}

// Flat FP64 parameter vector in the order W1, b1, ..., W4, b4 (host memory).
void mlp_get_params(Context &c, double *out) {
    Mlp &m = mlp_of(c);
    if (!m.ready) fail(BEM_ERR_NOT_BUILT, "bem_mlp_init has not been called");
    int64_t off = 0;
    for (int i = 0; i < 4; ++i) {
        int64_t nw = (int64_t)m.dims[i + 1] * m.dims[i];
        std::vector<float> a(nw), bb(m.dims[i + 1]);
        BEM_CUDA(cudaMemcpyAsync(a.data(), m.W[i].p, nw * sizeof(float), cudaMemcpyDeviceToHost, c.stream));
        BEM_CUDA(cudaMemcpyAsync(bb.data(), m.b[i].p, bb.size() * sizeof(float), cudaMemcpyDeviceToHost, c.stream));
        BEM_CUDA(cudaStreamSynchronize(c.stream));
        for (int64_t k = 0; k < nw; ++k) out[off++] = a[k];
        for (float v : bb) out[off++] = v;
    }
}

void mlp_set_params(Context &c, const double *in) {
    Mlp &m = mlp_of(c);
    if (!m.ready) fail(BEM_ERR_NOT_BUILT, "bem_mlp_init has not been called");
    int64_t off = 0;
    for (int i = 0; i < 4; ++i) {
        int64_t nw = (int64_t)m.dims[i + 1] * m.dims[i];
        std::vector<float> a(in + off, in + off + nw);
        off += nw;
        std::vector<float> bb(in + off, in + off + m.dims[i + 1]);
        off += m.dims[i + 1];
        BEM_CUDA(cudaMemcpyAsync(m.W[i].p, a.data(), nw * sizeof(float), cudaMemcpyHostToDevice, c.stream));
        BEM_CUDA(cudaMemcpyAsync(m.b[i].p, bb.data(), bb.size() * sizeof(float), cudaMemcpyHostToDevice, c.stream));
        refresh_weights(c, m, i);
        BEM_CUDA(cudaStreamSynchronize(c.stream));
    }
}

int64_t mlp_samples(Context &c) { return c.mlp ? c.mlp->ns : 0; }
MlpStats &mlp_stats(Context &c) { return mlp_of(c).stats; }
const int *mlp_dims(Context &c) { return mlp_of(c).dims; }

}  // namespace bem
