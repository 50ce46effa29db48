// M2M and L2L of the far field (Section 3.7): multipoles of the children summed into their
// parent, M_parent = sum_o T_o M_child(o), and local expansions handed down, L_child(o) += S_o
// L_parent, one dense P x P matrix per child octant o and level.
//
// One block takes up to 64 columns (64 / R children x R right-hand sides) of one octant against 64
// coefficients of the result. Degree n of the result needs only the degrees k <= n (M2M) or k >= n
// (L2L) of the source, so a block walks the columns of T_o that can be non-zero: half of the
// matrix. M2M runs as clusters of 8 blocks, one per octant, that join their sums through
// distributed shared memory in octant order (TwoSum): no row per translation in global memory, no
// reduction launch. Before, one level of a 192600-point cluster took 33 us up and 71 us down (44
// blocks of 128 x 128 outputs over all P columns, the operator loaded element by element).
//
// A block's columns are the children that exist in its octant, moved together, in groups of 16: a
// surface's tree has about four children per parent, a tree deeper than its points are dense has one. (A
// warp holds eight columns of every group and skips its half of the last one where that is empty.)
//
// The blocks are bound by the latency of a few K chunks where a level is small and by the FP32 pipe
// where it is large; the products run as packed pairs (fma.f32x2) over even and odd k, which both
// operands' 16-byte shared-memory loads deliver as they are.
#include "internal.h"

#include <cooperative_groups.h>

#include <cmath>

namespace cg = cooperative_groups;

namespace bem {
namespace {

constexpr int UD_THREADS = 256, UD_ROWS = 64, UD_COLS = 64, UD_STAGES = 3;
constexpr int UD_MAXF = 4;  // column tiles' worth of parents that a block looks through at most
constexpr int UD_PITCH_BYTES = 144;  // 128 bytes of one row's K chunk; 8 consecutive rows fall in different banks
template <class T>
constexpr int ud_kc() { return 128 / (int)sizeof(T); }
constexpr int UD_STAGE_BYTES = (UD_ROWS + UD_COLS) * UD_PITCH_BYTES;
constexpr int UD_RED_BYTES_PITCH = 4 * (UD_ROWS + 4);  // float; doubled for double
constexpr int UD_SMEM = UD_STAGES * UD_STAGE_BYTES;
static_assert(UD_COLS * UD_RED_BYTES_PITCH * 2 <= UD_SMEM, "the result tile reuses the stages");

// 16 bytes (V: elements) of a row, zero where !ok; rows of P elements are 16-byte aligned only when P
// is a multiple of 16 bytes' worth of elements, else element by element
template <class T, bool VEC>
__device__ __forceinline__ void ud_copy(unsigned char *dst, const T *src, int k, int kend, bool ok) {
    constexpr int V = 16 / (int)sizeof(T);
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if (VEC) {  // P and k multiples of V: the whole unit is inside or outside
        const bool in = ok && k < kend;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(in ? src + k : src), "r"(in ? 16 : 0)
                     : "memory");
    } else {
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const bool in = ok && k + v < kend;
            asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(d + v * (int)sizeof(T)),
                         "l"(in ? src + k + v : src), "n"((int)sizeof(T)), "r"(in ? (int)sizeof(T) : 0)
                         : "memory");
        }
    }
}

struct Acc32 {
    float2 v = make_float2(0.f, 0.f);
    __device__ __forceinline__ void fma4(const float4 &a, const float4 &b) {
        v = __ffma2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y), v);
        v = __ffma2_rn(make_float2(a.z, a.w), make_float2(b.z, b.w), v);
    }
    __device__ __forceinline__ float get() const { return v.x + v.y; }
};
struct Acc64 {
    double v = 0.0;
    __device__ __forceinline__ void fma4(const double2 &a, const double2 &b) {
        v = fma(a.x, b.x, v);
        v = fma(a.y, b.y, v);
    }
    __device__ __forceinline__ double get() const { return v; }
};
template <class T>
struct UdTypes {
    using Vec = float4;
    using Acc = Acc32;
};
template <>
struct UdTypes<double> {
    using Vec = double2;
    using Acc = Acc64;
};

// one staged K chunk: rows ty + 16 i (i < NI), columns tx + 16 j (j < NJ)
template <class T, int NI, int NJ>
__device__ __forceinline__ void ud_chunk(const unsigned char *st, int tx, int ty, typename UdTypes<T>::Acc (*acc)[4]) {
    using Vec = typename UdTypes<T>::Vec;
    const unsigned char *A = st + ty * UD_PITCH_BYTES, *B = st + (UD_ROWS + tx) * UD_PITCH_BYTES;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        Vec a[NI];
#pragma unroll
        for (int i = 0; i < NI; ++i) a[i] = *reinterpret_cast<const Vec *>(A + 16 * i * UD_PITCH_BYTES + q * 16);
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            const Vec b = *reinterpret_cast<const Vec *>(B + 16 * j * UD_PITCH_BYTES + q * 16);
#pragma unroll
            for (int i = 0; i < NI; ++i) acc[i][j].fma4(a[i], b);
        }
    }
}

template <class T, int NI>
__device__ __forceinline__ void ud_cols(const unsigned char *st, int tx, int ty, int nj, typename UdTypes<T>::Acc (*acc)[4]) {
    if (nj == 4) ud_chunk<T, NI, 4>(st, tx, ty, acc);
    else if (nj == 3) ud_chunk<T, NI, 3>(st, tx, ty, acc);
    else if (nj == 2) ud_chunk<T, NI, 2>(st, tx, ty, acc);
    else if (nj == 1) ud_chunk<T, NI, 1>(st, tx, ty, acc);
}
template <class T>
__device__ __forceinline__ void ud_rows(const unsigned char *st, int tx, int ty, int ni, int nj,
                                        typename UdTypes<T>::Acc (*acc)[4]) {
    if (ni == 4) ud_cols<T, 4>(st, tx, ty, nj, acc);
    else if (ni == 3) ud_cols<T, 3>(st, tx, ty, nj, acc);
    else if (ni == 2) ud_cols<T, 2>(st, tx, ty, nj, acc);
    else ud_cols<T, 1>(st, tx, ty, nj, acc);
}

// acc (zero before) = rows r0 .. r0 + rows - 1 of A times `cols` packed columns, source(c) the data of
// column c. All threads leave together, the stages free.
template <class T, bool UP, bool VEC, class F>
__device__ __forceinline__ void ud_product(int P, int r0, int rows, int cols, const T *A, F source,
                                           typename UdTypes<T>::Acc (*acc)[4]) {
    extern __shared__ __align__(16) unsigned char ud_smem[];
    constexpr int KC = ud_kc<T>(), V = 16 / (int)sizeof(T);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // a warp is 8 column x 4 row groups: its 16-byte loads read 8 (4) different rows, conflict-free
    const int tx = (warp & 1) * 8 + (lane & 7), ty = (warp >> 1) * 4 + (lane >> 3);
    const int ni = (rows + 15) / 16;
    const int nj = (cols - 8 * (warp & 1) + 15) / 16;  // column groups that this warp has a part in
    // the columns of the matrix that the rows can need
    int kbeg = 0, kend = P;
    if (UP) {
        int n = 1;
        while (n * n < r0 + rows) ++n;  // rows of degree < n
        kend = min(P, n * n);
    } else {
        int n = 0;
        while ((n + 1) * (n + 1) <= r0) ++n;  // degree of row r0
        kbeg = n * n / KC * KC;
    }
    // this thread's copies of every chunk: a 16-byte unit of the rows tid / 8 + 32 u, two of the
    // matrix and two of the sources (8 units per row, 64 + 64 rows; zeros past the last column, up to
    // the last group of 16)
    const T *src[4];
    const int row0 = tid >> 3, off = row0 * UD_PITCH_BYTES + (tid & 7) * 16, kk = kbeg + (tid & 7) * V;
    bool ok[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int row = row0 + 32 * u;
        if (u < 2) {
            ok[u] = r0 + row < P;
            src[u] = A + (ok[u] ? (size_t)(r0 + row) * P : 0);
        } else {
            ok[u] = row - UD_ROWS < cols;
            src[u] = ok[u] ? source(row - UD_ROWS) : A;
        }
    }
    const int nk = (kend - kbeg + KC - 1) / KC;
    auto load = [&](int t) {
        if (t < nk) {
            unsigned char *st = ud_smem + (t % UD_STAGES) * UD_STAGE_BYTES;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (u < 2 || row0 + 32 * (u - 2) < (cols + 15) / 16 * 16)
                    ud_copy<T, VEC>(st + off + 32 * u * UD_PITCH_BYTES, src[u], kk + t * KC, P, ok[u]);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");  // one group per chunk, empty past the end
    };
#pragma unroll
    for (int t = 0; t < UD_STAGES - 1; ++t) load(t);
    for (int t = 0; t < nk; ++t) {
        asm volatile("cp.async.wait_group %0;" ::"n"(UD_STAGES - 2) : "memory");
        __syncthreads();  // chunk t is there for everyone; the stage of chunk t - 1 is free
        load(t + UD_STAGES - 1);
        ud_rows<T>(ud_smem + (t % UD_STAGES) * UD_STAGE_BYTES, tx, ty, ni, nj, acc);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
}

// UP: Y[parent] = sum over octants (M2M); else Y[child] += the parent's share (L2L). Parents:
// global boxes pbase .. pbase + np - 1; child8[box][8]: their children by octant, -1 where empty.
// Blocks: x = 8 (tile of 64 / R parents) + octant, y = tile of result coefficients. The result tile in
// shared memory is indexed by the tile's columns (parent, right-hand side), zero where there is no child.
constexpr int UD_RP = UD_ROWS + 4;
template <class T, int R, bool UP, bool VEC>
__global__ void __launch_bounds__(UD_THREADS, sizeof(T) == 4 ? 3 : 2)
    k_updown(int P, int pbase, int np, const T *__restrict__ mats, const int32_t *__restrict__ child8, const T *X, T *Y) {
    extern __shared__ __align__(16) unsigned char ud_smem[];
    constexpr int TP = UD_COLS / R;
    __shared__ int s_child[UD_COLS], s_col[UD_COLS], s_half;
    const int oct = blockIdx.x & 7, q0 = (int)(blockIdx.x >> 3) * TP, r0 = blockIdx.y * UD_ROWS;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, rows = min(UD_ROWS, P - r0);
    bool here = false;
    int place = 0;
    if (tid < UD_COLS) {
        const int q = q0 + tid / R, ch = q < np ? child8[(int64_t)(pbase + q) * 8 + oct] : -1;
        s_child[tid] = ch;
        here = ch >= 0;
        const unsigned mask = __ballot_sync(0xffffffffu, here), below = (1u << lane) - 1u;
        place = here ? __popc(mask & below) : __popc(~mask & below);  // among the warp's
        if (tid == 31) s_half = __popc(mask);
    }
    const int cols = __syncthreads_count(here);
    // s_col: the columns that have a child, then the others
    if (tid < UD_COLS) s_col[place + (here ? (warp ? s_half : 0) : cols + (warp ? 32 - s_half : 0))] = tid;
    __syncthreads();
    T *red = reinterpret_cast<T *>(ud_smem);  // [column][UD_RP]
    if (cols || UP) {
        typename UdTypes<T>::Acc acc[4][4];
        if (cols)
            ud_product<T, UP, VEC>(P, r0, rows, cols, mats + (size_t)oct * P * P, [&](int c) {
                const int col = s_col[c];
                const int64_t box = UP ? s_child[col] : pbase + q0 + col / R;
                return X + ((size_t)box * R + col % R) * P;
            }, acc);
        const int tx = (warp & 1) * 8 + (lane & 7), ty = (warp >> 1) * 4 + (lane >> 3);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int col = s_col[tx + 16 * j];
#pragma unroll
            for (int i = 0; i < 4; ++i) red[col * UD_RP + ty + 16 * i] = acc[i][j].get();
        }
    }
    if constexpr (UP) {
        cg::cluster_group cl = cg::this_cluster();  // its 8 blocks are the octants of one tile
        cl.sync();
        for (int e = tid; e < (UD_COLS / 8) * UD_ROWS; e += UD_THREADS) {
            const int c = oct * (UD_COLS / 8) + e / UD_ROWS, row = e % UD_ROWS, q = q0 + c / R;
            if (row >= rows || q >= np) continue;
            T s = 0, comp = 0;
#pragma unroll
            for (int o = 0; o < 8; ++o) {
                const T v = cl.map_shared_rank(red, o)[c * UD_RP + row];
                const T t = s + v, bp = t - s;
                comp += (s - (t - bp)) + (v - bp);
                s = t;
            }
            Y[((size_t)(pbase + q) * R + c % R) * P + r0 + row] = s + comp;
        }
        cl.sync();  // no block leaves while another still reads its sums
    } else if (cols) {
        __syncthreads();
        for (int e = tid; e < UD_COLS * UD_ROWS; e += UD_THREADS) {
            const int c = e / UD_ROWS, row = e % UD_ROWS, ch = s_child[c];
            if (ch >= 0 && row < rows) Y[((size_t)ch * R + c % R) * P + r0 + row] += red[c * UD_RP + row];
        }
    }
}

// The same for parents of few children (in small orders the ranks of all octants cost more than they
// save where parents have about eight: M2M of 192600 points at p = 4, 17 us a product without and 21 with them):
// a tile has F x 64 / R parents (F = 2, 4), and its packed columns are all
// worked on in one pass where no octant (L2L: not the block's own) has more than 64 / R children, else in F
// passes over 64 / R parents each. The result tile is indexed by the packed columns.
template <class T, int R, bool UP, bool VEC>
__global__ void __launch_bounds__(UD_THREADS, sizeof(T) == 4 ? 3 : 2)
    k_updown_wide(int P, int pbase, int np, int F, const T *__restrict__ mats, const int32_t *__restrict__ child8,
                  const T *X, T *Y) {
    extern __shared__ __align__(16) unsigned char ud_smem[];
    constexpr int TP = UD_COLS / R, NO = UP ? 8 : 1, WARPS = UD_THREADS / 32;
    static_assert(TP * UD_MAXF <= UD_THREADS && (TP == 64 || TP == 16), "a thread per parent; whole or half warps per pass");
    __shared__ int16_t s_rank[NO][TP * UD_MAXF];  // a parent's place among its pass's columns, -1: no child
    __shared__ int s_cnt[NO][WARPS];
    __shared__ int s_par[TP], s_ch[TP];  // the block's own octant, by place: parent (in the tile) and child
    const int oct = blockIdx.x & 7, q0 = (int)(blockIdx.x >> 3) * TP * F, r0 = blockIdx.y * UD_ROWS;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, rows = min(UD_ROWS, P - r0);
    int own = -1, passes = 1;  // own: the child of this thread's parent in the block's octant
    {
        unsigned has[NO];
        int most = 0, ch[NO];
#pragma unroll
        for (int o = 0; o < NO; ++o) ch[o] = -1;
        if (tid < TP * F && q0 + tid < np) {
            const int32_t *row = child8 + (int64_t)(pbase + q0 + tid) * 8;
            own = row[oct];
            if constexpr (UP) {
                const int4 a = reinterpret_cast<const int4 *>(row)[0], b = reinterpret_cast<const int4 *>(row)[1];
                ch[0] = a.x, ch[1] = a.y, ch[2] = a.z, ch[3] = a.w;
                ch[4] = b.x, ch[5] = b.y, ch[6] = b.z, ch[7] = b.w;
            } else {
                ch[0] = own;
            }
        }
#pragma unroll
        for (int o = 0; o < NO; ++o) {
            has[o] = __ballot_sync(0xffffffffu, ch[o] >= 0);
            if (lane == 0) s_cnt[o][warp] = __popc(has[o]);
        }
        __syncthreads();
#pragma unroll
        for (int o = 0; o < NO; ++o) {
            int n = 0;
            for (int w = 0; w < WARPS; ++w) n += s_cnt[o][w];
            most = max(most, n);
        }
        if (most > TP) passes = F;  // the same in all blocks of a cluster
        if (tid < TP * F) {
#pragma unroll
            for (int o = 0; o < NO; ++o) {
                unsigned before = (1u << lane) - 1u;
                int n = 0;
                if (passes == 1) {
                    for (int w = 0; w < warp; ++w) n += s_cnt[o][w];
                } else if (TP == 64) {  // a pass is two warps
                    if (warp & 1) n = s_cnt[o][warp - 1];
                } else if (lane >= 16) {  // a pass is half a warp
                    before &= 0xffff0000u;
                }
                s_rank[o][tid] = (int16_t)((has[o] >> lane) & 1u ? n + __popc(has[o] & before) : -1);
            }
        }
    }
    const int pp = TP * F / passes;  // parents of a pass
    T *red = reinterpret_cast<T *>(ud_smem);  // [packed column][UD_RP]
    for (int p0 = 0; p0 < TP * F && q0 + p0 < np; p0 += pp) {
        const bool mine = own >= 0 && tid >= p0 && tid < p0 + pp;
        if (mine) {
            const int c = s_rank[UP ? oct : 0][tid];
            s_par[c] = tid;
            s_ch[c] = own;
        }
        const int cols = __syncthreads_count(mine) * R;
        if (cols) {
            typename UdTypes<T>::Acc acc[4][4];
            ud_product<T, UP, VEC>(P, r0, rows, cols, mats + (size_t)oct * P * P, [&](int c) {
                const int64_t box = UP ? s_ch[c / R] : pbase + q0 + s_par[c / R];
                return X + ((size_t)box * R + c % R) * P;
            }, acc);
            const int tx = (warp & 1) * 8 + (lane & 7), ty = (warp >> 1) * 4 + (lane >> 3);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) red[(tx + 16 * j) * UD_RP + ty + 16 * i] = acc[i][j].get();
        }
        if constexpr (UP) {
            cg::cluster_group cl = cg::this_cluster();
            cl.sync();
            for (int e = oct * UD_THREADS + tid; e < pp * R * UD_ROWS; e += 8 * UD_THREADS) {
                const int q = p0 + e / (UD_ROWS * R), r = e / UD_ROWS % R, row = e % UD_ROWS;
                if (row >= rows || q0 + q >= np) continue;
                T v[8], s = 0, comp = 0;
                bool first = true;
#pragma unroll
                for (int o = 0; o < 8; ++o)  // all eight in flight; an octant without the child gives column 0, left out below
                    v[o] = cl.map_shared_rank(red, o)[(max((int)s_rank[o][q], 0) * R + r) * UD_RP + row];
#pragma unroll
                for (int o = 0; o < 8; ++o) {
                    if (s_rank[o][q] < 0) continue;  // uniform in the warp
                    if (first) {
                        s = v[o];
                        first = false;
                        continue;
                    }
                    const T t = s + v[o], bp = t - s;
                    comp += (s - (t - bp)) + (v[o] - bp);
                    s = t;
                }
                Y[((size_t)(pbase + q0 + q) * R + r) * P + r0 + row] = s + comp;
            }
            cl.sync();  // no block leaves, or takes its next pass, while another still reads its sums
        } else {
            __syncthreads();
            for (int e = tid; e < cols * UD_ROWS; e += UD_THREADS) {
                const int c = e / UD_ROWS, row = e % UD_ROWS;
                if (row < rows) Y[((size_t)s_ch[c / R] * R + c % R) * P + r0 + row] += red[c * UD_RP + row];
            }
            __syncthreads();
        }
    }
}

template <class T, int R, bool UP, bool VEC>
void launch_vec(int P, int pbase, int np, int nchild, int num_sms, const T *mats, const int32_t *child8, const T *X, T *Y,
                cudaStream_t st) {
    // Wider tiles where parents have few children: the expected columns of an octant, F x 64 / 8 children per
    // parent, stay within 48 of its 64 (more would mean F passes), and four blocks per SM are left.
    // 40962 points of a sphere at depth 10, one child per parent at most levels: all columns multiplied M2M 2.65
    // and L2L 2.26 ms, those with a child 1.88 and 1.68 ms, with wider tiles 1.03 and 0.72 ms (FP32, p 14);
    // FP64, p 8: 9.2 and 7.7, 3.8 and 2.6, 2.3 and 1.7 ms. 3.21M points on 5000 spheres, 4 children per parent
    // and F = 1: 0.13 and 0.14 ms in every form.
    const int ry = div_up(P, UD_ROWS);
    int F = UD_MAXF;
    while (F > 1 && (F * (int64_t)nchild > 6 * (int64_t)np || (int64_t)8 * div_up(np, F * UD_COLS / R) * ry < 4 * num_sms)) F /= 2;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(8 * div_up(np, F * UD_COLS / R)), (unsigned)ry);
    cfg.blockDim = dim3(UD_THREADS);
    cfg.dynamicSmemBytes = UD_SMEM;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 8;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = UP ? 1 : 0;
    if (F == 1) {
        BEM_CUDA(cudaFuncSetAttribute(k_updown<T, R, UP, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, UD_SMEM));
        BEM_CUDA(cudaLaunchKernelEx(&cfg, k_updown<T, R, UP, VEC>, P, pbase, np, mats, child8, X, Y));
    } else {
        BEM_CUDA(cudaFuncSetAttribute(k_updown_wide<T, R, UP, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, UD_SMEM));
        BEM_CUDA(cudaLaunchKernelEx(&cfg, k_updown_wide<T, R, UP, VEC>, P, pbase, np, F, mats, child8, X, Y));
    }
    BEM_LAUNCH_CHECK();
}

template <class T, int R, bool UP>
void launch(int P, int pbase, int np, int nchild, int num_sms, const T *mats, const int32_t *child8, const T *X, T *Y,
            cudaStream_t st) {
    if (np <= 0) return;
    if (P % (16 / (int)sizeof(T)) == 0) launch_vec<T, R, UP, true>(P, pbase, np, nchild, num_sms, mats, child8, X, Y, st);
    else launch_vec<T, R, UP, false>(P, pbase, np, nchild, num_sms, mats, child8, X, Y, st);
}

}  // namespace

template <class T, int R>
void launch_m2m(int P, int pbase, int np, int nchild, int num_sms, const T *mats, const int32_t *child8, T *mp, cudaStream_t st) {
    launch<T, R, true>(P, pbase, np, nchild, num_sms, mats, child8, mp, mp, st);
}
template <class T, int R>
void launch_l2l(int P, int pbase, int np, int nchild, int num_sms, const T *mats, const int32_t *child8, T *lc, cudaStream_t st) {
    launch<T, R, false>(P, pbase, np, nchild, num_sms, mats, child8, lc, lc, st);
}

template void launch_m2m<float, 1>(int, int, int, int, int, const float *, const int32_t *, float *, cudaStream_t);
template void launch_m2m<float, 4>(int, int, int, int, int, const float *, const int32_t *, float *, cudaStream_t);
template void launch_m2m<double, 1>(int, int, int, int, int, const double *, const int32_t *, double *, cudaStream_t);
template void launch_m2m<double, 4>(int, int, int, int, int, const double *, const int32_t *, double *, cudaStream_t);
template void launch_l2l<float, 1>(int, int, int, int, int, const float *, const int32_t *, float *, cudaStream_t);
template void launch_l2l<float, 4>(int, int, int, int, int, const float *, const int32_t *, float *, cudaStream_t);
template void launch_l2l<double, 1>(int, int, int, int, int, const double *, const int32_t *, double *, cudaStream_t);
template void launch_l2l<double, 4>(int, int, int, int, int, const double *, const int32_t *, double *, cudaStream_t);

}  // namespace bem
