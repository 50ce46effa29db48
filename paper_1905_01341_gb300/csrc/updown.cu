// M2M and L2L of the far field (Section 3.7): multipoles of the children summed into their
// parent, M_parent = sum_o T_o M_child(o), and local expansions handed down, L_child(o) += S_o
// L_parent, one dense P x P matrix per child octant o and level.
//
// One block takes 64 columns (64 / R parents x R right-hand sides) of one octant against 64
// coefficients of the result. Degree n of the result needs only the degrees k <= n (M2M) or k >= n
// (L2L) of the source, so a block walks the columns of T_o that can be non-zero: half of the
// matrix. M2M runs as clusters of 8 blocks, one per octant, that join their sums through
// distributed shared memory in octant order (TwoSum): no row per translation in global memory, no
// reduction launch. Before, one level of a 192600-point cluster took 33 us up and 71 us down (44
// blocks of 128 x 128 outputs over all P columns, the operator loaded element by element).
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

// one staged K chunk: rows ty + 16 i (i < NI), columns tx + 16 j
template <class T, int NI>
__device__ __forceinline__ void ud_chunk(const unsigned char *st, int tx, int ty, typename UdTypes<T>::Acc (*acc)[4]) {
    using Vec = typename UdTypes<T>::Vec;
    const unsigned char *A = st + ty * UD_PITCH_BYTES, *B = st + (UD_ROWS + tx) * UD_PITCH_BYTES;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        Vec a[NI], b[4];
#pragma unroll
        for (int i = 0; i < NI; ++i) a[i] = *reinterpret_cast<const Vec *>(A + 16 * i * UD_PITCH_BYTES + q * 16);
#pragma unroll
        for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const Vec *>(B + 16 * j * UD_PITCH_BYTES + q * 16);
#pragma unroll
        for (int i = 0; i < NI; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j].fma4(a[i], b[j]);
    }
}

// UP: Y[parent] = sum over octants (M2M); else Y[child] += the parent's share (L2L). Parents:
// global boxes pbase .. pbase + np - 1; child8[box][8]: their children by octant, -1 where empty.
// Blocks: x = 8 (tile of parents) + octant, y = tile of result coefficients.
template <class T, int R, bool UP, bool VEC>
__global__ void __launch_bounds__(UD_THREADS, sizeof(T) == 4 ? 3 : 2) k_updown(int P, int pbase, int np, const T *__restrict__ mats,
                                                        const int32_t *__restrict__ child8, const T *X, T *Y) {
    extern __shared__ __align__(16) unsigned char ud_smem[];
    __shared__ int s_child[UD_COLS];
    constexpr int KC = ud_kc<T>(), TP = UD_COLS / R;
    const int oct = blockIdx.x & 7, tile = blockIdx.x >> 3, r0 = blockIdx.y * UD_ROWS;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // a warp is 8 column x 4 row groups: its 16-byte loads read 8 (4) different rows, conflict-free
    const int tx = (warp & 1) * 8 + (lane & 7), ty = (warp >> 1) * 4 + (lane >> 3);
    if (tid < UD_COLS) {
        const int q = tile * TP + tid / R;
        s_child[tid] = q < np ? child8[(int64_t)(pbase + q) * 8 + oct] : -1;
    }
    __syncthreads();
    const bool any = __syncthreads_or(tid < UD_COLS && s_child[tid] >= 0);
    const int rows = min(UD_ROWS, P - r0), ni = (rows + 15) / 16;
    typename UdTypes<T>::Acc acc[4][4];
    if (any) {
        // the columns of the matrix that rows r0 .. r0 + rows - 1 can need
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
        const T *A = mats + (size_t)oct * P * P;
        // this thread's copies of every chunk: two 16-byte units of the matrix and two of the sources
        constexpr int V = 16 / (int)sizeof(T);
        const T *src[4];
        int off[4], kk[4];
        bool ok[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int e = tid + u * UD_THREADS, row = e >> 3;  // 8 units per row, 64 + 64 rows
            kk[u] = (e & 7) * V;
            off[u] = row * UD_PITCH_BYTES + (e & 7) * 16;
            if (row < UD_ROWS) {
                ok[u] = r0 + row < P;
                src[u] = A + (ok[u] ? (size_t)(r0 + row) * P : 0);
            } else {
                const int c = row - UD_ROWS, ch = s_child[c];
                ok[u] = ch >= 0;
                const int64_t box = UP ? ch : pbase + tile * TP + c / R;
                src[u] = X + (ok[u] ? ((size_t)box * R + c % R) * P : 0);
            }
        }
        const int nk = (kend - kbeg + KC - 1) / KC;
        auto load = [&](int t) {
            if (t < nk) {
                unsigned char *st = ud_smem + (t % UD_STAGES) * UD_STAGE_BYTES;
#pragma unroll
                for (int u = 0; u < 4; ++u) ud_copy<T, VEC>(st + off[u], src[u], kbeg + t * KC + kk[u], P, ok[u]);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");  // one group per chunk, empty past the end
        };
#pragma unroll
        for (int t = 0; t < UD_STAGES - 1; ++t) load(t);
        for (int t = 0; t < nk; ++t) {
            asm volatile("cp.async.wait_group %0;" ::"n"(UD_STAGES - 2) : "memory");
            __syncthreads();  // chunk t is there for everyone; the stage of chunk t - 1 is free
            load(t + UD_STAGES - 1);
            const unsigned char *st = ud_smem + (t % UD_STAGES) * UD_STAGE_BYTES;
            if (ni == 4) ud_chunk<T, 4>(st, tx, ty, acc);
            else if (ni == 3) ud_chunk<T, 3>(st, tx, ty, acc);
            else if (ni == 2) ud_chunk<T, 2>(st, tx, ty, acc);
            else ud_chunk<T, 1>(st, tx, ty, acc);
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    constexpr int RP = UD_ROWS + 4;
    T *red = reinterpret_cast<T *>(ud_smem);  // [column][RP]
    if (any || UP) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) red[(tx + 16 * j) * RP + ty + 16 * i] = acc[i][j].get();
    }
    if constexpr (UP) {
        cg::cluster_group cl = cg::this_cluster();  // its 8 blocks are the octants of one tile
        cl.sync();
        for (int e = tid; e < (UD_COLS / 8) * UD_ROWS; e += UD_THREADS) {
            const int c = oct * (UD_COLS / 8) + e / UD_ROWS, row = e % UD_ROWS;
            const int q = tile * TP + c / R;
            if (row >= rows || q >= np) continue;
            T s = 0, comp = 0;
#pragma unroll
            for (int o = 0; o < 8; ++o) {
                const T v = cl.map_shared_rank(red, o)[c * RP + row];
                const T t = s + v, bp = t - s;
                comp += (s - (t - bp)) + (v - bp);
                s = t;
            }
            Y[((size_t)(pbase + q) * R + c % R) * P + r0 + row] = s + comp;
        }
        cl.sync();  // no block leaves while another still reads its sums
    } else {
        __syncthreads();
        if (!any) return;
        for (int e = tid; e < UD_COLS * UD_ROWS; e += UD_THREADS) {
            const int c = e / UD_ROWS, row = e % UD_ROWS, ch = s_child[c];
            if (ch >= 0 && row < rows) Y[((size_t)ch * R + c % R) * P + r0 + row] += red[c * RP + row];
        }
    }
}

template <class T, int R, bool UP, bool VEC>
void launch_vec(int P, int pbase, int np, const T *mats, const int32_t *child8, const T *X, T *Y, cudaStream_t st) {
    auto kern = k_updown<T, R, UP, VEC>;
    BEM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, UD_SMEM));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(8 * div_up(np, UD_COLS / R)), (unsigned)div_up(P, UD_ROWS));
    cfg.blockDim = dim3(UD_THREADS);
    cfg.dynamicSmemBytes = UD_SMEM;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 8;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = UP ? 1 : 0;
    BEM_CUDA(cudaLaunchKernelEx(&cfg, kern, P, pbase, np, mats, child8, X, Y));
    BEM_LAUNCH_CHECK();
}

template <class T, int R, bool UP>
void launch(int P, int pbase, int np, const T *mats, const int32_t *child8, const T *X, T *Y, cudaStream_t st) {
    if (np <= 0) return;
    if (P % (16 / (int)sizeof(T)) == 0) launch_vec<T, R, UP, true>(P, pbase, np, mats, child8, X, Y, st);
    else launch_vec<T, R, UP, false>(P, pbase, np, mats, child8, X, Y, st);
}

}  // namespace

template <class T, int R>
void launch_m2m(int P, int pbase, int np, const T *mats, const int32_t *child8, T *mp, cudaStream_t st) {
    launch<T, R, true>(P, pbase, np, mats, child8, mp, mp, st);
}
template <class T, int R>
void launch_l2l(int P, int pbase, int np, const T *mats, const int32_t *child8, T *lc, cudaStream_t st) {
    launch<T, R, false>(P, pbase, np, mats, child8, lc, lc, st);
}

template void launch_m2m<float, 1>(int, int, int, const float *, const int32_t *, float *, cudaStream_t);
template void launch_m2m<float, 4>(int, int, int, const float *, const int32_t *, float *, cudaStream_t);
template void launch_m2m<double, 1>(int, int, int, const double *, const int32_t *, double *, cudaStream_t);
template void launch_m2m<double, 4>(int, int, int, const double *, const int32_t *, double *, cudaStream_t);
template void launch_l2l<float, 1>(int, int, int, const float *, const int32_t *, float *, cudaStream_t);
template void launch_l2l<float, 4>(int, int, int, const float *, const int32_t *, float *, cudaStream_t);
template void launch_l2l<double, 1>(int, int, int, const double *, const int32_t *, double *, cudaStream_t);
template void launch_l2l<double, 4>(int, int, int, const double *, const int32_t *, double *, cudaStream_t);

}  // namespace bem
