// The direct all-pairs product (Section 3.9, brute force) with the one-point quadrature kernel
// of Eq. (ns1),
//   u_i = sum_{j != i} [ q_j / |r_i - r_j| + w_j n_j.(r_i - r_j) / |r_i - r_j|^3 ],
// q_j = f s_j X_L,j / (4 pi), w_j = g s_j X_M,j / (4 pi) (Eqs. (2.13), (3.27)), plus the identity
// diagonals f L_ii X_L,i + g M_ii X_M,i where the caller asks for them.
//
// Both precisions split every receiver block's sources over the CTAs of one thread-block cluster
// and join the partial sums through distributed shared memory in rank order: no scratch in
// global memory, no second launch, a fixed summation order. Without the split a product of N
// points ran as N / 128 blocks, each walking all N sources in sequence: 6 blocks for one bubble
// of 642 vertices (0.49 ms in FP64), 106 for 13446 points (0.52 ms in FP32), on 152 SMs.
// A layer whose coefficient is zero is not evaluated (HQ: single layer, HW: double layer).
#include "internal.h"

#include <cooperative_groups.h>

namespace cg = cooperative_groups;

namespace bem {
namespace {

constexpr double kInv4Pi = 0.0795774715459476678844418816862571810;
constexpr int DIR_SPLIT = 8;  // CTAs per cluster (the portable maximum): shares of the sources

template <int R>
struct DirArgs {
    double f[R], g[R];
    const double *xL[R];
    const double *xM[R];
    double *out[R];
    const double *ld, *md;  // identity diagonals to add, or null
};

// source strengths of right-hand side r
template <int R>
__device__ __forceinline__ double dir_q(const DirArgs<R> &a, int r, double sj, int64_t j) {
    return a.f[r] != 0.0 ? a.f[r] * sj * a.xL[r][j] : 0.0;
}
template <int R>
__device__ __forceinline__ double dir_w(const DirArgs<R> &a, int r, double sj, int64_t j) {
    return a.g[r] != 0.0 ? a.g[r] * sj * a.xM[r][j] : 0.0;
}

template <int R>
__device__ __forceinline__ void dir_store(const DirArgs<R> &a, int r, int64_t i, double v) {
    if (a.ld) {
        if (a.f[r] != 0.0) v += a.f[r] * a.ld[i] * a.xL[r][i];
        if (a.g[r] != 0.0) v += a.g[r] * a.md[i] * a.xM[r][i];
    }
    a.out[r][i] = v;
}

// ------------------------------------------------------------------------------ FP64
// RECV receivers per cluster, one lane each; the sources are shared by the cluster's 8 CTAs and, tile
// by tile, by a CTA's 4 warps x 32 / RECV lane groups. FP64 runs at 2 lanes per clock and SM on this
// part, so the kernel is bound by its FP64 instructions (about 15 per pair for the single layer, 22
// for both; 5124 points, both: 0.97 ms against 0.92): what counts is that every SM has the same share.
// 32 receivers where that gives several CTAs per SM; below, 8, for four times as many equal pieces
// (642 points: 168 CTAs of 32 receivers left 136 SMs waiting for the 16 that had two).
constexpr int D64_THREADS = 128, D64_WARPS = D64_THREADS / 32, D64_TILE = 128;

template <int R, bool HQ, bool HW, int RECV>
__global__ void __launch_bounds__(D64_THREADS) k_direct64(int64_t N, const double *__restrict__ xyz,
                                                          const double *__restrict__ s, const double *__restrict__ nrm,
                                                          DirArgs<R> a) {
    __shared__ double sx[D64_TILE], sy[D64_TILE], sz[D64_TILE];
    __shared__ double snx[HW ? D64_TILE : 1], sny[HW ? D64_TILE : 1], snz[HW ? D64_TILE : 1];
    __shared__ double sq[HQ ? R : 1][D64_TILE], sw[HW ? R : 1][D64_TILE];
    constexpr int GR = 32 / RECV, PARTS = D64_WARPS * GR;  // shares of a tile's sources
    __shared__ double red[PARTS][R][RECV];
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), nr = (int)cl.num_blocks();
    const int tid = threadIdx.x, part = (tid >> 5) * GR + (tid & 31) / RECV, rl = tid & (RECV - 1);
    const int64_t i = (int64_t)(blockIdx.x / nr) * RECV + rl;
    const int64_t ii = i < N ? i : N - 1;
    const double xi = xyz[ii], yi = xyz[N + ii], zi = xyz[2 * N + ii];
    const int64_t per = (N + nr - 1) / nr, j0 = rank * per, j1 = N < j0 + per ? N : j0 + per;
    double acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = 0.0;
    for (int64_t t0 = j0; t0 < j1; t0 += D64_TILE) {
        const int ns = (int)(j1 - t0 < D64_TILE ? j1 - t0 : D64_TILE);
        __syncthreads();
        if (tid < ns) {
            const int64_t j = t0 + tid;
            sx[tid] = xyz[j];
            sy[tid] = xyz[N + j];
            sz[tid] = xyz[2 * N + j];
            if (HW) {
                snx[tid] = nrm[j];
                sny[tid] = nrm[N + j];
                snz[tid] = nrm[2 * N + j];
            }
            const double sj = s[j] * kInv4Pi;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (HQ) sq[r][tid] = dir_q(a, r, sj, j);
                if (HW) sw[r][tid] = dir_w(a, r, sj, j);
            }
        }
        __syncthreads();
        const int e0 = part * ns / PARTS, e1 = (part + 1) * ns / PARTS;
#pragma unroll 4
        for (int e = e0; e < e1; ++e) {
            const double dx = xi - sx[e], dy = yi - sy[e], dz = zi - sz[e];
            const double r2 = dx * dx + dy * dy + dz * dz;
            const double rinv = (t0 + e == i) ? 0.0 : rsqrt(r2);
            if (HQ) {
#pragma unroll
                for (int r = 0; r < R; ++r) acc[r] += sq[r][e] * rinv;
            }
            if (HW) {
                const double nd3 = (snx[e] * dx + sny[e] * dy + snz[e] * dz) * (rinv * rinv * rinv);
#pragma unroll
                for (int r = 0; r < R; ++r) acc[r] += sw[r][e] * nd3;
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) red[part][r][rl] = acc[r];
    __syncthreads();
    // the CTA's own parts in order, then this rank joins the receivers rank, rank + nr, ... of the
    // group, the ranks in order
    for (int e = tid; e < R * RECV; e += D64_THREADS) {
        double v = 0.0;
#pragma unroll
        for (int w = 0; w < PARTS; ++w) v += (&red[w][0][0])[e];
        (&red[0][0][0])[e] = v;
    }
    cl.sync();
    for (int e = tid; e < R * RECV; e += D64_THREADS) {
        const int r = e / RECV, l = e % RECV;
        const int64_t k = (int64_t)(blockIdx.x / nr) * RECV + l;
        if (l % nr != rank || k >= N) continue;
        double v = 0.0;
        for (int c = 0; c < nr; ++c) v += cl.map_shared_rank(&red[0][0][0], c)[e];
        dir_store(a, r, k, v);
    }
    cl.sync();  // no CTA leaves while another still reads its sums
}

// ------------------------------------------------------------------------------ FP32
// Coordinates as hi + lo FP32 pairs; packed two-wide arithmetic (add/mul/fma .f32x2) over two
// sources, 128 receivers per cluster. Per pair the FP32 pipe has 9
// additions for the difference of the split coordinates and 4 (single layer) to 11 (both) further
// operations, the special-function unit one reciprocal square root; a thread reads 28 (single layer) to
// 44 bytes (both) of shared memory a pair, and that pipe bounds the kernel (74 % busy at 13446 points, both
// layers, 144 us; 103 us the single layer). Sums run over at most 64 sources per packed half in FP32 and are
// merged with TwoSum; the cluster's shares are joined in FP64.
// One receiver per thread: two halve the shared-memory reads, but leave half as many warps (both layers,
// one against two: 34 / 41 us at 5000 points, 144 / 174 at 13446, 330 / 318 at 20484, 1129 / 1061 at 40000).
constexpr int D32_THREADS = 128, D32_RI = 1, D32_RECV = D32_THREADS * D32_RI, D32_TILE = 128;

template <int R, bool HQ, bool HW>
struct D32Stage {
    float4 a[D32_TILE / 2];            // -x, -x', -y, -y'   (hi)
    float4 b[D32_TILE / 2];            // -z, -z' (hi), -x, -x' (lo)
    float4 c[D32_TILE / 2];            // -y, -y', -z, -z'   (lo)
    float4 d[HW ? D32_TILE / 2 : 1];   // n_x, n_x', n_y, n_y'
    float2 e[HW ? D32_TILE / 2 : 1];   // n_z, n_z'
    float2 q[HQ ? R : 1][D32_TILE / 2];
    float2 w[HW ? R : 1][D32_TILE / 2];
};

__device__ __forceinline__ void dir_comp_add(float &s, float &c, float v) {
    const float t = s + v, bp = t - s;
    c += (s - (t - bp)) + (v - bp);
    s = t;
}

// The hardware reciprocal square root without denormal handling: r^2 below 2^-126 counts as 0 and
// gives inf. SAFE uses rsqrtf, which covers the denormals.
template <bool SAFE>
__device__ __forceinline__ float dir_rsqrt(float x) {
    if (SAFE) return rsqrtf(x);
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Sources j0 <= j < j1 against the thread's receivers base + tid + 128 k, k < D32_RI (past the end: the
// last point); (accs, accc) the compensated sums.
// The pair i = j is left out by index, in the tiles that can hold it.
template <int R, bool HQ, bool HW, bool SAFE>
__device__ __forceinline__ void dir32_sources(D32Stage<R, HQ, HW> &sg, int64_t N, int64_t j0, int64_t j1, int64_t base,
                                              const float *__restrict__ hi, const float *__restrict__ lo,
                                              const double *__restrict__ s, const double *__restrict__ nrm,
                                              const DirArgs<R> &a, float (*accs)[R], float (*accc)[R]) {
    const int tid = threadIdx.x;
    float2 XH[D32_RI], YH[D32_RI], ZH[D32_RI], XL[D32_RI], YL[D32_RI], ZL[D32_RI];
    int64_t ri[D32_RI];
#pragma unroll
    for (int k = 0; k < D32_RI; ++k) {
        ri[k] = base + tid + k * D32_THREADS;
        const int64_t i = ri[k] < N ? ri[k] : N - 1;
        XH[k] = make_float2(hi[i], hi[i]);
        YH[k] = make_float2(hi[N + i], hi[N + i]);
        ZH[k] = make_float2(hi[2 * N + i], hi[2 * N + i]);
        XL[k] = make_float2(lo[i], lo[i]);
        YL[k] = make_float2(lo[N + i], lo[N + i]);
        ZL[k] = make_float2(lo[2 * N + i], lo[2 * N + i]);
    }
    auto pairs = [&](auto selfc, int64_t t0, int np, float2 (*part)[R]) {
        constexpr bool SELF = decltype(selfc)::value;
#pragma unroll(SAFE ? 1 : 4)
        for (int p = 0; p < np; ++p) {
            const float4 A = sg.a[p], B = sg.b[p], C = sg.c[p];
#pragma unroll
            for (int k = 0; k < D32_RI; ++k) {
                const float2 dx = __fadd2_rn(__fadd2_rn(XH[k], make_float2(A.x, A.y)), __fadd2_rn(XL[k], make_float2(B.z, B.w)));
                const float2 dy = __fadd2_rn(__fadd2_rn(YH[k], make_float2(A.z, A.w)), __fadd2_rn(YL[k], make_float2(C.x, C.y)));
                const float2 dz = __fadd2_rn(__fadd2_rn(ZH[k], make_float2(B.x, B.y)), __fadd2_rn(ZL[k], make_float2(C.z, C.w)));
                float2 r2 = __fmul2_rn(dx, dx);
                r2 = __ffma2_rn(dy, dy, r2);
                r2 = __ffma2_rn(dz, dz, r2);
                float2 v = make_float2(dir_rsqrt<SAFE>(r2.x), dir_rsqrt<SAFE>(r2.y));
                if (SELF) {
                    if (ri[k] == t0 + 2 * p) v.x = 0.f;
                    if (ri[k] == t0 + 2 * p + 1) v.y = 0.f;
                }
                if (HQ) {
#pragma unroll
                    for (int r = 0; r < R; ++r) part[k][r] = __ffma2_rn(sg.q[r][p], v, part[k][r]);
                }
                if (HW) {
                    const float4 D = sg.d[p];
                    float2 nd = __fmul2_rn(make_float2(D.x, D.y), dx);
                    nd = __ffma2_rn(make_float2(D.z, D.w), dy, nd);
                    nd = __ffma2_rn(sg.e[p], dz, nd);
                    const float2 nd3 = __fmul2_rn(nd, __fmul2_rn(__fmul2_rn(v, v), v));
#pragma unroll
                    for (int r = 0; r < R; ++r) part[k][r] = __ffma2_rn(sg.w[r][p], nd3, part[k][r]);
                }
            }
        }
    };
    // this thread's source of the next tile, loaded while the current one is evaluated
    float ph[3], pl[3];
    double pn[3], ps, pq[R], pw[R];
    auto fetch = [&](int64_t t0) {
        if (t0 + tid >= j1) return;
        const int64_t j = t0 + tid;
        ps = s[j];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            ph[d] = hi[d * N + j];
            pl[d] = lo[d * N + j];
            if (HW) pn[d] = nrm[d * N + j];
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (HQ) pq[r] = a.f[r] != 0.0 ? a.xL[r][j] : 0.0;
            if (HW) pw[r] = a.g[r] != 0.0 ? a.xM[r][j] : 0.0;
        }
    };
    fetch(j0);
    for (int64_t t0 = j0; t0 < j1; t0 += D32_TILE) {
        const int ns = (int)(j1 - t0 < D32_TILE ? j1 - t0 : D32_TILE);
        __syncthreads();
        {
            const int p = tid >> 1, h = tid & 1;
            float *A = reinterpret_cast<float *>(&sg.a[p]), *B = reinterpret_cast<float *>(&sg.b[p]),
                  *C = reinterpret_cast<float *>(&sg.c[p]);
            const bool in = tid < ns;
            // past the share's end: zero strength, far away (a finite r^2)
            A[h] = in ? -ph[0] : -1e18f;
            A[2 + h] = in ? -ph[1] : -1e18f;
            B[h] = in ? -ph[2] : -1e18f;
            B[2 + h] = in ? -pl[0] : 0.f;
            C[h] = in ? -pl[1] : 0.f;
            C[2 + h] = in ? -pl[2] : 0.f;
            if (HW) {
                float *D = reinterpret_cast<float *>(&sg.d[p]), *E = reinterpret_cast<float *>(&sg.e[p]);
                D[h] = in ? (float)pn[0] : 0.f;
                D[2 + h] = in ? (float)pn[1] : 0.f;
                E[h] = in ? (float)pn[2] : 0.f;
            }
            const double sj = ps * kInv4Pi;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (HQ) reinterpret_cast<float *>(&sg.q[r][p])[h] = in && a.f[r] != 0.0 ? (float)(a.f[r] * sj * pq[r]) : 0.f;
                if (HW) reinterpret_cast<float *>(&sg.w[r][p])[h] = in && a.g[r] != 0.0 ? (float)(a.g[r] * sj * pw[r]) : 0.f;
            }
        }
        fetch(t0 + D32_TILE);
        __syncthreads();
        float2 part[D32_RI][R];
#pragma unroll
        for (int k = 0; k < D32_RI; ++k)
#pragma unroll
            for (int r = 0; r < R; ++r) part[k][r] = make_float2(0.f, 0.f);
        const int np = (ns + 1) / 2;
        if (t0 < base + D32_RECV && t0 + D32_TILE > base) pairs(std::true_type{}, t0, np, part);
        else pairs(std::false_type{}, t0, np, part);
#pragma unroll
        for (int k = 0; k < D32_RI; ++k)
#pragma unroll
            for (int r = 0; r < R; ++r) dir_comp_add(accs[k][r], accc[k][r], part[k][r].x + part[k][r].y);
    }
}

template <int R, bool HQ, bool HW>
__global__ void __launch_bounds__(D32_THREADS) k_direct32(int64_t N, const float *__restrict__ hi,
                                                          const float *__restrict__ lo, const double *__restrict__ s,
                                                          const double *__restrict__ nrm, DirArgs<R> a) {
    __shared__ D32Stage<R, HQ, HW> sg;
    __shared__ float2 red[R][D32_RECV];
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), nr = (int)cl.num_blocks();
    const int tid = threadIdx.x;
    const int64_t base = (int64_t)(blockIdx.x / nr) * D32_RECV;
    const int64_t per = (N + nr - 1) / nr, j0 = rank * per, j1 = N < j0 + per ? N : j0 + per;
    float accs[D32_RI][R], accc[D32_RI][R];
    auto clear = [&]() {
#pragma unroll
        for (int k = 0; k < D32_RI; ++k)
#pragma unroll
            for (int r = 0; r < R; ++r) accs[k][r] = accc[k][r] = 0.f;
    };
    clear();
    dir32_sources<R, HQ, HW, false>(sg, N, j0, j1, base, hi, lo, s, nrm, a, accs, accc);
    // A sum that is not finite: points closer than 1e-19, or such inputs. Threads past the last receiver
    // hold a copy of it that meets its own source at r = 0: they have no say (with it, one CTA of every
    // product of N % 128 != 0 points took its share twice: 9600 points 64 us, 9601 points 103 us).
    bool odd = false;
#pragma unroll
    for (int k = 0; k < D32_RI; ++k)
#pragma unroll
        for (int r = 0; r < R; ++r) odd = odd || (base + tid + k * D32_THREADS < N && !isfinite(accs[k][r]));
    if (__syncthreads_or(odd)) {
        clear();
        dir32_sources<R, HQ, HW, true>(sg, N, j0, j1, base, hi, lo, s, nrm, a, accs, accc);
    }
#pragma unroll
    for (int k = 0; k < D32_RI; ++k)
#pragma unroll
        for (int r = 0; r < R; ++r) red[r][tid + k * D32_THREADS] = make_float2(accs[k][r], accc[k][r]);
    cl.sync();
    // this rank joins its share of the block's receivers, the cluster's sums in rank order
    const int share = D32_RECV / nr;
    for (int e = tid; e < R * share; e += D32_THREADS) {
        const int r = e / share, l = rank * share + e % share;
        if (base + l >= N) continue;
        double v = 0.0;
        for (int c = 0; c < nr; ++c) {
            const float2 p = cl.map_shared_rank(&red[0][0], c)[r * D32_RECV + l];
            v += (double)p.x + (double)p.y;
        }
        dir_store(a, r, base + l, v);
    }
    cl.sync();  // no CTA leaves while another still reads its sums
}

// `groups` receiver blocks of DIR_SPLIT CTAs each
template <class K, class... A>
void launch_cluster(K kern, int64_t groups, int threads, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(groups * DIR_SPLIT));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = DIR_SPLIT;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    BEM_CUDA(cudaLaunchKernelEx(&cfg, kern, args...));
    BEM_LAUNCH_CHECK();
}

template <int R, bool HQ, bool HW>
void launch64(int64_t N, const double *xyz, const double *s, const double *nrm, const DirArgs<R> &a, int num_sms,
              cudaStream_t st) {
    if (div_up(N, 32) * DIR_SPLIT >= 8 * num_sms)
        launch_cluster(k_direct64<R, HQ, HW, 32>, div_up(N, 32), D64_THREADS, st, N, xyz, s, nrm, a);
    else
        launch_cluster(k_direct64<R, HQ, HW, 8>, div_up(N, 8), D64_THREADS, st, N, xyz, s, nrm, a);
}
template <int R, bool HQ, bool HW>
void launch32(int64_t N, const float *hi, const float *lo, const double *s, const double *nrm, const DirArgs<R> &a,
              cudaStream_t st) {
    launch_cluster(k_direct32<R, HQ, HW>, div_up(N, D32_RECV), D32_THREADS, st, N, hi, lo, s, nrm, a);
}

// calls fn with the layers that the coefficients ask for (R > 1: both; no layer at all: the single
// layer with zero strengths)
template <int R, class F>
void with_layers(const DirArgs<R> &a, F fn) {
    if constexpr (R > 1) {
        fn(std::true_type{}, std::true_type{});
    } else if (a.g[0] == 0.0) {
        fn(std::true_type{}, std::false_type{});
    } else if (a.f[0] == 0.0) {
        fn(std::false_type{}, std::true_type{});
    } else {
        fn(std::true_type{}, std::true_type{});
    }
}

}  // namespace

template <int R>
void launch_direct(Context &c, int prec, const double *f, const double *const *xL, const double *g,
                   const double *const *xM, double *const *out, const double *ld, const double *md) {
    DirArgs<R> a{};
    for (int r = 0; r < R; ++r) {
        a.f[r] = f[r];
        a.g[r] = g[r];
        a.xL[r] = xL[r];
        a.xM[r] = xM[r];
        a.out[r] = out[r];
    }
    a.ld = ld;
    a.md = md;
    PhaseScope ps(c, PH_DIRECT);
    with_layers<R>(a, [&](auto hq, auto hw) {
        constexpr bool HQ = decltype(hq)::value, HW = decltype(hw)::value;
        if (prec == BEM_PREC_FP64) launch64<R, HQ, HW>(c.N, c.xyz.p, c.s.p, c.nrm.p, a, c.num_sms, c.stream);
        else launch32<R, HQ, HW>(c.N, c.dir_hi.p, c.dir_lo.p, c.s.p, c.nrm.p, a, c.stream);
    });
}

void launch_direct32_raw(int64_t N, const float *hi, const float *lo, const double *s, const double *nrm, double f,
                         const double *xL, double g, const double *xM, const double *ld, const double *md, double *out,
                         cudaStream_t st) {
    DirArgs<1> a{};
    a.f[0] = f;
    a.g[0] = g;
    a.xL[0] = xL;
    a.xM[0] = xM;
    a.out[0] = out;
    a.ld = ld;
    a.md = md;
    with_layers<1>(a, [&](auto hq, auto hw) {
        launch32<1, decltype(hq)::value, decltype(hw)::value>(N, hi, lo, s, nrm, a, st);
    });
}

template void launch_direct<1>(Context &, int, const double *, const double *const *, const double *,
                               const double *const *, double *const *, const double *, const double *);
template void launch_direct<4>(Context &, int, const double *, const double *const *, const double *,
                               const double *const *, double *const *, const double *, const double *);

}  // namespace bem
