// P2M and L2P of the FP32 far field (Section 3.7): points to multipoles at the leaves, local
// expansions to potentials at the points.
//
// Both evaluate the regular solid harmonics R_n^m (m >= 0) of a leaf's points column by column
// (fixed m, rising n). R_n^m = gamma_n^m p_n^m with the monic recurrence
//   p_m^m = (x + i y)^m,  p_n^m = z p_{n-1}^m - beta_n^m r^2 p_{n-2}^m,
//   beta_n^m = ((n-1)^2 - m^2) / ((2n-1)(2n-3)),
//   gamma_m^m = prod_{k<=m} -1/(2k),  gamma_n^m = gamma_{n-1}^m (2n-1) / ((n+m)(n-m)),
// so a step takes five packed operations (fma.f32x2, two points per lane) and the factors gamma are
// applied once per coefficient and leaf, not once per point. A leaf's block has two warps, each with
// its own points; a lane holds two points in each of one or two sets (two where a leaf has more than
// 128 points: every table value then serves both, and their recurrences are independent chains).
//
// P2M has to sum every value over the leaf's points, i.e. over the lanes: each lane writes its value
// into a row of shared memory (one row per value), and every 32 rows each lane adds up one row with
// 16-byte loads (rows 36 floats apart: neither side conflicts). The recurrence is
// linear, so for the single layer the strength is its starting value; otherwise the moments of the
// charges q, w n_x, w n_y, w n_z are formed and the dipole's gradient
//   n . grad R_n^m = n_z R_{n-1}^m - (n_x + i n_y)/2 R_{n-1}^{m-1} + (n_x - i n_y)/2 R_{n-1}^{m+1}
// is taken once per coefficient from those.
//
// Bound by instruction issue. The kernels before built every harmonic once per order group in shared
// memory (P2M, 128 threads and two barriers per 32 points) and rebuilt the divisor tables per leaf
// (both). Single layer, p = 14: P2M at 3.21M points 492 -> 242 us, at 192600 points 63 -> 41 us; L2P
// 288 -> 213 us and 62 -> 34 us; P2M of the double layer at 801000 points 399 -> 182 us. One warp per
// leaf with up to three sets per lane left the large leaves' warps running alone (54 us and 39 us at
// 192600 points).
#include "internal.h"

namespace bem {
namespace {

constexpr int PL_WARPS = 2;    // warps per leaf (block)
constexpr int PL_PITCH = 36;   // floats between the rows of the transposition buffer

struct Pair {
    float x, y;
};
struct Tables {
    Pair beta[kMaxPfmm][kMaxPfmm + 1];    // [m][n], broadcast pairs
    float gamma[kMaxPfmm][kMaxPfmm];      // [m][n]
    float scale[kMaxPfmm];                // 2^e_n of the orders above kPlainP32
};
constexpr Tables make_tables() {
    Tables t{};
    double gm = 1.0;
    for (int m = 0; m < kMaxPfmm; ++m) {
        if (m > 0) gm *= -0.5 / m;
        double g = gm;
        for (int n = m; n < kMaxPfmm; ++n) {
            if (n > m) g *= (2.0 * n - 1.0) / ((double)(n + m) * (n - m));
            t.gamma[m][n] = (float)g;
        }
        for (int n = m + 2; n <= kMaxPfmm; ++n) {
            const float b = (float)(((double)(n - 1) * (n - 1) - (double)m * m) / ((2.0 * n - 1.0) * (2.0 * n - 3.0)));
            t.beta[m][n] = {b, b};
        }
    }
    for (int n = 0; n < kMaxPfmm; ++n) {
        t.scale[n] = 1.f;
        for (int i = 0; i < expo32(kMaxPfmm, n); ++i) t.scale[n] *= 2.f;
    }
    return t;
}
__constant__ Tables kTab = make_tables();         // warp-uniform reads
__device__ const Tables kTabG = make_tables();    // reads that differ between the lanes

// position of (n, m) in the order of the columns, and the real storage index n^2 + ... decoded
__device__ __forceinline__ int col_idx(int p, int n, int m) { return m * p - m * (m - 1) / 2 + (n - m); }
__device__ __forceinline__ void coef_nm(int e, int &n, int &m, int &part) {
    n = (int)sqrtf((float)e);
    while (n * n > e) --n;
    while ((n + 1) * (n + 1) <= e) ++n;
    const int r = e - n * n;
    m = (r + 1) / 2;
    part = r > 0 && !(r & 1);  // 1: imaginary
}

// S sets of two points per lane: points base + 64 s + lane and + 32 (clamped to the last one)
template <int S>
struct Pts {
    float2 X[S], Y[S], Z[S], NR2[S], MR[S], MI[S];
    __device__ __forceinline__ void load(int lane, int base, int cnt, int64_t s0, int64_t N, const float *__restrict__ loc) {
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int64_t a = s0 + min(base + 64 * s + lane, cnt - 1), b = s0 + min(base + 64 * s + 32 + lane, cnt - 1);
            X[s] = make_float2(loc[a], loc[b]);
            Y[s] = make_float2(loc[N + a], loc[N + b]);
            Z[s] = make_float2(loc[2 * N + a], loc[2 * N + b]);
            const float2 r2 = __ffma2_rn(Z[s], Z[s], __ffma2_rn(Y[s], Y[s], __fmul2_rn(X[s], X[s])));
            NR2[s] = make_float2(-r2.x, -r2.y);
        }
    }
    // (x + i y)^m -> (x + i y)^(m + 1)
    __device__ __forceinline__ void raise() {
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const float2 r = __ffma2_rn(X[s], MR[s], __fmul2_rn(make_float2(-Y[s].x, -Y[s].y), MI[s]));
            MI[s] = __ffma2_rn(X[s], MI[s], __fmul2_rn(Y[s], MR[s]));
            MR[s] = r;
        }
    }
};

// ------------------------------------------------------------------------------ P2M
template <int R, bool HQ, bool HW>
__host__ __device__ constexpr int p2m_charges() { return R * ((HQ ? 1 : 0) + (HW ? 3 : 0)); }
// floats of moments per leaf: whole groups of 32 rows
template <int R, bool HQ, bool HW>
__host__ __device__ constexpr int p2m_moments(int p) {
    const int rs = 2 * p2m_charges<R, HQ, HW>(), spf = 32 / rs;
    return (p * (p + 1) / 2 + spf - 1) / spf * 32;
}

// moments of the points base .. base + 64 S - 1, written (first) or added to
// Ms[32 (step / spf) + (step % spf) 2 NC + 2 c + part]
template <int R, bool HQ, bool HW, int S>
__device__ __forceinline__ void p2m_pass(int p, int lane, int base, int cnt, int64_t s0, int64_t N,
                                         const float *__restrict__ loc, const float *__restrict__ nrm,
                                         const float *__restrict__ q, const float *__restrict__ w, float *buf, float *Ms,
                                         bool first) {
    constexpr int NC = p2m_charges<R, HQ, HW>(), RS = 2 * NC, SPF = 32 / RS;
    static_assert(RS * SPF == 32 || NC == 3, "rows per flush");
    Pts<S> P;
    P.load(lane, base, cnt, s0, N, loc);
    float2 wt[S][NC];
#pragma unroll
    for (int s = 0; s < S; ++s) {
        const int a = base + 64 * s + lane, b = a + 32;
        const bool va = a < cnt, vb = b < cnt;  // points past the leaf's end have zero charges
        const int64_t ia = s0 + min(a, cnt - 1), ib = s0 + min(b, cnt - 1);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            constexpr int per = (HQ ? 1 : 0) + (HW ? 3 : 0);
            if (HQ) wt[s][r * per] = make_float2(va ? q[r * N + ia] : 0.f, vb ? q[r * N + ib] : 0.f);
            if (HW) {
                const float2 ww = make_float2(va ? w[r * N + ia] : 0.f, vb ? w[r * N + ib] : 0.f);
#pragma unroll
                for (int d = 0; d < 3; ++d)
                    wt[s][r * per + (HQ ? 1 : 0) + d] = __fmul2_rn(ww, make_float2(nrm[d * N + ia], nrm[d * N + ib]));
            }
        }
        P.MR[s] = NC == 1 ? wt[s][0] : make_float2(1.f, 1.f);  // one charge: the recurrence starts from it
        P.MI[s] = make_float2(0.f, 0.f);
    }
    float *wp = buf + lane, *dst = Ms + lane;
    const float *const wend = buf + SPF * RS * PL_PITCH;
    auto flush = [&]() {
        __syncwarp();
        const float4 *row = reinterpret_cast<const float4 *>(buf + lane * PL_PITCH);
        float2 u = make_float2(0.f, 0.f), v = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float4 t = row[i];
            u = __fadd2_rn(u, make_float2(t.x, t.y));
            v = __fadd2_rn(v, make_float2(t.z, t.w));
        }
        const float2 t = __fadd2_rn(u, v);
        *dst = first ? t.x + t.y : *dst + (t.x + t.y);
        dst += 32;
        wp = buf + lane;
        __syncwarp();
    };
    for (int m = 0; m < p; ++m) {
        if (m > 0) P.raise();
        float2 cr[S], ci[S], pr[S], pi[S];
#pragma unroll
        for (int s = 0; s < S; ++s) {
            cr[s] = P.MR[s];
            ci[s] = P.MI[s];
            pr[s] = pi[s] = make_float2(0.f, 0.f);
        }
#pragma unroll 2
        for (int n = m; n < p; ++n) {
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                float2 vr, vi;
                if (NC == 1) {
                    vr = cr[0];
                    vi = ci[0];
#pragma unroll
                    for (int s = 1; s < S; ++s) {
                        vr = __fadd2_rn(vr, cr[s]);
                        vi = __fadd2_rn(vi, ci[s]);
                    }
                } else {
                    vr = __fmul2_rn(wt[0][c], cr[0]);
                    vi = __fmul2_rn(wt[0][c], ci[0]);
#pragma unroll
                    for (int s = 1; s < S; ++s) {
                        vr = __ffma2_rn(wt[s][c], cr[s], vr);
                        vi = __ffma2_rn(wt[s][c], ci[s], vi);
                    }
                }
                wp[0] = vr.x + vr.y;
                wp[PL_PITCH] = vi.x + vi.y;
                wp += 2 * PL_PITCH;
            }
            if (wp >= wend) flush();  // uniform in the warp
            const Pair b = kTab.beta[m][n + 1];
#pragma unroll
            for (int s = 0; s < S; ++s) {
                const float2 t = __fmul2_rn(make_float2(b.x, b.y), P.NR2[s]);
                const float2 nr = __ffma2_rn(P.Z[s], cr[s], __fmul2_rn(t, pr[s]));
                const float2 ni = __ffma2_rn(P.Z[s], ci[s], __fmul2_rn(t, pi[s]));
                pr[s] = cr[s];
                pi[s] = ci[s];
                cr[s] = nr;
                ci[s] = ni;
            }
        }
    }
    if (wp != buf + lane) flush();
}

template <int R, bool HQ, bool HW>
__global__ void __launch_bounds__(PL_WARPS * 32) k_p2m32(int p, const int32_t *__restrict__ bstart,
                                                         const int32_t *__restrict__ bcount, int64_t N,
                                                         const float *__restrict__ loc, const float *__restrict__ nrm,
                                                         const float *__restrict__ q, const float *__restrict__ w,
                                                         float *__restrict__ mp) {
    extern __shared__ __align__(16) float pl_smem[];
    constexpr int NC = p2m_charges<R, HQ, HW>(), RS = 2 * NC, SPF = 32 / RS, per = (HQ ? 1 : 0) + (HW ? 3 : 0);
    static_assert(PL_WARPS == 2, "the two warps' moments are added by name");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = blockIdx.x;
    const int mom = p2m_moments<R, HQ, HW>(p);
    float *buf = pl_smem + warp * (32 * PL_PITCH + mom), *Ms = buf + 32 * PL_PITCH;
    const int64_t s0 = bstart[b];
    const int cnt = bcount[b], P = p * p;
    // a warp without points (at most 64 in the leaf) has zero moments
    bool first = true;
    for (int base = 0; base < cnt; base += 64 * PL_WARPS * 2) {
        if (cnt - base > 64 * PL_WARPS) {
            const int mine = base + warp * 128;
            if (mine < cnt) {
                p2m_pass<R, HQ, HW, 2>(p, lane, mine, cnt, s0, N, loc, nrm, q, w, buf, Ms, first);
                first = false;
            }
        } else {
            const int mine = base + warp * 64;
            if (mine < cnt) {
                p2m_pass<R, HQ, HW, 1>(p, lane, mine, cnt, s0, N, loc, nrm, q, w, buf, Ms, first);
                first = false;
            }
        }
    }
    if (first)
        for (int e = lane; e < mom; e += 32) Ms[e] = 0.f;
    __syncthreads();
    const float *M0 = pl_smem + 32 * PL_PITCH, *M1 = M0 + 32 * PL_PITCH + mom;  // the two warps' moments
    // gamma times the moment of charge c, (n, m) with |m| <= n
    auto moment = [&](int c, int n, int m, float &re, float &im) {
        const int st = col_idx(p, n, m);
        const float g = kTabG.gamma[m][n];
        const int x = 32 * (st / SPF) + (st % SPF) * RS + 2 * c;
        re = g * (M0[x] + M1[x]);
        im = g * (M0[x + 1] + M1[x + 1]);
    };
    for (int e = threadIdx.x; e < P; e += PL_WARPS * 32) {
        int n, m, part;
        coef_nm(e, n, m, part);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            float re = 0.f, im = 0.f;
            if (HQ) moment(r * per, n, m, re, im);
            if (HW && n >= 1) {
                const int c = r * per + (HQ ? 1 : 0);
                float gr = 0.f, gi = 0.f, xr, xi, yr, yi;
                if (m <= n - 1) moment(c + 2, n - 1, m, gr, gi);
                if (m >= 1 || n >= 2) {  // R_{n-1}^{m-1}; R^{-1} = -conj(R^1)
                    moment(c, n - 1, m >= 1 ? m - 1 : 1, xr, xi);
                    moment(c + 1, n - 1, m >= 1 ? m - 1 : 1, yr, yi);
                    if (m == 0) {
                        xr = -xr;
                        yr = -yr;
                    }
                    gr -= 0.5f * (xr - yi);
                    gi -= 0.5f * (xi + yr);
                }
                if (m + 1 <= n - 1) {
                    moment(c, n - 1, m + 1, xr, xi);
                    moment(c + 1, n - 1, m + 1, yr, yi);
                    gr += 0.5f * (xr + yi);
                    gi += 0.5f * (xi - yr);
                }
                re += gr;
                im += gi;
            }
            if (p > kPlainP32) {
                re *= kTabG.scale[n];
                im *= kTabG.scale[n];
            }
            mp[((size_t)b * R + r) * P + e] = part ? -im : re;  // conjugate
        }
    }
}

// ------------------------------------------------------------------------------ L2P
// Points base .. base + 64 S - 1: far = sum L_n^m R_n^m, each column summed plainly, the columns
// merged with TwoSum. Ls[(n, m) in column order][R]: gamma times the coefficient as broadcast pairs
// (re, re, im, im) with the real form's factors (m = 0: 1, 0; m > 0: 2, -2).
template <int R, int S>
__device__ __forceinline__ void l2p_pass(int p, int lane, int base, int cnt, int64_t s0, int64_t N,
                                         const float *__restrict__ loc, const float4 *Ls, float *__restrict__ far) {
    Pts<S> P;
    P.load(lane, base, cnt, s0, N, loc);
    float2 as[S][R], ac[S][R];
#pragma unroll
    for (int s = 0; s < S; ++s) {
        P.MR[s] = make_float2(1.f, 1.f);
        P.MI[s] = make_float2(0.f, 0.f);
#pragma unroll
        for (int r = 0; r < R; ++r) as[s][r] = ac[s][r] = make_float2(0.f, 0.f);
    }
    const float4 *L = Ls;
    for (int m = 0; m < p; ++m) {
        if (m > 0) P.raise();
        float2 cr[S], ci[S], pr[S], pi[S], col[S][R];
#pragma unroll
        for (int s = 0; s < S; ++s) {
            cr[s] = P.MR[s];
            ci[s] = P.MI[s];
            pr[s] = pi[s] = make_float2(0.f, 0.f);
#pragma unroll
            for (int r = 0; r < R; ++r) col[s][r] = make_float2(0.f, 0.f);
        }
#pragma unroll 2
        for (int n = m; n < p; ++n, L += R) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float4 l = L[r];
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    col[s][r] = __ffma2_rn(make_float2(l.x, l.y), cr[s], col[s][r]);
                    col[s][r] = __ffma2_rn(make_float2(l.z, l.w), ci[s], col[s][r]);
                }
            }
            const Pair b = kTab.beta[m][n + 1];
#pragma unroll
            for (int s = 0; s < S; ++s) {
                const float2 t = __fmul2_rn(make_float2(b.x, b.y), P.NR2[s]);
                const float2 nr = __ffma2_rn(P.Z[s], cr[s], __fmul2_rn(t, pr[s]));
                const float2 ni = __ffma2_rn(P.Z[s], ci[s], __fmul2_rn(t, pi[s]));
                pr[s] = cr[s];
                pi[s] = ci[s];
                cr[s] = nr;
                ci[s] = ni;
            }
        }
#pragma unroll
        for (int s = 0; s < S; ++s)
#pragma unroll
            for (int r = 0; r < R; ++r) {  // packed TwoSum
                const float2 v = col[s][r], t = __fadd2_rn(as[s][r], v);
                const float2 ns = make_float2(-as[s][r].x, -as[s][r].y);
                const float2 bp = __fadd2_rn(t, ns);              // the part of v that arrived
                const float2 d = __fadd2_rn(t, make_float2(-bp.x, -bp.y));
                const float2 e0 = __fadd2_rn(as[s][r], make_float2(-d.x, -d.y));
                const float2 e1 = __fadd2_rn(v, make_float2(-bp.x, -bp.y));
                ac[s][r] = __fadd2_rn(ac[s][r], __fadd2_rn(e0, e1));
                as[s][r] = t;
            }
    }
#pragma unroll
    for (int s = 0; s < S; ++s) {
        const int a = base + 64 * s + lane, c = a + 32;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (a < cnt) far[r * N + s0 + a] = as[s][r].x + ac[s][r].x;
            if (c < cnt) far[r * N + s0 + c] = as[s][r].y + ac[s][r].y;
        }
    }
}

template <int R>
__global__ void __launch_bounds__(PL_WARPS * 32) k_l2p32(int p, const int32_t *__restrict__ bstart,
                                                         const int32_t *__restrict__ bcount, int64_t N,
                                                         const float *__restrict__ loc, const float *__restrict__ lc,
                                                         float *__restrict__ far) {
    extern __shared__ __align__(16) float pl_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = blockIdx.x;
    const int P = p * p;
    float4 *Ls = reinterpret_cast<float4 *>(pl_smem);
    for (int e = threadIdx.x; e < P; e += PL_WARPS * 32) {
        int n, m, part;
        coef_nm(e, n, m, part);
        float f = kTabG.gamma[m][n] * (m == 0 ? 1.f : (part ? -2.f : 2.f));
        if (p > kPlainP32) f *= kTabG.scale[n];
        float2 *dst = reinterpret_cast<float2 *>(Ls + (size_t)col_idx(p, n, m) * R) + part;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float v = f * lc[((size_t)b * R + r) * P + e];
            dst[2 * r] = make_float2(v, v);
            if (m == 0) dst[2 * r + 1] = make_float2(0.f, 0.f);
        }
    }
    __syncthreads();
    const int64_t s0 = bstart[b];
    const int cnt = bcount[b];
    for (int base = 0; base < cnt; base += 64 * PL_WARPS * 2) {
        if (cnt - base > 64 * PL_WARPS) {
            if (base + warp * 128 < cnt) l2p_pass<R, 2>(p, lane, base + warp * 128, cnt, s0, N, loc, Ls, far);
        } else {
            if (base + warp * 64 < cnt) l2p_pass<R, 1>(p, lane, base + warp * 64, cnt, s0, N, loc, Ls, far);
        }
    }
}

template <class K, class... A>
void launch_leaves(K kern, int nleaf, size_t smem, cudaStream_t st, A... args) {
    if (nleaf <= 0) return;
    if (smem > 48 * 1024)  // belongs to the current device: set before every launch
        BEM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    kern<<<(unsigned)nleaf, PL_WARPS * 32, smem, st>>>(args...);
    BEM_LAUNCH_CHECK();
}

}  // namespace

template <int R>
void launch_p2m32(int p, int nleaf, const int32_t *bstart, const int32_t *bcount, int64_t N, const float *loc,
                  const float *nrm, const float *q, const float *w, bool hq, bool hw, float *mp, cudaStream_t st) {
    auto go = [&](auto hqc, auto hwc) {
        constexpr bool HQ = decltype(hqc)::value, HW = decltype(hwc)::value;
        const size_t sm = (size_t)PL_WARPS * (32 * PL_PITCH + p2m_moments<R, HQ, HW>(p)) * sizeof(float);
        launch_leaves(k_p2m32<R, HQ, HW>, nleaf, sm, st, p, bstart, bcount, N, loc, nrm, q, w, mp);
    };
    if (!hw) {
        go(std::true_type{}, std::false_type{});
    } else if (!hq) {
        go(std::false_type{}, std::true_type{});
    } else {
        go(std::true_type{}, std::true_type{});
    }
}

template <int R>
void launch_l2p32(int p, int nleaf, const int32_t *bstart, const int32_t *bcount, int64_t N, const float *loc,
                  const float *lc, float *far, cudaStream_t st) {
    const size_t sm = (size_t)(p * (p + 1) / 2) * R * sizeof(float4);
    launch_leaves(k_l2p32<R>, nleaf, sm, st, p, bstart, bcount, N, loc, lc, far);
}

template void launch_p2m32<1>(int, int, const int32_t *, const int32_t *, int64_t, const float *, const float *,
                              const float *, const float *, bool, bool, float *, cudaStream_t);
template void launch_l2p32<1>(int, int, const int32_t *, const int32_t *, int64_t, const float *, const float *, float *,
                              cudaStream_t);
template void launch_l2p32<4>(int, int, const int32_t *, const int32_t *, int64_t, const float *, const float *, float *,
                              cudaStream_t);

}  // namespace bem
