// Near field of the FMM (Section 3.7, A^(sparse) X) with the one-point quadrature kernel of
// Eq. (ns1):
//   u_i += sum_{j != i} [ q_j / |r_i - r_j| + w_j n_j.(r_i - r_j) / |r_i - r_j|^3 ],
// q_j = f s_j X_L,j / (4 pi), w_j = g s_j X_M,j / (4 pi) (Eqs. (2.13), (3.27)).
//
// FP32 variants keep coordinates accurate by construction: the list kernel works in
// leaf-box units with coordinates relative to each leaf centre (integer box offsets are
// exact in FP32). Sums are formed per shared-memory tile in FP32 and merged with TwoSum
// compensation.
//
// The single-layer kernel of Eq. (ns1) is symmetric in r = |r_i - r_j|, so the FP32 single-RHS,
// single-layer products (every GMRES product) evaluate every pair of neighbour leaves A < B
// once, by A's units: one reciprocal square root feeds both q_j / r into r_i and q_i / r into
// r_j. B's shares are summed over A's receivers inside the warp, stored per (unit of A, B), and
// added to B's points by a second kernel in a fixed order: no atomics, deterministic results.
// Products with the double layer run one way: its exchanged dipole term (n_i instead of n_j)
// costs more arithmetic and registers than the shared square root saves (measured: 5.96 ms
// symmetric against 5.37 ms one way at the benchmark's size).
#include "internal.h"

#include <algorithm>
#include <type_traits>

namespace bem {
namespace {


template <class T>
__device__ __forceinline__ T rsqrt_t(T x);
// The hardware approximation (relative error below 2^-22) without the denormal handling of
// rsqrtf: r^2 is never denormal here (coordinates are in leaf-box units), and r^2 = 0 gives
// +inf, which the self-pair test replaces by 0.
template <>
__device__ __forceinline__ float rsqrt_t<float>(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
template <>
__device__ __forceinline__ double rsqrt_t<double>(double x) { return rsqrt(x); }

template <class T>
struct Comp {
    T s = 0, c = 0;
    __device__ __forceinline__ void add(T v) {
        T t = s + v;
        T bp = t - s;
        c += (s - (t - bp)) + (v - bp);
        s = t;
    }
    __device__ __forceinline__ double get() const { return (double)s + (double)c; }
};

template <class T>
struct V4 {
    using type = float4;
};
template <>
struct V4<double> {
    using type = double4;
};
template <class T>
struct V2 {
    using type = float2;
};
template <>
struct V2<double> {
    using type = double2;
};

// Near-field work is split into units of up to 64 receivers of one leaf (Tree::p2p_units) and these
// into items, ranges of the joined list of the (up to 27) neighbour leaves' sources
// (Tree::p2p_items). One warp takes an item and each lane keeps two receivers in registers, so a
// staged source feeds two pairs; a unit of fewer receivers splits each source tile over groups of
// lanes instead of leaving lanes idle. The sources are staged 32 at a time in the warp's own
// shared-memory slice as (x, y, z, q) and (n_x, n_y, n_z, w), positions
// relative to the target leaf's centre in leaf-box units. HQ / HW select the single- and
// double-layer terms, so a product with one layer only (every GMRES product) pays for that
// layer alone. The self pair has r^2 = 0 exactly (same coordinates, zero offset) and is
// skipped; only the target leaf's own tiles can hold it, so only they test r^2 (the paper's
// quadrature excludes j = i, Eq. (ns1); distinct vertices never coincide on a valid mesh).
constexpr int P2P_WARPS = 4;   // warps (work items) per block
constexpr int P2P_UNIT = 64;   // receivers per work unit
// receivers in an item's row of sums [receiver][R]: a multiple of 8 (with 64 for every item, leaves of one or
// two points took 1 KB a leaf and right-hand side in FP64)
__device__ __forceinline__ int p2p_row(int nr) { return (nr + 7) & ~7; }

template <class T, int R, bool HQ, bool HW>
struct P2PStage {
    using T4 = typename V4<T>::type;
    T4 a[32];                                  // x, y, z, q (first RHS)
    T4 b[HW ? 32 : 1];                         // n_x, n_y, n_z, w (first RHS)
    T q[(R > 1 && HQ) ? R - 1 : 1][32];        // q of the other RHS
    T w[(R > 1 && HW) ? R - 1 : 1][32];        // w of the other RHS
    int4 tab[27];                              // per neighbour: its offset, its points less its list positions
    int tend[27];                              // its end in the item's list
};

template <class T, int R, int KR, bool HQ, bool HW, bool SELF>
__device__ __forceinline__ void p2p_source(const P2PStage<T, R, HQ, HW> &sg, int s, const T *xi, const T *yi,
                                           const T *zi, T (*part)[R]) {
    using T4 = typename V4<T>::type;
    const T4 a = sg.a[s];
    T4 bb;
    if (HW) bb = sg.b[s];
#pragma unroll
    for (int k = 0; k < KR; ++k) {
        const T dx = xi[k] - a.x, dy = yi[k] - a.y, dz = zi[k] - a.z;
        const T r2 = dx * dx + dy * dy + dz * dz;
        const T rinv = SELF ? (r2 > (T)0 ? rsqrt_t<T>(r2) : (T)0) : rsqrt_t<T>(r2);
        if constexpr (R == 1 && HW) {
            // both layers as (q + w n.d / r^2) / r, the normal staged times its strength
            const T nd = bb.x * dx + bb.y * dy + bb.z * dz;
            const T ri2 = rinv * rinv;
            part[k][0] += (HQ ? a.w + nd * ri2 : nd * ri2) * rinv;
            continue;
        }
        if (HQ) {
            part[k][0] += a.w * rinv;
#pragma unroll
            for (int r = 1; r < R; ++r) part[k][r] += sg.q[r - 1][s] * rinv;
        }
        if (HW) {
            const T nd3 = (bb.x * dx + bb.y * dy + bb.z * dz) * (rinv * rinv * rinv);
            part[k][0] += bb.w * nd3;
#pragma unroll
            for (int r = 1; r < R; ++r) part[k][r] += sg.w[r - 1][s] * nd3;
        }
    }
}

// One staged tile of up to 32 sources against a lane's two receivers. The warp's lanes form G
// groups of 32/G lanes; group gi takes the sources gi * 32/G .. (gi + 1) * 32/G - 1 of the tile,
// so a unit of few receivers still keeps every lane busy (its groups' partial sums are merged
// at the end of the unit).
template <class T, int R, int G, bool HQ, bool HW, bool SELF>
__device__ __forceinline__ void p2p_tile(const P2PStage<T, R, HQ, HW> &sg, int ns, int gi, const T *xi, const T *yi,
                                         const T *zi, Comp<T> (*acc)[R]) {
    constexpr int SG = 32 / G;  // sources per group and tile
    T part[2][R];
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int r = 0; r < R; ++r) part[k][r] = (T)0;
    const int s0 = gi * SG;
    if (ns == 32) {  // full tile: fixed trip count
#pragma unroll 8
        for (int t = 0; t < SG; ++t) p2p_source<T, R, 2, HQ, HW, SELF>(sg, s0 + t, xi, yi, zi, part);
    } else {
        const int e = min(SG, ns - s0);  // may be <= 0 for the groups past the tile's end
#pragma unroll 2
        for (int t = 0; t < e; ++t) p2p_source<T, R, 2, HQ, HW, SELF>(sg, s0 + t, xi, yi, zi, part);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int r = 0; r < R; ++r) acc[k][r].add(part[k][r]);
}

// One FP64 work item (see the packed form below: up to 64 receivers of one leaf and a range of its list
// of neighbour sources) by one warp, its lanes split into G groups (G = 1 for 33..64 receivers, 2 for
// 17..32, 4 for 9..16, 8 for 1..8): lane = gi * (32/G) + rs holds the receivers rs and rs + 32/G and takes
// group gi's share of every source tile. Bound by the FP64 pipe (two lanes per clock and SM). With a warp
// per unit and all its neighbours, 784 warps at 40962 points, a part of the SMs ran two rounds and the SMs
// were active 59 % of the kernel's time: 5.62 -> 3.32 ms (both layers of 40962 points, p 16;
// with the layers taken as one factor of 1/r, two operations a pair fewer, 6.27 -> 5.62 before).
template <class T, int R, int G, bool HQ, bool HW>
__device__ __forceinline__ void p2p_item_g(P2PStage<T, R, HQ, HW> &sg, int lane, int4 it, int nr,
                                           const int32_t *__restrict__ bstart, const int32_t *__restrict__ bcount,
                                           const int32_t *__restrict__ nbr, const int32_t *__restrict__ ncnt,
                                           const int8_t *__restrict__ nd, int64_t N, const T *__restrict__ loc,
                                           const T *__restrict__ nrm, const T *__restrict__ q, const T *__restrict__ w,
                                           double2 *__restrict__ fwd, const int32_t *__restrict__ row) {
    constexpr int LG = 32 / G;  // lanes per group
    const int rs = lane & (LG - 1), gi = lane / LG;
    const int b = it.x, r0 = it.y;
    const int s0 = bstart[b];
    T xi[2], yi[2], zi[2];
    Comp<T> acc[2][R];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int li = rs + k * LG;
        const int64_t i = s0 + r0 + (li < nr ? li : 0);
        xi[k] = loc[i];
        yi[k] = loc[N + i];
        zi[k] = loc[2 * N + i];
    }
    auto stage = [&](int64_t j, int ox, int oy, int oz) {
        sg.a[lane] = typename V4<T>::type{loc[j] + (T)ox, loc[N + j] + (T)oy, loc[2 * N + j] + (T)oz, HQ ? q[j] : (T)0};
        if (HW) {
            const T wn = R == 1 ? w[j] : (T)1;
            sg.b[lane] = typename V4<T>::type{nrm[j] * wn, nrm[N + j] * wn, nrm[2 * N + j] * wn, w[j]};
        }
#pragma unroll
        for (int r = 1; r < R; ++r) {
            if (HQ) sg.q[r - 1][lane] = q[r * N + j];
            if (HW) sg.w[r - 1][lane] = w[r * N + j];
        }
    };
    if (it.z < 0) {  // the unit's first item: its own leaf, then the list from 0
        const int fc = bcount[b];
        for (int t0 = 0; t0 < fc; t0 += 32) {
            if (t0 + lane < fc) stage((int64_t)s0 + t0 + lane, 0, 0, 0);
            __syncwarp();
            p2p_tile<T, R, G, HQ, HW, true>(sg, min(32, fc - t0), gi, xi, yi, zi, acc);
            __syncwarp();
        }
    }
    const int lbeg = max(it.z, 0), lend = it.w;
    if (lbeg < lend) {
        // the list: per neighbour its end position and the shift from positions to points
        const int nn = ncnt[b];
        int cnt = 0, st = 0;
        int4 tb = make_int4(0, 0, 0, 0);
        if (lane < nn) {
            const int f = nbr[b * 27 + lane];
            if (f != b) cnt = bcount[f];
            st = bstart[f];
            tb.x = nd[(b * 27 + lane) * 4];
            tb.y = nd[(b * 27 + lane) * 4 + 1];
            tb.z = nd[(b * 27 + lane) * 4 + 2];
        }
        int end = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += v;
        }
        if (lane < 27) {
            tb.w = st - (end - cnt);
            sg.tab[lane] = tb;
            sg.tend[lane] = end;
        }
        __syncwarp();
        int k = 0, kend = sg.tend[0];
        int4 cur = sg.tab[0];
        for (int t0 = lbeg; t0 < lend; t0 += 32) {
            const int s = t0 + lane;
            if (s < lend) {
                if (s >= kend) {
                    do kend = sg.tend[++k];
                    while (s >= kend);
                    cur = sg.tab[k];
                }
                stage((int64_t)cur.w + s, cur.x, cur.y, cur.z);
            }
            __syncwarp();
            p2p_tile<T, R, G, HQ, HW, false>(sg, min(32, lend - t0), gi, xi, yi, zi, acc);
            __syncwarp();
        }
    }
    // merge the groups' partial sums into group 0 (a fixed butterfly: deterministic)
#pragma unroll
    for (int off = LG; off < 32; off <<= 1)
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const T os = __shfl_xor_sync(0xffffffffu, acc[k][r].s, off);
                const T oc = __shfl_xor_sync(0xffffffffu, acc[k][r].c, off);
                acc[k][r].add(os);
                acc[k][r].c += oc;
            }
    if (gi == 0) {
        fwd += (int64_t)*row * (8 * R);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int li = rs + k * LG;
            if (li < nr) {
#pragma unroll
                for (int r = 0; r < R; ++r) fwd[li * R + r] = make_double2(acc[k][r].s, acc[k][r].c);
            }
        }
    }
}

// FP32 form with packed two-wide arithmetic (add/mul/fma .f32x2: one instruction for two
// lanes' worth of FP32 work): each lane takes its two receivers against two sources at a time. A
// staged tile holds 16 source pairs, each as (-x, -x', -y, -y'), (-z, -z', q, q') (and
// (n_x, n_x', n_y, n_y'), (n_z, n_z', w, w') for the double layer); a receiver's coordinate is a
// broadcast pair, so x_i - x_j is one packed add of the negated source coordinate (exactly the
// scalar difference) and r^2, the sums and the double layer's n.(r_i - r_j) / r^3 are packed
// products; the reciprocal square roots stay scalar. Lanes past a tile's end stage a source of zero
// strength far outside the leaf's neighbourhood (finite r^2), so a partial tile runs whole pairs.
//
// Work items (Tree::p2p_items): the neighbour leaves that a unit evaluates, one after another in its
// neighbour list, count as one list of sources; an item is a unit and a range of that list, of about
// the same length for all items (the unit's own leaf belongs to its first item). Tiles run across
// the borders of the leaves (every staged source gets its own leaf's offset), so only an item's last
// tile is partial: with a tile per 32 sources of each leaf, about a sixth of the pair slots were
// empty at 90 to 130 points a leaf. And a small product has enough items of equal size to fill the
// chip: one warp per unit left the SMs active 59 % of the kernel's time at 192600 points. An item's
// sums go to its own row of `fwd`, joined per point by k_p2p_gather. Symmetric single-layer kernel
// with its gather, 192600 points: 207 -> 124 us; 3.21M points: 2.51 -> 2.35 ms.
template <int R, bool HQ, bool HW>
struct P2PStageX2 {
    float4 a[16];               // -x, -x', -y, -y'
    float4 b[16];               // -z, -z', q, q' (first RHS)
    float4 c[HW ? 16 : 1];      // n_x, n_x', n_y, n_y'
    float4 d[HW ? 16 : 1];      // n_z, n_z', w, w' (first RHS)
    float q[(R > 1 && HQ) ? R - 1 : 1][32];
    float w[(R > 1 && HW) ? R - 1 : 1][32];
    float4 tab[27];  // per neighbour: box offset x, y, z and (as an integer) first point - list position
    int32_t tend[27];  // per neighbour: end in the item's source list
};
template <int R, bool HQ, bool HW, bool SYM>
struct P2PStageSym : P2PStageX2<R, HQ, HW> {
    float tr[SYM ? 32 : 1][20];  // symmetric form: per-lane rows of the sources' shares, transposed
};

template <bool SELF>
__device__ __forceinline__ float2 rsqrt_x2(float2 r2) {
    float2 ri;
    ri.x = SELF ? (r2.x > 0.f ? rsqrt_t<float>(r2.x) : 0.f) : rsqrt_t<float>(r2.x);
    ri.y = SELF ? (r2.y > 0.f ? rsqrt_t<float>(r2.y) : 0.f) : rsqrt_t<float>(r2.y);
    return ri;
}

// The receivers' own strengths for the symmetric form (broadcast pairs, zero for lanes past the
// unit's end).
struct RecvX2 {
    float2 q[2];
};

// BACK (single layer): also accumulate the pair's share for the two sources, the sum over this
// lane's receivers of q_i / r
template <int R, bool HQ, bool HW, bool SELF, bool BACK = false>
__device__ __forceinline__ void p2p_source_x2(const P2PStageX2<R, HQ, HW> &sg, int p, const float2 *X,
                                              const float2 *Y, const float2 *Z, float2 (*part)[R],
                                              const RecvX2 *rv = nullptr, float2 *bk = nullptr) {
    const float4 A = sg.a[p], B = sg.b[p];
    const float2 mx = make_float2(A.x, A.y), my = make_float2(A.z, A.w), mz = make_float2(B.x, B.y);
    float4 C, D;
    if (HW) {
        C = sg.c[p];
        D = sg.d[p];
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float2 dx = __fadd2_rn(X[k], mx), dy = __fadd2_rn(Y[k], my), dz = __fadd2_rn(Z[k], mz);
        float2 r2 = __fmul2_rn(dx, dx);
        r2 = __ffma2_rn(dy, dy, r2);
        r2 = __ffma2_rn(dz, dz, r2);
        const float2 ri = rsqrt_x2<SELF>(r2);
        if (HQ) {
            part[k][0] = __ffma2_rn(make_float2(B.z, B.w), ri, part[k][0]);
#pragma unroll
            for (int r = 1; r < R; ++r)
                part[k][r] = __ffma2_rn(*reinterpret_cast<const float2 *>(&sg.q[r - 1][2 * p]), ri, part[k][r]);
            if (BACK) *bk = __ffma2_rn(rv->q[k], ri, *bk);
        }
        if (HW) {
            float2 nd = __fmul2_rn(make_float2(C.x, C.y), dx);
            nd = __ffma2_rn(make_float2(C.z, C.w), dy, nd);
            nd = __ffma2_rn(make_float2(D.x, D.y), dz, nd);
            const float2 nd3 = __fmul2_rn(nd, __fmul2_rn(__fmul2_rn(ri, ri), ri));
            part[k][0] = __ffma2_rn(make_float2(D.z, D.w), nd3, part[k][0]);
#pragma unroll
            for (int r = 1; r < R; ++r)
                part[k][r] = __ffma2_rn(*reinterpret_cast<const float2 *>(&sg.w[r - 1][2 * p]), nd3, part[k][r]);
        }
    }
}

// A staged tile in the symmetric form (one RHS): the forward sums and, per batch of up to 16
// sources of a group, each source's share summed over the unit's receivers (every group holds all
// of them), written to back[s] for the tile's sources s < ns. The sum over lanes goes through
// shared memory: every lane stores its row of the batch's values. One group of 32 lanes: lane
// (rg, cq) adds the rows rg + 8 i of the four columns of quad cq with 16-byte loads (the quads of a
// row rotate with the row, so neither the stores nor the loads conflict), then three exchanges join
// the row groups. More groups: lane rs adds up column rs over its group's rows, the groups' rows
// skewed so that their columns fall in different banks. The order of every sum is fixed, so the
// result is deterministic.
template <int G, bool HQ, bool HW>
__device__ __forceinline__ void p2p_tile_x2_sym(P2PStageSym<1, HQ, HW, true> &sg, int ns, int gi, int lane,
                                                const float2 *X, const float2 *Y, const float2 *Z, const RecvX2 &rv,
                                                Comp<float> (*acc)[1], float *__restrict__ back) {
    constexpr int SP = 16 / G, LG = 32 / G;
    constexpr int HP = SP < 8 ? SP : 8;  // source pairs per batch
    constexpr int NV = 2 * HP;           // sources per batch: values per lane
    constexpr int SK = G == 2 ? 4 : (G == 4 ? 2 : 1);  // row skew per group (see above)
    const int rs = lane & (LG - 1);
    float2 part[2][1];
    part[0][0] = part[1][0] = make_float2(0.f, 0.f);
    const int p0 = gi * SP;
#pragma unroll
    for (int h0 = 0; h0 < SP; h0 += HP) {
        float2 bk[HP];
#pragma unroll
        for (int t = 0; t < HP; ++t) bk[t] = make_float2(0.f, 0.f);
#pragma unroll
        for (int t = 0; t < HP; ++t) p2p_source_x2<1, HQ, HW, false, true>(sg, p0 + h0 + t, X, Y, Z, part, &rv, &bk[t]);
        if constexpr (G == 1) {
            float4 *tr = reinterpret_cast<float4 *>(&sg.tr[0][0]);  // [32 rows][4 quads]
            const int sw = (lane >> 1) & 3;
#pragma unroll
            for (int c4 = 0; c4 < 4; ++c4)
                tr[lane * 4 + (c4 ^ sw)] = make_float4(bk[2 * c4].x, bk[2 * c4].y, bk[2 * c4 + 1].x, bk[2 * c4 + 1].y);
            __syncwarp();
            const int cq = lane & 3, rg = lane >> 2;
            float2 u = make_float2(0.f, 0.f), v = make_float2(0.f, 0.f);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int row = rg + 8 * i;
                const float4 t4 = tr[row * 4 + (cq ^ ((row >> 1) & 3))];
                u = __fadd2_rn(u, make_float2(t4.x, t4.y));
                v = __fadd2_rn(v, make_float2(t4.z, t4.w));
            }
            // join the row groups (lane bits 4, 3, 2); bits 4 and 3 choose the column kept
            const bool b4 = lane & 16, b3 = lane & 8;
            const float s0 = b4 ? u.x : v.x, s1 = b4 ? u.y : v.y;
            const float k0 = (b4 ? v.x : u.x) + __shfl_xor_sync(0xffffffffu, s0, 16);
            const float k1 = (b4 ? v.y : u.y) + __shfl_xor_sync(0xffffffffu, s1, 16);
            float tot = (b3 ? k1 : k0) + __shfl_xor_sync(0xffffffffu, b3 ? k0 : k1, 8);
            tot += __shfl_xor_sync(0xffffffffu, tot, 4);
            __syncwarp();  // the next batch rewrites the rows
            const int src = 2 * h0 + 4 * cq + (b4 ? 2 : 0) + (b3 ? 1 : 0);
            if (!(lane & 4) && src < ns) back[src] = tot;
        } else {
            float4 *row = reinterpret_cast<float4 *>(&sg.tr[lane][0]);
#pragma unroll
            for (int c4 = 0; c4 < NV / 4; ++c4)
                row[c4] = make_float4(bk[2 * c4].x, bk[2 * c4].y, bk[2 * c4 + 1].x, bk[2 * c4 + 1].y);
            __syncwarp();
            float tot = 0.f;
            const int sk = G == 8 ? (gi >> 1) : SK * gi;
#pragma unroll
            for (int r = 0; r < LG; ++r) tot += sg.tr[gi * LG + ((r + sk) & (LG - 1))][rs];
            __syncwarp();  // the next batch rewrites the rows
            const int src = 2 * (p0 + h0) + (rs & (NV - 1));
            if (rs < NV && src < ns) back[src] = tot;
        }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) acc[k][0].add(part[k][0].x + part[k][0].y);
}

// one staged tile (16 source pairs, those past the tile's end of zero strength) against a lane's
// two receivers; group gi of G takes the pairs gi * 16/G .. (gi + 1) * 16/G - 1
template <int R, int G, bool HQ, bool HW, bool SELF>
__device__ __forceinline__ void p2p_tile_x2(const P2PStageX2<R, HQ, HW> &sg, int gi, const float2 *X,
                                            const float2 *Y, const float2 *Z, Comp<float> (*acc)[R]) {
    constexpr int SP = 16 / G;  // source pairs per group and tile
    float2 part[2][R];
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int r = 0; r < R; ++r) part[k][r] = make_float2(0.f, 0.f);
    const int p0 = gi * SP;
#pragma unroll(SELF ? 2 : 4)
    for (int t = 0; t < SP; ++t) p2p_source_x2<R, HQ, HW, SELF>(sg, p0 + t, X, Y, Z, part);
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int r = 0; r < R; ++r) acc[k][r].add(part[k][r].x + part[k][r].y);
}

// lane `lane` stages source j (in: the slot holds a source), displaced by the box offset o
template <int R, bool HQ, bool HW>
__device__ __forceinline__ void p2p_stage_x2(P2PStageX2<R, HQ, HW> &sg, int lane, bool in, int64_t j, float ox, float oy,
                                             float oz, int64_t N, const float *__restrict__ loc,
                                             const float *__restrict__ nrm, const float *__restrict__ q,
                                             const float *__restrict__ w) {
    const int sp = lane >> 1, h = lane & 1;
    float *a = reinterpret_cast<float *>(&sg.a[sp]), *b = reinterpret_cast<float *>(&sg.b[sp]);
    if (in) {
        a[h] = -(loc[j] + ox);
        a[2 + h] = -(loc[N + j] + oy);
        b[h] = -(loc[2 * N + j] + oz);
        b[2 + h] = HQ ? q[j] : 0.f;
        if (HW) {
            float *c = reinterpret_cast<float *>(&sg.c[sp]), *d = reinterpret_cast<float *>(&sg.d[sp]);
            c[h] = nrm[j];
            c[2 + h] = nrm[N + j];
            d[h] = nrm[2 * N + j];
            d[2 + h] = w[j];
        }
#pragma unroll
        for (int r = 1; r < R; ++r) {
            if (HQ) sg.q[r - 1][lane] = q[r * N + j];
            if (HW) sg.w[r - 1][lane] = w[r * N + j];
        }
    } else {  // zero strength, 1e4 leaf widths away
        a[h] = -1e4f;
        a[2 + h] = -1e4f;
        b[h] = -1e4f;
        b[2 + h] = 0.f;
        if (HW) {
            float *c = reinterpret_cast<float *>(&sg.c[sp]), *d = reinterpret_cast<float *>(&sg.d[sp]);
            c[h] = 0.f;
            c[2 + h] = 0.f;
            d[h] = 0.f;
            d[2 + h] = 0.f;
        }
#pragma unroll
        for (int r = 1; r < R; ++r) {
            if (HQ) sg.q[r - 1][lane] = 0.f;
            if (HW) sg.w[r - 1][lane] = 0.f;
        }
    }
}

// Symmetric form (SYM, one RHS): the list holds the neighbour leaves f > b; their tiles also
// produce the shares of the sources, written at back + the unit's region + list position; a
// neighbour f < b is left out (f's units evaluate the pair and b's points get their shares by the
// gather). Otherwise the list holds all neighbours. The leaf's own tiles are evaluated one way,
// all pairs i != j.
struct BackArgs {
    float *back;
    const int32_t *S;
    const int64_t *base;
};

// One item by one warp, its lanes split into G groups (G = 1 for 33..64 receivers, 2 for 17..32, 4
// for 9..16, 8 for 1..8): lane = gi * (32/G) + rs holds the receivers rs and rs + 32/G and takes
// group gi's share of every source tile.
template <int R, int G, bool HQ, bool HW, bool SYM>
__device__ __forceinline__ void p2p_item_gx2(P2PStageSym<R, HQ, HW, SYM> &sg, int lane, int4 it, int nr,
                                             const int32_t *__restrict__ bstart, const int32_t *__restrict__ bcount,
                                             const int32_t *__restrict__ nbr, const int32_t *__restrict__ ncnt,
                                             const int8_t *__restrict__ nd, int64_t N, const float *__restrict__ loc,
                                             const float *__restrict__ nrm, const float *__restrict__ q,
                                             const float *__restrict__ w, float2 *__restrict__ fwd, const int32_t *__restrict__ row,
                                             BackArgs ba) {
    constexpr int LG = 32 / G;
    const int rs = lane & (LG - 1), gi = lane / LG;
    const int b = it.x, r0 = it.y;
    const int s0 = bstart[b];
    float2 X[2], Y[2], Z[2];
    RecvX2 rv;
    Comp<float> acc[2][R];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int li = rs + k * LG;
        const bool valid = li < nr;
        const int64_t i = s0 + r0 + (valid ? li : 0);
        const float x = loc[i], y = loc[N + i], z = loc[2 * N + i];
        X[k] = make_float2(x, x);
        Y[k] = make_float2(y, y);
        Z[k] = make_float2(z, z);
        if (SYM) {
            const float qi = valid ? q[i] : 0.f;
            rv.q[k] = make_float2(qi, qi);
        }
    }
    if (it.z < 0) {  // the unit's first item: its own leaf, then the list from 0
        const int fc = bcount[b];
        for (int t0 = 0; t0 < fc; t0 += 32) {
            p2p_stage_x2<R, HQ, HW>(sg, lane, t0 + lane < fc, (int64_t)s0 + t0 + lane, 0.f, 0.f, 0.f, N, loc, nrm, q, w);
            __syncwarp();
            p2p_tile_x2<R, G, HQ, HW, true>(sg, gi, X, Y, Z, acc);
            __syncwarp();
        }
    }
    const int lbeg = max(it.z, 0), lend = it.w;
    if (lbeg < lend) {
        // the list: per neighbour its end position and the shift from positions to points
        const int nn = ncnt[b];
        int cnt = 0, st = 0;
        float4 tb = make_float4(0.f, 0.f, 0.f, 0.f);
        if (lane < nn) {
            const int f = nbr[b * 27 + lane];
            if (SYM ? f > b : f != b) cnt = bcount[f];
            st = bstart[f];
            tb.x = (float)nd[(b * 27 + lane) * 4];
            tb.y = (float)nd[(b * 27 + lane) * 4 + 1];
            tb.z = (float)nd[(b * 27 + lane) * 4 + 2];
        }
        int end = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += v;
        }
        if (lane < 27) {
            tb.w = __int_as_float(st - (end - cnt));
            sg.tab[lane] = tb;
            sg.tend[lane] = end;
        }
        __syncwarp();
        float *back_unit = nullptr;
        if (SYM) back_unit = ba.back + ba.base[b] + (int64_t)(r0 / P2P_UNIT) * ba.S[b];
        int k = 0, kend = sg.tend[0];
        float4 cur = sg.tab[0];
        for (int t0 = lbeg; t0 < lend; t0 += 32) {
            const int s = t0 + lane;
            const bool in = s < lend;
            if (in && s >= kend) {
                do kend = sg.tend[++k];
                while (s >= kend);
                cur = sg.tab[k];
            }
            p2p_stage_x2<R, HQ, HW>(sg, lane, in, (int64_t)__float_as_int(cur.w) + s, cur.x, cur.y, cur.z, N, loc, nrm, q,
                                    w);
            __syncwarp();
            if constexpr (SYM) p2p_tile_x2_sym<G, HQ, HW>(sg, min(32, lend - t0), gi, lane, X, Y, Z, rv, acc, back_unit + t0);
            else p2p_tile_x2<R, G, HQ, HW, false>(sg, gi, X, Y, Z, acc);
            __syncwarp();
        }
    }
    // merge the groups' partial sums into group 0 (a fixed butterfly: deterministic)
#pragma unroll
    for (int off = LG; off < 32; off <<= 1)
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float os = __shfl_xor_sync(0xffffffffu, acc[k][r].s, off);
                const float oc = __shfl_xor_sync(0xffffffffu, acc[k][r].c, off);
                acc[k][r].add(os);
                acc[k][r].c += oc;
            }
    if (gi == 0) {
        if (!SYM) fwd += (int64_t)*row * (8 * R);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int li = rs + k * LG;
            if (li < nr) {
#pragma unroll
                for (int r = 0; r < R; ++r) fwd[li * R + r] = make_float2(acc[k][r].s, acc[k][r].c);
            }
        }
    }
}

// Each warp takes the items blockIdx.x * P2P_WARPS + warp, then every gridDim.x * P2P_WARPS further:
// one item per warp when the grid covers all items, or a persistent grid of a fixed number of
// blocks per SM (leaving room on every SM for the far-field kernels that run concurrently on the
// other stream). Every item writes its own row, so the result does not depend on the grid.
template <int R, bool HQ, bool HW, bool SYM>
__global__ void __launch_bounds__(P2P_WARPS * 32, SYM ? 6 : (R == 1 ? 5 : 4)) k_p2p_items_x2(
    const int4 *__restrict__ items, const int32_t *__restrict__ irow, int64_t nitems, const int32_t *__restrict__ bstart,
    const int32_t *__restrict__ bcount, const int32_t *__restrict__ nbr, const int32_t *__restrict__ ncnt,
    const int8_t *__restrict__ nd, int64_t N, const float *__restrict__ loc, const float *__restrict__ nrm,
    const float *__restrict__ q, const float *__restrict__ w, float2 *__restrict__ fwd, BackArgs ba) {
    static_assert(!SYM || (R == 1 && !HW), "the symmetric form is single-RHS, single-layer");
    __shared__ P2PStageSym<R, HQ, HW, SYM> stage[P2P_WARPS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * P2P_WARPS;
    auto &sg = stage[warp];
    for (int64_t u = (int64_t)blockIdx.x * P2P_WARPS + warp; u < nitems; u += stride) {
        const int4 it = items[u];
        const int nr = min(P2P_UNIT, bcount[it.x] - it.y);  // uniform in the warp
        // where the row lies: the symmetric form looks it up first, the others, short of registers, at the end
        // (the other way round costs each about 1 %)
        float2 *f = SYM ? fwd + (int64_t)irow[u] * (8 * R) : fwd;
        if (nr > 32) p2p_item_gx2<R, 1, HQ, HW, SYM>(sg, lane, it, nr, bstart, bcount, nbr, ncnt, nd, N, loc, nrm, q, w, f, irow + u, ba);
        else if (nr > 16) p2p_item_gx2<R, 2, HQ, HW, SYM>(sg, lane, it, nr, bstart, bcount, nbr, ncnt, nd, N, loc, nrm, q, w, f, irow + u, ba);
        else if (nr > 8) p2p_item_gx2<R, 4, HQ, HW, SYM>(sg, lane, it, nr, bstart, bcount, nbr, ncnt, nd, N, loc, nrm, q, w, f, irow + u, ba);
        else p2p_item_gx2<R, 8, HQ, HW, SYM>(sg, lane, it, nr, bstart, bcount, nbr, ncnt, nd, N, loc, nrm, q, w, f, irow + u, ba);
    }
}

// Second pass: one warp per work unit (up to 64 points of leaf B, two per lane); every point adds
// its unit's items in order and, in the symmetric form, the shares that the units of B's neighbours
// A < B wrote for it, neighbour by neighbour in B's list, unit by unit, in a compensated FP32 sum
// (TwoSum; FP64 arithmetic is slow on this part). Lane k first looks up neighbour k's region;
// shuffles broadcast it.
constexpr int GATHER_WARPS = 8;
template <class T, int R, bool SYM>
__global__ void __launch_bounds__(GATHER_WARPS * 32) k_p2p_gather(
    const int2 *__restrict__ units, int64_t nunits, const int32_t *__restrict__ ioff, const int32_t *__restrict__ irow,
    const typename V2<T>::type *__restrict__ fwd,
    const int32_t *__restrict__ bstart, const int32_t *__restrict__ bcount, const int32_t *__restrict__ nbr,
    const int32_t *__restrict__ ncnt, const int32_t *__restrict__ gofs, const int32_t *__restrict__ ucnt,
    const int32_t *__restrict__ S, const int64_t *__restrict__ base, const float *__restrict__ back, int64_t N,
    double *__restrict__ out) {
    const int64_t uw = (int64_t)blockIdx.x * GATHER_WARPS + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (uw >= nunits) return;  // uniform in the warp
    const int2 un = units[uw];
    const int b = un.x, r0 = un.y;
    const int nr = min(P2P_UNIT, bcount[b] - r0);
    const bool v0 = lane < nr, v1 = lane + 32 < nr;
    const int64_t i0 = (int64_t)bstart[b] + r0 + lane;
    using T2 = typename V2<T>::type;
    Comp<T> a0[R], a1[R];
    const int row = p2p_row(nr) * R;  // the unit's items lie one after another
    const T2 *f = fwd + (int64_t)irow[ioff[uw]] * (8 * R) + lane * R;
    for (int i = ioff[uw], e = ioff[uw + 1]; i < e; ++i, f += row) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (v0) {
                const T2 x = f[r];
                a0[r].add(x.x);
                a0[r].c += x.y;
            }
            if (v1) {
                const T2 x = f[32 * R + r];
                a1[r].add(x.x);
                a1[r].c += x.y;
            }
        }
    }
    if constexpr (SYM) {
        const int nn = ncnt[b];
        int64_t my_off = 0;
        int my_S = 0, my_n = 0;
        if (lane < nn) {
            const int g = gofs[b * 27 + lane];
            if (g >= 0) {
                const int a = nbr[b * 27 + lane];
                my_off = base[a] + g;
                my_S = S[a];
                my_n = ucnt[a];
            }
        }
        const int j0 = r0 + lane, j1 = r0 + lane + 32;
        for (int k = 0; k < nn; ++k) {
            const int nk = __shfl_sync(0xffffffffu, my_n, k);
            if (nk == 0) continue;
            const int64_t off = __shfl_sync(0xffffffffu, my_off, k);
            const int sk = __shfl_sync(0xffffffffu, my_S, k);
            const float *p = back + off;
            int u = 0;
            for (; u + 2 <= nk; u += 2) {  // the loads of two units issued before their (ordered) sums
                const float *pu = p + (int64_t)u * sk, *pv = pu + sk;
                const float x0 = v0 ? pu[j0] : 0.f, x1 = v1 ? pu[j1] : 0.f;
                const float y0 = v0 ? pv[j0] : 0.f, y1 = v1 ? pv[j1] : 0.f;
                a0[0].add(x0);
                a1[0].add(x1);
                a0[0].add(y0);
                a1[0].add(y1);
            }
            for (; u < nk; ++u) {
                const float *pu = p + (int64_t)u * sk;
                a0[0].add(v0 ? pu[j0] : 0.f);
                a1[0].add(v1 ? pu[j1] : 0.f);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (v0) out[r * N + i0] = a0[r].get();
        if (v1) out[r * N + i0 + 32] = a1[r].get();
    }
}

// The FP64 items, as k_p2p_items_x2
template <class T, int R, bool HQ, bool HW>
__global__ void __launch_bounds__(P2P_WARPS * 32) k_p2p_items(
    const int4 *__restrict__ items, const int32_t *__restrict__ irow, int64_t nitems, const int32_t *__restrict__ bstart,
    const int32_t *__restrict__ bcount, const int32_t *__restrict__ nbr, const int32_t *__restrict__ ncnt,
    const int8_t *__restrict__ nd, int64_t N, const T *__restrict__ loc, const T *__restrict__ nrm,
    const T *__restrict__ q, const T *__restrict__ w, double2 *__restrict__ fwd) {
    __shared__ P2PStage<T, R, HQ, HW> stage[P2P_WARPS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * P2P_WARPS;
    auto &sg = stage[warp];
    // the loop bound is uniform in the warp; only warp-level barriers follow
    for (int64_t u = (int64_t)blockIdx.x * P2P_WARPS + warp; u < nitems; u += stride) {
        const int4 it = items[u];
        const int nr = min(P2P_UNIT, bcount[it.x] - it.y);  // uniform in the warp
        if (nr > 32) p2p_item_g<T, R, 1, HQ, HW>(sg, lane, it, nr, bstart, bcount, nbr, ncnt, nd, N, loc, nrm, q, w, fwd, irow + u);
        else if (nr > 16) p2p_item_g<T, R, 2, HQ, HW>(sg, lane, it, nr, bstart, bcount, nbr, ncnt, nd, N, loc, nrm, q, w, fwd, irow + u);
        else if (nr > 8) p2p_item_g<T, R, 4, HQ, HW>(sg, lane, it, nr, bstart, bcount, nbr, ncnt, nd, N, loc, nrm, q, w, fwd, irow + u);
        else p2p_item_g<T, R, 8, HQ, HW>(sg, lane, it, nr, bstart, bcount, nbr, ncnt, nd, N, loc, nrm, q, w, fwd, irow + u);
    }
}

}  // namespace

// scratch that follows the tree: an eighth more than asked for, so that a tree that changes slowly (time
// steps) does not allocate in every product
template <class T>
static void grow(DevBuf<T> &b, size_t n) {
    if (n > b.cap) b.resize(n + n / 8);
}

template <class T, int R, bool HQ, bool HW>
static void launch_units(Context &c, const T *q, const T *w, double *out_sorted, cudaStream_t st) {
    Tree &t = c.tree;
    const int L = t.L;
    const T *loc = sizeof(T) == 8 ? (const T *)t.loc64.p : (const T *)t.loc32.p;
    const T *nrm = sizeof(T) == 8 ? (const T *)t.nrm64.p : (const T *)t.nrm32.p;
    const int64_t nu = t.n_p2p_units;
    if (nu == 0) return;
    // With the far field running concurrently, ask for the SM configuration with the most shared
    // memory: the tensor-core M2L needs it, and an SM whose resident near-field blocks had it
    // configured for more L1 would first have to drain them. (A per-device attribute, set on
    // every launch; about a microsecond.)
    const int32_t *bst = t.bstart.p + t.base[L], *bcn = t.bcount.p + t.base[L];
    if constexpr (std::is_same<T, float>::value) {
        // FP32: the packed kernel over the work items, symmetric for one RHS and the single layer
        constexpr bool SYM = R == 1 && !HW;
        constexpr int li = SYM ? 0 : 1;
        auto kern = k_p2p_items_x2<R, HQ, HW, SYM>;
        if (c.tuned_overlap)
            BEM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                          (int)cudaSharedmemCarveoutMaxShared));
        const int64_t ni = t.n_p2p_items[li];
        int64_t blocks = div_up(ni, P2P_WARPS);
        if (c.tuned_p2p_blocks > 0) blocks = std::min<int64_t>(blocks, (int64_t)c.num_sms * c.tuned_p2p_blocks);
        grow(c.p2p_fwd, (size_t)t.n_p2p_rows[li] * 8 * R);
        const BackArgs ba{SYM ? t.back.p : nullptr, t.back_S.p, t.back_base.p};
        kern<<<(unsigned)blocks, P2P_WARPS * 32, 0, st>>>(t.p2p_items[li].p, t.p2p_irow[li].p, ni, bst, bcn, t.nbr.p, t.nbr_cnt.p,
                                                           t.nbr_d.p, c.N, loc, nrm, q, w, c.p2p_fwd.p, ba);
        BEM_LAUNCH_CHECK();
        k_p2p_gather<float, R, SYM><<<(unsigned)div_up(nu, GATHER_WARPS), GATHER_WARPS * 32, 0, st>>>(
            t.p2p_units.p, nu, t.p2p_ioff[li].p, t.p2p_irow[li].p, c.p2p_fwd.p, bst, bcn, t.nbr.p, t.nbr_cnt.p, t.back_gofs.p, t.p2p_ucnt.p,
            t.back_S.p, t.back_base.p, t.back.p, c.N, out_sorted);
    } else {
        if (c.tuned_overlap)
            BEM_CUDA(cudaFuncSetAttribute(k_p2p_items<T, R, HQ, HW>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                          (int)cudaSharedmemCarveoutMaxShared));
        const int64_t ni = t.n_p2p_items[1];
        int64_t blocks = div_up(ni, P2P_WARPS);
        if (c.tuned_p2p_blocks > 0) blocks = std::min<int64_t>(blocks, (int64_t)c.num_sms * c.tuned_p2p_blocks);
        grow(c.p2p_fwd64, (size_t)t.n_p2p_rows[1] * 8 * R);
        k_p2p_items<T, R, HQ, HW><<<(unsigned)blocks, P2P_WARPS * 32, 0, st>>>(
            t.p2p_items[1].p, t.p2p_irow[1].p, ni, bst, bcn, t.nbr.p, t.nbr_cnt.p, t.nbr_d.p, c.N, loc, nrm, q, w, c.p2p_fwd64.p);
        BEM_LAUNCH_CHECK();
        k_p2p_gather<double, R, false><<<(unsigned)div_up(nu, GATHER_WARPS), GATHER_WARPS * 32, 0, st>>>(
            t.p2p_units.p, nu, t.p2p_ioff[1].p, t.p2p_irow[1].p, c.p2p_fwd64.p, bst, bcn, t.nbr.p, t.nbr_cnt.p, nullptr, nullptr, nullptr,
            nullptr, nullptr, c.N, out_sorted);
    }
    BEM_LAUNCH_CHECK();
}

template <class T, int R>
void launch_p2p_list(Context &c, const T *q, const T *w, double *near_sorted, bool hq, bool hw, cudaStream_t st) {
    if (R > 1 || (hq && hw)) launch_units<T, R, true, true>(c, q, w, near_sorted, st);
    else if (hw) launch_units<T, R, false, true>(c, q, w, near_sorted, st);
    else launch_units<T, R, true, false>(c, q, w, near_sorted, st);  // also the all-zero product
}

template void launch_p2p_list<float, 1>(Context &, const float *, const float *, double *, bool, bool,
                                         cudaStream_t);
template void launch_p2p_list<float, 4>(Context &, const float *, const float *, double *, bool, bool,
                                         cudaStream_t);
template void launch_p2p_list<double, 1>(Context &, const double *, const double *, double *, bool, bool,
                                         cudaStream_t);
template void launch_p2p_list<double, 4>(Context &, const double *, const double *, double *, bool, bool,
                                         cudaStream_t);

}  // namespace bem
