// Octree of Section 3.7: the domain is scaled to a cube, refined uniformly to depth l_max,
// empty boxes are skipped, boxes are found by bit interleaving (Morton keys) and sorting, and
// the near-field (27-box neighbourhood) and M2L interaction lists are built.
//
// Everything runs on the device: bounding-cube reduction, 30-bit Morton keys, a stable LSD
// radix sort written here (8-bit digits, per-warp match ranking), per-level unique boxes by
// flag + scan. The 27 neighbours of every box come from its parent's: the neighbour at d is a
// child of the parent's neighbour, found in the table of children, so the near-field and M2L
// lists need no search.
#include "internal.h"

#include <algorithm>
#include <cmath>

namespace bem {

// ------------------------------------------------------------------------------ scratch
namespace {
struct Scratch {
    DevBuf<int32_t> a, b, c;
};
Scratch &scan_scratch(int depth) {
    static Scratch s[4];
    return s[depth];
}

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 4;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

// Exclusive scan of one tile per block; writes the tile total to sums[block].
__global__ void k_scan_tiles(const int32_t *__restrict__ in, int32_t *__restrict__ out, int64_t n,
                             int32_t *__restrict__ sums) {
    __shared__ int32_t warp_tot[SCAN_THREADS / 32];
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE + threadIdx.x * SCAN_ITEMS;
    int32_t v[SCAN_ITEMS];
    int32_t t = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        v[i] = (base + i < n) ? in[base + i] : 0;
        t += v[i];
    }
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int32_t incl = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_tot[w] = incl;
    __syncthreads();
    if (w == 0) {
        int32_t x = lane < SCAN_THREADS / 32 ? warp_tot[lane] : 0;
        int32_t xi = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int32_t y = __shfl_up_sync(0xffffffffu, xi, o);
            if (lane >= o) xi += y;
        }
        if (lane < SCAN_THREADS / 32) warp_tot[lane] = xi - x;
        if (lane == SCAN_THREADS / 32 - 1 && sums) sums[blockIdx.x] = xi;
    }
    __syncthreads();
    int32_t run = warp_tot[w] + incl - t;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        if (base + i < n) out[base + i] = run;
        run += v[i];
    }
}

__global__ void k_scan_add(int32_t *__restrict__ out, int64_t n, const int32_t *__restrict__ offs) {
    int64_t i = (int64_t)blockIdx.x * SCAN_TILE + threadIdx.x;
    int32_t o = offs[blockIdx.x];
    for (int k = 0; k < SCAN_ITEMS; ++k, i += SCAN_THREADS)
        if (i < n) out[i] += o;
}

__global__ void k_scan_total(const int32_t *in, const int32_t *ex, int64_t n, int32_t *total) {
    *total = (n > 0) ? ex[n - 1] + in[n - 1] : 0;
}

void scan_rec(const int32_t *in, int32_t *out, int64_t n, cudaStream_t st, int depth) {
    int nb = div_up(n, SCAN_TILE);
    if (nb <= 1) {
        k_scan_tiles<<<1, SCAN_THREADS, 0, st>>>(in, out, n, nullptr);
        BEM_LAUNCH_CHECK();
        return;
    }
    if (depth >= 3) fail(BEM_ERR_ARG, "scan too large");
    Scratch &s = scan_scratch(depth);
    s.a.resize(nb);
    s.b.resize(nb);
    k_scan_tiles<<<nb, SCAN_THREADS, 0, st>>>(in, out, n, s.a.p);
    BEM_LAUNCH_CHECK();
    scan_rec(s.a.p, s.b.p, nb, st, depth + 1);
    k_scan_add<<<nb, SCAN_THREADS, 0, st>>>(out, n, s.b.p);
    BEM_LAUNCH_CHECK();
}
}  // namespace

void exclusive_scan_i32(const int32_t *in, int32_t *out, int64_t n, int32_t *total_dev, cudaStream_t st) {
    if (n <= 0) return;
    scan_rec(in, out, n, st, 0);
    if (total_dev) {
        k_scan_total<<<1, 1, 0, st>>>(in, out, n, total_dev);
        BEM_LAUNCH_CHECK();
    }
}

// ------------------------------------------------------------------------------ radix sort
namespace {
constexpr int RS_THREADS = 256;
constexpr int RS_ITEMS = 8;
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;
constexpr int RS_WARPS = RS_THREADS / 32;

__global__ void k_rs_hist(const uint32_t *__restrict__ keys, int64_t n, int shift,
                          int32_t *__restrict__ hist, int nblocks) {
    __shared__ int32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    int64_t base = (int64_t)blockIdx.x * RS_TILE;
    for (int r = 0; r < RS_ITEMS; ++r) {
        int64_t i = base + r * RS_THREADS + threadIdx.x;
        if (i < n) atomicAdd(&h[(keys[i] >> shift) & 255u], 1);
    }
    __syncthreads();
    hist[(int64_t)threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

// Stable scatter: items keep their input order within a digit. Items are taken in rounds of
// RS_THREADS consecutive keys; a warp ranks equal digits with __match_any_sync and warps are
// ordered through a shared per-digit prefix.
__global__ void k_rs_scatter(const uint32_t *__restrict__ kin, const int32_t *__restrict__ vin,
                             uint32_t *__restrict__ kout, int32_t *__restrict__ vout, int64_t n,
                             int shift, const int32_t *__restrict__ offs, int nblocks) {
    __shared__ int32_t running[256];
    __shared__ int32_t total[256];
    __shared__ int32_t wcnt[RS_WARPS][256];
    int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    running[tid] = offs[(int64_t)tid * nblocks + blockIdx.x];
    int64_t base = (int64_t)blockIdx.x * RS_TILE;
    for (int r = 0; r < RS_ITEMS; ++r) {
        for (int k = 0; k < 8; ++k) wcnt[w][lane * 8 + k] = 0;
        int64_t i = base + r * RS_THREADS + tid;
        bool valid = i < n;
        uint32_t key = valid ? kin[i] : 0u;
        int32_t val = valid ? vin[i] : 0;
        int d = valid ? (int)((key >> shift) & 255u) : 256;
        unsigned peers = __match_any_sync(0xffffffffu, d);
        int rank = __popc(peers & ((1u << lane) - 1u));
        __syncwarp();
        if (valid && rank == 0) wcnt[w][d] = __popc(peers);
        __syncthreads();
        {
            int acc = 0;
            for (int ww = 0; ww < RS_WARPS; ++ww) {
                int t = wcnt[ww][tid];
                wcnt[ww][tid] = acc;
                acc += t;
            }
            total[tid] = acc;
        }
        __syncthreads();
        if (valid) {
            int pos = running[d] + wcnt[w][d] + rank;
            kout[pos] = key;
            vout[pos] = val;
        }
        __syncthreads();
        running[tid] += total[tid];
        __syncthreads();
    }
}
}  // namespace

// Sort (keys, vals) by the low `bits` bits of the keys, stably. Result ends in keys/vals.
void radix_sort_u32(uint32_t *keys, int32_t *vals, int64_t n, int bits, uint32_t *keys_tmp,
                    int32_t *vals_tmp, cudaStream_t st) {
    if (n <= 1) return;
    int nblocks = div_up(n, RS_TILE);
    static DevBuf<int32_t> hist, offs;
    hist.resize((size_t)256 * nblocks);
    offs.resize((size_t)256 * nblocks);
    uint32_t *ka = keys, *kb = keys_tmp;
    int32_t *va = vals, *vb = vals_tmp;
    int passes = 0;
    for (int shift = 0; shift < bits; shift += 8) {
        k_rs_hist<<<nblocks, RS_THREADS, 0, st>>>(ka, n, shift, hist.p, nblocks);
        BEM_LAUNCH_CHECK();
        exclusive_scan_i32(hist.p, offs.p, (int64_t)256 * nblocks, nullptr, st);
        k_rs_scatter<<<nblocks, RS_THREADS, 0, st>>>(ka, va, kb, vb, n, shift, offs.p, nblocks);
        BEM_LAUNCH_CHECK();
        std::swap(ka, kb);
        std::swap(va, vb);
        ++passes;
    }
    if (passes & 1) {
        BEM_CUDA(cudaMemcpyAsync(keys, ka, n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, st));
        BEM_CUDA(cudaMemcpyAsync(vals, va, n * sizeof(int32_t), cudaMemcpyDeviceToDevice, st));
    }
}

// ------------------------------------------------------------------------------ Morton helpers
namespace {
__device__ __forceinline__ uint32_t spread3(uint32_t x) {
    x &= 0x3ffu;
    x = (x | (x << 16)) & 0x030000FFu;
    x = (x | (x << 8)) & 0x0300F00Fu;
    x = (x | (x << 4)) & 0x030C30C3u;
    x = (x | (x << 2)) & 0x09249249u;
    return x;
}
__device__ __forceinline__ uint32_t compact3(uint32_t x) {
    x &= 0x09249249u;
    x = (x ^ (x >> 2)) & 0x030C30C3u;
    x = (x ^ (x >> 4)) & 0x0300F00Fu;
    x = (x ^ (x >> 8)) & 0xFF0000FFu;
    x = (x ^ (x >> 16)) & 0x000003FFu;
    return x;
}
__device__ __forceinline__ uint32_t morton(uint32_t gx, uint32_t gy, uint32_t gz) {
    return (spread3(gx) << 2) | (spread3(gy) << 1) | spread3(gz);
}
__device__ __forceinline__ void demorton(uint32_t k, int &gx, int &gy, int &gz) {
    gx = (int)compact3(k >> 2);
    gy = (int)compact3(k >> 1);
    gz = (int)compact3(k);
}
__global__ void k_bbox(int64_t N, const double *__restrict__ xyz, double *__restrict__ part) {
    // part[block][6] = min x,y,z, max x,y,z
    __shared__ double sm[6][256];
    double mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        for (int d = 0; d < 3; ++d) {
            double v = xyz[d * N + i];
            mn[d] = fmin(mn[d], v);
            mx[d] = fmax(mx[d], v);
        }
    }
    for (int d = 0; d < 3; ++d) {
        sm[d][threadIdx.x] = mn[d];
        sm[3 + d][threadIdx.x] = mx[d];
    }
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s)
            for (int d = 0; d < 3; ++d) {
                sm[d][threadIdx.x] = fmin(sm[d][threadIdx.x], sm[d][threadIdx.x + s]);
                sm[3 + d][threadIdx.x] = fmax(sm[3 + d][threadIdx.x], sm[3 + d][threadIdx.x + s]);
            }
        __syncthreads();
    }
    if (threadIdx.x < 6) part[blockIdx.x * 6 + threadIdx.x] = sm[threadIdx.x][0];
}

__global__ void k_keys(int64_t N, const double *__restrict__ xyz, double ox, double oy, double oz,
                       double inv_size, uint32_t *__restrict__ key, int32_t *__restrict__ idx) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double scale = inv_size * (double)(1 << kDeepLevel);
    int g[3];
    double o[3] = {ox, oy, oz};
    for (int d = 0; d < 3; ++d) {
        double u = (xyz[d * N + i] - o[d]) * scale;
        int gi = (int)floor(u);
        g[d] = min(max(gi, 0), (1 << kDeepLevel) - 1);
    }
    key[i] = morton(g[0], g[1], g[2]);
    idx[i] = (int32_t)i;
}

// Clusters: the key is (cluster << 24) | 24-bit Morton key of depth 8 in the cluster's own cube,
// so sorting groups clusters and shifting right by 3 (8 - l) gives (cluster << 3l) | box key.
constexpr int kClusterDeep = 8;

constexpr int CB_PARTS = 16;  // blocks per cluster (one took 219 us for 16 clusters of 359000 points)
__global__ void k_cluster_bbox(const int64_t *__restrict__ cvoff, int64_t N, const double *__restrict__ xyz,
                               double *__restrict__ out) {
    __shared__ double sm[6][256];
    const int c = blockIdx.x / CB_PARTS, part = blockIdx.x % CB_PARTS;
    double mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int64_t i = cvoff[c] + part * 256 + threadIdx.x; i < cvoff[c + 1]; i += 256 * CB_PARTS)
        for (int d = 0; d < 3; ++d) {
            double v = xyz[d * N + i];
            mn[d] = fmin(mn[d], v);
            mx[d] = fmax(mx[d], v);
        }
    for (int d = 0; d < 3; ++d) {
        sm[d][threadIdx.x] = mn[d];
        sm[3 + d][threadIdx.x] = mx[d];
    }
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s)
            for (int d = 0; d < 3; ++d) {
                sm[d][threadIdx.x] = fmin(sm[d][threadIdx.x], sm[d][threadIdx.x + s]);
                sm[3 + d][threadIdx.x] = fmax(sm[3 + d][threadIdx.x], sm[3 + d][threadIdx.x + s]);
            }
        __syncthreads();
    }
    if (threadIdx.x < 6) out[blockIdx.x * 6 + threadIdx.x] = sm[threadIdx.x][0];
}

// cube[c] = (origin x, y, z, 1 / size)
__global__ void k_keys_clusters(int64_t N, const double *__restrict__ xyz, const int32_t *__restrict__ vcid,
                                const double *__restrict__ cube, uint32_t *__restrict__ key, int32_t *__restrict__ idx) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int c = vcid[i];
    const double scale = cube[4 * c + 3] * (double)(1 << kClusterDeep);
    int g[3];
    for (int d = 0; d < 3; ++d) {
        double u = (xyz[d * N + i] - cube[4 * c + d]) * scale;
        int gi = (int)floor(u);
        g[d] = min(max(gi, 0), (1 << kClusterDeep) - 1);
    }
    key[i] = ((uint32_t)c << (3 * kClusterDeep)) | morton(g[0], g[1], g[2]);
    idx[i] = (int32_t)i;
}

// cnt[l] += number of i in [1, N) whose key first differs from the one before at level l (the prefix of
// every deeper level differs as well)
__global__ void __launch_bounds__(256) k_level_counts(int64_t N, int deep, const uint32_t *__restrict__ key,
                                                      int32_t *__restrict__ cnt) {
    __shared__ int32_t h[kDeepLevel + 1];
    if (threadIdx.x <= kDeepLevel) h[threadIdx.x] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t b = blockIdx.x * (int64_t)blockDim.x; b < N; b += stride) {  // uniform in the block
        const int64_t i = b + threadIdx.x;
        const uint32_t x = i >= 1 && i < N ? key[i] ^ key[i - 1] : 0u;
        const int l = x ? max(0, deep - (31 - __clz(x)) / 3) : -1;
        int mine = 0;
        for (int q = 0; q <= deep; ++q) {
            const int n = __popc(__ballot_sync(0xffffffffu, l == q));
            if (lane == q) mine = n;
        }
        if (lane <= deep && mine) atomicAdd(&h[lane], mine);
    }
    __syncthreads();
    if (threadIdx.x <= deep && h[threadIdx.x]) atomicAdd(&cnt[threadIdx.x], h[threadIdx.x]);
}

__global__ void k_flags_points(int64_t N, const uint32_t *__restrict__ key, int shift, int32_t *__restrict__ flag) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= N) return;
    flag[i] = (i == 0 || (key[i] >> shift) != (key[i - 1] >> shift)) ? 1 : 0;
}

// Leaf boxes straight from the sorted points: start, key and the leaf of every point.
__global__ void k_emit_leaves(int64_t N, const uint32_t *__restrict__ key, int shift,
                              const int32_t *__restrict__ flag, const int32_t *__restrict__ ex,
                              uint32_t *__restrict__ bkey, int32_t *__restrict__ bstart,
                              int32_t *__restrict__ leaf_of) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= N) return;
    int b = ex[i] + flag[i] - 1;
    leaf_of[i] = b;
    if (flag[i]) {
        bkey[b] = key[i] >> shift;
        bstart[b] = (int32_t)i;
    }
}

__global__ void k_flags_boxes(int n, const uint32_t *__restrict__ ckey, int32_t *__restrict__ flag) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    flag[i] = (i == 0 || (ckey[i] >> 3) != (ckey[i - 1] >> 3)) ? 1 : 0;
}

// Parents from children (children are sorted, so each parent's children are contiguous).
__global__ void k_emit_parents(int n, const uint32_t *__restrict__ ckey, const int32_t *__restrict__ cstart,
                               const int32_t *__restrict__ flag, const int32_t *__restrict__ ex,
                               uint32_t *__restrict__ pkey, int32_t *__restrict__ pstart,
                               int32_t *__restrict__ cparent, int pbase) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int b = ex[i] + flag[i] - 1;
    cparent[i] = pbase + b;
    if (flag[i]) {
        pkey[b] = ckey[i] >> 3;
        pstart[b] = cstart[i];
    }
}

__global__ void k_box_counts(int n, const int32_t *__restrict__ bstart, int32_t total, int32_t *__restrict__ bcount) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    bcount[i] = ((i + 1 < n) ? bstart[i + 1] : total) - bstart[i];
}

// nb27[box][27]: the boxes of the same level (and cluster) around every box, itself included, by offset
// (dx, dy, dz) in lexicographic order; -1 where empty. One level, from the level above.
__global__ void k_nb27(int n, int gbase, const uint32_t *__restrict__ bkey, const int32_t *__restrict__ parent,
                       const int32_t *__restrict__ child8, int32_t *__restrict__ nb27) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n * 27) return;
    const int b = gbase + e / 27, k = e % 27;
    const int d[3] = {k / 9 - 1, k / 3 % 3 - 1, k % 3 - 1};
    const int par = parent[b];
    if (par < 0) {  // a root: its cluster has no other box at this level
        nb27[(int64_t)b * 27 + k] = k == 13 ? b : -1;
        return;
    }
    const uint32_t oct = bkey[b] & 7u;
    int pk = 0, oc = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int c = (int)((oct >> (2 - a)) & 1u) + d[a];  // -1 .. 2 in the parent's children
        pk = pk * 3 + (c >> 1) + 1;
        oc = oc * 2 + (c & 1);
    }
    const int pn = nb27[(int64_t)par * 27 + pk];
    nb27[(int64_t)b * 27 + k] = pn >= 0 ? child8[(int64_t)pn * 8 + oc] : -1;
}

// Near field (Section 3.7, A^(sparse)): the non-empty leaves among the 27 around each leaf.
__global__ void k_neighbours(int nleaf, int gbase, const int32_t *__restrict__ nb27,
                             const int32_t *__restrict__ lcount, int32_t *__restrict__ nbr,
                             int32_t *__restrict__ ncnt, int8_t *__restrict__ nd,
                             unsigned long long *__restrict__ pairs) {
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    long long mine = 0;
    if (b < nleaf) {
        int c = 0;
        long long src = 0;
        for (int k = 0; k < 27; ++k) {
            const int g = nb27[(int64_t)(gbase + b) * 27 + k];
            if (g < 0) continue;
            nbr[b * 27 + c] = g - gbase;
            reinterpret_cast<char4 *>(nd)[b * 27 + c] =
                make_char4((signed char)(k / 9 - 1), (signed char)(k / 3 % 3 - 1), (signed char)(k % 3 - 1), 0);
            src += lcount[g - gbase];
            ++c;
        }
        ncnt[b] = c;
        mine = lcount[b] * (src - 1);
    }
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(pairs, (unsigned long long)mine);
}

// Compact index of an M2L offset (dx,dy,dz) in [-3,3]^3 with max |d| >= 2, in lexicographic
// order; must match the order in which the operator builder enumerates the offsets. It is the
// offset's position among all 343 offsets minus the near offsets (all |d| <= 1) before it.
__device__ __forceinline__ int m2l_class(int dx, int dy, int dz) {
    const int full = (dx + 3) * 49 + (dy + 3) * 7 + (dz + 3);
    auto below = [](int d) { return min(max(d + 1, 0), 3); };  // near values (-1, 0, 1) below d
    const bool nx = dx >= -1 && dx <= 1, ny = dy >= -1 && dy <= 1;
    const int near_before = below(dx) * 9 + (nx ? below(dy) * 3 + (ny ? below(dz) : 0) : 0);
    return full - near_before;
}

// M2L list of a box: children of the parent's neighbours that are not its own neighbours; one warp
// per box (levels 2 on). The 216 candidates run over the offsets (dx, dy, dz) in lexicographic order,
// so a box's pairs come out by ascending offset class. pass 0 counts, pass 1 writes (target,
// source, class) from off[box] on.
__global__ void __launch_bounds__(256) k_m2l_lists(int first, int nbox, const uint32_t *__restrict__ bkey,
                                                   const int32_t *__restrict__ parent,
                                                   const int32_t *__restrict__ nb27, const int32_t *__restrict__ child8,
                                                   int pass, int32_t *__restrict__ cnt, const int32_t *__restrict__ off,
                                                   int32_t *__restrict__ tgt, int32_t *__restrict__ src,
                                                   uint32_t *__restrict__ cls) {
    const int b = first + blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (b >= nbox) return;  // uniform in the warp
    const uint32_t oct = bkey[b] & 7u;
    const int bx = (oct >> 2) & 1, by = (oct >> 1) & 1, bz = oct & 1;
    const int32_t *pn = nb27 + (int64_t)parent[b] * 27;
    int n = 0;
    const int64_t o = pass ? off[b] : 0;
    for (int c0 = 0; c0 < 216; c0 += 32) {
        const int c = c0 + lane;
        int f = -1, dx = 0, dy = 0, dz = 0;
        if (c < 216) {
            // per axis i = 0..5: the parent's neighbour (i >> 1) - 1 and its child i & 1
            const int ix = c / 36, iy = c / 6 % 6, iz = c % 6;
            dx = ix - 2 - bx;
            dy = iy - 2 - by;
            dz = iz - 2 - bz;
            if (max(abs(dx), max(abs(dy), abs(dz))) > 1) {
                const int p = pn[(ix >> 1) * 9 + (iy >> 1) * 3 + (iz >> 1)];
                if (p >= 0) f = child8[(int64_t)p * 8 + (ix & 1) * 4 + (iy & 1) * 2 + (iz & 1)];
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, f >= 0);
        if (pass && f >= 0) {
            const int64_t q = o + n + __popc(m & ((1u << lane) - 1u));
            tgt[q] = b;
            src[q] = f;
            cls[q] = (uint32_t)m2l_class(dx, dy, dz);
        }
        n += __popc(m);
    }
    if (!pass && lane == 0) cnt[b] = n;
}

__global__ void k_iota(int64_t n, int32_t *a) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) a[i] = (int32_t)i;
}

// the pairs in class-sorted order, and every target-major pair's place in it
__global__ void k_m2l_order(int64_t n, const int32_t *__restrict__ order, const int32_t *__restrict__ ptgt,
                            const int32_t *__restrict__ psrc, int32_t *__restrict__ tgt, int32_t *__restrict__ src,
                            int32_t *__restrict__ by_tgt) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int k = order[i];
    tgt[i] = ptgt[k];
    src[i] = psrc[k];
    by_tgt[k] = (int32_t)i;
}

__global__ void __launch_bounds__(256) k_class_hist(int64_t n, const uint32_t *__restrict__ k, int32_t *__restrict__ h) {
    __shared__ int32_t s[kNumM2LClasses];
    for (int i = threadIdx.x; i < kNumM2LClasses; i += blockDim.x) s[i] = 0;
    __syncthreads();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(&s[k[i]], 1);
    __syncthreads();
    for (int i = threadIdx.x; i < kNumM2LClasses; i += blockDim.x)
        if (s[i]) atomicAdd(&h[i], s[i]);
}

// child8[box][8]: the children of every box by octant (the low bits of their keys), -1 where empty
__global__ void k_child8(int first, int nbox, const uint32_t *__restrict__ bkey, const int32_t *__restrict__ parent,
                         int32_t *__restrict__ child8) {
    const int i = first + blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nbox) child8[(int64_t)parent[i] * 8 + (bkey[i] & 7u)] = i;
}

// Sorted-order point data: leaf-local coordinates (units of the leaf box, centred), normals
// and weights.
__global__ void k_sorted_points(int64_t N, int L, int deep, const int32_t *__restrict__ perm,
                                const uint32_t *__restrict__ key, const double *__restrict__ xyz,
                                const double *__restrict__ nrm, const double *__restrict__ s,
                                const double *__restrict__ cube, const int32_t *__restrict__ vcid,
                                double *__restrict__ loc64, float *__restrict__ loc32,
                                double *__restrict__ n64, float *__restrict__ n32,
                                double *__restrict__ s_sorted, double *__restrict__ ih) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= N) return;
    int j = perm[i];
    int g[3];
    demorton((key[i] >> (3 * (deep - L))) & ((1u << (3 * L)) - 1u), g[0], g[1], g[2]);
    const int c = vcid ? vcid[j] : 0;
    double o[3] = {cube[4 * c], cube[4 * c + 1], cube[4 * c + 2]};
    double scale = cube[4 * c + 3] * (double)(1 << L);
    ih[i] = scale;
    for (int d = 0; d < 3; ++d) {
        double u = (xyz[d * N + j] - o[d]) * scale - ((double)g[d] + 0.5);
        loc64[d * N + i] = u;
        loc32[d * N + i] = (float)u;
        double nv = nrm[d * N + j];
        n64[d * N + i] = nv;
        n32[d * N + i] = (float)nv;
    }
    s_sorted[i] = s[j];
}
constexpr int P2P_ITEM_RECV = 64;  // receivers of a near-field unit
// Near-field work units: leaf b gets ceil(n_b / 64) units (b, 64 u).
__global__ void k_p2p_unit_count(int nleaf, const int32_t *__restrict__ bcount, int32_t *__restrict__ cnt) {
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < nleaf) cnt[b] = (bcount[b] + 63) / 64;
}

__global__ void k_p2p_unit_emit(int nleaf, const int32_t *__restrict__ bcount, const int32_t *__restrict__ off,
                                int2 *__restrict__ units) {
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nleaf) return;
    const int n = (bcount[b] + 63) / 64;
    for (int u = 0; u < n; ++u) units[off[b] + u] = make_int2(b, 64 * u);
}

// Symmetric near field: leaf A owns its pairs with the neighbours B > A. S_A = the floats one
// unit of A writes (the points of its owned neighbours, in neighbour-list order); the leaf's
// region holds its units' shares one after another, padded to 32 floats. all_A = the points of all
// neighbours but A itself.
__global__ void k_back_sizes(int nleaf, const int32_t *__restrict__ nbr, const int32_t *__restrict__ ncnt,
                             const int32_t *__restrict__ bcount, const int32_t *__restrict__ ucnt,
                             int32_t *__restrict__ S, int32_t *__restrict__ all, int32_t *__restrict__ blk32) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= nleaf) return;
    int s = 0, n = 0;
    for (int k = 0; k < ncnt[a]; ++k) {
        const int f = nbr[a * 27 + k];
        if (f > a) s += bcount[f];
        if (f != a) n += bcount[f];
    }
    S[a] = s;
    all[a] = n;
    blk32[a] = (int32_t)(((int64_t)ucnt[a] * s + 31) / 32);
}

// Items of a near-field unit (leaf b, receivers r0 ..): `len` list positions cut every `chunk` (times
// the lane groups that a small unit splits its tiles over); the first item also takes the leaf's
// own points, and so much less of the list.
struct UnitCut {
    int first, chunk, n;
};
__device__ __forceinline__ UnitCut unit_cut(int own, int r0, int len, int chunk) {
    const int nr = min(64, own - r0);
    const int c = chunk * (nr > 32 ? 1 : (nr > 16 ? 2 : (nr > 8 ? 4 : 8)));
    const int first = min(len, max(0, c - (own + 31) / 32 * 32));
    return {first, c, 1 + (len - first + c - 1) / c};
}
// receivers of a unit rounded up to 8, in eights
__device__ __forceinline__ int unit_row8(int own, int r0) { return (min(64, own - r0) + 7) / 8; }
// cnt[4][nu] + 1: per unit the items of the symmetric and of the one-way list, then the eights of their rows
__global__ void k_p2p_item_count(int64_t nu, const int2 *__restrict__ units, const int32_t *__restrict__ bcount,
                                 const int32_t *__restrict__ len0, const int32_t *__restrict__ len1, int chunk0, int chunk1,
                                 int32_t *__restrict__ cnt) {
    const int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (u >= nu) return;
    const int2 un = units[u];
    const int own = bcount[un.x], w8 = unit_row8(own, un.y);
    const int n0 = unit_cut(own, un.y, len0[un.x], chunk0).n, n1 = unit_cut(own, un.y, len1[un.x], chunk1).n;
    cnt[u] = n0;
    cnt[nu + u] = n1;
    cnt[2 * nu + u] = n0 * w8;
    cnt[3 * nu + u] = n1 * w8;
    if (u == 0) cnt[4 * nu] = 0;
}
// items, their rows and the units' first items, list by list, from the sums over cnt
__global__ void k_p2p_item_emit(int64_t nu, const int2 *__restrict__ units, const int32_t *__restrict__ bcount,
                                const int32_t *__restrict__ len, int chunk, const int32_t *__restrict__ ex, int list,
                                int32_t *__restrict__ ioff, int4 *__restrict__ items, int32_t *__restrict__ irow) {
    const int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (u >= nu) return;
    const int2 un = units[u];
    const int L = len[un.x], own = bcount[un.x], w8 = unit_row8(own, un.y);
    const UnitCut uc = unit_cut(own, un.y, L, chunk);
    const int32_t *ei = ex + list * nu, *er = ex + (2 + list) * nu;
    const int i0 = ei[u] - ei[0], row = er[u] - er[0];
    ioff[u] = i0;
    if (u + 1 == nu) ioff[nu] = i0 + uc.n;
    items[i0] = make_int4(un.x, un.y, -1, uc.first);  // -1: from 0, and the leaf's own points
    irow[i0] = row;
    for (int i = 1; i < uc.n; ++i) {
        items[i0 + i] = make_int4(un.x, un.y, uc.first + (i - 1) * uc.chunk, min(L, uc.first + i * uc.chunk));
        irow[i0 + i] = row + i * w8;
    }
}

__global__ void k_back_base(int nleaf, const int32_t *__restrict__ blkoff, int64_t *__restrict__ base) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a < nleaf) base[a] = 32 * (int64_t)blkoff[a];
}

// for neighbour k = A of leaf B with A < B: where B's share starts inside each unit of A (the
// owned neighbours of A before B in A's list, summed)
__global__ void k_back_gofs(int nleaf, const int32_t *__restrict__ nbr, const int32_t *__restrict__ ncnt,
                            const int32_t *__restrict__ bcount, int32_t *__restrict__ gofs) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nleaf * 27) return;
    const int b = e / 27, k = e % 27;
    int g = -1;
    if (k < ncnt[b]) {
        const int a = nbr[e];
        if (a < b) {
            int off = 0;
            for (int k2 = 0; k2 < ncnt[a]; ++k2) {
                const int f = nbr[a * 27 + k2];
                if (f == b) {
                    g = off;
                    break;
                }
                if (f > a) off += bcount[f];
            }
        }
    }
    gofs[e] = g;
}

}  // namespace

// ------------------------------------------------------------------------------ build
void build_tree(Context &c) {
    Tree &t = c.tree;
    cudaStream_t st = c.stream;
    const int64_t N = c.N;
    t.N = N;
    const int tb = 256;

    const bool clusters = c.C > 1;
    t.deep = clusters ? kClusterDeep : kDeepLevel;
    DevBuf<double> &cube = t.s_f64[0];  // per cluster: origin x, y, z, 1 / size
    cube.resize(4 * std::max<int64_t>(c.C, 1));
    std::vector<double> hcube(4 * std::max<int64_t>(c.C, 1));
    // 1. bounding cube (one per cluster)
    int nbb = std::min<int64_t>(div_up(N, tb), 1024);
    DevBuf<double> &part = t.s_f64[1];
    part.resize((size_t)nbb * 6);
    k_bbox<<<nbb, tb, 0, st>>>(N, c.xyz.p, part.p);
    BEM_LAUNCH_CHECK();
    std::vector<double> hp((size_t)nbb * 6);
    BEM_CUDA(cudaMemcpyAsync(hp.data(), part.p, hp.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
    BEM_CUDA(cudaStreamSynchronize(st));
    double mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int b = 0; b < nbb; ++b)
        for (int d = 0; d < 3; ++d) {
            mn[d] = std::min(mn[d], hp[b * 6 + d]);
            mx[d] = std::max(mx[d], hp[b * 6 + 3 + d]);
        }
    double ext = 0.0;
    for (int d = 0; d < 3; ++d) {
        if (!std::isfinite(mn[d]) || !std::isfinite(mx[d])) fail(BEM_ERR_NAN, "non-finite vertex coordinate");
        ext = std::max(ext, mx[d] - mn[d]);
    }
    if (ext <= 0.0) ext = 1.0;
    t.size = ext * (1.0 + 1.0 / 1024.0);
    for (int d = 0; d < 3; ++d) t.origin[d] = 0.5 * (mn[d] + mx[d]) - 0.5 * t.size;
    for (int d = 0; d < 3; ++d) hcube[d] = t.origin[d];
    hcube[3] = 1.0 / t.size;
    if (clusters) {
        std::vector<int64_t> cvoff(c.C + 1);
        for (int64_t k = 0; k <= c.C; ++k) cvoff[k] = c.vert_off[c.cluster_boff[k]];
        DevBuf<int64_t> &dcv = t.s_i64[0];
        DevBuf<double> &cb = t.s_f64[2];
        dcv.resize(c.C + 1);
        cb.resize(6 * c.C * CB_PARTS);
        BEM_CUDA(cudaMemcpyAsync(dcv.p, cvoff.data(), (c.C + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, st));
        k_cluster_bbox<<<(unsigned)(c.C * CB_PARTS), 256, 0, st>>>(dcv.p, N, c.xyz.p, cb.p);
        BEM_LAUNCH_CHECK();
        std::vector<double> hb(6 * c.C * CB_PARTS);
        BEM_CUDA(cudaMemcpyAsync(hb.data(), cb.p, hb.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
        BEM_CUDA(cudaStreamSynchronize(st));
        for (int64_t k = 0; k < c.C; ++k) {
            // the parts' boxes joined into the first one's place
            for (int q = 0; q < CB_PARTS; ++q)
                for (int d = 0; d < 3; ++d) {
                    const double lo = hb[6 * (k * CB_PARTS + q) + d], hi = hb[6 * (k * CB_PARTS + q) + 3 + d];
                    hb[6 * k + d] = q ? std::min(hb[6 * k + d], lo) : lo;
                    hb[6 * k + 3 + d] = q ? std::max(hb[6 * k + 3 + d], hi) : hi;
                }
            double e = 0.0;
            for (int d = 0; d < 3; ++d) e = std::max(e, hb[6 * k + 3 + d] - hb[6 * k + d]);
            if (!(e > 0.0)) e = 1.0;
            double size = e * (1.0 + 1.0 / 1024.0);
            for (int d = 0; d < 3; ++d) hcube[4 * k + d] = 0.5 * (hb[6 * k + d] + hb[6 * k + 3 + d]) - 0.5 * size;
            hcube[4 * k + 3] = 1.0 / size;
        }
    }
    BEM_CUDA(cudaMemcpyAsync(cube.p, hcube.data(), hcube.size() * sizeof(double), cudaMemcpyHostToDevice, st));

    // 2. Morton keys at the key depth and sort
    t.key.resize(N);
    t.perm.resize(N);
    DevBuf<uint32_t> &ktmp = t.s_u32[0];
    DevBuf<int32_t> &vtmp = t.s_i32[0];
    ktmp.resize(N);
    vtmp.resize(N);
    if (clusters)
        k_keys_clusters<<<div_up(N, tb), tb, 0, st>>>(N, c.xyz.p, c.vcid.p, cube.p, t.key.p, t.perm.p);
    else
        k_keys<<<div_up(N, tb), tb, 0, st>>>(N, c.xyz.p, t.origin[0], t.origin[1], t.origin[2], 1.0 / t.size,
                                              t.key.p, t.perm.p);
    BEM_LAUNCH_CHECK();
    radix_sort_u32(t.key.p, t.perm.p, N, clusters ? 32 : 3 * kDeepLevel, ktmp.p, vtmp.p, st);

    // 3. unique boxes per level; choose l_max
    DevBuf<int32_t> &lc = t.s_i32[1];
    lc.resize(kDeepLevel + 1);
    BEM_CUDA(cudaMemsetAsync(lc.p, 0, (kDeepLevel + 1) * sizeof(int32_t), st));
    k_level_counts<<<(unsigned)std::min<int64_t>(div_up(N, 256), 1024), 256, 0, st>>>(N, t.deep, t.key.p, lc.p);
    BEM_LAUNCH_CHECK();
    int32_t hc[kDeepLevel + 1] = {};
    BEM_CUDA(cudaMemcpyAsync(hc, lc.p, (t.deep + 1) * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    BEM_CUDA(cudaStreamSynchronize(st));
    for (int l = 1; l <= t.deep; ++l) hc[l] += hc[l - 1];
    int L = 2;
    const int forced = c.level_override > 0 ? c.level_override : c.prm.fixed_level;
    if (forced > 0) {
        L = std::min(forced, t.deep);
    } else {
        for (int l = 2; l <= t.deep; ++l)
            if ((double)N / (double)(hc[l] + 1) >= (double)std::max(c.prm.leaf_target, 1)) L = l;
    }
    t.L = L;
    t.nb.assign(L + 1, 0);
    t.base.assign(L + 2, 0);
    for (int l = 0; l <= L; ++l) {
        t.nb[l] = hc[l] + 1;
        t.base[l + 1] = t.base[l] + t.nb[l];
    }
    t.nbox = t.base[L + 1];

    // 4. boxes of every level
    t.bkey.resize(t.nbox);
    t.bstart.resize(t.nbox);
    t.bcount.resize(t.nbox);
    t.parent.resize(t.nbox);
    t.leaf_of.resize(N);
    DevBuf<int32_t> &flag = t.s_i32[2], &ex = t.s_i32[3];
    flag.resize(N);
    ex.resize(N);
    int shiftL = 3 * (t.deep - L);
    k_flags_points<<<div_up(N, tb), tb, 0, st>>>(N, t.key.p, shiftL, flag.p);
    BEM_LAUNCH_CHECK();
    exclusive_scan_i32(flag.p, ex.p, N, nullptr, st);
    k_emit_leaves<<<div_up(N, tb), tb, 0, st>>>(N, t.key.p, shiftL, flag.p, ex.p, t.bkey.p + t.base[L],
                                                 t.bstart.p + t.base[L], t.leaf_of.p);
    BEM_LAUNCH_CHECK();
    for (int l = L; l >= 1; --l) {
        int n = t.nb[l];
        k_flags_boxes<<<div_up(n, tb), tb, 0, st>>>(n, t.bkey.p + t.base[l], flag.p);
        BEM_LAUNCH_CHECK();
        exclusive_scan_i32(flag.p, ex.p, n, nullptr, st);
        k_emit_parents<<<div_up(n, tb), tb, 0, st>>>(n, t.bkey.p + t.base[l], t.bstart.p + t.base[l], flag.p, ex.p,
                                                      t.bkey.p + t.base[l - 1], t.bstart.p + t.base[l - 1],
                                                      t.parent.p + t.base[l], t.base[l - 1]);
        BEM_LAUNCH_CHECK();
    }
    BEM_CUDA(cudaMemsetAsync(t.parent.p, 0xff, t.nb[0] * sizeof(int32_t), st));  // roots have no parent
    for (int l = 0; l <= L; ++l) {
        int n = t.nb[l];
        k_box_counts<<<div_up(n, tb), tb, 0, st>>>(n, t.bstart.p + t.base[l], (int32_t)N, t.bcount.p + t.base[l]);
        BEM_LAUNCH_CHECK();
    }

    // 5. children of every box by octant, neighbours of every box, near-field lists at the leaf level
    t.child8.resize((size_t)t.nbox * 8);
    BEM_CUDA(cudaMemsetAsync(t.child8.p, 0xff, (size_t)t.nbox * 8 * sizeof(int32_t), st));
    k_child8<<<div_up(t.nbox - t.base[1], tb), tb, 0, st>>>(t.base[1], t.nbox, t.bkey.p, t.parent.p, t.child8.p);
    BEM_LAUNCH_CHECK();
    DevBuf<int32_t> &nb27 = t.s_i32[17];
    nb27.resize((size_t)t.nbox * 27);
    for (int l = 0; l <= L; ++l) {
        k_nb27<<<div_up((int64_t)t.nb[l] * 27, tb), tb, 0, st>>>(t.nb[l], t.base[l], t.bkey.p, t.parent.p, t.child8.p, nb27.p);
        BEM_LAUNCH_CHECK();
    }
    int nleaf = t.nb[L];
    t.nbr.resize((size_t)nleaf * 27);
    t.nbr_cnt.resize(nleaf);
    t.nbr_d.resize((size_t)nleaf * 27 * 4);
    DevBuf<unsigned long long> &pairs = t.s_u64[0];
    pairs.resize(1);
    BEM_CUDA(cudaMemsetAsync(pairs.p, 0, sizeof(unsigned long long), st));
    k_neighbours<<<div_up(nleaf, tb), tb, 0, st>>>(nleaf, t.base[L], nb27.p, t.bcount.p + t.base[L], t.nbr.p,
                                                    t.nbr_cnt.p, t.nbr_d.p, pairs.p);
    BEM_LAUNCH_CHECK();
    {
        DevBuf<int32_t> &ucnt = t.s_i32[4], &uoff = t.s_i32[5], &utot = t.s_i32[6];
        ucnt.resize(nleaf + 1);
        uoff.resize(nleaf + 1);
        utot.resize(2);  // units, 32-float blocks of shares
        k_p2p_unit_count<<<div_up(nleaf, tb), tb, 0, st>>>(nleaf, t.bcount.p + t.base[L], ucnt.p);
        BEM_LAUNCH_CHECK();
        exclusive_scan_i32(ucnt.p, uoff.p, nleaf, utot.p, st);
        // symmetric near field: per-leaf regions of the shares
        DevBuf<int32_t> &blk = t.s_i32[7], &blkoff = t.s_i32[8], &all = t.s_i32[22];
        blk.resize(nleaf + 1);
        blkoff.resize(nleaf + 1);
        all.resize(nleaf);
        t.back_S.resize(nleaf);
        t.back_base.resize(nleaf);
        t.back_gofs.resize((size_t)nleaf * 27);
        k_back_sizes<<<div_up(nleaf, tb), tb, 0, st>>>(nleaf, t.nbr.p, t.nbr_cnt.p, t.bcount.p + t.base[L], ucnt.p,
                                                        t.back_S.p, all.p, blk.p);
        BEM_LAUNCH_CHECK();
        exclusive_scan_i32(blk.p, blkoff.p, nleaf, utot.p + 1, st);
        k_back_base<<<div_up(nleaf, tb), tb, 0, st>>>(nleaf, blkoff.p, t.back_base.p);
        BEM_LAUNCH_CHECK();
        k_back_gofs<<<div_up((int64_t)nleaf * 27, tb), tb, 0, st>>>(nleaf, t.nbr.p, t.nbr_cnt.p, t.bcount.p + t.base[L],
                                                       t.back_gofs.p);
        BEM_LAUNCH_CHECK();
        int32_t tot2[2] = {0, 0};
        unsigned long long hpairs = 0;
        BEM_CUDA(cudaMemcpyAsync(tot2, utot.p, 2 * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
        BEM_CUDA(cudaMemcpyAsync(&hpairs, pairs.p, sizeof(hpairs), cudaMemcpyDeviceToHost, st));
        BEM_CUDA(cudaStreamSynchronize(st));
        const int64_t nu = tot2[0];
        t.p2p_pairs = (int64_t)hpairs;
        t.n_p2p_units = nu;
        t.p2p_units.resize(std::max<int64_t>(nu, 1));
        k_p2p_unit_emit<<<div_up(nleaf, tb), tb, 0, st>>>(nleaf, t.bcount.p + t.base[L], uoff.p, t.p2p_units.p);
        BEM_LAUNCH_CHECK();
        t.p2p_ucnt.resize(nleaf);
        BEM_CUDA(cudaMemcpyAsync(t.p2p_ucnt.p, ucnt.p, nleaf * sizeof(int32_t), cudaMemcpyDeviceToDevice, st));
        t.n_back = 32 * (int64_t)tot2[1];
        t.back.resize(std::max<int64_t>(t.n_back, 1));
        // Near-field items (one-way list: also FP64). The list length of an item: enough items for about six rounds of the warps that
        // the chip holds (24 per SM), so that the last round is a small part, but at least 64 and at
        // most 4096 positions (an item's set-up is about a quarter of a 64-source item's time, and
        // beyond 4096 nearly every unit is one item). Half the pairs in the symmetric list.
        const double per_item = (double)t.p2p_pairs / P2P_ITEM_RECV / ((double)c.num_sms * 24 * 6);
        DevBuf<int32_t> &icnt = t.s_i32[23], &iex = t.s_i32[18];
        icnt.resize(4 * nu + 1);
        iex.resize(4 * nu + 1);
        int chunk[2];
        const int32_t *len[2] = {t.back_S.p, all.p};
        for (int k = 0; k < 2; ++k) {
            const double want = k == 0 ? 0.5 * per_item : per_item;
            chunk[k] = std::min(4096, std::max(64, ((int)std::min(want, 1e6) + 31) / 32 * 32));
        }
        k_p2p_item_count<<<div_up(nu, tb), tb, 0, st>>>(nu, t.p2p_units.p, t.bcount.p + t.base[L], len[0], len[1], chunk[0],
                                                        chunk[1], icnt.p);
        BEM_LAUNCH_CHECK();
        exclusive_scan_i32(icnt.p, iex.p, 4 * nu + 1, nullptr, st);
        int32_t at[5];  // where each of the four lists begins, and the end
        BEM_CUDA(cudaMemcpy2DAsync(at, sizeof(int32_t), iex.p, nu * sizeof(int32_t), sizeof(int32_t), 5, cudaMemcpyDeviceToHost,
                                   st));
        BEM_CUDA(cudaStreamSynchronize(st));
        for (int k = 0; k < 2; ++k) {
            t.n_p2p_items[k] = at[k + 1] - at[k];
            t.n_p2p_rows[k] = at[k + 3] - at[k + 2];
            t.p2p_items[k].resize(std::max<int64_t>(t.n_p2p_items[k], 1));
            t.p2p_irow[k].resize(std::max<int64_t>(t.n_p2p_items[k], 1));
            t.p2p_ioff[k].resize(nu + 1);
            k_p2p_item_emit<<<div_up(nu, tb), tb, 0, st>>>(nu, t.p2p_units.p, t.bcount.p + t.base[L], len[k], chunk[k], iex.p,
                                                           k, t.p2p_ioff[k].p, t.p2p_items[k].p, t.p2p_irow[k].p);
            BEM_LAUNCH_CHECK();
        }
    }

    // 6. M2L pairs of levels 2..L: counted, then written target by target (m2l_tgt_off is their CSR)
    DevBuf<int32_t> &cnt = t.s_i32[9], &tot = t.s_i32[11];
    cnt.resize((size_t)t.nbox + 1);
    tot.resize(1);
    t.m2l_tgt_off.resize((size_t)t.nbox + 1);
    BEM_CUDA(cudaMemsetAsync(cnt.p, 0, ((size_t)t.nbox + 1) * sizeof(int32_t), st));
    const int first2 = t.base[2], lgrid = div_up(t.nbox - first2, 8);
    k_m2l_lists<<<lgrid, 256, 0, st>>>(first2, t.nbox, t.bkey.p, t.parent.p, nb27.p, t.child8.p, 0, cnt.p, nullptr, nullptr,
                                       nullptr, nullptr);
    BEM_LAUNCH_CHECK();
    exclusive_scan_i32(cnt.p, t.m2l_tgt_off.p, (int64_t)t.nbox + 1, tot.p, st);
    int32_t hm2l = 0;
    BEM_CUDA(cudaMemcpyAsync(&hm2l, tot.p, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    BEM_CUDA(cudaStreamSynchronize(st));
    const int64_t nm2l = hm2l;
    t.n_m2l = nm2l;
    DevBuf<int32_t> &ptgt = t.s_i32[12], &psrc = t.s_i32[13];
    DevBuf<uint32_t> &pcls = t.m2l_cls;  // sorted in place below: the class of every sorted pair
    ptgt.resize(nm2l);
    psrc.resize(nm2l);
    pcls.resize(std::max<int64_t>(nm2l, 1));
    t.m2l_src.resize(nm2l);
    t.m2l_tgt.resize(nm2l);
    t.m2l_by_tgt.resize(std::max<int64_t>(nm2l, 1));
    t.m2l_class_off.assign(kNumM2LClasses + 1, 0);
    if (nm2l > 0) {
        k_m2l_lists<<<lgrid, 256, 0, st>>>(first2, t.nbox, t.bkey.p, t.parent.p, nb27.p, t.child8.p, 1, nullptr,
                                           t.m2l_tgt_off.p, ptgt.p, psrc.p, pcls.p);
        BEM_LAUNCH_CHECK();
        // 7. sorted by offset class (stable: ascending target within a class). A target's pairs were
        // written by ascending class, so their places in the sorted order ascend as well.
        DevBuf<int32_t> &order = t.s_i32[14], &otmp = t.s_i32[15];
        DevBuf<uint32_t> &ctmp = t.s_u32[1];
        order.resize(nm2l);
        otmp.resize(nm2l);
        ctmp.resize(nm2l);
        DevBuf<int32_t> &hist = t.s_i32[16];
        hist.resize(kNumM2LClasses);
        BEM_CUDA(cudaMemsetAsync(hist.p, 0, kNumM2LClasses * sizeof(int32_t), st));
        k_class_hist<<<(unsigned)std::min<int64_t>(div_up(nm2l, 1024), 608), 256, 0, st>>>(nm2l, pcls.p, hist.p);
        BEM_LAUNCH_CHECK();
        k_iota<<<div_up(nm2l, tb), tb, 0, st>>>(nm2l, order.p);
        BEM_LAUNCH_CHECK();
        radix_sort_u32(pcls.p, order.p, nm2l, 9, ctmp.p, otmp.p, st);
        k_m2l_order<<<div_up(nm2l, tb), tb, 0, st>>>(nm2l, order.p, ptgt.p, psrc.p, t.m2l_tgt.p, t.m2l_src.p, t.m2l_by_tgt.p);
        BEM_LAUNCH_CHECK();
        std::vector<int32_t> hh(kNumM2LClasses);
        BEM_CUDA(cudaMemcpyAsync(hh.data(), hist.p, kNumM2LClasses * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
        BEM_CUDA(cudaStreamSynchronize(st));
        for (int k = 0; k < kNumM2LClasses; ++k) t.m2l_class_off[k + 1] = t.m2l_class_off[k] + hh[k];
    }

    // 8. sorted point data
    t.loc64.resize(3 * N);
    t.loc32.resize(3 * N);
    t.nrm64.resize(3 * N);
    t.nrm32.resize(3 * N);
    t.s_sorted.resize(N);
    t.ih.resize(N);
    k_sorted_points<<<div_up(N, tb), tb, 0, st>>>(N, L, t.deep, t.perm.p, t.key.p, c.xyz.p, c.nrm.p, c.s.p, cube.p,
                                                   clusters ? c.vcid.p : nullptr, t.loc64.p, t.loc32.p, t.nrm64.p,
                                                   t.nrm32.p, t.s_sorted.p, t.ih.p);
    BEM_LAUNCH_CHECK();
    BEM_CUDA(cudaStreamSynchronize(st));
}

}  // namespace bem
