// qw_tree.cu -- the locality order of the level bitmaps: a two-means tree over
// the data, built on the GPU.
//
// Each node of more than kGroupIds points is split in two: two centroids seeded
// by the points with the smallest and the largest projection on one LSH
// direction (the node's level mod m), three rounds of two-means, then the points
// ordered by their side of the bisecting hyperplane and cut where the side
// changes, rounded to a multiple of kGroupIds (the points nearest the
// hyperplane change sides), so that every 128-id group of the order lies
// inside one leaf of nearby points.  A node all of whose points fall on one
// side (copies of one point) is cut in the middle, and so is every node after
// kMaxUneven levels, which bounds the depth.  The order only decides which ids
// share a group: no result depends on it, only how many groups the bitmap path has
// to count.  FP32 sums serve where they are taken of what tells a node's points
// apart: every coordinate is read as its difference from the node's first point
// (exact to a rounding, so that an offset common to the data costs nothing), and a
// hyperplane's normal is divided by the largest component of the first one's (only
// the side and the order of distances count), so that no product leaves the range
// that the coordinates themselves fit.  Sums of a chunk's differences stay below FP32's
// largest number for coordinates up to about 1e33.
//
// All nodes of a level are split together.  A node's points are cut in chunks
// of whole blocks (256 rows, more for large nodes: at most kMaxChunks chunks
// per node); the kernels of a level work on chunks, those that combine a
// node's chunks (in chunk order: the tree is the same for every build) on
// nodes.  What bounds it is reading the rows five times a level: 17 ms at
// 1,000,000 x 128 (21 levels; 8.4 ms of it the side sums), against more than a
// second on 16 host cores in FP64, beside copying the data there.  The host
// only launches: it reads three counters per level.
#include "qw_internal.cuh"
#include "qw_scan.cuh"

#include <float.h>

#include <algorithm>

namespace qw {
namespace {

constexpr int TR_ROWS = 256;      // rows of a chunk's block, threads per block
constexpr int kMaxChunks = 608;   // per node: four per SM
constexpr int kMaxUneven = 48;    // levels before every cut goes through the middle
constexpr int kSmemSums = 24 * 1024;  // bytes of coordinate sums kept in shared memory

// Working memory of a build (device).
struct Tree {
    const float *X;
    const float *A;
    int64_t n;
    int d, m;
    int dv;                  // floats per row of v (d + 2, padded to 16 bytes)
    bool vec;                // rows in 16-byte pieces
    int32_t *perm, *perm2;   // the order, and the split nodes' next one
    float *t;                // signed distance to the node's hyperplane (times |v|)
    int32_t *lo, *hi, *c0;   // nodes of the level: range, first chunk
    int32_t *o;              // ... and data id of the first point
    int32_t *lo2, *hi2, *c02, *o2;
    int32_t *cut;            // per node, points of the first child
    int32_t *node, *node2;   // per chunk, its node
    float *v;                // per node, c2 - c1 scaled (d), the threshold, the scale
    float *part;             // per chunk, coordinate sums of both sides (2 d), of the
                             // differences from the node's first point
    int32_t *below;          // per chunk, points of the first side
    unsigned long long *kmin, *kmax;  // per chunk, smallest and largest (key, position)
    int32_t *ctl;            // next level: nodes, chunks, longest node
};

__host__ __device__ __forceinline__ int chunk_rows(int len)
{
    constexpr uint32_t most = TR_ROWS * kMaxChunks;
    return TR_ROWS * (int)(((uint32_t)len + most - 1) / most);
}

// Unsigned key in the order of a float.
__device__ __forceinline__ uint32_t fkey(float x)
{
    const uint32_t b = __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// Rows [b, e) of the chunk, and its node.
__device__ __forceinline__ void chunk_range(const Tree &T, int chunk, int &u, int &b, int &e)
{
    u = T.node[chunk];
    const int len = T.hi[u] - T.lo[u], cs = chunk_rows(len);
    b = T.lo[u] + (chunk - T.c0[u]) * cs;
    e = min(T.hi[u], b + cs);
}

// The node's first point: what its coordinates are taken relative to.
__device__ __forceinline__ const float *node_origin(const Tree &T, int u)
{
    return T.X + (int64_t)T.o[u] * T.d;
}

// f(position, (row - o) . w) for the rows at positions [b, e) of the order, a warp
// four rows at a time (their loads in flight together); every lane calls f.
template <class F>
__device__ __forceinline__ void rows_dot(const Tree &T, const float *__restrict__ w,
                                         const float *__restrict__ o, int b, int e, F &&f)
{
    constexpr int R = 4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, d = T.d;
    for (int j0 = b + warp * R; j0 < e; j0 += (TR_ROWS / 32) * R) {
        const float *x[R];
        float acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            x[r] = T.X + (int64_t)T.perm[min(j0 + r, e - 1)] * d;
            acc[r] = 0.0f;
        }
        if (T.vec) {
#pragma unroll 1  // (the rows' loads are in flight together; more registers cost blocks)
            for (int c = 4 * lane; c < d; c += 128) {
                const float4 y = *reinterpret_cast<const float4 *>(w + c);
                const float4 q = __ldg(reinterpret_cast<const float4 *>(o + c));
                float4 z[R];
#pragma unroll
                for (int r = 0; r < R; ++r) z[r] = __ldg(reinterpret_cast<const float4 *>(x[r] + c));
#pragma unroll
                for (int r = 0; r < R; ++r)
                    acc[r] = fmaf(z[r].x - q.x, y.x,
                                  fmaf(z[r].y - q.y, y.y,
                                       fmaf(z[r].z - q.z, y.z, fmaf(z[r].w - q.w, y.w, acc[r]))));
            }
        } else {
            for (int c = lane; c < d; c += 32) {
                const float y = w[c], q = __ldg(o + c);
#pragma unroll
                for (int r = 0; r < R; ++r) acc[r] = fmaf(__ldg(x[r] + c) - q, y, acc[r]);
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1)
                acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], off);
            if (j0 + r < e) f(j0 + r, acc[r]);
        }
    }
}

__global__ void tree_init_kernel(Tree T)
{
    const int64_t j0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t j = j0; j < T.n; j += (int64_t)gridDim.x * blockDim.x) T.perm[j] = (int32_t)j;
    if (j0 == 0) {
        T.lo[0] = 0;
        T.hi[0] = (int)T.n;
        T.c0[0] = 0;
        T.o[0] = 0;
    }
    const int cs = chunk_rows((int)T.n);
    if (j0 < ((int)T.n + cs - 1) / cs) T.node[j0] = 0;
}

// Per chunk, the positions of the smallest and largest projection on direction
// `dir` (ties: the first position).
__global__ void __launch_bounds__(TR_ROWS, 4) tree_seed_kernel(Tree T, int dir)
{
    __shared__ unsigned long long smin[TR_ROWS / 32], smax[TR_ROWS / 32];
    int u, b, e;
    chunk_range(T, blockIdx.x, u, b, e);
    unsigned long long mn = ~0ull, mx = 0ull;
    rows_dot(T, T.A + (int64_t)dir * T.d, node_origin(T, u), b, e, [&](int j, float t) {
        const unsigned long long k = (unsigned long long)fkey(t) << 32;
        mn = min(mn, k | (uint32_t)j);
        mx = max(mx, k | (0xffffffffu - (uint32_t)j));
    });
    if ((threadIdx.x & 31) == 0) {
        smin[threadIdx.x >> 5] = mn;
        smax[threadIdx.x >> 5] = mx;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < TR_ROWS / 32; ++w) {
            mn = min(mn, smin[w]);
            mx = max(mx, smax[w]);
        }
        T.kmin[blockIdx.x] = mn;
        T.kmax[blockIdx.x] = mx;
    }
}

// Block-wide sum (or largest) of one float per thread.
template <bool MAX>
__device__ __forceinline__ float block_reduce(float x, float *tmp)
{
    auto both = [](float a, float b) { return MAX ? fmaxf(a, b) : a + b; };
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) x = both(x, __shfl_xor_sync(0xffffffffu, x, off));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) tmp[threadIdx.x >> 5] = x;
    __syncthreads();
    float s = tmp[0];
    for (int w = 1; w < TR_ROWS / 32; ++w) s = both(s, tmp[w]);
    return s;
}

// Per node: the hyperplane between two centroids, v = c2 - c1 over the node's scale
// (the largest component between the seeds) and the threshold v . (c1 + c2) / 2, from
// the seeds (round 0) or from the sums of the chunks' sides.  A side without points
// leaves the hyperplane as it is.
__global__ void __launch_bounds__(TR_ROWS) tree_plane_kernel(Tree T, int n_chunks, int n_nodes,
                                                             bool seeds)
{
    __shared__ float tmp[TR_ROWS / 32];
    __shared__ unsigned long long s_mn, s_mx;
    __shared__ int s_below;
    const int u = blockIdx.x, d = T.d;
    const int k0 = T.c0[u], k1 = u + 1 < n_nodes ? T.c0[u + 1] : n_chunks;
    const int len = T.hi[u] - T.lo[u];
    float *v = T.v + (int64_t)u * T.dv;
    // the centroids, relative to the node's first point
    const float *x1 = nullptr, *x2 = nullptr, *o = node_origin(T, u);
    float r1 = 0.0f, r2 = 0.0f;
    if (seeds) {
        if (threadIdx.x == 0) {
            s_mn = ~0ull;
            s_mx = 0ull;
        }
        __syncthreads();
        for (int k = k0 + threadIdx.x; k < k1; k += TR_ROWS) {
            atomicMin(&s_mn, T.kmin[k]);
            atomicMax(&s_mx, T.kmax[k]);
        }
        __syncthreads();
        x1 = T.X + (int64_t)T.perm[(uint32_t)s_mn] * d;
        x2 = T.X + (int64_t)T.perm[0xffffffffu - (uint32_t)s_mx] * d;
    } else {
        if (threadIdx.x == 0) s_below = 0;
        __syncthreads();
        int mine = 0;
        for (int k = k0 + threadIdx.x; k < k1; k += TR_ROWS) mine += T.below[k];
        if (mine) atomicAdd(&s_below, mine);
        __syncthreads();
        const int n1 = s_below, n2 = len - n1;
        if (n1 == 0 || n2 == 0) return;
        r1 = 1.0f / (float)n1;
        r2 = 1.0f / (float)n2;
    }
    auto centroids = [&](int c, float &a, float &b) {
        if (seeds) {
            a = x1[c] - o[c];
            b = x2[c] - o[c];
        } else {
            a = b = 0.0f;
#pragma unroll 8
            for (int k = k0; k < k1; ++k) {
                a = fmaf(T.part[(int64_t)k * 2 * d + c], r1, a);
                b = fmaf(T.part[(int64_t)k * 2 * d + d + c], r2, b);
            }
        }
    };
    float most = seeds ? 0.0f : v[d + 1];
    if (seeds) {
        for (int c = threadIdx.x; c < d; c += TR_ROWS) most = fmaxf(most, fabsf(x2[c] - x1[c]));
        most = block_reduce<true>(most, tmp);
        if (threadIdx.x == 0) v[d + 1] = most;
    }
    float q = 0.0f;
    for (int c = threadIdx.x; c < d; c += TR_ROWS) {
        float a, b;
        centroids(c, a, b);
        const float w = most > 0.0f ? (b - a) / most : 0.0f;
        v[c] = w;
        q += w * (0.5f * a + 0.5f * b);
    }
    q = block_reduce<false>(q, tmp);
    if (threadIdx.x == 0) v[d] = q;
}

// Per chunk: each row's side of its node's hyperplane, and the coordinate sums
// of both sides.  A block takes 256 rows at a time: warps form the rows'
// projections, then threads own coordinates (256 / d threads share one, each a
// part of the rows) and add the rows, now in L1, side by side.  Held to five blocks
// per SM, 48 registers: 12.0 ms at 300,000 x 512.
__global__ void __launch_bounds__(TR_ROWS, 5) tree_assign_kernel(Tree T, bool in_smem)
{
    extern __shared__ float sums_s[];
    __shared__ uint8_t side[TR_ROWS];
    __shared__ int s_below;
    int u, b, e;
    chunk_range(T, blockIdx.x, u, b, e);
    const int d = T.d;
    const float *v = T.v + (int64_t)u * T.dv, *o = node_origin(T, u);
    const float thr = v[d];
    float *out = T.part + (int64_t)blockIdx.x * 2 * d;
    const int G = in_smem && d < TR_ROWS ? TR_ROWS / d : 1;   // threads per coordinate
    float *sums = in_smem ? sums_s : out;                // [group][side][coordinate]
    if (threadIdx.x == 0) s_below = 0;
    for (int c = threadIdx.x; c < G * 2 * d; c += TR_ROWS) sums[c] = 0.0f;
    __syncthreads();
    for (int r0 = b; r0 < e; r0 += TR_ROWS) {
        const int r1 = min(e, r0 + TR_ROWS);
        rows_dot(T, v, o, r0, r1, [&](int j, float t) {
            if ((threadIdx.x & 31) == 0) side[j - r0] = t < thr ? 0 : 1;
        });
        __syncthreads();
        const int n0 = __syncthreads_count((int)threadIdx.x < r1 - r0 && side[threadIdx.x] == 0);
        if (threadIdx.x == 0) s_below += n0;
        const int g = G > 1 ? threadIdx.x / d : 0;
        for (int c = G > 1 ? threadIdx.x % d : threadIdx.x; c < d && g < G; c += TR_ROWS) {
            float s0 = sums[g * 2 * d + c], s1 = sums[g * 2 * d + d + c];
            const float oc = __ldg(o + c);
#pragma unroll 8
            for (int j = r0 + g; j < r1; j += G) {
                const float x = __ldg(T.X + (int64_t)T.perm[j] * d + c) - oc;
                const bool second = side[j - r0] != 0;
                s0 += second ? 0.0f : x;
                s1 += second ? x : 0.0f;
            }
            sums[g * 2 * d + c] = s0;
            sums[g * 2 * d + d + c] = s1;
            if (G > 1) break;
        }
        __syncthreads();
    }
    if (in_smem)
        for (int c = threadIdx.x; c < 2 * d; c += TR_ROWS) {
            float s = sums[c];
            for (int g = 1; g < G; ++g) s += sums[g * 2 * d + c];
            out[c] = s;
        }
    if (threadIdx.x == 0) T.below[blockIdx.x] = s_below;
}

// Per chunk: the rows' signed distances and how many are below zero.
__global__ void __launch_bounds__(TR_ROWS, 4) tree_side_kernel(Tree T)
{
    __shared__ int s_below;
    int u, b, e;
    chunk_range(T, blockIdx.x, u, b, e);
    const float *v = T.v + (int64_t)u * T.dv;
    const float thr = v[T.d];
    if (threadIdx.x == 0) s_below = 0;
    __syncthreads();
    int mine = 0;
    rows_dot(T, v, node_origin(T, u), b, e, [&](int j, float t) {
        t -= thr;
        // keep an order where sums overflow
        if (!(fabsf(t) <= FLT_MAX)) t = t < 0.0f ? -FLT_MAX : FLT_MAX;
        if ((threadIdx.x & 31) == 0) T.t[j] = t;
        mine += t < 0.0f ? 1 : 0;
    });
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&s_below, mine);
    __syncthreads();
    if (threadIdx.x == 0) T.below[blockIdx.x] = s_below;
}

// Per node (one block): the cut, and the node's points written to perm2 with
// the first child's before the second's, each in their present order.  The
// points that change sides to reach the cut are the r = |cut - below| <= 128
// nearest to the hyperplane: every thread's nearest point of that side bounds
// them (the r-th smallest of the threads' minima has at least r points at or
// below it, and few more), so they are found among a short list instead of by
// sorting the node.
template <int NT>
__global__ void __launch_bounds__(NT) tree_split_kernel(Tree T, int n_chunks, int n_nodes,
                                                        bool even)
{
    constexpr int kList = 2048, E = 4;
    __shared__ uint32_t mins[NT];
    __shared__ uint32_t list[kList];
    __shared__ int hist[256];
    __shared__ int bc[4];
    __shared__ int tmp[NT / 32];
    __shared__ int s_below, s_n;
    const int u = blockIdx.x;
    const int lo = T.lo[u], len = T.hi[u] - lo;
    const int k0 = T.c0[u], k1 = u + 1 < n_nodes ? T.c0[u + 1] : n_chunks;
    if (threadIdx.x == 0) {
        s_below = 0;
        s_n = 0;
    }
    __syncthreads();
    int mine = 0;
    for (int k = k0 + threadIdx.x; k < k1; k += NT) mine += T.below[k];
    if (mine) atomicAdd(&s_below, mine);
    __syncthreads();
    const int below = s_below;
    const bool middle = even || below == 0 || below == len;
    const int last = (len - 1) / kGroupIds * kGroupIds;
    int cut = middle ? len / 2 : below;
    cut = (cut + kGroupIds / 2) / kGroupIds * kGroupIds;
    cut = max(kGroupIds, min(cut, last));
    const float *t = T.t + lo;
    // move: points with side 1 (grow) or side 0 whose |t| is below `bar`, and the
    // first `ties` of those at it
    const bool grow = cut > below;
    const int r = middle ? 0 : (grow ? cut - below : below - cut);
    uint32_t bar = 0;
    int ties = 0;
    if (r > 0) {
        auto key = [&](int j) {  // distance as ordered bits; ~0: not of the side that gives
            const float x = t[j];
            return (x < 0.0f) != grow ? __float_as_uint(fabsf(x)) : 0xffffffffu;
        };
        uint32_t mn = 0xffffffffu;
        for (int j = threadIdx.x; j < len; j += NT) mn = min(mn, key(j));
        mins[threadIdx.x] = mn;
        __syncthreads();
        // (fewer threads' minima than r: no bound)
        const uint32_t top = r <= NT ? block_kth_smallest<NT>(mins, NT, r, hist, bc) : 0xffffffffu;
        if (top != 0xffffffffu)
            for (int j = threadIdx.x; j < len; j += NT) {
                const uint32_t k = key(j);
                if (k <= top) {
                    const int p = atomicAdd(&s_n, 1);
                    if (p < kList) list[p] = k;
                }
            }
        __syncthreads();
        const int nl = s_n;
        auto all = [&](int j, uint32_t *k) {
            *k = key(j);
            return *k != 0xffffffffu;
        };
        bar = top != 0xffffffffu && nl <= kList ? block_kth_smallest<NT>(list, nl, r, hist, bc)
                                                : block_kth_smallest_if<NT>(len, r, all, hist, bc);
        // how many lie strictly below it
        __syncthreads();
        if (threadIdx.x == 0) s_n = 0;
        __syncthreads();
        int under = 0;
        for (int j = threadIdx.x; j < len; j += NT) under += key(j) < bar ? 1 : 0;
        if (under) atomicAdd(&s_n, under);
        __syncthreads();
        ties = r - s_n;
    }
    int32_t *out = T.perm2 + lo;
    const int32_t *in = T.perm + lo;
    int first = 0, tied = 0;  // points of the first child, ties so far
    for (int j0 = 0; j0 < len; j0 += NT * E) {
        bool f[E], tie[E];
        int nt = 0;
#pragma unroll
        for (int x = 0; x < E; ++x) {
            const int j = j0 + (int)threadIdx.x * E + x;
            f[x] = tie[x] = false;
            if (j < len) {
                if (middle) {
                    f[x] = j < cut;
                } else {
                    const float tj = t[j];
                    const bool neg = tj < 0.0f;
                    const uint32_t k = __float_as_uint(fabsf(tj));
                    const bool gives = r > 0 && neg != grow;
                    f[x] = neg != (gives && k < bar);
                    tie[x] = gives && k == bar;
                }
            }
            nt += tie[x] ? 1 : 0;
        }
        if (r > 0) {
            int tot;
            int at = tied + block_exclusive_scan<NT>(nt, tmp, &tot);
#pragma unroll
            for (int x = 0; x < E; ++x)
                if (tie[x]) f[x] = (at++ < ties) == grow;
            tied += tot;
        }
        int nf = 0;
#pragma unroll
        for (int x = 0; x < E; ++x) nf += f[x] ? 1 : 0;
        int tot;
        int at = first + block_exclusive_scan<NT>(nf, tmp, &tot);
#pragma unroll
        for (int x = 0; x < E; ++x) {
            const int j = j0 + (int)threadIdx.x * E + x;
            if (j < len) {
                // points of the second child before j: j minus those of the first
                out[f[x] ? at : cut + (j - at)] = in[j];
                at += f[x] ? 1 : 0;
            }
        }
        first += tot;
    }
    if (threadIdx.x == 0) T.cut[u] = cut;
}

// The next level's nodes (children of more than kGroupIds points) and chunks;
// one block, the nodes in order.
__global__ void __launch_bounds__(1024) tree_next_kernel(Tree T, int n_nodes)
{
    __shared__ int tmp[32];
    __shared__ int s_long;
    if (threadIdx.x == 0) s_long = 0;
    __syncthreads();
    int nodes = 0, chunks = 0;
    for (int u0 = 0; u0 < n_nodes; u0 += 1024) {
        const int u = u0 + (int)threadIdx.x;
        int lo[2] = {0, 0}, hi[2] = {0, 0}, nn = 0, nc = 0;
        if (u < n_nodes) {
            lo[0] = T.lo[u];
            hi[1] = T.hi[u];
            hi[0] = lo[1] = lo[0] + T.cut[u];
            for (int x = 0; x < 2; ++x) {
                const int len = hi[x] - lo[x];
                if (len <= kGroupIds) continue;
                ++nn;
                nc += (len + chunk_rows(len) - 1) / chunk_rows(len);
                atomicMax(&s_long, len);
            }
        }
        int tn, tc;
        int at = nodes + block_exclusive_scan<1024>(nn, tmp, &tn);
        int ct = chunks + block_exclusive_scan<1024>(nc, tmp, &tc);
        for (int x = 0; x < 2; ++x) {
            const int len = hi[x] - lo[x];
            if (len <= kGroupIds) continue;
            T.lo2[at] = lo[x];
            T.hi2[at] = hi[x];
            T.c02[at] = ct;
            T.o2[at] = T.perm[lo[x]];
            const int k = (len + chunk_rows(len) - 1) / chunk_rows(len);
            for (int y = 0; y < k; ++y) T.node2[ct + y] = at;
            ct += k;
            ++at;
        }
        nodes += tn;
        chunks += tc;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        T.ctl[0] = nodes;
        T.ctl[1] = chunks;
        T.ctl[2] = s_long;
    }
}

// The split nodes' order back into perm (points outside them keep their place).
__global__ void __launch_bounds__(TR_ROWS) tree_copy_kernel(Tree T)
{
    int u, b, e;
    chunk_range(T, blockIdx.x, u, b, e);
    for (int j = b + (int)threadIdx.x; j < e; j += TR_ROWS) T.perm[j] = T.perm2[j];
}

}  // namespace

qw_status locality_order(const float *X, int64_t n, int d, const float *A, int m, int32_t *perm,
                         cudaStream_t s)
{
    Tree T{};
    T.X = X;
    T.A = A;
    T.n = n;
    T.d = d;
    T.m = m;
    T.dv = (d + 5) / 4 * 4;
    T.vec = d % 4 == 0 && ((uintptr_t)X | (uintptr_t)A) % 16 == 0;
    // at most n / kGroupIds nodes a level (every node holds more than
    // kGroupIds points), and chunks for them
    const int64_t max_nodes = std::max<int64_t>(1, n / kGroupIds);
    const int64_t max_chunks = max_nodes + n / TR_ROWS + 1;
    const bool in_smem = (size_t)2 * std::max(d, TR_ROWS) * sizeof(float) <= kSmemSums;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t at = off;
        off += (bytes + 255) / 256 * 256;
        return at;
    };
    const size_t o_perm2 = take((size_t)n * 4), o_t = take((size_t)n * 4);
    const size_t o_node = take((size_t)max_chunks * 4), o_node2 = take((size_t)max_chunks * 4);
    size_t o_n[9];
    for (size_t &o : o_n) o = take((size_t)(max_nodes + 1) * 4);
    const size_t o_v = take((size_t)max_nodes * T.dv * 4);
    const size_t o_part = take((size_t)max_chunks * 2 * d * 4);
    const size_t o_below = take((size_t)max_chunks * 4);
    const size_t o_kmin = take((size_t)max_chunks * 8), o_kmax = take((size_t)max_chunks * 8);
    const size_t o_ctl = take(16);
    DevBuf mem;
    QW_TRY(mem.ensure(off));
    char *p = mem.as<char>();
    T.perm = perm;
    T.perm2 = reinterpret_cast<int32_t *>(p + o_perm2);
    T.t = reinterpret_cast<float *>(p + o_t);
    T.node = reinterpret_cast<int32_t *>(p + o_node);
    T.node2 = reinterpret_cast<int32_t *>(p + o_node2);
    int32_t **nodes[9] = {&T.lo, &T.hi, &T.c0, &T.o, &T.lo2, &T.hi2, &T.c02, &T.o2, &T.cut};
    for (int k = 0; k < 9; ++k) *nodes[k] = reinterpret_cast<int32_t *>(p + o_n[k]);
    T.v = reinterpret_cast<float *>(p + o_v);
    T.part = reinterpret_cast<float *>(p + o_part);
    T.below = reinterpret_cast<int32_t *>(p + o_below);
    T.kmin = reinterpret_cast<unsigned long long *>(p + o_kmin);
    T.kmax = reinterpret_cast<unsigned long long *>(p + o_kmax);
    T.ctl = reinterpret_cast<int32_t *>(p + o_ctl);

    tree_init_kernel<<<(unsigned)std::min<int64_t>((n + 255) / 256 + 3, 152 * 8), 256, 0, s>>>(T);
    QW_CUDA_TRY(cudaGetLastError());
    const int64_t cs = chunk_rows((int)n);
    // nodes, chunks, longest node of the level
    int32_t h[3] = {n > kGroupIds ? 1 : 0, (int32_t)((n + cs - 1) / cs), (int32_t)n};
    for (int level = 0; h[0] > 0; ++level) {
        const int nn = h[0], nc = h[1];
        const size_t smem =
            in_smem ? (size_t)2 * std::max(d, TR_ROWS / d * d) * sizeof(float) : 0;
        tree_seed_kernel<<<nc, TR_ROWS, 0, s>>>(T, level % m);
        tree_plane_kernel<<<nn, TR_ROWS, 0, s>>>(T, nc, nn, true);
        for (int it = 0; it < 3; ++it) {
            tree_assign_kernel<<<nc, TR_ROWS, smem, s>>>(T, in_smem);
            tree_plane_kernel<<<nn, TR_ROWS, 0, s>>>(T, nc, nn, false);
        }
        tree_side_kernel<<<nc, TR_ROWS, 0, s>>>(T);
        const bool even = level >= kMaxUneven;
        if (h[2] > 8192)
            tree_split_kernel<1024><<<nn, 1024, 0, s>>>(T, nc, nn, even);
        else
            tree_split_kernel<256><<<nn, 256, 0, s>>>(T, nc, nn, even);
        tree_copy_kernel<<<nc, TR_ROWS, 0, s>>>(T);
        tree_next_kernel<<<1, 1024, 0, s>>>(T, nn);
        QW_CUDA_TRY(cudaGetLastError());
        QW_CUDA_TRY(cudaMemcpyAsync(h, T.ctl, sizeof(h), cudaMemcpyDeviceToHost, s));
        QW_CUDA_TRY(cudaStreamSynchronize(s));
        std::swap(T.lo, T.lo2);
        std::swap(T.hi, T.hi2);
        std::swap(T.c0, T.c02);
        std::swap(T.o, T.o2);
        std::swap(T.node, T.node2);
    }
    QW_CUDA_TRY(cudaStreamSynchronize(s));  // mem is freed on return
    return QW_OK;
}

}  // namespace qw
