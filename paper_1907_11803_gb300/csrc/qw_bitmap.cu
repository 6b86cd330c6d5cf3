// qw_bitmap.cu -- the bitmap path of collision counting.
//
// The level path counts collisions by scanning the index entries of every
// projection's bucket range and incrementing one counter per entry: one
// shared-memory atomic per (entry, query), plus one counter byte per (id,
// query) kept in device memory between levels.  On workloads whose ranges are
// dense (a query's range holds a quarter of the ids of a projection) that is
// both atomic-bound and counter-traffic-bound.
//
// The bitmap path trades HBM capacity for that work.  At build time it stores,
// for every projection i, id tile t, level L (radius R = c^L, Section 2's
// virtual rehashing) and level-L bucket beta, the set of the tile's ids whose
// anchored bucket id satisfies floor(bid / R) == beta, as a bitmap of kTile
// bits (4 KiB).  A query collides with an object on projection i at radius R
// exactly when the object lies in the bucket beta_i = floor(g_i / R) of the
// query, so at every level the collision count of each id is the number of
// the m bitmaps B_i(beta_i) that contain it (Section 3.1).  Counts are summed
// bit-sliced (a carry-save adder tree keeps, per 32 ids, the seven bit planes
// of their counts in registers) and recomputed from scratch at every level:
// no atomics per entry and no counters kept between levels.
//
// Ids are numbered in a locality order (a two-means tree over the data, leaves
// of 128 ids; qw_tree.cu): a 128-id group holds nearby points.  Every bitmap carries a
// 256-bit summary (which groups it touches).  A group touched by fewer than l
// of the query's m buckets cannot hold a candidate, so a level runs in two
// passes: a filter on the summaries finds the live groups of every (query,
// tile), and only those are counted from the bitmaps.  Candidates go to a
// per-query list with their counts; the k + v bound and the tie rule (smallest
// original id) are applied per query at the end.  Results -- candidate sets,
// counts, statistics -- are those of the level path; a query whose candidates
// overflow the fixed lists is answered by the level path.
//
// Storage: per (projection, tile), sum over levels L of (span / c^L + 1)
// bitmaps, i.e. about (c / (c - 1)) * (span + 1) * 4 KiB, plus 32 bytes of
// summary each.  A level-L bitmap is the OR of its c children at level L - 1;
// the finest level comes from the data's bucket ids.
#include "qw_internal.cuh"
#include "qw_dir.cuh"
#include "qw_scan.cuh"
#include "qw_tma.cuh"

#include <algorithm>
#include <vector>

namespace qw {

qw_status bitmap_layout(const std::vector<int32_t> &span, int nT, int c, BitmapLayout *out)
{
    const int m = (int)span.size();
    out->base.assign(m, 0);
    out->nb.assign(m, 0);
    out->lvl.assign((size_t)m * kBmLevels, 0);
    out->J.assign(m, 0);
    int64_t total = 0;
    for (int i = 0; i < m; ++i) {
        int J = 0;
        int64_t R = 1;
        while (R <= (int64_t)span[i]) {
            R *= c;
            ++J;
        }
        if (J >= kBmLevels) {
            set_error("qw_build_index: too many levels for the bitmap table");
            return QW_ERR_RANGE;
        }
        int32_t acc = 0;
        R = 1;
        for (int L = 0; L <= J; ++L) {
            out->lvl[(size_t)i * kBmLevels + L] = acc;
            const int64_t nbk = (int64_t)span[i] / R + 1;
            if ((int64_t)acc + nbk > INT32_MAX) {
                set_error("qw_build_index: bitmap table too large");
                return QW_ERR_RANGE;
            }
            acc += (int32_t)nbk;
            R *= c;
        }
        out->J[i] = J;
        out->nb[i] = acc;
        out->base[i] = total;
        total += (int64_t)nT * acc;
    }
    out->total = total;
    return QW_OK;
}

namespace {

constexpr int BM_THREADS = kBmUint4;  // one thread per 16 bytes (128 ids) of a tile bitmap

// Level 0: bit j of bitmap (i, t, 0, bid) for every internal id j of tile t
// whose object has anchored bucket id bid on projection i, from the rows of
// ids in locality order, a 16-byte piece (16 / sizeof(T) projections) at a
// time.  A warp covers one 32-bit word (32 consecutive internal ids), and a
// word of a bucket belongs to that warp alone, so each bid's first lane stores
// it; the buffer is cleared first.  (Reading the projection-major ids through
// the order touched a line per id and projection: 720 us at 1,000,000 x 64
// projections, 394 us from the rows.)
template <typename T>
__global__ void __launch_bounds__(BM_THREADS) bm_fill_level0_kernel(IndexView ix, uint4 *bm)
{
    constexpr int P = 16 / (int)sizeof(T);
    const int t = blockIdx.x, i0 = blockIdx.y * P;
    const int len = (int)min((int64_t)kTile, ix.n - (int64_t)t * kTile);
    uint32_t *bw = reinterpret_cast<uint32_t *>(bm);
    const char *rows = static_cast<const char *>(ix.hloc) + (int64_t)t * kTile * ix.hloc_stride +
                       (int64_t)i0 * sizeof(T);
    const int lane = threadIdx.x & 31;
    const uint32_t below = (1u << lane) - 1u;
    __shared__ int64_t blk[P];
    if ((int)threadIdx.x < P && i0 + (int)threadIdx.x < ix.m) {
        const int i = i0 + threadIdx.x;
        blk[threadIdx.x] = ix.bm_base[i] + (int64_t)t * ix.bm_nb[i] + ix.bm_lvl[i * kBmLevels];
    }
    __syncthreads();
    for (int j = threadIdx.x; j - lane < len; j += BM_THREADS) {
        const bool valid = j < len;
        const uint4 v = valid ? __ldg(reinterpret_cast<const uint4 *>(
                                    rows + (int64_t)j * ix.hloc_stride))
                              : make_uint4(0, 0, 0, 0);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int u = 0; u < P; ++u) {
            if (i0 + u >= ix.m) break;
            const uint32_t word = w[u * (int)sizeof(T) / 4];
            const int sh = (u * (int)sizeof(T) % 4) * 8;
            const int64_t bid = valid ? (int64_t)(T)(word >> sh) : -1;
            const uint32_t same = __match_any_sync(0xffffffffu, (int32_t)bid);
            if (valid && (same & below) == 0)
                bw[(blk[u] + bid) * (kTile / 32) + (j >> 5)] = same;
        }
    }
}

// Row j of Xloc is data row perm[j]; inv is the inverse of perm.
__global__ void locality_copy_kernel(const float *__restrict__ X, const int32_t *__restrict__ perm,
                                     int64_t n, int d, float *__restrict__ Xloc,
                                     int32_t *__restrict__ inv)
{
    for (int64_t j = blockIdx.x; j < n; j += gridDim.x) {
        const int64_t src = perm[j];
        for (int c = threadIdx.x; c < d; c += blockDim.x) Xloc[j * d + c] = X[src * d + c];
        if (threadIdx.x == 0) inv[src] = (int32_t)j;
    }
}

// Per bitmap, one bit per 128-id group: the group has at least one id.  The
// summaries of one bucket over the tiles lie side by side (row bm_base[i] +
// k * nT + t for bitmap k of tile t's block of projection i), so that the
// filter reads four tiles of a bucket as one 128-byte line; nT zero rows at
// the end stand for buckets without data.
__global__ void __launch_bounds__(BM_THREADS) bm_summary_kernel(IndexView ix,
                                                                const uint4 *__restrict__ bm,
                                                                uint32_t *__restrict__ sum)
{
    const int t = blockIdx.x, i = blockIdx.y;
    const int nbk = ix.bm_nb[i];
    const int64_t b0 = ix.bm_base[i] + (int64_t)t * nbk;
    for (int k = 0; k < nbk; ++k) {
        const uint4 v = bm[(b0 + k) * kBmUint4 + threadIdx.x];
        const uint32_t word = __ballot_sync(0xffffffffu, (v.x | v.y | v.z | v.w) != 0);
        if ((threadIdx.x & 31) == 0)
            sum[(ix.bm_base[i] + (int64_t)k * ix.nT + t) * (kBmUint4 / 32) + (threadIdx.x >> 5)] =
                word;
    }
}

// Level L >= 1: bucket beta is the union of buckets c*beta .. c*beta + c - 1
// of level L - 1 (floor(floor(bid / R) / c) == floor(bid / (R c))).
__global__ void __launch_bounds__(BM_THREADS) bm_or_level_kernel(IndexView ix, uint4 *bm, int L,
                                                                 int64_t R, int c)
{
    const int t = blockIdx.x, i = blockIdx.y;
    if (L > ix.bm_J[i]) return;
    const int64_t sp = ix.span[i];
    const int64_t nbk = sp / R + 1;
    const int64_t nbk_child = sp / (R / c) + 1;
    const int64_t blk = ix.bm_base[i] + (int64_t)t * ix.bm_nb[i];
    const uint4 *child = bm + (blk + ix.bm_lvl[i * kBmLevels + L - 1]) * kBmUint4;
    uint4 *out = bm + (blk + ix.bm_lvl[i * kBmLevels + L]) * kBmUint4;
    for (int64_t beta = 0; beta < nbk; ++beta) {
        uint4 acc = make_uint4(0, 0, 0, 0);
        for (int u = 0; u < c; ++u) {
            const int64_t ch = beta * c + u;
            if (ch >= nbk_child) break;
            const uint4 x = child[ch * kBmUint4 + threadIdx.x];
            acc.x |= x.x;
            acc.y |= x.y;
            acc.z |= x.z;
            acc.w |= x.w;
        }
        out[beta * kBmUint4 + threadIdx.x] = acc;
    }
}


// Full adder on 32 lanes of bits: lo = a ^ b ^ c, hi = majority(a, b, c).
__device__ __forceinline__ void csa(uint32_t &hi, uint32_t &lo, uint32_t a, uint32_t b, uint32_t c)
{
    const uint32_t u = a ^ b;
    hi = (a & b) | (u & c);
    lo = u ^ c;
}

// Seven bit planes of the counts of 4 x 32 ids: bit k of the count of id
// (word w, bit b) is bit b of s[k][w].
struct Planes {
    uint32_t s[7][4];
};

// Add eight one-bit inputs per id (x[0..8)) to the planes.  Ones, twos and
// fours are carry-save; eights are a binary counter incremented by ripple.
__device__ __forceinline__ void add8(Planes &P, const uint4 (&x)[8])
{
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        uint32_t xs[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            xs[u] = w == 0 ? x[u].x : (w == 1 ? x[u].y : (w == 2 ? x[u].z : x[u].w));
        uint32_t t2a, t2b, t4a, t4b, t8;
        csa(t2a, P.s[0][w], P.s[0][w], xs[0], xs[1]);
        csa(t2b, P.s[0][w], P.s[0][w], xs[2], xs[3]);
        csa(t4a, P.s[1][w], P.s[1][w], t2a, t2b);
        csa(t2a, P.s[0][w], P.s[0][w], xs[4], xs[5]);
        csa(t2b, P.s[0][w], P.s[0][w], xs[6], xs[7]);
        csa(t4b, P.s[1][w], P.s[1][w], t2a, t2b);
        csa(t8, P.s[2][w], P.s[2][w], t4a, t4b);
        uint32_t cy = t8, nx;
        nx = P.s[3][w] & cy; P.s[3][w] ^= cy; cy = nx;
        nx = P.s[4][w] & cy; P.s[4][w] ^= cy; cy = nx;
        nx = P.s[5][w] & cy; P.s[5][w] ^= cy; cy = nx;
        P.s[6][w] ^= cy;  // counts stay below 128 (m <= 127)
    }
}


// Bits of word w whose count is >= l (l in 1..127).
__device__ __forceinline__ uint32_t count_ge_planes(const Planes &P, int w, int l)
{
    uint32_t gt = 0, eq = 0xffffffffu;
#pragma unroll
    for (int k = 6; k >= 0; --k) {
        const uint32_t sk = P.s[k][w];
        if ((l >> k) & 1) {
            eq &= sk;
        } else {
            gt |= eq & sk;
            eq &= ~sk;
        }
    }
    return gt | eq;
}

__device__ __forceinline__ int count_of(const Planes &P, int w, int b)
{
    int c = 0;
#pragma unroll
    for (int k = 0; k < 7; ++k) c |= (int)((P.s[k][w] >> b) & 1u) << k;
    return c;
}

__device__ __forceinline__ uint32_t word_of(const uint4 &v, int w)
{
    return w == 0 ? v.x : (w == 1 ? v.y : (w == 2 ? v.z : v.w));
}


// The candidate bits (count >= l) of the thread's 4 x 32 ids.
__device__ __forceinline__ uint4 candidates_of(const Planes &P, int l)
{
    uint4 cand;
    cand.x = count_ge_planes(P, 0, l);
    cand.y = count_ge_planes(P, 1, l);
    cand.z = count_ge_planes(P, 2, l);
    cand.w = count_ge_planes(P, 3, l);
    return cand;
}

// Bitmap number of the level-`level` bucket beta of projection i in tile t,
// or -1 when the bucket holds no data (beta below zero or past the span).
// Past the last stored level a single bucket (beta == 0) holds every id.
__device__ __forceinline__ int64_t bm_index(const IndexView &ix, int i, int t, int level,
                                            int64_t R, int64_t beta)
{
    const int J = ix.bm_J[i];
    int L = level;
    if (level > J) {
        if (beta != 0) return -1;
        L = J;
    } else if (beta < 0 || beta > (int64_t)ix.span[i] / R) {
        return -1;
    }
    return ix.bm_base[i] + (int64_t)t * ix.bm_nb[i] + ix.bm_lvl[i * kBmLevels + L] + beta;
}

// ---- the same level in two passes (the bitmap path's default)
//
// Pass 1 (bm_filter_kernel) reads only the bucket summaries (one bit per 128-id
// group): a bit-sliced sum over the m projections gives every group the number
// of the query's buckets that touch it, and the groups touched by at least l of
// them are live: no other can hold a candidate.  Each (query, tile)'s 256
// live bits are written (bm_amask) and their number summed over the level.
// Pass 2 counts the live groups from the bitmaps, in one of two forms chosen on
// the device from that number (both are launched, one returns at once):
//   bm_count_kernel, few queries per group: a warp takes one query's live
//     groups of four tiles, one per lane, and each lane reads the m words of its
//     group from the bitmaps;
//   bm_dense_kernel, many queries per group: a block keeps the words of every
//     bucket of a few groups in shared memory and counts them for every query
//     whose group is live.
// Both write the candidate word of a group with candidates (count >= l), add its
// candidates to the query's count, and clear the live bit of a group without:
// the bit then says that the group's word was written at this level.  Only a
// query's last level needs its candidates one by one, with their counts: they
// are listed after the loop (bm_list_kernel).
constexpr int FL_WARPS = 8;                   // warps per block in pass 1
constexpr int kSumWords = kBmUint4 / 32;      // summary words per bitmap (8)

// The dense form's table of one group: for every projection S rows of 16 bytes,
// the words of its buckets at the level, then zeros; S, a power of two, is above
// the most buckets of any projection, so row S - 1 is zero and stands for
// buckets without data.  A query names its rows in 4 bits each.
constexpr int kDenseTable = 66 * 1024;       // bytes of tables per block
constexpr int kDenseGroups = 16;             // most groups per block
constexpr int kDenseMin = 256;               // live groups per group of the index
constexpr int kDenseBlocks = 2 * 152;        // two per SM
constexpr int kDenseUnits = 200;             // fewest units (groups x query slices)

// Per level, in st.bm_ctl: [0] live groups, [1] the dense form's next unit,
// [2] S (0: more than 15 buckets), [3] groups per block, [4] queries that run.
enum { kCtlLive = 0, kCtlUnit = 1, kCtlRows = 2, kCtlGroups = 3, kCtlRun = 4 };

// The dense form's query slices, so that there are several units per block: slices
// of at least 1,024 of `run` queries.
__device__ __forceinline__ int dense_slices(int nT, int G, int run)
{
    const int chunks = nT * (kBmUint4 / G);
    return max(1, min((kDenseBlocks * 4 + chunks - 1) / chunks, (run + 1023) / 1024));
}

// The dense form pays when a group's table is read often enough (its words are
// loaded once per block instead of once per query) and its units fill the GPU: on a
// small index most blocks have none.  The lines lie where both forms take about the
// same time (live groups per group of the index: us count and dense).
//   1,000,000 points, 64 projections, S = 16: 135: 199 and 251, 175: 236 and 274,
//     295: 310 and 256, 386: 429 and 398, 689: 538 and 415, 1,969: 1,274 and 806;
//     S = 8: 125: 173 and 171, 256: 308 and 301, 539: 457 and 308; S = 4: 165: 385
//     and 118, 438: 534 and 258 (units 496 and more);
//   200,000 points, 48 projections, S = 16 and 448 units: 261: 64 and 55, 610: 106
//     and 84; S = 8 and 224 units: 262: 59 and 44; S = 4: 426 with 112 units 118 and
//     114, 1,186 with 224 224 and 160;
//   100,000 points, 64 projections, S = 4: 667 with 64 units 80 and 236, 774 with 128
//     111 and 160, 1,967 with 192 201 and 235, 2,338 with 256 291 and 231;
//   30,000 points, 40 projections, S = 4: 3,271 with 64 units 59 and 195; S = 8: 1,836
//     with 64 54 and 112, 5,504 with 192 88 and 114; S = 16: 5,501 with 384 86 and 84.
__device__ __forceinline__ bool dense_level(const IndexView &ix, const QueryState &st)
{
    const int S = (int)st.bm_ctl[kCtlRows], G = (int)st.bm_ctl[kCtlGroups];
    return S > 0 &&
           st.bm_ctl[kCtlLive] >= (uint32_t)kDenseMin * (uint32_t)ix.nT * kBmUint4 &&
           ix.nT * (kBmUint4 / G) * dense_slices(ix.nT, G, (int)st.bm_ctl[kCtlRun]) >= kDenseUnits;
}

// Buckets of projection i at a level (one past the last stored level).
__device__ __forceinline__ int buckets_at(const IndexView &ix, int i, int level, int64_t R)
{
    return level > ix.bm_J[i] ? 1 : (int)(floordiv64(ix.span[i], R) + 1);
}

// 16-byte words of a group's table (odd: the groups start in different banks).
__device__ __forceinline__ int table_words(int mp, int S) { return mp * S + 1; }

// The bucket of entry (query of the list at place e / bm_mp, projection e %
// bm_mp): its bitmap number at this level in tile 0 (tile t adds t * bm_nb[i];
// -1 when the bucket holds no data), its summary row (the zero rows then), and
// its row in the dense form's table (S - 1 then).  Rows are padded with empty
// buckets to multiples of 16 projections; eight lanes pack a word of table rows.
__device__ __forceinline__ void bucket_entry(const IndexView &ix, const QueryState &st, int level,
                                             int64_t R, int S, int64_t e)
{
    const int m = ix.m, mp = st.bm_mp;
    const int q = st.bm_run[e / mp], i = (int)(e % mp);
    const int64_t at = (int64_t)q * mp + i;
    int64_t b = -1;
    if (i < m) b = bm_index(ix, i, 0, level, R, floordiv64(st.g[(int64_t)q * m + i], R));
    st.bm_b0[at] = (int32_t)b;
    st.bm_srow[at] =
        (int32_t)(b >= 0 ? ix.bm_base[i] + (b - ix.bm_base[i]) * ix.nT : ix.bm_total);
    if (S == 0) return;
    uint32_t row = (uint32_t)S - 1u;
    if (b >= 0)
        row = (uint32_t)(b - ix.bm_base[i] - ix.bm_lvl[i * kBmLevels + min(level, ix.bm_J[i])]);
    row <<= 4 * (threadIdx.x & 7);
    const uint32_t mask = 0xffu << (threadIdx.x & 24);
#pragma unroll
    for (int off = 1; off < 8; off <<= 1) row |= __shfl_xor_sync(mask, row, off);
    if ((threadIdx.x & 7) == 0) st.bm_rows[at >> 3] = row;
}

// Before pass 1 (one block): the queries that run at this level, in order, and
// the level's counters: the passes walk this list and not the batch, most of
// which has stopped or not begun at most levels.  With `buckets` also their
// buckets (small batches: one launch less); else bm_bucket_kernel follows.
__global__ void __launch_bounds__(1024) bm_active_kernel(IndexView ix, int level, int64_t R, int nb,
                                                         QueryState st, const LoopCtl *ctl,
                                                         bool buckets)
{
    __shared__ int tmp[32];
    __shared__ int s_most;
    if (ctl) {
        level = ctl->level;
        R = ctl->R;
    }
    if (threadIdx.x == 0) s_most = 0;
    __syncthreads();
    if ((int)threadIdx.x < ix.m) atomicMax(&s_most, buckets_at(ix, threadIdx.x, level, R));
    constexpr int E = 8;
    int run = 0;
    for (int q0 = 0; q0 < nb; q0 += 1024 * E) {
        const int q1 = q0 + (int)threadIdx.x * E;
        int act[E], first[E];  // all of a thread's loads in flight
#pragma unroll
        for (int u = 0; u < E; ++u) {
            act[u] = q1 + u < nb ? st.active[q1 + u] : 0;
            first[u] = q1 + u < nb ? st.start[q1 + u] : 0;
        }
        uint32_t on = 0;
#pragma unroll
        for (int u = 0; u < E; ++u)
            if (act[u] && level >= first[u]) on |= 1u << u;
        int total;
        int at = run + block_exclusive_scan<1024>(__popc(on), tmp, &total);
#pragma unroll
        for (int u = 0; u < E; ++u)
            if ((on >> u) & 1u) st.bm_run[at++] = q1 + u;
        run += total;
    }
    __syncthreads();
    const int S = s_most < 4 ? 4 : (s_most < 8 ? 8 : (s_most < 16 ? 16 : 0));
    if (threadIdx.x == 0) {
        int G = kDenseGroups;
        while (G > 2 && table_words(st.bm_mp, S) * 16 * G > kDenseTable) G >>= 1;
        st.bm_ctl[kCtlLive] = 0;
        st.bm_ctl[kCtlUnit] = 0;
        st.bm_ctl[kCtlRows] = S;
        st.bm_ctl[kCtlGroups] = G;
        st.bm_ctl[kCtlRun] = run;
    }
    if (buckets)
        for (int64_t e = threadIdx.x; e < (int64_t)run * st.bm_mp; e += 1024)
            bucket_entry(ix, st, level, R, S, e);
}

__global__ void __launch_bounds__(256) bm_bucket_kernel(IndexView ix, int level, int64_t R,
                                                        QueryState st, const LoopCtl *ctl)
{
    if (ctl) {
        level = ctl->level;
        R = ctl->R;
    }
    const int S = (int)st.bm_ctl[kCtlRows];
    const int64_t total = (int64_t)st.bm_ctl[kCtlRun] * st.bm_mp;
    for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * 256)
        bucket_entry(ix, st, level, R, S, e);
}

// Eight one-bit inputs per lane bit added to one word's planes p[0..7).
__device__ __forceinline__ void add8_word(uint32_t (&p)[7], const uint32_t (&x)[8])
{
    uint32_t t2a, t2b, t4a, t4b, t8;
    csa(t2a, p[0], p[0], x[0], x[1]);
    csa(t2b, p[0], p[0], x[2], x[3]);
    csa(t4a, p[1], p[1], t2a, t2b);
    csa(t2a, p[0], p[0], x[4], x[5]);
    csa(t2b, p[0], p[0], x[6], x[7]);
    csa(t4b, p[1], p[1], t2a, t2b);
    csa(t8, p[2], p[2], t4a, t4b);
    uint32_t cy = t8, nx;
    nx = p[3] & cy; p[3] ^= cy; cy = nx;
    nx = p[4] & cy; p[4] ^= cy; cy = nx;
    nx = p[5] & cy; p[5] ^= cy; cy = nx;
    p[6] ^= cy;  // counts stay below 128
}

// One warp per (query, four tiles), tasks tile-major: the warps of a wave take
// the same tiles for many queries, whose summaries (and then bitmaps) serve all
// of them from L2.  Lane = (tile, summary word): the m summary words of a lane
// are summed bit-sliced, the four tiles of a bucket being one 128-byte line, and
// the compare gives the word's live groups.  Issue bound: about 6.5
// instructions per projection and four tiles.  (One warp per tile with a bit
// transpose of every word, for each group's own list of projections, issued
// about 30: 2,638 us per call on 3 million points and 10,000 queries; 584 so with
// the reads of 16 projections in flight, 545 with 32.)
__global__ void __launch_bounds__(FL_WARPS * 32) bm_filter_kernel(IndexView ix, int level, int l,
                                                                  QueryState st, const LoopCtl *ctl)
{
    if (ctl) level = ctl->level;
    const int lane = threadIdx.x & 31;
    const int nT = ix.nT, mp = st.bm_mp;
    const int par = level & 1;
    const int run = (int)st.bm_ctl[kCtlRun];
    const int64_t tasks = (int64_t)run * ((nT + 3) >> 2);
    uint32_t live = 0;
    unsigned long long items = 0, words = 0;
    for (int64_t k = (int64_t)blockIdx.x * FL_WARPS + (threadIdx.x >> 5); k < tasks;
         k += (int64_t)gridDim.x * FL_WARPS) {
        const int q = st.bm_run[k % run], t0 = (int)(k / run) * 4;
        const int t = t0 + (lane >> 3);
        // lanes past the last tile read its row again
        const int in_row = (min(t, nT - 1) - t0) * kSumWords + (lane & 7);
        const int4 *rows = reinterpret_cast<const int4 *>(st.bm_srow + (int64_t)q * mp);
        const uint32_t *sum = ix.bm_sum + (int64_t)t0 * kSumWords + in_row;
        uint32_t P[7] = {0, 0, 0, 0, 0, 0, 0};
#pragma unroll 4
        for (int i = 0; i < mp; i += 8) {
            const int4 ra = __ldg(rows + (i >> 2)), rb = __ldg(rows + (i >> 2) + 1);
            const int32_t r[8] = {ra.x, ra.y, ra.z, ra.w, rb.x, rb.y, rb.z, rb.w};
            uint32_t x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = __ldg(sum + (int64_t)r[u] * kSumWords);
            add8_word(P, x);
        }
        uint32_t gt = 0, eq = 0xffffffffu;
#pragma unroll
        for (int b = 6; b >= 0; --b) {
            if ((l >> b) & 1) {
                eq &= P[b];
            } else {
                gt |= eq & P[b];
                eq &= ~P[b];
            }
        }
        const uint32_t alive = t < nT ? gt | eq : 0u;
        if (t < nT)
            st.bm_amask[((int64_t)par * st.cln_par + (int64_t)q * nT + t0) * kSumWords + lane] = alive;
        live += __popc(alive);
        if (st.bm_prof) {
            // tiles with live groups; words of the buckets touching live groups
            const uint32_t any = __ballot_sync(0xffffffffu, alive != 0);
#pragma unroll
            for (int u = 0; u < 4; ++u) items += (any >> (8 * u)) & 0xffu ? 1 : 0;
#pragma unroll
            for (int b = 0; b < 7; ++b) words += (unsigned)__popc(alive & P[b]) << b;
        }
    }
    live = __reduce_add_sync(0xffffffffu, live);
    if (lane == 0 && live) atomicAdd(st.bm_ctl + kCtlLive, live);
    if (st.bm_prof) {
        words = __reduce_add_sync(0xffffffffu, (unsigned)words);
        if (lane == 0 && live) {
            atomicAdd(st.bm_prof + 0, items);
            atomicAdd(st.bm_prof + 1, (unsigned long long)live);
            atomicAdd(st.bm_prof + 2, words);
        }
    }
}

// What follows the count of a group with nc > 0 candidates.
__device__ __forceinline__ void emit_group(const QueryState &st, int nT, int level, int q, int t,
                                           int g, const uint4 &cand, int nc)
{
    const int64_t qt = (int64_t)q * nT + t;
    st.cbits[(int64_t)(level & 1) * st.cb_par + qt * kBmUint4 + g] = cand;
    atomicAdd(st.qbuf_n + (int64_t)(level & 1) * st.qbn_par + q, nc);
}

// Position of the n-th (0-based) set bit of v; n < popc(v).
__device__ __forceinline__ int nth_set_bit(uint32_t v, int n)
{
    int pos = 0;
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) {
        const int c = __popc(v & ((1u << w) - 1u));
        if (n >= c) {
            n -= c;
            v >>= w;
            pos += w;
        }
    }
    return pos;
}

// Bit transpose of a 32 x 32 block held one row per lane (bit b of lane i's
// word is element (i, b)): returns column `lane`, whose bit i is element
// (i, lane).  Five butterfly steps, each exchanging the off-diagonal halves
// of the blocks of that size.
__device__ __forceinline__ uint32_t transpose32(uint32_t a, int lane)
{
    const uint32_t keep[5] = {0x0000ffffu, 0x00ff00ffu, 0x0f0f0f0fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        const int j = 16 >> s;
        const uint32_t y = __shfl_xor_sync(0xffffffffu, a, j);
        a = (lane & j) ? (a & ~keep[s]) | ((y >> j) & keep[s])
                       : (a & keep[s]) | ((y << j) & ~keep[s]);
    }
    return a;
}

// The set bits of a warp's 32 words x (one per lane), 32 at a time: f(owner,
// bit, valid) per lane for the entries in order (lanes past the last repeat it,
// not valid).  With at most 8 of them in all, four lanes take each entry: f's
// last argument is then the lane's share (0..3 of 4), else 0 of 1, and lane
// share 0 is the valid one.
template <class F>
__device__ __forceinline__ void each_set_bit(uint32_t x, int lane, F &&f)
{
    int incl = __popc(x);
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += y;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    const bool four = total <= 8;
    for (int r0 = 0; r0 < total; r0 += 32) {
        // the (r0 + lane)-th set bit: the first word whose prefix passes it
        const int e = min(four ? lane >> 2 : r0 + lane, total - 1);
        int own = 0;
#pragma unroll
        for (int step = 16; step > 0; step >>= 1) {
            const int v = __shfl_sync(0xffffffffu, incl, own + step - 1);
            if (e >= v) own += step;
        }
        const uint32_t xw = __shfl_sync(0xffffffffu, x, own);
        const int before = __shfl_sync(0xffffffffu, incl, own) - __popc(xw);
        f(own, nth_set_bit(xw, e - before),
          four ? (lane >> 2) < total && (lane & 3) == 0 : r0 + lane < total, four);
    }
}

// Add the planes of another lane (lane ^ off) to this one's.
__device__ __forceinline__ void add_lane(Planes &P, int off)
{
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        uint32_t cy = 0;
#pragma unroll
        for (int k = 0; k < 7; ++k) {
            const uint32_t o = __shfl_xor_sync(0xffffffffu, P.s[k][w], off);
            csa(cy, P.s[k][w], P.s[k][w], o, cy);
        }
    }
}

// Count planes of group g of tile t from the m bitmaps whose numbers in tile 0
// are b0[0..m) (-1: no data; tile t adds t * nbs[i]), rows padded to 8.  With
// `four` (uniform over the warp) the four lanes of a quad have the same group and
// each reads every fourth run of eight projections: a quarter of the dependent
// rounds of loads where the warp's other lanes would idle.
__device__ __forceinline__ void count_planes(const IndexView &ix, const int32_t *b0,
                                             const int *nbs, int t, int g, Planes &P,
                                             bool four = false)
{
#pragma unroll
    for (int kk = 0; kk < 7; ++kk)
#pragma unroll
        for (int w = 0; w < 4; ++w) P.s[kk][w] = 0;
    const int4 *b4 = reinterpret_cast<const int4 *>(b0);
    const int step = four ? 32 : 8;
    for (int i0 = four ? 8 * (threadIdx.x & 3) : 0; i0 < ix.m; i0 += step) {
        const int4 ba = __ldg(b4 + (i0 >> 2)), bb = __ldg(b4 + (i0 >> 2) + 1);
        const int32_t bn[8] = {ba.x, ba.y, ba.z, ba.w, bb.x, bb.y, bb.z, bb.w};
        uint4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            v[u] = bn[u] >= 0
                       ? __ldg(ix.bm + ((int64_t)bn[u] + (int64_t)t * nbs[i0 + u]) * kBmUint4 + g)
                       : make_uint4(0, 0, 0, 0);
        add8(P, v);
    }
    if (four) {
        add_lane(P, 1);
        add_lane(P, 2);
    }
}

constexpr int kCountWarps = 152 * 3 * 8;  // resident at once, of blocks that count groups

// The bits of every word that part p of `parts` (a power of two up to 32) takes.
__device__ __forceinline__ uint32_t part_bits(int p, int parts)
{
    const int bits = 32 / parts;
    return (0xffffffffu >> (32 - bits)) << (bits * p);
}

// Few queries per group.  A warp takes the live bits of one query's four tiles
// (a word per lane), and its lanes the set bits, 32 at a time: a lane reads its
// group's word of each of the query's m bitmaps and sums them into bit planes.
// Bound by the latency of those 16-byte reads (about 20 sectors a request): see
// bm_dense_kernel for levels where many queries share a group.
// Where the queries that run give the resident warps less than a task each, a task is
// cut in up to 32 parts (equal runs of bits of every word): most groups are live
// where the data has few clusters or a query lies far from them, and 1,024 groups
// in one warp are 32 rounds of reads one after the other.  One query on 1,000,000
// points of one Gaussian, 64 dimensions, a whole call: 1,054 us with whole tasks,
// 400 so; 16 queries 1,634 and 711.
__global__ void __launch_bounds__(256, 3) bm_count_kernel(IndexView ix, int level, int l,
                                                          QueryState st, const LoopCtl *ctl)
{
    __shared__ int s_nb[QW_MAX_M + 16];
    __shared__ uint32_t s_keep[8][32];
    __shared__ int s_whole, s_parts;
    if (dense_level(ix, st)) return;
    if (ctl) level = ctl->level;
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const int m = ix.m, nT = ix.nT, mp = st.bm_mp;
    for (int i = threadIdx.x; i < mp; i += 256) s_nb[i] = i < m ? ix.bm_nb[i] : 0;
    if (threadIdx.x == 0) {
        const int whole = (int)st.bm_ctl[kCtlRun] * ((nT + 3) >> 2);  // (at most 2^23)
        int parts = 1;
        while (parts < 32 && whole * parts * 2 <= kCountWarps) parts *= 2;
        s_whole = whole;
        s_parts = parts;
    }
    __syncthreads();
    const int run = (int)st.bm_ctl[kCtlRun];
    for (int k = blockIdx.x * 8 + wi; k < s_whole * s_parts; k += gridDim.x * 8) {
        const int task = k % s_whole;
        const int q = st.bm_run[task % run], t0 = task / run * 4;
        uint32_t *am = st.bm_amask +
                       ((int64_t)(level & 1) * st.cln_par + (int64_t)q * nT + t0) * kSumWords + lane;
        uint32_t x = t0 + (lane >> 3) < nT ? *am : 0u;
        if (s_parts > 1) x &= part_bits(k / s_whole, s_parts);
        if (!__any_sync(0xffffffffu, x != 0)) continue;
        s_keep[wi][lane] = x;
        __syncwarp();
        each_set_bit(x, lane, [&](int own, int bit, bool valid, bool four) {
            const int t = t0 + (own >> 3), g = (own & 7) * 32 + bit;
            Planes P;
            count_planes(ix, st.bm_b0 + (int64_t)q * mp, s_nb, t, g, P, four);
            const uint4 cand = candidates_of(P, l);
            const int nc = __popc(cand.x) + __popc(cand.y) + __popc(cand.z) + __popc(cand.w);
            if (valid) {
                if (nc == 0) atomicAnd(&s_keep[wi][own], ~(1u << bit));
                else emit_group(st, nT, level, q, t, g, cand, nc);
            }
        });
        __syncwarp();
        const uint32_t keep = s_keep[wi][lane];
        if (keep != x) {
            if (s_parts == 1) *am = keep;
            else atomicAnd(am, keep | ~x);  // (the other bits are other warps')
        }
        __syncwarp();
    }
}

// Many queries per group.  A unit is (G groups of a tile, a slice of the queries
// that run); blocks take units from a counter.  A block loads the tables of the
// G groups (every bucket's word of every projection, so any query's count is m
// shared reads), then goes over its queries 8,192 at a time: the queries' live
// bits become one bit row per group; warps take pieces of the rows from a
// counter, and each set bit is an entry (group, query) of the warp's queue,
// counted 32 at a time, one per lane.  Nearly all of a warp's lanes then read
// the same group: for a projection, rows of one bucket list, consecutive 16-byte
// words, so quarter-warps meet no bank twice unless two of their queries are
// eight buckets apart.  Groups with candidates set a bit in a second set of
// rows, and the live bits of the others are cleared at the end.
//
// Bound by logic operations (35 per 16 projections and 32 ids, at 64 lanes a
// clock) and by shared memory (4 clocks per warp and projection).  41 million live
// (query, group) pairs on 3 million points: 2.4 ms, 3.6 by one lane per pair
// reading the bitmaps.  Two blocks per SM
// cover each other's loads, queue ends and barriers; with one block of whole
// rows dealt to the warps, three quarters of their time went into waiting for
// the warp with the busiest group.
constexpr int DN_THREADS = 256;
constexpr int DN_WARPS = DN_THREADS / 32;
constexpr int kDenseQ = 8192;   // queries of a segment
constexpr int kDensePiece = 16; // 32-query words of a row a warp takes at a time

struct DenseShared {
    uint32_t live[kDenseGroups][kDenseQ / 32];  // [group][query / 32]
    uint32_t some[kDenseGroups][kDenseQ / 32];  // ... with candidates
    uint32_t queue[DN_WARPS][64];         // group of the unit << 16 | place in the segment
    int nbk[QW_MAX_M];
    int64_t base[QW_MAX_M];               // first bitmap of the level in the tile
    int unit, next;
};

size_t dense_smem_bytes() { return kDenseTable + sizeof(DenseShared); }

// Sixteen one-bit inputs per id of the four words: two carry-save halves, then
// one carry into the planes of 16, 32 and 64.
__device__ __forceinline__ void add16_half(Planes &P, const uint4 (&x)[8], uint32_t (&t8)[4])
{
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        uint32_t t2a, t2b, t4a, t4b;
        csa(t2a, P.s[0][w], P.s[0][w], word_of(x[0], w), word_of(x[1], w));
        csa(t2b, P.s[0][w], P.s[0][w], word_of(x[2], w), word_of(x[3], w));
        csa(t4a, P.s[1][w], P.s[1][w], t2a, t2b);
        csa(t2a, P.s[0][w], P.s[0][w], word_of(x[4], w), word_of(x[5], w));
        csa(t2b, P.s[0][w], P.s[0][w], word_of(x[6], w), word_of(x[7], w));
        csa(t4b, P.s[1][w], P.s[1][w], t2a, t2b);
        csa(t8[w], P.s[2][w], P.s[2][w], t4a, t4b);
    }
}

// Count group g of tile t for query q, both the lane's own (every lane of the
// warp; lanes that are not valid write nothing), from the group's table.  Sets
// `bit` of *row when the group has a candidate.
template <int S>
__device__ __forceinline__ void dense_count(const IndexView &ix, const QueryState &st, int level,
                                            int l, const unsigned char *tab, int q, bool valid,
                                            int t, int g, uint32_t *row, int bit)
{
    const int mp = st.bm_mp;
    // 16 projections: two words of eight 4-bit rows
    const uint2 *rows = reinterpret_cast<const uint2 *>(st.bm_rows + (int64_t)q * (mp >> 3));
    Planes P;
#pragma unroll
    for (int kk = 0; kk < 7; ++kk)
#pragma unroll
        for (int w = 0; w < 4; ++w) P.s[kk][w] = 0;
    auto sixteen = [&](uint2 r, const unsigned char *tb) {
        uint32_t ta[4], tc[4];
        uint4 x[8];
        auto take = [&](uint32_t v, const unsigned char *at) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const uint32_t o = u == 0 ? (v << 4) & 0xf0u : (v >> (4 * u - 4)) & 0xf0u;
                x[u] = *reinterpret_cast<const uint4 *>(at + u * S * 16 + o);
            }
        };
        take(r.x, tb);
        add16_half(P, x, ta);
        take(r.y, tb + 8 * S * 16);
        add16_half(P, x, tc);
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            uint32_t cy;
            csa(cy, P.s[3][w], P.s[3][w], ta[w], tc[w]);
            uint32_t nx = P.s[4][w] & cy;
            P.s[4][w] ^= cy;
            cy = nx;
            nx = P.s[5][w] & cy;
            P.s[5][w] ^= cy;
            P.s[6][w] ^= nx;
        }
    };
    uint2 next = __ldg(rows);
    for (int i = 0; i < mp; i += 16) {
        const uint2 r = next;
        if (i + 16 < mp) next = __ldg(rows + (i >> 4) + 1);
        sixteen(r, tab + i * S * 16);
    }
    const uint4 cand = candidates_of(P, l);
    const int nc = __popc(cand.x) + __popc(cand.y) + __popc(cand.z) + __popc(cand.w);
    if (!valid || nc == 0) return;
    atomicOr(row, 1u << bit);
    emit_group(st, ix.nT, level, q, t, g, cand, nc);
}

__global__ void __launch_bounds__(DN_THREADS, 2) bm_dense_kernel(IndexView ix, int level, int64_t R,
                                                                 int l, QueryState st,
                                                                 const LoopCtl *ctl)
{
    extern __shared__ __align__(16) unsigned char dsm[];
    if (!dense_level(ix, st)) return;
    unsigned char *table = dsm;
    DenseShared &sh = *reinterpret_cast<DenseShared *>(dsm + kDenseTable);
    if (ctl) {
        level = ctl->level;
        R = ctl->R;
    }
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const int m = ix.m, nT = ix.nT, mp = st.bm_mp;
    const int nb = (int)st.bm_ctl[kCtlRun];  // queries that run
    const int S = (int)st.bm_ctl[kCtlRows], G = (int)st.bm_ctl[kCtlGroups];
    const int words = table_words(mp, S);
    const int per_tile = kBmUint4 / G;
    const int chunks = nT * per_tile;
    const int slices = dense_slices(nT, G, nb);
    const int per_slice = ((nb + slices - 1) / slices + 31) & ~31;
    uint32_t *amask = st.bm_amask + (int64_t)(level & 1) * st.cln_par * kSumWords;
    for (int i = threadIdx.x; i < m; i += DN_THREADS) sh.nbk[i] = buckets_at(ix, i, level, R);
    for (;;) {
        __syncthreads();  // the table and the rows of the previous unit are done with
        if (threadIdx.x == 0) sh.unit = (int)atomicAdd(st.bm_ctl + kCtlUnit, 1u);
        __syncthreads();
        const int unit = sh.unit;
        if (unit >= chunks * slices) break;
        // slices of one chunk one after the other: its bitmap words are in L2
        const int chunk = unit / slices, slice = unit % slices;
        const int t = chunk / per_tile, g0 = chunk % per_tile * G;
        const int w = g0 >> 5, sh0 = g0 & 31;
        for (int i = threadIdx.x; i < m; i += DN_THREADS)
            sh.base[i] = ix.bm_base[i] + (int64_t)t * ix.bm_nb[i] +
                         ix.bm_lvl[i * kBmLevels + min(level, ix.bm_J[i])];
        __syncthreads();
        // the tables: entries (projection, bucket, group), buckets past a
        // projection's (and projections past m) zero
#pragma unroll 4
        for (int e = threadIdx.x; e < mp * S * G; e += DN_THREADS) {
            const int g = e % G, b = e / G % S, i = e / (G * S);
            uint4 v = make_uint4(0, 0, 0, 0);
            if (i < m && b < sh.nbk[i]) v = __ldg(ix.bm + (sh.base[i] + b) * kBmUint4 + g0 + g);
            *reinterpret_cast<uint4 *>(table + ((size_t)g * words + i * S + b) * 16) = v;
        }
        const int q_end = min(nb, (slice + 1) * per_slice);
        for (int s0 = slice * per_slice; s0 < q_end; s0 += kDenseQ) {
            const int s1 = min(q_end, s0 + kDenseQ);
            const int nblk = (s1 - s0 + 31) >> 5;
            // live words (lane = query) -> rows (lane = group)
#pragma unroll 4
            for (int b = wi; b < nblk; b += DN_WARPS) {
                const int at = s0 + b * 32 + lane;
                const uint32_t x =
                    at < s1 ? amask[((int64_t)st.bm_run[at] * nT + t) * kSumWords + w] >> sh0 : 0u;
                uint32_t row = 0;
#pragma unroll
                for (int g = 0; g < kDenseGroups; ++g) {
                    const uint32_t y = __ballot_sync(0xffffffffu, (x >> g) & 1u);
                    row = lane == g ? y : row;
                }
                if (lane < G) {
                    sh.live[lane][b] = row;
                    sh.some[lane][b] = 0;
                }
            }
            if (threadIdx.x == 0) sh.next = 0;
            __syncthreads();
            const int pieces = (nblk + kDensePiece - 1) / kDensePiece;
            int held = 0;
            auto count32 = [&](uint32_t e, bool valid) {
                const int gl = (int)(e >> 16), ql = (int)(e & 0xffffu);
                const int q = st.bm_run[s0 + ql];
                const unsigned char *tab = table + (size_t)gl * words * 16;
                uint32_t *row = &sh.some[gl][ql >> 5];
                if (S == 4) dense_count<4>(ix, st, level, l, tab, q, valid, t, g0 + gl, row, ql & 31);
                else if (S == 8) dense_count<8>(ix, st, level, l, tab, q, valid, t, g0 + gl, row, ql & 31);
                else dense_count<16>(ix, st, level, l, tab, q, valid, t, g0 + gl, row, ql & 31);
            };
            for (;;) {
                int u = 0;
                if (lane == 0) u = atomicAdd(&sh.next, 1);
                u = __shfl_sync(0xffffffffu, u, 0);
                if (u >= G * pieces) break;
                const int gl = u / pieces, piece = u % pieces;
                const int b0 = piece * kDensePiece, b1 = min(nblk, b0 + kDensePiece);
                // the piece's words in the lanes
                const uint32_t xs = b0 + lane < b1 && lane < kDensePiece ? sh.live[gl][b0 + lane] : 0u;
                uint32_t full = __ballot_sync(0xffffffffu, xs != 0);
                while (full) {
                    const int o = __ffs(full) - 1;
                    full &= full - 1;
                    const uint32_t x = __shfl_sync(0xffffffffu, xs, o);
                    if ((x >> lane) & 1u)
                        sh.queue[wi][held + __popc(x & ((1u << lane) - 1u))] =
                            (uint32_t)gl << 16 | (uint32_t)((b0 + o) * 32 + lane);
                    held += __popc(x);
                    __syncwarp();
                    if (held >= 32) {
                        const uint32_t e = sh.queue[wi][lane];
                        const uint32_t rest = sh.queue[wi][32 + lane];
                        __syncwarp();
                        sh.queue[wi][lane] = rest;
                        held -= 32;
                        __syncwarp();
                        count32(e, true);
                    }
                }
            }
            if (held > 0) count32(sh.queue[wi][min(lane, held - 1)], lane < held);
            __syncthreads();
            // clear the live bits of groups without candidates
#pragma unroll 2
            for (int b = wi; b < nblk; b += DN_WARPS) {
                const int at = s0 + b * 32 + lane;
                const uint32_t none =
                    lane < G ? sh.live[lane][b] & ~sh.some[lane][b] : 0u;
                uint32_t gone = 0;
#pragma unroll
                for (int g = 0; g < kDenseGroups; ++g)
                    gone |= ((__shfl_sync(0xffffffffu, none, g) >> lane) & 1u) << g;
                if (at < s1 && gone)
                    atomicAnd(&amask[((int64_t)st.bm_run[at] * nT + t) * kSumWords + w],
                              ~(gone << sh0));
            }
            __syncthreads();
        }
    }
}

// ---- the same level in one pass (filter and count fused)
//
// One warp per (query, run of FL_TILES tiles), as in pass 1 above: the bucket
// summaries give every 128-id group the set of the query's buckets touching
// it, and the groups touched by at least l buckets are live.  The same warp
// then counts its live groups, 32 at a time (lane k takes the k-th live group
// of the tile): the m bitmap numbers of the tile stay in the lanes' registers
// (lane j holds projections j and j + 32) and are broadcast by shuffles, so a
// group's m word loads depend on nothing but its own projection mask, which
// the filter step left in shared memory.  Results (candidate words and counts, profile counters)
// are those of the two passes; every live group's bit stays set and its word is
// written.
constexpr int FL_TILES = 8;  // tiles per warp unless the caller picks 4 or 16

template <int NROW>
__device__ __forceinline__ void load_summaries(const IndexView &ix, const int32_t (&srow)[NROW],
                                               int t, uint4 (&sv)[NROW][2])
{
#pragma unroll
    for (int r = 0; r < NROW; ++r) {
        const uint4 *p =
            reinterpret_cast<const uint4 *>(ix.bm_sum + ((int64_t)srow[r] + t) * kSumWords);
        sv[r][0] = __ldg(p);
        sv[r][1] = __ldg(p + 1);
    }
}

template <int NROW, int TPW>
__global__ void __launch_bounds__(FL_WARPS * 32, 2) bm_fused_kernel(IndexView ix, int level,
                                                                   int l, int nb, QueryState st,
                                                                   const LoopCtl *ctl)
{
    constexpr int MW = (NROW + 1) / 2;
    __shared__ unsigned long long wmk[FL_WARPS][kSumWords][MW][32];
    __shared__ uint32_t wlive[FL_WARPS][kSumWords];
    if (ctl) level = ctl->level;
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const int m = ix.m, nT = ix.nT;
    const int nch = (nT + TPW - 1) / TPW;
    const int64_t tasks = (int64_t)nb * nch;
    const int par = level & 1;
    unsigned long long p_items = 0, p_groups = 0, p_words = 0;
    for (int64_t k = (int64_t)blockIdx.x * FL_WARPS + wi; k < tasks;
         k += (int64_t)gridDim.x * FL_WARPS) {
        // tile-major: the warps of a wave take one run of tiles for many
        // queries, so the bitmaps they touch (and the count pass after them)
        // stay in L2 across queries
        const int q = (int)(k % nb);
        const int t0 = (int)(k / nb) * TPW, t1 = min(nT, t0 + TPW);
        if (!st.active[q] || level < st.start[q]) continue;
        int64_t b0[NROW];
        int32_t nbp[NROW], srow[NROW];
#pragma unroll
        for (int r = 0; r < NROW; ++r) {
            const int i = lane + 32 * r;
            b0[r] = i < m ? st.bm_b0[(int64_t)q * st.bm_mp + i] : -1;
            srow[r] = i < m ? st.bm_srow[(int64_t)q * st.bm_mp + i] : (int32_t)ix.bm_total;
            nbp[r] = i < m ? ix.bm_nb[i] : 0;
        }
        uint4 sv[NROW][2];
        load_summaries<NROW>(ix, srow, t0, sv);
        for (int t = t0; t < t1; ++t) {
            const int64_t qt = (int64_t)q * nT + t;
            int n_alive = 0;
#pragma unroll
            for (int w = 0; w < kSumWords; ++w) {
                int cnt = 0;
                unsigned long long mk[MW];
#pragma unroll
                for (int h = 0; h < MW; ++h) mk[h] = 0ull;
#pragma unroll
                for (int r = 0; r < NROW; ++r) {
                    const uint32_t c = transpose32(word_of(sv[r][w >> 2], w & 3), lane);
                    cnt += __popc(c);
                    mk[r >> 1] |= (unsigned long long)c << (32 * (r & 1));
                }
#pragma unroll
                for (int h = 0; h < MW; ++h) wmk[wi][w][h][lane] = mk[h];
                const uint32_t xw = __ballot_sync(0xffffffffu, cnt >= l);
                if (lane == 0) wlive[wi][w] = xw;
                n_alive += __popc(xw);
            }
            __syncwarp();
            // the next tile's summaries load while this tile is counted
            if (t + 1 < t1) load_summaries<NROW>(ix, srow, t + 1, sv);
            if (lane < kSumWords)
                st.bm_amask[((int64_t)par * st.cln_par + qt) * kSumWords + lane] = wlive[wi][lane];
            if (n_alive == 0) continue;
            // this tile's bitmap numbers, one per lane and row
            int64_t bt[NROW];
#pragma unroll
            for (int r = 0; r < NROW; ++r) bt[r] = b0[r] >= 0 ? b0[r] + (int64_t)t * nbp[r] : -1;
            for (int base = 0; base < n_alive; base += 32) {
                // the (base + lane)-th live group of the tile
                const int kk = base + lane;
                int g = -1;
                {
                    int acc = 0;
#pragma unroll
                    for (int w = 0; w < kSumWords; ++w) {
                        const uint32_t xw = wlive[wi][w];
                        const int c = __popc(xw);
                        if (g < 0 && kk < acc + c) g = w * 32 + nth_set_bit(xw, kk - acc);
                        acc += c;
                    }
                }
                unsigned long long mk[MW];
#pragma unroll
                for (int h = 0; h < MW; ++h)
                    mk[h] = g >= 0 ? wmk[wi][g >> 5][h][g & 31] : 0ull;
                Planes P;
#pragma unroll
                for (int kq = 0; kq < 7; ++kq)
#pragma unroll
                    for (int w = 0; w < 4; ++w) P.s[kq][w] = 0;
                int words = 0;
#pragma unroll
                for (int h = 0; h < MW; ++h) words += __popcll(mk[h]);
                for (int i0 = 0; i0 < m; i0 += 8) {
                    uint4 xv[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int i = i0 + u;
                        const int r = i >> 5;
                        int64_t bn = 0;
#pragma unroll
                        for (int rr = 0; rr < NROW; ++rr)
                            if (rr == r) bn = __shfl_sync(0xffffffffu, bt[rr], i & 31);
                        const bool on = i < m && ((mk[i >> 6] >> (i & 63)) & 1ull);
                        xv[u] = on ? __ldg(ix.bm + bn * kBmUint4 + g) : make_uint4(0, 0, 0, 0);
                    }
                    add8(P, xv);
                }
                uint4 cand = make_uint4(0, 0, 0, 0);
                int nc = 0;
                if (g >= 0) {
                    cand = candidates_of(P, l);
                    st.cbits[(int64_t)par * st.cb_par + qt * kBmUint4 + g] = cand;
                    nc = __popc(cand.x) + __popc(cand.y) + __popc(cand.z) + __popc(cand.w);
                    p_words += (unsigned long long)words;
                }
                const int tot = __reduce_add_sync(0xffffffffu, nc);
                if (lane == 0 && tot) atomicAdd(st.qbuf_n + (int64_t)par * st.qbn_par + q, tot);
            }
            p_items += 1;
            p_groups += (unsigned long long)n_alive;
        }
    }
    if (st.bm_prof) {
        p_words = __reduce_add_sync(0xffffffffu, (unsigned)p_words);
        if (lane == 0 && (p_items || p_words)) {
            atomicAdd(st.bm_prof + 0, p_items);
            atomicAdd(st.bm_prof + 1, p_groups);
            atomicAdd(st.bm_prof + 2, p_words);
        }
    }
}

// ---- the same level with the bitmaps staged by TMA
//
// One persistent CTA per SM walks the (query, tile) items of the batch,
// item k = blockIdx.x + j * gridDim.x (consecutive queries are in signature
// order, so the CTAs working at one time share most bitmaps in L2).  A
// producer warp streams stages of 8 bitmaps into a ring in shared memory: its
// lanes compute the 64 bitmap addresses of an item in parallel (bucket ids of
// the next item prefetched a step ahead), lane 0 issues one 4 KiB bulk copy
// per present bitmap and writes a small header per stage (item, which
// bitmaps are present, first / last stage of the item, end of work).  Eight
// consumer warps follow the stage stream: each adds a stage into its bit
// planes straight from shared memory and, at an item's last stage, writes the
// item's candidate words, their group bits (a warp holds one word of them) and
// count.  Consumers never wait on a global load for control flow.
constexpr int kRing = 6;
constexpr int kPerStage = 8;                       // bitmaps per stage
constexpr int kStageBytesBm = kPerStage * kTile / 8;  // 32 KiB
constexpr int TMA_CONSUMERS = BM_THREADS;          // 8 warps, one 16-byte word each
constexpr int TMA_THREADS = TMA_CONSUMERS + 32;    // + the producer warp
constexpr uint32_t kFirstStage = 1, kLastStage = 2, kDone = 4;

struct StageHdr {
    int32_t q, t;
    uint32_t mask;   // which of the stage's bitmaps are present
    uint32_t flags;  // kFirstStage | kLastStage | kDone
};

struct TmaShared {
    uint64_t full[kRing];
    uint64_t empty[kRing];
    StageHdr hdr[kRing];
    int64_t pt[QW_MAX_M + 8];      // bitmap numbers of the current item (-1: empty)
    int64_t lbase[QW_MAX_M];       // per projection: bm_base + bm_lvl[min(level, J)]
    int32_t nbk[QW_MAX_M];         // per projection: buckets at this level (0: past J)
    int32_t pnb[QW_MAX_M];         // per projection: bitmaps per tile
};

size_t tma_smem_bytes() { return sizeof(TmaShared) + 128 + (size_t)kRing * kStageBytesBm; }

__global__ void __launch_bounds__(TMA_THREADS, 1) bm_level_tma_kernel(IndexView ix, int level,
                                                                      int64_t R, int l, int nb,
                                                                      QueryState st,
                                                                      const LoopCtl *ctl, int *err)
{
    extern __shared__ __align__(128) unsigned char smraw[];
    TmaShared &sh = *reinterpret_cast<TmaShared *>(smraw);
    unsigned char *ring = smraw + ((sizeof(TmaShared) + 127) / 128) * 128;
    if (ctl) {
        level = ctl->level;
        R = ctl->R;
    }
    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const int m = ix.m, nT = ix.nT;
    const int nst = (m + kPerStage - 1) / kPerStage;  // stages per item
    const int64_t items = (int64_t)nb * nT;
    if (tid == 0) {
        for (int k = 0; k < kRing; ++k) {
            mbar_init(&sh.full[k], 1);
            mbar_init(&sh.empty[k], TMA_CONSUMERS / 32);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = tid; i < m; i += TMA_THREADS) {
        const int J = ix.bm_J[i];
        const int L = level > J ? J : level;
        sh.lbase[i] = ix.bm_base[i] + ix.bm_lvl[i * kBmLevels + L];
        sh.nbk[i] = level > J ? 0 : (int32_t)((int64_t)ix.span[i] / R + 1);
        sh.pnb[i] = ix.bm_nb[i];
    }
    __syncthreads();
    bool stuck = false;
    if (warp == TMA_CONSUMERS / 32) {
        // ---- producer warp
        constexpr int kPL = (QW_MAX_M + 31) / 32;  // projections per lane
        uint32_t it = 0;
        int64_t k = blockIdx.x;
        int64_t gn[kPL];
        int act_n = 0, start_n = 0;
        auto prefetch = [&](int64_t kk) {
            if (kk >= items) return;
            const int qq = (int)(kk % nb);
            act_n = st.active[qq];
            start_n = st.start[qq];
#pragma unroll
            for (int u = 0; u < kPL; ++u) {
                const int i = lane + 32 * u;
                gn[u] = i < m ? st.g[(int64_t)qq * m + i] : 0;
            }
        };
        prefetch(k);
        for (; k < items && !stuck; k += gridDim.x) {
            // tile-major item order (one tile's bitmaps serve many queries in L2)
            const int q = (int)(k % nb), t = (int)(k / nb);
            int64_t g[kPL];
#pragma unroll
            for (int u = 0; u < kPL; ++u) g[u] = gn[u];
            const bool runs = act_n && level >= start_n;
            prefetch(k + gridDim.x);  // in flight while this item is issued
            if (!runs) continue;
#pragma unroll
            for (int u = 0; u < kPL; ++u) {
                const int i = lane + 32 * u;
                if (i < m) {
                    const int64_t beta = floordiv64(g[u], R);
                    const int nbk = sh.nbk[i];
                    // past the last stored level one bucket (beta == 0) holds every id
                    const bool present = nbk == 0 ? beta == 0 : (beta >= 0 && beta < nbk);
                    sh.pt[i] = present ? sh.lbase[i] + (int64_t)t * sh.pnb[i] + (nbk ? beta : 0)
                                       : -1;
                }
            }
            __syncwarp();
            if (lane == 0) {
                for (int j = 0; j < nst && !stuck; ++j, ++it) {
                    const int slot = (int)(it % kRing);
                    if (it >= (uint32_t)kRing)
                        mbar_wait(&sh.empty[slot], ((it / kRing) - 1) & 1, err, stuck);
                    if (stuck) break;
                    uint32_t mask = 0;
#pragma unroll
                    for (int u = 0; u < kPerStage; ++u) {
                        const int i = j * kPerStage + u;
                        if (i < m && sh.pt[i] >= 0) mask |= 1u << u;
                    }
                    StageHdr &h = sh.hdr[slot];
                    h.q = q;
                    h.t = t;
                    h.mask = mask;
                    h.flags = (j == 0 ? kFirstStage : 0u) | (j == nst - 1 ? kLastStage : 0u);
                    mbar_arrive_expect_tx(&sh.full[slot], (uint32_t)__popc(mask) * (kTile / 8));
#pragma unroll
                    for (int u = 0; u < kPerStage; ++u)
                        if ((mask >> u) & 1u)
                            bulk_g2s(ring + (size_t)slot * kStageBytesBm + (size_t)u * (kTile / 8),
                                     ix.bm + sh.pt[j * kPerStage + u] * kBmUint4, kTile / 8,
                                     &sh.full[slot]);
                }
            }
            stuck = __shfl_sync(0xffffffffu, stuck, 0);
            __syncwarp();
        }
        if (lane == 0) {
            if (!stuck) {
                // end of work
                const int slot = (int)(it % kRing);
                if (it >= (uint32_t)kRing)
                    mbar_wait(&sh.empty[slot], ((it / kRing) - 1) & 1, err, stuck);
                if (!stuck) {
                    sh.hdr[slot].flags = kDone;
                    sh.hdr[slot].mask = 0;
                    mbar_arrive_expect_tx(&sh.full[slot], 0);
                    ++it;
                }
            }
            if (stuck) {
                // no bulk copy may still be writing shared memory at exit
                for (uint32_t d = 0; d < (uint32_t)kRing && d < it; ++d) {
                    const uint32_t jt = it - 1 - d;
                    bool again = false;
                    mbar_wait(&sh.full[jt % kRing], (jt / kRing) & 1, err, again);
                }
            }
        }
        return;
    }
    // ---- consumers: thread tid owns 16-byte word tid (128 ids) of every bitmap
    uint32_t it = 0;
    Planes P;
    for (;; ++it) {
        const int slot = (int)(it % kRing);
        mbar_wait(&sh.full[slot], (it / kRing) & 1, err, stuck);
        if (stuck) break;
        const StageHdr h = sh.hdr[slot];
        if (h.flags & kDone) break;
        const int64_t qt = (int64_t)h.q * nT + h.t;
        if (h.flags & kFirstStage) {
#pragma unroll
            for (int kk = 0; kk < 7; ++kk)
#pragma unroll
                for (int w = 0; w < 4; ++w) P.s[kk][w] = 0;
        }
        const uint4 *stage = reinterpret_cast<const uint4 *>(ring + (size_t)slot * kStageBytesBm);
        uint4 x[kPerStage];
#pragma unroll
        for (int u = 0; u < kPerStage; ++u)
            x[u] = ((h.mask >> u) & 1u) ? stage[u * kBmUint4 + tid] : make_uint4(0, 0, 0, 0);
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.empty[slot]);
        add8(P, x);
        if (!(h.flags & kLastStage)) continue;
        // ---- the item's epilogue (consumers only: the producer does not take part)
        const uint4 cand = candidates_of(P, l);
        const int nc = __popc(cand.x) + __popc(cand.y) + __popc(cand.z) + __popc(cand.w);
        if (nc) st.cbits[(int64_t)(level & 1) * st.cb_par + qt * kBmUint4 + tid] = cand;
        const uint32_t some = __ballot_sync(0xffffffffu, nc != 0);
        const int tot = __reduce_add_sync(0xffffffffu, nc);
        if (lane == 0) {
            st.bm_amask[((int64_t)(level & 1) * st.cln_par + qt) * kSumWords + warp] = some;
            if (tot) atomicAdd(st.qbuf_n + (int64_t)(level & 1) * st.qbn_par + h.q, tot);
        }
    }
}

// ---- the candidates of the queries' last levels
//
// bm_final_bucket_kernel: the bitmap numbers of every query's buckets at its
// last level (the two-pass and fused levels leave them in bm_b0).
__global__ void bm_final_bucket_kernel(IndexView ix, int nb, QueryState st)
{
    const int m = ix.m, mp = st.bm_mp;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < (int64_t)nb * mp;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int q = (int)(e / mp), i = (int)(e % mp);
        const int L = st.levels[q] - 1;
        const int64_t R = st.finalR[q];
        st.bm_b0[e] = L >= 0 && i < m ? (int32_t)bm_index(ix, i, 0, L, R,
                                                          floordiv64(st.g[(int64_t)q * m + i], R))
                                      : -1;
    }
}

// Append this thread's candidates (128 ids, ascending) to the query's list
// from position pos: (internal id << 32) | (prev << 8) | count.
__device__ __forceinline__ void append_candidates(const Planes &P, const uint4 &cand,
                                                  const uint4 &prev, uint64_t *list, int pos,
                                                  int64_t id_base)
{
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        uint32_t x = word_of(cand, w);
        const uint32_t pw = word_of(prev, w);
        while (x) {
            const int b = __ffs(x) - 1;
            x &= x - 1;
            if (pos < kQCap)
                list[pos] = ((uint64_t)(id_base + w * 32 + b) << 32) |
                            ((uint64_t)((pw >> b) & 1u) << 8) | (uint64_t)count_of(P, w, b);
            ++pos;
        }
    }
}

// The candidate word of group g of a (query, tile) at level L (zero where the
// level wrote none).
__device__ __forceinline__ uint4 rd_word(const QueryState &st, int L, int64_t qt, int g)
{
    const int64_t pc = (int64_t)(L & 1) * st.cln_par + qt;
    if (!((st.bm_amask[pc * kSumWords + (g >> 5)] >> (g & 31)) & 1u)) return make_uint4(0, 0, 0, 0);
    return st.cbits[(int64_t)(L & 1) * st.cb_par + qt * kBmUint4 + g];
}

// Lists the last level's candidates of every query that has at most kQCap of
// them and no slot of the list rebuild below: the counts of its groups with candidates once more from the bitmaps
// (few of the groups counted on the way there), and whether each was a candidate
// of the previous level (its word there, if the query ran it).  A warp takes
// four tiles of a query, as bm_count_kernel does, or one of `parts` parts of their
// groups where the query has more than kListPart candidates, or where they are more
// than 32 and there are warps to spare (else part 0 takes them all).  Listing during the levels
// instead, every candidate of every level behind a returning atomic, took most
// of the count pass where candidates are many (606 queries whose last level
// takes in all 300,000 points: 2.3 ms of a level of 0.17).
constexpr int kListPart = 2048;

__global__ void __launch_bounds__(256, 3) bm_list_kernel(IndexView ix, int l, int nb, int parts,
                                                          bool spare, QueryState st)
{
    __shared__ int s_nb[QW_MAX_M + 16];
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const int m = ix.m, nT = ix.nT, mp = st.bm_mp;
    for (int i = threadIdx.x; i < mp; i += 256) s_nb[i] = i < m ? ix.bm_nb[i] : 0;
    __syncthreads();
    const int tasks = nb * ((nT + 3) >> 2) * parts;
    for (int k = blockIdx.x * 8 + wi; k < tasks; k += gridDim.x * 8) {
        const int q = k % nb, t0 = k / nb / parts * 4, part = k / nb % parts;
        const int L = st.levels[q] - 1;
        if (L < 0) continue;
        const int n = st.qbuf_n[(int64_t)(L & 1) * st.qbn_par + q];
        if (n == 0 || n > kQCap || (st.bm_ovf[q] & 8)) continue;
        const bool ran_prev = L > st.start[q];
        uint32_t x =
            t0 + (lane >> 3) < nT
                ? st.bm_amask[((int64_t)(L & 1) * st.cln_par + (int64_t)q * nT + t0) * kSumWords + lane]
                : 0u;
        if (parts > 1) {
            if (n > kListPart || (spare && __reduce_add_sync(0xffffffffu, __popc(x)) > 32))
                x &= part_bits(part, parts);
            else if (part)
                continue;
        }
        if (!__any_sync(0xffffffffu, x != 0)) continue;
        uint64_t *list = st.qbuf + (int64_t)q * kQCap;
        each_set_bit(x, lane, [&](int own, int bit, bool valid, bool four) {
            const int t = t0 + (own >> 3), g = (own & 7) * 32 + bit;
            const int64_t qt = (int64_t)q * nT + t;
            const uint4 prev = ran_prev ? rd_word(st, L - 1, qt, g) : make_uint4(0, 0, 0, 0);
            Planes P;
            count_planes(ix, st.bm_b0 + (int64_t)q * mp, s_nb, t, g, P, four);
            const uint4 cand = candidates_of(P, l);
            int nc = __popc(cand.x) + __popc(cand.y) + __popc(cand.z) + __popc(cand.w);
            if (!valid) nc = 0;
            int incl = nc;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += y;
            }
            int pos = 0;
            if (lane == 31 && incl) pos = atomicAdd(st.cross + q, incl);
            pos = __shfl_sync(0xffffffffu, pos, 31);
            if (nc)
                append_candidates(P, cand, prev, list, pos + incl - nc,
                                  (int64_t)t * kTile + (int64_t)g * 128);
        });
    }
}
// Sort keys[0..n) ascending in shared memory (n padded to P2 with ~0).
__device__ __forceinline__ void smem_bitonic(uint64_t *keys, int n, int P2)
{
    for (int i = n + (int)threadIdx.x; i < P2; i += blockDim.x) keys[i] = ~0ull;
    __syncthreads();
    for (int kk = 2; kk <= P2; kk <<= 1) {
        for (int jj = kk >> 1; jj > 0; jj >>= 1) {
            for (int x = threadIdx.x; x < (P2 >> 1); x += blockDim.x) {
                const int a = 2 * x - (x & (jj - 1));
                const int c = a + jj;
                const bool up = (a & kk) == 0;
                if ((keys[a] > keys[c]) == up) {
                    const uint64_t tmp = keys[a];
                    keys[a] = keys[c];
                    keys[c] = tmp;
                }
            }
            __syncthreads();
        }
    }
}

// The k + v bound on the bitmap path, one block per query, from the list of
// its last level's candidates: the boundary count c* and how many ids at c*
// are kept follow from the counts exactly as on the level path (Section 3.1,
// readings R4/R5); candidates of the previous level and those above c* are
// kept, and of those at c* the ones with the smallest original ids (radix
// selection of the take-th smallest id of the tie class).  The kept list is
// written with its counts in no particular order, or in ascending original id
// when `sorted`, plus the per-query statistics.  A tie class longer than its
// list (kEqCap ids) is selected from the candidate list itself.  A query whose
// candidate list overflowed keeps nothing here and is marked (bm_ovf); the
// list rebuild below shortens its list and this selection runs again on it (a
// query whose rebuilt list would still overflow goes to the level path).
constexpr int SEL_THREADS = 256;
constexpr int SEL_U = 4;  // list entries in flight per thread
static_assert(kHistBins <= 256, "count histogram shares the radix histogram");

__global__ void __launch_bounds__(SEL_THREADS) bm_select_kernel(IndexView ix, int l, int cap,
                                                                QueryState st,
                                                                int64_t *__restrict__ stats_out,
                                                                bool sorted)
{
    extern __shared__ uint64_t keys[];
    __shared__ int hist[256];
    __shared__ int bc[4];
    __shared__ int tmp[SEL_THREADS / 32];
    __shared__ int s_np, s_nd, s_ne, s_nt, s_cstar, s_take, s_keep;
    const int q = blockIdx.x;
    const int m = ix.m;
    const int lane = threadIdx.x & 31;
    const uint32_t below = (1u << lane) - 1u;
    const int jf = st.levels[q] - 1;
    const int n = st.qbuf_n[(int64_t)(jf & 1) * st.qbn_par + q];
    const int nc = st.ncand[q];
    const uint64_t *E = st.qbuf + (int64_t)q * kQCap;
    int32_t *cand = st.cand + (int64_t)q * cap;
    int32_t *col = st.cand_col + (int64_t)q * cap;
    int32_t *eq = st.eqbuf + (int64_t)q * kEqCap;
    // a rebuilt list (flag 4) holds only the kept entries and the tie class
    const bool ovf_list = n > kQCap || (n != nc && !(st.bm_ovf[q] & 4));
    const int nl = ovf_list ? 0 : n;
    if (threadIdx.x == 0) {
        s_np = 0;
        s_nd = 0;
        s_ne = 0;
        s_nt = 0;
    }
    for (int c = threadIdx.x; c < kHistBins; c += SEL_THREADS) hist[c] = 0;
    __syncthreads();
    // counts of the candidates not of the previous level, and how many are
    for (int j0 = 0; j0 < nl; j0 += SEL_THREADS * SEL_U) {
        uint64_t e[SEL_U];
#pragma unroll
        for (int u = 0; u < SEL_U; ++u) {
            const int j = j0 + u * SEL_THREADS + threadIdx.x;
            e[u] = j < nl ? E[j] : 1ull << 9;  // bit 9: no entry
        }
        int n_pf = 0;
#pragma unroll
        for (int u = 0; u < SEL_U; ++u) {
            if (j0 + u * SEL_THREADS >= nl) break;
            const bool pf = (e[u] >> 8) & 1u;
            const bool other = !((e[u] >> 8) & 3u);
            n_pf += __popc(__ballot_sync(0xffffffffu, pf));
            const uint32_t bin = other ? 1u + (uint32_t)(e[u] & 0xffu) : 1024u;
            const uint32_t peers = __match_any_sync(0xffffffffu, bin);
            if (other && lane == __ffs(peers) - 1) atomicAdd(&hist[bin], __popc(peers));
        }
        if (lane == 0 && n_pf) atomicAdd(&s_np, n_pf);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int cstar = l - 1, take = 0;
        const int np = s_np;
        if (nc > cap) {
            const int need = cap - np;
            int acc = 0;
            for (int c = m; c >= l; --c) {
                const int hc = hist[1 + c];
                if (acc + hc >= need) {
                    cstar = c;
                    take = need - acc;
                    break;
                }
                acc += hc;
            }
        }
        int kept = np + take;
        for (int c = max(cstar + 1, l); c <= m; ++c) kept += hist[1 + c];
        s_cstar = cstar;
        s_take = take;
        s_keep = min(kept, cap);
    }
    __syncthreads();
    const int cstar = s_cstar, take = s_take, keep = s_keep;
    // kept outright, and the tie class at c* (original ids); one slot
    // reservation per warp
    const int32_t *perm = ix.perm;
    for (int j0 = 0; j0 < nl; j0 += SEL_THREADS * SEL_U) {
        uint64_t e[SEL_U];
        int32_t orig[SEL_U];
        uint32_t bk[SEL_U], bt[SEL_U];
        int nK = 0, nT = 0;
#pragma unroll
        for (int u = 0; u < SEL_U; ++u) {
            const int j = j0 + u * SEL_THREADS + threadIdx.x;
            e[u] = j < nl ? E[j] : 1ull << 9;
        }
#pragma unroll
        for (int u = 0; u < SEL_U; ++u) {
            bk[u] = bt[u] = 0u;
            if (j0 + u * SEL_THREADS >= nl) continue;
            const int c = (int)(e[u] & 0xffu);
            const bool in = !((e[u] >> 9) & 1u);
            const bool kp = in && (((e[u] >> 8) & 1u) || c > cstar);
            const bool ti = in && !kp && c == cstar && take > 0;
            if (kp || ti) orig[u] = perm[e[u] >> 32];
            bk[u] = __ballot_sync(0xffffffffu, kp);
            bt[u] = __ballot_sync(0xffffffffu, ti);
            nK += __popc(bk[u]);
            nT += __popc(bt[u]);
        }
        int baseK = 0, baseT = 0;
        if (lane == 0) {
            if (nK) baseK = atomicAdd(&s_nd, nK);
            if (nT) baseT = atomicAdd(&s_ne, nT);
        }
        baseK = __shfl_sync(0xffffffffu, baseK, 0);
        baseT = __shfl_sync(0xffffffffu, baseT, 0);
#pragma unroll
        for (int u = 0; u < SEL_U; ++u) {
            if (j0 + u * SEL_THREADS >= nl) break;
            if ((bk[u] >> lane) & 1u) {
                const int d = baseK + __popc(bk[u] & below);
                if (d < cap) {
                    cand[d] = orig[u];
                    col[d] = (int)(e[u] & 0xffu);
                }
            } else if ((bt[u] >> lane) & 1u) {
                const int t = baseT + __popc(bt[u] & below);
                if (t < kEqCap) eq[t] = orig[u];
            }
            baseK += __popc(bk[u]);
            baseT += __popc(bt[u]);
        }
    }
    __syncthreads();
    const int nd = s_nd, ne = s_ne;
    const bool ovf = ovf_list || nd + take != keep || take > ne;
    if (ovf) {
        if (threadIdx.x == 0) {
            atomicOr(st.bm_ovf + q, 1);
            st.nkeep[q] = 0;
        }
        for (int p = threadIdx.x; p < cap; p += SEL_THREADS) {
            cand[p] = -1;
            col[p] = 0;
        }
        return;
    }
    if (take > 0 && ne > kEqCap) {
        // a tie class larger than its list: select from the candidate list
        // itself (members: not of the previous level, count c*), keyed by
        // original id
        auto tie = [&](int j, uint32_t *u) {
            const uint64_t e = E[j];
            if (((e >> 8) & 1u) || (int)(e & 0xffu) != cstar) return false;
            *u = (uint32_t)perm[e >> 32];
            return true;
        };
        const uint32_t T =
            take < ne ? block_kth_smallest_if<SEL_THREADS>(nl, take, tie, hist, bc) : 0xffffffffu;
        for (int j0 = 0; j0 < nl; j0 += SEL_THREADS) {
            const int j = j0 + threadIdx.x;
            uint32_t id = 0u;
            const bool in = j < nl && tie(j, &id) && id <= T;
            const uint32_t b = __ballot_sync(0xffffffffu, in);
            int base = 0;
            if (lane == 0 && b) base = atomicAdd(&s_nt, __popc(b));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (in) {
                cand[nd + base + __popc(b & below)] = (int32_t)id;
                col[nd + base + __popc(b & below)] = cstar;
            }
        }
        __syncthreads();
    } else if (take > 0) {
        // the take smallest ids of the tie class: those <= its take-th smallest
        // (ids are distinct, so exactly take of them)
        const uint32_t T = take < ne ? block_kth_bound<SEL_THREADS>(
                                           reinterpret_cast<const uint32_t *>(eq), ne, take, 0, 256,
                                           hist, bc, tmp)
                                     : 0xffffffffu;
        for (int j0 = 0; j0 < ne; j0 += SEL_THREADS) {
            const int j = j0 + threadIdx.x;
            const uint32_t id = j < ne ? (uint32_t)eq[j] : 0u;
            const bool in = j < ne && id <= T;
            const uint32_t b = __ballot_sync(0xffffffffu, in);
            int base = 0;
            if (lane == 0 && b) base = atomicAdd(&s_nt, __popc(b));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (in) {
                cand[nd + base + __popc(b & below)] = (int32_t)id;
                col[nd + base + __popc(b & below)] = cstar;
            }
        }
        __syncthreads();
    }
    if (sorted) {
        int P2 = 2;
        while (P2 < keep) P2 <<= 1;
        for (int i = threadIdx.x; i < keep; i += SEL_THREADS)
            keys[i] = ((uint64_t)(uint32_t)cand[i] << 32) | (uint32_t)col[i];
        smem_bitonic(keys, keep, P2);
        for (int i = threadIdx.x; i < keep; i += SEL_THREADS) {
            cand[i] = (int32_t)(keys[i] >> 32);
            col[i] = (int32_t)(keys[i] & 0xffffffffu);
        }
    }
    for (int p = keep + threadIdx.x; p < cap; p += SEL_THREADS) {
        cand[p] = -1;
        col[p] = 0;
    }
    if (threadIdx.x == 0) {
        st.nkeep[q] = keep;
        if (stats_out) {
            int64_t *so = stats_out + (int64_t)q * QW_NSTAT;
            so[0] = st.levels[q];
            so[1] = st.finalR[q];
            so[2] = nc;
            so[3] = keep;
            so[4] = st.term[q];
            so[5] = st.scan_last[q];
            so[6] = st.scan_full[q];
            so[7] = st.nprev[q];
        }
    }
}

// ---- a last level that overflows the candidate list
//
// A query's list holds up to kQCap candidates.  When one doubling of the radius
// sweeps whole clusters into a query's last level, that level can hold more, or
// so many that listing and selecting from them one by one costs more than counting
// them twice: from kQDirect on (4,000 queries with 430 million
// candidates, 325 of them with nearly every point: list, rebuild and selection
// 2.39 ms with the line at 32,768, 2.44 at 16,384, 2.40 at 65,536, 2.57 without
// it).  Of them the k + v bound keeps only the previous level's candidates, every
// candidate whose count is above the boundary count c*, and the smallest
// original ids of the tie class at c* (Section 3.1, readings R4/R5).  The kernels
// below rebuild the list of such a query with only those entries, from the candidate words of its last level
// (still in place: a stopped query's tiles are not touched by later levels)
// and the level bitmaps, each read once:
//   rd_compact  lists the queries (slots) and their buckets;
//   rd_count    one lane per 128-id group holding candidates: the counts
//               from the m bitmap words of the last level, the previous
//               level's candidate word (at a learned first level: their
//               counts there, from that level's bitmaps), stored as seven bit
//               planes and the word (128 bytes per group); the histogram of
//               the counts of the candidates not of the previous level;
//   rd_plan 0   c* and how many ids at c* are kept, as the selection derives
//               them;
//   rd_scan     when the tie class at c* holds more than kRdTieList ids: walks
//               the original ids upward (data id -> internal id -> candidate
//               word, stored count, previous-level word) and lists the take
//               smallest tie members, so that the list stays short;
//   rd_emit     the other kept entries (and a short tie class) from the
//               stored planes, written as the count kernels write them;
//   rd_plan 2   the list lengths.
// The selection then runs on the rebuilt list as on any other, with the same
// result as from the whole list.  A query whose rebuilt list would still
// overflow keeps the level-path answer, and so do the slots beyond one
// store's worth (kRdStoreBytes).
// candidates listed whole (more, if there is a slot: counted first); above any k + v
constexpr int kQDirect = 32768;
static_assert(kQDirect > QW_MAX_CAND, "a slot holds more candidates than are kept");
constexpr int kRdTieList = kEqCap;  // larger tie classes are cut by the original-id walk
constexpr int kRdStoreWords = 8;  // uint4 per group: 7 count planes, previous-level word
constexpr int RD_THREADS = 256;

// Count planes of group g of tile t from the bitmaps of one level: bq[i] is
// the bucket's bitmap in tile 0 (-1: no data), tile t adds t * bm_nb[i].
__device__ __forceinline__ void rd_planes(const IndexView &ix, const int64_t *bq, int t, int g,
                                          Planes &P)
{
    const int m = ix.m;
#pragma unroll
    for (int kk = 0; kk < 7; ++kk)
#pragma unroll
        for (int w = 0; w < 4; ++w) P.s[kk][w] = 0;
    for (int i0 = 0; i0 < m; i0 += 8) {
        uint4 x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = i0 + u;
            const int64_t b = i < m ? bq[i] : -1;
            x[u] = b >= 0 ? __ldg(ix.bm + (b + (int64_t)t * ix.bm_nb[i]) * kBmUint4 + g)
                          : make_uint4(0, 0, 0, 0);
        }
        add8(P, x);
    }
}

// Bits of word w whose count equals c.
__device__ __forceinline__ uint32_t count_eq_planes(const Planes &P, int w, int c)
{
    uint32_t eq = 0xffffffffu;
#pragma unroll
    for (int k = 0; k < 7; ++k) eq &= ((c >> k) & 1) ? P.s[k][w] : ~P.s[k][w];
    return eq;
}

// One warp per query: slots for the queries with more than `over` and at most
// `upto` candidates, as long as the store has places for those that could also
// be listed whole.  Marks them (bm_ovf flag 8).
__global__ void rd_compact_kernel(IndexView ix, int cgrow, QueryState st, int nb, int over,
                                  int upto, int wave)
{
    const int q = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (q >= nb) return;
    const int L = st.levels[q] - 1;
    if (L < 0) return;
    const int n = st.qbuf_n[(int64_t)(L & 1) * st.qbn_par + q];
    if (n <= over || n > upto) return;
    int slot = 0;
    if (lane == 0) slot = atomicAdd(st.rd_ctl, 1);
    slot = __shfl_sync(0xffffffffu, slot, 0);
    if (n <= kQCap && slot >= wave) return;
    if (lane == 0) {
        if (n > kQCap) atomicAdd(st.rd_ctl + 1, 1);
        st.bm_ovf[q] |= 8;
        RdPlan p;
        memset(&p, 0, sizeof(p));
        p.q = q;
        p.mode = 1;
        p.prev_recount = (L - 1 < st.start[q] && L > 0) ? 1 : 0;
        st.rd_plan[slot] = p;
    }
    int32_t *h = st.rd_hist + (int64_t)slot * kHistBins;
    for (int c = lane; c < kHistBins; c += 32) h[c] = 0;
    const int64_t R = st.finalR[q];
    int64_t *bq = st.rd_bq + (int64_t)slot * QW_MAX_M;
    for (int i = lane; i < ix.m; i += 32) {
        const int64_t gi = st.g[(int64_t)q * ix.m + i];
        bq[i] = L > 0 ? bm_index(ix, i, 0, L - 1, R / cgrow, floordiv64(gi, R / cgrow)) : -1;
    }
}

// A warp takes an eighth of the groups with candidates of four tiles of a slot
// (groups 4 p .. 4 p + 3 of every mask word), as bm_count_kernel takes live
// groups; the slots' tasks alternate, so that after the first of a slot most
// counts are known to lie below its c* and stay out of the histogram.  4,000
// queries, 1,000,000 points, 1,100 slots: 1,283 us in quarters, slot by slot and
// with the whole histogram, 1,164 so; 262 slots with all of 3,000,000 points 986
// and 935 us; 606 with all of 300,000 290 and 223.
constexpr int kRdParts = 8;

__device__ __forceinline__ uint32_t rd_task(const IndexView &ix, const QueryState &st, int64_t k,
                                            int nslot, int lane, int *slot, int *t0, int *q, int *L)
{
    const int part = (int)(k / nslot % kRdParts);
    *t0 = (int)(k / nslot / kRdParts) * 4;
    *slot = (int)(k % nslot);
    *q = st.rd_plan[*slot].q;
    *L = st.levels[*q] - 1;
    const uint32_t x = *t0 + (lane >> 3) < ix.nT
                           ? st.bm_amask[((int64_t)(*L & 1) * st.cln_par + (int64_t)*q * ix.nT +
                                          *t0) * kSumWords + lane]
                           : 0u;
    return x & part_bits(part, kRdParts);
}

__global__ void __launch_bounds__(RD_THREADS, 3) rd_count_kernel(IndexView ix, int l, int cap,
                                                                  QueryState st, int wave)
{
    __shared__ int sh_hist[RD_THREADS / 32][kHistBins];
    __shared__ int s_nb[QW_MAX_M + 16];
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < st.bm_mp; i += RD_THREADS) s_nb[i] = i < ix.m ? ix.bm_nb[i] : 0;
    for (int c = lane; c < kHistBins; c += 32) sh_hist[wi][c] = 0;
    __syncthreads();
    int *hist = sh_hist[wi];
    const int nT = ix.nT;
    const int nslot = min(st.rd_ctl[0], wave);
    const int64_t tasks = (int64_t)nslot * ((nT + 3) >> 2) * kRdParts;
    for (int64_t k = (int64_t)blockIdx.x * (RD_THREADS / 32) + wi; k < tasks;
         k += (int64_t)gridDim.x * (RD_THREADS / 32)) {
        int slot, t0, q, L;
        const uint32_t x = rd_task(ix, st, k, nslot, lane, &slot, &t0, &q, &L);
        if (!__any_sync(0xffffffffu, x != 0)) continue;
        const bool recount = st.rd_plan[slot].prev_recount;
        const int floor = max(l, __ldcg(&st.rd_plan[slot].floor));
        int my_np = 0;
        each_set_bit(x, lane, [&](int own, int bit, bool valid, bool four) {
            const int t = t0 + (own >> 3), g = (own & 7) * 32 + bit;
            const int64_t qt = (int64_t)q * nT + t;
            uint4 pw = make_uint4(0, 0, 0, 0);
            Planes P;
            if (recount) {
                rd_planes(ix, st.rd_bq + (int64_t)slot * QW_MAX_M, t, g, P);
                pw = candidates_of(P, l);
            } else if (L > 0) {
                pw = rd_word(st, L - 1, qt, g);
            }
            count_planes(ix, st.bm_b0 + (int64_t)q * st.bm_mp, s_nb, t, g, P, four);
            const uint4 cw = candidates_of(P, l);
            uint32_t oth[4] = {0, 0, 0, 0};  // candidates not of the previous level
            int n_oth = 0;
            if (valid) {
                uint4 *store = st.rd_store +
                               ((int64_t)slot * nT * kBmUint4 + (int64_t)t * kBmUint4 + g) *
                                   kRdStoreWords;
#pragma unroll
                for (int kk = 0; kk < 7; ++kk)
                    store[kk] = make_uint4(P.s[kk][0], P.s[kk][1], P.s[kk][2], P.s[kk][3]);
                store[7] = pw;
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    my_np += __popc(word_of(cw, w) & word_of(pw, w));
                    oth[w] = word_of(cw, w) & ~word_of(pw, w);
                    if (floor > l) oth[w] &= count_ge_planes(P, w, floor);
                    n_oth += __popc(oth[w]);
                }
            }
            // the histogram of their counts: a warp with many of them compares
            // the planes with every count (one addition per warp and count);
            // adding one by one meets the same few shared words over and over
            if (__reduce_add_sync(0xffffffffu, n_oth) > 256) {
                for (int c = floor; c <= ix.m; ++c) {
                    int here = 0;
#pragma unroll
                    for (int w = 0; w < 4; ++w)
                        if (oth[w]) here += __popc(count_eq_planes(P, w, c) & oth[w]);
                    here = __reduce_add_sync(0xffffffffu, here);
                    if (lane == 0 && here) atomicAdd(&hist[c], here);
                }
            } else {
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    uint32_t left = oth[w];
                    while (left) {
                        const int b = __ffs(left) - 1;
                        left &= left - 1;
                        atomicAdd(&hist[count_of(P, w, b)], 1);
                    }
                }
            }
        });
        my_np = __reduce_add_sync(0xffffffffu, my_np);
        if (lane == 0 && my_np) atomicAdd(&st.rd_plan[slot].np, my_np);
        __syncwarp();
        int32_t *h = st.rd_hist + (int64_t)slot * kHistBins;
        for (int c = lane; c < kHistBins; c += 32)
            if (hist[c]) {
                atomicAdd(h + c, hist[c]);
                hist[c] = 0;
            }
        __syncwarp();
        // k + v or more of them with at least c so far: c* is no lower
        int above = 0, c = 0;
        for (int c0 = ix.m; c0 >= floor && c == 0; c0 -= 32) {
            int incl = c0 - lane >= floor ? __ldcg(h + c0 - lane) : 0;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += y;
            }
            const uint32_t full = __ballot_sync(0xffffffffu, above + incl >= cap);
            if (full) c = c0 - (__ffs(full) - 1);
            above += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lane == 0 && c > floor) atomicMax(&st.rd_plan[slot].floor, c);
    }
}

__global__ void rd_plan_kernel(int l, int m, int cap, int cgrow, QueryState st, int wave, int stage)
{
    const int slot = blockIdx.x * blockDim.x + threadIdx.x;
    if (slot >= min(st.rd_ctl[0], wave)) return;
    RdPlan p = st.rd_plan[slot];
    const int q = p.q;
    const int L = st.levels[q] - 1;
    if (stage == 0) {
        if (!p.prev_recount) p.np = st.nprev[q];
        if (st.recount[q] && (st.finalR[q] / cgrow > st.top[q] || p.np >= cap)) {
            // a learned first level after the level where the plain path stops:
            // answered again from level 0
            atomicOr(st.bm_ovf + q, 2);
            p.mode = 0;
        } else {
            // histogram of counts -> the count c* at which the bound is reached
            const int32_t *h = st.rd_hist + (int64_t)slot * kHistBins;
            const int need = cap - p.np;
            int acc = 0, cstar = -1, take = 0;
            for (int c = m; c >= l; --c) {
                if (acc + h[c] >= need) {
                    cstar = c;
                    take = need - acc;
                    break;
                }
                acc += h[c];
            }
            if (cstar < 0) {
                p.mode = 0;  // cannot happen with more than k + v candidates
            } else {
                p.cstar = cstar;
                p.take = take;
                // a short tie class is listed whole, a long one cut by rd_scan
                p.mode = h[cstar] <= kRdTieList ? 1 : 2;
            }
        }
    } else if (p.mode == 0) {
        // nothing was listed: the selection marks the query
        st.qbuf_n[(int64_t)(L & 1) * st.qbn_par + q] = kQCap + 1;
    } else {
        // the rebuilt list (more than kQCap entries: the level path answers)
        st.qbuf_n[(int64_t)(L & 1) * st.qbn_par + q] = p.pos;
        st.bm_ovf[q] |= 4;
        if (st.recount[q]) {
            st.nprev[q] = p.np;
            st.recount[q] = 0;
        }
    }
    st.rd_plan[slot] = p;
}

// The stored planes of group g of tile t of a slot.
__device__ __forceinline__ void rd_stored(const QueryState &st, int slot, int nT, int t, int g,
                                          Planes &P, uint4 &pw)
{
    const uint4 *store = st.rd_store +
                         ((int64_t)slot * nT * kBmUint4 + (int64_t)t * kBmUint4 + g) * kRdStoreWords;
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        const uint4 v = store[k];
        P.s[k][0] = v.x;
        P.s[k][1] = v.y;
        P.s[k][2] = v.z;
        P.s[k][3] = v.w;
    }
    pw = store[7];
}

// The kept entries of every rebuilt slot, warps as in rd_count_kernel:
// previous-level candidates, counts above c*, and (a short tie class) the tie
// class.
__global__ void __launch_bounds__(RD_THREADS, 3) rd_emit_kernel(IndexView ix, int l, QueryState st,
                                                                 int wave)
{
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const int m = ix.m, nT = ix.nT;
    const int nslot = min(st.rd_ctl[0], wave);
    const int64_t tasks = (int64_t)nslot * ((nT + 3) >> 2) * kRdParts;
    for (int64_t k = (int64_t)blockIdx.x * (RD_THREADS / 32) + wi; k < tasks;
         k += (int64_t)gridDim.x * (RD_THREADS / 32)) {
        int slot, t0, q, L;
        const uint32_t x = rd_task(ix, st, k, nslot, lane, &slot, &t0, &q, &L);
        if (!__any_sync(0xffffffffu, x != 0)) continue;
        const int mode = st.rd_plan[slot].mode, cstar = st.rd_plan[slot].cstar;
        if (mode == 0) continue;
        uint64_t *E = st.qbuf + (int64_t)q * kQCap;
        each_set_bit(x, lane, [&](int own, int bit, bool valid, bool) {
            const int t = t0 + (own >> 3), g = (own & 7) * 32 + bit;
            Planes P;
            uint4 pw;
            rd_stored(st, slot, nT, t, g, P, pw);
            uint32_t kw[4];
            int my_n = 0;
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const uint32_t c_w = count_ge_planes(P, w, l), p_w = word_of(pw, w);
                const uint32_t oth = c_w & ~p_w;
                kw[w] = (c_w & p_w) | (cstar < m ? count_ge_planes(P, w, cstar + 1) & oth : 0u);
                if (mode == 1) kw[w] |= count_eq_planes(P, w, cstar) & oth;
                if (!valid) kw[w] = 0u;
                my_n += __popc(kw[w]);
            }
            int incl = my_n;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += y;
            }
            int pos = 0;
            if (lane == 31 && incl) pos = atomicAdd(&st.rd_plan[slot].pos, incl);
            pos = __shfl_sync(0xffffffffu, pos, 31) + incl - my_n;
            if (my_n)
                append_candidates(P, make_uint4(kw[0], kw[1], kw[2], kw[3]), pw, E, pos,
                                  (int64_t)t * kTile + (int64_t)g * 128);
        });
    }
}

// One block per slot with a long tie class: data ids 0, 1, 2, ... are tested
// kScanPer * RS_THREADS at a time (thread t takes ids o0 + u * RS_THREADS + t, so the loads
// of each u are coalesced and the kScanPer chains of dependent reads are in
// flight together; tie member: a candidate of the last level, not of the
// previous one, with count c*) until `take` members are found; those are the
// take smallest original ids of the tie class (reading R5), listed with count
// c*.  The walk reads about take * n / (tie class size) ids.
constexpr int kScanPer = 4;
constexpr int RS_THREADS = 1024;

__global__ void __launch_bounds__(RS_THREADS) rd_scan_kernel(IndexView ix, QueryState st,
                                                              int wave)
{
    constexpr int NW = RS_THREADS / 32;
    __shared__ int s_wc[kScanPer][NW];
    __shared__ int s_base;
    const int nslot = min(st.rd_ctl[0], wave);
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    for (int slot = blockIdx.x; slot < nslot; slot += gridDim.x) {
        const RdPlan pl = st.rd_plan[slot];
        if (pl.mode != 2 || pl.take <= 0) continue;
        const int q = pl.q, L = st.levels[q] - 1;
        uint64_t *E = st.qbuf + (int64_t)q * kQCap;
        if (threadIdx.x == 0) s_base = atomicAdd(&st.rd_plan[slot].pos, pl.take);
        __syncthreads();
        const int base = s_base;
        int found = 0;
        for (int64_t o0 = 0; o0 < ix.n && found < pl.take; o0 += RS_THREADS * kScanPer) {
            int64_t iid[kScanPer];
#pragma unroll
            for (int u = 0; u < kScanPer; ++u) {
                const int64_t o = o0 + u * RS_THREADS + threadIdx.x;
                iid[u] = o < ix.n ? (int64_t)ix.inv[o] : -1;
            }
            uint4 cw[kScanPer];
#pragma unroll
            for (int u = 0; u < kScanPer; ++u) {
                const int64_t id = iid[u] >= 0 ? iid[u] : 0;
                const int t = (int)(id / kTile), g = (int)((id % kTile) >> 7);
                cw[u] = iid[u] >= 0 ? rd_word(st, L, (int64_t)q * ix.nT + t, g)
                                    : make_uint4(0, 0, 0, 0);
            }
            bool tie[kScanPer];
#pragma unroll
            for (int u = 0; u < kScanPer; ++u) {
                tie[u] = false;
                const int64_t id = iid[u] >= 0 ? iid[u] : 0;
                const int t = (int)(id / kTile), g = (int)((id % kTile) >> 7), b = (int)(id & 127);
                if (iid[u] >= 0 && ((word_of(cw[u], b >> 5) >> (b & 31)) & 1u)) {
                    // the id's bit of each stored plane and of the previous
                    // level's word (word b / 32 of each 16-byte record)
                    const uint32_t *rec = reinterpret_cast<const uint32_t *>(
                        st.rd_store + ((int64_t)slot * ix.nT * kBmUint4 + (int64_t)t * kBmUint4 + g) *
                                          kRdStoreWords) + (b >> 5);
                    int cnt = 0;
#pragma unroll
                    for (int k = 0; k < 7; ++k) cnt |= (int)((rec[4 * k] >> (b & 31)) & 1u) << k;
                    tie[u] = !((rec[4 * 7] >> (b & 31)) & 1u) && cnt == pl.cstar;
                }
            }
            uint32_t bal[kScanPer];
#pragma unroll
            for (int u = 0; u < kScanPer; ++u) {
                bal[u] = __ballot_sync(0xffffffffu, tie[u]);
                if (lane == 0) s_wc[u][wi] = __popc(bal[u]);
            }
            __syncthreads();
            // ties before (u, this warp) in id order: all of the earlier u,
            // then the earlier warps of this u
            int total = 0;
#pragma unroll
            for (int u = 0; u < kScanPer; ++u) {
                int before = 0, tot_u = 0;
#pragma unroll
                for (int w = 0; w < NW; ++w) {
                    const int c = s_wc[u][w];
                    if (w < wi) before += c;
                    tot_u += c;
                }
                if (tie[u]) {
                    const int rank = found + total + before + __popc(bal[u] & lt);
                    if (rank < pl.take && base + rank < kQCap)
                        E[base + rank] = ((uint64_t)iid[u] << 32) | (uint64_t)pl.cstar;
                }
                total += tot_u;
            }
            found += total;
            __syncthreads();  // s_wc is rewritten next
        }
    }
}

// Learned starts on the bitmap path: a query that stopped at its first level
// L > 0 never counted level L - 1, whose candidates come first under the k + v
// bound (reading R5).  Those are exactly the final candidates whose level-(L-1)
// count reaches l (buckets nest, so C(L-1) is a subset of C(L)).  The count of
// a candidate is taken from its row of anchored bucket ids: on projection i it
// collides at radius R' = c^(L-1) when floor(h_i / R') == floor(g_i / R'), i.e.
// when h_i lies in [beta_i R', (beta_i + 1) R' - 1].  One block per query, one
// thread per candidate: the row is read in 16-byte pieces and compared with
// the bounds (packed like the row, in shared memory) 4, 2 or 1 ids per 32-bit
// word by SIMD compares.
// The plain path would have stopped earlier if |C(L-1)| >= k + v or if radius
// c^(L-1) already exceeded every useful radius of the query: such queries are
// marked for the level path.  A query's candidates are split over
// kRcSplits blocks (a long list would otherwise leave one block working
// alone); their counts add up in nprev, and a second kernel compares the sum
// with k + v.
constexpr int RC_THREADS = 128;
constexpr int kRcSplits = 8;
constexpr int kRcPer = 8;  // candidates per thread of a piece
constexpr int kRcChunks = (QW_MAX_M * 4 + 15) / 16;  // 16-byte pieces of the widest row

// Ids of a 32-bit word within [lo, hi] (element-wise, inclusive).
template <typename T> __device__ __forceinline__ int in_range(uint32_t h, uint32_t lo, uint32_t hi);
template <> __device__ __forceinline__ int in_range<uint8_t>(uint32_t h, uint32_t lo, uint32_t hi)
{
    // a >= b per byte in its bit 7: the difference of the low bits borrows from
    // bit 7 unless they are >=, and bit 7 itself decides where the two differ
    const uint32_t top = 0x80808080u;
    const uint32_t d0 = (h | top) - (lo & ~top), d1 = (hi | top) - (h & ~top);
    const uint32_t ge = (h & ~lo) | (~(h ^ lo) & d0), le = (hi & ~h) | (~(hi ^ h) & d1);
    return __popc(ge & le & top);
}
template <> __device__ __forceinline__ int in_range<uint16_t>(uint32_t h, uint32_t lo, uint32_t hi)
{
    return __popc(__vcmpgeu2(h, lo) & __vcmpleu2(h, hi)) >> 4;
}
template <> __device__ __forceinline__ int in_range<uint32_t>(uint32_t h, uint32_t lo, uint32_t hi)
{
    return (h >= lo && h <= hi) ? 1 : 0;
}

template <typename T>
__global__ void __launch_bounds__(RC_THREADS) bm_recount_kernel(IndexView ix, int l, int cap,
                                                                int cgrow, QueryState st)
{
    __shared__ uint4 blo[kRcChunks], bhi[kRcChunks];
    __shared__ int s_nprev;
    const int q = blockIdx.x;
    const int split = blockIdx.y, nsplit = gridDim.y;
    if (!st.recount[q]) return;
    const int m = ix.m;
    const int L = st.levels[q] - 1;
    const int64_t R = st.finalR[q] / cgrow;  // radius of level L - 1
    const int n = st.qbuf_n[(int64_t)(L & 1) * st.qbn_par + q];
    uint64_t *E = st.qbuf + (int64_t)q * kQCap;
    if (n > kQCap) return;  // the selection marks the query for the level path
    if (split > 0 && split * RC_THREADS * kRcPer >= n) return;
    if (R > st.top[q]) {
        // the plain path stops at level L - 1 by radius: not this answer
        if (threadIdx.x == 0 && split == 0) atomicOr(st.bm_ovf + q, 2);
        return;
    }
    const int chunks = ix.hloc_stride / 16;
    // per projection, the ids of the level-(L-1) bucket in the width of the row
    // (an empty range as lo = max, hi = 0; padding never matches)
    const int64_t tmax = sizeof(T) == 4 ? (int64_t)INT32_MAX : ((int64_t)1 << (8 * sizeof(T))) - 1;
    T *lo_t = reinterpret_cast<T *>(blo), *hi_t = reinterpret_cast<T *>(bhi);
    for (int i = threadIdx.x; i < chunks * (16 / (int)sizeof(T)); i += RC_THREADS) {
        int64_t lo = tmax, hi = 0;
        if (i < m) {
            const int64_t beta = floordiv64(st.g[(int64_t)q * m + i], R);
            const int64_t a = beta * R, b = beta * R + R - 1;
            if (b >= 0 && a <= tmax) {
                lo = a > 0 ? a : 0;
                hi = b < tmax ? b : tmax;
            }
        }
        lo_t[i] = (T)lo;
        hi_t[i] = (T)hi;
    }
    if (threadIdx.x == 0) s_nprev = 0;
    __syncthreads();
    const char *H = static_cast<const char *>(ix.hloc);
    int mine = 0;
    // the splits take pieces of kRcPer candidates per thread in turn
    const int piece = RC_THREADS * kRcPer;
    for (int i = threadIdx.x;; i += RC_THREADS) {
        const int j = (i / piece * nsplit + split) * piece + i % piece;
        if (j >= n) break;
        const uint64_t e = E[j];
        const uint4 *row = reinterpret_cast<const uint4 *>(H + (int64_t)(e >> 32) * ix.hloc_stride);
        int c = 0;
#pragma unroll 4
        for (int v = 0; v < chunks; ++v) {
            const uint4 h = __ldg(row + v);
            const uint4 a = blo[v], b = bhi[v];
            c += in_range<T>(h.x, a.x, b.x) + in_range<T>(h.y, a.y, b.y) +
                 in_range<T>(h.z, a.z, b.z) + in_range<T>(h.w, a.w, b.w);
        }
        if (c >= l) {
            E[j] = e | (1ull << 8);
            ++mine;
        }
    }
    mine = __reduce_add_sync(0xffffffffu, mine);
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&s_nprev, mine);
    __syncthreads();
    // nprev of a query stopped at its first level starts at 0 (the decision
    // kernel set it from the empty count before that level)
    if (threadIdx.x == 0 && s_nprev) atomicAdd(st.nprev + q, s_nprev);
}

// After the split recount: a query whose |C(L-1)| reaches k + v would have
// stopped at level L - 1 on the plain path; it is marked for the level path.
__global__ void recount_decide_kernel(QueryState st, int nb, int cap, int cgrow)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nb || !st.recount[q]) return;
    const int L = st.levels[q] - 1;
    if (st.qbuf_n[(int64_t)(L & 1) * st.qbn_par + q] > kQCap) return;
    if (st.finalR[q] / cgrow > st.top[q]) return;
    if (st.nprev[q] >= cap) atomicOr(st.bm_ovf + q, 2);
}

// Rows of anchored bucket ids in locality order from the projection-major ids:
// a block takes 64 data ids, reads their ids of every projection in coalesced
// runs, assembles the rows in shared memory and writes each to its place in the
// order in 16-byte pieces.  (One thread per entry through the order: 941 us at
// 1,000,000 x 64, 80 us so.)
constexpr int kHlocIds = 64;

template <typename T>
__global__ void __launch_bounds__(256) hloc_kernel(const int32_t *__restrict__ Ht,
                                                   const int32_t *__restrict__ inv,
                                                   const int32_t *__restrict__ o, int64_t n, int m,
                                                   int stride, char *__restrict__ out)
{
    extern __shared__ __align__(16) char rows[];
    const int pad = stride + 16;  // consecutive rows in other banks
    const int64_t j0 = (int64_t)blockIdx.x * kHlocIds;
    const int r = threadIdx.x % kHlocIds;
    for (int e = threadIdx.x; e < kHlocIds * pad / 16; e += 256)
        reinterpret_cast<uint4 *>(rows)[e] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    if (j0 + r < n)
        for (int i = threadIdx.x / kHlocIds; i < m; i += 256 / kHlocIds)
            reinterpret_cast<T *>(rows + r * pad)[i] = (T)(Ht[(int64_t)i * n + j0 + r] - o[i]);
    __syncthreads();
    const int pieces = stride / 16;
    for (int e = threadIdx.x; e < kHlocIds * pieces; e += 256) {
        const int row = e / pieces, p = e % pieces;
        if (j0 + row < n)
            *reinterpret_cast<uint4 *>(out + (int64_t)inv[j0 + row] * stride + 16 * p) =
                *reinterpret_cast<const uint4 *>(rows + row * pad + 16 * p);
    }
}

// Workload indices of the batch's queries to answer again: list[0] those whose
// candidates overflowed the bitmap path's lists (flag 1: the level path), list
// [1] those whose learned first level was too late (flag 2 alone: the bitmap
// path from level 0); count[0], count[1] their numbers.
__global__ void bm_overflow_list_kernel(const QueryState st, int nb, const int32_t *order_perm,
                                        int64_t b0, int32_t *list0, int32_t *list1,
                                        int32_t *count)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nb) return;
    const int f = st.bm_ovf[q] & 3;
    if (!f) return;
    // a learned first level that was too late is answered again from level 0
    // on the bitmap path, whatever else happened to the query
    const int which = (f & 2) ? 1 : 0;
    const int pos = atomicAdd(count + which, 1);
    (which == 0 ? list0 : list1)[pos] = order_perm ? order_perm[b0 + q] : (int32_t)(b0 + q);
}

// Data objects per bid of every projection, then the exclusive prefix over
// bids: bid_prefix[off[i] + b] = objects with bid < b.
__global__ void bid_count_kernel(IndexView ix, int64_t *prefix, const int64_t *off)
{
    const int t = blockIdx.x, i = blockIdx.y;
    const int64_t dslot = (int64_t)i * ix.nT + t;
    const int32_t *ub = ix.dir_bid + ix.dir_start[dslot];
    const int32_t *uo = ix.dir_off + ix.dir_start[dslot];
    const int cnt = ix.dir_cnt[dslot];
    const int len = (int)min((int64_t)kTile, ix.n - (int64_t)t * kTile);
    for (int u = threadIdx.x; u < cnt; u += blockDim.x) {
        const int e1 = (u + 1 < cnt) ? uo[u + 1] : len;
        atomicAdd(reinterpret_cast<unsigned long long *>(prefix + off[i] + ub[u] + 1),
                  (unsigned long long)(e1 - uo[u]));
    }
}

__global__ void bid_scan_kernel(IndexView ix, int64_t *prefix, const int64_t *off)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ix.m) return;
    int64_t *P = prefix + off[i];
    int64_t acc = 0;
    for (int64_t b = 1; b <= (int64_t)ix.span[i] + 1; ++b) {
        acc += P[b];
        P[b] = acc;
    }
}

}  // namespace

qw_status launch_bitmap_build(const IndexView &ix, int c, int maxJ, uint4 *bm, uint32_t *bm_sum,
                              int64_t total_bitmaps, cudaStream_t s)
{
    const dim3 grid((unsigned)ix.nT, (unsigned)ix.m);
    const int P = 16 / ix.hloc_bytes;
    const dim3 fgrid((unsigned)ix.nT, (unsigned)((ix.m + P - 1) / P));
    if (ix.hloc_bytes == 1) bm_fill_level0_kernel<uint8_t><<<fgrid, BM_THREADS, 0, s>>>(ix, bm);
    else if (ix.hloc_bytes == 2) bm_fill_level0_kernel<uint16_t><<<fgrid, BM_THREADS, 0, s>>>(ix, bm);
    else bm_fill_level0_kernel<uint32_t><<<fgrid, BM_THREADS, 0, s>>>(ix, bm);
    QW_CUDA_TRY(cudaGetLastError());
    int64_t R = 1;
    for (int L = 1; L <= maxJ; ++L) {
        R *= c;
        bm_or_level_kernel<<<grid, BM_THREADS, 0, s>>>(ix, bm, L, R, c);
        QW_CUDA_TRY(cudaGetLastError());
    }
    QW_CUDA_TRY(cudaMemsetAsync(bm_sum + total_bitmaps * (kBmUint4 / 32), 0,
                                (size_t)ix.nT * (kBmUint4 / 8), s));
    bm_summary_kernel<<<grid, BM_THREADS, 0, s>>>(ix, bm, bm_sum);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

qw_status launch_bid_prefix(const IndexView &ix, int64_t *prefix, const int64_t *off,
                            cudaStream_t s)
{
    bid_count_kernel<<<dim3((unsigned)ix.nT, (unsigned)ix.m), 128, 0, s>>>(ix, prefix, off);
    QW_CUDA_TRY(cudaGetLastError());
    bid_scan_kernel<<<(ix.m + 63) / 64, 64, 0, s>>>(ix, prefix, off);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

ScanStats scan_stats_of(const IndexView &ix, int c)
{
    ScanStats ss;
    ss.prefix = ix.bid_prefix;
    ss.off = ix.prefix_off;
    ss.span = ix.span;
    ss.m = ix.m;
    ss.cgrow = c;
    return ss;
}

template <int TPW>
static void launch_fused(const IndexView &ix, int nb, int level, int l, QueryState &st,
                         const LoopCtl *ctl, cudaStream_t s)
{
    const int64_t tasks = (int64_t)nb * ((ix.nT + TPW - 1) / TPW);
    const int blocks = (int)std::max<int64_t>(
        1, std::min<int64_t>((tasks + FL_WARPS - 1) / FL_WARPS, 152 * 16));
    if (ix.m <= 32)
        bm_fused_kernel<1, TPW><<<blocks, FL_WARPS * 32, 0, s>>>(ix, level, l, nb, st, ctl);
    else if (ix.m <= 64)
        bm_fused_kernel<2, TPW><<<blocks, FL_WARPS * 32, 0, s>>>(ix, level, l, nb, st, ctl);
    else
        bm_fused_kernel<4, TPW><<<blocks, FL_WARPS * 32, 0, s>>>(ix, level, l, nb, st, ctl);
}

// Up to four (query, projection) entries per thread of one block cost less than a
// launch.
static bool buckets_in_one_block(int nb, int mp) { return (int64_t)nb * mp <= 4096; }

int bm_level_launches(int nb, int mp, int loads, int part)
{
    if (loads == QW_LOADS_TMA) return 1;
    const int buckets = part == 2 ? 0 : buckets_in_one_block(nb, mp) ? 1 : 2;
    const int counts = part == 1 ? 0 : loads == QW_LOADS_FUSED ? 1 : nb >= kDenseMin ? 3 : 2;
    return buckets + counts;
}

qw_status launch_bm_level(const IndexView &ix, int nb, int level, int64_t R, int64_t Rp, int l,
                          int cgrow, QueryState &st, int *err, int loads, cudaStream_t s,
                          const LoopCtl *ctl, int part, int tpw)
{
    (void)Rp;
    (void)cgrow;
    if (loads != QW_LOADS_TMA) {
        if (part != 2) {
            const int64_t qi = (int64_t)nb * st.bm_mp;
            const bool one = buckets_in_one_block(nb, st.bm_mp);
            bm_active_kernel<<<1, 1024, 0, s>>>(ix, level, R, nb, st, ctl, one);
            QW_CUDA_TRY(cudaGetLastError());
            if (!one) {
                bm_bucket_kernel<<<(unsigned)std::min<int64_t>((qi + 255) / 256, 152 * 8), 256, 0,
                                   s>>>(ix, level, R, st, ctl);
                QW_CUDA_TRY(cudaGetLastError());
            }
        }
        if (part == 1) return QW_OK;
        if (loads == QW_LOADS_FUSED) {
            if (tpw == 4) launch_fused<4>(ix, nb, level, l, st, ctl, s);
            else if (tpw == 16) launch_fused<16>(ix, nb, level, l, st, ctl, s);
            else launch_fused<8>(ix, nb, level, l, st, ctl, s);
            QW_CUDA_TRY(cudaGetLastError());
            return QW_OK;
        }
        // two passes: filter on the summaries, then count the live groups
        const int64_t tasks = (int64_t)nb * ((ix.nT + 3) / 4);
        const int64_t blocks =
            std::max<int64_t>(1, std::min<int64_t>((tasks + 7) / 8, 152 * 24));
        bm_filter_kernel<<<(unsigned)blocks, FL_WARPS * 32, 0, s>>>(ix, level, l, st, ctl);
        QW_CUDA_TRY(cudaGetLastError());
        const int64_t cblocks = std::max(blocks, std::min<int64_t>(tasks * 4, kCountWarps / 8));
        bm_count_kernel<<<(unsigned)cblocks, 256, 0, s>>>(ix, level, l, st, ctl);
        QW_CUDA_TRY(cudaGetLastError());
        // fewer queries than the dense form asks of an average group never take it
        if (nb >= kDenseMin) {
            const size_t smem = dense_smem_bytes();
            QW_TRY(allow_smem(bm_dense_kernel, smem));
            bm_dense_kernel<<<kDenseBlocks, DN_THREADS, smem, s>>>(ix, level, R, l, st, ctl);
            QW_CUDA_TRY(cudaGetLastError());
        }
        return QW_OK;
    }
    int dev = 0, n_sm = 0;
    QW_CUDA_TRY(cudaGetDevice(&dev));
    QW_CUDA_TRY(cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev));
    const size_t smem = tma_smem_bytes();
    QW_TRY(allow_smem(bm_level_tma_kernel, smem));
    const int64_t items = (int64_t)nb * ix.nT;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(n_sm, items));
    bm_level_tma_kernel<<<grid, TMA_THREADS, smem, s>>>(ix, level, R, l, nb, st, ctl, err);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

qw_status launch_locality_copy(const float *X, const int32_t *perm, int64_t n, int d, float *Xloc,
                               int32_t *inv, cudaStream_t s)
{
    if (n == 0) return QW_OK;
    locality_copy_kernel<<<(unsigned)std::min<int64_t>(n, 152 * 64), 128, 0, s>>>(X, perm, n, d,
                                                                                 Xloc, inv);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

qw_status launch_bm_recount(const IndexView &ix, int nb, int l, int cap, int cgrow, QueryState &st,
                            cudaStream_t s)
{
    if (nb == 0) return QW_OK;
    const dim3 grid((unsigned)nb, kRcSplits);
    if (ix.hloc_bytes == 1)
        bm_recount_kernel<uint8_t><<<grid, RC_THREADS, 0, s>>>(ix, l, cap, cgrow, st);
    else if (ix.hloc_bytes == 2)
        bm_recount_kernel<uint16_t><<<grid, RC_THREADS, 0, s>>>(ix, l, cap, cgrow, st);
    else
        bm_recount_kernel<uint32_t><<<grid, RC_THREADS, 0, s>>>(ix, l, cap, cgrow, st);
    QW_CUDA_TRY(cudaGetLastError());
    recount_decide_kernel<<<(nb + 255) / 256, 256, 0, s>>>(st, nb, cap, cgrow);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

qw_status launch_hloc_build(const IndexView &ix, const int32_t *Ht, void *hloc, cudaStream_t s)
{
    if (ix.n == 0) return QW_OK;
    const unsigned blocks = (unsigned)((ix.n + kHlocIds - 1) / kHlocIds);
    const size_t smem = (size_t)kHlocIds * (ix.hloc_stride + 16);
    char *out = static_cast<char *>(hloc);
    if (ix.hloc_bytes == 1)
        hloc_kernel<uint8_t><<<blocks, 256, smem, s>>>(Ht, ix.inv, ix.o, ix.n, ix.m, ix.hloc_stride, out);
    else if (ix.hloc_bytes == 2)
        hloc_kernel<uint16_t><<<blocks, 256, smem, s>>>(Ht, ix.inv, ix.o, ix.n, ix.m, ix.hloc_stride, out);
    else
        hloc_kernel<uint32_t><<<blocks, 256, smem, s>>>(Ht, ix.inv, ix.o, ix.n, ix.m, ix.hloc_stride, out);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

qw_status launch_bm_collect(const IndexView &ix, int nb, int l, int cap, QueryState &st,
                            int64_t *stats_out, bool sorted, cudaStream_t s)
{
    int P2 = 2;
    while (P2 < cap) P2 <<= 1;
    // (within the 48 KiB that every launch may have)
    static_assert(QW_MAX_CAND * sizeof(uint64_t) + 2048 <= 48 << 10, "keys and the block's counts");
    const size_t smem = sorted ? (size_t)P2 * sizeof(uint64_t) : 0;
    bm_select_kernel<<<nb, SEL_THREADS, smem, s>>>(ix, l, cap, st, stats_out, sorted);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

// (the final buckets, one or two passes for slots, the listing; the rebuild's five;
// the selection and the list of queries to answer again)
int bm_select_launches(int nb, bool staged, int wave_slots, bool learned)
{
    return (staged ? 1 : 0) + (nb > wave_slots ? 2 : 1) + 1 + 5 + (learned ? 2 : 0) + 2;
}

qw_status launch_bm_list(const IndexView &ix, int nb, int l, int cgrow, QueryState &st,
                         bool staged, int wave_slots, cudaStream_t s)
{
    if (nb == 0) return QW_OK;
    if (staged) {
        const int64_t e = (int64_t)nb * st.bm_mp;
        bm_final_bucket_kernel<<<(unsigned)std::min<int64_t>((e + 255) / 256, 152 * 8), 256, 0, s>>>(
            ix, nb, st);
        QW_CUDA_TRY(cudaGetLastError());
    }
    // slots of the rebuild: the lists that would overflow and the long ones; where
    // the store (wave_slots) has no place for every query, the former first
    const unsigned qb = (unsigned)(((int64_t)nb * 32 + 127) / 128);
    QW_CUDA_TRY(cudaMemsetAsync(st.rd_ctl, 0, 2 * sizeof(int32_t), s));
    rd_compact_kernel<<<qb, 128, 0, s>>>(ix, cgrow, st, nb, nb <= wave_slots ? kQDirect : kQCap,
                                         INT32_MAX, wave_slots);
    if (nb > wave_slots)
        rd_compact_kernel<<<qb, 128, 0, s>>>(ix, cgrow, st, nb, kQDirect, kQCap, wave_slots);
    const int64_t quads = (int64_t)nb * ((ix.nT + 3) / 4);
    int parts = quads <= 65536 ? 4 : 1;
    while (parts < 32 && quads * parts * 2 <= kCountWarps) parts *= 2;
    bm_list_kernel<<<(unsigned)std::min<int64_t>((quads * parts + 7) / 8, 152 * 24), 256, 0, s>>>(
        ix, l, nb, parts, quads * parts <= kCountWarps, st);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

int bm_reduce_wave(int nT)
{
    return (int)std::max<int64_t>(1, kRdStoreBytes / ((int64_t)nT * kBmUint4 * kRdStoreWords * 16));
}

qw_status launch_bm_reduce(const IndexView &ix, int nb, int l, int cap, int cgrow,
                           QueryState &st, int wave_slots, cudaStream_t s)
{
    if (nb == 0) return QW_OK;
    // one store's worth of slots (wave_slots); queries past it keep the
    // level-path answer
    const unsigned grid = 152 * 12;
    const unsigned pb = (unsigned)((wave_slots + 127) / 128);
    rd_count_kernel<<<grid, RD_THREADS, 0, s>>>(ix, l, cap, st, wave_slots);
    rd_plan_kernel<<<pb, 128, 0, s>>>(l, ix.m, cap, cgrow, st, wave_slots, 0);
    rd_scan_kernel<<<152 * 2, RS_THREADS, 0, s>>>(ix, st, wave_slots);
    rd_emit_kernel<<<grid, RD_THREADS, 0, s>>>(ix, l, st, wave_slots);
    rd_plan_kernel<<<pb, 128, 0, s>>>(l, ix.m, cap, cgrow, st, wave_slots, 2);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

qw_status launch_bm_overflow_list(const QueryState &st, int nb, const int32_t *order_perm,
                                  int64_t b0, int32_t *list0, int32_t *list1, int32_t *count,
                                  cudaStream_t s)
{
    bm_overflow_list_kernel<<<(nb + 255) / 256, 256, 0, s>>>(st, nb, order_perm, b0, list0, list1,
                                                             count);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

}  // namespace qw
