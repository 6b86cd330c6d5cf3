// qw_query.cu -- the query side of collision counting with virtual rehashing.
//
// For every query of a batch the host runs levels L = 0, 1, 2, ... with radius
// R = c^L (Section 2, C2LSH virtual rehashing).  At radius R the bucket of
// projection i is floor(bid / R); a data object collides with the query on
// projection i when its bid lies in [beta_i R, beta_i R + R - 1],
// beta_i = floor(g_i / R), g_i = h_i(q) - o_i.  Its collision count is the
// number of such projections, and it is a candidate when the count reaches
// the threshold l (Section 3.1).
//
// Ranges nest from one level to the next, so a level only scans the entries
// of the two new flanks of every projection's range and adds them to the
// running counts.  Counts live in one byte per (query, data id): 7 bits of
// count (m <= 127) and a flag bit meaning "was a candidate at the previous
// level", which orders the truncation to k + v candidates.
//
// One CTA owns one (index tile, query): it stages the tile's counters in
// shared memory, range-searches the tile's bucket directory for the flank
// boundaries of all m projections, increments the counters of every id in the
// flanks, counts the ids whose count reaches l, and writes the counters back.
#include "qw_internal.cuh"
#include "qw_count.cuh"
#include "qw_dir.cuh"
#include "qw_scan.cuh"

#include <algorithm>
#include <climits>

#include <cuda_pipeline.h>

namespace qw {
namespace {

constexpr int LV_THREADS = 256;
constexpr int kWordsPerTile = kTile / 4;
constexpr int kUnroll = 4;

// One warp per query.
__global__ void query_setup_kernel(const int32_t *__restrict__ HQ, int nb, int m,
                                   const int32_t *__restrict__ o,
                                   const int32_t *__restrict__ span, QueryState st)
{
    const int q = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (q >= nb) return;
    int64_t top = 0;
    for (int i = lane; i < m; i += 32) {
        int64_t g = (int64_t)HQ[(int64_t)q * m + i] - (int64_t)o[i];
        st.g[(int64_t)q * m + i] = g;
        top = max(top, max((int64_t)span[i], g));
        // with probes a query bucket id below the data collides once R > -g
        if (st.probes > 0) top = max(top, -g);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
        top = max(top, (int64_t)__shfl_xor_sync(0xffffffffu, (long long)top, off));
    if (lane != 0) return;
    st.top[q] = top;
    st.active[q] = 1;
    st.ncand[q] = 0;
    st.nprev[q] = 0;
    st.cross[q] = 0;
    st.term[q] = 0;
    st.levels[q] = 0;
    st.finalR[q] = 0;
    st.scan_level[q] = 0;
    st.scan_last[q] = 0;
    st.scan_full[q] = 0;
    st.nkeep[q] = 0;
    st.start[q] = 0;
    st.fb[q] = 0;
    if (st.recount) st.recount[q] = 0;
    if (st.bm_ovf) st.bm_ovf[q] = 0;
    if (st.qbuf_n) {
        st.qbuf_n[q] = 0;
        st.qbuf_n[st.qbn_par + q] = 0;
    }
    atomicMax(st.max_top, (unsigned long long)top);
}

// Queries that stopped at a learned first level > 0 start over from level 0;
// fb_count[0] += their number, fb_count[1] += levels skipped by the others.
__global__ void fallback_kernel(int nb, QueryState st)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nb) return;
    if (!st.fb[q]) {
        if (st.start[q]) atomicAdd(st.fb_count + 1, (unsigned long long)st.start[q]);
        return;
    }
    st.fb[q] = 0;
    st.start[q] = 0;
    st.active[q] = 1;
    st.ncand[q] = 0;
    st.nprev[q] = 0;
    st.cross[q] = 0;
    st.term[q] = 0;
    st.levels[q] = 0;
    st.finalR[q] = 0;
    st.scan_level[q] = 0;
    st.scan_last[q] = 0;
    st.scan_full[q] = 0;
    if (st.qbuf_n) {
        st.qbuf_n[q] = 0;
        st.qbuf_n[st.qbn_par + q] = 0;
    }
    atomicAdd(st.fb_count, 1ull);
}

// One level of one (tile, query).  Bound by the shared-memory pipe: an atomic of
// a warp takes two passes over the banks on average (ids of a bucket cycle
// through the banks in uneven groups), 93 % of the pipe at a deep level, and at
// the first levels by instructions, 65 % of the issue slots.  1,000 queries on
// 500,000 points, 64 projections, levels 0-4: 635 792 979 1345 1984 us with one
// thread per projection searching its ends in turn, every thread stepping over
// all flanks and the ids outside whole chunks masked in the main loop;
// 424 466 592 864 1399 us so.  Forty registers (six blocks per SM) gain nothing
// here and cost QALSH's searches 20 %.
__global__ void __launch_bounds__(LV_THREADS) level_kernel(IndexView ix, int level, int64_t R,
                                                           int64_t Rp, int l, int cgrow,
                                                           QueryState st, int64_t words_per_query,
                                                           const LoopCtl *ctl)
{
    __shared__ __align__(16) uint32_t cnt_s[kWordsPerTile];
    __shared__ int32_t f_end[4][QW_MAX_M];
    __shared__ uint32_t f_run[2 * QW_MAX_M];        // flank's tile offsets: lo | hi << 16
    __shared__ int32_t f_cpref[2 * QW_MAX_M + 1];   // exclusive prefix of its whole chunks
    __shared__ int32_t wsum[LV_THREADS / 32];
    __shared__ int hist[kHistBins];
    __shared__ int32_t red_count;
    __shared__ unsigned long long red_scan;

    const int t = blockIdx.x;
    const int q = blockIdx.y;
    if (!st.active[q]) return;
    if (ctl) {
        level = ctl->level;
        R = ctl->R;
        Rp = ctl->Rp;
    }
    const int qstart = st.start[q];
    if (level < qstart) return;
    // the query's first level counts its whole range from zeroed counters
    const bool first = level == qstart;
    const int m = ix.m;
    const int64_t n = ix.n;
    const int64_t tbase = (int64_t)t * kTile;
    const int len = (int)min((int64_t)kTile, n - tbase);
    if (threadIdx.x == 0) {
        red_count = 0;
        red_scan = 0;
    }
    for (int c = threadIdx.x; c < kHistBins; c += LV_THREADS) hist[c] = 0;

    // the tile's counters on their way into shared memory while the flanks are
    // searched for
    uint4 *cg = reinterpret_cast<uint4 *>(st.counters + (int64_t)q * words_per_query +
                                          (int64_t)t * kWordsPerTile);
    uint4 *cs = reinterpret_cast<uint4 *>(cnt_s);
    if (first) {
#pragma unroll
        for (int r = 0; r < kWordsPerTile / 4 / LV_THREADS; ++r)
            cs[r * LV_THREADS + threadIdx.x] = make_uint4(0, 0, 0, 0);
    } else {
#pragma unroll
        for (int r = 0; r < kWordsPerTile / 4 / LV_THREADS; ++r)
            __pipeline_memcpy_async(cs + r * LV_THREADS + threadIdx.x,
                                    cg + r * LV_THREADS + threadIdx.x, 16);
        __pipeline_commit();
    }

    // 1. flank boundaries: the ends of this level's range of every projection
    //    and, unless it is the first, of the previous level's (ranges nest, so
    //    only the two new flanks are read; the ends of a previous range without
    //    data coincide); one search per thread, end b of projection i in
    //    f_end[b][i]
    const int ends = (first ? 2 : 4) * m;
    for (int j = threadIdx.x; j < ends; j += LV_THREADS) {
        const int b = j / m, i = j - b * m;
        const int64_t rad = b < 2 ? R : Rp;
        int pos;
        if (ix.qkey) {
            // QALSH: the run of the tile's sorted projections inside the
            // interval p_i(q) +- qhalf R
            const double h = __dmul_rn(ix.qhalf, (double)rad);
            const double pq = __longlong_as_double((long long)st.g[(int64_t)q * m + i]);
            const double *kk = ix.qkey + (int64_t)i * ix.nT * kTile + tbase;
            int lo = 0, hi = len;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                const double dk = __dsub_rn(kk[mid], pq);
                if ((b & 1) ? !(dk > h) : dk < -h) lo = mid + 1; else hi = mid;
            }
            pos = lo;
        } else {
            const int64_t dslot = (int64_t)i * ix.nT + t;
            const int64_t ds = ix.dir_start[dslot];
            const int64_t sp1 = (int64_t)ix.span[i] + 1;
            const int cnt = ix.dir_cnt[dslot];
            // the level's bid range, widened to P buckets on each side with probes
            const int64_t P = st.probes;
            int64_t lo = (floordiv64(st.g[(int64_t)q * m + i], rad) - P) * rad;
            if (b & 1) lo += (2 * P + 1) * rad;
            pos = dir_lower(ix.dir_bid + ds, ix.dir_off + ds, cnt, len, clamp64(lo, 0, sp1));
        }
        f_end[b][i] = pos;
    }
    if (first && level > 0 && !ix.qkey && threadIdx.x < m) {
        // entries in the ranges of the skipped levels, for the statistics
        const int i = threadIdx.x;
        const int64_t gi = st.g[(int64_t)q * m + i];
        const int64_t sp1 = (int64_t)ix.span[i] + 1;
        const int64_t dslot = (int64_t)i * ix.nT + t;
        const int32_t *ub = ix.dir_bid + ix.dir_start[dslot];
        const int32_t *uo = ix.dir_off + ix.dir_start[dslot];
        const int cnt = ix.dir_cnt[dslot];
        const int64_t P = st.probes;
        unsigned long long skipped = 0;
        int64_t Rs = R;
        for (int L2 = level - 1; L2 >= 0; --L2) {
            Rs /= cgrow;
            const int64_t lo3 = (floordiv64(gi, Rs) - P) * Rs;
            const int64_t A3 = clamp64(lo3, 0, sp1), B3 = clamp64(lo3 + (2 * P + 1) * Rs, 0, sp1);
            skipped += (unsigned long long)(dir_lower(ub, uo, cnt, len, B3) -
                                            dir_lower(ub, uo, cnt, len, A3));
        }
        if (skipped) atomicAdd(reinterpret_cast<unsigned long long *>(st.scan_full + q), skipped);
    }
    __syncthreads();
    unsigned long long my_scan = 0;
    int my_c0 = 0, my_c1 = 0;
    if (threadIdx.x < m) {
        const int i = threadIdx.x;
        const int pA = f_end[0][i], pB = f_end[1][i];
        int s0 = pA, e0 = pB, s1 = 0, e1 = 0;
        if (!first) {
            e0 = f_end[2][i];
            s1 = f_end[3][i];
            e1 = pB;
        }
        static_assert(kTile <= 65535, "tile offsets are packed in pairs");
        f_run[2 * i] = (uint32_t)s0 | (uint32_t)e0 << 16;
        f_run[2 * i + 1] = (uint32_t)s1 | (uint32_t)e1 << 16;
        my_c0 = max((e0 >> 3) - ((s0 + 7) >> 3), 0);
        my_c1 = max((e1 >> 3) - ((s1 + 7) >> 3), 0);
        my_scan = (unsigned long long)(pB - pA);
    }
    {
        int total;
        const int excl = block_exclusive_scan<LV_THREADS>(my_c0 + my_c1, wsum, &total);
        if (threadIdx.x < m) {
            f_cpref[2 * threadIdx.x] = excl;
            f_cpref[2 * threadIdx.x + 1] = excl + my_c0;
        }
        if (threadIdx.x == 0) f_cpref[2 * m] = total;
    }
    if (my_scan) atomicAdd(&red_scan, my_scan);

    // 2. flag the previous level's candidates, if the query has any
    const uint32_t bias = ge_bias(l);
    if (!first) {
        __pipeline_wait_prior(0);
        if (st.ncand[q] > 0) {
#pragma unroll
            for (int r = 0; r < kWordsPerTile / 4 / LV_THREADS; ++r) {
                uint4 x = cs[r * LV_THREADS + threadIdx.x];
                const uint4 f = make_uint4(ge_bits(x.x, bias), ge_bits(x.y, bias),
                                           ge_bits(x.z, bias), ge_bits(x.w, bias));
                if (!(f.x | f.y | f.z | f.w)) continue;
                cs[r * LV_THREADS + threadIdx.x] =
                    make_uint4(x.x | f.x, x.y | f.y, x.z | f.z, x.w | f.w);
            }
        }
    }
    __syncthreads();

    // 3. count every id in the flanks.  The tile's slots start 16-byte aligned,
    //    so chunk k of a tile's ids is its offsets 8 k .. 8 k + 7.  First the
    //    ids outside a flank's whole chunks (at most 14), 16 places per flank,
    //    kUnroll loads in flight per thread; then the whole chunks, a
    //    contiguous share of the flattened chunk space per warp, so that a lane
    //    steps over its warp's flanks only, kUnroll 16-byte loads in flight and
    //    no id to leave out.
    const uint16_t *lid = ix.lid + tbase;
    const int64_t pstride = (int64_t)ix.nT * kTile;
    for (int j0 = threadIdx.x; j0 < 32 * m; j0 += LV_THREADS * kUnroll) {
        int id[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const int j = j0 + u * LV_THREADS;
            id[u] = -1;
            if (j >= 32 * m) continue;
            const int lo = (int)(f_run[j >> 4] & 0xffffu), hi = (int)(f_run[j >> 4] >> 16);
            const int c0 = (lo + 7) & ~7, c1 = hi & ~7;
            const int k = lo + (j & 15);
            const int at = (c1 > c0 && k >= c0) ? k + (c1 - c0) : k;
            if (at < hi) id[u] = __ldg(lid + (j >> 5) * pstride + at);
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u)
            if (id[u] >= 0) count_id(cnt_s, (uint32_t)id[u]);
    }
    {
        const int total = f_cpref[2 * m];
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const int share = (total + LV_THREADS / 32 - 1) / (LV_THREADS / 32);
        const int wend = min((warp + 1) * share, total);
        int s = -1, c_hi = 0;  // the flank of the lane's last chunk
        const uint4 *p = nullptr;
        if (warp * share < wend) {
            // the last flank that starts at or before the warp's first chunk
            for (int k = lane; k < 2 * m; k += 32)
                if (f_cpref[k] <= warp * share) s = k;
            s = __reduce_max_sync(0xffffffffu, s) - 1;
        }
        for (int e0 = warp * share + lane; e0 < wend; e0 += 32 * kUnroll) {
            uint4 v[kUnroll];
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) {
                const int e = e0 + u * 32;
                if (e >= wend) continue;
                if (e >= c_hi) {
                    do c_hi = f_cpref[++s + 1]; while (e >= c_hi);
                    p = reinterpret_cast<const uint4 *>(lid + (s >> 1) * pstride) +
                        (((f_run[s] & 0xffffu) + 7) >> 3) - f_cpref[s];
                }
                v[u] = __ldg(p + e);
            }
#pragma unroll
            for (int u = 0; u < kUnroll; ++u)
                if (e0 + u * 32 < wend) count_chunk(cnt_s, v[u], 0xffu);
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();

    // 4. counters back to global memory (one bulk copy), and this tile's
    //    candidate profile: previous-level candidates, the others by count
    if (threadIdx.x == 0) {
        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(
                         __cvta_generic_to_global(cg)),
                     "r"((uint32_t)__cvta_generic_to_shared(cs)), "r"((uint32_t)kTile)
                     : "memory");
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    }
    int my_prev = 0, my_count = 0;
#pragma unroll
    for (int r = 0; r < kWordsPerTile / 4 / LV_THREADS; ++r) {
        const uint4 x = cs[r * LV_THREADS + threadIdx.x];
        const uint32_t wv[4] = {x.x, x.y, x.z, x.w};
        const uint32_t ge[4] = {ge_bits(x.x, bias), ge_bits(x.y, bias), ge_bits(x.z, bias),
                                ge_bits(x.w, bias)};
        if (!(ge[0] | ge[1] | ge[2] | ge[3])) continue;
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            my_count += __popc(ge[h]);
            my_prev += __popc(ge[h] & wv[h]);
            for (uint32_t left = ge[h] & ~wv[h]; left; left &= left - 1)
                atomicAdd(&hist[1 + ((wv[h] >> (__ffs(left) - 8)) & 0x7fu)], 1);
        }
    }
    my_prev = __reduce_add_sync(0xffffffffu, my_prev);
    my_count = __reduce_add_sync(0xffffffffu, my_count);
    if ((threadIdx.x & 31) == 0) {
        if (my_prev) atomicAdd(&hist[0], my_prev);
        if (my_count) atomicAdd(&red_count, my_count);
    }
    __syncthreads();
    int *th = st.tile_hist + ((int64_t)q * ix.nT + t) * kHistBins;
    for (int c = threadIdx.x; c < kHistBins; c += LV_THREADS) th[c] = hist[c];
    if (threadIdx.x == 0) {
        if (red_count) atomicAdd(st.cross + q, red_count);
        if (red_scan) atomicAdd(reinterpret_cast<unsigned long long *>(st.scan_level + q), red_scan);
        // the copy has read the counters before the block's memory goes
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    }
}

// Entries of projection i's data with bid in the level-R range of g.
__device__ __forceinline__ int64_t range_entries(const ScanStats &ss, int i, int64_t g, int64_t R)
{
    const int64_t sp1 = (int64_t)ss.span[i] + 1;
    const int64_t lo = floordiv64(g, R) * R;
    const int64_t A = clamp64(lo, 0, sp1), B = clamp64(lo + R, 0, sp1);
    const int64_t *P = ss.prefix + ss.off[i];
    return P[B] - P[A];
}

// One warp per query: the lanes add the entries-scanned statistics over the
// projections (bitmap path), lane 0 takes the decision.
__global__ void decide_kernel(int nb, int level, int64_t R, int cap, QueryState st,
                              LoopCtl *ctl, ScanStats ss)
{
    const int q = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (q >= nb || !st.active[q]) return;
    if (ctl) {
        level = ctl->level;
        R = ctl->R;
    }
    if (level < st.start[q]) {
        // not started yet: the device-driven loop must go on
        if (ctl && lane == 0) atomicAdd(&ctl->active, 1u);
        return;
    }
    const bool first = level == st.start[q];
    int64_t sl = 0, skipped = 0;
    if (ss.prefix) {
        // the same sums as the level kernel's, from the bid prefix counts: this
        // level's ranges, and at a learned first level > 0 the ranges of the
        // levels it skipped
        for (int i = lane; i < ss.m; i += 32) {
            const int64_t g = st.g[(int64_t)q * ss.m + i];
            sl += range_entries(ss, i, g, R);
            if (first && level > 0) {
                int64_t Rs = R;
                for (int L2 = level - 1; L2 >= 0; --L2) {
                    Rs /= ss.cgrow;
                    skipped += range_entries(ss, i, g, Rs);
                }
            }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            sl += __shfl_down_sync(0xffffffffu, sl, off);
            skipped += __shfl_down_sync(0xffffffffu, skipped, off);
        }
    }
    if (lane != 0) return;
    // all reads before the first write: one latency instead of one each
    if (!ss.prefix) sl = st.scan_level[q];
    const int32_t before = st.ncand[q];  // |C_R| of the previous level
    // |C_R| of this level (the bitmap path counts its list, the level path sums tiles)
    const int32_t nc = st.qbuf_n ? st.qbuf_n[(int64_t)(level & 1) * st.qbn_par + q] : st.cross[q];
    const int64_t full = st.scan_full[q], top = st.top[q];
    if (st.level_passes) atomicAdd(st.level_passes, 1ull);
    st.cross[q] = 0;
    st.scan_level[q] = 0;
    st.scan_last[q] = sl;
    st.scan_full[q] = full + skipped + sl;
    st.levels[q] = level + 1;
    st.finalR[q] = R;
    const bool enough = nc >= cap;        // the k + v bound (Section 3.1)
    const bool past = R > top;            // no further level can change C_R
    if ((enough || past) && first && level > 0) {
        if (ss.recount_first) {
            // bitmap path: stop here; the previous level's candidates are
            // recounted from the bitmaps afterwards (and checked)
            st.recount[q] = 1;
        } else {
            // stopped at a learned first level: the previous level is unknown,
            // so the query is answered again from level 0
            st.fb[q] = 1;
            st.active[q] = 0;
            return;
        }
    }
    if (enough || past) {
        st.term[q] = enough ? 2 : 3;
        st.active[q] = 0;
        st.nprev[q] = before;
    } else {
        if (ctl) atomicAdd(&ctl->active, 1u);
        // the next level's candidate list starts empty (bitmap path)
        if (st.qbuf_n) st.qbuf_n[(int64_t)((level + 1) & 1) * st.qbn_par + q] = 0;
    }
    st.ncand[q] = nc;
}

// Graph mode: the level loop runs on the device.  The first pass starts at
// the smallest first level of the batch (0 unless every query has a learned
// start above it): levels below it would do no work.
__global__ void loop_min_start_kernel(LoopCtl *ctl, QueryState st, int nb)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    int s = q < nb ? st.start[q] : INT_MAX;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s = min(s, __shfl_down_sync(0xffffffffu, s, off));
    if ((threadIdx.x & 31) == 0 && s != INT_MAX) atomicMin(&ctl->min_start, s);
}

__global__ void loop_reset_kernel(LoopCtl *ctl)
{
    ctl->min_start = INT_MAX;
    ctl->active = 0;
}

__global__ void loop_init_kernel(LoopCtl *ctl, int cgrow)
{
    const int L = ctl->min_start == INT_MAX ? 0 : ctl->min_start;
    int64_t R = 1, Rp = 1;
    for (int j = 0; j < L; ++j) {
        Rp = R;
        R *= cgrow;
    }
    ctl->level = L;
    ctl->R = R;
    ctl->Rp = Rp;
    ctl->pass = 0;
    ctl->active = 0;
}

// After a level's decision: stop once R exceeds every query's last useful
// radius (after this level no query can still be active), else go to the
// next level.  Mirrors the host loop; level 63 would overflow R and is an
// error (flag 8).
__global__ void loop_ctl_kernel(LoopCtl *ctl, const unsigned long long *max_top, int cgrow,
                                int kernels, cudaGraphConditionalHandle h, int *err)
{
    const int64_t R = ctl->R;
    // stop once R exceeds every useful radius, or no query is left to run
    bool more = (unsigned long long)R <= *max_top && ctl->active > 0;
    ctl->active = 0;
    ctl->iters += 1;
    ctl->kernels += (unsigned long long)kernels;
    if (more && ctl->level > 62) {
        atomicOr(err, 8);
        more = false;
    }
    if (more) {
        ctl->level += 1;
        ctl->Rp = R;
        ctl->R = R * cgrow;
    }
    cudaGraphSetConditional(h, more ? 1u : 0u);
}

// Learned start, graph mode: after the fallback kernel marked the queries that
// stopped at their learned first level, run the loop again from level 0 if
// there are any.
__global__ void second_pass_kernel(QueryState st, LoopCtl *ctl, cudaGraphConditionalHandle h)
{
    ctl->level = 0;
    ctl->R = 1;
    ctl->Rp = 1;
    ctl->pass = 1;
    ctl->active = 0;
    ctl->fb_total += st.fb_count[0];
    ctl->skipped_total += st.fb_count[1];
    cudaGraphSetConditional(h, st.fb_count[0] > 0 ? 1u : 0u);
}

constexpr int CL_THREADS = 256;

// Plan the kept candidates of one query from the per-tile profiles of its
// last level: all ids with count >= l when there are at most k + v of them;
// otherwise the previous level's candidates, then by count descending, then by
// id ascending, up to k + v.  The boundary count c* splits the ids with count
// above it (all kept) from those equal to it (the first take_eq by id kept).
// Writes, per tile, where its kept ids start in the query's list and how many
// count-c* ids precede it; and the query's statistics.
__global__ void __launch_bounds__(CL_THREADS) select_plan_kernel(
    int nT, int m, int l, int cap, QueryState st, int64_t *__restrict__ stats_out)
{
    __shared__ int tot[kHistBins];
    __shared__ int s_cstar, s_take_eq;
    __shared__ int scan_tmp[CL_THREADS / 32];
    const int q = blockIdx.x;
    const int nc = st.ncand[q];
    const int np = st.nprev[q];
    const int *qh = st.tile_hist + (int64_t)q * nT * kHistBins;
    if (threadIdx.x == 0) {
        s_cstar = l - 1;
        s_take_eq = 0;
    }
    if (nc > cap) {
        for (int c = threadIdx.x; c < kHistBins; c += CL_THREADS) {
            int sum = 0;
            for (int t = 0; t < nT; ++t) sum += qh[(int64_t)t * kHistBins + c];
            tot[c] = sum;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            const int need = cap - np;
            int acc = 0;
            for (int c = m; c >= l; --c) {
                const int hc = tot[1 + c];
                if (acc + hc >= need) {
                    s_cstar = c;
                    s_take_eq = need - acc;
                    break;
                }
                acc += hc;
            }
        }
    }
    __syncthreads();
    const int cstar = s_cstar, take_eq = s_take_eq;
    // per tile: kept ids above c*, and ids at c*, then prefixes over tiles
    int eq_base = 0, out_base = 0;
    for (int t0 = 0; t0 < nT; t0 += CL_THREADS) {
        const int t = t0 + threadIdx.x;
        int above = 0, eq = 0;
        if (t < nT) {
            const int *th = qh + (int64_t)t * kHistBins;
            above = th[0];
            for (int c = max(cstar + 1, l); c <= m; ++c) above += th[1 + c];
            eq = (cstar >= l) ? th[1 + cstar] : 0;
        }
        int eq_tot;
        const int eq_ex = eq_base + block_exclusive_scan<CL_THREADS>(eq, scan_tmp, &eq_tot);
        const int kept = above + min(max(take_eq - eq_ex, 0), eq);
        int kept_tot;
        const int out_ex = out_base + block_exclusive_scan<CL_THREADS>(kept, scan_tmp, &kept_tot);
        if (t < nT) {
            st.tile_plan[((int64_t)q * nT + t) * 3 + 0] = out_ex;
            st.tile_plan[((int64_t)q * nT + t) * 3 + 1] = eq_ex;
            st.tile_plan[((int64_t)q * nT + t) * 3 + 2] = kept;
        }
        eq_base += eq_tot;
        out_base += kept_tot;
    }
    if (threadIdx.x == 0) {
        const int keep = min(out_base, cap);
        st.nkeep[q] = keep;
        st.qplan[q * 2 + 0] = cstar;
        st.qplan[q * 2 + 1] = take_eq;
        if (stats_out) {
            int64_t *so = stats_out + (int64_t)q * QW_NSTAT;
            so[0] = st.levels[q];
            so[1] = st.finalR[q];
            so[2] = nc;
            so[3] = keep;
            so[4] = st.term[q];
            so[5] = st.scan_last[q];
            so[6] = st.scan_full[q];
            so[7] = np;
        }
    }
    // pad the list (the emit kernel fills [0, keep))
    const int keep = min(out_base, cap);
    for (int p = keep + threadIdx.x; p < cap; p += CL_THREADS) {
        st.cand[(int64_t)q * cap + p] = -1;
        st.cand_col[(int64_t)q * cap + p] = 0;
    }
}

// Emit the kept ids of one (tile, query) in ascending order at the tile's
// planned position.  The block reads the tile's counters as eight coalesced
// rows of 16 ids per thread; a thread counts its ids kept outright and those at
// c* per row, and one scan over the (row, warp) totals of both gives every
// thread its first output slot.  Bound by reading the counters (32 KiB per tile
// and query): 568 us for 1,000 queries on 500,000 points with a thread per 128
// consecutive ids walking its words in local memory, 174 us so.
constexpr int EM_ROWS = kTile / (CL_THREADS * 16);  // 8
constexpr int EM_WARPS = CL_THREADS / 32;

// First places of the (row, warp, lane) entries, in that order, of v[r]: tot is
// EM_ROWS * EM_WARPS words of shared memory.  Returns them in v.
__device__ __forceinline__ void emit_scan(uint32_t (&v)[EM_ROWS], uint32_t *tot)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t mine[EM_ROWS];
#pragma unroll
    for (int r = 0; r < EM_ROWS; ++r) {
        uint32_t incl = v[r];
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += y;
        }
        mine[r] = incl - v[r];
        if (lane == 31) tot[r * EM_WARPS + warp] = incl;
    }
    __syncthreads();
    static_assert(EM_ROWS * EM_WARPS == 64, "two totals per lane");
    if (warp == 0) {
        const uint32_t x = tot[2 * lane], y = tot[2 * lane + 1];
        uint32_t incl = x + y;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t z = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += z;
        }
        tot[2 * lane] = incl - x - y;
        tot[2 * lane + 1] = incl - y;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < EM_ROWS; ++r) v[r] = mine[r] + tot[r * EM_WARPS + warp];
}

__global__ void __launch_bounds__(CL_THREADS, 4) select_emit_kernel(
    int nT, int l, int cap, QueryState st, int64_t words_per_query)
{
    __shared__ uint32_t tot[EM_ROWS * EM_WARPS];
    const int t = blockIdx.x;
    const int q = blockIdx.y;
    const int cstar = st.qplan[q * 2 + 0], take_eq = st.qplan[q * 2 + 1];
    const int *plan = st.tile_plan + ((int64_t)q * nT + t) * 3;
    if (plan[2] == 0) return;  // nothing kept in this tile: skip its counters
    const int out0 = plan[0];
    const int eq0 = plan[1];
    const int64_t tbase = (int64_t)t * kTile;
    // counters are allocated for whole tiles; ids past n hold zero
    const uint4 *cb = reinterpret_cast<const uint4 *>(
                          reinterpret_cast<const uint8_t *>(st.counters + (int64_t)q * words_per_query) +
                          tbase) + threadIdx.x;
    // bit 7 of the bytes to keep outright (previous-level candidates and counts
    // above c*), and of the others at c*
    const uint32_t bias = ge_bias(l), abias = ge_bias(min(max(cstar + 1, l), 128));
    const bool ties = cstar >= l;
    const uint32_t cbias = ge_bias(min(max(cstar, l), 128));
    auto at_of = [&](uint32_t x) { return ge_bits(x, cbias); };  // at c* where not kept outright
    auto above_of = [&](uint32_t x) { return ge_bits(x, abias) | (ge_bits(x, bias) & x); };
    uint4 v[EM_ROWS];
#pragma unroll
    for (int r = 0; r < EM_ROWS; ++r) v[r] = cb[r * CL_THREADS];
    // ids kept outright in the low half, ids at c* in the high one: at most
    // kTile together
    uint32_t first[EM_ROWS];
    int any = 0;
#pragma unroll
    for (int r = 0; r < EM_ROWS; ++r) {
        const uint32_t w[4] = {v[r].x, v[r].y, v[r].z, v[r].w};
        first[r] = 0;
        if (!(ge_bits(w[0], bias) | ge_bits(w[1], bias) | ge_bits(w[2], bias) |
              ge_bits(w[3], bias)))
            continue;
        any |= 1 << r;
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const uint32_t ab = above_of(w[h]);
            first[r] += (uint32_t)__popc(ab);
            if (ties) first[r] += (uint32_t)__popc(at_of(w[h]) & ~ab) << 16;
        }
    }
    emit_scan(first, tot);
    if (!any) return;
    const int left_eq = max(take_eq - eq0, 0);  // ids at c* that this tile may keep
    int32_t *cand = st.cand + (int64_t)q * cap, *col = st.cand_col + (int64_t)q * cap;
#pragma unroll
    for (int r = 0; r < EM_ROWS; ++r) {
        if (!((any >> r) & 1)) continue;
        const uint32_t w[4] = {v[r].x, v[r].y, v[r].z, v[r].w};
        int rk = (int)(first[r] >> 16);
        int pos = out0 + (int)(first[r] & 0xffffu) + min(rk, left_eq);
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const uint32_t ab = above_of(w[h]), eq = ties ? at_of(w[h]) & ~ab : 0u;
            for (uint32_t left = ab | eq; left; left &= left - 1) {
                const int sh = __ffs(left) - 8;
                if (!((ab >> sh) & 0x80u) && rk++ >= left_eq) continue;
                if (pos < cap) {
                    cand[pos] = (int32_t)(tbase + (r * CL_THREADS + (int)threadIdx.x) * 16 + h * 4 +
                                          (sh >> 3));
                    col[pos] = (int)((w[h] >> sh) & 0x7fu);
                }
                ++pos;
            }
        }
    }
}

__global__ void candidates_out_kernel(const int32_t *__restrict__ cand,
                                      const int32_t *__restrict__ cand_col, int64_t total,
                                      int64_t *__restrict__ ids_out, int32_t *__restrict__ col_out)
{
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        ids_out[e] = (int64_t)cand[e];
        if (col_out) col_out[e] = cand_col[e];
    }
}

__global__ void sum_i32_kernel(const int32_t *__restrict__ v, int n, unsigned long long *out)
{
    unsigned long long acc = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) acc += v[i];
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if ((threadIdx.x & 31) == 0 && acc) atomicAdd(out, acc);
}

}  // namespace

qw_status launch_sum_i32(const int32_t *v, int n, unsigned long long *out, cudaStream_t s)
{
    sum_i32_kernel<<<std::min(152, (n + 255) / 256 + 1), 256, 0, s>>>(v, n, out);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

qw_status launch_candidates_out(const QueryState &st, int nb, int cap, int64_t *cand_ids,
                                int32_t *cand_col, cudaStream_t s)
{
    const int64_t total = (int64_t)nb * cap;
    int64_t blocks = std::min<int64_t>((total + 255) / 256, 152 * 8);
    candidates_out_kernel<<<(unsigned)blocks, 256, 0, s>>>(st.cand, st.cand_col, total, cand_ids,
                                                           cand_col);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

qw_status launch_query_setup(const IndexView &ix, const int32_t *HQ, int nb, QueryState &st,
                             cudaStream_t s)
{
    QW_CUDA_TRY(cudaMemsetAsync(st.max_top, 0, sizeof(unsigned long long), s));
    query_setup_kernel<<<(unsigned)(((int64_t)nb * 32 + 127) / 128), 128, 0, s>>>(HQ, nb, ix.m, ix.o, ix.span, st);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

// A learned first level never lies past the query's own last useful level,
// the first L with c^L > top (there the radius rule stops the plain path, and
// the level loops run at least that far for every query of the batch); a
// later prediction would leave the query unstarted.
__global__ void clamp_start_kernel(QueryState st, int nb, int cgrow)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nb) return;
    int L = 0;
    for (int64_t R = 1; R <= st.top[q]; R *= cgrow) ++L;
    if (st.start[q] > L) st.start[q] = L;
}

qw_status launch_clamp_start(int nb, QueryState &st, int cgrow, cudaStream_t s)
{
    if (nb == 0) return QW_OK;
    clamp_start_kernel<<<(nb + 127) / 128, 128, 0, s>>>(st, nb, cgrow);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

qw_status launch_level(const IndexView &ix, int nb, int level, int64_t R, int64_t Rp, int l,
                       int cgrow, QueryState &st, cudaStream_t s, const LoopCtl *ctl)
{
    const int64_t wpq = (int64_t)ix.nT * kWordsPerTile;
    level_kernel<<<dim3((unsigned)ix.nT, (unsigned)nb), LV_THREADS, 0, s>>>(ix, level, R, Rp, l,
                                                                           cgrow, st, wpq, ctl);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

qw_status launch_loop_init(LoopCtl *ctl, const QueryState &st, int nb, int cgrow, cudaStream_t s)
{
    loop_reset_kernel<<<1, 1, 0, s>>>(ctl);
    QW_CUDA_TRY(cudaGetLastError());
    loop_min_start_kernel<<<(nb + 255) / 256, 256, 0, s>>>(ctl, st, nb);
    QW_CUDA_TRY(cudaGetLastError());
    loop_init_kernel<<<1, 1, 0, s>>>(ctl, cgrow);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

qw_status launch_loop_ctl(LoopCtl *ctl, const unsigned long long *max_top, int cgrow, int kernels,
                          cudaGraphConditionalHandle h, int *err, cudaStream_t s)
{
    loop_ctl_kernel<<<1, 1, 0, s>>>(ctl, max_top, cgrow, kernels, h, err);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

qw_status launch_fallback_graph(int nb, QueryState &st, LoopCtl *ctl, cudaGraphConditionalHandle h,
                                cudaStream_t s)
{
    fallback_kernel<<<(nb + 127) / 128, 128, 0, s>>>(nb, st);
    QW_CUDA_TRY(cudaGetLastError());
    second_pass_kernel<<<1, 1, 0, s>>>(st, ctl, h);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

qw_status launch_fallback(int nb, QueryState &st, cudaStream_t s)
{
    fallback_kernel<<<(nb + 127) / 128, 128, 0, s>>>(nb, st);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

qw_status launch_decide(int nb, int level, int64_t R, int cap, QueryState &st, cudaStream_t s,
                        LoopCtl *ctl, const ScanStats &ss)
{
    decide_kernel<<<(unsigned)(((int64_t)nb * 32 + 127) / 128), 128, 0, s>>>(nb, level, R, cap, st,
                                                                            ctl, ss);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

qw_status launch_select_plan(const IndexView &ix, int nb, int l, int cap, QueryState &st,
                             int64_t *stats_out, cudaStream_t s)
{
    select_plan_kernel<<<nb, CL_THREADS, 0, s>>>(ix.nT, ix.m, l, cap, st, stats_out);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

qw_status launch_collect(const IndexView &ix, int nb, int l, int cap, QueryState &st,
                         int64_t *stats_out, cudaStream_t s)
{
    const int64_t wpq = (int64_t)ix.nT * kWordsPerTile;
    QW_TRY(launch_select_plan(ix, nb, l, cap, st, stats_out, s));
    select_emit_kernel<<<dim3((unsigned)ix.nT, (unsigned)nb), CL_THREADS, 0, s>>>(ix.nT, l, cap, st,
                                                                                wpq);
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

}  // namespace qw
