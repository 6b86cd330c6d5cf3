// qw_project.cu -- the projection step of the hash family (Section 3):
//   h_i(v) = floor((a_i . v + b_i) / w),   a_i ~ N(0, I), b_i ~ U[0, w).
//
// Pass 1 (FP32, tiled over rows x projections) computes t = a_i . v with FP32
// fused multiply-adds summed over j = 0..d-1 in order, then u = (t + b_i) / w
// with FP32 operations.  Each fused multiply-add rounds once, and in a
// recursive sum the rounding errors add up without being amplified, so the
// error of t is at most u / (1 - u) * sum_j |s_j|, s_j the computed partial
// sums (u = 2^-24).  |s_j| is at most (1 + 2 d u) times the product of the
// norms of the first j coordinates of a_i and of v (Cauchy-Schwarz), and so, by
// the same inequality over j,
//   sum_j |s_j| <= (1 + 2 d u) W(a_i) W(v),  W(x)^2 = sum_j (d - j) x_j^2
// (j from 0): one number per row and one per projection, formed in FP32 and
// enlarged by 1 % for their own rounding, where a sum of magnitudes per entry
// would take as many registers as the sums themselves.  Adding b and dividing
// by w add at most 3u |u| + u.  Whenever the distance of u to the nearest
// integer is not larger than that bound (or than 1e-5, i.e. 1e-5 w in
// projection units, whichever is larger), floor(u) is not trusted and the entry
// goes to the block's list: 0.15 % of them at d = 128 on the benchmark's data, and
// more as the rows' norm grows against w.  1,000,000 x 128 x 64, unit spread about
// 0, 10, 100, 1,000 and 10,000, w = 4: 0.03, 0.3, 2.5, 25 and 100 % of the entries,
// 512, 514, 710, 2,465 and 8,102 us (with an error sum per entry and FP64 for all
// that it left open 1,498, 1,975, 6,595, 36,772 and 62,457).
//
// Pass 2 (same block) recomputes the listed entries, eight lanes each, in
// pairs of floats: products and sums are split into a rounded value and its
// exact error (fused multiply-add; Knuth's two-sum), the errors summed apart,
// so t is known to about 2^-40 of sum_j |a_j v_j|.  Where even that leaves the
// floor open, the entry is recomputed in FP64 with the dot product summed in
// index order, each product and sum correctly rounded (no fused multiply-add),
// then (t + b) / w in double and floor: the same sequence of IEEE operations as
// the FP64 definition, so the bucket id equals it exactly.  (FP64 runs at two
// lanes a clock and SM here: recomputing all listed entries with it took 405 us
// of a 1,000,000 x 128 x 64 block, beside 1,055 us for pass 1.)
#include "qw_internal.cuh"
#include "qw_tc.cuh"

#include <cuda_bf16.h>
#include <float.h>

#include <algorithm>

namespace qw {
namespace {

constexpr int BK = 16;   // dimension chunk
constexpr int NT = 256;  // threads
// rows, and entries, up to which project_rows_kernel serves
constexpr int64_t kFewRows = 256, kFewEntries = (int64_t)1 << 20;
constexpr float kU = 5.9604645e-08f;  // 2^-24

// What the second pass and the epilogues need of a call.
struct HashArgs {
    const float *V;
    int64_t nv;
    int d;
    const float *A;
    const float *b;
    int m;
    float w;
    int32_t *H;
    int64_t ld_row, ld_col;
    int *err;
    unsigned long long *fixups;
    bool vec;  // rows of V and A in 16-byte pieces (d a multiple of 4, bases aligned)
};

// (hi, lo) += a * v, the product and the sum of the high parts without loss.
__device__ __forceinline__ void pair_fma(float &hi, float &lo, float a, float v)
{
    const float p = __fmul_rn(a, v);
    const float pe = fmaf(a, v, -p);
    const float s = __fadd_rn(hi, p);
    const float z = __fsub_rn(s, hi);
    const float se = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, z)), __fsub_rn(p, z));
    hi = s;
    lo = __fadd_rn(lo, __fadd_rn(se, pe));
}

// a_i . v_r as a pair of floats over the eight lanes of a group (lane8 = 0..7;
// every lane of the warp calls it; idle groups pass valid = false).
__device__ __forceinline__ float2 pair_dot(const HashArgs &h, int64_t r, int i, bool valid,
                                           int lane8)
{
    float hi = 0.0f, lo = 0.0f;
    if (valid) {
        const float *v = h.V + r * (int64_t)h.d, *a = h.A + (int64_t)i * h.d;
        if (h.vec) {
#pragma unroll 4
            for (int j = 4 * lane8; j < h.d; j += 32) {
                const float4 x = __ldg(reinterpret_cast<const float4 *>(v + j));
                const float4 y = __ldg(reinterpret_cast<const float4 *>(a + j));
                pair_fma(hi, lo, y.x, x.x);
                pair_fma(hi, lo, y.y, x.y);
                pair_fma(hi, lo, y.z, x.z);
                pair_fma(hi, lo, y.w, x.w);
            }
        } else {
            for (int j = lane8; j < h.d; j += 8) pair_fma(hi, lo, __ldg(a + j), __ldg(v + j));
        }
    }
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {
        const float oh = __shfl_xor_sync(0xffffffffu, hi, off);
        const float ol = __shfl_xor_sync(0xffffffffu, lo, off);
        const float s = __fadd_rn(hi, oh);
        const float z = __fsub_rn(s, hi);
        const float se = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, z)), __fsub_rn(oh, z));
        hi = s;
        lo = __fadd_rn(__fadd_rn(lo, ol), se);
    }
    return make_float2(hi, lo);
}

// W(x) from its FP32 sum of weighted squares, an upper bound (squares
// that underflow lose less than d 2^-149 each; overflow gives +inf, and then
// every entry of the vector takes the FP64 pass).
__device__ __forceinline__ float norm_bound(float sumsq, int d)
{
    return sqrtf(sumsq + (float)d * ((float)d * 1.4e-45f)) * 1.01f;
}

// Whether u, within rel S / w + 2^-50 |u| or so of the definition's value, may lie
// in another bucket than that.
__device__ __forceinline__ bool open_at(double u, double rel, double S, double w, int d)
{
    const double E = 1.05 * (rel * S + (double)d * 1e-44) / w + fabs(u) * 8.9e-16;
    const double frac = u - floor(u);
    return !(fmin(frac, 1.0 - frac) > E);
}

// (v . a + bias) / w of each open lane's rows v and a, as far as its bucket needs
// it (see settle_entry; apart from it so that its registers are not the callers').
__device__ __noinline__ double open_value(const float *v, const float *a, int d, double bias,
                                          double w, double S, bool open)
{
    const int lane = threadIdx.x & 31;
    double u = 0.0;
    uint32_t mask = __ballot_sync(0xffffffffu, open);
    if (__popc(mask) <= 8) {
        for (; mask; mask &= mask - 1) {
            const int src = __ffs(mask) - 1;
            const float *vr = reinterpret_cast<const float *>(
                __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(v), src));
            const float *ar = reinterpret_cast<const float *>(
                __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(a), src));
            double s = 0.0;
#pragma unroll 4
            for (int j = lane; j < d; j += 32) s = fma((double)__ldg(ar + j), (double)__ldg(vr + j), s);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1)
                s = __dadd_rn(s, __shfl_xor_sync(0xffffffffu, s, off));
            if (lane == src) {
                u = __ddiv_rn(__dadd_rn(s, bias), w);
                open = open_at(u, (double)(d + d / 32 + 8) * 1.1102230246251565e-16, S, w, d);
            }
        }
    }
    if (open) {
        double s = 0.0;
#pragma unroll 8
        for (int j = 0; j < d; ++j)
            s = __dadd_rn(s, __dmul_rn((double)__ldg(a + j), (double)__ldg(v + j)));
        u = __ddiv_rn(__dadd_rn(s, bias), w);
    }
    return u;
}

// Bucket id of each lane's entry (r, i) from its dot product as a pair and S >=
// sum_j |a_j v_j| (W(a) W(v), whose weights are at least 1); every lane of the
// warp calls it, those without an entry with valid = false.  With L terms per lane
// every one of the 2 L additions to the low part, and of the 6 of the lanes' sums,
// rounds a value of at most u (L + 4) S: 2 (L + 4)^2 u^2 S in all; the FP64
// definition is within d 2^-53 S + 2^-51 |u| w of the real value, and so is u
// below.  An entry that this leaves open is summed in FP64 by the warp (d / 32
// fused steps per lane and five sums: (d / 32 + 8) 2^-53 S), and only one that is
// open then takes the definition's own sequence, d dependent additions (67 us at
// d = 512).  At d = 512 one entry in 50,000 is open after the pairs, so a call met
// the sequence in some block: 2,000 rows x 64 took 107 us, 40
// so.  Where more than eight lanes are open they take the sequence side by side
// at once.
__device__ __forceinline__ void settle_entry(const HashArgs &h, int64_t r, int i, float2 t,
                                             double S, bool valid)
{
    const double w = (double)h.w, bias = valid ? (double)h.b[i] : 0.0;
    double u = __ddiv_rn(__dadd_rn(__dadd_rn((double)t.x, (double)t.y), bias), w);
    const double L = (double)(h.d / 8 + 8);
    const bool open = valid && open_at(u, 2.0 * L * L * 3.552713678800501e-15 +
                                              (double)h.d * 1.1102230246251565e-16, S, w, h.d);
    if (__any_sync(0xffffffffu, open)) {
        const double x = open_value(h.V + r * (int64_t)h.d, h.A + (int64_t)i * h.d, h.d, bias, w,
                                    S, open);
        if (open) u = x;
    }
    if (!valid) return;
    const double f = floor(u);
    int32_t *hp = h.H + r * h.ld_row + (int64_t)i * h.ld_col;
    if (!(f >= -2147483647.0 && f <= 2147483646.0)) {
        atomicOr(h.err, 2);
        *hp = 0;
    } else {
        *hp = (int32_t)f;
    }
}

// Pass 1's error of t per unit of W(a) W(v), over w.
__device__ __forceinline__ float sum_unit(int d, float w)
{
    return kU * (1.0f + 4.0f * (float)d * kU) * 1.01f / w;
}

// Whether floor(u) of pass 1 is taken for u = (t + b) / w, E the error of t over w:
// not near an edge, not out of int32, not a NaN.
__device__ __forceinline__ bool sure_at(float u, float f, float E)
{
    const float frac = u - f;                       // exact
    const float eps = fmaxf(E + 4.0f * kU * (fabsf(u) + 1.0f), 1e-5f);
    return fminf(frac, 1.0f - frac) > eps && f >= -2147483520.0f && f <= 2147483520.0f;
}

// Pass 2 of a block: its `count` listed entries (local row << 7 | local
// column; uint16 holds 512 rows of 128), a round of blockDim.x entries at a time: eight lanes per entry form
// the dot products, then one thread per entry settles the bucket id.  vn, an:
// W of the block's rows and projections.  Block-wide.
__device__ void settle_listed(const HashArgs &h, const uint16_t *list, int count, float2 *sums,
                              const float *vn, const float *an, int64_t row0, int col0)
{
    const int nthr = blockDim.x, lane8 = threadIdx.x & 7;
    for (int base = 0; base < count; base += nthr) {
        const int nn = min(nthr, count - base);
        for (int s0 = 0; s0 < nn; s0 += nthr / 8) {
            const int s = s0 + (threadIdx.x >> 3);
            const bool valid = s < nn;
            const int e = valid ? list[base + s] : 0;
            const float2 t = pair_dot(h, row0 + (e >> 7), col0 + (e & 127), valid, lane8);
            if (valid && lane8 == 0) sums[s] = t;
        }
        __syncthreads();
        if ((int)(threadIdx.x & ~31u) < nn) {  // whole warps
            const bool valid = (int)threadIdx.x < nn;
            const int e = list[base + (valid ? (int)threadIdx.x : 0)];
            settle_entry(h, row0 + (e >> 7), col0 + (e & 127), sums[valid ? threadIdx.x : 0],
                         (double)vn[e >> 7] * (double)an[e & 127], valid);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0 && count && h.fixups) atomicAdd(h.fixups, (unsigned long long)count);
}

// Few rows: every entry straight in pairs of floats (pass 2 alone), 32
// entries per block.  The tiled kernel gives at most one block per 64 rows,
// whose dependent chunks take 11.5 us at d = 128 whatever the rows; this form
// takes 5.6 us for 16 rows of 64 projections and 15.8 for 300, hence the limit.
// The entries counted are those that the tiled kernel would list.
__global__ void __launch_bounds__(NT) project_rows_kernel(HashArgs h)
{
    const int64_t e = (int64_t)blockIdx.x * (NT / 8) + (threadIdx.x >> 3);
    const int lane8 = threadIdx.x & 7;
    const bool valid = e < h.nv * h.m;
    const int64_t r = valid ? e / h.m : 0;
    const int i = valid ? (int)(e % h.m) : 0;
    const float2 t = pair_dot(h, r, i, valid, lane8);
    // S from the two weighted norms, eight lanes each
    float sv = 0.0f, sa = 0.0f;
    if (valid)
        for (int j = lane8; j < h.d; j += 8) {
            const float x = __ldg(h.V + r * h.d + j), y = __ldg(h.A + (int64_t)i * h.d + j);
            const float wt = (float)(h.d - j);
            sv = fmaf(wt * x, x, sv);
            sa = fmaf(wt * y, y, sa);
        }
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {
        sv += __shfl_xor_sync(0xffffffffu, sv, off);
        sa += __shfl_xor_sync(0xffffffffu, sa, off);
    }
    const float wv = norm_bound(sv, h.d), wa = norm_bound(sa, h.d);
    const bool mine = valid && lane8 == 0;
    if (h.fixups) {
        const float u = __fmul_rn(__fadd_rn(t.x, valid ? __ldg(h.b + i) : 0.0f), __frcp_rn(h.w));
        const uint32_t near = __ballot_sync(
            0xffffffffu, mine && !sure_at(u, floorf(u), wa * sum_unit(h.d, h.w) * wv));
        if (near && (threadIdx.x & 31) == 0) atomicAdd(h.fixups, (unsigned long long)__popc(near));
    }
    settle_entry(h, r, i, t, (double)wv * (double)wa, mine);
}

// A (32 TM) x (8 TN) tile of entries per block, TM x TN per thread, the operands
// of 16 coordinates at a time in shared memory (8- and 16-byte reads; the next
// 16 are in registers meanwhile).  Shared memory returns 128 bytes a clock, so a
// thread that reads TM + TN floats for TM TN products is bound by it below
// 8 x 8 (16 clocks of reads against 16 of products per warp and coordinate;
// 8 x 4 measured 654 us on 1,000,000 x 128 x 64, the first form with 4 x 4 and
// 4-byte reads 1,055 us, this one 459 us).  TM = 2 serves row counts
// that would leave SMs without a block of 256 rows; where its blocks of 64 rows leave
// SMs without one too, gridDim.z blocks form the same tile and each settles and
// writes its share of the rows: on data far from the origin, where the first pass
// leaves most entries open, a block's second pass takes far longer than its first.
// 300 rows of 512 coordinates about 0, 1,000 and 100,000 (w = 4): 32, 253 and 1,788
// us with a block per tile, 32, 42 and 145 so; 2,000 rows of 128: 12, 39 and 135, now
// 12, 20 and 56.
template <int TM, int TN>
__global__ void __launch_bounds__(NT, 2) project_fp32_kernel(HashArgs h)
{
    constexpr int BM = 32 * TM, BN = 8 * TN;
    constexpr int PV = BM / 64;  // staged 16-byte pieces of V per thread
    static_assert((TM == 2 || TM == 8) && (TN == 4 || TN == 8), "tile shapes");
    struct Tiles {
        float V[BK][BM + 4];
        float A[BK][BN + 4];
    };
    __shared__ __align__(16) union {
        Tiles t[2];  // the chunk being summed and the next
        struct {
            float2 sums[NT];
            uint16_t list[BM * BN];
        } fix;
    } sm;
    __shared__ float vn[BM], an[BN];
    __shared__ int n_list;

    const int tid = threadIdx.x;
    const int tx = tid & 7;    // projections 4 tx .. (and 32 + 4 tx ..)
    const int ty = tid >> 3;   // rows 4 ty .. and 128 + 4 ty .. (TM = 2: 2 ty ..)
    const int64_t row0 = (int64_t)blockIdx.x * BM;
    const int col0 = blockIdx.y * BN;
    const int d = h.d, m = h.m;
    if (tid == 0) n_list = 0;
    auto row_of = [&](int i) { return TM == 8 ? (i < 4 ? 0 : 128) + 4 * ty + (i & 3) : 2 * ty + i; };
    auto col_of = [&](int j) { return (j < 4 ? 0 : 32) + 4 * tx + (j & 3); };

    // staging: piece p of a thread is coordinates 4 (tid & 3) .. + 3 of row
    // tid / 4 + 64 p of V, and of projection tid / 4 of A
    const int sc = 4 * (tid & 3), sr = tid >> 2;
    float4 rv[PV], ra;
    float sqv[PV], sqa = 0.0f;
#pragma unroll
    for (int p = 0; p < PV; ++p) sqv[p] = 0.0f;
    auto load4 = [&](const float *base, int64_t row, bool in, int k) {
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (in && k < d) {
            const float *p = base + row * d + k;
            if (h.vec) {
                x = __ldg(reinterpret_cast<const float4 *>(p));
            } else {
                x.x = __ldg(p);
                if (k + 1 < d) x.y = __ldg(p + 1);
                if (k + 2 < d) x.z = __ldg(p + 2);
                if (k + 3 < d) x.w = __ldg(p + 3);
            }
        }
        return x;
    };
    auto fetch = [&](int k0) {
#pragma unroll
        for (int p = 0; p < PV; ++p)
            rv[p] = load4(h.V, row0 + sr + 64 * p, row0 + sr + 64 * p < h.nv, k0 + sc);
        ra = load4(h.A, col0 + sr, sr < BN && col0 + sr < m, k0 + sc);
    };
    // squares weighted with d - j (coordinates past d are zero)
    auto sq = [](float acc, float4 x, float wt) {
        acc = fmaf(wt * x.x, x.x, acc);
        acc = fmaf((wt - 1.0f) * x.y, x.y, acc);
        acc = fmaf((wt - 2.0f) * x.z, x.z, acc);
        return fmaf((wt - 3.0f) * x.w, x.w, acc);
    };

    float acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = 0.0f;
    auto stage = [&](Tiles &t, int k0) {
        const float wt = (float)(d - k0 - sc);
#pragma unroll
        for (int p = 0; p < PV; ++p) {
            sqv[p] = sq(sqv[p], rv[p], wt);
            t.V[sc + 0][sr + 64 * p] = rv[p].x;
            t.V[sc + 1][sr + 64 * p] = rv[p].y;
            t.V[sc + 2][sr + 64 * p] = rv[p].z;
            t.V[sc + 3][sr + 64 * p] = rv[p].w;
        }
        if (sr < BN) {
            sqa = sq(sqa, ra, wt);
            t.A[sc + 0][sr] = ra.x;
            t.A[sc + 1][sr] = ra.y;
            t.A[sc + 2][sr] = ra.z;
            t.A[sc + 3][sr] = ra.w;
        }
    };
    fetch(0);
    stage(sm.t[0], 0);
    __syncthreads();
    for (int k0 = 0, c = 0; k0 < d; k0 += BK, c ^= 1) {
        const Tiles &t = sm.t[c];
        if (k0 + BK < d) fetch(k0 + BK);
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            float v[TM], a[TN];
            if constexpr (TM == 8) {
                const float4 v0 = *reinterpret_cast<const float4 *>(&t.V[kk][4 * ty]);
                const float4 v1 = *reinterpret_cast<const float4 *>(&t.V[kk][128 + 4 * ty]);
                v[0] = v0.x; v[1] = v0.y; v[2] = v0.z; v[3] = v0.w;
                v[4] = v1.x; v[5] = v1.y; v[6] = v1.z; v[7] = v1.w;
            } else {
                const float2 v0 = *reinterpret_cast<const float2 *>(&t.V[kk][2 * ty]);
                v[0] = v0.x; v[1] = v0.y;
            }
            const float4 a0 = *reinterpret_cast<const float4 *>(&t.A[kk][4 * tx]);
            a[0] = a0.x; a[1] = a0.y; a[2] = a0.z; a[3] = a0.w;
            if constexpr (TN == 8) {
                const float4 a1 = *reinterpret_cast<const float4 *>(&t.A[kk][32 + 4 * tx]);
                a[4] = a1.x; a[5] = a1.y; a[6] = a1.z; a[7] = a1.w;
            }
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(v[i], a[j], acc[i][j]);
        }
        // the other tile was last read before the previous barrier
        if (k0 + BK < d) stage(sm.t[c ^ 1], k0 + BK);
        __syncthreads();
    }
    // W of the rows and projections: the four lanes of a staged row hold pieces
#pragma unroll
    for (int off = 1; off < 4; off <<= 1) {
#pragma unroll
        for (int p = 0; p < PV; ++p) sqv[p] += __shfl_xor_sync(0xffffffffu, sqv[p], off);
        sqa += __shfl_xor_sync(0xffffffffu, sqa, off);
    }
    if ((tid & 3) == 0) {
#pragma unroll
        for (int p = 0; p < PV; ++p) vn[sr + 64 * p] = norm_bound(sqv[p], d);
        if (sr < BN) an[sr] = norm_bound(sqa, d);
    }
    __syncthreads();  // the tiles become the list

    const float w = h.w;
    // dividing by w as a product with its reciprocal: one more rounding, 3 u |u|
    // in all (a reciprocal below the normal range is off by less than the 1e-5)
    const float rw = __frcp_rn(w);
    const float unit = sum_unit(d, w);
    const bool out_rows = h.ld_col == 1 && (h.ld_row & 3) == 0 && (m & 3) == 0 &&
                          (reinterpret_cast<uintptr_t>(h.H) & 15) == 0;
    const bool out_cols = TM == 8 && h.ld_row == 1 && (h.ld_col & 3) == 0 && row0 + BM <= h.nv &&
                          (reinterpret_cast<uintptr_t>(h.H) & 15) == 0;
    float bias[TN], na[TN];
#pragma unroll
    for (int j = 0; j < TN; ++j) {
        const int i = col0 + col_of(j);
        bias[j] = i < m ? __ldg(h.b + i) : 0.0f;
        na[j] = an[col_of(j)] * unit;
    }
    // the floors replace the sums (their bits)
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int lr = row_of(i);
        if (TM == 2 && lr % gridDim.z != blockIdx.z) continue;  // another block's share
        const float wv = vn[lr];
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const int lc = col_of(j);
            const float u = __fmul_rn(__fadd_rn(acc[i][j], bias[j]), rw);
            const float f = floorf(u);
            const bool sure = sure_at(u, f, na[j] * wv);  // else the second pass decides
            acc[i][j] = __int_as_float(sure ? (int32_t)f : 0);
            if (!sure && row0 + lr < h.nv && col0 + lc < m)
                sm.fix.list[atomicAdd(&n_list, 1)] = (uint16_t)(lr << 7 | lc);
        }
        // 16-byte stores along the contiguous direction where it is aligned
        const int64_t r = row0 + lr;
        if (out_rows) {
#pragma unroll
            for (int j = 0; j < TN; j += 4)
                if (r < h.nv && col0 + col_of(j) < m)
                    *reinterpret_cast<float4 *>(h.H + r * h.ld_row + col0 + col_of(j)) =
                        make_float4(acc[i][j], acc[i][j + 1], acc[i][j + 2], acc[i][j + 3]);
        } else if (!out_cols) {
#pragma unroll
            for (int j = 0; j < TN; ++j)
                if (r < h.nv && col0 + col_of(j) < m)
                    h.H[r * h.ld_row + (int64_t)(col0 + col_of(j)) * h.ld_col] =
                        __float_as_int(acc[i][j]);
        }
    }
    if (out_cols) {
        if constexpr (TM == 8) {
#pragma unroll
            for (int j = 0; j < TN; ++j) {
                const int i = col0 + col_of(j);
                if (i >= m) continue;
                float *p = reinterpret_cast<float *>(h.H + (int64_t)i * h.ld_col + row0 + 4 * ty);
                *reinterpret_cast<float4 *>(p) =
                    make_float4(acc[0][j], acc[1][j], acc[2][j], acc[3][j]);
                *reinterpret_cast<float4 *>(p + 128) =
                    make_float4(acc[4][j], acc[5][j], acc[6][j], acc[7][j]);
            }
        }
    }
    __syncthreads();
    settle_listed(h, sm.fix.list, n_list, sm.fix.sums, vn, an, row0, col0);
}

// ---- the same projection on the tensor cores (tcgen05, BF16 in, FP32 out)
//
// Every FP32 input is split into two BF16 numbers, v = v_hi + v_lo + e with
// v_hi = bf16(v), v_lo = bf16(v - v_hi) (v - v_hi is exact in FP32) and
// |e| <= 2^-16 |v|; likewise a = a_hi + a_lo + e_a.  A CTA of 128 threads
// takes 128 rows and every projection; the three products that matter,
//   D_hh = X_hi A_hi^T,  D_hl = X_lo A_hi^T,  D_lh = X_hi A_lo^T,
// go to three FP32 accumulators in tensor memory (M = 128, N = m rounded up to
// 16, K = 16 per instruction, one issuing thread), and t = D_hh + (D_hl + D_lh)
// is formed in FP32 in the epilogue.  Error of t, for any order of the
// tensor cores' internal additions:
//   - dropped terms a_lo v_lo and those with e, e_a: <= 3.01 * 2^-16 S;
//   - accumulation, taking every addition inside the tensor core to lose at
//     most two units in the last place (2^-22 relative; rounding or
//     truncation): <= (d - 1) * 2^-22 * S for D_hh, and 2^-8 of that for the
//     two small accumulators;
//   - the two FP32 additions of the epilogue: <= 2^-23 S,
// with S = sum_j |a_j v_j| <= ||a|| ||v|| (Cauchy-Schwarz; norms formed in
// FP32 and enlarged by 1 %).  As in the CUDA-core pass, every entry whose
// value lies within that bound (and at least 1e-5 w) of a bucket edge is
// listed and settled by the block's second pass (settle_listed), so the bucket
// ids are those of the FP64 definition whatever the tensor cores' rounding.
constexpr int PT_ROWS = 128;  // rows per CTA (the MMA's M)
constexpr int PT_KC = 64;     // input coordinates per staged chunk

// gridDim.y blocks form the same 128 rows and each settles and writes its share (as
// above, where the rows give few blocks).
__global__ void __launch_bounds__(PT_ROWS, 1) project_tc_kernel(HashArgs h, uint32_t ncols)
{
    const float *__restrict__ V = h.V, *__restrict__ A = h.A, *__restrict__ b = h.b;
    const int64_t nv = h.nv;
    const int d = h.d, m = h.m;
    const float w = h.w;
    extern __shared__ __align__(1024) unsigned char ptsm[];
    __shared__ int n_list;
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tbase_s;
    __shared__ int s_stuck;
    __shared__ float vnorm2[PT_ROWS], anorm2[128];
    const int tid = threadIdx.x, warp = tid >> 5;
    const int N = (m + 15) & ~15;                      // projections, padded
    unsigned char *xhi = ptsm;                         // 128 x PT_KC BF16
    unsigned char *xlo = xhi + PT_ROWS * PT_KC * 2;
    unsigned char *ahi = xlo + PT_ROWS * PT_KC * 2;    // N x PT_KC BF16
    unsigned char *alo = ahi + 128 * PT_KC * 2;
    const int64_t r0 = (int64_t)blockIdx.x * PT_ROWS;
    if (tid == 0) {
        s_stuck = 0;
        n_list = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem(&bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    vnorm2[tid] = 0.0f;
    anorm2[tid] = 0.0f;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         tc_smem(&tbase_s)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = tbase_s;
    const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
    const uint32_t idesc = tc_idesc_bf16(PT_ROWS, N);
    uint32_t phase = 0;
    // split a float into BF16 hi + lo
    auto split = [](float v, __nv_bfloat16 &hi, __nv_bfloat16 &lo) {
        hi = __float2bfloat16_rn(v);
        lo = __float2bfloat16_rn(v - __bfloat162float(hi));
    };
    for (int k0 = 0; k0 < d; k0 += PT_KC) {
        // stage the chunk: rows of V (4 consecutive coordinates per piece)
        for (int p = tid; p < PT_ROWS * (PT_KC / 4); p += PT_ROWS) {
            const int r = p / (PT_KC / 4), c = (p % (PT_KC / 4)) * 4;
            const int64_t gr = r0 + r;
            __align__(8) __nv_bfloat16 h4[4], l4[4];
            float sq = 0.0f;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int gc = k0 + c + u;
                const float v = (gr < nv && gc < d) ? V[gr * d + gc] : 0.0f;
                sq = fmaf(v, v, sq);
                split(v, h4[u], l4[u]);
            }
            if (sq != 0.0f) atomicAdd(&vnorm2[r], sq);
            *reinterpret_cast<uint2 *>(xhi + tc_off(r, c, PT_KC)) = *reinterpret_cast<const uint2 *>(h4);
            *reinterpret_cast<uint2 *>(xlo + tc_off(r, c, PT_KC)) = *reinterpret_cast<const uint2 *>(l4);
        }
        // and rows of A (projections past m are zero)
        for (int p = tid; p < N * (PT_KC / 4); p += PT_ROWS) {
            const int r = p / (PT_KC / 4), c = (p % (PT_KC / 4)) * 4;
            __align__(8) __nv_bfloat16 h4[4], l4[4];
            float sq = 0.0f;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int gc = k0 + c + u;
                const float v = (r < m && gc < d) ? A[(int64_t)r * d + gc] : 0.0f;
                sq = fmaf(v, v, sq);
                split(v, h4[u], l4[u]);
            }
            if (sq != 0.0f) atomicAdd(&anorm2[r], sq);
            *reinterpret_cast<uint2 *>(ahi + tc_off(r, c, PT_KC)) = *reinterpret_cast<const uint2 *>(h4);
            *reinterpret_cast<uint2 *>(alo + tc_off(r, c, PT_KC)) = *reinterpret_cast<const uint2 *>(l4);
        }
        tc_fence_async_smem();
        tc_fence_before();
        __syncthreads();
        const bool go = s_stuck == 0;
        if (tid == 0 && go) {
            tc_fence_after();
#pragma unroll
            for (int s2 = 0; s2 < PT_KC / 16; ++s2) {
                const uint32_t acc = (k0 | s2) != 0 ? 1u : 0u;
                const uint32_t kb = (uint32_t)(2 * s2) * 128;  // 16 k = two core matrices
                const uint64_t dxh = tc_desc(xhi + kb, 128, PT_KC * 16);
                const uint64_t dxl = tc_desc(xlo + kb, 128, PT_KC * 16);
                const uint64_t dah = tc_desc(ahi + kb, 128, PT_KC * 16);
                const uint64_t dal = tc_desc(alo + kb, 128, PT_KC * 16);
                tc_mma(tbase, dxh, dah, idesc, acc);                    // X_hi A_hi^T
                tc_mma(tbase + (uint32_t)N, dxl, dah, idesc, acc);      // X_lo A_hi^T
                tc_mma(tbase + 2u * (uint32_t)N, dxh, dal, idesc, acc); // X_hi A_lo^T
            }
            tc_commit(&bar);
        }
        if (go) {
            if (!tc_wait(&bar, phase)) s_stuck = 1;
            phase ^= 1;
        }
        tc_fence_after();
        __syncthreads();  // the chunk buffers are rewritten next
    }
    // epilogue: row = thread
    const int64_t r = r0 + tid;
    const bool stuck = s_stuck != 0;
    const float unit = kU;
    // the sums of squares become norm bounds
    vnorm2[tid] = norm_bound(vnorm2[tid], d);
    anorm2[tid] = norm_bound(anorm2[tid], d);
    __syncthreads();
    const float vn = vnorm2[tid];
    // the operand tiles (the MMAs are done) become the list and its sums
    uint16_t *list = reinterpret_cast<uint16_t *>(ptsm);
    float2 *sums = reinterpret_cast<float2 *>(ptsm + PT_ROWS * 128 * sizeof(uint16_t));
    const float cacc = (3.01f * 1.52587890625e-05f                 // 3.01 * 2^-16
                        + (float)(d > 1 ? d - 1 : 0) * 2.384185791e-07f * 1.01f  // (d-1) 2^-22
                        + 2.0f * unit) * 1.01f;
    for (int n0 = 0; n0 < N; n0 += 16) {
        float hh[16], hl[16], lh[16];
        tc_ld16(tbase + lane_base + (uint32_t)n0, hh);
        tc_ld16(tbase + lane_base + (uint32_t)(N + n0), hl);
        tc_ld16(tbase + lane_base + (uint32_t)(2 * N + n0), lh);
        if (r >= nv || tid % gridDim.y != blockIdx.y) continue;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const int i = n0 + j;
            if (i >= m) continue;
            const float t = __fadd_rn(hh[j], __fadd_rn(hl[j], lh[j]));
            const float u = __fdiv_rn(__fadd_rn(t, b[i]), w);
            const float f = floorf(u);
            // out of int32, NaN, or a wait that gave up: the second pass decides
            bool open = stuck || !(f >= -2147483520.0f && f <= 2147483520.0f);
            if (!open) {
                const float frac = u - f;
                const float near = fminf(frac, 1.0f - frac);
                const float eps = fmaxf(cacc * anorm2[i] * vn / w + 4.0f * unit * (fabsf(u) + 1.0f),
                                        1e-5f);
                open = !(near > eps);
                if (!open) h.H[r * h.ld_row + (int64_t)i * h.ld_col] = (int32_t)f;
            }
            if (open) list[atomicAdd(&n_list, 1)] = (uint16_t)(tid * 128 + i);
        }
    }
    __syncthreads();
    settle_listed(h, list, n_list, sums, vnorm2, anorm2, r0, 0);
    if (tid == 0 && stuck) atomicOr(h.err, 16);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase),
                     "r"(ncols)
                     : "memory");
    }
}

}  // namespace

qw_status launch_hash(const float *V, int64_t nv, int d, const float *A, const float *b, int m,
                      float w, int32_t *H, int64_t ld_row, int64_t ld_col, int *err,
                      unsigned long long *fixups, cudaStream_t s, bool tensor_cores)
{
    if (nv == 0) return QW_OK;
    if (!((ld_row == m && ld_col == 1) || (ld_row == 1 && ld_col == nv))) return QW_ERR_ARG;
    HashArgs h;
    h.V = V;
    h.nv = nv;
    h.d = d;
    h.A = A;
    h.b = b;
    h.m = m;
    h.w = w;
    h.H = H;
    h.ld_row = ld_row;
    h.ld_col = ld_col;
    h.err = err;
    h.fixups = fixups;
    h.vec = d % 4 == 0 && ((uintptr_t)V | (uintptr_t)A) % 16 == 0;
    // blocks of one tile: one per SM in all, at least two rows each
    auto shares = [](int64_t tiles) {
        return std::max<int64_t>(1, std::min<int64_t>(32, 152 / tiles));
    };
    if (tensor_cores && m <= 128) {
        const int N = (m + 15) & ~15;
        uint32_t ncols = 32;
        while (ncols < (uint32_t)(3 * N)) ncols <<= 1;
        // shared memory sized so that the CTAs resident on an SM never ask
        // for more than its 512 TMEM columns (no allocation waits)
        constexpr size_t per = (size_t)(2 * PT_ROWS + 2 * 128) * PT_KC * 2;
        static_assert(per >= PT_ROWS * 128 * sizeof(uint16_t) + PT_ROWS * sizeof(float2),
                      "the list of open entries fits the operand tiles");
        static_assert(per <= (size_t)80 << 10, "the operand tiles fit the smaller size");
        const size_t smem = ncols > 256 ? (size_t)120 << 10 : (size_t)80 << 10;
        QW_TRY(allow_smem(project_tc_kernel, (size_t)120 << 10));
        const int64_t blocks = (nv + PT_ROWS - 1) / PT_ROWS;
        if (blocks > 2147483647LL) return QW_ERR_ARG;
        const dim3 grid((unsigned)blocks, (unsigned)shares(blocks));
        project_tc_kernel<<<grid, PT_ROWS, smem, s>>>(h, ncols);
    } else if (nv <= kFewRows && nv * m <= kFewEntries) {
        project_rows_kernel<<<(unsigned)((nv * m + NT / 8 - 1) / (NT / 8)), NT, 0, s>>>(h);
    } else {
        const int bn = m <= 32 ? 32 : 64;
        const int64_t cb = (m + bn - 1) / bn;
        // 256 rows per block from 100 blocks on, else 64: with fewer, the smaller
        // blocks' use of every SM outweighs their reads of A (64 and 256 rows, us, 128
        // dimensions x 64 projections: 75 blocks 52 and 57, 118 71 and 58, 196 84 and
        // 68, 301 101 and 70, 1,172 259 and 181; 512 x 64: 75 96 and 111, 118 137 and
        // 110; 128 x 32: 75 45 and 49, 118 57 and 48; 64 x 127: 64 50 and 57, 150 57
        // and 57, 236 73 and 62)
        const bool wide = (nv + 255) / 256 * cb >= 100;
        const int64_t rb = wide ? (nv + 255) / 256 : (nv + 63) / 64;
        if (rb > 2147483647LL) return QW_ERR_ARG;
        const dim3 grid((unsigned)rb, (unsigned)cb, wide ? 1u : (unsigned)shares(rb * cb));
        if (bn == 32 && wide) project_fp32_kernel<8, 4><<<grid, NT, 0, s>>>(h);
        else if (bn == 32) project_fp32_kernel<2, 4><<<grid, NT, 0, s>>>(h);
        else if (wide) project_fp32_kernel<8, 8><<<grid, NT, 0, s>>>(h);
        else project_fp32_kernel<2, 8><<<grid, NT, 0, s>>>(h);
    }
    QW_CUDA_TRY(cudaGetLastError());
    return QW_OK;
}

}  // namespace qw
