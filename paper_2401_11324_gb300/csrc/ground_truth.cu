// Exact k nearest neighbours on the GPU: the ground truth that recall@k
// (§6.3, k-recall@k) is measured against.  Distances are squared L2, exact
// integers for u8/i8 data and FP64 for f32 data, the latter summed in
// ascending dimension order with each difference, product and sum rounded
// (no fused multiply-add); ties go to the smaller id.  The only FP64 on the
// GPU in this library besides the offline k-means.
//
// The k-th distance among any subset of the points is at least the k-th over
// all n, so every true neighbour lies within it.  (1) Each query's exact k
// nearest among 1,024 points (spread evenly over the ids) give a first
// threshold.  (2) A tile of queries held in shared memory streams over 16
// times as many points, one point per thread, and appends every point within a
// query's threshold to that query's candidate list (about 16 k of them); their
// k-th distance is the next threshold, and so on until all n points have been
// streamed over; integer rows of up to 256 dimensions and FP32 rows of up to
// 208 on the tensor cores (ground_truth_tc.cuh), others as above.  (3) One warp per query picks the k smallest candidates of
// the last list by (distance, id).  A list that overflows its capacity is
// detected and its pass rerun with room for the longest list.
//
// Step (1) kept each query's k nearest sorted in one warp, a serial chain per
// insertion: over 262,144 points it took 294 of 375 ms (10,000 u8 queries,
// d = 128, 1M points, k = 100).  Over 1,024, with the distances in shared memory
// and a radix selection, it takes 1.2.  The streamed levels are a contraction:
// with a point per thread (vabsdiff4 + dp4a) they took 73 ms, on the tensor
// cores 6.1; the sorted selection took 3.9 ms one neighbour after the other, 0.1
// gathered and sorted.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "bang.h"
#include "bang_internal.h"
#include "ground_truth_tc.cuh"

namespace {

constexpr uint32_t kNo = 0xFFFFFFFFu;
constexpr int kW = 32;
constexpr uint32_t kMaxK = 256;
constexpr uint32_t kTileQ = 128;         // at most this many queries per CTA in pass 2
constexpr uint32_t kSample = 1024;       // points of the first threshold
constexpr uint64_t kQueries = 1u << 16;  // queries at a time
constexpr uint32_t kLeastQueries = 64;   // at least, where memory is short
constexpr uint32_t kLevel = 16;          // each further level streams over this many times as many

struct GtArgs {
    const void *base, *queries;
    int dtype;
    uint64_t n;                  // points of this level: ids i * stride, i < n
    uint64_t stride;
    uint32_t nq, d, k;
    const double *thr;           // nq thresholds (pass 2)
    double *thr_out;             // pass 1
    uint32_t *cnt;               // nq candidate counts
    double *cd;                  // nq x cap candidate distances
    uint32_t *ci;                // nq x cap candidate ids
    uint64_t cap;
    uint32_t *out_ids;
    double *out_dist;
    uint32_t tileq;              // queries per CTA in pass 2 (46 KB of rows at most)
    uint32_t words;              // integer rows readable as 32-bit words (d % 4 == 0, aligned)
    uint32_t regrow;             // integer rows of 16..128 bytes in 16-byte steps, 16-byte aligned
};

// Squared distance of two rows of 32-bit words of packed bytes (int8 offset
// by 128 on both sides, so byte differences are unsigned).
__device__ __forceinline__ uint32_t word_dist(uint32_t a, uint32_t b, uint32_t acc, bool i8)
{
    if (i8) { a ^= 0x80808080u; b ^= 0x80808080u; }
    const uint32_t t = __vabsdiffu4(a, b);
    return __dp4a(t, t, acc);
}

__device__ __forceinline__ double dist_rows(const GtArgs &g, const void *qrow, uint64_t i)
{
    if (g.dtype == 2) {
        const float *q = static_cast<const float *>(qrow);
        const float *x = static_cast<const float *>(g.base) + i * g.d;
        double acc = 0.0;
        for (uint32_t j = 0; j < g.d; ++j) {
            const double t = __dsub_rn(static_cast<double>(q[j]), static_cast<double>(__ldg(x + j)));
            acc = __dadd_rn(acc, __dmul_rn(t, t));
        }
        return acc;
    }
    if (g.words) {
        const uint32_t *q = static_cast<const uint32_t *>(qrow);
        const uint32_t *x = reinterpret_cast<const uint32_t *>(static_cast<const unsigned char *>(g.base) + i * g.d);
        uint32_t acc = 0;       // at most d * 255^2 < 2^32 (d <= 4096)
        for (uint32_t w = 0; w < g.d / 4u; ++w) acc = word_dist(q[w], __ldg(x + w), acc, g.dtype == 1);
        return static_cast<double>(acc);
    }
    int64_t acc = 0;
    if (g.dtype == 0) {
        const uint8_t *q = static_cast<const uint8_t *>(qrow);
        const uint8_t *x = static_cast<const uint8_t *>(g.base) + i * g.d;
        for (uint32_t j = 0; j < g.d; ++j) {
            const int32_t t = static_cast<int32_t>(q[j]) - static_cast<int32_t>(__ldg(x + j));
            acc += t * t;
        }
    } else {
        const int8_t *q = static_cast<const int8_t *>(qrow);
        const int8_t *x = static_cast<const int8_t *>(g.base) + i * g.d;
        for (uint32_t j = 0; j < g.d; ++j) {
            const int32_t t = static_cast<int32_t>(q[j]) - static_cast<int32_t>(__ldg(x + j));
            acc += t * t;
        }
    }
    return static_cast<double>(acc);
}

__device__ __forceinline__ const void *query_row(const GtArgs &g, uint32_t q)
{
    const size_t esz = g.dtype == 2 ? 4 : 1;
    return static_cast<const unsigned char *>(g.queries) + static_cast<uint64_t>(q) * g.d * esz;
}

// (distance, id) order; distances are >= +0, so their bit patterns order like
// their values.
__device__ __forceinline__ bool less_pair(uint64_t da, uint32_t ia, uint64_t db, uint32_t ib)
{
    return da < db || (da == db && ia < ib);
}

// Step 2: blockIdx.y = tile of kTileQ queries (rows in shared memory);
// threads stride over the points.
__global__ void collect(const GtArgs g)
{
    extern __shared__ __align__(16) unsigned char qs[];
    const uint32_t q0 = blockIdx.y * g.tileq;
    const uint32_t nt = g.nq - q0 < g.tileq ? g.nq - q0 : g.tileq;
    const size_t rowb = static_cast<size_t>(g.d) * (g.dtype == 2 ? 4 : 1);
    for (size_t i = threadIdx.x; i < nt * rowb; i += blockDim.x)
        qs[i] = static_cast<const unsigned char *>(query_row(g, q0))[i];
    __shared__ double th[kTileQ];
    if (threadIdx.x < nt) th[threadIdx.x] = g.thr[q0 + threadIdx.x];
    __syncthreads();
    for (uint64_t i0 = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; i0 < g.n;
         i0 += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
        const uint64_t i = i0 * g.stride;
        uint4 xr[8];                     // the point's row, for the register path
        const uint32_t nv = g.d / 16u;
        if (g.regrow) {
            const uint4 *x = reinterpret_cast<const uint4 *>(static_cast<const unsigned char *>(g.base) + i * g.d);
#pragma unroll
            for (int c = 0; c < 8; ++c) xr[c] = static_cast<uint32_t>(c) < nv ? __ldg(x + c) : make_uint4(0u, 0u, 0u, 0u);
        }
        for (uint32_t t = 0; t < nt; ++t) {
            double dv;
            if (g.regrow) {
                const uint4 *qv = reinterpret_cast<const uint4 *>(qs + t * rowb);
                uint32_t acc = 0;
                const bool i8 = g.dtype == 1;
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    if (static_cast<uint32_t>(c) < nv) {
                        const uint4 a = qv[c], b = xr[c];
                        acc = word_dist(a.x, b.x, acc, i8);
                        acc = word_dist(a.y, b.y, acc, i8);
                        acc = word_dist(a.z, b.z, acc, i8);
                        acc = word_dist(a.w, b.w, acc, i8);
                    }
                }
                dv = static_cast<double>(acc);
            } else {
                dv = dist_rows(g, qs + t * rowb, i);
            }
            if (dv <= th[t]) {
                const uint32_t q = q0 + t;
                const uint32_t slot = atomicAdd(g.cnt + q, 1u);
                if (slot < g.cap) {
                    g.cd[static_cast<uint64_t>(q) * g.cap + slot] = dv;
                    g.ci[static_cast<uint64_t>(q) * g.cap + slot] = static_cast<uint32_t>(i);
                }
            }
        }
    }
}

// An upper bound of the k-th smallest of m >= k distances, as FP32 bits: its
// FP32 value rounded up (integer distances are exact), by four rounds of 8-bit
// digits.  One warp; hist: 256 words of shared memory.
__device__ __forceinline__ uint32_t value_bits(double d) { return __float_as_uint(__double2float_ru(d)); }

template <typename Bits>
__device__ __forceinline__ uint32_t kth_bits(Bits bits, uint32_t m, uint32_t k, uint32_t *hist, int lane)
{
    uint32_t prefix = 0, mask = 0, want = k;     // the want-th among the values with this prefix
    for (int shift = 24; shift >= 0; shift -= 8) {
        for (int b = lane; b < 256; b += kW) hist[b] = 0;
        __syncwarp();
        for (uint32_t j = lane; j < m; j += kW) {
            const uint32_t v = bits(j);
            if ((v & mask) == prefix) atomicAdd(&hist[(v >> shift) & 255u], 1u);
        }
        __syncwarp();
        uint32_t h[8], sum = 0;                  // this lane's bins: 8 lane .. 8 lane + 7
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            h[b] = hist[lane * 8 + b];
            sum += h[b];
        }
        uint32_t below = sum;
#pragma unroll
        for (int o = 1; o < kW; o <<= 1) {
            const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, below, o);
            if (lane >= o) below += up;
        }
        below -= sum;
        const bool here = below < want && want <= below + sum;
        uint32_t bin = 0, left = here ? want - below : 0u;
        if (here) {
#pragma unroll
            for (int b = 0; b < 7; ++b)
                if (bin == static_cast<uint32_t>(b) && left > h[b]) {
                    left -= h[b];
                    ++bin;
                }
            bin += lane * 8u;
        }
        const int src = __ffs(__ballot_sync(0xFFFFFFFFu, here)) - 1;
        bin = __shfl_sync(0xFFFFFFFFu, bin, src);
        want = __shfl_sync(0xFFFFFFFFu, left, src);
        prefix |= bin << shift;
        mask |= 255u << shift;
        __syncwarp();
    }
    return prefix;
}

constexpr int kKthWarps = 4;

// Step 1: one warp per query, the distances of the first level's points (at
// most kSample) in shared memory, as the bits that kth_bits selects by.
constexpr int kSampleWarps = 4;
__global__ void __launch_bounds__(kSampleWarps * kW) sample_threshold(const GtArgs g)
{
    __shared__ uint32_t bits[kSampleWarps][kSample];
    __shared__ uint32_t hist[kSampleWarps][256];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t q = blockIdx.x * kSampleWarps + wid;
    if (q >= g.nq) return;
    const void *qr = query_row(g, q);
    const uint32_t m = static_cast<uint32_t>(g.n);
    for (uint32_t i = lane; i < m; i += kW) bits[wid][i] = value_bits(dist_rows(g, qr, i * g.stride));
    __syncwarp();
    double t = __longlong_as_double(0x7FF0000000000000ll);       // fewer than k points: every point is a candidate
    if (m >= g.k) {
        const uint32_t *bw = bits[wid];
        t = static_cast<double>(__uint_as_float(kth_bits([bw](uint32_t j) { return bw[j]; }, m, g.k, hist[wid], lane)));
    }
    if (lane == 0) g.thr_out[q] = t == t ? t : __longlong_as_double(0x7FF0000000000000ll);   // (NaN rows)
}

// The threshold of the next level from a query's list.  One warp per query.
__global__ void __launch_bounds__(kKthWarps * kW) kth_threshold(const GtArgs g)
{
    __shared__ uint32_t hist[kKthWarps][256];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t q = blockIdx.x * kKthWarps + wid;
    if (q >= g.nq) return;
    const uint32_t m = g.cnt[q];                 // at most cap, checked by the host
    const double *cd = g.cd + static_cast<uint64_t>(q) * g.cap;
    if (m < g.k) return;                         // the level's points differ: the old threshold stays the best
    const double t = static_cast<double>(
        __uint_as_float(kth_bits([cd](uint32_t j) { return value_bits(cd[j]); }, m, g.k, hist[wid], lane)));
    if (lane == 0 && t <= g.thr_out[q]) g.thr_out[q] = t;
}

// Step 3: one warp per query, the k smallest candidates in (distance, id)
// order: those within the bound of the k-th (k of them, and what ties with it
// or rounds to it) are gathered and bitonic-sorted in shared memory; when more
// than kSortMax are, the k smallest are taken one after the other.
constexpr uint32_t kSortMax = 512;
__global__ void __launch_bounds__(kKthWarps * kW) select_k(const GtArgs g)
{
    __shared__ uint32_t hist[kKthWarps][256];
    __shared__ uint64_t sd[kKthWarps][kSortMax];
    __shared__ uint32_t si[kKthWarps][kSortMax];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t q = blockIdx.x * kKthWarps + wid;
    if (q >= g.nq) return;
    const uint32_t m = static_cast<uint32_t>(g.cnt[q] < g.cap ? g.cnt[q] : g.cap);
    const double *cd = g.cd + static_cast<uint64_t>(q) * g.cap;
    const uint32_t *ci = g.ci + static_cast<uint64_t>(q) * g.cap;
    const uint32_t bound = m >= g.k ? kth_bits([cd](uint32_t j) { return value_bits(cd[j]); }, m, g.k, hist[wid], lane)
                                      : 0xFFFFFFFFu;
    uint32_t c = 0;                              // gathered
    for (uint32_t j0 = 0; j0 < m && c <= kSortMax; j0 += kW) {
        const uint32_t j = j0 + lane;
        const bool in = j < m && value_bits(cd[j]) <= bound;
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, in);
        const uint32_t at = c + __popc(bal & ((1u << lane) - 1u));
        if (in && at < kSortMax) {
            sd[wid][at] = static_cast<uint64_t>(__double_as_longlong(cd[j]));
            si[wid][at] = ci[j];
        }
        c += __popc(bal);
    }
    if (c <= kSortMax) {
        uint32_t P = kW;
        while (P < c) P <<= 1;
        for (uint32_t i = c + lane; i < P; i += kW) {
            sd[wid][i] = ~0ull;
            si[wid][i] = kNo;
        }
        __syncwarp();
        for (uint32_t size = 2; size <= P; size <<= 1)
            for (uint32_t j = size >> 1; j > 0; j >>= 1) {
                for (uint32_t t = lane; t < P / 2; t += kW) {
                    const uint32_t i = ((t & ~(j - 1u)) << 1) | (t & (j - 1u)), l = i | j;
                    const uint64_t xd = sd[wid][i], yd = sd[wid][l];
                    const uint32_t xi = si[wid][i], yi = si[wid][l];
                    const bool up = (i & size) == 0;
                    if (less_pair(yd, yi, xd, xi) == up) {
                        sd[wid][i] = yd;
                        si[wid][i] = yi;
                        sd[wid][l] = xd;
                        si[wid][l] = xi;
                    }
                }
                __syncwarp();
            }
        for (uint32_t r = lane; r < g.k; r += kW) {
            const uint64_t o = static_cast<uint64_t>(q) * g.k + r;
            const bool have = r < c;
            g.out_ids[o] = have ? si[wid][r] : kNo;
            g.out_dist[o] = __longlong_as_double(have ? static_cast<long long>(sd[wid][r]) : 0x7FF0000000000000ll);
        }
        return;
    }
    uint64_t pd = 0;             // the last pair taken (exclusive lower bound)
    uint32_t pi = 0;
    bool first = true;
    for (uint32_t r = 0; r < g.k; ++r) {
        uint64_t bd = ~0ull;
        uint32_t bi = kNo;
        for (uint32_t j = lane; j < m; j += kW) {
            const uint64_t dj = static_cast<uint64_t>(__double_as_longlong(cd[j]));
            const uint32_t ij = ci[j];
            if (!first && !less_pair(pd, pi, dj, ij)) continue;          // already taken
            if (less_pair(dj, ij, bd, bi)) { bd = dj; bi = ij; }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const uint64_t od = __shfl_xor_sync(0xFFFFFFFFu, bd, o);
            const uint32_t oi = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
            if (less_pair(od, oi, bd, bi)) { bd = od; bi = oi; }
        }
        const uint64_t o = static_cast<uint64_t>(q) * g.k + r;
        if (lane == 0) {
            g.out_ids[o] = bi;
            g.out_dist[o] = bi == kNo ? __longlong_as_double(0x7FF0000000000000ll)
                                      : __longlong_as_double(static_cast<long long>(bd));
        }
        pd = bd;
        pi = bi;
        first = false;
    }
}

template <typename T> struct DArr {
    T *p = nullptr;
    ~DArr() { if (p) cudaFree(p); }
    cudaError_t alloc(uint64_t count)
    {
        if (p) cudaFree(p);
        p = nullptr;
        return cudaMalloc(&p, sizeof(T) * (count ? count : 1));
    }
};

// The tensor-core form of a level (ground_truth_tc.cuh): its operands and
// scratch.  From kTcLeast points a level; below, the launches cost as much.
constexpr uint64_t kTcLeast = 8192;
struct TcLevel {
    const void *B, *Q;
    int dtype;
    uint32_t d, nq, nblk, qper, qgroups;
    int sms;
    bool on;
    uint32_t state[2] = {0u, 0u};          // copy of flags: values out of the filter's range, a wait gave up
    DArr<unsigned char> qtiles, ptiles;
    DArr<float> pnorm, lim, qq;
    DArr<uint32_t> flags;

    TcLevel(const void *base, const void *queries, int dt, uint32_t dim, uint32_t count, int sm)
        : B(base), Q(queries), dtype(dt), d(dim), nq(count), sms(sm)
    {
        nblk = (d + 15u) / 16u * (dt == 2 ? 2u : 1u);
        on = nblk <= (dt == 2 ? gt_tc::kMaxBlocks : 16u);    // integer sums above 256 dimensions pass 2^24
        qper = nblk <= 8u ? 256u : 128u;
        qgroups = (nq + qper - 1u) / qper;
    }
    cudaError_t prepare(uint64_t n, cudaStream_t st)
    {
        if (!on || n < kTcLeast) {
            on = false;
            return cudaSuccess;
        }
        const uint32_t qt = (nq + gt_tc::kTileP - 1u) / gt_tc::kTileP;
        const uint64_t pt = ((n < gt_tc::kTcPoints ? n : gt_tc::kTcPoints) + gt_tc::kTileP - 1u) / gt_tc::kTileP;
        cudaError_t e = qtiles.alloc(static_cast<uint64_t>(qt) * nblk * gt_tc::kBlock);
        if (e == cudaSuccess) e = ptiles.alloc(pt * nblk * gt_tc::kBlock);
        if (e == cudaSuccess) e = pnorm.alloc(pt * gt_tc::kTileP);
        if (e == cudaSuccess) e = lim.alloc(nq);
        if (e == cudaSuccess) e = qq.alloc(nq);
        if (e == cudaSuccess) e = flags.alloc(2);
        if (e == cudaErrorMemoryAllocation) {      // up to 0.9 GB that the other form does without
            cudaGetLastError();
            qtiles.alloc(0);
            ptiles.alloc(0);
            on = false;
            return cudaSuccess;
        }
        if (e != cudaSuccess) return e;
        if ((e = cudaMemsetAsync(flags.p, 0, 8, st)) != cudaSuccess) return e;
        // the limit belongs to the kernel and outlasts this call: the same for every
        // thread, as others launch with theirs between this call's levels
        constexpr int kMost = 227 * 1024;
        e = dtype == 2 ? cudaFuncSetAttribute(gt_tc::collect_tc<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost)
                       : cudaFuncSetAttribute(gt_tc::collect_tc<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost);
        if (e != cudaSuccess) return e;
        gt_tc::convert<<<qt, gt_tc::kTileP, 0, st>>>(Q, dtype, d, nblk, 0, nq, 1, qtiles.p, nullptr, flags.p);
        return cudaGetLastError();
    }
    // Appends every pair of the level within its query's threshold (g.cnt zeroed).
    cudaError_t collect(const GtArgs &g, cudaStream_t st)
    {
        gt_tc::limits<<<(nq + 127u) / 128u, 128, 0, st>>>(Q, dtype, d, nq, g.thr, lim.p, qq.p);
        gt_tc::TcArgs a;
        std::memset(&a, 0, sizeof a);
        a.base = B; a.queries = Q; a.dtype = dtype; a.d = d; a.nblk = nblk; a.nq = nq; a.stride = g.stride;
        a.ptiles = ptiles.p; a.qtiles = qtiles.p; a.pnorm = pnorm.p; a.lim = lim.p; a.qq = qq.p; a.thr = g.thr;
        a.cnt = g.cnt; a.cd = g.cd; a.ci = g.ci; a.cap = g.cap; a.err = flags.p + 1;
        const uint32_t smem = gt_tc::smem_bytes(nblk);
        for (uint64_t first = 0; first < g.n; first += gt_tc::kTcPoints) {
            a.first = first;
            a.count = g.n - first < gt_tc::kTcPoints ? g.n - first : gt_tc::kTcPoints;
            const uint32_t nt = static_cast<uint32_t>((a.count + gt_tc::kTileP - 1u) / gt_tc::kTileP);
            gt_tc::convert<<<nt, gt_tc::kTileP, 0, st>>>(B, dtype, d, nblk, first, a.count, g.stride, ptiles.p, pnorm.p, flags.p);
            // shares of the tiles: of the counts that give up to 8 blocks an SM,
            // the one whose last wave leaves the fewest tiles waiting
            uint32_t best = 1;
            uint64_t cost = ~0ull;
            for (uint32_t x = 1; x <= nt && static_cast<uint64_t>(x) * qgroups <= 8ull * sms + qgroups; ++x) {
                const uint64_t waves = (static_cast<uint64_t>(x) * qgroups + sms - 1u) / sms;
                const uint64_t t = waves * ((nt + x - 1u) / x + 4u);     // a block's start costs about 4 tiles
                if (t < cost) { cost = t; best = x; }
            }
            a.tiles_per_cta = (nt + best - 1u) / best;
            const dim3 grid((nt + a.tiles_per_cta - 1u) / a.tiles_per_cta, qgroups);
            if (dtype == 2) gt_tc::collect_tc<1><<<grid, gt_tc::kThreads, smem, st>>>(a);
            else gt_tc::collect_tc<0><<<grid, gt_tc::kThreads, smem, st>>>(a);
            const cudaError_t e = cudaGetLastError();
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    }
};

bool is_dev(const void *p)
{
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

int gtfail(int code, const std::string &m)
{
    bang::set_error(m);
    return code;
}

}  // namespace

#define GT_TRY(x)                                                                           \
    do {                                                                                    \
        cudaError_t e_ = (x);                                                               \
        if (e_ != cudaSuccess) {                                                            \
            cudaGetLastError();                                                             \
            return gtfail(e_ == cudaErrorMemoryAllocation ? BANG_ENOMEM : BANG_ECUDA,      \
                          std::string(#x) + ": " + cudaGetErrorString(e_));                 \
        }                                                                                   \
    } while (0)

namespace {

// The k nearest of n points (B) for m queries (Q), all on the device but the
// results where they go to the host.
int truth_of(int device, const void *B, const void *Q, bang_dtype dtype, uint64_t n, uint32_t m, uint32_t d, uint32_t k,
             uint32_t tileq, bool tensor, uint32_t *ids, double *dist, bool dev_out, cudaStream_t st)
{
    const size_t esz = dtype == BANG_F32 ? 4 : 1;
    DArr<double> thr, cd, odist;
    DArr<uint32_t> cnt, ci, oids;
    GT_TRY(thr.alloc(m));
    GT_TRY(cnt.alloc(m));
    GtArgs g;
    std::memset(&g, 0, sizeof g);
    g.base = B;
    g.queries = Q;
    g.dtype = dtype;
    g.nq = m;
    g.d = d;
    g.k = k;
    g.thr_out = thr.p;
    g.thr = thr.p;
    g.cnt = cnt.p;
    g.tileq = tileq;
    {
        const uintptr_t ab = reinterpret_cast<uintptr_t>(B), aq = reinterpret_cast<uintptr_t>(Q);
        g.words = dtype != BANG_F32 && d % 4 == 0 && ab % 4 == 0 && aq % 4 == 0;
        g.regrow = dtype != BANG_F32 && d % 16 == 0 && d <= 128 && ab % 16 == 0;
    }
    g.n = n < kSample ? n : kSample;
    g.stride = n / g.n;
    sample_threshold<<<(m + kSampleWarps - 1) / kSampleWarps, kSampleWarps * kW, 0, st>>>(g);
    GT_TRY(cudaGetLastError());
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    const uint32_t tiles = (m + tileq - 1) / tileq;
    std::vector<uint32_t> c(m);
    uint64_t cap = 0;
    TcLevel tc(B, Q, dtype, d, m, sms);
    tc.on = tc.on && tensor;
    GT_TRY(tc.prepare(n, st));
    for (uint64_t seen = g.n;; seen = g.n) {
        g.n = seen < n / kLevel ? seen * kLevel : n;     // the last level takes every point
        g.stride = n / g.n;
        // expected list length about k * (points now / points before); room for twice that, then the longest
        uint64_t room = 2ull * k * ((g.n + seen - 1) / seen) + 256;
        for (int attempt = 0;; ++attempt) {
            if (room > cap) {
                GT_TRY(cd.alloc(room * m));
                GT_TRY(ci.alloc(room * m));
                cap = room;
            }
            GT_TRY(cudaMemsetAsync(cnt.p, 0, m * 4, st));
            g.cd = cd.p;
            g.ci = ci.p;
            g.cap = cap;
            if (tc.on && g.n >= kTcLeast) GT_TRY(tc.collect(g, st));
            else {
                // fewer queries a block where the level's points alone would not fill the GPU
                const uint64_t have = (g.n + 255u) / 256u * tiles, want = 4ull * sms;
                g.tileq = have < want ? static_cast<uint32_t>(std::max<uint64_t>(1u, tileq * have / want)) : tileq;
                const uint32_t ty = (m + g.tileq - 1u) / g.tileq;
                const uint32_t tx = static_cast<uint32_t>((static_cast<uint64_t>(sms) * 8 + ty - 1) / ty) + 1;
                collect<<<dim3(tx, ty), 256, g.tileq * d * esz, st>>>(g);
            }
            GT_TRY(cudaGetLastError());
            GT_TRY(cudaMemcpyAsync(c.data(), cnt.p, m * 4, cudaMemcpyDeviceToHost, st));
            if (tc.on) GT_TRY(cudaMemcpyAsync(tc.state, tc.flags.p, sizeof tc.state, cudaMemcpyDeviceToHost, st));
            GT_TRY(cudaStreamSynchronize(st));
            if (tc.on && tc.state[1]) return gtfail(BANG_ETIMEOUT, "bang_ground_truth: a tensor-core wait gave up");
            if (tc.on && tc.state[0]) {          // values the filter cannot bound: this level again without it
                tc.on = false;
                --attempt;
                continue;
            }
            room = *std::max_element(c.begin(), c.end());
            if (room <= cap) break;
            if (attempt == 1) return gtfail(BANG_ECUDA, "bang_ground_truth: candidate lists kept growing");
        }
        if (g.n == n) break;
        kth_threshold<<<(m + kKthWarps - 1) / kKthWarps, kKthWarps * kW, 0, st>>>(g);
        GT_TRY(cudaGetLastError());
    }
    if (!dev_out) {
        GT_TRY(oids.alloc(static_cast<uint64_t>(m) * k));
        GT_TRY(odist.alloc(static_cast<uint64_t>(m) * k));
    }
    g.out_ids = dev_out ? ids : oids.p;
    g.out_dist = dev_out ? dist : odist.p;
    select_k<<<(m + kKthWarps - 1) / kKthWarps, kKthWarps * kW, 0, st>>>(g);
    GT_TRY(cudaGetLastError());
    if (!dev_out) {
        GT_TRY(cudaMemcpyAsync(ids, oids.p, static_cast<uint64_t>(m) * k * 4, cudaMemcpyDeviceToHost, st));
        GT_TRY(cudaMemcpyAsync(dist, odist.p, static_cast<uint64_t>(m) * k * 8, cudaMemcpyDeviceToHost, st));
    }
    GT_TRY(cudaStreamSynchronize(st));
    return BANG_OK;
}

}  // namespace

extern "C" int bang_ground_truth(int device, const void *base, const void *queries, bang_dtype dtype,
                                 uint64_t n, uint32_t nq, uint32_t d, uint32_t k, uint32_t *out_ids,
                                 double *out_dist, void *stream)
{
    if (!base || !queries || !out_ids || !out_dist) return gtfail(BANG_EINVAL, "bang_ground_truth: NULL argument");
    if (dtype != BANG_U8 && dtype != BANG_I8 && dtype != BANG_F32)
        return gtfail(BANG_EINVAL, "bang_ground_truth: unknown dtype");
    if (n == 0 || n >= (1ull << 32) - 1 || d == 0 || d > 4096 || k == 0 || k > kMaxK)
        return gtfail(BANG_EINVAL, "bang_ground_truth: need 0 < n < 2^32 - 1, 0 < d <= 4096, 1 <= k <= 256");
    if (bang::pointer_kind(base, device) == 2 || bang::pointer_kind(queries, device) == 2 ||
        bang::pointer_kind(out_ids, device) == 2 || bang::pointer_kind(out_dist, device) == 2)
        return gtfail(BANG_EINVAL, "bang_ground_truth: a buffer is memory of another GPU");
    if (nq == 0) return BANG_OK;
    const size_t esz = dtype == BANG_F32 ? 4 : 1;
    // query rows in dynamic shared memory; with the thresholds (static) under 48 KB
    const uint32_t tileq = static_cast<uint32_t>(std::min<size_t>(kTileQ, (46u * 1024u) / (d * esz)));
    if (tileq == 0) return gtfail(BANG_EINVAL, "bang_ground_truth: rows too long");
    int prev = -1;
    cudaGetDevice(&prev);
    if (cudaSetDevice(device) != cudaSuccess) {
        cudaGetLastError();
        return gtfail(BANG_ECUDA, "bang_ground_truth: cannot select the device");
    }
    struct Restore { int d; ~Restore() { if (d >= 0) cudaSetDevice(d); } } restore{prev};
    cudaStream_t st = static_cast<cudaStream_t>(stream);

    DArr<unsigned char> dbase, dq;
    const void *B = base, *Q = queries;
    if (!is_dev(base)) {
        GT_TRY(dbase.alloc(n * d * esz));
        GT_TRY(cudaMemcpyAsync(dbase.p, base, n * d * esz, cudaMemcpyHostToDevice, st));
        B = dbase.p;
    }
    if (!is_dev(queries)) {
        GT_TRY(dq.alloc(static_cast<uint64_t>(nq) * d * esz));
        GT_TRY(cudaMemcpyAsync(dq.p, queries, static_cast<uint64_t>(nq) * d * esz, cudaMemcpyHostToDevice, st));
        Q = dq.p;
    }
    const bool dev_out = is_dev(out_ids);
    // kQueries queries at a time, fewer where their candidate lists do not fit
    // (they are longer than those of a single pass over the points), in the end
    // without the tensor cores' operands
    uint64_t block = kQueries;
    bool tensor = true;
    for (uint64_t q0 = 0; q0 < nq;) {
        const uint32_t m = static_cast<uint32_t>(nq - q0 < block ? nq - q0 : block);
        const int rc = truth_of(device, B, static_cast<const unsigned char *>(Q) + q0 * d * esz, dtype, n, m, d, k, tileq,
                                tensor, out_ids + q0 * k, out_dist + q0 * k, dev_out, st);
        if (rc == BANG_ENOMEM && m > kLeastQueries) {
            block = (m + 1u) / 2u;
            continue;
        }
        if (rc == BANG_ENOMEM && tensor) {
            tensor = false;
            continue;
        }
        if (rc != BANG_OK) return rc;
        q0 += m;
    }
    return BANG_OK;
}
