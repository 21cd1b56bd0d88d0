// GPU product quantisation (§4: the vector is split into M contiguous
// subspaces, the first d mod M of them one dimension wider; 256 centroids
// per subspace by k-means; a point's code is its nearest centroid in each
// subspace).  Training runs Lloyd iterations from the given initial points:
// assignment to the nearest centroid (FP64 distance summed in ascending
// dimension order, each difference, product and sum rounded; ties to the
// smaller centroid), then every centroid becomes the FP64 mean of its
// points, summed in training-sample order (a centroid with no points keeps
// its position).  Encoding uses the FP32 codebook the same way.  Every sum
// has a fixed order, so codebook and codes are the same bytes on every run.
//
// Assignment and encoding: one thread per (point, subspace), the subspace's
// centroids in shared memory.  What bounds them is arithmetic, 256 distances
// a thread, and FP64 runs at a sixtieth of the FP32 rate here.  So every
// distance is computed in FP32 first, keeping the smallest and the second
// smallest; the FP64 distances are computed only where the second lies within
// both values' rounding errors of the smallest (`cut`), and then only for the
// centroids that do.  The result is the FP64 one always.
// Update: integer sums are exact in any order, so uint8 and int8 points are
// added with shared-memory atomics, a block per part of the sample; float
// points keep the order: one warp per (subspace, centroid) looks for its points
// in the assignments (4 bytes a lane), reads 32 points at a time and sums them.
// 100,000 training points of u8, d = 128, M = 32: assignment 24.2 -> 0.45 ms an
// iteration; update 16.6 ms with a thread per (subspace, centroid), 1.0 with the
// warp, under 0.1 with the atomics; encoding 400,000 points 130 -> 1.6 ms.  The
// whole call with 10 iterations: 538 -> 7.6 ms.
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "bang.h"
#include "bang_internal.h"

namespace {

constexpr uint32_t kMaxDsub = 16;       // dimensions per subspace

struct PArgs {
    const void *X;              // n x d elements of dtype (device)
    int dtype;
    uint32_t d, M;
    const uint32_t *off;        // M + 1
    const uint64_t *sample;     // ns row ids
    uint64_t ns, n;
    uint64_t ns_pad;            // assignments per subspace, a multiple of 4
    double *cent;               // 256 * d, subspace s at 256 * off[s], centroid c at + c * ds
    uint8_t *asg;               // M x ns_pad assignments
    unsigned long long *isum, *icnt;    // integer points: sums like cent, counts like the centroids
    const float *cb;            // 256 * d codebook (encode)
    uint8_t *codes;             // n x M
};

__device__ __forceinline__ double elem(const PArgs &a, uint64_t i)
{
    if (a.dtype == 0) return static_cast<double>(static_cast<const uint8_t *>(a.X)[i]);
    if (a.dtype == 1) return static_cast<double>(static_cast<const int8_t *>(a.X)[i]);
    return static_cast<double>(static_cast<const float *>(a.X)[i]);
}

// Nearest centroid of x among the 256 in c (FP32, row-major DS wide), where
// it is certain; otherwise false and the candidates' upper bound in cut.
// cerr: bound on |c_j| for centroids that were rounded to FP32, 0 for exact
// ones.  Error of an FP32 distance a against the FP64 one: each difference is
// off by at most 2^-24 (|x_j - c_j| + |c_j|), each product and sum by 2^-24
// relative, so by at most alpha a + beta sqrt(a) with alpha = (DS + 4) 2^-23
// and beta = 2^-22 sqrt(DS) cerr.  A centroid whose a exceeds the smallest, m,
// by more than 3 alpha m + 6 beta sqrt(m) + 16 beta^2 cannot be nearer.
template <uint32_t DS>
__device__ __forceinline__ bool nearest32(const float (&x)[kMaxDsub], const float *c, uint32_t ds, float cerr,
                                          uint32_t &best, float &cut)
{
    const uint32_t w = DS ? DS : ds;
    float m1 = __int_as_float(0x7F800000), m2 = m1;
    uint32_t i1 = 0;
#pragma unroll 4
    for (uint32_t cc = 0; cc < 256; ++cc) {
        float a = 0.0f;
        if (DS == 4) {
            const float4 v = reinterpret_cast<const float4 *>(c)[cc];
            float t = x[0] - v.x; a = t * t;
            t = x[1] - v.y; a = __fmaf_rn(t, t, a);
            t = x[2] - v.z; a = __fmaf_rn(t, t, a);
            t = x[3] - v.w; a = __fmaf_rn(t, t, a);
        } else {
#pragma unroll
            for (uint32_t j = 0; j < (DS ? DS : kMaxDsub); ++j)
                if (DS || j < ds) {
                    const float t = x[j] - c[cc * w + j];
                    a = __fmaf_rn(t, t, a);
                }
        }
        m2 = fminf(m2, fmaxf(m1, a));
        if (a < m1) {
            m1 = a;
            i1 = cc;
        }
    }
    best = i1;
    const float alpha = static_cast<float>(w + 4u) * 0x1p-23f, beta = 0x1p-22f * sqrtf(static_cast<float>(w)) * cerr;
    cut = m1 + 3.0f * alpha * m1 + 6.0f * beta * sqrtf(m1) + 16.0f * beta * beta;
    cut = cut * (1.0f + 0x1p-20f) + 1e-30f;      // the bound's own rounding; products that underflow
    return m1 < 1e37f && m2 > cut;               // beyond: overflow, infinities, NaN
}

// The FP64 rule: distances in ascending dimension order, each difference,
// product and sum rounded, ties to the smaller centroid; over the centroids
// whose FP32 distance is at most cut (all when cut is not finite).
template <typename C>
__device__ __noinline__ uint32_t nearest64(const float *x, const float *c32, const C *c, uint32_t ds, float cut)
{
    double best = __longlong_as_double(0x7FF0000000000000ll);     // +inf
    uint32_t bc = 0;
    for (uint32_t cc = 0; cc < 256; ++cc) {
        float a = 0.0f;
        for (uint32_t j = 0; j < ds; ++j) {
            const float t = x[j] - c32[cc * ds + j];
            a = __fmaf_rn(t, t, a);
        }
        if (a > cut && cut < 1e37f) continue;
        double acc = 0.0;
        for (uint32_t j = 0; j < ds; ++j) {
            const double t = __dsub_rn(static_cast<double>(x[j]), static_cast<double>(c[cc * ds + j]));
            acc = __dadd_rn(acc, __dmul_rn(t, t));
        }
        if (acc < best) { best = acc; bc = cc; }
    }
    return bc;
}

template <typename C>
__device__ __forceinline__ uint32_t nearest(const float (&x)[kMaxDsub], const float *c32, const C *c, uint32_t ds,
                                            float cerr)
{
    uint32_t best;
    float cut;
    bool sure;
    if (ds == 4) sure = nearest32<4>(x, c32, ds, cerr, best, cut);
    else if (ds == 2) sure = nearest32<2>(x, c32, ds, cerr, best, cut);
    else if (ds == 3) sure = nearest32<3>(x, c32, ds, cerr, best, cut);
    else sure = nearest32<0>(x, c32, ds, cerr, best, cut);
    if (sure) return best;
    float xv[kMaxDsub];
    for (uint32_t j = 0; j < kMaxDsub; ++j) xv[j] = x[j];
    return nearest64(xv, c32, c, ds, cut);
}

__device__ __forceinline__ float elem32(const PArgs &a, uint64_t i)      // exact
{
    if (a.dtype == 0) return static_cast<float>(static_cast<const uint8_t *>(a.X)[i]);
    if (a.dtype == 1) return static_cast<float>(static_cast<const int8_t *>(a.X)[i]);
    return static_cast<const float *>(a.X)[i];
}

// This thread's sub-vector (zeros beyond ds).
__device__ __forceinline__ void load_sub(const PArgs &a, uint64_t row, uint32_t ds, float (&x)[kMaxDsub])
{
#pragma unroll
    for (uint32_t j = 0; j < kMaxDsub; ++j) x[j] = j < ds ? elem32(a, row + j) : 0.0f;
}

// blockIdx.y = subspace; threads over the training sample.
__global__ void __launch_bounds__(256) assign(const PArgs a)
{
    __shared__ __align__(16) float c32[256 * kMaxDsub];
    __shared__ float big[256];
    const uint32_t s = blockIdx.y, o = a.off[s], ds = a.off[s + 1] - o;
    const double *c = a.cent + 256ull * o;
    float mx = 0.0f;
    for (uint32_t i = threadIdx.x; i < 256 * ds; i += blockDim.x) {
        c32[i] = __double2float_rn(c[i]);
        mx = fmaxf(mx, fabsf(c32[i]));
    }
    big[threadIdx.x] = mx;
    __syncthreads();
    for (uint32_t h = 128; h > 0; h >>= 1) {
        if (threadIdx.x < h) big[threadIdx.x] = fmaxf(big[threadIdx.x], big[threadIdx.x + h]);
        __syncthreads();
    }
    const float cerr = big[0];
    for (uint64_t i = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; i < a.ns;
         i += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
        float x[kMaxDsub];
        load_sub(a, a.sample[i] * a.d + o, ds, x);
        a.asg[static_cast<uint64_t>(s) * a.ns_pad + i] = static_cast<uint8_t>(nearest(x, c32, c, ds, cerr));
    }
}

// Integer points: sums and counts per centroid of this block's part of the
// sample, added to the subspace's (blockIdx.y).  At most 2^20 points a block
// keep the 32-bit sums exact.
constexpr uint64_t kIntPart = 1u << 20;
__global__ void __launch_bounds__(256) update_int(const PArgs a)
{
    __shared__ int sum[256 * kMaxDsub];
    __shared__ uint32_t cnt[256];
    const uint32_t s = blockIdx.y, o = a.off[s], ds = a.off[s + 1] - o;
    for (uint32_t i = threadIdx.x; i < 256 * ds; i += blockDim.x) sum[i] = 0;
    cnt[threadIdx.x] = 0;
    __syncthreads();
    const uint64_t per = (a.ns + gridDim.x - 1) / gridDim.x;             // <= kIntPart
    const uint64_t end = per * (blockIdx.x + 1) < a.ns ? per * (blockIdx.x + 1) : a.ns;
    for (uint64_t i = per * blockIdx.x + threadIdx.x; i < end; i += blockDim.x) {
        const uint32_t c = a.asg[static_cast<uint64_t>(s) * a.ns_pad + i];
        const uint64_t row = a.sample[i] * a.d + o;
        atomicAdd(&cnt[c], 1u);
        for (uint32_t j = 0; j < ds; ++j)
            atomicAdd(&sum[c * ds + j], a.dtype == 0 ? static_cast<int>(static_cast<const uint8_t *>(a.X)[row + j])
                                                     : static_cast<int>(static_cast<const int8_t *>(a.X)[row + j]));
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < 256 * ds; i += blockDim.x)
        if (sum[i]) atomicAdd(a.isum + 256ull * o + i, static_cast<unsigned long long>(static_cast<long long>(sum[i])));
    if (cnt[threadIdx.x]) atomicAdd(a.icnt + 256ull * s + threadIdx.x, static_cast<unsigned long long>(cnt[threadIdx.x]));
}

__global__ void mean_int(const PArgs a)
{
    const uint32_t s = blockIdx.x, cc = threadIdx.x;      // 256 threads
    const uint32_t o = a.off[s], ds = a.off[s + 1] - o;
    const unsigned long long cnt = a.icnt[256ull * s + cc];
    if (cnt == 0) return;
    for (uint32_t j = 0; j < ds; ++j) {
        const uint64_t i = 256ull * o + static_cast<uint64_t>(cc) * ds + j;
        a.cent[i] = __ddiv_rn(static_cast<double>(static_cast<long long>(a.isum[i])), static_cast<double>(cnt));
    }
}

// One warp per (subspace, centroid): the mean of its points in sample order.
// Matches are queued in order, 32 at a time are read (a point a lane) and
// summed (a dimension a lane).
constexpr uint32_t kUpWarps = 4;
__global__ void __launch_bounds__(32 * kUpWarps) update(const PArgs a)
{
    __shared__ uint64_t rows[kUpWarps][32];
    __shared__ float val[kUpWarps][kMaxDsub][33];
    const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
    const uint32_t job = blockIdx.x * kUpWarps + w;
    if (job >= a.M * 256u) return;
    const uint32_t s = job >> 8, cc = job & 255u;
    const uint32_t o = a.off[s], ds = a.off[s + 1] - o;
    const uint32_t *as = reinterpret_cast<const uint32_t *>(a.asg + static_cast<uint64_t>(s) * a.ns_pad);
    const uint32_t pat = cc * 0x01010101u;
    double sum = 0.0;                    // lane j < ds: dimension j
    uint64_t cnt = 0;
    uint32_t queued = 0;
    auto drain = [&]() {
        __syncwarp();
        if (lane < queued)
            for (uint32_t j = 0; j < ds; ++j) val[w][j][lane] = elem32(a, rows[w][lane] + j);
        __syncwarp();
        if (lane < ds)
            for (uint32_t t = 0; t < queued; ++t) sum = __dadd_rn(sum, static_cast<double>(val[w][lane][t]));
        cnt += queued;
        queued = 0;
        __syncwarp();
    };
    const uint64_t nw = (a.ns + 3u) / 4u;
    for (uint64_t i0 = 0; i0 < nw; i0 += 32u * 8u) {
        uint32_t v[8];                   // 1,024 assignments requested at once
#pragma unroll
        for (uint32_t t = 0; t < 8; ++t) {
            const uint64_t i = i0 + 32u * t + lane;
            v[t] = i < nw ? as[i] : 0u;
        }
#pragma unroll
        for (uint32_t t = 0; t < 8; ++t) {
            const uint64_t i = (i0 + 32u * t + lane) * 4u;
            uint32_t hit = __vcmpeq4(v[t], pat) & 0x08040201u;           // bit 9 b: byte b matches
            hit = (hit | hit >> 8 | hit >> 16 | hit >> 24) & 0xFu;       // bit b
            if (i + 3u >= a.ns) hit &= i >= a.ns ? 0u : (1u << (a.ns - i)) - 1u;
            uint32_t any = __ballot_sync(0xFFFFFFFFu, hit != 0u);
            while (any) {                // lanes in order, then bytes in order
                const int src = __ffs(any) - 1;
                any &= any - 1u;
                uint32_t h = __shfl_sync(0xFFFFFFFFu, hit, src);
                if (queued + __popc(h) > 32u) drain();
                if (static_cast<int>(lane) == src)
                    for (uint32_t q = queued, hh = h; hh; hh &= hh - 1u, ++q)
                        rows[w][q] = a.sample[i + __ffs(hh) - 1] * a.d + o;
                queued += __popc(h);
            }
        }
    }
    drain();
    if (cnt == 0 || lane >= ds) return;
    a.cent[256ull * o + static_cast<uint64_t>(cc) * ds + lane] = __ddiv_rn(sum, static_cast<double>(cnt));
}

__global__ void to_float(const double *cent, uint64_t count, float *cb)
{
    for (uint64_t i = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; i < count;
         i += static_cast<uint64_t>(gridDim.x) * blockDim.x)
        cb[i] = __double2float_rn(cent[i]);
}

// blockIdx.y = subspace; threads over the points.
__global__ void __launch_bounds__(256) encode(const PArgs a)
{
    __shared__ __align__(16) float c[256 * kMaxDsub];
    const uint32_t s = blockIdx.y, o = a.off[s], ds = a.off[s + 1] - o;
    for (uint32_t i = threadIdx.x; i < 256 * ds; i += blockDim.x) c[i] = a.cb[256ull * o + i];
    __syncthreads();
    for (uint64_t i = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; i < a.n;
         i += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
        float x[kMaxDsub];
        load_sub(a, i * a.d + o, ds, x);
        a.codes[i * a.M + s] = static_cast<uint8_t>(nearest(x, c, c, ds, 0.0f));
    }
}

__global__ void init_cent(const PArgs a, const uint64_t *init)
{
    const uint32_t s = blockIdx.x, cc = threadIdx.x;
    const uint32_t o = a.off[s], ds = a.off[s + 1] - o;
    const uint64_t row = init[static_cast<uint64_t>(s) * 256 + cc] * a.d + o;
    for (uint32_t j = 0; j < ds; ++j) a.cent[256ull * o + static_cast<uint64_t>(cc) * ds + j] = elem(a, row + j);
}

template <typename T> struct DArr {
    T *p = nullptr;
    ~DArr() { if (p) cudaFree(p); }
    cudaError_t alloc(uint64_t count) { return cudaMalloc(&p, sizeof(T) * (count ? count : 1)); }
};

int pfail(int code, const std::string &m)
{
    bang::set_error(m);
    return code;
}

bool is_dev(const void *p)
{
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

}  // namespace

#define PQ_TRY(x)                                                                           \
    do {                                                                                    \
        cudaError_t e_ = (x);                                                               \
        if (e_ != cudaSuccess) {                                                            \
            cudaGetLastError();                                                             \
            return pfail(e_ == cudaErrorMemoryAllocation ? BANG_ENOMEM : BANG_ECUDA,       \
                         std::string(#x) + ": " + cudaGetErrorString(e_));                  \
        }                                                                                   \
    } while (0)

extern "C" int bang_build_pq(int device, const void *base, bang_dtype dtype, uint64_t n, uint32_t d,
                             uint32_t M, const uint64_t *sample, uint64_t ns, const uint64_t *init,
                             uint32_t iters, float *codebook, uint8_t *codes, void *stream)
{
    if (!base || !sample || !init || !codebook || !codes)
        return pfail(BANG_EINVAL, "bang_build_pq: NULL argument");
    if (dtype != BANG_U8 && dtype != BANG_I8 && dtype != BANG_F32)
        return pfail(BANG_EINVAL, "bang_build_pq: unknown dtype");
    if (n == 0 || d == 0 || M == 0 || M > d || ns == 0 || iters > 1000)
        return pfail(BANG_EINVAL, "bang_build_pq: need n, d, ns > 0, 1 <= M <= d, iters <= 1000");
    if ((d + M - 1) / M > kMaxDsub) return pfail(BANG_EINVAL, "bang_build_pq: subspaces wider than 16 dimensions");
    if (bang::pointer_kind(base, device) == 2 || bang::pointer_kind(codebook, device) == 2 ||
        bang::pointer_kind(codes, device) == 2)
        return pfail(BANG_EINVAL, "bang_build_pq: base, codebook or codes is memory of another GPU");
    if (is_dev(sample) || is_dev(init)) return pfail(BANG_EINVAL, "bang_build_pq: sample and init must be host memory");
    for (uint64_t i = 0; i < ns; ++i)
        if (sample[i] >= n) return pfail(BANG_EINVAL, "bang_build_pq: sample id >= n");
    for (uint64_t i = 0; i < 256ull * M; ++i)
        if (init[i] >= n) return pfail(BANG_EINVAL, "bang_build_pq: init id >= n");
    int prev = -1;
    cudaGetDevice(&prev);
    if (cudaSetDevice(device) != cudaSuccess) {
        cudaGetLastError();
        return pfail(BANG_ECUDA, "bang_build_pq: cannot select the device");
    }
    struct Restore { int d; ~Restore() { if (d >= 0) cudaSetDevice(d); } } restore{prev};
    cudaStream_t st = static_cast<cudaStream_t>(stream);

    std::vector<uint32_t> off(M + 1);
    for (uint32_t s = 0, o = 0; s <= M; ++s) {        // first d mod M subspaces one wider (§6.3)
        off[s] = o;
        if (s < M) o += d / M + (s < d % M ? 1u : 0u);
    }
    const uint32_t esz = dtype == BANG_F32 ? 4u : 1u;
    DArr<uint8_t> X, asg, dcodes;
    DArr<uint32_t> doff;
    DArr<uint64_t> dsample, dinit;
    DArr<double> cent;
    DArr<float> cb;
    const void *Xd = base;
    if (!is_dev(base)) {
        PQ_TRY(X.alloc(n * d * esz));
        PQ_TRY(cudaMemcpyAsync(X.p, base, n * d * esz, cudaMemcpyHostToDevice, st));
        Xd = X.p;
    }
    PQ_TRY(doff.alloc(M + 1));
    PQ_TRY(cudaMemcpyAsync(doff.p, off.data(), (M + 1) * 4, cudaMemcpyHostToDevice, st));
    PQ_TRY(dsample.alloc(ns));
    PQ_TRY(cudaMemcpyAsync(dsample.p, sample, ns * 8, cudaMemcpyHostToDevice, st));
    PQ_TRY(dinit.alloc(256ull * M));
    PQ_TRY(cudaMemcpyAsync(dinit.p, init, 256ull * M * 8, cudaMemcpyHostToDevice, st));
    PQ_TRY(cent.alloc(256ull * d));
    PQ_TRY(cb.alloc(256ull * d));
    const uint64_t ns_pad = (ns + 3u) & ~3ull;
    PQ_TRY(asg.alloc(ns_pad * M));
    DArr<unsigned long long> isum;
    if (dtype != BANG_F32) PQ_TRY(isum.alloc(256ull * d + 256ull * M));
    const bool codes_dev = is_dev(codes);
    if (!codes_dev) PQ_TRY(dcodes.alloc(n * M));

    PArgs a;
    std::memset(&a, 0, sizeof a);
    a.X = Xd;
    a.dtype = dtype;
    a.d = d;
    a.M = M;
    a.off = doff.p;
    a.sample = dsample.p;
    a.ns = ns;
    a.ns_pad = ns_pad;
    a.isum = isum.p;
    a.icnt = isum.p ? isum.p + 256ull * d : nullptr;
    a.n = n;
    a.cent = cent.p;
    a.asg = asg.p;
    a.cb = cb.p;
    a.codes = codes_dev ? codes : dcodes.p;
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    init_cent<<<M, 256, 0, st>>>(a, dinit.p);
    // whole waves: four blocks of assign (and of update_int) fit an SM, six of
    // encode (one block more per subspace made the 608 that fit 640: 0.52 ms
    // an iteration instead of 0.45)
    const uint32_t bx = static_cast<uint32_t>(sms) * 4u / M ? static_cast<uint32_t>(sms) * 4u / M : 1u;
    const uint32_t be = static_cast<uint32_t>(sms) * 6u / M ? static_cast<uint32_t>(sms) * 6u / M : 1u;
    const uint64_t least = (ns + kIntPart - 1) / kIntPart;       // parts that keep 32-bit sums exact
    const uint32_t parts = static_cast<uint32_t>(least > bx ? least : bx);
    for (uint32_t it = 0; it < iters; ++it) {
        assign<<<dim3(bx, M), 256, 0, st>>>(a);
        if (dtype == BANG_F32) {
            update<<<M * 256u / kUpWarps, 32 * kUpWarps, 0, st>>>(a);
        } else {
            PQ_TRY(cudaMemsetAsync(isum.p, 0, (256ull * d + 256ull * M) * 8u, st));
            update_int<<<dim3(parts, M), 256, 0, st>>>(a);
            mean_int<<<M, 256, 0, st>>>(a);
        }
    }
    to_float<<<256, 256, 0, st>>>(cent.p, 256ull * d, cb.p);
    encode<<<dim3(be * 3, M), 256, 0, st>>>(a);
    PQ_TRY(cudaGetLastError());
    PQ_TRY(cudaMemcpyAsync(codebook, cb.p, 256ull * d * 4, cudaMemcpyDefault, st));
    if (!codes_dev) PQ_TRY(cudaMemcpyAsync(codes, dcodes.p, n * M, cudaMemcpyDeviceToHost, st));
    PQ_TRY(cudaStreamSynchronize(st));
    return BANG_OK;
}
