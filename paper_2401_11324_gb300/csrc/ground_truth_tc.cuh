// Ground truth, step 2 on the tensor cores (tcgen05): every pair's distance
// against the query's limit as a dense queries x points contraction,
//   |q|^2 + |x|^2 - 2 q.x <= threshold   <=>   xx - 2 v <= lim.
//
// Integer data (uint8, int8; d <= 256): the values are exact in FP16 and the
// sums (at most 256 * 255^2 < 2^24) in the FP32 accumulator, so a pair that
// passes the filter gets its exact distance from v.  FP32 data (d <= 208):
// both sides are split into two BF16 parts (three products).  What is left out
// and the rounding of up to 624 FP32 additions put v off by less than
// 2^-13 |q| |x|, so 2 v by less than 2^-13 (|q|^2 + |x|^2); the filter is twice
// that wider and a pair that passes gets its FP64 distance from the rows.
//
// The points are converted once per level (at most kTcPoints at a time) into
// tiles of 256 points laid out as the MMA reads them: per 16 dimensions (and
// part) one block of 256 x 16 16-bit values in no-swizzle K-major core
// matrices, 8 KB; so a tile is one contiguous stretch and is fetched by bulk
// copies into a ring of 32 KB stages.  A CTA keeps 256 queries in shared memory
// (128 when a tile has more than 8 blocks; three stages above 16) and streams over its share of the
// tiles: one warp copies, one issues the MMAs (M = 128, N = 256), and two
// groups of eight warps read the two TMEM accumulators, half the columns each,
// one accumulator while the other is being computed.  Few pairs pass: they are
// kept in shared memory, 4 per thread, and appended to the query's list with
// one atomic, by all lanes of a warp together (so the first level, where a tenth
// of the pairs passes, took 0.64 ms instead of 0.87).  The filter
// sets the pace (216 instructions per 32 x 32 pairs; 10^10 pairs take the MMAs
// alone 1.4 ms): with four warps a group, two a scheduler, the three levels of
// 10,000 queries over 1M points took 7.5 ms (tensor pipe 23 %), with eight 6.1
// (27 %; half the issue rate, the warps waiting for the accumulators most);
// packed FP32 arithmetic with a three-way minimum and loads one step ahead
// changed nothing.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace gt_tc {

constexpr uint32_t kTileP = 256;            // points per tile, queries per tile
constexpr uint32_t kBlock = 8192;           // bytes of one 256 x 16 block
constexpr uint32_t kStageBlocks = 4;
__host__ __device__ constexpr uint32_t stages(uint32_t nblk) { return nblk <= 16u ? 4u : 3u; }
constexpr uint32_t kKeep = 4;               // pairs kept per thread before they are appended
constexpr uint32_t kFilter = 512;           // filtering threads: two per accumulator row
constexpr uint32_t kThreads = 128 + kFilter;
constexpr uint32_t kMaxBlocks = 26;         // 26 x 4 KB of queries beside three stages
constexpr uint64_t kTcPoints = 1u << 20;    // points converted at a time (832 MB at most)
constexpr long long kWaitCycles = 6000000000ll;      // about 3 s

struct TcArgs {
    const void *base, *queries;             // raw rows
    int dtype;
    uint32_t d, nblk;                       // blocks per tile
    uint32_t nq;
    uint64_t first, count, stride;          // this launch's points: ids (first + i) * stride, i < count
    const unsigned char *ptiles, *qtiles;
    const float *pnorm;                     // per point of the launch: xx as the filter takes it
    const float *lim, *qq;                  // per query
    const double *thr;
    uint32_t *cnt;
    double *cd;
    uint32_t *ci;
    uint64_t cap;
    uint32_t tiles_per_cta;
    unsigned int *err;
};

__device__ __forceinline__ uint32_t saddr(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

// Bounded wait of one thread; gives up when another role has (bad not null).
__device__ __forceinline__ bool wait(uint32_t bar, uint32_t parity, volatile uint32_t *bad)
{
    long long began = 0;
    for (uint32_t i = 0;; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred P;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, P;\n\t}\n"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if (bad && *bad) return false;
        if (i == 0) began = clock64();
        else if (clock64() - began > kWaitCycles) {
            if (bad) *bad = 1u;
            return false;
        }
    }
}
__device__ __forceinline__ void init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void arrive(uint32_t bar)
{
    asm volatile("{\n\t.reg .b64 t;\n\tmbarrier.arrive.shared::cta.b64 t, [%0];\n\t}\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void expect(uint32_t bar, uint32_t bytes)
{
    asm volatile("{\n\t.reg .b64 t;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 t, [%0], %1;\n\t}\n" ::"r"(bar), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}
// No-swizzle K-major operand: K-adjacent core matrices 128 bytes apart,
// M/N-adjacent ones 256.
__device__ __forceinline__ uint64_t desc(uint32_t a)
{
    return static_cast<uint64_t>((a & 0x3FFFFu) >> 4) | (static_cast<uint64_t>(128u >> 4) << 16) |
           (static_cast<uint64_t>(256u >> 4) << 32) | (static_cast<uint64_t>(1u) << 46);
}
__device__ __forceinline__ void mma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void ld32(uint32_t taddr, float (&v)[32])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
        "%12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, "
        "%30, %31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
          "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
          "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ float value(const void *X, int dtype, uint64_t i)
{
    if (dtype == 0) return static_cast<float>(static_cast<const uint8_t *>(X)[i]);
    if (dtype == 1) return static_cast<float>(static_cast<const int8_t *>(X)[i]);
    return static_cast<const float *>(X)[i];
}

// One 256-row tile per block, a row per thread: rows (first + i) * stride of
// X, i < count, zero rows beyond.  norm (may be null): the filter's xx,
// +infinity beyond count.  *odd is set when an FP32 row's norm is not finite
// or too large for the filter.
__global__ void __launch_bounds__(kTileP) convert(const void *X, int dtype, uint32_t d, uint32_t nblk, uint64_t first,
                                                  uint64_t count, uint64_t stride, unsigned char *tiles, float *norm,
                                                  unsigned int *odd)
{
    const uint32_t r = threadIdx.x;
    const uint64_t i = static_cast<uint64_t>(blockIdx.x) * kTileP + r;
    const bool valid = i < count;
    const uint64_t row = (first + i) * stride * d;
    unsigned char *t = tiles + static_cast<uint64_t>(blockIdx.x) * nblk * kBlock + (r >> 3) * 256u + (r & 7u) * 16u;
    const uint32_t parts = dtype == 2 ? 2u : 1u;
    double n2 = 0.0;
    uint32_t n2i = 0;
    const bool vec = dtype != 2 && d % 16u == 0 && (reinterpret_cast<uintptr_t>(X) & 15u) == 0;
    for (uint32_t kb = 0; kb < nblk / parts; ++kb) {
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        if (vec && valid) w = *reinterpret_cast<const uint4 *>(static_cast<const unsigned char *>(X) + row + kb * 16u);
        const uint32_t wb[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (uint32_t half = 0; half < 2; ++half) {
            uint32_t h[4] = {0u, 0u, 0u, 0u}, l[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (uint32_t e = 0; e < 8; ++e) {
                const uint32_t j = kb * 16u + half * 8u + e;
                float x = 0.0f;
                if (vec) {
                    const uint32_t b = (wb[half * 2u + (e >> 2)] >> (8u * (e & 3u))) & 0xFFu;
                    x = dtype == 0 ? static_cast<float>(b) : static_cast<float>(static_cast<int8_t>(b));
                } else if (valid && j < d) {
                    x = value(X, dtype, row + j);
                }
                uint32_t hb, lb = 0;
                if (dtype == 2) {
                    n2 += static_cast<double>(x) * static_cast<double>(x);
                    const __nv_bfloat16 xh = __float2bfloat16_rn(x);
                    hb = __bfloat16_as_ushort(xh);
                    lb = __bfloat16_as_ushort(__float2bfloat16_rn(x - __bfloat162float(xh)));
                } else {
                    const int v = static_cast<int>(x);
                    n2i += static_cast<uint32_t>(v * v);
                    hb = __half_as_ushort(__float2half_rn(x));
                }
                h[e >> 1] |= hb << (16u * (e & 1u));
                l[e >> 1] |= lb << (16u * (e & 1u));
            }
            unsigned char *o = t + static_cast<uint64_t>(kb) * parts * kBlock + half * 128u;
            *reinterpret_cast<uint4 *>(o) = make_uint4(h[0], h[1], h[2], h[3]);
            if (dtype == 2) *reinterpret_cast<uint4 *>(o + kBlock) = make_uint4(l[0], l[1], l[2], l[3]);
        }
    }
    if (dtype == 2 && valid && !(n2 < 1e30)) *odd = 1u;
    if (norm) {
        float v = __uint_as_float(0x7F800000u);
        if (valid) v = dtype == 2 ? __double2float_rd(n2 * (1.0 - 0x1p-12)) : static_cast<float>(n2i);
        norm[i] = v;
    }
}

// The filter's limit of every query for its threshold, and |q|^2.
__global__ void limits(const void *Q, int dtype, uint32_t d, uint32_t nq, const double *thr, float *lim, float *qq)
{
    const uint32_t q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nq) return;
    double n2 = 0.0;
    for (uint32_t j = 0; j < d; ++j) {
        const double x = value(Q, dtype, static_cast<uint64_t>(q) * d + j);
        n2 += x * x;
    }
    qq[q] = static_cast<float>(n2);              // exact for integers (below 2^24)
    // integers: xx - 2 v is exact below 2^24, else within 2 of it
    lim[q] = __double2float_ru(thr[q] - n2 + (dtype == 2 ? n2 * 0x1p-12 + 1e-35 : 4.0));
}

// FP64 distance as the ground truth defines it.
__device__ __forceinline__ double exact64(const float *q, const float *x, uint32_t d)
{
    double acc = 0.0;
    for (uint32_t j = 0; j < d; ++j) {
        const double t = __dsub_rn(static_cast<double>(q[j]), static_cast<double>(x[j]));
        acc = __dadd_rn(acc, __dmul_rn(t, t));
    }
    return acc;
}

inline uint32_t smem_bytes(uint32_t nblk)
{
    const uint32_t a = nblk <= 8u ? nblk * kBlock : nblk * kBlock / 2u;
    return a + stages(nblk) * kStageBlocks * kBlock + 2u * kTileP * 4u + kKeep * kFilter * 12u + 256u;
}

// DT: 0 integer data (FP16 operands), 1 FP32 data (BF16 operands, two parts).
template <int DT>
__global__ void __launch_bounds__(kThreads, 1) collect_tc(const TcArgs a)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31u;
    const bool two = a.nblk <= 8u;               // 256 queries per CTA, else 128
    const uint32_t abytes = two ? a.nblk * kBlock : a.nblk * kBlock / 2u;
    unsigned char *A = smem, *B = A + abytes;
    const uint32_t kStages = stages(a.nblk);
    float *nrm = reinterpret_cast<float *>(B + kStages * kStageBlocks * kBlock);      // 2 x 256
    double *kd = reinterpret_cast<double *>(nrm + 2u * kTileP);
    uint32_t *ki = reinterpret_cast<uint32_t *>(kd + kKeep * kFilter);
    uint64_t *bars = reinterpret_cast<uint64_t *>(ki + kKeep * kFilter);
    const uint32_t b0 = saddr(bars);
    // full / empty stage, full / empty norms, full / empty accumulator, queries
    const uint32_t full = b0, empty = b0 + 32u, nfull = b0 + 64u, nempty = b0 + 80u, tfull = b0 + 96u,
                   tempty = b0 + 112u, qbar = b0 + 128u;
    volatile uint32_t *bad = reinterpret_cast<volatile uint32_t *>(bars + 17);
    uint32_t *slot = reinterpret_cast<uint32_t *>(bars + 18);
    if (tid == 0) {
        for (uint32_t s = 0; s < kStages; ++s) {
            init(full + 8u * s, 1);
            init(empty + 8u * s, 1);
        }
        for (uint32_t s = 0; s < 2; ++s) {
            init(nfull + 8u * s, 1);
            init(nempty + 8u * s, two ? 16 : 8);          // one arrival per warp
            init(tfull + 8u * s, 1);
            init(tempty + 8u * s, 8);
        }
        init(qbar, 1);
        *bad = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(saddr(slot)), "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = *slot;
    const uint32_t ntiles_all = static_cast<uint32_t>((a.count + kTileP - 1) / kTileP);
    const uint32_t t0 = blockIdx.x * a.tiles_per_cta;
    const uint32_t nt = t0 >= ntiles_all ? 0u : (ntiles_all - t0 < a.tiles_per_cta ? ntiles_all - t0 : a.tiles_per_cta);
    const uint32_t nch = (a.nblk + kStageBlocks - 1u) / kStageBlocks;
    const uint32_t q0 = blockIdx.y * (two ? 256u : 128u);

    if (warp == 0 && lane == 0) {
        // ---- copies
        const unsigned char *qt = a.qtiles + static_cast<uint64_t>(q0 / kTileP) * a.nblk * kBlock;
        expect(qbar, abytes);
        if (two) {
            for (uint32_t o = 0; o < abytes; o += kBlock) copy(saddr(A + o), qt + o, kBlock, qbar);
        } else {                                 // the upper or lower 128 rows of every block
            for (uint32_t b = 0; b < a.nblk; ++b)
                copy(saddr(A + b * kBlock / 2u), qt + b * kBlock + ((q0 & 128u) ? kBlock / 2u : 0u), kBlock / 2u, qbar);
        }
        uint32_t it = 0, nit = 0;
        bool ok = true;
        for (uint32_t t = 0; t < nt && ok; ++t) {
            const uint32_t ns = t & 1u;
            ok = wait(nempty + 8u * ns, ((t >> 1) & 1u) ^ 1u, bad);
            if (!ok) break;
            nit = t + 1u;
            expect(nfull + 8u * ns, kTileP * 4u);
            copy(saddr(nrm + ns * kTileP), a.pnorm + static_cast<uint64_t>(t0 + t) * kTileP, kTileP * 4u, nfull + 8u * ns);
            const unsigned char *src = a.ptiles + static_cast<uint64_t>(t0 + t) * a.nblk * kBlock;
            for (uint32_t c = 0; c < nch; ++c, ++it) {
                const uint32_t s = it % kStages;
                const uint32_t nb = a.nblk - c * kStageBlocks < kStageBlocks ? a.nblk - c * kStageBlocks : kStageBlocks;
                ok = wait(empty + 8u * s, ((it / kStages) & 1u) ^ 1u, bad);
                if (!ok) break;
                expect(full + 8u * s, nb * kBlock);
                copy(saddr(B + s * kStageBlocks * kBlock), src + c * kStageBlocks * kBlock, nb * kBlock, full + 8u * s);
            }
        }
        // every copy issued has landed before the block ends (also after a failure)
        wait(qbar, 0u, nullptr);
        for (uint32_t i = it > kStages ? it - kStages : 0u; i < it; ++i)
            wait(full + 8u * (i % kStages), (i / kStages) & 1u, nullptr);
        for (uint32_t t = nit > 2u ? nit - 2u : 0u; t < nit; ++t) wait(nfull + 8u * (t & 1u), (t >> 1) & 1u, nullptr);
    } else if (warp == 1 && lane == 0) {
        // ---- MMAs
        constexpr uint32_t fmt = DT == 0 ? 0u : 1u;          // FP16 or BF16
        constexpr uint32_t idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((kTileP >> 3) << 17) | ((128u >> 4) << 24);
        bool ok = wait(qbar, 0u, bad);
        uint32_t it = 0;
        const uint32_t ablk = two ? kBlock : kBlock / 2u;
        for (uint32_t t = 0; t < nt && ok; ++t, it += nch) {
            for (uint32_t h = 0; h < (two ? 2u : 1u) && ok; ++h) {
                const uint32_t g = two ? h : (t & 1u);       // accumulator
                const uint32_t use = two ? t : t >> 1;       // how often it was used before
                ok = wait(tempty + 8u * g, (use & 1u) ^ 1u, bad);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                uint32_t acc = 0;
                for (uint32_t c = 0; c < nch && ok; ++c) {
                    const uint32_t i = it + c, s = i % kStages;
                    if (h == 0) ok = wait(full + 8u * s, (i / kStages) & 1u, bad);
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    const uint32_t nb = a.nblk - c * kStageBlocks < kStageBlocks ? a.nblk - c * kStageBlocks : kStageBlocks;
                    const uint32_t bs = saddr(B + s * kStageBlocks * kBlock);
                    const uint32_t as = saddr(A) + c * kStageBlocks * ablk + (two ? h * (kBlock / 2u) : 0u);
                    for (uint32_t b = 0; b < nb; b += DT == 0 ? 1u : 2u) {
                        mma(tmem + g * 256u, desc(as + b * ablk), desc(bs + b * kBlock), idesc, acc);
                        acc = 1;
                        if (DT == 1) {           // high x low, low x high
                            mma(tmem + g * 256u, desc(as + b * ablk), desc(bs + (b + 1u) * kBlock), idesc, 1u);
                            mma(tmem + g * 256u, desc(as + (b + 1u) * ablk), desc(bs + b * kBlock), idesc, 1u);
                        }
                    }
                    if (!two || h == 1) commit(empty + 8u * s);
                }
                if (ok) commit(tfull + 8u * g);
            }
        }
    } else if (warp >= 4) {
        // ---- filter: this thread's query against half of the tile's points
        const uint32_t g = (warp - 4u) >> 3, half = ((warp - 4u) >> 2) & 1u, r = (warp & 3u) * 32u + lane, me = tid - 128u;
        const uint32_t q = q0 + (two ? g * 128u : 0u) + r;
        const bool mine = q < a.nq;
        const float lim = mine ? a.lim[q] : __uint_as_float(0xFF800000u);
        const float qq = mine ? a.qq[q] : 0.0f;
        const double thr = mine ? a.thr[q] : 0.0;
        uint32_t kept = 0;
        auto flush = [&]() {
            if (kept == 0u) return;
            const uint32_t at = atomicAdd(a.cnt + q, kept);
            for (uint32_t i = 0; i < kept; ++i)
                if (at + i < a.cap) {
                    a.cd[static_cast<uint64_t>(q) * a.cap + at + i] = kd[i * kFilter + me];
                    a.ci[static_cast<uint64_t>(q) * a.cap + at + i] = ki[i * kFilter + me];
                }
            kept = 0;
        };
        for (uint32_t t = two ? 0u : g; t < nt; t += two ? 1u : 2u) {
            const uint32_t use = two ? t : t >> 1, ns = t & 1u;
            const bool ok = wait(tfull + 8u * g, use & 1u, bad) && wait(nfull + 8u * ns, (t >> 1) & 1u, bad);
            if (!__all_sync(0xFFFFFFFFu, ok)) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const float4 *xn = reinterpret_cast<const float4 *>(nrm + ns * kTileP);
            for (uint32_t c0 = half * (kTileP / 2u); c0 < (half + 1u) * (kTileP / 2u); c0 += 32) {
                float v[32];
                ld32(tmem + g * 256u + (((warp & 3u) * 32u) << 16) + c0, v);
                uint32_t pass = 0;
#pragma unroll
                for (int i = 0; i < 32; i += 4) {
                    const float4 x4 = xn[(c0 + i) / 4u];
                    pass |= fmaf(-2.0f, v[i], x4.x) <= lim ? 1u << i : 0u;
                    pass |= fmaf(-2.0f, v[i + 1], x4.y) <= lim ? 2u << i : 0u;
                    pass |= fmaf(-2.0f, v[i + 2], x4.z) <= lim ? 4u << i : 0u;
                    pass |= fmaf(-2.0f, v[i + 3], x4.w) <= lim ? 8u << i : 0u;
                }
                while (pass) {
                    const int i = __ffs(pass) - 1;
                    pass &= pass - 1u;
                    const uint64_t p = static_cast<uint64_t>(t0 + t) * kTileP + c0 + i;
                    if (p >= a.count) break;                 // the last tile's padding
                    const uint64_t id = (a.first + p) * a.stride;
                    double dist;
                    if (DT == 0) {
                        float vi = 0.0f;
#pragma unroll
                        for (int e = 0; e < 32; ++e) vi = e == i ? v[e] : vi;
                        const int x2 = static_cast<int>(nrm[ns * kTileP + c0 + i]);
                        dist = static_cast<double>(static_cast<int>(qq) + x2 - 2 * static_cast<int>(vi));
                    } else {
                        dist = exact64(static_cast<const float *>(a.queries) + static_cast<uint64_t>(q) * a.d,
                                       static_cast<const float *>(a.base) + id * a.d, a.d);
                    }
                    if (dist <= thr) {
                        if (kept == kKeep) flush();
                        kd[kept * kFilter + me] = dist;
                        ki[kept * kFilter + me] = static_cast<uint32_t>(id);
                        ++kept;
                    }
                }
                // all lanes at once, so that the warp waits for one atomic's
                // round trip and not for one per lane
                if (__any_sync(0xFFFFFFFFu, kept >= kKeep - 1u)) flush();
                __syncwarp();
            }
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) {
                arrive(tempty + 8u * g);
                arrive(nempty + 8u * ns);
            }
        }
        if (mine) flush();
    }
    __syncthreads();
    if (tid == 0 && *bad) atomicExch(a.err, 1u);
    if (warp == 2) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512u) : "memory");
    }
}

}  // namespace gt_tc
