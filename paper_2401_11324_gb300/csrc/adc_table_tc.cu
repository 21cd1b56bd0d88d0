// PQ distance tables on the tensor cores (§4.1's PQDistTable as a dense
// queries x centroids contraction), tcgen05 (sm_100 family) form.
//
//   T[q][s][c] = ||q_s||^2 + ||C_s[c]||^2 - 2 q_s . C_s[c]
//
// The cross term is a GEMM per subspace: A = the queries' dimensions of the
// 16-wide K block(s) holding subspace s (128 queries per CTA, BF16), B = the
// 256 centroids of s written into the same 16-wide block with zeros outside
// the subspace's dimensions.  Accuracy: uint8/int8 queries are exact in BF16;
// FP32 queries and the centroids are split into three BF16 parts each (about
// 24 significant bits), and the products that matter (high x all, middle x
// high and middle, low x high) are summed in the FP32 accumulator, which
// gives the cross term to about FP32 accuracy; the norms are FP32.  Tables come out FP32 or
// BF16 (the reduced-precision search form reads BF16 tables).  The TF32 form
// (a.tf32 with centroid tiles rounded to TF32 on the host) rounds both
// operands to TF32 first; a TF32 value is exactly the sum of two BF16 parts,
// so the same MMAs then form exact TF32 x TF32 products with FP32
// accumulation: the numerics of a TF32 GEMM, at about its tensor-pipe cost
// (two BF16 MMAs per TF32 MMA).
//
// Per CTA: 128 threads; thread t owns query row t of the tile (TMEM lane t)
// and writes that row of the query operand when a subspace starts another K
// block (four 4-dimension subspaces share one).
// Operands live in shared memory in the no-swizzle K-major layout: 8-row x
// 16-byte core matrices, K-adjacent cores 128 bytes apart, M/N-adjacent
// cores 256 bytes apart.  One thread issues the MMAs; completion is signalled
// through an mbarrier; every wait is bounded and reports failure in *err.
//
// What bounds it is the table's own bytes (M * 256 entries a query).  A thread's
// TMEM row is one query's entries of the subspace, so storing from registers
// made every warp store touch 32 rows at 16 bytes each; the entries go through
// shared memory instead (rows padded by 16 bytes against bank conflicts) and
// a warp stores 512 contiguous bytes of one row at a time.  The next subspace's
// centroids are fetched by bulk copies during the epilogue, and shared memory is
// sized by the blocks the subspaces really span, so that two CTAs share an SM.
// 10,000 u8 queries, M = 32, FP32 out (328 MB): 268 -> 115 us for the call (2.8 TB/s).
#include <cuda_runtime.h>

#include <cstdint>
#include <cuda_bf16.h>

#include "adc_table_tc.h"

namespace bang {
namespace {

constexpr uint32_t kTile = 128;            // queries per CTA (UMMA M)
constexpr uint32_t kN = 256;               // centroids per subspace (UMMA N)
constexpr uint32_t kACore = 4096;          // bytes of one 128 x 16 BF16 operand
constexpr uint32_t kBCore = 8192;          // bytes of one 256 x 16 BF16 operand
constexpr uint32_t kMaxWaitSpins = 1u << 26;
constexpr uint32_t kSubPerCta = 4;         // subspaces per CTA (grid y covers the rest)

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Shared-memory matrix descriptor: start, leading (K) and stride (M/N) byte
// offsets, fixed version bits for this architecture, no swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr)
{
    uint64_t d = 0;
    d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
    d |= static_cast<uint64_t>(128u >> 4) << 16;   // K-adjacent core matrices
    d |= static_cast<uint64_t>(256u >> 4) << 32;   // M/N-adjacent core matrices
    d |= static_cast<uint64_t>(1u) << 46;
    return d;
}

// Instruction descriptor: FP32 accumulator, BF16 A and B, both K-major,
// N = 256, M = 128.
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((kN >> 3) << 17) | ((kTile >> 4) << 24);

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(kIdesc), "r"(accumulate));
}

__device__ __forceinline__ void mma_commit(uint32_t mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(mbar)
                 : "memory");
}

__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity)
{
    for (uint32_t i = 0; i < kMaxWaitSpins; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred P;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, P;\n\t}\n"
            : "=r"(ok)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float *v)
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

// Round to TF32 (10 mantissa bits), to nearest with ties to even: the
// operands of the TF32 form, whose products the split parts then carry
// exactly (a TF32 value is the sum of two BF16 values).
__device__ __forceinline__ float tf32_rne(float x)
{
    uint32_t u = __float_as_uint(x);
    u += 0xFFFu + ((u >> 13) & 1u);
    return __uint_as_float(u & ~0x1FFFu);
}

// Offset of element (row, k) of a K-major no-swizzle operand with 16 K
// columns: core (row/8, k/8), 8 rows of 16 bytes per core.
__device__ __forceinline__ uint32_t core_off(uint32_t row, uint32_t k)
{
    return ((row >> 3) * 2u + (k >> 3)) * 128u + (row & 7u) * 16u + (k & 7u) * 2u;
}

__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t mbar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(mbar)
                 : "memory");
}

constexpr uint32_t kRowPad = 128u * 4u + 16u;      // staged row: 128 FP32 entries (256 BF16) and the padding

template <int DT>
__global__ void __launch_bounds__(128) adc_table_tc_kernel(TcTableArgs a)
{
    using E = typename TcElem<DT>::T;
    extern __shared__ __align__(1024) unsigned char smem[];
    const uint32_t t = threadIdx.x, warp = t >> 5;
    // carve: query operand (parts x nbmax K blocks x 4 KB), centroid operand
    // (3 parts x nbmax x 8 KB), centroid norms (2 x 256 floats), staged rows,
    // mbarriers (MMAs done, centroids here), TMEM address
    constexpr uint32_t kAParts = DT == 2 ? 3u : 1u;   // integer queries are exact in BF16
    const uint32_t nbmax = a.nbmax;
    unsigned char *Abuf = smem;
    unsigned char *Bbuf = Abuf + kAParts * nbmax * kACore;
    float *cn2 = reinterpret_cast<float *>(Bbuf + 3u * nbmax * kBCore);
    unsigned char *stage = reinterpret_cast<unsigned char *>(cn2 + 2u * kN);
    uint64_t *mbar = reinterpret_cast<uint64_t *>(stage + kTile * kRowPad);
    uint64_t *bbar = mbar + 1;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(mbar + 2);
    const uint32_t lane = t & 31u;
    unsigned char *wstage = stage + warp * 32u * kRowPad;      // this warp's rows

    const uint32_t q0 = blockIdx.x * kTile;
    const uint32_t q = q0 + t;
    const bool valid = q < a.nq;
    const E *qp = static_cast<const E *>(a.queries) + static_cast<uint64_t>(valid ? q : 0u) * a.d;

    if (t == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(mbar)) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(bbar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                         smem_u32(tmem_slot)),
                     "r"(kN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    bool ok = true;

    // this CTA's subspaces: group blockIdx.y of kSubPerCta
    const uint32_t s_begin = blockIdx.y * kSubPerCta;
    const uint32_t s_end = s_begin + kSubPerCta < a.M ? s_begin + kSubPerCta : a.M;
    // centroid tiles of subspace s (three parts per K block, prepared at load
    // time) and its norms, as bulk copies
    auto fetch = [&](uint32_t s) {
        const uint32_t o = a.off[s], kb0 = o / 16u, nb = (a.off[s + 1] - 1u) / 16u - kb0 + 1u;
        const uint32_t bytes = nb * 3u * kBCore;
        asm volatile("{\n\t.reg .b64 t;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 t, [%0], %1;\n\t}\n" ::"r"(
                         smem_u32(bbar)),
                     "r"(bytes + kN * 4u)
                     : "memory");
        const unsigned char *src = a.btiles + static_cast<uint64_t>(a.bfirst[s]) * kBCore;
        for (uint32_t i = 0; i < bytes; i += kBCore) bulk_copy(smem_u32(Bbuf + i), src + i, kBCore, smem_u32(bbar));
        bulk_copy(smem_u32(cn2 + (s & 1u) * kN), a.cnorm + s * kN, kN * 4u, smem_u32(bbar));
    };
    if (t == 0 && s_begin < s_end) fetch(s_begin);
    uint32_t have0 = 0xFFFFFFFFu, have1 = 0;          // K blocks the query operand holds
    for (uint32_t s = s_begin; s < s_end; ++s) {
        const uint32_t o = a.off[s], ds = a.off[s + 1] - o;
        const uint32_t kb0 = o / 16u, kb1 = (o + ds - 1u) / 16u;
        const uint32_t nb = kb1 - kb0 + 1u;              // <= nbmax (computed on the host)
        const float *cn = cn2 + (s & 1u) * kN;
        // ---- this thread's query row over the subspace's K blocks (zero
        // beyond d and nq), split into BF16 parts
        for (uint32_t b = 0; b < nb && (have0 != kb0 || have1 != kb1); ++b)
#pragma unroll
            for (uint32_t half = 0; half < 2; ++half) {
                uint32_t hw[4], mw[4], lw[4];
#pragma unroll
                for (uint32_t e = 0; e < 8; ++e) {
                    const uint32_t j = (kb0 + b) * 16u + half * 8u + e;
                    float x = (valid && j < a.d) ? static_cast<float>(qp[j]) : 0.0f;
                    if (a.tf32) x = tf32_rne(x);
                    const __nv_bfloat16 h = __float2bfloat16_rn(x);
                    const uint32_t sh = 16u * (e & 1u);
                    if ((e & 1u) == 0) hw[e >> 1] = mw[e >> 1] = lw[e >> 1] = 0;
                    hw[e >> 1] |= static_cast<uint32_t>(__bfloat16_as_ushort(h)) << sh;
                    if (kAParts > 1) {
                        const float r1 = x - __bfloat162float(h);
                        const __nv_bfloat16 m = __float2bfloat16_rn(r1);
                        const __nv_bfloat16 l = __float2bfloat16_rn(r1 - __bfloat162float(m));
                        mw[e >> 1] |= static_cast<uint32_t>(__bfloat16_as_ushort(m)) << sh;
                        lw[e >> 1] |= static_cast<uint32_t>(__bfloat16_as_ushort(l)) << sh;
                    }
                }
                const uint32_t e = core_off(t, half * 8u);
                *reinterpret_cast<uint4 *>(Abuf + b * kACore + e) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
                if (kAParts > 1) {
                    *reinterpret_cast<uint4 *>(Abuf + (nbmax + b) * kACore + e) = make_uint4(mw[0], mw[1], mw[2], mw[3]);
                    *reinterpret_cast<uint4 *>(Abuf + (2u * nbmax + b) * kACore + e) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
                }
            }
        have0 = kb0;
        have1 = kb1;
        // make generic-proxy shared stores visible to the tensor cores
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        // every thread sees the centroids (and norms) arrive; the vote keeps the outcome uniform
        ok = __syncthreads_and(mbar_wait(smem_u32(bbar), (s - s_begin) & 1u)) != 0;
        if (!ok) break;
        if (t == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            uint32_t acc = 0;
            for (uint32_t b = 0; b < nb; ++b) {
                const uint64_t ah = smem_desc(smem_u32(Abuf + b * kACore));
                const uint64_t bh = smem_desc(smem_u32(Bbuf + (3u * b) * kBCore));
                const uint64_t bm = smem_desc(smem_u32(Bbuf + (3u * b + 1u) * kBCore));
                const uint64_t bl = smem_desc(smem_u32(Bbuf + (3u * b + 2u) * kBCore));
                mma_bf16(tmem, ah, bh, acc); acc = 1;
                mma_bf16(tmem, ah, bm, 1);
                mma_bf16(tmem, ah, bl, 1);
                if (kAParts > 1) {
                    const uint64_t am = smem_desc(smem_u32(Abuf + (nbmax + b) * kACore));
                    const uint64_t al = smem_desc(smem_u32(Abuf + (2u * nbmax + b) * kACore));
                    mma_bf16(tmem, am, bh, 1);
                    mma_bf16(tmem, am, bm, 1);
                    mma_bf16(tmem, al, bh, 1);
                }
            }
            mma_commit(smem_u32(mbar));
        }
        // every thread waits with a bound
        ok = __syncthreads_and(mbar_wait(smem_u32(mbar), (s - s_begin) & 1u)) != 0;
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        if (!ok) break;
        if (t == 0 && s + 1u < s_end) fetch(s + 1u);     // the centroid operand is free
        // ---- epilogue: ||q_s||^2 + ||c||^2 - 2 q.c, clamped at 0
        float qn = 0.0f;
        for (uint32_t j = o; j < o + ds; ++j) {
            const float x = valid ? static_cast<float>(qp[j]) : 0.0f;
            qn = __fmaf_rn(x, x, qn);
        }
        const uint32_t esz = a.out_bf16 ? 2u : 4u;
        unsigned char *mine = wstage + lane * kRowPad;
        const uint32_t rows = a.nq - q0 > warp * 32u ? a.nq - q0 - warp * 32u : 0u;    // this warp's valid rows
        for (uint32_t c0 = 0; c0 < kN; c0 += 32) {
            float v[32];
            tmem_ld32(tmem + ((warp * 32u) << 16) + c0, v);
#pragma unroll
            for (int i = 0; i < 32; i += 4) {
                const float4 n4 = *reinterpret_cast<const float4 *>(cn + c0 + i);
                const float nn[4] = {n4.x, n4.y, n4.z, n4.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float x = __fadd_rn(__fadd_rn(qn, nn[e]), -2.0f * v[i + e]);
                    v[i + e] = x > 0.0f ? x : 0.0f;
                }
            }
            // 512 bytes of every row (128 FP32 or 256 BF16 entries) are staged, then stored
            if (a.out_bf16) {
                uint4 *st = reinterpret_cast<uint4 *>(mine + c0 * 2u);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    uint32_t w[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        w[e] = static_cast<uint32_t>(__bfloat16_as_ushort(__float2bfloat16_rn(v[8 * i + 2 * e]))) |
                               (static_cast<uint32_t>(__bfloat16_as_ushort(__float2bfloat16_rn(v[8 * i + 2 * e + 1]))) << 16);
                    st[i] = make_uint4(w[0], w[1], w[2], w[3]);
                }
            } else {
                float4 *st = reinterpret_cast<float4 *>(mine + (c0 & 127u) * 4u);
#pragma unroll
                for (int i = 0; i < 8; ++i) st[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            }
            const uint32_t done = (c0 + 32u) * esz;          // bytes of the row so far
            if ((done & 511u) == 0u) {
                __syncwarp();
                unsigned char *dst = static_cast<unsigned char *>(a.out) +
                                     (static_cast<uint64_t>(q0 + warp * 32u) * a.M + s) * kN * esz + (done - 512u) + lane * 16u;
                const uint64_t step = static_cast<uint64_t>(a.M) * kN * esz;
                const unsigned char *src = wstage + lane * 16u;
#pragma unroll 8
                for (uint32_t r = 0; r < 32u; ++r)
                    if (r < rows) *reinterpret_cast<uint4 *>(dst + r * step) = *reinterpret_cast<const uint4 *>(src + r * kRowPad);
                __syncwarp();
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        __syncthreads();                               // TMEM and B buffer free for the next subspace
    }
    if (!ok && t == 0) {
        atomicExch(a.err, 1u);
        mbar_wait(smem_u32(bbar), 0u);                  // copies in flight land before the block ends
        mbar_wait(smem_u32(bbar), 1u);
    }
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kN) : "memory");
    }
}

}  // namespace

namespace {
uint32_t smem_for(uint32_t nbmax, int dtype)
{
    return (dtype == 2 ? 3u : 1u) * nbmax * kACore + 3u * nbmax * kBCore + 2u * kN * 4u + kTile * kRowPad + 32u;
}
}  // namespace

uint32_t tc_table_smem_bytes(uint32_t d, int dtype)
{
    (void)d;
    return smem_for(kMaxKbPerSub, dtype);
}

cudaError_t launch_tc_tables(const TcTableArgs &args, int dtype, cudaStream_t st)
{
    TcTableArgs a = args;
    a.nbmax = 1;                     // the first d mod M subspaces are one dimension wider
    for (uint32_t s = 0, o = 0; s < a.M; ++s) {
        const uint32_t ds = a.d / a.M + (s < a.d % a.M ? 1u : 0u), nb = (o + ds - 1u) / 16u - o / 16u + 1u;
        if (nb > a.nbmax) a.nbmax = nb;
        o += ds;
    }
    if (a.nbmax > kMaxKbPerSub) return cudaErrorInvalidValue;        // refused at load time
    const uint32_t smem = smem_for(a.nbmax, dtype);
    const dim3 grid((a.nq + kTile - 1) / kTile, (a.M + kSubPerCta - 1) / kSubPerCta);
    cudaError_t e;
    // the limit belongs to the kernel, not to this call: every thread sets the
    // same one, or one thread's layout would refuse another's launch
#define BANG_TC_LAUNCH(DT)                                                                          \
    e = cudaFuncSetAttribute(adc_table_tc_kernel<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024); \
    if (e != cudaSuccess) return e;                                                                 \
    adc_table_tc_kernel<DT><<<grid, 128, smem, st>>>(a)
    if (dtype == 0) { BANG_TC_LAUNCH(0); }
    else if (dtype == 1) { BANG_TC_LAUNCH(1); }
    else { BANG_TC_LAUNCH(2); }
#undef BANG_TC_LAUNCH
    return cudaGetLastError();
}

}  // namespace bang
