// Team form of the search kernel (search_kernel.cuh states the method and the
// order of every sum; the results are the same bits): a CTA of 1 + E warps
// searches one query.
//
// The one-warp form is a serial chain: an expansion waits for the node's row,
// then for the new neighbours' code rows, and its distances, filter, choice
// and merge follow one another in the same warp, while the query's table
// (32 KB in FP32) lets only five such chains live on an SM.  What one
// expansion reads and computes, though, depends on its node alone: the row,
// the neighbours' distances and the node's exact distance are the same
// whenever they are asked for.  So here the first warp (the control warp)
// keeps only what is sequential (Bloom filter, choice of the next node, merge,
// top-k) and E expander warps work ahead of it: each takes one of the best
// unvisited worklist entries, reads its row, measures its neighbours and
// leaves ids and distances in a slot.  Nearly every such entry is expanded
// next or soon after, because an entry leaves the worklist only by being
// expanded or by falling off its end.  The order of the expansions, and with
// it every result, stays the control warp's.
//
// An expander skips the neighbours whose two filter bits are already set:
// bits are never cleared, so such a neighbour is still seen when its node's
// turn comes.  The control warp tests the others again against the filter as
// it stands then, which gives exactly the test of §4.3.
//
// What bounds it: the control warp's chain of dependent warp-wide steps
// (about 3,400 cycles per expansion against 4,200 of the one-warp form's whole
// iteration; the waits for rows and code rows, 40 % of it there, are gone).
// So where the entry after u* is ready too, both are expanded in one step (a
// quarter to a third of the steps); an expander takes about 3,000 cycles, hence
// three.  10,000 u8 queries, 1M points, L = 224, FP32 table, HBM: 7.02 -> 5.06 ms;
// 3,000 float queries, d = 96, M = 48, L = 128: 4.33 -> 2.57 ms; one query at
// L = 64: 156 -> 112 us.
//
// Slots are handed over through two mbarriers each (request, result); every
// wait is bounded.  A control warp whose wait gave up ends the query with
// status 3 and sets SearchArgs::gave_up.  Whichever side gave up, the two may
// then count a slot's phases differently, so the CTA starts its next query with
// new barriers.
#pragma once

#include "search_kernel.cuh"

namespace bang {

constexpr uint32_t kTeamMaxExpanders = 3;
constexpr long long kTeamWaitCycles = 6000000000ll;     // about 3 s

// Shared-memory carve-up of the team form, in bytes.
struct TeamLayout {
    uint32_t off_T, off_bloom, off_L, off_Nk, off_bits, off_Ck, off_slot, off_qw, off_head, off_bar, off_q,
        off_offs, off_lo, off_wid, slot_bytes, total;
    __host__ __device__ TeamLayout(uint32_t M, uint32_t log2z, uint32_t L, uint32_t k, uint32_t d, uint32_t R,
                                   int mode, uint32_t E)
    {
        const uint32_t tsz = mode == kModeF32 ? 4u : mode == kModeBF16 ? 2u : mode == kModeQ8 ? 1u : 0u;
        const uint32_t rw = R > 64u ? 128u : 64u;         // what the kernel's lanes cover
        uint32_t o = 0;
        off_T = o;      o += SmemLayout::up16(M * 256u * tsz);
        off_bloom = o;  o += SmemLayout::up16((1u << log2z) / 8u);
        off_L = o;      o += SmemLayout::up16(L * 8u);
        off_Nk = o;     o += 32u * 8u;                    // new keys, 32 at a time
        off_bits = o;   o += 128u;                        // output positions of a merge (L <= 1024)
        off_Ck = o;     o += SmemLayout::up16(k > (uint32_t)kRegK && mode != kModeExact ? k * 8u : 0u);
        slot_bytes = rw * (log2z <= 16u ? 12u : 16u);     // ids, distances, filter positions
        off_slot = o;   o += E * slot_bytes;
        off_qw = o;     o += mode == kModeExact ? 128u : 0u;   // the query's bytes (integer vectors, d <= 128)
        off_head = o;   o += SmemLayout::up16(E * 12u + 8u);   // node, count, exact distance; query ticket; a wait gave up
        off_bar = o;    o += SmemLayout::up16(E * 16u);
        // table-build scratch, dead before the first slot is used
        const uint32_t sq = SmemLayout::up16(mode != kModeExact ? d * 4u : 0u),
                       so = SmemLayout::up16(mode != kModeExact ? (M + 1u) * 4u : 0u),
                       sl = SmemLayout::up16(mode == kModeQ8 ? M * 4u : 0u);
        uint32_t b = E * slot_bytes >= sq + so + 2u * sl ? off_slot : o;
        const bool own = b != off_slot;
        off_q = b;      b += sq;
        off_offs = b;   b += so;
        off_lo = b;     b += sl;
        off_wid = b;    b += sl;
        total = own ? b : o;
    }
};

__device__ __forceinline__ uint32_t team_smem_addr(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void team_bar_init(uint32_t bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void team_bar_inval(uint32_t bar)
{
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];\n" ::"r"(bar) : "memory");
}
// New barriers, by all threads together.  Out of line, so that the search's
// loops are compiled as if it were not there.
static __device__ __noinline__ void team_start_over(uint32_t bar0, uint32_t count, volatile uint32_t *gave_up)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        for (uint32_t i = 0; i < count; ++i) {
            team_bar_inval(bar0 + 8u * i);
            team_bar_init(bar0 + 8u * i);
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        *gave_up = 0u;
    }
    __syncthreads();
}
__device__ __forceinline__ void team_arrive(uint32_t bar)
{
    asm volatile("{\n\t.reg .b64 t;\n\tmbarrier.arrive.release.cta.shared::cta.b64 t, [%0];\n\t}\n" ::"r"(bar)
                 : "memory");
}
__device__ __forceinline__ bool team_test(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred P;\n\t"
        "mbarrier.test_wait.parity.acquire.cta.shared::cta.b64 P, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, P;\n\t}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0u;
}
// One lane's wait; false when it gave up, after about `limit` cycles.
__device__ __forceinline__ bool team_wait_lane(uint32_t bar, uint32_t parity, long long limit)
{
    uint32_t ok = 0;
    long long began = 0;
    for (uint32_t i = 0;; ++i) {
        asm volatile(
            "{\n\t.reg .pred P;\n\t"
            "mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 P, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, P;\n\t}\n"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if (i == 0) began = clock64();
        else if (clock64() - began > limit) return false;
    }
}
// Whole warp: one answer for all lanes.
__device__ __forceinline__ bool team_wait(uint32_t bar, uint32_t parity, long long limit)
{
    return __all_sync(0xFFFFFFFFu, team_wait_lane(bar, parity, limit)) != 0;
}
// The same, and with `ask` whether another barrier's phase is over by then (bit
// 1 beside bit 0): each lane asks for itself while the other side may arrive at
// any moment, so that answer needs the vote as well.  One vote for both.
__device__ __forceinline__ uint32_t team_wait_ask(uint32_t bar, uint32_t parity, long long limit, bool ask,
                                                  uint32_t bar2, uint32_t parity2)
{
    uint32_t got = team_wait_lane(bar, parity, limit) ? 1u : 0u;
    if (ask && team_test(bar2, parity2)) got |= 2u;
    return __reduce_and_sync(0xFFFFFFFFu, got);
}

__device__ __forceinline__ bool team_seen(const volatile uint32_t *bloom, uint32_t p1, uint32_t p2)
{
    const uint32_t w1 = bloom[p1 >> 5], w2 = bloom[p2 >> 5];
    return ((w1 >> (p1 & 31u)) & (w2 >> (p2 & 31u)) & 1u) != 0u;
}

// The table of one query, subspaces shared out over the CTA's warps; the
// caller synchronises before (query, offsets) and after.  Entries are those
// of build_table.
template <int MODE>
__device__ __forceinline__ void team_build_table(const SearchArgs &a, const float *qv, const uint32_t *offs, void *T,
                                                 float *lo, float *wid, int lane, uint32_t warp, uint32_t nwarps)
{
    float v[8];
    if constexpr (MODE == kModeQ8) {
        for (uint32_t s = warp; s < a.M; s += nwarps) {
            subspace_entries(a, qv, offs, s, lane, v);
            uint32_t mn = __float_as_uint(v[0]), mx = mn;
#pragma unroll
            for (int t = 1; t < 8; ++t) {
                const uint32_t b = __float_as_uint(v[t]);
                mn = b < mn ? b : mn;
                mx = b > mx ? b : mx;
            }
            const float fmn = __uint_as_float(__reduce_min_sync(0xFFFFFFFFu, mn));
            const float fmx = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, mx));
            if (lane == 0) {
                lo[s] = fmn;
                wid[s] = __fsub_rn(fmx, fmn);
            }
        }
        __syncthreads();
        float g = 0.0f;
        for (uint32_t s = lane; s < a.M; s += kWarp) g = wid[s] > g ? wid[s] : g;
        g = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(g)));   // widths are >= +0
        const float inv = g > 0.0f ? __fdiv_rn(255.0f, g) : 0.0f;
        for (uint32_t s = warp; s < a.M; s += nwarps) {
            subspace_entries(a, qv, offs, s, lane, v);
            const float los = lo[s];
            uint8_t *Ts = static_cast<uint8_t *>(T) + s * 256u;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                uint32_t qv8 = 0;
                if (g > 0.0f) {
                    qv8 = __float2uint_rn(__fmul_rn(__fsub_rn(v[t], los), inv));
                    qv8 = qv8 < 255u ? qv8 : 255u;
                }
                Ts[lane + kWarp * t] = static_cast<uint8_t>(qv8);
            }
        }
    } else {
        for (uint32_t s = warp; s < a.M; s += nwarps) {
            subspace_entries(a, qv, offs, s, lane, v);
            unsigned char *Ts = static_cast<unsigned char *>(T) + s * 256u * (MODE == kModeBF16 ? 2u : 4u);
#pragma unroll
            for (int t = 0; t < 8; ++t) store_entry<MODE>(Ts, lane + kWarp * t, v[t]);
        }
    }
}

// Ordering bits of the distances of the m neighbours listed in ids, into db.
// One warp.  PQ: a lane per neighbour (2 or 4 lanes on the 8-bit table when
// few are left, exact in any order).  Exact: a lane per neighbour for integer
// rows of 16-byte multiples, else the warp per neighbour.
template <int DT, int RPL, int DCH, int MODE>
__device__ __forceinline__ void team_distances(const SearchArgs &a, const TableRef &tr, const uint32_t *qw,
                                               const VecShare<DT, DCH> &qs, const uint32_t *ids, uint32_t *db,
                                               uint32_t m, int lane)
{
    using E = typename Elem<DT>::T;
    if constexpr (MODE != kModeExact) {
        if (MODE == kModeQ8 && m <= 16u) {
            const uint32_t P = m <= 8u ? 4u : 2u;
            const uint32_t j = static_cast<uint32_t>(lane) / P, part = static_cast<uint32_t>(lane) % P;
            const uint8_t *T8 = static_cast<const uint8_t *>(tr.T);
            uint32_t s = 0;
            if (j < m) {
                const uint8_t *row = a.codes + static_cast<uint64_t>(ids[j]) * a.Mpad;
                s = P == 4u ? adc_q8_part<4>(T8, row, a.M, a.Mpad, part) : adc_q8_part<2>(T8, row, a.M, a.Mpad, part);
            }
            s += __shfl_xor_sync(0xFFFFFFFFu, s, 1);
            if (P == 4u) s += __shfl_xor_sync(0xFFFFFFFFu, s, 2);
            if (j < m && part == 0u) db[j] = s;
            return;
        }
#pragma unroll
        for (int t = 0; t < RPL; ++t) {
            const uint32_t j = lane + kWarp * t;
            if (j < m) db[j] = pq_dist_bits<MODE>(tr, a.codes + static_cast<uint64_t>(ids[j]) * a.Mpad, a.M, a.Mpad);
        }
    } else if (DT != 2 && DCH == 1 && (a.d & 15u) == 0 && a.vecb_ok) {
        const uint32_t nv = a.d / 16u;               // 16-byte chunks per row, <= 8
        const uint32_t bias = DT == 1 ? 0x80808080u : 0u;
        for (uint32_t j0 = 0; j0 < m; j0 += kWarp) {
            const uint32_t j = j0 + static_cast<uint32_t>(lane);
            const bool act = j < m;
            const uint4 *row = reinterpret_cast<const uint4 *>(static_cast<const E *>(a.base) +
                                                               static_cast<uint64_t>(act ? ids[j] : 0u) * a.vstride);
            uint4 xv[8];
#pragma unroll
            for (int c = 0; c < 8; ++c)
                xv[c] = (act && static_cast<uint32_t>(c) < nv) ? __ldg(row + c) : make_uint4(0u, 0u, 0u, 0u);
            uint32_t acc = 0;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                if (static_cast<uint32_t>(c) < nv) {
                    const uint4 q4 = reinterpret_cast<const uint4 *>(qw)[c];
                    const uint32_t xw[4] = {xv[c].x ^ bias, xv[c].y ^ bias, xv[c].z ^ bias, xv[c].w ^ bias};
                    const uint32_t w4[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint32_t df = __vabsdiffu4(w4[i], xw[i]);
                        acc = __dp4a(df, df, acc);
                    }
                }
            }
            if (act) db[j] = acc;
        }
    } else {
        for (uint32_t j0 = 0; j0 < m; j0 += 4) {
            VecShare<DT, DCH> xs[4];
#pragma unroll
            for (int t = 0; t < 4; ++t)
                if (j0 + t < m)
                    load_share<DT, DCH>(static_cast<const E *>(a.base) + static_cast<uint64_t>(ids[j0 + t]) * a.vstride,
                                        a.d, a.vecb_ok != 0, lane, xs[t]);
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                if (j0 + t < m) {
                    const uint32_t e = exact_distance_bits<DT, DCH>(qs, xs[t]);
                    if (lane == 0) db[j0 + t] = e;
                }
            }
        }
    }
}

// Registers per thread: five FP32 queries of four warps fill an SM's 65,536 at
// 96; the other tables take six to eight queries of three or four warps at 80
// (at 64 the spills cost 25-50 % on the 8-bit table).
constexpr int team_regs(int dch, int mode) { return dch > 1 ? 128 : mode == kModeF32 ? 96 : 80; }

template <int DT, int RPL, int DCH, int MODE>
__global__ void __maxnreg__(team_regs(DCH, MODE)) team_kernel(const SearchArgs a)
{
    using E = typename Elem<DT>::T;
    constexpr bool kPQ = MODE != kModeExact;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const uint32_t warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5, nexp = nwarps - 1u;
    const TeamLayout lay(a.M, a.log2z, a.L, a.k, a.d, a.R, MODE, nexp);
    void *T = smem + lay.off_T;
    uint32_t *bloom = reinterpret_cast<uint32_t *>(smem + lay.off_bloom);
    uint64_t *Lk = reinterpret_cast<uint64_t *>(smem + lay.off_L);
    uint64_t *Nk = reinterpret_cast<uint64_t *>(smem + lay.off_Nk);
    uint32_t *obits = reinterpret_cast<uint32_t *>(smem + lay.off_bits);
    uint64_t *Ck = reinterpret_cast<uint64_t *>(smem + lay.off_Ck);
    uint32_t *qw = reinterpret_cast<uint32_t *>(smem + lay.off_qw);
    volatile uint32_t *head = reinterpret_cast<volatile uint32_t *>(smem + lay.off_head);   // 3 words per slot
    volatile uint32_t *ticket = head + 3u * nexp, *gave_up = ticket + 1;
    const uint32_t bar0 = team_smem_addr(smem + lay.off_bar);   // slot e: request at +16e, result at +16e+8
    float *qv = reinterpret_cast<float *>(smem + lay.off_q);
    uint32_t *offs = reinterpret_cast<uint32_t *>(smem + lay.off_offs);
    float *lo8 = reinterpret_cast<float *>(smem + lay.off_lo);
    float *wid8 = reinterpret_cast<float *>(smem + lay.off_wid);

    const uint32_t d = a.d, kstride = a.k;
    constexpr uint32_t rw = kWarp * RPL;
    const uint32_t zmask = (1u << a.log2z) - 1u;
    const uint32_t nwords = (1u << a.log2z) / 32u;
    const bool z16 = a.log2z <= 16u;             // both filter positions fit one word

    if (threadIdx.x == 0) {
        for (uint32_t i = 0; i < 2u * nexp; ++i) team_bar_init(bar0 + 8u * i);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        *gave_up = 0u;
    }
    __syncthreads();

    uint32_t phase = 0;                  // expander: its request's parity; control: bit e, slot e's result parity
    uint32_t next_static = blockIdx.x;
    for (;;) {
        // ---- next query: from the work counter (persistent launch) or by grid stride
        uint32_t qi;
        if (a.queue) {
            if (threadIdx.x == 0) *ticket = atomicAdd(a.queue, 1u);
            __syncthreads();
            qi = *ticket;
            __syncthreads();             // read by all before the next one is written
        } else {
            qi = next_static;
            next_static += gridDim.x;
        }
        if (qi >= a.nq) break;
        const uint32_t q = a.order ? a.order[qi] : qi;
        const uint32_t k = a.k_per_q ? a.k_per_q[q] : a.k;
        const uint32_t L = a.L_per_q ? a.L_per_q[q] : a.L;
        const bool regk = k <= static_cast<uint32_t>(kRegK);
        if (k == 0 || k > a.k || L < k || L > a.L) {     // per-query arguments out of range
            for (uint32_t i = threadIdx.x; i < kstride; i += blockDim.x) {
                a.out_ids[static_cast<uint64_t>(q) * kstride + i] = kNone;
                a.out_dist[static_cast<uint64_t>(q) * kstride + i] = __uint_as_float(0x7F800000u);
            }
            if (threadIdx.x == 0) {
                if (a.out_iters) a.out_iters[q] = 0;
                if (a.out_status) a.out_status[q] = -1;
                if (a.out_ndist) a.out_ndist[q] = 0;
                if (a.cand_n) a.cand_n[q] = 0;
            }
            continue;
        }
        // ---- query, filter and table: the whole CTA
        const E *qp = static_cast<const E *>(a.queries) + static_cast<uint64_t>(q) * d;
        if (kPQ) {
            for (uint32_t j = threadIdx.x; j < d; j += blockDim.x) qv[j] = static_cast<float>(qp[j]);
            for (uint32_t i = threadIdx.x; i <= a.M; i += blockDim.x) offs[i] = a.off[i];
        }
        VecShare<DT, DCH> qs;
        load_share<DT, DCH>(qp, d, a.vec_ok != 0, lane, qs);
        if (!kPQ && DT != 2 && DCH == 1 && warp == 0) qw[lane] = qs.w[0];
        for (uint32_t w = threadIdx.x; w < nwords; w += blockDim.x) bloom[w] = 0u;
        __syncthreads();
        bool table_failed = false;
        if ((MODE == kModeBF16 || MODE == kModeF32) && a.tables) {   // precomputed on the tensor cores
            constexpr uint32_t esz = MODE == kModeBF16 ? 2u : 4u;
            table_failed = *a.tables_err != 0u;
            const uint4 *src = reinterpret_cast<const uint4 *>(static_cast<const unsigned char *>(a.tables) +
                                                               static_cast<uint64_t>(q) * a.M * 256u * esz);
            uint4 *dst = reinterpret_cast<uint4 *>(T);
            for (uint32_t i = threadIdx.x; i < a.M * 256u * esz / 16u; i += blockDim.x) dst[i] = src[i];
        } else if constexpr (kPQ) {
            team_build_table<MODE>(a, qv, offs, T, lo8, wid8, lane, warp, nwarps);
        }
        __syncthreads();
        const TableRef tr{T, qv, offs, a.codebook, 0u, a.M};

        if (warp != 0) {
            // ================= expander: one slot, one node at a time
            const uint32_t e = warp - 1u;
            uint32_t *ids = reinterpret_cast<uint32_t *>(smem + lay.off_slot + e * lay.slot_bytes);
            uint32_t *db = ids + rw;
            const uint32_t req = bar0 + 16u * e;
            for (;;) {
                if (!team_wait(req, phase, a.wait_cycles)) {
                    if (lane == 0) *gave_up = 1u;
                    break;
                }
                phase ^= 1u;
                const uint32_t u = head[3u * e];
                if (u == kNone) break;                   // the query is done
                NodeData<DT, RPL, DCH> nd;
                load_node<DT, RPL, DCH, kPQ, false>(a, u, lane, nd);
                unpack_ids<RPL>(a, lane, nd.nb);
                uint32_t m = 0;
#pragma unroll
                for (int r = 0; r < RPL; ++r) {
                    const uint32_t id = nd.nb[r];
                    const uint32_t p1 = fnv1a32_id(id) & zmask, p2 = fnv1a64_id_folded(id) & zmask;
                    const bool open = id != kNone && !team_seen(bloom, p1, p2);
                    const uint32_t bal = __ballot_sync(0xFFFFFFFFu, open);
                    if (open) {
                        const uint32_t j = m + __popc(bal & ((1u << lane) - 1u));
                        ids[j] = id;
                        db[rw + j] = z16 ? p1 | (p2 << 16) : p1;
                        if (!z16) db[2 * rw + j] = p2;
                    }
                    m += __popc(bal);
                }
                __syncwarp();
                team_distances<DT, RPL, DCH, MODE>(a, tr, qw, qs, ids, db, m, lane);
                uint32_t xd = 0;
                if (kPQ && !a.cand) xd = exact_distance_bits<DT, DCH>(qs, nd.x);
                if (lane == 0) {
                    head[3u * e + 1u] = m;
                    head[3u * e + 2u] = xd;
                }
                __syncwarp();
                if (lane == 0) team_arrive(req + 8u);
            }
        } else {
            // ================= control
            const uint32_t iter_cap = a.iter_cap ? a.iter_cap : 8u * L + 64u;
            const uint32_t lt = (1u << lane) - 1u;
            const uint32_t mybar = bar0 + 16u * static_cast<uint32_t>(lane);
            // lane e < nexp: the node in slot e (kNone: free) and its distance
            uint32_t sid = kNone, sdb = 0;
            auto post = [&](uint32_t e, uint64_t key) {
                if (static_cast<uint32_t>(lane) == e) {
                    sid = key_id(key);
                    sdb = static_cast<uint32_t>(key >> 32);
                    head[3u * e] = sid;
                    team_arrive(mybar);
                }
            };
            auto result = [&](uint32_t e) { return bar0 + 16u * e + 8u; };
            // start: worklist = {medoid}, medoid marked seen
            const uint32_t s0 = a.entry ? a.entry[q] : a.medoid;
            uint32_t dm_bits = 0;
            if (!kPQ) {
                VecShare<DT, DCH> xs;
                load_share<DT, DCH>(static_cast<const E *>(a.base) + static_cast<uint64_t>(s0) * a.vstride, d,
                                    a.vecb_ok != 0, lane, xs);
                dm_bits = exact_distance_bits<DT, DCH>(qs, xs);
            } else {
                dm_bits = pq_dist_bits<MODE>(tr, a.codes + static_cast<uint64_t>(s0) * a.Mpad, a.M, a.Mpad);
            }
            uint64_t ukey = make_key(dm_bits, s0);       // u*, the next node to expand
            if (lane == 0) {
                Lk[0] = ukey;
                const uint32_t p1 = fnv1a32_id(s0) & zmask, p2 = fnv1a64_id_folded(s0) & zmask;
                atomicOr(&bloom[p1 >> 5], 1u << (p1 & 31u));
                atomicOr(&bloom[p2 >> 5], 1u << (p2 & 31u));
            }
            __syncwarp();
            uint32_t nl = 1, nc = 0, iters = 0, ndist = 1, first = 0;    // first: u*'s index
            bool have_next = !table_failed;
            int32_t status = table_failed ? 2 : 0;
            uint64_t ck = ~0ull;             // register top-k (k <= kRegK): lane i holds rank i
            // the first unvisited entry after u* and the one after that (~0:
            // none; both3: the second is known), with their indexes plus one
            uint64_t lkey = ~0ull, lkey3 = ~0ull;
            uint32_t lpos = 0, lpos3 = 0;
            bool both3 = true;
            uint32_t *const cand = a.cand + static_cast<uint64_t>(q) * a.cand_cap;
            uint32_t *const trace = a.trace + static_cast<uint64_t>(q) * a.trace_cap;
            const uint32_t ncand = a.cand && !a.cand_list ? a.cand_cap : 0u, ntrace = a.trace ? a.trace_cap : 0u;
            auto rerank = [&](uint64_t ek) {     // the exact key of an expanded node into the top-k
                if (regk) {
                    const uint32_t pos = __popc(__ballot_sync(0xFFFFFFFFu, ck < ek));
                    if (pos < k) {
                        const uint64_t up = shfl_up_u64(ck, 1);
                        if (static_cast<uint32_t>(lane) == pos) ck = ek;
                        else if (static_cast<uint32_t>(lane) > pos) ck = up;
                    }
                    nc = nc + 1 < k ? nc + 1 : k;
                } else if (!(nc == k && ek >= Ck[k - 1])) {
                    uint32_t less = 0;
                    uint64_t keepk[kMaxK / kWarp];
#pragma unroll
                    for (int t = 0; t < kMaxK / kWarp; ++t) {
                        const uint32_t i = lane + kWarp * t;
                        keepk[t] = i < nc ? Ck[i] : 0ull;
                        less += (i < nc && keepk[t] < ek) ? 1u : 0u;
                    }
                    const uint32_t pos = __reduce_add_sync(0xFFFFFFFFu, less);
                    __syncwarp();
#pragma unroll
                    for (int t = 0; t < kMaxK / kWarp; ++t) {
                        const uint32_t i = lane + kWarp * t;
                        if (i < nc && i >= pos && i + 1 < k) Ck[i + 1] = keepk[t];
                    }
                    if (lane == 0) Ck[pos] = ek;
                    nc = nc + 1 < k ? nc + 1 : k;
                    __syncwarp();
                }
            };
            if (have_next && q + 1u != a.mute) post(0u, ukey);
            else if (lane == 0) sid = have_next ? key_id(ukey) : kNone;      // (tests: a request that gets lost)

            while (have_next) {
                if (iters >= iter_cap) {
                    status = 1;
                    break;
                }
                const uint32_t u = key_id(ukey), u2 = key_id(lkey);
                // (one bit at most: the leading-zero count is half of __ffs)
                const uint32_t se = 31u - __clz(__ballot_sync(0xFFFFFFFFu, sid == u));
                const uint32_t s2 = 31u - __clz(__ballot_sync(0xFFFFFFFFu, sid == u2));     // ~0: in no slot
                // Two expansions at once: the entry after u* is next after it
                // unless one of u*'s new neighbours is nearer.  When its slot
                // is ready too and both nodes' neighbours fit the warp, they
                // are filtered together, u*'s first.
                bool pair = lkey != ~0ull && s2 < nexp && both3 && iters + 1u < iter_cap;
                const uint32_t got = team_wait_ask(result(se), (phase >> se) & 1u, a.wait_cycles, pair, result(s2),
                                                   (phase >> (s2 & 31u)) & 1u);
                if (!(got & 1u)) {
                    status = 3;
                    break;
                }
                pair = (got & 2u) != 0u;
                const uint32_t m = head[3u * se + 1u], xd = head[3u * se + 2u];
                uint32_t m2 = 0, xd2 = 0;
                if (pair) {
                    m2 = head[3u * s2 + 1u];
                    xd2 = head[3u * s2 + 2u];
                    pair = m + m2 <= static_cast<uint32_t>(kWarp);
                }
                const uint32_t *ent = reinterpret_cast<const uint32_t *>(smem + lay.off_slot + se * lay.slot_bytes) + lane;
                if (pair && static_cast<uint32_t>(lane) >= m)
                    ent = reinterpret_cast<const uint32_t *>(smem + lay.off_slot + s2 * lay.slot_bytes) + (lane - m);
                const uint32_t mt = pair ? m + m2 : m;
                uint32_t id = ent[0], db = ent[rw], p1 = ent[2 * rw], p2 = z16 ? p1 >> 16 : ent[3 * rw];
                p1 &= zmask;
                // ---- filter seen neighbours, §4.3: test all, then insert all.
                // Bit t of fresh: entry lane + 32 t is new.
                uint32_t fresh = static_cast<uint32_t>(lane) < mt && !team_seen(bloom, p1, p2) ? 1u : 0u;
                const bool second = pair && static_cast<uint32_t>(lane) >= m;
                if (m > static_cast<uint32_t>(kWarp)) {
#pragma unroll 1
                    for (uint32_t t = 1; t * kWarp < m; ++t) {
                        const uint32_t x1 = ent[2 * rw + t * kWarp], x2 = z16 ? x1 >> 16 : ent[3 * rw + t * kWarp];
                        if (lane + t * kWarp < m && !team_seen(bloom, x1 & zmask, x2)) fresh |= 1u << t;
                    }
                    __syncwarp();
#pragma unroll 1
                    for (uint32_t t = 1; t * kWarp < m; ++t) {
                        const uint32_t x1 = ent[2 * rw + t * kWarp], x2 = z16 ? x1 >> 16 : ent[3 * rw + t * kWarp];
                        if ((fresh >> t) & 1u) {
                            atomicOr(&bloom[(x1 & zmask) >> 5], 1u << (x1 & zmask & 31u));
                            atomicOr(&bloom[x2 >> 5], 1u << (x2 & 31u));
                        }
                        ndist += __popc(__ballot_sync(0xFFFFFFFFu, (fresh >> t) & 1u));
                    }
                }
                __syncwarp();
                if ((fresh & 1u) && !second) {
                    atomicOr(&bloom[p1 >> 5], 1u << (p1 & 31u));
                    atomicOr(&bloom[p2 >> 5], 1u << (p2 & 31u));
                }
                const uint64_t last = nl == L ? Lk[L - 1] >> 1 : ~0ull;
                const uint64_t key0 = make_key(db, id);
                if (pair) {
                    __syncwarp();
                    if (__any_sync(0xFFFFFFFFu, fresh && !second && key0 < lkey)) {
                        pair = false;                    // a new neighbour of u* comes first
                        if (second) fresh = 0u;
                    } else if (second && fresh) {        // against the filter with u*'s neighbours in it
                        fresh = team_seen(bloom, p1, p2) ? 0u : 1u;
                    }
                    __syncwarp();
                    if (second && fresh) {
                        atomicOr(&bloom[p1 >> 5], 1u << (p1 & 31u));
                        atomicOr(&bloom[p2 >> 5], 1u << (p2 & 31u));
                    }
                }
                ndist += __popc(__ballot_sync(0xFFFFFFFFu, fresh & 1u));
                phase ^= 1u << se;
                if (static_cast<uint32_t>(lane) == se) sid = kNone;      // read: free again
                if (lane == 0) {
                    Lk[first] = ukey | 1ull;             // visited
                    if (iters < ncand) cand[iters] = u;
                    if (iters < ntrace) trace[iters] = u;
                    if (pair) {
                        Lk[lpos - 1u] = lkey | 1ull;
                        if (iters + 1u < ncand) cand[iters + 1u] = u2;
                        if (iters + 1u < ntrace) trace[iters + 1u] = u2;
                    }
                }
                const bool paired = pair;
                ++iters;
                if (pair) {
                    ++iters;
                    phase ^= 1u << s2;
                    if (static_cast<uint32_t>(lane) == s2) sid = kNone;
                    lkey = lkey3;
                    lpos = lpos3;
                }
                // ---- merge, §4.6-§4.7: as in the one-warp form (output
                // position = own index + rank in the other list), 32 new keys
                // at a time.  New keys behind the last entry of a full worklist
                // would land at L or later and are dropped.
                uint64_t best = lkey;
                uint32_t npos = 0;               // position of `best`, plus one
#pragma unroll 1
                for (uint32_t t = 0;;) {
                    const uint64_t key = t == 0 ? key0 : make_key(ent[rw + t * kWarp], ent[t * kWarp]);
                    const bool keep = ((fresh >> t) & 1u) && (key >> 1) < last;
                    const uint32_t bal = __ballot_sync(0xFFFFFFFFu, keep);
                    const uint32_t nm = __popc(bal);
                    ++t;
                    const bool done = t * kWarp >= m;
                    if (nm > 0) {
                        const uint64_t kb = warp_min_key(keep ? key : ~0ull);
                        best = kb < best ? kb : best;
                    }
                    // next node, §4.5: the best new neighbour or the first
                    // unvisited worklist entry; handed out at once when no
                    // expander has it (the slot just read is free)
                    if (done && best != ~0ull && !__any_sync(0xFFFFFFFFu, sid == key_id(best))) post(se, best);
                    npos = lpos;                 // in the untouched prefix, if not met below
                    if (nm > 0) {
                        if (keep) Nk[__popc(bal & lt)] = key;
                        obits[lane] = 0u;
                        __syncwarp();
                        const uint32_t nl2 = nl + nm < L ? nl + nm : L;
                        const uint32_t nw = (nl2 + 31u) >> 5;
                        uint64_t x = 0;
                        uint32_t xpos = 0xFFFFFFFFu, lo = 0xFFFFFFFFu, met = 0;
                        if (static_cast<uint32_t>(lane) < nm) {
                            x = Nk[lane];
                            lo = 0;              // #{worklist keys < x}
                            for (uint32_t b = 1u << ((31 - __clz(nl)) & ~1); b != 0u; b >>= 2) {   // powers of 4
                                const uint32_t c1 = lo + b, c2 = c1 + b, c3 = c2 + b;
                                const uint32_t mm = static_cast<uint32_t>(c1 <= nl && Lk[c1 - 1u] < x) +
                                                    static_cast<uint32_t>(c2 <= nl && Lk[c2 - 1u] < x) +
                                                    static_cast<uint32_t>(c3 <= nl && Lk[c3 - 1u] < x);
                                lo += b * mm;
                            }
                            xpos = lo;
                            for (uint32_t tt = 0; tt < nm; tt += 4) {            // Nk is 32 keys long
                                const uint64_t k0 = Nk[tt], k1 = Nk[tt + 1], k2 = Nk[tt + 2], k3 = Nk[tt + 3];
                                xpos += (k0 < x) + (tt + 1 < nm && k1 < x) + (tt + 2 < nm && k2 < x) +
                                        (tt + 3 < nm && k3 < x);
                            }
                        }
                        const uint32_t rmin = __reduce_min_sync(0xFFFFFFFFu, lo);
                        if (xpos < L) atomicOr(&obits[xpos >> 5], 1u << (xpos & 31u));
                        __syncwarp();
                        // new keys at or below the chunk in hand: all of them,
                        // less those of the chunks already done, from the end
                        uint32_t upto = __popc(__ballot_sync(0xFFFFFFFFu, xpos < L));
                        const int32_t cmin = static_cast<int32_t>(rmin >> 5);
                        constexpr int kG = 4;    // chunks read before they are written
#pragma unroll 1
                        for (int32_t ctop = static_cast<int32_t>(nw) - 1; ctop >= cmin; ctop -= kG) {
                            uint64_t mv[kG];
                            uint32_t dst[kG];
#pragma unroll
                            for (int g = 0; g < kG; ++g) {
                                const int32_t c = ctop - g;
                                mv[g] = 0;
                                dst[g] = 0xFFFFFFFFu;
                                if (c >= cmin) {
                                    const uint32_t w = obits[c];
                                    upto -= __popc(w);
                                    const uint32_t below = upto + __popc(w & lt);
                                    const uint32_t p = static_cast<uint32_t>(c) * 32u + lane;
                                    if (p < nl2 && p >= rmin && !((w >> lane) & 1u)) {
                                        mv[g] = Lk[p - below];
                                        dst[g] = p;
                                        if (mv[g] == best) met = p + 1;
                                    }
                                }
                            }
                            __syncwarp();
#pragma unroll
                            for (int g = 0; g < kG; ++g)
                                if (dst[g] != 0xFFFFFFFFu) Lk[dst[g]] = mv[g];
                            __syncwarp();
                        }
                        if (xpos < L) {
                            Lk[xpos] = x;
                            if (x == best) met = xpos + 1;
                        }
                        __syncwarp();
                        nl = nl2;
                        met = __reduce_max_sync(0xFFFFFFFFu, met);
                        if (met) npos = met;
                    }
                    if (done) break;
                }
                have_next = best != ~0ull;
                if (have_next && m > static_cast<uint32_t>(kWarp)) {     // several merges: look it up
                    for (uint32_t b0 = 0; b0 < nl; b0 += kWarp) {
                        const uint32_t at = __ballot_sync(0xFFFFFFFFu, b0 + lane < nl && Lk[b0 + lane] == best);
                        if (at) {
                            npos = b0 + static_cast<uint32_t>(__ffs(at));
                            break;
                        }
                    }
                }
                first = npos - 1;
                ukey = best;
                __syncwarp();
                // ---- the unvisited entries after the new u*; free slots go to
                // the nearest that no slot holds, after finished slots whose
                // nodes are no longer among the nearest are taken back
                lkey = lkey3 = ~0ull;
                lpos = lpos3 = 0;
                both3 = true;
                if (have_next) {
                    uint64_t key = first + lane < nl ? Lk[first + lane] : ~0ull;
                    uint32_t un = __ballot_sync(0xFFFFFFFFu, (key & 1ull) == 0ull) & ~1u;
                    if (un) {
                        uint32_t i = static_cast<uint32_t>(__ffs(un)) - 1u;
                        lkey = shfl_u64(key, static_cast<int>(i));
                        lpos = first + i + 1u;
                        uint32_t rest = un & (un - 1u);
                        if (rest) {
                            i = static_cast<uint32_t>(__ffs(rest)) - 1u;
                            lkey3 = shfl_u64(key, static_cast<int>(i));
                            lpos3 = first + i + 1u;
                        } else {
                            both3 = first + kWarp >= nl;
                        }
                        if (nexp > 1u) {
                            uint32_t want = un;          // the nearest nexp - 1
                            uint32_t beyond = rest;
                            for (uint32_t c = 2; c < nexp; ++c) beyond &= beyond - 1u;
                            want ^= beyond;
                            bool held = false;
                            for (uint32_t e = 0; e < nexp; ++e)
                                held |= __shfl_sync(0xFFFFFFFFu, sid, static_cast<int>(e)) == key_id(key);
                            want &= ~__ballot_sync(0xFFFFFFFFu, held);
                            if (want) {
                                // beyond the nearest nexp - 1, or off a full worklist
                                const uint32_t far = beyond ? __shfl_sync(0xFFFFFFFFu, static_cast<uint32_t>(key >> 32),
                                                                          __ffs(beyond) - 1)
                                                            : nl == L ? static_cast<uint32_t>(Lk[L - 1] >> 32) : 0xFFFFFFFFu;
                                bool idle = sid == kNone;
                                if (!idle && sdb >= far && sid != key_id(best) && (beyond || sdb > far))
                                    idle = team_test(mybar + 8u, (phase >> lane) & 1u);
                                idle = idle && static_cast<uint32_t>(lane) < nexp;
                                phase ^= __ballot_sync(0xFFFFFFFFu, idle && sid != kNone);
                                if (idle) sid = kNone;
                                uint32_t freeb = __ballot_sync(0xFFFFFFFFu, idle);
#pragma unroll 1
                                while (freeb && want) {
                                    post(static_cast<uint32_t>(__ffs(freeb)) - 1u, shfl_u64(key, __ffs(want) - 1));
                                    freeb &= freeb - 1u;
                                    want &= want - 1u;
                                }
                            }
                        }
                    } else {
                        both3 = false;
                        for (uint32_t b0 = first + kWarp; b0 < nl; b0 += kWarp) {
                            key = b0 + lane < nl ? Lk[b0 + lane] : ~0ull;
                            un = __ballot_sync(0xFFFFFFFFu, (key & 1ull) == 0ull);
                            if (un) {
                                const uint32_t i = static_cast<uint32_t>(__ffs(un)) - 1u;
                                lkey = shfl_u64(key, static_cast<int>(i));
                                lpos = b0 + i + 1u;
                                break;
                            }
                        }
                    }
                }
                // ---- re-rank candidates: exact distances of the nodes just expanded (§4.8)
                if (kPQ && !a.cand) {
                    rerank(make_key(xd, u));
                    if (paired) rerank(make_key(xd2, u2));
                }
                __syncwarp();
            }

            // ---- end of the query: the expanders finish and stop
            for (uint32_t e = 0; e < nexp; ++e) {
                if (__shfl_sync(0xFFFFFFFFu, sid, static_cast<int>(e)) != kNone) {
                    if (!team_wait(result(e), (phase >> e) & 1u, a.wait_cycles)) status = 3;
                    phase ^= 1u << e;
                }
                if (static_cast<uint32_t>(lane) == e) {
                    head[3u * e] = kNone;
                    team_arrive(mybar);
                }
            }
            // ---- output (see search_kernel)
            const uint64_t o0 = static_cast<uint64_t>(q) * kstride;
            if (kPQ && a.cand) {
                if (a.cand_list) {
                    for (uint32_t i = lane; i < nl; i += kWarp)
                        a.cand[static_cast<uint64_t>(q) * a.cand_cap + i] = key_id(Lk[i]);
                    if (lane == 0) a.cand_n[q] = nl;
                } else if (lane == 0) {
                    a.cand_n[q] = iters < a.cand_cap ? iters : a.cand_cap;
                }
            } else {
                const uint32_t have = kPQ ? nc : (nl < k ? nl : k);
                for (uint32_t i = lane; i < kstride; i += kWarp) {
                    uint32_t oid = kNone;
                    float od = __uint_as_float(0x7F800000u);
                    if (i < have) {              // regk: have <= 32, rank i is lane i's register
                        const uint64_t key = !kPQ ? Lk[i] : regk ? ck : Ck[i];
                        const uint32_t bits = static_cast<uint32_t>(key >> 32);
                        oid = key_id(key);
                        od = DT == 2 ? __uint_as_float(bits) : static_cast<float>(bits);
                    }
                    a.out_ids[o0 + i] = oid;
                    a.out_dist[o0 + i] = od;
                }
            }
            if (lane == 0) {
                if (a.out_iters) a.out_iters[q] = iters;
                if (a.out_status) a.out_status[q] = status;
                if (a.out_ndist) a.out_ndist[q] = ndist;
                if (status == 3) {
                    *gave_up = 1u;
                    if (a.gave_up) *reinterpret_cast<volatile uint32_t *>(a.gave_up) = 1u;
                }
            }
        }
        __syncthreads();                 // every warp is done with the query's shared memory
        if (*gave_up) {                  // the same for all: nobody waits on a barrier now
            team_start_over(bar0, 2u * nexp, gave_up);
            phase = 0;
        }
    }
}

// ---- Which form: expanders per query, 0 for one warp.
//
// A team answers a query sooner (1.1 to 2.1 times, measured) and takes three or
// four times the warps.  What counts is how many queries an SM holds at once in
// either form, by shared memory and registers, and how often it has to be
// filled for all of them (waves).  Where the team costs no resident query it is
// the faster form nearly everywhere; where it costs some, its gain has to make
// up for the waves it adds.  Where it does is read off 4,900 measured points:
// ten shapes (uint8, int8, FP32; d = 96 to 200, M = 30 to 74, 32 to 68
// neighbours), all modes, filters of 2^14 to 2^17 bits, L = 32 to 256, 1 to
// 10,000 queries, graph and vectors in HBM or host memory, plain and batched,
// indexes inside the L2 cache (60,000 and 100,000 points) and beyond it
// (700,000).  29 points are more than 2 % slower than one warp, by 11 % at most
// (by shared memory alone, as it was before: 326, by up to 45 %).  For example,
// us per call with one warp / two / three expanders, [chosen]; queries that an
// SM holds in brackets:
//   u8 d = 128, M = 32  FP32  L = 150     1 query   (5 5 5)   296 /   241 / [200]
//   the same                          1,200 queries (5 5 5)   652 /   556 / [481]
//   the same, 8-bit, 2^17             1,200         (8 7 6)  [405]/   596 /  609
//   int8 M = 50, 8-bit, 2^16          1,400         (9 8 6)   800 /  [617]/  566
//   u8 d = 130, exact                 1,200        (20 5 4) [1,028]/ 1,542 / 1,279
//   FP32 d = 128, exact, host, L = 64   600        (21 8 6) [5,652]/ 5,620 / 5,815
// (u8 and int8 rows of 16-byte multiples, exact: measured again with the
// registers that search_kernel has now, 60,000 and 300,000 points.)
// At most three expanders: a fourth changed nothing, the control warp is then
// the slower side.

// Queries that share an SM: with `bytes` of shared memory each, and teams of E
// expanders with `regs` registers a thread (16,384 in each quarter of the SM).
inline uint32_t fit_smem(uint32_t bytes)
{
    return bytes > 227u * 1024u ? 0u : 228u * 1024u / (((bytes + 127u) & ~127u) + 1024u);
}
inline uint32_t team_fit(const SearchArgs &a, int mode, uint32_t E)
{
    const uint32_t regs = static_cast<uint32_t>(team_regs(a.d > 128u ? 4 : 1, mode));
    const uint32_t s = fit_smem(TeamLayout(a.M, a.log2z, a.L, a.k, a.d, a.R, mode, E).total);
    const uint32_t r = 16384u / (32u * regs) * 4u / (1u + E);
    return s < r ? s : r;
}

// f1, f2, f3: the queries an SM holds with one warp, two and three expanders.
inline uint32_t team_choice(const SearchArgs &a, int dtype, int mode, uint32_t sms, uint32_t f1, uint32_t f2,
                            uint32_t f3)
{
    if (a.overlapped) {
        // launches that fill the SMs together, all in the same form: 24
        // requests, BF16 table, L up to 256 (8 7 6): two expanders 1.02 times
        // as fast as one warp, three 1.06; the form chosen launch by launch,
        // so that both kinds share the SMs, 0.92.  A few small requests, where
        // most SMs have one query, gain up to twofold.
        return fit_smem(TeamLayout(a.M, a.log2z, a.L, a.k, a.d, a.R, mode, 2).total) > 7u ? 0u : 3u;
    }
    const uint32_t share = (a.nq + sms - 1u) / sms, need = share < f1 ? share : f1;
    const auto waves = [&](uint32_t f) { return f ? (a.nq + sms * f - 1u) / (sms * f) : ~0u; };
    const uint32_t w1 = waves(f1), w2 = waves(f2), w3 = waves(f3);
    const bool flt = dtype == 2, wide = a.d > 128u, wide_r = a.R > 64u;
    const bool lanes = !flt && !wide && a.d % 16u == 0u && a.vecb_ok;    // exact: a lane per row
    // beyond the L2 cache a hop takes longer, and the team hides it
    const bool far = static_cast<uint64_t>(a.n) * (4ull * a.R + a.Mpad + a.d * (flt ? 4ull : 1ull)) > (96ull << 20);
    if (mode == kModeExact) {
        if (a.base_link && share > 1u) {
            // every neighbour measured is a row over the host link, which
            // expansions in vain and neighbours measured twice load
            if (flt) return f3 >= need && share <= 2u && a.L >= 64u ? 3u : 0u;
            if (lanes) {
                if (share <= 2u) return a.L >= 96u && f3 >= need ? 3u : a.L >= 48u && f2 >= need ? 2u : 0u;
                // rows that fill a 128-byte line: 5 to 10 % better than one
                // warp's whole-row loads where the search is long
                if (a.d > 112u && !wide_r && a.L >= 96u) return 2u;
                return share <= 4u && a.L >= 160u && f2 >= need ? 2u : 0u;
            }
        }
        if (wide && !a.vecb_ok) return f3 >= need && share <= 4u ? 3u : 0u;   // rows read byte by byte
        if (f3 >= need) return 3u;
        if (f2 >= need) return 2u;
        if (a.base_link) return 0u;
        if (wide) return flt && share <= (a.L >= 128u ? 8u : 6u) ? 3u : 0u;
        return share <= 9u && (flt || (far && !lanes)) ? 3u : 0u;
    }
    // short code rows in the 8-bit table, several waves: one warp has the fewest instructions
    if (mode == kModeQ8 && a.Mpad <= 32u && a.R > 32u && f1 >= 7u && w1 >= 4u) return 0u;
    if (f3 >= need) return 3u;
    const uint32_t e = f3 == f2 || (w3 == w2 && !flt && (wide || (mode == kModeF32 && w2 <= 2u))) ? 3u : 2u;
    if (f2 >= need) return e;
    // from here on a team costs resident queries
    if (mode == kModeF32) {
        if (w1 > 1u) return e;
        return !wide && a.Mpad <= 32u && !flt && a.vecb_ok && !wide_r ? 0u : 3u;
    }
    if (w1 == 1u) {              // one warp per query holds them all at once
        if (wide) return flt ? (w2 == 2u ? 2u : 0u) : w3 == 2u && !a.queue ? 3u : 0u;
        if (f1 <= 7u) return a.Mpad > 32u ? e : 0u;
        return far && !lanes && !flt && f1 <= 12u ? 2u : 0u;
    }
    if (f1 <= 6u) return e;
    if (wide) return wide_r && f1 > 7u && !flt ? (w1 == 2u && w2 <= 3u ? e : 0u) : f1 <= 9u ? e : 0u;
    if (f1 == 7u) return !wide_r || w1 <= (far ? 4u : 3u) ? e : 0u;
    if (f1 > 10u) return 0u;
    if (wide_r) return w1 == 2u && w2 <= (far ? 3u : 2u) ? 2u : 0u;
    if (w2 <= w1) return 2u;
    return a.Mpad >= 64u && f1 <= 9u && ((w1 <= 3u && (far || a.Mpad >= 80u)) || (far && !lanes)) ? 2u : 0u;
}

// bytes1: the one-warp form's shared memory per query.
inline uint32_t team_expanders(const SearchArgs &a, int dtype, int mode, uint32_t sms, uint32_t bytes1)
{
    const uint32_t f1 = fit_smem(bytes1), f2 = team_fit(a, mode, 2), f3 = team_fit(a, mode, 3);
    if (f1 == 0u || f2 == 0u) return 0u;
    const uint32_t e = team_choice(a, dtype, mode, sms, f1 < 32u ? f1 : 32u, f2, f3);
    return e == 3u && f3 == 0u ? 2u : e;          // three slots may not fit where two do
}

template <int DT, int RPL, int DCH, int MODE>
cudaError_t launch_team_one(const SearchArgs &a, uint32_t nexp, int sms, cudaStream_t st)
{
    const auto kern = team_kernel<DT, RPL, DCH, MODE>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e != cudaSuccess) return e;
    static std::atomic<uint32_t> carveout_set{0};      // the hint stays with the function (see launch_one)
    if (carveout_set.load() != a.carveout) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 a.carveout ? static_cast<int>(a.carveout) : -1);
        if (e != cudaSuccess) return e;
        carveout_set.store(a.carveout);
    }
    const size_t smem = TeamLayout(a.M, a.log2z, a.L, a.k, a.d, a.R, MODE, nexp).total;
    const int threads = static_cast<int>(kWarp * (1u + nexp));
    uint32_t grid = a.nq;
    if (a.queue) {                     // persistent: a multiple of the resident CTAs
        int per_sm = 0;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem)) != cudaSuccess) return e;
        const uint64_t want = static_cast<uint64_t>(sms) * (per_sm > 0 ? per_sm : 1) *
                              (a.grid_mult ? a.grid_mult : 1u);
        grid = static_cast<uint32_t>(want < a.nq ? want : a.nq);
    }
    kern<<<grid, threads, smem, st>>>(a);
    return cudaGetLastError();
}

// Launch of one mode.  The one-warp form (search_kernel.cuh) stays where it is
// faster (above) and for what the team form does not do: the per-phase clock
// and the neighbour-code layout.
template <int MODE> cudaError_t launch_team(const SearchArgs &args, int dtype, size_t smem, cudaStream_t st)
{
    SearchArgs a = args;
    if (a.wait_cycles == 0) a.wait_cycles = kTeamWaitCycles;
    int dev = 0, sms = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const bool one = a.phase_cycles || a.ncodes;
    const uint32_t nexp = a.form ? a.form - 1u : one ? 0u : team_expanders(a, dtype, MODE, static_cast<uint32_t>(sms), static_cast<uint32_t>(smem));
    if (a.form > 1u && (one || nexp > kTeamMaxExpanders ||
                        TeamLayout(a.M, a.log2z, a.L, a.k, a.d, a.R, MODE, nexp).total > 227u * 1024u))
        return cudaErrorInvalidValue;            // asked for by name, but not possible here
    if (a.form_out) *a.form_out = 1u + nexp;
    if (nexp == 0) return launch_mode<MODE>(a, dtype, smem, st);
    const bool narrow = a.d <= 128, wide_r = a.R > 64;
#define BANG_DISPATCH(DT)                                                                                    \
    return wide_r ? (narrow ? launch_team_one<DT, 4, 1, MODE>(a, nexp, sms, st)                              \
                            : launch_team_one<DT, 4, 4, MODE>(a, nexp, sms, st))                             \
                  : (narrow ? launch_team_one<DT, 2, 1, MODE>(a, nexp, sms, st)                              \
                            : launch_team_one<DT, 2, 4, MODE>(a, nexp, sms, st))
    if (dtype == 0) { BANG_DISPATCH(0); }
    if (dtype == 1) { BANG_DISPATCH(1); }
    BANG_DISPATCH(2);
#undef BANG_DISPATCH
}

}  // namespace bang
