// GEMM for more than 128 activation rows (batched verify passes, prefill): the launch is bound by the tensor cores and
// by how fast operands reach them, not by the weight stream.
//
//   D[f][r] = sum_k W[f][k] * (X_hi[r][k] + X_lo[r][k])
//
// A pair of CTAs (cluster of two, cta_group::2) owns a tile of 256 weight rows x NP <= 256 activation rows: each CTA
// loads its 128 weight rows and half of the activation rows, one tcgen05.mma works on both CTAs' shared memory, and CTA
// `c` holds features 128 c .. 128 c + 127 of the tile in its tensor memory (lane = feature, column = row).  The second
// terms of two-term activations are a second B operand added into the same accumulator.
//
// Why this tile: per 64-wide k-step an SM fetches 16 KB of weights and NP/2 x 128 B (twice with two terms) of activations
// from L2 for NP x 4 KFLOP of its tensor cores' work; at NP = 256 that is 48 B (two-term) or 64 B (one-term) a clock,
// where the 128 x 128-row tile of gemm_tc_kernel asks for 94 and 128 -- more than the L2 delivers.
//
// Persistent: P <= 74 pairs.  Whole rounds of P items (item = weight tile x row tile, row tiles fastest so that concurrent
// pairs share weight tiles) are dealt out one per pair; the items left over -- all of them, where there are fewer than P --
// are cut into equal ranges of k-steps (unless they nearly fill a round: wide_shape()), on average at most eight to an item (nine can touch one).  A pair that holds part of an item stores its fp32 partial tile and counts in; the pair that
// comes last adds the parts in k order (bit-reproducible) and runs the epilogue.  Nobody waits for another pair.  The cut
// items come first, so that this exchange (20-25 us where nothing follows) hides under the whole ones.  Where there is a whole
// round nothing beyond the rest is cut: pairs at different depths of K share no operands in L2 (the down projection of 1536
// rows with all its 84 items cut read 2.4 GB from HBM, 380 us instead of 288).  A launch of fewer than P items works that way
// throughout; use_wide() says from how many k-steps a pair on it is still the faster one.  Two accumulators in tensor memory: the epilogue of one item runs
// under the main loop of the next.
//
// Warp roles: warp 0 = TMA producer, warp 1 = tensor memory + MMA issuer (first CTA of the pair), warps 2..9 = epilogue.
// Every mbarrier wait is bounded.  One that gives up records GLANCE_E_TIMEOUT and tells the other CTA of the pair: from the
// item that it concerns on neither stores results, a cut item with a given-up part is finished by nobody (its counter still
// returns to zero), and before the pair leaves it waits for the copies and MMAs that it has in flight.
#include <cuda.h>

#include <algorithm>

#include "gemm_epilogue.cuh"

namespace glance {

namespace {

using namespace tc;

constexpr int NEPI = 8;                      // epilogue warps: two per tensor memory lane quarter, 16-column chunks in turn
constexpr int NTHR = 64 + 32 * NEPI;
constexpr int CSTEP = NEPI / 4 * 16;         // columns that the warps of a lane quarter cover together
constexpr int PAIR = 2 * BM;                 // weight rows of a pair's tile
constexpr int MAX_STAGES = 8;
constexpr int FLIGHT = 4;                    // parts of a cut item in flight (3: down at 512 rows 113.5 instead of 110 us)
constexpr size_t PLANE = (size_t)kWideRows * BM;   // floats of one CTA's partial tile
constexpr int GIVEN_UP = 1 << 16;            // added to a cut item's arrival counter by a part that has no result

struct alignas(8) WideBars {
    uint64_t full[MAX_STAGES], empty[MAX_STAGES];
    uint64_t acc_full[2], acc_empty[2];
    uint64_t drained;
    uint32_t tmem_base;
    int abort_flag;
    int issued;                              // k-steps that this CTA's producer has gone through
};

__device__ __forceinline__ void tma_load_pair(void *dst, const CUtensorMap *map, uint32_t bar_cluster, int c0, int c1, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;"
        ::"r"(smem_u32(dst)), "l"(map), "r"(bar_cluster), "r"(c0), "r"(c1), "l"(policy) : "memory");
}
// boxes of wide_make_map(): 16-row groups of gate and up rows / of the two halves of a head
__device__ __forceinline__ void tma_load_pair_4d(void *dst, const CUtensorMap *map, uint32_t bar_cluster, int c0, int c3, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %5, %5, %4}], [%2], %6;"
        ::"r"(smem_u32(dst)), "l"(map), "r"(bar_cluster), "r"(c0), "r"(c3), "r"(0), "l"(policy) : "memory");
}
__device__ __forceinline__ void tma_load_pair_5d(void *dst, const CUtensorMap *map, uint32_t bar_cluster, int c0, int c4, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %5, %5, %5, %4}], [%2], %6;"
        ::"r"(smem_u32(dst)), "l"(map), "r"(bar_cluster), "r"(c0), "r"(c4), "r"(0), "l"(policy) : "memory");
}
// bf16 x bf16 -> fp32, both operands K-major, M = 256 over the pair
__device__ __forceinline__ uint32_t idesc_pair(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(PAIR >> 4) << 24);
}
__device__ __forceinline__ void umma_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
}
// arrives on the barrier at this offset in both CTAs once every MMA issued so far has completed
__device__ __forceinline__ void umma_commit_pair(uint64_t *bar) {
    asm volatile(
        "{\n\t.reg .b16 m;\n\t"
        "mov.b16 m, 3;\n\t"
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], m;\n\t}"
        ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar_cluster) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster) : "memory");
}
__device__ __forceinline__ void epilogue_sync() { asm volatile("bar.sync 1, %0;" ::"n"(32 * NEPI) : "memory"); }
// the same barrier, and whether every epilogue thread says yes
__device__ __forceinline__ bool epilogue_all(bool yes) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "bar.red.and.pred q, 1, %2, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r) : "r"((uint32_t)yes), "n"(32 * NEPI) : "memory");
    return r != 0;
}
// Bounded wait; giving up (or finding that another role did) also stops the other CTA of the pair.
__device__ __forceinline__ bool pair_wait(WideBars &bars, uint64_t *bar, uint32_t parity, int32_t *status, uint64_t limit_ns) {
    if (mbar_wait(bar, parity, &bars.abort_flag, status, limit_ns)) return true;
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(map_to_rank(smem_u32(&bars.abort_flag), cluster_rank() ^ 1u)), "r"(1) : "memory");
    return false;
}
// takes bytes that no copy will deliver off a barrier's count
__device__ __forceinline__ void mbar_complete_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.complete_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bounded_wait(uint64_t *bar, uint32_t parity, uint64_t limit_ns) {
    const uint64_t t0 = global_ns();
    while (!mbar_try_wait(bar, parity))
        if (global_ns() - t0 > limit_ns) break;
}

// The work of one pair, in order: its range [u0, u1) of the cut items' k-steps, then `rounds` whole items.
struct Deal {
    int ks, P, C, pair, cut, rounds, items;  // k-steps per item; pairs; pairs that share the cut items; this pair; ...
    long long U, u0, u1;                     // units of the cut items; this pair's range
    __device__ Deal(const TcGemmArgs &a, int pair_) {
        ks = a.K / BK; P = a.wide_pairs; C = a.wide_cutters; pair = pair_; cut = a.wide_cut; rounds = a.wide_rounds; items = a.wide_items;
        U = (long long)cut * ks;
        u0 = pair < C ? start_of(pair) : 0;
        u1 = pair < C ? start_of(pair + 1) : 0;
    }
    __device__ long long start_of(int p) const { return p * U / C; }
    __device__ int holder_of(long long u) const { return (int)(((u + 1) * C - 1) / U); }
};
struct Segment {
    int item, k0, k1;
};
// i-th segment of the pair; false when there is none
__device__ __forceinline__ bool segment(const Deal &d, int i, Segment &s) {
    if (d.u1 > d.u0) {
        const int first = (int)(d.u0 / d.ks), n = (int)((d.u1 - 1) / d.ks) - first + 1;
        if (i < n) {
            s.item = first + i;
            s.k0 = i == 0 ? (int)(d.u0 - (long long)first * d.ks) : 0;
            s.k1 = (int)min((long long)d.ks, d.u1 - (long long)s.item * d.ks);
            return true;
        }
        i -= n;
    }
    s.item = d.cut + i * d.P + d.pair;
    if (i >= d.rounds || s.item >= d.items) return false;
    s.k0 = 0;
    s.k1 = d.ks;
    return true;
}

// Modes as in gemm_tc.cuh: 1 SwiGLU, 2 arg-max (+ logits, sampling, entropy), 3 residual, 4 rotary + K/V write.
// Modes 1 and 4 combine features half a block apart (gate and up; a rotary pair).  Their weight rows are fetched in
// groups of 16, partners next to each other, so that partners are in one warp's part of the tile; a tensor map with
// the groups as dimensions of their own brings them in this order with one copy (eight 16-row copies per k-step held the
// main loop of the QKV launch at 0.77 us per k-step, one copy at 0.55).
template <int MODE>
__global__ void __launch_bounds__(NTHR, 1) gemm_wide_kernel(const __grid_constant__ CUtensorMap map_w,
                                                           const __grid_constant__ CUtensorMap map_x, TcGemmArgs a) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ WideBars bars;
    __shared__ float row_scale[2][kWideRows];
    // per row: what the four lane quarters found (sum of squares / packed arg-max key)
    __shared__ float part_f[MODE == 3 ? 4 : 1][kWideRows];
    __shared__ unsigned long long part_k[MODE == 2 ? 4 : 1][kWideRows];
    // 16 rows x 32 features of an epilogue warp, transposed on the way from tensor memory: a lane then works on four
    // consecutive features of a row with 16-byte accesses (2-byte stores, one per row and lane, took 1.3 us per chunk)
    constexpr int TS = 36;
    __shared__ __align__(16) float turn[NEPI][16 * TS];
    __shared__ int sh_seen;                               // a cut item's counter: the others that are there

    const int NP = a.np, half_rows = NP / 2, stages = a.stages, terms = a.x_lo_row > 0 ? 2 : 1;
    const int x_bytes = half_rows * 128, stage_bytes = BM * 128 + terms * x_bytes;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int FT = MODE == 1 ? BM : PAIR;                 // output features of a tile
    const Deal deal(a, blockIdx.x >> 1);
    const uint64_t wait_limit = a.wait_limit_ns ? a.wait_limit_ns : kWaitLimitNs;

    // optional phase timestamps of the first CTA (test hook; a.trace is nullptr in normal use)
    unsigned long long *trace = (a.trace && blockIdx.x == 0) ? a.trace : nullptr;
    if (trace && threadIdx.x == 0) trace[0] = global_ns();
    if (a.trace && threadIdx.x == 0) atomicMin(a.trace + 14, (unsigned long long)global_ns());
    pdl_launch_dependents();
    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(&bars.full[s], 1);
            mbar_init(&bars.empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&bars.acc_full[b], 1);
            mbar_init(&bars.acc_empty[b], 2 * NEPI);      // one arrival per epilogue warp of both CTAs
        }
        mbar_init(&bars.drained, 1);
        bars.abort_flag = 0;
        bars.issued = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars.tmem_base)), "r"(a.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    cluster_sync_all();                                   // the peer's barriers and tensor memory exist
    tc_fence_after();
    const uint32_t tmem_base = bars.tmem_base;
    const uint32_t acc_cols = a.tmem_cols / 2;            // columns between the two accumulators
    if (trace && threadIdx.x == 0) trace[1] = global_ns();

    if (warp == 0) {
        // ---------------- TMA producer (both CTAs; every byte is counted on the first CTA's barrier) ----------------
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(&map_w) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"(&map_x) : "memory");
            // The loop is a serial chain for one thread: ring position and phase are carried along and coordinates are
            // worked out per segment (with four integer divisions per k-step it issued one every 0.5 us)
            // weights pass through L2 once; activations, partial tiles and tables should stay in it
            const uint64_t w_policy = l2_evict_first(), x_policy = l2_evict_last();
            int cw = 0, cx = 0;                           // the segment's weight and activation coordinates
            auto load_w = [&](int kt, unsigned char *slot, uint32_t bar) {
                if (MODE == 1) tma_load_pair_4d(slot, &map_w, bar, kt * BK, cw, w_policy);
                else if (MODE == 4) tma_load_pair_5d(slot, &map_w, bar, kt * BK, cw, w_policy);
                else tma_load_pair(slot, &map_w, bar, kt * BK, cw, w_policy);
            };
            auto load_x = [&](int kt, unsigned char *slot, uint32_t bar) {
                tma_load_pair(slot + BM * 128, &map_x, bar, kt * BK, cx, x_policy);
                if (terms == 2) tma_load_pair(slot + BM * 128 + x_bytes, &map_x, bar, kt * BK, a.x_lo_row + cx, x_policy);
            };
            const uint32_t full0 = map_to_rank(smem_u32(&bars.full[0]), 0u);
            int s = 0;                                    // ring slot of the next k-step, and the phase it waits for
            uint32_t phase = 1;
            bool waited = false, alive = true;
            int n = 0;                                    // k-steps so far
            Segment sg;
            for (int i = 0; alive && segment(deal, i, sg); ++i) {
                const int f = sg.item / a.wide_row_tiles * FT + (int)rank * (FT / 2);
                cw = MODE == 1 ? f / 16 : MODE == 4 ? f / a.head_dim : f;
                cx = (sg.item % a.wide_row_tiles) * NP + (int)rank * half_rows;
                int k = sg.k0;
                if (!waited) {
                    // weights depend on no kernel: they travel while the predecessor finishes
                    const int pre = min(sg.k1 - sg.k0, stages);
                    for (int j = 0; j < pre; ++j) {
                        if (j + 1 == a.stall_kstep1) continue;        // test hook: this slot is never filled
                        if (rank == 0) mbar_expect_tx(&bars.full[j], (uint32_t)(2 * stage_bytes));
                        load_w(k + j, smem + (size_t)j * stage_bytes, full0 + 8 * j);
                    }
                    pdl_wait();
                    waited = true;
                    if (trace) trace[2] = global_ns();
                    for (int j = 0; j < pre; ++j)
                        if (j + 1 != a.stall_kstep1) load_x(k + j, smem + (size_t)j * stage_bytes, full0 + 8 * j);
                    k += pre;
                    n = pre;
                    s = pre;
                    if (s == stages) { s = 0; phase = 0; }
                }
                for (; k < sg.k1; ++k) {
                    if (!pair_wait(bars, &bars.empty[s], phase, a.status, wait_limit)) { alive = false; break; }
                    unsigned char *slot = smem + (size_t)s * stage_bytes;
                    if (++n != a.stall_kstep1) {          // (test hook)
                        if (rank == 0) mbar_expect_tx(&bars.full[s], (uint32_t)(2 * stage_bytes));
                        load_w(k, slot, full0 + 8 * s);
                        load_x(k, slot, full0 + 8 * s);
                    }
                    if (++s == stages) { s = 0; phase ^= 1; }
                }
            }
            if (!waited) pdl_wait();
            bars.issued = n;
            // the last arrivals on this CTA's slots, which MMAs of the first CTA signal, come in before it may leave
            for (int i = 0; alive && i < stages; ++i) {
                alive = pair_wait(bars, &bars.empty[s], phase, a.status, wait_limit);
                if (++s == stages) { s = 0; phase ^= 1; }
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer: one thread of the pair ----------------
        if (lane == 0 && rank == 0) {
            const uint32_t idesc = idesc_pair(NP);
            int s = 0;
            uint32_t phase = 0;
            bool ok = true, first = true;
            Segment sg;
            for (int i = 0; ok && segment(deal, i, sg); ++i) {
                const int b = i & 1;
                if (!pair_wait(bars, &bars.acc_empty[b], ((uint32_t)(i >> 1) & 1u) ^ 1u, a.status, wait_limit)) break;
                tc_fence_after();
                const uint32_t acc = tmem_base + (uint32_t)b * acc_cols;
                for (int k = sg.k0; k < sg.k1; ++k) {
                    if (!pair_wait(bars, &bars.full[s], phase, a.status, wait_limit)) { ok = false; break; }
                    if (trace && first) trace[3] = global_ns();
                    first = false;
                    tc_fence_after();
                    const uint32_t slot = smem_u32(smem + (size_t)s * stage_bytes);
                    const uint64_t adesc = umma_desc(slot);
                    for (int t = 0; t < terms; ++t) {
                        const uint64_t bdesc = umma_desc(slot + BM * 128 + (uint32_t)(t * x_bytes));
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk)
                            umma_pair(acc, adesc + (uint64_t)(kk * 2), bdesc + (uint64_t)(kk * 2), idesc, (k > sg.k0 || t > 0 || kk > 0) ? 1u : 0u);
                    }
                    umma_commit_pair(&bars.empty[s]);
                    if (++s == stages) { s = 0; phase ^= 1; }
                }
                if (ok) umma_commit_pair(&bars.acc_full[b]);
            }
        }
    } else {
        // ---------------- epilogue ----------------
        pdl_wait();
        const int q = warp & 3;                           // tensor memory lane quarter of this warp
        const int c0 = ((warp - 2) >> 2) * 16;            // this warp's first column; its chunks are CSTEP columns apart
        const int t = threadIdx.x - 64;
        const uint32_t acc_empty0 = map_to_rank(smem_u32(&bars.acc_empty[0]), 0u);
        bool alive = true;                                // no wait has given up so far (the same in every warp)
        unsigned long long loop_end = 0;                  // test hook: end of this CTA's main loop so far
        Segment sg;
        for (int i = 0; segment(deal, i, sg); ++i) {
            const int b = i & 1;
            const int tile = sg.item / a.wide_row_tiles, r0 = (sg.item % a.wide_row_tiles) * NP;
            const int rows = min(NP, a.R - r0);
            const int f_quarter = tile * FT + (int)rank * (FT / 2) + q * (FT / 8);   // first feature of this lane quarter
            // ---- a part of an item: store it, and go on only if every other part is there
            int n_parts = 1, my_part = 0, first_holder = 0, first_slot = 0;
            if (sg.k1 - sg.k0 < deal.ks) {
                first_holder = deal.holder_of((long long)sg.item * deal.ks);
                // a pair's first plane takes the item its range starts in, the second the one it runs into; only the
                // item's first holder can have started earlier
                first_slot = deal.start_of(first_holder) >= (long long)sg.item * deal.ks ? 0 : 1;
                n_parts = deal.holder_of((long long)(sg.item + 1) * deal.ks - 1) - first_holder + 1;
                my_part = deal.pair - first_holder;
            }
            auto plane_of = [&](int part) {
                const int slot = (first_holder + part) * 2 + (part == 0 ? first_slot : 0);
                return reinterpret_cast<float4 *>(a.wide_planes + ((size_t)slot * 2 + rank) * PLANE) + q * 32 + lane;
            };
            // row scales, fetched while the main loop runs
            if (MODE != 3 && t < NP) {
                float inv = 1.f;
                if (a.ssq && t < rows) {
                    const float *src = a.ssq + r0 + t;
                    float ss = 0.f;
                    for (int j0 = 0; j0 < a.n_ssq; j0 += 8) {      // eight loads in flight, added in plane order
                        float p[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) p[j] = j0 + j < a.n_ssq ? __ldcg(src + (size_t)(j0 + j) * a.ssq_stride) : 0.f;
#pragma unroll
                        for (int j = 0; j < 8; ++j) ss += p[j];
                    }
                    inv = rsqrtf(ss / (float)a.K + a.eps);
                }
                row_scale[b][t] = inv;
            }
            bool ok = alive && pair_wait(bars, &bars.acc_full[b], (uint32_t)(i >> 1) & 1u, a.status, wait_limit);
            ok = __all_sync(0xffffffffu, ok);
            tc_fence_after();
            const uint32_t acc = tmem_base + (uint32_t)b * acc_cols + ((uint32_t)(q * 32) << 16);
            if (trace && t == 0 && i == 0) trace[4] = global_ns();
            if (a.trace && t == 0) loop_end = global_ns();
            int32_t *counter = a.wide_counters + sg.item * 2 + rank;
            if (n_parts > 1 && t == 0) sh_seen = *reinterpret_cast<volatile int32_t *>(counter);
            // One decision for the CTA; behind this barrier the row scales are there and part_f / part_k are free.  It holds
            // for all later items too: a barrier that was given up in one phase may read as complete in the next.
            alive = ok = epilogue_all(ok);
            bool finish = ok;
            if (n_parts > 1) {
                int seen = sh_seen;
                finish = (seen & (GIVEN_UP - 1)) == n_parts - 1;                // all others are there
                if (!finish) {
                    float4 *pl = plane_of(my_part);
                    for (int c = c0; ok && c < NP; c += CSTEP) {
                        uint32_t v[16];
                        tmem_ld16(acc + (uint32_t)c, v);
                        tmem_ld_wait();
#pragma unroll
                        for (int j = 0; j < 16; j += 4)
                            if (c + j < rows)
                                __stcg(pl + (size_t)((c + j) >> 2) * BM, make_float4(__uint_as_float(v[j]), __uint_as_float(v[j + 1]), __uint_as_float(v[j + 2]), __uint_as_float(v[j + 3])));
                    }
                    __threadfence();
                    epilogue_sync();
                    if (t == 0) sh_seen = atomicAdd(counter, ok ? 1 : 1 + GIVEN_UP);
                    epilogue_sync();
                    seen = sh_seen;
                    finish = (seen & (GIVEN_UP - 1)) == n_parts - 1;
                }
                if (finish) {
                    __threadfence();
                    if (t == 0) *counter = 0;             // ready for the next launch
                    finish = ok && seen < GIVEN_UP;
                }
                epilogue_sync();                          // sh_seen may be written again
            }
            if (trace && t == 0 && i == 0) trace[7] = finish ? global_ns() : 0;
            if (finish) {
                float *tn = turn[warp - 2];
                for (int c = c0; c < NP; c += CSTEP) {
                    const int n = min(16, rows - c);      // rows of this chunk (warp-uniform)
                    if (n <= 0) break;
                    const int rr = r0 + c;
                    // operands of the chunk's rows: in flight together with the parts below
                    const int lr = lane >> 3, lf = (lane & 7) * 4;   // mode 3: rows lr + 4 u, features lf..lf+3 of the quarter's 32
                    float4 xa[4], xb[2];
                    if (MODE == 3) {
                        const int f = f_quarter + lf;
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            xa[u] = lr + 4 * u < n && f < a.Nout ? __ldcg(reinterpret_cast<const float4 *>(a.x + (size_t)(rr + lr + 4 * u) * a.Nout + f))
                                                                : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                    // mode 4: a lane takes rows (lane >> 2) + 8 u, features 4 (lane & 3) .. + 3 of the quarter's 16 in the
                    // first half of a head, and the same ones of the second half
                    int head = 0, fi = 0;
                    bool rotate = false;
                    long long kv_base[2] = {-1, -1};
                    if (MODE == 4) {
                        const int half = a.head_dim >> 1, in_tile = q * 16;
                        head = (tile * FT + (int)rank * BM) / a.head_dim + in_tile / half;
                        fi = in_tile % half + (lane & 3) * 4;
                        rotate = head < a.Hq + a.Hkv;
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const int r = (lane >> 2) + 8 * u;
                            const bool need = rotate && r < n;
                            xa[u] = need ? __ldg(reinterpret_cast<const float4 *>(a.rope_cos + (size_t)(rr + r) * half + fi)) : make_float4(1.f, 1.f, 1.f, 1.f);
                            xb[u] = need ? __ldg(reinterpret_cast<const float4 *>(a.rope_sin + (size_t)(rr + r) * half + fi)) : make_float4(0.f, 0.f, 0.f, 0.f);
                            if (r < n && head >= a.Hq) kv_base[u] = __ldg(a.kvrow + rr + r);
                        }
                    }
                    float v[16];
                    auto take_own = [&](bool first) {
                        uint32_t w[16];
                        tmem_ld16(acc + (uint32_t)c, w);
                        tmem_ld_wait();
#pragma unroll
                        for (int j = 0; j < 16; ++j) v[j] = first ? __uint_as_float(w[j]) : v[j] + __uint_as_float(w[j]);
                    };
                    if (n_parts == 1) {
                        take_own(true);
                    } else {                              // parts in k order: the sum does not depend on who came last
#pragma unroll
                        for (int j = 0; j < 16; ++j) v[j] = 0.f;
                        for (int p0 = 0; p0 < n_parts; p0 += FLIGHT) {
                            float4 in[FLIGHT][4];
#pragma unroll
                            for (int u = 0; u < FLIGHT; ++u) {
                                const bool there = p0 + u < n_parts && p0 + u != my_part;
                                const float4 *pl = plane_of(p0 + u) + (size_t)(c >> 2) * BM;
#pragma unroll
                                for (int m = 0; m < 4; ++m)
                                    in[u][m] = there && 4 * m < n ? __ldcg(pl + (size_t)m * BM) : make_float4(0.f, 0.f, 0.f, 0.f);
                            }
#pragma unroll
                            for (int u = 0; u < FLIGHT; ++u) {
                                if (p0 + u == my_part) {
                                    take_own(false);
                                } else {
#pragma unroll
                                    for (int m = 0; m < 4; ++m) {
                                        v[4 * m] += in[u][m].x;
                                        v[4 * m + 1] += in[u][m].y;
                                        v[4 * m + 2] += in[u][m].z;
                                        v[4 * m + 3] += in[u][m].w;
                                    }
                                }
                            }
                        }
                    }
                    __syncwarp();                         // the previous chunk's reads of `turn` are done
#pragma unroll
                    for (int j = 0; j < 16; ++j) tn[j * TS + lane] = v[j];
                    __syncwarp();
                    if (MODE == 1) {
                        // 16 gate features, then the 16 up features: rows (lane >> 2) + 8 u, four features a lane
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const int r = (lane >> 2) + 8 * u, fo = (lane & 3) * 4, f = f_quarter + fo;
                            if (r < n && f < a.F) {
                                const float sc = row_scale[b][c + r];
                                const float4 g = *reinterpret_cast<const float4 *>(tn + r * TS + fo);
                                const float4 w = *reinterpret_cast<const float4 *>(tn + r * TS + 16 + fo);
                                const float g0 = g.x * sc, g1 = g.y * sc, g2 = g.z * sc, g3 = g.w * sc;
                                const float4 y = make_float4(g0 / (1.f + __expf(-g0)) * (w.x * sc), g1 / (1.f + __expf(-g1)) * (w.y * sc),
                                                             g2 / (1.f + __expf(-g2)) * (w.z * sc), g3 / (1.f + __expf(-g3)) * (w.w * sc));
                                const size_t o = (size_t)(rr + r) * a.F + f;
                                store_two_term(a.act + o, a.act_lo ? a.act_lo + o : nullptr, y);
                            }
                        }
                    } else if (MODE == 3) {
                        const int f = f_quarter + lf;
                        const bool valid = f < a.Nout;    // Nout is a multiple of 4
                        float4 gain = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (valid) {
                            const uint2 gg = __ldg(reinterpret_cast<const uint2 *>(a.gain + f));
                            const __nv_bfloat162 g01 = *reinterpret_cast<const __nv_bfloat162 *>(&gg.x), g23 = *reinterpret_cast<const __nv_bfloat162 *>(&gg.y);
                            gain = make_float4(__low2float(g01), __high2float(g01), __low2float(g23), __high2float(g23));
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int r = lr + 4 * u;
                            float sq = 0.f;
                            if (r < n && valid) {
                                const float4 y = *reinterpret_cast<const float4 *>(tn + r * TS + lf);
                                float4 x = xa[u];
                                x.x += y.x; x.y += y.y; x.z += y.z; x.w += y.w;
                                const size_t o = (size_t)(rr + r) * a.Nout + f;
                                *reinterpret_cast<float4 *>(a.x + o) = x;
                                store_two_term(a.xb + o, a.xb_lo ? a.xb_lo + o : nullptr, make_float4(x.x * gain.x, x.y * gain.y, x.z * gain.z, x.w * gain.w));
                                if (a.hidden_out) store_two_term(a.hidden_out + o, nullptr, x);
                                sq = ((x.x * x.x + x.y * x.y) + x.z * x.z) + x.w * x.w;
                            }
#pragma unroll
                            for (int o = 4; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
                            if ((lane & 7) == 0) part_f[q][c + r] = sq;
                        }
                    } else if (MODE == 4) {
                        const int half = a.head_dim >> 1;
                        const bool is_q = head < a.Hq, is_k = !is_q && rotate;
                        const int kvh = is_k ? head - a.Hq : head - a.Hq - a.Hkv;
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const int r = (lane >> 2) + 8 * u;
                            if (r < n && head < a.Nout / a.head_dim) {
                                const float sc = row_scale[b][c + r];
                                float4 y = *reinterpret_cast<const float4 *>(tn + r * TS + (lane & 3) * 4);
                                float4 z = *reinterpret_cast<const float4 *>(tn + r * TS + 16 + (lane & 3) * 4);
                                y.x *= sc; y.y *= sc; y.z *= sc; y.w *= sc;
                                z.x *= sc; z.y *= sc; z.z *= sc; z.w *= sc;
                                if (rotate) {
                                    const float4 cs = xa[u], sn = xb[u], y0 = y;
                                    y = make_float4(y.x * cs.x - z.x * sn.x, y.y * cs.y - z.y * sn.y, y.z * cs.z - z.z * sn.z, y.w * cs.w - z.w * sn.w);
                                    z = make_float4(z.x * cs.x + y0.x * sn.x, z.y * cs.y + y0.y * sn.y, z.z * cs.z + y0.z * sn.z, z.w * cs.w + y0.w * sn.w);
                                }
                                if (is_q) {
                                    if (rr + r < a.Rq) {
                                        const size_t o = ((size_t)(rr + r) * a.Hq + head) * a.head_dim + fi;
                                        store_two_term(a.q + o, a.q_lo ? a.q_lo + o : nullptr, y);
                                        store_two_term(a.q + o + half, a.q_lo ? a.q_lo + o + half : nullptr, z);
                                    }
                                } else if (kv_base[u] >= 0) {
                                    bf16 *dst = a.pool_layer + (size_t)kv_base[u] + (is_k ? 0 : a.v_off) + (size_t)kvh * a.head_stride + fi;
                                    store_two_term(dst, nullptr, y);
                                    store_two_term(dst + half, nullptr, z);
                                }
                            }
                        }
                    } else {
                        // row lane >> 1, features 16 (lane & 1) .. + 15 of the quarter's 32
                        const int r = lane >> 1, fo = (lane & 1) * 16, f = f_quarter + fo;
                        const bool in = r < n;
                        const float sc = in ? row_scale[b][c + r] : 0.f;
                        float y[16];
#pragma unroll
                        for (int m = 0; m < 16; m += 4) {
                            const float4 w = *reinterpret_cast<const float4 *>(tn + r * TS + fo + m);
                            y[m] = w.x * sc; y[m + 1] = w.y * sc; y[m + 2] = w.z * sc; y[m + 3] = w.w * sc;
                        }
                        const int row = min(rr + r, a.R - 1);
                        if (a.Y && in) {
                            float *dst = a.Y + (size_t)row * a.ldy + f;
#pragma unroll
                            for (int m = 0; m < 16; m += 4) {
                                if ((a.ldy & 3) == 0 && f + m + 3 < a.Nout) {
                                    *reinterpret_cast<float4 *>(dst + m) = make_float4(y[m], y[m + 1], y[m + 2], y[m + 3]);
                                } else {
#pragma unroll
                                    for (int k = 0; k < 4; ++k)
                                        if (f + m + k < a.Nout) dst[m + k] = y[m + k];
                                }
                            }
                        }
                        if (a.ent_out && __any_sync(0xffffffffu, in && row % a.ent_N == 0)) {
                            // soft-max statistics of a root row's 32 features
                            float mx = -INFINITY, l = 0.f, tt = 0.f;
#pragma unroll
                            for (int m = 0; m < 16; ++m)
                                if (f + m < a.Nout) mx = fmaxf(mx, y[m]);
                            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
#pragma unroll
                            for (int m = 0; m < 16; ++m)
                                if (f + m < a.Nout) {
                                    const float e = __expf(y[m] - mx);
                                    l += e;
                                    tt += e * y[m];
                                }
                            l += __shfl_xor_sync(0xffffffffu, l, 1);
                            tt += __shfl_xor_sync(0xffffffffu, tt, 1);
                            // the last pair tile's second half may lie wholly behind the vocabulary: it has no parts
                            // (a part is kept for every 32 features of ceil(Nout / 128) tiles of 128)
                            if (in && (lane & 1) == 0 && row % a.ent_N == 0 && (tile * 2 + (int)rank) * BM < a.Nout) {
                                const int part = (tile * 2 + (int)rank) * 4 + q;
                                float *dst = a.ent_part + ((size_t)part * a.ent_batch + row / a.ent_N) * 3;
                                dst[0] = mx; dst[1] = l; dst[2] = tt;
                            }
                        }
                        if (a.sample_pos) {
                            const uint32_t pos = (uint32_t)(a.sample_pos[row] + 1);
#pragma unroll
                            for (int m = 0; m < 16; m += 4) {
                                const uint4 w = philox4x32_10(make_uint4((uint32_t)((f + m) >> 2), pos, 0u, 0u),
                                                              make_uint2((uint32_t)a.sample_seed, (uint32_t)(a.sample_seed >> 32)));
                                y[m] = y[m] * a.sample_inv_t + gumbel_from_word(w.x);
                                y[m + 1] = y[m + 1] * a.sample_inv_t + gumbel_from_word(w.y);
                                y[m + 2] = y[m + 2] * a.sample_inv_t + gumbel_from_word(w.z);
                                y[m + 3] = y[m + 3] * a.sample_inv_t + gumbel_from_word(w.w);
                            }
                        }
                        unsigned long long key = 0ull;
#pragma unroll
                        for (int m = 0; m < 16; ++m)
                            if (f + m < a.Nout) {
                                const unsigned long long k = pack_val_id(y[m], f + m);
                                key = k > key ? k : key;
                            }
                        const unsigned long long other = __shfl_xor_sync(0xffffffffu, key, 1);
                        key = other > key ? other : key;
                        if ((lane & 1) == 0) part_k[q][c + r] = key;
                    }
                }
                if (MODE == 2 || MODE == 3) {
                    epilogue_sync();
                    if (t < rows) {
                        if (MODE == 3) {
                            const int plane = tile * 2 + (int)rank;           // 128 features
                            if (plane * BM < a.Nout)
                                a.ssq_out[(size_t)plane * a.ssq_stride + r0 + t] = ((part_f[0][t] + part_f[1][t]) + part_f[2][t]) + part_f[3][t];
                        } else {
                            unsigned long long key = part_k[0][t];
#pragma unroll
                            for (int k = 1; k < 4; ++k) key = part_k[k][t] > key ? part_k[k][t] : key;
                            atomicMax(a.keys + r0 + t, key);
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(acc_empty0 + (uint32_t)(b * 8));   // this warp is done with the accumulator
        }
        if (a.trace && t == 0) {
            if (trace) trace[8] = global_ns();
            if (loop_end) {                               // (0: this pair had nothing to do)
                atomicMax(a.trace + 12, loop_end);
                atomicMin(a.trace + 13, loop_end);
            }
            atomicMax(a.trace + 15, (unsigned long long)global_ns());
        }
    }
    tc_fence_before();
    cluster_sync_all();                                   // neither CTA leaves while the other still uses its memory
    if (*reinterpret_cast<volatile int *>(&bars.abort_flag)) {       // set in both CTAs or in neither
        // MMAs in flight read both CTAs' shared memory and write both CTAs' tensor memory; copies in flight write shared
        // memory and are counted on the first CTA's barriers
        if (warp == 1 && lane == 0) {
            if (rank == 0) umma_commit_pair(&bars.drained);
            bounded_wait(&bars.drained, 0, wait_limit);
        } else if (warp == 0 && lane == 0 && rank == 0) {
            int theirs;
            asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(theirs) : "r"(map_to_rank(smem_u32(&bars.issued), 1u)) : "memory");
            const int mine = bars.issued, most = max(mine, theirs);
            for (int j = max(0, most - stages); j < most; ++j) {
                if (j + 1 == a.stall_kstep1) continue;    // issued by neither
                if (j >= mine) mbar_expect_tx(&bars.full[j % stages], (uint32_t)stage_bytes);           // the peer's copies only
                else if (j >= theirs) mbar_complete_tx(&bars.full[j % stages], (uint32_t)stage_bytes);  // without the peer's
            }
            for (int j = max(0, most - stages); j < most; ++j)
                if (j + 1 != a.stall_kstep1) bounded_wait(&bars.full[j % stages], (uint32_t)(j / stages) & 1u, wait_limit);
        }
        __syncwarp();
        cluster_sync_all();
    }
    if (trace && threadIdx.x == 0) trace[9] = global_ns();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(a.tmem_cols) : "memory");
    }
    if (MODE == 2) finish_argmax<NTHR>(a, 4 * ((a.Nout + BM - 1) / BM));
}

template <int MODE>
cudaError_t launch_mode(const TcGemmArgs &a, const CUtensorMap &mw, const CUtensorMap &mx, size_t smem, cudaStream_t st) {
    static bool once = false;
    if (!once) {
        cudaError_t e = cudaFuncSetAttribute(gemm_wide_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWideSmem);
        if (e != cudaSuccess) return e;
        once = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * a.wide_pairs, 1, 1);
    cfg.blockDim = dim3(NTHR, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, gemm_wide_kernel<MODE>, mw, mx, a);
}

}  // namespace

bool wide_make_map(CUtensorMap *map, int mode, const void *W, int Nout, int K, int head_dim) {
    if (mode == 1) {          // [F / 16 groups][gate, up][16 rows][K]
        const uint64_t F = (uint64_t)Nout / 2, dims[4] = {(uint64_t)K, 16, 2, F / 16}, rows[3] = {1, F, 16};
        const uint32_t box[4] = {BK, 16, 2, 4};
        return tc_make_map_nd(map, W, 4, dims, rows, box);
    }
    if (mode == 4) {          // [heads][half / 16 groups][first, second half][16 rows][K]
        const uint64_t d = (uint64_t)head_dim, half = d / 2, dims[5] = {(uint64_t)K, 16, 2, half / 16, (uint64_t)Nout / d}, rows[4] = {1, half, 16, d};
        const uint32_t box[5] = {BK, 16, 2, (uint32_t)(half / 16), (uint32_t)(BM / d)};
        return tc_make_map_nd(map, W, 5, dims, rows, box);
    }
    return tc_make_map(map, W, (uint64_t)K, (uint64_t)Nout, BM);
}

WideShape wide_shape(int mode, int Nout, int K, int R) {
    WideShape s;
    const int feats = mode == 1 ? Nout / 2 : Nout, ft = mode == 1 ? BM : PAIR;
    s.row_tiles = (R + kWideRows - 1) / kWideRows;
    s.np = ((R + s.row_tiles - 1) / s.row_tiles + 31) / 32 * 32;
    s.items = (feats + ft - 1) / ft * s.row_tiles;
    s.steps = (long long)s.items * (K / BK);
    // a part of fewer than eight k-steps would cost more in the exchange than it saves
    s.pairs = (int)std::max(1LL, std::min<long long>(kWidePairs, s.steps / 8));
    s.rounds = s.items / s.pairs;
    s.cut = s.items % s.pairs;
    // A rest that nearly fills a round is dealt out whole: the pairs left over idle for an item, which takes them
    // (P - rest) / P of its k-steps' time, and the exchange of the parts (20 us where no whole item follows) is saved
    // (1280 rows at the 7B widths, 70 items: O 64 -> 53 us, down 270 -> 230).
    const double step_us = 0.2 + s.np * (mode == 1 || mode == 3 ? 2 : 1) * 0.00095;
    if (s.cut * 5 >= s.pairs * 4 && (1.0 - (double)s.cut / s.pairs) * (K / BK) * step_us < 15.0) {
        s.cut = 0;
        ++s.rounds;
    }
    s.cutters = std::max(1, std::min({s.pairs, 8 * s.cut, (int)((long long)s.cut * (K / BK) / 4)}));
    return s;
}

namespace {

struct Ring {
    int stages;
    uint32_t tmem_cols;
    size_t smem;
};

Ring ring_of(const WideShape &s, bool two_term) {
    Ring r;
    const int stage_bytes = BM * 128 + (two_term ? 2 : 1) * (s.np / 2) * 128;
    r.stages = std::min(MAX_STAGES, (kWideSmem - 1024) / stage_bytes);
    r.tmem_cols = 32;
    while ((int)r.tmem_cols < 2 * s.np) r.tmem_cols <<= 1;
    r.smem = std::max((size_t)r.stages * stage_bytes + 1024, least_smem(r.tmem_cols));
    return r;
}

}  // namespace

CtaSize wide_cta_size(int mode, int Nout, int K, int R, bool two_term) {
    const Ring r = ring_of(wide_shape(mode, Nout, K, R), two_term);
    return CtaSize{(long long)r.smem, (long long)r.tmem_cols};
}

cudaError_t launch_gemm_wide(int mode, TcGemmArgs a, const WideShape &s, const CUtensorMap &map_w, const CUtensorMap &map_x,
                             cudaStream_t st) {
    a.np = s.np;
    a.wide_pairs = s.pairs; a.wide_row_tiles = s.row_tiles; a.wide_rounds = s.rounds; a.wide_cut = s.cut; a.wide_items = s.items;
    a.wide_cutters = s.cutters;
    const Ring r = ring_of(s, a.x_lo_row > 0);
    a.stages = r.stages;
    a.tmem_cols = r.tmem_cols;
    if (s.cut > kWideCut || s.pairs > kWidePairs || s.np > kWideRows) return cudaErrorInvalidValue;
    if (mode == 1) return launch_mode<1>(a, map_w, map_x, r.smem, st);
    if (mode == 2) return launch_mode<2>(a, map_w, map_x, r.smem, st);
    if (mode == 3) return launch_mode<3>(a, map_w, map_x, r.smem, st);
    return launch_mode<4>(a, map_w, map_x, r.smem, st);
}

}  // namespace glance
