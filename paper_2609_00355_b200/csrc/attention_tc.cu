// Split-KV paged attention on the 5th-generation tensor cores (tcgen05 + TMEM) for the packed tree rows
// (Definition 1: ancestor-masked target pass) and the draft block (Section 3.2).
//
// One CTA = (128 packed query rows of one kv head, one key split).  The G query heads that share a kv
// head are packed into the row dimension (packed row = node * G + g), so each K/V page is fetched once
// per CTA for all of them.  Per 128-key tile (= two KV pages, TMA-loaded with 128-byte swizzle):
//     S[128 x 128] = Q K^T          tcgen05.mma, A = Q (K-major, two bf16 terms hi + lo: the rounding of a query
//                                   would otherwise reach every score of its row), B = K pages (K-major),
//                                   accumulator in TMEM
//     P            = 2^(S' - m)     softmax warps (one thread per row) read S from TMEM, apply the scale and the
//                                   ancestor mask, write P back into TMEM over the scores as two bf16 terms (32 keys
//                                   take the 32 columns of their scores: 16 of hi pairs, 16 of lo pairs)
//     O[128 x d]  += P V            tcgen05.mma, A = P_hi and P_lo in tensor memory, B = V pages (MN-major),
//                                   accumulator in TMEM
// Why 128 keys: a 128 x 64 x 16 MMA reads its 4 KB of Q from shared memory for 32 clocks of arithmetic and takes 59, a
// 128 x 128 x 16 one takes 64; 24 MMAs per 64 keys measure 1270 clocks, 32 per 128 keys 2053.
//
// The softmax warps form two groups: one takes the CTA's even key tiles, the other the odd ones, each with an S/P
// buffer, its own running maximum, row sums and accumulator in TMEM.  The tensor pipe works off P V and the next scores
// of one group (2053 clocks) while the other group's exponentials run; the two accumulators are combined like two key
// splits when the loop ends.  The running reference maximum m of a row is only raised when a tile exceeds it by more
// than 2^8 (the accumulator is then rescaled in TMEM), so exponentials stay far inside fp32/bf16 range and O is almost
// never touched between tiles.  Loops over columns are kept rolled where they can be: every launch finds its
// instructions cold, and a CTA of a short context runs this code two or three times.
// Measured per layer at the 7B widths against 64-key tiles with two threads a row and two S/P buffers a group, us: 128 rows
// over 8704 positions 72 -> 46, 8 x 64 rows over 1024..4096 97 -> 71, 1280 rows of a prefill 97 -> 42, 64 rows over 1536
// 17.8 -> 16.2, one row 15 -> 13.3.  What is left of a long loop is the softmax warps (1.85 us per 128-key tile for
// 1.05 of MMAs), of a short one the start and the merge.
// Warp roles: warp 0 = TMA producer, warp 1 = TMEM allocator + MMA issuer, warps 2..9 = softmax / epilogue.
// The key splits of a tile form a thread-block cluster and are merged through distributed shared memory
// (one asynchronous bulk copy per owner CTA, byte-counted on the owner's mbarrier).  Every mbarrier wait is
// bounded; a wait that gives up records GLANCE_E_TIMEOUT.
#include "kernels.cuh"
#include "tc_ptx.cuh"

namespace glance {

namespace {

using namespace tc;

constexpr int QT = 128;           // packed query rows per CTA (UMMA M)
constexpr int KT = 2 * kPage;     // keys per tile (UMMA N of S, K of P V); a split with an odd number of pages ends in half a tile
constexpr int NG = 2;             // softmax groups; tile i belongs to group i % NG, and so do its K, V and S/P buffers
constexpr int MAX_SPLITS = 8;     // the splits of a tile form one thread-block cluster
constexpr float kRescaleThreshold = 8.f;   // log2 units

__device__ __forceinline__ float ex2_approx(float x) {   // 2^x, hardware approximation; 2^-inf = +0
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
constexpr int CK = 32;                   // keys whose scores and probabilities share 32 columns of tensor memory
constexpr int P_TERMS = 2;               // bf16 terms of a probability
constexpr int NSOFT = 128 * NG;          // softmax / epilogue threads: one per row and group
constexpr int ECG = NG;                  // column groups of the epilogue: a row's d outputs are split over them
constexpr int NTHREADS = 64 + NSOFT;
static_assert(CK == 32, "the visibility bit set of 32 keys is one word");

// 16 accumulator columns of a row, combined over the softmax groups: sum_g w[g] * O_g.  Warp-collective.  Only the
// first `groups` accumulators are read (a group without tiles never wrote its TMEM columns).
__device__ __forceinline__ void load_combined(uint32_t tmem_O, uint32_t addr, int d, int groups, const float (&w)[NG], float (&out)[16]) {
    uint32_t v[NG][16];
#pragma unroll
    for (int gi = 0; gi < NG; ++gi)
        if (gi < groups) tmem_ld16(tmem_O + (uint32_t)(gi * d) + addr, v[gi]);
    tmem_ld_wait();
#pragma unroll
    for (int j = 0; j < 16; ++j) out[j] = 0.f;
#pragma unroll
    for (int gi = 0; gi < NG; ++gi)
        if (gi < groups) {
#pragma unroll
            for (int j = 0; j < 16; ++j) out[j] = fmaf(w[gi], __uint_as_float(v[gi][j]), out[j]);
        }
}

template <int D>
struct Smem {
    static constexpr int SLABS = D / 64;                 // 64-element (128-byte) column slabs of a d-wide tile
    static constexpr int SLAB = KT * 128;                // one slab of a K or V tile: the rows of both its pages
    static constexpr int KV_BYTES = SLABS * SLAB;        // a K or V tile: 32 KB at d = 128
    static constexpr int Q_BYTES = 2 * SLABS * QT * 128; // both query planes: 64 KB at d = 128
    static constexpr int OPER_BYTES = Q_BYTES + 2 * NG * KV_BYTES;      // Q, two K tiles, two V tiles
    static constexpr int ROWF = D + 4;                   // floats per merged row: O, m, l, padding
    // Split merge, in the operand buffers once every CTA of the cluster is done with its own: the rows of this CTA, and
    // behind them the rows received (each owner gets <= ceil(QT/S) rows from each of S CTAs)
    static constexpr int RECV_AT = QT * ROWF * 4;
    static constexpr int RECV_BYTES = (QT + MAX_SPLITS) * ROWF * 4;
    // tensor memory columns: one S/P buffer of 128 and one accumulator (d) per group
    static constexpr uint32_t O_COL = NG * KT;
    static constexpr uint32_t TMEM_COLS = 512;
    // d 64 would fit twice into an SM's shared memory, and clusters whose CTAs hold the columns crosswise would wait for each
    // other in a cluster barrier
    static constexpr int TOTAL = OPER_BYTES + 1024 > (int)least_smem(TMEM_COLS) ? OPER_BYTES + 1024 : (int)least_smem(TMEM_COLS);
    static_assert(O_COL + NG * D <= TMEM_COLS, "tensor memory budget");
    static_assert(RECV_AT + RECV_BYTES <= OPER_BYTES, "the merge fits the operand buffers");
    static_assert(RECV_AT % 16 == 0 && ROWF % 4 == 0, "bulk copies start on 16-byte boundaries");
};

struct alignas(8) AttnBars {
    uint64_t q_ready, k_full[NG], k_empty[NG], v_full[NG], v_empty[NG], s_full[NG], p_full[NG], all_done, v_zero, merge;
    uint32_t tmem_base;
    int abort_flag;
};

template <int D>
__global__ void __launch_bounds__(NTHREADS, 1) attn_tc_kernel(const __grid_constant__ CUtensorMap map_kv, AttnParams p) {
    constexpr int SLABS = Smem<D>::SLABS, SLAB = Smem<D>::SLAB, KV_BYTES = Smem<D>::KV_BYTES;
    constexpr int CH = D / 8;                            // 16-byte chunks per row
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char *sQ = smem;                                        // hi plane, lo plane
    unsigned char *sK = sQ + Smem<D>::Q_BYTES;                       // tiles [slab][128 keys][128 bytes], one per group
    unsigned char *sV = sK + NG * KV_BYTES;
    __shared__ AttnBars bars;
    __shared__ float red_m[NG][QT], red_l[NG][QT];        // the groups' reference maxima and row sums

    unsigned long long *trace = (p.trace && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0) ? p.trace : nullptr;
    if (trace && threadIdx.x == 0) trace[0] = global_ns();
    if (p.trace && threadIdx.x == 0) atomicMin(p.trace + 14, (unsigned long long)global_ns());   // grid span: first start
    pdl_launch_dependents();
    const int G = p.Hq / p.Hkv;
    const int PR = p.T * G;
    // a chain's query tiles see more keys the later they are: the longest of all heads start first
    int qt = blockIdx.x, kvh = blockIdx.y;
    if (p.causal) {
        const int i = blockIdx.y * gridDim.x + blockIdx.x;
        qt = (int)gridDim.x - 1 - i / p.Hkv;
        kvh = i % p.Hkv;
    }
    const int s = blockIdx.z / p.S, split = blockIdx.z % p.S;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        mbar_init(&bars.q_ready, NSOFT / 32);            // one arrival per softmax warp
        for (int b = 0; b < NG; ++b) {
            mbar_init(&bars.k_full[b], 1);
            mbar_init(&bars.k_empty[b], 1);
            mbar_init(&bars.v_full[b], 1);
            mbar_init(&bars.v_empty[b], 1);
            mbar_init(&bars.s_full[b], 1);
            mbar_init(&bars.p_full[b], 4);               // one arrival per warp of the group
        }
        mbar_init(&bars.all_done, 1);
        mbar_init(&bars.v_zero, 1);
        mbar_init(&bars.merge, 1);
        bars.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (p.S > 1) {
            // split merge: this CTA owns a band of the tile's rows and receives that band from each of the S CTAs
            const int rpc = (QT + p.S - 1) / p.S;
            const int mine = max(0, min(rpc, QT - (int)cluster_rank() * rpc));
            if (mine > 0) mbar_expect_tx(&bars.merge, (uint32_t)(p.S * mine * Smem<D>::ROWF * 4));
        }
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars.tmem_base)), "r"(Smem<D>::TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // S / P buffer of group g: columns 128 g; its accumulator: O_COL + d g
    const uint32_t tmem_S = bars.tmem_base, tmem_O = bars.tmem_base + Smem<D>::O_COL;
    volatile int *abort_flag = &bars.abort_flag;

    if (trace && threadIdx.x == 0) trace[1] = global_ns();
    // Sequence lengths change in a commit, a prefill's advance (between its passes too) or a truncation, page tables in the
    // caller's work, and each of these has finished before any kernel of the pass starts: the pass's row-setup kernel is
    // launched without programmatic overlap and releases none of its dependents early.  So both may be read before the
    // dependency wait.  Pages entirely below seq_len - block_B hold committed
    // context that no kernel of this pass writes, so the producer prefetches them before the wait as well.
    const int P = p.seq_len[s];
    // keys any row of this tile sees: all of them, or, in a chain, those up to the tile's last node
    const int n_keys = P + (p.causal ? (min((qt + 1) * QT, PR) - 1) / G + 1 : p.T);
    const int n_pages = (n_keys + kPage - 1) / kPage;
    // ceil-distribution of pages: the extra ones go to the first splits, because the last split already carries the
    // costlier masked tiles and the partial page
    const int pg_begin = (int)(((long long)split * n_pages + p.S - 1) / p.S);
    const int pg_end = (int)(((long long)(split + 1) * n_pages + p.S - 1) / p.S);
    const int np = pg_end - pg_begin;                    // pages of this CTA
    const int nt = (np + 1) / 2;                         // tiles, the last one may have one page only
    const int32_t *pt = p.page_table + (size_t)s * p.geom.max_pages_per_seq;
    // second terms of queries / probabilities on pure-context tiles (see AttnParams::lo_skip)
    const bool skip_q_lo = (p.lo_skip & 1) && P >= p.lo_skip_min_keys;
    const bool skip_p_lo = (p.lo_skip & 2) && P >= p.lo_skip_min_keys;
    if (warp != 0) {
        pdl_wait();                                      // q, the tree rows' K/V and the outputs belong to other kernels
        if (trace && threadIdx.x == 64) trace[2] = global_ns();
    }

    if (warp == 0) {
        // ---------------- TMA producer: K tiles and V tiles in separate rings of two ----------------
        int issued_k = 0, issued_v = 0;
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(&map_kv) : "memory");
            bool waited = false;
            // Rows written by this pass lie in [P - block_B, P + T): the head's refreshed context rows and the new
            // tree / block rows.  Pages entirely below that are committed context that no kernel of the pass writes,
            // so they may be fetched before the dependency wait.
            auto load_tile = [&](int i, int kv, unsigned char *dst, uint64_t *bar) {
                const int pages = min(2, np - 2 * i);
                mbar_expect_tx(bar, (uint32_t)(pages * (KV_BYTES / 2)));
                for (int h = 0; h < pages; ++h) {
                    const int pg = pg_begin + 2 * i + h;
                    if (!waited && (pg + 1) * kPage > P - kMaxBlock) {
                        pdl_wait();
                        waited = true;
                    }
                    int page = (pg < p.geom.max_pages_per_seq) ? pt[pg] : -1;
                    if (page < 0 || page >= p.geom.n_pages) {
                        page = 0;
                        set_status(p.status, GLANCE_E_BOUNDS);
                    }
                    const int row = ((page * 2 + kv) * p.geom.n_kv_heads + kvh) * kPage;
#pragma unroll
                    for (int sl = 0; sl < SLABS; ++sl) tma_load_2d(dst + sl * SLAB + h * (kPage * 128), &map_kv, bar, sl * 64, row);
                }
            };
            // K and V tiles advance independently, each as far ahead as its ring allows: one thread polls both rings
            uint64_t stall_t0 = 0;
            uint32_t spins = 0;
            while (issued_k < nt || issued_v < nt) {
                bool progressed = false;
                const int ks = issued_k & 1, vs = issued_v & 1;
                if (issued_k < nt && mbar_try_wait(&bars.k_empty[ks], ((uint32_t)(issued_k >> 1) & 1u) ^ 1u)) {
                    load_tile(issued_k, 0, sK + ks * KV_BYTES, &bars.k_full[ks]);
                    ++issued_k;
                    progressed = true;
                }
                if (issued_v < nt && mbar_try_wait(&bars.v_empty[vs], ((uint32_t)(issued_v >> 1) & 1u) ^ 1u)) {
                    load_tile(issued_v, 1, sV + vs * KV_BYTES, &bars.v_full[vs]);
                    ++issued_v;
                    progressed = true;
                }
                if (progressed) {
                    stall_t0 = 0;
                } else if ((++spins & 63u) == 0) {
                    // bounded: no slot of either ring has come free for the whole limit, or another role gave up
                    if (*abort_flag) break;
                    const uint64_t now = global_ns();
                    if (stall_t0 == 0) stall_t0 = now;
                    else if (now - stall_t0 > kWaitLimitNs) {
                        *abort_flag = 1;
                        set_status(p.status, GLANCE_E_TIMEOUT);
                        break;
                    }
                }
            }
            if (!waited) pdl_wait();
        }
        // The page that holds the last key may continue with rows that belong to nobody (any bits, NaN included):
        // this warp zeroes them in the V tile once it has landed, and tells the MMA issuer.  The wait is exact:
        // this thread issued the copy, and no later copy can follow into the slot before that tile's second MMA.
        const int last_valid = n_keys - (pg_begin + 2 * (nt - 1)) * kPage;      // keys of this CTA's last tile
        const int last_rows = (np - 2 * (nt - 1)) * kPage;                      // rows of the pages that it has
        if (nt > 0 && last_valid < last_rows) {
            const int i = nt - 1, slot = i & 1;
            int got = 0;
            if (lane == 0) got = (issued_v == nt && mbar_wait(&bars.v_full[slot], (uint32_t)(i >> 1) & 1u, abort_flag, p.status)) ? 1 : 0;
            got = __shfl_sync(0xffffffffu, got, 0);
            if (got) {
                unsigned char *v = sV + slot * KV_BYTES;
                for (int it = lane; it < (last_rows - last_valid) * CH; it += 32) {
                    const int r = last_valid + it / CH, c = it % CH;
                    *reinterpret_cast<int4 *>(v + (c >> 3) * SLAB + r * 128 + (((c & 7) ^ (r & 7)) << 4)) = make_int4(0, 0, 0, 0);
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars.v_zero);
            }
        }
        if (lane == 0) {
            if (*abort_flag) {
                // copies already issued must land before the CTA may exit
                for (int k = 0; k < 2; ++k) {
                    const int issued = k ? issued_v : issued_k;
                    uint64_t *full = k ? bars.v_full : bars.k_full;
                    for (int i = max(0, issued - NG); i < issued; ++i) {
                        const uint64_t t0 = global_ns();
                        while (!mbar_try_wait(&full[i & 1], (uint32_t)(i >> 1) & 1u))
                            if (global_ns() - t0 > kWaitLimitNs) break;
                    }
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        // The scores of the first two tiles are issued up front; after P V of tile i the scores of tile i + 2 follow into
        // the buffer that P V has just read (MMAs of one thread execute in order).
        if (lane == 0 && nt > 0) {
            const uint32_t idesc_o = umma_idesc_bmn(D);           // M 128, N d, B = V is MN-major
            const int planes = p.q_lo ? 2 : 1;
            auto pages_of = [&](int i) { return min(2, np - 2 * i); };
            auto in_context = [&](int i) { return (pg_begin + 2 * i + pages_of(i)) * kPage <= P; };
            auto issue_s = [&](int i) -> bool {
                const int b = i & 1;
                const int planes_i = (skip_q_lo && in_context(i)) ? 1 : planes;
                const uint32_t idesc_s = umma_idesc(pages_of(i) * kPage);       // M 128, N = the tile's keys
                if (!mbar_wait(&bars.k_full[b], (uint32_t)(i >> 1) & 1u, abort_flag, p.status)) return false;
                tc_fence_after();
                const uint32_t kbase = smem_u32(sK + b * KV_BYTES);
#pragma unroll 1
                for (int pl = 0; pl < planes_i; ++pl) {
                    const uint32_t qbase = smem_u32(sQ) + (uint32_t)(pl * SLABS * QT * 128);
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks) {
                        const int sl = ks >> 2, kk = ks & 3;
                        umma_f16(tmem_S + (uint32_t)(b * KT), umma_desc(qbase + sl * QT * 128) + (uint64_t)(kk * 2),
                                 umma_desc(kbase + sl * SLAB) + (uint64_t)(kk * 2), idesc_s, (pl | ks) > 0 ? 1u : 0u);
                    }
                }
                umma_commit(&bars.k_empty[b]);            // K tile free once these MMAs have read it
                umma_commit(&bars.s_full[b]);
                return true;
            };
            bool ok = mbar_wait(&bars.q_ready, 0, abort_flag, p.status);
            for (int i = 0; i < NG && i < nt && ok; ++i) ok = issue_s(i);
            for (int i = 0; i < nt && ok; ++i) {
                const int b = i & 1;
                const uint32_t ph = (uint32_t)(i >> 1) & 1u;
                if (!mbar_wait(&bars.v_full[b], ph, abort_flag, p.status)) { ok = false; break; }
                // the rows after the last key have been zeroed by the producer warp
                if (i == nt - 1 && n_keys < pg_end * kPage && !mbar_wait(&bars.v_zero, 0, abort_flag, p.status)) { ok = false; break; }
                if (!mbar_wait(&bars.p_full[b], ph, abort_flag, p.status)) { ok = false; break; }
                tc_fence_after();
                const uint32_t vbase = smem_u32(sV + b * KV_BYTES);
                const int p_terms = (skip_p_lo && in_context(i)) ? 1 : P_TERMS;
                const int chunks = pages_of(i) * (kPage / CK);
                // 32 keys: two k-steps of 16 for either term
#pragma unroll 1
                for (int c = 0; c < chunks; ++c)
#pragma unroll
                    for (int kk = 0; kk < 2; ++kk)
                        for (int pt = 0; pt < p_terms; ++pt)
                            umma_f16_ts(tmem_O + (uint32_t)(b * D), tmem_S + (uint32_t)(b * KT + c * CK + pt * (CK / 2) + kk * 8),
                                        umma_desc_mn(vbase + (c * CK + kk * 16) * 128, SLAB), idesc_o, (i >= NG || (c | kk | pt) > 0) ? 1u : 0u);
                umma_commit(&bars.v_empty[b]);            // V tile free once these MMAs have read it
                if (i + NG < nt && !issue_s(i + NG)) { ok = false; break; }
            }
            if (ok) umma_commit(&bars.all_done);         // every MMA of this CTA has completed when this barrier flips
        }
        __syncwarp();
    } else {
        // ---------------- softmax / epilogue warps ----------------
        // 8 warps in two groups of 4: warp (group, q) serves the TMEM lane quarter q, one query row per thread.
        const int q = warp & 3;                           // TMEM lane quarter this warp may access
        const int grp = (warp - 2) >> 2;                  // softmax group: takes tiles i with i % NG == grp
        const int row = q * 32 + lane;
        const int tsm = threadIdx.x - 64;                 // 0..NSOFT-1
        int pr = qt * QT + row;
        const bool row_valid = pr < PR;
        if (!row_valid) pr = PR - 1;
        const int node = pr / G, g = pr % G;
        // Q tile (both planes) -> shared memory in the K-major 128-byte-swizzled operand layout (async copies, all in
        // flight).  A thread keeps one 16-byte chunk column and walks rows NSOFT / CH apart: the row's source offset
        // (two integer divisions) is computed once per row and serves both planes.
        {
            static_assert(NSOFT % CH == 0 && QT % (NSOFT / CH) == 0, "a thread's chunks share one chunk column");
            constexpr int RSTEP = NSOFT / CH;             // rows between a thread's consecutive chunks
            const int c = tsm % CH;
            const uint32_t dst0 = smem_u32(sQ) + (uint32_t)((c >> 3) * QT * 128);
#pragma unroll 2
            for (int k = 0; k < QT / RSTEP; ++k) {
                const int r = tsm / CH + k * RSTEP;
                // rows beyond the last query are zeros, not read: with one query a head, 121 of the tile's 128 rows would
                // otherwise fetch the same two lines (plain decoding 2951 -> 2917 us a token)
                int prr = qt * QT + r;
                const uint32_t take = prr < PR ? 16u : 0u;
                if (prr >= PR) prr = PR - 1;
                const size_t off = ((size_t)(s * p.T + prr / G) * p.Hq + kvh * G + prr % G) * D + c * 8;
                const uint32_t dst = dst0 + (uint32_t)(r * 128 + (((c & 7) ^ (r & 7)) << 4));
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(p.q + off), "r"(take));
                if (p.q_lo)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + (uint32_t)(SLABS * QT * 128)), "l"(p.q_lo + off), "r"(take));
            }
        }
        asm volatile("cp.async.commit_group;" ::);
        // the row's ancestor words travel while the copies are in flight
        uint64_t anc0 = ~0ull, anc1 = ~0ull;               // no mask: every extra key is visible
        if (p.anc && !p.causal) {
            const uint64_t *a = p.anc + ((size_t)s * p.T + node) * p.W;
            anc0 = a[0];
            anc1 = p.W > 1 ? a[1] : 0ull;
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        fence_async_smem();
        __syncwarp();                                     // every lane's rows are written and fenced: one arrival per warp
        if (lane == 0) mbar_arrive(&bars.q_ready);
        if (trace && threadIdx.x == 64) trace[3] = global_ns();

        const uint32_t lane_addr = (uint32_t)(q * 32) << 16;
        const float sl2 = rsqrtf((float)D) * 1.4426950408889634f;
        const uint32_t tmem_Sg = tmem_S + lane_addr + (uint32_t)(grp * KT);     // this group's scores, and its accumulator
        const uint32_t tmem_Og = tmem_O + lane_addr + (uint32_t)(grp * D);
        float m_ref = -INFINITY, l_run = 0.f;
        bool ok = true;
        for (int i = grp; i < nt; i += NG) {
            const int key0 = (pg_begin + 2 * i) * kPage;
            const int pages = min(2, np - 2 * i);
            // The scores were issued behind P V of the group's previous tile, so this wait covers that MMA too: buffer
            // and accumulator are the group's own until it hands the tile over.
            ok = mbar_wait(&bars.s_full[grp], (uint32_t)(i >> 1) & 1u, abort_flag, p.status);
            ok = __all_sync(0xffffffffu, ok);             // TMEM accesses are warp-collective
            if (!ok) break;                               // a warp that leaves stops arriving at p_full: every wait is bounded
            if (trace && threadIdx.x == 64 && i == 0) trace[4] = global_ns();
            tc_fence_after();
            if (key0 + pages * kPage > P) {
                // Visibility of 32 keys as one bit set: committed keys (< P) are visible, keys past the last one are not,
                // extra key b is visible if bit b of the row's ancestor set is (all of them without a mask).
                // b0 = index of the first key among the extra keys; negative inside the context.
#pragma unroll 1
                for (int c = 0; c < pages * (kPage / CK); ++c) {
                    const int b0 = key0 + c * CK - P;
                    uint32_t vis;
                    if (p.causal) {
                        const int n_vis = node + 1 - b0;  // leading visible keys
                        vis = n_vis >= 32 ? 0xffffffffu : n_vis <= 0 ? 0u : ((1u << n_vis) - 1u);
                    } else if (b0 >= 0) {
                        const uint64_t lo = b0 >= 64 ? anc1 : anc0, hi = b0 >= 64 ? 0ull : anc1;
                        const int sh = b0 & 63;
                        vis = (uint32_t)(sh == 0 ? lo : ((lo >> sh) | (hi << (64 - sh))));
                    } else {
                        const int nctx = -b0;             // leading committed keys
                        vis = nctx >= 32 ? 0xffffffffu : (((uint32_t)anc0 << nctx) | ((1u << nctx) - 1u));
                    }
                    const int n_valid = p.T - b0;         // keys that exist
                    if (n_valid < 32) vis &= n_valid <= 0 ? 0u : ((1u << n_valid) - 1u);
                    if (__all_sync(0xffffffffu, vis == 0xffffffffu)) continue;
                    uint32_t v[32];
                    tmem_ld32(tmem_Sg + (uint32_t)(c * CK), v);
                    tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = ((vis >> j) & 1u) ? v[j] : 0xff800000u;    // -inf
                    tmem_st32(tmem_Sg + (uint32_t)(c * CK), v);
                }
                tmem_st_wait();
            }
            // maximum of the row's raw scores; the scale is folded into the exponent (sl2 > 0 keeps the order)
            float mt = -INFINITY;
#pragma unroll 1
            for (int h = 0; h < pages; ++h) {
                uint32_t v[2][32];
                tmem_ld32(tmem_Sg + (uint32_t)(h * kPage), v[0]);
                tmem_ld32(tmem_Sg + (uint32_t)(h * kPage + CK), v[1]);
                tmem_ld_wait();
                float m4[4] = {mt, mt, mt, mt};
#pragma unroll
                for (int j = 0; j < 32; j += 4)
#pragma unroll
                    for (int u = 0; u < 4; ++u) m4[u] = fmaxf(m4[u], fmaxf(__uint_as_float(v[0][j + u]), __uint_as_float(v[1][j + u])));
                mt = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
            }
            mt *= sl2;
            float factor = 1.f;
            if (m_ref == -INFINITY) {
                m_ref = mt;                               // nothing accumulated for this row yet
            } else if (mt > m_ref + kRescaleThreshold) {
                factor = exp2f(m_ref - mt);
                m_ref = mt;
            }
            if (__any_sync(0xffffffffu, factor != 1.f)) {
                l_run *= factor;
#pragma unroll 1
                for (int c = 0; c < D; c += 32) {
                    uint32_t v[32];
                    tmem_ld32(tmem_Og + (uint32_t)c, v);
                    tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) * factor);
                    tmem_st32(tmem_Og + (uint32_t)c, v);
                }
            }
            // P = 2^(S' - m_ref) as bf16 pairs over the scores of the same 32 keys: hi terms, then lo terms (what the hi
            // term lost to rounding); both are A operands of the second MMA
            const float m_sub = (m_ref == -INFINITY) ? 0.f : m_ref;   // a fully masked row keeps -inf - 0 = -inf -> 2^-inf = 0
            const float2 scale2 = make_float2(sl2, sl2), shift2 = make_float2(-m_sub, -m_sub);
            float2 rs0 = make_float2(0.f, 0.f), rs1 = rs0;
#pragma unroll 1
            for (int h = 0; h < pages; ++h) {
                uint32_t v[2][32];
                tmem_ld32(tmem_Sg + (uint32_t)(h * kPage), v[0]);
                tmem_ld32(tmem_Sg + (uint32_t)(h * kPage + CK), v[1]);
                tmem_ld_wait();
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    uint32_t w[32];
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const float2 e = fma2(make_float2(__uint_as_float(v[u][2 * j]), __uint_as_float(v[u][2 * j + 1])), scale2, shift2);
                        const float2 pp = make_float2(ex2_approx(e.x), ex2_approx(e.y));
                        if (j & 1) rs1 = add2(rs1, pp);
                        else rs0 = add2(rs0, pp);
                        __nv_bfloat162 h2 = __floats2bfloat162_rn(pp.x, pp.y);
                        w[j] = *reinterpret_cast<uint32_t *>(&h2);
                        const float2 left = add2(pp, make_float2(-__uint_as_float(w[j] << 16), -__uint_as_float(w[j] & 0xffff0000u)));
                        __nv_bfloat162 l2 = __floats2bfloat162_rn(left.x, left.y);
                        w[16 + j] = *reinterpret_cast<uint32_t *>(&l2);
                    }
                    tmem_st32(tmem_Sg + (uint32_t)(h * kPage + u * CK), w);
                }
            }
            l_run += (rs0.x + rs0.y) + (rs1.x + rs1.y);
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();                                 // single arrivals of every thread would serialise on the barrier word
            if (lane == 0) mbar_arrive(&bars.p_full[grp]);
            if (trace && threadIdx.x == 64 && i == 0) trace[5] = global_ns();
        }
        if (trace && threadIdx.x == 64) trace[6] = global_ns();
        // the groups' row sums and reference maxima meet here: every thread combines them in fixed order (this needs
        // no accumulator and runs while the last second MMA completes)
        red_m[grp][row] = m_ref;
        red_l[grp][row] = l_run;
        asm volatile("bar.sync 1, %0;" ::"n"(NSOFT) : "memory");
        float m_all = -INFINITY, l_row = 0.f, w[NG];
#pragma unroll
        for (int gi = 0; gi < NG; ++gi) m_all = fmaxf(m_all, red_m[gi][row]);
#pragma unroll
        for (int gi = 0; gi < NG; ++gi) {
            // weight of the group's accumulator; a group without tiles, or with no visible key in this row, has none
            const float gm = red_m[gi][row];
            w[gi] = (gi < nt && gm != -INFINITY) ? ex2_approx(gm - m_all) : 0.f;
            l_row += w[gi] * red_l[gi][row];
        }
        // The accumulators are read below by every softmax thread: the issuer commits a one-shot barrier after its last MMA.
        if (nt > 0) {
            ok = ok && mbar_wait(&bars.all_done, 0, abort_flag, p.status);
            ok = __all_sync(0xffffffffu, ok);
            tc_fence_after();
        }
        ok = ok && (*abort_flag == 0);
        ok = __all_sync(0xffffffffu, ok);
        if (trace && threadIdx.x == 64) trace[7] = global_ns();
        // ---------------- epilogue ----------------
        constexpr int OC = D / ECG;                       // output columns of a thread
        if (p.S == 1) {
            const float inv = 1.f / l_row;
            const bool aligned = (((uintptr_t)p.out | (uintptr_t)p.out_lo) & 15) == 0;     // (rows start on multiples of 128 bytes)
            const size_t off = ((size_t)(s * p.T + node) * p.Hq + kvh * G + g) * D + grp * OC;
#pragma unroll 1
            for (int c = 0; ok && c < OC; c += 16) {
                float v[16];
                load_combined(tmem_O, lane_addr + (uint32_t)(grp * OC + c), D, min(nt, NG), w, v);
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] *= inv;
                if (row_valid && aligned) {
#pragma unroll
                    for (int j = 0; j < 16; j += 8) store_two_term8(p.out + off + c + j, p.out_lo ? p.out_lo + off + c + j : nullptr, v + j);
                } else if (row_valid) {
#pragma unroll
                    for (int j = 0; j < 16; j += 4)
                        store_two_term(p.out + off + c + j, p.out_lo ? p.out_lo + off + c + j : nullptr, make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]));
                }
            }
        } else {
            // ---------------- merge of the key splits inside the cluster (reduce-scatter by rows) ----------------
            // The S CTAs of one (sequence, kv head, q tile) form a cluster.  CTA `rank` owns rows [rank*RPC, +RPC).
            // Every CTA stages its unnormalised O rows with (m, l) in its own (now idle) operand buffers, then one
            // asynchronous shared-to-shared copy per owner ships that owner's band into the owner's receive region
            // and counts its bytes on the owner's merge barrier; the owner combines the S bands in split order.
            constexpr int ROWF = Smem<D>::ROWF;
            const int RPC = (QT + p.S - 1) / p.S;
            const uint32_t rank = cluster_rank();
            float *stage = reinterpret_cast<float *>(smem);
            unsigned char *recv = smem + Smem<D>::RECV_AT;
            // This CTA's MMAs have all completed and every page it asked for has been consumed: its operand buffers may
            // receive rows.  The copies below start when every CTA of the cluster has got here.
            cluster_arrive();
            const bool live = nt > 0 && ok;
            float *dst = stage + (size_t)row * ROWF + grp * OC;
#pragma unroll 1
            for (int c = 0; c < OC; c += 16) {
                float v[16];
                if (live) {
                    load_combined(tmem_O, lane_addr + (uint32_t)(grp * OC + c), D, min(nt, NG), w, v);
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = 0.f;
                }
#pragma unroll
                for (int j = 0; j < 16; j += 4)
                    *reinterpret_cast<float4 *>(dst + c + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
            }
            if (grp == 0) {
                stage[(size_t)row * ROWF + D] = live ? m_all : -INFINITY;
                stage[(size_t)row * ROWF + D + 1] = live ? l_row : 0.f;
            }
            fence_async_smem();                           // staged rows visible to the asynchronous copy engine
            cluster_wait();
            asm volatile("bar.sync 1, %0;" ::"n"(NSOFT) : "memory");
            if (trace && threadIdx.x == 64) trace[8] = global_ns();
            if (warp == 2 && lane < p.S) {
                const uint32_t owner = (uint32_t)lane;
                const int rows = max(0, min(RPC, QT - (int)owner * RPC));
                if (rows > 0)
                    dsmem_bulk_copy(map_to_rank(smem_u32(recv) + (uint32_t)(rank * RPC * ROWF * 4), owner),
                                    smem_u32(stage) + (uint32_t)(owner * RPC * ROWF * 4), (uint32_t)(rows * ROWF * 4),
                                    map_to_rank(smem_u32(&bars.merge), owner));
            }
            __syncwarp();
            if (trace && threadIdx.x == 64) trace[9] = global_ns();
            const int row_lo = (int)rank * RPC;
            const int own_rows = max(0, min(RPC, QT - row_lo));
            bool got = true;
            if (own_rows > 0) got = mbar_wait(&bars.merge, 0, abort_flag, p.status);
            __syncwarp();
            // Everything bound for this CTA has landed: that is all its peers need to know before they may leave
            // (a CTA's staged rows are read by the copies it sent).  The matching wait is at the end of the kernel.
            cluster_arrive();
            if (trace && threadIdx.x == 64) trace[10] = global_ns();
            const float *rows = reinterpret_cast<const float *>(recv);
            const int my_rows = got ? max(0, min(own_rows, PR - qt * QT - row_lo)) : 0;
            constexpr int SEG = D / 8;                    // items per row: two 4-float pieces, half a row apart
#pragma unroll 1
            for (int item = tsm; item < my_rows * SEG; item += NSOFT) {
                const int lr = item / SEG, c0 = (item % SEG) * 4, c1 = D / 2 + c0;
                const float *rp0 = rows + (size_t)lr * ROWF;
                const size_t sstride = (size_t)RPC * ROWF;      // floats between the same row of consecutive splits
                // all loads first (the values of up to MAX_SPLITS splits), then the arithmetic
                float ms[MAX_SPLITS], ls[MAX_SPLITS];
                float4 va[MAX_SPLITS], vb[MAX_SPLITS];
                float M = -INFINITY;
#pragma unroll
                for (int sp = 0; sp < MAX_SPLITS; ++sp) {
                    ms[sp] = -INFINITY; ls[sp] = 0.f;
                    va[sp] = vb[sp] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (sp < p.S) {
                        const float *rp = rp0 + sp * sstride;
                        ms[sp] = rp[D];
                        ls[sp] = rp[D + 1];
                        va[sp] = *reinterpret_cast<const float4 *>(rp + c0);
                        vb[sp] = *reinterpret_cast<const float4 *>(rp + c1);
                        M = fmaxf(M, ms[sp]);
                    }
                }
                float4 acc = make_float4(0.f, 0.f, 0.f, 0.f), bcc = acc;
                float den = 0.f;
#pragma unroll
                for (int sp = 0; sp < MAX_SPLITS; ++sp) {  // split order: bit-reproducible
                    const float ws = ex2_approx(ms[sp] - M);   // 2^-inf = 0 for an empty split
                    den += ws * ls[sp];
                    acc.x += ws * va[sp].x; acc.y += ws * va[sp].y; acc.z += ws * va[sp].z; acc.w += ws * va[sp].w;
                    bcc.x += ws * vb[sp].x; bcc.y += ws * vb[sp].y; bcc.z += ws * vb[sp].z; bcc.w += ws * vb[sp].w;
                }
                const float inv = 1.f / den;
                const int prr = qt * QT + row_lo + lr;
                const size_t off = ((size_t)(s * p.T + prr / G) * p.Hq + kvh * G + prr % G) * D;
                store_two_term(p.out + off + c0, p.out_lo ? p.out_lo + off + c0 : nullptr,
                               make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv));
                store_two_term(p.out + off + c1, p.out_lo ? p.out_lo + off + c1 : nullptr,
                               make_float4(bcc.x * inv, bcc.y * inv, bcc.z * inv, bcc.w * inv));
            }
        }
        tc_fence_before();
    }
    if (trace && threadIdx.x == 64) trace[11] = global_ns();
    if (p.trace && threadIdx.x == 64) atomicMax(p.trace + 15, (unsigned long long)global_ns());  // grid span: last end
    if (p.S > 1) {
        __syncwarp();
        if (warp < 2) {                                  // the two arrivals of the softmax warps' merge
            cluster_arrive();
            cluster_wait();
            cluster_arrive();
        }
        // no CTA leaves while its staged rows may still be read by a copy in flight, or a peer may still write to it
        cluster_wait();
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(bars.tmem_base), "r"(Smem<D>::TMEM_COLS) : "memory");
    }
}

template <int D>
cudaError_t launch_d(const AttnParams &p, const CUtensorMap &map_kv, dim3 grid, cudaStream_t st) {
    static bool once = false;
    if (!once) {
        cudaError_t e = cudaFuncSetAttribute(attn_tc_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem<D>::TOTAL);
        if (e != cudaSuccess) return e;
        once = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(NTHREADS, 1, 1);
    cfg.dynamicSmemBytes = Smem<D>::TOTAL;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;      // the key splits of one tile form a cluster
    attr[1].val.clusterDim.x = 1;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = p.S;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, attn_tc_kernel<D>, map_kv, p);
}

// largest number of co-resident clusters of `cs` CTAs of this kernel (queried once per cluster size)
template <int D>
int max_active_clusters(int cs) {
    static int cache[MAX_SPLITS + 1] = {0};
    if (cache[cs] == 0) {
        cudaFuncSetAttribute(attn_tc_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem<D>::TOTAL);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(1, 1, cs);
        cfg.blockDim = dim3(NTHREADS, 1, 1);
        cfg.dynamicSmemBytes = Smem<D>::TOTAL;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 1;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = cs;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, attn_tc_kernel<D>, &cfg) != cudaSuccess || n < 1) n = 148 / cs - 4;
        cache[cs] = n < 1 ? 1 : n;
    }
    return cache[cs];
}

}  // namespace

CtaSize attention_tc_cta_size(int d) {
    return d == 128 ? CtaSize{Smem<128>::TOTAL, Smem<128>::TMEM_COLS} : CtaSize{Smem<64>::TOTAL, Smem<64>::TMEM_COLS};
}

int attention_tc_q_tiles(int T, int G) { return (T * G + QT - 1) / QT; }

// Key splits per (sequence, kv head, q tile): the splits of a tile form a cluster, and all clusters of the
// launch should be resident at once (a second wave would double the kernel's latency).  A launch that cannot fit
// one wave split (several sequences), but fits unsplit, gets two splits: that halves the longest sequence's loop, which sets
// the launch's duration, while larger clusters lose more than they gain once clusters queue for SMs (a cluster starts
// only when enough SMs of one GPC are free together: with 64-key tiles 8 sequences of 1024-4096 positions took 100 / 84 /
// 102 / 154 us per layer with 1 / 2 / 4 / 8 splits; with 128-key tiles two splits take 70).
// Beyond one CTA per SM unsplit (a long prefill, many sequences) there is nothing to fill, and it stays unsplit.
int attention_tc_splits(int T, int G, int Hkv, int batch, int d) {
    const int base = attention_tc_q_tiles(T, G) * Hkv * batch;
    for (int s = MAX_SPLITS; s > 1; --s) {
        const int fit = d == 128 ? max_active_clusters<128>(s) : max_active_clusters<64>(s);
        if (base <= fit) return s;
    }
    return base <= 148 ? 2 : 1;
}

cudaError_t launch_attention_tc(const AttnParams &p, const CUtensorMap &map_kv, cudaStream_t st) {
    const int G = p.Hq / p.Hkv;
    dim3 grid(attention_tc_q_tiles(p.T, G), p.Hkv, p.batch * p.S);
    if (p.d == 128) return launch_d<128>(p, map_kv, grid, st);
    return launch_d<64>(p, map_kv, grid, st);
}

}  // namespace glance
