// Candidate-tree construction (Algorithm 1 lines 2-3) and greedy walk + KV commit (lines 5-12).
#include "kernels.cuh"
#include "tc_ptx.cuh"

namespace glance {

// ------------------------------------------------------------------------------------------
// Best-first tree builder: one warp per sequence.
//
// Keeps the min(N-1, sum_l k^l) prefixes of highest score under the total order
// (score desc, depth asc, path key asc).  The frontier holds, for every kept node, its best child that is not kept yet;
// a node's children score no higher than the node and fall with their rank (log-probabilities are <= 0 and
// non-increasing in rank, fp32 addition is monotone), so repeatedly popping the best frontier entry enumerates the order
// exactly.  A node's score is one fp32 add from its parent's score.
//
// A pop is a serial chain, so it is kept short: warp maximum, ballot, one shuffle.  Node i and its frontier entry live in
// slot i / 32 of lane i % 32.  The popped entry's lane moves on to its next child by itself, the popped score is the warp
// maximum itself, and the new node's lane receives the image of its first child ready made; everything else (tables, path
// keys) is fetched or computed off the chain.  Equal scores, which alone need the 64-bit tie word, take a separate path,
// and the ancestor masks are built in parallel at the end.  63 pops: 29.0 -> 16.2 us a call.
// ------------------------------------------------------------------------------------------
// Path keys are ranks as 4-bit digits, the first edge in the most significant digit that the largest block uses.
__device__ __forceinline__ unsigned long long path_digit(int depth, int rank) { return (unsigned long long)rank << (4 * (15 - depth)); }

template <int SLOTS>
__global__ void __launch_bounds__(32) build_tree_kernel(int N, int L, int k, const int32_t *root, const int32_t *ids,
                                                        const float *lp, glance_tree out) {
    __shared__ int n_parent[SLOTS * 32];
    __shared__ float s_lp[kMaxBlock * kMaxTopk + 1];
    __shared__ int s_id[kMaxBlock * kMaxTopk];
    const int s = blockIdx.x, lane = threadIdx.x;
    const int W = (N + 63) >> 6;
    // Candidates and outputs belong to other kernels before the wait.  Dependents may start after it and not before: some
    // read sequence lengths ahead of their own wait, which a commit in front of this kernel may still be changing.
    tc::pdl_wait();
    tc::pdl_launch_dependents();
    const int32_t *sid = ids + (size_t)s * L * k;
    const float *slp = lp + (size_t)s * L * k;
    for (int e = lane; e < L * k; e += 32) {
        s_lp[e] = slp[e];
        s_id[e] = sid[e];
    }
    const int32_t root_tok = root[s];
    __syncwarp();

    // node u * 32 + lane: score, meta = depth | rank << 4 | parent << 8, path key.  Its frontier entry, the candidate child
    // of rank next[u]: order-preserving image of the candidate's score (0 = none); the log-probabilities of the rank after
    // it and of its own best child, from which `succ` and `kid` -- the images that take its place and that open the new
    // node's entry when it is popped -- are worked out while the next warp maximum is under way.
    float score[SLOTS], lp_succ[SLOTS], lp_kid[SLOTS];
    uint32_t meta[SLOTS], front[SLOTS];
    int next[SLOTS];
    unsigned long long key[SLOTS];
    constexpr int kNone = kMaxBlock * kMaxTopk;          // entry of s_lp behind the table
#pragma unroll
    for (int u = 0; u < SLOTS; ++u) {
        score[u] = 0.f; lp_succ[u] = 0.f; lp_kid[u] = 0.f; meta[u] = 0u; front[u] = 0u; next[u] = 0; key[u] = 0ull;
    }
    if (lane == 0 && L >= 1 && N > 1) {
        front[0] = float_key(__fadd_rn(0.f, s_lp[0]));
        lp_succ[0] = s_lp[1];
        lp_kid[0] = s_lp[k];
    }
    int nc = 1;
    while (nc < N) {
        uint32_t mine = front[0];
#pragma unroll
        for (int u = 1; u < SLOTS; ++u) mine = max(mine, front[u]);
        const uint32_t best = __reduce_max_sync(0xffffffffu, mine);
        uint32_t succ[SLOTS], kid[SLOTS];
#pragma unroll
        for (int u = 0; u < SLOTS; ++u) {
            succ[u] = next[u] + 1 < k ? float_key(__fadd_rn(score[u], lp_succ[u])) : 0u;
            kid[u] = (int)(meta[u] & 15u) + 1 < L ? float_key(__fadd_rn(key_float(front[u]), lp_kid[u])) : 0u;
        }
        if (best == 0u) break;                           // no candidate is left
        int slot = 0, holders = 0, wl = 0;
#pragma unroll
        for (int u = SLOTS - 1; u >= 0; --u) {
            const uint32_t b = __ballot_sync(0xffffffffu, front[u] == best);
            holders += __popc(b);
            if (b) { slot = u; wl = __ffs(b) - 1; }
        }
        if (holders > 1) {
            // equal scores: shallower first, then the smaller path key ((depth, key) identifies a candidate)
            unsigned long long t = 0ull;
            int tu = 0;
#pragma unroll
            for (int u = 0; u < SLOTS; ++u) {
                const int depth = (int)(meta[u] & 15u) + 1;
                const unsigned long long tie = ((unsigned long long)(15 - depth) << 60) | (~(key[u] + path_digit(depth, next[u])) & 0x0fffffffffffffffull);
                if (front[u] == best && (t == 0ull || tie > t)) { t = tie; tu = u; }
            }
            bool in = mine == best;
            const uint32_t hi = __reduce_max_sync(0xffffffffu, in ? (uint32_t)(t >> 32) : 0u);
            in = in && (uint32_t)(t >> 32) == hi;
            const uint32_t lo = __reduce_max_sync(0xffffffffu, in ? (uint32_t)t : 0u);
            in = in && (uint32_t)t == lo;
            wl = __ffs(__ballot_sync(0xffffffffu, in)) - 1;
            slot = __shfl_sync(0xffffffffu, tu, wl);
        }
        // what the new node takes over from the popped entry's lane
        // (slots are chosen by bits: a comparison of u with an index would turn the registers into local memory)
        const uint32_t slot_bit = 1u << slot;
        uint32_t m = 0u, opens = 0u;
        unsigned long long pk = 0ull;
#pragma unroll
        for (int u = 0; u < SLOTS; ++u)
            if ((slot_bit >> u) & 1u) {
                opens = kid[u];
                m = (meta[u] & 15u) | ((uint32_t)next[u] << 4);
                pk = key[u];
            }
        opens = __shfl_sync(0xffffffffu, opens, wl);
        m = __shfl_sync(0xffffffffu, m, wl);
        pk = __shfl_sync(0xffffffffu, pk, wl);
        const int depth = (int)(m & 15u) + 1, rank = (int)(m >> 4);
        const int i = nc++;
        const uint32_t popped = lane == wl ? slot_bit : 0u, fresh = lane == (i & 31) ? 1u << (i >> 5) : 0u;
        const float lp_s = s_lp[min((depth - 1) * k + rank + 2, kNone)];        // both used a pop later at the earliest
        const float lp_c = s_lp[min(depth * k + 1, kNone)], lp_g = s_lp[min((depth + 1) * k, kNone)];
#pragma unroll
        for (int u = 0; u < SLOTS; ++u) {
            if ((popped >> u) & 1u) {                    // the popped entry moves on to its node's next child
                front[u] = succ[u];
                next[u] = rank + 1;
                lp_succ[u] = lp_s;
            }
            if ((fresh >> u) & 1u) {                     // the new node, and its first child
                front[u] = opens;
                score[u] = key_float(best);
                meta[u] = (uint32_t)depth | ((uint32_t)rank << 4) | ((uint32_t)(slot * 32 + wl) << 8);
                key[u] = pk + path_digit(depth, rank);
                next[u] = 0;
                lp_succ[u] = lp_c;
                lp_kid[u] = lp_g;
            }
        }
    }
    // ancestor masks: every node climbs to the root
    uint64_t anc_lo[SLOTS], anc_hi[SLOTS];
#pragma unroll
    for (int u = 0; u < SLOTS; ++u) n_parent[u * 32 + lane] = u * 32 + lane == 0 ? -1 : (int)(meta[u] >> 8);
    __syncwarp();
#pragma unroll
    for (int u = 0; u < SLOTS; ++u) {
        anc_lo[u] = anc_hi[u] = 0ull;
        const int i = u * 32 + lane;
        for (int v = i < nc ? i : -1, left = kMaxBlock + 1; v >= 0 && left > 0; v = n_parent[v], --left) {
            if (v < 64) anc_lo[u] |= 1ull << v;
            else anc_hi[u] |= 1ull << (v - 64);
        }
    }
    __syncwarp();
    if (lane == 0) out.n_nodes[s] = nc;
    const size_t o = (size_t)s * N;
    uint64_t *anc = out.anc + o * W;
#pragma unroll
    for (int u = 0; u < SLOTS; ++u) {
        const int i = u * 32 + lane;
        if (i >= N) continue;
        // padding rows: never entered by the walk, visible to themselves only
        const bool real = i < nc, inner = real && i > 0;
        const int depth = (int)(meta[u] & 15u), rank = (int)((meta[u] >> 4) & 15u);
        out.token[o + i] = inner ? s_id[(depth - 1) * k + rank] : real ? root_tok : 0;
        out.parent[o + i] = inner ? (int)(meta[u] >> 8) : -1;
        out.depth[o + i] = inner ? depth : 0;
        out.rank[o + i] = inner ? rank : 0;
        out.score[o + i] = inner ? score[u] : 0.f;
        for (int w = 0; w < W; ++w)
            anc[(size_t)i * W + w] = real ? (w == 0 ? anc_lo[u] : anc_hi[u]) : (((i >> 6) == w) ? (1ull << (i & 63)) : 0ull);
    }
}

// Programmatic launch: the block is placed while the predecessor drains and waits for it inside.
template <typename... P, typename... A>
void launch_early(void (*kernel)(P...), dim3 grid, int threads, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, args...);
}

void launch_build_tree(int batch, int N, int L, int k, const int32_t *root, const int32_t *ids, const float *lp,
                       const glance_tree &out, cudaStream_t st) {
    if (N <= 32) launch_early(build_tree_kernel<1>, dim3(batch), 32, st, N, L, k, root, ids, lp, out);
    else if (N <= 64) launch_early(build_tree_kernel<2>, dim3(batch), 32, st, N, L, k, root, ids, lp, out);
    else launch_early(build_tree_kernel<4>, dim3(batch), 32, st, N, L, k, root, ids, lp, out);
}

// ------------------------------------------------------------------------------------------
// Walk + commit in one kernel: latency-bound (a dozen rows of a few KB per layer), so it is one wave of blocks and few
// dependent steps.
//
// Grid (batch, n_layers * 2).  Every block repeats the walk -- all nodes find out in parallel whether their parent's
// decision names them (the lowest such child of a node is its successor), then one thread follows the successors -- and
// compacts its own (layer, K|V): cache row P + path[d] -> row P + d for d = 1..a.  Heads are disjoint; within a head items go
// in ascending d, and path is strictly increasing with path[d] >= d, so a row that a step overwrites can be the source of
// that step or of an earlier one only.  A block holds a thousand items in registers before it stores any, and a row
// overwritten in one trip is read by no later one.  The block that is the last of its sequence to have read seq_len
// publishes the outputs and advances the sequence state; nothing else in the kernel reads what it writes, so nobody waits
// for the copies.  Eight sequences, 13 rows each, 28 layers, with a small copy in front: 23.2 -> 6.5 us in a graph, 26.6 ->
// 18.5 us as two calls of the host (one block per head made 1.5 waves, each with a walk of warp-wide searches, a fence and a serial publication).
// ------------------------------------------------------------------------------------------
constexpr int kCommitThreads = 256;
constexpr int kCommitItems = 4;                          // 16-byte pieces a thread holds at once

__global__ void __launch_bounds__(kCommitThreads) walk_commit_kernel(WalkCommit p) {
    __shared__ int sh_path[kMaxBlock + 1];
    __shared__ int sh_a, sh_root, sh_last, sh_P;
    __shared__ int sh_am[kMaxTreeN], sh_tok[kMaxTreeN], sh_succ[kMaxTreeN];
    __shared__ int sh_page[4];
    __shared__ long long sh_src[kMaxBlock], sh_dst[kMaxBlock];    // row offsets (head 0) of step d, -1 = nothing to move
    const int s = blockIdx.x, t = threadIdx.x;
    const int L = p.B - 1;
    tc::pdl_wait();                                      // launched early; everything it reads belongs to other kernels
    // the tree, and the length.  A block counts itself in once it has read the length (acquire: not before).
    int par = -1;
    if (t == kCommitThreads - 1) {
        int P;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(P) : "l"(p.seq_len + s) : "memory");
        sh_P = P;
        sh_last = atomicAdd(&p.counters[s], 1) == (int)gridDim.y - 1;
    }
    static_assert(kMaxTreeN < kCommitThreads, "one thread per node, and one for the length");
    int nn = 0;
    if (p.argmax) {
        nn = p.n_nodes[s];
        nn = nn < 1 ? 1 : (nn > p.N ? p.N : nn);
        if (t < p.N) {
            sh_am[t] = p.argmax[(size_t)s * p.N + t];
            sh_tok[t] = p.token[(size_t)s * p.N + t];
            par = p.parent[(size_t)s * p.N + t];
            sh_succ[t] = kMaxTreeN;
        }
    }
    __syncthreads();
    const int P = sh_P;
    const int32_t *pt = p.page_table + (size_t)s * p.geom.max_pages_per_seq;
    if (t >= kCommitThreads - 4) {                       // the pages of rows P .. P + N - 1
        const int j = t - (kCommitThreads - 4), pg = P / kPage + j;
        sh_page[j] = P >= 0 && pg < p.geom.max_pages_per_seq && j * kPage <= p.N + kPage ? pt[pg] : -1;
    }
    if (p.argmax && t >= 1 && t < nn && par >= 0 && par < p.N && sh_tok[t] == sh_am[par]) atomicMin(&sh_succ[par], t);
    __syncthreads();
    if (t == 0) {
        if (p.argmax) {
            int v = 0, a = 0;
            sh_path[0] = 0;
            while (a < L && sh_succ[v] < kMaxTreeN) {
                v = sh_succ[v];
                sh_path[++a] = v;
            }
            sh_a = a;
            sh_root = sh_am[v];
        } else {
            int len = p.forced_len[s];
            len = len < 1 ? 1 : (len > p.B ? p.B : len);
            int prev = -1;
            bool ok = true;
            for (int d = 0; d < len; ++d) {
                int v = p.forced_path[(size_t)s * p.B + d];
                if (v <= prev || v >= p.N || (d == 0 && v != 0)) ok = false;
                prev = v;
                sh_path[d] = ok ? v : d;
            }
            if (!ok) set_status(p.status, GLANCE_E_BOUNDS);
            sh_a = len - 1;
            sh_root = p.forced_root[s];
        }
    }
    __syncthreads();
    const int a = sh_a;
    const int layer = blockIdx.y >> 1, kv = blockIdx.y & 1;
    if (t < a) {
        const int d = t + 1, from = P % kPage + sh_path[d], to = P % kPage + d;      // relative to the first page
        const int spage = P < 0 ? -1 : sh_page[from / kPage], dpage = P < 0 ? -1 : sh_page[to / kPage];
        const bool ok = spage >= 0 && spage < p.geom.n_pages && dpage >= 0 && dpage < p.geom.n_pages;
        if (!ok) set_status(p.status, GLANCE_E_BOUNDS);
        sh_src[t] = ok ? (long long)p.geom.row(spage, kv, 0, from % kPage) : -1;
        sh_dst[t] = ok ? (long long)p.geom.row(dpage, kv, 0, to % kPage) : -1;
    }
    if (sh_last && t < 32) {
        // every block of the sequence has read the length: publish
        const int d = t;
        if (d < p.B) {
            if (p.path) p.path[(size_t)s * p.B + d] = d <= a ? sh_path[d] : -1;
            if (p.out_tokens)
                p.out_tokens[(size_t)s * p.B + d] = d < a ? (p.argmax ? sh_tok[sh_path[d + 1]] : -1) : d == a ? sh_root : -1;
        }
        if (t == 0) {
            if (p.accept_len) p.accept_len[s] = a;
            p.feat_count[s] = a + 1;
            p.seq_len[s] = P + a + 1;
            p.root[s] = sh_root;
            p.counters[s] = 0;
        }
    }
    __syncthreads();

    // compaction
    bf16 *base = p.kv_pool + (size_t)layer * p.geom.layer_stride();
    const int chunks = p.geom.head_dim * 2 / 16;        // 16-byte pieces per row
    const int per_head = a * chunks, items = per_head * p.geom.n_kv_heads;
    const size_t head_step = (size_t)kPage * p.geom.head_dim;
    for (int it0 = 0; it0 < items; it0 += kCommitThreads * kCommitItems) {
        int4 val[kCommitItems];
        int4 *dst[kCommitItems];
#pragma unroll
        for (int u = 0; u < kCommitItems; ++u) {
            const int it = it0 + u * kCommitThreads + t;
            dst[u] = nullptr;
            if (it < items) {
                const int head = it / per_head, rem = it - head * per_head, d = rem / chunks, c = rem - d * chunks;
                const long long from = sh_src[d], to = sh_dst[d];
                if (from != to) {                        // (both -1: refused above)
                    val[u] = *(reinterpret_cast<const int4 *>(base + from + head * head_step) + c);
                    dst[u] = reinterpret_cast<int4 *>(base + to + head * head_step) + c;
                }
            }
        }
        __syncthreads();                                // all sources of these items are in registers
#pragma unroll
        for (int u = 0; u < kCommitItems; ++u)
            if (dst[u]) *dst[u] = val[u];
        __syncthreads();
    }

    // features of the accepted path (every tap slice): hidden[path[i]] -> feat[i], in 16-byte pieces shared out over
    // all blocks of the sequence (nothing reads feat before the next draft pass)
    const int CH = p.H >> 3;                            // H is a multiple of 64
    const int per_tap = (a + 1) * CH;
    const int total = p.n_taps * per_tap;
    for (int it = blockIdx.y * blockDim.x + t; it < total; it += gridDim.y * blockDim.x) {
        const int tap = it / per_tap, rem = it - tap * per_tap;
        const int i = rem / CH, c = rem - i * CH;
        const int4 *src = reinterpret_cast<const int4 *>(p.hidden + ((size_t)tap * p.batch * p.N + (size_t)s * p.N + sh_path[i]) * p.H) + c;
        int4 *dst = reinterpret_cast<int4 *>(p.feat + ((size_t)tap * p.batch * p.B + (size_t)s * p.B + i) * p.H) + c;
        *dst = *src;
    }
}

void launch_walk_commit(const WalkCommit &p, cudaStream_t st) {
    launch_early(walk_commit_kernel, dim3(p.batch, p.n_layers * 2), kCommitThreads, st, p);
}

}  // namespace glance
