"""The work that users of this framework have it do, as cases that can be prepared, run, checked and timed.

Every case is a plain dict with a "kind":

  tree     glance_build_tree alone: the candidate tree of one sequence or a small batch.  The smallest call.
  commit   glance_accept_commit alone: the walk and the in-place compaction of the paged cache.
  topk     glance_topk_static: top-k + log-softmax of a caller's logits, for callers without a workspace.
  draft    glance_draft_block: one pass of the block head over a filled context.
  round    a whole speculative round (draft, tree, verify, commit), replayed as one CUDA graph.
  decode   plain decoding through the same calls: a verify pass over single-node trees, then commit, as one CUDA graph.
  prefill  glance_prefill of an image prefix and a text part, possibly behind earlier positions.

Model widths are the repository's own (tiny, small, 7b); a model's depth, the sequences' lengths, the batch and the
round's shape (block, top-k, tree rows) belong to the case.  Weights are random with the repository's recipe, the
context's K/V rows have the scale that the model's own projections give, candidates follow the controlled marginals.

What a walk accepts is given by the case and not by the model: the commit takes decisions that follow one path of the
tree, as a caller with a sampler of its own passes them.  With random weights the arg-max of a row is decided by
margins of the size of the rounding error, so token ids that such margins decide are not among the outputs; the
logits, log-probabilities, hidden states and cache rows that they come from are.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2609_00355_b200 import binding, synth

# model widths: n_layers is the full depth, a case may take fewer layers
WIDTHS = {name: {k: getattr(synth.CONFIGS[name], k) for k in
                 ("n_layers", "hidden", "n_q_heads", "n_kv_heads", "head_dim", "ffn", "vocab")}
          for name in ("tiny", "small", "7b")}
THETA, EPS, PAGE = 1e6, 1e-6, 64


def listed():
    return [
        # one sequence's tree at the benchmark's shape: a single small launch, all latency
        dict(name="tree", kind="tree", batch=1, block=16, topk=8, nodes=64),
        # eight sequences that accept long paths at the largest tree: the most rows that a commit moves
        dict(name="commit-batch8", kind="commit", model="7b", layers=28, batch=8, block=16, nodes=128, accept=13, lo=1024, hi=4096),
        # a caller's logits at the full vocabulary
        dict(name="topk-static", kind="topk", batch=1, block=16, topk=8, vocab=152064),
        # the drafter alone: one-layer head over an image + text context
        dict(name="draft-7b", kind="draft", model="7b", taps=1, batch=1, block=16, topk=8, nodes=64, lo=1536, hi=1536),
        # a small model, odd context length: launches and latency count
        dict(name="round-small", kind="round", model="small", layers=8, taps=1, batch=1, block=8, topk=4, nodes=32, lo=701, hi=701, accept=3, sample=False),
        # plain greedy decoding of one sequence: one row through the whole model
        dict(name="decode-7b", kind="decode", model="7b", layers=28, batch=1, lo=1536, hi=1536),
        # the benchmark's round: one sequence, 64 tree rows
        dict(name="round-7b", kind="round", model="7b", layers=28, taps=1, batch=1, block=16, topk=8, nodes=64, lo=1536, hi=1536, accept=4, sample=False),
        # three sequences in sampling mode with the paper's five-layer multi-tap head and the entropy log
        dict(name="round-7b-taps5", kind="round", model="7b", layers=28, taps=5, batch=3, block=16, topk=8, nodes=48, lo=900, hi=2100, accept=3, sample=True),
        # a document-sized image prefix and the widest tree
        dict(name="round-long", kind="round", model="7b", layers=28, taps=1, batch=1, block=16, topk=8, nodes=128, lo=8704, hi=8704, accept=2, sample=False),
        # small-batch serving: eight ragged sequences
        dict(name="round-batch8", kind="round", model="7b", layers=28, taps=1, batch=8, block=16, topk=8, nodes=64, lo=1024, hi=4096, accept=3, sample=False),
        # a new request at the benchmark's shape: image rows, then the text
        dict(name="prefill-7b", kind="prefill", model="7b", layers=28, taps=1, nodes=64, prior=0, n_img=1280, n_txt=256),
        # a new request of the small model, ragged in both parts
        dict(name="prefill-small", kind="prefill", model="small", layers=8, taps=1, nodes=32, prior=0, n_img=577, n_txt=131),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["tree", "commit", "topk", "draft", "round", "round", "round", "decode", "prefill", "prefill"])
    block = rng.choice([4, 8, 13, 16])
    if kind == "tree":
        return dict(kind=kind, batch=rng.randint(1, 8), block=block, topk=rng.randint(2, 16), nodes=_log_int(rng, 8, 128))
    if kind == "topk":
        vocab, topk, batch = _log_int(rng, 1000, 152064), rng.randint(1, 16), rng.randint(1, 4)
        while batch > 1 and batch * (block - 1) * -(-vocab // 1024) * (8 * topk + 8) > 1000000:
            batch -= 1
        return dict(kind=kind, batch=batch, block=block, topk=topk, vocab=vocab)
    model = rng.choice(["tiny", "small", "7b", "7b"])
    layers = _log_int(rng, 2, WIDTHS[model]["n_layers"])
    if kind == "commit":
        nodes = _log_int(rng, 2 * block + 2, 128)
        lo = _log_int(rng, 64, 2048)
        return dict(kind=kind, model=model, layers=layers, batch=rng.randint(1, 8), block=block, nodes=nodes,
                    accept=rng.randint(0, block - 1), lo=lo, hi=2 * lo)
    if kind == "decode":
        batch = rng.choice([1, 1, 2, 5])
        lo = _log_int(rng, 64, 6000)
        return dict(kind=kind, model=model, layers=layers, batch=batch, lo=lo, hi=lo if batch == 1 else lo + lo // 2)
    taps = rng.choice([1, 1, 1, 2]) if layers >= 2 else 1
    if kind == "prefill":
        nodes = rng.choice([16, 32, 64, 128])
        most = min(4096, nodes * 24 * 28 // layers, 1536 * 28 // layers)
        total = _log_int(rng, 24, most)
        n_img = rng.choice([0, total // 2, (3 * total) // 4, total - 1])
        return dict(kind=kind, model=model, layers=layers, taps=taps, nodes=nodes, prior=rng.choice([0, 0, rng.randint(1, 1500)]),
                    n_img=n_img, n_txt=total - n_img)
    batch = rng.choice([1, 1, 1, 2, 4, 8])
    lo = _log_int(rng, 64, 8704 if batch == 1 else 2048)
    hi = lo if batch == 1 else 2 * lo
    topk, nodes = rng.randint(2, 12), _log_int(rng, 8, 128 if batch <= 4 else 64)
    if kind == "draft":
        return dict(kind=kind, model=model, taps=taps, batch=batch, block=block, topk=topk, nodes=nodes, lo=lo, hi=hi)
    return dict(kind=kind, model=model, layers=layers, taps=taps, batch=batch, block=block, topk=topk, nodes=nodes, lo=lo, hi=hi,
                accept=rng.randint(0, min(block - 1, 4)), sample=rng.random() < 0.25)


# ---- inputs --------------------------------------------------------------------------------------------------------
def _config(c):
    """The case's model and round shape as the repository's configuration record."""
    w = dict(WIDTHS[c.get("model", "tiny")])
    taps = c.get("taps", 1)
    w["n_layers"] = c.get("layers", max(2, taps) if c["kind"] == "draft" else 1)
    head_taps = tuple(i * (w["n_layers"] - 1) // (taps - 1) for i in range(taps)) if taps > 1 else ()
    return synth.RoundConfig(name="case", n_img=0, n_txt=0, block_B=c.get("block", 16), topk=c.get("topk", 1),
                             tree_N=c.get("nodes", 1), p_m=0.8, rounds=1, batch=c.get("batch", 1), rms_eps=EPS,
                             rope_theta=THETA, head_taps=head_taps, **w)


def _lengths(c):
    """Committed positions of every sequence: the case's, whatever the seed."""
    return [int(v) for v in np.random.default_rng((c["lo"], c["hi"], 1)).integers(c["lo"], c["hi"] + 1, size=c.get("batch", 1))]


def _last_commits(cfg, lens):
    """Rows that each sequence committed last: between one and a whole block."""
    return np.minimum(np.random.default_rng((sum(lens), 2)).integers(1, cfg.block_B + 1, size=cfg.batch), lens).astype(np.int32)


def _normal(shape, std, gen):
    return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(0.0, std, generator=gen)


def _gain(n, gen):
    return (torch.rand(n, device="cuda", generator=gen) * 0.5 + 0.75).to(torch.bfloat16)


def _weights(cfg, seed, read=True, target_layers=True):
    """(target, head) dicts.  `read` False: the call never reads the model, so every matrix is a view of one buffer;
    `target_layers` False: the call reads the head and the vocabulary matrices only."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    H, F, V, d = cfg.hidden, cfg.ffn, cfg.vocab, cfg.head_dim
    qkv, std = (cfg.n_q_heads + 2 * cfg.n_kv_heads) * d, 0.02
    if not read:
        buf = torch.zeros(max(V, 2 * F, qkv) * H, dtype=torch.bfloat16, device="cuda")
        mat, vec = (lambda r, k: buf[: r * k].view(r, k)), (lambda n: buf[:n])
    else:
        mat, vec = (lambda r, k: _normal((r, k), std, gen)), (lambda n: _gain(n, gen))
    layer = lambda: {"ln1": vec(H), "wqkv": mat(qkv, H), "wo": mat(H, cfg.n_q_heads * d), "ln2": vec(H), "wgu": mat(2 * F, H),
                     "wd": mat(H, F)}
    head_layer = lambda: dict(layer(), ctx_norm=vec(H))
    head = dict(head_layer(), mask_embed=mat(1, H)[0], final_norm=vec(H), more=[head_layer() for _ in range(cfg.head_layers - 1)])
    target = {"embed": mat(V, H), "lm_head": mat(V, H), "final_norm": vec(H)}
    if read and target_layers:
        target["layers"] = [layer() for _ in range(cfg.n_layers)]
    else:
        target["layers"] = [{k: head[k] for k in ("ln1", "wqkv", "wo", "ln2", "wgu", "wd")}] * cfg.n_layers
    return target, head


def _fill_context(eng, cfg, lens, seed):
    """Committed context of every sequence: K/V rows of the scale that the projections give, pending root token, the
    tapped features of the rows committed last."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 1000003)
    rng = np.random.default_rng((seed, 2))
    sigma = 0.02 * math.sqrt(cfg.hidden)
    pps = eng.pages_per_seq
    # pages handed out in order, as by a freshly started allocator
    eng.page_table.copy_(torch.arange(cfg.batch * pps, dtype=torch.int32, device="cuda").view(cfg.batch, pps))
    eng.kv_pool.normal_(0.0, sigma, generator=gen)
    eng.head_kv_all.normal_(0.0, sigma, generator=gen)
    eng.feat_all.normal_(0.0, 1.0, generator=gen)
    eng.seq_len.copy_(torch.tensor(lens, dtype=torch.int32))
    eng.root.copy_(torch.from_numpy(rng.integers(0, cfg.vocab, size=cfg.batch).astype(np.int32)))
    eng.feat_count.copy_(torch.from_numpy(_last_commits(cfg, lens)))


def _candidates(cfg, seed):
    """Candidate ids and log-probabilities [batch][L][k] of the controlled marginals, one match probability a sequence."""
    rng = np.random.default_rng((seed, 3))
    ids = np.stack([np.stack([rng.choice(cfg.vocab, size=cfg.topk, replace=False) for _ in range(cfg.L)]) for _ in range(cfg.batch)])
    lp = np.stack([synth.controlled_marginals(float(rng.uniform(0.4, 0.9)), cfg.topk, cfg.L) for _ in range(cfg.batch)])
    # no two depths alike, as with drafted marginals; still non-increasing in rank
    lp = lp - np.sort(rng.uniform(0.0, 0.05, size=lp.shape), axis=-1)
    return ids.astype(np.int32), lp.astype(np.float32)


def _decisions(parent, token, n_nodes, accept, vocab, rng):
    """Decisions [N] that walk one random path of at most `accept` edges and then leave the tree; the path's nodes."""
    out = rng.integers(0, vocab, size=len(token)).astype(np.int32)
    path, v = [0], 0
    while True:
        kids = [i for i in range(1, n_nodes) if parent[i] == v]
        if len(path) > accept or not kids:
            taken = {int(token[i]) for i in kids}
            while int(out[v]) in taken:
                out[v] = (out[v] + 1) % vocab
            return out, path
        v_next = kids[0] if rng.random() < 0.7 else int(rng.choice(kids))
        out[v], v = token[v_next], v_next
        path.append(v)


def _commit_tree(N, L, accept, vocab, rng):
    """A tree whose accepted path sits behind the nodes 1..accept of a branch that was drafted as more likely, so that
    every accepted row moves and no row that is read is also written."""
    a = min(accept, L, (N - 1) // 2)
    token = rng.choice(vocab, size=N, replace=False).astype(np.int32)
    parent, depth = np.full(N, -1, np.int32), np.zeros(N, np.int32)
    for i in range(1, a + 1):
        parent[i], depth[i] = i - 1, i
    path = [0] + sorted(int(v) for v in rng.choice(np.arange(a + 1, N), size=a, replace=False))
    for d in range(1, a + 1):
        parent[path[d]], depth[path[d]] = path[d - 1], d
    for i in range(a + 1, N):
        if i not in path:
            parent[i], depth[i] = 0, 1
    return token, parent, depth, path


@functools.lru_cache(maxsize=None)
def _stream():
    """One stream for every state of this process, as a serving loop has one: passes follow one another on it."""
    return torch.cuda.Stream()


def _engine(cfg, weights, lens, extra):
    return binding.Engine(cfg, weights[0], weights[1], batch=cfg.batch, stream=_stream(), max_len=max(lens) + extra + PAGE)


def _rows(pool, seq, pps, first, count):
    """Views of the cache rows first..first+count-1 of one sequence in a pool [layers][pages][2][Hkv][64][d]."""
    out = []
    while count > 0:
        page, slot = seq * pps + first // PAGE, first % PAGE
        n = min(count, PAGE - slot)
        out.append(pool[:, page, :, :, slot : slot + n])
        first, count = first + n, count - n
    return out


def _span(pool, count):
    """Views of the cache rows 0..count-1 of sequence 0 (pages in order)."""
    full, rest = count // PAGE, count % PAGE
    return ([pool[:, :full]] if full else []) + ([pool[:, full, :, :, :rest]] if rest else [])


def prepare(case, seed):
    c, kind = case, case["kind"]
    with torch.cuda.stream(_stream()):
        if kind == "topk":
            gen = torch.Generator(device="cuda")
            gen.manual_seed(seed)
            L = c["block"] - 1
            return dict(kind=kind, k=c["topk"], logits=torch.randn(c["batch"], c["block"], c["vocab"], device="cuda", generator=gen) * 1.2,
                        ids=torch.zeros(c["batch"], L, c["topk"], dtype=torch.int32, device="cuda"),
                        lp=torch.zeros(c["batch"], L, c["topk"], device="cuda"))
        cfg = _config(c)
        rng = np.random.default_rng((seed, 4))
        if kind == "tree":
            eng = _engine(cfg, _weights(cfg, seed, read=False), [0], cfg.tree_N)
            ids, lp = _candidates(cfg, seed)
            eng.root.copy_(torch.from_numpy(rng.integers(0, cfg.vocab, size=cfg.batch).astype(np.int32)))
            return dict(kind=kind, eng=eng, ids=torch.from_numpy(ids).cuda(), lp=torch.from_numpy(lp).cuda())
        if kind == "prefill":
            eng = _engine(cfg, _weights(cfg, seed), [c["prior"] + c["n_img"] + c["n_txt"]], cfg.tree_N)
            _fill_context(eng, cfg, [c["prior"]], seed)
            img, ids = synth.make_context(cfg, "cuda", seed=seed + 1, n_img=c["n_img"], n_txt=c["n_txt"])
            total = c["prior"] + c["n_img"] + c["n_txt"]
            return dict(kind=kind, eng=eng, img=img, ids=ids, seq_len0=eng.seq_len.clone(),
                        out=dict(kv=_span(eng.kv_pool, total), head_kv=_span(eng.head_kv_all, total), seq_len=eng.seq_len,
                                 feat_count=eng.feat_count))
        lens = _lengths(c)
        reads = kind != "commit"
        eng = _engine(cfg, _weights(cfg, seed, read=reads, target_layers=kind != "draft"), lens, max(cfg.tree_N, cfg.block_B))
        _fill_context(eng, cfg, lens, seed)
        if kind == "draft":
            logits = torch.zeros(cfg.batch * cfg.block_B, cfg.vocab, device="cuda")
            count = eng.feat_count.tolist()
            return dict(kind=kind, eng=eng, logits=logits,
                        out=dict(lp=eng.topk_lp, logits=logits,
                                 head_kv=[_rows(eng.head_kv_all, s, eng.pages_per_seq, lens[s] - count[s], count[s]) for s in range(cfg.batch)]))
        state = dict(kind=kind, eng=eng, snap=eng.snapshot_state(), lens=lens)
        N = cfg.tree_N
        if kind == "commit":
            eng.hidden_all.normal_(0.0, 1.0, generator=torch.Generator(device="cuda").manual_seed(seed + 5))
            made = [_commit_tree(N, cfg.L, c["accept"], cfg.vocab, rng) for _ in range(cfg.batch)]
            eng.tree.token.copy_(torch.from_numpy(np.stack([m[0] for m in made])))
            eng.tree.parent.copy_(torch.from_numpy(np.stack([m[1] for m in made])))
            eng.tree.depth.copy_(torch.from_numpy(np.stack([m[2] for m in made])))
            eng.tree.n_nodes.fill_(N)
            walks = []
            for token, _, _, path in made:
                dec = rng.integers(0, cfg.vocab, size=N).astype(np.int32)
                for u, v in zip(path, path[1:]):
                    dec[u] = token[v]
                while int(dec[path[-1]]) in set(token.tolist()):
                    dec[path[-1]] = (dec[path[-1]] + 1) % cfg.vocab
                walks.append((dec, path))
        elif kind == "decode":
            eng.tree.token.copy_(eng.root[:, None])
            eng.tree.anc.fill_(1)
            walks = [(rng.integers(0, cfg.vocab, size=1).astype(np.int32), [0]) for _ in lens]
        else:
            ids, lp = _candidates(cfg, seed)
            state["ids"], state["lp"] = torch.from_numpy(ids).cuda(), torch.from_numpy(lp).cuda()
            eng.glance_build_tree(state["ids"], state["lp"])
            parent, token, nodes = eng.tree.parent.cpu().numpy(), eng.tree.token.cpu().numpy(), eng.tree.n_nodes.tolist()
            walks = [_decisions(parent[s], token[s], nodes[s], c["accept"], cfg.vocab, rng) for s in range(cfg.batch)]
        state["decisions"] = torch.from_numpy(np.stack([w[0] for w in walks])).cuda()
        keep = 1 + (len(walks[0][1]) - 1 if kind == "commit" else 0 if kind == "decode" else min(c["accept"], N - 1))
        state["sample_seed"] = seed if c.get("sample") else None
        out = dict(accept_len=eng.accept_len, path=eng.path, tokens=eng.out_tokens, seq_len=eng.seq_len, root=eng.root,
                   feat_count=eng.feat_count, feat=eng.feat_all,
                   kv=[_rows(eng.kv_pool, s, eng.pages_per_seq, lens[s], keep) for s in range(cfg.batch)])
        if kind != "commit":
            state["logits"] = out["logits"] = torch.zeros(cfg.batch * N, cfg.vocab, device="cuda")
            out["hidden"] = eng.hidden_all
        if kind == "round":
            out["lp"] = eng.topk_lp
            if c.get("sample"):
                out["entropy"] = torch.zeros(cfg.batch, device="cuda")
                eng.glance_log_root_entropy(out["entropy"])
            count = state["snap"][3].tolist()
            out["head_kv"] = [_rows(eng.head_kv_all, s, eng.pages_per_seq, lens[s] - count[s], count[s]) for s in range(cfg.batch)]
        state["out"] = out
        if kind in ("round", "decode"):
            _step(state)                                     # kernel attributes and descriptors are set up on first use
            state["graph"] = eng.capture(lambda: _step(state))
        return state


def _step(state):
    """The state of before the step, then the calls of one step."""
    eng, kind = state["eng"], state["kind"]
    eng.restore_state(state["snap"])
    if kind == "round":
        eng.glance_draft_block()
        eng.glance_build_tree(state["ids"], state["lp"])
    if kind in ("round", "decode"):
        if state["sample_seed"] is not None:
            eng.glance_verify_tree_sample(state["sample_seed"], 1.0, logits_dbg=state["logits"])
        else:
            eng.glance_verify_tree(logits_dbg=state["logits"])
    eng.glance_accept_commit(argmax=state["decisions"])


def run(state):
    kind = state["kind"]
    with torch.cuda.stream(_stream()):
        if kind == "topk":
            rc = binding.glance_topk_static(state["logits"], state["k"], state["ids"], state["lp"])
            if rc != 0:
                raise RuntimeError("glance_topk_static: %d" % rc)
            return dict(ids=state["ids"], lp=state["lp"])
        eng = state["eng"]
        if kind == "tree":
            eng.glance_build_tree(state["ids"], state["lp"])
            t = eng.tree
            return dict(token=t.token, parent=t.parent, depth=t.depth, rank=t.rank, score=t.score, anc=t.anc, n_nodes=t.n_nodes)
        if kind == "draft":
            eng.glance_draft_block(logits_dbg=state["logits"])
        elif kind == "prefill":
            eng.seq_len.copy_(state["seq_len0"])
            eng.prefill_context(0, state["img"], state["ids"])
        elif kind == "commit":
            eng.seq_len.copy_(state["snap"][0])
            eng.glance_accept_commit(argmax=state["decisions"])
        else:
            state["graph"].replay()
        return state["out"]


# ---- what a pass cannot do without, and how close results have to be ----------------------------------------------------
def work(case):
    c, kind = case, case["kind"]
    if kind == "topk":
        n = c["batch"] * (c["block"] - 1)
        return dict(bytes=n * (4 * c["vocab"] + 8 * c["topk"]), flops=4 * n * c["vocab"])
    cfg = _config(c)
    H, F, V, d, Hq, Hkv, N, B = cfg.hidden, cfg.ffn, cfg.vocab, cfg.head_dim, cfg.n_q_heads, cfg.n_kv_heads, cfg.tree_N, cfg.block_B
    if kind == "tree":
        return dict(bytes=cfg.batch * (8 * cfg.L * cfg.topk + N * (20 + 8 * ((N + 63) // 64))), flops=0)
    row = 4 * Hkv * d                                        # bytes of one position's K and V in one layer
    mats = (Hq + 2 * Hkv) * d * H + H * Hq * d + 3 * F * H   # weights of one layer
    ctx = (c["lo"] + c["hi"]) // 2 * cfg.batch if kind != "prefill" else 0
    if kind == "commit":
        moved = cfg.batch * (min(c["accept"], cfg.L, (N - 1) // 2) * row * cfg.n_layers + (c["accept"] + 1) * 2 * H)
        return dict(bytes=2 * moved, flops=0)
    if kind == "prefill":
        T = c["n_img"] + c["n_txt"]
        keys = T * c["prior"] + T * (T + 1) // 2
        by = 2 * (cfg.n_layers * mats + cfg.head_layers * 2 * Hkv * d * H + V * H) + T * 2 * H + (cfg.n_layers * (T + c["prior"]) + cfg.head_layers * T) * row
        return dict(bytes=by, flops=2 * T * (cfg.n_layers * mats + cfg.head_layers * 2 * Hkv * d * H) + 4 * cfg.n_layers * keys * Hq * d + 2 * V * H)
    by = fl = 0
    if kind in ("draft", "round"):
        R = cfg.batch * B
        by += 2 * (cfg.head_layers * mats + V * H) + cfg.head_layers * ctx * row + (4 * R * V if kind == "draft" else 0)
        fl += 2 * R * (cfg.head_layers * mats + V * H) + 4 * cfg.head_layers * B * (ctx + cfg.batch * B) * Hq * d
    if kind in ("decode", "round"):
        R = cfg.batch * N
        by += 2 * (cfg.n_layers * mats + V * H) + cfg.n_layers * ctx * row + 4 * R * V
        fl += 2 * R * (cfg.n_layers * mats + V * H) + 4 * cfg.n_layers * N * (ctx + cfg.batch * N) * Hq * d
    return dict(bytes=by, flops=fl)


def tolerance(case):
    if case["kind"] in ("tree", "commit"):
        return "exact"                                       # whole numbers, one fp32 add a node, bytes that move
    if case["kind"] == "topk":
        return {"rel": 1e-6, "max": 1e-5}                    # fp32 log-sum-exp in another order
    # bf16 operands and cache rows, fp32 sums: up to 1.5e-2 off 64 bits after 28 layers, and two such results differ by
    # up to twice that
    return {"rel": 0.03, "max": 0.4}


# ---- the same in 64 bits, plain torch ----------------------------------------------------------------------------------
def _norm64(x, gain):
    return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + EPS) * gain.double()


def _rope64(x, pos):
    """x [R][heads][d] rotated by the rows' positions (pairs i, i + d/2)."""
    half = x.shape[-1] // 2
    ang = pos.double()[:, None] * THETA ** (-torch.arange(half, device=x.device, dtype=torch.float64) / half)
    cs, sn = ang.cos()[:, None], ang.sin()[:, None]
    a, b = x[..., :half], x[..., half:]
    return torch.cat([a * cs - b * sn, b * cs + a * sn], -1)


def _attend64(q, k, v, mask):
    """q [T][Hq][d] against k, v [n][Hkv][d]; mask [T][n] (True: visible) or None."""
    T, Hq, d = q.shape
    Hkv = k.shape[1]
    out = torch.empty_like(q)
    for h in range(Hq):
        s = q[:, h] @ k[:, h * Hkv // Hq].T / math.sqrt(d)
        if mask is not None:
            s.masked_fill_(~mask, -math.inf)
        out[:, h] = torch.softmax(s, -1) @ v[:, h * Hkv // Hq]
    return out.reshape(T, Hq * d)


def _qkv64(cfg, n, w, pos):
    y = (n @ w["wqkv"].double().T).view(n.shape[0], -1, cfg.head_dim)
    q, k, v = y.split([cfg.n_q_heads, cfg.n_kv_heads, cfg.n_kv_heads], 1)
    return _rope64(q, pos), _rope64(k, pos), v


def _rest64(x, att, w):
    x = x + att @ w["wo"].double().T
    g, u = (_norm64(x, w["ln2"]) @ w["wgu"].double().T).chunk(2, -1)
    return x + (g * torch.sigmoid(g) * u) @ w["wd"].double().T


def _logits64(n, lm_head):
    return torch.cat([n @ part.double().T for part in lm_head.split(16384)], 1)


def _context(pool_layer, seq, pps, count):
    """K, V [count][Hkv][d] of one sequence from a pool layer [pages][2][Hkv][64][d] (pages in order)."""
    pages = pool_layer[seq * pps : (seq + 1) * pps]
    k, v = (pages[:, i].transpose(1, 2).reshape(-1, pages.shape[2], pages.shape[4])[:count].double() for i in (0, 1))
    return k, v


def _draft64(cfg, tw, hw, eng, lens, root, feat, count):
    """(log-probabilities of the k best [batch][L][k], logits, refreshed head rows) of the draft pass."""
    B = cfg.block_B
    x = hw["mask_embed"].double().expand(cfg.batch, B, cfg.hidden).clone()
    x[:, 0] = tw["embed"][root.long()].double()
    x = x.reshape(cfg.batch * B, -1)
    pos = torch.cat([torch.arange(P, P + B, device="cuda") for P in lens])
    fresh = [[] for _ in lens]
    for i, w in enumerate([hw] + hw["more"]):
        q, k, v = _qkv64(cfg, _norm64(x, w["ln1"]), w, pos)
        att = []
        for s, P in enumerate(lens):
            at = torch.arange(P - count[s], P, device="cuda")
            _, fk, fv = _qkv64(cfg, _norm64(feat[i, s, : count[s]].double(), w["ctx_norm"]), w, at)
            ck, cv = _context(eng.head_kv_all[i], s, eng.pages_per_seq, P - count[s])
            fresh[s].append(torch.stack([fk, fv]).transpose(1, 2))       # [2][Hkv][count][d]
            r = slice(s * B, (s + 1) * B)
            att.append(_attend64(q[r], torch.cat([ck, fk, k[r]]), torch.cat([cv, fv, v[r]]), None))
        x = _rest64(x, torch.cat(att), w)
    logits = _logits64(_norm64(x, hw["final_norm"]), tw["lm_head"])
    lp = torch.log_softmax(logits, -1).view(cfg.batch, B, -1)[:, 1:].topk(cfg.topk, -1).values
    return lp, logits, [torch.stack(f) for f in fresh]


def _target64(cfg, tw, eng, lens, x, pos, masks):
    """(tapped hidden states, per layer new K and V, last residual) of a pass of T rows for each sequence."""
    T = x.shape[0] // len(lens)
    taps, hidden, kv = cfg.head_taps or (cfg.n_layers - 1,), {}, []
    for l, w in enumerate(tw["layers"]):
        q, k, v = _qkv64(cfg, _norm64(x, w["ln1"]), w, pos)
        att = []
        for s, P in enumerate(lens):
            ck, cv = _context(eng.kv_pool[l], s, eng.pages_per_seq, P)
            r = slice(s * T, (s + 1) * T)
            seen = torch.cat([torch.ones(T, P, dtype=torch.bool, device="cuda"), masks[s]], 1)
            att.append(_attend64(q[r], torch.cat([ck, k[r]]), torch.cat([cv, v[r]]), seen))
        x = _rest64(x, torch.cat(att), w)
        kv.append(torch.stack([k, v]))                       # [2][rows][Hkv][d]
        hidden[l] = x
    return torch.stack([hidden[t] for t in taps]), torch.stack(kv), x


def _as_rows(block, first):
    """Rows [layers][2][Hkv][count][d] cut at the page boundaries that _rows() cuts at."""
    out, done = [], 0
    while done < block.shape[3]:
        n = min(block.shape[3] - done, PAGE - (first + done) % PAGE)
        out.append(block[:, :, :, done : done + n])
        done += n
    return out


def _as_span(prior, block, eng_pool, total):
    """The whole sequence's rows in the layout of _span(): earlier rows as they were, then `block`."""
    pages = -(-total // PAGE)
    rows = eng_pool[:, :pages].double().permute(0, 2, 3, 1, 4, 5).flatten(3, 4).clone()      # [layers][2][Hkv][pos][d]
    rows[:, :, :, prior:total] = block
    rows = rows.unflatten(3, (pages, PAGE)).permute(0, 3, 1, 2, 4, 5)
    full, rest = total // PAGE, total % PAGE
    return ([rows[:, :full]] if full else []) + ([rows[:, full, :, :, :rest]] if rest else [])


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("tree", "commit"):
        return None                                          # compared bit by bit
    state = prepare(case, seed)
    torch.cuda.synchronize()
    if kind == "topk":
        lp = torch.log_softmax(state["logits"][:, 1:].double(), -1).topk(c["topk"], -1)
        return dict(ids=lp.indices, lp=lp.values)
    eng, cfg = state["eng"], state["eng"].cfg
    tw, hw = eng._keep
    if kind == "draft":
        lens, count = eng.seq_len.tolist(), eng.feat_count.tolist()
        lp, logits, fresh = _draft64(cfg, tw, hw, eng, lens, eng.root, eng.feat_all, count)
        return dict(lp=lp, logits=logits, head_kv=[_as_rows(f, lens[s] - count[s]) for s, f in enumerate(fresh)])
    if kind == "prefill":
        prior, T = c["prior"], c["n_img"] + c["n_txt"]
        x = torch.cat([state["img"].double(), tw["embed"][state["ids"].long()].double()])
        pos = torch.arange(prior, prior + T, device="cuda")
        hidden, kv, _ = _target64(cfg, tw, eng, [prior], x, pos, [torch.ones(T, T, dtype=torch.bool, device="cuda").tril()])
        head = [torch.stack(_qkv64(cfg, _norm64(hidden[i], w["ctx_norm"]), w, pos)[1:]) for i, w in enumerate([hw] + hw["more"])]
        return dict(kv=_as_span(prior, kv.transpose(2, 3), eng.kv_pool, prior + T),
                    head_kv=_as_span(prior, torch.stack(head).transpose(2, 3), eng.head_kv_all, prior + T), seq_len=None, feat_count=None)
    lens, N = state["lens"], cfg.tree_N
    _, root, feat, count = state["snap"]
    out = dict(accept_len=None, path=None, tokens=None, seq_len=None, root=None, feat_count=None)
    eng.restore_state(state["snap"])
    if kind == "round":
        out["lp"], _, fresh = _draft64(cfg, tw, hw, eng, lens, root, feat, count.tolist())
        out["head_kv"] = [_as_rows(f, lens[s] - int(count[s])) for s, f in enumerate(fresh)]
    x = tw["embed"][eng.tree.token.flatten().long()].double()
    pos = (eng.tree.depth + torch.tensor(lens, device="cuda")[:, None]).flatten()
    bit = torch.arange(N, device="cuda")
    masks = [((eng.tree.anc[s][:, bit // 64] >> (bit % 64)) & 1).bool() for s in range(cfg.batch)]
    hidden, kv, last = _target64(cfg, tw, eng, lens, x, pos, masks)
    out["logits"] = _logits64(_norm64(last, tw["final_norm"]), tw["lm_head"])
    out["hidden"] = hidden.view(-1, cfg.batch, N, cfg.hidden)
    if c.get("sample"):
        lp = torch.log_softmax(out["logits"].view(cfg.batch, N, -1)[:, 0], -1)
        out["entropy"] = -(lp.exp() * lp).sum(-1)
    eng.glance_accept_commit(argmax=state["decisions"])
    torch.cuda.synchronize()
    paths = [[v for v in p if v >= 0] for p in eng.path.tolist()]
    out["feat"] = feat.double()                              # rows beyond the accepted ones stay as they were
    for s, p in enumerate(paths):
        out["feat"][:, s, : len(p)] = out["hidden"][:, s, p]
    # cache row P + d holds node path[d] of the accepted path; behind it the verify pass's row d stays
    keep = 1 + min(c.get("accept", 0), N - 1)
    paths = [(p + list(range(len(p), keep)))[:keep] for p in paths]
    kv = kv.view(cfg.n_layers, 2, cfg.batch, N, cfg.n_kv_heads, cfg.head_dim)
    out["kv"] = [_as_rows(kv[:, :, s, p].transpose(2, 3), lens[s]) for s, p in enumerate(paths)]
    return out
