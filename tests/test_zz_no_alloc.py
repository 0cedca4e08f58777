"""glance_topk_static: the workspace-free top-k entry point (GPU).

Some callers may not allocate device memory (their process gave the whole GPU to its own arena, or they run
inside a callback where allocation calls are forbidden), so this entry point keeps its scratch in a fixed
array inside the library.  The test drives it through the C ABI twice in a row -- the array keeps the first
call's contents -- and compares its output (a) with what glance_draft_block returned for the same logits and
(b) with the oracle's per-offset top-k and log-softmax of those logits.
"""
import numpy as np
import pytest
import torch

from oracle import glance_oracle as O
from paper_2609_00355_b200 import synth

pytestmark = pytest.mark.gpu

MARGIN = 0.05          # ids are compared where consecutive ranks are further apart than this
TOL = 2e-2             # of the logit scale


def test_topk_static_matches_draft_block_and_oracle_twice():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_00355_b200 import binding
    cfg = synth.CONFIGS["small"].replace(n_layers=1, n_img=40, n_txt=24, rounds=2)     # vocabulary 32000: 32 warps per row
    tw, hw = synth.make_weights(cfg, "cuda")
    eng = binding.Engine(cfg, tw, hw, batch=2)
    for s in range(2):
        img, ids = synth.make_context(cfg, "cuda", seed=5 + s)
        eng.prefill_context(s, img, ids)
    B, V, k, L = cfg.block_B, cfg.vocab, cfg.topk, cfg.L
    for call in range(2):
        logits = torch.zeros(2, B, V, dtype=torch.float32, device="cuda")
        eng.glance_draft_block(logits_dbg=logits)
        eng.check_device_status()
        ids_ref, lp_ref = eng.topk_ids.clone(), eng.topk_lp.clone()
        ids = torch.full((2, L, k), -1, dtype=torch.int32, device="cuda")
        lp = torch.full((2, L, k), float("nan"), dtype=torch.float32, device="cuda")
        assert binding.glance_topk_static(logits, k, ids, lp) == 0
        torch.cuda.synchronize()
        # Same logits on both sides (the draft pass exported the ones its fused top-k worked on): both select the k
        # largest under (logit desc, id asc), so the ids are identical; the log-sum-exp is added up in a different
        # order (1024-entry spans here, 128-feature tiles there), so the log-probabilities agree to rounding --
        # checked within the 2e-2 (relative to the logit scale) tolerance of the other parity tests, and far tighter
        assert torch.equal(ids, ids_ref)
        scale = float(logits.abs().max())
        assert float((lp - lp_ref).abs().max()) <= TOL * scale
        assert float((lp - lp_ref).abs().max()) <= 1e-4
        # against the oracle on the same logits: log-probabilities within the tolerance, ids identical wherever
        # the oracle's gap between consecutive ranks exceeds the margin
        lg_cpu = logits.cpu()
        for s in range(2):
            oid, olp = O.topk_logprobs(lg_cpu[s], k)
            assert float(np.abs(lp[s].cpu().numpy() - olp).max()) <= TOL * scale
            for j in range(L):
                srt = np.sort(lg_cpu[s, j + 1].numpy())[::-1][:k + 1]
                for r in range(k):
                    clear_above = r == 0 or srt[r - 1] - srt[r] > MARGIN
                    clear_below = srt[r] - srt[r + 1] > MARGIN
                    if clear_above and clear_below:
                        assert int(ids[s, j, r]) == int(oid[j, r]), (call, s, j, r)
        # move the state on so that the second call sees different logits and stale scratch from the first
        eng.glance_build_tree()
        eng.glance_verify_tree()
        eng.glance_accept_commit()
    # a request larger than the built-in scratch is refused with a clear status and launches nothing
    big = torch.zeros(1, 2, 8, dtype=torch.float32, device="cuda")
    lib = binding.load_library()
    rc = lib.glance_topk_static(big.data_ptr(), 64, 16, 1 << 24, 16, ids.data_ptr(), lp.data_ptr(), None)
    assert rc == -3 and lib.glance_status_string(rc) == b"capacity exceeded"
    # so is one with more rows than a launch dimension takes, although its scratch would fit
    rc = lib.glance_topk_static(big.data_ptr(), 65536, 2, 8, 1, ids.data_ptr(), lp.data_ptr(), None)
    assert rc == -3
    assert lib.glance_topk_static(None, 1, 2, 8, 1, ids.data_ptr(), lp.data_ptr(), None) == -1


@pytest.mark.parametrize("V,k,kind", [(2, 1, "random"), (16, 16, "random"), (1000, 7, "ties"), (1025, 16, "random"), (33000, 16, "ties"),
                                      (262144, 16, "random"), (262145, 3, "random"), (600000, 16, "random"), (600000, 16, "stripes"),
                                      (70000, 5, "inf"),
                                      # one CTA and a cluster of them, and the last vocabulary that a cluster takes
                                      (8192, 16, "random"), (8193, 16, "ties"), (9000, 16, "inf"), (196608, 16, "random"), (196609, 2, "ties")])
def test_topk_static_edges_of_spans_and_lists(V, k, kind):
    """One span, its remainders, more spans than threads, many equal values, -inf entries, and keys concentrated in a few
    spans, against the exact (logit desc, id asc) order on the CPU."""
    from paper_2609_00355_b200 import binding
    rng = np.random.default_rng(V + k)
    x = rng.standard_normal((1, 3, V)).astype(np.float32)
    if kind == "ties":
        x = np.round(x * 2) / 2
    elif kind == "stripes":                               # the best keys all in spans that one thread of the merge shares
        x[..., : V // 1024 * 1024].reshape(1, 3, -1, 1024)[:, :, 0::256] += 20
    elif kind == "inf":
        x[..., 10:] = -np.inf
    g = torch.from_numpy(x).cuda()
    ids = torch.full((1, 2, k), -1, dtype=torch.int32, device="cuda")
    lp = torch.full((1, 2, k), float("nan"), dtype=torch.float32, device="cuda")
    for _ in range(2):
        assert binding.glance_topk_static(g, k, ids, lp) == 0
    torch.cuda.synchronize()
    for j in range(2):
        row = x[0, j + 1].astype(np.float64)
        order = np.lexsort((np.arange(V), -row))[:k]
        assert ids[0, j].cpu().tolist() == order.tolist()
        m = row.max()
        ref = row[order] - (m + np.log(np.exp(row - m).sum()))
        got = lp[0, j].cpu().numpy()
        fin = np.isfinite(ref)
        assert np.array_equal(np.isfinite(got), fin)
        # fp32 sums of V terms in blocks of 32 and more: 1e-6 of the log-sum-exp's scale
        assert np.abs(got[fin] - ref[fin]).max() <= 4e-6 * max(1.0, float(np.abs(row[np.isfinite(row)]).max()) + np.log(V))


@pytest.mark.parametrize("batch,B,V,k", [(2, 16, 152064, 8), (2, 16, 152064, 4), (4, 16, 152064, 4), (10, 16, 8193, 16), (32, 16, 8192, 4),
                                         (1, 16, 65000, 16), (6, 16, 65000, 16), (2, 16, 8192, 16)])
def test_topk_static_many_rows(batch, B, V, k):
    """More rows than clusters are resident, in one launch and in two, and lists of more than 128 keys, against the exact
    (logit desc, id asc) order; the log-probabilities against 64 bits (fp32 sums of V terms: 1e-6 of the scale)."""
    from paper_2609_00355_b200 import binding
    g = torch.Generator(device="cuda").manual_seed(V + k)
    x = torch.randn(batch, B, V, generator=g, device="cuda") * 1.2
    ids = torch.full((batch, B - 1, k), -1, dtype=torch.int32, device="cuda")
    lp = torch.full((batch, B - 1, k), float("nan"), dtype=torch.float32, device="cuda")
    for _ in range(2):
        assert binding.glance_topk_static(x, k, ids, lp) == 0
    rows = x[:, 1:]
    val, idx = torch.sort(rows, dim=-1, descending=True, stable=True)
    assert torch.equal(ids.long(), idx[..., :k])
    ref = val[..., :k].double() - torch.logsumexp(rows.double(), dim=-1, keepdim=True)
    assert float((lp.double() - ref).abs().max()) <= 4e-6 * (float(rows.abs().max()) + np.log(V))
