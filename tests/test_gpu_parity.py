"""GPU parity tests: every call goes through the C-ABI library and is compared with the CPU oracle."""
import threading

import numpy as np
import pytest
import torch

import oracle
import parity
from helpers import to_bf16_bits
from paper_2603_17803_b200 import binding as B
from paper_2603_17803_b200 import workloads as W
from paper_2603_17803_b200.session import Session

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def run_separate_calls(sess):
    sess.select()
    sess.resolve()
    sess.gather()
    sess.sparse_attn()


def small(name, **kw):
    return W.scaled(W.CONFIGS[name], **kw)


CASES = {
    # several score tiles, a ragged tail, a partial last page; sized for an oracle run of seconds
    "c1_small": small("c1_tiny", ctx_len=16 * 700 + 5, top_k=48),
    "c2_small": small("c2_128k", ctx_len=16 * 1500 + 9, top_k=96, n_topics=12),
    "c3_small": small("c3_batched", batch=3, ctx_len=16 * 400 + 1, top_k=40, n_topics=8),
    "c4_small": small("c4_long", batch=2, ctx_len=32 * 900 + 17, top_k=64, n_topics=16),
    "c5_small": small("c5_skewed", batch=5, ctx_range=(16 * 20, 16 * 900), top_k=32, n_topics=10),
    "k_exceeds_pages": small("c5_skewed", batch=3, ctx_range=(1, 16 * 12), top_k=24, n_topics=3),
}


@pytest.mark.parametrize("name", list(CASES))
def test_separate_calls_match_oracle(name):
    w = W.generate(CASES[name], seed=11, device=DEV)
    sess = Session(w, keep_scores=True, keep_gathered=True)
    run_separate_calls(sess)
    info = parity.check_step(w, sess)
    assert info["heads"] == w.cfg.batch * w.cfg.n_q_heads
    sess.close()


@pytest.mark.parametrize("name", list(CASES))
def test_fused_step_equals_composition(name):
    w = W.generate(CASES[name], seed=12, device=DEV)
    a = Session(w, keep_scores=True, keep_gathered=True)
    run_separate_calls(a)
    torch.cuda.synchronize()
    b = Session(w, keep_scores=True, keep_gathered=True, ksum=a.ksum)
    b.step()
    info = parity.check_step(w, b)
    for f in ("sel", "n_sel", "n_tok", "k_out", "v_out", "queue_load"):
        assert torch.equal(getattr(a.o, f), getattr(b.o, f)), f
    n = int(a.o.n_uniq[0])
    assert int(b.o.n_uniq[0]) == n
    assert torch.equal(a.o.uniq[:n], b.o.uniq[:n]) and torch.equal(a.o.queue_of[:n], b.o.queue_of[:n])
    assert torch.equal(a.o.scores, b.o.scores)
    assert (a.o.out - b.o.out).abs().max().item() <= 1e-4
    assert (a.o.lse - b.o.lse).abs().max().item() <= 1e-4
    # fused step without the optional outputs gives the same required outputs
    c = Session(w, ksum=a.ksum)
    c.step()
    torch.cuda.synchronize()
    assert torch.equal(c.o.sel, b.o.sel) and torch.equal(c.o.out, b.o.out) and torch.equal(c.o.queue_load, b.o.queue_load)
    for s in (a, b, c):
        s.close()


def test_workspace_canaries_catch_a_stray_write():
    """Every Session.close() checks the canaries between the workspace regions (the stand-in for a memory checker
    on this path).  Here one canary byte is overwritten from the host side -- a torch fill, no kernel of the
    library involved -- to show that the check fires, and where."""
    w = W.generate(CASES["c1_small"], seed=3, device=DEV)
    sess = Session(w)
    sess.step()
    assert B.swarm_check_workspace(sess.ctx) == 0
    sess.workspace[7] = 0                                   # inside the canary in front of the first region
    assert B.swarm_check_workspace(sess.ctx) == 1
    sess.workspace[-3] = 1                                  # and inside the one behind the last region
    damaged = B.swarm_check_workspace(sess.ctx)
    assert damaged & 1 and damaged >> 1 and (damaged >> 1) & ((damaged >> 1) - 1) == 0
    with pytest.raises(RuntimeError, match="canaries"):
        sess.close()


@pytest.mark.parametrize("name", ["c2_small", "c3_small", "c5_small", "k_exceeds_pages"])
def test_overlapped_tail_gives_the_same_step(name):
    """Cluster resolution on a tail stream (swarm_set_tail_stream): consecutive steps with changing queries are
    enqueued without waiting in between, so a step's resolution runs beside the next step's scoring and
    selection; every step's outputs must equal those of the plain step bit for bit (integers) / within rounding
    (attention), and the last one must match the oracle."""
    w = W.generate(CASES[name], seed=14, device=DEV)
    plain = Session(w)
    tail_stream, stream = torch.cuda.Stream(), torch.cuda.Stream()
    tail = Session(w, ksum=plain.ksum, tail_stream=tail_stream)
    qs = [w.q, (w.q.float() * -1.0).to(torch.bfloat16), (w.q.float() * 0.5 + 0.125).to(torch.bfloat16), w.q]
    want = []
    for q in qs:
        plain.set_query(q)
        plain.step()
        torch.cuda.synchronize()
        n = int(plain.o.n_uniq[0])
        want.append(dict(sel=plain.o.sel.clone(), uniq=plain.o.uniq[:n].clone(), queue_of=plain.o.queue_of[:n].clone(),
                         load=plain.o.queue_load.clone(), out=plain.o.out.clone(), lse=plain.o.lse.clone()))
    # the tail session needs one set of outputs per step in flight: give every step its own
    outs = []
    with torch.cuda.stream(stream):
        for q in qs:
            o = type(tail.o)(**{f: (getattr(tail.o, f).clone() if getattr(tail.o, f) is not None else None)
                                for f in tail.o.__dataclass_fields__})
            outs.append(o)
            tail.o = o
            tail.outputs = B.make_outputs(**{k_: getattr(o, k_) for k_ in o.__dataclass_fields__})
            tail.set_query(q)
            tail.step(stream=stream)
        tail.tail_join(stream)
        stream.synchronize()
    assert tail.status() == 0
    for o, ref in zip(outs, want):
        n = len(ref["uniq"])
        assert int(o.n_uniq[0]) == n
        assert torch.equal(o.sel, ref["sel"]) and torch.equal(o.uniq[:n], ref["uniq"])
        assert torch.equal(o.queue_of[:n], ref["queue_of"]) and torch.equal(o.queue_load, ref["load"])
        assert (o.out - ref["out"]).abs().max().item() <= 1e-4 and (o.lse - ref["lse"]).abs().max().item() <= 1e-4
    parity.check_step(w, tail)
    # the same chain recorded into a CUDA graph (the capture has to join the tail stream) and replayed twice
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        with torch.cuda.graph(g, stream=stream):
            for _ in range(3):
                tail.step(stream=stream)
            tail.tail_join(stream)
        g.replay()
        g.replay()
        stream.synchronize()
    parity.check_step(w, tail)
    plain.close()
    tail.close()


@pytest.mark.parametrize("hq,hkv", [(16, 2), (8, 2), (6, 3), (5, 5), (6, 2)])
def test_fp32_pipe_scorer_matches_oracle(hq, hkv):
    """The scorer on the fp32 pipes (what shapes beyond the streaming kernel's limits fall back to), forced by
    swarm_set_scorer: groups of 8, 4, 2 and 1 query heads per KV head (its four instantiations; a group of 3 runs
    the single-head one three times), ragged tails, requests of unequal length, then the whole step on top."""
    cfg = small("c5_skewed", batch=3, n_q_heads=hq, n_kv_heads=hkv, ctx_range=(16 * 9, 16 * 333), top_k=24, n_topics=5)
    w = W.generate(cfg, seed=31, device=DEV)
    ref = Session(w, keep_scores=True, keep_gathered=True)
    ref.step()
    sess = Session(w, keep_scores=True, keep_gathered=True, scorer=B.SCORER_FP32, ksum=ref.ksum)
    run_separate_calls(sess)
    info = parity.check_step(w, sess)
    assert info["heads"] == cfg.batch * hq
    sess.step()
    parity.check_step(w, sess)
    # the two scorers agree far inside the tolerance of the score rule
    torch.cuda.synchronize()
    a, b = ref.o.scores, sess.o.scores
    live = torch.isfinite(a)
    assert torch.equal(live, torch.isfinite(b))
    assert ((a[live] - b[live]).abs() <= 1e-5 * a[live].abs() + 1e-4).all()
    with pytest.raises(B.SwarmError):
        B.swarm_set_scorer(sess.ctx, 3)
    B.swarm_set_scorer(sess.ctx, B.SCORER_TENSOR)
    sess.step()
    parity.check_step(w, sess)
    ref.close()
    sess.close()


@pytest.mark.parametrize("name", ["c1_tiny", "c2_128k"])
def test_full_size_configs_match_oracle(name):
    """The two configurations the oracle handles whole, at full size, through the fused step."""
    w = W.generate(W.CONFIGS[name], seed=0, device=DEV)
    sess = Session(w, keep_scores=True, keep_gathered=True)
    sess.step()
    info = parity.check_step(w, sess)
    assert info["exact_heads"] >= info["heads"] - 4      # band differences are legal but rare
    sess.close()


@pytest.mark.parametrize("name,reqs,heads", [("c3_batched", [0, 9], [0, 5, 31]), ("c4_long", [1], [0, 17, 63])])
def test_full_size_sampled(name, reqs, heads):
    """Full-size launch configuration; stage 3 checked whole, the other stages on sampled requests/heads."""
    w = W.generate(W.CONFIGS[name], seed=0, device=DEV)
    sess = Session(w, keep_scores=True)
    sess.step()
    parity.check_step(w, sess, requests=reqs, heads=heads)
    sess.close()


def test_c5_full_size_sampled():
    w = W.generate(W.CONFIGS["c5_skewed"], seed=0, device=DEV)
    sess = Session(w, keep_scores=True)
    sess.step()
    lens = w.ctx_len.cpu().numpy()
    reqs = sorted({int(np.argmin(lens)), int(np.argmax(lens)), 7})
    parity.check_step(w, sess, requests=reqs, heads=[0, 13, 31])
    # more fetched clusters than the resolution kernel stages in shared memory: the submission order too
    sess.enable_submit_order()
    sess.step()
    assert check_submit_order(w, sess) > 20000
    sess.close()


def test_caller_supplied_selection_and_misplaced_partial_page():
    """swarm_gather / swarm_sparse_attn on a selection the caller wrote (ascending, a subset of the pages, the
    partial last page included): parity with the oracle; the same pages with the partial page NOT last are
    refused for that page (status bit, slot zero-filled) instead of attending its padding rows."""
    cfg = small("c2_128k", ctx_len=16 * 300 + 5, top_k=20, n_topics=4)
    w = W.generate(cfg, seed=17, device=DEV)
    sess = Session(w, keep_gathered=True)
    P = cfg.max_pages()
    rng = np.random.default_rng(2)
    sel = np.full((1, cfg.n_q_heads, cfg.top_k), -1, dtype=np.int32)
    n_sel = np.zeros((1, cfg.n_q_heads), dtype=np.int32)
    for h in range(cfg.n_q_heads):
        n = int(rng.integers(1, cfg.top_k + 1))
        pages = np.sort(rng.choice(P - 1, size=n - 1, replace=False)) if n > 1 else np.zeros(0, np.int64)
        sel[0, h, :n] = np.concatenate([pages, [P - 1]])     # the partial page, last
        n_sel[0, h] = n
    sel_t, n_sel_t = torch.from_numpy(sel).to(DEV), torch.from_numpy(n_sel).to(DEV)
    sess.gather(sel_t, n_sel_t)
    sess.sparse_attn()
    torch.cuda.synchronize()
    assert sess.status() == 0
    tabs = parity.host_tables(w)
    pool = parity.bits_u16(w.kv_pool)
    kg, vg, n_tok = oracle.gather(pool, sel, n_sel, tabs["page_base"], tabs["ctx_len"], cfg.n_kv_heads, cfg.head_dim, cfg.page_size)
    assert np.array_equal(parity.bits_u16(sess.o.k_out), kg) and np.array_equal(parity.bits_u16(sess.o.v_out), vg)
    assert np.array_equal(sess.o.n_tok.cpu().numpy(), n_tok)
    out_ref, lse_ref = oracle.attention(parity.bits_u16(w.q), kg, vg, n_tok)
    parity.check_attention(sess.o.out.cpu().numpy(), sess.o.lse.cpu().numpy(), out_ref, lse_ref)
    # the partial page first: flagged and skipped
    h = int(np.argmax(n_sel[0] >= 2))
    n = int(n_sel[0, h])
    sel[0, h, :n] = np.concatenate([[P - 1], sel[0, h, :n - 1]])
    sess.gather(torch.from_numpy(sel).to(DEV), n_sel_t)
    torch.cuda.synchronize()
    assert sess.status() == B.DEV_BAD_PAGE
    assert not sess.o.k_out[0, h, : cfg.page_size].any()
    sess.close()


@pytest.mark.parametrize("splits", [1, 2, 7, 64])
def test_split_count_is_unobservable(splits):
    w = W.generate(CASES["c2_small"], seed=5, device=DEV)
    sess = Session(w, keep_gathered=True)
    B.swarm_set_attn_splits(sess.ctx, splits)
    run_separate_calls(sess)
    parity.check_step(w, sess)
    sess.step()
    parity.check_step(w, sess)
    sess.close()


@pytest.mark.parametrize("flags", [B.ORDER_BY_ID, B.UNIT_LOAD, B.ORDER_BY_ID | B.UNIT_LOAD])
@pytest.mark.parametrize("name", ["c3_small", "c5_small"])
def test_scheduling_flags(name, flags):
    w = W.generate(CASES[name], seed=6, device=DEV)
    sess = Session(w, flags=flags)
    sess.step()
    parity.check_step(w, sess, flags=flags)
    sess.close()


@pytest.mark.parametrize("replication,D", [("one", 5), ("all", 7), ("all", 32), ("two", 32)])
def test_replication_extremes(replication, D):
    cfg = small("c3_batched", batch=2, ctx_len=16 * 300, top_k=50, n_topics=6, replication=replication, n_queues=D)
    w = W.generate(cfg, seed=7, device=DEV)
    sess = Session(w, flags=B.UNIT_LOAD if replication == "all" else 0)
    sess.step()
    parity.check_step(w, sess, flags=B.UNIT_LOAD if replication == "all" else 0)
    load = sess.o.queue_load.cpu().numpy()[:D]
    if replication == "all":
        assert load.max() - load.min() <= 1
    sess.close()


@pytest.mark.parametrize("replication", ["two", "half_two"])
@pytest.mark.parametrize("D,sizes", [(2, (8,)), (3, (8, 1)), (4, (7,)), (8, (8,)), (8, (1, 2, 3)), (8, (40, 63)),
                                     (8, (900, 1023)), (8, (1500, 60000)), (8, (0,)), (8, (0, 9)), (9, (8,)), (12, (8, 1)),
                                     (15, (3, 4, 5, 6)), (16, (8,)), (16, (62, 63)), (16, (64, 70)), (17, (8,))])
def test_schedules_of_two_replicas(replication, D, sizes):
    """The serial pass over two-replica clusters runs equal weights on up to 8 queues in 32 stretches while the loads fit a
    byte, other weights and up to 16 queues level by level, and the rest one by one: queue counts and weights on both
    sides of every limit, single-replica clusters that spread the starting loads, and stretches that end in a
    remainder.  Every cluster is activated."""
    cfg = small("c3_batched", batch=3, ctx_len=16 * 1501, top_k=1501, n_q_heads=2, n_kv_heads=2, n_topics=6,
                replication=replication, n_queues=D)
    w = W.generate(cfg, seed=D, device=DEV)
    rng = np.random.default_rng(D * 1000 + len(sizes))
    w.cluster_size.copy_(torch.from_numpy(rng.choice(sizes, size=w.n_clusters).astype(np.uint16).view(np.int16)))
    for flags in (0, B.ORDER_BY_ID) if len(sizes) == 1 else (0,):
        sess = Session(w, flags=flags)
        sess.step()
        torch.cuda.synchronize()
        assert sess.status() == 0
        o = sess.o
        uniq, _, _ = parity.check_resolve(w, parity.host_tables(w), o.sel.cpu().numpy(), o.n_sel.cpu().numpy(), o.uniq.cpu().numpy(),
                                          o.queue_of.cpu().numpy(), o.n_uniq.cpu().numpy()[0], o.queue_load.cpu().numpy(), flags)
        assert len(uniq) == w.n_clusters
        sess.close()


@pytest.mark.parametrize("batch,replication,sizes", [(2, "two", (8,)), (2, "two", (1, 2, 7)), (2, "hot_three", (3, 5)), (4, "two", (2,)),
                                                     (4, "two", (1, 9))])
def test_schedules_longer_than_the_shared_list(batch, replication, sizes):
    """8192 and 16384 activated clusters, below and above the capacity of the serial pass's list in shared memory (9928
    clusters, 5944 with a submission order)."""
    cfg = small("c3_batched", batch=batch, ctx_len=16 * 8192, top_k=8192, n_q_heads=1, n_kv_heads=1, n_topics=4, cluster_pages=2,
                replication=replication, n_queues=12)
    w = W.generate(cfg, seed=batch, device=DEV)
    rng = np.random.default_rng(batch)
    w.cluster_size.copy_(torch.from_numpy(rng.choice(sizes, size=w.n_clusters).astype(np.uint16).view(np.int16)))
    for order in (False, True):
        sess = Session(w)
        if order:
            sess.enable_submit_order()
        sess.step()
        torch.cuda.synchronize()
        assert sess.status() == 0
        o = sess.o
        parity.check_resolve(w, parity.host_tables(w), o.sel.cpu().numpy(), o.n_sel.cpu().numpy(), o.uniq.cpu().numpy(),
                             o.queue_of.cpu().numpy(), o.n_uniq.cpu().numpy()[0], o.queue_load.cpu().numpy())
        if order:
            check_submit_order(w, sess)
        sess.close()


@pytest.mark.parametrize("order", [False, True])
@pytest.mark.parametrize("over", [-16, -15, 0, 1])
def test_schedules_at_the_capacity_of_the_shared_list(over, order):
    """The serial pass keeps lists of up to 9928 clusters in shared memory, 5944 with a submission order, and lets blank
    clusters follow them: lists that end 16 and 15 places short of the capacity, at it and behind it.  A cluster per
    page, every page selected."""
    n = (5944 if order else 9928) + over
    cfg = small("c1_tiny", ctx_len=16 * n, top_k=n, n_q_heads=1, n_kv_heads=1, cluster_pages=1, n_queues=12)
    w = W.generate(cfg, seed=n, device=DEV)
    two = w.cluster_replica_mask.clone()
    rng = np.random.default_rng(n)
    third = torch.from_numpy(1 << rng.integers(0, 12, size=n).astype(np.int32)).to(DEV)
    every_third = torch.arange(n, device=DEV) % 3 == 0
    # all of two replicas, equal and unequal weights; two or three replicas; in id order with single replicas among them
    for masks, sizes, flags in ((two, (8,), 0), (two, (1, 2, 7), 0), (torch.where(every_third, two | third, two), (3, 5), 0),
                                (torch.where(every_third, third, two), (4, 9), B.ORDER_BY_ID)):
        w.cluster_replica_mask = masks.contiguous()
        w.cluster_size.copy_(torch.from_numpy(rng.choice(sizes, size=n).astype(np.uint16).view(np.int16)))
        sess = Session(w, flags=flags)
        if order:
            sess.enable_submit_order()
        sess.o.queue_of.fill_(255)
        sess.step()
        torch.cuda.synchronize()
        assert sess.status() == 0
        o = sess.o
        uniq, _, _ = parity.check_resolve(w, parity.host_tables(w), o.sel.cpu().numpy(), o.n_sel.cpu().numpy(), o.uniq.cpu().numpy(),
                                          o.queue_of.cpu().numpy(), o.n_uniq.cpu().numpy()[0], o.queue_load.cpu().numpy(), flags)
        assert len(uniq) == n
        if order:
            assert check_submit_order(w, sess, flags) == n
        sess.close()


def test_all_equal_scores_pick_lowest_ids_and_signed_zero_ties():
    cfg = small("c1_tiny", ctx_len=16 * 300, top_k=20)
    w = W.generate(cfg, seed=8, device=DEV)
    w.q.zero_()                                          # every score is exactly 0
    sess = Session(w, keep_scores=True)
    sess.step()
    torch.cuda.synchronize()
    assert torch.equal(sess.o.sel[0, 3].cpu(), torch.arange(20, dtype=torch.int32))
    parity.check_step(w, sess)
    # planted duplicates straddling the k-th place: make the scorer reproduce chosen scores exactly
    # (q = e_0 and kmin = kmax = the wanted score in coordinate 0), then compare with the oracle's top-k
    P = cfg.max_pages()
    sc = torch.zeros((1, 8, P), device=DEV)
    sc[0, 1] = torch.arange(P, device=DEV) % 7
    sc[0, 2] = -(torch.arange(P, device=DEV) % 5).float()
    sc[0, 3] = (torch.arange(P, device=DEV) // 50).float()
    ref, _ = oracle.topk(sc.cpu().numpy(), w.ctx_len.cpu().numpy(), 16, 20)
    ksum = torch.zeros_like(sess.ksum)
    ksum[:, :, :, 0] = sc[0].t()[:, :, None].to(torch.bfloat16)
    w.q.zero_()
    w.q[..., 0] = 1.0
    sess2 = Session(w, keep_scores=True, ksum=ksum)
    sess2.select()
    torch.cuda.synchronize()
    assert torch.equal(sess2.o.scores[0, :, :P], sc[0])
    assert np.array_equal(sess2.o.sel.cpu().numpy()[0], ref[0])
    sess.close()
    sess2.close()


def test_structured_attention_outputs_of_order_one():
    """Dominant key and constant V: outputs of magnitude 1, so the tolerance is meaningful."""
    cfg = small("c1_tiny", ctx_len=16 * 200, top_k=30)
    w = W.generate(cfg, seed=9, device=DEV)
    q = w.q.float()
    # plant, for head 2, a key in page 77 aligned with q and strong enough to dominate
    w.kv_pool[77, 2, 0, 5] = (40.0 * q[0, 2] / q[0, 2].norm()).to(torch.bfloat16)
    w.kv_pool[:, 4, 1] = 1.5                              # head 4: constant V
    sess = Session(w, keep_gathered=True)
    sess.step()
    parity.check_step(w, sess)
    out = sess.o.out.cpu()
    assert (out[0, 2] - w.kv_pool[77, 2, 1, 5].float().cpu()).abs().max() < 2e-2
    assert (out[0, 4] - 1.5).abs().max() < 1e-5
    sess.close()


def test_corrupt_tables_set_status_bits_and_never_trap():
    cfg = small("c3_batched", batch=2, ctx_len=16 * 100, top_k=16, n_topics=4)
    w = W.generate(cfg, seed=10, device=DEV)
    sess = Session(w)
    sess.step()
    torch.cuda.synchronize()
    assert sess.status() == 0
    good_mask = w.cluster_replica_mask.clone()
    w.cluster_replica_mask.zero_()                        # no replica anywhere
    sess.step()
    assert sess.status() & B.DEV_BAD_REPLICA
    assert int(sess.o.queue_of[0]) == 0xFF
    w.cluster_replica_mask.copy_(good_mask)
    good_p2c = w.page2cluster.clone()
    w.page2cluster.fill_(10 ** 6)                         # cluster ids out of range
    sess.step()
    assert sess.status() & B.DEV_BAD_CLUSTER
    w.page2cluster.copy_(good_p2c)
    bad_sel = sess.o.sel.clone()
    bad_sel[0, 0, 0] = 10 ** 6                            # page id out of range, fed to the stage calls
    sess.resolve(sel=bad_sel)
    assert sess.status() & B.DEV_BAD_PAGE
    good_len = w.ctx_len.clone()
    w.ctx_len[0] = 0
    sess.select()
    assert sess.status() & B.DEV_BAD_LENGTH
    w.ctx_len.copy_(good_len)
    sess.step()                                           # the ctx is still usable
    torch.cuda.synchronize()
    assert sess.status() == 0
    parity.check_step(w, sess)
    sess.close()


def test_invalid_arguments_are_rejected_on_the_host():
    ok = dict(batch=1, n_q_heads=8, n_kv_heads=2, page_size=16, top_k=4, n_queues=4, max_pages_per_req=8,
              max_clusters_total=4, n_pool_pages=8)
    for bad, code in [(dict(head_dim=64), B.ERR_UNSUPPORTED), (dict(page_size=8), B.ERR_UNSUPPORTED),
                      (dict(n_queues=33), B.ERR_INVALID_ARG), (dict(n_kv_heads=3), B.ERR_INVALID_ARG),
                      (dict(top_k=0), B.ERR_INVALID_ARG), (dict(flags=64), B.ERR_INVALID_ARG)]:
        with pytest.raises(B.SwarmError) as e:
            B.swarm_create(B.make_shape(**{**ok, **bad}))
        assert e.value.code == code
    shape = B.make_shape(**ok)
    ctx = B.swarm_create(shape)
    t = torch.zeros(1024, dtype=torch.int32, device=DEV)
    with pytest.raises(B.SwarmError) as e:                # no workspace yet
        B.swarm_select(ctx, B.make_inputs(q=t, ksum=t, page_base=t, ctx_len=t), None, t, t)
    assert e.value.code == B.ERR_WORKSPACE_TOO_SMALL
    with pytest.raises(B.SwarmError) as e:
        B.swarm_set_workspace(ctx, torch.empty(16, dtype=torch.uint8, device=DEV))
    assert e.value.code == B.ERR_WORKSPACE_TOO_SMALL
    with pytest.raises(B.SwarmError) as e:                # the flag array lives in the workspace
        B.swarm_cluster_flags(ctx)
    assert e.value.code == B.ERR_WORKSPACE_TOO_SMALL
    ws = torch.empty(B.swarm_workspace_bytes(shape), dtype=torch.uint8, device=DEV)
    B.swarm_set_workspace(ctx, ws)
    with pytest.raises(B.SwarmError) as e:                # null input
        B.swarm_select(ctx, B.make_inputs(q=t, ksum=None, page_base=t, ctx_len=t), None, t, t)
    assert e.value.code == B.ERR_INVALID_ARG
    with pytest.raises(B.SwarmError) as e:                # misaligned pointer
        B.swarm_select(ctx, B.make_inputs(q=t[1:], ksum=t, page_base=t, ctx_len=t), None, t, t)
    assert e.value.code == B.ERR_INVALID_ARG
    addr, n = B.swarm_cluster_flags(ctx)
    assert n == 4 and ws.data_ptr() <= addr and addr + n <= ws.data_ptr() + ws.numel()
    for half in (B.swarm_step_begin, B.swarm_step_end):    # the halves validate like the whole step
        with pytest.raises(B.SwarmError) as e:
            half(ctx, B.make_inputs(q=t, ksum=t, page_base=t, ctx_len=t), B.make_outputs(sel=t, n_sel=t))
        assert e.value.code == B.ERR_INVALID_ARG
    B.swarm_destroy(ctx)


def test_step_host_round_trip():
    w = W.generate(CASES["c2_small"], seed=13, device=DEV)
    sess = Session(w)
    sess.step()
    torch.cuda.synchronize()
    want_out, want_load = sess.o.out.cpu().clone(), sess.o.queue_load.cpu().clone()
    q_host = w.q.cpu().pin_memory()
    out_host = torch.empty_like(want_out).pin_memory()
    lse_host = torch.empty((1, 32), dtype=torch.float32).pin_memory()
    n_host = torch.zeros(1, dtype=torch.int32).pin_memory()
    load_host = torch.zeros(w.cfg.n_queues, dtype=torch.int32).pin_memory()
    sess.o.out.zero_()
    sess.step_host(q_host, out_host, lse_host, n_host, load_host)
    assert torch.equal(out_host, want_out)
    assert torch.equal(load_host, want_load[: w.cfg.n_queues])
    assert int(n_host[0]) == int(sess.o.n_uniq[0])
    # on a stream of its own the call records a graph and replays it; repeated calls give the same bytes
    stream = torch.cuda.Stream()
    for _ in range(3):
        out_host.zero_(); lse_host.zero_(); n_host.zero_(); load_host.zero_()
        sess.step_host(q_host, out_host, lse_host, n_host, load_host, stream=stream)
        assert torch.equal(out_host, want_out) and torch.equal(load_host, want_load[: w.cfg.n_queues])
        assert torch.equal(lse_host.view(-1), sess.o.lse.cpu().view(-1)) and int(n_host[0]) == int(sess.o.n_uniq[0])
    # pageable (and odd-offset) destinations take the copy path and give the same bytes
    out_page = torch.empty(want_out.numel() + 1, dtype=torch.float32)[1:].view_as(want_out)
    lse_page = torch.empty((1, 32), dtype=torch.float32)
    n_page, load_page = torch.zeros(1, dtype=torch.int32), torch.zeros(w.cfg.n_queues, dtype=torch.int32)
    sess.step_host(q_host, out_page, lse_page, n_page, load_page)
    assert torch.equal(out_page, want_out) and torch.equal(load_page, want_load[: w.cfg.n_queues])
    assert int(n_page[0]) == int(sess.o.n_uniq[0])
    # a mix: pinned out, no lse, pageable counters
    out_host.zero_()
    sess.step_host(q_host, out_host, None, n_page, None)
    assert torch.equal(out_host, want_out)
    sess.close()


@pytest.mark.parametrize("name", ["c3_small", "c5_small", "k_exceeds_pages"])
def test_step_host_follows_a_query_buffer_rewritten_between_calls(name):
    """The same pinned buffers, new contents every call: every call's results are those of its own query and are
    complete in host memory when the call returns (the recorded graph, the fetch of q and the completion word
    are all reused from call to call)."""
    w = W.generate(CASES[name], seed=17, device=DEV)
    cfg = w.cfg
    sess = Session(w)
    ref = Session(w, ksum=sess.ksum)
    g = torch.Generator(device="cpu").manual_seed(5)
    q_host = torch.empty_like(w.q, device="cpu").pin_memory()
    out_host = torch.empty((cfg.batch, cfg.n_q_heads, cfg.head_dim), dtype=torch.float32).pin_memory()
    lse_host = torch.empty((cfg.batch, cfg.n_q_heads), dtype=torch.float32).pin_memory()
    n_host = torch.zeros(1, dtype=torch.int32).pin_memory()
    load_host = torch.zeros(cfg.n_queues, dtype=torch.int32).pin_memory()
    stream = torch.cuda.Stream()
    for it in range(40):
        q = (w.q.cpu().float() + 0.5 * torch.randn(w.q.shape, generator=g)).to(torch.bfloat16)
        q_host.copy_(q)
        out_host.fill_(float("nan")); lse_host.fill_(float("nan")); n_host.fill_(-1); load_host.fill_(-1)
        sess.step_host(q_host, out_host, lse_host, n_host, load_host, stream=stream)
        got = (out_host.clone(), lse_host.clone(), int(n_host[0]), load_host.clone())   # read at once, no synchronize
        ref.set_query(q.to(DEV))
        ref.step()
        torch.cuda.synchronize()
        assert torch.equal(got[0], ref.o.out.cpu()), f"call {it}"
        assert torch.equal(got[1], ref.o.lse.cpu()) and got[2] == int(ref.o.n_uniq[0])
        assert torch.equal(got[3], ref.o.queue_load.cpu()[: cfg.n_queues])
        assert torch.equal(sess.o.sel, ref.o.sel) and torch.equal(sess.o.uniq[: got[2]], ref.o.uniq[: got[2]])
    assert sess.status() == 0
    sess.close()
    ref.close()


def test_step_can_be_captured_in_a_cuda_graph():
    w = W.generate(CASES["c3_small"], seed=14, device=DEV)
    sess = Session(w)
    sess.step()
    torch.cuda.synchronize()
    n = int(sess.o.n_uniq[0])
    sess.o.uniq[n:].zero_()                               # entries beyond n_uniq are not written
    want = {f: getattr(sess.o, f).clone() for f in ("sel", "out", "lse", "queue_load", "uniq", "n_uniq")}
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        sess.step(stream=s)                               # warm-up on the capture stream
        s.synchronize()
        with torch.cuda.graph(graph, stream=s):
            sess.step(stream=s)
    for f in want:
        getattr(sess.o, f).zero_()
    graph.replay()
    torch.cuda.synchronize()
    for f, t in want.items():
        assert torch.equal(getattr(sess.o, f), t), f
    sess.close()


def test_paged_attention_alone_matches_gathered_attention():
    w = W.generate(CASES["c4_small"], seed=15, device=DEV)
    sess = Session(w, keep_gathered=True)
    run_separate_calls(sess)
    torch.cuda.synchronize()
    out, lse = sess.o.out.clone(), sess.o.lse.clone()
    sess.o.out.zero_()
    sess.sparse_attn_paged()
    torch.cuda.synchronize()
    assert (sess.o.out - out).abs().max().item() <= 1e-5 and (sess.o.lse - lse).abs().max().item() <= 1e-5
    parity.check_step(w, sess)
    out2 = sess.o.out.clone()
    sess.o.out.zero_()
    sess.sparse_attn_paged(reuse_last_selection=True)     # bitmaps left in the workspace by the calls above
    torch.cuda.synchronize()
    assert torch.equal(sess.o.out, out2)
    sess.close()


@pytest.mark.parametrize("name", ["c1_small", "c2_small", "c3_small", "c5_small"])
def test_paged_attention_reuses_the_bitmaps_a_step_left(name):
    """A fused step hands its page bitmaps to its own attention kernel in whichever form is fastest; whatever
    that is, a later swarm_sparse_attn_paged without a selection finds them in the workspace."""
    w = W.generate(CASES[name], seed=16, device=DEV)
    sess = Session(w)
    sess.step()
    sess.step()
    torch.cuda.synchronize()
    out, lse = sess.o.out.clone(), sess.o.lse.clone()
    sess.o.out.zero_()
    sess.o.lse.zero_()
    sess.sparse_attn_paged(reuse_last_selection=True)
    torch.cuda.synchronize()
    assert sess.status() == 0
    assert (sess.o.out - out).abs().max().item() <= 1e-5 and (sess.o.lse - lse).abs().max().item() <= 1e-5
    parity.check_step(w, sess)
    sess.close()


@pytest.mark.parametrize("name", ["c1_small", "c2_small", "c3_small", "c4_small", "c5_small"])
@pytest.mark.parametrize("tail", [False, True])
def test_index_prefetch_changes_no_result(name, tail):
    """swarm_set_index_prefetch: the scorer asks for its first index blocks before it waits for the previous
    step's attention kernel (which releases its SMs early for it).  Back-to-back steps with the switch on give the
    results of the switch off, bit for bit, and match the oracle."""
    w = W.generate(CASES[name], seed=17, device=DEV)
    tstream = torch.cuda.Stream() if tail else None
    ref = Session(w, tail_stream=tstream)
    for _ in range(2):
        ref.step()
    if tail:
        ref.tail_join()
    torch.cuda.synchronize()
    sess = Session(w, ksum=ref.ksum, tail_stream=tstream, index_prefetch=True)
    for _ in range(4):                                     # each step's scorer is launched behind the previous step's attention
        sess.step()
    if tail:
        sess.tail_join()
    torch.cuda.synchronize()
    assert sess.status() == 0
    for key in ("sel", "n_sel", "out", "lse"):
        assert torch.equal(getattr(ref.o, key), getattr(sess.o, key)), key
    n_q = w.cfg.n_queues
    assert int(ref.o.n_uniq[0]) == int(sess.o.n_uniq[0]) and torch.equal(ref.o.queue_load[:n_q], sess.o.queue_load[:n_q])
    parity.check_step(w, sess)
    B.swarm_set_index_prefetch(sess.ctx, False)            # and off again
    sess.step()
    if tail:
        sess.tail_join()
    torch.cuda.synchronize()
    assert sess.status() == 0 and torch.equal(ref.o.out, sess.o.out)
    sess.close()
    ref.close()


@pytest.mark.parametrize("between", ["medoid_rows", "admission", "gathered_attention"])
@pytest.mark.parametrize("name", ["c2_small", "c3_small"])
def test_index_update_one_operation_ahead_of_a_prefetching_step(name, between):
    """The contract of the index prefetch: the operation directly before the step writes none of the index, one further up
    may.  The pool is rewritten between turns, its summaries are built again, one other call follows, then the step."""
    w = W.generate(CASES[name], seed=18, device=DEV)
    pools = [w.kv_pool.clone(), W.generate(CASES[name], seed=19, device=DEV).kv_pool]
    want = []
    for pool in pools:
        w.kv_pool.copy_(pool)
        ref = Session(w)
        torch.cuda.synchronize()
        ref.step()
        parity.check_step(w, ref)
        want.append({k: getattr(ref.o, k).clone() for k in ("sel", "n_sel", "out", "lse")})
        ref.close()
    sess = Session(w, keep_gathered=True, index_prefetch=True)
    sess.enable_medoid_index(5)
    sess.outputs = B.make_outputs(**{k: None if k in ("k_out", "v_out", "n_tok") else getattr(sess.o, k) for k in sess.o.__dataclass_fields__})
    sess.select()
    sess.gather()
    score = torch.rand(w.n_clusters, device=DEV)
    resident = torch.zeros(w.n_clusters, dtype=torch.uint8, device=DEV)
    for turn in range(6):
        w.kv_pool.copy_(pools[turn % 2])
        B.swarm_build_summaries(sess.ctx, sess.inputs, sess.ksum)
        if between == "medoid_rows":
            B.swarm_build_medoid_index(sess.ctx, sess.inputs, sess.medoid_page, sess.medoid_ksum, sess.cluster_ctx_len)
        elif between == "admission":
            B.swarm_cache_admit(score, w.cluster_size, w.n_pool_pages // 4, resident)
        else:
            sess.sparse_attn()
        sess.step()
        torch.cuda.synchronize()
        assert sess.status() == 0
        for k, v in want[turn % 2].items():
            assert torch.equal(getattr(sess.o, k), v), (turn, k)
    sess.close()


@pytest.mark.parametrize("scorer", [B.SCORER_AUTO, B.SCORER_FP32])
def test_medoid_step_directly_behind_its_index_build(scorer):
    """The pseudo lengths and the rows are rewritten right in front of the step that reads them, with either scorer."""
    w = W.generate(CASES["c5_small"], seed=20, device=DEV)
    sess = Session(w, scorer=scorer)
    sess.enable_medoid_index(7, keep_scores=True)
    torch.cuda.synchronize()
    sess.step_medoid()
    check_medoid_step(w, sess, 7)
    keys = ("sel_clusters", "n_sel_clusters", "cluster_scores")
    want = {k: getattr(sess, k).clone() for k in keys}
    out = sess.o.out.clone()
    for _ in range(6):
        sess.medoid_ksum.zero_()
        sess.cluster_ctx_len.fill_(1)
        B.swarm_build_medoid_index(sess.ctx, sess.inputs, sess.medoid_page, sess.medoid_ksum, sess.cluster_ctx_len)
        sess.step_medoid()
        torch.cuda.synchronize()
        assert sess.status() == 0 and torch.equal(sess.o.out, out)
        for k, v in want.items():
            assert torch.equal(getattr(sess, k), v), k
    sess.close()


@pytest.mark.parametrize("name", ["c3_small", "c5_small"])
def test_resident_filter_and_cache_counters(name):
    """Eq. 8 with the resident term, activation frequencies and Eq. 6 scores, against the oracle on the GPU's
    own selection; two steps in a row so the counters accumulate; then detached again."""
    w = W.generate(CASES[name], seed=16, device=DEV)
    sess = Session(w)
    C = w.n_clusters
    g = torch.Generator(device="cpu").manual_seed(5)
    resident = (torch.rand(C, generator=g) < 0.3).to(torch.uint8).to(DEV)
    freq0 = torch.randint(-3, 10, (C,), generator=g, dtype=torch.int32)
    freq = freq0.to(DEV)
    score = torch.zeros(C, dtype=torch.float32, device=DEV)
    n_hit = torch.zeros(4, dtype=torch.int32, device=DEV)
    t_base, t_tr = 80.0, 2.5
    B.swarm_set_cache(sess.ctx, resident=resident, freq=freq, score=score, n_hit=n_hit, t_base=t_base, t_transfer=t_tr)
    tabs = parity.host_tables(w)
    want_freq = freq0.numpy().copy()
    for step_no in range(2):
        if step_no == 0:
            sess.step()
        else:                                             # the separate call takes the same path
            sess.resolve()
        torch.cuda.synchronize()
        assert sess.status() == 0
        uniq, qof, load, hits, want_freq, want_score = oracle.resolve_cached(
            sess.o.sel.cpu().numpy(), sess.o.n_sel.cpu().numpy(), tabs["page_base"], tabs["page2cluster"],
            tabs["cluster_base"], tabs["replica_mask"], tabs["cluster_size"], resident.cpu().numpy(), want_freq,
            w.cfg.n_queues, t_base, t_tr)
        n = int(sess.o.n_uniq[0])
        assert n == len(uniq) and hits > 0
        assert np.array_equal(sess.o.uniq[:n].cpu().numpy(), uniq)
        assert np.array_equal(sess.o.queue_of[:n].cpu().numpy(), qof)
        assert np.array_equal(sess.o.queue_load.cpu().numpy()[: w.cfg.n_queues], load)
        assert int(n_hit[0]) == hits
        assert np.array_equal(freq.cpu().numpy(), want_freq)
        assert np.allclose(score.cpu().numpy(), want_score, rtol=1e-6, atol=1e-6)
    B.swarm_set_cache(sess.ctx)                           # detached: plain merge again
    sess.step()
    parity.check_step(w, sess)
    assert np.array_equal(freq.cpu().numpy(), want_freq)
    sess.close()


EDGE_SHAPES = {
    # group of 16 heads per KV head (two head tiles in the scorer and in attention), 32-token pages
    "g16_s32": small("c4_long", batch=2, n_q_heads=32, n_kv_heads=2, ctx_len=32 * 300 + 5, top_k=24, n_topics=6),
    # odd number of KV heads, group of 2
    "hkv3_g2": small("c2_128k", batch=2, n_q_heads=6, n_kv_heads=3, ctx_len=16 * 500 + 3, top_k=33, n_topics=5),
    # more KV heads than one scorer block holds (two KV groups), MHA
    "hkv16_g1": small("c1_tiny", batch=1, n_q_heads=16, n_kv_heads=16, ctx_len=16 * 260, top_k=17),
    # a single page per head, a single queue
    "k1_d1": small("c3_batched", batch=3, ctx_len=16 * 150 + 1, top_k=1, n_topics=4, n_queues=1, replication="one"),
    # group of 12 heads: a full head tile of 8 plus a partial one of 4
    "g12": small("c2_128k", batch=1, n_q_heads=24, n_kv_heads=2, ctx_len=16 * 400, top_k=40, n_topics=6),
    # more (request, KV head) groups than fit one wave of attention CTAs with short page ranges: two waves, the
    # last groups cut into one range more than the others
    "two_waves": small("c3_batched", batch=12, ctx_len=16 * 300 + 7, top_k=128, n_topics=8),
}


@pytest.mark.parametrize("name", list(EDGE_SHAPES))
def test_unusual_shapes(name):
    w = W.generate(EDGE_SHAPES[name], seed=17, device=DEV)
    a = Session(w, keep_scores=True, keep_gathered=True)
    run_separate_calls(a)
    parity.check_step(w, a)
    b = Session(w, keep_scores=True, keep_gathered=True, ksum=a.ksum)
    b.step()
    parity.check_step(w, b)
    assert torch.equal(a.o.sel, b.o.sel) and (a.o.out - b.o.out).abs().max().item() <= 1e-4
    a.close()
    b.close()


# ---- local window (Sec. 4.2, Tier 1 (2)): the last W pages of every request are always selected ------------
@pytest.mark.parametrize("name,window", [("c1_small", 1), ("c2_small", 16), ("c3_small", 2), ("c4_small", 8), ("c5_small", 3),
                                         ("k_exceeds_pages", 8), ("k_exceeds_pages", 24)])
def test_local_window(name, window):
    cfg = CASES[name]
    window = min(window, cfg.top_k)
    w = W.generate(cfg, seed=23, device=DEV)
    a = Session(w, keep_scores=True, keep_gathered=True, local_window_pages=window)
    a.step()
    parity.check_step(w, a)
    sel, n_sel = a.o.sel.cpu().numpy(), a.o.n_sel.cpu().numpy()
    ctx = w.ctx_len.cpu().numpy()
    for b in range(cfg.batch):
        P = -(-int(ctx[b]) // cfg.page_size)
        w_eff = min(window, P)
        for h in range(cfg.n_q_heads):
            n = int(n_sel[b, h])
            assert list(sel[b, h, n - w_eff:n]) == list(range(P - w_eff, P))
    b_ = Session(w, keep_scores=True, keep_gathered=True, ksum=a.ksum, local_window_pages=window)
    run_separate_calls(b_)
    parity.check_step(w, b_)
    assert torch.equal(a.o.sel, b_.o.sel)
    a.close()
    b_.close()


def test_local_window_covering_all_of_k_and_longer_than_a_request():
    cfg = small("c3_batched", batch=3, ctx_len=16 * 40, top_k=12, n_topics=4)
    w = W.generate(cfg, seed=29, device=DEV)
    w.ctx_len[1] = 16 * 5 + 3                               # 6 pages < window
    a = Session(w, keep_scores=True, keep_gathered=True, local_window_pages=12)
    a.step()
    parity.check_step(w, a)
    a.close()
    with pytest.raises(B.SwarmError):
        Session(w, local_window_pages=13)


# ---- every list-length variant of the selection kernel, with and without a local window --------------------
@pytest.mark.parametrize("pages,top_k,window", [(4097, 1, 0), (4999, 100, 3), (8192, 512, 0), (9001, 700, 9)])
def test_selection_of_many_long_lists(pages, top_k, window):
    """136 lists longer than a register-resident CTA takes when there are many: keys in shared memory, row lengths that
    16-byte loads reach and do not, tied scores in one request, contexts that end anywhere (the last request has one page)."""
    cfg = small("c5_skewed", batch=17, n_q_heads=8, n_kv_heads=1, ctx_range=None, ctx_len=16 * pages - 5, top_k=top_k, n_topics=8)
    w = W.generate(cfg, seed=pages, device=DEV)
    lens = torch.randint(1, 16 * pages - 4, (17,), generator=torch.Generator().manual_seed(pages), dtype=torch.int32)
    lens[0], lens[-1] = 16 * pages - 5, 7
    w.ctx_len.copy_(lens)
    w.q[3].zero_()                                          # every score of request 3 is 0
    sess = Session(w, keep_scores=True, local_window_pages=min(window, top_k))
    sess.step()
    torch.cuda.synchronize()
    assert sess.status() == 0
    sc, sel = sess.o.scores.cpu().numpy(), sess.o.sel.cpu().numpy()
    want, n_want = oracle.topk(sc, lens.numpy(), cfg.page_size, top_k, min(window, top_k))
    assert np.array_equal(sel, want) and np.array_equal(sess.o.n_sel.cpu().numpy(), n_want)
    parity.check_resolve(w, parity.host_tables(w), sel, sess.o.n_sel.cpu().numpy(), sess.o.uniq.cpu().numpy(), sess.o.queue_of.cpu().numpy(),
                         sess.o.n_uniq.cpu().numpy()[0], sess.o.queue_load.cpu().numpy())
    sess.close()


@pytest.mark.parametrize("heads", [4, 136])
@pytest.mark.parametrize("pages,top_k,window", [(32769, 150, 0), (40000, 64, 0), (40000, 39000, 7), (48160, 150, 5), (48160, 48000, 0), (48161, 150, 0)])
def test_selection_where_more_pages_tie_than_a_signed_half_word_holds(pages, top_k, window, heads):
    """Long lists with nearly all scores equal, as few lists and as many, up to the longest one with its keys in shared
    memory (48160 pages) and one page more.  The keys of all but 100 pages are zero, so those tie at score 0 behind
    the 100; for the first head the query is zero and every page ties."""
    cfg = small("c1_tiny", ctx_len=16 * pages - 3, top_k=top_k, n_q_heads=heads, n_kv_heads=1)
    w = W.generate(cfg, seed=pages, device=DEV)
    keep = torch.randperm(pages, generator=torch.Generator().manual_seed(pages))[:100].to(DEV)
    some = w.kv_pool[keep, :, 0].clone()
    w.kv_pool[:, :, 0] = 0
    w.kv_pool[keep, :, 0] = some
    w.q[0, 0] = 0
    sess = Session(w, keep_scores=True, local_window_pages=window)
    lens = w.ctx_len.cpu().numpy()

    def check():
        torch.cuda.synchronize()
        assert sess.status() == 0
        sc, sel, n_sel = (t.cpu().numpy() for t in (sess.o.scores, sess.o.sel, sess.o.n_sel))
        assert (sc == 0).sum(axis=-1).min() >= pages - 100
        want, n_want = oracle.topk(sc, lens, cfg.page_size, top_k, window)
        assert np.array_equal(sel, want) and np.array_equal(n_sel, n_want)
        return sel, n_sel

    sess.select()
    check()
    if heads == 4:                                          # inside the step it marks the selected pages' clusters too
        sess.step()
        sel, n_sel = check()
        parity.check_resolve(w, parity.host_tables(w), sel, n_sel, sess.o.uniq.cpu().numpy(), sess.o.queue_of.cpu().numpy(),
                             sess.o.n_uniq.cpu().numpy()[0], sess.o.queue_load.cpu().numpy())
    sess.close()


@pytest.mark.parametrize("pages", [900, 2000, 4000, 8000, 16000, 30000, 45000])
@pytest.mark.parametrize("window", [0, 5])
def test_selection_at_every_list_length(pages, window):
    cfg = small("c1_tiny", batch=2, n_q_heads=2, n_kv_heads=1, ctx_len=16 * pages - 7, top_k=100, n_topics=8)
    w = W.generate(cfg, seed=31, device=DEV)
    w.ctx_len[1] = 16 * (pages // 3) + 1                    # a shorter request beside the long one
    sess = Session(w, keep_scores=True, local_window_pages=window)
    sess.select()
    torch.cuda.synchronize()
    assert sess.status() == 0
    sc = sess.o.scores.cpu().numpy()
    sel, n_sel = sess.o.sel.cpu().numpy(), sess.o.n_sel.cpu().numpy()
    ctx = w.ctx_len.cpu().numpy()
    want, n_want = oracle.topk(sc, ctx, cfg.page_size, cfg.top_k, window)
    assert np.array_equal(n_sel, n_want) and np.array_equal(sel, want)
    # the fused step marks the same pages and attends to them
    sess.step()
    torch.cuda.synchronize()
    assert np.array_equal(sess.o.sel.cpu().numpy(), want)
    parity.check_step(w, sess, requests=[1], heads=[1])
    sess.close()


# ---- medoid index (Sec. 4.2 Tier 1 (1)): clusters are scored by their medoid page and retrieved whole -------
def check_medoid_step(w, sess, k_c, flags=0, window=0):
    torch.cuda.synchronize()
    assert sess.status() == 0
    cfg = w.cfg
    tabs = parity.host_tables(w)
    ptr, members, medoid = (t.cpu().numpy() for t in (sess.cluster_page_ptr, sess.cluster_pages, sess.medoid_page))
    ksum = W.bits_u16(sess.ksum)
    rows_gpu = W.bits_u16(sess.medoid_ksum)
    rows_ref = oracle.medoid_rows(ksum, tabs["page_base"], tabs["cluster_base"], medoid)
    assert np.array_equal(rows_gpu[: len(rows_ref)], rows_ref), "medoid index rows differ"
    sel_c, n_sel_c = sess.sel_clusters.cpu().numpy(), sess.n_sel_clusters.cpu().numpy()
    r = oracle.medoid_step(W.bits_u16(w.q), ksum, W.bits_u16(w.kv_pool), tabs["page_base"], tabs["ctx_len"],
                           tabs["page2cluster"], tabs["cluster_base"], tabs["replica_mask"], tabs["cluster_size"],
                           ptr, members, medoid, Hkv=cfg.n_kv_heads, S=cfg.page_size, k_c=k_c, D=cfg.n_queues,
                           flags=flags, sel_override=(sel_c, n_sel_c), window=window)
    cb = tabs["cluster_base"]
    exact = 0
    for b in range(cfg.batch):
        n_c = int(cb[b + 1] - cb[b])
        if sess.cluster_scores is not None:
            sc = sess.cluster_scores[b].cpu().numpy()
            parity.check_scores(sc, r.score64[b], r.cond[b], n_c)
            on_gpu_scores, _ = oracle.topk(sc[None, :, :n_c], np.array([n_c * cfg.page_size], np.int32),
                                           cfg.page_size, k_c)
            assert np.array_equal(on_gpu_scores[0], sel_c[b]), "not the exact top-k of the GPU's own cluster scores"
        for h in range(cfg.n_q_heads):
            parity.check_selection(sel_c[b, h], int(n_sel_c[b, h]), r.score64[b, h], n_c, k_c)
            exact += int(np.array_equal(sel_c[b, h], r.sel_clusters[b, h]))
    o = sess.o
    n = int(o.n_uniq.cpu().numpy()[0])
    assert n == len(r.uniq) and np.array_equal(o.uniq.cpu().numpy()[:n], r.uniq)
    assert np.array_equal(o.queue_of.cpu().numpy()[:n], r.queue_of)
    assert np.array_equal(o.queue_load.cpu().numpy()[: cfg.n_queues], r.load)
    parity.check_attention(o.out.cpu().numpy(), o.lse.cpu().numpy(), r.out, r.lse)
    return exact


@pytest.mark.parametrize("name,k_c", [("c1_small", 6), ("c2_small", 12), ("c3_small", 5), ("c4_small", 9),
                                      ("c5_small", 4), ("k_exceeds_pages", 7)])
def test_medoid_step_matches_oracle(name, k_c):
    w = W.generate(CASES[name], seed=37, device=DEV)
    sess = Session(w)
    sess.enable_medoid_index(k_c, keep_scores=True)
    sess.step_medoid()
    exact = check_medoid_step(w, sess, k_c)
    assert exact >= 0.9 * w.cfg.batch * w.cfg.n_q_heads
    # the page step still works on the same session afterwards, and the medoid step again after it
    sess.step()
    torch.cuda.synchronize()
    first = sess.sel_clusters.clone()
    sess.step_medoid()
    torch.cuda.synchronize()
    assert torch.equal(first, sess.sel_clusters)
    check_medoid_step(w, sess, k_c)
    sess.close()


def test_medoid_step_rejects_bad_arguments_and_flags_bad_members():
    w = W.generate(CASES["c3_small"], seed=41, device=DEV)
    sess = Session(w, keep_gathered=True)
    sess.enable_medoid_index(4)
    with pytest.raises(B.SwarmError):                       # gathered outputs are not part of this step
        B.swarm_step_medoid(sess.ctx, sess.inputs, sess.medoid_index, sess.outputs)
    bad = B.make_medoid_index(medoid_ksum=sess.medoid_ksum, cluster_page_ptr=sess.cluster_page_ptr,
                              cluster_pages=sess.cluster_pages, cluster_ctx_len=sess.cluster_ctx_len, top_k_clusters=0,
                              max_clusters_per_req=sess.max_clusters_per_req)
    with pytest.raises(B.SwarmError):
        B.swarm_step_medoid(sess.ctx, sess.inputs, bad, sess.medoid_outputs)
    sess.cluster_pages.fill_(1 << 20)                       # members outside every request: flagged, never followed
    sess.step_medoid()
    torch.cuda.synchronize()
    assert sess.status() & B.DEV_BAD_PAGE
    sess.cluster_page_ptr.fill_(1 << 40)                    # member offsets beyond the member array: skipped
    sess.step_medoid()
    torch.cuda.synchronize()
    assert sess.status() & B.DEV_BAD_CLUSTER
    sess.close()


def test_medoid_step_full_size_c2():
    w = W.generate(W.CONFIGS["c2_128k"], seed=43, device=DEV)
    sess = Session(w)
    sess.enable_medoid_index(32, keep_scores=True)          # 32 clusters of 8 pages: the page step's 256 pages per head
    sess.step_medoid()
    check_medoid_step(w, sess, 32)
    sess.close()


# ---- batched submission order (Sec. 5.1): heads of all buckets per batch -----------------------------------
def check_submit_order(w, sess, flags=0):
    torch.cuda.synchronize()
    tabs = parity.host_tables(w)
    n = int(sess.o.n_uniq.cpu().numpy()[0])
    uniq = sess.o.uniq.cpu().numpy()[:n]
    queue_of = sess.o.queue_of.cpu().numpy()[:n]
    want, rounds = oracle.submit_order(queue_of, tabs["replica_mask"][uniq], w.cfg.n_queues, flags)
    info = sess.submit_info.cpu().numpy()
    assert info[0] == rounds and info[1] == len(want)
    assert np.array_equal(sess.submit_order.cpu().numpy()[: len(want)], want)
    return len(want)


@pytest.mark.parametrize("flags", [0, B.ORDER_BY_ID])
@pytest.mark.parametrize("name", ["c2_small", "c3_small", "c5_small"])
def test_submit_order_matches_oracle(name, flags):
    w = W.generate(CASES[name], seed=47, device=DEV)
    sess = Session(w, flags=flags)
    sess.enable_submit_order()
    sess.step()
    parity.check_step(w, sess, flags=flags)
    assert check_submit_order(w, sess, flags) > 0
    sess.submit_order.fill_(-1)
    sess.select()
    sess.resolve()                                          # the separate call writes it too
    check_submit_order(w, sess, flags)
    sess.enable_medoid_index(5)
    sess.step_medoid()
    check_submit_order(w, sess, flags)
    B.swarm_set_submit_order(sess.ctx, None, None)          # detached: nothing is written any more
    sess.submit_order.fill_(-7)
    sess.step()
    torch.cuda.synchronize()
    assert int(sess.submit_order.max()) == -7
    sess.close()


def test_submit_order_full_size_and_bad_masks():
    w = W.generate(W.CONFIGS["c3_batched"], seed=53, device=DEV)     # 3071 clusters, half of them with two replicas
    sess = Session(w)
    sess.enable_submit_order()
    sess.step()
    assert check_submit_order(w, sess) > 2000
    w.cluster_replica_mask[::7] = 0                         # no replica anywhere: never submitted
    sess.step()
    torch.cuda.synchronize()
    assert sess.status() & B.DEV_BAD_REPLICA
    check_submit_order(w, sess)
    sess.close()


@pytest.mark.parametrize("batch,topics", [(1, 4), (11, 4)])
def test_submit_order_at_the_ends_of_its_range(batch, topics):
    """A list shorter than the warps that rank it (20 clusters), and one whose keys (45056) come to shared memory in two parts."""
    pages = 40 if batch == 1 else 8192
    cfg = small("c3_batched", batch=batch, ctx_len=16 * pages, top_k=pages, n_q_heads=1, n_kv_heads=1, n_topics=topics, cluster_pages=2,
                replication="two", n_queues=12)
    w = W.generate(cfg, seed=batch, device=DEV)
    sess = Session(w)
    sess.enable_submit_order()
    sess.step()
    torch.cuda.synchronize()
    assert sess.status() == 0
    assert check_submit_order(w, sess) == w.n_clusters
    sess.close()


# ---- Algorithm 1 (offline co-activation clustering) ---------------------------------------------------------
def check_clusters(dist, tau, cap=None):
    density, ptr, members, medoid = B.swarm_build_clusters(dist, tau, members_cap=cap)
    torch.cuda.synchronize()
    d_host = dist.cpu().numpy()
    # the rule: every step agrees with Eq. 5's plain average (double, from scratch) outside a band of 1e-5 * tau
    # around the radius; where no decision falls inside the band the clustering is the plain oracle's exactly
    near = oracle.replay_clusters(d_host, tau, ptr.cpu().numpy(), members.cpu().numpy(), medoid.cpu().numpy(), near_rtol=1e-5)
    rho_p, ptr_p, members_p, medoid_p, near_p = oracle.build_clusters_plain(d_host, tau, members_cap=cap, near_rtol=1e-5)
    assert np.array_equal(density.cpu().numpy(), rho_p)
    if near == 0 and near_p == 0:
        assert np.array_equal(ptr.cpu().numpy(), ptr_p) and np.array_equal(members.cpu().numpy(), members_p)
        assert np.array_equal(medoid.cpu().numpy(), medoid_p)
    # and, beyond the rule, the fp32 reading of the oracle (running sum in joining order) bit for bit
    rho, ptr_ref, members_ref, medoid_ref = oracle.build_clusters(d_host, tau, members_cap=cap)
    assert np.array_equal(density.cpu().numpy(), rho)
    assert np.array_equal(medoid.cpu().numpy(), medoid_ref)
    assert np.array_equal(ptr.cpu().numpy(), ptr_ref)
    assert np.array_equal(members.cpu().numpy(), members_ref)
    return len(medoid_ref), len(members_ref)


@pytest.mark.parametrize("n,topics,tau", [(5, 1, 0.5), (37, 3, 0.4), (256, 8, 0.38), (1000, 20, 0.4),
                                          (1027, 12, 0.33), (2048, 64, 0.45), (3000, 30, 0.05), (600, 4, 1.0),
                                          (8192, 64, 0.4)])
def test_algorithm1_matches_oracle(n, topics, tau):
    dist = W.coactivation_distances(n, topics, seed=n, device=DEV)
    n_clusters, n_members = check_clusters(dist, tau, cap=64 * n if tau < 1.0 else None)
    assert n_members >= n and n_clusters >= 1
    if tau == 0.05:
        assert n_clusters == n                              # radius below every distance: singletons
    if tau == 1.0:
        assert n_clusters == 1 and n_members == n           # radius above every distance: one cluster


@pytest.mark.parametrize("n,frac,symmetric", [(1, 0.5, True), (33, 0.5, False), (129, 0.9, False), (513, 0.45, True),
                                              (1025, 0.999, True), (1026, 0.999, False), (1300, 0.9, True),
                                              (2049, 0.03, False), (2304, 0.5, True)])
def test_algorithm1_on_unstructured_distances(n, frac, symmetric):
    """Uniform random distances, candidate lists that threads hold (up to 384), that are sorted by counting (up to 1024) and
    longer ones, asymmetric matrices, ties (distances on a grid of 1/512)."""
    g = torch.Generator(device=DEV).manual_seed(n)
    dist = torch.randint(0, 512, (n, n), generator=g, device=DEV).to(torch.float32) / 512
    if symmetric:
        dist = torch.minimum(dist, dist.T).contiguous()
        tau = 1.0 - (1.0 - frac) ** 0.5                     # a fraction `frac` of the entries lies within tau
    else:
        tau = frac
    dist.fill_diagonal_(0.0)
    rho, ptr_ref, members_ref, medoid_ref = oracle.build_clusters(dist.cpu().numpy(), tau, members_cap=400 * n)
    density, ptr, members, medoid = B.swarm_build_clusters(dist, tau, members_cap=400 * n)
    assert np.array_equal(density.cpu().numpy(), rho) and np.array_equal(medoid.cpu().numpy(), medoid_ref)
    assert np.array_equal(ptr.cpu().numpy(), ptr_ref) and np.array_equal(members.cpu().numpy(), members_ref)
    if len(members_ref) > n:                                # one place too few: flagged, nothing written past the end
        with pytest.raises(B.SwarmError):
            B.swarm_build_clusters(dist, tau, members_cap=max(n, len(members_ref) - 1))


@pytest.mark.parametrize("n", [2, 32, 34, 384, 385, 386, 1025, 1026])
def test_algorithm1_at_the_ends_of_its_candidate_lists(n):
    """Nearly every entry a candidate of every other: lists that end at a block of 32, at the 384 candidates that threads
    hold and at the 1024 that are sorted by counting.  Distances in general position (few ties)."""
    g = torch.Generator(device=DEV).manual_seed(n)
    dist = torch.rand((n, n), generator=g, device=DEV)
    dist.fill_diagonal_(0.0)
    check = [oracle.build_clusters(dist.cpu().numpy(), tau, members_cap=400 * n) for tau in (0.999, 0.55)]
    for tau, (rho, ptr_ref, members_ref, medoid_ref) in zip((0.999, 0.55), check):
        density, ptr, members, medoid = B.swarm_build_clusters(dist, tau, members_cap=400 * n)
        assert np.array_equal(density.cpu().numpy(), rho) and np.array_equal(medoid.cpu().numpy(), medoid_ref)
        assert np.array_equal(ptr.cpu().numpy(), ptr_ref) and np.array_equal(members.cpu().numpy(), members_ref)


@pytest.mark.parametrize("n,reach", [(1024, 513), (1024, 514), (3075, 769), (3075, 770), (2050, 2050), (8193, 8193)])
def test_algorithm1_on_lists_whose_sums_are_kept_by_entry(n, reach):
    """Eight entries within the radius of the first `reach`, which lie at random from one another, about half of them within
    it: lists of reach - 1 and about half as many candidates of which some join.  The lengths are those at which the sums of
    candidates behind the first 384 move from the candidates' order to the entries' (8 (reach - 1 - 384) > n), and lists of
    all entries."""
    g = torch.Generator(device=DEV).manual_seed(n + reach)
    dist = torch.rand((n, n), generator=g, device=DEV)
    dist[reach:] = 2.0
    dist[:, reach:] = 2.0
    dist[:8, :reach] = 0.25 + dist[:8, :reach] / 16
    dist[:reach, :8] = dist[:8, :reach].T
    dist.fill_diagonal_(0.0)
    rho, ptr_ref, members_ref, medoid_ref = oracle.build_clusters(dist.cpu().numpy(), 0.5, members_cap=400 * n)
    assert rho.max() == reach - 1 and len(medoid_ref) > n - reach
    density, ptr, members, medoid = B.swarm_build_clusters(dist, 0.5, members_cap=400 * n)
    assert np.array_equal(density.cpu().numpy(), rho) and np.array_equal(medoid.cpu().numpy(), medoid_ref)
    assert np.array_equal(ptr.cpu().numpy(), ptr_ref) and np.array_equal(members.cpu().numpy(), members_ref)


def test_algorithm1_with_more_members_than_the_scratch_holds():
    """40 entries sit within reach of all 600, the others only of those: about 555 clusters of 41 members, more than the 16
    memberships per entry that the binding makes room for by itself, and many more clusters than a round grows."""
    n, hubs, tau = 600, 40, 0.1
    d = np.ones((n, n), dtype=np.float32)
    d[:hubs, :] = d[:, :hubs] = 0.03125
    np.fill_diagonal(d, 0.0)
    n_clusters, n_members = check_clusters(torch.from_numpy(d).to(DEV), tau, cap=64 * n)
    assert n_members > 16 * n and n_clusters > 500


def test_algorithm1_hand_case_and_capacity():
    d = np.full((5, 5), 0.9, dtype=np.float32)
    np.fill_diagonal(d, 0.0)
    for (i, j), v in {(0, 1): 0.1, (0, 2): 0.2, (1, 2): 0.3, (3, 4): 0.1, (2, 3): 0.4, (2, 4): 0.5}.items():
        d[i, j] = d[j, i] = v
    dist = torch.from_numpy(d).to(DEV)
    density, ptr, members, medoid = B.swarm_build_clusters(dist, 0.5)
    assert density.tolist() == [2, 2, 4, 2, 2] and ptr.tolist() == [0, 3, 6]
    assert members.tolist() == [2, 0, 1, 3, 4, 2] and medoid.tolist() == [2, 3]
    with pytest.raises(B.SwarmError):                       # six memberships do not fit five slots
        B.swarm_build_clusters(dist, 0.5, members_cap=5)
    with pytest.raises(B.SwarmError):
        B.swarm_build_clusters(dist, -1.0)


def test_algorithm1_on_a_stream_beside_pending_work():
    """The outputs may be memory that work still pending on the current stream is about to write: the call's stream waits
    for it."""
    n, cap = 64, 300000
    dist = W.coactivation_distances(n, 4, seed=3, device=DEV)
    want = B.swarm_build_clusters(dist, 0.4, members_cap=cap)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(3):
        blocks = [torch.empty(words, dtype=torch.int32, device=DEV) for words in (cap + 4 * n, cap + 3 * n + 12)]
        torch.cuda._sleep(20_000_000)                       # about 10 ms in front of the writes
        for t in blocks:
            t.fill_(7)
        del blocks, t
        got = B.swarm_build_clusters(dist, 0.4, members_cap=cap, stream=side)
        for a, b in zip(got, want):
            assert torch.equal(a, b)


def test_algorithm1_from_two_threads_on_streams_of_their_own():
    """Two threads cluster different matrices at the same time, one of them beside decode steps of a third stream."""
    dists = [W.coactivation_distances(n, n // 32, seed=n, device=DEV) for n in (2048, 1500)]
    want = [B.swarm_build_clusters(d, 0.4) for d in dists]
    w = W.generate(CASES["c2_small"], seed=21, device=DEV)
    sess = Session(w)
    sess.step()
    torch.cuda.synchronize()
    out = sess.o.out.clone()
    wrong = []

    def work(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(25):
                got = B.swarm_build_clusters(dists[i], 0.4)
                if not all(torch.equal(a, b) for a, b in zip(got, want[i])):
                    wrong.append(i)

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for _ in range(200):
        sess.step()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not wrong and sess.status() == 0 and torch.equal(sess.o.out, out)
    sess.close()


def test_algorithm1_clusters_drive_the_medoid_step():
    """Clusters with replicas built on the GPU from a distance matrix, then used as the index of the medoid step."""
    cfg = small("c2_128k", ctx_len=16 * 640, top_k=32, n_topics=8)
    w = W.generate(cfg, seed=59, device=DEV)
    P = cfg.max_pages()
    dist = W.coactivation_distances(P, 16, seed=61, device=DEV)
    density, ptr, members, medoid = B.swarm_build_clusters(dist, 0.4, members_cap=64 * P)
    C = len(medoid)
    assert len(members) > P                                 # some pages sit in several clusters
    # cluster tables of the workload replaced by the ones just built (one request)
    sizes = (ptr[1:] - ptr[:-1]).to(torch.int16)
    rng = np.random.default_rng(3)
    mask = torch.from_numpy(np.array([(1 << int(a)) | (1 << int(b)) for a, b in
                                      zip(rng.integers(0, 8, C), rng.integers(0, 8, C))], dtype=np.int32)).to(DEV)
    w.cluster_base = torch.tensor([0, C], dtype=torch.int64, device=DEV)
    w.cluster_replica_mask, w.cluster_size = mask, sizes
    w.page2cluster = torch.zeros(P, dtype=torch.int32, device=DEV)      # not read by the medoid step
    sess = Session(w)
    k_c = 6
    sess.cluster_page_ptr, sess.cluster_pages, sess.medoid_page = ptr.to(torch.int64), members, medoid
    sess.max_clusters_per_req = C
    sess.medoid_ksum = torch.empty((C, cfg.n_kv_heads, 2, cfg.head_dim), dtype=torch.bfloat16, device=DEV)
    sess.cluster_ctx_len = torch.empty(4, dtype=torch.int32, device=DEV)
    B.swarm_build_medoid_index(sess.ctx, sess.inputs, medoid, sess.medoid_ksum, sess.cluster_ctx_len)
    sess.medoid_index = B.make_medoid_index(medoid_ksum=sess.medoid_ksum, cluster_page_ptr=sess.cluster_page_ptr,
                                            cluster_pages=members, cluster_ctx_len=sess.cluster_ctx_len,
                                            top_k_clusters=k_c, max_clusters_per_req=C)
    i32 = dict(dtype=torch.int32, device=DEV)
    sess.sel_clusters = torch.empty((1, cfg.n_q_heads, k_c), **i32)
    sess.n_sel_clusters = torch.empty((1, cfg.n_q_heads), **i32)
    sess.cluster_scores = None
    o = sess.o
    sess.medoid_outputs = B.make_outputs(sel=sess.sel_clusters, n_sel=sess.n_sel_clusters, uniq=o.uniq,
                                         queue_of=o.queue_of, n_uniq=o.n_uniq, queue_load=o.queue_load, out=o.out,
                                         lse=o.lse)
    sess.step_medoid()
    torch.cuda.synchronize()
    assert sess.status() == 0
    # oracle: scores/top-k over the medoids, union of the members, scheduling of the selected clusters
    tabs = parity.host_tables(w)
    ksum = W.bits_u16(sess.ksum)
    rows = oracle.medoid_rows(ksum, tabs["page_base"], tabs["cluster_base"], medoid.cpu().numpy())
    len_c = np.array([C * cfg.page_size], np.int32)
    s64, s32, cond = oracle.scores(W.bits_u16(w.q), rows, tabs["cluster_base"], len_c, cfg.n_kv_heads, cfg.page_size, C)
    sel_c, n_sel_c = sess.sel_clusters.cpu().numpy(), sess.n_sel_clusters.cpu().numpy()
    for h in range(cfg.n_q_heads):
        parity.check_selection(sel_c[0, h], int(n_sel_c[0, h]), s64[0, h], C, k_c)
    sel_p, n_sel_p = oracle.expand_clusters(sel_c, n_sel_c, tabs["cluster_base"], ptr.cpu().numpy(), members.cpu().numpy())
    ident = np.arange(C, dtype=np.int32)                     # scheduling sees the selected clusters themselves
    uniq, queue_of, load = oracle.resolve(sel_c, n_sel_c, tabs["cluster_base"], ident, tabs["cluster_base"],
                                          tabs["replica_mask"], tabs["cluster_size"], cfg.n_queues, 0)
    n = int(o.n_uniq.cpu().numpy()[0])
    assert n == len(uniq) and np.array_equal(o.uniq.cpu().numpy()[:n], uniq)
    assert np.array_equal(o.queue_of.cpu().numpy()[:n], queue_of)
    assert np.array_equal(o.queue_load.cpu().numpy()[: cfg.n_queues], load)
    k_g, v_g, n_tok = oracle.gather(W.bits_u16(w.kv_pool), sel_p, n_sel_p, tabs["page_base"], tabs["ctx_len"],
                                    cfg.n_kv_heads, cfg.head_dim, cfg.page_size)
    out, lse = oracle.attention(W.bits_u16(w.q), k_g, v_g, n_tok)
    parity.check_attention(o.out.cpu().numpy(), o.lse.cpu().numpy(), out, lse)
    sess.close()

    # entry-level scheduling (the paper's exact model): every page of the selected clusters is a unit of its own,
    # with the copies Eq. 7 gives it -- one per cluster that stores it
    entry_masks = oracle.entry_replica_masks(ptr.cpu().numpy(), members.cpu().numpy(), P, cfg.n_queues)
    assert (np.array([bin(int(x)).count("1") for x in entry_masks]) > 1).any()
    sess = Session(w, max_clusters_total=P)
    sess.medoid_ksum = torch.empty((C, cfg.n_kv_heads, 2, cfg.head_dim), dtype=torch.bfloat16, device=DEV)
    len_dev = torch.empty(4, dtype=torch.int32, device=DEV)
    B.swarm_build_medoid_index(sess.ctx, sess.inputs, medoid, sess.medoid_ksum, len_dev)
    masks_dev = torch.from_numpy(entry_masks.view(np.int32)).to(DEV)
    ptr64 = ptr.to(torch.int64)                               # kept alive: the index holds its address
    index = B.make_medoid_index(medoid_ksum=sess.medoid_ksum, cluster_page_ptr=ptr64, cluster_pages=members,
                                cluster_ctx_len=len_dev,
                                top_k_clusters=k_c, max_clusters_per_req=C, entry_replica_mask=masks_dev)
    sel_c2 = torch.empty((1, cfg.n_q_heads, k_c), **i32)
    n_sel_c2 = torch.empty((1, cfg.n_q_heads), **i32)
    o = sess.o
    outs = B.make_outputs(sel=sel_c2, n_sel=n_sel_c2, uniq=o.uniq, queue_of=o.queue_of, n_uniq=o.n_uniq,
                          queue_load=o.queue_load, out=o.out, lse=o.lse)
    sess.enable_submit_order()
    B.swarm_step_medoid(sess.ctx, sess.inputs, index, outs)
    torch.cuda.synchronize()
    assert sess.status() == 0
    assert np.array_equal(sel_c2.cpu().numpy(), sel_c)        # same selection as before
    ones = np.ones(P, dtype=np.uint16)
    ident_p = np.arange(P, dtype=np.int32)
    uniq, queue_of, load = oracle.resolve(sel_p, n_sel_p, tabs["page_base"], ident_p, tabs["page_base"], entry_masks, ones,
                                          cfg.n_queues, oracle.UNIT_LOAD)
    n = int(o.n_uniq.cpu().numpy()[0])
    assert n == len(uniq) and np.array_equal(o.uniq.cpu().numpy()[:n], uniq)
    assert np.array_equal(o.queue_of.cpu().numpy()[:n], queue_of)
    assert np.array_equal(o.queue_load.cpu().numpy()[: cfg.n_queues], load) and int(load.sum()) == n
    want_order, rounds = oracle.submit_order(queue_of, entry_masks[uniq], cfg.n_queues)
    assert np.array_equal(sess.submit_order.cpu().numpy()[:n], want_order)
    parity.check_attention(o.out.cpu().numpy(), o.lse.cpu().numpy(), out, lse)
    sess.close()


@pytest.mark.parametrize("name,k_c,window", [("c2_small", 12, 3), ("c5_small", 4, 2), ("k_exceeds_pages", 7, 5),
                                             ("c4_small", 9, 64), ("c3_small", 1, 40)])
def test_medoid_step_with_local_window(name, k_c, window):
    """The paper's whole Tier-1 step: clusters chosen through the medoid index, attended whole, plus the local
    window (requests shorter than the window are attended densely)."""
    cfg = CASES[name]
    window = min(window, cfg.top_k)                         # the shape allows 0 <= W <= top_k
    w = W.generate(cfg, seed=83, device=DEV)
    sess = Session(w, local_window_pages=window)
    sess.enable_medoid_index(k_c, keep_scores=True)
    sess.step_medoid()
    check_medoid_step(w, sess, k_c, window=window)
    sess.step()                                             # the page step with the same window still works
    parity.check_step(w, sess)
    sess.step_medoid()
    check_medoid_step(w, sess, k_c, window=window)
    sess.close()


def test_medoid_step_entry_level_with_local_window():
    """Entry-level scheduling: the window's pages are units of their own, like the members of the selected clusters."""
    cfg = small("c2_128k", ctx_len=16 * 300 + 7, top_k=32, n_topics=6)
    window = 5
    w = W.generate(cfg, seed=89, device=DEV)
    P = cfg.max_pages()
    ptr, members, medoid = W.cluster_members(w)
    entry_masks = oracle.entry_replica_masks(ptr.cpu().numpy(), members.cpu().numpy(), P, cfg.n_queues)
    # give every third page a second copy so that the scheduling has something to decide
    entry_masks = entry_masks.copy()
    entry_masks[::3] |= np.uint32(1) << ((np.arange(P)[::3] // 3) % cfg.n_queues).astype(np.uint32)
    sess = Session(w, local_window_pages=window, max_clusters_total=P)
    sess.enable_medoid_index(4)
    masks_dev = torch.from_numpy(entry_masks.view(np.int32)).to(DEV)
    index = B.make_medoid_index(medoid_ksum=sess.medoid_ksum, cluster_page_ptr=sess.cluster_page_ptr,
                                cluster_pages=sess.cluster_pages, cluster_ctx_len=sess.cluster_ctx_len, top_k_clusters=4,
                                max_clusters_per_req=sess.max_clusters_per_req, entry_replica_mask=masks_dev)
    B.swarm_step_medoid(sess.ctx, sess.inputs, index, sess.medoid_outputs)
    torch.cuda.synchronize()
    assert sess.status() == 0
    tabs = parity.host_tables(w)
    sel_c, n_sel_c = sess.sel_clusters.cpu().numpy(), sess.n_sel_clusters.cpu().numpy()
    sel_p, n_sel_p = oracle.expand_clusters(sel_c, n_sel_c, tabs["cluster_base"], ptr.cpu().numpy(), members.cpu().numpy(),
                                            tabs["ctx_len"], cfg.page_size, window)
    assert all(set(range(P - window, P)) <= set(sel_p[0, h, : n_sel_p[0, h]].tolist()) for h in range(cfg.n_q_heads))
    uniq, queue_of, load = oracle.resolve(sel_p, n_sel_p, tabs["page_base"], np.arange(P, dtype=np.int32), tabs["page_base"],
                                          entry_masks, np.ones(P, dtype=np.uint16), cfg.n_queues, oracle.UNIT_LOAD)
    o = sess.o
    n = int(o.n_uniq.cpu().numpy()[0])
    assert n == len(uniq) and np.array_equal(o.uniq.cpu().numpy()[:n], uniq)
    assert np.array_equal(o.queue_of.cpu().numpy()[:n], queue_of)
    assert np.array_equal(o.queue_load.cpu().numpy()[: cfg.n_queues], load)
    k_g, v_g, n_tok = oracle.gather(W.bits_u16(w.kv_pool), sel_p, n_sel_p, tabs["page_base"], tabs["ctx_len"],
                                    cfg.n_kv_heads, cfg.head_dim, cfg.page_size)
    out, lse = oracle.attention(W.bits_u16(w.q), k_g, v_g, n_tok)
    parity.check_attention(o.out.cpu().numpy(), o.lse.cpu().numpy(), out, lse)
    sess.close()


def test_medoid_step_full_size_c3_and_wide_groups():
    w = W.generate(W.CONFIGS["c3_batched"], seed=67, device=DEV)      # 16 requests, 256 clusters each
    sess = Session(w)
    sess.enable_medoid_index(16, keep_scores=True)
    sess.step_medoid()
    check_medoid_step(w, sess, 16)
    sess.close()
    for name in ("g16_s32", "hkv3_g2", "k1_d1"):                      # 16-head groups on 32-token pages, odd KV heads, one queue
        w = W.generate(EDGE_SHAPES[name], seed=71, device=DEV)
        sess = Session(w)
        sess.enable_medoid_index(3, keep_scores=True)
        sess.step_medoid()
        check_medoid_step(w, sess, 3)
        sess.close()


# ---- admission of clusters to the fast tier by their Eq. 6 score -------------------------------------------
@pytest.mark.parametrize("n,cap_frac", [(5, 0.7), (200, 0.3), (1024, 0.5), (3000, 0.25), (5000, 0.0), (5000, 2.0)])
def test_cache_admission_matches_oracle(n, cap_frac):
    g = torch.Generator(device="cpu").manual_seed(n)
    score = torch.randint(0, 40, (n,), generator=g).to(torch.float32) * 0.25      # many ties
    size = torch.randint(1, 17, (n,), generator=g, dtype=torch.int16)
    cap = int(cap_frac * int(size.sum()))
    resident = torch.full((n + 16,), 7, dtype=torch.uint8, device=DEV)
    info = torch.zeros(4, dtype=torch.int32, device=DEV)
    B.swarm_cache_admit(score.to(DEV), size.to(DEV), cap, resident, info)
    torch.cuda.synchronize()
    want, n_in, used = oracle.cache_admit(score.numpy(), size.numpy().view(np.uint16), cap)
    assert np.array_equal(resident.cpu().numpy()[:n], want) and int(resident[n:].min()) == 7
    assert info.cpu().numpy()[:2].tolist() == [n_in, used]


def test_cache_admission_feeds_the_resident_filter():
    """Scores maintained by the step (Eq. 6) -> admission -> the next step fetches only what is not resident."""
    w = W.generate(CASES["c3_small"], seed=73, device=DEV)
    sess = Session(w)
    C = w.n_clusters
    resident = torch.zeros(C + 16, dtype=torch.uint8, device=DEV)
    freq = torch.zeros(C, dtype=torch.int32, device=DEV)
    score = torch.zeros(C, dtype=torch.float32, device=DEV)
    n_hit = torch.zeros(4, dtype=torch.int32, device=DEV)
    B.swarm_set_cache(sess.ctx, resident=resident, freq=freq, score=score, n_hit=n_hit, t_base=80.0, t_transfer=2.5)
    sess.step()                                             # nothing resident yet: every activated cluster scores
    torch.cuda.synchronize()
    n_first = int(sess.o.n_uniq[0])
    assert int(n_hit[0]) == 0 and int((freq > 0).sum()) == n_first
    B.swarm_cache_admit(score, w.cluster_size, 10_000_000, resident)       # room for everything with a score
    want, _, _ = oracle.cache_admit(score.cpu().numpy(), w.cluster_size.cpu().numpy().view(np.uint16), 10_000_000)
    assert np.array_equal(resident.cpu().numpy()[:C], want) and want.all()
    sess.step()                                             # same query: everything activated is resident now
    torch.cuda.synchronize()
    assert int(sess.o.n_uniq[0]) == 0 and int(n_hit[0]) == n_first
    sess.close()


# ---- the selector report: its figures recomputed on the host in fp64 from the selectors' own lists -------------
@pytest.mark.parametrize("name,k_c", [("c2_small", 12), ("c5_small", 4)])
def test_selector_report_figures(name, k_c):
    from helpers import from_bf16_bits
    from paper_2603_17803_b200 import selector_report as R
    w = W.generate(CASES[name], seed=79, device=DEV)
    rep = R.compare(w, k_c, keep_lists=True)
    cfg, tabs = w.cfg, parity.host_tables(w)
    S, d, g = cfg.page_size, cfg.head_dim, cfg.n_q_heads // cfg.n_kv_heads
    q = from_bf16_bits(W.bits_u16(w.q)).astype(np.float64)
    pool = W.bits_u16(w.kv_pool)
    ptr, members, _ = (t.cpu().numpy() for t in W.cluster_members(w))
    for sel_name in ("pages", "medoids"):
        lists, n_lists = rep[sel_name]["lists"]
        if sel_name == "medoids":                           # the pages those clusters hold
            sel_p, n_p = oracle.expand_clusters(lists, n_lists, tabs["cluster_base"], ptr, members)
        else:
            sel_p, n_p = lists, n_lists
        att_n, mass_r, top_r = [], [], []
        for b in range(cfg.batch):
            ctx = int(tabs["ctx_len"][b])
            P = -(-ctx // S)
            pb = int(tabs["page_base"][b])
            for h in range(cfg.n_q_heads):
                keys = from_bf16_bits(pool[pb:pb + P, h // g, 0]).astype(np.float64).reshape(P * S, d)
                logit = keys @ q[b, h] / np.sqrt(d)
                logit[ctx:] = -np.inf
                prob = np.exp(logit - logit.max())
                mass = (prob / prob.sum()).reshape(P, S).sum(1)
                pages = sel_p[b, h, : n_p[b, h]]
                att_n.append(len(pages))
                mass_r.append(mass[pages].sum())
                best = np.argsort(-mass, kind="stable")[: min(cfg.top_k, P)]
                top_r.append(np.isin(best, pages).mean())
        got = rep[sel_name]
        assert got["attended_pages"] == pytest.approx(np.mean(att_n), rel=1e-6)
        assert got["mass_recall"] == pytest.approx(np.mean(mass_r), abs=2e-4)
        assert got["topk_recall"] == pytest.approx(np.mean(top_r), abs=5e-3)     # near-ties of mass order differently in fp32
        uniq, _, load = oracle.resolve(sel_p, n_p, tabs["page_base"], tabs["page2cluster"], tabs["cluster_base"],
                                       tabs["replica_mask"], tabs["cluster_size"], cfg.n_queues)
        assert got["io_clusters"] == len(uniq) and got["io_pages"] == int(tabs["cluster_size"][uniq].sum())
        assert got["io_pages"] == int(load.sum()) and got["max_queue_load"] == int(load.max())
    # whole clusters attended: the medoid selector's I/O is exactly what its heads attend, no partial clusters
    assert rep["medoids"]["io_pages"] >= rep["medoids"]["attended_pages"]


# ---- the step in two halves: query heads spread over several ctxs (one per GPU in production) ------------------
def test_begin_then_end_is_the_step():
    w = W.generate(CASES["c5_small"], seed=97, device=DEV)
    a, b_ = Session(w), Session(w)
    a.step()
    b_.step_begin()
    flags = b_.cluster_flags()
    assert flags.numel() == w.n_clusters and int(flags.sum()) == int(a.o.n_uniq[0])   # every activated cluster, once
    b_.step_end()
    torch.cuda.synchronize()
    assert int(flags.sum()) == 0                            # consumed
    for name in ("sel", "n_sel", "queue_load", "out", "lse"):
        assert torch.equal(getattr(a.o, name), getattr(b_.o, name)), name
    n = int(a.o.n_uniq[0])
    assert torch.equal(a.o.uniq[:n], b_.o.uniq[:n]) and torch.equal(a.o.queue_of[:n], b_.o.queue_of[:n])
    parity.check_step(w, b_)
    a.close()
    b_.close()


@pytest.mark.parametrize("name,world", [("c2_small", 2), ("c2_small", 4), ("c3_small", 8), ("c5_small", 2)])
def test_head_sharded_step_on_one_device(name, world):
    """`world` ctxs, each with the K/V of its own KV heads, run one after the other on this device; the flag
    exchange (an all-reduce by maximum across GPUs in production) is a plain maximum here.  Every shard must
    derive the unsharded schedule, and the shards' heads together the unsharded selection and attention."""
    from paper_2603_17803_b200 import sharding
    w = W.generate(CASES[name], seed=101, device=DEV)
    full = Session(w)
    full.step()
    parity.check_step(w, full)
    shards = [sharding.shard_workload(w, r, world) for r in range(world)]
    sess = [Session(s, ksum=None) for s in shards]
    for s in sess:
        s.step_begin()
    torch.cuda.synchronize()
    own = [int(s.cluster_flags().sum()) for s in sess]
    union = torch.stack([s.cluster_flags() for s in sess]).amax(0)
    n = int(full.o.n_uniq[0])
    assert int(union.sum()) == n and max(own) <= n
    for s in sess:
        s.cluster_flags().copy_(union)
        s.step_end()
    torch.cuda.synchronize()
    hq = w.cfg.n_q_heads // world
    for r, s in enumerate(sess):
        assert s.status() == 0
        assert int(s.o.n_uniq[0]) == n
        assert torch.equal(s.o.uniq[:n], full.o.uniq[:n]) and torch.equal(s.o.queue_of[:n], full.o.queue_of[:n])
        assert torch.equal(s.o.queue_load[: w.cfg.n_queues], full.o.queue_load[: w.cfg.n_queues])
        assert torch.equal(s.o.sel, full.o.sel[:, r * hq:(r + 1) * hq])
        d_out = (s.o.out - full.o.out[:, r * hq:(r + 1) * hq]).abs().max().item()
        d_lse = (s.o.lse - full.o.lse[:, r * hq:(r + 1) * hq]).abs().max().item()
        assert d_out <= parity.ATTN_ATOL and d_lse <= parity.LSE_ATOL   # split counts differ between the layouts
        assert int(s.cluster_flags().sum()) == 0
    # sharding.sharded_step without a process group is the plain step
    sharding.sharded_step(sess[0])
    torch.cuda.synchronize()
    parity.check_step(shards[0], sess[0])
    for s in sess:
        s.close()
    full.close()


@pytest.mark.parametrize("page,ctx_len", [(16, [16 * 37 + 1, 5, 16 * 3]), (32, [32 * 9 + 31, 1, 33])])
def test_summaries_of_special_values(page, ctx_len):
    """Minima and maxima are whole values: denormals are kept, -0 lies below +0, infinities count, NaN does not."""
    cfg = W.scaled(W.CONFIGS["c5_skewed"], batch=len(ctx_len), ctx_range=(1, max(ctx_len)), page_size=page, top_k=2, n_topics=2)
    w = W.generate(cfg, seed=5, device=DEV)
    assert int((w.page_base[1:] - w.page_base[:-1]).min()) >= 1
    lens = [min(n, int(w.page_base[b + 1] - w.page_base[b]) * page) for b, n in enumerate(ctx_len)]
    w.ctx_len.copy_(torch.tensor(lens, dtype=torch.int32))
    values = np.array([0x0000, 0x8000, 0x0001, 0x8001, 0x007F, 0x807F, 0x3F80, 0xBF80, 0x7F7F, 0xFF7F, 0x7F80, 0xFF80, 0x7FC0, 0xFFC1], dtype=np.uint16)
    bits = np.random.default_rng(7).choice(values, size=w.kv_pool.shape, p=[.3, .3] + [.4 / 12] * 12)
    w.kv_pool.copy_(torch.from_numpy(bits.view(np.int16)).view(torch.bfloat16))
    sess = Session(w)
    torch.cuda.synchronize()
    got = sess.ksum.view(torch.int16).cpu().numpy().view(np.uint16)
    key = np.where(bits & 0x8000, 0x7FFF - (bits & 0x7FFF).astype(np.int32), 0x8000 + bits.astype(np.int32))   # sign-magnitude order
    nan = (bits & 0x7FFF) > 0x7F80
    for b, n in enumerate(lens):
        base = int(w.page_base[b])
        for p in range(-(-n // page)):
            tok = slice(0, min(page, n - p * page))
            for part, empty, reduce in ((0, 0x7F80, np.argmin), (1, 0xFF80, np.argmax)):
                k = np.where(nan[base + p, :, 0, tok], 1 << 20 if part == 0 else -1, key[base + p, :, 0, tok])
                at = reduce(k, axis=1)
                want = np.take_along_axis(bits[base + p, :, 0, tok], at[:, None], axis=1)[:, 0]
                want = np.where(nan[base + p, :, 0, tok].all(axis=1), empty, want)
                assert np.array_equal(got[base + p, :, part], want), (b, p, part)
    sess.close()


@pytest.mark.parametrize("own_stream", [True, False])
@pytest.mark.parametrize("name", ["c2_small", "c3_small", "c5_small"])
def test_step_host_directly_behind_an_index_build(name, own_stream):
    """The host step's scorer asks for its first summaries while the queries travel: still after whatever precedes the call in its
    stream, here the summaries of a pool rewritten every turn (the recorded graph on a stream of its own; plain launches)."""
    w = W.generate(CASES[name], seed=23, device=DEV)
    pools = [w.kv_pool.clone(), w.kv_pool.flip(1)]          # (the KV heads in the other order)
    q_host = w.q.cpu().pin_memory()
    out_host = torch.empty((w.cfg.batch, w.cfg.n_q_heads, w.cfg.head_dim), dtype=torch.float32).pin_memory()
    want = []
    for pool in pools:
        w.kv_pool.copy_(pool)
        ref = Session(w)
        torch.cuda.synchronize()
        ref.step()
        torch.cuda.synchronize()
        want.append((ref.o.sel.clone(), ref.o.out.cpu()))
        ref.close()
    sess = Session(w)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream() if own_stream else None
    for turn in range(8):
        with torch.cuda.stream(stream or torch.cuda.current_stream()):
            w.kv_pool.copy_(pools[turn % 2])
            B.swarm_build_summaries(sess.ctx, sess.inputs, sess.ksum)
            sess.step_host(q_host, out_host, stream=stream)
        assert torch.equal(out_host, want[turn % 2][1]), turn
        torch.cuda.synchronize()
        assert sess.status() == 0 and torch.equal(sess.o.sel, want[turn % 2][0])
    sess.close()


@pytest.mark.parametrize("n", [3, 146, 147, 148, 149, 297, 1483])
def test_algorithm1_order_of_equal_densities(n):
    """The walk starts with the densest entries, ties with the lower index first: a few densities shared by many entries, entries
    around multiples of the CTAs that count them (each its own stretch)."""
    rng = np.random.default_rng(n)
    kind = rng.integers(0, 5, size=n)                     # five blocks of near entries, far from the others
    dist = np.where(kind[:, None] == kind[None, :], 0.125, 0.875).astype(np.float32)
    np.fill_diagonal(dist, 0.0)
    dist[rng.integers(0, n, size=n // 3), rng.integers(0, n, size=n // 3)] = 0.375   # some rows of other densities
    np.fill_diagonal(dist, 0.0)
    for tau in (0.0625, 0.25, 0.5):                       # nobody near, the blocks, the blocks and the odd ones
        rho, ptr_ref, members_ref, medoid_ref = oracle.build_clusters(dist, tau, members_cap=64 * n)
        density, ptr, members, medoid = B.swarm_build_clusters(torch.from_numpy(dist).to(DEV), tau, members_cap=64 * n)
        assert np.array_equal(density.cpu().numpy(), rho) and np.array_equal(medoid.cpu().numpy(), medoid_ref)
        assert np.array_equal(ptr.cpu().numpy(), ptr_ref) and np.array_equal(members.cpu().numpy(), members_ref)


@pytest.mark.parametrize("shift", [0, 1, 4])
@pytest.mark.parametrize("pages", [5, 16 * 8, 16 * 128 + 3, 2 * 1024 + 1])
def test_cache_bookkeeping_at_row_ends_and_unaligned_arrays(pages, shift):
    """Counters and scores of four clusters at a time where the arrays allow it, one by one otherwise: cluster counts around
    multiples of 4 and of a row of 1024, arrays that start off a 16-byte boundary.  A cluster per page, a third of them selected."""
    cfg = small("c1_tiny", ctx_len=16 * pages, top_k=max(1, pages // 3), n_q_heads=1, n_kv_heads=1, cluster_pages=1, n_queues=6)
    w = W.generate(cfg, seed=pages, device=DEV)
    C = w.n_clusters
    rng = np.random.default_rng(pages + shift)
    w.cluster_size.copy_(torch.from_numpy(rng.integers(1, 12, size=C).astype(np.uint16).view(np.int16)))
    resident0, freq0 = (rng.random(C) < 0.4).astype(np.uint8), rng.integers(-2, 9, size=C).astype(np.int32)
    guard = 77
    resident, freq = torch.full((C + 32,), guard, dtype=torch.uint8, device=DEV), torch.full((C + 32,), guard, dtype=torch.int32, device=DEV)
    score = torch.full((C + 32,), float(guard), device=DEV)
    resident[shift:shift + C], freq[shift:shift + C] = torch.from_numpy(resident0).to(DEV), torch.from_numpy(freq0).to(DEV)
    n_hit = torch.zeros(4, dtype=torch.int32, device=DEV)
    sess = Session(w)
    B.swarm_set_cache(sess.ctx, resident=resident[shift:], freq=freq[shift:], score=score[shift:], n_hit=n_hit, t_base=80.0, t_transfer=2.5)
    tabs = parity.host_tables(w)
    for turn in range(2):
        if turn == 0:
            sess.step()
        else:
            sess.resolve()                                # the separate call takes the same path
        torch.cuda.synchronize()
        assert sess.status() == 0
        uniq, qof, load, hits, freq0, score0 = oracle.resolve_cached(
            sess.o.sel.cpu().numpy(), sess.o.n_sel.cpu().numpy(), tabs["page_base"], tabs["page2cluster"], tabs["cluster_base"],
            tabs["replica_mask"], tabs["cluster_size"], resident0, freq0, cfg.n_queues, 80.0, 2.5)
        n = int(sess.o.n_uniq[0])
        assert n == len(uniq) and int(n_hit[0]) == hits
        assert np.array_equal(sess.o.uniq[:n].cpu().numpy(), uniq) and np.array_equal(sess.o.queue_of[:n].cpu().numpy(), qof)
        assert np.array_equal(freq[shift:shift + C].cpu().numpy(), freq0)
        assert np.allclose(score[shift:shift + C].cpu().numpy(), score0, rtol=1e-6, atol=1e-6)
        for t in (freq, score):                           # nothing beside the arrays is touched
            assert bool((t[:shift] == guard).all()) and bool((t[shift + C:] == guard).all())
    B.swarm_set_cache(sess.ctx)
    sess.close()


@pytest.mark.parametrize("shift", [0, 1, 4])
@pytest.mark.parametrize("pages", [5, 16 * 8, 2 * 1024 + 1])
def test_resolutions_in_a_row_with_cache_state(pages, shift):
    """Separate resolutions and admissions directly behind one another, with nothing between them on the host: every kernel lets the next
    one start early, and each still counts on what the one before it left in the caller's arrays, which end with the last cluster."""
    cfg = small("c1_tiny", ctx_len=16 * pages, top_k=max(1, pages // 3), n_q_heads=2, n_kv_heads=1, cluster_pages=1, n_queues=6)
    w = W.generate(cfg, seed=pages, device=DEV)
    C, T_BASE, T_TR = w.n_clusters, 80.0, 2.5
    rng = np.random.default_rng(pages + shift)
    resident0, freq0 = (rng.random(C) < 0.4).astype(np.uint8), rng.integers(0, 4, size=C).astype(np.int32)
    resident, freq = (torch.zeros(shift + C, dtype=t, device=DEV) for t in (torch.uint8, torch.int32))
    score = torch.zeros(shift + C, device=DEV)
    n_hit = torch.zeros(4, dtype=torch.int32, device=DEV)
    sess = Session(w)
    sess.select()
    other = [torch.roll(sess.o.sel, 1, dims=1)] + [torch.flip((sess.o.sel + 1 + i) % pages, dims=[2]).contiguous() for i in range(2)]
    sels = [sess.o.sel, *(o.contiguous() for o in other)]
    kinds = ["resolve", "resolve", "admit", "resolve", "resolve", "resolve", "admit", "resolve", "admit", "resolve"]
    if shift:                                               # an admission takes arrays on 16-byte boundaries only
        kinds = [k for k in kinds if k == "resolve"]
    capacity = max(1, int(w.cluster_size.sum()) // 3)
    B.swarm_set_cache(sess.ctx, resident=resident[shift:], freq=freq[shift:], score=score[shift:], n_hit=n_hit, t_base=T_BASE, t_transfer=T_TR)
    for _ in range(6):                                      # the races this would show do not occur every time
        resident[shift:], freq[shift:] = torch.from_numpy(resident0).to(DEV), torch.from_numpy(freq0).to(DEV)
        torch.cuda.synchronize()
        for turn, kind in enumerate(kinds):
            if kind == "resolve":
                sess.resolve(sel=sels[turn % len(sels)])
            else:
                B.swarm_cache_admit(score[shift:], w.cluster_size, capacity, resident[shift:])
        torch.cuda.synchronize()
        assert sess.status() == 0
        tabs = parity.host_tables(w)
        want_res, want_freq, want_score = resident0, freq0, None
        for turn, kind in enumerate(kinds):
            if kind == "resolve":
                uniq, qof, load, hits, want_freq, want_score = oracle.resolve_cached(
                    sels[turn % len(sels)].cpu().numpy(), sess.o.n_sel.cpu().numpy(), tabs["page_base"], tabs["page2cluster"], tabs["cluster_base"],
                    tabs["replica_mask"], tabs["cluster_size"], want_res, want_freq, cfg.n_queues, T_BASE, T_TR)
            else:
                want_res, _, _ = oracle.cache_admit(want_score, tabs["cluster_size"], capacity)
        assert np.array_equal(freq[shift:].cpu().numpy(), want_freq) and np.array_equal(resident[shift:].cpu().numpy(), want_res)
        n = int(sess.o.n_uniq[0])
        assert n == len(uniq) and int(n_hit[0]) == hits
        assert np.array_equal(sess.o.uniq[:n].cpu().numpy(), uniq) and np.array_equal(sess.o.queue_of[:n].cpu().numpy(), qof)
        assert np.allclose(score[shift:].cpu().numpy(), want_score, rtol=1e-6, atol=1e-6)
    B.swarm_set_cache(sess.ctx)
    sess.close()


@pytest.mark.parametrize("shift", [0, 4])
@pytest.mark.parametrize("name", ["c1_small", "c3_small", "c5_small"])
def test_second_half_directly_behind_an_admission(name, shift):
    """The resolution of a step in two halves counts on what an admission between the halves has written, although the admission lets
    the second half start before it has written anything; the attention does not notice either."""
    w = W.generate(CASES[name], seed=31, device=DEV)
    C, T_BASE, T_TR = w.n_clusters, 80.0, 2.5
    rng = np.random.default_rng(C)
    wish = [torch.from_numpy(rng.integers(0, 9, size=C).astype(np.float32)).to(DEV) for _ in range(3)]   # scores that decide the admissions
    capacity = int(w.cluster_size.sum()) // 3
    sizes = w.cluster_size.cpu().numpy().view(np.uint16)
    admitted = [oracle.cache_admit(x.cpu().numpy(), sizes, capacity)[0] for x in wish]
    resident, freq = torch.zeros(C, dtype=torch.uint8, device=DEV), torch.zeros(shift + C, dtype=torch.int32, device=DEV)
    score, n_hit = torch.zeros(shift + C, device=DEV), torch.zeros(4, dtype=torch.int32, device=DEV)
    sess = Session(w)
    sess.step()
    torch.cuda.synchronize()
    out, lse = sess.o.out.clone(), sess.o.lse.clone()
    B.swarm_set_cache(sess.ctx, resident=resident, freq=freq[shift:], score=score[shift:], n_hit=n_hit, t_base=T_BASE, t_transfer=T_TR)
    for _ in range(4):
        turns = 5
        freq.zero_()
        torch.cuda.synchronize()
        for turn in range(turns):
            sess.step_begin()
            B.swarm_cache_admit(wish[turn % 3], w.cluster_size, capacity, resident)
            sess.step_end()
        torch.cuda.synchronize()
        assert sess.status() == 0
        tabs = parity.host_tables(w)
        want_freq = np.zeros(C, dtype=np.int32)
        for turn in range(turns):
            uniq, qof, load, hits, want_freq, want_score = oracle.resolve_cached(
                sess.o.sel.cpu().numpy(), sess.o.n_sel.cpu().numpy(), tabs["page_base"], tabs["page2cluster"], tabs["cluster_base"],
                tabs["replica_mask"], tabs["cluster_size"], admitted[turn % 3], want_freq, w.cfg.n_queues, T_BASE, T_TR)
        n = int(sess.o.n_uniq[0])
        assert n == len(uniq) and int(n_hit[0]) == hits
        assert np.array_equal(freq[shift:].cpu().numpy(), want_freq)
        assert np.array_equal(sess.o.uniq[:n].cpu().numpy(), uniq) and np.array_equal(sess.o.queue_of[:n].cpu().numpy(), qof)
        assert np.allclose(score[shift:].cpu().numpy(), want_score, rtol=1e-6, atol=1e-6)
        assert (sess.o.out - out).abs().max().item() <= 1e-4 and (sess.o.lse - lse).abs().max().item() <= 1e-4   # (other ranges: other sums)
    B.swarm_set_cache(sess.ctx)
    sess.close()


def test_counters_that_a_step_does_not_move_can_be_moved_by_others():
    """A step writes the counters of the activated and the resident clusters.  The others, among them neighbours in the same 16 bytes, belong
    to whoever wants them meanwhile: a second stream counts them up beside the steps, and no count is lost on either side."""
    w = W.generate(small("c2_128k", ctx_len=16 * 4096, top_k=64, n_topics=0, cluster_pages=1), seed=37, device=DEV)
    C, steps = w.n_clusters, 60
    sess = Session(w)
    sess.step()
    torch.cuda.synchronize()
    resident = (torch.arange(C, device=DEV) % 5 == 0).to(torch.uint8)
    moved = resident != 0
    moved[sess.o.uniq[: int(sess.o.n_uniq[0])].long()] = True
    others = torch.nonzero(~moved).flatten()
    words = moved[: C // 4 * 4].view(-1, 4).sum(1)
    assert int(((words > 0) & (words < 4)).sum()) > 100      # 16 bytes shared by both sides
    freq, score = torch.zeros(C, dtype=torch.int32, device=DEV), torch.zeros(C, device=DEV)
    B.swarm_set_cache(sess.ctx, resident=resident, freq=freq, score=score, t_base=80.0, t_transfer=2.5)
    want = torch.zeros(C, dtype=torch.int32, device=DEV)
    sess.step()                                             # what one step does to the counters
    torch.cuda.synchronize()
    once = freq.clone()
    freq.zero_()
    ones = torch.ones(len(others), dtype=torch.int32, device=DEV)
    side, main = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    rounds = 0
    for _ in range(steps):
        sess.step(stream=main)
        with torch.cuda.stream(side):
            for _ in range(4):
                freq.index_add_(0, others, ones)
                rounds += 1
    torch.cuda.synchronize()
    assert sess.status() == 0
    want = once * steps
    want[others] += rounds
    assert torch.equal(freq, want)
    B.swarm_set_cache(sess.ctx)
    sess.close()


def test_resolution_directly_behind_an_update_of_its_tables():
    """The separate call finds its tables as the operations in front of it in the stream left them."""
    w = W.generate(CASES["c3_small"], seed=29, device=DEV)
    sess = Session(w)
    sess.step()
    torch.cuda.synchronize()
    big = torch.empty(64 << 20, device=DEV)
    masks, sizes = w.cluster_replica_mask.clone(), w.cluster_size.clone()
    for turn in range(4):
        big.fill_(float(turn))                            # (a while of work in front)
        w.cluster_size.copy_(sizes + turn)
        w.cluster_replica_mask.mul_(0).add_(masks.roll(turn))
        sess.resolve()
        torch.cuda.synchronize()
        assert sess.status() == 0
        o = sess.o
        parity.check_resolve(w, parity.host_tables(w), o.sel.cpu().numpy(), o.n_sel.cpu().numpy(), o.uniq.cpu().numpy(), o.queue_of.cpu().numpy(),
                             o.n_uniq.cpu().numpy()[0], o.queue_load.cpu().numpy())
    sess.close()


@pytest.mark.parametrize("name", ["c1_small", "c3_small", "c5_small"])
def test_resolution_directly_behind_a_selection(name):
    """The kernel in front of the separate call is the selection, which lets the resolution start before it has written anything: queries
    that change every turn, nothing waits on the host, and every turn's schedule is that of its own selection."""
    w = W.generate(CASES[name], seed=29, device=DEV)
    sess = Session(w)
    qs = [w.q, (w.q.float() * -1.0).to(torch.bfloat16), (w.q.float() * 0.5 + 0.125).to(torch.bfloat16)]
    got = []
    for turn in range(9):
        sess.set_query(qs[turn % 3])
        torch.cuda.synchronize()                            # (the two calls enqueued together, the device idle in front of them)
        sess.select()
        sess.resolve()
        o = sess.o
        got.append([x.clone() for x in (o.sel, o.n_sel, o.uniq, o.queue_of, o.n_uniq, o.queue_load)])
    torch.cuda.synchronize()
    assert sess.status() == 0
    assert not torch.equal(got[0][0], got[1][0])
    tabs = parity.host_tables(w)
    for sel, n_sel, uniq, queue_of, n_uniq, load in ([x.cpu().numpy() for x in g] for g in got):
        parity.check_resolve(w, tabs, sel, n_sel, uniq, queue_of, n_uniq[0], load)
    sess.close()


@pytest.mark.parametrize("batch,hq,pages,cluster_pages,k_c,window", [(1, 4, 1023, 1, 70, 0), (2, 2, 1025, 1, 5, 3), (3, 2, 2049, 1, 300, 0), (1, 2, 4097, 1, 3964, 0),
                                                                     (1, 2, 4097, 1, 3965, 0), (2, 66, 4500, 1, 40, 2), (2, 4, 1500, 41, 9, 0)])
def test_medoid_step_at_the_limits_of_its_selection(batch, hq, pages, cluster_pages, k_c, window):
    """The selection expands its clusters itself while the bitmap row and the list fit 16 KiB (3964 clusters of 4097 pages, not 3965) and its
    keys fit registers (not 132 lists of 4500 clusters); every CTA size, and clusters of more members than lanes look at in one turn."""
    cfg = small("c3_batched", batch=batch, ctx_len=16 * pages - 3, n_q_heads=hq, n_kv_heads=2, top_k=8, n_topics=3, cluster_pages=cluster_pages)
    w = W.generate(cfg, seed=pages + k_c, device=DEV)
    sess = Session(w, local_window_pages=window)
    sess.enable_medoid_index(k_c, keep_scores=True)
    for _ in range(2):
        sess.step_medoid()
        check_medoid_step(w, sess, k_c, window=window)
    sess.step()                                             # the page step on the same scratch
    parity.check_step(w, sess)
    sess.close()
