"""Timed cases of the retrieval path: what a serving program asks of this library, through its public entry points.

The decode side is ``Session.step`` (score, select, resolve, attend) over the five benchmark configurations, from one
request with one query head per KV head at 32K tokens to 64 ragged requests of up to 256K; the same step as a chain of
layers, driven from host buffers, with the medoid selector, with the fast-tier bookkeeping, and as its four separate
calls.  The index side is what runs when pages are written (key summaries, medoid rows) and when co-activation
profiles are clustered (Algorithm 1).

Every case is drawn from the seed on the GPU, with the structure of the repository's synthetic workloads.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2603_17803_b200 import binding as B
from paper_2603_17803_b200 import workloads as W
from paper_2603_17803_b200.session import Session

D = 128                                     # head dimension of the library
POOL_BYTES = 35 << 30                       # pool of the largest listed case (64 ragged requests of up to 256K tokens)


def _decode(name, op="step", *, batch=1, q_heads=32, kv_heads=8, page=16, top_k=256, queues=8, ctx=131072,
            ragged=False, topics=64, mixed=False, replication="two", window=0, layers=1):
    """A decode case.  ``ragged``: context lengths uniform in [ctx / 64, ctx]; ``mixed``: clusters of 4..16 pages with
    Zipf topic popularity instead of clusters of 8; ``window``: pages of the local window."""
    return dict(name=name, op=op, batch=batch, q_heads=q_heads, kv_heads=kv_heads, page=page, top_k=top_k,
                queues=queues, ctx=ctx, ragged=ragged, topics=topics, mixed=mixed, replication=replication,
                window=window, layers=layers)


def listed():
    return [
        # one small request, a query head per KV head, keys without topics: launches and hand-offs count
        _decode("step_32k_one_request", q_heads=8, top_k=64, queues=4, ctx=32768, topics=0),
        # a Llama-3-8B-shaped layer at 128K tokens, the library's headline
        _decode("step_128k_one_request"),
        # batched decode at 32K tokens per request, half of the clusters with two replicas
        _decode("step_batch16_32k", batch=16, top_k=128, ctx=32768, topics=32, replication="half_two"),
        # long context: 4 requests of 512K tokens, pages of 32, eight query heads per KV head
        _decode("step_batch4_512k", batch=4, q_heads=64, page=32, top_k=512, queues=16, ctx=524288, topics=128),
        # skewed serving mix: 64 requests of 4K..256K tokens, clusters of 4..16 pages, hot ones on three queues
        _decode("step_batch64_ragged", batch=64, top_k=128, queues=12, ctx=262144, ragged=True, mixed=True,
                replication="hot_three"),
        # a decoder's layers one after the other, their cluster schedules overlapped (tail stream, index prefetch)
        _decode("layers_128k_overlapped", "layers", layers=4),
        # a host program that holds the query and wants the results: synchronous, pinned host buffers both ways
        _decode("step_128k_from_host", "host"),
        # cluster-granular selection by medoids with a local window, odd context length
        _decode("medoid_step_ragged", "medoid", batch=5, top_k=256, ctx=100003, ragged=True, window=8),
        # the four stages as separate calls (selection shown to an I/O layer, K/V copied out, attention over the copies)
        _decode("four_calls_ragged", "stages", batch=6, q_heads=32, top_k=100, queues=6, ctx=50021, ragged=True),
        # the step with the fast tier in play: resident filter, counters, scores, submission order, then a new admission
        _decode("cached_step_and_admission", "cache", batch=16, top_k=128, queues=12, ctx=131072, ragged=True,
                mixed=True, replication="hot_three"),
        # index of freshly written pages: key summaries and medoid rows of a batch of prompts
        _decode("index_build_ragged", "index", batch=16, top_k=128, ctx=60000, ragged=True),
        # offline clustering of a co-activation profile (Algorithm 1)
        dict(name="algorithm1_8192_entries", op="cluster", entries=8192, topics=64),
    ]


def draw(rng):
    """One more case of the same ranges: any of the operations, sizes spread over their logarithms."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["step", "step", "step", "step", "layers", "host", "medoid", "stages", "cache", "index", "cluster"])
    if op == "cluster":
        n = log_int(256, 8192)
        return dict(op=op, entries=n, topics=max(2, n // rng.choice([32, 64, 128])))
    kv_heads = rng.choice([4, 8, 8])
    page = rng.choice([16, 16, 32])
    ctx = log_int(4096, 524288) if op in ("step", "medoid") else log_int(4096, 131072)
    batch = log_int(1, 64)
    limit = POOL_BYTES // {"layers": 16, "index": 12}.get(op, 4)
    while batch > 1 and batch * ctx * kv_heads * 4 * D > limit:
        batch //= 2
    top_k = log_int(16, 512)
    group = rng.choice([1, 2, 4, 4, 8])
    while op == "stages" and top_k > 16 and batch * kv_heads * group * top_k * page * 4 * D > 1 << 30:
        top_k //= 2
    mixed = rng.random() < 0.4
    c = _decode("", op, batch=batch, q_heads=kv_heads * group, kv_heads=kv_heads, page=page, top_k=top_k,
                queues=rng.choice([4, 6, 8, 12, 16]), ctx=ctx, ragged=batch > 1 and rng.random() < 0.5,
                topics=rng.choice([16, 32, 64, 128]), mixed=mixed,
                replication="hot_three" if mixed else rng.choice(["two", "two", "half_two"]),
                window=rng.choice([0, 0, 4]) if op in ("step", "medoid") else 0, layers=4 if op == "layers" else 1)
    del c["name"]
    return c


def _lengths(c):
    """Context lengths: they belong to the case, as the layout of the clusters does, not to the seed."""
    if not c["ragged"]:
        return np.full(c["batch"], c["ctx"], dtype=np.int64)
    return np.random.default_rng(c["ctx"]).integers(max(1, c["ctx"] // 64), c["ctx"] + 1, size=c["batch"])


def _workload(c, seed):
    """One layer's inputs, structured like the library's benchmark workloads: the keys of a page are a topic's centroid
    plus noise, the pages of a topic form the clusters, a request's heads mostly follow its topic."""
    rng, layout = np.random.default_rng(seed), np.random.default_rng(7)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    batch, kv, S, T, n_queues = c["batch"], c["kv_heads"], c["page"], c["topics"], c["queues"]
    lengths = _lengths(c)
    pages = -(-lengths // S)
    page_base = np.concatenate([[0], np.cumsum(pages)])
    weights = 1.0 / np.arange(1, max(T, 1) + 1) ** (1.2 if c["mixed"] else 0.0)
    weights /= weights.sum()
    topics, p2c, sizes, n_rep, cluster_base = [], [], [], [], [0]
    for P in (int(p) for p in pages):
        if T == 0:                          # keys without topics: clusters of random pages
            topic, order = np.zeros(P, dtype=np.int64), rng.permutation(P)
        elif c["mixed"]:
            topic = rng.choice(T, size=P, p=weights)
            order = np.argsort(topic, kind="stable")
        else:
            topic = np.empty(P, dtype=np.int64)
            topic[rng.permutation(P)] = np.arange(P) * T // P
            order = np.argsort(topic, kind="stable")
        runs = [P] if T == 0 or c["mixed"] else np.bincount(topic, minlength=T)
        cut = []
        for run_pages in (int(r) for r in runs if r):
            if c["mixed"]:
                part = layout.integers(4, 17, size=run_pages // 4 + 1)
                ends = np.minimum(np.cumsum(part), run_pages)
            else:
                ends = np.minimum(np.arange(8, run_pages + 8, 8), run_pages)
            cut.append(np.diff(np.concatenate([[0], np.unique(ends)])))
        cut = np.concatenate(cut)
        C = len(cut)
        of_page = np.empty(P, dtype=np.int32)
        of_page[order] = np.repeat(np.arange(C, dtype=np.int32), cut)
        rep = np.full(C, 2 if c["replication"] == "two" else 1)
        if c["replication"] == "half_two":
            rep[rng.permutation(C)[: C // 2]] = 2
        elif c["replication"] == "hot_three":
            rep[: max(1, C // 10)] = 3      # clusters run from the hottest topic down
        topics.append(topic)
        p2c.append(of_page)
        sizes.append(cut)
        n_rep.append(rep)
        cluster_base.append(cluster_base[-1] + C)
    n_rep = np.concatenate(n_rep)
    C = len(n_rep)
    primary = np.arange(C) % n_queues       # the first copy walks round-robin over the queues, the others lie elsewhere
    other = np.argsort(rng.random((C, n_queues - 1)), axis=1)[:, :2] + 1
    mask = 1 << primary
    for r in (2, 3):
        mask = np.where(n_rep >= r, mask | (1 << (primary + other[:, r - 2]) % n_queues), mask)

    pool = torch.empty((int(page_base[-1]), kv, 2, S, D), dtype=torch.bfloat16, device="cuda").normal_(generator=gen)
    q = torch.randn((batch, c["q_heads"], D), generator=gen, device="cuda")
    if T > 0:
        centroids = torch.randn((batch, T, kv, D), generator=gen, device="cuda")
        for b in range(batch):
            topic = torch.from_numpy(topics[b]).cuda()
            for lo in range(0, int(pages[b]), 8192):
                keys = pool[page_base[b] + lo:page_base[b] + min(lo + 8192, int(pages[b])), :, 0]
                keys.mul_(0.3).add_(centroids[b, topic[lo:lo + 8192], :, None].to(torch.bfloat16))
        head_topic = np.where(rng.random((batch, c["q_heads"])) < 0.75, rng.choice(T, size=(batch, 1), p=weights),
                              rng.choice(T, size=(batch, c["q_heads"]), p=weights))
        kv_of = torch.arange(c["q_heads"], device="cuda") // (c["q_heads"] // kv)
        q = q * 0.3 + centroids[torch.arange(batch, device="cuda")[:, None], torch.from_numpy(head_topic).cuda(), kv_of]
    cfg = W.WorkloadConfig("case", batch=batch, n_layers=c["layers"], n_q_heads=c["q_heads"], n_kv_heads=kv, page_size=S,
                           top_k=c["top_k"], n_queues=n_queues, ctx_len=int(lengths.max()), n_topics=T)

    def dev(x, kind):
        return torch.from_numpy(np.ascontiguousarray(x.astype(kind))).cuda()

    return W.Workload(cfg=cfg, seed=seed, q=q.to(torch.bfloat16), kv_pool=pool, page_base=dev(page_base, np.int64),
                      ctx_len=dev(lengths, np.int32), page2cluster=dev(np.concatenate(p2c), np.int32),
                      cluster_base=dev(np.asarray(cluster_base), np.int64), cluster_replica_mask=dev(mask, np.int32),
                      cluster_size=dev(np.concatenate(sizes), np.int16), topic_of_page=np.concatenate(topics),
                      centroids=None)


def _distances(n, topics, seed):
    """Co-activation distances on the GPU, the distribution of ``workloads.coactivation_distances``: near entries share
    a latent topic, a tenth of them belong to two; symmetric, zero diagonal."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    kw = dict(generator=g, device="cuda")
    first = torch.randint(0, topics, (n,), **kw)
    second = torch.where(torch.rand(n, **kw) < 0.1, torch.randint(0, topics, (n,), **kw), first)
    same = (first[:, None] == first) | (second[:, None] == first) | (first[:, None] == second)
    d = torch.where(same, 0.25, 0.85) + (torch.rand((n, n), **kw) - 0.5) * 0.3
    d = d.clamp_(0.0, 1.0)
    d = torch.minimum(d, d.T).contiguous()
    return d.fill_diagonal_(0.0)


def _session(c, seed, layer=0, **kw):
    s = Session(_workload(c, seed * 16 + layer), local_window_pages=c["window"], **kw)
    s.o.uniq.fill_(-1)                      # entries past n_uniq are not written by a step: a defined value for them
    s.o.queue_of.fill_(255)
    return s


def prepare(case, seed):
    c, op = case, case["op"]
    if op == "cluster":
        n, i32 = c["entries"], dict(dtype=torch.int32, device="cuda")
        return dict(op=op, dist=_distances(n, c["topics"], seed), clusters=torch.zeros(n + 1, **i32),
                    members=torch.zeros(16 * n, **i32), medoids=torch.zeros(n, **i32))
    if op == "layers":
        tail = torch.cuda.Stream()
        sessions = [_session(c, seed, layer=i, tail_stream=tail, index_prefetch=True) for i in range(c["layers"])]
        return dict(op=op, sessions=sessions)
    s = _session(c, seed, keep_scores=op == "stages", keep_gathered=op == "stages")
    st = dict(op=op, s=s)
    if op == "host":
        st["stream"] = torch.cuda.Stream()
        st["q"] = s.w.q.cpu().pin_memory()
        st["out"], st["lse"] = torch.empty(s.o.out.shape).pin_memory(), torch.empty(s.o.lse.shape).pin_memory()
        st["n_uniq"] = torch.zeros(4, dtype=torch.int32).pin_memory()
        st["load"] = torch.zeros(max(4, c["queues"]), dtype=torch.int32).pin_memory()
        torch.cuda.synchronize()            # the session's set-up ran on another stream
    elif op == "medoid":
        s.enable_medoid_index(top_k_clusters=max(1, c["top_k"] // 8))
    elif op == "cache":
        n = s.w.n_clusters
        g = torch.Generator(device="cuda").manual_seed(seed)
        st["resident"] = (torch.rand(n, generator=g, device="cuda") < 0.25).to(torch.uint8)
        st["freq"] = torch.randint(0, 50, (n,), generator=g, device="cuda", dtype=torch.int32)
        st["score"] = torch.zeros(n, device="cuda")
        st["n_hit"] = torch.zeros(4, dtype=torch.int32, device="cuda")
        B.swarm_set_cache(s.ctx, resident=st["resident"], freq=st["freq"], score=st["score"], n_hit=st["n_hit"],
                          t_base=80.0, t_transfer=4.0)
        s.enable_submit_order()
        st["capacity"] = s.w.n_pool_pages // 4
        st["next_resident"] = torch.zeros(n, dtype=torch.uint8, device="cuda")
        st["admitted"] = torch.zeros(4, dtype=torch.int32, device="cuda")
    elif op == "index":
        _, _, st["medoid_page"] = W.cluster_members(s.w)
        st["rows"] = torch.empty((s.w.n_clusters, c["kv_heads"], 2, D), dtype=torch.bfloat16, device="cuda")
        st["len"] = torch.zeros(max(4, c["batch"]), dtype=torch.int32, device="cuda")
    return st


def _step_outputs(s):
    o = s.o
    return dict(sel=o.sel, n_sel=o.n_sel, uniq=o.uniq, queue_of=o.queue_of, n_uniq=o.n_uniq, queue_load=o.queue_load,
                out=o.out, lse=o.lse)


def run(st):
    op = st["op"]
    if op == "cluster":
        density, ptr, members, medoid = B.swarm_build_clusters(st["dist"], 0.4)
        for keep, new in (("clusters", ptr), ("members", members), ("medoids", medoid)):   # the program's own tables
            st[keep][: new.numel()].copy_(new)
        return dict(density=density, clusters=st["clusters"], members=st["members"], medoids=st["medoids"])
    if op == "layers":
        for s in st["sessions"]:
            s.step()
        for s in st["sessions"]:
            s.tail_join()
        return [_step_outputs(s) for s in st["sessions"]]
    s = st["s"]
    if op == "step":
        s.step()
        return _step_outputs(s)
    if op == "host":
        s.step_host(st["q"], st["out"], st["lse"], st["n_uniq"], st["load"], stream=st["stream"])
        return dict(out=st["out"], lse=st["lse"], n_uniq=st["n_uniq"], queue_load=st["load"], sel=s.o.sel,
                    n_sel=s.o.n_sel, uniq=s.o.uniq, queue_of=s.o.queue_of)
    if op == "medoid":
        s.step_medoid()
        return dict(_step_outputs(s), sel=s.sel_clusters, n_sel=s.n_sel_clusters)
    if op == "stages":
        s.select()
        s.resolve()
        s.gather()
        s.sparse_attn()
        return dict(_step_outputs(s), scores=s.o.scores, k_out=s.o.k_out, v_out=s.o.v_out, n_tok=s.o.n_tok)
    if op == "cache":
        s.step()
        B.swarm_cache_admit(st["score"], s.w.cluster_size, st["capacity"], st["next_resident"], st["admitted"])
        return dict(_step_outputs(s), submit_order=s.submit_order, submit_info=s.submit_info, freq=st["freq"],
                    score=st["score"], n_hit=st["n_hit"], next_resident=st["next_resident"], admitted=st["admitted"])
    B.swarm_build_summaries(s.ctx, s.inputs, s.ksum)
    B.swarm_build_medoid_index(s.ctx, s.inputs, st["medoid_page"], st["rows"], st["len"])
    return dict(ksum=s.ksum, rows=st["rows"], len=st["len"])


def work(case):
    """Bytes and operations of one pass.  K/V of a decode step: the heads of a group share the pages they have in
    common; in the synthetic topics a further head adds about a third of its own."""
    c, op = case, case["op"]
    if op == "cluster":
        n = c["entries"]
        return dict(bytes=4.0 * n * n, flops=1.0 * n * n)
    pages = float(np.sum(-(-_lengths(c) // c["page"])))
    kv, g, S = c["kv_heads"], c["q_heads"] // c["kv_heads"], c["page"]
    block = 2 * S * D * 2.0                 # K and V of one (page, KV head)
    clusters = pages / (10 if c["mixed"] else 8)
    if op == "index":
        return dict(bytes=pages * kv * (block / 2 + 512) + clusters * kv * 512 * 2, flops=2.0 * pages * kv * S * D)
    per_head = min(c["top_k"] + c["window"], pages / c["batch"])
    distinct = min(per_head * (1 + (g - 1) / 3), pages / c["batch"])
    rows = clusters if op == "medoid" else pages
    slots = c["batch"] * c["q_heads"] * per_head
    small = c["batch"] * c["q_heads"] * (D * 6 + per_head * 4)
    nbytes = rows * kv * 512 + c["batch"] * kv * distinct * block + small
    if op == "stages":                      # the copies are written and read once each
        nbytes += slots * block * 2 + c["batch"] * c["q_heads"] * (pages / c["batch"]) * 4
    if op == "cache":
        nbytes += clusters * (1 + 2 * 4 + 4 * 2 + 2 + 1)
    flops = 2.0 * rows * c["q_heads"] * 2 * D + 4.0 * slots * S * D
    return dict(bytes=nbytes * c["layers"], flops=flops * c["layers"])


def tolerance(case):
    if case["op"] in ("cluster", "index"):
        return "exact"
    # fp32 sums over bf16 operands; selections, schedules, counters and copied bytes are whole values
    return {"rel": 1e-5, "differ": 0.0}
