"""Timing cases of the SpecAttn verification hot path, through the package's public entry points.

Five kinds of work, each a thing a serving program does with this library:

  step    one verification step from a launch plan (``VerifyStep.run``): one selection, then one
          sparse attention call per target layer, everything resident on the GPU
  host    the same step from pinned host buffers (``VerifyStep.run_host``)
  rows    top-p nucleus of single probability rows (``select_topp``, one head, one query)
  select  selection alone over draft attention maps, with the variants of Alg. 2 (one nucleus per
          speculated query, a fixed number of bisection steps, chunk granularity, per-head lists)
  verify  attention of one layer (``sparse_verify``), over lists or dense, with or without the
          in-flight tokens behind the context

Shapes and value laws are those of the package's five benchmark configurations; the inputs are
drawn on the GPU from the seed alone.
"""
from __future__ import annotations

import functools
import math

import torch

import paper_2510_27641_b200 as sa
from paper_2510_27641_b200.step import VerifyStep

HEAD_DIM = 128
FAMILIES = ("uniform", "zipf", "quantised")


# ---- the cases ---------------------------------------------------------------------------------
def _step(name, kind="step", **kw):
    c = {"name": name, "kind": kind, "layers": 1, "draft_layers": 1, "batch": 1, "ctx": 4096, "ctx_min": 0,
         "heads": 12, "gamma": 4, "q_heads": 32, "kv_heads": 8, "page": 16, "paged": True, "p": 0.9, "groups": 1}
    c.update(kw)
    return c


def _rows(name, **kw):
    c = {"name": name, "kind": "rows", "family": "zipf", "rows": 256, "n": 1024, "p": 0.9}
    c.update(kw)
    return c


def _select(name, **kw):
    c = {"name": name, "kind": "select", "draft_layers": 4, "batch": 8, "ctx": 32768, "ctx_min": 0, "heads": 12,
         "gamma": 5, "p": 0.95, "groups": 1, "per_step": False, "bisect": 0, "chunk": 1}
    c.update(kw)
    return c


def _verify(name, **kw):
    c = {"name": name, "kind": "verify", "batch": 4, "ctx": 131072, "ctx_min": 0, "gamma": 4, "q_heads": 64,
         "kv_heads": 8, "page": 16, "dense": False, "kept": 1024, "chunk": 1, "page_lists": False, "tail": 0}
    c.update(kw)
    return c


def listed():
    return [
        # one short conversation, one layer at a time: the latency of the launches
        _step("step_b1_4k", paged=False),
        # the serving workload: an 8B-shaped target (28 of its layers), batch 8, 32k context
        _step("step_b8_32k", layers=28, draft_layers=4, batch=8, ctx=32768, gamma=5, p=0.95),
        # a ragged batch as a continuous-batching server has it
        _step("step_ragged_b32", batch=32, ctx=65536, ctx_min=2048),
        # long context, a 70B-shaped target (16 of its layers)
        _step("step_b4_128k", layers=16, draft_layers=4, batch=4, ctx=131072, heads=16, q_heads=64),
        # one list per KV head, odd lengths, larger pages, a small batch
        _step("step_per_head_b3", layers=4, draft_layers=2, batch=3, ctx=11003, ctx_min=5003, heads=16, gamma=3,
              page=32, groups=8, p=0.95),
        # a step whose draft model lives elsewhere: inputs and results cross PCIe
        _step("host_b2_8k", kind="host", layers=8, draft_layers=2, batch=2, ctx=8192, gamma=5, p=0.95),
        # top-p filtering of probability rows: short peaked, odd-length tied, long flat
        _rows("rows_1k_zipf"),
        _rows("rows_8k_quantised", family="quantised", n=8191, p=0.5),
        _rows("rows_128k_uniform", family="uniform", n=131072),
        # selection as the paper's listing has it: a nucleus per speculated query, united, ten
        # bisection steps, chunks of 16 positions
        _select("select_alg2_chunk16", per_step=True, bisect=10, chunk=16),
        # full attention over a long cache, as the layers that keep every position run it
        _verify("verify_dense_128k", dense=True),
        # chunk lists with the tokens being verified behind them
        _verify("verify_chunk16_tail", batch=16, ctx=16000, q_heads=32, kept=2048, chunk=16, page_lists=True, tail=5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the ranges that the listed ones stand for; never larger than the largest of them."""
    kind = rng.choice(["step", "step", "step", "rows", "rows", "select", "verify", "verify", "host"])
    gamma, p = rng.randint(2, 7), round(rng.uniform(0.8, 0.97), 3)
    q_heads = 64 if rng.random() < 0.35 else 32
    if kind == "rows":
        n = _log_int(rng, 1024, 131072)
        return {k: v for k, v in _rows("", family=rng.choice(FAMILIES), rows=_log_int(rng, 16, 256), n=n,
                                       p=rng.choice([0.5, 0.9, 0.99])).items() if k != "name"}
    batch, ctx, ragged = _log_int(rng, 1, 32), _log_int(rng, 1500, 131072), rng.random() < 0.4
    while batch * ctx > (8 if ragged else 4) * 131072:
        batch = (batch + 1) // 2
    ctx_min = max(1000, ctx // rng.randint(2, 16)) if batch > 1 and ragged else 0
    page = rng.choice([16, 16, 32, 64])
    if kind in ("step", "host"):
        heads, groups = rng.choice([(12, 1), (16, 1), (16, 8)])
        if kind == "host":
            batch, ctx, ctx_min = min(batch, 4), min(ctx, 8192 + ctx % 4096), min(ctx_min, 4096)
        # K/V of all layers stays below 6 M positions (fewer in ragged batches, whose flatter rows
        # keep more of them), the draft maps below 60 M values
        layers = min(_log_int(rng, 1, 28), ((2 if ctx_min else 6) << 20) // (batch * ctx)) or 1
        draft_layers = max(1, min(rng.randint(1, 4), layers, (60 << 20) // (batch * ctx * heads * gamma)))
        c = _step("", kind=kind, layers=layers, draft_layers=draft_layers, batch=batch, ctx=ctx, ctx_min=ctx_min,
                  heads=heads, gamma=gamma, q_heads=q_heads, page=page, paged=rng.random() < 0.8, p=p, groups=groups)
    elif kind == "select":
        c = _select("", draft_layers=max(1, min(rng.randint(1, 4), (60 << 20) // (batch * ctx * 12 * gamma))),
                    batch=batch, ctx=ctx, ctx_min=ctx_min, gamma=gamma, p=p,
                    per_step=rng.random() < 0.5, bisect=rng.choice([0, 10]), chunk=rng.choice([1, 16, 16, 32]))
    else:
        dense, chunk = rng.random() < 0.3, rng.choice([1, 1, 16])
        c = _verify("", batch=batch, ctx=ctx, ctx_min=ctx_min, gamma=gamma, q_heads=q_heads, page=page, dense=dense,
                    kept=0 if dense else max(32, ctx // rng.randint(4, 24)), chunk=1 if dense else chunk,
                    page_lists=not dense and chunk == 16, tail=rng.choice([0, gamma + 1]))
    return {k: v for k, v in c.items() if k != "name"}


# ---- inputs ------------------------------------------------------------------------------------
def _round_up(x, m):
    return (x + m - 1) // m * m


def _lengths(c):
    """Context lengths: all equal, or spread evenly over the logarithm of [ctx_min, ctx]."""
    if not c["ctx_min"] or c["batch"] == 1:
        return [c["ctx"]] * c["batch"]
    lo, hi, n = math.log(c["ctx_min"]), math.log(c["ctx"]), c["batch"]
    return [int(round(math.exp(lo + (hi - lo) * i / (n - 1)))) for i in range(n)]


def _sequences(c):
    """(length, sink, slope) of every sequence; ragged batches differ in sink and recency too."""
    lens = _lengths(c)
    if not c["ctx_min"]:
        return [(n, 8.0, 0.002) for n in lens]
    return [(n, 4.0 + (8.0 * i * 5 % (8 * len(lens))) / len(lens), (16.0 * ((i * 7) % len(lens)) / len(lens)) / n)
            for i, n in enumerate(lens)]


def _attention_rows(gen, n, rows, sink, slope):
    """Softmax over n positions of 3 z + sink on the first four + a recency ramp, float32 [*rows, n]."""
    logit = torch.randn(*rows, n, generator=gen, device=gen.device) * 3.0
    logit += slope * torch.arange(n, dtype=torch.float32, device=gen.device)
    logit[..., :4] += sink
    return torch.softmax(logit, dim=-1)


def _order(c, gen):
    """The sequences of a ragged batch in a seeded order."""
    seqs = _sequences(c)
    return [seqs[i] for i in torch.randperm(len(seqs), generator=gen, device=gen.device).tolist()]


def _fill_draft(maps, seqs, gen):
    for b, (n, sink, slope) in enumerate(seqs):
        maps[b, :, :, :n] = _attention_rows(gen, n, maps.shape[1:3], sink, slope)


def _nucleus_rows(c, gen):
    """Probability rows [rows, n] of one of the three families."""
    shape = (c["rows"], c["n"])
    if c["family"] == "uniform":
        a = torch.rand(shape, generator=gen, device=gen.device)
    elif c["family"] == "zipf":
        base = torch.arange(1, c["n"] + 1, dtype=torch.float64, device=gen.device).pow(-1.2).float()
        a = base[torch.rand(shape, generator=gen, device=gen.device).argsort(dim=1)]
    else:
        a = torch.exp2(-torch.randint(0, 64, shape, generator=gen, device=gen.device) / 4.0)
    return a / a.sum(dim=1, keepdim=True)


def _pool(c, n_pages, gen):
    return torch.randn(n_pages, 2, c["page"], c["kv_heads"], HEAD_DIM, generator=gen, device=gen.device,
                       dtype=torch.bfloat16)


def _layer_map(c, gen):
    """Monotone map target layer -> draft layer that uses every draft layer."""
    rest = torch.randint(0, c["draft_layers"], (c["layers"] - c["draft_layers"],), generator=gen, device=gen.device)
    return sorted(list(range(c["draft_layers"])) + rest.tolist())


def _cache(c, gen, extra=0):
    """Pages per sequence, pages in the pool and the block table (None: contiguous cache)."""
    per_seq = (c["ctx"] + extra + c["page"] - 1) // c["page"]
    n_pages = c["batch"] * per_seq
    table = None
    if c.get("paged", True):
        table = torch.randperm(n_pages, generator=gen, device=gen.device).to(torch.int32).view(c["batch"], per_seq)
    return per_seq, n_pages, table


def _head_group(c):
    return None if c["groups"] == 1 else [h * c["groups"] // c["heads"] for h in range(c["heads"])]


def _prepare_step(c, gen):
    seqs = _order(c, gen)
    kv_len = torch.tensor([s[0] for s in seqs], dtype=torch.int32, device=gen.device)
    per_seq, n_pages, table = _cache(c, gen)
    step = VerifyStep(layer_map=_layer_map(c, gen), n_draft_layers=c["draft_layers"], batch=c["batch"],
                      n_draft_heads=c["heads"], gamma=c["gamma"], L_stride=_round_up(c["ctx"], 4),
                      n_q_heads=c["q_heads"], p=c["p"], kv_pools=[_pool(c, n_pages, gen) for _ in range(c["layers"])],
                      kv_len=kv_len, block_table=table, pages_per_seq=per_seq, n_groups=c["groups"],
                      head_group=_head_group(c),
                      # the caller knows that its batch is ragged, the library's host side does not
                      select_form=sa.SELECT_FORM_TWO_LAUNCH if c["ctx_min"] else sa.SELECT_FORM_AUTO)
    for maps in step.draft_probs:
        _fill_draft(maps, seqs, gen)
    for q in step.q:
        q.normal_(generator=gen)
    state = {"case": c, "step": step}
    if c["kind"] == "host":
        def pinned(t):
            h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
            h.copy_(t)
            return h
        state["draft"] = [pinned(t) for t in step.draft_probs]
        state["q"] = [pinned(t) for t in step.q]
        state["out"] = [pinned(torch.zeros_like(t)) for t in step.out]
        state["lse"] = [pinned(torch.zeros_like(t)) for t in step.lse]
    return state


def _prepare_select(c, gen):
    if c["kind"] == "rows":
        probs = torch.zeros(c["rows"], 1, 1, _round_up(c["n"], 4), device=gen.device)
        probs[:, 0, 0, :c["n"]] = _nucleus_rows(c, gen)
        maps, lens, groups = [probs], [c["n"]] * c["rows"], 1
    else:
        seqs, groups = _order(c, gen), c["groups"]
        lens = [s[0] for s in seqs]
        maps = [torch.zeros(c["batch"], c["heads"], c["gamma"], _round_up(c["ctx"], 4), device=gen.device)
                for _ in range(c["draft_layers"])]
        for m in maps:
            _fill_draft(m, seqs, gen)
    lists = (len(maps), len(lens), groups)
    return {"case": c, "maps": maps, "kv_len": torch.tensor(lens, dtype=torch.int32, device=gen.device),
            # the list buffers that the program keeps: entries beyond a list's count stay as they are
            "idx": torch.full((*lists, maps[0].shape[3]), -1, dtype=torch.int32, device=gen.device),
            "counts": torch.full(lists, -1, dtype=torch.int32, device=gen.device),
            "row_status": torch.full(lists, -1, dtype=torch.int32, device=gen.device)}


def _lists(c, lens, gen):
    """Ascending lists of about `kept` positions, half of them recent, in whole chunks."""
    k = c["chunk"]
    stride = _round_up(max(lens), k)
    idx = torch.zeros(c["batch"], 1, stride, dtype=torch.int32, device=gen.device)
    counts = torch.zeros(c["batch"], 1, dtype=torch.int32, device=gen.device)
    for b, n in enumerate(lens):
        chunks = (n + k - 1) // k
        take = max(1, min(chunks, c["kept"] * n // (c["ctx"] * k)))
        key = torch.rand(chunks, generator=gen, device=gen.device)
        key[chunks - take // 2:] += 1.0
        first = key.topk(take).indices.sort().values * k
        pos = (first[:, None] + torch.arange(k, device=gen.device)).flatten()
        pos = pos[pos < n]
        idx[b, 0, :len(pos)] = pos.to(torch.int32)
        counts[b, 0] = len(pos)
    return idx, counts


def _prepare_verify(c, gen):
    lens = [s[0] for s in _order(c, gen)]
    per_seq, n_pages, table = _cache(c, gen, c["tail"])
    idx, counts = (None, None) if c["dense"] else _lists(c, lens, gen)
    q = torch.randn(c["batch"], c["gamma"] + 1, c["q_heads"], HEAD_DIM, generator=gen, device=gen.device,
                    dtype=torch.bfloat16)
    return {"case": c, "q": q, "kv": _pool(c, n_pages, gen), "table": table, "idx": idx, "counts": counts,
            "kv_len": torch.tensor(lens, dtype=torch.int32, device=gen.device)}


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = case["kind"]
    if kind in ("step", "host"):
        return _prepare_step(case, gen)
    if kind == "verify":
        return _prepare_verify(case, gen)
    return _prepare_select(case, gen)


# ---- one pass ----------------------------------------------------------------------------------
def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "step":
        s = state["step"]
        s.run()
        return {"out": s.out, "lse": s.lse, "status": s.status, "idx": s.idx, "counts": s.counts,
                "row_status": s.row_status, "diag": s.diag}
    if kind == "host":
        s = state["step"]
        s.run_host(state["draft"], state["q"], state["out"], state["lse"])
        return {"out": state["out"], "lse": state["lse"], "status": s.status, "idx": s.idx, "counts": s.counts,
                "row_status": s.row_status, "diag": s.diag}
    if kind == "verify":
        return sa.sparse_verify(state["q"], state["kv"], state["kv_len"], block_table=state["table"],
                                idx=state["idx"], counts=state["counts"], dense=c["dense"], tail_len=c["tail"],
                                flags=sa.VERIFY_PAGE_LISTS if c["page_lists"] else 0)
    options = {}
    if kind == "select":
        options = {"per_step": c["per_step"], "bisect_iters": c["bisect"], "chunk": c["chunk"]}
        if c["ctx_min"]:
            options["form"] = sa.SELECT_FORM_TWO_LAUNCH
    idx, counts, status, _ = sa.select_topp(state["maps"], state["kv_len"], list(range(len(state["maps"]))), c["p"],
                                            idx=state["idx"], counts=state["counts"],
                                            row_status=state["row_status"], **options)
    return idx, counts, status


# ---- what a pass cannot do without -------------------------------------------------------------
def _count(a, p):
    """Size of the top-p nucleus of each row of a [rows, n]."""
    v = a.double().sort(dim=-1, descending=True).values
    s = v.cumsum(dim=-1)
    return ((s < p * s[..., -1:]).sum(dim=-1) + 1).clamp(max=a.shape[-1])


@functools.lru_cache(maxsize=None)
def _kept(items):
    """Positions kept over all lists of one draft layer (or all rows), from one sample of the inputs."""
    c = dict(items)
    gen = torch.Generator(device="cuda" if torch.cuda.is_available() else "cpu")
    gen.manual_seed(0)
    if c["kind"] == "rows":
        sample = dict(c, rows=min(c["rows"], 8))
        return int(_count(_nucleus_rows(sample, gen), c["p"]).double().mean() * c["rows"])
    total, seen = 0, {}
    for seq in _sequences(c):
        if seq not in seen:
            n, sink, slope = seq
            per_group = c["heads"] // c["groups"]
            a = _attention_rows(gen, n, (per_group, c["gamma"]), sink, slope).sum(dim=0)
            if not c.get("per_step"):
                a = a.sum(dim=0, keepdim=True)
            k = c.get("chunk", 1)
            a = torch.nn.functional.pad(a, (0, -n % k)).view(a.shape[0], -1, k).sum(dim=-1)
            mask = torch.zeros(a.shape[1], dtype=torch.bool, device=a.device)
            for row, m in zip(a, _count(a, c["p"]).tolist()):
                mask[row.topk(m).indices] = True
            seen[seq] = min(n, int(mask.sum()) * k) * c["groups"]
        total += seen[seq]
    return total


def work(case):
    c = case
    kind = c["kind"]
    if kind == "rows":
        return {"bytes": 4 * c["rows"] * c["n"] + 4 * _kept(tuple(sorted(c.items()))), "flops": 0}
    total_len, b, f = sum(_lengths(c)), 0, 0
    if kind in ("step", "host", "select"):
        kept = _kept(tuple(sorted(c.items())))
        b += c["draft_layers"] * (4 * c["heads"] * c["gamma"] * total_len + 4 * kept)
        f += c["draft_layers"] * c["heads"] * c["gamma"] * total_len
        if kind == "select":
            return {"bytes": b, "flops": f}
        layers, rows = c["layers"], kept * c["kv_heads"] // c["groups"]
    else:
        layers = 1
        kept = total_len if c["dense"] else sum(max(1, c["kept"] * n // c["ctx"]) for n in _lengths(c))
        rows = (kept + c["tail"] * c["batch"]) * c["kv_heads"]
    n_q = c["gamma"] + 1
    # K and V rows once, the lists once, queries in bf16, outputs and LSE in float32
    lists = 0 if c.get("dense") else 4 * kept
    b += layers * (rows * 4 * HEAD_DIM + lists + c["batch"] * n_q * c["q_heads"] * (6 * HEAD_DIM + 4))
    f += layers * rows * n_q * (c["q_heads"] // c["kv_heads"]) * 4 * HEAD_DIM
    return {"bytes": b, "flops": f}


def tolerance(case):
    """Lists are whole numbers and the same.  Attention runs on exact bf16 products with float32
    sums and weights carried to 2^-16, so outputs agree to 32-bit sums; the masses are binary64."""
    return "exact" if case["kind"] in ("rows", "select") else {"rel": 1e-5, "max": 2e-4}
