"""End-to-end parity of a whole verification step (select -> sparse verify per target layer)
against the CPU oracle, on the benchmark configurations at reduced and at full shapes."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl
from gpu_util import check_attention, compare_lists, dev, to_dev
from workloads import bf16

pytestmark = pytest.mark.gpu


def _build(cfg, n_groups=1, head_group=None, dense_first=0, layer_map=None, **step_kw):
    from paper_2510_27641_b200.step import VerifyStep
    si = wl.make_step_inputs(cfg)
    if layer_map is not None:
        # a chosen map (e.g. one target layer per draft layer): the draft rows of a layer depend
        # only on (seed, draft layer), so they are the full configuration's
        si.layer_map = np.asarray(layer_map, np.int32)
        sink, slope = (8.0, 0.002)
        assert not cfg.ragged
        si.draft_probs = [wl.draft_probs(cfg.seed, u, si.kv_len, cfg.n_draft_heads, cfg.gamma, si.L_stride, sink, slope)
                          if u in set(si.layer_map.tolist()) else None for u in range(cfg.n_draft_layers)]
    if dense_first:
        si.layer_map[:dense_first] = -1
    pools = [wl.kv_pool(cfg.seed, j, si.n_pages, cfg.page_size, cfg.n_kv_heads, cfg.head_dim, device=dev())
             for j in range(cfg.n_target_layers)]
    kv_len = to_dev(si.kv_len)
    bt = None if si.block_table is None else to_dev(si.block_table)
    step = VerifyStep(layer_map=si.layer_map.tolist(), n_draft_layers=cfg.n_draft_layers, batch=cfg.batch,
                      n_draft_heads=cfg.n_draft_heads, gamma=cfg.gamma, L_stride=si.L_stride,
                      n_q_heads=cfg.n_q_heads, p=cfg.p, kv_pools=pools, kv_len=kv_len, block_table=bt,
                      pages_per_seq=si.pages_per_seq, n_groups=n_groups, head_group=head_group, **step_kw)
    step.load_inputs([None if x is None else torch.from_numpy(x) for x in si.draft_probs],
                     [bf16.bits_to_torch(q) for q in si.q])
    return si, pools, step


def _check_step(cfg, si, pools, step, layers, n_groups=1, head_group=None):
    oi, oc, os_, od = oracle.select_topp(si.draft_probs, si.layer_map, si.kv_len, cfg.p,
                                         n_groups=n_groups, head_group=head_group)
    B, G = cfg.batch, n_groups

    def row(i):
        u, b, g = i // (B * G), (i // G) % B, i % G
        return oracle.aggregate(si.draft_probs[u][b], L=int(si.kv_len[b]), head_group=head_group, g=g)[0]

    st = compare_lists(row, cfg.p, step.idx.cpu().numpy(), step.counts.cpu().numpy(),
                       step.row_status.cpu().numpy(), oi, oc, os_, od)
    worst = (0.0, 0.0)
    for j in layers:
        u = int(si.layer_map[j])
        kv_bits = bf16.torch_to_bits(pools[j].cpu())
        # the oracle attends the GPU's own lists, so attention parity does not hinge on a
        # near-boundary row having taken the neighbouring threshold
        idx = step.idx[u].cpu().numpy() if u >= 0 else None
        cnt = step.counts[u].cpu().numpy() if u >= 0 else None
        ro, rl = oracle.sparse_verify(si.q[j], kv_bits, wl.kv_strides(cfg.page_size, cfg.n_kv_heads, cfg.head_dim),
                                      si.block_table, si.kv_len, idx, cnt, n_kv_heads=cfg.n_kv_heads,
                                      page_size=cfg.page_size, n_groups=n_groups, dense=u < 0,
                                      pages_per_seq=si.pages_per_seq)
        e = check_attention(step.out[j], step.lse[j], ro, rl)
        worst = (max(worst[0], e[0]), max(worst[1], e[1]))
    assert int(step.status.abs().sum()) == 0
    return st, worst


def test_config0_full_size():
    cfg = wl.config0()
    si, pools, step = _build(cfg)
    step.run()
    torch.cuda.synchronize()
    st, worst = _check_step(cfg, si, pools, step, [0])
    assert st["n"] == 1


def test_config1_shape_reduced_layers_and_context():
    cfg = wl.config1().scaled(n_target_layers=5, n_draft_layers=3, batch=3, ctx=6000)
    si, pools, step = _build(cfg, dense_first=1)
    step.run()
    torch.cuda.synchronize()
    st, worst = _check_step(cfg, si, pools, step, range(5))
    assert st["n"] == len(set(si.layer_map.tolist()) - {-1}) * 3


def test_overlapped_selection_schedule_matches_the_oracle_and_the_plain_schedule():
    """One selection per draft layer, all but the first on a second stream under the attention of
    earlier layers (a layer waits for its own draft layer's lists only): same lists, same outputs,
    launched directly and replayed from a CUDA graph; the map visits the draft layers out of order
    and comes back to one, and starts with a dense layer."""
    cfg = wl.config1().scaled(n_target_layers=8, n_draft_layers=4, batch=3, ctx=6000)
    lmap = [2, 2, 0, 3, 0, 2, 3, 3]
    si, pools, plain = _build(cfg, dense_first=1, layer_map=lmap)
    plain.run()
    torch.cuda.synchronize()
    si2, pools2, step = _build(cfg, dense_first=1, layer_map=lmap, overlap_select=True)
    assert step.overlap and step.launches_per_step == 3 + len(step.plans) + 8
    step.run()
    torch.cuda.synchronize()
    st, worst = _check_step(cfg, si2, pools2, step, range(8))
    assert st["n"] == 3 * 3

    def same():
        used = sorted(set(si.layer_map.tolist()) - {-1})
        for u in used:
            assert torch.equal(step.counts[u], plain.counts[u]) and torch.equal(step.idx[u], plain.idx[u])
        for j in range(8):
            assert torch.equal(step.out[j], plain.out[j]) and torch.equal(step.lse[j], plain.lse[j])
        assert int(step.status.abs().sum()) == 0
    same()
    # replayed from a graph (the second stream joins the capture and is joined again at the end)
    for o in step.out:
        o.fill_(float("nan"))
    step.counts.fill_(-1)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        step.run()
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    same()


def test_config3_ragged_reduced():
    cfg = wl.config3().scaled(batch=9, ctx=9000, ctx_min=300)
    si, pools, step = _build(cfg)
    step.run()
    torch.cuda.synchronize()
    st, worst = _check_step(cfg, si, pools, step, [0])
    assert st["n"] == 9 and len(set(si.kv_len.tolist())) > 5


def test_config4_shape_reduced_with_per_head_lists():
    cfg = wl.config4(n_target_layers=2).scaled(batch=2, ctx=20000, n_draft_layers=2)
    hg = (np.arange(16) * 8 // 16).astype(np.int32)
    si, pools, step = _build(cfg, n_groups=8, head_group=hg.tolist())
    step.run()
    torch.cuda.synchronize()
    st, worst = _check_step(cfg, si, pools, step, [0, 1], n_groups=8, head_group=hg)
    # p = 1 on the same kernel equals the dense flag
    from paper_2510_27641_b200.step import VerifyStep
    step1 = VerifyStep(layer_map=si.layer_map.tolist(), n_draft_layers=2, batch=2, n_draft_heads=16, gamma=4,
                       L_stride=si.L_stride, n_q_heads=64, p=1.0, kv_pools=pools, kv_len=step.kv_len,
                       block_table=step.block_table)
    step1.load_inputs([None if x is None else torch.from_numpy(x) for x in si.draft_probs],
                      [bf16.bits_to_torch(q) for q in si.q])
    step1.run()
    import paper_2510_27641_b200 as sa
    # (dense calls of this shape -- 40 query rows per KV head over a 20000-position cache -- go to
    # the tcgen05 engine by default; the bitwise comparison pins both sides to one engine)
    stepd = VerifyStep(layer_map=[-1, -1], n_draft_layers=2, batch=2, n_draft_heads=16, gamma=4,
                       L_stride=si.L_stride, n_q_heads=64, p=1.0, kv_pools=pools, kv_len=step.kv_len,
                       block_table=step.block_table, verify_flags=sa.VERIFY_ENGINE_MMA_SYNC)
    stepd.load_inputs([None, None], [bf16.bits_to_torch(q) for q in si.q])
    stepd.run()
    torch.cuda.synchronize()
    for j in range(2):
        assert torch.equal(step1.out[j], stepd.out[j]) and torch.equal(step1.lse[j], stepd.lse[j])
    # the default engine choice for the dense call agrees within the tolerance of the operation
    stepa = VerifyStep(layer_map=[-1, -1], n_draft_layers=2, batch=2, n_draft_heads=16, gamma=4,
                       L_stride=si.L_stride, n_q_heads=64, p=1.0, kv_pools=pools, kv_len=step.kv_len,
                       block_table=step.block_table)
    stepa.load_inputs([None, None], [bf16.bits_to_torch(q) for q in si.q])
    stepa.run()
    torch.cuda.synchronize()
    assert int(stepa.status.abs().sum()) == 0
    for j in range(2):
        assert float((stepa.out[j] - stepd.out[j]).abs().max()) <= 2e-5
        assert float((stepa.lse[j] - stepd.lse[j]).abs().max()) <= 2e-5
    u = int(si.layer_map[0])
    assert step1.counts[u].cpu().numpy().ravel().tolist() == [20000, 20000]


def test_host_buffer_step_matches_device_resident_step():
    cfg = wl.config1().scaled(n_target_layers=4, n_draft_layers=2, batch=2, ctx=3000)
    si, pools, step = _build(cfg)
    step.run()
    torch.cuda.synchronize()
    ref_out = [o.clone() for o in step.out]
    ref_lse = [l.clone() for l in step.lse]
    ref_idx, ref_cnt = step.idx.clone(), step.counts.clone()
    # wipe device-side inputs and results, then run the whole step from pinned host memory
    for t in step.draft_probs:
        if t is not None:
            t.zero_()
    for j in range(4):
        step.q[j].zero_()
        step.out[j].zero_()
    step.counts.fill_(-1)
    dp_host = [None if x is None else torch.from_numpy(x).pin_memory() for x in si.draft_probs]
    q_host = [bf16.bits_to_torch(q).pin_memory() for q in si.q]
    out_host = [torch.zeros(o.shape, dtype=torch.float32).pin_memory() for o in step.out]
    lse_host = [torch.zeros(l.shape, dtype=torch.float32).pin_memory() for l in step.lse]
    step.run_host(dp_host, q_host, out_host, lse_host)
    # work enqueued on the caller's stream afterwards sees the step complete (the call joins its
    # copy lanes back into that stream): a device-side copy of the last layer's output, taken
    # without any synchronisation in between
    seen = step.out[3].clone()
    torch.cuda.synchronize()
    assert torch.equal(step.counts, ref_cnt) and torch.equal(seen, ref_out[3])
    for j in range(4):
        assert torch.equal(out_host[j], ref_out[j].cpu()) and torch.equal(lse_host[j], ref_lse[j].cpu())
    # two steps back to back reuse the lanes and their events
    for t in out_host:
        t.zero_()
    step.run_host(dp_host, q_host, out_host, lse_host)
    step.run_host(dp_host, q_host, out_host, lse_host)
    torch.cuda.synchronize()
    for j in range(4):
        assert torch.equal(out_host[j], ref_out[j].cpu()) and torch.equal(lse_host[j], ref_lse[j].cpu())


def test_host_buffer_steps_with_changing_inputs_match_the_oracle():
    """Two steps from host buffers whose draft rows differ (so the lists, their lengths and the
    work partitions change between the steps): each step must match the oracle on its own
    inputs -- a launch that read the previous step's partition or lists would not."""
    cfg = wl.config1().scaled(n_target_layers=6, n_draft_layers=3, batch=3, ctx=5000)
    si, pools, step = _build(cfg, layer_map=[0, 0, 1, 1, 2, 2])
    sp = wl.kv_strides(cfg.page_size, cfg.n_kv_heads, cfg.head_dim)
    q_host = [bf16.bits_to_torch(q).pin_memory() for q in si.q]
    out_host = [torch.zeros(o.shape, dtype=torch.float32).pin_memory() for o in step.out]
    lse_host = [torch.zeros(l.shape, dtype=torch.float32).pin_memory() for l in step.lse]
    kv_bits = [bf16.torch_to_bits(pl.cpu()) for pl in pools]
    prev_counts = None
    for k, (p_sink, p_slope) in enumerate([(8.0, 0.002), (2.0, 0.0004), (8.0, 0.002)]):
        probs = [wl.draft_probs(cfg.seed + 17 * k, u, si.kv_len, cfg.n_draft_heads, cfg.gamma, si.L_stride,
                                p_sink, p_slope) for u in range(3)]
        dp_host = [torch.from_numpy(x).pin_memory() for x in probs]
        step.run_host(dp_host, q_host, out_host, lse_host)
        torch.cuda.synchronize()
        oi, oc, os_, od = oracle.select_topp(probs, si.layer_map, si.kv_len, cfg.p)
        st = compare_lists(lambda i: oracle.aggregate(probs[i // 3][i % 3], L=int(si.kv_len[i % 3]))[0], cfg.p,
                           step.idx.cpu().numpy(), step.counts.cpu().numpy(), step.row_status.cpu().numpy(),
                           oi, oc, os_, od)
        assert st["n"] == 9
        if prev_counts is not None:
            assert not np.array_equal(prev_counts, oc)     # the partitions really changed
        prev_counts = oc.copy()
        for j in range(6):
            u = int(si.layer_map[j])
            ro, rl = oracle.sparse_verify(si.q[j], kv_bits[j], sp, si.block_table, si.kv_len,
                                          step.idx[u].cpu().numpy(), step.counts[u].cpu().numpy(),
                                          n_kv_heads=cfg.n_kv_heads, page_size=cfg.page_size, n_groups=1, dense=False,
                                          pages_per_seq=si.pages_per_seq)
            check_attention(out_host[j], lse_host[j], ro, rl)
        assert int(step.status.abs().sum()) == 0


@pytest.mark.parametrize("which", ["cfg1", "cfg3", "cfg4_p0.8", "cfg4_p0.9", "cfg4_p0.95"])
def test_full_size_sampled_outputs(which):
    """Full batch / context of configs 1, 3 and 4: every list is compared (config 1: the lists
    of all four draft layers, one target layer mapped to each; config 4: two target layers at
    each p of the configuration); attention is checked on sampled (layer, sequence, kv head)
    units whose K/V rows are regenerated on the CPU from the hashed pool definition."""
    lmap = None
    if which == "cfg1":
        cfg = wl.config1().scaled(n_target_layers=4)
        lmap = [0, 1, 2, 3]
    elif which == "cfg3":
        cfg = wl.config3()
    else:
        cfg = wl.config4(n_target_layers=2, p=float(which.split("_p")[1]))   # 70B-shaped, ctx 131072
    si, pools, step = _build(cfg, layer_map=lmap)
    step.run()
    torch.cuda.synchronize()
    oi, oc, os_, od = oracle.select_topp(si.draft_probs, si.layer_map, si.kv_len, cfg.p)
    B = cfg.batch

    def row(i):
        u, b = i // B, i % B
        return oracle.aggregate(si.draft_probs[u][b], L=int(si.kv_len[b]))[0]

    st = compare_lists(row, cfg.p, step.idx.cpu().numpy(), step.counts.cpu().numpy(),
                       step.row_status.cpu().numpy(), oi, oc, os_, od)
    assert st["n"] == len(set(si.layer_map.tolist())) * B
    rng = np.random.default_rng(0)
    sp, sk, ss, sh = wl.kv_strides(cfg.page_size, cfg.n_kv_heads, cfg.head_dim)
    grp = cfg.n_q_heads // cfg.n_kv_heads
    d = cfg.head_dim
    for _ in range(6):
        j = int(rng.integers(0, cfg.n_target_layers))
        b = int(rng.integers(0, B))
        hk = int(rng.integers(0, cfg.n_kv_heads))
        u = int(si.layer_map[j])
        c = int(step.counts[u, b, 0])
        pos = step.idx[u, b, 0, :c].cpu().numpy().astype(np.int64)
        page = si.block_table[b, pos // cfg.page_size].astype(np.int64)
        base = page * sp + (pos % cfg.page_size) * ss + hk * sh
        flat = torch.from_numpy(base)[:, None] + torch.arange(d)[None, :]
        K = bf16.torch_to_bits(wl.kv_values(cfg.seed, j, flat))
        V = bf16.torch_to_bits(wl.kv_values(cfg.seed, j, flat + sk))
        qrows = si.q[j][b][:, hk * grp:(hk + 1) * grp, :].reshape(-1, d)
        ro, rl = oracle.attend_rows(qrows, K, V)
        go = step.out[j][b, :, hk * grp:(hk + 1) * grp, :].reshape(-1, d)
        gl = step.lse[j][b, :, hk * grp:(hk + 1) * grp].reshape(-1)
        check_attention(go, gl, ro, rl)
    assert int(step.status.abs().sum()) == 0


@pytest.mark.parametrize("engine", ["default", "mma_sync"])
def test_full_size_dense_baseline_of_config4(engine):
    """Config 4's p = 1 baseline at full size: 4 sequences x 131072 positions, 64 q / 8 kv heads,
    gamma = 4 (40 query rows per KV head).  The default engine choice for this shape is the
    tcgen05 kernel; the other run forces mma.sync.  Sampled (sequence, kv head) units are
    recomputed by the oracle over all 131072 positions, with K/V regenerated on the CPU."""
    import paper_2510_27641_b200 as sa
    from paper_2510_27641_b200.step import VerifyStep
    cfg = wl.config4(n_target_layers=1, p=1.0)
    si = wl.make_step_inputs(cfg)
    pools = [wl.kv_pool(cfg.seed, 0, si.n_pages, cfg.page_size, cfg.n_kv_heads, cfg.head_dim, device=dev())]
    flags = 0 if engine == "default" else sa.VERIFY_ENGINE_MMA_SYNC
    step = VerifyStep(layer_map=[-1], n_draft_layers=cfg.n_draft_layers, batch=cfg.batch,
                      n_draft_heads=cfg.n_draft_heads, gamma=cfg.gamma, L_stride=si.L_stride,
                      n_q_heads=cfg.n_q_heads, p=1.0, kv_pools=pools, kv_len=to_dev(si.kv_len),
                      block_table=to_dev(si.block_table), pages_per_seq=si.pages_per_seq, verify_flags=flags)
    step.load_inputs([None] * cfg.n_draft_layers, [bf16.bits_to_torch(si.q[0])])
    step.run()
    torch.cuda.synchronize()
    assert int(step.status.abs().sum()) == 0
    sp, sk, ss, sh = wl.kv_strides(cfg.page_size, cfg.n_kv_heads, cfg.head_dim)
    grp, d, L = cfg.n_q_heads // cfg.n_kv_heads, cfg.head_dim, cfg.ctx
    rng = np.random.default_rng(1)
    for _ in range(2):
        b, hk = int(rng.integers(0, cfg.batch)), int(rng.integers(0, cfg.n_kv_heads))
        pos = np.arange(L, dtype=np.int64)
        page = si.block_table[b, pos // cfg.page_size].astype(np.int64)
        base = page * sp + (pos % cfg.page_size) * ss + hk * sh
        flat = torch.from_numpy(base)[:, None] + torch.arange(d)[None, :]
        K = bf16.torch_to_bits(wl.kv_values(cfg.seed, 0, flat))
        V = bf16.torch_to_bits(wl.kv_values(cfg.seed, 0, flat + sk))
        qrows = si.q[0][b][:, hk * grp:(hk + 1) * grp, :].reshape(-1, d)
        ro, rl = oracle.attend_rows(qrows, K, V)
        go = step.out[0][b, :, hk * grp:(hk + 1) * grp, :].reshape(-1, d)
        gl = step.lse[0][b, :, hk * grp:(hk + 1) * grp].reshape(-1)
        check_attention(go, gl, ro, rl)


def test_graft_entry_smoke_runs():
    """The repository's smoke entry point (one small step checked against the oracle) stays in
    working order as the launch plan of a step changes."""
    import importlib
    import sys
    from pathlib import Path
    root = str(Path(__file__).resolve().parents[1])
    if root not in sys.path:
        sys.path.insert(0, root)
    importlib.import_module("__graft_entry__").smoke()


@pytest.mark.parametrize("pinned,layers", [(False, 3), (True, 3), (True, 70)])
def test_host_buffer_step_from_pageable_memory_and_with_many_layers(pinned, layers):
    """Query and result blocks move by a kernel where the GPU can address them and by copy-engine transfers
    elsewhere (pageable memory); more layers than one launch of that kernel takes."""
    cfg = wl.config1().scaled(n_target_layers=layers, n_draft_layers=2, batch=1, ctx=600, n_q_heads=8, n_kv_heads=2)
    si, pools, step = _build(cfg)
    step.run()
    torch.cuda.synchronize()
    ref_out, ref_lse = [o.cpu() for o in step.out], [l.cpu() for l in step.lse]
    put = (lambda t: t.pin_memory()) if pinned else (lambda t: t)
    dp_host = [None if x is None else put(torch.from_numpy(x)) for x in si.draft_probs]
    q_host = [put(bf16.bits_to_torch(q)) for q in si.q]
    out_host = [put(torch.zeros(o.shape, dtype=torch.float32)) for o in step.out]
    lse_host = [put(torch.zeros(l.shape, dtype=torch.float32)) for l in step.lse]
    for t in step.q + step.out:
        t.zero_()
    step.run_host(dp_host, q_host, out_host, lse_host)
    torch.cuda.synchronize()
    for j in range(layers):
        assert torch.equal(out_host[j], ref_out[j]) and torch.equal(lse_host[j], ref_lse[j])


def _capture_host_step(step, *host):
    """Records a step from host buffers into a graph that is never launched.  Returns the launches of the
    library's kernels, and per kernel node the number of copy nodes that it waits for."""
    from cuda.bindings import runtime as rt
    import paper_2510_27641_b200 as sa

    def ok(r):
        assert r[0] == rt.cudaError_t.cudaSuccess, r[0]
        return r[1] if len(r) == 2 else r[1:]

    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    n0 = sa.kernel_launch_count()
    ok(rt.cudaStreamBeginCapture(stream.cuda_stream, rt.cudaStreamCaptureMode.cudaStreamCaptureModeRelaxed))
    try:
        step.run_host(*host, stream=stream)
    finally:
        graph = rt.cudaStreamEndCapture(stream.cuda_stream)
    graph = ok(graph)
    launches = sa.kernel_launch_count() - n0
    nodes = ok(rt.cudaGraphGetNodes(graph, ok(rt.cudaGraphGetNodes(graph))[1]))[0]
    before = {}
    for node in nodes:
        n = ok(rt.cudaGraphNodeGetDependencies_v2(node))[-1]
        before[int(node)] = [int(d) for d in ok(rt.cudaGraphNodeGetDependencies_v2(node, n))[0][:n]] if n else []
    kind = {int(node): ok(rt.cudaGraphNodeGetType(node)) for node in nodes}

    def copies(node):
        seen, todo = set(), list(before[node])
        while todo:
            d = todo.pop()
            if d not in seen:
                seen.add(d)
                todo += before[d]
        return sum(kind[d] == rt.cudaGraphNodeType.cudaGraphNodeTypeMemcpy for d in seen)

    waits = [copies(n) for n, k in kind.items() if k == rt.cudaGraphNodeType.cudaGraphNodeTypeKernel]
    ok(rt.cudaGraphDestroy(graph) + (None,))
    return launches, waits


def _host_step(layers, ctx=600):
    cfg = wl.config1().scaled(n_target_layers=layers, n_draft_layers=2, batch=1, ctx=ctx, n_q_heads=8, n_kv_heads=2)
    si, pools, step = _build(cfg, layer_map=[j * 2 // layers for j in range(layers)])
    dp_host = [torch.from_numpy(x).pin_memory() for x in si.draft_probs]
    q_host = [bf16.bits_to_torch(q).pin_memory() for q in si.q]
    out_host = [torch.zeros(o.shape, dtype=torch.float32).pin_memory() for o in step.out]
    lse_host = [torch.zeros(l.shape, dtype=torch.float32).pin_memory() for l in step.lse]
    step.run_host(dp_host, q_host, out_host, lse_host)   # makes the lanes and their events
    torch.cuda.synchronize()
    return step, dp_host, q_host, out_host, lse_host


def test_host_blocks_beyond_a_registered_range_are_left_to_the_copy_engine():
    """A host block of which only the first page is registered must not be read by the kernel that moves small
    blocks.  (The step is recorded, not run.)"""
    import mmap
    from cuda.bindings import runtime as rt
    import paper_2510_27641_b200 as sa
    step, dp_host, q_host, out_host, lse_host = _host_step(2)
    size = q_host[1].numel() * 2
    assert size > 4096
    memory = mmap.mmap(-1, 4 * 4096)
    block = torch.frombuffer(memory, dtype=torch.bfloat16, count=q_host[1].numel()).view(q_host[1].shape)
    registered = []
    for pages, by_kernel in ((4, True), (1, False)):
        assert rt.cudaHostRegister(block.data_ptr(), pages * 4096, 0)[0] == rt.cudaError_t.cudaSuccess
        try:
            n, _ = _capture_host_step(step, dp_host, [block, block], out_host, lse_host)
            registered.append(n)
        except sa.SpecAttnError as e:   # the runtime may refuse such a copy, as it may any other
            assert not by_kernel and e.code == -7
        finally:
            assert rt.cudaHostUnregister(block.data_ptr())[0] == rt.cudaError_t.cudaSuccess
    assert len(registered) == 1 or registered[1] == registered[0] - 1   # both query blocks are one launch


def test_query_blocks_for_the_copy_engine_do_not_wait_behind_the_draft_rows():
    """Query blocks that the kernel does not take (here: unaligned) reach the GPU ahead of the draft rows: the
    first selection waits for its own layer's rows, not for every layer's."""
    layers = 4
    step, dp_host, q_host, out_host, lse_host = _host_step(layers)
    ref_out, ref_lse = [o.clone() for o in out_host], [l.clone() for l in lse_host]
    odd = []
    for q in q_host:
        flat = torch.empty(q.numel() + 1, dtype=q.dtype).pin_memory()
        odd.append(flat[1:].view(q.shape))
        odd[-1].copy_(q)
    _, waits = _capture_host_step(step, dp_host, odd, out_host, lse_host)
    assert min(w for w in waits if w > 0) <= layers + 1   # the queries and one draft layer of two
    for t in step.q + step.out + out_host:
        t.zero_()
    step.run_host(dp_host, odd, out_host, lse_host)
    torch.cuda.synchronize()
    for j in range(layers):
        assert torch.equal(out_host[j], ref_out[j]) and torch.equal(lse_host[j], ref_lse[j])
