"""GPU parity of specattn_sparse_verify (through the C ABI) against the CPU oracle's fp64
attention restricted to the listed rows (Eq. 1 over the index set of Eq. 2-3)."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl
from gpu_util import bf16_to_dev, check_attention, dev, to_dev
from workloads import bf16

pytestmark = pytest.mark.gpu

_ENGINE = {"flags": 0}


@pytest.fixture(params=["mma_sync", "tcgen05"], autouse=True)
def engine(request):
    """Every case runs once per implementation of the operation (forced through the flags)."""
    import paper_2510_27641_b200 as sa
    _ENGINE["flags"] = sa.VERIFY_ENGINE_MMA_SYNC if request.param == "mma_sync" else sa.VERIFY_ENGINE_TCGEN05
    yield request.param
    _ENGINE["flags"] = 0


def _make_case(seed, B, T, Hq, Hkv, page, lens, G=1, counts=None, shuffle=True, d=128, tail=0):
    rng = np.random.default_rng(seed)
    lens = np.asarray(lens, np.int32)
    pages_per_seq = max(1, (int(lens.max()) + tail + page - 1) // page)   # room for the in-flight tokens
    n_pages = B * pages_per_seq
    kv = wl.kv_pool(seed, 0, n_pages, page, Hkv, d)                      # torch bf16 on CPU
    bt = wl.block_table(seed, B, pages_per_seq, n_pages, shuffle=shuffle)
    q = wl.queries(seed, 0, B, T, Hq, d)
    stride = max(1, int(lens.max()))
    idx = np.zeros((B, G, stride), np.int32)
    cnt = np.zeros((B, G), np.int32)
    for b in range(B):
        for g in range(G):
            c = int(counts[b][g]) if counts is not None else int(rng.integers(0, lens[b] + 1))
            c = min(c, int(lens[b]))
            sel = np.sort(rng.choice(int(lens[b]), size=c, replace=False)) if c else np.zeros(0, np.int64)
            idx[b, g, :c] = sel
            cnt[b, g] = c
    return dict(q=q, kv=kv, bt=bt, lens=lens, idx=idx, cnt=cnt, page=page, Hkv=Hkv, G=G,
                pages_per_seq=pages_per_seq, tail=tail)


def _run(case, dense=False, use_bt=True, sm_scale=0.0, workspace=None):
    import paper_2510_27641_b200 as sa
    kv_d = case["kv"].to(dev())
    out, lse, status = sa.sparse_verify(
        bf16_to_dev(case["q"]), kv_d, to_dev(case["lens"]),
        block_table=to_dev(case["bt"]) if use_bt else None, pages_per_seq=case["pages_per_seq"],
        idx=None if dense else to_dev(case["idx"]), counts=None if dense else to_dev(case["cnt"]),
        n_groups=case["G"], dense=dense, sm_scale=sm_scale, workspace=workspace, tail_len=case.get("tail", 0),
        flags=_ENGINE["flags"])
    torch.cuda.synchronize()
    return out, lse, status


def _oracle(case, dense=False, use_bt=True, scale=0.0):
    kv_bits = bf16.torch_to_bits(case["kv"])
    page, Hkv = case["page"], case["Hkv"]
    return oracle.sparse_verify(case["q"], kv_bits, wl.kv_strides(page, Hkv, 128),
                                case["bt"] if use_bt else None, case["lens"], case["idx"], case["cnt"],
                                n_kv_heads=Hkv, page_size=page, n_groups=case["G"], dense=dense,
                                scale=scale, pages_per_seq=case["pages_per_seq"], tail_len=case.get("tail", 0))


@pytest.mark.parametrize("T,Hq,Hkv", [(5, 32, 8), (6, 32, 8), (5, 64, 8), (2, 8, 2), (8, 16, 2), (1, 4, 4)])
def test_query_block_shapes(T, Hq, Hkv):
    case = _make_case(10 + T, 3, T, Hq, Hkv, 16, [700, 130, 1], counts=[[300], [130], [1]])
    out, lse, status = _run(case)
    check_attention(out, lse, *_oracle(case))
    assert status.cpu().numpy().tolist() == [0, 0, 0]


def test_list_lengths_around_tile_edges_and_empty_lists():
    lens = [2000] * 14
    counts = [[c] for c in (0, 1, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129)]
    case = _make_case(20, 14, 5, 32, 8, 16, lens, counts=counts)
    out, lse, _ = _run(case)
    check_attention(out, lse, *_oracle(case))
    assert torch.all(out[0] == 0) and torch.all(torch.isneginf(lse[0]))


def test_long_lists_are_split_across_ctas_and_merged():
    # one sequence, 2 kv heads: every unit is cut among ~74 CTAs and merged by the last arriver
    case = _make_case(21, 1, 6, 8, 2, 16, [40000], counts=[[33333]])
    out, lse, _ = _run(case)
    check_attention(out, lse, *_oracle(case))
    # bitwise reproducible regardless of which CTA happens to arrive last
    out2, lse2, _ = _run(case)
    assert torch.equal(out, out2) and torch.equal(lse, lse2)


@pytest.mark.parametrize("T,Hq,counts", [
    (5, 64, [700, 1250, 2100]),      # 40 query rows (two warps per slab): units of 44 - 132 atoms, cut in 2 - 8 parts
    (6, 32, [1100, 1700, 2600]),     # 24 rows (CTA pairs): units above 64 atoms, cut in three or more parts
    (6, 32, [300, 640, 1000]),       # 24 rows: units of up to 64 atoms take the pair's path, cut in two
])
def test_units_cut_in_few_parts_merge_like_the_oracle(T, Hq, counts):
    """Short lists on few sequences: every unit is cut into a handful of parts (odd and even
    numbers of them), merged by the CTA that arrives last -- alone, with the slab's second warp,
    or through the pair's shared memory, depending on the shape.  Results are the oracle's and do
    not depend on who arrives last."""
    case = _make_case(31, 3, T, Hq, 8, 16, [9000, 9000, 9000], counts=[[c] for c in counts])
    out, lse, status = _run(case)
    assert int(status.abs().sum()) == 0
    check_attention(out, lse, *_oracle(case))
    for _ in range(3):
        out2, lse2, _ = _run(case)
        assert torch.equal(out, out2) and torch.equal(lse, lse2)


def test_ragged_batch_with_shared_workspace_reuse():
    import paper_2510_27641_b200 as sa
    rng = np.random.default_rng(3)
    lens = rng.integers(1, 6000, size=12).tolist()
    case = _make_case(22, 12, 5, 32, 8, 16, lens)
    out, lse, _ = _run(case)
    ref = _oracle(case)
    check_attention(out, lse, *ref)
    # the same workspace serves consecutive calls on a stream
    kv_d = case["kv"].to(dev())
    q_d, len_d, bt_d = bf16_to_dev(case["q"]), to_dev(case["lens"]), to_dev(case["bt"])
    idx_d, cnt_d = to_dev(case["idx"]), to_dev(case["cnt"])
    o = torch.empty_like(out)
    l = torch.empty_like(lse)
    args = sa.make_verify_args(q_d, kv_d, len_d, block_table=bt_d, idx=idx_d, counts=cnt_d, out=o, lse=l)
    ws = sa.verify_workspace(args)
    for _ in range(3):
        o.fill_(float("nan"))
        sa.sparse_verify(q_d, kv_d, len_d, block_table=bt_d, idx=idx_d, counts=cnt_d, out=o, lse=l, workspace=ws,
                         flags=_ENGINE["flags"])
        torch.cuda.synchronize()
        assert torch.equal(o, out) and torch.equal(l, lse)


def test_dense_flag_equals_full_list_and_contiguous_cache():
    lens = [1000, 37, 2048]
    case = _make_case(23, 3, 5, 32, 8, 16, lens, counts=[[1000], [37], [2048]], shuffle=False)
    o_d, l_d, _ = _run(case, dense=True)
    check_attention(o_d, l_d, *_oracle(case, dense=True))
    o_f, l_f, _ = _run(case)                      # the p = 1 list
    assert torch.equal(o_d, o_f) and torch.equal(l_d, l_f)
    o_c, l_c, _ = _run(case, use_bt=False)        # identity block table == contiguous addressing
    assert torch.equal(o_c, o_f) and torch.equal(l_c, l_f)
    check_attention(o_c, l_c, *_oracle(case, use_bt=False))


def test_per_kv_head_lists_page_sizes_and_scale():
    for page in (1, 8, 16, 48):
        case = _make_case(24 + page, 2, 5, 16, 4, page, [900, 333], G=4)
        out, lse, _ = _run(case, sm_scale=0.05)
        check_attention(out, lse, *_oracle(case, scale=0.05))


@pytest.mark.parametrize("T,tail", [(5, 5), (6, 6), (5, 2), (4, 7), (6, 1)])
def test_causal_tail_of_in_flight_tokens(T, tail):
    # list lengths chosen so that the tail starts at every offset of a 64-token tile, straddles
    # tiles, follows an empty list, and follows lists cut between CTAs
    lens = [300, 300, 300, 300, 300, 300, 3000, 5000]
    counts = [[0], [1], [31], [60], [63], [64], [2999], [4097]]
    case = _make_case(40 + T, 8, T, 32, 8, 16, lens, counts=counts, tail=tail)
    out, lse, status = _run(case)
    check_attention(out, lse, *_oracle(case))
    assert int(status.abs().sum()) == 0
    # dense context + tail = ordinary causal decode attention of the verified tokens
    case_d = _make_case(50 + T, 2, T, 16, 2, 16, [130, 64], counts=[[130], [64]], tail=tail)
    o_d, l_d, _ = _run(case_d, dense=True)
    check_attention(o_d, l_d, *_oracle(case_d, dense=True))
    o_f, l_f, _ = _run(case_d)
    assert torch.equal(o_d, o_f) and torch.equal(l_d, l_f)


def test_precision_when_few_tokens_dominate():
    # two nearly tied dominant keys with large opposite values: exposes bf16 rounding of P
    case = _make_case(30, 1, 5, 32, 8, 16, [64], counts=[[2]])
    kvb = bf16.torch_to_bits(case["kv"]).copy()
    vals = bf16.to_f32(kvb)
    pages = case["bt"][0]
    for k, pos in enumerate(case["idx"][0, 0, :2]):
        vals[pages[pos // 16], 1, pos % 16] = 4.0 if k == 0 else -4.0
        vals[pages[pos // 16], 0, pos % 16] *= 0.01
    case["kv"] = bf16.bits_to_torch(bf16.from_f32(vals)).reshape(case["kv"].shape)
    out, lse, _ = _run(case)
    check_attention(out, lse, *_oracle(case))


def test_bad_positions_and_pages_are_flagged_not_followed():
    import paper_2510_27641_b200 as sa
    case = _make_case(31, 3, 5, 32, 8, 16, [500, 500, 500], counts=[[100], [100], [100]])
    case["idx"][1, 0, 5] = 500          # == kv_len: out of range
    case["idx"][1, 0, 6] = -3
    case["bt"][2, 0:32] = 10 ** 6       # page id far outside the pool
    out, lse, status = _run(case)
    st = status.cpu().numpy()
    assert st[0] == 0 and st[1] == sa.ROW_BAD_INDEX and st[2] == sa.ROW_BAD_INDEX
    assert torch.all(torch.isfinite(out))
    ref_o, ref_l = _oracle(dict(case, idx=case["idx"][:1], cnt=case["cnt"][:1], lens=case["lens"][:1],
                                bt=case["bt"][:1], q=case["q"][:1]))
    check_attention(out[:1], lse[:1], ref_o, ref_l)


def test_argument_errors():
    import paper_2510_27641_b200 as sa
    case = _make_case(32, 1, 5, 32, 8, 16, [64], counts=[[10]])
    q_d, kv_d = bf16_to_dev(case["q"]), case["kv"].to(dev())
    len_d, bt_d = to_dev(case["lens"]), to_dev(case["bt"])
    idx_d, cnt_d = to_dev(case["idx"]), to_dev(case["cnt"])
    with pytest.raises(sa.SpecAttnError) as e:     # 9 queries x group 8 = 72 rows > 64
        q9 = torch.zeros((1, 9, 64, 128), dtype=torch.bfloat16, device=dev())
        sa.sparse_verify(q9, kv_d, len_d, block_table=bt_d, idx=idx_d, counts=cnt_d)
    assert e.value.code == -6
    tiny = torch.zeros(1024, dtype=torch.uint8, device=dev())
    with pytest.raises(sa.SpecAttnError) as e:
        sa.sparse_verify(q_d, kv_d, len_d, block_table=bt_d, idx=idx_d, counts=cnt_d, workspace=tiny)
    assert e.value.code == -5
    with pytest.raises(sa.SpecAttnError) as e:     # misaligned K/V base
        kv_off = kv_d.view(-1)[4:4 + 3 * 32768].view(3, 2, 16, 8, 128)
        sa.sparse_verify(q_d, kv_off, len_d, block_table=bt_d, idx=idx_d, counts=cnt_d)
    assert e.value.code == -4


def test_back_to_back_launches_with_many_segments_per_cta():
    # 256 units of ~125 atoms: every CTA walks several units, launches overlap through programmatic
    # stream serialization, and short last tiles make consecutive completion signals arrive within
    # nanoseconds of each other -- the case in which a completion barrier must not be missed
    import paper_2510_27641_b200 as sa
    case = _make_case(60, 32, 8, 64, 8, 16, [2100] * 32, counts=[[2000]] * 32)
    kv_d = case["kv"].to(dev())
    q_d, len_d, bt_d = bf16_to_dev(case["q"]), to_dev(case["lens"]), to_dev(case["bt"])
    idx_d, cnt_d = to_dev(case["idx"]), to_dev(case["cnt"])
    out, lse, status = _run(case)
    assert int(status.abs().sum()) == 0
    o, l = torch.empty_like(out), torch.empty_like(lse)
    st = torch.zeros_like(status)
    args = sa.make_verify_args(q_d, kv_d, len_d, block_table=bt_d, idx=idx_d, counts=cnt_d, out=o, lse=l)
    ws = sa.verify_workspace(args)
    for _ in range(100):
        sa.sparse_verify(q_d, kv_d, len_d, block_table=bt_d, idx=idx_d, counts=cnt_d, out=o, lse=l, status=st,
                         workspace=ws, flags=_ENGINE["flags"])
    torch.cuda.synchronize()
    assert int(st.abs().sum()) == 0
    assert torch.equal(o, out) and torch.equal(l, lse)


def test_precomputed_work_partition_gives_the_same_results_and_is_ignored_when_it_does_not_fit():
    import ctypes as C
    import paper_2510_27641_b200 as sa
    if _ENGINE["flags"] != sa.VERIFY_ENGINE_MMA_SYNC:
        pytest.skip("only the mma.sync engine reads plans")
    rng = np.random.default_rng(5)
    lens = rng.integers(1, 5000, size=10).tolist()
    case = _make_case(70, 10, 5, 32, 8, 16, lens)
    kv_d = case["kv"].to(dev())
    q_d, len_d, bt_d = bf16_to_dev(case["q"]), to_dev(case["lens"]), to_dev(case["bt"])
    idx_d, cnt_d = to_dev(case["idx"]), to_dev(case["cnt"])
    ref_o, ref_l, _ = _run(case)

    def run(plan, tail_len=0, cnt=cnt_d):
        o = torch.full_like(ref_o, float("nan"))
        l = torch.full_like(ref_l, float("nan"))
        a = sa.make_verify_args(q_d, kv_d, len_d, block_table=bt_d, idx=idx_d, counts=cnt, out=o, lse=l,
                                flags=_ENGINE["flags"], tail_len=tail_len)
        a.workspace_t = sa.verify_workspace(a)
        a.workspace, a.workspace_bytes = a.workspace_t.data_ptr(), a.workspace_t.numel()
        a.plan = None if plan is None else plan.data_ptr()
        rc = sa.lib().specattn_sparse_verify(C.byref(a), None)
        assert rc == 0
        torch.cuda.synchronize()
        return o, l, a

    o0, l0, a0 = run(None)
    plan = sa.verify_plan_buffer(a0)
    sa.verify_plan(a0, plan)
    torch.cuda.synchronize()
    hdr = plan[:8].cpu().tolist()
    assert hdr[1] == 10 * 8 and hdr[6] == 0 and hdr[7] == 0 and hdr[4] >= 1
    o1, l1, _ = run(plan)
    assert torch.equal(o0, o1) and torch.equal(l0, l1) and torch.equal(o0, ref_o)
    # a plan made for other lists of the same shape is the caller's mistake; one whose header
    # does not fit the launch (here: another tail_len) is ignored and the kernel partitions itself
    case_t = _make_case(70, 10, 5, 32, 8, 16, lens, tail=3)
    ref_t = _oracle(case_t)
    kv_t = case_t["kv"].to(dev())
    o = torch.empty_like(ref_o)
    l = torch.empty_like(ref_l)
    at = sa.make_verify_args(bf16_to_dev(case_t["q"]), kv_t, to_dev(case_t["lens"]), block_table=to_dev(case_t["bt"]),
                             idx=to_dev(case_t["idx"]), counts=to_dev(case_t["cnt"]), out=o, lse=l,
                             flags=_ENGINE["flags"], tail_len=3)
    ws = sa.verify_workspace(at)
    at.workspace, at.workspace_bytes = ws.data_ptr(), ws.numel()
    at.plan = plan.data_ptr()
    assert sa.lib().specattn_sparse_verify(C.byref(at), None) == 0
    torch.cuda.synchronize()
    check_attention(o, l, *ref_t)
    # several plans in one launch: the same bits as one launch each (here 11: two launches of <= 8)
    variants = []
    for k in range(11):
        cnt_k = torch.clamp(cnt_d - 3 * k, min=0)
        _, _, ak = run(None, cnt=cnt_k)
        variants.append((ak, cnt_k))
    singles = []
    for ak, _ in variants:
        pk = sa.verify_plan_buffer(ak)
        sa.verify_plan(ak, pk)
        singles.append(pk)
    many = [sa.verify_plan_buffer(ak) for ak, _ in variants]
    n0 = sa.kernel_launch_count()
    sa.verify_plan_many([ak for ak, _ in variants], many)
    torch.cuda.synchronize()
    assert sa.kernel_launch_count() - n0 == 2
    for pk, pm in zip(singles, many):
        assert torch.equal(pk, pm)
    # argument errors
    small = torch.zeros(4, dtype=torch.int32, device=dev())
    with pytest.raises(sa.SpecAttnError):
        sa.verify_plan_many([a0], [small])
    assert sa.lib().specattn_verify_plan(C.byref(a0), small.data_ptr(), 16, None) == -5
    assert sa.lib().specattn_verify_plan(C.byref(a0), None, 1 << 20, None) == -1


def test_kv_len_beyond_the_block_table_is_flagged_not_followed():
    """A device-side kv_len (dense call) or a listed position that lies beyond what the
    sequence's row of the block table covers must not index the table out of its row: those
    positions are flagged SPECATTN_ROW_BAD_INDEX and read position 0 instead; the other
    sequences are unaffected."""
    import paper_2510_27641_b200 as sa
    case = _make_case(33, 3, 5, 32, 8, 16, [480, 480, 480], counts=[[100], [100], [100]])
    assert case["pages_per_seq"] == 30
    # dense: sequence 1 claims one page more than its block-table row holds
    over = dict(case, lens=np.array([480, 496, 480], np.int32))
    for use_bt in (True, False):
        out, lse, status = _run(over, dense=True, use_bt=use_bt)
        st = status.cpu().numpy()
        assert st[0] == 0 and st[1] == sa.ROW_BAD_INDEX and st[2] == 0
        assert torch.all(torch.isfinite(out))
        ref_o, ref_l = _oracle(case, dense=True, use_bt=use_bt)
        check_attention(out[[0, 2]], lse[[0, 2]], ref_o[[0, 2]], ref_l[[0, 2]])
    # listed: the same claim lets position 485 through the kv_len check, not through the table's
    over["idx"] = case["idx"].copy()
    over["idx"][1, 0, 99] = 485
    out, lse, status = _run(over)
    st = status.cpu().numpy()
    assert st[0] == 0 and st[1] == sa.ROW_BAD_INDEX and st[2] == 0
    ref_o, ref_l = _oracle(case)
    check_attention(out[[0, 2]], lse[[0, 2]], ref_o[[0, 2]], ref_l[[0, 2]])


def test_a_bounded_wait_that_runs_out_is_reported_and_the_next_call_is_correct():
    """Failure path of the device-side waits, without faulting anything: with the test-only flag
    one producer warp of CTA 0 withholds the completion signal of its first tile; the waits on it
    give up at their poll limit, the kernel returns normally with SPECATTN_ROW_TIMEOUT in
    status[0], and -- after the workspace is re-initialised -- the next ordinary call on the same
    buffers is correct."""
    import ctypes as C
    import time
    import paper_2510_27641_b200 as sa
    case = _make_case(34, 2, 5, 32, 8, 16, [3000, 2000], counts=[[2500], [1500]])
    kv_d = case["kv"].to(dev())
    q_d, len_d, bt_d = bf16_to_dev(case["q"]), to_dev(case["lens"]), to_dev(case["bt"])
    idx_d, cnt_d = to_dev(case["idx"]), to_dev(case["cnt"])
    o = torch.zeros((2, 5, 32, 128), dtype=torch.float32, device=dev())
    l = torch.zeros((2, 5, 32), dtype=torch.float32, device=dev())
    st = torch.zeros(2, dtype=torch.int32, device=dev())
    a = sa.make_verify_args(q_d, kv_d, len_d, block_table=bt_d, idx=idx_d, counts=cnt_d, out=o, lse=l, status=st,
                            flags=_ENGINE["flags"] | sa.VERIFY_TEST_LOSE_ARRIVAL)
    ws = sa.verify_workspace(a)
    a.workspace, a.workspace_bytes = ws.data_ptr(), ws.numel()
    torch.cuda.synchronize()
    t0 = time.time()
    assert sa.lib().specattn_sparse_verify(C.byref(a), None) == 0
    torch.cuda.synchronize()           # returns: the kernel gave up instead of spinning for ever
    elapsed = time.time() - t0
    assert int(st[0]) & sa.ROW_TIMEOUT
    assert elapsed < 30.0
    # recovery: fresh counters, same buffers, no test flag
    assert sa.lib().specattn_verify_workspace_init(ws.data_ptr(), ws.numel(), None) == 0
    st.zero_()
    a.flags = _ENGINE["flags"]
    assert sa.lib().specattn_sparse_verify(C.byref(a), None) == 0
    torch.cuda.synchronize()
    assert int(st.abs().sum()) == 0
    check_attention(o, l, *_oracle(case))


def _chunk_lists(case, rng, chunk=16, frac=0.4):
    """Replaces the case's lists by lists of whole aligned chunks (the form specattn_select_topp
    emits with chunk = 16, 32 or 64): a random subset of each sequence's chunks, always including
    the last one (cut at kv_len) for half of the lists."""
    B, G = case["cnt"].shape
    for b in range(B):
        L = int(case["lens"][b])
        n_chunks = (L + chunk - 1) // chunk
        for g in range(G):
            take = rng.random(n_chunks) < frac
            if n_chunks and (b + g) % 2 == 0:
                take[-1] = True
            pos = np.concatenate([np.arange(j * chunk, min(L, (j + 1) * chunk)) for j in np.flatnonzero(take)]
                                 or [np.zeros(0, np.int64)])
            case["idx"][b, g, :len(pos)] = pos
            case["idx"][b, g, len(pos):] = 0
            case["cnt"][b, g] = len(pos)


@pytest.mark.parametrize("page,chunk", [(16, 16), (32, 16), (16, 64), (64, 32)])
def test_page_granular_lists_and_dense_calls(page, chunk):
    """Lists of whole aligned chunks flagged SPECATTN_VERIFY_PAGE_LISTS, and dense calls, read K/V
    page-wise (tiled bulk tensor copies in the tcgen05 engine): page sizes 16 to 64, partial last
    pages and chunks, shuffled block table, per-kv-head lists, lists cut between CTAs.  The slots
    of a last page beyond kv_len are poisoned with NaN: they must not reach the result."""
    import paper_2510_27641_b200 as sa
    rng = np.random.default_rng(page * 100 + chunk)
    lens = [5000, 777, 16, 1, 4096, 3333]
    case = _make_case(80 + page, 6, 5, 32, 8, page, lens, G=1)
    _chunk_lists(case, rng, chunk)
    kv = case["kv"].clone()
    for b, L in enumerate(lens):                       # poison what lies beyond kv_len in the last page
        if L % page:
            pg = int(case["bt"][b, L // page])
            kv[pg, :, L % page:] = float("nan")
    poisoned = dict(case, kv=kv)
    flags0 = _ENGINE["flags"]
    try:
        _ENGINE["flags"] = flags0 | sa.VERIFY_PAGE_LISTS
        out, lse, status = _run(poisoned)
        assert int(status.abs().sum()) == 0
        check_attention(out, lse, *_oracle(case))
        o_d, l_d, status = _run(poisoned, dense=True)
        assert int(status.abs().sum()) == 0
        check_attention(o_d, l_d, *_oracle(case, dense=True))
        # the flag changes how rows are fetched, not the results
        _ENGINE["flags"] = flags0
        out0, lse0, _ = _run(case)
        assert float((out - out0).abs().max()) <= 2e-5
        assert float(torch.nan_to_num(lse - lse0, nan=0.0).abs().max()) <= 2e-5    # (-inf) - (-inf): empty lists
    finally:
        _ENGINE["flags"] = flags0


def test_page_granular_per_head_lists_tails_and_contiguous_cache():
    import paper_2510_27641_b200 as sa
    rng = np.random.default_rng(7)
    flags0 = _ENGINE["flags"]
    try:
        _ENGINE["flags"] = flags0 | sa.VERIFY_PAGE_LISTS
        # per-kv-head lists; in-flight tokens behind the lists (they start in the middle of a page)
        case = _make_case(90, 3, 5, 16, 4, 16, [2000, 1000, 37], G=4, tail=5)
        _chunk_lists(case, rng, 16)
        out, lse, status = _run(case)
        assert int(status.abs().sum()) == 0
        check_attention(out, lse, *_oracle(case))
        # dense + tail: ordinary causal decode attention of the verified tokens, page-wise
        o_d, l_d, _ = _run(case, dense=True)
        check_attention(o_d, l_d, *_oracle(case, dense=True))
        # contiguous cache (no block table), one long sequence cut among all CTAs
        case = _make_case(91, 1, 6, 8, 2, 32, [40000], shuffle=False)
        _chunk_lists(case, rng, 32, frac=0.8)
        out, lse, _ = _run(case, use_bt=False)
        check_attention(out, lse, *_oracle(case, use_bt=False))
        o_d, l_d, _ = _run(case, dense=True, use_bt=False)
        check_attention(o_d, l_d, *_oracle(case, dense=True, use_bt=False))
        # a list that breaks the promise is flagged, and nothing faults
        case = _make_case(92, 2, 5, 32, 8, 16, [3000, 3000])
        _chunk_lists(case, rng, 16)
        case["idx"][1, 0, 16 * 3] += 5
        out, lse, status = _run(case)
        st = status.cpu().numpy()
        assert st[0] == 0 and torch.all(torch.isfinite(out))
        if flags0 == sa.VERIFY_ENGINE_TCGEN05:
            assert st[1] == sa.ROW_BAD_INDEX
    finally:
        _ENGINE["flags"] = flags0


@pytest.mark.parametrize("hkv,counts", [
    (2, [1200, 0, 33, 130, 64]),                       # up to eight parts a unit: 8, 4, 2, 1 and an empty list
    (8, [65, 127, 513]),                               # up to four
    (8, [900, 17, 260, 0, 1024, 700]),                 # pairs, or more parts through global memory
    (8, [300] * 9 + [2048]),                           # one long list among short ones
    (8, [40 + 16 * i for i in range(20)]),             # more units than SMs
])
def test_mixed_list_lengths_cut_into_parts_of_one_cluster(hkv, counts):
    """Units of one call cut into different numbers of parts (a power of two up to the cluster size),
    with and without a precomputed partition: same results, within the oracle's tolerance."""
    import ctypes as C
    import paper_2510_27641_b200 as sa
    case = _make_case(95, len(counts), 5, 4 * hkv, hkv, 16, [max(2 * c, 50) for c in counts], counts=[[c] for c in counts])
    out, lse, status = _run(case)
    assert int(status.abs().sum()) == 0
    check_attention(out, lse, *_oracle(case))
    kv_d = case["kv"].to(dev())
    o, l, st = torch.empty_like(out), torch.empty_like(lse), torch.zeros_like(status)
    keep = [bf16_to_dev(case["q"]), to_dev(case["lens"]), to_dev(case["bt"]), to_dev(case["idx"]), to_dev(case["cnt"])]
    a = sa.make_verify_args(keep[0], kv_d, keep[1], block_table=keep[2], idx=keep[3], counts=keep[4], out=o, lse=l,
                            status=st, flags=_ENGINE["flags"])
    ws, plan = sa.verify_workspace(a), sa.verify_plan_buffer(a)
    a.workspace, a.workspace_bytes, a.plan = ws.data_ptr(), ws.numel(), plan.data_ptr()
    sa.verify_plan(a, plan)
    assert sa.lib().specattn_sparse_verify(C.byref(a), C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    torch.cuda.synchronize()
    assert torch.equal(o, out) and torch.equal(l, lse)


@pytest.mark.parametrize("kept", [40, 2500])
def test_a_call_that_clears_its_own_workspace_and_status(kept):
    """Workspace and status full of ones: with the two flags the call clears what it uses itself; with a
    given status and without its flag, earlier status bits stay."""
    import ctypes as C
    import paper_2510_27641_b200 as sa
    case = _make_case(96, 3, 5, 32, 8, 16, [3000] * 3, counts=[[kept], [kept // 2], [kept]])
    keep = [bf16_to_dev(case["q"]), case["kv"].to(dev()), to_dev(case["lens"]), to_dev(case["bt"]), to_dev(case["idx"]),
            to_dev(case["cnt"])]
    out, lse, status = _run(case)
    for init_status in (True, False):
        o, l = torch.empty_like(out), torch.empty_like(lse)
        st = torch.full_like(status, 1)
        a = sa.make_verify_args(keep[0], keep[1], keep[2], block_table=keep[3], idx=keep[4], counts=keep[5], out=o, lse=l,
                                status=st, flags=_ENGINE["flags"] | sa.VERIFY_INIT_WORKSPACE |
                                (sa.VERIFY_INIT_STATUS if init_status else 0) | sa.VERIFY_LISTS_STABLE)
        ws = torch.full((sa.verify_workspace_bytes(a),), 255, dtype=torch.uint8, device=dev())
        a.workspace, a.workspace_bytes = ws.data_ptr(), ws.numel()
        assert sa.lib().specattn_sparse_verify(C.byref(a), C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
        torch.cuda.synchronize()
        assert torch.equal(o, out) and torch.equal(l, lse)
        assert st.tolist() == ([0, 0, 0] if init_status else [1, 1, 1])


@pytest.mark.parametrize("stride,lens,counts", [
    (6145, 12300, [6145]),          # long by idx_stride: pairs
    (6144, 12300, [6144]),          # the line
    (6000, 8000, [6000, 300]),      # one unit far above the average: parts anywhere
])
def test_long_and_skewed_lists_of_33_and_more_query_rows(stride, lens, counts):
    """Either side of the line between larger clusters and pairs, and a small batch whose longest list a cluster
    cannot cut finely enough; with and without a precomputed partition."""
    import ctypes as C
    import paper_2510_27641_b200 as sa
    case = _make_case(97, len(counts), 5, 32, 4, 16, [lens] * len(counts), counts=[[c] for c in counts])
    case["idx"] = case["idx"][:, :, :stride].copy()
    out, lse, status = _run(case)
    assert int(status.abs().sum()) == 0
    check_attention(out, lse, *_oracle(case))
    o, l, st = torch.empty_like(out), torch.empty_like(lse), torch.zeros_like(status)
    keep = [bf16_to_dev(case["q"]), case["kv"].to(dev()), to_dev(case["lens"]), to_dev(case["bt"]), to_dev(case["idx"]),
            to_dev(case["cnt"])]
    a = sa.make_verify_args(keep[0], keep[1], keep[2], block_table=keep[3], idx=keep[4], counts=keep[5], out=o, lse=l,
                            status=st, flags=_ENGINE["flags"])
    ws, plan = sa.verify_workspace(a), sa.verify_plan_buffer(a)
    a.workspace, a.workspace_bytes, a.plan = ws.data_ptr(), ws.numel(), plan.data_ptr()
    sa.verify_plan(a, plan)
    assert sa.lib().specattn_sparse_verify(C.byref(a), C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    torch.cuda.synchronize()
    assert torch.equal(o, out) and torch.equal(l, lse)


def test_a_plan_for_clusters_of_another_size_is_ignored():
    """A plan names the cluster size of the launch it was made for, which depends on the query rows and on idx_stride
    too.  A plan of calls with 16 query rows serves one with 40 where both are launched alike and is ignored
    elsewhere; and a plan whose header names another size, and which deals no work at all, changes nothing."""
    import ctypes as C
    import paper_2510_27641_b200 as sa
    if _ENGINE["flags"] != sa.VERIFY_ENGINE_MMA_SYNC:
        pytest.skip("only the mma.sync engine reads plans")

    def prepare(T, stride):
        case = _make_case(98, 2, T, 64, 8, 16, [12300] * 2, counts=[[700], [1500]])
        case["idx"] = case["idx"][:, :, :stride].copy()
        keep = [bf16_to_dev(case["q"]), case["kv"].to(dev()), to_dev(case["lens"]), to_dev(case["bt"]), to_dev(case["idx"]),
                to_dev(case["cnt"])]
        out = torch.full((2, T, 64, 128), float("nan"), device=dev())
        lse = torch.full((2, T, 64), float("nan"), device=dev())
        a = sa.make_verify_args(keep[0], keep[1], keep[2], block_table=keep[3], idx=keep[4], counts=keep[5], out=out, lse=lse,
                                flags=_ENGINE["flags"])
        ws = sa.verify_workspace(a)
        a.workspace, a.workspace_bytes = ws.data_ptr(), ws.numel()
        return case, a, out, lse, keep + [ws]

    def call(a, out, lse, plan=None):
        out.fill_(float("nan"))
        lse.fill_(float("nan"))
        a.plan = None if plan is None else plan.data_ptr()
        assert sa.lib().specattn_sparse_verify(C.byref(a), None) == 0
        torch.cuda.synchronize()
        return out.clone(), lse.clone()

    few = prepare(2, 6144)               # 16 query rows
    plan = sa.verify_plan_buffer(few[1])
    sa.verify_plan(few[1], plan)
    for stride in (6144, 6145):         # larger clusters, pairs
        case, a, out, lse, keep = prepare(5, stride)   # 40 query rows
        ref = call(a, out, lse)
        check_attention(*ref, *_oracle(case))
        got = call(a, out, lse, plan)
        assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
        own = sa.verify_plan_buffer(a)
        sa.verify_plan(a, own)
        words = own.cpu()
        size = int(words[3]) >> 8
        assert size in (1, 2, 4, 8)
        other = words.clone()
        other[3] = (1 if size > 1 else 2) << 8             # ranges, in a launch of another cluster size
        other[8 + 2 * (2 * 8 + 1):] = 0                    # no CTA has work
        got = call(a, out, lse, other.to(dev()))
        assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])


@pytest.mark.parametrize("batch,n_q,n_q_heads,tokens,parts,cluster", [
    (1, 5, 64, 13000, 15, 1),    # 40 rows: more parts than a cluster has CTAs, wherever there is room
    (1, 5, 64, 1100, 8, 8),
    (1, 5, 32, 1100, 8, 8),      # 20 rows
    (4, 5, 32, 500, 2, 4),       # four parts of eight atoms each would take most of the GPU
    (4, 5, 32, 1100, 4, 4),
    (4, 5, 64, 500, 4, 4),
    (6, 5, 32, 300, 2, 2),
    (6, 5, 64, 800, 2, 2),
])
def test_how_units_are_cut(batch, n_q, n_q_heads, tokens, parts, cluster):
    """Parts per unit where the two ways of merging them, or two numbers of parts, come close (8 KV heads, equal lists)."""
    import paper_2510_27641_b200 as sa
    if _ENGINE["flags"] != sa.VERIFY_ENGINE_MMA_SYNC or torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the plan of the mma.sync engine on 148 SMs")
    d = dev()
    keep = [torch.zeros(batch, n_q, n_q_heads, 128, dtype=torch.bfloat16, device=d),
            torch.zeros(1, 2, 16, 8, 128, dtype=torch.bfloat16, device=d),
            torch.full((batch,), 65536, dtype=torch.int32, device=d), torch.zeros(batch, 4096, dtype=torch.int32, device=d),
            torch.zeros(batch, 1, 65536, dtype=torch.int32, device=d),
            torch.full((batch, 1), tokens, dtype=torch.int32, device=d), torch.zeros(4, device=d), torch.zeros(4, device=d)]
    a = sa.make_verify_args(keep[0], keep[1], keep[2], block_table=keep[3], idx=keep[4], counts=keep[5], out=keep[6],
                            lse=keep[7], flags=_ENGINE["flags"])
    plan = sa.verify_plan_buffer(a)
    sa.verify_plan(a, plan)
    words = plan[:8].cpu().tolist()
    assert words[3] & 0xff == cluster and words[4] == 8 * batch * parts


@pytest.mark.parametrize("counts,tail", [
    ([0, 1, 15, 16, 17, 33, 64, 65, 127, 128, 129, 300], 3),   # edges of a 16-token tile and of four of them, in-flight tokens
    ([5, 2100, 40, 900, 17, 0, 64, 1300, 3, 700], 0),          # long lists among short ones, cut in up to four parts
    ([4100] + [260] * 9, 0),                                   # one unit far above the average
    ([17 * i for i in range(20)], 2),                          # more units than SMs
    ([60, 3, 0, 17] * 9 + [33], 0),                            # as many units as CTAs where two share an SM
    ([40 + 13 * (i % 7) for i in range(50)], 1),               # more: several units and parts of units a CTA, both query buffers in turn
])
@pytest.mark.parametrize("T,Hq", [(1, 32), (3, 32), (5, 32), (6, 32), (7, 32), (5, 64), (6, 64), (7, 64), (8, 64)])
def test_many_units_by_all_their_query_rows(T, Hq, counts, tail):
    """More units than half of the SMs, 4 to 64 query rows (every number of eight-row blocks a warp or a row group may have):
    the oracle's results, the same bits with a precomputed partition and again on the same workspace, and a call
    with the smaller workspace that other shapes need agrees."""
    import ctypes as C
    import paper_2510_27641_b200 as sa
    if _ENGINE["flags"] != sa.VERIFY_ENGINE_MMA_SYNC:
        pytest.skip("the mma.sync engine's rule")
    case = _make_case(99, len(counts), T, Hq, 8, 16, [max(2 * c, 50) for c in counts], counts=[[c] for c in counts], tail=tail)
    out, lse, status = _run(case)
    assert int(status.abs().sum()) == 0
    ref = _oracle(case)
    check_attention(out, lse, *ref)
    kv_d = case["kv"].to(dev())
    o, l, st = torch.empty_like(out), torch.empty_like(lse), torch.zeros_like(status)
    keep = [bf16_to_dev(case["q"]), to_dev(case["lens"]), to_dev(case["bt"]), to_dev(case["idx"]), to_dev(case["cnt"])]
    a = sa.make_verify_args(keep[0], kv_d, keep[1], block_table=keep[2], idx=keep[3], counts=keep[4], out=o, lse=l,
                            status=st, flags=_ENGINE["flags"], tail_len=tail)
    ws, plan = sa.verify_workspace(a), sa.verify_plan_buffer(a)
    a.workspace, a.workspace_bytes = ws.data_ptr(), ws.numel()
    sa.verify_plan(a, plan)
    for p in (plan.data_ptr(), None, plan.data_ptr()):
        a.plan = p
        o.fill_(float("nan"))
        assert sa.lib().specattn_sparse_verify(C.byref(a), C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
        torch.cuda.synchronize()
        assert torch.equal(o, out) and torch.equal(l, lse)
    few = sa.make_verify_args(keep[0][:1], kv_d, keep[1][:1], block_table=keep[2][:1], idx=keep[3][:1], counts=keep[4][:1], out=o, lse=l)
    a.workspace_bytes = sa.verify_workspace_bytes(few)   # (8 units: one CTA per SM)
    assert a.workspace_bytes <= ws.numel()
    assert sa.lib().specattn_sparse_verify(C.byref(a), C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    torch.cuda.synchronize()
    assert int(st.abs().sum()) == 0
    check_attention(o, l, *ref)


@pytest.mark.parametrize("B,kept", [(64, 60), (40, 400)])   # two CTAs per SM: several units each, one or two
@pytest.mark.parametrize("T,Hq", [(4, 32), (5, 32), (7, 64)])
def test_queries_that_the_launch_right_before_wrote(T, Hq, B, kept):
    """SPECATTN_VERIFY_LISTS_STABLE vouches for lists and K/V rows, not for the queries: they may be the previous launch's
    output, whatever segment of a CTA reads them.  Other queries at every turn, written by a copy kernel or by
    another attention launch (which lets this one begin early); every turn gives the bits of an unflagged call."""
    import ctypes as C
    import paper_2510_27641_b200 as sa
    case = _make_case(100 + T, B, T, Hq, 8, 16, [500] * B, counts=[[kept]] * B)
    d = dev()
    kv, lens, bt, idx, cnt = case["kv"].to(d), to_dev(case["lens"]), to_dev(case["bt"]), to_dev(case["idx"]), to_dev(case["cnt"])
    shape, n = (B, T, Hq, 128), 6
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    keep = []

    def call(q, kv, lens, bt, idx, cnt, out, flags):
        lse = torch.empty(shape[:3], device=d)
        a = sa.make_verify_args(q, kv, lens, block_table=bt, idx=idx, counts=cnt, out=out, lse=lse, flags=_ENGINE["flags"] | flags)
        ws = sa.verify_workspace(a)
        a.workspace, a.workspace_bytes = ws.data_ptr(), ws.numel()
        keep.append((a, ws, lse, q, idx))
        return lambda: sa.lib().specattn_sparse_verify(C.byref(a), stream)

    # The writing launch attends one key a sequence, so that its binary32 output is that V row: finite queries when read
    # as bf16.  Sequences 1 and 2 have long lists, whose first key takes all the weight: they are written late.
    long, few = 3000, 8 * 16
    wkv = wl.kv_pool(7, 0, 8 * B, 16, 8, 128).to(d)
    wbt = torch.arange(8 * B, device=d).view(B, 8).repeat(1, 1 + long // few).to(torch.int32)
    wbt[1:3, 8:] = torch.arange(8 * B, device=d)[torch.arange(wbt.shape[1] - 8, device=d) % (5 * B) + 3 * B].to(torch.int32)
    wq = torch.zeros(shape, dtype=torch.bfloat16, device=d)
    wq[..., 0] = 16
    wkv[:, 0, :, :, 0] = -100
    wkv[:, 0, :n, :, 0] = 100          # (slots that a list holds at most one of)
    wlens = torch.full((B,), few, dtype=torch.int32, device=d)
    wcnt = torch.ones(B, 1, dtype=torch.int32, device=d)
    wout = torch.empty(shape, device=d)
    read = wout.view(torch.bfloat16).view(-1)[:wq.numel()].view(shape)
    rest = torch.arange(16, long, device=d)
    rest = rest[rest % 16 >= n].to(torch.int32)
    wlens[1:3], wcnt[1:3] = long, 1 + len(rest)
    writers, queries = [], []
    for i in range(n):
        widx = torch.zeros(B, 1, long, dtype=torch.int32, device=d)
        widx[:, 0, 0] = i
        widx[1:3, 0, 1:1 + len(rest)] = rest
        writers.append(call(wq, wkv, wlens, wbt, widx, wcnt, wout, 0))
        assert writers[i]() == 0
        torch.cuda.synchronize()
        queries.append(read.clone())
        assert torch.all(torch.isfinite(queries[i])) and (i == 0 or not torch.equal(queries[i], queries[i - 1]))
    case["q"] = bf16.torch_to_bits(queries[0].cpu()).reshape(shape)
    want, got = torch.empty(n, *shape, device=d), torch.empty(n, *shape, device=d)
    for i in range(n):
        assert call(queries[i], kv, lens, bt, idx, cnt, want[i], 0)() == 0
    torch.cuda.synchronize()
    check_attention(want[0], keep[-n][2], *_oracle(case))
    q = torch.empty(shape, dtype=torch.bfloat16, device=d)
    for source in (q, read):
        flagged = [call(source, kv, lens, bt, idx, cnt, got[i], sa.VERIFY_LISTS_STABLE) for i in range(n)]
        torch.cuda.synchronize()
        got.fill_(float("nan"))
        for i in list(range(n)) * 3:
            if source is q:
                q.copy_(queries[i])
            else:
                assert writers[i]() == 0
            assert flagged[i]() == 0
        torch.cuda.synchronize()
        assert torch.equal(got, want)


@pytest.mark.parametrize("tokens", [19000, 38400, 65536])   # up to 148 parts, 255 or more of them, and as many as there are CTAs
@pytest.mark.parametrize("T", [2, 4, 5, 6])
def test_one_long_list_among_empty_ones_is_dealt_alike_with_and_without_a_plan(T, tokens):
    """80 units, one of them with a list: its parts, more than 255 of them where two CTAs share an SM, find one another by
    what a plan says as they do without one.  Bits, and attention over the whole list."""
    import ctypes as C
    import paper_2510_27641_b200 as sa
    if _ENGINE["flags"] != sa.VERIFY_ENGINE_MMA_SYNC:
        pytest.skip("only the mma.sync engine reads plans")
    d, B, pps = dev(), 80, tokens // 16 + 1
    kv = wl.kv_pool(5, 0, pps, 16, 1, 128).to(d)
    q = bf16_to_dev(wl.queries(5, 0, B, T, 4, 128))
    bt = torch.zeros(B, pps, dtype=torch.int32, device=d)
    bt[33] = torch.randperm(pps, generator=torch.Generator().manual_seed(5)).to(torch.int32).to(d)
    lens, cnt = (torch.zeros(B, dtype=torch.int32, device=d) for _ in range(2))
    lens[33] = cnt[33] = tokens
    idx = torch.arange(tokens, dtype=torch.int32, device=d).repeat(B, 1, 1)
    out = [torch.full((B, T, 4, 128), float("nan"), device=d) for _ in range(2)]
    lse = [torch.full((B, T, 4), float("nan"), device=d) for _ in range(2)]
    a = sa.make_verify_args(q, kv, lens, block_table=bt, idx=idx, counts=cnt.view(B, 1), out=out[0], lse=lse[0], flags=_ENGINE["flags"])
    ws, plan = sa.verify_workspace(a), sa.verify_plan_buffer(a)
    a.workspace, a.workspace_bytes = ws.data_ptr(), ws.numel()
    sa.verify_plan(a, plan)
    for i in range(2):
        a.out, a.lse, a.plan = out[i].data_ptr(), lse[i].data_ptr(), plan.data_ptr() if i else None
        assert sa.lib().specattn_sparse_verify(C.byref(a), C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    torch.cuda.synchronize()
    assert torch.equal(out[0], out[1]) and torch.equal(lse[0], lse[1])
    rows = kv[bt[33].long()].transpose(1, 2).reshape(-1, 2, 128)[:tokens].double()      # [token, K / V, dim]
    s = q[33].double().reshape(-1, 128) @ rows[:, 0].T / 128 ** 0.5
    check_attention(out[1][33].reshape(-1, 128), lse[1][33].reshape(-1), (s.softmax(-1) @ rows[:, 1]).cpu().numpy(),
                    s.logsumexp(-1).cpu().numpy())
    others = torch.arange(B, device=d) != 33
    assert torch.all(out[1][others] == 0) and torch.all(torch.isneginf(lse[1][others]))


@pytest.mark.parametrize("counts", [
    [700] * 10,         # units cut in clusters: the CTA that gives up leaves with its peers
    [2000] + [0] * 11,  # parts that merge through global memory
    [20] * 40,          # several units a CTA, the queries of the second on their way when the first is given up
])
@pytest.mark.parametrize("T,Hq", [(4, 32), (5, 32), (5, 64), (7, 64)])
def test_a_bounded_wait_that_runs_out_with_many_units(T, Hq, counts):
    """As above where two CTAs share an SM and where two units' queries are held at a time: flagged, no hang, and the next
    call on a fresh workspace is correct."""
    import ctypes as C
    import paper_2510_27641_b200 as sa
    if _ENGINE["flags"] != sa.VERIFY_ENGINE_MMA_SYNC:
        pytest.skip("the mma.sync engine's kernels")
    case = _make_case(35, len(counts), T, Hq, 8, 16, [max(2 * c, 50) for c in counts], counts=[[c] for c in counts])
    keep = [bf16_to_dev(case["q"]), case["kv"].to(dev()), to_dev(case["lens"]), to_dev(case["bt"]), to_dev(case["idx"]),
            to_dev(case["cnt"])]
    o = torch.zeros((len(counts), T, Hq, 128), dtype=torch.float32, device=dev())
    l, st = torch.zeros((len(counts), T, Hq), device=dev()), torch.zeros(len(counts), dtype=torch.int32, device=dev())
    a = sa.make_verify_args(keep[0], keep[1], keep[2], block_table=keep[3], idx=keep[4], counts=keep[5], out=o, lse=l, status=st)
    ws = sa.verify_workspace(a)
    a.workspace, a.workspace_bytes = ws.data_ptr(), ws.numel()
    for flags, lost in ((sa.VERIFY_TEST_LOSE_ARRIVAL, sa.ROW_TIMEOUT), (0, 0)):
        assert sa.lib().specattn_verify_workspace_init(ws.data_ptr(), ws.numel(), None) == 0
        st.zero_()
        a.flags = _ENGINE["flags"] | flags
        assert sa.lib().specattn_sparse_verify(C.byref(a), None) == 0
        torch.cuda.synchronize()
        assert int(st[0]) & sa.ROW_TIMEOUT == lost
    assert int(st.abs().sum()) == 0
    check_attention(o, l, *_oracle(case))


def test_how_units_are_cut_with_one_cta_per_sm_and_few_query_rows():
    """144 units of unequal lengths, 16 query rows, the workspace of one CTA per SM: ranges, as with 32 rows (the wider
    choice of shares is for two CTAs per SM)."""
    import paper_2510_27641_b200 as sa
    if _ENGINE["flags"] != sa.VERIFY_ENGINE_MMA_SYNC or torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the plan of the mma.sync engine on 148 SMs")
    d, B = dev(), 18
    counts = torch.tensor([[int(300 * 0.1 ** (b / 17))] for b in range(B)], dtype=torch.int32, device=d)
    words = []
    for T in (4, 8):
        q = torch.zeros(B, T, 32, 128, dtype=torch.bfloat16, device=d)
        keep = [torch.zeros(1, 2, 16, 8, 128, dtype=torch.bfloat16, device=d), torch.full((B,), 512, dtype=torch.int32, device=d),
                torch.zeros(B, 32, dtype=torch.int32, device=d), torch.zeros(B, 1, 512, dtype=torch.int32, device=d), torch.zeros(4, device=d)]

        def args(n, ws=None):
            return sa.make_verify_args(q[:n], keep[0], keep[1][:n], block_table=keep[2][:n], idx=keep[3][:n], counts=counts[:n],
                                       out=keep[4], lse=keep[4], flags=_ENGINE["flags"], workspace=ws)

        a = args(B, torch.empty(sa.verify_workspace_bytes(args(1)), dtype=torch.uint8, device=d))
        plan = sa.verify_plan_buffer(a)
        sa.verify_plan(a, plan)
        words.append(plan[:8].cpu().tolist())
    assert words[0] == words[1] and words[0][3] & 0xff == 0


@pytest.mark.parametrize("n_q,counts,ctas,cluster", [
    (5, [2000] + [100] * 9, 104, 4),   # the long list in four parts
    (4, [2000] * 16, 256, 4),
    (5, [2000] * 18, 288, 2),          # more units than clusters of four have pairs of CTAs for
    (6, [3000] * 10, 240, 1),          # three parts a unit, anywhere
    (2, [100] * 20, 160, 2),           # a unit per CTA at most
    (5, [3000] * 38, 296, 0),          # ranges
    (5, [60, 3] * 18 + [0], 296, 1),   # a CTA per unit, the empty ones' idle
    (5, [3000] + [60] * 36, 296, 0),
])
def test_how_units_are_cut_with_two_ctas_per_sm(n_q, counts, ctas, cluster):
    """CTAs with work and the clusters they merge in, 8 KV heads, up to 24 query rows, more units than half of the SMs."""
    import paper_2510_27641_b200 as sa
    if _ENGINE["flags"] != sa.VERIFY_ENGINE_MMA_SYNC or torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the plan of the mma.sync engine on 148 SMs")
    d, B = dev(), len(counts)
    keep = [torch.zeros(B, n_q, 32, 128, dtype=torch.bfloat16, device=d), torch.zeros(1, 2, 16, 8, 128, dtype=torch.bfloat16, device=d),
            torch.full((B,), 4096, dtype=torch.int32, device=d), torch.zeros(B, 256, dtype=torch.int32, device=d),
            torch.zeros(B, 1, 4096, dtype=torch.int32, device=d), torch.tensor([[c] for c in counts], dtype=torch.int32, device=d),
            torch.zeros(4, device=d)]
    a = sa.make_verify_args(keep[0], keep[1], keep[2], block_table=keep[3], idx=keep[4], counts=keep[5], out=keep[6],
                            lse=keep[6], flags=_ENGINE["flags"])
    plan = sa.verify_plan_buffer(a)
    sa.verify_plan(a, plan)
    words = plan[:8].cpu().tolist()
    assert words[3] & 0xff == cluster and words[4] == ctas


@pytest.mark.parametrize("T", [2, 5, 6])
@pytest.mark.parametrize("page,bt", [(16, True), (24, True), (1, True), (16, False)])
def test_many_units_with_a_list_per_kv_head(T, page, bt):
    """8, 20 and 24 query rows of 96 units (two CTAs per SM): lists per KV head, pages that are no power of two, a
    contiguous cache, in-flight tokens, a scale of the caller's."""
    rng = np.random.default_rng(page)
    lens = rng.integers(1, 700, size=12).tolist()
    case = _make_case(110 + page, 12, T, 32, 8, page, lens, G=8, shuffle=bt, tail=2)
    out, lse, status = _run(case, use_bt=bt, sm_scale=0.11)
    assert int(status.abs().sum()) == 0
    check_attention(out, lse, *_oracle(case, use_bt=bt, scale=0.11))


@pytest.mark.parametrize("T", [3, 5])
def test_many_units_with_bad_positions_and_pages(T):
    """Flagged, not followed, where two CTAs share an SM; the other sequences keep their results."""
    import paper_2510_27641_b200 as sa
    case = _make_case(111, 12, T, 32, 8, 16, [500] * 12, counts=[[100 + 7 * b] for b in range(12)])
    case["idx"][3, 0, 5] = 500
    case["idx"][3, 0, 101] = -3
    case["bt"][7, 0:32] = 10 ** 6
    out, lse, status = _run(case)
    bad = [sa.ROW_BAD_INDEX if b in (3, 7) else 0 for b in range(12)]
    assert status.cpu().tolist() == bad and torch.all(torch.isfinite(out))
    good = [b for b in range(12) if not bad[b]]
    part = dict(case, idx=case["idx"][good], cnt=case["cnt"][good], lens=case["lens"][good], bt=case["bt"][good], q=case["q"][good])
    check_attention(out[good], lse[good], *_oracle(part))


@pytest.mark.parametrize("counts", [[900] * 10, [300] * 40])   # units in parts; whole
@pytest.mark.parametrize("T,step", [(3, 0.02), (5, 0.02), (6, 0.3), (5, -0.02)])
def test_scores_that_grow_along_a_list(T, step, counts):
    """The reference maximum of a row is raised (and all that was summed up rescaled) tile after tile, by less than 2^8 a
    tile and by more, in every warp and part; or never, where scores fall."""
    case = _make_case(112, len(counts), T, 32, 8, 16, [c + 50 for c in counts], counts=[[c] for c in counts])
    vals = bf16.to_f32(bf16.torch_to_bits(case["kv"]))
    for b, c in enumerate(counts):
        for i, pos in enumerate(case["idx"][b, 0, :c]):
            vals[case["bt"][b, pos // 16], 0, pos % 16, :, 0] = step * i * 128 ** 0.5 / 16     # (log2 of a weight: 1.44 step a key)
    q = bf16.to_f32(case["q"])
    q[..., 0] = 16
    case["q"] = bf16.from_f32(q)
    case["kv"] = bf16.bits_to_torch(bf16.from_f32(vals)).reshape(case["kv"].shape)
    out, lse, status = _run(case)
    assert int(status.abs().sum()) == 0
    check_attention(out, lse, *_oracle(case))
