"""specattn_sparse_verify_static: the attention entry point for callers that cannot allocate
device memory (a custom call inside another runtime's graph gets only its inputs and outputs;
a serving engine's pool may own the whole GPU).  Its scratch is a fixed array inside the
library, so the test checks that two calls in a row -- the second one meeting whatever the
first left in that array -- both reproduce the regular entry point's results."""
import ctypes as C
import gc

import numpy as np
import pytest
import torch

import workloads as wl
from gpu_util import LSE_TOL, OUT_TOL, bf16_to_dev, dev, lse_err, to_dev

pytestmark = pytest.mark.gpu


def _case(seed, B, T, Hq, Hkv, lens, counts):
    rng = np.random.default_rng(seed)
    page = 16
    pps = (max(lens) + page - 1) // page
    kv = wl.kv_pool(seed, 0, B * pps, page, Hkv, 128, device=dev())
    bt = to_dev(wl.block_table(seed, B, pps))
    q = bf16_to_dev(wl.queries(seed, 0, B, T, Hq, 128))
    idx = np.zeros((B, 1, max(lens)), np.int32)
    for b in range(B):
        idx[b, 0, :counts[b]] = np.sort(rng.choice(lens[b], size=counts[b], replace=False))
    return q, kv, bt, to_dev(np.asarray(lens, np.int32)), to_dev(idx), to_dev(np.asarray(counts, np.int32).reshape(B, 1))


def test_static_scratch_entry_point_matches_the_regular_one_twice_in_a_row():
    import paper_2510_27641_b200 as sa
    cases = [_case(41, 3, 6, 32, 8, [5000, 300, 40], [3100, 300, 0]),      # units split across CTAs
             _case(42, 2, 5, 32, 8, [900, 2000], [17, 1999]),
             # two CTAs per SM: cut units, several units a CTA
             _case(45, 12, 5, 32, 8, [900] * 12, [70 * i for i in range(12)]),
             _case(46, 12, 4, 32, 8, [900] * 12, [70 * i for i in range(12)]),
             _case(47, 40, 6, 32, 8, [300] * 40, [7 * i for i in range(40)])]
    for q, kv, bt, kv_len, idx, cnt in cases:
        ref_out, ref_lse, ref_status = sa.sparse_verify(q, kv, kv_len, block_table=bt, idx=idx, counts=cnt)
        torch.cuda.synchronize()
        for call in range(2):
            out = torch.full_like(ref_out, float("nan"))
            lse = torch.full_like(ref_lse, float("nan"))
            status = torch.zeros_like(ref_status)
            args = sa.make_verify_args(q, kv, kv_len, block_table=bt, idx=idx, counts=cnt, out=out, lse=lse,
                                       status=status)          # no workspace: none is needed
            # nothing is allocated: neither through torch's caching allocator (its allocation
            # counter stands still) nor from the driver (the device's free memory stands still)
            gc.collect()
            torch.cuda.synchronize()
            n_alloc = torch.cuda.memory_stats()["allocation.all.allocated"]
            free_before = torch.cuda.mem_get_info()[0]
            sa.sparse_verify_static(args)
            torch.cuda.synchronize()
            assert torch.cuda.memory_stats()["allocation.all.allocated"] == n_alloc
            assert torch.cuda.mem_get_info()[0] == free_before
            # the same kernel over the same work partition, and a cut unit is merged in a fixed
            # order whoever arrives last: the results agree bit for bit (a fortiori within the
            # tolerance the other tests grant the operation: OUT_TOL, LSE_TOL)
            assert torch.equal(out, ref_out), f"call {call}"
            assert torch.equal(lse, ref_lse), f"call {call}"
            assert float((out - ref_out).abs().max()) <= OUT_TOL
            assert lse_err(lse.cpu().numpy().astype(np.float64), ref_lse.cpu().numpy().astype(np.float64)) <= LSE_TOL
            assert torch.equal(status, ref_status)


def test_static_scratch_entry_point_rejects_shapes_beyond_its_buffer():
    import paper_2510_27641_b200 as sa
    # 8 queries x group of 8 = 64 query rows per KV head: four 16-row slabs need ~10 MB of scratch
    q, kv, bt, kv_len, idx, cnt = _case(43, 1, 8, 64, 8, [64], [10])
    out = torch.empty((1, 8, 64, 128), dtype=torch.float32, device=dev())
    lse = torch.empty((1, 8, 64), dtype=torch.float32, device=dev())
    args = sa.make_verify_args(q, kv, kv_len, block_table=bt, idx=idx, counts=cnt, out=out, lse=lse)
    assert sa.verify_workspace_bytes(args) > (6 << 20)
    n0 = sa.kernel_launch_count()
    with pytest.raises(sa.SpecAttnError) as e:
        sa.sparse_verify_static(args)
    assert e.value.code == -8 and "static" in str(e.value)
    assert sa.kernel_launch_count() == n0
    assert sa.lib().specattn_sparse_verify_static(None, None) == -1
    # argument errors are found before anything is enqueued: a missing output pointer
    q, kv, bt, kv_len, idx, cnt = _case(44, 1, 5, 32, 8, [64], [10])
    out = torch.empty((1, 5, 32, 128), dtype=torch.float32, device=dev())
    lse = torch.empty((1, 5, 32), dtype=torch.float32, device=dev())
    args = sa.make_verify_args(q, kv, kv_len, block_table=bt, idx=idx, counts=cnt, out=out, lse=lse)
    args.out = None
    assert sa.lib().specattn_sparse_verify_static(C.byref(args), None) == -1
    assert sa.kernel_launch_count() == n0


@pytest.mark.parametrize("T,rows_of", [(5, "all"), (6, "all"), (4, "all"), (5, "few"), (4, "few")])
def test_a_plan_serves_the_workspace_that_it_was_made_for(T, rows_of):
    """12 sequences (two CTAs per SM with the full workspace, one with the former smaller one), planned: the call with the
    library's own scratch and the one with a workspace of either size read their plan -- one that deals no work leaves
    the outputs alone -- and give the bits that they give without one."""
    import paper_2510_27641_b200 as sa
    q, kv, bt, kv_len, idx, cnt = _case(48, 12, T, 32, 8, [900] * 12, [75 * i + 1 for i in range(12)])
    out, lse = torch.empty((12, T, 32, 128), device=dev()), torch.empty((12, T, 32), device=dev())
    flags = sa.VERIFY_ENGINE_MMA_SYNC
    a = sa.make_verify_args(q, kv, kv_len, block_table=bt, idx=idx, counts=cnt, out=out, lse=lse, flags=flags)
    # (a buffer sized for another number of query rows serves this one too)
    wide = sa.make_verify_args(q.repeat(1, 1, 2, 1)[:, :4].contiguous(), kv, kv_len, block_table=bt, idx=idx, counts=cnt, out=out, lse=lse)
    plan = sa.verify_plan_buffer(wide)
    assert plan.numel() == sa.verify_plan_buffer(a).numel()
    ws = sa.verify_workspace(a)
    if rows_of == "few":
        one = sa.make_verify_args(q[:1], kv, kv_len[:1], block_table=bt[:1], idx=idx[:1], counts=cnt[:1], out=out, lse=lse)
        ws = ws[:sa.verify_workspace_bytes(one)]
        assert ws.numel() < sa.verify_workspace_bytes(a)

    def call():
        out.fill_(float("nan"))
        lse.fill_(float("nan"))
        if static:
            sa.sparse_verify_static(a)
        else:
            assert sa.lib().specattn_sparse_verify(C.byref(a), None) == 0
        torch.cuda.synchronize()
        return out.clone(), lse.clone()

    for static in ((False, True) if rows_of == "all" else (False,)):
        a.workspace, a.workspace_bytes = (None, 0) if static else (ws.data_ptr(), ws.numel())
        a.plan = None
        ref = call()
        sa.verify_plan(a, plan)
        a.plan = plan.data_ptr()
        got = call()
        assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
        assert not torch.any(torch.isnan(ref[0]))
        idle = plan.clone()
        idle[4] = 0                 # no CTA has work
        a.plan = idle.data_ptr()
        assert torch.all(torch.isnan(call()[0]))
