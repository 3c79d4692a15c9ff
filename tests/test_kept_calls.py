"""The argument structs that the one-call entry points keep per shape (CPU: the library is a recorder)."""
import numpy as np
import pytest
import torch

import paper_2510_27641_b200 as sa


class _Recorder:
    """Stands in for the shared library: remembers the scalar fields of every call."""

    def __init__(self):
        self.calls, self.sms = [], 148

    def specattn_select_topp(self, ref, stream):
        a = ref._obj
        self.calls.append((round(a.p, 6), [a.layer_map[j] for j in range(a.n_target_layers)], a.bisect_iters))
        return 0

    def specattn_select_workspace_bytes(self, ref):
        return 0

    def specattn_sparse_verify(self, ref, stream):
        self.calls.append((round(ref._obj.sm_scale, 6), ref._obj.workspace_bytes))
        return 0

    def specattn_verify_workspace_bytes(self, ref):
        return 1000 * self.sms


@pytest.fixture
def recorder(monkeypatch):
    r = _Recorder()
    monkeypatch.setattr(sa, "lib", lambda: r)
    monkeypatch.setattr(sa, "_stream_ptr", lambda stream: 0)
    monkeypatch.setattr(sa, "_calls", sa._Calls())
    monkeypatch.setattr(sa, "_raw_device", lambda: 0)
    return r


def _select(p, layer_map=(0, 1), **kw):
    maps = [torch.zeros(1, 2, 1, 8), torch.zeros(1, 2, 1, 8)]
    return sa.select_topp(maps, torch.zeros(1, dtype=torch.int32), layer_map, p, **kw)


def test_scalars_that_change_in_place_are_taken_by_value(recorder):
    p, m = torch.tensor(0.5), torch.tensor([0, 1])
    _select(p)
    p.fill_(0.75)
    _select(p)
    _select(p, m)
    m[1] = 0
    _select(p, m)
    assert recorder.calls == [(0.5, [0, 1], 0), (0.75, [0, 1], 0), (0.75, [0, 1], 0), (0.75, [0, 0], 0)]


def test_scalars_without_a_hash_are_accepted(recorder):
    _select(np.array(0.25), np.array([1, 0]), bisect_iters=np.array(3))
    _select(0.25, [1, 0], bisect_iters=3)
    assert recorder.calls == [(0.25, [1, 0], 3)] * 2
    assert len(sa._calls.made) == 1


def test_a_workspace_is_sized_for_the_device_of_the_call(recorder, monkeypatch):
    q, kv = torch.zeros(1, 2, 8, 128, dtype=torch.bfloat16), torch.zeros(4, 2, 16, 2, 128, dtype=torch.bfloat16)
    call = lambda: sa.sparse_verify(q, kv, torch.zeros(1, dtype=torch.int32), pages_per_seq=4, dense=True,
                                    sm_scale=0.5)
    call()
    monkeypatch.setattr(sa, "_raw_device", lambda: 1)
    recorder.sms = 160
    call()
    assert recorder.calls == [(0.5, 148000), (0.5, 160000)]
