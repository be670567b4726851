"""A one-call step that is refused has enqueued nothing: its queries, outputs and pages are as they were, and the call may be
repeated with what it lacked."""
import ctypes

import numpy as np
import pytest

import paper_2505_21889_b200 as efim
from paper_2505_21889_b200 import binding as B
from paper_2505_21889_b200 import build as efim_build

INVALID_ARG, OUT_OF_RANGE, WORKSPACE = 1, 3, 4

BATCHES = [
    ([600, 5, 300], [20, 70, 3]),          # several sequences, not cut
    ([16000, 9000], [16, 16]),             # cut key ranges
    ([240], [16]),                         # one sequence: one kernel
    ([16000], [16]),                       # one sequence, cut
]


@pytest.mark.parametrize("cached,new", BATCHES)
@pytest.mark.parametrize("in_place", [False, True])
def test_a_refused_step_launches_nothing(cached, new, in_place):
    """Without a GPU a launch is answered with EFIM_ERR_CUDA (5): every refusal has to come before the first one.  (The
    addresses are never used.)"""
    efim_build.build()
    lib = efim.load_library()
    cache = B._CacheDesc(0x10000, 0x20000, 4096, 16, 8, 2, 128)
    rope = B._RopeDesc(0x30000, 32768, 0)
    q, k, v, out, ws = 0x1000000, 0x2000000, 0x3000000, 0x1000000 if in_place else 0x4000000, 0x5000000

    def batch(cached, new, pages=1024):
        c, n = np.array(cached, np.int32), np.array(new, np.int32)
        bd = B._BatchDesc(len(c), pages, int(n.sum()), 0x40000, 0x41000, 0x42000, 0x43000, c.ctypes.data, n.ctypes.data)
        bd.keep = c, n
        return bd
    bd, other = batch(cached, new), batch(cached[:-1] + [cached[-1] + 1], new)
    need = lib.efim_prefill_workspace_bytes(ctypes.byref(cache), ctypes.byref(bd))

    def plan_of(b):
        blob = np.zeros(lib.efim_prefill_plan_bytes(ctypes.byref(cache), ctypes.byref(b)), np.uint8)
        assert lib.efim_prefill_plan(ctypes.byref(cache), ctypes.byref(b), blob.ctypes.data, blob.size) == 0
        return blob

    def step(b=bd, plan=None, plan_bytes=None, q=q, out=out, ws=ws, ws_bytes=need):
        return lib.efim_append_prefill_step(ctypes.byref(cache), ctypes.byref(b), ctypes.byref(rope), q, k, v, out, None, 0.0,
                                            plan.ctypes.data if plan is not None else None,
                                            (plan.size if plan_bytes is None else plan_bytes) if plan is not None else 0, 0, ws,
                                            ws_bytes, None, None)
    mine = plan_of(bd)
    for plan in (None, mine):
        assert step(plan=plan, ws=None) == WORKSPACE
        assert step(plan=plan, ws_bytes=need - 1) == WORKSPACE
        assert step(plan=plan, ws=ws + 16) == INVALID_ARG
        assert step(plan=plan, out=out + 8) == INVALID_ARG
        assert step(plan=plan, q=None) == INVALID_ARG
        assert step(batch(cached, new, pages=4), plan=plan) == OUT_OF_RANGE
        blind = batch(cached, new)
        blind.h_cached_len = None
        assert step(blind, plan=plan) == INVALID_ARG
    assert step(plan=plan_of(other)) == INVALID_ARG
    assert step(plan=mine, plan_bytes=mine.size - 1) == INVALID_ARG


@pytest.mark.gpu
@pytest.mark.parametrize("cached,new", BATCHES)
@pytest.mark.parametrize("in_place", [False, True])
def test_a_refused_step_may_be_repeated(cached, new, in_place):
    """Refused for its workspace and for its plan, then repeated with the right ones: the bits of the two calls."""
    import torch
    import tests.gpu_harness as H
    from tests.test_gpu_parity import _custom
    w = _custom(8, 2, 128, cached, new, seed=23)
    a, b = H.DeviceWorkload(w), H.DeviceWorkload(w)
    a.gpu_kv_append()
    a.gpu_prefill()
    other = _custom(8, 2, 128, cached[:-1] + [cached[-1] + 1], new, seed=23)
    stale = efim.efim_prefill_plan(b.cache, efim.Batch(other.cached_len, other.new_len, other.block_table))
    ws = torch.empty(efim.efim_prefill_workspace_bytes(b.cache, b.batch), dtype=torch.uint8, device="cuda")
    out = b.q if in_place else torch.full_like(b.q, float("nan"))
    before = [t.view(torch.int16).clone() for t in (b.q, out, b.k_pool, b.v_pool)]

    def step(workspace, plan=None):
        efim.efim_append_prefill_step(b.cache, b.batch, b.rope, b.q, b.k_new, b.v_new, out, b.lse, 0.0, workspace, b.status,
                                      plan=plan)
    for workspace, plan, code in ((ws[:ws.numel() - 256], None, WORKSPACE), (ws[:ws.numel() - 256], efim.efim_prefill_plan(
            b.cache, b.batch), WORKSPACE), (ws, stale, INVALID_ARG)):
        with pytest.raises(efim.EfimError) as e:
            step(workspace, plan)
        assert e.value.code == code
        torch.cuda.synchronize()
        for t, was in zip((b.q, out, b.k_pool, b.v_pool), before):
            assert torch.equal(t.view(torch.int16), was)
    step(ws)
    torch.cuda.synchronize()
    assert int(a.status.item()) == int(b.status.item()) == 0
    assert torch.equal(a.out.view(torch.int16), out.view(torch.int16)) and torch.equal(a.lse, b.lse)
    assert torch.equal(a.k_pool.view(torch.int16), b.k_pool.view(torch.int16))
    assert torch.equal(a.v_pool.view(torch.int16), b.v_pool.view(torch.int16))
