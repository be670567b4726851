"""Kernels whose warps look a token's sequence up 32 candidates at a time: batches of more than one and of more than two such
trips, with sequences that bring nothing among them; every number of warps per token of the append; and one-call steps, whose
append rotates the queries too."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
BAD_PAGE, BAD_POSITION = 1, 2            # EFIM_DEV_*


def _new_lengths(batch, tokens, seed):
    """`tokens` spread over `batch` sequences, a third of which bring none; the first and the last one among those."""
    rng = np.random.default_rng([batch, tokens, seed])
    takes = np.flatnonzero(rng.random(batch) > 0.33)
    takes = takes[(takes > 0) & (takes < batch - 1)] if batch > 4 else np.arange(batch)
    return np.bincount(rng.choice(takes, tokens), minlength=batch).astype(np.int32)


@pytest.mark.parametrize("Hq,Hkv,D,batch,tokens,interleaved", [
    (40, 40, 128, 33, 70, False),      # eight warps per token, more heads than their first pass covers
    (6, 2, 64, 1100, 592, True),       # eight, as many tokens as they are for at most; three trips
    (5, 1, 128, 32, 593, False),       # four, as few as they are for at least
    (4, 4, 64, 300, 1185, False),      # two, few rows per token
    (28, 4, 128, 65, 1300, True),      # two, many rows per token
    (48, 24, 128, 2, 1250, False),     # four again: more rows still
    (4, 4, 64, 1025, 2400, True),      # one
])
def test_append_of_many_sequences(Hq, Hkv, D, batch, tokens, interleaved):
    import torch
    import tests.gpu_harness as H
    from oracle import efim_oracle as orc
    from tests.test_gpu_parity import _custom
    new = _new_lengths(batch, tokens, D)
    cached = np.random.default_rng(batch).integers(0, 40, batch).astype(np.int32)
    w = _custom(Hq, Hkv, D, cached, new, seed=tokens, extra=0)
    dw = H.DeviceWorkload(w, interleaved=interleaved)
    dw.gpu_kv_append()
    torch.cuda.synchronize()
    assert int(dw.status.item()) == 0
    kp, vp, bt, _ = w.compact_host_pool()
    q_rot = orc.kv_append(kp, vp, bt, w.cached_len, w.new_len, dw.q_bits, dw.k_bits, dw.v_bits, w.rope_base, interleaved)
    used = np.array(sorted(set(w.block_table[w.block_table >= 0].tolist())), np.int64)
    assert np.array_equal(dw.pages_from_device("v", used), vp)
    H.assert_rope_close(dw.pages_from_device("k", used), kp, "k pages")
    H.assert_rope_close(H.torch_to_bits(dw.q), q_rot, "q")


@pytest.mark.parametrize("Hq,Hkv,D,batch,tokens", [
    (32, 8, 128, 3, 40),               # four rows a warp
    (6, 2, 64, 40, 30),                # two
    (3, 1, 128, 1100, 9),              # one; three trips
])
def test_merge_of_cut_sequences_among_many(Hq, Hkv, D, batch, tokens):
    """Few tokens over long contexts, cut into key chunks, in batches whose other sequences bring nothing."""
    import paper_2505_21889_b200 as efim
    from tests.test_gpu_parity import _check_turn, _custom
    new = _new_lengths(batch, tokens, D)
    cached = np.where(new > 0, 3000 + 7 * np.arange(batch), 5).astype(np.int32)
    dw, _ = _check_turn(_custom(Hq, Hkv, D, cached, new, seed=batch), use_rope=False)
    assert efim.efim_prefill_launch_count(dw.cache, dw.batch) == 2


def _step(dw, rope, q, k, v, out, ws, plan=None):
    import paper_2505_21889_b200 as efim
    efim.efim_append_prefill_step(dw.cache, dw.batch, rope, q, k, v, out, dw.lse, 0.0, ws, dw.status, plan=plan)


@pytest.mark.parametrize("where", ["beside", "on q", "on k", "on v"])
@pytest.mark.parametrize("Hq,Hkv,D,cached,new", [
    (32, 8, 128, [6000, 5, 700], [20, 70, 3]),          # cut key ranges: several work items read the rows
    (7, 1, 64, [0, 33, 100, 16], [300, 1, 40, 5]),      # row blocks that end inside a token
])
def test_step_with_its_output_on_other_rows(Hq, Hkv, D, cached, new, where):
    """The one-call step leaves the rotated queries where the outputs go, if nothing that the append reads lies there: the bits of
    the two calls wherever the output is."""
    import torch
    import paper_2505_21889_b200 as efim
    import tests.gpu_harness as H
    from tests.test_gpu_parity import _custom
    w = _custom(Hq, Hkv, D, cached, new, seed=Hq)
    a, b = H.DeviceWorkload(w), H.DeviceWorkload(w)
    a.gpu_kv_append()
    a.gpu_prefill()
    n_q, n_k, odd = b.q.numel(), b.k_new.numel(), 8 * D
    mem = torch.zeros(3 * n_q + 2 * n_k + odd, dtype=torch.bfloat16, device="cuda")
    q, k, v = mem[:n_q], mem[2 * n_q: 2 * n_q + n_k], mem[2 * n_q + n_k: 2 * n_q + 2 * n_k]
    for dst, src in ((q, b.q), (k, b.k_new), (v, b.v_new)):
        dst.copy_(src.flatten())
    start = {"beside": n_q, "on q": 0, "on k": n_q + odd, "on v": 2 * n_q + n_k}[where]
    out = mem[start: start + n_q]
    ws = torch.empty(efim.efim_prefill_workspace_bytes(b.cache, b.batch), dtype=torch.uint8, device="cuda")
    _step(b, b.rope, q.view_as(b.q), k.view_as(b.k_new), v.view_as(b.v_new), out.view_as(b.q), ws)
    torch.cuda.synchronize()
    assert int(a.status.item()) == int(b.status.item()) == 0
    assert torch.equal(a.out.view(torch.int16), out.view_as(b.q).view(torch.int16)) and torch.equal(a.lse, b.lse)
    assert torch.equal(a.k_pool.view(torch.int16), b.k_pool.view(torch.int16))
    assert torch.equal(a.v_pool.view(torch.int16), b.v_pool.view(torch.int16))


@pytest.mark.parametrize("interleaved", [False, True])
def test_step_rotates_queries_whose_keys_have_no_page(interleaved):
    """A rejected page drops its keys and nothing else: the token's query attends over the others, as it does when the attention
    kernel rotates the rows (the form of the call without k and v, here over the pages of the first one)."""
    import torch
    import paper_2505_21889_b200 as efim
    import tests.gpu_harness as H
    from tests.test_gpu_parity import _custom
    w = _custom(8, 2, 128, [60, 200], [40, 9], seed=5)
    w.block_table[0, 5] = w.num_pages + 3               # keys 80 .. 95 of the first sequence, new ones
    dw = H.DeviceWorkload(w, interleaved=interleaved)
    ws = torch.empty(efim.efim_prefill_workspace_bytes(dw.cache, dw.batch), dtype=torch.uint8, device="cuda")
    short = efim.Rope(w.rope_base, w.head_dim, 205, interleaved)        # and the last positions of the second have no table row
    outs = []
    for k, v in ((dw.k_new, dw.v_new), (None, None)):
        out = torch.full_like(dw.q, float("nan"))
        _step(dw, short, dw.q, k, v, out, ws)
        torch.cuda.synchronize()
        outs.append(out.view(torch.int16).clone())
        assert int(dw.status.item()) == BAD_PAGE | BAD_POSITION
    assert torch.equal(*outs) and torch.isfinite(out.float()).all()


@pytest.mark.parametrize("interleaved", [False, True])
@pytest.mark.parametrize("Hq,Hkv,tokens", [(8, 2, 40), (8, 2, 700), (48, 24, 1250), (8, 2, 1400), (8, 2, 2500)])   # 8, 4, 4, 2, 1 warps
def test_step_in_place_over_rejected_tokens(Hq, Hkv, tokens, interleaved):
    """The output on the queries themselves: tokens whose keys have no page attend with their rotated query, tokens beyond the
    rotary table with a zero query, as they do where the attention kernel rotates the rows."""
    import torch
    import paper_2505_21889_b200 as efim
    import tests.gpu_harness as H
    from tests.test_gpu_parity import _custom
    w = _custom(Hq, Hkv, 128, [60, tokens + 60], [tokens, 10], seed=6)
    w.block_table[0, 5] = w.num_pages + 3                 # keys 80 .. 95 of the first sequence, new ones
    dw = H.DeviceWorkload(w, interleaved=interleaved)
    ws = torch.empty(efim.efim_prefill_workspace_bytes(dw.cache, dw.batch), dtype=torch.uint8, device="cuda")
    short = efim.Rope(w.rope_base, w.head_dim, tokens + 68, interleaved)     # the last two positions have no table row
    outs = []
    for k, v, in_place in ((dw.k_new, dw.v_new, True), (None, None, False)):
        q = dw.q.clone()
        out = q if in_place else torch.empty_like(q)
        _step(dw, short, q, k, v, out, ws)
        torch.cuda.synchronize()
        outs.append(out.view(torch.int16).clone())
        assert int(dw.status.item()) == BAD_PAGE | BAD_POSITION
        dw.status.zero_()
    assert torch.equal(*outs) and torch.isfinite(out.float()).all()


@pytest.mark.parametrize("interleaved", [False, True])
@pytest.mark.parametrize("Hq,Hkv,D", [(32, 8, 128), (24, 8, 128), (8, 8, 64), (24, 8, 64)])
def test_attention_of_many_items_rotates_on_load(Hq, Hkv, D, interleaved):
    """The attention-only form of the step, whose CTAs rotate the queries of their second and later items as they load
    them: the bits of efim_kv_append, which rotates them in memory, followed by the attention; the queries stay."""
    import torch
    import paper_2505_21889_b200 as efim
    import tests.gpu_harness as H
    from tests.test_gpu_items import _items, _lengths_of_every_shape
    from tests.test_gpu_parity import _custom
    w = _custom(Hq, Hkv, D, *_lengths_of_every_shape(Hq, Hkv, D), seed=Hq + D)
    a = H.DeviceWorkload(w, interleaved=interleaved)
    assert _items(a) >= 3 * torch.cuda.get_device_properties(0).multi_processor_count
    q = a.q.clone()
    a.gpu_kv_append()
    a.gpu_prefill()
    ws = torch.empty(efim.efim_prefill_workspace_bytes(a.cache, a.batch), dtype=torch.uint8, device="cuda")
    out, lse = torch.empty_like(q), torch.empty_like(a.lse)
    for _ in range(2):
        out.fill_(float("nan"))
        efim.efim_append_prefill_step(a.cache, a.batch, a.rope, q, None, None, out, lse, 0.0, ws, a.status)
        torch.cuda.synchronize()
        assert int(a.status.item()) == 0
        assert torch.equal(a.out.view(torch.int16), out.view(torch.int16)) and torch.equal(a.lse, lse)
        assert torch.equal(q.view(torch.int16), H.bits_to_torch(a.q_bits).view(torch.int16))


class _KernelNodeParams(ctypes.Structure):       # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3), ("shared", ctypes.c_uint),
                ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p), ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def _blocks_of(call):
    """Blocks of the one kernel that a call enqueues, read off a graph it is captured into."""
    import torch
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    cu, handle = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(graph.raw_cuda_graph())
    nodes, n, p = (ctypes.c_void_p * 2)(), ctypes.c_size_t(2), _KernelNodeParams()
    assert cu.cuGraphGetNodes(handle, nodes, ctypes.byref(n)) == 0 and n.value == 1
    assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(nodes[0]), ctypes.byref(p)) == 0
    return p.grid[0]


@pytest.mark.parametrize("Hq,Hkv,D,tokens,with_q,without", [
    (28, 4, 128, 3000, 2, 1),              # warps per token
    (48, 8, 64, 2400, 2, 1),
    (32, 32, 128, 1200, 4, 4),             # k and v alone are as many rows
    (4, 4, 64, 3000, 1, 1),
])
def test_append_without_queries_has_the_warps_that_its_rows_keep_busy(Hq, Hkv, D, tokens, with_q, without):
    """Beyond what is resident at once, a token has as many warps as the rows that are moved keep busy: without q those of k
    and v."""
    import paper_2505_21889_b200 as efim
    import tests.gpu_harness as H
    from tests.test_gpu_parity import _custom
    dw = H.DeviceWorkload(_custom(Hq, Hkv, D, [5, 40], [tokens - 10, 10], seed=1))
    for q, warps in ((dw.q, with_q), (None, without)):
        blocks = _blocks_of(lambda: efim.efim_kv_append(dw.cache, dw.batch, dw.rope, q, dw.k_new, dw.v_new, dw.status))
        assert blocks == -(-tokens * warps * 32 // 256)


@pytest.mark.parametrize("Hq,Hkv,D", [(32, 8, 128), (6, 2, 64), (3, 1, 128)])
def test_merge_of_rows_without_a_finite_score(Hq, Hkv, D):
    """All scores of a row that is cut into key chunks are minus infinity (their keys are -3e38, the queries 3e38): output 0 and
    lse -inf, whatever its values hold - a partial without weight is not looked at."""
    import torch
    import paper_2505_21889_b200 as efim
    import tests.gpu_harness as H
    from tests.test_gpu_parity import _custom
    w = _custom(Hq, Hkv, D, [9000, 40], [20, 3], seed=D + Hq)      # (more than 32 rows to a kv head)
    dw = H.DeviceWorkload(w, use_rope=False)
    assert efim.efim_prefill_launch_count(dw.cache, dw.batch) == 2
    dw.k_pool.fill_(-3e38)
    dw.v_pool.fill_(float("inf"))
    dw.q[:20].fill_(3e38)
    dw.gpu_prefill()
    torch.cuda.synchronize()
    assert int(dw.status.item()) == 0
    assert bool((dw.out[:20].float() == 0).all()) and bool((dw.lse[:20] == float("-inf")).all())


@pytest.mark.parametrize("Hq,Hkv,D,cached,new", [
    (6, 2, 64, [4000, 10, 5000, 4500], [300, 5, 330, 280]),
    (5, 1, 128, [3000, 0, 4000], [500, 7, 620]),
])
def test_merge_of_many_rows_at_other_head_counts(Hq, Hkv, D, cached, new):
    """Cut key ranges and more rows than eight chunks in flight are for, where four heads are not a divisor of all."""
    import torch
    import paper_2505_21889_b200 as efim
    from tests.test_gpu_parity import _check_turn, _custom
    assert sum(new) * Hq > 32 * torch.cuda.get_device_properties(0).multi_processor_count
    dw, _ = _check_turn(_custom(Hq, Hkv, D, cached, new, seed=Hq), use_rope=False)
    assert efim.efim_prefill_launch_count(dw.cache, dw.batch) == 2


@pytest.mark.parametrize("Hq,Hkv,D,cached,new,rows_per_sm", [
    (16, 1, 128, [2000, 900, 7], [200, 150, 4], 32),       # one row a warp, four chunks in flight
    (32, 8, 128, [1500, 900, 7], [300, 90, 4], 80),        # four rows a warp
    (28, 4, 64, [2000, 900, 7], [300, 150, 4], 80),
    (6, 2, 64, [3000, 10], [2000, 5], 80),                 # two
    (14, 2, 128, [3000, 2000], [600, 300], 80),
])
def test_merge_forms_of_many_rows(Hq, Hkv, D, cached, new, rows_per_sm):
    """Cut key ranges on either side of where a warp takes more than one row."""
    import torch
    import paper_2505_21889_b200 as efim
    from tests.test_gpu_parity import _check_turn, _custom
    rows = sum(new) * Hq / torch.cuda.get_device_properties(0).multi_processor_count
    assert rows > 80 if rows_per_sm == 80 else 32 < rows <= 80
    dw, _ = _check_turn(_custom(Hq, Hkv, D, cached, new, seed=Hq), use_rope=False)
    assert efim.efim_prefill_launch_count(dw.cache, dw.batch) == 2
