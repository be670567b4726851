"""Append-prefill launches whose CTAs walk several work items each, of one query tile, two and at most 32 rows in turn:
whatever one item leaves behind (ring positions, barrier phases, queries, O, staged output rows) the next one must not see."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hq,Hkv,D", [(32, 8, 128), (56, 8, 128), (8, 8, 64), (24, 8, 64)])
def test_items_of_every_shape_in_turn(Hq, Hkv, D):
    """160 sequences (more than 8 items per SM, so in order of sequence and not of cost); rows around the edges of the
    32-row groups and of the tiles, contexts around page and step edges, empty ones among them.  (Without rotation, so
    that the oracle's queries and keys are the kernel's bit for bit: in a row of one key a single bf16 tie that rounds the
    other way moves the lse by up to 2.7e-3.)"""
    from tests.test_gpu_parity import _check_turn, _custom
    _check_turn(_custom(Hq, Hkv, D, *_lengths_of_every_shape(Hq, Hkv, D), seed=Hq + D), use_rope=False)


def _lengths_of_every_shape(Hq, Hkv, D):
    """Cached and new tokens of 160 sequences."""
    G = Hq // Hkv
    rng = np.random.default_rng([Hq, Hkv, D])
    rows = np.array([G, 20, 31, 32, 33, 64, 100, 128, 129, 200, 256, 257, 300, 520])
    new = np.maximum(1, rng.permutation(np.tile(rows, 12))[:160] // G).astype(np.int32)
    return rng.choice([0, 1, 15, 16, 79, 80, 81, 160, 200, 239], 160).astype(np.int32), new


def _items(dw):
    """Number of work items in the plan of a workload's batch (the seventh word of the plan)."""
    import paper_2505_21889_b200 as efim
    plan = efim.efim_prefill_plan(dw.cache, dw.batch)
    return int(np.frombuffer(bytes(bytearray(np.asarray(plan)[:32].view(np.uint8))), np.int32)[6])


@pytest.mark.parametrize("interleaved", [False, True])
@pytest.mark.parametrize("Hq,Hkv,D", [(32, 8, 128), (24, 8, 128), (8, 8, 64), (24, 8, 64)])
def test_items_of_every_shape_rotated_on_load(Hq, Hkv, D, interleaved):
    """The same batches as one-call steps, whose CTAs rotate the queries of their second and later items as they load them:
    the bits of efim_kv_append, which rotates them in memory, followed by the attention."""
    import torch
    import paper_2505_21889_b200 as efim
    import tests.gpu_harness as H
    from tests.test_gpu_parity import _custom
    w = _custom(Hq, Hkv, D, *_lengths_of_every_shape(Hq, Hkv, D), seed=Hq + D)
    a, b = H.DeviceWorkload(w, interleaved=interleaved), H.DeviceWorkload(w, interleaved=interleaved)
    assert _items(a) >= 3 * torch.cuda.get_device_properties(0).multi_processor_count
    a.gpu_kv_append()
    a.gpu_prefill()
    ws = torch.empty(efim.efim_prefill_workspace_bytes(b.cache, b.batch), dtype=torch.uint8, device="cuda")
    for _ in range(2):
        b.out.fill_(float("nan"))
        efim.efim_append_prefill_step(b.cache, b.batch, b.rope, b.q, b.k_new, b.v_new, b.out, b.lse, 0.0, ws, b.status)
        torch.cuda.synchronize()
        assert int(a.status.item()) == int(b.status.item()) == 0
        assert torch.equal(a.out.view(torch.int16), b.out.view(torch.int16)) and torch.equal(a.lse, b.lse)
        assert torch.equal(a.k_pool.view(torch.int16), b.k_pool.view(torch.int16))


@pytest.mark.parametrize("Hq,Hkv,D,cached,new", [
    (32, 8, 64, [849, 472, 698, 78, 63, 600, 43, 820, 527, 225, 117, 432], [1, 8, 1, 35, 32, 32, 8, 50, 64, 1, 8, 32]),
    (24, 8, 128, [647, 606, 35, 261, 177, 737, 776, 180, 115, 612, 541, 163, 67], [1, 6, 1, 66, 6, 46, 6, 66, 1, 46, 11, 6, 33]),
])
def test_items_of_cut_key_ranges_in_turn(Hq, Hkv, D, cached, new):
    """More items than SMs, of all three shapes and of sequences cut into key chunks: partials leave through the staged stores
    of a CTA's second item too."""
    import torch
    import paper_2505_21889_b200 as efim
    from tests.test_gpu_parity import _check_turn, _custom
    dw, _ = _check_turn(_custom(Hq, Hkv, D, cached, new, seed=D), use_rope=False)
    assert _items(dw) > torch.cuda.get_device_properties(0).multi_processor_count
    assert efim.efim_prefill_launch_count(dw.cache, dw.batch) == 2


@pytest.mark.parametrize("Hq,Hkv,D,cached,new,interleaved,max_position,bad_page", [
    (4, 4, 64, [240], [16], False, None, False),
    (32, 8, 128, [0], [64], False, None, False),               # 256 rows, nothing cached
    (28, 4, 128, [79, 300], [36, 0], True, None, False),       # the last key of a step is new; an idle sequence beside it
    (8, 8, 128, [0, 80], [0, 256], False, None, False),        # the first key of a step is new
    (16, 1, 128, [81], [1], True, None, False),
    (24, 8, 64, [1000], [33], False, 1010, False),             # positions beyond the rotary table
    (8, 2, 128, [250], [40], False, None, True),               # a new token's page id outside the pool
])
def test_rows_appended_by_the_attention_kernel(Hq, Hkv, D, cached, new, interleaved, max_position, bad_page):
    """A step of one sequence of at most 256 rows (one launch) against efim_kv_append without q and the attention-only
    step: out, lse, pools and status bit for bit."""
    import torch
    import paper_2505_21889_b200 as efim
    import tests.gpu_harness as H
    from tests.test_gpu_parity import _custom
    w = _custom(Hq, Hkv, D, cached, new, seed=3 * D + Hq)
    if bad_page:
        w.block_table[0, cached[0] // 16 + 1] = w.num_pages + 5
    a, b = H.DeviceWorkload(w, interleaved=interleaved), H.DeviceWorkload(w, interleaved=interleaved)
    rope = efim.Rope(w.rope_base, D, max_position or int((w.cached_len + w.new_len).max()), interleaved)
    ws = torch.empty(max(efim.efim_prefill_workspace_bytes(a.cache, a.batch), 256), dtype=torch.uint8, device="cuda")
    efim.efim_kv_append(a.cache, a.batch, rope, None, a.k_new, a.v_new, a.status)
    efim.efim_append_prefill_step(a.cache, a.batch, rope, a.q, None, None, a.out, a.lse, 0.0, ws, a.status)
    for _ in range(2):                                         # (again over pages that hold the tokens already)
        efim.efim_append_prefill_step(b.cache, b.batch, rope, b.q, b.k_new, b.v_new, b.out, b.lse, 0.0, ws, b.status)
    torch.cuda.synchronize()
    assert int(a.status.item()) == int(b.status.item()) == (2 if max_position else 1 if bad_page else 0)
    assert torch.equal(a.out.view(torch.int16), b.out.view(torch.int16)) and torch.equal(a.lse, b.lse)
    assert torch.equal(a.k_pool.view(torch.int16), b.k_pool.view(torch.int16))
    assert torch.equal(a.v_pool.view(torch.int16), b.v_pool.view(torch.int16))


def _kernels_of(call):
    """Number of kernels a call enqueues: the nodes of a graph it is captured into (these calls copy nothing)."""
    import ctypes
    import torch
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    n = ctypes.c_size_t()
    assert ctypes.CDLL("libcudart.so.12").cudaGraphGetNodes(ctypes.c_void_p(graph.raw_cuda_graph()), None, ctypes.byref(n)) == 0
    return n.value


class _OneSequenceStep:
    """The same step twice over: as one call (`b`), and as efim_kv_append without q followed by the attention only (`a`)."""

    def __init__(self, w, interleaved=False, max_position=None):
        import torch
        import paper_2505_21889_b200 as efim
        import tests.gpu_harness as H
        self.efim, self.torch = efim, torch
        self.a, self.b = H.DeviceWorkload(w, interleaved=interleaved), H.DeviceWorkload(w, interleaved=interleaved)
        self.rope = efim.Rope(w.rope_base, w.head_dim, max_position or int((w.cached_len + w.new_len).max()), interleaved)
        self.ws = torch.empty(max(efim.efim_prefill_workspace_bytes(self.a.cache, self.a.batch), 256), dtype=torch.uint8,
                              device="cuda")
        assert efim.efim_prefill_launch_count(self.a.cache, self.a.batch) == 1       # not cut

    def two_calls(self, sm_scale=0.0, lse=True):
        a = self.a
        self.efim.efim_kv_append(a.cache, a.batch, self.rope, None, a.k_new, a.v_new, a.status)
        self.efim.efim_append_prefill_step(a.cache, a.batch, self.rope, a.q, None, None, a.out, a.lse if lse else None, sm_scale,
                                           self.ws, a.status)

    def one_call(self, sm_scale=0.0, lse=True, out=None, out_lse=None):
        b = self.b
        out_lse = (b.lse if out_lse is None else out_lse) if lse else None
        self.efim.efim_append_prefill_step(b.cache, b.batch, self.rope, b.q, b.k_new, b.v_new, b.out if out is None else out,
                                           out_lse, sm_scale, self.ws, b.status)

    def same(self, out=None, out_lse=None):
        a, b, i16, equal = self.a, self.b, self.torch.int16, self.torch.equal
        self.torch.cuda.synchronize()
        return (equal(a.out.view(i16), (b.out if out is None else out).view(i16))
                and equal(a.lse, b.lse if out_lse is None else out_lse)
                and equal(a.k_pool.view(i16), b.k_pool.view(i16)) and equal(a.v_pool.view(i16), b.v_pool.view(i16)))


@pytest.mark.parametrize("what", ["nothing", "out on k", "out on v", "lse on k", "lse on v"])
def test_outputs_may_overlap_the_new_rows(what):
    """A step whose output or lse lies on its new k or v rows equals append, then attention; it takes two kernels then, as the
    append has to have read all rows before the first output is stored."""
    import torch
    from tests.test_gpu_parity import _custom
    s = _OneSequenceStep(_custom(8, 8, 128, [100], [20], seed=11))
    s.two_calls()
    args = {}
    rows = s.b.k_new if what.endswith("k") else s.b.v_new
    if what.startswith("out"):
        args["out"] = rows
    if what.startswith("lse"):
        args["out_lse"] = rows.view(torch.uint8).flatten()[256:256 + 20 * 8 * 4].view(torch.float32).view(20, 8)
    s.one_call(**args)
    assert s.same(**args) and int(s.b.status.item()) == 0
    assert _kernels_of(lambda: s.one_call(**args)) == (1 if what == "nothing" else 2)


@pytest.mark.parametrize("Hq,Hkv,D,cached,new,old,renewed", [
    (32, 8, 128, 300, 16, 1, 19),          # a page of the first step is the one that the new tokens fill
    (8, 8, 64, 330, 40, 7, 21),            # ... of a later step, and the second of three pages
    (4, 4, 64, 17, 16, 0, 2),              # within the first step
])
def test_a_page_named_twice(Hq, Hkv, D, cached, new, old, renewed):
    """A table that names one page for cached keys and again for new ones: the cached keys are what the step writes there, as
    they are behind an append of its own.  (New k and v each time: a copy made too early would bring the old ones.)"""
    import torch
    from tests.test_gpu_parity import _custom
    w = _custom(Hq, Hkv, D, [cached], [new], seed=5)
    w.block_table[0, old] = w.block_table[0, renewed]
    s = _OneSequenceStep(w)
    assert _kernels_of(s.one_call) == 1
    gen = torch.Generator(device="cuda").manual_seed(3)
    for _ in range(20):
        for x, y in ((s.a.k_new, s.b.k_new), (s.a.v_new, s.b.v_new)):
            x.copy_(torch.randn(x.shape, device="cuda", generator=gen))
            y.copy_(x)
        s.two_calls()
        s.one_call()
        assert s.same()


@pytest.mark.parametrize("Hq,Hkv,D,new,kernels", [(4, 4, 64, 128, 1), (4, 4, 64, 129, 2), (32, 8, 128, 32, 1), (32, 8, 128, 33, 2),
                                                  (16, 1, 128, 8, 1), (16, 1, 128, 16, 2), (8, 8, 128, 256, 2)])
def test_one_kernel_up_to_one_query_tile(Hq, Hkv, D, new, kernels):
    """A step of one sequence is one kernel up to 128 rows, where that is the faster form, and two beyond; the same bits."""
    from tests.test_gpu_parity import _custom
    s = _OneSequenceStep(_custom(Hq, Hkv, D, [0], [new], seed=new))
    s.two_calls()
    assert _kernels_of(s.one_call) == kernels
    s.one_call()
    assert s.same()


def test_one_sequence_step_whose_list_is_copied():
    """One sequence brings new tokens, in a batch too long for lists in the launch parameters: its rows are appended by a kernel
    of their own, as only kernels with the list in the parameters can."""
    from tests.test_gpu_parity import _custom
    new = np.zeros(257, np.int32)
    new[100] = 20
    s = _OneSequenceStep(_custom(8, 8, 128, np.full(257, 40, np.int32), new, seed=4))
    s.two_calls()
    s.one_call()
    assert s.same() and int(s.b.status.item()) == 0


@pytest.mark.parametrize("Hq,Hkv,D,new", [(32, 8, 128, 36), (8, 8, 64, 100), (32, 8, 128, 5), (32, 8, 128, 40)])
def test_nan_queries_of_one_sequence_do_not_slow_another(Hq, Hkv, D, new):
    """The rows past a sequence in a block of 32 may hold the next sequence's queries; NaN there must not change what the
    sequence gets, nor make its warps redo their steps (which took 1.25 times as long and more)."""
    import torch
    import paper_2505_21889_b200 as efim
    import tests.gpu_harness as H
    from tests.test_gpu_parity import _custom
    dw = H.DeviceWorkload(_custom(Hq, Hkv, D, [16384, 0], [new, 8], seed=8), use_rope=False)
    ws = torch.empty(efim.efim_prefill_workspace_bytes(dw.cache, dw.batch), dtype=torch.uint8, device="cuda")
    clean = dw.q.clone()
    poisoned = dw.q.clone()
    poisoned[new:] = float("nan")
    out = {}
    times = {"clean": [], "poisoned": []}
    for _ in range(15):
        for what, q in (("clean", clean), ("poisoned", poisoned)):
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            start.record()
            for _ in range(10):
                efim.efim_append_prefill_attn(dw.cache, dw.batch, q, dw.out, dw.lse, 0.0, ws, dw.status)
            end.record()
            torch.cuda.synchronize()
            times[what].append(start.elapsed_time(end))
            out[what] = dw.out[:new].clone()
    assert torch.equal(out["clean"].view(torch.int16), out["poisoned"].view(torch.int16))
    assert dw.out[new:].isnan().all()
    ratio = np.median(times["poisoned"]) / np.median(times["clean"])
    assert ratio < 1.1, f"{ratio:.3f} times as long behind NaN queries"


@pytest.mark.parametrize("Hq,Hkv,D,cached,new,interleaved,max_position,sm_scale,lse", [
    (8, 8, 128, [0, 80], [0, 128], False, None, 0.0, True),     # 128 rows; the first key of a step is new; an idle sequence
    (32, 8, 128, [79], [32], True, None, 0.3, True),            # the last key of a step is new
    (24, 8, 64, [200], [33], False, 210, 0.0, True),            # positions beyond the rotary table
    (24, 8, 64, [200], [33], True, 210, 0.0, True),
    (64, 2, 128, [100], [4], False, None, 0.05, False),         # 32 heads a group; no lse
    (16, 1, 128, [0], [8], False, None, 0.0, False),
])
def test_rows_appended_by_the_only_kernel(Hq, Hkv, D, cached, new, interleaved, max_position, sm_scale, lse):
    """Steps that are one kernel, against efim_kv_append without q and the attention-only step, bit for bit."""
    from tests.test_gpu_parity import _custom
    s = _OneSequenceStep(_custom(Hq, Hkv, D, cached, new, seed=D + Hq), interleaved, max_position)
    for d in (s.a, s.b):
        d.lse.fill_(7.0)
    s.two_calls(sm_scale, lse)
    s.one_call(sm_scale, lse)
    assert s.same()
    assert int(s.a.status.item()) == int(s.b.status.item()) == (2 if max_position else 0)
    assert bool((s.b.lse == 7.0).all()) == (not lse)
    assert _kernels_of(lambda: s.one_call(sm_scale, lse)) == 1


@pytest.mark.parametrize("Hq,Hkv,D", [(64, 2, 128), (32, 1, 64), (32, 2, 64)])
def test_rows_of_wide_groups_as_boxes(Hq, Hkv, D):
    """32 and 16 query heads to a kv head: a box of 32 rows is one token's, or two tokens'."""
    from tests.test_gpu_parity import _check_turn, _custom
    _check_turn(_custom(Hq, Hkv, D, [70, 0, 200, 31], [1, 9, 8, 17], seed=Hq), use_rope=False)
