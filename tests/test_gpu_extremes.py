"""GPU: infinities, NaN and values near the ends of bf16's range in the cache and in q, against the
oracle on the same bits.  Attention is a weighted mean: a key whose score is -inf has no weight, a NaN
that a row sees makes the row NaN, an infinite value makes its dimension infinite."""
import numpy as np
import pytest
import torch

from oracle import efim_oracle as orc

pytestmark = pytest.mark.gpu

HQ, HKV = 8, 2
# new tokens at 4 query heads per kv head: 32-row CTAs, one query tile, two query tiles
SHAPES = [5, 20, 60]


class _Rows:
    """One sequence per entry of `cached` (`new` tokens each) over pages in order; pools and q are device tensors to be
    edited before a call."""

    def __init__(self, cached, new, D=128, seed=0):
        import paper_2505_21889_b200 as efim
        self.efim = efim
        self.cached, self.new, self.D = np.array(cached, np.int32), np.full(len(cached), new, np.int32), D
        need = -(-(self.cached + self.new) // 16)
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        shape = (int(need.sum()), HKV, 16, D)
        self.k = torch.randn(shape, generator=g, device="cuda").bfloat16()
        self.v = torch.randn(shape, generator=g, device="cuda").bfloat16()
        self.q = torch.randn((int(self.new.sum()), HQ, D), generator=g, device="cuda").bfloat16()
        first = np.concatenate([[0], np.cumsum(need)])
        self.table = np.zeros((len(cached), int(need.max())), np.int32)
        for s in range(len(cached)):
            self.table[s, :need[s]] = np.arange(first[s], first[s + 1])
        self.status = torch.zeros(1, dtype=torch.int32, device="cuda")

    def _call(self, fn):
        out = torch.full_like(self.q, 7.0)
        lse = torch.full(self.q.shape[:2], 7.0, dtype=torch.float32, device="cuda")
        fn(out, lse)
        torch.cuda.synchronize()
        assert int(self.status.item()) == 0
        return out.float().cpu().numpy().astype(np.float64), lse.cpu().numpy().astype(np.float64)

    def prefill(self):
        efim = self.efim
        cache, batch = efim.Cache(self.k, self.v, HQ), efim.Batch(self.cached, self.new, self.table)
        ws = torch.empty(max(efim.efim_prefill_workspace_bytes(cache, batch), 256), dtype=torch.uint8, device="cuda")
        return self._call(lambda out, lse: efim.efim_append_prefill_attn(cache, batch, self.q, out, lse, 0.0, ws,
                                                                         self.status))

    def decode(self):
        """One query row per sequence (new = 1) over all its keys."""
        efim = self.efim
        cache, total = efim.Cache(self.k, self.v, HQ), self.cached + self.new
        ws = torch.empty(max(efim.efim_decode_workspace_bytes(cache, len(total), int(total.max())), 256),
                         dtype=torch.uint8, device="cuda")
        ctx, table = torch.from_numpy(total).cuda(), torch.from_numpy(self.table).cuda()
        return self._call(lambda out, lse: efim.efim_decode_attn(cache, len(total), ctx, int(total.max()), table, self.q,
                                                                 out, lse, 0.0, ws, self.status))

    def _bits(self):
        from tests.gpu_harness import torch_to_bits
        return torch_to_bits(self.q), torch_to_bits(self.k), torch_to_bits(self.v)

    def prefill_oracle(self):
        q, k, v = self._bits()
        with np.errstate(all="ignore"):
            return orc.append_prefill_attention(q, k, v, self.table, self.cached, self.new, HQ)

    def decode_oracle(self):
        q, k, v = self._bits()
        with np.errstate(all="ignore"):
            return orc.decode_attention(q, k, v, self.table, self.cached + self.new, HQ)


@pytest.mark.parametrize("new", SHAPES)
@pytest.mark.parametrize("cached", [300, 6000])                # 6000: the key range is cut, partials are merged
def test_prefill_first_keys_of_infinitely_low_score(cached, new):
    """The keys of a row's first steps have the score -inf: they have no weight, and the reference comes
    from the first finite score."""
    r = _Rows([cached], new)
    r.q[:, :, 0] = 1.0
    r.k[:10] = 0.0                                             # 160 keys: two steps
    r.k[:10, :, :, 0] = -torch.inf
    out, lse = r.prefill()
    o, want = r.prefill_oracle()
    assert np.abs(out - o).max() <= 2e-2 and np.abs(lse - want).max() <= 1e-3


@pytest.mark.parametrize("new", SHAPES)
@pytest.mark.parametrize("cached", [300, 6000])
def test_prefill_values_near_the_end_of_the_range(cached, new):
    """Peaked rows over values of up to 1e36: the weighted mean of finite values is finite.  Bound: output and
    probabilities are rounded to bf16 (2^-9 each), so the 2-norm error stays below 2 * 2^-9."""
    r = _Rows([cached], new)
    r.k *= 8.0
    r.v = (r.v.float() * 2e35).bfloat16()
    out, lse = r.prefill()
    o, want = r.prefill_oracle()
    assert np.isfinite(out).all()
    assert np.linalg.norm((out - o) / 2e35) <= 2.0 ** -8 * np.linalg.norm(o / 2e35)
    assert np.abs(lse - want).max() <= 1e-3


@pytest.mark.parametrize("new", SHAPES)
def test_prefill_key_far_above_the_others_is_returned_exactly(new):
    """A key 2^30 times as heavy as any other, behind the row's first steps: its probability is 1 without
    rounding, so the output is its value bit for bit (the others move it by 700 * 2^-30).  Against the
    others it is 2^30.0054 = 2^30 * 1.00378, halfway between two bf16 values: rounded there, most
    outputs would move to the neighbouring value."""
    r = _Rows([700], new)
    r.k.zero_()
    r.q[:, :, 0] = 1.0
    r.q[:, :, 1] = 1.0
    r.k[31, :, 4, 0] = 235.0                                   # position 500; (235 + 0.3046875) log2(e) / sqrt(128)
    r.k[31, :, 4, 1] = 0.3046875
    out, _ = r.prefill()
    v = r.v[31, :, 4].float().cpu().numpy()
    assert np.array_equal(out, np.broadcast_to(np.repeat(v, HQ // HKV, axis=0), out.shape))


@pytest.mark.parametrize("new,pos", [(5, 200), (20, 200), (60, 100)])
def test_prefill_heaviest_key_in_the_second_step_is_weighted_without_rounding(new, pos):
    """A key 2^7.0055 = 128 * 1.0038 times as heavy as each of the others, in the second step of its stream, and
    values of zero everywhere else: the output is its value times its exact weight.  Rounded to bf16 against
    the first step's reference the weight would be off by 0.0038 and nearly every output with it."""
    from oracle.efim_oracle import bf16_to_f64, f64_to_bf16
    r = _Rows([300], new)
    r.k.zero_()
    r.v[:, :, :, :] = torch.where(torch.arange(16, device="cuda")[None, None, :, None] == pos % 16, r.v, 0)
    r.v[:pos // 16], r.v[pos // 16 + 1:] = 0.0, 0.0
    r.q[:, :, :2] = 1.0
    r.k[pos // 16, :, pos % 16, 0] = 54.75                     # (54.75 + 0.1875) log2(e) / sqrt(128)
    r.k[pos // 16, :, pos % 16, 1] = 0.1875
    out, _ = r.prefill()
    o, _ = r.prefill_oracle()
    assert (out == bf16_to_f64(f64_to_bf16(o))).mean() >= 0.99


def _same_or_nan(out, lse, o, want):
    """Equal within the attention tolerances, and NaN exactly where the oracle has NaN."""
    assert np.array_equal(np.isnan(out), np.isnan(o)) and np.array_equal(np.isnan(lse), np.isnan(want))
    ok, lok = ~np.isnan(o), ~np.isnan(want)
    assert ok.any() and not ok.all()
    assert np.abs(out[ok] - o[ok]).max() <= 2e-2 and np.abs(lse[lok] - want[lok]).max() <= 1e-3


@pytest.mark.parametrize("new", SHAPES)
@pytest.mark.parametrize("cached", [300, 6000])
@pytest.mark.parametrize("where", ["q", "k", "many_k"])
def test_prefill_nan_scores_make_their_rows_nan(where, cached, new):
    """A NaN in a query row, in one cached key or in all keys of a stretch longer than any chunk: the rows
    that see it are NaN, out and lse, and no key is silently left out; all others are untouched."""
    r = _Rows([cached], new)
    if where == "q":
        r.q[1, 1, 3] = torch.nan
    elif where == "k":
        r.k[2, 0, 5, 7] = torch.nan                            # position 37, kv head 0
    else:
        r.k[:cached // 16 - 1, 0] = torch.nan
    out, lse = r.prefill()
    _same_or_nan(out, lse, *r.prefill_oracle())


@pytest.mark.parametrize("D", [128, 64])
@pytest.mark.parametrize("total", [200, 1500])                 # 1500: several chunks, merged
def test_decode_keys_of_infinitely_low_score(total, D):
    """The first 160 keys (whole pages of three or four warps) and single later ones have the score -inf: no weight."""
    r = _Rows([total - 1], 1, D=D)
    r.q[:, :, 0] = 1.0
    for key in list(range(160)) + [170, total - 1]:
        r.k[key // 16, :, key % 16] = 0.0
        r.k[key // 16, :, key % 16, 0] = -torch.inf
    out, lse = r.decode()
    o, want = r.decode_oracle()
    assert np.abs(out - o).max() <= 2e-2 and np.abs(lse - want).max() <= 1e-3


@pytest.mark.parametrize("total", [200, 1500, 5000])           # one chunk; a few; more than eight (merge on four warps)
@pytest.mark.parametrize("where", ["q", "k", "last_k", "many_k"])
def test_decode_nan_scores_make_their_rows_nan(where, total):
    """A NaN in a query row, in one key, in the last 256 keys (whole chunks) or in all but the first 16: the heads
    that see it are NaN, out and lse; the other kv head and the other row are untouched."""
    r = _Rows([total - 1, total // 2], 1)
    if where == "q":
        r.q[0, 1, 3] = torch.nan
    elif where == "k":
        r.k[2, 0, 5, 7] = torch.nan
    else:
        pages = -(-total // 16)                                # of the first row
        r.k[pages - 16 if where == "last_k" and pages > 32 else 1:pages, 0] = torch.nan
    out, lse = r.decode()
    _same_or_nan(out, lse, *r.decode_oracle())


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("D", [128, 64])
@pytest.mark.parametrize("total", [200, 1500, 5000])
def test_decode_infinite_values(total, D, fused):
    """Infinite values in the cache, and in the new token of a fused step: their dimensions are infinite, NaN where
    both signs or a NaN meet, and every other dimension is what it was."""
    r = _Rows([total - 1, total // 2], 1, D=D)
    first = [0, 37, total // 2, total - 1]                     # keys of the first row
    for n, key in enumerate(first):
        r.v[key // 16, 0, key % 16, 5 + 8 * n] = torch.inf
        r.v[key // 16, 1, key % 16, 6 + 8 * n] = -torch.inf
    r.v[2, :, 5, 40], r.v[3, :, 7, 40] = torch.inf, -torch.inf # both signs
    r.v[1, :, 3, 41] = torch.nan
    if fused:
        from paper_2505_21889_b200 import efim_decode_step, Cache, efim_decode_workspace_bytes
        lens = r.cached + r.new
        spot = [(int(r.table[s, (n - 1) // 16]), int(n - 1) % 16) for s, n in enumerate(lens)]
        k_new = torch.stack([r.k[p, :, t] for p, t in spot])
        v_new = torch.stack([r.v[p, :, t] for p, t in spot])
        o, want = r.decode_oracle()
        for p, t in spot:                                      # what is in the slot before is not looked at
            r.k[p, :, t], r.v[p, :, t] = torch.nan, torch.nan
        cache = Cache(r.k, r.v, HQ)
        ws = torch.empty(max(efim_decode_workspace_bytes(cache, 2, total), 256), dtype=torch.uint8, device="cuda")
        ctx, table = torch.from_numpy(lens).cuda(), torch.from_numpy(r.table).cuda()
        out, lse = r._call(lambda out, lse: efim_decode_step(cache, 2, ctx, total, table, None, r.q, k_new, v_new, out, lse,
                                                             0.0, ws, r.status))
    else:
        o, want = r.decode_oracle()
        out, lse = r.decode()
    assert np.array_equal(np.isnan(out), np.isnan(o)) and np.isnan(o).any()
    assert np.array_equal(np.isposinf(out), np.isposinf(o)) and np.array_equal(np.isneginf(out), np.isneginf(o))
    ok = np.isfinite(o)
    assert np.abs(out[ok] - o[ok]).max() <= 2e-2 and np.abs(lse - want).max() <= 1e-3


def test_decode_probabilities_keep_fp32_precision():
    """46 keys of weight 1 and value 1 against 93 of weight p = 2^(-7.28125 log2(e) / sqrt(128)) = 0.5254 and value -w: the
    mean cancels to 3e-8, so that the error of p is what is left.  Rounded to one bf16 term p is off by 2^-8.1, to
    two by 2^-17.2.  Bound: the exponential and the two sums are good to 2^-21 of sums of weight 1."""
    from oracle.efim_oracle import bf16_to_f64, f64_to_bf16
    r = _Rows([138], 1)
    r.k.zero_()
    r.q[:, :, 0] = 1.0
    w = 0.94140625
    heavy = np.array([i % 3 == 0 and i < 138 for i in range(139)])
    for i in range(139):
        r.k[i // 16, :, i % 16, 0] = 0.0 if heavy[i] else -7.28125
        r.v[i // 16, :, i % 16] = 1.0 if heavy[i] else -w
    out, _ = r.decode()
    o, _ = r.decode_oracle()
    limit = 2.0 ** -21
    assert np.abs(o).max() < 1e-7 and np.abs(out - o).max() <= limit
    # the bound sees a p of one or two bf16 terms (planted here, in 64 bits)
    p = np.exp(-7.28125 / np.sqrt(128.0))
    high = bf16_to_f64(f64_to_bf16(p))
    for terms in (high, high + bf16_to_f64(f64_to_bf16(p - high))):
        assert abs((heavy.sum() - (~heavy).sum() * terms * w) / (heavy.sum() + (~heavy).sum() * p)) > 4 * limit
