"""Kernels whose warps look a token's sequence up 32 candidates at a time: batches of more than one and of more than two such
trips, with sequences that bring nothing among them; and every number of warps per token of the append."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


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
