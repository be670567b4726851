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
    G = Hq // Hkv
    rng = np.random.default_rng([Hq, Hkv, D])
    rows = np.array([G, 20, 31, 32, 33, 64, 100, 128, 129, 200, 256, 257, 300, 520])
    new = np.maximum(1, rng.permutation(np.tile(rows, 12))[:160] // G).astype(np.int32)
    cached = rng.choice([0, 1, 15, 16, 79, 80, 81, 160, 200, 239], 160).astype(np.int32)
    _check_turn(_custom(Hq, Hkv, D, cached, new, seed=Hq + D), use_rope=False)
