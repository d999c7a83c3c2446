"""The rules of the multi-layer calls, on the host: KV heads per unit of the selection (one selection per
layer), items per unit of the scoring."""
import ctypes

import numpy as np
import pytest

import ckv_synth as cs
import paper_2508_02401_gb300 as ckv
from paper_2508_02401_gb300 import build as ckv_build


@pytest.mark.parametrize("layers,seqs,length,budget,kv_heads,want", [
    (8, 1, 8192, 256, 8, 1), (32, 1, 8192, 256, 8, 2), (32, 4, 8192, 256, 8, 4), (32, 8, 2048, 256, 8, 8),
    (32, 1, 32768, 1024, 8, 2), (8, 1, 131072, 1024, 8, 1), (8, 8, 300, 100, 3, 2), (8, 12, 300, 100, 3, 3),
    (8, 8, 300, 100, 5, 4), (32, 1, 600, 100, 1, 1)])
def test_heads_per_unit(layers, seqs, length, budget, kv_heads, want):
    """152 CTAs, four score rows, layer-adaptive budgets; the first six are shapes that the rule was fitted to."""
    ckv_build.build()
    wl = cs.Workload(name="rule", num_layers=layers, num_q_heads=4 * kv_heads, num_kv_heads=kv_heads, window=32,
                     heads_per_group=1, budget_mean=budget, seqlens=(length,) * seqs, seed=1)
    b, r = np.sort(wl.budgets().astype(np.int32))[::-1].copy(), np.full(layers, 4, np.int32)
    got = ckv.load().ckv_internal_select_heads_per_unit(
        b.ctypes.data_as(ctypes.c_void_p), r.ctypes.data_as(ctypes.c_void_p), layers, seqs, seqs * length, kv_heads, 152)
    assert got == want


def _items(tiles, batches, ctas=152, lse=False):
    t, out = np.array(tiles, np.int32), np.zeros(len(tiles), np.int32)
    total = ckv.load().ckv_internal_plan_items(
        t.ctypes.data_as(ctypes.c_void_p), len(t), batches, ctas, int(lse), out.ctypes.data_as(ctypes.c_void_p))
    assert total == batches * out.sum()
    return out.tolist()


@pytest.mark.parametrize("lse", [False, True])
def test_long_launches_cut_each_sequence_by_its_own_length(lse):
    """32 layers of 8 KV heads: a sequence's items are the same alone and beside any other, 12 tiles from 160
    to 512 tiles and 14 otherwise, and never more than the CTAs."""
    ckv_build.build()
    tiles = [161, 64, 64, 1024, 512, 513, 159, 160, 1, 0]
    want = [14, 5, 5, 74, 43, 37, 12, 14, 1, 0]
    assert _items(tiles, 256, lse=lse) == want
    for t, m in zip(tiles, want):
        if t >= 64:
            assert _items([t], 256, lse=lse) == [m]
    assert _items([161, 20000], 128, ctas=8, lse=lse) == [1, 8]


@pytest.mark.parametrize("tiles,batches,want", [
    ([16], 8, [16]), ([64], 8, [16]), ([128], 8, [19]), ([256], 8, [19]), ([32, 32], 16, [4, 4]),  # 1 or 2 rounds
    ([64], 64, [16]), ([256], 32, [64]), ([256, 0, 3], 40, [64, 0, 1]),                            # 3 to 6
    ([256], 56, [22]), ([300, 100], 100, [25, 8])])                                               # more, or many units
def test_given_lse_items(tiles, batches, want):
    """Full rounds of short items in a launch of one or two rounds, four tiles up to six rounds."""
    ckv_build.build()
    assert _items(tiles, batches, lse=True) == want
