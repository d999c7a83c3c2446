"""The multi-layer selection with one selection per layer, whose units serve 1, 2, 4 or all KV heads:
KV-head counts that the heads of a unit do and do not divide, budgets with and without row-copy jobs,
scoring grids of 1 to all CTAs.  The first test's calls have fewer units than the GPU has SMs, so that a
unit serves one head; those of the second have more, and the rule's choice is asserted.  Positions and
rows against the oracle, every output between canaries."""
import ctypes

import numpy as np
import pytest
import torch

import ckv_synth as cs
import oracle
import paper_2508_02401_gb300 as ckv
from tests import gpu_util as gu
from tests import test_gpu_layers as layers

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("max_ctas", [1, 3, 7, 12, 0])
@pytest.mark.parametrize("kv_heads,budget", [(8, 64), (3, 100), (8, 1600), (3, 1600), (2, 3000)])
def test_heads_split_over_units(kv_heads, budget, max_ctas):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    oracle.build()
    wl = cs.Workload(name="heads", num_layers=3, num_q_heads=4 * kv_heads, num_kv_heads=kv_heads, window=16, heads_per_group=2,
                     scope="layer", heads_per_layer=3, pool_kernel=5, pool_type="avg", seed=91,
                     budget_mean=budget, seqlens=(3000, 40, 2500))
    cfg = ckv.Config.from_workload(wl, max_ctas=max_ctas)
    lis = [wl.layer(l) for l in range(wl.num_layers)]
    res = layers._run_layers(wl, cfg, lis, with_scores=False)
    for l, li in enumerate(lis):
        gu.check_layer(wl, l, li, res[l], gu.run_oracle(wl, l, li, want_kv=False))


def _rule(wl, heads, ctas):
    """The library's choice of KV heads per unit for the workload's layers, at most 32 of them."""
    b = np.sort(wl.budgets().astype(np.int32))[::-1].copy()
    r = np.full(len(b), heads, np.int32)
    return ckv.load().ckv_internal_select_heads_per_unit(
        b.ctypes.data_as(ctypes.c_void_p), r.ctypes.data_as(ctypes.c_void_p), len(b), wl.num_seqs,
        int(wl.cu_seqlens()[-1]), wl.num_kv_heads, ctas)


def _ragged(n, longest):
    return tuple(longest - 17 * i for i in range(n))


# layers, KV heads, lengths, budget, KV heads per unit on 152 SMs
SPLIT = [(8, 8, _ragged(4, 330), 100, 2), (8, 8, _ragged(6, 330), 100, 4), (8, 8, _ragged(12, 430), 100, 8),
         (8, 3, _ragged(8, 330), 100, 2), (8, 3, _ragged(12, 430), 100, 3), (8, 5, _ragged(8, 330), 100, 4),
         (24, 8, (1700,), 1600, 2), (8, 8, _ragged(6, 1750), 1600, 4), (8, 3, _ragged(8, 1750), 1600, 2),
         (8, 3, _ragged(12, 1800), 1600, 3), (8, 5, _ragged(8, 1750), 1600, 4), (33, 3, _ragged(4, 1750), 1400, 3)]


@pytest.mark.parametrize("case", range(len(SPLIT)))
def test_units_that_serve_several_heads(case):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    oracle.build()
    n, kv_heads, lens, budget, heads = SPLIT[case]
    wl = cs.Workload(name="split", num_layers=n, num_q_heads=2 * kv_heads, num_kv_heads=kv_heads, window=16,
                     heads_per_group=1, scope="layer", heads_per_layer=3, pool_kernel=5, pool_type="avg", seed=92,
                     budget_mean=budget, budget_uniform=True, seqlens=lens)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert _rule(wl.with_(num_layers=min(n, 32)), 3, sms) == heads
    cfg = ckv.Config.from_workload(wl)
    lis = [wl.layer(l) for l in range(n)]
    res = layers._run_layers(wl, cfg, lis, with_scores=False)
    for l, li in enumerate(lis):
        gu.check_layer(wl, l, li, res[l], gu.run_oracle(wl, l, li, want_kv=False))
