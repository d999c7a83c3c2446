"""The multi-layer selection with one selection per layer: the KV heads are split over units of 1, 2, 4
or all heads by the number of units per CTA, which max_ctas varies here, with KV-head counts that the
units do and do not divide, and budgets with and without row-copy jobs.  Positions and rows against
the oracle, every output between canaries."""
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
