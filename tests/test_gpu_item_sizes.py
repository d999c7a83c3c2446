"""The two-pass kernel's work items: their length follows the launch (one full round, several rounds, more
units than CTAs, long units), for one layer and several, at capped grids and ragged lengths.  Scores
and selections against the oracle, every output between canaries."""
import pytest
import torch

import ckv_synth as cs
import oracle
import paper_2508_02401_gb300 as ckv
from tests import gpu_util as gu
from tests import test_gpu_layers as layers

pytestmark = pytest.mark.gpu

# 8 units a layer and sequence: 19 items a unit fill 152 CTAs
CASES = [((129,), 1), ((2432,), 1), ((2433,), 1), ((8192,), 2), ((17024,), 1), ((17025,), 1), ((20480, 100), 1),
         ((3000, 1, 700, 2000), 2), ((300,) * 20, 1)]


@pytest.mark.parametrize("max_ctas", [0, 37, 2])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_item_lengths(case, max_ctas):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    oracle.build()
    lens, n = CASES[case]
    wl = cs.Workload(name="items", num_layers=n, num_q_heads=32, num_kv_heads=8, seqlens=lens, window=32,
                     heads_per_group=2, budget_mean=64, pool_kernel=7, seed=33)
    cfg = ckv.Config.from_workload(wl, max_ctas=max_ctas)
    lis = [wl.layer(l) for l in range(n)]
    res = layers._run_layers(wl, cfg, lis, with_scores=True)
    for l, li in enumerate(lis):
        gu.check_layer(wl, l, li, res[l], gu.run_oracle(wl, l, li, want_kv=False))
