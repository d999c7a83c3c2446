"""The multi-layer selection's row-copy jobs: the rows that a unit keeps beyond the first 1024 are
copied by whichever CTA is free, in jobs of a fixed number of rows.  Budgets at the first job's edges
and in its middle, sequences kept whole and just above the limit, budgets that differ by layer, one
selection per layer, and more long sequences than the job table takes (no jobs).  Positions and rows
against the oracle, every output between canaries."""
import pytest
import torch

import ckv_synth as cs
import oracle
import paper_2508_02401_gb300 as ckv
from tests import gpu_util as gu
from tests import test_gpu_layers as layers

pytestmark = pytest.mark.gpu

SEQS = (3000, 1024, 700, 5000, 1025)
CASES = [dict(budget_mean=b, budget_uniform=True, seqlens=SEQS) for b in (1024, 1025, 1536, 1537, 2900, 4990)] + [
    dict(budget_mean=1400, num_layers=5, seqlens=(9000, 2000)),
    dict(budget_mean=2100, budget_uniform=True, scope="layer", heads_per_layer=3, num_q_heads=16, num_kv_heads=4,
         seqlens=(3000, 40, 2500)),
    dict(budget_mean=1029, budget_uniform=True, num_kv_heads=1, num_q_heads=2, heads_per_group=1,
         seqlens=tuple(1030 + (i % 3) for i in range(66))),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_rows_beyond_the_first_are_copied(case):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    oracle.build()
    kw = dict(name="jobs", num_layers=2, num_q_heads=8, num_kv_heads=2, window=32, heads_per_group=2,
              pool_kernel=7, seed=77)
    kw.update(CASES[case])
    wl = cs.Workload(**kw)
    cfg = ckv.Config.from_workload(wl)
    lis = [wl.layer(l) for l in range(wl.num_layers)]
    res = layers._run_layers(wl, cfg, lis, with_scores=False)
    for l, li in enumerate(lis):
        gu.check_layer(wl, l, li, res[l], gu.run_oracle(wl, l, li, want_kv=False))
