"""Bounded waits that run out, kernel by kernel: the call returns, the status word reports it, and the
same call with the default limit is clean and matches the oracle.  The limit is shortened with
ckv_set_wait_limit_us; no flag, barrier or check is removed, every wait still ends."""
import numpy as np
import pytest
import torch

import ckv_synth as cs
import oracle
import paper_2508_02401_gb300 as ckv
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    ckv.load()
    oracle.build()


@pytest.mark.parametrize("heads", [1, 2], ids=["N32", "N64"])
@pytest.mark.parametrize("max_ctas,path", [(4, ckv.SCORE_RELOAD), (0, ckv.SCORE_RELOAD), (0, ckv.SCORE_RESIDENT)],
                         ids=["reload4", "reload", "resident"])
def test_the_two_pass_kernels_give_up_and_return(max_ctas, path, heads):
    """The waits for the other CTAs of a sequence outlast 1 us on either kernel, at either width."""
    wl = cs.Workload(name="limits", num_layers=1, num_q_heads=32, num_kv_heads=8, seqlens=(30000, 5000),
                     window=32, heads_per_group=heads, budget_mean=300, budget_uniform=True, seed=15)
    li = wl.layer(0)
    cfg = ckv.Config.from_workload(wl, max_ctas=max_ctas, score_path=path)
    ckv.ckv_set_wait_limit_us(1)
    try:
        for _ in range(3):
            g = gu.run_gpu(wl, 0, li, cfg=cfg, scores=False, check_status=False)
            assert g["status"][0] == 2, g["status"]
    finally:
        ckv.ckv_set_wait_limit_us(0)
    g = gu.run_gpu(wl, 0, li, cfg=cfg)
    g.pop("scores")
    gu.check_layer(wl, 0, li, g, gu.run_oracle(wl, 0, li, groups=(0, 7), want_kv=False), groups=(0, 7))
