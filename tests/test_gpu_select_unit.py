"""The one-block selection at the edges of its positions per thread (2, 4, 8 and 16 positions for up
to 2048, 4096, 8192 and 16384 tokens), alone and with shorter sequences, with either scope, through
ckv_compress_layer against the oracle."""
import pytest
import torch

import ckv_synth as cs
import oracle
import paper_2508_02401_gb300 as ckv
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scope", ["kv_head", "layer"])
@pytest.mark.parametrize("longest", [130, 2047, 2048, 2049, 4096, 4097, 8192, 8193, 16384])
def test_one_block_selection(longest, scope):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    ckv.load()
    oracle.build()
    heads = dict(heads_per_group=2) if scope == "kv_head" else dict(heads_per_group=1, heads_per_layer=3)
    wl = cs.Workload(name="unit", num_layers=1, num_q_heads=8, num_kv_heads=2, seqlens=(longest, 70, 129),
                     window=32, budget_mean=100, budget_uniform=True, scope=scope, seed=31, **heads)
    li = wl.layer(0)
    gu.check_layer(wl, 0, li, gu.run_gpu(wl, 0, li), gu.run_oracle(wl, 0, li))
