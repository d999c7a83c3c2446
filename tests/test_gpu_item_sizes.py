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
from tests import test_gpu_wait_limits as limits

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


# The given-lse kernel's items: such that one or two rounds are full, of four tiles in a launch of up to six
# rounds (of 14-tile items), of 12 or 14 tiles in one of more rounds or of more units than CTAs; a unit
# has at most as many items as CTAs.
# 8 units a layer on 8 CTAs: 84 tiles (10752 tokens) are six rounds, 85 are seven.
LSE_CASES = [((129,), 1, 0), ((16300,), 1, 0), ((20001, 900), 1, 0), ((2433,), 2, 0), ((10752,), 1, 8), ((10753,), 1, 8), ((20480,), 1, 8), ((65537,), 1, 8),
             ((8192, 100), 2, 0), ((900, 1, 3000), 1, 37), ((300,) * 20, 1, 0), ((2000,), 1, 1)]


@pytest.mark.parametrize("case", range(len(LSE_CASES)))
def test_given_lse_item_lengths(case):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    oracle.build()
    lens, n, max_ctas = LSE_CASES[case]
    kv_heads = 1 if max_ctas == 1 else 8
    wl = cs.Workload(name="items_lse", num_layers=n, num_q_heads=2 * kv_heads, num_kv_heads=kv_heads, seqlens=lens,
                     window=32, heads_per_group=2, budget_mean=64, pool_kernel=7, seed=34)
    cfg, batch = ckv.Config.from_workload(wl, max_ctas=max_ctas), ckv.Batch(wl.cu_seqlens())
    ios = limits._layers(wl, cfg, batch, lse=True)
    out = []
    for io, _ in ios:
        out.append(gu.Guarded(tuple(io.scores.shape), torch.float32, float("nan")))
        io.scores = out[-1].view
    ws = ckv.new_layers_workspace(cfg, [io for io, _ in ios], batch)
    ckv.ckv_score_windows_lse(cfg, [io for io, _ in ios], batch, ws)
    assert ckv.ckv_read_device_status(ws) == (0, 0)
    for l, (g, (_, li)) in enumerate(zip(out, ios)):
        g.check()
        o = gu.run_oracle(wl, l, li, want_kv=False)
        gu.assert_close_rows(g.view.cpu().numpy(), o["scores"])
