"""The automatic choice of the one-layer scoring kernel: small calls take the TMEM-resident kernel, as
do all at N = 32, the others the two-pass kernel.  Around the limits of the rule (key tiles and units per CTA),
with both layouts of K, the scores agree with the two-pass kernel's and the layer with the oracle."""
import numpy as np
import pytest
import torch

import ckv_synth as cs
import oracle
import paper_2508_02401_gb300 as ckv
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

# 8 groups: two tiles for each of 152 CTAs are 38 per unit (4864 tokens), four 76; 76 units are 9 sequences
CASES = [((130,), 2), ((2048,), 2), ((4864,), 2), ((4865,), 2), ((500,) * 9, 2), ((400,) * 10, 2),
         ((4000, 33, 1, 3000), 2), ((1500,), 4), ((4864,), 1), ((4865,), 1), ((9728,), 1), ((9729,), 1)]


@pytest.mark.parametrize("interleaved", [False, True])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_small_calls_agree_with_the_two_pass_kernel(case, interleaved):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    ckv.load()
    oracle.build()
    lens, heads = CASES[case]
    wl = cs.Workload(name="auto", num_layers=1, num_q_heads=32, num_kv_heads=8, seqlens=lens, window=32,
                     heads_per_group=heads, budget_mean=100, budget_uniform=True, outlier_channels=8, seed=91)
    li = wl.layer(0)
    if not interleaved:
        gu.check_layer(wl, 0, li, gu.run_gpu(wl, 0, li), gu.run_oracle(wl, 0, li))
    batch = ckv.Batch(wl.cu_seqlens())
    q, k = gu.to_dev(li.q_win), gu.to_dev(li.k)
    strides = {}
    if interleaved:
        k = torch.stack([k, torch.zeros_like(k)], dim=1).contiguous()[:, 0]
        strides = dict(tok_stride=2 * 8 * 128, head_stride=128)
    got = []
    for path in (ckv.SCORE_AUTO, ckv.SCORE_RELOAD):
        cfg = ckv.Config.from_workload(wl, score_path=path)
        _, n_sel = ckv.ckv_keep_lengths(cfg, 0, batch)
        sc = gu.Guarded((n_sel, batch.total_tokens), torch.float32, float("nan"))
        ws = ckv.new_workspace(cfg, 0, batch)
        ckv.ckv_score_window(cfg, 0, batch, q, k, sc.view, ws, **strides)
        assert ckv.ckv_read_device_status(ws) == (0, 0)
        sc.check()
        got.append(sc.view.cpu().numpy().astype(np.float64))
    # each side is within 1e-3 of the oracle (fp32 logits of up to about 40 in base-2 units: 2e-5)
    gu.assert_close_rows(got[0], got[1], rtol=1e-4)


@pytest.mark.parametrize("static", [False, True], ids=["workspace", "static"])
def test_a_small_call_of_more_sequences_than_the_resident_kernel_takes(static):
    """65540 sequences, all but three of them empty: few key tiles, but more sequences than the resident
    kernel's tables hold, so the two-pass kernel takes the call (N = 64)."""
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    ckv.load()
    oracle.build()
    w, S, full = 33, 65540, {0: 700, 40000: 129, 65539: 1000}
    lens = np.zeros(S, np.int64)
    for s, n in full.items():
        lens[s] = n
    cu = np.concatenate([[0], np.cumsum(lens)])
    cfg = ckv.Config(num_layers=1, num_q_heads=1, num_kv_heads=1, window=w, pool_kernel=7, pool_type=ckv.POOL_MAX,
                     head_order=ckv.POOL_THEN_SUM, head_mask=np.ones((1, 1), np.uint8),
                     budgets=np.array([64], np.int32))
    batch = ckv.Batch(cu)
    gen = torch.Generator("cuda").manual_seed(5)
    q = torch.zeros((S, w, 1, 128), dtype=torch.bfloat16, device="cuda")
    for s in full:
        q[s] = torch.randn((w, 1, 128), device="cuda", generator=gen).bfloat16()
    k = torch.randn((int(cu[-1]), 1, 128), device="cuda", generator=gen).bfloat16()
    sc = gu.Guarded((1, batch.total_tokens), torch.float32, float("nan"))
    if static:
        status = torch.full((2,), -1, dtype=torch.int32, device="cuda")
        ckv.ckv_score_window_static(cfg, 0, batch, q, k, sc.view, status)
        assert status.tolist() == [0, 0]
    else:
        ws = ckv.new_workspace(cfg, 0, batch)
        ckv.ckv_score_window(cfg, 0, batch, q, k, sc.view, ws)
        assert ckv.ckv_read_device_status(ws) == (0, 0)
    sc.check()
    got = sc.view.cpu().numpy()
    for s in full:
        ref = oracle.window_scores(gu.to_host(q[s, :, 0]), gu.to_host(k[int(cu[s]):int(cu[s + 1]), 0]))[0]
        gu.assert_close_rows(got[:, cu[s]:cu[s + 1]], ref.reshape(1, -1))
