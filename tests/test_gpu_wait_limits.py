"""Bounded waits that run out, kernel by kernel: the call returns, the status word reports it, and the
same call with the default limit is clean and matches the oracle.  The limit is shortened with
ckv_set_wait_limit_us; no flag, barrier or check is removed, every wait still ends."""
import time

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


def _layers(wl, cfg, batch, lse=False):
    """Every layer's inputs and outputs for a multi-layer call; with the rows' lse of the oracle."""
    cu, w, ios = wl.cu_seqlens(), wl.window, []
    for l in range(wl.num_layers):
        li = wl.layer(l)
        idx, ck, ko, vo, _ = ckv.new_outputs(cfg, l, batch)
        _, n_sel = ckv.ckv_keep_lengths(cfg, l, batch)
        io = ckv.LayerIO(layer=l, q_win=gu.to_dev(li.q_win), k=gu.to_dev(li.k), v=gu.to_dev(li.v), idx=idx,
                         cu_keep_dev=ck, k_out=ko, v_out=vo,
                         scores=torch.zeros((n_sel, batch.total_tokens), dtype=torch.float32, device="cuda"))
        if lse:
            x = np.zeros((wl.num_q_heads, wl.num_seqs * w), np.float32)
            for s in range(wl.num_seqs):
                for h in np.nonzero(wl.head_mask()[l])[0]:
                    kv = li.k[int(cu[s]):int(cu[s + 1]), h // wl.group_size]
                    x[h, s * w:(s + 1) * w] = oracle.window_scores(li.q_win[s, :, h], kv)[1]
            io.lse = torch.from_numpy(x).cuda()
        ios.append((io, li))
    return ios


@pytest.mark.parametrize("heads", [1, 2], ids=["N32", "N64"])
def test_the_given_lse_kernel_of_many_layers_reports_its_waits(heads):
    """Its waits are all within a CTA; those for the first query rows and key tiles last 1.5 to 4 us, so
    a limit of 1 us runs out in every call, in the scoring kernel itself (details 33 to 35)."""
    wl = cs.Workload(name="limits_lse", num_layers=2, num_q_heads=8, num_kv_heads=2, seqlens=(40000, 900),
                     window=32, heads_per_group=heads, budget_mean=200, budget_uniform=True, seed=7)
    cfg, batch = ckv.Config.from_workload(wl), ckv.Batch(wl.cu_seqlens())
    layers = _layers(wl, cfg, batch, lse=True)
    ios = [io for io, _ in layers]
    ws = ckv.new_layers_workspace(cfg, ios, batch)
    ckv.ckv_set_wait_limit_us(1)
    try:
        for _ in range(5):
            ckv.ckv_score_windows_lse(cfg, ios, batch, ws)
            code, detail = ckv.ckv_read_device_status(ws)
            assert code == 2 and detail in (33, 34, 35), (code, detail)
    finally:
        ckv.ckv_set_wait_limit_us(0)
    ckv.ckv_score_windows_lse(cfg, ios, batch, ws)
    assert ckv.ckv_read_device_status(ws) == (0, 0)
    for l, (io, li) in enumerate(layers):
        o = gu.run_oracle(wl, l, li, want_kv=False)
        gu.assert_close_rows(io.scores.cpu().numpy(), o["scores"])


def test_a_wait_that_is_suspended_gives_up():
    """A limit above those that are polled (about 100 us): two CTAs share one unit of 782 key tiles, and
    pass 2 waits for pass 1's 391 of them."""
    wl = cs.Workload(name="limits_long", num_layers=1, num_q_heads=2, num_kv_heads=1, seqlens=(100000,),
                     window=32, heads_per_group=2, budget_mean=300, budget_uniform=True, seed=3)
    li = wl.layer(0)
    cfg = ckv.Config.from_workload(wl, max_ctas=2, score_path=ckv.SCORE_RELOAD)
    ckv.ckv_set_wait_limit_us(150)
    try:
        g = gu.run_gpu(wl, 0, li, cfg=cfg, scores=False, check_status=False)
    finally:
        ckv.ckv_set_wait_limit_us(0)
    assert g["status"][0] == 2, g["status"]
    g = gu.run_gpu(wl, 0, li, cfg=cfg)
    gu.check_layer(wl, 0, li, g, gu.run_oracle(wl, 0, li, want_kv=False))


def _fill(ios):
    for io in ios:
        io.idx.fill_(-7)


def _check_clean(wl, cfg, batch, layers):
    """The call with the default limit: status clean, positions and rows as the oracle's."""
    ios = [io for io, _ in layers]
    for io in ios:
        io.pooled_out = torch.zeros((cfg.num_vectors, batch.total_tokens), dtype=torch.float32, device="cuda")
    ws = ckv.new_layers_workspace(cfg, ios, batch)
    ckv.ckv_compress_layers_lse(cfg, ios, batch, ws)
    assert ckv.ckv_read_device_status(ws) == (0, 0)
    for l, (io, li) in enumerate(layers):
        g = dict(cfg=cfg, cu_keep=ckv.ckv_keep_lengths(cfg, l, batch)[0], pooled=io.pooled_out.cpu().numpy(),
                 idx=io.idx.cpu().numpy(), cu_keep_dev=io.cu_keep_dev.cpu().numpy(),
                 k_out=gu.to_host(io.k_out), v_out=gu.to_host(io.v_out))
        gu.check_layer(wl, l, li, g, gu.run_oracle(wl, l, li, want_kv=False))


def test_a_selection_that_gives_up_releases_its_row_copy_jobs():
    """Four score rows a selection are staged in one buffer, so that every chunk waits for its loads, longer
    than 1 us: the units of the long sequence give up.  Those of the short ones, kept whole, stage
    nothing; their CTAs go on to the long units' row-copy jobs and must not wait for them."""
    wl = cs.Workload(name="limits_stage", num_layers=1, num_q_heads=8, num_kv_heads=2, seqlens=(60000,) + (1000,) * 12,
                     window=16, heads_per_group=4, budget_mean=1100, budget_uniform=True, seed=41)
    cfg, batch = ckv.Config.from_workload(wl), ckv.Batch(wl.cu_seqlens())
    layers = _layers(wl, cfg, batch, lse=True)
    ios = [io for io, _ in layers]
    ws = ckv.new_layers_workspace(cfg, ios, batch)
    ckv.ckv_compress_layers_lse(cfg, ios, batch, ws)  # loads the kernels
    assert ckv.ckv_read_device_status(ws) == (0, 0)
    _fill(ios)
    ckv.ckv_set_wait_limit_us(1)
    try:
        t0 = time.perf_counter()
        ckv.ckv_compress_layers_lse(cfg, ios, batch, ws)
        assert ckv.ckv_read_device_status(ws)[0] == 2
        took = time.perf_counter() - t0
    finally:
        ckv.ckv_set_wait_limit_us(0)
    idx = ios[0].idx.cpu().numpy()
    assert np.all(idx[:, :1100] == -7) and np.all(idx[:, 1100:] >= 0)  # who gave up, and who did not
    assert took < 1.0, took  # a job that waits for a unit that gave up waits about 2 s
    _check_clean(wl, cfg, batch, layers)


def test_a_row_copy_job_whose_unit_takes_longer_than_the_limit_is_reported():
    """The units of the short sequences, kept whole, end within some 25 us; their CTAs go on to the jobs of
    the long sequence's units, which take about 100 us: a limit of 30 us runs out there (detail 251) and
    nowhere before, as the given-lse scoring's waits take a few microseconds."""
    wl = cs.Workload(name="limits_jobs", num_layers=1, num_q_heads=8, num_kv_heads=2, seqlens=(131072,) + (600,) * 12,
                     window=32, heads_per_group=2, budget_mean=1100, budget_uniform=True, seed=43)
    cfg, batch = ckv.Config.from_workload(wl), ckv.Batch(wl.cu_seqlens())
    layers = _layers(wl, cfg, batch, lse=True)
    ios = [io for io, _ in layers]
    ws = ckv.new_layers_workspace(cfg, ios, batch)
    ckv.ckv_set_wait_limit_us(30)
    try:
        ckv.ckv_compress_layers_lse(cfg, ios, batch, ws)
        assert ckv.ckv_read_device_status(ws) == (2, 251)
    finally:
        ckv.ckv_set_wait_limit_us(0)
    _check_clean(wl, cfg, batch, layers)
