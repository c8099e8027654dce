"""A tuned group capacity stands for the automatic one: calls with few cells keep their larger groups and calls with many small
cells their half warps (seen in the number of launches, as many as without tuning), also calls of other shapes than the tuned
one; an explicit capacity ends both."""
import numpy as np
import pytest
import torch

from paper_2407_19151_gb300 import workloads as W

from _parity import device_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["few", "half"])
def test_rules_stay_with_a_tuned_capacity(name):
    import paper_2407_19151_gb300 as mcc
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    wl = W.three_species(n_cells=100, mean_count=400.0, sigma=0.3, data_seed=5) if name == "few" else \
        W.three_species(n_cells=36 * sms, mean_count=40.0, data_seed=6)
    ctx, mc = mcc.context(0), int(wl.counts.sum(1).max())
    v, w, off = device_state(wl, "f32")

    def launches():
        p = mcc.Params(method=wl.method, dt=wl.dt, fE=wl.fE, seed=wl.seed, step=3)
        before = ctx.launch_count()
        x = [a.clone() for a in v]
        mcc.mcc_step_fused(*x, w, off, wl.n_cells, 3, list(zip(wl.q, wl.m)), wl.lnL, p, max_cell=mc)
        return ctx.launch_count() - before, x

    try:
        automatic, x0 = launches()
        caps0 = ctx.group_capacities()
        ctx.tune_group_capacity(224)
        assert ctx.group_capacities()[:3] == [224, 448, 896] != caps0[:3]
        tuned, x1 = launches()
        ctx.set_group_capacity(224)
        explicit, _ = launches()
        ctx.set_group_capacity(0)
        assert ctx.group_capacities() == caps0
    finally:
        ctx.set_group_capacity(0)
    mcc.sync_status(0)
    assert tuned == automatic != explicit
    if name == "half":  # every cell on a half warp either way
        assert all(torch.equal(a, b) for a, b in zip(x0, x1))


def test_autotuned_context_keeps_the_rules(tmp_path, monkeypatch):
    import paper_2407_19151_gb300 as mcc
    monkeypatch.setenv("MCC_AUTOTUNE_CACHE", str(tmp_path / "autotune.json"))
    wl = W.three_species(n_cells=3000, mean_count=300.0, data_seed=7).weight_ordered()
    small = W.three_species(n_cells=100, mean_count=400.0, sigma=0.3, data_seed=5)
    ctx, sp = mcc.context(0), list(zip(wl.q, wl.m))
    p = mcc.Params(method=wl.method, dt=wl.dt, fE=wl.fE, seed=wl.seed)

    def launches():
        v, w, off = device_state(small, "f32")
        before = ctx.launch_count()
        mcc.mcc_step_fused(*v, w, off, small.n_cells, 3, sp, small.lnL, p, max_cell=int(small.counts.sum(1).max()))
        return ctx.launch_count() - before

    try:
        want = launches()
        v, w, off = device_state(wl, "f32")
        mcc.autotune(*v, w, off, wl.n_cells, 3, sp, wl.lnL, p, int(wl.counts.sum(1).max()), persist=False)
        assert launches() == want
    finally:
        ctx.set_group_capacity(0)
        ctx.set_tile_cap(0)
    mcc.sync_status(0)
