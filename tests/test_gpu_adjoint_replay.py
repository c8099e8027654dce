"""The adjoint's forward repeats the FP64 step bit for bit, also where a correction takes more pairs than the step kernel's first
warp or its first chunk of 128, and several passes: the prefix sums over the pairs' caps associate as the step kernel's."""
import pytest
import torch

from paper_2407_19151_gb300 import workloads as W

from _parity import device_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fE", [0.05, 0.01, 0.004, 0.0015])
@pytest.mark.parametrize("mean", [60.0, 1300.0])
@pytest.mark.parametrize("order", ["any", "weight"])
def test_adjoint_forward_repeats_the_step(fE, mean, order):
    import paper_2407_19151_gb300 as mcc
    from paper_2407_19151_gb300 import _binding as B
    wl = W.three_species(n_cells=30, mean_count=mean, precision="f64", data_seed=8)
    if order == "weight":
        wl = wl.weight_ordered()
    p = mcc.Params(method=wl.method, dt=wl.dt, fE=fE, seed=wl.seed, step=3)
    sp, mc = list(zip(wl.q, wl.m)), int(wl.counts.sum(1).max())
    v, w, off = device_state(wl, "f64")
    x = [a.clone() for a in v]
    for k, (a, b) in enumerate(mcc.default_interactions(3)):
        out = [torch.empty_like(y) for y in x]
        B.mcc_adjoint(*x, w, off, wl.n_cells, 3, sp, wl.lnL, a, b, k, p, mc, out=out)
        x = out
    corr, _ = mcc.mcc_step_fused(*v, w, off, wl.n_cells, 3, sp, wl.lnL, p)
    mcc.sync_status(0)
    if fE < 0.005 and mean > 1000:
        assert corr.max() > 300  # well beyond a chunk in some species
    for a, b in zip(x, v):
        assert torch.equal(a, b)
