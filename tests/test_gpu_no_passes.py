"""max_corr_passes = 0: no energy pair is allowed, so every interaction with an energy violation fails. The FP64 step, the mixed
step, the adjoint's forward and the oracle agree on it, under each fail policy that continues."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2407_19151_gb300 import workloads as W

from _parity import F32_TOL, F64_TOL, device_state, gpu_velocities, oracle_state, velocity_error

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("policy", [0, 1])
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_no_passes(policy, prec):
    import paper_2407_19151_gb300 as mcc
    wl = W.three_species(n_cells=40, mean_count=90.0, precision=prec)
    kw = dict(method=wl.method, dt=wl.dt, fE=wl.fE, seed=wl.seed, step=3, max_corr_passes=0, fail_policy=policy)
    v, w, off = device_state(wl, prec)
    corr, fail = mcc.mcc_step_fused(*v, w, off, wl.n_cells, 3, list(zip(wl.q, wl.m)), wl.lnL, mcc.Params(**kw))
    mcc.sync_status(0)
    st = oracle_state(wl, prec)
    ocorr, ofail = O.step(st, wl.q, wl.m, wl.lnL, O.Params(**kw), n_steps=1)
    assert ofail.sum() > wl.n_cells
    np.testing.assert_array_equal(fail.cpu().numpy(), ofail)
    np.testing.assert_array_equal(corr.cpu().numpy(), ocorr)
    assert velocity_error(gpu_velocities(v), st.v(), wl.offsets).max() < (F64_TOL if prec == "f64" else F32_TOL)


def test_no_passes_adjoint_forward():
    import paper_2407_19151_gb300 as mcc
    from paper_2407_19151_gb300 import _binding as B
    wl = W.three_species(n_cells=20, mean_count=90.0, precision="f64")
    p = mcc.Params(method=wl.method, dt=wl.dt, fE=wl.fE, seed=wl.seed, step=3, max_corr_passes=0)
    sp, mc = list(zip(wl.q, wl.m)), int(wl.counts.sum(1).max())
    v, w, off = device_state(wl, "f64")
    x = [a.clone() for a in v]
    for k, (a, b) in enumerate(mcc.default_interactions(3)):
        out = [torch.empty_like(y) for y in x]
        B.mcc_adjoint(*x, w, off, wl.n_cells, 3, sp, wl.lnL, a, b, k, p, mc, out=out)
        x = out
    mcc.mcc_step_fused(*v, w, off, wl.n_cells, 3, sp, wl.lnL, p)
    mcc.sync_status(0)
    for a, b in zip(x, v):
        assert (a - b).abs().max() <= F64_TOL * b.abs().max()
