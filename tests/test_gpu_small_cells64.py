"""FP64 steps around the line where small cells run on six CTAs per SM (cells of at most 320 particles, more than four per SM):
whole steps against the oracle within the FP64 bound for every particle."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2407_19151_gb300 import workloads as W

from _parity import F64_TOL, device_state, gpu_velocities, oracle_state, velocity_error

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case", ["few", "many", "line", "beam"])
def test_small_cells(case):
    import paper_2407_19151_gb300 as mcc
    n = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    if case == "few":
        wl = W.equilibration(n_cells=n, mean_count=6.0, data_seed=3, method=W.N97, precision="f64")
    elif case == "many":
        wl = W.equilibration(n_cells=n + 1, mean_count=6.0, data_seed=4, method=W.TA77, precision="f64")
    elif case == "line":
        wl = W.equilibration(n_cells=n + 1, mean_count=128.0, data_seed=5, method=W.N97, precision="f64")
    else:
        wl = W.relativistic_beam(n_cells=n + 1, count_hi=300, data_seed=6, precision="f64")
    v, w, off = device_state(wl, "f64")
    par = dict(method=wl.method, relativistic=case == "beam", dt=wl.dt, c=wl.c, fE=wl.fE, seed=wl.seed, step=2)
    corr, fail = mcc.mcc_step_fused(*v, w, off, wl.n_cells, wl.n_species, list(zip(wl.q, wl.m)), wl.lnL, mcc.Params(**par))
    mcc.sync_status(0)
    st = oracle_state(wl, "f64")
    ocorr, ofail = O.step(st, wl.q, wl.m, wl.lnL, O.Params(**par), n_steps=1)
    np.testing.assert_array_equal(fail.cpu().numpy(), ofail)
    np.testing.assert_array_equal(corr.cpu().numpy(), ocorr)
    assert velocity_error(gpu_velocities(v), st.v(), wl.offsets).max() < F64_TOL
