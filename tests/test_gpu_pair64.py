"""FP64 pair kinematics (tabulated N97 root, logarithm and azimuth) over the whole range of scattering lengths, from far below
the short-length series to isotropic: one scatter against the oracle within the FP64 bound for every particle."""
import numpy as np
import pytest

import oracle as O
from paper_2407_19151_gb300 import workloads as W

from _parity import F64_TOL, device_state, gpu_velocities, oracle_state, velocity_error

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", [W.TA77, W.N97])
@pytest.mark.parametrize("dt_scale", [1e-9, 1e-3, 0.3, 4.0, 60.0, 1e9])
@pytest.mark.parametrize("rel", [False, True])
def test_scatter_over_lengths(method, dt_scale, rel):
    import paper_2407_19151_gb300 as mcc
    if rel:
        wl = W.relativistic_beam(n_cells=60, count_hi=300, precision="f64")
    else:
        wl = W.three_species(n_cells=60, mean_count=90, precision="f64")
    v, w, off = device_state(wl, "f64")
    par = dict(method=method, relativistic=rel, dt=wl.dt * dt_scale, c=wl.c, seed=wl.seed, step=9, correct=False)
    mcc.mcc_step_fused(*v, w, off, wl.n_cells, wl.n_species, list(zip(wl.q, wl.m)), wl.lnL, mcc.Params(**par))
    mcc.sync_status(0)
    st = oracle_state(wl, "f64")
    O.step(st, wl.q, wl.m, wl.lnL, O.Params(**par), n_steps=1)
    err = velocity_error(gpu_velocities(v), st.v(), wl.offsets)
    assert np.isfinite(err).all() and err.max() < F64_TOL
