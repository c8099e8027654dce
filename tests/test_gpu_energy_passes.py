"""Energy correction over several passes on the one-CTA kernel: pass p + 1 pairs across the pairs of pass p, so it must see all
of their velocities. A small fE needs many passes; the step equals the oracle (FP64 bound) and repeats bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_2407_19151_gb300 import workloads as W

from _parity import F64_TOL, device_state, gpu_velocities, oracle_state, velocity_error

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mean,fE", [(60, 0.004), (512, 0.01), (1500, 0.02)])
def test_several_passes(mean, fE):
    import paper_2407_19151_gb300 as mcc
    wl = W.three_species(n_cells=96, mean_count=float(mean), precision="f64", data_seed=5)
    par = dict(method=wl.method, dt=wl.dt, fE=fE, seed=wl.seed, step=2)
    runs = []
    for _ in range(2):
        v, w, off = device_state(wl, "f64")
        corr, fail = mcc.mcc_step_fused(*v, w, off, wl.n_cells, wl.n_species, list(zip(wl.q, wl.m)), wl.lnL,
                                        mcc.Params(**par))
        mcc.sync_status(0)
        runs.append((gpu_velocities(v), corr.cpu().numpy(), fail.cpu().numpy()))
    st = oracle_state(wl, "f64")
    ocorr, ofail = O.step(st, wl.q, wl.m, wl.lnL, O.Params(**par), n_steps=1)
    for got, corr, fail in runs:
        np.testing.assert_array_equal(fail, ofail)
        np.testing.assert_array_equal(corr, ocorr)
        assert np.quantile(velocity_error(got, st.v(), wl.offsets), 0.999) < F64_TOL
    np.testing.assert_array_equal(runs[0][0], runs[1][0])
