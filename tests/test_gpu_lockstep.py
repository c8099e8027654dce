"""Groups of a CTA in lockstep (mixed path): batches that are not full, cells of several size classes side by side, and cells
whose corrections fail, which are visited again without the failed interaction. Bounds: those of the mixed path at these
cell sizes (2e-6 for 99.9% of particles, 1e-5 for all); failures counted exactly."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2407_19151_gb300 import workloads as W

from _parity import F32_TOL, device_state, gpu_velocities, oracle_state, velocity_error

pytestmark = pytest.mark.gpu


def _both(wl, rel=False, **kw):
    import paper_2407_19151_gb300 as mcc
    v, w, off = device_state(wl, "f32")
    par = dict(method=wl.method, relativistic=rel, dt=wl.dt, c=wl.c, seed=wl.seed, step=3, **kw)
    corr, fail = mcc.mcc_step_fused(*v, w, off, wl.n_cells, wl.n_species, list(zip(wl.q, wl.m)), wl.lnL,
                                    mcc.Params(**par))
    mcc.sync_status(0)
    st = oracle_state(wl, "f32")
    ocorr, ofail = O.step(st, wl.q, wl.m, wl.lnL, O.Params(**par), n_steps=1)
    err = velocity_error(gpu_velocities(v), st.v(), wl.offsets)
    return err, corr.cpu().numpy(), fail.cpu().numpy(), ocorr, ofail


@pytest.mark.parametrize("n_cells", [1, 7, 8, 9, 17, 160])
@pytest.mark.parametrize("passes,fE", [(8, 0.05), (1, 0.004)])
def test_batches_and_retries(n_cells, passes, fE):
    wl = W.three_species(n_cells=n_cells, mean_count=350.0, data_seed=77 + n_cells).weight_ordered()
    err, corr, fail, ocorr, ofail = _both(wl, fE=fE, max_corr_passes=passes)
    if passes == 1 and n_cells >= 17:
        assert ofail.sum() > n_cells  # every batch holds cells to visit again
    np.testing.assert_array_equal(fail, ofail)
    assert np.abs(corr - ocorr).max() <= 2  # a crossing pair may be its neighbour's neighbour; a recount would be tens
    assert np.quantile(err, 0.999) < F32_TOL and err.max() < 1e-5


@pytest.mark.parametrize("n_cells", [5, 33])
def test_relativistic_batches(n_cells):
    wl = W.relativistic_beam(n_cells=n_cells, data_seed=11 + n_cells, count_hi=700)
    err, corr, fail, ocorr, ofail = _both(wl, rel=True, fE=wl.fE)
    np.testing.assert_array_equal(fail, ofail)
    assert np.quantile(err, 0.999) < F32_TOL


@pytest.mark.parametrize("n_cells", [3, 304, 305, 608, 609, 1216, 1217])
def test_few_cells_on_larger_groups(n_cells):
    # around the cell counts where the group size changes on 152 SMs (some cells are empty): the same cells on the size
    # classes themselves, which an explicit capacity selects, give the same step up to the order of float-float sums
    # (2^-44), so stored velocities within two float ulps of their population's speed, and the same counts
    import paper_2407_19151_gb300 as mcc
    wl = W.equilibration(n_cells=n_cells, mean_count=12.0, data_seed=n_cells, method=W.N97, precision="f32")
    ctx = mcc.context(0)
    runs = []
    for per_warp in (0, 280):
        ctx.set_group_capacity(per_warp)
        try:
            v, w, off = device_state(wl, "f32")
            res = torch.full((2 * n_cells,), -1.0, dtype=torch.float64, device="cuda")
            p = mcc.Params(method=wl.method, dt=wl.dt, fE=wl.fE, seed=wl.seed, step=3, residual=res)
            corr, fail = mcc.mcc_step_fused(*v, w, off, wl.n_cells, wl.n_species, list(zip(wl.q, wl.m)), wl.lnL, p)
            mcc.sync_status(0)
        finally:
            ctx.set_group_capacity(0)
        assert (res >= 0).all()  # every cell visited
        runs.append((gpu_velocities(v), corr.cpu().numpy(), fail.cpu().numpy()))
    np.testing.assert_array_equal(runs[0][1], runs[1][1])
    np.testing.assert_array_equal(runs[0][2], runs[1][2])
    assert velocity_error(runs[0][0], runs[1][0], wl.offsets).max() <= 2.0 ** -22
