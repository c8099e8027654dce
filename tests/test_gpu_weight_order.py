"""Weight orders where a counting sort on linear buckets can go wrong: equal weights, ties, clusters that fill one bucket,
neighbours within the keys' tie width, for every size class; and the cell sort's two orders on such keys."""
import numpy as np
import pytest

import oracle as O
from paper_2407_19151_gb300 import workloads as W

from _parity import F32_TOL, device_state, gpu_velocities, oracle_state, velocity_error

pytestmark = pytest.mark.gpu


def _weights(kind, n, rng):
    if kind == "decades":
        return 10.0 ** rng.uniform(0, 4, n)
    if kind == "equal":
        return np.full(n, 3.0)
    if kind == "ties":
        return rng.integers(1, 5, n).astype(float)
    if kind == "clusters":  # nearly all in one bucket
        return np.where(rng.random(n) < 0.9, 1.0 + 1e-6 * rng.random(n), 10.0 ** rng.uniform(0, 3, n))
    return 1.0 + 2.0 ** -33 * rng.integers(0, 4, n)  # "within": most neighbours tie to 2^-32


KINDS = ["decades", "equal", "ties", "clusters", "within"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("mean", [30, 500, 1000, 2000])
def test_step_order(kind, mean):
    import paper_2407_19151_gb300 as mcc
    # more cells than the GPU's warps, so that they run on the size classes: the tail of the cells is small
    wl = W.three_species(n_cells=40, mean_count=float(mean), data_seed=mean)
    wl.w[:] = _weights(kind, wl.n, np.random.default_rng(mean))
    ctx = mcc.context(0)
    v, w, off = device_state(wl, "f32")
    par = dict(method=wl.method, dt=wl.dt * (wl.w.max() * 1e-4) ** -1, fE=wl.fE, seed=wl.seed, step=5)
    ctx.set_group_capacity(300)  # the size classes, also for few cells
    try:
        corr, fail = mcc.mcc_step_fused(*v, w, off, wl.n_cells, wl.n_species, list(zip(wl.q, wl.m)), wl.lnL,
                                        mcc.Params(**par))
        mcc.sync_status(0)
    finally:
        ctx.set_group_capacity(0)
    st = oracle_state(wl, "f32")
    ocorr, ofail = O.step(st, wl.q, wl.m, wl.lnL, O.Params(**par), n_steps=1)
    np.testing.assert_array_equal(fail.cpu().numpy(), ofail)
    # a wrong order pairs other particles: their velocities then differ by far more than the mixed path's bound
    err = velocity_error(gpu_velocities(v), st.v(), wl.offsets)
    assert np.quantile(err, 0.99) < F32_TOL


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n,C,S", [(7, 2, 2), (3001, 40, 3), (40_000, 90, 1), (50_000, 31, 3), (120_000, 700, 3)])
@pytest.mark.parametrize("layout", ["shuffled", "binned", "pushed"])
def test_cell_sort(kind, n, C, S, layout):
    import torch
    import paper_2407_19151_gb300 as mcc
    rng = np.random.default_rng(n + len(kind))
    cell = rng.integers(0, C, n).astype(np.int32)
    sp = rng.integers(0, S, n).astype(np.int32)
    if layout != "shuffled":
        by = np.argsort(cell.astype(np.int64) * S + sp, kind="stable")
        cell, sp = cell[by].copy(), sp[by].copy()
    if layout == "pushed":  # a sixth moved to a neighbouring cell
        move = rng.random(n) < 1 / 6
        cell[move] = (cell[move] + rng.choice([-1, 1], int(move.sum()))) % C
    w = _weights(kind, n, rng)
    dev = [torch.from_numpy(a).cuda() for a in (cell, sp, w)]
    for perm, off, ref in ((*mcc.mcc_bin(dev[0], dev[1], C, S), O.bin_particles(cell, sp, C, S)),
                           (*mcc.mcc_bin_weighted(*dev, C, S), O.bin_particles_weighted(cell, sp, w, C, S)),
                           (*mcc.mcc_bin_static(dev[0], dev[1], C, S), O.bin_particles(cell, sp, C, S))):
        np.testing.assert_array_equal(perm.cpu().numpy(), ref[0])
        np.testing.assert_array_equal(off.cpu().numpy(), ref[1])
    mcc.sync_status(0)
