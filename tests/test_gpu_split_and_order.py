"""The unfused calls around the tile that four CTAs per SM share (cells above it go in a second launch), and the cell order
built by several CTAs (calls with many cells)."""
import numpy as np
import pytest

import oracle as O
from paper_2407_19151_gb300 import workloads as W

from _parity import F64_TOL, device_state, gpu_velocities, oracle_state, velocity_error

pytestmark = pytest.mark.gpu


def _with_counts(wl, counts):
    """The workload's first species populations cut to the given (cells, species) counts."""
    counts = np.asarray(counts, dtype=np.int64)
    big = W.three_species(n_cells=len(counts), mean_count=12000.0, sigma=0.01, precision=wl.precision, data_seed=3)
    keep = np.concatenate([big.offsets[k] + np.arange(c) for k, c in enumerate(counts.reshape(-1))])
    return W.Workload("cut", len(counts), big.q, big.m, big.lnL, counts, big.vx[keep], big.vy[keep], big.vz[keep],
                      big.w[keep], big.dt, big.method, precision=wl.precision, seed=big.seed)


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_unfused_calls_over_cell_sizes(prec):
    import torch
    import paper_2407_19151_gb300 as mcc
    # cells of 0, 1 and 2 particles, sizes through the small tile (about 640 FP64, 950 float) and up to three times it
    tot = [0, 1, 2, 5, 300] + list(range(600, 720, 7)) + list(range(900, 1000, 11)) + [1500, 2400, 3000]
    wl = _with_counts(W.three_species(n_cells=1, precision=prec),
                      [[t // 3 + (t % 3 > 0), t // 3 + (t % 3 > 1), t // 3] for t in tot])
    v, w, off = device_state(wl, prec)
    sp = list(zip(wl.q, wl.m))
    kw = dict(method=wl.method, dt=wl.dt, fE=wl.fE, seed=wl.seed, step=4)
    p = mcc.Params(**kw)
    total = np.zeros(wl.n_cells, dtype=np.int64)
    for k, (a, b) in enumerate(mcc.default_interactions(3)):
        pairs = mcc.mcc_pair(off, wl.n_cells, 3, a, b, k, p.seed, p.step)
        backup = mcc.mcc_scatter(*v, w, off, wl.n_cells, 3, sp, wl.lnL, a, b, k, pairs, p)
        corr, fail = mcc.mcc_correct(*v, w, off, wl.n_cells, 3, sp, a, b, k, p, backup)
        total += fail.cpu().numpy()
    mcc.sync_status(0)
    st = oracle_state(wl, prec)
    _, ofail = O.step(st, wl.q, wl.m, wl.lnL, O.Params(**kw), n_steps=1)
    err = velocity_error(gpu_velocities(v), st.v(), wl.offsets)
    np.testing.assert_array_equal(total, ofail)
    if prec == "f64":
        assert err.max() < F64_TOL
    else:  # float velocities between the calls: the stated bounds of the one-CTA float kernel
        assert np.quantile(err, 0.99) < 2e-6 and err.max() < 2e-4


@pytest.mark.parametrize("n_cells", [16384, 16385, 50_001])
def test_order_of_many_cells(n_cells):
    import dataclasses
    import paper_2407_19151_gb300 as mcc
    # one call equals two calls on its halves (cells are independent): every cell visited once, whatever its place
    wl = W.three_species(n_cells=n_cells, mean_count=9.0, sigma=1.2, data_seed=1)
    sp = list(zip(wl.q, wl.m))
    p = mcc.Params(method=wl.method, dt=wl.dt, fE=wl.fE, seed=wl.seed, step=2)
    mc = int(wl.counts.sum(1).max())
    ctx = mcc.context(0)
    ctx.set_group_capacity(300)
    try:
        v, w, off = device_state(wl, "f32")
        corr, fail = mcc.mcc_step_fused(*v, w, off, n_cells, 3, sp, wl.lnL, p, max_cell=mc)
        u, _, _ = device_state(wl, "f32")
        h = n_cells // 2
        cut = int(wl.offsets[3 * h])
        got = []
        for lo, hi, c0, c1 in ((0, cut, 0, h), (cut, wl.n, h, n_cells)):
            o = off[3 * c0:3 * c1 + 1] - off[3 * c0]
            got.append(mcc.mcc_step_fused(*(x[lo:hi] for x in u), w[lo:hi], o, c1 - c0, 3, sp, wl.lnL,
                                          dataclasses.replace(p, cell_base=c0), max_cell=mc))
        mcc.sync_status(0)
    finally:
        ctx.set_group_capacity(0)
    for x, y in zip(v, u):
        assert (x == y).all()
    assert (corr.cpu().numpy() == np.concatenate([g[0].cpu().numpy() for g in got])).all()
    assert (fail.cpu().numpy() == np.concatenate([g[1].cpu().numpy() for g in got])).all()
