"""The lines by which a call picks its kernels, with cells that reach them: few cells on groups of 64, 128 and 256 threads (at the
cell counts and at the largest cell where each begins), FP64 steps of small cells on six CTAs per SM (largest cell 319 to 321).
Every case holds empty cells and cells of 1 to 5 particles. The number of launches shows which size classes ran; results against
the oracle within the stated bounds (mixed path 2e-6 for 99.9% of the particles)."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle as O
from paper_2407_19151_gb300 import workloads as W

from _parity import F32_TOL, F64_TOL, device_state, gpu_velocities, oracle_state, velocity_error

pytestmark = pytest.mark.gpu


def _cells(tot, precision):
    """Three-species cells of the given totals, cut from larger ones."""
    tot = np.asarray(tot, dtype=np.int64)
    counts = np.stack([(tot + 2) // 3, (tot + 1) // 3, tot // 3], 1)
    base = W.three_species(n_cells=len(tot), mean_count=float(tot.max() + 30), sigma=0.0, data_seed=9, precision=precision)
    keep = np.concatenate([base.offsets[k] + np.arange(c) for k, c in enumerate(counts.reshape(-1))])
    cut = lambda x: np.ascontiguousarray(x[keep])  # noqa: E731
    return dataclasses.replace(base, counts=counts, vx=cut(base.vx), vy=cut(base.vy), vz=cut(base.vz), w=cut(base.w))


def _totals(n, largest):
    rng = np.random.default_rng(n + largest)
    tot = rng.integers(max(6, largest // 4), largest + 1, n)
    tot[rng.permutation(n)[: n // 4]] = rng.integers(0, 6, n // 4)  # empty and tiny cells among them
    tot[-1], tot[0] = 0, largest
    return tot


def _step(mcc, wl, prec):
    v, w, off = device_state(wl, prec)
    kw = dict(method=wl.method, dt=wl.dt, fE=wl.fE, seed=wl.seed, step=3)
    ctx = mcc.context(0)
    before = ctx.launch_count()
    corr, fail = mcc.mcc_step_fused(*v, w, off, wl.n_cells, 3, list(zip(wl.q, wl.m)), wl.lnL, mcc.Params(**kw),
                                    max_cell=int(wl.counts.sum(1).max()))
    launches = ctx.launch_count() - before
    mcc.sync_status(0)
    st = oracle_state(wl, prec)
    ocorr, ofail = O.step(st, wl.q, wl.m, wl.lnL, O.Params(**kw), n_steps=1)
    err = velocity_error(gpu_velocities(v), st.v(), wl.offsets)
    return launches, err, corr.cpu().numpy(), fail.cpu().numpy(), ocorr, ofail


# (cells: so many per SM and so many more, largest cell, class from which the call runs)
@pytest.mark.parametrize("per_sm,more,largest,cls", [
    (0, 3, 700, 3), (2, 0, 600, 3), (2, 1, 600, 2), (4, 0, 300, 2), (4, 1, 300, 1), (8, 0, 150, 1), (8, 1, 150, 0),
    (0, 100, 511, 2), (0, 100, 512, 3), (0, 100, 255, 1), (0, 100, 256, 2), (0, 100, 127, 0), (0, 100, 128, 1)])
def test_few_cells(per_sm, more, largest, cls):
    import paper_2407_19151_gb300 as mcc
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + more
    wl = _cells(_totals(n, largest) if n > 5 else [largest, 0, 1], "f32")
    caps = [-1] * cls + mcc.context(0).group_capacities()[cls:]
    launches, err, _, fail, _, ofail = _step(mcc, wl, "f32")
    # the cells' order, then the classes that can hold a cell
    assert launches == 1 + sum(k == cls or caps[k - 1] < largest for k in range(cls, 5))
    big = np.repeat(wl.counts.sum(1) >= 24, wl.counts.sum(1))  # (tiny cells have a bound of their own, 5e-4)
    assert np.quantile(err[big], 0.999) < F32_TOL and err.max() < 5e-4
    np.testing.assert_array_equal(fail[wl.counts.sum(1) >= 24], ofail[wl.counts.sum(1) >= 24])


@pytest.mark.parametrize("largest", [319, 320, 321])
@pytest.mark.parametrize("extra", [0, 1])
def test_small_cells_fp64(largest, extra):
    import paper_2407_19151_gb300 as mcc
    wl = _cells(_totals(4 * torch.cuda.get_device_properties(0).multi_processor_count + extra, largest), "f64")
    _, err, corr, fail, ocorr, ofail = _step(mcc, wl, "f64")
    np.testing.assert_array_equal(fail, ofail)
    np.testing.assert_array_equal(corr, ocorr)
    assert err.max() < F64_TOL
