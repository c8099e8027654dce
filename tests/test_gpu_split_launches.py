"""The unfused calls on both sides of one cell per SM (one launch up to there, two that may overlap beyond), with cells on both sides
of the first launch's tile: the separate calls equal the oracle, and a captured scatter and correction equal direct ones."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2407_19151_gb300 import workloads as W

from _parity import F64_TOL, device_state, gpu_velocities, oracle_state, velocity_error
from test_gpu_split_and_order import _with_counts

pytestmark = pytest.mark.gpu


def _workload(extra, prec):
    n = torch.cuda.get_device_properties(0).multi_processor_count + extra
    tot = np.resize([0, 1, 2, 30, 300, 640, 700, 960, 1200, 2400], n)
    return _with_counts(W.three_species(n_cells=1, precision=prec), np.stack([(tot + 2) // 3, (tot + 1) // 3, tot // 3], 1))


def _calls(mcc, wl, v, w, off, p, pairs=None):
    sp, total = list(zip(wl.q, wl.m)), 0
    for k, (a, b) in enumerate(mcc.default_interactions(3)):
        pr = pairs[k] if pairs else mcc.mcc_pair(off, wl.n_cells, 3, a, b, k, p.seed, p.step)
        backup = mcc.mcc_scatter(*v, w, off, wl.n_cells, 3, sp, wl.lnL, a, b, k, pr, p)
        total = total + mcc.mcc_correct(*v, w, off, wl.n_cells, 3, sp, a, b, k, p, backup)[1]
    return total


@pytest.mark.parametrize("extra", [0, 1, 60])
def test_separate_calls(extra):
    import paper_2407_19151_gb300 as mcc
    wl = _workload(extra, "f64")
    v, w, off = device_state(wl, "f64")
    kw = dict(method=wl.method, dt=wl.dt, fE=wl.fE, seed=wl.seed, step=4)
    total = _calls(mcc, wl, v, w, off, mcc.Params(**kw))
    mcc.sync_status(0)
    st = oracle_state(wl, "f64")
    _, ofail = O.step(st, wl.q, wl.m, wl.lnL, O.Params(**kw), n_steps=1)
    np.testing.assert_array_equal(total.cpu().numpy(), ofail)
    assert velocity_error(gpu_velocities(v), st.v(), wl.offsets).max() < F64_TOL


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("rel", [False, True])
def test_two_launches_equal_one(prec, rel):
    """Cells are independent: a call on all of them (two launches) gives what calls on a third of them (one launch) give."""
    import paper_2407_19151_gb300 as mcc
    wl = _workload(60, prec)
    v, w, off = device_state(wl, prec)
    u = [x.clone() for x in v]
    sp = list(zip(wl.q, wl.m))
    kw = dict(method=wl.method, relativistic=rel, c=9.0, dt=wl.dt, fE=wl.fE, seed=wl.seed, step=4)
    p, n = mcc.Params(**kw), wl.n_cells
    a, b, k = 0, 1, 1
    pairs = mcc.mcc_pair(off, n, 3, a, b, k, p.seed, p.step)
    want = O.pairs(wl.offsets, n, 3, a, b, k, p.seed, p.step)
    for x, y in zip(pairs, want):
        np.testing.assert_array_equal(x.cpu().numpy()[want[0] >= 0], np.asarray(y)[want[0] >= 0])
    backup = mcc.mcc_scatter(*v, w, off, n, 3, sp, wl.lnL, a, b, k, pairs, p)
    corr, fail = mcc.mcc_correct(*v, w, off, n, 3, sp, a, b, k, p, backup)
    got = []
    for c0 in range(0, n, (n + 2) // 3):
        c1 = min(n, c0 + (n + 2) // 3)
        p0, p1 = int(wl.offsets[3 * c0]), int(wl.offsets[3 * c1])
        o = off[3 * c0:3 * c1 + 1] - p0
        x, ws = [y[p0:p1].clone() for y in u], w[p0:p1].clone()
        pr = (pairs[0][p0:p1] - p0, pairs[1][p0:p1] - p0, pairs[2][p0:p1].clone())
        q = mcc.Params(**kw, cell_base=c0)
        bk = mcc.mcc_scatter(*x, ws, o, c1 - c0, 3, sp, wl.lnL, a, b, k, pr, q)
        got.append((*x, *mcc.mcc_correct(*x, ws, o, c1 - c0, 3, sp, a, b, k, q, bk)))
    mcc.sync_status(0)
    for x, parts in zip((*v, corr, fail), zip(*got)):
        assert torch.equal(x, torch.cat(parts))


def test_captured_calls():
    import paper_2407_19151_gb300 as mcc
    wl = _workload(60, "f64")
    v, w, off = device_state(wl, "f64")
    u = [x.clone() for x in v]
    p = mcc.Params(method=wl.method, dt=wl.dt, fE=wl.fE, seed=wl.seed, step=4)
    pairs = [mcc.mcc_pair(off, wl.n_cells, 3, a, b, k, p.seed, p.step)
             for k, (a, b) in enumerate(mcc.default_interactions(3))]
    t0 = [x.clone() for x in v]
    _calls(mcc, wl, t0, w, off, p, pairs)  # warm-up
    for _ in range(2):
        direct = _calls(mcc, wl, v, w, off, p, pairs)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        captured = _calls(mcc, wl, u, w, off, p, pairs)
    g.replay()
    g.replay()
    torch.cuda.synchronize()
    mcc.sync_status(0)
    for a, b in zip((*v, direct), (*u, captured)):
        assert torch.equal(a, b)
