"""Small cells two to a warp (mixed path, calls with many cells) against the one-warp groups, which an explicit capacity selects:
sizes from empty to beyond the line between them, unordered, tied and stored weight orders, both angle samplers, relativistic
pairs and cells visited again after a failed correction. The two differ in the order of float-float sums (2^-44), which now
and then moves a float of the pair kinematics by an ulp: equal counts, and stored velocities within two float ulps of their
population's speed."""
import numpy as np
import pytest
import torch

from paper_2407_19151_gb300 import workloads as W

from _parity import device_state, gpu_velocities, velocity_error

pytestmark = pytest.mark.gpu


def _cells():  # enough for every warp of the GPU to hold two, with room for the larger cells of a case
    return 4 * 16 * torch.cuda.get_device_properties(0).multi_processor_count + 3


@pytest.mark.parametrize("case", ["tiny", "line", "ta77", "stored", "retries", "beam"])
def test_half_warps(case):
    import paper_2407_19151_gb300 as mcc
    n, kw, rel = _cells(), {}, False
    if case == "tiny":
        wl = W.equilibration(n_cells=n, mean_count=4.0, data_seed=5, method=W.N97, precision="f32")
    elif case == "line":
        wl = W.equilibration(n_cells=n, mean_count=61.0, data_seed=6, method=W.N97, precision="f32")
    elif case == "ta77":
        wl = W.equilibration(n_cells=n, mean_count=25.0, data_seed=7, method=W.TA77, precision="f32")
    elif case == "stored":
        wl = W.three_species(n_cells=n, mean_count=45.0, data_seed=8).weight_ordered()
    elif case == "retries":
        wl = W.three_species(n_cells=n, mean_count=45.0, data_seed=9)
        kw = dict(max_corr_passes=1, fE=0.004)
    else:
        wl, rel = W.relativistic_beam(n_cells=n, data_seed=10, count_hi=250, precision="f32"), True
    kw.setdefault("fE", wl.fE)
    ctx = mcc.context(0)
    runs = []
    for per_warp in (0, 280):
        ctx.set_group_capacity(per_warp)
        try:
            v, w, off = device_state(wl, "f32")
            res = torch.full((2 * n,), -1.0, dtype=torch.float64, device="cuda")
            p = mcc.Params(method=wl.method, relativistic=rel, dt=wl.dt, c=wl.c, seed=wl.seed, step=3, residual=res, **kw)
            corr, fail = mcc.mcc_step_fused(*v, w, off, wl.n_cells, wl.n_species, list(zip(wl.q, wl.m)), wl.lnL, p)
            mcc.sync_status(0)
        finally:
            ctx.set_group_capacity(0)
        assert (res >= 0).all()  # every cell visited
        runs.append((gpu_velocities(v), corr.cpu().numpy(), fail.cpu().numpy()))
    if case == "retries":
        assert runs[0][2].sum() > n // 10
    np.testing.assert_array_equal(runs[0][1], runs[1][1])
    np.testing.assert_array_equal(runs[0][2], runs[1][2])
    assert velocity_error(runs[0][0], runs[1][0], wl.offsets).max() <= 2.0 ** -22


def test_overlapped_classes_captured():
    # every size class in one step, whose kernels overlap: a captured step replayed twice gives the two steps of a direct call, and
    # so does a call that records events between the kernels, bit for bit
    import paper_2407_19151_gb300 as mcc
    wl = W.three_species(n_cells=_cells(), mean_count=110.0, sigma=0.9, data_seed=12).weight_ordered()
    species, mc = list(zip(wl.q, wl.m)), int(np.diff(wl.offsets[:: wl.n_species]).max())
    assert mc > 1500
    kw = dict(method=wl.method, dt=wl.dt, fE=wl.fE, seed=wl.seed)

    def step(v, p, n):
        return mcc.mcc_step_fused(*v, w, off, wl.n_cells, wl.n_species, species, wl.lnL, p, n_steps=n, max_cell=mc)

    v0, w, off = device_state(wl, "f32")
    v1, v2 = [x.clone() for x in v0], [x.clone() for x in v0]
    warm = [x.clone() for x in v0]
    step(v0, mcc.Params(step=4, **kw), 2)
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2 * (mcc.GROUP_CLASSES + 1))]
    for e in ev:
        e.record()
    step(v2, mcc.Params(step=4, launch_events=ev, **kw), 2)
    counter = torch.tensor([4], dtype=torch.int64, device="cuda")
    pd = mcc.Params(step=0, **kw)
    pd.step_device = counter
    step(warm, pd, 1)
    torch.cuda.synchronize()
    counter.fill_(4)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        step(v1, pd, 1)
    g.replay()
    g.replay()
    torch.cuda.synchronize()
    mcc.sync_status(0)
    assert int(counter.item()) == 6
    for a, b, c in zip(v0, v1, v2):
        assert torch.equal(a, b) and torch.equal(a, c)
