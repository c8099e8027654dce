"""A problem stepped in parts (chunks of the host pipeline, shards of ShardedStep) equals the same problem in one call bit for bit,
also where the whole problem and its parts lie on different sides of the lines by which a call picks the size of its groups:
few cells on larger groups, many small cells on half warps, FP64 steps of small cells on more CTAs per SM."""
import numpy as np
import pytest
import torch

from paper_2407_19151_gb300 import sharding
from paper_2407_19151_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _case(name):
    """Workload, relativistic; the counts put whole and quarters on different sides of a line for 152 SMs."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if name == "few":  # whole on 64 threads and more, quarters on 256
        wl = W.three_species(n_cells=7 * sms, mean_count=300.0, data_seed=31)
        assert 2 * wl.n_cells <= 16 * sms and wl.counts.sum(1).max() >= 512
    elif name == "few small":  # quarters on 64 threads
        wl = W.equilibration(n_cells=10 * sms, mean_count=70.0, data_seed=32, method=W.TA77, precision="f32")
        assert 128 <= wl.counts.sum(1).max() < 256
    elif name == "half":  # half warps in the whole only
        wl = W.three_species(n_cells=36 * sms, mean_count=40.0, data_seed=33).weight_ordered()
        assert (wl.counts.sum(1) < 128).sum() >= 32 * sms
    elif name == "beam":
        wl = W.relativistic_beam(n_cells=60 * sms, data_seed=34, count_hi=700, precision="f32")
        assert (wl.counts.sum(1) < 128).sum() >= 32 * sms
    else:  # "f64": six CTAs per SM in the whole only
        wl = W.three_species(n_cells=4 * sms + 40, mean_count=90.0, sigma=0.2, data_seed=35, precision="f64")
        assert wl.counts.sum(1).max() <= 320
    return wl, name == "beam"


CASES = ["few", "few small", "half", "beam", "f64"]


def _whole(mcc, wl, p, n_steps):
    dt = torch.float64 if wl.precision == "f64" else torch.float32
    v = [torch.from_numpy(np.ascontiguousarray(x)).to("cuda", dt) for x in (wl.vx, wl.vy, wl.vz)]
    corr, fail = mcc.mcc_step_fused(*v, torch.from_numpy(wl.w).cuda(), torch.from_numpy(wl.offsets).cuda(), wl.n_cells,
                                    wl.n_species, list(zip(wl.q, wl.m)), wl.lnL, p, n_steps=n_steps)
    mcc.sync_status(0)
    return [x.cpu().numpy() for x in v], corr.cpu().numpy(), fail.cpu().numpy()


@pytest.mark.parametrize("name", CASES)
def test_chunks_equal_one_call(name):
    import paper_2407_19151_gb300 as mcc
    from paper_2407_19151_gb300.host_pipeline import step_host
    wl, rel = _case(name)
    p = mcc.Params(method=wl.method, relativistic=rel, dt=wl.dt, c=wl.c, fE=wl.fE, seed=wl.seed, step=5)
    v, corr, fail = _whole(mcc, wl, p, 2)
    dt = torch.float64 if wl.precision == "f64" else torch.float32
    host = [torch.from_numpy(np.ascontiguousarray(x)).to(dt).pin_memory() for x in (wl.vx, wl.vy, wl.vz)]
    hc, hf = step_host(*host, torch.from_numpy(wl.w).pin_memory(), wl.offsets, wl.n_cells, wl.n_species,
                       list(zip(wl.q, wl.m)), wl.lnL, p, n_steps=2, chunks=4)
    mcc.sync_status(0)
    for a, b in zip(host, v):
        np.testing.assert_array_equal(a.numpy(), b)
    np.testing.assert_array_equal(hc, corr)
    np.testing.assert_array_equal(hf, fail)


@pytest.mark.parametrize("name", CASES)
def test_shards_equal_one_call(name):
    import paper_2407_19151_gb300 as mcc
    wl, rel = _case(name)
    kw = dict(method=wl.method, relativistic=rel, dt=wl.dt, c=wl.c, fE=wl.fE, seed=wl.seed, step=2)
    v, _, fail = _whole(mcc, wl, mcc.Params(**kw), 2)
    dt = np.float64 if wl.precision == "f64" else np.float32
    arrays = [np.asarray(x, dtype=dt) for x in (wl.vx, wl.vy, wl.vz)]
    got, fails = [], 0
    for r in range(4):
        sh = sharding.ShardedStep(wl.offsets, wl.n_cells, wl.n_species, list(zip(wl.q, wl.m)), wl.lnL, mcc.Params(**kw),
                                  cell_range=sharding.shard_cells(wl.offsets, wl.n_species, 4, r))
        sh.load(*arrays, wl.w)
        fails += sh.step(2)[1]
        got.append(sh.velocities())
    mcc.sync_status(0)
    np.testing.assert_array_equal(np.concatenate(got), np.stack(v, axis=1).astype(np.float64))
    assert fails == fail.sum()


def test_part_of_a_problem_refuses_wrong_counts():
    import paper_2407_19151_gb300 as mcc
    wl = W.three_species(n_cells=20, mean_count=30.0)
    for whole in ((19, 0), (20, 21), (30, -1)):
        with pytest.raises(mcc.MccError):
            _whole(mcc, wl, mcc.Params(method=wl.method, dt=wl.dt, seed=1, whole_cells=whole[0], whole_small=whole[1]), 1)
