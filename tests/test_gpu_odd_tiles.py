"""Weight orders of cells that fill a tile of odd capacity to its last slot, the last species a power of two (every bucket of its
counting sort has a slot of its own): whole steps on unordered weights equal those on the same cells in a tile with room to
spare, in groups of one warp, of several and of half a warp."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2407_19151_gb300 import workloads as W

from _parity import device_state

pytestmark = pytest.mark.gpu


def _cells(n_cells, counts):
    base = W.three_species(n_cells=n_cells, mean_count=3.0 * max(counts) + 30.0, sigma=0.0, data_seed=4)
    keep = np.concatenate([base.offsets[3 * c + k] + np.arange(counts[k]) for c in range(n_cells) for k in range(3)])
    cut = lambda x: np.ascontiguousarray(x[keep])  # noqa: E731
    return dataclasses.replace(base, counts=np.tile(np.asarray(counts, dtype=np.int64), (n_cells, 1)), vx=cut(base.vx),
                               vy=cut(base.vy), vz=cut(base.vz), w=cut(base.w))


@pytest.mark.parametrize("counts,caps,room", [
    ((300, 213, 512), (64, 1025), (64, 1026)),   # 512 threads, full to the last slot
    ((250, 518, 257), (64, 1025), (64, 1026)),   # the last slot unused
    ((20, 25, 32), (77, 0), (78, 0)),            # one warp
    ((40, 1, 64), (105, 0), (106, 0)),
])
def test_full_odd_tile(counts, caps, room):
    import paper_2407_19151_gb300 as mcc
    wl = _cells(24, counts)
    assert wl.counts.sum(1).max() in caps
    ctx, runs = mcc.context(0), []
    for cap in (caps, room):
        ctx.set_group_capacity(*cap)
        try:
            v, w, off = device_state(wl, "f32")
            p = mcc.Params(method=wl.method, dt=wl.dt, fE=wl.fE, seed=wl.seed, step=3)
            corr, fail = mcc.mcc_step_fused(*v, w, off, wl.n_cells, 3, list(zip(wl.q, wl.m)), wl.lnL, p, n_steps=2)
            mcc.sync_status(0)
        finally:
            ctx.set_group_capacity(0)
        runs.append((v, corr, fail))
    for a, b in zip((*runs[0][0], *runs[0][1:]), (*runs[1][0], *runs[1][1:])):
        assert torch.equal(a, b)


def test_full_odd_tile_of_half_warps():
    import paper_2407_19151_gb300 as mcc
    n = 32 * torch.cuda.get_device_properties(0).multi_processor_count + 5
    wl = _cells(n, (19, 10, 8))
    runs = []
    for mc in (37, 38):  # the tile of half warps holds the largest cell: full, or with room
        v, w, off = device_state(wl, "f32")
        p = mcc.Params(method=wl.method, dt=wl.dt, fE=wl.fE, seed=wl.seed, step=3)
        corr, fail = mcc.mcc_step_fused(*v, w, off, n, 3, list(zip(wl.q, wl.m)), wl.lnL, p, max_cell=mc)
        mcc.sync_status(0)
        runs.append((v, corr, fail))
    for a, b in zip((*runs[0][0], *runs[0][1:]), (*runs[1][0], *runs[1][1:])):
        assert torch.equal(a, b)
