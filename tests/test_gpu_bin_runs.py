"""Cell sorts of nearly binned input: bit-exact against the oracle over the ways a warp groups its keys (a match over all lanes, or
runs of neighbours) and a segment maps its indices to buckets (one linear piece, three, or the bitonic network)."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


def _binned(sizes, S, rng):
    """Keys of `sizes` particles per segment, in segment order."""
    key = np.repeat(np.arange(len(sizes)), sizes)
    return (key // S).astype(np.int32), (key % S).astype(np.int32)


def _case(name):
    rng = np.random.default_rng(23)
    S = 3
    if name == "sizes":  # every size around the warp, the bucket counts and the warp sort's limit, a fifth moved
        sizes = np.repeat([0, 1, 2, 11, 12, 13, 14, 24, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 400, 511, 512,
                           513, 600], 12)
        cell, sp = _binned(rng.permutation(sizes), S, rng)
        C = len(sizes) // S
        move = rng.random(len(cell)) < 0.2
        cell[move] = (cell[move] + rng.choice([-9, -1, 1, 9], move.sum())) % C
    elif name in ("low", "high"):  # what moved in comes from one side only, the far end of the arrays
        sizes = np.full(300, 170)
        cell, sp = _binned(sizes, S, rng)
        C = 100
        move = rng.random(len(cell)) < 0.25
        cell[move] = rng.integers(0, C, move.sum())
        far = (cell // 50) == (1 if name == "low" else 0)  # only one half of the cells receives
        cell[move & ~far] = _binned(sizes, S, rng)[0][move & ~far]
    elif name.startswith("moved"):
        C = 400
        cell, sp = _binned(np.full(C * S, 120), S, rng)
        move = rng.random(len(cell)) < float(name[5:])
        cell[move] = rng.integers(0, C, move.sum())
    elif name == "turns":  # species in turns within binned cells
        C = 500
        n = C * S * 90
        cell, sp = (np.arange(n) // (S * 90)).astype(np.int32), (np.arange(n) % S).astype(np.int32)
    elif name == "random species":
        C = 500
        n = C * S * 90
        cell, sp = (np.arange(n) // (S * 90)).astype(np.int32), rng.integers(0, S, n).astype(np.int32)
    elif name == "few":  # at the number of segments below which every warp takes the match
        C = 170
        cell, sp = rng.integers(0, C, 50_001).astype(np.int32), rng.integers(0, S, 50_001).astype(np.int32)
    else:  # "shuffled": just above it
        C = 171
        cell, sp = rng.integers(0, C, 50_001).astype(np.int32), rng.integers(0, S, 50_001).astype(np.int32)
    return np.ascontiguousarray(cell), np.ascontiguousarray(sp), C, S


@pytest.mark.parametrize("name", ["sizes", "low", "high", "moved0.02", "moved0.17", "moved0.6", "moved0.95", "turns",
                                  "random species", "few", "shuffled"])
def test_nearly_binned(name):
    import paper_2407_19151_gb300 as mcc
    from paper_2407_19151_gb300 import _binding as B
    cell, sp, C, S = _case(name)
    w = 10.0 ** np.random.default_rng(5).uniform(0, 4, len(cell))
    c, s = torch.from_numpy(cell).cuda(), torch.from_numpy(sp).cuda()
    rperm, roff = O.bin_particles(cell, sp, C, S)
    for perm, off in (mcc.mcc_bin(c, s, C, S), B.mcc_bin_static(c, s, C, S)):
        np.testing.assert_array_equal(off.cpu().numpy(), roff)
        np.testing.assert_array_equal(perm.cpu().numpy(), rperm)
    perm, off = mcc.mcc_bin_weighted(c, s, torch.from_numpy(w).cuda(), C, S)
    mcc.sync_status(0)
    rperm, roff = O.bin_particles_weighted(cell, sp, w, C, S)
    np.testing.assert_array_equal(off.cpu().numpy(), roff)
    np.testing.assert_array_equal(perm.cpu().numpy(), rperm)


@pytest.mark.parametrize("n", [63_999_999, 64_000_000])
def test_gather_on_both_sides_of_the_streaming_line(n):
    import paper_2407_19151_gb300 as mcc
    g = torch.Generator(device="cuda").manual_seed(3)
    perm = torch.randperm(n, device="cuda", generator=g).int()
    x = torch.arange(n, device="cuda", dtype=torch.float64)
    assert torch.equal(mcc.mcc_gather(x, perm), perm.double())
