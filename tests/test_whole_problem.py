"""The cell counts of the whole problem that shards and chunks hand to the step (host logic, CPU)."""
import numpy as np

from paper_2407_19151_gb300 import Params, sharding
from paper_2407_19151_gb300 import _binding as B


class _Backend:
    def load(self, vx, vy, vz, w, view):
        return {}

    def zeros(self, n):
        return np.zeros(n)

    def step(self, st, n_cells, S, species, lnL, params, n_steps, max_cell, fail):
        self.seen = (n_cells, params.cell_base, params.whole_cells, params.whole_small, max_cell)


def _offsets(counts):
    off = np.zeros(counts.size + 1, dtype=np.int64)
    np.cumsum(counts.reshape(-1), out=off[1:])
    return off


def test_shards_carry_the_whole_problems_counts():
    tot = np.array([0, 1, B.SMALL_CELL - 1, B.SMALL_CELL, B.SMALL_CELL + 1, 700, 3, 500])
    off = _offsets(np.stack([(tot + 1) // 2, tot // 2], 1))
    n = int(off[-1])
    for world in (1, 3):
        for r in range(world):
            be = _Backend()
            sh = sharding.ShardedStep(off, len(tot), 2, [(1.0, 1.0)] * 2, 10.0, Params(), backend=be,
                                      cell_range=sharding.shard_cells(off, 2, world, r))
            sh.load(*[np.zeros(n)] * 4).advance(1)
            if sh.n_cells:
                assert be.seen == (sh.n_cells, sh.c0, len(tot), 4, 700)


def test_a_part_of_a_part_keeps_the_outer_counts():
    off = _offsets(np.full((10, 2), 40))
    assert sharding.whole_problem(off, 2, Params()) == dict(whole_cells=10, whole_small=10)
    assert sharding.whole_problem(off, 2, Params(whole_cells=99, whole_small=7)) == dict(whole_cells=99, whole_small=7)
