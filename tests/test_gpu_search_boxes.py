"""The pair search over box shapes that its rules tell apart: the columns each
cluster looks at (rows before its own are skipped, periodic images of rows and
of z are looked at only where they can hold a partner), the z index that gives
a column's candidates, the scan of the columns (within the scatter up to 1,024
columns, a kernel of its own above) and the per-column sort (one CTA per column
with few columns, one warp with many).

Random points without exclusions: every pair within rlist by the FP32 distance
contract has its mask bit exactly once, so the pair sets are compared bit for
bit; there is no tolerance. The same for the pruned list at positions moved
since the search, whose clusters the prune first compares by their boxes.
"""
import numpy as np
import pytest
import torch

import oracle
from gpu_common import expand_counted_pairs, pair_set

pytestmark = pytest.mark.gpu

# box edges (nm) and atoms: one axis long or just above 2 rlist, partly filled columns, a column that holds
# everything, fewer atoms than a cluster, more than 1,024 columns in a flat box (sorted by CTA and, past 4
# columns per SM, by warp)
BOXES = [((1.61, 1.61, 9.0), 700), ((9.0, 1.61, 1.61), 700), ((1.61, 9.0, 1.61), 700), ((1.61, 1.61, 1.61), 5),
         ((2.0, 3.1, 4.3), 333), ((5.0, 1.7, 1.7), 1500), ((6.3, 6.1, 1.62), 9001), ((40.0, 41.0, 1.61), 12007)]
RLIST, R_INNER = 0.8, 0.7


def check(pl, nb, box, n, seed):
    rng = np.random.default_rng(seed)
    L = np.asarray(box, dtype=np.float32)
    x = (rng.random((n, 3)) * L).astype(np.float32)
    if n > 100:  # a dense slab at both faces of z, and atoms on the faces
        x[: n // 4, 2] = (x[: n // 4, 2] * np.float32(0.05)) % L[2]
        x[-3:] = np.stack([np.zeros_like(L), np.nextafter(L, np.float32(0)), L])
    eo, ei = np.zeros(n + 1, np.int32), np.zeros(0, np.int32)
    pl.search(torch.from_numpy(x).cuda(), L, RLIST)
    assert pl.status() == 0
    counted = expand_counted_pairs(pl.export(nb.NB_LIST_OUTER), oracle.image_f32(x, x, L), L, RLIST)
    ref = oracle.pairs_f32(x, x, L, RLIST, eo, ei)
    assert len(pair_set(counted)) == len(counted)
    assert pair_set(counted) == pair_set(ref)
    # moved by at most 0.035 nm, less than half the margin of 0.1 nm between rlist and r_inner
    moved = (x + rng.uniform(-0.02, 0.02, x.shape)).astype(np.float32)
    pl.prune(torch.from_numpy(moved).cuda(), R_INNER)
    assert pl.status() == 0
    counted = expand_counted_pairs(pl.export(nb.NB_LIST_INNER), oracle.image_f32(x, moved, L), L, R_INNER)
    ref = oracle.pairs_f32(x, moved, L, R_INNER, eo, ei)
    assert len(pair_set(counted)) == len(counted)
    assert pair_set(counted) == pair_set(ref)


@pytest.mark.parametrize("box, n", BOXES, ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_every_pair_once(box, n):
    from paper_2405_01420_gb300 import nb
    pl = nb.Pairlist(n)
    for seed in range(3):  # the column counts are 0 again after each search
        check(pl, nb, box, n, seed)
    pl.close()


def test_one_list_over_changing_boxes():
    """A pair list whose box, and with it the grid, changes from search to search."""
    from paper_2405_01420_gb300 import nb
    n = 1500
    pl = nb.Pairlist(n)
    for seed, box in enumerate([(3.0, 3.0, 3.0), (9.0, 1.61, 1.61), (1.7, 1.7, 6.0), (3.0, 3.0, 3.0)]):
        check(pl, nb, box, n, seed)
    pl.close()
