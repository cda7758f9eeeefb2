"""The kernels over 8x8 tiles take the clusters in order of list length. The
order belongs to one search's clusters; replays of captured calls change the
clusters without a call of the library, so these sequences mix captured and
eager calls over frames that fall into different numbers of clusters, both
growing and shrinking. Every result is compared with the oracle (forces) or
with a list made eagerly for that frame, without orders (adjoint).
"""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_common import compare_forces, to_dev

pytestmark = pytest.mark.gpu

N_WATERS = 2000  # 6,000 atoms: above the size up to which an unpruned list is never ordered
RC, R_INNER, RLIST = 0.9, 0.94, 1.0
BETA = synth.ewald_beta(RC)


class Frames:
    def __init__(self):
        from paper_2405_01420_gb300 import nb
        self.nb = nb
        boxes = [synth.water_box(N_WATERS, seed) for seed in (1, 2, 3, 4)]
        b = boxes[0]
        self.n, self.box = b.n_atoms, b.box
        self.d = to_dev(b)
        self.args = (self.d["q"], self.d["type"], self.d["lj"], RC, BETA)
        self.g = torch.from_numpy(np.random.default_rng(8).normal(size=(self.n, 3)).astype(np.float32)).cuda()
        xs = []
        for k in boxes:
            x = torch.from_numpy(k.coords).cuda()
            pl = nb.Pairlist(self.n)
            pl.search(x, self.box, RLIST, self.d["excl_off"], self.d["excl_idx"])
            xs.append((pl.stats()["n_clusters"], x))
            pl.close()
        xs.sort(key=lambda v: v[0])
        assert xs[0][0] < xs[-1][0], "the frames need different cluster counts"
        self.small, self.large = xs[0][1], xs[-1][1]
        self.refs = {}

    def pair(self, grow):
        return (self.small, self.large) if grow else (self.large, self.small)

    def search(self, pl, x):
        pl.search(x, self.box, RLIST, self.d["excl_off"], self.d["excl_idx"])

    def ref(self, x):
        key = x.data_ptr()
        if key not in self.refs:
            d = self.d
            f = oracle.energy_forces(x.cpu().numpy(), d["q"].cpu().numpy(), d["type"].cpu().numpy(),
                                     d["lj"].cpu().numpy(), self.box, RC, BETA, d["excl_off"].cpu().numpy(),
                                     d["excl_idx"].cpu().numpy())[0]
            pl = self.nb.Pairlist(self.n, sort_lists=False)
            self.search(pl, x)
            self.refs[key] = (f, pl.backward(x, *self.args, self.g))
            pl.close()
        return self.refs[key]

    def call(self, pl, what, x, out=None):
        if what == "forces":
            F = torch.empty((self.n, 3), device="cuda") if out is None else out
            pl.forces(x, *self.args, F, want_energy=False)
            return F
        return pl.backward(x, *self.args, self.g)

    def check(self, what, got, frame):
        f, adj = self.ref(frame)
        if what == "forces":
            compare_forces(got.cpu().numpy(), f)
        else:  # the same FP32 pair terms in another order of summation
            for a, b in zip(got[:2], adj[:2]):
                assert (a - b).abs().max() <= 1e-4 * b.abs().max()
            for c in range(2):
                a, b = got[2][..., c], adj[2][..., c]
                assert (a - b).abs().max() <= 1e-3 * b.abs().max()


@pytest.fixture(scope="module")
def fr():
    return Frames()


def captured(fn):
    """fn() captured in a CUDA graph (fn has run eagerly before); returns the graph and fn's result."""
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        out = fn()
    torch.cuda.synchronize()
    return g, out


@pytest.mark.parametrize("grow", [True, False])
@pytest.mark.parametrize("what", ["forces", "backward"])
@pytest.mark.parametrize("prune", [True, False])
def test_eager_calls_over_a_captured_search(fr, prune, what, grow):
    """Search (and prune) captured; 8x8 force or adjoint calls issued eagerly between its replays."""
    first, second = fr.pair(grow)
    pl = fr.nb.Pairlist(fr.n)
    x = first.clone()

    def lists():
        fr.search(pl, x)
        if prune:
            pl.prune(x, R_INNER)

    lists()
    graph, _ = captured(lists)
    pl.set_flags(cluster_tiles=True)
    for frame in (first, second, first):
        x.copy_(frame)
        graph.replay()
        fr.check(what, fr.call(pl, what, x), frame)
    assert pl.status() == 0
    pl.close()


@pytest.mark.parametrize("grow", [True, False])
@pytest.mark.parametrize("what", ["forces", "backward"])
@pytest.mark.parametrize("prune, sort_lists, by_prune", [(True, True, True), (True, False, True), (False, True, True),
                                                         (True, True, False)])
def test_a_captured_call_over_eager_searches(fr, prune, sort_lists, by_prune, what, grow):
    """An 8x8 call captured when its list had an order, or was to get it, replayed over later lists, ordered
    or not."""
    first, second = fr.pair(grow)
    pl = fr.nb.Pairlist(fr.n, cluster_tiles=by_prune)
    x = first.clone()

    def lists():
        fr.search(pl, x)
        if prune:
            pl.prune(x, R_INNER)

    lists()
    if by_prune:
        fr.call(pl, what, x)
    pl.set_flags(cluster_tiles=True)
    F = torch.empty((fr.n, 3), device="cuda")
    graph, out = captured(lambda: fr.call(pl, what, x, F))
    graph.replay()
    fr.check(what, out, first)
    pl.set_flags(cluster_tiles=False, sort_lists=sort_lists)
    x.copy_(second)
    lists()
    graph.replay()
    fr.check(what, out, second)
    assert pl.status() == 0
    pl.close()
