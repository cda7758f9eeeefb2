"""One pair force whatever the call: on isolated pairs of atoms, where a force
is a single term and no order of summation can change it, the gathered-tile
force kernel gives the same bits with and without energies, and the Ewald
adjoint the same radial factor. Every comparison is of bits; there is no
tolerance.

The pairs sit on a lattice wider than the cutoff allows a second neighbour.
All other terms that reach an atom's accumulator are zeros, which change no
value.
"""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

CELLS, SPACING = 6, 3.0  # 216 pairs in an 18 nm box
RC, RLIST, R_INNER = 1.0, 1.1, 1.04
BETA = synth.ewald_beta(RC)
F_COULOMB = np.float32(138.935458)


def dimers(seed, r):
    """Pairs at distances r (one per pair) in random directions; atoms in random order, and each atom's partner."""
    rng = np.random.default_rng(seed)
    c = (np.stack(np.meshgrid(*[np.arange(CELLS)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.5) * SPACING
    u = rng.normal(size=c.shape)
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    x = np.concatenate([c, c + u * r[:, None]]).astype(np.float32)
    n = len(x)
    order = rng.permutation(n)
    inv = np.argsort(order)
    partner = inv[(order + n // 2) % n]
    return x[order], order < n // 2, partner


def prepared(nb, x, coul="ewald"):
    box = np.full(3, CELLS * SPACING, np.float32)
    pl = nb.Pairlist(len(x))
    if coul != "ewald":
        pl.set_coulomb("rf" if coul == "rf" else "ewald", shift=coul == "shift")
    xd = torch.from_numpy(x).cuda()
    pl.search(xd, box, RLIST)
    pl.prune(xd, R_INNER)
    return pl, xd


def bits(t):
    return (t + 0.0).view(torch.int32)  # -0 + 0 = 0: a zero force has no sign


@pytest.mark.parametrize("coul", ["ewald", "shift", "rf"])
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_forces_with_and_without_energies(coul, seed):
    from paper_2405_01420_gb300 import nb
    rng = np.random.default_rng(seed + 100)
    r = rng.uniform(0.12, 0.98, CELLS ** 3)
    x, _, partner = dimers(seed, r)
    n, nt = len(x), 4
    lj = synth.combine_geometric(rng.uniform(1e-3, 3e-3, nt), rng.uniform(1e-6, 3e-6, nt)).astype(np.float32)
    lj[0] = lj[:, 0] = 0.0
    args = [torch.from_numpy(a).cuda() for a in (rng.normal(0, 0.5, n).astype(np.float32),
                                                 rng.integers(0, nt, n).astype(np.int32), lj)] + [RC, BETA]
    pl, xd = prepared(nb, x, coul)
    F, _ = pl.forces(xd, *args, want_energy=False)
    FE, _ = pl.forces(xd, *args)
    assert pl.status() == 0
    pl.close()
    assert torch.isfinite(F).all() and (F.abs().amax(1) > 0).float().mean() > 0.99
    assert torch.equal(bits(F), bits(FE))
    assert torch.equal(bits(F), bits(-F[torch.from_numpy(partner).cuda()]))


@pytest.mark.parametrize("energy", [False, True])
def test_the_adjoints_ewald_factor_is_the_forces(energy):
    """Without LJ, with charges 1 and 1/f (whose product with f is exactly 1) the force on the first atom
    along x is fl(B dx), and so is dL/dq of the unit charge for g = x on the first atom."""
    from paper_2405_01420_gb300 import nb
    qf = np.float32(1) / F_COULOMB
    qf = next(q for q in (qf, np.nextafter(qf, np.float32(0)), np.nextafter(qf, np.float32(1)))
              if np.float32(q * F_COULOMB) == 1)
    rng = np.random.default_rng(7)
    x, first, partner = dimers(7, rng.uniform(0.12, 0.98, CELLS ** 3))
    n = len(x)
    q = torch.from_numpy(np.where(first, qf, np.float32(1)).astype(np.float32)).cuda()
    t, lj = torch.zeros(n, dtype=torch.int32, device="cuda"), torch.zeros((1, 1, 2), device="cuda")
    g = np.zeros((n, 3), np.float32)
    g[first, 0] = 1.0
    pl, xd = prepared(nb, x)
    F, _ = pl.forces(xd, q, t, lj, RC, BETA, want_energy=energy)
    _, gq, _ = pl.backward(xd, q, t, lj, RC, BETA, torch.from_numpy(g).cuda())
    assert pl.status() == 0
    pl.close()
    f = torch.from_numpy(first).cuda()
    assert torch.equal(bits(F[f, 0]), bits(gq[torch.from_numpy(partner).cuda()][f]))


@pytest.mark.parametrize("energy", [False, True])
@pytest.mark.parametrize("coul", ["ewald", "rf"])
def test_close_atoms_without_lj(coul, energy):
    """Atoms without LJ 1e-5 nm apart: 1/r^8 overflows FP32, the Coulomb force does not."""
    from paper_2405_01420_gb300 import nb
    x, _, _ = dimers(9, np.full(CELLS ** 3, 1e-5))
    n = len(x)
    q = torch.full((n,), 0.4, device="cuda")
    t, lj = torch.zeros(n, dtype=torch.int32, device="cuda"), torch.zeros((1, 1, 2), device="cuda")
    pl, xd = prepared(nb, x, coul)
    F, _ = pl.forces(xd, q, t, lj, RC, BETA, want_energy=energy)
    assert pl.status() == 0
    pl.close()
    assert torch.isfinite(F).all()
