"""The gathered-tile force kernel without energies, in each launch shape its
size rule picks (first items by index; from the counter at 5 and at 6 CTAs
per SM), and with energies beside it, against the oracle.

Without energies the kernel evaluates the pair force in its own form (one
rational for the Ewald force, 12 C12/r^6 - 6 C6 in one step), so every
Coulomb flavour is checked on its own. Tolerance: per atom 1e-4 of rms(F),
as for every force test here. The two forms differ by FP32 rounding of the
same pair set, so per pair by less than 1e-6 of its force; the largest pair
force is below 100 rms(F) in these boxes and an atom has up to 10 such
pairs, which leaves 1e-3 rms(F) as a bound no correct form can miss.
"""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_common import compare_forces

pytestmark = pytest.mark.gpu

# waters, rc, rlist, r_inner: below one half per warp, one to two, past the index rule, past the 6-CTA rule
SIZES = [(64, 0.5, 0.6, 0.55), (512, 0.9, 1.0, 0.95), (3999, 1.0, 1.1, 1.04), (13001, 1.0, 1.1, 1.04),
         (41003, 0.9, 1.0, 0.95)]


@pytest.mark.parametrize("size", SIZES, ids=lambda s: f"{3 * s[0]}")
@pytest.mark.parametrize("coul", ["ewald", "shift", "rf"])
def test_forces_without_energies(size, coul):
    from paper_2405_01420_gb300 import nb
    n_waters, rc, rlist, r_inner = size
    b = synth.water_box(n_waters, 11)
    beta = synth.ewald_beta(rc)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    x, q, t, lj = d(b.coords), d(b.q), d(b.type), d(b.ljparams)
    pl = nb.Pairlist(b.n_atoms)
    if coul != "ewald":
        pl.set_coulomb("rf" if coul == "rf" else "ewald", shift=coul == "shift")
    pl.search(x, b.box, rlist, d(b.excl_off), d(b.excl_idx))
    pl.prune(x, r_inner)
    # the accumulators and outputs of an earlier call must not show in the next
    F = torch.full((b.n_atoms, 3), float("nan"), device="cuda")
    for _ in range(2):
        pl.forces(x, q, t, lj, rc, beta, F, want_energy=False)
    FE, _ = pl.forces(x, q, t, lj, rc, beta)
    assert pl.status() == 0
    got, with_e = F.cpu().numpy(), FE.cpu().numpy()
    pl.close()
    if coul == "rf":  # the force vanishes at rc for a conducting boundary, so the FP64 pair set will do
        Fo = oracle.energy_forces_coul(b.coords, b.q, b.type, b.ljparams, b.box, rc, 0.0, b.excl_off, b.excl_idx,
                                       kind="rf")[0]
    else:
        Fo = oracle.energy_forces(b.coords, b.q, b.type, b.ljparams, b.box, rc, beta, b.excl_off, b.excl_idx)[0]
    compare_forces(got, Fo)
    compare_forces(with_e, Fo)
    compare_forces(got, with_e.astype(np.float64), tol=1e-3)


def test_without_energies_at_beta_zero():
    """beta = 0: the rational is 1 and the Ewald force is the bare Coulomb force."""
    from paper_2405_01420_gb300 import nb
    b = synth.water_box(700, 5)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    x, q, t, lj = d(b.coords), d(b.q), d(b.type), d(b.ljparams)
    pl = nb.Pairlist(b.n_atoms)
    pl.search(x, b.box, 0.9, d(b.excl_off), d(b.excl_idx))
    pl.prune(x, 0.85)
    F, _ = pl.forces(x, q, t, lj, 0.8, 0.0, want_energy=False)
    FE, _ = pl.forces(x, q, t, lj, 0.8, 0.0)
    assert pl.status() == 0
    # the bare force does not vanish at the cutoff: both forms decide the same pair set
    compare_forces(F.cpu().numpy(), FE.cpu().numpy().astype(np.float64))
    pl.close()
