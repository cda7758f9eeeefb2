"""The gathered-tile force kernel without energies in the middle of its range
of sizes: first items from the work counter at 5 CTAs per SM, between the
sizes whose warps start by index and those that the reaction field runs at 6
CTAs. The size is checked against both ends of that range on the device at
hand, so that a moved line cannot leave the kernel without a test.

Tolerances: against the oracle 1e-4 of rms(F), as for every force test here.
With and without energies every pair's force has the same bits, and only the
order of an atom's FP32 sums differs: about 150 additions, each rounding by at
most 2^-25 of a partial sum that stays below 30 rms(F), so about
sqrt(150) 3e-8 30 = 1.1e-5 of rms(F) if all were at that bound; 2e-5.
"""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_common import compare_forces, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("coul", ["ewald", "rf"])
def test_forces_from_the_counter(coul):
    from paper_2405_01420_gb300 import nb
    rc = 1.0
    beta = synth.ewald_beta(rc)
    b = synth.water_box(20001, 17)
    d = to_dev(b)
    pl = nb.Pairlist(b.n_atoms)
    if coul == "rf":
        pl.set_coulomb("rf")
    pl.search(d["coords"], b.box, 1.1, d["excl_off"], d["excl_idx"])
    pl.prune(d["coords"], 1.04)
    halves = 2 * (b.n_atoms // 8 + pl.stats()["n_columns"])
    warps = 5 * 4 * torch.cuda.get_device_properties(0).multi_processor_count
    assert 3.5 * warps < halves < 10 * warps
    args = (d["coords"], d["q"], d["type"], d["lj"], rc, beta)
    F, _ = pl.forces(*args, want_energy=False)
    FE, _ = pl.forces(*args)
    assert pl.status() == 0
    pl.close()
    if coul == "rf":
        Fo = oracle.energy_forces_coul(b.coords, b.q, b.type, b.ljparams, b.box, rc, 0.0, b.excl_off, b.excl_idx,
                                       kind="rf")[0]
    else:
        Fo = oracle.energy_forces(b.coords, b.q, b.type, b.ljparams, b.box, rc, beta, b.excl_off, b.excl_idx)[0]
    compare_forces(F.cpu().numpy(), Fo)
    compare_forces(F.cpu().numpy(), FE.cpu().numpy().astype(np.float64), tol=2e-5)
