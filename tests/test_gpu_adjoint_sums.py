"""The LJ gradient of the gathered-tile adjoint is handed from a CTA's warps
to its last one through shared memory; a warp whose sums are not seen there
yet is missing from the result. Calls on one input are repeated and compared.

Tolerance: a half's FP32 sums are the same from call to call (one lane order),
and only the order of their FP64 addition differs. With fewer than 2^14
additions the two results differ by at most 2^15 * 2^-53 = 4e-12 of the sum of
the terms' magnitudes, which for the box here exceeds the gradient's entries
by less than 100 times; 1e-9 of the largest entry leaves more than twice that.
One warp's share is 1/2,432 of the sum on 152 SMs.
"""
import numpy as np
import pytest
import torch

import synth
from gpu_common import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ntype", [1, 2, 3, 4])
def test_lj_gradient_is_whole_on_every_call(ntype):
    from paper_2405_01420_gb300 import nb
    b = synth.water_box(1700, 31)
    rng = np.random.default_rng(5)
    types = rng.integers(0, ntype, b.n_atoms).astype(np.int32)
    c6 = rng.uniform(1e-3, 3e-3, ntype)
    c12 = rng.uniform(1e-6, 3e-6, ntype)
    lj = synth.combine_geometric(c6, c12).astype(np.float32)
    d = to_dev(b)
    t, ljd = torch.from_numpy(types).cuda(), torch.from_numpy(lj).cuda()
    rc = 0.9
    beta = synth.ewald_beta(rc)
    pl = nb.Pairlist(b.n_atoms)
    pl.search(d["coords"], b.box, 1.0, d["excl_off"], d["excl_idx"])
    pl.prune(d["coords"], 0.95)
    F, _ = pl.forces(d["coords"], d["q"], t, ljd, rc, beta, want_energy=False)
    out = torch.stack([pl.backward(d["coords"], d["q"], t, ljd, rc, beta, F)[2] for _ in range(100)])
    assert pl.status() == 0
    pl.close()
    for c in range(2):  # C6 and C12 gradients differ by orders of magnitude
        g = out[..., c]
        assert torch.isfinite(g).all()
        assert (g - g[0]).abs().max() <= 1e-9 * g[0].abs().max()
