"""Deferred checks and molecules of a species that the parameters do not have
(index in [n_species, 8)): their pairs carry no force, energy, virial or
gradient, so what is left are the results of the other molecules alone.

Tolerances are those of the force and adjoint tests: 1e-12 of max(|F_ic|,
||F_i||), energy and virial 1e-12 of the sums of magnitudes, gradients 1e-10 of
the largest."""
import numpy as np
import pytest
import torch

import oracle
from oracle import torch_ref
from paper_cs_0702131_gb300 import synth
from paper_cs_0702131_gb300.aica import Mesh
from gpu_helpers import assert_forces

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("species", [2, 3])
@pytest.mark.parametrize("shift", [False, True])
def test_pairs_of_unknown_species_carry_nothing(species, shift):
    rng = np.random.default_rng(species)
    a = synth.A_FCC_08
    L = np.full(3, 5 * a)
    box = dict(L=L, periodic=np.array([1, 1, 1], np.int32))
    x = synth.wrap(synth.jitter(synth.fcc_sites(5, 5, 5, a), 0.05, rng), L, box["periodic"])
    n = len(x)
    sp = (rng.permutation(n) % species).astype(np.int32)
    unknown = rng.permutation(n)[:40]
    known = np.setdiff1d(np.arange(n), unknown)
    sp[unknown] = species + np.arange(40) % (8 - species)
    eps, sigma = np.array([1.0, 1.5, 0.7])[:species], np.array([1.0, 0.88, 1.1])[:species]
    m = Mesh(synth.hex_mesh((4, 4, 4), (0, 0, 0), L, 0.15, rng), box)
    m.build_lists(2.5, 1e-3)
    m.set_deferred(True)
    m.bin(torch.tensor(x, device="cuda"), torch.tensor(sp, device="cuda"), outputs=False)
    F, ev, _ = m.forces(eps, sigma, "fp64", shift=shift)
    F, ev = F.cpu().numpy(), ev.cpu().numpy()
    ref = oracle.lj(x[known], sp[known], eps, sigma, 2.5, box, shift=shift)
    assert not F[unknown].any()
    assert_forces(F[known], ref, 1e-12)
    assert abs(ev[0] - ref["U"]) <= 1e-12 * ref["Uabs"]
    assert np.abs(ev[1:] - ref["W"]).max() <= 1e-12 * ref["Wabs"]

    v = rng.standard_normal((n, 3))
    gp, ge, gs = (t.cpu().numpy() for t in
                  m.forces_backward(eps, sigma, torch.tensor(v, device="cuda"), "fp64"))
    gx, re, rs, _ = torch_ref.vjp(x[known], sp[known], eps, sigma, 2.5, box, v[known])
    assert not gp[unknown].any()
    assert np.abs(gp[known] - gx).max() <= 1e-10 * np.abs(gx).max()
    np.testing.assert_allclose(ge, re, rtol=1e-10, atol=1e-10 * np.abs(re).max())
    np.testing.assert_allclose(gs, rs, rtol=1e-10, atol=1e-10 * np.abs(rs).max())
    m.check()
    m.close()
