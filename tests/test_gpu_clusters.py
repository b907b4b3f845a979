"""The cluster kernels where their tiles, buffers and shares have their
edges: forces, energy, virial, counts and the adjoint against the oracle, for
clusters of a few to 256 molecules (one to eight tiles, several buffer
fills, a cluster that meets its own images), one and two species, with and
without the energy shift, meshes with fewer clusters than resident warps, and
meshes most of whose cells are empty.

Tolerances are those of the force and adjoint tests: forces 1e-12 (FP64) or
1e-5 (FP32) of max(|F_ic|, ||F_i||), energy and virial 1e-12 / 1e-6 of the sums
of magnitudes, gradients 1e-10 / 2e-4 of the largest."""
import numpy as np
import pytest
import torch

import oracle
from oracle import torch_ref
from paper_cs_0702131_gb300 import synth
from gpu_helpers import assert_forces, gpu_setup

pytestmark = pytest.mark.gpu


def _fluid(n, hexes, tets, species, seed=7, keep=None):
    """FCC fluid of 4 n^3 molecules (or `keep` of them) in hexes^3 hexahedra."""
    rng = np.random.default_rng(seed)
    a = synth.A_FCC_08
    L = np.full(3, n * a)
    box = dict(L=L, periodic=np.array([1, 1, 1], np.int32))
    pos = synth.wrap(synth.jitter(synth.fcc_sites(n, n, n, a), 0.05, rng), L, box["periodic"])
    if keep is not None:
        pos = pos[rng.permutation(len(pos))[:keep]]
    sp = (rng.permutation(len(pos)) % species).astype(np.int32)
    mesh = synth.hex_mesh((hexes,) * 3, (0, 0, 0), L, 0.15, rng, tets=tets)
    return dict(pos=pos, species=sp, eps=np.array([1.0, 1.5])[:species], sigma=np.array([1.0, 0.88])[:species],
                rc=2.5, box=box, mesh=mesh, skin=1e-3)


CASES = [  # (n, hexes, tets, species, kept molecules): molecules per cluster
    (4, 1, False, 1, None),     # 256: one cluster and its own images, eight tiles
    (4, 2, False, 2, None),     # 32 on average: a tile and a little more
    (5, 2, True, 1, None),      # 62
    (5, 3, False, 1, None),     # 18.5
    (4, 3, True, 2, None),      # 9.5: fewer clusters than warps
    (6, 6, False, 2, 40),       # mostly empty cells
    (4, 2, True, 1, 1),         # one molecule
]


@pytest.mark.parametrize("prec", ["fp64"])
@pytest.mark.parametrize("shift", [False, True])
@pytest.mark.parametrize("n,hexes,tets,species,keep", CASES)
def test_forces_at_the_edges(n, hexes, tets, species, keep, shift, prec):
    c = _fluid(n, hexes, tets, species, keep=keep)
    m, *_ = gpu_setup(c)
    assert m.get_option("cluster_path") == 1
    F, ev, cnt = m.forces(c["eps"], c["sigma"], prec, shift=shift)
    ref = oracle.lj(c["pos"], c["species"], c["eps"], c["sigma"], c["rc"], c["box"], shift=shift)
    assert_forces(F.double().cpu().numpy(), ref, 1e-12 if prec == "fp64" else 1e-5)
    te = 1e-12 if prec == "fp64" else 1e-6
    ev, cnt = ev.cpu().numpy(), cnt.cpu().numpy()
    assert abs(ev[0] - ref["U"]) <= te * ref["Uabs"]
    assert np.abs(ev[1:] - ref["W"]).max() <= te * ref["Wabs"]
    assert cnt[3] + cnt[4] + cnt[5] == ref["pairs"]
    m.close()


@pytest.mark.parametrize("prec", ["fp64"])
@pytest.mark.parametrize("n,hexes,tets,species,keep", CASES)
def test_adjoint_at_the_edges(n, hexes, tets, species, keep, prec):
    c = _fluid(n, hexes, tets, species, keep=keep)
    m, *_ = gpu_setup(c)
    v = np.random.default_rng(3).normal(size=c["pos"].shape)
    gx, ge, gs, _ = torch_ref.vjp(c["pos"], c["species"], c["eps"], c["sigma"], c["rc"], c["box"], v)
    dt, tol = (torch.float64, 1e-10) if prec == "fp64" else (torch.float32, 2e-4)
    gp, ge_g, gs_g = m.forces_backward(c["eps"], c["sigma"], torch.tensor(v, dtype=dt, device="cuda"), prec)
    assert np.abs(gp.double().cpu().numpy() - gx).max() <= tol * np.abs(gx).max()
    np.testing.assert_allclose(ge_g.cpu().numpy(), ge, rtol=tol, atol=tol * np.abs(ge).max())
    np.testing.assert_allclose(gs_g.cpu().numpy(), gs, rtol=tol, atol=tol * np.abs(gs).max())
    m.close()


def test_fp64_equals_the_cell_kernel():
    """The cluster kernel against the cell kernel, which serves the vertex
    criterion with a guard distance that lists every pair of this mesh."""
    c = _fluid(5, 3, False, 2)
    m, *_ = gpu_setup(c)
    F, ev, cnt = m.forces(c["eps"], c["sigma"], "fp64")
    m.build_lists(c["rc"], 1.5, criterion="vertex")
    assert m.get_option("cluster_path") == 0
    G, ew, cmt = m.forces(c["eps"], c["sigma"], "fp64")
    assert cnt[3:].sum() == cmt[3:].sum() and cnt[3] == cmt[3]
    assert (F - G).abs().max() <= 1e-12 * F.abs().max()
    assert (ev - ew).abs().max() <= 1e-12 * ew.abs().max()
    m.close()
