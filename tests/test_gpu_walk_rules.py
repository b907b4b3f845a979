"""Point location from previous cells at the edges of its rules: as many
molecules as the search has warps and one more (nobody walks, or warps with
enough walkers do), moves of a fraction of a cell to unrelated positions (walks
that arrive, run out or are not begun), meshes of tetrahedra, of convex and of
other hexahedra, and of both tetrahedra and hexahedra.  The cells must be those
of a search without previous cells, and those of the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_cs_0702131_gb300 import synth
from paper_cs_0702131_gb300.aica import Mesh

pytestmark = pytest.mark.gpu

L = np.full(3, 15.0)
BOX = dict(L=L, periodic=np.array([1, 1, 1], np.int32))


def _mixed(rng):
    """Two stacks, one of tetrahedra and one of hexahedra, that meet at z = 7.5
    without being neighbours: a walk ends there."""
    lo, hi = np.zeros(3), L.copy()
    hi[2] = 7.5
    a = synth.hex_mesh((6, 6, 3), lo, hi, 0.15, rng, tets=True)
    lo[2], hi[2] = 7.5, 15.0
    b = synth.hex_mesh((6, 6, 3), lo, hi, 0.15, rng)
    off = a["points"].shape[0]
    return dict(points=np.concatenate([a["points"], b["points"]]),
                face_offsets=np.concatenate([a["face_offsets"], b["face_offsets"][1:] + a["face_offsets"][-1]]),
                face_vertices=np.concatenate([a["face_vertices"], b["face_vertices"] + off]),
                owner=np.concatenate([a["owner"], b["owner"] + a["n_cells"]]),
                neighbour=np.concatenate([a["neighbour"],
                                          np.where(b["neighbour"] < 0, -1, b["neighbour"] + a["n_cells"])]),
                n_cells=a["n_cells"] + b["n_cells"])


def _mesh(kind):
    rng = np.random.default_rng(2)
    if kind == "mixed":
        return _mixed(rng)
    return synth.hex_mesh((6, 6, 6), (0, 0, 0), L, 0.0 if kind == "cube" else 0.2, rng, tets=kind == "tet")


@pytest.mark.parametrize("n", [4864, 4865, 40000])
@pytest.mark.parametrize("dist", [0.01, 0.5, 3.0, None])
@pytest.mark.parametrize("kind", ["tet", "hex", "cube", "mixed"])
def test_previous_cells_equal_search(kind, dist, n):
    mesh = _mesh(kind)
    rng = np.random.default_rng(n)
    pos = rng.uniform(0, 15.0, size=(n, 3))
    moved = (rng.uniform(0, 15.0, size=(n, 3)) if dist is None
             else synth.random_displacement(pos, dist, rng, L, BOX["periodic"]))
    sp = torch.zeros(n, dtype=torch.int32, device="cuda")
    a, b = Mesh(mesh, BOX), Mesh(mesh, BOX)
    a.bin(torch.tensor(pos, device="cuda"), sp)
    walked = a.bin(torch.tensor(moved, device="cuda"), sp)
    searched = b.bin(torch.tensor(moved, device="cuda"), sp)
    for x, y in zip(walked, searched):
        assert torch.equal(x, y)
    if n == 4865:
        cell, _ = oracle.locate(oracle.cell_geometry(mesh), BOX, moved)
        np.testing.assert_array_equal(walked[0].cpu().numpy(), cell)
    a.close()
    b.close()
