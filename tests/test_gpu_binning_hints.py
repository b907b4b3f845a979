"""Re-binning from the previous cells where the FP32 filter cannot decide:
molecules exactly on mesh planes (all of them go to the exact pass, a warp
takes 1 to 32 at a time), and the walk through cells that need not be convex.
The cells must be those of a search without hints, and on an undistorted grid
those of the floor rule (points on a cell's low faces belong to it)."""
import numpy as np
import pytest
import torch

from paper_cs_0702131_gb300 import synth
from paper_cs_0702131_gb300.aica import Mesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 4864, 4865, 9729, 160000])
def test_molecules_on_mesh_planes(n):
    g, w = 8, 2.0                                  # 8^3 cubes of edge 2: planes exactly representable
    L = np.full(3, g * w)
    mesh = synth.hex_mesh((g,) * 3, (0, 0, 0), L, 0.0, np.random.default_rng(0))
    m = Mesh(mesh, dict(L=L, periodic=np.array([1, 1, 1], np.int32)))
    rng = np.random.default_rng(n)
    pos = rng.uniform(0, g * w, size=(n, 3))
    axis = rng.integers(0, 3, n)
    pos[np.arange(n), axis] = w * rng.integers(0, g, n)
    k = np.floor(pos / w).astype(int)
    want = (k[:, 0] * g + k[:, 1]) * g + k[:, 2]
    p = torch.tensor(pos, device="cuda")
    sp = torch.zeros(n, dtype=torch.int32, device="cuda")
    for _ in range(2):                             # without and with previous cells
        cell, order, off = m.bin(p, sp)
        np.testing.assert_array_equal(cell.cpu().numpy(), want)
        np.testing.assert_array_equal(order.cpu().numpy(), np.argsort(want, kind="stable"))
    m.close()


@pytest.mark.parametrize("tets", [False, True])
@pytest.mark.parametrize("dist", [0.05, 0.5, 3.0])
def test_walk_equals_search(tets, dist):
    rng = np.random.default_rng(3)
    L = np.full(3, 16.0)
    mesh = synth.hex_mesh((7, 7, 7), (0, 0, 0), L, 0.2, rng, tets=tets)
    box = dict(L=L, periodic=np.array([1, 1, 1], np.int32))
    pos = rng.uniform(0, 16.0, size=(3000, 3))
    moved = synth.random_displacement(pos, dist, rng, L, box["periodic"])
    sp = torch.zeros(len(pos), dtype=torch.int32, device="cuda")
    a, b = Mesh(mesh, box), Mesh(mesh, box)
    a.bin(torch.tensor(pos, device="cuda"), sp)
    walked = a.bin(torch.tensor(moved, device="cuda"), sp)
    searched = b.bin(torch.tensor(moved, device="cuda"), sp)
    for x, y in zip(walked, searched):
        assert torch.equal(x, y)
    a.close()
    b.close()
