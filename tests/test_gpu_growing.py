"""Binnings of a growing number of molecules: buffers grow between calls, and
words that the calls hand on as zero must be zero in the new buffers too."""
import numpy as np
import pytest
import torch

from paper_cs_0702131_gb300 import synth
from paper_cs_0702131_gb300.aica import Mesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("deferred", [False, True])
def test_growing_binnings(deferred):
    g, w = 6, 2.0
    L = np.full(3, g * w)
    m = Mesh(synth.hex_mesh((g,) * 3, (0, 0, 0), L, 0.0, np.random.default_rng(0)),
             dict(L=L, periodic=np.array([1, 1, 1], np.int32)))
    m.set_deferred(deferred)
    rng = np.random.default_rng(1)
    for n in (1, 2, 100, 129, 300, 1000, 1023, 1024, 1025, 5000, 70000, 300000, 7):
        for _ in range(2):                     # without and with previous cells
            x = rng.uniform(0, g * w, size=(n, 3))
            k = np.floor(x / w).astype(int)
            want = (k[:, 0] * g + k[:, 1]) * g + k[:, 2]
            cell, order, off = m.bin(torch.tensor(x, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda"))
            np.testing.assert_array_equal(cell.cpu().numpy(), want)
            np.testing.assert_array_equal(order.cpu().numpy(), np.argsort(want, kind="stable"))
            assert int(off[-1]) == n
    m.check()
    m.close()
