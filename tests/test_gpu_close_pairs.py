"""FP64 forces, energy and virial of two molecules at any distance, near the
cluster's origin and far from it, against exact rational arithmetic.

Along one axis r^2 carries one rounding (u = 2^-53), its reciprocal two, so
r^-6 at most 11 u: with h = A / r^12 and l = B / r^6 the force f = (h - l) / r
rounds to within 20 u |f| + 16 u (h + l) / r, the energy likewise, and the virial
r f one u more."""
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_cs_0702131_gb300 import synth
from paper_cs_0702131_gb300.aica import Mesh

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def mesh():
    L = np.full(3, 12.0)
    m = Mesh(synth.hex_mesh((4, 4, 4), (0, 0, 0), L, 0.0, np.random.default_rng(0)),
             dict(L=L, periodic=np.array([1, 1, 1], np.int32)))
    m.build_lists(2.5, 1e-3)
    assert m.get_option("cluster_path") == 1
    yield m
    m.close()


def _check(m, x, eps=1.0, sigma=1.0):
    r = Fraction(x[0][0]) - Fraction(x[1][0])              # along x
    pos = torch.tensor(x, dtype=torch.float64, device="cuda")
    m.bin(pos, torch.zeros(2, dtype=torch.int32, device="cuda"))
    F, ev, cnt = m.forces(np.array([eps]), np.array([sigma]), "fp64")
    F, ev = F.cpu().numpy(), ev.cpu().numpy()
    assert int(cnt[3:].sum()) == 1
    s6 = (Fraction(sigma) / r) ** 6
    h, l = 48 * Fraction(eps) * s6 * s6, 24 * Fraction(eps) * s6
    f, u = (h - l) / r, (h - 2 * l) / 12
    tol_f = Fraction(U) * (20 * abs(f) + 16 * (h + l) / r)
    tol_u = Fraction(U) * (20 * abs(u) + 16 * (h + 2 * l) / 12)
    for i, s in ((0, 1), (1, -1)):
        assert abs(Fraction(F[i, 0]) - s * f) <= tol_f, float(r)
        assert F[i, 1] == 0 and F[i, 2] == 0
    assert abs(Fraction(ev[0]) - u) <= tol_u, float(r)
    assert abs(Fraction(ev[1]) - r * f) <= r * (tol_f + Fraction(U) * abs(f)), float(r)
    assert not ev[2:].any()


@pytest.mark.parametrize("exp", [-60, -52, -51, -50, -49, -40, -20, -10, -5, -2, -1, 0, 1])
def test_at_the_origin(mesh, exp):
    """From r^2 = 2^-120 to 4: both sides of the range in which the reciprocal
    starts from FP32 (2^-100)."""
    for mant in (1.0, 1.2345678901234567, 1.9999999999999998):
        r = mant * 2.0 ** exp
        if r < 2.5:
            _check(mesh, [[r, 0.0, 0.0], [0.0, 0.0, 0.0]])


@pytest.mark.parametrize("exp", [-40, -30, -20, -12, -8, -5, -4, -3, -2, -1, 0])
@pytest.mark.parametrize("at", [1.5, 5.75, 9.25])
def test_far_from_the_origin(mesh, at, exp):
    """The virial of a pair is r x F also where the molecules' coordinates are
    much larger than r."""
    _check(mesh, [[at + 1.25 * 2.0 ** exp, 2.0, 2.5], [at, 2.0, 2.5]])
