"""Error bits and the largest species after a replayed graph.  A captured
(deferred) binning writes the device's flag words without a host call; the
checked calls that follow must report what it flagged, and the next checked
binning must start from clean words."""
import numpy as np
import pytest
import torch

import oracle
from paper_cs_0702131_gb300 import synth
from paper_cs_0702131_gb300.aica import AicaError, Mesh
from gpu_helpers import assert_forces

pytestmark = pytest.mark.gpu

EPS, SIGMA = np.array([1.0, 1.5]), np.array([1.0, 0.88])


@pytest.fixture(params=[False, True], ids=["hex", "tet"])
def captured(request):
    """A mesh open along z, good molecules, and a captured binning of the buffers."""
    rng = np.random.default_rng(11)
    a = synth.A_FCC_08
    L = np.full(3, 5 * a)
    box = dict(L=L, periodic=np.array([1, 1, 0], np.int32))
    x = synth.jitter(synth.fcc_sites(5, 5, 5, a), 0.05, rng)
    x[:, 2] = np.clip(x[:, 2], 0.01, L[2] - 0.01)
    x = synth.wrap(x, L, box["periodic"])
    m = Mesh(synth.hex_mesh((4, 4, 4), (0, 0, 0), L, 0.15, rng, tets=request.param), box)
    m.build_lists(2.5, 1e-3)
    good = torch.tensor(x, device="cuda")
    pos, sp = good.clone(), torch.zeros(len(x), dtype=torch.int32, device="cuda")
    m.bin(pos, sp)
    m.set_deferred(True)
    m.bin(pos, sp, outputs=False)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        m.bin(pos, sp, outputs=False)
    m.set_deferred(False)
    ref = oracle.lj(x, np.zeros(len(x), np.int32), EPS[:1], SIGMA[:1], 2.5, box)
    yield m, g, pos, sp, good, ref
    del g
    m.close()


def _good_call(m, good, ref):
    m.bin(good, torch.zeros(len(good), dtype=torch.int32, device="cuda"))
    F, _, cnt = m.forces(EPS[:1], SIGMA[:1], "fp64")
    assert_forces(F.cpu().numpy(), ref, 1e-12)
    assert int(cnt[3:].sum()) == ref["pairs"]


@pytest.mark.parametrize("call", ["forces", "backward", "bin"])
def test_molecule_outside_in_a_replay(captured, call):
    m, g, pos, sp, good, ref = captured
    for _ in range(2):
        _good_call(m, good, ref)
        pos[17, 2] = -1.0                        # outside the mesh
        g.replay()
        torch.cuda.synchronize()
        pos[17, 2] = good[17, 2]
        if call == "forces":
            with pytest.raises(AicaError):
                m.forces(EPS[:1], SIGMA[:1], "fp64")
        elif call == "backward":
            with pytest.raises(AicaError):
                m.forces_backward(EPS[:1], SIGMA[:1], torch.ones_like(good), "fp64")
        _good_call(m, good, ref)                 # the replay's error is not this call's
    m.check()


def test_species_of_a_replay(captured):
    m, g, pos, sp, good, ref = captured
    for bad in (1, 99):                          # more species than the next call has; out of range
        _good_call(m, good, ref)
        sp[3] = bad
        g.replay()
        torch.cuda.synchronize()
        sp[3] = 0
        _good_call(m, good, ref)


def test_check_reports_a_replay_once(captured):
    m, g, pos, sp, good, ref = captured
    _good_call(m, good, ref)
    pos[17, 2] = -1.0
    g.replay()
    torch.cuda.synchronize()
    pos[17, 2] = good[17, 2]
    with pytest.raises(AicaError):
        m.check()
    m.check()
    m.forces(EPS[:1], SIGMA[:1], "fp64")
    _good_call(m, good, ref)
