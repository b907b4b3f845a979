"""Calls in turn on one mesh: each leaves the accumulators, sums and counters
that the next one starts from, so precision, kernel, refinement, adjoint,
molecule number, failed and deferred binnings and replayed graphs alternate here.

Tolerances are those of the force and adjoint tests: forces 1e-12 (FP64) or
1e-5 (FP32) of max(|F_ic|, ||F_i||), energy 1e-12 / 1e-6 of the sum of
magnitudes, FP64 position gradients 1e-10 of the largest; counts are equal."""
import numpy as np
import pytest
import torch

import oracle
from oracle import torch_ref
from paper_cs_0702131_gb300 import synth
from paper_cs_0702131_gb300.aica import AicaError
from gpu_helpers import assert_forces, gpu_setup

pytestmark = pytest.mark.gpu


def _fluid(hexes, tets, seed=3):
    rng = np.random.default_rng(seed)
    a = synth.A_FCC_08
    L = np.full(3, 6 * a)
    box = dict(L=L, periodic=np.array([1, 1, 1], np.int32))
    pos = synth.wrap(synth.jitter(synth.fcc_sites(6, 6, 6, a), 0.05, rng), L, box["periodic"])
    pos = pos[rng.permutation(len(pos))]
    mesh = synth.hex_mesh((hexes,) * 3, (0, 0, 0), L, 0.15, rng, tets=tets)
    sp = (np.arange(len(pos)) % 2).astype(np.int32)
    return dict(pos=pos, species=sp, eps=np.array([1.0, 1.5]), sigma=np.array([1.0, 0.88]), rc=2.5, box=box,
                mesh=mesh, skin=1e-3)


def _bin(m, c, n):
    m.bin(torch.tensor(c["pos"][:n], device="cuda"), torch.tensor(c["species"][:n], device="cuda"))


def _check(out, ref, prec):
    F, ev, cnt = out
    assert_forces(F.double().cpu().numpy(), ref, 1e-12 if prec == "fp64" else 1e-5)
    assert abs(float(ev[0]) - ref["U"]) <= (1e-12 if prec == "fp64" else 1e-6) * ref["Uabs"]
    assert int(cnt[3:6].sum()) == ref["pairs"]


@pytest.mark.parametrize("hexes,tets", [(3, False), (5, True)])   # cells of 32 molecules (bin_cells), of 1.4 (bin_slots)
def test_calls_in_turn(hexes, tets):
    c = _fluid(hexes, tets)
    m, *_ = gpu_setup(c)
    N = len(c["pos"])
    refs = {n: oracle.lj(c["pos"][:n], c["species"][:n], c["eps"], c["sigma"], c["rc"], c["box"]) for n in (N, N - 301)}
    rng = np.random.default_rng(5)
    v = rng.standard_normal((N, 3))
    gp_ref = torch_ref.vjp(c["pos"], c["species"], c["eps"], c["sigma"], c["rc"], c["box"], v)[0]
    refined = None
    for n in (N, N - 301, N):
        _bin(m, c, n)
        for prec, opt, val in (("fp32", None, 0), ("fp64", None, 0), ("fp32", "fp32_kernel", 1), ("fp32", None, 0),
                               ("fp32", "fp32_refine_tol", 0.0), ("fp64", None, 0), ("fp32", None, 0)):
            old = m.get_option(opt) if opt else None
            if opt:
                m.set_option(opt, val)
            out = m.forces(c["eps"], c["sigma"], prec)
            if opt is None:
                _check(out, refs[n], prec)
            if opt is None and prec == "fp32" and n == N:
                refined = m.get_option("refined") if refined is None else refined
                assert abs(m.get_option("refined") - refined) <= 0.02 * refined + 2   # last bits of FP32 sums
            if opt:
                m.set_option(opt, old)
            if n == N:
                gp = m.forces_backward(c["eps"], c["sigma"], torch.tensor(v, device="cuda"), "fp64")[0].cpu().numpy()
                assert np.abs(gp - gp_ref).max() <= 1e-10 * np.abs(gp_ref).max()
    bad = torch.tensor(c["species"], device="cuda")
    bad[17] = 99
    for _ in range(2):                # an error, then the same call without it
        with pytest.raises(AicaError):
            m.bin(torch.tensor(c["pos"], device="cuda"), bad)
        _bin(m, c, N)
        _check(m.forces(c["eps"], c["sigma"]), refs[N], "fp32")
    m.set_deferred(True)              # an error that nobody asked for must not reach the next checked call
    m.bin(torch.tensor(c["pos"], device="cuda"), bad)
    m.set_deferred(False)
    _bin(m, c, N)
    _check(m.forces(c["eps"], c["sigma"], "fp64"), refs[N], "fp64")
    m.close()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_replayed_graph_and_eager_calls(prec):
    c = _fluid(5, True)
    m, *_ = gpu_setup(c)
    N = len(c["pos"])
    ref = oracle.lj(c["pos"], c["species"], c["eps"], c["sigma"], c["rc"], c["box"])
    pos, sp = torch.tensor(c["pos"], device="cuda"), torch.tensor(c["species"], device="cuda")
    m.set_deferred(True)
    out = m.forces(c["eps"], c["sigma"], prec)      # also allocates
    m.bin(pos, sp, outputs=False)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        m.bin(pos, sp, outputs=False)
        m.forces(c["eps"], c["sigma"], prec, out=out[0], ev=out[1], counts=out[2])
    for other in ("fp64", "fp32"):
        for _ in range(2):
            for t in out:
                t.fill_(-7)
            g.replay()
            torch.cuda.synchronize()
            _check(out, ref, prec)
        _check(m.forces(c["eps"], c["sigma"], other), ref, other)
    m.check()
    del g
    m.close()
