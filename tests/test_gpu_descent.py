"""Steepest descent against its definition, one step at a time: x + h F with the forces that
the force kernels of their own give at the same state (get_forces).  One launch with several
blocks to a CTA (more blocks than resident CTAs), the launches per step of large systems, and
the FP64 form.  And two captured steps, each with a launch that fills the GPU, at once."""
import threading

import numpy as np
import pytest

import oracle
from tests.helpers import mixture, oracle_params, quantized

pytestmark = pytest.mark.gpu

bbmd = pytest.importorskip("paper_1105_5613_gb300.bbmd")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1105_5613_gb300 import build as b

    b.build()
    bbmd.load()


def make(ncell, shape, shake=0.12, **kw):
    n, L, pos, vel, sp = mixture(ncell, shake=shake)
    return bbmd.Sim(bbmd.ka_params(block_z=shape, **kw), n, L, sp, pos, vel), n, L, sp


# 186 624 particles in 2 x 2 x 1 blocks: 1900 blocks, at most 608 resident CTAs; 55 296 in
# 4 x 4 x 2: one wave; 530 604: beyond the one-launch descent
@pytest.mark.parametrize("ncell,shape,kw", [(36, 1, {}), (36, 2, {"nbr_mode": bbmd.NBR_CELL}), (24, 8, {}),
                                            (51, 4, {}), (10, 2, {"precision": bbmd.PREC_FP64}),
                                            (14, 8, {"precision": bbmd.PREC_FP64, "nbr_mode": bbmd.NBR_CELL})])
def test_a_step_follows_the_forces(ncell, shape, kw):
    sim, n, L, sp = make(ncell, shape, **kw)
    # positions come as doubles of 61-bit integers: half a unit in the last place of each read
    tol = 2 * np.spacing(L)
    before = sim.observe(0)["n_rebuilds"]
    for k in range(12):
        hmax, dmax = (1e-5, 10.0) if k % 2 else (1.0, 0.08)
        F = sim.get_forces()
        x0, _, i0 = sim.get_state()
        sim.minimize(1, hmax, dmax)
        x1, _, i1 = sim.get_state()
        h = hmax
        err = tol
        fm = float(np.sqrt(np.square(F.astype(np.float32)).sum(1).max()))  # (taken in FP32)
        if dmax / fm < hmax:
            h = dmax / fm
            err = tol + 1e-6 * dmax
        step = (x1 + i1 * L) - (x0 + i0 * L)
        assert np.abs(step - h * F).max() <= err + 4 * np.spacing(np.abs(i1 * L).max()), k
    assert sim.observe(0)["n_rebuilds"] > before
    if n < 200000:
        # the lists of the descent's rebuilds miss no pair: FP64 energies from them
        xq, _, _ = quantized(sim.get_state()[0], L)
        uo = oracle.forces(xq, sp, L, oracle_params(bbmd.ka_params()), "cells")[1]
        _, u = sim.get_forces(energies=True)
        assert np.abs(u - uo).max() <= 1e-9 * max(1.0, np.abs(uo).max())
    sim.close()


@pytest.mark.parametrize("ncell,shape,kw", [(36, 1, {}), (36, 1, {"nbr_mode": bbmd.NBR_CELL}),
                                            (10, 2, {"precision": bbmd.PREC_FP64})])
def test_one_call_equals_single_steps(ncell, shape, kw):
    a, b = make(ncell, shape, **kw)[0], make(ncell, shape, **kw)[0]
    a.minimize(25, 1e-3, 0.05)
    for _ in range(25):
        b.minimize(1, 1e-3, 0.05)
    for x, y in zip(a.get_state(), b.get_state()):
        assert np.array_equal(x, y)
    assert a.observe(0)["n_rebuilds"] == b.observe(0)["n_rebuilds"] > 1
    a.close()
    b.close()


def test_two_captured_steps_at_once():
    def pair():
        return [make(36, 1, 0.1)[0], make(34, 2, 0.1, precision=bbmd.PREC_FP64)[0]]

    def run(s):
        for _ in range(10):
            s.step(12, 0.005)

    ref, sims = pair(), pair()
    for s in ref:
        run(s)
    threads = [threading.Thread(target=run, args=(s,)) for s in sims]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for s, r in zip(sims, ref):
        for x, y in zip(s.get_state(), r.get_state()):
            assert np.array_equal(x, y)
        assert s.observe(0)["n_rebuilds"] == r.observe(0)["n_rebuilds"] > 5
    for s in sims + ref:
        s.close()
