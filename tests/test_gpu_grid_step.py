"""The one-launch step and steepest descent of small systems against the phase-by-phase
launches: bit for bit the same states, from three cells per axis to just past the size
where every block has a CTA of its own; two handles stepping from two threads at once."""
import threading

import numpy as np
import pytest

from tests.helpers import mixture

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


def make(ncell, shape, shift=1, mode=0, shake=0.12, **kw):
    n, L, pos, vel, sp = mixture(ncell, shake=shake)
    p = bbmd.ka_params(block_z=shape, shift=shift, nbr_mode=mode, **kw)
    return bbmd.Sim(p, n, L, sp, pos, vel)


# step_profiled launches every phase on its own: the same steps
@pytest.mark.parametrize("ncell,shape", [(6, 1), (6, 2), (10, 1), (10, 4), (16, 8), (17, 1), (21, 2),
                                         (30, 4), (33, 8)])
@pytest.mark.parametrize("thermo", [None, (bbmd.THERMO_NH, 2.0, 1.5, 0.5)])
@pytest.mark.parametrize("shift,mode", [(1, 0), (2, 1)])
def test_step_equals_phase_launches(ncell, shape, thermo, shift, mode):
    a, b = make(ncell, shape, shift, mode), make(ncell, shape, shift, mode)
    for k in (1, 23):
        a.step(k, 0.005, thermo)
        b.step_profiled(k, 0.005, thermo)
        for x, y in zip(a.get_state(), b.get_state()):
            assert np.array_equal(x, y)
    oa, ob = a.observe(bbmd.OBS_ENERGY), b.observe(bbmd.OBS_ENERGY)
    assert oa["n_rebuilds"] == ob["n_rebuilds"] > 1 and oa["step"] == ob["step"] == 24
    assert oa["ke"] == ob["ke"] and oa["xi"] == ob["xi"] and oa["pe"] == ob["pe"]
    a.close()
    b.close()


@pytest.mark.parametrize("ncell,shape,kw", [(36, 1, {}), (36, 4, {"mode": 1}),
                                            (10, 2, {"precision": bbmd.PREC_FP64}),
                                            (14, 8, {"precision": bbmd.PREC_FP64, "mode": 1})])
def test_captured_step_equals_phase_launches(ncell, shape, kw):
    # past one wave of blocks, and the FP64 form: one launch per phase, trigger and sort chain
    # as one
    a, b = make(ncell, shape, **kw), make(ncell, shape, **kw)
    a.step(24, 0.005, (bbmd.THERMO_NH, 2.0, 1.5, 0.5))
    b.step_profiled(24, 0.005, (bbmd.THERMO_NH, 2.0, 1.5, 0.5))
    for x, y in zip(a.get_state(), b.get_state()):
        assert np.array_equal(x, y)
    oa, ob = a.observe(0), b.observe(0)
    assert oa["n_rebuilds"] == ob["n_rebuilds"] > 1 and oa["xi"] == ob["xi"]
    a.close()
    b.close()


def test_cut_lists_fall_back_and_grow():
    # lists that hold the lattice but not the liquid: forces come from the stencil until the
    # next synchronising call grows them
    a, b = (make(10, 1, shake=0.0, list_capacity=88) for _ in range(2))
    for _ in range(3):
        a.step(20, 0.005)
        b.step_profiled(20, 0.005)
        assert np.array_equal(a.get_state()[0], b.get_state()[0])
    a.close()
    b.close()


@pytest.mark.parametrize("ncell,shape", [(6, 2), (10, 1), (16, 4)])
def test_minimize_lowers_the_energy_like_single_calls(ncell, shape):
    # one call of 40 steps = 40 calls of one step (each ends with the forces)
    a, b = make(ncell, shape, shake=0.25), make(ncell, shape, shake=0.25)
    e0 = a.observe(bbmd.OBS_ENERGY)["pe"]
    a.minimize(40, 1e-3, 0.05)
    for _ in range(40):
        b.minimize(1, 1e-3, 0.05)
    assert np.array_equal(a.get_state()[0], b.get_state()[0])
    oa, ob = a.observe(bbmd.OBS_ENERGY), b.observe(bbmd.OBS_ENERGY)
    assert oa["pe"] == ob["pe"] < e0 and oa["n_rebuilds"] == ob["n_rebuilds"] > 1
    a.minimize(0, 1e-3, 0.05)
    assert np.array_equal(a.get_state()[0], b.get_state()[0])
    a.close()
    b.close()


def test_two_handles_from_two_threads():
    sims = [make(17, 1), make(20, 1)]
    ref = [make(17, 1), make(20, 1)]
    for s in ref:
        s.step(400, 0.005)
    want = [s.get_state() for s in ref]
    threads = [threading.Thread(target=lambda s=s: [s.step(40, 0.005) for _ in range(10)]) for s in sims]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for s, w in zip(sims, want):
        for x, y in zip(s.get_state(), w):
            assert np.array_equal(x, y)
    for s in sims + ref:
        s.close()
