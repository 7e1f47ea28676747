"""Failure detection of the launches that run several phases, without a GPU fault: a wait
limit that cannot be met makes the launch give up.  Every call on the handle then reports
BBMD_ERR_TIMEOUT (and returns, whatever half-done state it looks at), and the device stays
usable: a new handle steps like one made before."""
import numpy as np
import pytest

from tests.helpers import mixture

pytestmark = pytest.mark.gpu

bbmd = pytest.importorskip("paper_1105_5613_gb300.bbmd")

NH = (bbmd.THERMO_NH, 2.0, 2.0, 0.5)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1105_5613_gb300 import build as b

    b.build()
    bbmd.load()


def make(ncell, shape, **kw):
    n, L, pos, vel, sp = mixture(ncell, shake=0.1)
    return bbmd.Sim(bbmd.ka_params(block_z=shape, **kw), n, L, sp, pos, vel)


def every_call_times_out(sim, mode=bbmd.NBR_VERLET):
    ids = np.arange(0, sim.n, 7)
    calls = [lambda: sim.observe(bbmd.OBS_ENERGY | bbmd.OBS_VIRIAL), lambda: sim.observe(bbmd.OBS_GR, nbins=100),
             lambda: sim.get_forces(energies=True), lambda: sim.get_forces_ids(ids), sim.get_state,
             lambda: sim.step_profiled(3, 0.005, NH), lambda: sim.minimize(5)]
    if mode == bbmd.NBR_VERLET:
        calls.append(sim.get_neighbors)
    for _ in range(2):
        for f in calls:
            with pytest.raises(bbmd.BBMDError) as e:
                f()
            assert e.value.code == 7  # BBMD_ERR_TIMEOUT
        sim.step(300, 0.005, NH)  # (asynchronous)


def still_works(ncell, shape, want, **kw):
    sim = make(ncell, shape, **kw)
    sim.step(30, 0.005, NH)
    for x, y in zip(sim.get_state(), want):
        assert np.array_equal(x, y)
    sim.close()


# one launch for many steps (four and eight warps a block, list and cell mode); the captured
# step, whose trigger and sort chain are one launch (mixed and FP64)
@pytest.mark.parametrize("ncell,shape,kw", [(10, 1, {}), (16, 4, {}), (16, 8, {"nbr_mode": bbmd.NBR_CELL}),
                                            (17, 1, {}), (36, 1, {}),
                                            (14, 2, {"precision": bbmd.PREC_FP64})])
def test_a_barrier_wait_that_runs_out(ncell, shape, kw):
    ref = make(ncell, shape, **kw)
    ref.step(30, 0.005, NH)
    want = ref.get_state()
    ref.close()
    sim = make(ncell, shape, **kw)
    with pytest.raises(bbmd.BBMDError) as e:
        sim.set_wait_limits(barrier_ns=0)
    assert e.value.code == 1  # BBMD_ERR_ARG
    sim.step(5, 0.005, NH)
    sim.set_wait_limits(barrier_ns=1)
    sim.step(400, 0.005, NH)
    mode = kw.get("nbr_mode", bbmd.NBR_VERLET)
    every_call_times_out(sim, mode)
    sim.set_wait_limits()  # a longer limit does not bring the state back
    every_call_times_out(sim, mode)
    sim.close()
    still_works(ncell, shape, want, **kw)


@pytest.mark.parametrize("ncell,shape", [(10, 1), (16, 4), (36, 1)])
def test_a_barrier_wait_of_a_descent_that_runs_out(ncell, shape):
    sim = make(ncell, shape)
    sim.set_wait_limits(barrier_ns=1)
    with pytest.raises(bbmd.BBMDError) as e:
        sim.minimize(50)
    assert e.value.code == 7
    every_call_times_out(sim)
    sim.close()
