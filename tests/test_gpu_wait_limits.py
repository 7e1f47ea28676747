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


def moved_at_most(sim, pos, L, dist):
    """The positions on the device (get_state fills its arrays whatever status it returns)."""
    now = np.empty_like(pos)
    dp = bbmd.C.POINTER(bbmd.C.c_double)
    rc = bbmd.load().bbmd_get_state(sim.h, now.ctypes.data_as(dp), None, None)
    assert rc == 7  # BBMD_ERR_TIMEOUT
    d = now - pos
    d -= L * np.round(d / L)
    return np.abs(d).max() <= dist


# a staging wait that gives up ends the launch of many steps: none is taken on old forces
@pytest.mark.parametrize("ncell,shape,kw", [(10, 1, {}), (16, 4, {}), (16, 2, {"nbr_mode": bbmd.NBR_CELL})])
def test_a_staging_wait_that_gives_up(ncell, shape, kw):
    ref = make(ncell, shape, **kw)
    ref.step(30, 0.005, NH)
    want = ref.get_state()
    ref.close()
    sim = make(ncell, shape, **kw)
    pos, vel, _ = sim.get_state()
    L = mixture(ncell)[1]
    mode = kw.get("nbr_mode", bbmd.NBR_VERLET)
    sim.set_wait_limits(staging_tries=0)
    sim.step(400, 0.005)
    assert moved_at_most(sim, pos, L, 2 * 0.005 * 2 * np.abs(vel).max())
    every_call_times_out(sim, mode)
    sim.close()
    sim = make(ncell, shape, **kw)
    sim.set_wait_limits(staging_tries=0)
    with pytest.raises(bbmd.BBMDError) as e:
        sim.minimize(400, 1e-3, 0.05)
    assert e.value.code == 7
    assert moved_at_most(sim, pos, L, 2 * 0.05)
    sim.close()
    still_works(ncell, shape, want, **kw)


def test_a_staging_wait_of_a_replica_that_gives_up():
    sys = [mixture(m, shake=0.1) for m in (8, 9, 10)]
    ns, boxes, pos, vel, sp = zip(*sys)
    b = bbmd.Batch(bbmd.ka_params(), ns, boxes, sp, pos, vel)
    assert b.uses_persistent()
    b.step(3, 0.005)
    b.replica(1).set_wait_limits(staging_tries=0)
    b.step(400, 0.005)
    for r in range(3):
        with pytest.raises(bbmd.BBMDError) as e:
            b.replica(r).observe(0)
        assert e.value.code == 7, r
    v = np.abs(vel[1]).max()
    start = bbmd.Sim(bbmd.ka_params(block_z=4), ns[1], boxes[1], sp[1], pos[1], vel[1])
    start.step(3, 0.005)
    p3, _, _ = start.get_state()
    start.close()
    assert moved_at_most(b.replica(1), p3, boxes[1], 2 * 0.005 * 2 * v)
    b.close()
