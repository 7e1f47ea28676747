"""g(r) pair counts against the oracle (whole numbers, equal) over the searches the call
chooses from: the build cells (two and more to each side, rows that wrap, few particles a
cell, several cells a tile, particles moved since the build), the coarse grid and all
pairs; wide and very narrow bins (where every pair is decided by the FP64 rule)."""
import numpy as np
import pytest

import oracle
from inputs import generate as gen
from tests.helpers import mixture, quantized

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


def check(sim, sp, L, nbins, rmax):
    pos, _, _ = sim.get_state()
    _, xfix, k = quantized(pos, L)
    want = oracle.gr_counts(xfix, sp, L, k, nbins, rmax)
    o = sim.observe(bbmd.OBS_GR, nbins=nbins, rmax=rmax)
    assert np.array_equal(o["gr_counts"], want)
    assert np.array_equal(sim.gr_counts_noalloc(nbins, rmax), want)


@pytest.mark.parametrize("ncell", [6, 9, 10, 13])
@pytest.mark.parametrize("nbins,rmax", [(500, 5.0), (1, 2.5), (333, 3.0), (4096, 1.3)])
@pytest.mark.parametrize("prec,mode", [(0, 0), (1, 1)])
def test_counts_after_steps(ncell, nbins, rmax, prec, mode):
    n, L, pos, vel, sp = mixture(ncell, shake=0.1)
    sim = bbmd.Sim(bbmd.ka_params(precision=prec, nbr_mode=mode), n, L, sp, pos, vel)
    sim.step(7, 0.005)  # moved since the last rebuild
    check(sim, sp, L, nbins, rmax)
    sim.close()


@pytest.mark.parametrize("frac_b", [0.0, 0.8])
@pytest.mark.parametrize("rmax", [1.7, 4.0])
def test_counts_with_small_cells(frac_b, rmax):
    # four particles a cell: tiles of eight cells, four cells to each side
    n, L, pos, vel, sp = mixture(11, shake=0.1, frac_b=frac_b)
    p = bbmd.ka_params(potential=bbmd.POT_SOFT, shift=bbmd.SHIFT_FORCE)
    for a in range(2):
        for b in range(2):
            p.rcut[a][b] = 1.2
    sim = bbmd.Sim(p, n, L, sp, pos, vel)
    sim.step(20, 0.001)
    check(sim, sp, L, 400, rmax)
    sim.close()


def test_counts_in_a_ragged_box():
    n0 = 4 * 9 ** 3
    side = gen.box_for(n0, 1.2)
    rng = np.random.default_rng(8)
    pos = np.concatenate([gen.fcc_lattice(9, side) + [k * side, 0.0, 0.0] for k in range(2)])
    keep = np.sort(rng.permutation(2 * n0)[:2 * n0 - 117])
    box = np.array([2 * side, side, side])
    pos = np.mod(pos + rng.uniform(-0.1, 0.1, pos.shape), box)[keep]
    sp = gen.assign_species(len(keep), len(keep) // 3, 4)
    sim = bbmd.Sim(bbmd.ka_params(), len(keep), box, sp, pos, np.zeros_like(pos))
    check(sim, sp, box, 250, 5.0)
    sim.close()


def test_counts_across_the_seam_of_a_long_box():
    # 1071 cells do not fill the long side: a run past the seam is off by the gap they leave
    side = gen.box_for(2048, 1.2)
    rng = np.random.default_rng(12)
    pos = gen.fcc_lattice(8, side) + rng.uniform(-0.1, 0.1, (2048, 3))
    box = np.array([3000.7, 15.1, 15.9])
    pos = np.mod(pos - 0.5 * side, box)
    sp = gen.assign_species(2048, 400, 2)
    sim = bbmd.Sim(bbmd.ka_params(stencil_capacity=2200, block_z=2), 2048, box, sp, pos, np.zeros((2048, 3)))
    check(sim, sp, box, 500, 5.0)
    sim.close()
