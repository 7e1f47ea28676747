"""Energies in cell mode of a state whose density varies: a dense cube in a thin gas fits the
staged region of the forces' block shape (36 x 4 or 16 x 6 cells at the mean density) but not
the smaller region that the energy pass prefers (4 x 4 x 4 cells).  Bars as in
test_gpu_parity: u_i 1e-9 and potential energy 1e-10 relative."""
import numpy as np
import pytest

import oracle
from inputs import generate as gen
from tests.helpers import oracle_params, quantized

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


def cube_in_gas(cells, m, spacing):
    """An FCC cube of 4 m^3 particles at density 1.2 in the middle of a box of `cells` cells a
    side, and a simple cubic gas of about the given spacing around it."""
    L = cells * 2.81
    side = gen.box_for(4 * m ** 3, 1.2)
    rng = np.random.default_rng(1)
    cube = gen.fcc_lattice(m, side) + 0.5 * (L - side) + rng.uniform(-0.05, 0.05, (4 * m ** 3, 3))
    g = int(round(L / spacing))
    gas = (np.stack(np.meshgrid(*[np.arange(g)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.5) * (L / g)
    gas = gas[np.abs(gas - 0.5 * L).max(1) > 0.5 * side + 0.9]
    return np.concatenate([cube, gas]), L


@pytest.mark.parametrize("shape,spacing", [(8, 1.6), (8, 1.5), (4, 1.5), (0, 1.6), (0, 1.5)])
def test_energies_of_a_state_beyond_the_smaller_region(shape, spacing):
    pos, L = cube_in_gas(8, 7, spacing)
    n = len(pos)
    sp = (np.arange(n) % 5 == 0).astype(np.uint8)
    p = bbmd.ka_params(nbr_mode=bbmd.NBR_CELL, block_z=shape)
    sim = bbmd.Sim(p, n, L, sp, pos, np.zeros_like(pos))
    assert sim.info()["block_z"] in (4, 8)
    xq, _, _ = quantized(pos, L)
    _, uo, _, PEo = oracle.forces(xq, sp, L, oracle_params(p), "cells")
    for _ in range(2):
        assert abs(sim.observe(bbmd.OBS_ENERGY)["pe"] - PEo) <= 1e-10 * np.abs(uo).sum()
        _, u = sim.get_forces(energies=True)
        assert np.abs(u - uo).max() <= 1e-9 * max(1.0, np.abs(uo).max())
    sim.close()


def test_energies_first_asked_for_per_particle():
    pos, L = cube_in_gas(8, 7, 1.5)
    n = len(pos)
    sp = np.zeros(n, np.uint8)
    p = bbmd.ka_params(nbr_mode=bbmd.NBR_CELL, block_z=8)
    sim = bbmd.Sim(p, n, L, sp, pos, np.zeros_like(pos))
    xq, _, _ = quantized(pos, L)
    uo = oracle.forces(xq, sp, L, oracle_params(p), "cells")[1]
    _, u = sim.get_forces(energies=True)
    assert np.abs(u - uo).max() <= 1e-9 * max(1.0, np.abs(uo).max())
    sim.close()
