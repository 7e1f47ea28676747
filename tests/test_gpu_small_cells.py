"""Neighbour search with few particles a cell (a short cutoff): a group of 32 staged
candidates then reaches past its row of cells, into the lane's own."""
import numpy as np
import pytest

import oracle
from tests.helpers import force_errors, mixture, oracle_params, quantized

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


@pytest.mark.parametrize("shape", [1, 2, 4, 8])
@pytest.mark.parametrize("frac_b", [0.0, 0.2, 0.8])
def test_lists_and_forces_with_small_cells(frac_b, shape):
    n, L, pos, vel, sp = mixture(11, shake=0.2, frac_b=frac_b)
    p = bbmd.ka_params(potential=bbmd.POT_SOFT, shift=bbmd.SHIFT_FORCE, block_z=shape)
    for a in range(2):
        for b in range(2):
            p.rcut[a][b] = 1.2
    xq, xfix, k = quantized(pos, L)
    po = oracle_params(p)
    sim = bbmd.Sim(p, n, L, sp, pos, vel)
    off, nbr = sim.get_neighbors()
    offo, nbro = oracle.neighbors(xfix, sp, L, k, oracle.list_R2(po, 0.3), "cells", rcell=1.5)
    assert np.array_equal(off, offo) and np.array_equal(nbr, nbro)
    sim.close()
    p.nbr_mode = bbmd.NBR_CELL
    sim = bbmd.Sim(p, n, L, sp, pos, vel)
    e = force_errors(sim.get_forces(), oracle.forces(xq, sp, L, po, "cells")[0])
    assert np.median(e) <= 1e-5 and e.max() <= 1e-4, (np.median(e), e.max())
    sim.close()
