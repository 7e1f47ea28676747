"""FP64 pair kernels (the FP64 form and the energy passes of both precisions) where their
FP32 classification, queues and half-pair sums can go wrong: coarse position units (a long
box), three cells per axis (a region that holds a cell twice), ragged sizes, every block
shape, with and without a stored list.  Bars as in test_gpu_parity: forces of the FP64 form
1e-10, u_i 1e-9, potential energy 1e-10 and virial 1e-6 relative."""
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


def clump(n, box, seed):
    """n particles of a shaken FCC lump (density about 1.2) across the x seam of box."""
    m = 6
    side = gen.box_for(4 * m ** 3, 1.2)
    rng = np.random.default_rng(seed)
    pos = gen.fcc_lattice(m, side) + rng.uniform(-0.1, 0.1, (4 * m ** 3, 3))
    pos = pos[rng.choice(4 * m ** 3, n, replace=False)]
    pos[:, 0] -= 0.5 * side
    return np.mod(pos, box), gen.assign_species(n, n // 5, seed)


@pytest.mark.parametrize("box,n,shape", [
    ((300000.0, 9.0, 9.0), 864, 1),   # position unit 2^-43: upper words of 2^-11
    ((300000.0, 11.3, 9.0), 337, 2),
    ((9.0, 9.0, 9.0), 864, 1),        # three cells per axis
    ((9.0, 9.0, 9.0), 33, 2),
    ((12.1, 9.0, 11.7), 861, 4),
    ((12.1, 12.3, 9.0), 863, 8),
])
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("pot,shift", [(0, 1), (1, 2)])
@pytest.mark.parametrize("prec", [0, 1])
def test_fp64_pass_against_brute_force(box, n, shape, mode, pot, shift, prec):
    box = np.array(box)
    pos, sp = clump(n, box, 5 * n + shape)
    # (a staged region may hold every particle, some of them several times; the mean density
    # does not tell that of the lump)
    p = bbmd.ka_params(precision=prec, potential=pot, shift=shift, nbr_mode=mode, block_z=shape,
                       stencil_capacity=3 * n + 64)
    sim = bbmd.Sim(p, n, box, sp, pos, np.zeros((n, 3)))
    # the oracle gets the same lump moved to the origin: near x = 3e5 a double does not hold a
    # 61-bit position
    _, xfix, k = quantized(pos, box)
    move = np.ldexp([5.0, 0.0, 0.0], k).astype(np.int64)
    xq = oracle.dequantize((xfix + move) % np.ldexp(box, k).astype(np.int64), k)
    Fo, uo, Wo, PEo = oracle.forces(xq, sp, box, oracle_params(p))
    F, u = sim.get_forces(energies=True)
    assert np.abs(u - uo).max() <= 1e-9 * max(1.0, np.abs(uo).max())
    if prec == bbmd.PREC_FP64:
        rel = np.linalg.norm(F - Fo, axis=1) / np.maximum(np.linalg.norm(Fo, axis=1), 1e-3)
        assert rel.max() <= 1e-10, rel.max()
    o = sim.observe(bbmd.OBS_ENERGY | bbmd.OBS_VIRIAL)
    assert abs(o["pe"] - PEo) <= 1e-10 * np.abs(uo).sum()
    assert abs(o["virial"] - Wo) <= 1e-6 * abs(Wo)
    again = sim.observe(bbmd.OBS_ENERGY | bbmd.OBS_VIRIAL)
    assert again["pe"] == o["pe"] and again["virial"] == o["virial"]
    sim.close()
