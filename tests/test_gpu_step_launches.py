"""Kernels counted per step: one launch for all steps of a small system; six a captured step
(integrate, trigger and sort, list build, two force kernels, finalize); fifteen with a launch
per sort kernel."""
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


@pytest.mark.parametrize("ncell,first,per_step", [(10, 2, 0), (36, 1, 6), (64, 1, 15)])
def test_launches_per_step(ncell, first, per_step):
    n = 4 * ncell ** 3
    L = mixture(6)[1] * ncell / 6
    sim = bbmd.Sim(bbmd.ka_params(block_z=1), n, L, np.zeros(n, np.uint8), None, None, T0=1.0)
    assert sim.step_launches() == 0
    sim.step(12, 0.005)
    assert sim.step_launches() == first + 12 * per_step
    sim.close()
