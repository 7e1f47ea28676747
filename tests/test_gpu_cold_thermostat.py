"""Kinetic energy of very cold particles in the Nose-Hoover step: a chunk of 32 is summed
exactly and rounded once, to 2^-32.  512 particles, one to a cell and out of each other's
reach, every one with 4.499 x 2^-40: 32 of them are 0.56 units of 2^-32, where values
rounded to 2^-40 one by one would make half a unit."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("units", [4.499, 4.45, 0.3, 1.0])
def test_kinetic_energy_of_a_cold_chunk(units):
    cells, side = 8, 2.81
    L = cells * side
    g = np.arange(cells)
    pos = (np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3) + 0.5) * side
    n = len(pos)
    vel = np.zeros((n, 3))
    vel[:, 0] = np.where(np.arange(n) % 2, 1.0, -1.0) * np.sqrt(2.0 * units * 2.0 ** -40)
    p = bbmd.ka_params(block_z=8)  # blocks of 32 cells: chunks of 32 particles
    sim = bbmd.Sim(p, n, L, np.zeros(n, np.uint8), pos, vel)
    K0 = n * units * 2.0 ** -40
    dof = 3 * n - 3
    T, tau, dt = 2.0 * K0 / dof, 0.5, 0.001
    Q = dof * T * tau * tau
    # the opening half of the step, then the closing one from the energy that the step sums
    half = lambda xi, K: (xi + 0.25 * dt * (2 * K - dof * T) / Q, K)
    xi, K = half(0.0, K0)
    K *= np.exp(-xi * dt)
    xi, K = half(xi, K)
    opened = xi
    xi, K1 = half(opened, K)
    xi, _ = half(xi, K1 * np.exp(-xi * dt))
    sim.step_profiled(1, dt, (bbmd.THERMO_NH, T, T, tau))
    # each of the n / 32 chunks is off by half a unit of 2^-32 at most; a unit of energy moves xi
    # by dt / Q over the two quarter updates (1 % for the scale between them and FP32 velocities)
    bound = 1.01 * (n // 32) * 2.0 ** -33 * dt / Q
    assert abs(sim.observe(0)["xi"] - xi) <= bound
    sim.close()
