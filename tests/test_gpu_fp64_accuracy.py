"""Rounding of the FP64 pair kernels: no further from a wider evaluation (numpy's long double,
the same integer positions and decisions) than plain FP64 arithmetic with correctly rounded
divisions and square roots is, summed pair by pair.  Root mean squares over 12 000 force
components or 4000 energies scatter by about a per cent; the bar is 15 %."""
import numpy as np
import pytest

import oracle
from tests.helpers import mixture, quantized

pytestmark = pytest.mark.gpu

bbmd = pytest.importorskip("paper_1105_5613_gb300.bbmd")
spatial = pytest.importorskip("scipy.spatial")

EPS = np.array([1.0, 1.5, 1.5, 0.5])
SIG = np.array([1.0, 0.8, 0.8, 0.88])
NCELL = 10


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1105_5613_gb300 import build as b

    b.build()
    bbmd.load()


def system(shake=0.13):
    n, L, pos, vel, sp = mixture(NCELL, seed=3, shake=shake)
    return n, L, pos, sp


def evaluate(real, pos, sp, L, pot, shift):
    """(F, u) of the quantised positions in arithmetic of type `real`, every particle's pairs
    added one after the other."""
    n = len(pos)
    xq, xfix, k = quantized(pos, L)
    x = xfix.astype(np.int64)
    Lf = np.int64(np.rint(np.ldexp(L, k)))
    pairs = spatial.cKDTree(np.mod(xq, L), boxsize=L).query_pairs(2.5 + 1e-9, output_type="ndarray")
    i = np.concatenate([pairs[:, 0], pairs[:, 1]])
    j = np.concatenate([pairs[:, 1], pairs[:, 0]])
    o = np.argsort(i, kind="stable")
    i, j = i[o], j[o]
    d = x[j] - x[i]
    d = np.where(d > Lf >> 1, d - Lf, np.where(d < -(Lf >> 1), d + Lf, d))
    kind = sp[i].astype(int) * 2 + sp[j]
    dd = np.ldexp(d.astype(np.float64), -k)  # the cutoff decision is FP64's for both
    near = (dd[:, 0] ** 2 + dd[:, 1] ** 2) + dd[:, 2] ** 2 < ((2.5 * SIG) * (2.5 * SIG))[kind]
    i, d, kind = i[near], np.ldexp(d[near].astype(real), -k), kind[near]
    eps, sig, rc = EPS.astype(real)[kind], SIG.astype(real)[kind], (2.5 * SIG).astype(real)[kind]
    c = real(1 if pot == bbmd.POT_LJ else 0)
    r2 = (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]
    ir2 = real(1) / r2
    s2 = sig * sig * ir2
    s6 = s2 * s2 * s2
    f = 48 * eps * ir2 * s6 * (s6 - c / 2)
    V = 4 * eps * s6 * (s6 - c)
    q2 = sig * sig / (rc * rc)
    q6 = q2 * q2 * q2
    if shift != bbmd.SHIFT_NONE:
        V = V - 4 * eps * q6 * (q6 - c)
    if shift == bbmd.SHIFT_FORCE:
        dc = -48 * eps * q6 * (q6 - c / 2) / rc
        r = np.sqrt(r2)
        f = f + dc / r
        V = V - (r - rc) * dc
    first = np.searchsorted(i, np.arange(n))
    count = np.bincount(i, minlength=n)
    F, u = np.zeros((n, 3), real), np.zeros(n, real)
    for t in range(count.max()):
        has = np.nonzero(count > t)[0]
        p = first[has] + t
        F[has] -= f[p, None] * d[p]
        u[has] += V[p]
    return F, u / 2


def rms(a, b):
    return float(np.sqrt(np.mean(np.square(a.astype(np.longdouble) - b))))


@pytest.mark.parametrize("pot", [bbmd.POT_LJ, bbmd.POT_SOFT])
@pytest.mark.parametrize("shift", [bbmd.SHIFT_ENERGY, bbmd.SHIFT_FORCE])
@pytest.mark.parametrize("mode", [bbmd.NBR_VERLET, bbmd.NBR_CELL])
def test_forces_round_like_plain_fp64(pot, shift, mode):
    n, L, pos, sp = system()
    wide, _ = evaluate(np.longdouble, pos, sp, L, pot, shift)
    plain, _ = evaluate(np.float64, pos, sp, L, pot, shift)
    p = bbmd.ka_params(precision=bbmd.PREC_FP64, potential=pot, shift=shift, nbr_mode=mode)
    sim = bbmd.Sim(p, n, L, sp, pos, np.zeros_like(pos))
    assert rms(sim.get_forces(), wide) <= 1.15 * rms(plain, wide)
    sim.close()


@pytest.mark.parametrize("pot", [bbmd.POT_LJ, bbmd.POT_SOFT])
@pytest.mark.parametrize("shift", [bbmd.SHIFT_NONE, bbmd.SHIFT_ENERGY, bbmd.SHIFT_FORCE])
@pytest.mark.parametrize("prec,mode", [(bbmd.PREC_FP64, bbmd.NBR_VERLET), (bbmd.PREC_MIXED, bbmd.NBR_VERLET),
                                       (bbmd.PREC_MIXED, bbmd.NBR_CELL)])
def test_energies_round_like_plain_fp64(pot, shift, prec, mode):
    # (a small shake: attraction and repulsion of the order of their sum, as in a liquid)
    n, L, pos, sp = system(0.05)
    _, wide = evaluate(np.longdouble, pos, sp, L, pot, shift)
    _, plain = evaluate(np.float64, pos, sp, L, pot, shift)
    p = bbmd.ka_params(precision=prec, potential=pot, shift=shift, nbr_mode=mode)
    sim = bbmd.Sim(p, n, L, sp, pos, np.zeros_like(pos))
    _, u = sim.get_forces(energies=True)
    assert rms(u, wide) <= 1.15 * rms(plain, wide)
    sim.close()
