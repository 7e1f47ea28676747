"""The build with two staging buffers (BBMD_STAGE_BUFFERS=2): block i + 1 is described and
copied while block i is computed.  Lists, forces and steps equal the default build's, with
several blocks to a CTA (shape 2 x 2 x 2 alone is rebuilt for it)."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUN = """
import sys
import numpy as np
from paper_1105_5613_gb300 import bbmd
from tests.helpers import mixture

out = {}
for ncell, mode in ((10, 0), (10, 1), (44, 0), (44, 1)):  # (one block a CTA, three and more)
    n, L, pos, vel, sp = mixture(ncell, shake=0.1)
    sim = bbmd.Sim(bbmd.ka_params(block_z=2, nbr_mode=mode), n, L, sp, pos, vel)
    key = f"{ncell}_{mode}_"
    out[key + "F"] = sim.get_forces()
    if mode == 0:
        out[key + "off"], out[key + "nbr"] = sim.get_neighbors(np.arange(0, n, 97))
    sim.step(12, 0.005, (bbmd.THERMO_NH, 2.0, 2.0, 0.5))
    sim.minimize(3)
    out[key + "x"], out[key + "v"], _ = sim.get_state()
    sim.close()
np.savez(sys.argv[1], **out)
"""


@pytest.fixture(scope="module")
def variant(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1105_5613_gb300 import build as b

    b.build()
    out = str(tmp_path_factory.mktemp("two_buffers"))
    nvcc = b._nvcc()
    z2 = os.path.join(out, "k_force_z2.o")
    subprocess.run([nvcc, *b.ARCH, *b.FLAGS, "-DBBMD_BLOCK_Z=2", "-DBBMD_STAGE_BUFFERS=2", "-c",
                    os.path.join(b.CSRC, "k_force.cu"), "-o", z2], check=True)
    objs = [z2 if o == "k_force_z2.o" else os.path.join(b.OUT, o) for _, o, _ in b.SOURCES]
    lib = os.path.join(out, "libbbmd.so")
    subprocess.run([nvcc, *b.ARCH, "-shared", "-o", lib, *objs, "-lcudart"], check=True)
    return b.LIB, lib, out


def test_two_staging_buffers_equal_one(variant):
    default, two, out = variant
    res = []
    for k, lib in enumerate((default, two)):
        path = os.path.join(out, f"{k}.npz")
        subprocess.run([sys.executable, "-c", RUN, path], check=True, cwd=ROOT,
                       env={**os.environ, "BBMD_LIB": lib, "PYTHONPATH": ROOT})
        res.append(np.load(path))
    assert sorted(res[0].files) == sorted(res[1].files)
    for f in res[0].files:
        assert np.array_equal(res[0][f], res[1][f]), f
