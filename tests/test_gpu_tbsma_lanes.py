"""The many-body passes of small systems (several lanes per atom, blocks shared by CTAs) and their
fused integration, bit for bit against one lane per atom (the energy pass) and against separate
integration kernels: the sums are exact integers and the update the same operations."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1305_4196_gb300 import mdgb as M  # noqa: E402
from paper_1305_4196_gb300 import workloads as W  # noqa: E402

P = W.copper_tbsma()
# cells of the crystal, sites left empty: from 8 lanes per atom to one, whole and ragged blocks
SIZES = [((9, 9, 9), 0), ((9, 10, 13), 77), ((18, 18, 18), 5), ((24, 22, 20), 1001), ((36, 30, 33), 3)]


def make(cells, missing):
    pos, box = W.fcc_lattice(*cells, 3.615)
    pos = W.gaussian_jitter(pos, box, 0.08, 3, stream=2)
    keep = np.sort(np.random.default_rng(missing).permutation(len(pos))[missing:])
    pos = np.ascontiguousarray(pos[keep])
    s = M.System(len(pos), box, r_cut=P["rc"], skin=0.4, mass=P["mass"], dt=0.1)
    s.set_tbsma(P["A"], P["xi"], P["p"], P["q"], P["r0"], P["rc"])
    s.set_state(pos, W.thermal_velocities(np.full(len(pos), P["mass"]), 0.05, 3))
    return s


@pytest.mark.parametrize("cells,missing", SIZES)
def test_lanes_and_fused_steps_are_bit_identical(cells, missing, monkeypatch):
    a = make(cells, missing)
    F = a.forces()
    monkeypatch.setenv("MDGB_NO_FUSE", "1")
    b = make(cells, missing)
    b.energy_virial()  # one lane per atom; its forces stay
    assert np.array_equal(F, b.forces())
    for n in (1, 13):
        a.step(n)
        b.step(n)
        for x, y in zip(a.get_state(), b.get_state()):
            assert np.array_equal(x, y)
        assert np.array_equal(a.forces(), b.forces())
    a.close()
    b.close()
