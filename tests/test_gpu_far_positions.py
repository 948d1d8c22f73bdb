"""Positions any number of box lengths away are mapped into the box at the first binning."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1305_4196_gb300 import mdgb as M  # noqa: E402
from paper_1305_4196_gb300 import workloads as W  # noqa: E402

KINDS = {"full": {}, "fp64": dict(precision=M.MD_FP64), "half": dict(list_kind=M.MD_LIST_HALF_COLOUR8),
         "atomic_free": dict(list_kind=M.MD_LIST_HALF_ATOMIC_FREE)}


def _liquid():
    """2,048 atoms in a box of 14 sigma, positions on a grid of 2^-20: a shift by whole box lengths is
    exact, so every result has to be the same bit for bit."""
    w = W.lj_fcc(8, rho=2048 / 14.0 ** 3, seed=5, jitter=0.05)
    assert np.allclose(w.box, 14.0)
    pos = np.minimum(np.floor(np.mod(w.pos, 14.0) * 2.0 ** 20) / 2.0 ** 20, 14.0 - 2.0 ** -20)
    return pos, w.vel


@pytest.mark.parametrize("kind", list(KINDS))
@pytest.mark.parametrize("first", ["forces", "bin", "step"])
def test_positions_anywhere(kind, first):
    pos, vel = _liquid()
    n, box = len(pos), np.full(3, 14.0)
    rng = np.random.default_rng(7)
    k = rng.integers(-3, 4, (n, 3))
    k[:4] = [[2, 0, -2], [-2, 5, 0], [1000, -1000, 3], [0, 0, 2 ** 20]]
    res = []
    for shift in (np.zeros((n, 3)), k):
        s = M.System(n, box, r_cut=2.5, skin=0.3, **KINDS[kind])
        s.set_state(np.ascontiguousarray(pos + shift * 14.0), vel)
        if first == "bin":
            s.bin_cells()
            x, _, image = s.get_state()
            assert np.array_equal(x, pos) and np.array_equal(image, shift)
        if first == "step":
            s.step(3)
        f = s.forces()
        x, v, image = s.get_state()
        res.append((f, x, v, image - shift, np.array(s.energy_virial()[:2])))
        s.close()
    for a, b in zip(*res):
        assert np.array_equal(a, b)
