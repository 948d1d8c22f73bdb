"""Positions any number of box lengths away are mapped into the box at the first binning, and an atom
that later moves by more than one box length between builds is an error on every path that builds."""
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


@pytest.mark.parametrize("L", [14.0, 13.37])
def test_edges_of_the_mapping(L):
    """Coordinates at and beside -L, 0, L, 2 L and further: in the box after the binning, and at the place that
    the image counters give to the last bit of the coordinate."""
    edges = [e * L for e in (-3.0, -2.0, -1.0, 0.0, 1.0, 2.0, 3.0, 4097.0)]
    xs = np.array(sorted({f(e) for e in edges for f in (
        lambda e: e, lambda e: np.nextafter(e, np.inf), lambda e: np.nextafter(e, -np.inf),
        lambda e: e * (1 + 2.0 ** -21), lambda e: e * (1 - 2.0 ** -21), lambda e: e + 0.3, lambda e: e - 0.3)}))
    rng = np.random.default_rng(2)
    pos = rng.uniform(0, L, (len(xs), 3))
    pos[:, 1] = xs
    s = M.System(len(xs), np.full(3, L))
    s.set_state(pos, np.zeros_like(pos))
    s.bin_cells()
    x, _, image = s.get_state()
    assert (x >= 0).all() and (x <= L).all()
    assert np.array_equal(x[:, ::2], pos[:, ::2]) and not image[:, ::2].any()
    assert (np.abs(x[:, 1] + image[:, 1] * L - xs) <= 2.0 ** -51 * np.maximum(np.abs(xs), L)).all()
    s.close()


@pytest.mark.parametrize("x", [2.0 ** 31 * 14.0, -1.0e300])
def test_positions_beyond_the_image_counters(x):
    pos, vel = _liquid()
    pos[9, 1] = x
    s = M.System(len(pos), np.full(3, 14.0))
    for call in (s.forces, s.build_neighbors, s.bin_cells, lambda: s.step(1), s.energy_virial):
        s.set_state(pos, vel)
        with pytest.raises(M.MDError):
            call()
    s.close()


@pytest.mark.parametrize("kind", list(KINDS))
@pytest.mark.parametrize("no_graphs", ["0", "1"])
@pytest.mark.parametrize("steps", [1, 2, 5])
def test_an_atom_that_escapes_is_an_error(monkeypatch, kind, no_graphs, steps):
    """2.5 box lengths in one step: the build in that step reports it, in graphs and launched from the
    host, also when further steps follow."""
    monkeypatch.setenv("MDGB_NO_GRAPHS", no_graphs)
    pos, vel = _liquid()
    vel[9, 1] = 2.5 * 14.0 / 0.005
    s = M.System(len(pos), np.full(3, 14.0), dt=0.005, **KINDS[kind])
    s.set_state(pos, vel)
    with pytest.raises(M.MDError) as e:
        s.step(steps)
    assert e.value.code == M.MD_ERR_NONFINITE
    s.close()
