"""Colour-phase half lists of a box whose every tile is the whole box, at the largest tiles that the force kernel's
shared memory takes (tile coordinates, reaction sums and its static arrays together)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from oracle import oracle as O  # noqa: E402
from paper_1305_4196_gb300 import mdgb as M  # noqa: E402

NX, L, R_CUT, SKIN = 12, 20.0, 4.0, 0.3  # four cells a side, three lattice cells wide


@pytest.mark.parametrize("n", [6751, 6752, 6783])
def test_forces_energies_and_steps_at_the_limit(n):
    rng = np.random.default_rng(n)
    a = L / NX
    cells = np.stack(np.meshgrid(*[np.arange(NX)] * 3, indexing="ij"), -1).reshape(-1, 1, 3)
    basis = np.array([[0.25, 0.25, 0.25], [0.75, 0.75, 0.25], [0.75, 0.25, 0.75], [0.25, 0.75, 0.75]])
    pos = ((cells + basis) * a).reshape(-1, 3)
    pos = pos[np.sort(rng.permutation(len(pos))[:n])]
    pos = pos + np.clip(0.05 * rng.normal(size=pos.shape), -0.2, 0.2)
    vel = rng.normal(size=pos.shape)
    vel -= vel.mean(0)
    box = np.full(3, L)
    s = M.System(n, box, r_cut=R_CUT, skin=SKIN, list_kind=M.MD_LIST_HALF_COLOUR8)
    s.set_state(pos, vel)
    F = s.forces()
    assert s.info()["tile_cap"] == (6752 if n == 6751 else 6784)  # (the next one exceeds an SM's shared memory)
    P = O.LJParams.single(rc=R_CUT)
    Fref, pe_ref, _ = O.lj_forces(pos, box, P)
    mag = np.sqrt((Fref ** 2).sum(1))
    err = np.sqrt(((F - Fref) ** 2).sum(1)) / np.maximum(mag, np.sqrt((mag ** 2).mean()))
    assert err.max() <= 2e-5
    assert abs(s.energy_virial()[0] - pe_ref) <= 1e-6 * abs(pe_ref)
    s.step(3)
    x, _, image = s.get_state()
    ref = O.run_nve(pos, vel, box, P, 0.005, SKIN, 3)
    assert np.abs(x + image * box - (ref["pos"] + ref["image"] * box)).max() < 1e-6
    s.close()
