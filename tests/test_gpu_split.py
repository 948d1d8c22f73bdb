"""Mixed full-list forces of systems with few blocks, whose blocks are shared by CTAs with two,
four or eight lanes per atom: forces against the oracle (bar 2e-5, as in test_gpu_parity), and
the fused steps bit for bit against separate force and integration kernels."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from oracle import oracle as O  # noqa: E402
from paper_1305_4196_gb300 import mdgb as M  # noqa: E402
from paper_1305_4196_gb300 import workloads as W  # noqa: E402

KA = O.LJParams([[1.0, 1.5], [1.5, 0.5]], [[1.0, 0.8], [0.8, 0.88]], 2.5 * np.array([[1.0, 0.8], [0.8, 0.88]]),
                [1.0, 1.3])


def system(n, rho, two, gas=False):
    if gas:  # short lists, empty cells, a first list capacity of a few chunks
        box = np.array([24.0, 36.0, 30.0])
        pos = W.wrap(W.fcc_lattice(6, 9, 8, 4.0)[0] + 0.3, box)[:n]
        w = W.System(pos, W.thermal_velocities(np.ones(len(pos)), 0.5, 3), np.zeros(len(pos), np.int32), box)
    else:
        w = W.fcc_vacancies(n, rho, 0.8, seed=n)
    P = KA if two else O.LJParams.single()
    sp = W.species_shuffle(w.n, 0.2, 5) if two else w.species
    s = M.System(w.n, w.box, r_cut=float(P.rc.max()), skin=0.3, eps=P.eps, sigma=P.sig, mass=P.mass,
                 rcut=P.rc if two else None)
    s.set_state(w.pos, w.vel, sp)
    return s, w, P, sp


@pytest.mark.parametrize("two", [False, True])
@pytest.mark.parametrize("n,rho,gas", [(1501, 0.8442, False), (5003, 1.1, False), (16001, 0.8442, False),
                                       (33333, 0.8442, False), (61001, 0.8442, False), (1700, 0.0, True)])
def test_forces_and_fused_steps(n, rho, gas, two, monkeypatch):
    s, w, P, sp = system(n, rho, two, gas)
    F = s.forces()
    Fr, pe, _ = O.lj_forces(w.pos, w.box, P, sp) if two else O.lj_forces(w.pos, w.box, P)
    mag = np.sqrt((Fr ** 2).sum(1))
    e = np.sqrt(((F - Fr) ** 2).sum(1)) / np.maximum(mag, max(np.sqrt((mag ** 2).mean()), 1e-6))
    assert e.max() <= 2e-5
    assert abs(s.energy_virial()[0] - pe) <= 1e-6 * max(abs(pe), 1e-6)
    s.step(21)
    a = s.get_state()
    monkeypatch.setenv("MDGB_NO_FUSE", "1")
    t, _, _, _ = system(n, rho, two, gas)
    t.step(21)
    for x, y in zip(a, t.get_state()):
        assert np.array_equal(x, y)
    s.close()
    t.close()


def test_close_pairs_leave_their_lanes():
    """Pairs at 0.6 sigma (terms beyond the split sums) in three blocks: the exact finish."""
    w = W.fcc_vacancies(9001, 0.8, 0.5, seed=3)
    pos = w.pos.copy()
    for k in (0, 4000, 8000):
        pos[k + 1] = pos[k] + np.where(pos[k] + 0.35 < w.box, 0.35, -0.35)
    P = O.LJParams.single()
    s = M.System(w.n, w.box)
    s.set_state(pos, w.vel, w.species)
    F = s.forces()
    Fr = O.lj_forces(pos, w.box, P)[0]
    mag = np.sqrt((Fr ** 2).sum(1))
    e = np.sqrt(((F - Fr) ** 2).sum(1)) / np.maximum(mag, np.sqrt(np.median(mag) ** 2))
    assert e.max() <= 2e-5
    s.close()


@pytest.mark.parametrize("two", [False, True])
@pytest.mark.parametrize("n,rho", [(1501, 0.8442), (4999, 1.3), (13001, 0.75), (61001, 0.8442)])
def test_half_list_lanes(n, rho, two):
    """Four lanes per atom in the colour launches: blocks of more own atoms than lanes (several
    rounds), counted reaction sums in whole-box tiles, ordinary blocks."""
    w = W.fcc_vacancies(n, rho, 0.8, seed=n)
    P = KA if two else O.LJParams.single()
    sp = W.species_shuffle(w.n, 0.2, 5) if two else w.species
    s = M.System(w.n, w.box, r_cut=float(P.rc.max()), skin=0.3, eps=P.eps, sigma=P.sig, mass=P.mass,
                 rcut=P.rc if two else None, list_kind=M.MD_LIST_HALF_COLOUR8)
    s.set_state(w.pos, w.vel, sp)
    F = s.forces()
    Fr = (O.lj_forces(w.pos, w.box, P, sp) if two else O.lj_forces(w.pos, w.box, P))[0]
    mag = np.sqrt((Fr ** 2).sum(1))
    e = np.sqrt(((F - Fr) ** 2).sum(1)) / np.maximum(mag, np.sqrt((mag ** 2).mean()))
    assert e.max() <= 2e-5
    q = np.rint(F * 2.0 ** 32).astype(np.int64)
    assert np.array_equal(q.sum(0), np.zeros(3, np.int64))  # every reaction is the exact negative
    s.close()
