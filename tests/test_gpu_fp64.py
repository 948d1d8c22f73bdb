"""FP64 full-list forces, energy and virial against the oracle over the forms the launch picks:
one, two, four and eight lanes per atom, tiles that leave no room for the entry queues, several
species, close pairs, and length units whose squares lie outside the FP32 range the tests use.
Bars as in test_gpu_parity: 1e-12 relative (FP64 rounding of ~100 terms stays below 1e-13)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from oracle import oracle as O  # noqa: E402
from paper_1305_4196_gb300 import mdgb as M  # noqa: E402
from paper_1305_4196_gb300 import workloads as W  # noqa: E402


def check(pos, box, sp, P, r_cut, skin):
    s = M.System(len(pos), box, r_cut=r_cut, skin=skin, eps=P.eps, sigma=P.sig, mass=P.mass, precision=M.MD_FP64,
                 rcut=P.rc if P.nsp > 1 else None)
    s.set_state(pos, np.zeros_like(pos), sp)
    F = s.forces()
    pe, _, vir = s.energy_virial()
    F2 = s.forces()
    s.close()
    Fr, per, virr = O.lj_forces(pos, box, P, sp) if P.nsp > 1 else O.lj_forces(pos, box, P)
    mag = np.sqrt((Fr ** 2).sum(1))
    e = np.sqrt(((F - Fr) ** 2).sum(1)) / np.maximum(mag, np.sqrt((mag ** 2).mean()))
    assert e.max() <= 1e-12
    assert np.array_equal(F, F2)
    assert abs(pe - per) <= 1e-12 * abs(per)
    assert np.abs(vir - virr).max() <= 1e-12 * np.abs(virr).max()


@pytest.mark.parametrize("n,rho,close", [
    (2047, 0.8442, False),   # eight blocks, eight lanes per atom
    (8209, 1.86, True),      # a whole-box tile with no room for the queues
    (21001, 0.8442, True),   # four lanes, two CTAs per block
    (60001, 0.8442, False),  # two lanes, three CTAs per block
    (150001, 0.8442, True),  # two lanes, a CTA per block
])
def test_forms_match_oracle(n, rho, close):
    w = W.fcc_vacancies(n, rho, 1.0, seed=n)
    pos = w.pos.copy()
    if close:  # two atoms 0.3 sigma apart: terms of 10^9
        pos[1] = np.where(pos[0] + 0.17 < w.box, pos[0] + 0.17, pos[0] - 0.17)
    check(pos, w.box, w.species, O.LJParams.single(), 2.5, 0.3)


@pytest.mark.parametrize("scale", [1.0, 3.4e-10, 1.0e-14, 30.0])
def test_length_units(scale):
    w = W.fcc_vacancies(3001, 0.8442, 1.0, seed=7)
    P = O.LJParams.single(sig=scale, rc=2.5 * scale)
    check(w.pos * scale, w.box * scale, w.species, P, 2.5 * scale, 0.3 * scale)


@pytest.mark.parametrize("n_cells", [8, 15])
def test_two_species(n_cells):
    w = W.lj_fcc(n_cells, rho=1.2, seed=5, jitter=0.05)
    sig = np.array([[1.0, 0.8], [0.8, 0.88]])
    P = O.LJParams([[1.0, 1.5], [1.5, 0.5]], sig, 2.5 * sig, [1.0, 1.0])
    check(w.pos, w.box, W.species_shuffle(w.n, 0.2, 5), P, float(P.rc.max()), 0.3)
