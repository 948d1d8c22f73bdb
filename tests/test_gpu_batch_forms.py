"""The form each system of an ensemble takes, by atoms and SMs: systems of at most 512 atoms, or of at most
half a CTA's share of all atoms, one CTA each; larger ones of the one-CTA kind shared out as tasks;
the rest block tasks.  The shared and the one-CTA form of a system agree bit for bit
(forces and energies), and its forces with the oracle's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import oracle as O  # noqa: E402
from paper_1305_4196_gb300 import batch as BA  # noqa: E402
from paper_1305_4196_gb300 import workloads as W  # noqa: E402


def test_forms_and_their_results():
    small = [W.fcc_vacancies(n, 0.85, 1.0, seed=n) for n in (512, 513, 1999, 3571)]  # (3,571: a box below 6 cells)
    filler = W.lj_fcc(20, rho=0.8, seed=5, jitter=0.05)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    many = 4 * 3571 * sms // filler.n + 1  # half a CTA's share (two CTAs per SM) above 3,571 atoms
    few, lots = BA.from_systems(small + [filler]), BA.from_systems(small + [filler] * many)
    assert few.launch_shape()[0].tolist() == [0, 2, 2, 2, 1]
    assert lots.launch_shape()[0].tolist() == [0, 0, 0, 0] + [1] * many
    for steps in (0, 3):
        if steps:
            few.step(steps)
            lots.step(steps)
        a, b = few.forces(), lots.forces()
        ea, eb = few.energies(), lots.energies()
        o = 0
        pos = few.get_state()[0]
        for k, s in enumerate(small):
            assert np.array_equal(a[o:o + s.n], b[o:o + s.n])
            assert ea[0][k] == eb[0][k] and ea[1][k] == eb[1][k]
            Fref = O.lj_forces(pos[o:o + s.n], s.box, O.LJParams.single())[0]
            mag = np.sqrt((Fref ** 2).sum(1))
            err = np.sqrt(((a[o:o + s.n] - Fref) ** 2).sum(1)) / np.maximum(mag, np.sqrt((mag ** 2).mean()))
            assert err.max() <= 2e-5
            o += s.n
    few.close()
    lots.close()
