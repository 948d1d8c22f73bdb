"""One-CTA systems of an ensemble shared out as tasks (few atoms per CTA of the launch) against the same
systems run by one CTA each (in an ensemble of many atoms), bit for bit: positions, velocities,
forces and energies after step counts of either parity, with and without forces from the call before."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1305_4196_gb300 import batch as BA  # noqa: E402
from paper_1305_4196_gb300 import workloads as W  # noqa: E402

R_CUT, SKIN = 2.5, 0.3


def system(n_cells, n, rho, seed):
    s = W.lj_fcc(n_cells, rho=rho * 4 * n_cells ** 3 / n, seed=seed, T=1.0, jitter=0.05)
    keep = np.sort(np.random.default_rng(seed).permutation(s.n)[:n])
    return s.pos[keep], s.vel[keep], s.box


def ensemble(parts):
    b = BA.Batch([len(p) for p, _, _ in parts], np.stack([x for _, _, x in parts]), r_cut=R_CUT, skin=SKIN, dt=0.002)
    b.set_state(np.concatenate([p for p, _, _ in parts]), np.concatenate([v for _, v, _ in parts]))
    return b


def test_shared_systems_equal_one_cta_systems():
    # ragged chunks of 512 atoms, a whole number of them, and the largest that fits no block system
    small = [system(6, 513, 0.8, 1), system(7, 1024, 0.85, 2), system(8, 1999, 0.9, 3), system(10, 3571, 0.9, 4)]
    pos, vel, box = system(20, 32000, 0.8, 5)
    filler = [(pos, vel, box)] * 74  # 2.4 million atoms: more than 3,571 for half a CTA's share
    n = sum(len(p) for p, _, _ in small)
    # (with one of them, so that the width of the FP64 decision band is the same)
    a, b = ensemble(small + filler[:1]), ensemble(small + filler)
    for e in (a, b):
        assert e.layout()[0][:len(small)].tolist() == [0] * len(small)
    for k, steps in enumerate((1, 4, 0, 7)):
        if steps:
            a.step(steps)
            b.step(steps)
        if k % 2 == 0:  # the next step finds forces, or those of the step call only
            assert np.array_equal(a.forces()[:n], b.forces()[:n])
            for x, y in zip(a.energies(), b.energies()):
                assert np.array_equal(x[:len(small)], y[:len(small)])
        for x, y in zip(a.get_state(), b.get_state()):
            assert np.array_equal(x[:n], y[:n])
