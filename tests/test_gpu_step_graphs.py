"""Steps run as one graph per chunk (a loop and what is left over) against the same kernels
launched from the host, bit for bit, over step counts with every remainder, in one call and split
into calls, beyond a chunk, and with timing switched on in between."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1305_4196_gb300 import mdgb as M  # noqa: E402
from paper_1305_4196_gb300 import workloads as W  # noqa: E402

KINDS = {"fused": {}, "fp64": dict(precision=M.MD_FP64), "half": dict(list_kind=M.MD_LIST_HALF_COLOUR8),
         "every_k": dict(rebuild=M.MD_REBUILD_EVERY_K, rebuild_k=3), "copper": {}}


def make(kind):
    if kind == "copper":
        P = W.copper_tbsma()
        pos, box = W.fcc_lattice(9, 9, 9, 3.615)
        pos = W.gaussian_jitter(pos, box, 0.08, 3, stream=2)
        s = M.System(len(pos), box, r_cut=P["rc"], skin=0.4, mass=P["mass"], dt=0.1)
        s.set_tbsma(P["A"], P["xi"], P["p"], P["q"], P["r0"], P["rc"])
        s.set_state(pos, W.thermal_velocities(np.full(len(pos), P["mass"]), 0.05, 3))
        return s
    w = W.lj_fcc(9, seed=4, T=1.2, jitter=0.05)
    s = M.System(w.n, w.box, **KINDS[kind])
    s.set_state(w.pos, w.vel, w.species)
    return s


@pytest.mark.parametrize("kind", list(KINDS))
def test_graphs_equal_host_launches(kind, monkeypatch):
    counts = [1, 2, 3, 4, 5, 7, 8, 9, 14] + ([203] if kind == "fused" else [])
    a = make(kind)
    monkeypatch.setenv("MDGB_NO_GRAPHS", "1")
    b = make(kind)
    for k, n in enumerate(counts):
        a.set_timing(k == 5)
        a.step(n)
        b.step(n)
        for x, y in zip(a.get_state(), b.get_state()):
            assert np.array_equal(x, y), (kind, n)
        assert a.energy_virial()[0] == b.energy_virial()[0]
    assert a.info()["n_steps"] == sum(counts) and a.info()["n_builds"] == b.info()["n_builds"]
    a.close()
    b.close()
