"""Derivatives of the forces over species counts and atom counts that leave lanes, groups of own
atoms and whole blocks partly empty, against the FP64 oracle.  Bars as for the other derivative
tests: 1e-11 (FP64) and 2e-5 (FP32 pair terms) of the largest value."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import oracle as O  # noqa: E402
from paper_1305_4196_gb300 import build as B  # noqa: E402
from paper_1305_4196_gb300 import workloads as W  # noqa: E402

B.build()
from paper_1305_4196_gb300 import mdgb as M  # noqa: E402

TOL = {"fp64": 1e-11, "mixed": 2e-5}
PREC = {"fp64": M.MD_FP64, "mixed": M.MD_MIXED}


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nsp,n_cells,keep", [(1, 10, None), (1, 10, 33), (2, 14, 10975), (2, 10, 1), (3, 10, 3999),
                                              (4, 11, 5000)])
def test_derivatives_over_species_and_sizes(precision, nsp, n_cells, keep):
    s = W.lj_fcc(n_cells, rho=1.0, seed=nsp, jitter=0.05)
    rng = np.random.default_rng(10 * nsp + n_cells)
    pos = s.pos if keep is None else s.pos[np.sort(rng.permutation(s.n)[:keep])]
    n = len(pos)
    sp = rng.integers(0, nsp, n).astype(np.int32)
    a = 1.0 + 0.1 * np.arange(nsp)
    eps, sig = np.sqrt(np.outer(a, a)), (1.0 - 0.02 * np.add.outer(np.arange(nsp), np.arange(nsp)))
    rc = 2.3 * sig
    P = O.LJParams(eps, sig, rc, [1.0] * nsp)
    G = rng.normal(size=(n, 3))
    sysm = M.System(n, s.box, r_cut=float(rc.max()), skin=0.3, eps=eps, sigma=sig, mass=[1.0] * nsp,
                    precision=PREC[precision], rcut=rc)
    sysm.set_state(np.ascontiguousarray(pos), np.zeros_like(pos), sp)
    gx, ge, gs = sysm.forces_backward(G)
    gx_ref, ge_ref, gs_ref = O.lj_force_grad(pos, s.box, P, G, sp)
    de, ds = sysm.energy_param_grad()
    de_ref, ds_ref = O.lj_energy_param_grad(pos, s.box, P, sp)
    for v, ref in [(gx, gx_ref), (ge, ge_ref), (gs, gs_ref), (de, de_ref), (ds, ds_ref)]:
        assert np.abs(v - ref).max() <= TOL[precision] * np.abs(ref).max()
