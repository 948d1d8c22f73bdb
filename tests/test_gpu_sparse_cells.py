"""Forces and derivatives of systems whose cells hold few atoms or none, and of small blocks shared by several CTAs
(staging of the tile and adding it back across cell borders), against the FP64 oracle.  Bars as in the other
tests: 1e-12 (FP64 forces), 1e-11 (FP64 derivatives), 2e-5 (mixed)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from oracle import oracle as O  # noqa: E402
from paper_1305_4196_gb300 import mdgb as M  # noqa: E402


def scattered(n, box, seed):
    """n atoms no closer than 0.9: sites of a simple cubic lattice of side >= 1.0, jittered by 0.05."""
    rng = np.random.default_rng(seed)
    k = np.floor(box).astype(int)
    sites = np.stack(np.meshgrid(*[np.arange(x) for x in k], indexing="ij"), -1).reshape(-1, 3)
    pick = sites[np.sort(rng.permutation(len(sites))[:n])]
    return np.ascontiguousarray((pick + 0.5 + rng.uniform(-0.05, 0.05, pick.shape)) * (box / k))


def energy_bar(s, pos, box, r_cut, precision):
    """Bound of the energy's error.  Mixed: a coordinate difference is off by at most 2 (2^-25 + 2^-23) cell widths
    (cell-relative coordinates rounded to FP32, then in the block's frame, up to two widths), which
    moves a pair's energy by |force| times that, and the FP32 terms round to some 2^-21.  FP64: 2^-29 as much."""
    i, j = O.neighbor_pairs(pos, box, r_cut).T
    d = pos[i] - pos[j]
    d -= box * np.rint(d / box)
    r2 = (d * d).sum(1)
    s6 = r2 ** -3.0
    shift = np.sqrt(3.0) * 2 * (2.0 ** -25 + 2.0 ** -23) * (box / np.array(s.info()["ncell"])).max()
    bar = (24 * np.abs(2 * s6 * s6 - s6) / np.sqrt(r2) * shift + 4 * (s6 * s6 + s6) * 2.0 ** -21).sum()
    return bar if precision == M.MD_MIXED else 2.0 ** -29 * bar


@pytest.mark.parametrize("precision,kind,tol", [(M.MD_FP64, M.MD_LIST_FULL, 1e-12),
                                                (M.MD_FP64, M.MD_LIST_HALF_COLOUR8, 1e-12),
                                                (M.MD_MIXED, M.MD_LIST_HALF_COLOUR8, 2e-5)],
                         ids=["fp64", "fp64-half", "mixed-half"])
@pytest.mark.parametrize("n,side,r_cut", [(1, 12.0, 2.5), (40, 23.0, 2.5), (3000, 33.0, 1.2), (12000, 29.0, 1.2),
                                          (1500, 12.0, 2.5), (4000, 24.0, 4.0)])
def test_sparse_and_shared_blocks(precision, kind, tol, n, side, r_cut):
    box = side * np.array([1.0, 1.1, 1.25])
    pos = scattered(n, box, seed=n)
    P = O.LJParams.single(rc=r_cut)
    s = M.System(n, box, r_cut=r_cut, skin=0.3, precision=precision, list_kind=kind)
    s.set_state(pos, np.zeros_like(pos))
    F = s.forces()
    Fref, pe_ref, _ = O.lj_forces(pos, box, P)
    mag = np.sqrt((Fref ** 2).sum(1))
    bar = np.maximum(np.maximum(mag, np.sqrt((mag ** 2).mean())), 1e-300)
    assert (np.sqrt(((F - Fref) ** 2).sum(1)) <= tol * bar).all()
    assert abs(s.energy_virial()[0] - pe_ref) <= energy_bar(s, pos, box, r_cut, precision)
    if precision == M.MD_FP64 and kind == M.MD_LIST_FULL:
        G = np.random.default_rng(1).normal(size=(n, 3))
        for v, ref in zip(s.forces_backward(G), O.lj_force_grad(pos, box, P, G)):
            assert np.abs(v - ref).max() <= 1e-11 * np.abs(ref).max()
    s.close()
