"""Neighbour lists where the builder's stages change over: cells of more than 32 atoms, batches
of 64 candidates that are all neighbours (a row of open entries runs over), lists longer than
the first capacity, blocks shared by several CTAs and cells of a few atoms."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from oracle import oracle as O  # noqa: E402
from paper_1305_4196_gb300 import mdgb as M  # noqa: E402
from paper_1305_4196_gb300 import workloads as W  # noqa: E402


@pytest.mark.parametrize("lst", ["full", "half"])
@pytest.mark.parametrize("nx,ny,nz,rho", [
    (10, 10, 10, 2.6),   # 65 atoms per cell, 240 neighbours: rows run over, three groups of own atoms
    (12, 13, 14, 4.1),   # 137 atoms per cell, 370 neighbours: every batch runs over, lists regrow
    (8, 9, 14, 0.8442),  # 4 cells a side: blocks shared by several CTAs
    (23, 7, 15, 0.25),   # 8 atoms per cell, unequal sides
    (30, 30, 31, 0.8442),  # more blocks than two per SM: one CTA each
])
def test_lists_match_oracle(nx, ny, nz, rho, lst):
    a = W.lattice_constant(rho)
    pos, box = W.fcc_lattice(nx, ny, nz, a)
    pos = W.gaussian_jitter(pos, box, 0.04 * a, 17, stream=2)[:-3]  # an odd count, three vacancies
    s = M.System(len(pos), box, list_kind=M.MD_LIST_FULL if lst == "full" else M.MD_LIST_HALF_COLOUR8)
    s.set_state(pos, np.zeros_like(pos))
    s.build_neighbors()
    assert np.array_equal(s.neighbors(), O.neighbor_pairs(pos, box, 2.8))
    s.close()
