"""Lists of a box whose every tile is all of its 16,000 atoms: near the chip's limit the list builder runs four
warps per CTA instead of eight (no force kernel takes such a tile, a list query does)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from oracle import oracle as O  # noqa: E402
from paper_1305_4196_gb300 import mdgb as M  # noqa: E402
from paper_1305_4196_gb300 import workloads as W  # noqa: E402


@pytest.mark.parametrize("kw", [{}, dict(precision=M.MD_FP64), dict(list_kind=M.MD_LIST_HALF_COLOUR8)],
                         ids=["full", "fp64", "half"])
@pytest.mark.parametrize("n", [15776, 15808, 16000])
def test_lists_of_a_tile_near_the_limit(kw, n):
    box = np.full(3, 11.3)  # four cells a side at a list radius of 2.8
    pos = W.random_gas(n, box, seed=n)
    s = M.System(n, box, r_cut=2.5, skin=0.3, **kw)
    s.set_state(pos, np.zeros_like(pos))
    s.build_neighbors()
    assert s.info()["max_tile"] == n + 1
    assert np.array_equal(s.neighbors(), O.neighbor_pairs(pos, box, 2.8))
    s.close()
