"""A list build that is refused because the tile cannot fit on the chip leaves cells, positions and
images of the binning before it consistent, in the caller's order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1305_4196_gb300 import mdgb as M  # noqa: E402


@pytest.mark.parametrize("kw", [{}, dict(precision=M.MD_FP64), dict(list_kind=M.MD_LIST_HALF_COLOUR8)],
                         ids=["full", "fp64", "half"])
def test_cells_after_a_refused_build(kw):
    rng = np.random.default_rng(3)
    n, L = 24000, 11.5  # four cells a side: every tile is the whole box, and too large
    pos, vel = rng.uniform(0, L, (n, 3)), rng.normal(size=(n, 3))
    s = M.System(n, np.full(3, L), r_cut=2.5, skin=0.3, **kw)
    s.set_state(pos, vel)
    for call in (s.build_neighbors, s.forces):
        with pytest.raises(M.MDError) as e:
            call()
        assert e.value.code == M.MD_ERR_CELL_OVERFLOW
        nc = np.array(s.info()["ncell"])
        c = np.floor(pos * (nc / L)).astype(int)
        assert np.array_equal(s.cells(), c[:, 0] + nc[0] * (c[:, 1] + nc[1] * c[:, 2]))
        x, v, image = s.get_state()
        assert np.array_equal(x, pos) and np.array_equal(v, vel) and not image.any()
    s.close()
