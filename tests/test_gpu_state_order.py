"""The permuted state after builds: positions, velocities and images come back exactly in the caller's
order, on every list kind, with a tile that outgrows its capacity at the first build (the list builder
takes the state to its new order and then starts again), and after a second build."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1305_4196_gb300 import mdgb as M  # noqa: E402

KINDS = {"full": {}, "fp64": dict(precision=M.MD_FP64), "half": dict(list_kind=M.MD_LIST_HALF_COLOUR8),
         "atomic_free": dict(list_kind=M.MD_LIST_HALF_ATOMIC_FREE)}


@pytest.mark.parametrize("kind", list(KINDS))
@pytest.mark.parametrize("n,cluster", [(1, 0), (4099, 0), (4099, 700), (60001, 900)])
def test_state_keeps_the_callers_order(kind, n, cluster):
    rng = np.random.default_rng(n + cluster)
    L = max(24.0, (n / 0.3) ** (1 / 3))
    pos = rng.uniform(0, L, (n, 3))
    if cluster:  # one dense spot: many times the mean tile
        pos[rng.permutation(n)[:cluster]] = 0.5 * L + rng.normal(0, 0.8, (cluster, 3))
    vel = rng.normal(size=(n, 3))
    s = M.System(n, np.full(3, L), **KINDS[kind])
    s.set_state(pos, vel)
    if kind == "atomic_free" and cluster:  # its lists take at most 63 atoms per cell
        with pytest.raises(M.MDError):
            s.build_neighbors()
        return
    for _ in range(2):
        s.build_neighbors()
        x, v, image = s.get_state()
        assert np.array_equal(x + image * L, pos) and np.array_equal(v, vel)
    s.close()
