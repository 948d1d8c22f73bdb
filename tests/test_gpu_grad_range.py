"""Parameter derivatives whose FP32 terms are finite and whose sums leave FP32's range: the same terms
scaled by a power of two give the same sums scaled, as in FP64; and terms that overflow are seen."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1305_4196_gb300 import mdgb as M  # noqa: E402
from paper_1305_4196_gb300 import workloads as W  # noqa: E402


@pytest.mark.parametrize("nsp", [1, 2, 3, 4])
def test_sums_beyond_fp32(nsp):
    s = W.lj_fcc(10, rho=1.0, seed=nsp, jitter=0.02)
    sp = np.random.default_rng(nsp).integers(0, nsp, s.n).astype(np.int32)
    sysm = M.System(s.n, s.box, eps=np.ones((nsp, nsp)), sigma=np.full((nsp, nsp), 1.05), mass=[1.0] * nsp)
    sysm.set_state(s.pos, s.vel, sp)
    L = s.box[0]
    G = L / (2 * np.pi) * np.sin(2 * np.pi * s.pos / L)  # (dL/dF differs by about the distance of a pair)
    _, ge, gs = sysm.forces_backward(G)
    for k in (60, 121, 124):  # (124: the sums of a warp's atoms reach beyond FP32, their terms do not)
        _, he, hs = sysm.forces_backward(G * 2.0 ** k)
        assert np.isfinite(he).all() and np.isfinite(hs).all()
        # the same terms, exactly scaled: only the order of FP64 additions differs
        for a, b in ((ge, he), (gs, hs)):
            assert np.abs(b / 2.0 ** k - a).max() <= 1e-11 * np.abs(a).max()
    _, ie, _ = sysm.forces_backward(G * 2.0 ** 127)  # terms that are not finite
    assert not np.isfinite(ie).all()
    sysm.close()
