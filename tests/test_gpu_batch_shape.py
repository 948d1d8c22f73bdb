"""Launches of ensembles whose tile comes near a limit of shared memory: what a CTA may take at all, and
what still lets an SM hold two.  The launch is sized by the block system's tile (64 cells of 1.6 times the
mean occupancy and 4 atoms, one float4 each) and the list build beside it (three floats per atom and
35.5 KB)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import oracle as O  # noqa: E402
from paper_1305_4196_gb300 import batch as BA  # noqa: E402
from paper_1305_4196_gb300 import mdgb as M  # noqa: E402
from paper_1305_4196_gb300 import workloads as W  # noqa: E402

SKIN = 0.3


def sized(m):
    """(atoms, box side, cutoff) of a system on 6 cells a side whose tile is sized for m + 4 atoms per cell."""
    n = round((m - 0.5) / 1.6 * 6 ** 3)
    L = (n / 0.9) ** (1.0 / 3.0)
    return n, L, L / 7.9 - SKIN


def layout_bytes(m):
    tile = 64 * (m + 4)
    return -(-max(16 * (tile + 1), (tile + 228) // 4 * 12 * 4 + 32768) // 16) * 16


@pytest.mark.parametrize("m,ctas", [(92, 2), (93, 1), (213, 1), (214, 1), (215, None)])
def test_launch_near_the_limits(m, ctas):
    """Two CTAs per SM up to 109,664 bytes, one up to 224,256, refused beyond."""
    n, L, rc = sized(m)
    size = layout_bytes(m)
    assert (2 if size <= 109664 else 1 if size <= 224256 else None) == ctas
    if ctas is None:
        with pytest.raises(M.MDError) as e:
            BA.Batch([n], [[L, L, L]], r_cut=rc, skin=SKIN)
        assert e.value.code == M.MD_ERR_CELL_OVERFLOW
        return
    b = BA.Batch([n], [[L, L, L]], r_cut=rc, skin=SKIN)
    form, per_sm, smem = b.launch_shape()
    assert form.tolist() == [1] and smem == size and per_sm == ctas
    s = W.fcc_vacancies(n, 0.9, 0.7, seed=m)
    b.set_state(s.pos, s.vel)
    F = b.forces()
    Fref, pe, _ = O.lj_forces(s.pos, s.box, O.LJParams.single(rc=rc))
    frms = np.sqrt((Fref ** 2).sum(1).mean())
    assert np.abs(F - Fref).max() <= 2e-5 * max(frms, np.abs(Fref).max())
    assert abs(b.energies()[0][0] - pe) <= 1e-6 * abs(pe)
    b.close()


@pytest.mark.parametrize("short_of", [1, 30, 200, 400, 600])
def test_lists_of_a_tile_that_fills_its_memory(short_of):
    """A dense bar through a dilute box: the fullest tile comes within short_of atoms of its slots, where the
    list build has room for the buffers of six or seven warps (600: all eight)."""
    n, L, rc = sized(40)
    w, target = L / 6, (64 * 44 - short_of) // 4  # atoms of the bar in each of the six layers of cells
    rng = np.random.default_rng(short_of)
    sites, _ = W.fcc_lattice(14, 14, 14, L / 14)
    sites = np.mod(sites + 0.21, L)
    cell = np.floor(sites / w).astype(int)
    bar = ((cell[:, :2] >= 1) & (cell[:, :2] <= 4)).all(1)
    keep = [rng.permutation(np.nonzero(bar & (cell[:, 2] == z))[0])[:target] for z in range(6)]
    assert all(len(k) == target for k in keep)
    rest = rng.permutation(np.nonzero(~bar)[0])[:n - 6 * target]
    idx = np.sort(np.concatenate(keep + [rest]))
    assert len(idx) == n
    pos = np.ascontiguousarray(sites[idx])
    b = BA.Batch([n], [[L, L, L]], r_cut=rc, skin=SKIN)
    assert b.launch_shape()[2] == layout_bytes(40)
    b.set_state(pos, np.zeros_like(pos))
    F = b.forces()
    Fref = O.lj_forces(pos, np.full(3, L), O.LJParams.single(rc=rc))[0]
    frms = np.sqrt((Fref ** 2).sum(1).mean())
    assert np.abs(F - Fref).max() <= 2e-5 * max(frms, np.abs(Fref).max())
    b.close()
