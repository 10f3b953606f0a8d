"""GPU tests of the spatial point order at its kernels' edges, and of the
density over tiles cut from it."""
import numpy as np
import pytest

from paper_2512_16677_gb300 import synth
from tolerances import TOL

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2512_16677_gb300 import buildlib
    buildlib.build()


def _context(m, mode, points):
    from paper_2512_16677_gb300 import qmckl
    c = qmckl.Context(mode)
    c.set_molecule(m)
    c.set_points_device(torch.from_numpy(np.ascontiguousarray(points)).cuda())
    return c


@pytest.mark.parametrize("n", [50, 1023, 1025, 4096, 4097, 5121, 262144, 262145, 600001])
def test_order_is_the_stable_cell_sort(cfg, n):
    """One block up to 4096 points, blocks of 1024 keys up to 262 144, more
    keys per block beyond; many points of one cell, some outside the box."""
    m = cfg(1)
    rng = np.random.default_rng(n)
    pts = rng.normal(scale=4.0, size=(n, 3))
    pts[: n // 3] = pts[0]                      # a run of equal keys
    c = _context(m, "bf16x3", pts)
    c.mo_vgl_device()
    perm, _ = c.tile_layout()
    lo = (m.nucl_coord.min(axis=0) - 4.0).astype(np.float32)
    hi = (m.nucl_coord.max(axis=0) + 4.0).astype(np.float32)
    inv = (np.float32(32.0) / np.maximum(hi - lo, np.float32(1e-3))).astype(np.float32)
    f = (pts.astype(np.float32) - lo) * inv
    cell = np.where(f <= 0, 0, np.where(f >= 31, 31, np.trunc(f))).astype(np.uint32)
    key = np.zeros(n, dtype=np.uint32)
    for bit in range(5):
        for axis in range(3):
            key |= ((cell[:, axis] >> bit) & 1) << (3 * bit + axis)
    np.testing.assert_array_equal(perm, np.argsort(key, kind="stable"))


@pytest.mark.parametrize("mode", ["tf32", "bf16x3"])
@pytest.mark.parametrize("n", [65536, 65613])
def test_density_over_ordered_tiles(cfg, mode, n):
    """From 65 536 points on, the density's tiles come from the spatial order:
    the same values as in the caller's order, near and far from the nuclei
    (tiles that nothing reaches), and the oracle's on a sample."""
    from oracle import density, oracle
    oracle.build()
    m = cfg(6)
    rng = np.random.default_rng(n)
    pts = rng.uniform(m.nucl_coord.min(axis=0) - 30.0, m.nucl_coord.max(axis=0) + 30.0, (n, 3))
    w = synth.occupations(m)
    c = _context(m, mode, pts)
    got = c.density_device(w).cpu().numpy()
    c.set_spatial_order(False)
    c.set_points_device(torch.from_numpy(pts).cuda())
    np.testing.assert_array_equal(got, c.density_device(w).cpu().numpy())
    c.synchronize()
    idx = rng.choice(n, 120, replace=False)
    ref, size = density.density(m, w, points=pts[idx])
    assert (np.abs(got[idx] - ref) / (size + 1e-300)).max() <= TOL[mode][0]
