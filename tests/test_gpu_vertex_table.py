"""The vertex index's hash table and packed sort against the oracle, bit for bit: one
voxel, coordinates at both ends of the 21-bit range (every pass of the sort has
work), corners just inside and just outside the 1e-3 limit, and ids written to
an array that is not 16-byte aligned."""
import numpy as np
import pytest
import torch

from oracle import vertex as VX
from paper_2511_02510_gb300 import litevoxel as L

pytestmark = pytest.mark.gpu


def index(geom, unit, shift=0):
    g = torch.as_tensor(geom, device="cuda")
    n = g.shape[0]
    buf = torch.empty(8 * n + shift, dtype=torch.int32, device="cuda")
    vidx = buf[shift:].view(n, 8)
    nv, st = torch.zeros(1, dtype=torch.int64, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    L.lv_build_vertex_index(g, unit, vidx, nv, st)
    return vidx.cpu().numpy().astype(np.int64), int(nv), int(st)


def lattice(n, lo, hi, seed, unit=1.0):
    """n voxels of half-size 1 to 4 units at integer centres in [lo, hi]."""
    rng = np.random.default_rng(seed)
    h = rng.integers(1, 5, n)
    return np.concatenate([rng.integers(lo, hi + 1, (n, 3)), h[:, None]], 1).astype(np.float32) * np.float32(unit)


@pytest.mark.parametrize("n,lo,hi,unit,shift", [
    (1, 5, 5, 1.0, 0), (257, -3, 3, 0.25, 0), (1000, -20, 20, 1.0, 1), (5000, -(1 << 20) + 4, (1 << 20) - 5, 1.0, 0),
    (20001, -700, 300, 2.0 ** -9, 0), (3000, 40, 90, 0.3, 2),
])
def test_index_bit_exact(n, lo, hi, unit, shift):
    geom = lattice(n, lo, hi, n, unit)
    u = float(np.float32(unit))
    ref, nref = VX.vertex_index(geom, u)
    vidx, nv, st = index(geom, u, shift)
    assert st == 0 and nv == nref
    np.testing.assert_array_equal(vidx, ref)


@pytest.mark.parametrize("off,good", [(0.9e-3, True), (0.995e-3, True), (1.005e-3, False), (0.4, False)])
def test_distance_limit(off, good):
    geom = lattice(64, 0, 50, 3)
    geom[17, 1] += np.float32(off)
    _, _, st = index(geom, 1.0)
    x = (geom[17, 1].astype(np.float64) + np.array([-1, 1]) * geom[17, 3].astype(np.float64))
    assert (np.abs(x - np.rint(x)).max() <= 1e-3) == good
    assert (st == 0) == good


def test_out_of_range_reports():
    geom = lattice(8, 0, 9, 1)
    geom[3, 0] = float(1 << 20)
    assert index(geom, 1.0)[2] == L.LV_ERR_INVALID_ARG
