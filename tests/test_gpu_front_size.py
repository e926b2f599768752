"""The sorted front of a very long list is never a few entries: one voxel close to the
camera before a crowd at nearly one depth makes the first range of keys a single
entry, and the front goes on past it, so that pixels which stop within the crowd's
first entries need no second pass.  Every output is that of the whole order."""
import numpy as np
import pytest
import torch

from paper_2511_02510_gb300 import synth
from test_gpu_front import FILLERS, run

pytestmark = pytest.mark.gpu


def open_tiles(ctx):
    """Count of tiles whose pixels were open at the end of the sorted part: word 7 of the work counters,
    the third 256-byte block of the forward's workspace."""
    torch.cuda.synchronize()
    return int(ctx.workspace[512:544].view(torch.int32)[7])


@pytest.mark.parametrize("tile,persistent", [(32, False), (32, True), (16, False)])
def test_front_goes_past_an_outlier(tile, persistent):
    rng = np.random.default_rng(3)
    cam = synth.look_at_camera((0.5, 0.5, -1.0), (0.5, 0.5, 1.0), 64, 32, 60.0, z_near=1e-3)
    fx, cx, cy = cam["fx"], cam["cx"], cam["cy"]
    # an opaque lattice over the whole left half at depth 10, then 60,000 voxels within 0.04 behind it: one bin
    # of the 2048 between the outlier's depth and theirs
    gx, gy = np.meshgrid(np.arange(0.0, 33.0, 2.0), np.arange(0.0, 33.0, 2.0))
    m = 60000
    u = np.concatenate([[tile / 2 + 0.5], gx.ravel(), rng.uniform(0.0, 32.0, m)])
    v = np.concatenate([[tile / 2 + 0.5], gy.ravel(), rng.uniform(0.0, 32.0, m)])
    d = np.concatenate([[0.02], np.full(gx.size, 10.0), rng.uniform(10.005, 10.04, m)])
    c = np.stack([0.5 - (u - cx) * d / fx, 0.5 - (v - cy) * d / fx, d - 1.0], 1)
    half = 2.0 * d / fx
    half[0] = 1e-5
    dens = np.full(len(c), 200.0)
    dens[0] = 0.0
    at = np.sort(rng.choice(len(c) + FILLERS, len(c), replace=False))
    order = rng.permutation(len(c))
    c, half, dens = c[order], half[order], dens[order]
    small = synth.constant_voxel_scene(c, half, dens, rng.uniform(0.1, 0.9, (len(c), 3)))
    big = np.empty((len(c) + FILLERS, 3))
    big[:] = [0.5, 0.5, -9.0]
    big_half, big_dens = np.full(len(big), 0.01), np.full(len(big), 1.0)
    big[at], big_half[at], big_dens[at] = c, half, dens
    large = synth.constant_voxel_scene(big, big_half, big_dens, np.full((len(big), 3), 0.5))
    large["sh"][at] = small["sh"]
    a, sa, dda, _ = run(small, cam, tile=tile, persistent=persistent)
    b, sb, ddb, _ = run(large, cam, tile=tile, persistent=persistent)
    for name in ("rgb", "depth", "T", "n_contrib", "n_samples"):
        assert torch.equal(getattr(a, name), getattr(b, name)), name
    ids = torch.as_tensor(at, device="cuda")
    for name in ("wmax_packed", "z_min", "delta_min", "seen"):
        assert torch.equal(getattr(a, name), getattr(b, name)[ids]), name
    assert float((dda - ddb[ids]).abs().max()) <= 1e-4 * float(dda.abs().max())
    left = a.T.view(32, 64)[:, :32]
    assert float(left.max()) < 1e-4  # every pixel of the crowded tiles stops
    assert open_tiles(b) == 0
