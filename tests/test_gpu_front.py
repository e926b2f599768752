"""Composites over partly sorted lists: in large scenes only the front of a very
long list is depth-sorted before the composite, and the rest for the tiles whose
pixels are still open, whose march then goes on in a second launch.  Voxels
behind the camera make a scene large without being seen; without them the same
lists are sorted whole, and every output has to be the same bits.  (The whole
order against the oracle is checked too.)"""
import numpy as np
import pytest
import torch

from gpu_helpers import gpu_pairs
from paper_2511_02510_gb300 import synth
from paper_2511_02510_gb300.raster import RasterContext, Scene

pytestmark = pytest.mark.gpu

FILLERS = (1 << 19) + 1  # scenes of more voxels sort only the front of a list above 16384 entries


def scenes(counts, density, equal, tile, seed):
    """A (32 * len(counts)) x 32 view with counts[t] voxels of about a pixel in a tile of its t-th 32 columns,
    the first `equal` of t = 0 at one depth: alone, and with the voxels behind the camera in between."""
    rng = np.random.default_rng(seed)
    cam = synth.look_at_camera((0.5, 0.5, -1.0), (0.5, 0.5, 1.0), 32 * len(counts), 32, 60.0, z_near=1e-3)
    fx, cx, cy = cam["fx"], cam["cx"], cam["cy"]
    cents = []
    for t, m in enumerate(counts):
        d = np.exp(rng.uniform(np.log(0.5), np.log(40.0), m))
        if t == 0:
            d[:equal] = 2.0
        h = 0.5 * tile
        u, v = 32.0 * t + h + rng.uniform(-h + 1.5, h - 1.5, m), h + rng.uniform(-h + 1.5, h - 1.5, m)
        cents.append(np.stack([0.5 - (u - cx) * d / fx, 0.5 - (v - cy) * d / fx, d - 1.0], 1))
    c = np.concatenate(cents)
    c = c[rng.permutation(len(c))]
    half = 1.2e-2 * (c[:, 2] + 1.0)
    at = np.sort(rng.choice(len(c) + FILLERS, len(c), replace=False))
    big = np.empty((len(c) + FILLERS, 3))
    big[:] = [0.5, 0.5, -9.0]
    big_half = np.full(len(big), 0.01)
    big[at], big_half[at] = c, half
    small = synth.constant_voxel_scene(c, half, density, rng.uniform(0.1, 0.9, (len(c), 3)))
    large = synth.constant_voxel_scene(big, big_half, density, np.full((len(big), 3), 0.5))
    large["sh"][at], large["density"][at] = small["sh"], small["density"]
    return small, large, at, cam


def run(sc, cam, **kw):
    scene = Scene.from_numpy(sc, "cuda")
    ctx = RasterContext([cam], scene.n, **kw)
    vox = scene.voxels()
    ctx.fit_capacity(vox)
    ctx.reset_stats()
    ctx.forward(vox)
    g = torch.linspace(-1.0, 1.0, 3 * ctx.n_pix, device="cuda").view(-1, 3)
    d_density, d_sh = ctx.backward(vox, g, g[:, 0].contiguous(), g[:, 1].contiguous())
    ctx.check()
    return ctx, scene, d_density, d_sh


@pytest.mark.parametrize("counts,density,equal,tile,persistent,segment", [
    ([40000, 16385, 16384, 300], 0.02, 0, 32, False, False),   # every pixel stays open
    ([40000, 30000, 5000, 300], 1.5, 0, 16, False, False),     # some stop in the front, some in the rest
    ([60000, 20000, 300, 5], 0.02, 9000, 32, True, False),     # more equal depths than a sort takes
    ([30000, 20000, 300, 5], 0.02, 20000, 8, True, True),      # the nearest sorted part is equal depths
    ([30000, 20000, 300, 5], 60.0, 0, 32, True, False),        # every pixel stops in the front
])
def test_partly_sorted_lists_give_the_same_bits(ora, counts, density, equal, tile, persistent, segment):
    small, large, at, cam = scenes(counts, density, equal, tile, 7)
    kw = dict(tile=tile, persistent=persistent, exact_segment=segment)
    a, sa, dda, dsa = run(small, cam, **kw)
    b, sb, ddb, dsb = run(large, cam, **kw)
    for name in ("rgb", "depth", "T", "n_contrib", "n_samples"):
        assert torch.equal(getattr(a, name), getattr(b, name)), name
    ids = torch.as_tensor(at, device="cuda")
    for name in ("wmax_packed", "z_min", "delta_min", "seen"):
        assert torch.equal(getattr(a, name), getattr(b, name)[ids]), name
    # atomic sums in another order: FP32 rounding of the sums
    for x, y in ((dda, ddb[ids]), (dsa, dsb[ids])):
        assert float((x - y).abs().max()) <= 1e-4 * float(x.abs().max())
    # the calls that read whole lists complete them
    keys, vox, ranges, pairs = gpu_pairs(b, sb.n)
    ref = ora.pairs(large, [cam], ts=tile)
    assert pairs == ref["n_pairs"]
    np.testing.assert_array_equal(keys, ref["keys"])
    np.testing.assert_array_equal(vox, ref["vals"])
    np.testing.assert_array_equal(ranges, ref["ranges"])
