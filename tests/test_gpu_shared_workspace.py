"""The calls that take a forward's workspace as const only read it, also where the
forward left very long lists partly sorted: its bytes stay, calls on two streams over
one workspace give the bits of one call, and the lists and pixels they give are those
of the whole order."""
import numpy as np
import pytest
import torch

from gpu_helpers import gpu_pairs
from paper_2511_02510_gb300 import litevoxel as L
from test_gpu_front import run, scenes

pytestmark = pytest.mark.gpu


def pairs_of(ctx, n, keys, vox):
    L.lv_debug_pairs(n, ctx.cams_arr, ctx.n_views, ctx.opts, ctx.workspace, ctx.pair_capacity, keys, vox, None)


def pixels_of(ctx, scene, px, rgb, T):
    L.lv_render_pixels_f64(scene.voxels(), ctx.cams_arr, ctx.n_views, ctx.opts, ctx.workspace, ctx.pair_capacity, px,
                           rgb, T)


# dense voxels: every pixel stops in a list's sorted front; then the densities fall, and the FP64 march
# goes through the rest: of plain lists, with more equal depths there than one sort takes, and by segment
@pytest.mark.parametrize("counts,equal,tile,segment", [
    ([30000, 20000, 300, 5], 0, 32, False),
    ([60000, 20000, 300, 5], 9000, 32, True),
    ([30000, 20000, 300, 5], 0, 8, False),
])
def test_const_workspace_is_only_read(ora, counts, equal, tile, segment):
    small, large, at, cam = scenes(counts, 60.0, equal, tile, 11)
    a, sa, _, _ = run(small, cam, tile=tile, persistent=False, exact_segment=segment)
    b, sb, _, _ = run(large, cam, tile=tile, persistent=False, exact_segment=segment)
    for s in (sa, sb):
        s.density.mul_(0.02 / 60.0)
    px = torch.arange(0, b.n_pix, 7, device="cuda")
    before = b.workspace.clone()
    ref = ora.pairs(large, [cam], ts=tile)
    keys, vox, ranges, pairs = gpu_pairs(b, sb.n)
    assert pairs == ref["n_pairs"]
    np.testing.assert_array_equal(keys, ref["keys"])
    np.testing.assert_array_equal(vox, ref["vals"])
    np.testing.assert_array_equal(ranges, ref["ranges"])

    def buffers():
        return (torch.empty((px.numel(), 3), dtype=torch.float64, device="cuda"),
                torch.empty(px.numel(), dtype=torch.float64, device="cuda"),
                torch.zeros(pairs, dtype=torch.int64, device="cuda"),
                torch.zeros(pairs, dtype=torch.int32, device="cuda"))

    whole, one, two, three = buffers(), buffers(), buffers(), buffers()
    pixels_of(a, sa, px, whole[0], whole[1])
    pixels_of(b, sb, px, one[0], one[1])
    pairs_of(b, sb.n, one[2], one[3])
    # each sample's terms are within some 50 roundings of FP64, and a pixel has at most its list's samples
    for x, y in zip(whole[:2], one[:2]):
        assert float((x - y).abs().max()) <= max(counts) * 50 * 2.0 ** -53
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(3):
        for s, o in ((s1, two), (s2, three)):
            with torch.cuda.stream(s):
                pixels_of(b, sb, px, o[0], o[1])
                pairs_of(b, sb.n, o[2], o[3])
    torch.cuda.synchronize()
    for x, y, z in zip(one, two, three):
        assert torch.equal(x, y) and torch.equal(x, z)
    assert torch.equal(b.workspace, before)
