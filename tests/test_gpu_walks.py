"""The composites' walks give the same bits however they are batched: one view of few
strips takes the kernels that look ahead, a schedule cut to fewer SMs and a batch of
48 equal views the others.  Lists shorter than, equal to and just beyond the walks'
batches and rounds, with pixels that stop at once, late or never."""
import pytest
import torch

from paper_2511_02510_gb300.raster import RasterContext, Scene
from test_gpu_front import scenes

pytestmark = pytest.mark.gpu

COUNTS = [1, 15, 16, 17, 33, 96, 97, 129, 300, 2000]


def run(sc, cams, **kw):
    scene = Scene.from_numpy(sc, "cuda")
    ctx = RasterContext(cams, scene.n, **kw)
    vox = scene.voxels()
    ctx.fit_capacity(vox)
    ctx.reset_stats()
    ctx.forward(vox)
    g = torch.linspace(-1.0, 1.0, 3 * ctx.n_pix // len(cams), device="cuda").repeat(len(cams)).view(-1, 3)
    d_density, d_sh = ctx.backward(vox, g, g[:, 0].contiguous(), g[:, 1].contiguous())
    ctx.check()
    return ctx, d_density, d_sh


@pytest.mark.parametrize("density", [0.02, 1.5, 60.0])
@pytest.mark.parametrize("tile,segment", [(8, False), (16, True), (32, False)])
def test_walks_give_the_same_bits(density, tile, segment):
    sc, _, _, cam = scenes(COUNTS, density, 0, tile, 5)
    views = 48
    a, dda, dsa = run(sc, [cam], tile=tile, exact_segment=segment)  # 320 strips: looks ahead
    b, ddb, dsb = run(sc, [cam], tile=tile, exact_segment=segment, persistent=True, persistent_sms=3)
    many = [run(sc, [cam] * views, tile=tile, exact_segment=segment, persistent=p) for p in (False, True)]
    n = a.n_pix
    for name in ("rgb", "depth", "T", "n_contrib", "n_samples"):
        x = getattr(a, name)
        assert torch.equal(x, getattr(b, name)), name
        for c, _, _ in many:
            y = getattr(c, name)
            assert all(torch.equal(x, y[v * n:(v + 1) * n]) for v in range(views)), name
    for name in ("wmax_packed", "z_min", "delta_min", "seen"):
        for c in [b] + [m[0] for m in many]:
            assert torch.equal(getattr(a, name), getattr(c, name)), name
    # atomic sums in another order: FP32 rounding of the sums
    for x, y in [(dda, ddb), (dsa, dsb)] + [(dda, m[1] / views) for m in many] + [(dsa, m[2] / views) for m in many]:
        assert float((x - y).abs().max()) <= 1e-4 * float(x.abs().max())
