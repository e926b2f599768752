"""The batch changes no launch, so the autotuner times a tile and schedule once: the time
stands for every accepted batch, and no candidate gets more chances than another."""
import pytest
import torch

from paper_2511_02510_gb300 import litevoxel as L
from paper_2511_02510_gb300 import synth

pytestmark = pytest.mark.gpu


def test_one_time_per_tile_and_schedule():
    sc = synth.scene_tiny()
    arrays = [torch.as_tensor(sc[k]).cuda() for k in ("geom", "density", "sh")]
    vox = L.make_voxels(*arrays)
    cams = L.make_cameras([synth.orbit_camera(128, 96, 60.0, 3.0, 20.0, 15.0)])
    base, cap = L.make_opts(batch=64), 400000
    ws = torch.empty(L.lv_autotune_workspace_size(vox.n, cams, 1, base, cap), dtype=torch.uint8, device="cuda")
    before = L.launch_count()
    best, ms = L.lv_autotune(vox, cams, 1, base, cap, 2, ws)
    passes = L.launch_count() - before
    assert best.batch == 32
    for t in range(3):
        for p in range(2):
            row = list(ms[6 * t + 3 * p:6 * t + 3 * p + 3])
            assert row[0] > 0 and row[1] == row[0] and row[2] == (-1 if t == 2 else row[0])
    # six candidates of three forward + backward passes each, of at most 16 launches
    assert passes <= 6 * 3 * 16
