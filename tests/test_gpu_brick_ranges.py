"""Stored value ranges of the bricks: exactly those of a brick's stored voxels (ghost layer included).

A plane of bright voxels one row past a brick's ghost layer must leave the brick transparent; in the
ghost layer it must not.  The image cannot tell (a wide range only skips less), the count of executed
samples can: rays along z through voxel centres take 2 nz samples, all of them in bricks of one y row,
which are skipped together or not at all."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("brick", [8, 16, 32, 64, 128, 256])
def test_ranges_hold_the_stored_voxels_only(storage, brick):
    import paper_1012_2909_gb300 as vr
    nx, ny, nz = brick + 3, 2 * brick + 5, brick + 2
    tf = synth.viridis_ramp_tf()
    tf[:, 3] = np.where(-1.0 + 21.0 * np.arange(256) / 255.0 < 6.0, 0.0, 1e-3)
    cam = dict(type=0, eye=[0.0, 0.0, -8.0], right=[1.0, 0.0, 0.0], up=[0.0, 1.0, 0.0], fwd=[0.0, 0.0, 1.0],
               win=[0.0, float(nx), 0.0, float(ny)], width=nx, height=ny)
    r = vr.Renderer(0, brick=brick, ert=2.0)
    counter = torch.zeros(1, dtype=torch.int64, device="cuda")
    for y in (brick - 2, brick, brick + 1, 2 * brick - 2):
        vol = torch.zeros((nz, ny, nx), device="cuda")
        vol[:, y] = 15.0
        r.load_cube(vol, storage)
        r.set_transfer_function(tf, -1.0, 20.0)
        r.set_camera(cam)
        counter.zero_()
        vr.vr_set_sample_counter(r.ctx, counter)
        r.render("composite")
        vr.vr_set_sample_counter(r.ctx, None)
        rows = 0  # pixel rows of the brick rows whose stored voxels, y0 - 1 .. y0 + brick, hold the plane
        for y0 in range(0, ny, brick):
            if y0 - 1 <= y <= y0 + brick:
                rows += min(brick, ny - y0)
        assert int(counter.item()) == rows * nx * 2 * nz
    r.close()
