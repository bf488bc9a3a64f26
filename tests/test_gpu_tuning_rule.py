"""Setting a launch shape whose lanes per segment are the ones reported leaves the rule for them in force:
setting back what was read, or with another tile or block only, changes nothing.  Seen by the rounding of
the sort-last image, which the lanes decide."""
import json

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def scene():
    import paper_1012_2909_gb300 as vr
    dims = (70, 64, 66)
    r = vr.Renderer(0, brick=64)
    r.load_cube(synth.generate(synth.cube_params(*dims, seed=12, nsrc=6)), "f32")
    r.set_transfer_function(synth.viridis_ramp_tf(), -1.0, 20.0)
    r.set_camera(synth.orbit_view(dims, 50.0, 301, 201))  # rays less than a voxel apart
    r.set_path("sortlast")
    return r


def test_reported_lanes_set_back_leave_the_rule(tmp_path):
    import paper_1012_2909_gb300 as vr
    r = scene()

    def image():
        return r.render("composite").cpu().numpy()

    by_rule = image()
    t = vr.vr_get_tuning(r.ctx)
    assert t == dict(tile_w=8, tile_h=4, block=256, group=8)
    vr.vr_set_tuning(r.ctx, t)
    np.testing.assert_array_equal(image(), by_rule)
    vr.vr_set_tuning(r.ctx, dict(t, tile_w=16, tile_h=2, block=128))
    np.testing.assert_array_equal(image(), by_rule)
    r.set_path("ray")  # an image-order result carries lanes that were not timed
    best = vr.vr_autotune(r.ctx, "composite", torch.empty((1, 201, 301, 4), device="cuda"), reps=1)
    vr.vr_set_tuning(r.ctx, best)
    r.set_path("sortlast")
    np.testing.assert_array_equal(image(), by_rule)
    # lanes that were chosen stay chosen, also when they are the default's
    vr.vr_set_tuning(r.ctx, dict(t, group=16))
    vr.vr_set_tuning(r.ctx, t)
    eight = image()
    assert (eight != by_rule).any()
    vr.vr_set_tuning(r.ctx, vr.vr_get_tuning(r.ctx))
    np.testing.assert_array_equal(image(), eight)
    vr.vr_set_tuning(r.ctx, dict(t, group=4))
    np.testing.assert_array_equal(image(), by_rule)
    r.close()
    # so do lanes from a file of measured shapes, in a renderer of its own
    cache = str(tmp_path / "tune.json")
    for wanted in (None, 8, 4):
        r = scene()
        if wanted:
            with open(cache) as f:
                table = {k: dict(v, group=wanted) for k, v in json.load(f).items()}
            with open(cache, "w") as f:
                json.dump(table, f)
        r.set_path("brick")
        assert vr.autotune(r, "mip", reps=1, cache=cache)["cached"] == bool(wanted)
        r.set_path("sortlast")
        if wanted:
            np.testing.assert_array_equal(r.render("composite").cpu().numpy(), eight if wanted == 8 else by_rule)
        r.close()
