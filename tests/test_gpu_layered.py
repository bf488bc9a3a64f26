"""The layered composite of a cube in core (one thread per ray over its bricks) against the
streamed cube's layers (one launch per visibility layer, state carried in memory): the same
ownership, positions and operations, so the same image bit for bit."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DIMS = (75, 130, 41)  # ragged against every brick edge


def _cams():
    w, h = 61, 37  # ragged against the 8 x 4 tiles
    views = [synth.look_at(DIMS, d, w, h) for d in ((0.4, 0.3, 1.0), (-0.7, 0.5, -0.6), (0.0, 0.0, -1.0))]
    views.append(synth.look_at(DIMS, (0.3, -0.2, 1.0), w, h, dist_factor=0.2))  # eye inside
    views.append(synth.ortho_view(DIMS, w, h, rx_deg=-35.0, ry_deg=160.0))
    views.append(dict(synth.axis_view(DIMS, w, h), eye=[8.0, 3.0, -10.0]))  # along z, on voxel centres
    views.append(synth.look_at(DIMS, (1.0, 0.0, 0.0), w, h, fov_deg=5.0, up_hint=(0.0, 0.0, 1.0)) |
                 {"eye": [500.0, 500.0, 500.0]})  # miss
    return views


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("brick,ert,single", [(32, 0.99, False), (64, 2.0, True), (32, 0.3, True)])
def test_layered_equals_layer_launches(storage, brick, ert, single):
    import paper_1012_2909_gb300 as vr
    p = synth.cube_params(*DIMS, seed=5, nsrc=9)
    tf = synth.viridis_ramp_tf()
    tf[:30, 3] = 0.0  # some bricks transparent or nearly so
    fn, user = synth.region_callback(p, 2)
    got = []
    for streamed in (False, True):
        r = vr.Renderer(0, brick=brick, ert=ert, single_store=single)
        if streamed:
            vr.vr_load_cube_streamed(r.ctx, fn, user, DIMS, storage, 1 << 27)
        else:
            r.load_cube(synth.generate(p), storage)
            r.set_path("layered")
        r.set_transfer_function(tf, -1.0, 20.0)
        r.set_camera(_cams())
        got.append(r.render("composite").cpu().numpy())
        r.close()
    assert np.count_nonzero(got[0][:-1]) > 0 and not got[0][-1].any()
    np.testing.assert_array_equal(got[0], got[1])
