"""Lanes per segment of the staged-cell passes on either side of the rule's spacings: the maxima are
those of every tuning, bit for bit, and the sort-last image is the oracle's (1e-4, as elsewhere)."""
import numpy as np
import pytest

import oracle
import synth
from tests.parity import compare

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("size", [(19, 13), (61, 43), (129, 97), (401, 299)])  # some 16 to 0.6 voxels a pixel
def test_group_rule(storage, size):
    import paper_1012_2909_gb300 as vr
    dims = (190, 101, 150)
    vol = synth.generate(synth.cube_params(*dims, seed=5, nsrc=4))
    tf = synth.viridis_ramp_tf()
    cam = synth.orbit_view(dims, 73.0, *size)
    r = vr.Renderer(0, brick=64)
    r.load_cube(vol, storage)
    r.set_transfer_function(tf, -1.0, 20.0)
    r.set_camera(cam)
    r.set_path("sortlast")
    img = r.render("composite").cpu().numpy().reshape(-1, 4)
    sc = oracle.Scene(oracle.round_storage(vol, storage), tf, -1.0, 20.0, 0.5, 2.0)
    pix = np.random.default_rng(2).choice(size[0] * size[1], min(1500, size[0] * size[1]), replace=False)
    compare(img[pix], sc, cam, "composite", pixels=pix, tol=1e-4, path="sortlast")
    r.set_path("brick")
    by_rule = r.render("mip", with_max=True)[1].clone()
    assert torch.isfinite(by_rule).any()
    for group in (4, 8):
        vr.vr_set_tuning(r.ctx, dict(tile_w=8, tile_h=4, block=256, group=group))
        assert torch.equal(r.render("mip", with_max=True)[1], by_rule)
    r.close()
