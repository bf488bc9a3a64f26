"""The marcher's and the layered composite's compiled forms (default brick edge and tables of up to
256 entries) and their general ones, against the oracle: bricks and tables on either side of the
line, steps of several voxels, views inside, along an axis and from far away.

Tolerance 1e-4 per channel, as for every FP32 render of the rounded cube (rays flagged by the
oracle may take its alternative outcomes)."""
import pytest

import oracle
import synth
from tests.parity import compare

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DIMS = (131, 37, 150)  # two bricks of 128 along x and z, ragged


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("brick,ntf,step", [(128, 256, 0.5), (128, 257, 0.5), (64, 256, 0.5), (256, 256, 3.7),
                                            (128, 256, 3.7), (128, 2, 40.0)])
def test_forms_against_oracle(storage, brick, ntf, step):
    import paper_1012_2909_gb300 as vr
    vol = synth.generate(synth.cube_params(*DIMS, seed=12, nsrc=9))
    tf = synth.viridis_ramp_tf(ntf)
    w, h = 43, 29
    cams = [synth.look_at(DIMS, (0.6, 0.3, 1.0), w, h), synth.look_at(DIMS, (-1.0, 0.1, -0.4), w, h),
            synth.look_at(DIMS, (0.2, -0.3, 1.0), w, h, dist_factor=0.1),
            synth.ortho_view(DIMS, w, h, rx_deg=-15.0, ry_deg=200.0),
            dict(synth.axis_view(DIMS, w, h), eye=[90.0, 4.0, -3.0]),
            synth.look_at(DIMS, (0.5, 0.6, -0.8), w, h, fov_deg=0.06, dist_factor=1000.0)]
    sc = oracle.Scene(oracle.round_storage(vol, storage), tf, -1.0, 20.0, step, 0.9)
    r = vr.Renderer(0, brick=brick, step=step, ert=0.9)
    r.load_cube(vol, storage)
    r.set_transfer_function(tf, -1.0, 20.0)
    r.set_camera(cams)
    for mode, path in (("composite", "ray"), ("mip", "ray"), ("composite", "layered")):
        r.set_path(path)
        img = r.render(mode).cpu().numpy()
        for i, c in enumerate(cams):
            compare(img[i].reshape(-1, 4), sc, c, mode, tol=1e-4, path=path)
    r.close()
