"""Small cubes under many pixels: a staged cell's pixels are split into row bands among CTAs.  The
same maxima as the image-order marcher's and the same sort-last image as the oracle's, for one
camera and several, image sizes around the bands' limits, and fewer rows than bands.

Tolerances as elsewhere: 1e-4 against the oracle; 2e-3 between the two paths' maxima (values up to
20, positions within 3e-5 voxel on the staged path)."""
import numpy as np
import pytest

import oracle
import synth
from tests.parity import compare

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("dims,size,ncam", [((33, 20, 40), (701, 333), 1), ((33, 20, 40), (901, 7), 2),
                                            ((70, 50, 64), (640, 480), 3), ((5, 4, 3), (1024, 257), 1)])
def test_bands(storage, dims, size, ncam):
    import paper_1012_2909_gb300 as vr
    vol = synth.generate(synth.cube_params(*dims, seed=3, nsrc=3))
    tf = synth.viridis_ramp_tf()
    cams = [synth.orbit_view(dims, 20.0 + 100.0 * i, *size) for i in range(ncam)]
    r = vr.Renderer(0, brick=64)
    r.load_cube(vol, storage)
    r.set_transfer_function(tf, -1.0, 20.0)
    r.set_camera(cams)
    got = {}
    for path in ("ray", "brick"):
        r.set_path(path)
        got[path] = r.render("mip", with_max=True)[1].cpu().numpy()
    hit = np.isfinite(got["ray"])
    assert hit.any() and np.array_equal(hit, np.isfinite(got["brick"]))
    assert np.abs(got["ray"][hit] - got["brick"][hit]).max() <= 2e-3
    r.set_path("sortlast")
    img = r.render("composite").cpu().numpy()
    sc = oracle.Scene(oracle.round_storage(vol, storage), tf, -1.0, 20.0, 0.5, 2.0)
    pix = np.random.default_rng(2).choice(size[0] * size[1], 1500, replace=False)
    for i, c in enumerate(cams):
        compare(img[i].reshape(-1, 4)[pix], sc, c, "composite", pixels=pix, tol=1e-4, path="sortlast")
    r.close()
