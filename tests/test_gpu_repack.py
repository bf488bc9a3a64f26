"""The brick store made from a device cube (one launch) and from a host cube (slab by slab),
with and without the copy shifted by one element: the same images, and the oracle's values."""
import numpy as np
import pytest

import oracle
import synth
from tests.parity import compare

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("brick,dims", [(8, (17, 8, 9)), (16, (1, 33, 15)), (32, (64, 31, 65)), (256, (130, 3, 257))])
def test_store_from_device_and_host(storage, brick, dims):
    import paper_1012_2909_gb300 as vr
    vol = synth.generate(synth.cube_params(*dims, seed=21, nsrc=3))
    tf = synth.viridis_ramp_tf()
    cams = [synth.look_at(dims, d, 45, 27) for d in ((0.5, 0.4, 1.0), (-1.0, 0.2, -0.3))]
    sc = oracle.Scene(oracle.round_storage(vol, storage), tf, -1.0, 20.0, 0.5, 0.99)
    ref = None
    for source in ("device", "host"):
        for single in (False, True):
            r = vr.Renderer(0, brick=brick, single_store=single)
            for first in (vol[::-1].copy(), vol):  # a second load replaces the first
                r.load_cube(torch.from_numpy(first).cuda() if source == "device" else first, storage)
            r.set_transfer_function(tf, -1.0, 20.0)
            r.set_camera(cams)
            got = [r.render("composite").cpu().numpy(), r.render("mip").cpu().numpy()]
            r.close()
            if ref is None:
                ref = got
                for i, c in enumerate(cams):
                    compare(got[0][i].reshape(-1, 4), sc, c, "composite", tol=1e-4)
                    compare(got[1][i].reshape(-1, 4), sc, c, "mip", tol=1e-4)
            for a, b in zip(ref, got):
                np.testing.assert_array_equal(a, b)


def test_replaced_cubes_equal_fresh_ones():
    """A renderer that loads cube after cube, with and without taking over the buffers (the same
    bricks, or another size or type width), against a fresh renderer for each."""
    import paper_1012_2909_gb300 as vr
    tf = synth.viridis_ramp_tf()
    kept = vr.Renderer(0, brick=64)
    for i, (dims, storage, host) in enumerate((((90, 70, 65), "f16", False), ((100, 66, 128), "bf16", False),
                                               ((100, 66, 128), "f32", False), ((90, 70, 65), "f32", True),
                                               ((90, 70, 60), "f16", True), ((90, 70, 65), "f16", False))):
        vol = synth.generate(synth.cube_params(*dims, seed=40 + i, nsrc=5))
        src = vol if host else torch.from_numpy(vol).cuda()
        got = []
        for r in (kept, vr.Renderer(0, brick=64)):
            r.load_cube(src, storage)
            r.set_transfer_function(tf, -1.0, 20.0)
            r.set_camera(synth.look_at(dims, (0.4, 0.3, 1.0), 45, 27))
            for mode, path in (("composite", "ray"), ("composite", "layered"), ("composite", "sortlast"), ("mip", "brick")):
                r.set_path(path)
                got.append(r.render(mode).cpu().numpy())
            assert r.cube_info()["nx"] == dims[0] and r.cube_info()["nz"] == dims[2]
        for a, b in zip(got[:4], got[4:]):
            np.testing.assert_array_equal(a, b)
