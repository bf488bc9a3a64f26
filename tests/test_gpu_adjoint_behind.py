"""Table gradient entry by entry, for entries reached only behind others: every entry keeps the relative
precision of FP32 terms, however small the transmittance in front of it.

15 slabs of one value, rising by one table node from slab to slab, one opacity throughout and no
termination: slab j is seen through 0.8^(8 j), down to 1e-11.  Slabs of 2, 8 and 32 samples: as many or
fewer lanes of a warp on one table interval.  Colours fall by 0.62 from node to node, so that no term of
the opacity gradient cancels by more than a factor of some 12.

Tolerance 2e-4 of each entry: the transmittance is a product of up to 480 factors, each rounded twice
(480 * 2 * 2^-24 = 5.7e-5), in front of the sample and behind it; the difference of a sample's colour and
what is behind it multiplies the rounding of the latter (about 1e-6) by 12; the lookup's weights (about
one half) are off by 15 * 2^-23 = 2e-6."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("n,brick,thick", [(16, 128, 4), (16, 16, 4), (512, 128, 4), (1024, 16, 4), (16, 128, 1),
                                           (16, 128, 16)])
def test_every_entry(n, brick, thick, storage):
    import paper_1012_2909_gb300 as vr
    nx, ny, nz = 9, 7, 15 * thick
    vol = np.empty((nz, ny, nx), np.float32)
    vol[:] = (np.arange(nz) // thick + 0.5)[:, None, None]
    node = np.minimum(np.arange(n), 16)  # larger tables: the nodes from 16 on are not reached
    tf = np.stack([0.62 ** node, 0.5 * 0.62 ** node, 0.9 * 0.62 ** node, np.full(n, 1.0 - 0.8 ** (4.0 / thick))], 1).astype(np.float32)
    cam = dict(type=0, eye=[0.0, 0.0, -8.0], right=[1.0, 0.0, 0.0], up=[0.0, 1.0, 0.0], fwd=[0.0, 0.0, 1.0],
               win=[0.0, float(nx), 0.0, float(ny)], width=nx, height=ny)
    dimg = np.random.default_rng(3).uniform(0.5, 1.0, (1, ny, nx, 4)).astype(np.float32)
    dimg[..., 3] = 0.0
    r = vr.Renderer(0, brick=brick, ert=2.0)
    r.load_cube(vol, storage)
    r.set_transfer_function(tf, 0.0, float(n - 1))
    r.set_camera(cam)
    dtf = torch.empty((n, 4), device="cuda")
    dvol = torch.empty(vol.shape, device="cuda")
    ref = oracle.backward(oracle.Scene(vol, tf, 0.0, float(n - 1), 0.5, 2.0), [cam], dimg.astype(np.float64),
                          "composite")[0]
    for voxels in (None, dvol):
        vr.vr_render_backward(r.ctx, "composite", torch.from_numpy(dimg).cuda(), dtf, voxels)
        got = dtf.cpu().numpy().astype(np.float64)
        assert (ref[:16] > 0).all() and not ref[16:].any() and not got[16:].any()
        err = np.abs(got[:16] - ref[:16]) / ref[:16]
        print(n, brick, thick, storage, "largest relative error of an entry", err.max(axis=0))
        assert err.max() <= 2e-4
    r.close()
