"""Table gradients: the fixed-point histograms of a ray and the FP32 path for what they cannot hold.

Tolerance 1e-4 against the FP64 adjoint (relative to the largest entry): the gradient sums FP32 products
of some 1e-6 relative error (sample values, transmittance products over up to 2000 samples); a histogram
rounds a sample by 2^-22 of the ray's bound at most."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DIMS = (24, 20, 28)


def _grad(tf, step, ert, scale=1.0, spoil=None):
    import paper_1012_2909_gb300 as vr
    vol = synth.generate(synth.cube_params(*DIMS, seed=8, nsrc=4))
    views = synth.random_views(DIMS, 2, seed=4, width=21, height=13)
    r = vr.Renderer(0, brick=16, step=step, ert=ert)
    r.load_cube(vol, "f32")
    r.set_transfer_function(tf, -1.0, 20.0)
    r.set_camera(views)
    dimg = np.random.default_rng(1).normal(size=(2, 13, 21, 4)).astype(np.float32)
    if spoil is not None:
        dimg[0, 6, 10, 1] = spoil
    d = (torch.from_numpy(dimg) * scale).cuda()
    dtf = torch.empty((len(tf), 4), device="cuda")
    dvol = torch.empty(vol.shape, device="cuda")
    vr.vr_render_backward(r.ctx, "composite", d, dtf, dvol)
    out = dtf.cpu().numpy().astype(np.float64), dvol.cpu().numpy()
    only = torch.empty_like(dtf)  # the table alone: no voxel gradients
    vr.vr_render_backward(r.ctx, "composite", d, only, None)
    np.testing.assert_allclose(only.cpu().numpy(), out[0], rtol=1e-4, atol=1e-5 * np.abs(out[0]).max())
    r.close()
    return out, oracle.Scene(vol, tf, -1.0, 20.0, step, ert), views, dimg


def _table(n, alpha):
    t = synth.hidden_tf(5, n)
    t[:, 3] = np.linspace(0.0, 1.0, n) * alpha
    return t


@pytest.mark.parametrize("n", [2, 256, 1024])
@pytest.mark.parametrize("alpha,step", [(1.0, 0.5), (0.05, 0.02), (1.3, 0.5)])  # ends early; 70 chunks; beyond [0, 1]
def test_against_oracle(n, alpha, step):
    (dtf, dvol), sc, views, dimg = _grad(_table(n, alpha), step, 2.0)
    ref, ref_vol = oracle.backward(sc, views, dimg.astype(np.float64), "composite")
    assert np.abs(dtf - ref).max() <= 1e-4 * np.abs(ref).max()
    assert np.linalg.norm(dvol - ref_vol) <= 1e-3 * np.linalg.norm(ref_vol)  # table kinks (one-sided slopes)


def test_scales_and_non_finite():
    tf = _table(256, 1.0)
    base = _grad(tf, 0.5, 0.99)[0][0]
    for scale in (2.0 ** -90, 2.0 ** 60):
        got = _grad(tf, 0.5, 0.99, scale=scale)[0][0]
        assert np.abs(got / scale - base).max() <= 1e-5 * np.abs(base).max()
    got = _grad(tf, 0.5, 0.99, spoil=1e31)[0][0]  # one ray through the FP32 path
    assert np.isfinite(got).all() and np.abs(got[:, 1]).max() > 1e28
    assert np.isnan(_spoilt(tf, np.nan)).any()


def _spoilt(tf, value):
    import paper_1012_2909_gb300 as vr
    vol = synth.generate(synth.cube_params(*DIMS, seed=8, nsrc=4))
    r = vr.Renderer(0, brick=16)
    r.load_cube(vol, "f32")
    r.set_transfer_function(tf, -1.0, 20.0)
    r.set_camera(synth.random_views(DIMS, 1, seed=4, width=21, height=13))
    d = torch.zeros((1, 13, 21, 4), device="cuda")
    d[0, 6, 10, 1] = value
    dtf = torch.empty((len(tf), 4), device="cuda")
    vr.vr_render_backward(r.ctx, "composite", d, dtf, None)
    out = dtf.cpu().numpy()
    r.close()
    return out
