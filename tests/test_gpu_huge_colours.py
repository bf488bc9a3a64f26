"""A ray that ends before an interval whose end colours lie further apart than FP32 reaches: the samples
fetched together with its last one are not part of its image."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("n,brick", [(4, 128), (4, 32), (300, 128)])
@pytest.mark.parametrize("path", ["ray", "layered"])
def test_samples_past_the_end_add_nothing(path, n, brick, storage):
    import paper_1012_2909_gb300 as vr
    vol = np.full((20, 5, 6), 2.5, np.float32)
    vol[0] = 0.0
    tf = np.full((n, 4), 0.5, np.float32)
    tf[:, 3] = 1.0
    tf[2, :3], tf[3, :3] = 3e38, -3e38  # the interval of 2.5
    r = vr.Renderer(0, brick=brick)
    r.load_cube(vol, storage)
    r.set_transfer_function(tf, 0.0, float(n - 1))
    r.set_camera(dict(type=0, eye=[0.0, 0.0, -8.0], right=[1.0, 0.0, 0.0], up=[0.0, 1.0, 0.0], fwd=[0.0, 0.0, 1.0],
                      win=[0.0, 6.0, 0.0, 5.0], width=6, height=5))
    r.set_path(path)
    img = r.render("composite").cpu().numpy()
    np.testing.assert_array_equal(img, np.broadcast_to(np.float32([0.5, 0.5, 0.5, 1.0]), img.shape))
    r.close()


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("brick", [128, 32])
@pytest.mark.parametrize("path", ["ray", "layered"])
def test_transmittance_beyond_fp32(path, brick, storage):
    """Opacity -9: the transmittance grows by 10 a sample and the colour sum ends at -inf, not at NaN."""
    import paper_1012_2909_gb300 as vr
    tf = np.full((4, 4), 0.5, np.float32)
    tf[:, 3] = -9.0
    r = vr.Renderer(0, brick=brick)
    r.load_cube(np.full((41, 5, 6), 1.5, np.float32), storage)
    r.set_transfer_function(tf, 0.0, 3.0)
    r.set_camera(dict(type=0, eye=[0.0, 0.0, -8.0], right=[1.0, 0.0, 0.0], up=[0.0, 1.0, 0.0], fwd=[0.0, 0.0, 1.0],
                      win=[0.0, 6.0, 0.0, 5.0], width=6, height=5))
    r.set_path(path)
    img = r.render("composite").cpu().numpy()
    np.testing.assert_array_equal(img, np.full_like(img, -np.inf))
    r.close()
