"""Discs thousands of image widths across, far away (a sky or a ground plane):
the products of their projected ellipse underflow in float32, and they must
still cover the image."""
import numpy as np
import pytest

import oracle
import scenegen as sg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_17545_gb300 import render as R
    return R


@pytest.mark.parametrize("z,scale,focal", [(1000.0, 8e4, 60.0), (1000.0, 5e3, 1000.0), (1e4, 1e5, 2000.0)])
@pytest.mark.parametrize("tilt", [0.0, 0.2])
@pytest.mark.parametrize("samples", [1, 4])
def test_far_wide_discs_cover_the_image(R, z, scale, focal, tilt, samples):
    f32 = lambda a: np.ascontiguousarray(a, np.float32)  # noqa: E731
    q = np.array([[np.cos(tilt), np.sin(tilt), 0.0, 0.0]])
    scene = sg.Scene(0, f32([[3.0, 5.0, z]]), f32(q), f32([[scale, 0.7 * scale]]), f32([[[0.3, 0.1, -0.2]]]),
                     f32([[0.0, 0.0, 0.9 * z]]), f32(q), f32([[scale, scale]]), f32([0.5]), f32([[[0.1, 0.2, 0.3]]]))
    scene.g_scale = f32([[scale, scale]])        # a 2D Gaussian of the same kind, in front
    cam = sg.Camera(70, 45, focal, focal, 35.0, 22.5, np.concatenate([np.eye(3), np.zeros((3, 1))], 1), 0.01, (.1, .2, .3))
    gs = R.GESScene.from_arrays(scene)
    out = R.render(gs, cam, dict(samples=samples))
    gs.close()
    ref = oracle.render(scene, cam, dict(samples=samples), culled=False)
    assert (ref["id"] == 0).all() and (ref["wg"] > 0.4).all()
    assert (out["id"].cpu().numpy().reshape(ref["id"].shape) == 0).all()
    assert np.abs(out["rgb"].cpu().numpy() - ref["rgb"]).max() <= 2e-4
