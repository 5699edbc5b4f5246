"""The translucent backward on either side of the tile count where its sweep
changes its registers per thread (three CTAs per SM hold all tiles up to 456),
against the float64 oracle."""
import numpy as np
import pytest

import oracle
import scenegen as sg

pytestmark = pytest.mark.gpu

GRAD_TOL = 1e-3


@pytest.fixture(scope="module")
def R():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_17545_gb300 import render as R
    return R


@pytest.mark.parametrize("width,height", [(24 * 16, 19 * 16), (24 * 16 + 1, 19 * 16)])   # 456 and 475 tiles
@pytest.mark.parametrize("front", [False, True])
def test_gradients_on_either_side(R, width, height, front):
    import torch
    scene = sg.random_scene(11, 3000, 0, n_objects=3, sphere_frac=1.0, centre_box=0.6, surfel_scale=(0.02, 0.05))
    cam = sg.look_at((0.0, 0.0, -3.0), (0.0, 0.0, 0.0), (0.0, 1.0, 0.0), width, height, 60.0)
    rng = np.random.default_rng(12)
    w = rng.uniform(0.3, 3.0, scene.n_surfels).astype(np.float32)
    w64 = w.astype(np.float64)
    g = rng.standard_normal((3, height, width)).astype(np.float32).astype(np.float64)
    g[:, oracle.render_translucent(scene, cam, w64, front)["amb"] != 0] = 0.0
    ref = oracle.backward_translucent(scene, cam, w64, g, front)
    gs = R.GESScene.from_arrays(scene)
    wt = torch.from_numpy(w).cuda()
    out = R.render_translucent(gs, cam, wt, front)
    got = R.render_translucent_backward(gs, cam, wt, out, torch.as_tensor(g, dtype=torch.float32, device="cuda"), front)
    gs.close()
    # the tolerance of the other translucent gradients: relative to each array's largest
    for k in ("s_pos", "s_rot", "s_scale", "s_w", "s_sh"):
        want = np.asarray(ref[k])
        err = np.abs(got[k].double().cpu().numpy().reshape(want.shape) - want).max()
        assert np.abs(want).max() > 0 and err <= GRAD_TOL * np.abs(want).max(), (k, err, np.abs(want).max())
