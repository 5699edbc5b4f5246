"""Translucent gradients of faint surfels at small and large scales.

The backward sums moments over the disc in fixed point and applies the scales
afterwards, so the step of the sums must follow the scales.  Surfels behind a
transmittance of 1e-4 or 1e-2, a hundred pixels to a few hundred each, against
the float64 oracle."""
import numpy as np
import pytest

import oracle
import scenegen as sg

pytestmark = pytest.mark.gpu

W, H = 65, 49


@pytest.fixture(scope="module")
def R():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_17545_gb300 import render as R
    return R


def _scene(s, aspect, T, n=60):
    """n faint discs of scales around (aspect s, s) at 20 s, behind two wide ones that leave T."""
    rng = np.random.default_rng(1)
    f32 = lambda a: np.ascontiguousarray(a, np.float32)  # noqa: E731
    z = 20.0 * s
    pos = np.concatenate([[[0, 0, 0.5 * z], [0, 0, 0.6 * z]],
                          np.stack([rng.uniform(-.5, .5, n), rng.uniform(-.4, .4, n), rng.uniform(1.0, 1.3, n)], 1) * z])
    q = np.concatenate([np.tile([1.0, 0, 0, 0], (2, 1)), [1.0, 0, 0, 0] + 0.3 * rng.standard_normal((n, 4))])
    scale = np.concatenate([np.full((2, 2), 40.0 * z), s * rng.uniform(.7, 1.3, (n, 2)) * [aspect, 1.0]])
    scene = sg.Scene(0, f32(pos), f32(q / np.linalg.norm(q, axis=1, keepdims=True)), f32(scale),
                     f32(rng.uniform(-1, 1, (n + 2, 1, 3))), *(f32(np.zeros(x)) for x in ((0, 3), (0, 4), (0, 3), (0,), (0, 1, 3))))
    w = f32(np.concatenate([[1 - T ** 0.5] * 2, rng.uniform(0.006, 0.02, n)]))
    cam = sg.Camera(W, H, 60.0, 60.0, 0.5 * W, 0.5 * H, np.concatenate([np.eye(3), np.zeros((3, 1))], 1),
                    0.01 * min(1.0, z), (.1, .2, .3))
    return scene, cam, w


@pytest.mark.parametrize("s,aspect,T", [(1e-4, 1.0, 1.2e-4), (1e-5, 1.0, 1.2e-4), (1.0, 100.0, 1e-2), (100.0, 1.0, 1e-2)])
@pytest.mark.parametrize("unit", [1.0, 1e-30])
def test_faint_gradients_at_every_scale(R, s, aspect, T, unit):
    import torch
    scene, cam, w = _scene(s, aspect, T)
    w64 = w.astype(np.float64)
    g = np.random.default_rng(3).standard_normal((3, H, W)).astype(np.float32).astype(np.float64)
    g[:, oracle.render_translucent(scene, cam, w64, False)["amb"] != 0] = 0.0
    ref = oracle.backward_translucent(scene, cam, w64, g, False)
    gs = R.GESScene.from_arrays(scene)
    wt = torch.from_numpy(w).cuda()
    out = R.render_translucent(gs, cam, wt, False)
    # dL/dC in units of 1e-30: the gradients scale with it
    grads = R.render_translucent_backward(gs, cam, wt, out, torch.as_tensor(g, dtype=torch.float32, device="cuda") * unit, False)
    gs.close()
    for k in ("s_pos", "s_rot", "s_scale", "s_w", "s_sh"):
        got = grads[k].double().cpu().numpy().reshape(len(w), -1)[2:] / unit
        want = np.asarray(ref[k]).reshape(len(w), -1)[2:]
        # half a step of max |dL/dC| 2^-24 for each of the image's 9 x 13 blocks,
        # and float32 along the chain: the hit's cancellation (z = 20 s) times
        # a few units of 6e-8
        tol = 0.5 * 2.0 ** -24 * 117 * np.abs(g).max() + 1e-5 * np.abs(want).max()
        assert np.abs(want).max() > 0 and np.abs(got - want).max() <= tol, (k, np.abs(got - want).max(), tol)
