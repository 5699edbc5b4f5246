"""SH gradient rows, which a warp stores together, at every degree and around
the 32 rows of a warp and the 256 of a CTA.

A row is Y_k(direction) times the colour gradient, so its first entry gives the
whole row: float32 bases of unit directions are within 1e-5 of the float64
ones (values up to 3, gradients up to 10, a few units of 6e-8 each)."""
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


def _check_rows(rows, pos, eye, deg):
    rows = rows.cpu().numpy().astype(np.float64)
    d = eye - pos.astype(np.float64)
    Y = np.stack([oracle.sh_basis(deg, v / np.linalg.norm(v))[0] for v in d]).reshape(len(d), -1)
    g = rows[:, 0, :] / Y[:, :1]
    err = np.abs(rows - Y[:, :, None] * g[:, None, :])
    assert (err <= 1e-5 * np.abs(g).max(1)[:, None, None]).all()
    return np.abs(g).max(1) > 0


@pytest.mark.parametrize("deg", [0, 1, 2, 3])
@pytest.mark.parametrize("n,m,dim", [(1, 1, 3), (31, 33, 3), (33, 31, 2), (256, 257, 3), (257, 255, 2)])
def test_rows_are_bases_times_one_gradient(R, deg, n, m, dim):
    import torch
    scene = sg.random_scene(deg + n, n, m, n_objects=2, sphere_frac=1.0, centre_box=0.5, sh_degree=deg,
                            surfel_scale=(0.05, 0.1), gauss_logscale=(-3.0, 0.5))
    if dim == 2:
        scene.g_scale = scene.g_scale[:, :2].copy()
    eye = np.array([0.0, 0.0, -3.0])
    cam = sg.look_at(tuple(eye), (0.0, 0.0, 0.0), (0.0, 1.0, 0.0), 97, 61, 60.0)
    gs = R.GESScene.from_arrays(scene)
    dl = torch.as_tensor(np.random.default_rng(n).standard_normal((3, 61, 97)), dtype=torch.float32, device="cuda")
    fwd = R.render(gs, cam, with_aux=True)
    gr = R.render_backward(gs, cam, fwd, dl)
    hit = _check_rows(gr["s_sh"], scene.s_pos, eye, deg)
    won = np.isin(np.arange(n), fwd["id"].cpu().numpy())
    assert not hit[~won].any() and (n < 31 or hit.any())
    hit = _check_rows(gr["g_sh"], scene.g_pos, eye, deg)
    assert m < 31 or hit.any()
    w = torch.full((n,), 0.5, device="cuda")
    t = R.render_translucent(gs, cam, w)
    hit = _check_rows(R.render_translucent_backward(gs, cam, w, t, dl)["s_sh"], scene.s_pos, eye, deg)
    assert n < 31 or hit.any()
    gs.close()
