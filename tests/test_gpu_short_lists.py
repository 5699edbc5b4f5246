"""Tiles whose lists have an entry per lane or fewer take a path of their own
(raster_short), a block at a time in a view and several in a batch, and the
batch's tile order keeps them apart.  Lists of 0 to 34 entries of either kind
over one tile of an image of ragged edges, with exact depth ties, all kernels'
variants: the single view and the geometry maps against the float64 oracle,
the batches bit for bit against the single view."""
import numpy as np
import pytest

import oracle
import scenegen as sg

pytestmark = pytest.mark.gpu

W, H = 45, 39          # 3 x 3 tiles, the last ones cut inside a block


@pytest.fixture(scope="module")
def R():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_17545_gb300 import render as R
    return R


def _scene(n, m, dim):
    """n fronto-parallel discs over the middle tile, each depth used by several
    of them (exact ties: the lower index wins), and m Gaussians about them."""
    rng = np.random.default_rng(100 * n + m)
    f32 = lambda a: np.ascontiguousarray(a, np.float32)  # noqa: E731
    z = rng.choice(np.linspace(2.0, 3.0, max(1, n // 3)), n)
    s_pos = np.stack([rng.uniform(-.25, .25, n), rng.uniform(-.2, .2, n), z], 1)
    g_pos = np.stack([rng.uniform(-.3, .3, m), rng.uniform(-.25, .25, m), rng.uniform(1.6, 3.4, m)], 1)
    q = rng.standard_normal((m, 4))
    if dim == 2:
        q[:, 1:3] *= 0.2        # not edge-on
    return sg.Scene(1, f32(s_pos), f32(np.tile([1.0, 0, 0, 0], (n, 1))), f32(rng.uniform(0.02, 0.08, (n, 2))),
                    f32(rng.uniform(0, 1, (n, 4, 3))), f32(g_pos), f32(q / np.linalg.norm(q, axis=1, keepdims=True)),
                    f32(rng.uniform(0.01, 0.03, (m, dim))), f32(rng.uniform(0.1, 0.9, m)), f32(rng.uniform(0, 1, (m, 4, 3))))


def _cam(w=W, h=H):
    return sg.Camera(w, h, 50.0, 50.0, 0.5 * w, 0.5 * h, np.concatenate([np.eye(3), np.zeros((3, 1))], 1), 0.01, (.1, .2, .3))


@pytest.mark.parametrize("n,m", [(0, 0), (1, 0), (0, 1), (5, 7), (31, 32), (32, 31), (32, 32), (33, 4), (4, 33), (34, 34)])
@pytest.mark.parametrize("dim", [3, 2])
@pytest.mark.parametrize("samples", [1, 4])
def test_views_and_batches_of_short_lists(R, n, m, dim, samples):
    import torch
    scene, cam, opts = _scene(n, m, dim), _cam(), dict(samples=samples)
    gs = R.GESScene.from_arrays(scene, device="cuda")
    out = R.render(gs, cam, opts)
    ref = oracle.render(scene, cam, opts)
    ids, want = out["id"].cpu().numpy().reshape(-1, H, W), ref["id"].reshape(-1, H, W)
    # Only a sample on a disc's rim may differ: 34 discs with rims of at most 45
    # pixels and a band of 1e-5 pixels, 0.015 samples in all, so none does.
    assert (ids == want).all()
    ok = ref["amb"] == 0
    assert np.abs(out["rgb"].cpu().numpy() - ref["rgb"])[:, ok].max(initial=0.0) <= 2e-4
    geo = R.render_geom(gs, cam, opts)
    assert torch.equal(geo["rgb"], out["rgb"])
    gref = oracle.render_geom(scene, cam, opts)
    for k in ("dg", "ng"):
        g, r = geo[k].cpu().numpy().reshape(-1, H, W), np.asarray(gref[k]).reshape(-1, H, W)
        # sums of alpha times depths up to 3.4: the colour's bound per unit
        assert np.abs(g - r)[:, ok].max(initial=0.0) <= 2e-4 * (1.0 + np.abs(r).max())
    cams = [_cam(), _cam(W + 16, H - 7), _cam()]
    one = [R.render(gs, c, opts) for c in cams]
    for (rgb, depth), w in zip(R.render_batch([gs], cams, opts=opts), one):
        assert torch.equal(rgb, w["rgb"]) and torch.equal(depth, w["depth"])
    if samples == 1 and n in (5, 33):
        # whole tiles at a time: a batch of four tiles and more for each warp of the GPU
        many = [cams[k % 2] for k in range(2400)]
        for k, (rgb, depth) in enumerate(R.render_batch([gs], many, opts=opts)):
            if k % 97 < 2:
                assert torch.equal(rgb, one[k % 2]["rgb"]) and torch.equal(depth, one[k % 2]["depth"])
    gs.close()
