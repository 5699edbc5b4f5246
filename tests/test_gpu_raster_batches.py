"""The raster's batches of 32 surfel records and its cull words at their edges.

A warp tests its 8x4 block's surfels a record per lane, 32 at a time (few left
over: one at a time), and a tile-list entry carries a rounded cull key beside
the block mask.  Stacks of discs of every batch remainder over one block, with
exact depth ties (the lower index must win, inside a batch and across two),
and depth-test keys at the ends of the float range, against the oracle."""
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


def _stack(n, m, seed):
    """n fronto-parallel discs around the axis, each depth used by several of
    them (exact ties), and m small Gaussians in front of and behind them."""
    rng = np.random.default_rng(seed)
    f32 = lambda a: np.ascontiguousarray(a, np.float32)  # noqa: E731
    z = rng.choice(np.linspace(2.0, 3.0, max(1, n // 3)), n)
    s_pos = np.stack([rng.uniform(-0.05, 0.05, n), rng.uniform(-0.05, 0.05, n), z], 1)
    rot = np.tile([1.0, 0.0, 0.0, 0.0], (n, 1))
    g_pos = np.stack([rng.uniform(-0.2, 0.2, m), rng.uniform(-0.2, 0.2, m), rng.uniform(1.5, 3.5, m)], 1)
    q = rng.standard_normal((m, 4))
    return sg.Scene(1, f32(s_pos), f32(rot), f32(rng.uniform(0.02, 0.08, (n, 2))), f32(rng.uniform(0, 1, (n, 4, 3))),
                    f32(g_pos), f32(q / np.linalg.norm(q, axis=1, keepdims=True)),
                    f32(rng.uniform(0.01, 0.03, (m, 3))), f32(rng.uniform(0.1, 0.9, m)), f32(rng.uniform(0, 1, (m, 4, 3))))


def _camera(width, height):
    return sg.Camera(width, height, 40.0, 40.0, 0.5 * width, 0.5 * height,
                     np.concatenate([np.eye(3), np.zeros((3, 1))], 1), 0.01, (0.1, 0.2, 0.3))


@pytest.mark.parametrize("samples", [1, 4])
@pytest.mark.parametrize("n", [1, 8, 9, 12, 13, 31, 32, 33, 63, 64, 65, 97, 400])
def test_batch_remainders_and_ties(R, n, samples):
    scene, cam = _stack(n, 5, n), _camera(19, 13)
    gs = R.GESScene.from_arrays(scene, device="cuda")
    out = R.render(gs, cam, dict(samples=samples))
    ref = oracle.render(scene, cam, dict(samples=samples))
    ids, want = out["id"].cpu().numpy().reshape(samples, 13, 19), ref["id"].reshape(samples, 13, 19)
    # The planes are parallel to the image, so discs of one depth tie exactly on
    # both sides (1/z has no gradient) and the lower index wins.  Ids could only
    # differ at a disc's rim: 400 discs of at most 4 pixels with a band of 1e-5
    # of their area, 0.02 pixels in all.
    assert (ids == want).all()
    assert n < 9 or len(set(scene.s_pos[:, 2])) < n
    ok = (ids == want).all(0) & (ref["amb"] == 0)
    assert np.abs(out["rgb"].cpu().numpy() - ref["rgb"])[:, ok].max(initial=0.0) <= 2e-4
    gs.close()


@pytest.mark.parametrize("eps", [3e38, -3e38, 0.0, 1e-30, -0.7])
def test_depth_keys_at_the_ends_of_the_float_range(R, eps):
    scene, cam = _stack(40, 300, 7), _camera(33, 21)
    opts = dict(eps_mode=2, eps_value=eps)
    gs = R.GESScene.from_arrays(scene, device="cuda")
    out = R.render(gs, cam, opts)
    ref = oracle.render(scene, cam, opts)
    ok = (out["id"].cpu().numpy() == ref["id"]) & (ref["amb"] == 0)
    assert ok.mean() > 0.5
    assert np.abs(out["rgb"].cpu().numpy() - ref["rgb"])[:, ok].max() <= 2e-4
    # W_G sums alphas in (1/255, 1): the colour's bound carries over
    assert np.abs(out["aux"].cpu().numpy() - ref["wg"])[ok].max() <= 2e-4 * (1.0 + ref["wg"].max())
    gs.close()
