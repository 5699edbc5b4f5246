"""Batches of many small views: a warp finds its item's view 32 at a time, and
the views whose long tiles a CTA's warps share are found the same way.  View
counts around 32 and 32 x 32, one late view with long lists, against the
single-view renders bit for bit."""
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_17545_gb300 import render as R
    return R


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 34, 65, 1024, 1026, 1057])
def test_many_small_views(R, n):
    import torch
    small = R.GESScene.from_arrays(sg.random_scene(3, 300, 200, n_objects=2, sphere_frac=1.0, centre_box=0.5))
    large = R.GESScene.from_arrays(sg.random_scene(4, 150_000, 50_000, n_objects=2, sphere_frac=1.0, centre_box=0.5))
    # odd sizes of 1 to 12 tiles
    cams = [sg.look_at((0.02 * (v % 7), 0.0, -3.0), (0.0, 0.0, 0.0), (0.0, 1.0, 0.0), 13 + 5 * (v % 8), 9 + 7 * (v % 5), 50.0)
            for v in range(n)]
    late = (2 * n) // 3
    sov = [1 if v == late else 0 for v in range(n)]
    scenes = [small, large]
    for _ in range(2):      # the graph's first call and a replay
        outs = R.render_batch(scenes, cams, sov)
        torch.cuda.synchronize()
        for v in range(n):
            if v % 7 and v not in (late, n - 1):
                continue
            one = R.render(scenes[sov[v]], cams[v])
            assert torch.equal(outs[v][0], one["rgb"]) and torch.equal(outs[v][1], one["depth"]), v
    for s in scenes:
        s.close()
