"""The translucent render's per-tile sort at its edges.

Lists of up to 256, 512 and 1024 entries are sorted in registers (1, 2 and 4
keys per thread), longer ones in shared memory and then in global memory.
Stacks of discs over one tile, of every length around those edges, blended in
depth order, against the oracle."""
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


@pytest.mark.parametrize("n", [1, 2, 31, 33, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 4096, 4097])
def test_lists_of_every_length_blend_in_order(R, n):
    import torch
    rng = np.random.default_rng(n)
    f32 = lambda a: np.ascontiguousarray(a, np.float32)  # noqa: E731
    z = 2.0 + rng.permutation(n) / 64.0        # far outside the order's rounding
    pos = np.stack([rng.uniform(-0.02, 0.02, n) * z, rng.uniform(-0.02, 0.02, n) * z, z], 1)
    scene = sg.Scene(0, f32(pos), f32(np.tile([1.0, 0, 0, 0], (n, 1))), f32(rng.uniform(0.5, 1.0, (n, 2)) * z[:, None]),
                     f32(rng.uniform(-1, 1, (n, 1, 3))), *(f32(np.zeros(s)) for s in ((0, 3), (0, 4), (0, 3), (0,), (0, 1, 3))))
    w = f32(rng.uniform(0.004, 0.03, n))       # nearly clear: about 550 discs of the longest lists are blended
    cam = sg.Camera(16, 16, 60.0, 60.0, 8.0, 8.0, np.concatenate([np.eye(3), np.zeros((3, 1))], 1), 0.01, (0.2, 0.4, 0.6))
    gs = R.GESScene.from_arrays(scene, device="cuda")
    out = R.render_translucent(gs, cam, torch.from_numpy(w).cuda(), front_first=False)
    ref = oracle.render_translucent(scene, cam, w, front_first=False)
    ok = (ref["amb"] & 2) == 0
    assert ok.mean() > 0.5
    # up to n blends of a pixel, each rounded: 2 u n on T and on the colour, 2e-4 the renders' own bound
    tol = 2e-4 + 2.0 * 6e-8 * n
    assert np.abs(out["rgb"].cpu().numpy() - ref["rgb"])[:, ok].max(initial=0.0) <= tol
    assert np.abs(out["T"].cpu().numpy() - ref["T"])[ok].max(initial=0.0) <= tol
    gs.close()
