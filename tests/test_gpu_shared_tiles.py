"""Long tiles whose blocks all warps of a CTA share: 2D Gaussians and the
geometry maps, whose extra sums and planes the merge carries as well, at one
and four samples, against the float64 oracle."""
import numpy as np
import pytest

import oracle
from test_gpu_short_lists import H, R, W, _cam, _scene  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(260, 0), (0, 260), (300, 700), (1500, 300)])     # more than 256 entries over the middle tile
@pytest.mark.parametrize("dim", [3, 2])
@pytest.mark.parametrize("samples", [1, 4])
def test_geometry_maps_of_shared_tiles(R, n, m, dim, samples):  # noqa: F811
    import torch
    scene, cam, opts = _scene(n, m, dim), _cam(), dict(samples=samples)
    gs = R.GESScene.from_arrays(scene, device="cuda")
    out, geo = R.render(gs, cam, opts), R.render_geom(gs, cam, opts)
    gs.close()
    assert torch.equal(geo["rgb"], out["rgb"]) and torch.equal(geo["depth"], out["depth"])
    ref, gref = oracle.render(scene, cam, opts), oracle.render_geom(scene, cam, opts)
    assert ((out["id"].cpu().numpy() != ref["id"]).reshape(-1, H, W)[:, (ref["amb"] & 1) == 0]).sum() == 0
    ok = ref["amb"] == 0
    assert ok.mean() > 0.5
    assert np.abs(out["rgb"].cpu().numpy() - ref["rgb"])[:, ok].max() <= 2e-4
    # sums of up to 700 terms alpha x with x to 3.4, each as the colour's: its bound per unit of the largest
    for k in ("dg", "ng"):
        g, r = geo[k].cpu().numpy().reshape(-1, H, W), np.asarray(gref[k]).reshape(-1, H, W)
        assert np.abs(g - r)[:, ok].max() <= 2e-4 * (1.0 + np.abs(r).max())
