"""The set-up's staged SH rows against its direct loads.

Degree-3 rows that start on 16 bytes go through shared memory, others are read
by their own thread; both evaluate the colours with the same operations, so a
scene gives the same bits from a buffer one element off.  Counts around the
32 primitives of a warp and the 512 of a round, all storage types, both
Gaussian kinds, and an image with too many tiles for the staged kernel."""
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


def _off_by_one(t):
    """The same values in a buffer that starts one element after an aligned one."""
    import torch
    flat = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)[1:]
    flat.copy_(t.reshape(-1))
    return flat.view(t.shape)


@pytest.mark.parametrize("n,m", [(1, 1), (31, 33), (32, 0), (0, 64), (513, 511), (20_001, 9_999)])
@pytest.mark.parametrize("dtype", ["float32", "float16", "bfloat16"])
@pytest.mark.parametrize("dim", [3, 2])
def test_staged_and_direct_rows_give_the_same_bits(R, n, m, dtype, dim):
    import torch
    scene = sg.random_scene(n + m, n, m, n_objects=3, sphere_frac=1.0, centre_box=0.7)
    if dim == 2:
        scene.g_scale = scene.g_scale[:, :2].copy()
    gs = R.GESScene.from_arrays(scene, sh_dtype=getattr(torch, dtype))
    t = dict(gs.t, s_sh=_off_by_one(gs.t["s_sh"]), g_sh=_off_by_one(gs.t["g_sh"]))
    assert n + m < 2 or any(t[k].data_ptr() % 16 for k in ("s_sh", "g_sh") if t[k].numel())
    off = R.GESScene(3, **t)
    for w, h in ((97, 61), (2048, 1100)):
        cam = sg.look_at((0.0, 0.0, -3.0), (0.0, 0.0, 0.0), (0.0, 1.0, 0.0), w, h, 60.0)
        a, b = R.render(gs, cam), R.render(off, cam)
        for k in ("rgb", "depth", "id", "aux"):
            assert torch.equal(a[k], b[k]), (k, w, h)
        batch = R.render_batch([gs, off], [cam, cam], [0, 1])      # each scene one view: no colour pass
        assert torch.equal(batch[0][0], a["rgb"]) and torch.equal(batch[1][0], a["rgb"])
    gs.close()
    off.close()
