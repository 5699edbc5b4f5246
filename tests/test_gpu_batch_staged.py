"""render_batch where the set-up stages SH rows in shared memory.

A batch whose scenes have one view each and degree-3 rows that start on 16
bytes takes the staged set-up; the call's kept graph holds that choice, so rows
that start elsewhere (by an update, or in another scene of the same counts)
need a graph of their own.  Every call gives the bits of the single-view render
of unaligned rows, which are read directly."""
import pytest

import scenegen as sg
from test_gpu_staged_setup import R, _off_by_one  # noqa: F401

pytestmark = pytest.mark.gpu

SIZES = ((97, 61), (161, 117))


def _cam(w, h):
    return sg.look_at((0.0, 0.0, -3.0), (0.0, 0.0, 0.0), (0.0, 1.0, 0.0), w, h, 60.0)


def _scene(R, seed, n, m, dim, dtype):  # noqa: F811
    import torch
    scene = sg.random_scene(seed, n, m, n_objects=3, sphere_frac=1.0, centre_box=0.7)
    if dim == 2:
        scene.g_scale = scene.g_scale[:, :2].copy()
    return R.GESScene.from_arrays(scene, sh_dtype=getattr(torch, dtype))


def _unaligned(R, gs):  # noqa: F811
    t = dict(gs.t, s_sh=_off_by_one(gs.t["s_sh"]), g_sh=_off_by_one(gs.t["g_sh"]))
    assert t["s_sh"].data_ptr() % 16 and t["g_sh"].data_ptr() % 16
    return R.GESScene(3, **t)


@pytest.mark.parametrize("dtypes", [("float32", "float32"), ("float16", "float16"), ("bfloat16", "bfloat16"),
                                    ("float32", "float16")])
@pytest.mark.parametrize("dim", [3, 2])
def test_the_kept_graph_follows_the_rows_alignment(R, dim, dtypes):  # noqa: F811
    import torch
    scenes = [_scene(R, 5 + k, 1500 + 700 * k, 2100 - 900 * k, dim, d) for k, d in enumerate(dtypes)]
    off = [_unaligned(R, s) for s in scenes]
    cams = [_cam(w, h) for w, h in SIZES]
    want = [R.render(s, c) for s, c in zip(off, cams)]

    def check(ss):
        for _ in range(2):      # a graph's first call and a replay
            for (rgb, depth), r in zip(R.render_batch(ss, cams, [0, 1]), want):
                assert torch.equal(rgb, r["rgb"]) and torch.equal(depth, r["depth"])

    check(scenes)                                   # staged
    aligned = dict(s_sh=scenes[1].t["s_sh"], g_sh=scenes[1].t["g_sh"])
    scenes[1].update(s_sh=off[1].t["s_sh"], g_sh=off[1].t["g_sh"])
    check(scenes)                                   # by update
    scenes[1].update(**aligned)
    check(scenes)                                   # and back
    check([scenes[0], off[1]])                      # another scene of the same counts
    scenes[1].update(s_sh=off[1].t["s_sh"])
    check(scenes)                                   # one array alone
    for s in scenes + off:
        s.close()
