"""Renders in which nothing is restricted leave the search for active sub-bricks out: the same pixels,
counts and depths as with a brush that every value passes, in both forms of the march, for fixed and
jittered lattices, alone and in a batch, with and without skipping and visibility skipping."""
import numpy as np
import pytest
import torch

from paper_2207_12011_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,store,r_in,r_out", [(2, "f32", 0.2, 1.0), (5, "f16", 0.0, 0.9), (33, "f32", 0.547, 1.0), (64, "f16", 0.547, 1.0),
                                                (64, "f32", 0.3, 1.2), (96, "f32", 0.9, 1.0)])
def test_open_renders_match_a_brush_that_all_pass(n, store, r_in, r_out):
    import paper_2207_12011_gb300.raypc as rp
    vol = synth.make_shell_volume(n, seed=n, device="cuda")
    tf = synth.make_tf(vol, "T_anom")
    rgbs = np.array(tf.rgbs, dtype=np.float32).reshape(-1, 4)
    rgbs[:100, 3] = 0.0
    cams = [synth.orbit_camera(35, 20, 2.8), synth.orbit_camera(80, -10, 0.8)]       # outside, and inside the sphere
    lo, hi = np.full(6, -np.inf, np.float32), np.full(6, np.inf, np.float32)
    with rp.Context(0) as ctx:
        v = ctx.load_volume(vol, store=store, r_in=r_in, r_out=r_out)
        v.build_bricks()
        v.set_tf(rgbs, tf.color_var, tf.v_lo, tf.v_hi)

        def frames(mask):
            v.set_brush(lo, hi, mask)
            out = []
            for cam in cams:
                for step in (0.0, 3.3 / n):
                    for kw in ({}, {"skip": False}, {"skip": False, "ert": False}, {"tf_skip": True}, {"variant": 2}, {"variant": 3}):
                        out += v.render(cam, 61, 47, step=step, counts=True, **kw)
                    out += v.render(cam, 61, 47, step=step, counts=True, depth=True)
                    for p in range(3):
                        out += v.render_progressive(cam, 61, 47, 5, p, None, step=step, counts=True)
            with rp.Batch(ctx, 3) as batch:
                views = [dict(vol=v, cam=c, w=50 + 13 * i, h=40, lo=lo, hi=hi, mask=mask, counts=True, skip=s)
                         for i, (c, s) in enumerate(zip(cams + cams[:1], (True, False, None)))]
                for o in batch.render(views):
                    out += o
                torch.cuda.synchronize()
            return [t.clone() for t in out]

        got, want = frames(0), frames(1)
        assert any(int((t[..., 1] > 0).sum()) for t in got if t.dtype == torch.int32) or n < 8
        assert len(got) == len(want) and all(torch.equal(a, b) for a, b in zip(got, want))
