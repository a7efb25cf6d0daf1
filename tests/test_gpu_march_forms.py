"""The two forms of the ray march (narrow: packed search index and 32-bit offsets; wide: any
shell radius, eye distance and volume size) and the tiled empty-space distance, at the sizes
where they can go wrong: edges 4k + 1, grids of one sub-brick, several tiles per axis, shells
and eyes beyond the narrow form's bounds."""
import numpy as np
import pytest
import torch

import oracle
from paper_2207_12011_gb300 import synth
from test_gpu_parity import _chebyshev_distance_brute, bits, load, stored

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rp():
    import paper_2207_12011_gb300.raypc as rp
    rp.lib()
    return rp


@pytest.mark.parametrize("n,store", [(2, "f32"), (5, "f16"), (9, "f32"), (33, "f16"), (64, "f32"), (65, "f32")])
@pytest.mark.parametrize("r_out,dist", [(1.0, 2.9), (1.0, 0.8), (1.25, 3.1), (1.0, 9000.0)])
def test_march_forms_match_oracle(rp, n, store, r_out, dist):
    """Per-pixel counts equal the oracle's and images agree within the storage tolerance, single
    frames with and without skipping and batched, for eyes inside and outside the sphere. The
    oracle colours a sample at its FP64 position, which the FP32 one leaves by up to |eye| 2^-23:
    images of the far eye are compared between the forms only."""
    vol = synth.make_shell_volume(n, seed=5)
    tf = synth.make_tf(vol, "T_anom")
    brush = synth.make_brush(vol, "c1")
    # a far eye sees the sphere under a small angle; rounding of |eye| rules its samples
    cam = synth.orbit_camera(25, 15, dist, 45.0 if dist < 10 else 0.016)
    with rp.Context(0) as ctx:
        v = ctx.load_volume(vol.cuda(), store=store, r_in=0.4, r_out=r_out)
        v.build_bricks()
        v.set_brush(brush.lo, brush.hi, brush.active_mask)
        v.set_tf(tf.rgbs, tf.color_var, tf.v_lo, tf.v_hi)
        ref, rc = oracle.render(stored(vol, store), 0.4, r_out, cam.as_array(), 45, 31, 1.0 / n, brush.lo, brush.hi,
                                brush.active_mask, tf.rgbs, tf.color_var, tf.v_lo, tf.v_hi, ert=False)
        assert int(rc[..., 0].sum()) > 0
        imgs = []
        for skip in (True, False):
            img, cnt = v.render(cam, 45, 31, skip=skip, counts=True, ert=False)
            imgs.append(img)
            assert np.array_equal(cnt.cpu().numpy().astype(np.uint32), rc), skip
            assert dist > 10 or np.abs(img.cpu().numpy() - ref).max() <= (1e-3 if store == "f32" else 4e-3)
        assert torch.equal(*imgs)
        with rp.Batch(ctx, 3) as b:
            near = synth.orbit_camera(80, -30, 2.8)
            q = dict(vol=v, w=45, h=31, lo=brush.lo, hi=brush.hi, mask=brush.active_mask, counts=True, ert=False)
            for views in ([dict(q, cam=cam)], [dict(q, cam=near), dict(q, cam=cam), dict(q, cam=near)]):
                for view, (i2, c2) in zip(views, b.render(views)):
                    i1, c1 = v.render(view["cam"], 45, 31, counts=True, ert=False)
                    assert torch.equal(i1, i2) and torch.equal(c1, c2)


def test_skip_off_without_room_for_the_distance(rp):
    """A render without skipping needs no distance grid: under a budget with no room for it, it
    reads the activity bits and gives the same pixels; one with skipping is refused."""
    n = 64
    vol = synth.make_shell_volume(n, seed=6)
    tf = synth.make_tf(vol, "T_anom")
    brush = synth.make_brush(vol, "c2")
    cam = synth.orbit_camera(40, 10, 2.9)

    def frame(budget, skip):
        with rp.Context(0, hbm_budget_bytes=budget) as ctx:
            v = load(ctx, vol, "f32", brush=brush, tf=tf)
            used = ctx.memory_used()
            img, cnt = v.render(cam, 70, 50, skip=skip, counts=True)
            return used, img.clone(), cnt.clone()

    used, img, cnt = frame(0, True)
    _, img2, cnt2 = frame(used + 64, False)
    assert torch.equal(img, img2) and torch.equal(cnt, cnt2)
    with pytest.raises(rp.RaypcError):
        frame(used + 64, True)


@pytest.mark.parametrize("n", [2, 4, 5, 29, 33, 65, 130, 517])
def test_distance_tiles_match_brute_force(rp, n):
    """The distance of every sub-brick (one tile, ragged tiles, several tiles per axis; rows that
    start inside a word) equals 3x3x3 dilations of the activity bits."""
    g = torch.Generator(device="cuda").manual_seed(n)
    vol = torch.rand((1, n, n, n), generator=g, device="cuda")
    nsb = (n + 3) // 4
    with rp.Context(0) as ctx:
        v = ctx.load_volume(vol, store="f16", r_in=0.0, r_out=1.0)
        v.build_bricks()
        # few active sub-bricks: the largest of the sub-brick maxima
        _, mx, _ = v.sub_bricks(classify=False)
        top = torch.sort(mx.flatten(), descending=True).values
        lo = float(top[min(top.numel() - 1, max(0, top.numel() // 3000))])
        v.set_brush([lo], [2.0], 1)
        _, _, act = v.sub_bricks()
        active = bits(rp, act, nsb ** 3).reshape(nsb, nsb, nsb)
        assert np.array_equal(v.skip_distance().cpu().numpy(), _chebyshev_distance_brute(active))
