"""What a context keeps between calls under streams and graphs: a call that reads it must not depend
on work that another stream has yet to do, or that was recorded and not run."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2207_12011_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rp():
    import paper_2207_12011_gb300.raypc as rp
    rp.lib()
    return rp


def skip_list(rp, ctx, v, stream, out):
    """The raw call, into buffers that exist."""
    rp._call("raypc_get_skip_list", ctx.handle, v.id, 0, *(ctypes.c_void_p(t.data_ptr()) for t in out), rp._stream(stream))


def test_skip_list_after_a_recorded_one(rp):
    n = 64
    vol = synth.make_shell_volume(n, device="cuda")
    a, b = synth.make_brush(vol, "c1"), synth.make_brush(vol, "c2")
    nb = (n + 7) // 8
    with rp.Context(0) as ctx:
        v = ctx.load_volume(vol)
        v.build_bricks()
        word = lambda k: torch.empty(k, dtype=torch.int32, device="cuda")  # noqa: E731
        out = [word((nb ** 3 + 31) // 32), word((nb ** 3 + 31) // 32), word(nb ** 3), word(1)]
        cur = torch.cuda.current_stream()
        lists = {}
        for name, br in (("a", a), ("b", b)):
            v.set_brush(br.lo, br.hi, br.active_mask)
            skip_list(rp, ctx, v, cur, out)
            torch.cuda.synchronize()
            lists[name] = [t.clone() for t in out]
        assert not torch.equal(lists["a"][0], lists["b"][0])
        v.set_brush(a.lo, a.hi, a.active_mask)
        torch.cuda.synchronize()
        side, g, rec = torch.cuda.Stream(), torch.cuda.CUDAGraph(), [torch.zeros_like(t) for t in out]
        with torch.cuda.graph(g, stream=side):
            skip_list(rp, ctx, v, torch.cuda.current_stream(), rec)
        skip_list(rp, ctx, v, cur, out)                      # the recorded one has not run
        torch.cuda.synchronize()
        k = int(out[3])
        for got, want in zip(out, lists["a"]):
            assert torch.equal(got[:k] if got is out[2] else got, want[:k] if got is out[2] else want)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(rec[0], lists["a"][0]) and torch.equal(rec[3], lists["a"][3])
        del g


@pytest.mark.parametrize("store", ["f32", "f16"])
def test_recorded_render_without_skipping(rp, store):
    """A render without skipping depends on the activity and the classes alone, which update, levels and
    brush edit leave current: recorded once, it shows the values of each later time step, and a render
    with the transfer function's visibility in between leaves it alone."""
    n, w, h = 96, 80, 60
    steps = [synth.make_shell_volume(n, seed=s, device="cuda") for s in (1, 2)]
    steps[1] = steps[1].flip(3).contiguous()
    tf = synth.make_tf(steps[0], "T_anom")
    rgbs = np.array(tf.rgbs, dtype=np.float32).reshape(-1, 4)
    rgbs[:128, 3] = 0.0                                      # half of the range is invisible
    brush = synth.make_brush(steps[0], "c2")
    cam = synth.orbit_camera(**synth.DEFAULT_CAMERA)
    with rp.Context(0) as ctx:
        v = ctx.load_volume(steps[0], store=store)

        def step(i):
            v.update(steps[i])
            v.build_bricks()
            v.set_brush(brush.lo, brush.hi, brush.active_mask)

        def render(**kw):
            img, cnt = v.render(cam, w, h, counts=True, **kw)
            torch.cuda.synchronize()
            return img.clone(), cnt.clone()

        step(0)
        v.set_tf(rgbs, tf.color_var, tf.v_lo, tf.v_hi)
        first = render(skip=False)
        render(skip=True)                                    # the grid is current when the graph is recorded
        img, cnt = torch.empty((h, w, 4), device="cuda"), torch.empty((h, w, 2), dtype=torch.int32, device="cuda")
        side, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=side):
            v.render(cam, w, h, skip=False, out=img, counts=cnt, stream=torch.cuda.current_stream())

        def replayed():
            img.zero_(), cnt.zero_()
            g.replay()
            torch.cuda.synchronize()
            return img, cnt

        same = lambda a, b: all(torch.equal(x, y) for x, y in zip(a, b))  # noqa: E731
        assert same(replayed(), first)
        for skip in (True, False):
            render(tf_skip=True, skip=skip)
            assert same(replayed(), first)
        step(1)
        got = [t.clone() for t in replayed()]
        second = render(skip=False)
        assert same(got, second) and not same(second, first)
        g2 = torch.cuda.CUDAGraph()
        step(0)
        torch.cuda.synchronize()
        with torch.cuda.graph(g2, stream=side):              # recorded and not run: it leaves nothing behind
            v.render(cam, w, h, skip=False, out=img, counts=cnt, stream=torch.cuda.current_stream())
        assert same(render(skip=True), first)
        step(1)
        assert same(render(skip=True), second)
        del g, g2


def test_visibility_skipping_under_a_tight_budget(rp):
    """Renders with skipping, with and without the transfer function's visibility, in turn, where the
    budget has room for one distance grid."""
    n, w, h = 64, 70, 50
    vol = synth.make_shell_volume(n, seed=6, device="cuda")
    tf, brush = synth.make_tf(vol, "T_anom"), synth.make_brush(vol, "c2")
    rgbs = np.array(tf.rgbs, dtype=np.float32).reshape(-1, 4)
    rgbs[:128, 3] = 0.0
    cam = synth.orbit_camera(40, 10, 2.9)

    def frames(budget):
        with rp.Context(0, hbm_budget_bytes=budget) as ctx:
            v = ctx.load_volume(vol)
            v.build_bricks()
            v.set_brush(brush.lo, brush.hi, brush.active_mask)
            v.set_tf(rgbs, tf.color_var, tf.v_lo, tf.v_hi)
            used = [ctx.memory_used()]
            out = []
            for tf_skip in (False, True, False, True):
                out.append(v.render(cam, w, h, tf_skip=tf_skip)[0].clone())
                used.append(ctx.memory_used())
            return used, out

    used, want = frames(0)
    assert used[2] > used[1] > used[0]
    used, got = frames(used[1])
    assert used[-1] == used[1] and all(torch.equal(a, b) for a, b in zip(got, want))
