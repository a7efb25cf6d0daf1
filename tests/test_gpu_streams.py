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
