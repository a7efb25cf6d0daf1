"""Scratch that a context keeps between calls: counted as memory used, within the budget, and given
back to whatever the context allocates next."""
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


def test_scratch_counts_and_makes_way(rp):
    n, order = 160, (0, 1, 2, 3, 4, 5)
    vol = synth.make_shell_volume(n, device="cuda").half()
    edges = np.array(synth.make_edges(vol.float(), order, 256), dtype=np.float32)

    def load(ctx):
        v = ctx.load_volume(vol, store="f16")
        v.build_bricks()
        return v

    def counts(v):
        out = v.pc_histogram(order, edges, use_brush=False)
        torch.cuda.synchronize()
        return out

    cells = int(rp.pc_histogram_noalloc(vol, order, edges, lo=[0.0] * 6, hi=[1.0] * 6, active_mask=0,
                                        use_brush=False)[0].long().sum())
    with rp.Context(0) as ctx:
        v = load(ctx)
        one = ctx.memory_used()
        want = counts(v)
        held = ctx.memory_used() - one
        assert held >= 6 * cells                             # a byte per listed cell and axis
        before = rp.kernel_launches()
        counts(v)
        listed = rp.kernel_launches() - before
        assert ctx.memory_used() - one == held               # used again, not grown
    # room for two volumes: the list fits beside one, and makes way for the second
    with rp.Context(0, hbm_budget_bytes=2 * one + (1 << 20)) as ctx:
        v = load(ctx)
        assert torch.equal(counts(v), want)
        assert one + 6 * cells <= ctx.memory_used() <= 2 * one + (1 << 20)
        w = load(ctx)
        assert 2 * one <= ctx.memory_used() <= 2 * one + (1 << 20)
        assert torch.equal(counts(w), want) and torch.equal(counts(v), want)      # without room for a list
        assert ctx.memory_used() <= 2 * one + (64 << 20)     # the copies that a call cannot do without
        w.free()
        before = rp.kernel_launches()
        assert torch.equal(counts(v), want) and rp.kernel_launches() - before == listed
    with pytest.raises(rp.RaypcError):
        with rp.Context(0, hbm_budget_bytes=one // 2) as ctx:
            load(ctx)


def test_streams_within_one_budget(rp):
    """Listed calls on several streams at once, each of which would fit the budget alone."""
    n, order = 160, (0, 1, 2, 3, 4, 5)
    vol = synth.make_shell_volume(n, device="cuda").half()
    edges = np.array(synth.make_edges(vol.float(), order, 256), dtype=np.float32)
    with rp.Context(0) as ctx:
        v = ctx.load_volume(vol, store="f16")
        one = ctx.memory_used()
        want = v.pc_histogram(order, edges, use_brush=False)
        torch.cuda.synchronize()
        held = ctx.memory_used() - one
    budget = one + held + held // 2
    with rp.Context(0, hbm_budget_bytes=budget) as ctx:
        v = ctx.load_volume(vol, store="f16")
        torch.cuda.synchronize()
        streams = [torch.cuda.Stream() for _ in range(4)]
        outs = [torch.empty_like(want) for _ in streams]
        for _ in range(5):
            for s, o in zip(streams, outs):
                v.pc_histogram(order, edges, use_brush=False, out=o, stream=s)
            torch.cuda.synchronize()
            assert all(torch.equal(o, want) for o in outs)
            assert ctx.memory_used() <= budget + (64 << 20)
