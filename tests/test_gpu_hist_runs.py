"""Histograms that count straight into L2, with few bins: neighbouring cells share bin pairs and many
cells meet in one counter. By runs of pairs (no copies, or no restriction) and of whole tuples
(copies and a brush), even edges that are no multiple of a chunk among them. Exact counts."""
import numpy as np
import pytest
import torch

import oracle
from paper_2207_12011_gb300 import synth
from test_gpu_parity import load, stored

pytestmark = pytest.mark.gpu
R_IN, R_OUT = 0.547, 1.0


@pytest.fixture(scope="module")
def rp():
    import paper_2207_12011_gb300.raypc as rp
    rp.lib()
    return rp


@pytest.mark.parametrize("n,store,order", [(62, "f32", (0, 1, 2, 3, 4, 5)), (64, "f16", (3, 1)), (126, "f16", (0, 1, 2, 3, 4, 5, 0, 2)),
                                           (128, "f32", (0, 1, 2)), (130, "f16", (5, 4, 3, 2, 1, 0))])
def test_few_bins(rp, n, store, order):
    vol = synth.make_shell_volume(n, seed=n)
    st = stored(vol, store)
    brush = synth.make_brush(vol, "c3")
    cells = torch.from_numpy(st).cuda()
    cells = cells.half() if store == "f16" else cells
    with rp.Context(0) as ctx:
        for mask in (0, brush.active_mask):
            v = load(ctx, vol, store)
            v.set_brush(brush.lo, brush.hi, mask)
            for bins in (2, 5, 16):
                edges = np.ascontiguousarray(synth.make_edges(torch.from_numpy(st), order, bins).astype(np.float32))
                want = oracle.histogram(st, R_IN, R_OUT, brush.lo, brush.hi, mask, order, edges, use_brush=True)[0]
                got = v.pc_histogram(order, edges, use_brush=True).cpu().numpy().astype(np.uint32)
                assert np.array_equal(got, want), (mask, bins)
                got = rp.pc_histogram_noalloc(cells, order, edges, lo=brush.lo, hi=brush.hi, active_mask=mask, use_brush=True)
                assert np.array_equal(got.cpu().numpy().astype(np.uint32), want), (mask, bins)
            v.free()


def test_even_edges_take_no_longer_than_odd_ones(rp):
    """An even edge that is no multiple of a chunk goes the chunked way, an odd one cell by cell: with few
    bins and no scratch the chunked way took over three times as long as the other."""
    def ms(n):
        cells = synth.make_shell_volume(n, device="cuda").half()
        edges = synth.make_edges(cells.float(), range(6), 4)
        best = []
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            rp.pc_histogram_noalloc(cells, range(6), edges, lo=[0.0] * 6, hi=[1.0] * 6, active_mask=0, use_brush=False)
            b.record()
            torch.cuda.synchronize()
            best.append(a.elapsed_time(b))
        return min(best)

    ms(250)
    assert ms(250) < 1.5 * ms(251)


def test_more_slots_than_the_chunked_kernel_has(rp):
    """A large brushed call with more axes and brushed variables than fit the chunked kernel's load slots
    takes no list: its counts spread over copies, which a second kernel sums."""
    n, bins = 324, 64
    vol = synth.make_shell_volume(n, device="cuda").half()
    order = (0, rp.AXIS_POS(rp.POS_R), 2, rp.AXIS_POS(rp.POS_X), rp.AXIS_POS(rp.POS_Y), rp.AXIS_POS(rp.POS_Z))
    edges = np.array(synth.make_edges(vol.float(), (0, 0, 2, 0, 0, 0), bins), dtype=np.float32)
    edges[1] = np.linspace(0.5, 1, bins + 1)
    edges[3:] = np.linspace(-1, 1, bins + 1)
    brush = synth.make_brush(vol.float(), "c3")
    mask = brush.active_mask | 0b111010                      # four brushed variables beside the two axes
    with rp.Context(0) as ctx:
        v = ctx.load_volume(vol, store="f16", r_in=R_IN, r_out=R_OUT)
        v.build_bricks()
        v.set_brush(brush.lo, brush.hi, mask)
        v.pc_histogram(order, edges)
        before = rp.kernel_launches()
        got = v.pc_histogram(order, edges).cpu().numpy().astype(np.uint32)
        assert rp.kernel_launches() - before == 2
        st = vol.float().cpu().numpy()
        want = oracle.histogram(st, R_IN, R_OUT, brush.lo, brush.hi, mask, order, edges, use_brush=True)[0]
        assert np.array_equal(got, want)
