"""Histograms where the listing and counting kernels can go wrong: bins shared by more cells than a
16-bit counter holds, counters of 32 and 16 bits and tables that fit neither, 2 to 8 axes, edges of
even and odd lengths, bins that the affine guess misses (repeated, infinite and uneven edges, edges at
and between binary16 values), NaN and infinite values, position axes and brushes, chunks and slabs
that run full, and calls that have no room for a list. Whole counts: all comparisons are exact."""
import numpy as np
import pytest
import torch

import oracle
from paper_2207_12011_gb300 import synth
from test_gpu_parity import POS, load, stored

pytestmark = pytest.mark.gpu
R_IN, R_OUT = 0.547, 1.0


@pytest.fixture(scope="module")
def rp():
    import paper_2207_12011_gb300.raypc as rp
    rp.lib()
    return rp


@pytest.fixture(scope="module")
def ctx(rp):
    return rp.Context(0)


def field(n, kind):
    vol = synth.make_shell_volume(n, seed=n)
    if kind == "constant":                                   # every cell in one bin of each pair but one
        for v in range(5):
            vol[v] = 0.25 * v
    elif kind == "nonfinite":
        vol[1, ::7, ::5, ::3] = float("nan")
        vol[2, ::5, ::3, ::7] = float("inf")
        vol[3, ::3, ::7, ::5] = -float("inf")
    return vol


def edges_of(kind, st, order, bins):
    e = synth.make_edges(torch.from_numpy(np.nan_to_num(st, nan=0.0, posinf=1.0, neginf=0.0)), order, bins).astype(np.float32)
    if kind == "uneven":                                      # the guess is many bins off, some bins are empty
        e = np.sort(e[:, :1] + (e[:, -1:] - e[:, :1]) * np.linspace(0, 1, bins + 1) ** 3, axis=1).astype(np.float32)
        e[:, bins // 2] = e[:, bins // 2 - 1]
        e[0, 0], e[-1, -1] = -np.inf, np.inf
    elif kind == "halves":                                    # at binary16 values and one float beside them
        h = e.astype(np.float16).astype(np.float32)
        h[:, 1::3] = np.nextafter(h[:, 1::3], np.float32(np.inf))
        h[:, 2::3] = np.nextafter(h[:, 2::3], np.float32(-np.inf))
        e = np.maximum.accumulate(h, axis=1)
    elif kind == "one":                                       # every edge the same
        e[:] = e[:, bins // 3:bins // 3 + 1]
    return np.ascontiguousarray(e)


def oracle_counts(st, brush, order, edges, use, pos=None):
    return oracle.histogram(st, R_IN, R_OUT, brush.lo, brush.hi, brush.active_mask, order, edges, use_brush=use,
                            pos=pos if use else None)[0]


@pytest.mark.parametrize("n,store,kind,ekind,bins,order", [
    (128, "f16", "smooth", "even", 256, (0, 1, 2, 3, 4, 5)),
    (128, "f32", "smooth", "halves", 224, (0, 1, 2, 3, 4, 5, 0, 2)),
    (130, "f16", "smooth", "halves", 225, (5, 3)),
    (132, "f32", "constant", "even", 256, (0, 1, 2, 3, 4, 5)),
    (134, "f16", "constant", "even", 300, (0, 1, 2, 3, 4, 5, 0)),
    (136, "f16", "constant", "one", 2, (0, 1, 5)),
    (128, "f16", "nonfinite", "even", 256, (0, 1, 2, 3)),
    (130, "f32", "nonfinite", "uneven", 100, (3, 2, 1, 0)),
    (136, "f16", "nonfinite", "halves", 257, (1, 2, 3, 4, 5)),
    (128, "f16", "smooth", "uneven", 320, (0, 1, 2)),
    (129, "f16", "smooth", "even", 64, (0, 4, 5)),
    (96, "f16", "smooth", "uneven", 37, (0, 1, 2, 3, 4, 5)),
    (62, "f32", "smooth", "even", 512, (0, 1)),
    (50, "f16", "nonfinite", "even", 16, (0, 1, 2, 3)),
])
def test_counts_match_oracle(ctx, rp, n, store, kind, ekind, bins, order):
    vol = field(n, kind)
    st = stored(vol, store)
    brush = synth.make_brush(synth.make_shell_volume(n, seed=n), "c2")
    edges = edges_of(ekind, st, order, bins)
    v = load(ctx, vol, store, brush=brush)
    cells = torch.from_numpy(st).cuda()
    cells = cells.half() if store == "f16" else cells
    for use in (False, True):
        want = oracle_counts(st, brush, order, edges, use)
        got = v.pc_histogram(order, edges, use_brush=use).cpu().numpy().astype(np.uint32)
        assert np.array_equal(got, want), use
        direct = rp.pc_histogram_noalloc(cells, order, edges, lo=brush.lo, hi=brush.hi, active_mask=brush.active_mask,
                                         use_brush=use)
        assert np.array_equal(direct.cpu().numpy().astype(np.uint32), want), use
    v.free()


@pytest.mark.parametrize("n,store", [(324, "f16"), (328, "f16"), (326, "f32"), (332, "f32")])
def test_brushed_lists(ctx, rp, n, store):
    """Brushed calls of listed size, rows (edge no multiple of a chunk) and sub-brick groups, alone
    and with a position brush and position axes, from the volume's classification and from the server's."""
    vol = field(n, "smooth")
    st = stored(vol, store)
    for bname, pos in (("c3", None), ("c1", POS)):
        brush = synth.make_brush(vol, bname)
        v = load(ctx, vol, store, brush=brush)
        order = (0, 1, 2, 3, 4, 5)
        edges = edges_of("even", st, order, 256)
        if pos is not None:
            v.set_position_brush(*pos)
            order = (0, rp.AXIS_POS(rp.POS_R), 3, rp.AXIS_POS(rp.POS_X))
            edges[1], edges[2], edges[3] = np.linspace(0.5, 1, 257), edges[3], np.linspace(-1, 1, 257)
            edges = edges[:4]
        for use in (True, False):
            got = v.pc_histogram(order, edges, use_brush=use).cpu().numpy().astype(np.uint32)
            assert np.array_equal(got, oracle_counts(st, brush, order, edges, use, pos)), (bname, use)
        with rp.Server(ctx) as srv:
            rid = srv.submit_histogram(v, order, edges, lo=brush.lo, hi=brush.hi, mask=brush.active_mask, pos=pos)
            res = srv.poll(rid, timeout_us=10_000_000)
            assert np.array_equal(res["hist"].cpu().numpy().astype(np.uint32), oracle_counts(st, brush, order, edges, True, pos))
            srv.release(rid)
        v.free()


@pytest.mark.parametrize("n,store,order,bins", [
    (448, "f16", (0, 1, 2, 3, 4, 5), 256),                    # eight rows per warp
    (400, "f16", (0, 1, 2, 3, 4, 5, 0, 1), 300),              # two slabs
    (402, "f32", (5, 4, 3, 2, 1, 0, 5, 4), 300),
])
def test_large_lists_match_direct_counts(ctx, rp, n, store, order, bins):
    src = synth.make_shell_volume(n, device="cuda")
    cells = src.half() if store == "f16" else src
    brush = synth.make_brush(cells.float(), "c3")
    edges = synth.make_edges(cells.float(), order, bins)
    v = ctx.load_volume(src, store=store, r_in=R_IN, r_out=R_OUT)
    v.build_bricks(n_lod=0)
    v.set_brush(brush.lo, brush.hi, brush.active_mask)
    for use in (True, False):
        got = v.pc_histogram(order, edges, use_brush=use)
        want = rp.pc_histogram_noalloc(cells, order, edges, lo=brush.lo, hi=brush.hi, active_mask=brush.active_mask,
                                       use_brush=use, r_in=R_IN, r_out=R_OUT)
        assert torch.equal(got, want) and int(got.sum()) > 0, use
    v.free()


def test_no_room_for_a_list(rp):
    """A budget that the volume fills, and a graph that records the call: the counts stay the same."""
    n, order = 128, (0, 1, 2, 3, 4, 5)
    vol = field(n, "smooth")
    st = stored(vol, "f16")
    brush = synth.make_brush(vol, "c2")
    edges = edges_of("even", st, order, 256)
    want = oracle_counts(st, brush, order, edges, False)
    wide = rp.Context(0)
    v = load(wide, vol, "f16", brush=brush)
    v.pc_histogram(order, edges, use_brush=False)
    out = torch.empty(want.shape, dtype=torch.int32, device="cuda")
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        v.pc_histogram(order, edges, use_brush=False, out=out, stream=torch.cuda.current_stream())
    for _ in range(2):
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy().astype(np.uint32), want)
    del g
    used = wide.memory_used()
    v.free()
    tight = rp.Context(0, hbm_budget_bytes=used + (1 << 20))
    v = load(tight, vol, "f16", brush=brush)
    assert np.array_equal(v.pc_histogram(order, edges, use_brush=False).cpu().numpy().astype(np.uint32), want)
    v.free()
