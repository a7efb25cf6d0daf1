"""Histograms whose counts meet in few bins, so that a block's 16-bit counters fill many times: hot
bins in the low half of a word, in the high half and in both, 256 and 300 bins, and one hot pair
beside even ones (whose blocks then help it). The fields are made of known bins, so the counts follow
from the number of in-shell cells. Whole counts: all comparisons are exact."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
R_IN, R_OUT = 0.547, 1.0


@pytest.fixture(scope="module")
def rp():
    import paper_2207_12011_gb300.raypc as rp
    rp.lib()
    return rp


def shell(n):
    d2 = (torch.arange(n, device="cuda") * 2 + 1 - n) ** 2
    s = d2.view(-1, 1, 1) + d2.view(1, -1, 1) + d2.view(1, 1, -1)
    return (s >= int(np.ceil((R_IN * n) ** 2))) & (s <= int(np.floor((R_OUT * n) ** 2)))


def middle(bin_, bins):
    """The middle of a bin of linspace(0, 1, bins + 1)."""
    return (bin_ + 0.5) / bins


def bins_of_kind(kind, n, bins):
    """Bin numbers of six variables, int64 [6, n, n, n] (expanded where constant)."""
    g = torch.Generator(device="cuda").manual_seed(n + bins)
    const = lambda b: torch.full((1, 1, 1), b, device="cuda", dtype=torch.int64).expand(n, n, n)  # noqa: E731
    rnd = lambda: torch.randint(0, bins, (n, n, n), generator=g, device="cuda")  # noqa: E731
    lo, hi = 10, bins - 6
    if kind == "halves":          # keys bin_a * pitch + bin_b: rows below the middle in the low halves of the words
        return [const(b) for b in (lo, lo, hi, hi, lo, lo)]
    if kind == "word":            # two hot counters of one word: half the rows of bins apart
        a = torch.where(torch.arange(n, device="cuda").view(1, 1, -1) % 2 == 0, lo, lo + bins // 2).expand(n, n, n)
        return [a, const(lo), a, const(hi), a, const(lo)]
    return [const(lo), const(hi), rnd(), rnd(), rnd(), rnd()]


@pytest.mark.parametrize("n,bins", [(256, 256), (256, 300), (386, 256)])
@pytest.mark.parametrize("kind", ["halves", "word", "one pair"])
def test_counters_that_fill(rp, n, bins, kind):
    inside = shell(n)
    cells = int(inside.sum())
    pairs = 5
    blocks = -(-torch.cuda.get_device_properties(0).multi_processor_count // pairs)
    assert cells // (2 if kind == "word" else 1) // blocks > 1 << 16      # a block's share of a hot bin wraps 16 bits
    which = bins_of_kind(kind, n, bins)
    vol = torch.stack([middle(w.float(), bins) for w in which]).half()
    edges = np.tile(np.linspace(0, 1, bins + 1, dtype=np.float32), (6, 1))
    for w, x in zip(which, vol):                                          # binary16 keeps the values in their bins
        assert torch.equal(torch.bucketize(x.float(), torch.from_numpy(edges[0, 1:-1]).cuda(), right=True), w.contiguous())
    want = torch.stack([torch.bincount((which[p] * bins + which[p + 1])[inside], minlength=bins * bins).view(bins, bins)
                        for p in range(pairs)]).int()
    with rp.Context(0) as ctx:
        v = ctx.load_volume(vol, store="f16", r_in=R_IN, r_out=R_OUT)
        v.build_bricks()
        got = v.pc_histogram(range(6), edges, use_brush=False)
        assert torch.equal(got, want)
    direct = rp.pc_histogram_noalloc(vol, range(6), edges, lo=[0.0] * 6, hi=[1.0] * 6, active_mask=0, use_brush=False,
                                     r_in=R_IN, r_out=R_OUT)
    assert torch.equal(direct, want)


def test_one_hot_bin_takes_no_longer_than_many(rp):
    """A constant field's cells all meet in one 16-bit counter per pair: its histogram has to take about
    as long as one whose cells spread (every thread at the counter's limit took 2.5 times as long)."""
    n, bins = 256, 256
    edges = np.tile(np.linspace(0, 1, bins + 1, dtype=np.float32), (6, 1))
    out = torch.empty((5, bins, bins), dtype=torch.int32, device="cuda")
    spread = torch.rand((6, n, n, n), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    with rp.Context(0) as ctx:
        def ms(vol):
            v = ctx.load_volume(vol, store="f32", r_in=R_IN, r_out=R_OUT)
            v.build_bricks()
            best = []
            for _ in range(8):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                v.pc_histogram(range(6), edges, use_brush=False, out=out)
                b.record()
                torch.cuda.synchronize()
                best.append(a.elapsed_time(b))
            v.free()
            return min(best)

        ms(spread)
        assert ms(torch.full_like(spread, 0.3)) < 1.75 * ms(spread)
