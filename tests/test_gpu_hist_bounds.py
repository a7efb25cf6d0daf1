"""Listed histograms at the bounds of their counters: the most bins of 32-bit counters and of 16-bit
ones, and one more of each, with bins in the first and the last row and column of the table."""
import numpy as np
import pytest
import torch

import oracle
from paper_2207_12011_gb300 import synth
from test_gpu_parity import load, stored

pytestmark = pytest.mark.gpu
R_IN, R_OUT = 0.547, 1.0


@pytest.mark.parametrize("bins", [217, 218, 309, 310])
@pytest.mark.parametrize("store", ["f32", "f16"])
def test_bins_at_the_bounds(bins, store):
    import paper_2207_12011_gb300.raypc as rp
    n, order = 128, (0, 1, 2, 3)
    vol = synth.make_shell_volume(n, seed=2)
    st = stored(vol, store)
    edges = np.stack([np.linspace(np.quantile(st[a], 0.02), np.quantile(st[a], 0.98), bins + 1) for a in order]).astype(np.float32)
    with rp.Context(0) as ctx:
        v = load(ctx, vol, store)
        got = v.pc_histogram(order, edges, use_brush=False).cpu().numpy().astype(np.uint32)
    lo, hi = np.full(6, -np.inf, np.float32), np.full(6, np.inf, np.float32)
    want = oracle.histogram(st, R_IN, R_OUT, lo, hi, 0, order, edges, use_brush=False)[0]
    assert np.array_equal(got, want) and got[0, 0].any() and got[0, -1].any() and got[:, :, -1].any()
