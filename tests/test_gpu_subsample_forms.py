"""Line subsamples at the edges of the select and the compaction: fewer rows than segments, one row and
several rows per segment, more rows than the launch has warps, one cell, all but one and all cells,
and a thin and an empty shell. Cells, values and flags are exact."""
import numpy as np
import pytest
import torch

import oracle
from paper_2207_12011_gb300 import synth
from test_gpu_parity import stored

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,store,r_in,r_out,seed", [
    (2, "f32", 0.0, 1.0, 1), (17, "f16", 0.547, 1.0, 2), (90, "f32", 0.547, 1.0, 3), (91, "f16", 0.0, 1.0, 0xFFFFFFFF),
    (100, "f32", 0.97, 0.975, 4), (128, "f16", 0.547, 1.0, 5), (150, "f32", 0.3, 0.8, 6), (64, "f32", 0.9999, 0.99991, 7),
])
def test_subsample_matches_oracle(n, store, r_in, r_out, seed):
    import paper_2207_12011_gb300.raypc as rp
    ctx = rp.Context(0)
    vol = synth.make_shell_volume(max(n, 8), seed=n)[:, :n, :n, :n].contiguous()
    st = stored(vol, store)
    v = ctx.load_volume(vol.cuda(), store=store, r_in=r_in, r_out=r_out)
    v.build_bricks(n_lod=0)
    lo, hi = np.full(6, -np.inf, np.float32), np.full(6, np.inf, np.float32)
    lo[1], hi[4] = np.nanmedian(st[1]), np.nanmedian(st[4])
    v.set_brush(lo, hi, 0b010010)
    order = (0, 4, 1)
    N = oracle.pc_subsample(st, r_in, r_out, lo, hi, 0b010010, seed, n ** 3, [0])[0].size
    for k in sorted({1, 2, 33, N // 3, max(N - 1, 0), N, N + 7}):
        cells, vals, flags = v.pc_subsample(seed, k, order)
        oc, ov, of = oracle.pc_subsample(st, r_in, r_out, lo, hi, 0b010010, seed, k, order)
        assert np.array_equal(cells.cpu().numpy(), oc), k
        assert np.array_equal(vals.cpu().numpy().view(np.uint32), np.asarray(ov, np.float32).view(np.uint32)), k
        assert np.array_equal(flags.cpu().numpy(), of), k
    v.free()
