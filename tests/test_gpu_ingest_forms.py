"""Ingest, level and brick passes at the edges of their forms: rows of one run, ragged and odd rows,
several column chunks, sources that are not 16-byte aligned, half quadrants at the grid's end, and
updates whose passes write one or two coarser levels on the way."""
import numpy as np
import pytest
import torch

import oracle
from paper_2207_12011_gb300 import synth
from test_gpu_parity import oracle_levels, stored

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rp():
    import paper_2207_12011_gb300.raypc as rp
    rp.lib()
    return rp


def source(n, dtype, seed, aligned=True):
    """Two random fields as a device tensor, optionally one element off a 16-byte boundary."""
    g = torch.Generator(device="cuda").manual_seed(1000 * seed + n)
    flat = torch.randn(2 * n ** 3 + 1, generator=g, device="cuda").to(dtype)
    flat = flat[:-1] if aligned else flat[1:]
    t = flat.view(2, n, n, n)
    assert (t.data_ptr() % 16 == 0) == aligned and t.is_contiguous()
    return t


TF = np.tile(np.array([0.5, 0.6, 0.7, 3.0], np.float32), (256, 1))


def check(v, src, store, n_lod):
    """Levels, their ranges, and through a brushed frame of each the x-pairs the render reads."""
    levels = oracle_levels(stored(src.float().cpu(), store), n_lod, store)
    for lod, want in enumerate(levels):
        assert np.array_equal(v.export(lod).float().cpu().numpy(), want), lod
        for edge, got in ((8, v.bricks(lod)), (4, v.sub_bricks(lod, classify=False)[:2])):
            for a, b in zip(got, oracle.brick_minmax(want, edge)):
                assert np.array_equal(a.cpu().numpy(), b.reshape(a.shape)), (lod, edge)
    lo, hi = np.float32([-0.2, -0.3]), np.float32([0.5, 0.4])
    v.set_brush(lo, hi, 3)
    cam = synth.orbit_camera(20 + src.shape[-1], 25, 2.8)
    for lod, want in enumerate(levels):
        m = want.shape[1]
        _, cnt = v.render(cam, 61, 47, lod=lod, counts=True, ert=False, step=0.03)
        _, ref = oracle.render(want, 0.1, 1.0, cam.as_array(), 61, 47, 0.03, lo, hi, 3, TF, 0, 0.0, 1.0, ert=False)
        assert m < 2 or np.array_equal(cnt.cpu().numpy().astype(np.uint32), ref), lod


@pytest.mark.parametrize("store", ["f32", "f16"])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float16])
@pytest.mark.parametrize("n,aligned", [(4, True), (5, True), (12, True), (30, False), (36, True), (36, False), (67, True),
                                       (128, True), (132, True), (144, True), (272, True)])
def test_passes_match_oracle(rp, store, dtype, n, aligned):
    n_lod = 2 if n >= 8 else 1
    with rp.Context(0) as ctx:
        src = source(n, dtype, 1, aligned)
        v = ctx.load_volume(src, store=store, r_in=0.1)
        v.set_tf(TF, 0, 0.0, 1.0)
        v.build_bricks(n_lod=n_lod)                    # every level from the one above it
        check(v, src, store, n_lod)
        for seed, lods in ((2, n_lod), (3, 1), (4, n_lod)):
            src = source(n, dtype, seed, aligned)       # the update writes what it can on the way
            v.update(src)
            v.build_bricks(n_lod=lods)
            check(v, src, store, lods)
        src = source(n, dtype, 5, aligned)              # an update that no build follows, then one that one does
        v.update(src)
        src = source(n, dtype, 6, aligned)
        v.update(src)
        v.build_bricks(n_lod=n_lod)
        v.build_bricks(n_lod=n_lod)                    # built again from the levels themselves
        check(v, src, store, n_lod)
