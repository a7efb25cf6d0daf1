"""The largest magnitudes of a level's stored values, which decide how its cells are classified:
they belong to the values that the level holds, on whatever stream they came in."""
import numpy as np
import pytest
import torch

import oracle
from paper_2207_12011_gb300 import synth
from test_gpu_parity import bits, stored

pytestmark = pytest.mark.gpu
R_IN, R_OUT = 0.3, 1.0


@pytest.fixture(scope="module")
def rp():
    import paper_2207_12011_gb300.raypc as rp
    rp.lib()
    return rp


def field(n, seed, nans):
    """Two smooth variables; with nans, some values of the first are NaN."""
    vol = synth.make_shell_volume(n, seed=seed)[:2].contiguous()
    if nans:
        vol[0, ::5, ::7, ::3] = float("nan")
    return vol


def wide_brush(vol):
    """Every number of the first variable passes; the second is cut at two of its values."""
    s = vol[1].flatten().sort().values
    return np.array([-1e30, float(s[len(s) // 5])], np.float32), np.array([1e30, float(s[-len(s) // 8])], np.float32), 0b11


def check_classes(rp, v, st, brush, lod=0, stream=None):
    """Activity and classes of a level under the volume's brush against the oracle on its values."""
    n = st.shape[1]
    nsb = (n + 3) // 4
    lo, hi, mask = brush
    words = v.sub_bricks(lod, stream=stream)[2]
    got = v.cell_classes(lod, stream=stream)
    torch.cuda.synchronize()
    mn, mx = oracle.brick_minmax(st, 4)
    want, _ = oracle.classify(mn, mx, n, R_IN, R_OUT, lo, hi, mask, bs=4)
    act = bits(rp, words, nsb ** 3).reshape(nsb, nsb, nsb).astype(bool)
    assert np.array_equal(act, want.reshape(act.shape).astype(bool))
    idx = np.arange(n) // 4
    sel = act[idx[:, None, None], idx[None, :, None], idx[None, None, :]]
    sel[n - 1], sel[:, n - 1], sel[:, :, n - 1] = False, False, False
    got, ref = got.cpu().numpy().view(np.uint16), oracle.cell_classes(st, lo, hi, mask)
    assert np.array_equal(got[sel], ref[sel]), np.argwhere((got != ref) & sel)[:4]


@pytest.mark.parametrize("store", ["f32", "f16"])
def test_load_on_a_stream_beside_a_busy_default_stream(rp, store):
    """A volume that comes in on a stream of its own, and its coarser level, while the default stream
    has work queued: nothing of theirs waits for, or is undone by, the default stream's order."""
    n = 48
    vol = field(n, 3, True)
    src, brush, st = vol.cuda(), wide_brush(torch.nan_to_num(vol)), stored(vol, store)
    busy = torch.empty((4096, 4096), device="cuda", dtype=torch.bfloat16).normal_()
    side = torch.cuda.Stream()
    with rp.Context(0) as ctx:
        torch.cuda.synchronize()
        for _ in range(200):
            busy @ busy
        v = ctx.load_volume(src, store=store, r_in=R_IN, r_out=R_OUT, stream=side)
        v.build_bricks(n_lod=1, stream=side)
        torch.cuda.synchronize()
        v.set_brush(*brush, stream=side)
        check_classes(rp, v, st, brush, stream=side)
        coarse = oracle.lod_mean(st)
        coarse = coarse.astype(np.float16).astype(np.float32) if store == "f16" else coarse
        check_classes(rp, v, coarse, brush, lod=1, stream=side)


@pytest.mark.parametrize("store", ["f32", "f16"])
@pytest.mark.parametrize("n", [48, 128])                     # level 1 by its own pass, and from the ingest
def test_recorded_time_steps_in_turn(rp, store, n):
    """Two time steps with NaN and a finite one, whose update, levels and brush edit are recorded in
    graphs: replayed in turn, and after a direct update, each leaves the classes of its own values."""
    steps = [field(n, 3, True), field(n, 5, True).flip(1) * 7, field(n, 5, False)]
    brush = wide_brush(steps[2])
    srcs, sts = [s.cuda() for s in steps], [stored(s, store) for s in steps]
    side = torch.cuda.Stream()
    with rp.Context(0) as ctx:
        v = ctx.load_volume(srcs[1], store=store, r_in=R_IN, r_out=R_OUT)

        def step(i):
            s = torch.cuda.current_stream()
            v.update(srcs[i], stream=s)
            v.build_bricks(n_lod=1, stream=s)
            v.set_brush(*brush, stream=s)
            return v.cell_classes(stream=s)

        v.build_bricks(n_lod=1)
        step(0)                                              # the buffers exist from here on
        torch.cuda.synchronize()
        graphs, outs = [], []
        for i in range(3):
            graphs.append(torch.cuda.CUDAGraph())
            with torch.cuda.graph(graphs[i], stream=side):
                outs.append(step(i))
        for i in (0, 1, 0, 2, 1, None, 0, 2):
            if i is None:
                step(1)
            else:
                graphs[i].replay()
            torch.cuda.synchronize()
            if i is not None:
                check_classes(rp, v, sts[i], brush)
                assert torch.equal(outs[i], v.cell_classes())
        del graphs


def test_update_with_nan_takes_the_time_of_one_without(rp):
    """Masked data has NaN in half of its cells: their ingest moves the same bytes as any other and has
    to take about its time (one atomic per thread that met a NaN took five times as long)."""
    n = 256
    vol = synth.make_shell_volume(n, device="cuda").half()
    masked = vol.clone()
    masked[:, ::2] = float("nan")
    with rp.Context(0) as ctx:
        v = ctx.load_volume(vol, store="f16")

        def ms(src):
            best = []
            for _ in range(8):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                v.update(src)
                b.record()
                torch.cuda.synchronize()
                best.append(a.elapsed_time(b))
            return min(best)

        ms(vol)
        assert ms(masked) < 2.0 * ms(vol)


@pytest.mark.parametrize("store", ["f32", "f16"])
@pytest.mark.parametrize("n", [2, 3, 6, 17, 34, 45, 66, 128, 130])
def test_classes_of_masked_fields(rp, store, n):
    """Fields with NaN in whole regions, in single cells on and beside sub-brick borders and in their
    last planes, and infinite values in one variable: both levels' classes against the oracle."""
    vol = synth.make_shell_volume(n, seed=n)[:3].contiguous()
    if n < 20:
        vol = vol + torch.randn(vol.shape, generator=torch.Generator().manual_seed(n))
    brush2 = wide_brush(vol)
    lo, hi = np.append(brush2[0], -np.inf).astype(np.float32), np.append(brush2[1], np.float32(vol[2].median())).astype(np.float32)
    for kind in ("region", "cells", "last", "inf"):
        x = vol.clone()
        if kind == "region":
            x[0, : n // 2, :, n // 3:] = float("nan")
            x[1, :, n // 2:, : n // 2] = float("nan")
        elif kind == "cells":
            for c in range(0, n, 4):
                x[0, c, c, c] = float("nan")
                x[1, (c + 3) % n, c, (c + 1) % n] = float("nan")
                x[2, c, (c + 2) % n, n - 1 - c] = float("nan")
        elif kind == "last":
            x[0, -1], x[1, :, -1], x[2, :, :, -1] = (float("nan"),) * 3
        else:
            x[1, n // 2, n // 3, n // 4] = float("inf")
            x[2, n // 4, n // 2, n // 3] = -float("inf")
        st = stored(x, store)
        with rp.Context(0) as ctx:
            v = ctx.load_volume(x.cuda(), store=store, r_in=R_IN, r_out=R_OUT)
            v.build_bricks(n_lod=1 if n >= 4 else 0)
            v.update(x.cuda())                               # level 1 from the ingest where it fits
            v.build_bricks(n_lod=1 if n >= 4 else 0)
            v.set_brush(lo, hi, 0b111)
            for lod in range(2 if n >= 4 else 1):
                if lod:
                    st = oracle.lod_mean(st)
                    st = st.astype(np.float16).astype(np.float32) if store == "f16" else st
                m = st.shape[1]
                act = bits(rp, v.sub_bricks(lod)[2], ((m + 3) // 4) ** 3)
                if act.any() and m > 2:
                    check_classes(rp, v, st, (lo, hi, 0b111), lod)
