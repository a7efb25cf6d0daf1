"""Classification and cell classes where their fast forms can go wrong: binary16 bounds at, between
and beyond the stored values, zeros of both signs, levels with a far outlier or with NaN and infinite
values (decided cell by cell), odd and tiny edges, groups cut by rows and words, and a volume that
turns finite again."""
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


def fields(n, kind, seed=3):
    """Four fields of mixed scale and sign; coarse steps make stored values meet the bounds."""
    rng = np.random.default_rng(seed + n)
    x = rng.normal(size=(4, n, n, n)).astype(np.float32)
    for a in range(1, 4):                                   # neighbours correlate, so that some cells are decided
        x += np.roll(x, 1, axis=a)
    x[1] *= 300.0
    x[2] = np.round(x[2] * 4) / 4                            # many equal values, zeros of both signs
    x[3] *= 1e-4
    if kind == "outlier":
        x[0, n // 2, n // 2, n // 2] = 60000.0
    elif kind == "nonfinite":
        x[0, n // 2, n // 2, n // 2] = np.nan
        x[1, n // 3, n // 3, n // 3] = np.inf
        x[2, n // 3, n // 2, n // 3] = -np.inf
    return torch.from_numpy(x)


def brushes(st):
    """Bounds at stored values, just beside them, at zero, open, empty and beyond binary16."""
    s = [np.sort(v[np.isfinite(v)].reshape(-1)) for v in st]
    q = lambda v, f: np.float32(s[v][int(f * (len(s[v]) - 1))])  # noqa: E731
    up, dn = np.float32(np.inf), np.float32(-np.inf)
    nx, pv = lambda a: np.nextafter(a, up), lambda a: np.nextafter(a, dn)  # noqa: E731
    yield [q(0, .2), q(1, .1), q(2, .2), q(3, .3)], [q(0, .9), q(1, .95), q(2, .8), q(3, .9)], 0b1111
    yield [nx(q(0, .2)), pv(q(1, .1)), 0.0, q(3, .01)], [pv(q(0, .9)), nx(q(1, .9)), up, q(3, .99)], 0b1111
    yield [-0.0, dn, -0.0, 0.0], [up, 0.0, 0.25, 1e30], 0b1111
    yield [-70000.0, -1e30, q(2, .1), dn], [70000.0, q(1, .7), q(2, .1), up], 0b0111
    yield [q(0, .5), dn, dn, dn], [q(0, .4), up, up, up], 0b0001


@pytest.mark.parametrize("store", ["f32", "f16"])
@pytest.mark.parametrize("n,kind", [(2, "plain"), (3, "plain"), (6, "plain"), (17, "plain"), (34, "outlier"), (45, "plain"),
                                    (64, "plain"), (66, "nonfinite"), (77, "nonfinite"), (130, "plain")])
def test_classes_match_oracle(rp, store, n, kind):
    vol = fields(n, kind)
    st = stored(vol, store)
    nsb = (n + 3) // 4
    idx = np.arange(n) // 4
    with rp.Context(0) as ctx:
        v = ctx.load_volume(vol.cuda(), store=store, r_in=R_IN, r_out=R_OUT)
        v.build_bricks()
        mn, mx = oracle.brick_minmax(st, 4)
        for lo, hi, mask in brushes(st):
            lo, hi = np.asarray(lo, np.float32), np.asarray(hi, np.float32)
            v.set_brush(lo, hi, mask)
            _, _, words = v.sub_bricks()
            want, _ = oracle.classify(mn, mx, n, R_IN, R_OUT, lo, hi, mask, bs=4)
            act = bits(rp, words, nsb ** 3).reshape(nsb, nsb, nsb).astype(bool)
            assert np.array_equal(act, want.reshape(act.shape).astype(bool))
            sel = act[idx[:, None, None], idx[None, :, None], idx[None, None, :]]
            sel[n - 1], sel[:, n - 1], sel[:, :, n - 1] = False, False, False
            got = v.cell_classes().cpu().numpy().view(np.uint16)
            ref = oracle.cell_classes(st, lo, hi, mask)
            assert np.array_equal(got[sel], ref[sel]), np.argwhere((got != ref) & sel)[:4]


@pytest.mark.parametrize("store", ["f32", "f16"])
def test_classes_after_updates(rp, store):
    """Time steps with and without non-finite values in turn, through the separate and the fused
    level passes, each against the oracle on its own values."""
    n = 128
    with rp.Context(0) as ctx:
        v = None
        for step, kind in enumerate(("plain", "nonfinite", "plain", "outlier", "plain")):
            vol = fields(n, kind, seed=20 + step)
            if v is None:
                v = ctx.load_volume(vol.cuda(), store=store, r_in=R_IN, r_out=R_OUT)
            else:
                v.update(vol.cuda())
            v.build_bricks(n_lod=1)
            st = stored(vol, store)
            lo, hi, mask = next(iter(brushes(st)))
            v.set_brush(lo, hi, mask)
            for lod, level in enumerate((st, oracle.lod_mean(st))):
                if lod and store == "f16":
                    level = level.astype(np.float16).astype(np.float32)
                m = level.shape[1]
                _, _, words = v.sub_bricks(lod)
                nsb = (m + 3) // 4
                act = bits(rp, words, nsb ** 3).reshape(nsb, nsb, nsb).astype(bool)
                idx = np.arange(m) // 4
                sel = act[idx[:, None, None], idx[None, :, None], idx[None, None, :]]
                sel[m - 1], sel[:, m - 1], sel[:, :, m - 1] = False, False, False
                got = v.cell_classes(lod).cpu().numpy().view(np.uint16)
                ref = oracle.cell_classes(level, np.asarray(lo, np.float32), np.asarray(hi, np.float32), mask)
                assert sel.any() and np.array_equal(got[sel], ref[sel]), (step, lod)
