"""FP16 sources: the same values as FP32 ones give, and no longer to take them in (half the bytes)."""
import pytest
import torch

from paper_2207_12011_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,store", [(251, "f32"), (251, "f16"), (256, "f32"), (252, "f16")])
def test_f16_sources(n, store):
    import paper_2207_12011_gb300.raypc as rp
    half = synth.make_shell_volume(n, device="cuda").half()
    full = half.float()
    with rp.Context(0) as ctx:
        v = ctx.load_volume(full, store=store)
        v.build_bricks(n_lod=1)

        def ms(src):
            best = []
            for _ in range(8):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                v.update(src)
                b.record()
                torch.cuda.synchronize()
                best.append(a.elapsed_time(b))
            v.build_bricks(n_lod=1)
            return min(best), [v.export(lod).clone() for lod in (0, 1)], [t.clone() for t in v.sub_bricks(1, classify=False)[:2]]

        ms(full)
        (tf, lf, bf), (th, lh, bh) = ms(full), ms(half)
        assert all(torch.equal(a, b) for a, b in zip(lf + bf, lh + bh))
        assert th < 1.15 * tf
