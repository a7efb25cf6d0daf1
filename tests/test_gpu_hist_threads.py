"""Histograms of several contexts at once, from threads of one process: calls of different sizes set
the same kernels' limits."""
import threading

import numpy as np
import pytest
import torch

from paper_2207_12011_gb300 import synth

pytestmark = pytest.mark.gpu


def test_two_contexts_with_tables_of_different_sizes():
    import paper_2207_12011_gb300.raypc as rp
    n = 128
    vol = synth.make_shell_volume(n, device="cuda").half()
    kinds = [(2, 218), (2, 256)]                             # listed, with tables of different sizes
    tables = [np.array(synth.make_edges(vol.float(), [a % 6 for a in range(k)], b), dtype=np.float32) for k, b in kinds]
    errors, counts = [], {}

    def work(t):
        try:
            s = torch.cuda.Stream()
            with rp.Context(0) as ctx:
                v = ctx.load_volume(vol, store="f16", stream=s)
                v.build_bricks(stream=s)
                outs = [torch.empty((k - 1, b, b), dtype=torch.int32, device="cuda") for k, b in kinds]
                for i in range(6000):
                    j = t % len(kinds)
                    v.pc_histogram([a % 6 for a in range(kinds[j][0])], tables[j], use_brush=False, out=outs[j], stream=s)
                s.synchronize()
                counts[t] = [int(o.long().sum()) for o in outs]
        except Exception as e:                                # noqa: BLE001 (reported by the test)
            errors.append(e)

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    assert len({counts[t][t % len(kinds)] for t in counts}) == 1 and counts[0][0] > 0      # every in-shell cell, once
