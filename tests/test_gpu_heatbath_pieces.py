"""Heatbath sweeps on a device with too little memory for a whole class's scratch: the class is
updated in pieces, with the same chain."""
import numpy as np
import pytest

from paper_1112_5280_gb300 import lqcd, synth

pytestmark = pytest.mark.gpu

MIB = 1 << 20
DIMS = (16, 18, 14, 34)  # 68544 half-sites: 9.4 MiB of scratch, no multiple of a CTA's links


def test_sweeps_in_pieces():
    import torch

    ctx = lqcd.Context(0)
    rng = np.random.default_rng(3)
    pool = synth.random_links((2, 2, 2, 2), 0.5, seed=3)
    links = pool[rng.integers(0, 16, int(np.prod(DIMS)))]
    out = []
    for left in (None, 8 * MIB):
        g = ctx.gauge(DIMS, links)
        g.heatbath(5.7, 1, seed=9)  # its double-float copy is there from now on
        rest = None
        if left:
            ctx.release_cache()  # the scratch too
            torch.cuda.synchronize()
            rest = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")
        fails = g.heatbath(5.7, 2, seed=9, sweep0=1)
        del rest
        torch.cuda.empty_cache()
        out.append((fails, g.download()))
        g.close()
    assert out[0][0] == out[1][0] and np.array_equal(out[0][1], out[1][1])
    ctx.close()
