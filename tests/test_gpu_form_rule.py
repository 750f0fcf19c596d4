"""The FP32 Dslash without a tuning table on either side of the lines of the form rule: the default
against both forms named in a table, bit for bit, Wilson and twisted."""
import json

import numpy as np
import pytest

from paper_1112_5280_gb300 import lqcd, synth

pytestmark = pytest.mark.gpu

# tiles of 64 sites: two launches fit at 8 CTAs per SM only, one at 6, one at 8, two waves either
# way, two against three, more than four
SIZES = {512: (16, 16, 16, 16), 686: (14, 14, 14, 32), 1024: (16, 16, 16, 32), 1536: (16, 16, 16, 48),
         2048: (16, 16, 16, 64), 3780: (24, 24, 20, 42)}


@pytest.mark.parametrize("tiles", list(SIZES))
@pytest.mark.parametrize("compress", [12, 18])
def test_default_is_bitwise_both_forms(tmp_path, tiles, compress):
    dims = SIZES[tiles]
    assert int(np.prod(dims)) == 128 * tiles
    rng = np.random.default_rng(4)
    pool = synth.random_links((2, 2, 2, 2), 0.5, seed=3)
    psi = rng.standard_normal((128 * tiles, 4, 3, 2)).view(np.complex128)[..., 0]
    ctx = lqcd.Context(0)
    g = ctx.gauge(dims, pool[rng.integers(0, 16, 128 * tiles)], "f32", compress)
    fin, fout = ctx.field(dims, "f32", lqcd.EVEN, data=psi), ctx.field(dims, "f32", lqcd.EVEN)

    def mhat():
        out = []
        for mu in (0.0, 0.03):
            lqcd.apply_Mhat(g, 0.14, fin, fout, mu=mu)
            out.append(fout.download())
        return out

    lqcd.tune_clear()
    default = mhat()
    assert all(np.abs(x).max() > 1 for x in default)
    lqcd.autotune_dslash([ctx.gauge((4, 4, 4, 4), synth.unit_links((4, 4, 4, 4)), "f32")], "f32")
    path = tmp_path / "tune.json"
    lqcd.tune_save(path)
    doc = json.loads(path.read_text())
    try:
        for form in (0, 3):
            doc["entries"] = [{"prec": 1, "nr": compress, "nrhs": 0, "bucket": tiles.bit_length() - 1, "ntiles": tiles,
                               "ctas_per_sm": 0, "form": form, "group": 0, "candidates": 2, "us_best": 1.0,
                               "us_default": 1.0}]
            path.write_text(json.dumps(doc))
            lqcd.tune_clear()
            lqcd.tune_load(path)
            assert all(np.array_equal(a, b) for a, b in zip(default, mhat()))
    finally:
        lqcd.tune_clear()
    ctx.close()
