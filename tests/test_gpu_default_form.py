"""The FP32 Dslash without a tuning table: the default form against the other one named in a
table, Wilson and twisted, on launches below and beyond one wave of resident CTAs (152 SMs x
8 tiles of 64 sites: 77824 half-sites). The two forms run the same operations in the same
order, so the results are the same bits."""
import json

import numpy as np
import pytest

from paper_1112_5280_gb300 import lqcd, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(4, 4, 2, 6), (20, 18, 16, 28)])  # 96 and 80640 half-sites
@pytest.mark.parametrize("compress", [12, 18])
@pytest.mark.parametrize("mu", [0.0, 0.03])
def test_default_form_is_bitwise_form_0(tmp_path, dims, compress, mu):
    ctx = lqcd.Context(0)
    rng = np.random.default_rng(4)
    v = int(np.prod(dims))
    U = synth.random_links((2, 2, 2, 2), 0.5, seed=3)
    U = U[rng.integers(0, 16, v)]  # any SU(3) links will do
    psi = synth.gaussian_spinor(dims, seed=5)
    g = ctx.gauge(dims, U, "f32", compress)
    fin, fout = ctx.field(dims, "f32", lqcd.EVEN, data=psi), ctx.field(dims, "f32", lqcd.EVEN)

    def mhat():
        lqcd.apply_Mhat(g, 0.14, fin, fout, mu=mu)
        return fout.download()

    lqcd.tune_clear()
    default = mhat()
    g1 = ctx.gauge((4, 4, 4, 8), synth.unit_links((4, 4, 4, 8)), prec="f32")
    lqcd.autotune_dslash([g1], "f32")
    path = tmp_path / "tune.json"
    lqcd.tune_save(path)
    doc = json.loads(path.read_text())
    ntiles = (v // 2 + 63) // 64
    doc["entries"] = [{"prec": 1, "nr": compress, "nrhs": 0, "bucket": ntiles.bit_length() - 1, "ntiles": ntiles,
                       "ctas_per_sm": 0, "form": 0, "group": 0, "candidates": 2, "us_best": 1.0, "us_default": 1.0}]
    path.write_text(json.dumps(doc))
    lqcd.tune_clear()
    lqcd.tune_load(path)
    try:
        assert np.array_equal(default, mhat())
    finally:
        lqcd.tune_clear()
    ctx.close()
