"""Packed FP32 hops (slots that load their own links) against scalar ones (slots that share link
loads), bit for bit over whole solves: a loaded tuning table names the shared form, which the
engine's own rule does not take for three slots on such small lattices. Ragged last tiles,
coinciding neighbours, both t boundaries, 18 and 12 link reals."""
import json

import numpy as np
import pytest

from paper_1112_5280_gb300 import lqcd, synth

pytestmark = pytest.mark.gpu

CODE = {"f32": 1, "f16": 2, "bf16": 3}
TILE, NRHS = 64, 3


@pytest.fixture
def tag(tmp_path):
    """The device tag of a saved table."""
    ctx = lqcd.Context(0)
    lqcd.tune_clear()
    lqcd.autotune_dslash([ctx.gauge((4, 4, 4, 4), synth.unit_links((4, 4, 4, 4)), "f32")], "f32")
    lqcd.tune_save(tmp_path / "tag.json")
    lqcd.tune_clear()
    ctx.close()
    yield json.loads((tmp_path / "tag.json").read_text())["device"]
    lqcd.tune_clear()


@pytest.mark.parametrize("dims,t_bc", [((6, 6, 4, 10), -1), ((2, 4, 2, 18), 1), ((2, 2, 2, 2), -1)])
@pytest.mark.parametrize("prec", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("compress", [18, 12])
def test_packed_hops_equal_scalar_hops(tag, tmp_path, dims, t_bc, prec, compress):
    blocks = (int(np.prod(dims)) // 2 + TILE - 1) // TILE
    ctx = lqcd.Context(0)
    g = ctx.gauge(dims, synth.random_links(dims, 0.5, seed=61), "f64", 18, t_bc)
    src = [ctx.field(dims, data=synth.gaussian_spinor(dims, seed=62 + k)) for k in range(NRHS)]

    def run(links):
        x = [ctx.field(dims) for _ in src]
        opts = lqcd.solve_opts(sloppy_prec=prec, sloppy_compress=compress, multi_rhs_links=links)
        infos = lqcd.solve_multi(g, src, 0.13, 1e-10, x, opts)
        assert all(i["status"] == 0 for i in infos)
        return [i["iters"] for i in infos], [f.download() for f in x]

    own = run(-1)
    for group in (2, 3):
        entry = {"prec": CODE[prec], "nr": compress, "nrhs": NRHS, "bucket": blocks.bit_length() - 1,
                 "ntiles": blocks * NRHS, "ctas_per_sm": 0, "form": 2, "group": group, "candidates": 1,
                 "us_best": 1.0, "us_default": 1.0}
        path = tmp_path / f"g{group}.json"
        path.write_text(json.dumps({"format": "lqcd-tune", "version": 2, "device": tag, "entries": [entry]}))
        lqcd.tune_clear()
        lqcd.tune_load(path)
        shared = run(1)
        lqcd.tune_clear()
        assert shared[0] == own[0]
        assert all(np.array_equal(a, b) for a, b in zip(shared[1], own[1]))
    ctx.close()
