"""One slot with more than 58 MiB of links reads them past L1, two slots on one gauge field of
that size do not: operators and solves are the same bit for bit, for every precision with that
choice, with a ragged last tile."""
import numpy as np
import pytest

from paper_1112_5280_gb300 import lqcd, synth

pytestmark = pytest.mark.gpu

DIMS = (22, 20, 26, 58)  # 5183.75 tiles; 60.7 MiB of FP16 links with 12 reals
BYTES = {"f32": 4, "f16": 2, "bf16": 2}


@pytest.fixture(scope="module")
def data():
    rng = np.random.default_rng(8)
    pool = synth.random_links((2, 2, 2, 2), 0.5, seed=8)
    vol = int(np.prod(DIMS))
    spinors = [rng.standard_normal((vol, 4, 3, 2)).view(np.complex128)[..., 0] for _ in range(2)]
    return pool[rng.integers(0, 16, vol)], spinors


def _in_range(prec, compress):
    return 58 << 20 < np.prod(DIMS) * 4 * compress * BYTES[prec] <= 256 << 20


@pytest.mark.parametrize("prec", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("compress", [12, 18])
@pytest.mark.parametrize("dagger", [False, True])
def test_operator(data, prec, compress, dagger):
    assert _in_range(prec, compress)
    links, spinors = data
    ctx = lqcd.Context(0)
    g = ctx.gauge(DIMS, links, prec, compress)
    fins = [ctx.field(DIMS, prec, lqcd.ODD, data=s) for s in spinors]
    both = [ctx.field(DIMS, prec, lqcd.EVEN) for _ in fins]
    one = ctx.field(DIMS, prec, lqcd.EVEN)
    lqcd.DslashBatch([g, g], fins, both, lqcd.EVEN, dagger).apply()
    for i, o in zip(fins, both):
        lqcd.dslash_eo(g, i, one, lqcd.EVEN, dagger)
        want = o.download()
        assert np.array_equal(one.download(), want) and np.abs(want).max() > 1
    ctx.close()


@pytest.mark.parametrize("prec,mu", [("f32", 0.02), ("f16", 0.0), ("bf16", 0.02)])
def test_solve(data, prec, mu):
    assert _in_range(prec, 12)
    links, spinors = data
    ctx = lqcd.Context(0)
    g = ctx.gauge(DIMS, links)
    srcs = [ctx.field(DIMS, data=s) for s in spinors]
    xs = [ctx.field(DIMS) for _ in srcs]
    one = ctx.field(DIMS)
    opts = lqcd.solve_opts(sloppy_prec=prec, mu=mu)
    infos = lqcd.solve_multi(g, srcs, 0.1, 1e-8, xs, opts)
    assert all(i["status"] == 0 for i in infos)
    for s, x, i in zip(srcs, xs, infos):
        assert lqcd.solve_fields(g, s, 0.1, 1e-8, one, opts)["iters"] == i["iters"]
        assert np.array_equal(one.download(), x.download())
    ctx.close()
