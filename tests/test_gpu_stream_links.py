"""Launches over several gauge fields whose links exceed half of L2 (64 MiB) read FP32 links
past L1; smaller ones and slots on one gauge field do not. The route changes no bit: a batch
equals its applications one by one, and a batched solve its solo solves."""
import numpy as np
import pytest

from paper_1112_5280_gb300 import lqcd, synth

pytestmark = pytest.mark.gpu


def _links(dims, seed):
    """Any SU(3) links: a few matrices spread over the lattice."""
    pool = synth.random_links((2, 2, 2, 2), 0.5, seed=seed)
    return pool[np.random.default_rng(seed).integers(0, 16, int(np.prod(dims)))]


@pytest.mark.parametrize("compress", [12, 18])
@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("shapes", [[(16, 12, 12, 28)] * 6, [(20, 18, 16, 32), (18, 16, 16, 28), (16, 12, 12, 18), (4, 4, 4, 4)]])
def test_batch_equals_single(compress, dagger, shapes):
    ctx = lqcd.Context(0)
    gs = [ctx.gauge(d, _links(d, 40 + k), "f32", compress) for k, d in enumerate(shapes)]
    assert sum(np.prod(d) * 4 * compress * 4 for d in shapes) > (64 << 20)
    fins = [ctx.field(d, "f32", lqcd.ODD, data=synth.gaussian_spinor(d, seed=50 + k)) for k, d in enumerate(shapes)]
    a, b = ([ctx.field(d, "f32", lqcd.EVEN) for d in shapes] for _ in range(2))
    lqcd.DslashBatch(gs, fins, a, lqcd.EVEN, dagger).apply()
    for g, i, o, r in zip(gs, fins, b, a):
        lqcd.dslash_eo(g, i, o, lqcd.EVEN, dagger)
        assert np.array_equal(o.download(), r.download())
    ctx.close()


@pytest.mark.parametrize("mu", [0.0, 0.02])
def test_batched_solves_equal_solo(mu):
    ctx = lqcd.Context(0)
    shapes = [(16, 12, 12, 28), (16, 12, 14, 24), (16, 16, 12, 24), (18, 12, 12, 24), (16, 12, 14, 26), (16, 16, 8, 10)]
    assert sum(np.prod(d) * 4 * 12 * 4 for d in shapes) > (64 << 20)
    gs = [ctx.gauge(d, _links(d, 60 + k)) for k, d in enumerate(shapes)]
    srcs = [ctx.field(d, data=synth.gaussian_spinor(d, seed=70 + k)) for k, d in enumerate(shapes)]
    xs, ys = ([ctx.field(d) for d in shapes] for _ in range(2))
    kappas = [0.10 + 0.004 * k for k in range(len(shapes))]
    opts = lqcd.solve_opts(sloppy_prec="f32", mu=mu)
    infos = lqcd.solve_batch(gs, srcs, kappas, 1e-9, xs, opts)
    assert all(i["status"] == 0 for i in infos)
    for g, s, k, x, y in zip(gs, srcs, kappas, xs, ys):
        lqcd.solve_fields(g, s, k, 1e-9, y, opts)
        assert np.array_equal(x.download(), y.download())
    ctx.close()
