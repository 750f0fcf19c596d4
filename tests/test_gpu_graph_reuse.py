"""The solver's captured graph is used again for a solve whose launches have the same shape:
other links, sources, kappas and tolerances of one lattice, and changes of shape in between
(another lattice, several systems, the twisted operator, the normal equations, a grid cap),
give the bits of the same solve on a context of its own."""
import numpy as np
import pytest

from paper_1112_5280_gb300 import lqcd, synth

pytestmark = pytest.mark.gpu

SMALL, OTHER = (4, 4, 4, 8), (6, 4, 4, 6)


def _solve(ctx, dims, seed, kappa, prec, mu=0.0, n=1, normal=False):
    g = ctx.gauge(dims, synth.random_links(dims, 0.5, seed=seed))
    srcs = [ctx.field(dims, data=synth.gaussian_spinor(dims, seed=seed + 1 + k)) for k in range(n)]
    xs = [ctx.field(dims) for _ in srcs]
    opts = lqcd.solve_opts(sloppy_prec=prec, mu=mu)
    if normal:
        infos = [lqcd.solve_normal(g, srcs[0], kappa, 1e-10, xs[0], opts)]
    else:
        infos = lqcd.solve_multi(g, srcs, kappa, 1e-10, xs, opts)
    assert all(i["status"] == 0 and i["true_resid"] <= 1e-10 for i in infos)
    return [x.download() for x in xs], [i["iters"] for i in infos]


@pytest.mark.parametrize("prec", ["f16", "f32", "f64", "df64"])
def test_reused_graph_gives_the_same_bits(prec):
    jobs = [dict(dims=SMALL, seed=11, kappa=0.13), dict(dims=SMALL, seed=21, kappa=0.15),
            dict(dims=SMALL, seed=31, kappa=0.12, mu=0.02), dict(dims=SMALL, seed=41, kappa=0.14, n=3),
            dict(dims=OTHER, seed=51, kappa=0.14), dict(dims=SMALL, seed=61, kappa=0.14, normal=True),
            dict(dims=SMALL, seed=11, kappa=0.13)]
    one = lqcd.Context(0)
    together = []
    for i, j in enumerate(jobs):
        if i == len(jobs) - 1:
            lqcd.set_grid_multiplier(0, 1)
        try:
            together.append(_solve(one, prec=prec, **j))
        finally:
            lqcd.set_grid_multiplier(0, 0)
    one.close()
    for j, (xs, iters) in zip(jobs, together):
        own = lqcd.Context(0)
        ys, own_iters = _solve(own, prec=prec, **j)
        assert iters == own_iters
        assert all(np.array_equal(x, y) for x, y in zip(xs, ys))
        own.close()
