"""A CG step whose |Mhat p|^2 is zero or not finite, found while the next launch runs: the slot
stops with its status and its last accepted solution, and its neighbours go on untouched."""
import numpy as np
import pytest

from paper_1112_5280_gb300 import lqcd, synth

pytestmark = pytest.mark.gpu

DIMS = (4, 4, 4, 8)


def _constant(dims):
    return np.full((int(np.prod(dims)), 4, 3), 1 + 1j)


# On unit links with periodic time the constant spinor is an eigenvector of the hopping term
# with eigenvalue 8, so Mhat = 1 - 64 kappa^2 takes it to zero, exactly, at kappa = 1/8. A
# kappa whose square is near the largest number of the storage overflows |Mhat p|^2.
FAILURES = {"breakdown": lambda prec: (0.125, lqcd.EBREAKDOWN),
            "nonfinite": lambda prec: (1e80 if prec == "f64" else 1e17, lqcd.ENONFINITE)}


@pytest.mark.parametrize("prec", ["f64", "df64", "f32", "f16"])
@pytest.mark.parametrize("failure", list(FAILURES))
@pytest.mark.parametrize("use_graph", [1, 0])
def test_failed_step_stops_its_slot_only(prec, failure, use_graph):
    kappa, status = FAILURES[failure](prec)
    opts = lqcd.solve_opts(sloppy_prec=prec, use_graph=use_graph)
    ctx = lqcd.Context(0)
    unit = ctx.gauge(DIMS, synth.unit_links(DIMS), t_bc=1)
    const = ctx.field(DIMS, data=_constant(DIMS))
    g = ctx.gauge(DIMS, synth.random_links(DIMS, 0.5, seed=5))
    src = ctx.field(DIMS, data=synth.gaussian_spinor(DIMS, seed=6))

    x = ctx.field(DIMS)
    info = lqcd.solve_normal(unit, const, kappa, 1e-10, x, opts)
    assert info["status"] == status and info["iters"] == 0
    assert not x.download().any()  # the initial solution

    want = ctx.field(DIMS)
    alone = lqcd.solve_normal(g, src, 0.14, 1e-10, want, opts)
    eng = lqcd.Engine(ctx, opts, max_slots=2)
    bad = eng.submit(unit, const, kappa, 1e-10, normal=True)
    good = eng.submit(g, src, 0.14, 1e-10, normal=True)
    while eng.step():
        pass
    with pytest.raises(lqcd.LqcdError) as err:
        eng.result(bad, x)
    assert err.value.code == status
    assert not x.download().any()
    assert eng.result(good, x)["iters"] == alone["iters"]
    assert np.array_equal(x.download(), want.download())
    eng.close()
    ctx.close()
