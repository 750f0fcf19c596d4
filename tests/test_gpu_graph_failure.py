"""A step whose graph cannot be captured (the legacy default stream takes no capture) reports the
error and leaves the engine able to go on: the next step builds the graph of the present slots,
and every solution is that of an engine without the failure, in the same number of steps."""
import numpy as np
import pytest

from paper_1112_5280_gb300 import lqcd, synth

pytestmark = pytest.mark.gpu

LEGACY_STREAM = 1  # cudaStreamLegacy
SYSTEMS = [((6, 4, 4, 8), 0.15, 1e-11), ((4, 4, 4, 8), 0.10, 1e-6)]  # the second finishes first


def _run(fail):
    """Both systems; fail: after the submission of the second (grow) or when it is done (shrink)."""
    ctx = lqcd.Context(0)
    eng = lqcd.Engine(ctx, lqcd.solve_opts(sloppy_prec="f32"), max_slots=4)
    ids, xs, objs = [], [], []

    def submit(k):
        dims, kappa, tol = SYSTEMS[k]
        g = ctx.gauge(dims, synth.random_links(dims, 0.5, seed=3 + k))
        src = ctx.field(dims, data=synth.gaussian_spinor(dims, seed=7 + k))
        objs.extend((g, src))
        xs.append(ctx.field(dims))
        ids.append(eng.submit(g, src, kappa, tol))

    def failing_step():
        ctx.set_stream(LEGACY_STREAM)
        with pytest.raises(lqcd.LqcdError):
            eng.step()
        ctx.set_stream(None)

    submit(0)
    assert eng.step() == 1
    submit(1)
    if fail == "grow":
        failing_step()
        failing_step()
    steps, active, done = 0, 2, []
    while active:
        if fail == "shrink" and active == 1:
            failing_step()
            fail = None
        active = eng.step()
        steps += 1
        done += eng.completed()
    assert done == [ids[1], ids[0]]
    out = [(eng.result(i, x)["iters"], x.download()) for i, x in zip(ids, xs)]
    eng.close()
    ctx.close()
    return steps, out


@pytest.mark.parametrize("fail", ["grow", "shrink"])
def test_engine_goes_on_after_a_failed_capture(fail):
    want_steps, want = _run(None)
    steps, got = _run(fail)
    assert steps == want_steps
    for (iters, x), (want_iters, y) in zip(got, want):
        assert iters == want_iters and np.array_equal(x, y)
