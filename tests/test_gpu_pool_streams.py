"""Objects destroyed while work outside the context's stream still reads them: their memory does
not go to the next object before that work is done."""
import numpy as np
import pytest

from paper_1112_5280_gb300 import lqcd, synth

pytestmark = pytest.mark.gpu

DIMS = (6, 4, 4, 10)
SLEEP = 200_000_000  # clock cycles, about 0.1 s: the host is through long before


def _others(ctx, n):
    """New objects of the destroyed ones' sizes, full of other values."""
    other = synth.gaussian_spinor(DIMS, seed=99)
    return [ctx.field(DIMS, "f32", data=other) for _ in range(n)] + [ctx.gauge(DIMS, synth.random_links(DIMS, 0.6, seed=98), "f32")]


def test_destroyed_while_a_graph_replays():
    import torch

    st, elsewhere = torch.cuda.Stream(), torch.cuda.Stream()
    ctx = lqcd.Context(0, stream=st)
    psi = synth.gaussian_spinor(DIMS, seed=4)
    g = ctx.gauge(DIMS, synth.random_links(DIMS, 0.6, seed=9), "f32")
    a, b = ctx.field(DIMS, "f32", data=psi), ctx.field(DIMS, "f32")
    out = torch.zeros((int(np.prod(DIMS)), 4, 3), dtype=torch.complex128, device="cuda")

    def chain():
        lqcd.apply_M(g, 0.14, a, b)
        b.download(out)

    chain()
    ctx.sync()
    want = out.cpu().numpy()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        torch.cuda._sleep(SLEEP)
        chain()
    out.zero_()
    torch.cuda.synchronize()
    with torch.cuda.stream(elsewhere):
        graph.replay()
    for o in (a, b, g):
        o.close()
    objs = _others(ctx, 2)
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy(), want) and np.abs(want).max() > 1
    del graph, objs
    ctx.close()


def test_destroyed_while_another_context_copies():
    import torch

    st = torch.cuda.Stream()
    one, two = lqcd.Context(0), lqcd.Context(0, stream=st)
    psi = synth.gaussian_spinor(DIMS, seed=4)
    a, b = one.field(DIMS, "f32", data=psi), two.field(DIMS, "f32")
    want = a.download()
    with torch.cuda.stream(st):
        torch.cuda._sleep(SLEEP)
    b.copy_from(a)
    a.close()
    objs = _others(one, 2)
    assert np.array_equal(b.download(), want)
    del objs
    one.close()
    two.close()
