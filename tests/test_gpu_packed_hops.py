"""The packed FP32 hops give the bits of the scalar ones: solves whose Dslash shares link loads
(scalar hops) against solves whose slots load their own (packed hops), on lattices with a
ragged last tile and with coinciding neighbours, both t boundaries, 18 and 12 link reals."""
import numpy as np
import pytest

from paper_1112_5280_gb300 import lqcd, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,t_bc", [((6, 6, 4, 10), -1), ((2, 4, 2, 18), 1), ((2, 2, 2, 2), -1)])
@pytest.mark.parametrize("prec", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("compress", [18, 12])
def test_packed_hops_equal_scalar_hops(dims, t_bc, prec, compress):
    ctx = lqcd.Context(0)
    g = ctx.gauge(dims, synth.random_links(dims, 0.5, seed=61), "f64", 18, t_bc)
    src = [ctx.field(dims, data=synth.gaussian_spinor(dims, seed=62 + k)) for k in range(3)]
    got = []
    for links in (1, -1):
        x = [ctx.field(dims) for _ in src]
        opts = lqcd.solve_opts(sloppy_prec=prec, sloppy_compress=compress, multi_rhs_links=links)
        infos = lqcd.solve_multi(g, src, 0.13, 1e-10, x, opts)
        assert all(i["status"] == 0 for i in infos)
        got.append(([i["iters"] for i in infos], [f.download() for f in x]))
    assert got[0][0] == got[1][0]
    for a, b in zip(got[0][1], got[1][1]):
        assert np.array_equal(a, b)
    ctx.close()


@pytest.mark.parametrize("dagger", [False, True])
def test_plain_f16_12_either_side_of_one_wave(dagger):
    """Operators of up to 8 CTAs per SM and larger launches use two register budgets: one
    16^3x32 application (1024 tiles) against two in a batch (2048), bit for bit."""
    dims = (16, 16, 16, 32)
    ctx = lqcd.Context(0)
    g = ctx.gauge(dims, synth.random_links(dims, 0.5, seed=71), "f16", 12)
    ins = [ctx.field(dims, "f16", lqcd.EVEN, synth.gaussian_spinor(dims, seed=72 + k)) for k in range(2)]
    outs = [ctx.field(dims, "f16", lqcd.ODD) for _ in range(4)]
    batch = lqcd.DslashBatch([g, g], ins, outs[:2], 1, dagger)
    batch.apply()
    for k in range(2):
        lqcd.dslash_eo(g, ins[k], outs[2 + k], 1, dagger)
        a, b = outs[k].download(), outs[2 + k].download()
        assert np.array_equal(a, b) and np.abs(a).max() > 1
    batch.close()
    ctx.close()
