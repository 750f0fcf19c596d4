"""Twisted Dslash epilogues at the edges of a 64-site tile, and beside Wilson slots.

Operator launches run the epilogue without the reduction code; the double-float form does its
epilogue on packed pairs and skips factors of one, which an untwisted slot of a twisted launch
must not show. Bars: those of the operators' parity (FP64 and DF64 1e-12, FP32 1e-5, FP16 4e-3,
BF16 3e-2 of the largest component).
"""
import numpy as np
import pytest

import oracle
from paper_1112_5280_gb300 import lqcd, synth

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-12, "df64": 1e-12, "f32": 1e-5, "f16": 4e-3, "bf16": 3e-2}


@pytest.fixture(scope="module")
def ctx():
    c = lqcd.Context(0)
    yield c
    c.close()


# V/2 = 8, 56, 64, 72 and 136 sites: below, at and past one tile of 64, and past two
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 2, 2, 14), (2, 4, 4, 4), (2, 2, 2, 18), (2, 2, 2, 34)])
@pytest.mark.parametrize("prec", sorted(TOL))
def test_twisted_operators_at_tile_edges(ctx, dims, prec):
    U = synth.random_links(dims, 0.5, seed=41)
    psi = synth.gaussian_spinor(dims, seed=42)
    g = ctx.gauge(dims, U, prec=prec)
    ev = synth.parity_of_sites(dims) == 0
    fe, fo = ctx.field(dims, prec, lqcd.EVEN, data=psi), ctx.field(dims, prec, lqcd.EVEN)
    for dag in (False, True):
        lqcd.apply_Mhat(g, 0.15, fe, fo, dagger=dag, mu=0.4)
        got = fo.download()[ev]
        ref = oracle.apply_Mhat(dims, U, 0.15, psi * ev[:, None, None], dagger=dag, mu=0.4)[ev]
        assert np.abs(got - ref).max() < TOL[prec] * np.abs(ref).max()


@pytest.mark.parametrize("sloppy", ["df64", "f32", "f16"])
def test_wilson_slot_beside_a_twisted_one(ctx, sloppy):
    dims = (2, 2, 4, 18)
    eng = lqcd.Engine(ctx, lqcd.solve_opts(sloppy_prec=sloppy), max_slots=4)
    items = []
    for seed, mu in ((1, 0.0), (2, 0.2), (3, 0.0)):
        g = ctx.gauge(dims, synth.random_links(dims, 0.4, seed=seed))
        src = ctx.field(dims, data=synth.gaussian_spinor(dims, seed=seed + 10))
        items.append((eng.submit(g, src, 0.13, 1e-10, mu=mu), mu, g, src))
    while eng.step() > 0:
        pass
    for rid, mu, g, src in items:
        x, alone = ctx.field(dims), ctx.field(dims)
        assert eng.result(rid, x)["status"] == 0
        lqcd.solve_fields(g, src, 0.13, 1e-10, alone, lqcd.solve_opts(sloppy_prec=sloppy, mu=mu))
        assert np.array_equal(x.download(), alone.download())
    eng.close()
