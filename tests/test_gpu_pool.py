"""Device buffers kept by a context between objects of one size: their content, their bound and
when they are given back."""
import numpy as np
import pytest

from paper_1112_5280_gb300 import lqcd, synth

pytestmark = pytest.mark.gpu

GIB = 1 << 30


def _free():
    import torch

    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_reused_buffers_hold_nothing_of_the_last_object():
    dims = (4, 4, 4, 6)
    ctx = lqcd.Context(0)
    psi = synth.gaussian_spinor(dims, seed=1)
    for prec in ("f64", "df64", "f32", "f16"):  # FP64 and double-float fields have one size
        f = ctx.field(dims, prec, lqcd.FULL, data=psi)
        f.close()
        assert not ctx.field(dims, prec, lqcd.FULL).download().any()
    want = None
    for compress in (18, 12, 18):  # FP32 links of 18 and 12 reals, and a new configuration
        U = synth.random_links(dims, 0.4, seed=compress)
        g = ctx.gauge(dims, U, "f32", compress)
        assert np.array_equal(g.download(), U)
        a, b = ctx.field(dims, "f32", data=psi), ctx.field(dims, "f32")
        lqcd.apply_M(g, 0.13, a, b)
        got = b.download()
        if compress == 18:
            assert want is None or np.array_equal(got, want)
            want = got
        for o in (a, b, g):
            o.close()
    ctx.close()


def test_pool_is_bounded_and_given_back():
    dims = (16, 16, 16, 32)  # 25.2 MB per FP64 field
    ctx = lqcd.Context(0)
    ctx.field(dims, "f64").close()
    ctx.release_cache()
    empty = _free()
    fields = [ctx.field(dims, "f64") for _ in range(80)]  # 2 GB
    for f in fields:
        f.close()
    held = empty - _free()
    assert 0 < held <= GIB + (64 << 20)  # allocation granularity
    ctx.release_cache()
    assert empty - _free() <= 32 << 20
    ctx.close()


def test_newest_buffers_stay():
    """A full pool makes room for the buffers freed last."""
    ctx = lqcd.Context(0)
    large, small = (16, 16, 16, 32), (8, 8, 8, 16)
    old = [ctx.field(large, "f64") for _ in range(50)]  # 1.26 GB
    for f in old:
        f.close()
    keep = [ctx.field(small, "f64") for _ in range(8)]
    for f in keep:
        f.close()
    before = _free()
    again = [ctx.field(small, "f64") for _ in range(8)]
    assert _free() == before  # from the pool
    for f in again:
        f.close()
    ctx.close()
