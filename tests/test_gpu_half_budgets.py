"""The half-precision operators in both register budgets, on either side of the lines between
them: an application on its own against the same one in a batch of another size, bit for bit."""
import numpy as np
import pytest

from paper_1112_5280_gb300 import lqcd, synth

pytestmark = pytest.mark.gpu

# tiles of 64 sites; with two or three in a batch the launch lies on the other side of a line
SIZES = {512: (16, 16, 16, 16), 648: (18, 16, 12, 24), 768: (16, 16, 16, 24), 1216: (16, 16, 16, 38), 1520: (20, 16, 16, 38), 1792: (16, 16, 16, 56)}


@pytest.mark.parametrize("tiles", list(SIZES))
@pytest.mark.parametrize("prec", ["f16", "bf16"])
@pytest.mark.parametrize("compress", [12, 18])
def test_single_equals_batch(tiles, prec, compress):
    dims = SIZES[tiles]
    assert int(np.prod(dims)) == 128 * tiles
    rng = np.random.default_rng(4)
    pool = synth.random_links((2, 2, 2, 2), 0.5, seed=3)
    ctx = lqcd.Context(0)
    g = ctx.gauge(dims, pool[rng.integers(0, 16, 128 * tiles)], prec, compress)
    psi = [rng.standard_normal((128 * tiles, 4, 3, 2)).view(np.complex128)[..., 0] for _ in range(2)]
    fins = [ctx.field(dims, prec, lqcd.EVEN, p) for p in psi]
    one = ctx.field(dims, prec, lqcd.ODD)
    want = []
    for f in fins:
        lqcd.dslash_eo(g, f, one, 1)
        want.append(one.download())
        assert np.abs(want[-1]).max() > 1
    for n in (2, 3):
        outs = [ctx.field(dims, prec, lqcd.ODD) for _ in range(n)]
        batch = lqcd.DslashBatch([g] * n, [fins[k % 2] for k in range(n)], outs, 1)
        batch.apply()
        for k, o in enumerate(outs):
            assert np.array_equal(o.download(), want[k % 2])
        batch.close()
    ctx.close()


@pytest.mark.parametrize("tiles", list(SIZES))
@pytest.mark.parametrize("prec", ["f64", "bf16"])
def test_twisted_against_untwisted(tiles, prec):
    """T(1, t) (D psi) of the twisted operator's launches at mu = 0+: mu so small that the twist
    rounds to one gives the untwisted operator's bits."""
    dims = SIZES[tiles]
    rng = np.random.default_rng(5)
    pool = synth.random_links((2, 2, 2, 2), 0.5, seed=6)
    ctx = lqcd.Context(0)
    g = ctx.gauge(dims, pool[rng.integers(0, 16, 128 * tiles)], prec, 18)
    psi = rng.standard_normal((128 * tiles, 4, 3, 2)).view(np.complex128)[..., 0]
    fin = ctx.field(dims, prec, lqcd.EVEN, psi)
    a, b = ctx.field(dims, prec, lqcd.EVEN), ctx.field(dims, prec, lqcd.EVEN)
    lqcd.apply_Mhat(g, 0.13, fin, a)
    lqcd.apply_Mhat(g, 0.13, fin, b, mu=1e-200)
    want = a.download()
    assert np.array_equal(b.download(), want) and np.abs(want).max() > 1
    ctx.close()
