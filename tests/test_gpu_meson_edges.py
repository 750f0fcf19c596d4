"""The meson kernel at the edges of its split: a slice's half-sites below, at and beyond one
CTA's 128 threads, one and two sites per thread, and requests that need only some of the
spin sums. The fields are noise (the contraction does not ask for solutions); the reference
is the oracle's contraction of the same fields.

Bar: every C(t) is a sum of FP64 products, so its error is rounding of the largest |C|
(which bounds the sums of magnitudes to within the spin count); 1e-12 of it, as for the
solved propagators."""
import numpy as np
import pytest

from oracle import contract
from paper_1112_5280_gb300 import lqcd, synth

pytestmark = pytest.mark.gpu


# half-sites of a slice: 4, 128 (one CTA), 200, 864 (two sites per thread, last CTA ragged)
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (8, 8, 4, 6), (10, 4, 10, 4), (12, 12, 12, 24)])
@pytest.mark.parametrize("codes", [[1], [2, 5], [9, 0, 4], list(range(10))])
def test_meson_split_edges(dims, codes):
    ctx = lqcd.Context(0)
    host = [synth.gaussian_spinor(dims, seed=300 + k) for k in range(12)]
    props = [ctx.field(dims, "f64", lqcd.FULL, data=p) for p in host]
    got = lqcd.meson_correlator(props, codes)
    ref = contract.meson_correlator(dims, host, codes)
    scale = np.abs(contract.meson_correlator(dims, host, [1])).max()  # C_g5: the largest
    assert got.shape == (len(codes), dims[3])
    assert np.abs(got - ref).max() < 1e-12 * scale
    ctx.close()
