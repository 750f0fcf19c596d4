"""Layout kernels at the edges of their tiles: half-lattices below, at and beyond one tile of
32 half-sites and with a ragged last tile, every precision and subset, host and device
arrays, and values at the ends of the conversions' ranges.

Every result here is determined exactly: a copy moves reals, and a conversion rounds once
(FP64 -> FP32 / FP16 / BF16 to nearest, double-float as hi + lo with hi the FP32 value and
lo the FP32 value of the rest), so the comparisons are for equality."""
import numpy as np
import pytest

from paper_1112_5280_gb300 import lqcd, synth

pytestmark = pytest.mark.gpu

DIMS = [(2, 2, 2, 2), (4, 2, 2, 4), (4, 4, 2, 2), (6, 2, 4, 6), (10, 6, 2, 4)]  # V/2 = 8, 32, 32, 144, 240


@pytest.fixture(scope="module")
def ctx():
    c = lqcd.Context(0)
    yield c
    c.close()


def _rounded(x, prec):
    """The FP64 values that a field of this precision holds."""
    v = np.ascontiguousarray(x).view(np.float64)
    with np.errstate(over="ignore"):
        if prec == "f32":
            v = v.astype(np.float32).astype(np.float64)
        elif prec == "f16":
            v = v.astype(np.float16).astype(np.float64)
        elif prec == "bf16":  # nearest even on the 16 high bits of the FP32 pattern, from FP64
            import torch
            v = torch.from_numpy(v.copy()).to(torch.bfloat16).double().numpy()
        elif prec == "df64":
            hi = v.astype(np.float32)
            lo = (v - hi.astype(np.float64)).astype(np.float32)
            v = hi.astype(np.float64) + lo.astype(np.float64)
    return v.view(np.complex128)


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("prec", ["f64", "df64", "f32", "f16", "bf16"])
def test_spinor_round_trip(ctx, dims, prec):
    import torch

    psi = synth.gaussian_spinor(dims, seed=5).astype(np.complex64).astype(np.complex128)  # one rounding only
    if prec == "f64" or prec == "df64":
        psi = synth.gaussian_spinor(dims, seed=5)
    psi.reshape(-1)[::7] = 0.0
    want = _rounded(psi, prec)
    even = (synth.parity_of_sites(dims) == 0)[:, None, None]
    for subset, mask in ((lqcd.FULL, True), (lqcd.EVEN, even), (lqcd.ODD, ~even)):
        f = ctx.field(dims, prec, subset, data=psi)
        got = f.download(np.full(psi.shape, -7.0 + 0j))
        assert np.array_equal(got, np.where(mask, want, -7.0))
        dev = torch.full(psi.shape, -7.0, dtype=torch.complex128, device="cuda")
        src = torch.from_numpy(psi).cuda()
        torch.cuda.synchronize()
        f.zero()
        f.upload(src)
        f.download(dev)
        ctx.sync()
        assert np.array_equal(dev.cpu().numpy(), np.where(mask, want, -7.0))


@pytest.mark.parametrize("dims", DIMS)
def test_links_and_momenta_round_trip(ctx, dims):
    U = synth.random_links(dims, 0.7, seed=6)
    g = ctx.gauge(dims, U)
    assert np.array_equal(g.download(), U)
    P = synth.gaussian_momenta(dims, 8)
    assert np.array_equal(ctx.mom(dims, P).download(), P)


def test_unaligned_device_source(ctx):
    """A device array that starts on an 8-byte boundary only is accepted, as before."""
    import ctypes
    import torch

    dims = (4, 4, 2, 2)
    psi = synth.gaussian_spinor(dims, seed=5)
    buf = torch.zeros(psi.size * 2 + 1, dtype=torch.float64, device="cuda")
    buf[1:] = torch.from_numpy(psi.view(np.float64).reshape(-1)).cuda()
    out = torch.zeros_like(buf)
    torch.cuda.synchronize()
    f = ctx.field(dims, "f64")
    assert buf.data_ptr() % 16 == 0
    lib = lqcd.load()
    assert lib.lqcd_field_upload_dev(f.h, ctypes.c_void_p(buf.data_ptr() + 8)) == 0
    assert lib.lqcd_field_download_dev(f.h, ctypes.c_void_p(out.data_ptr() + 8)) == 0
    ctx.sync()
    assert torch.equal(out, buf)


@pytest.mark.parametrize("scale", [1.0, 0.37])
def test_conversion_range(ctx, scale):
    """FP64 <-> double-float <-> FP32 over the whole exponent range, ties and zeros included."""
    dims = (6, 2, 4, 6)
    rng = np.random.default_rng(3)
    n = int(np.prod(dims)) * 24
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    m[::5] &= ~np.uint64((1 << 29) - 1)                       # exactly FP32
    m[1::5] = (m[1::5] & ~np.uint64((1 << 29) - 1)) | np.uint64(1 << 28)  # ties of the FP32 rounding
    m[2::25] = 0                                              # powers of two
    e = rng.integers(1023 - 140, 1023 + 126, n).astype(np.uint64)
    v = ((rng.integers(0, 2, n).astype(np.uint64) << np.uint64(63)) | (e << np.uint64(52)) | m).view(np.float64)
    v[:4] = [0.0, -0.0, 1.0, -1.0]
    psi = v.reshape(-1, 12, 2).copy().view(np.complex128).reshape(int(np.prod(dims)), 4, 3)
    f64 = ctx.field(dims, "f64", data=psi)
    for prec in ("df64", "f32"):
        f = ctx.field(dims, prec)
        f.copy_from(f64, scale)
        want = _rounded((psi.view(np.float64) * scale).view(np.complex128), prec)
        assert np.array_equal(f.download().view(np.float64), want.view(np.float64))
        back = ctx.field(dims, "f64")
        back.copy_from(f)
        assert np.array_equal(back.download().view(np.float64), want.view(np.float64))


def test_layout_under_capture():
    """Uploads, conversions and downloads of device arrays in a captured graph, beside the
    operators, a memset and a copy on a side stream, on a borrowed stream: each replay follows
    the source tensor."""
    import torch

    dims = (6, 2, 4, 6)
    st = torch.cuda.Stream()
    ctx = lqcd.Context(0, stream=st)
    g = ctx.gauge(dims, synth.random_links(dims, 0.6, seed=9), "f32")
    src = torch.zeros((int(np.prod(dims)), 4, 3), dtype=torch.complex128, device="cuda")
    out = torch.full_like(src, -7.0)
    stage = torch.zeros_like(src)
    side = torch.cuda.Stream()
    f, a, b = ctx.field(dims, "f64"), ctx.field(dims, "f32"), ctx.field(dims, "f32")

    def chain():
        f.zero()
        side.wait_stream(st)
        with torch.cuda.stream(side):
            src.copy_(stage)
        st.wait_stream(side)
        f.upload(src)
        a.zero()
        a.copy_from(f, 0.5)
        lqcd.apply_M(g, 0.14, a, b)
        b.copy_from(b, 2.0)
        b.download(out)

    torch.cuda.synchronize()
    chain()
    ctx.sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        chain()
    for seed in (3, 4):
        stage.copy_(torch.from_numpy(synth.gaussian_spinor(dims, seed=seed)))
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        got = out.cpu().numpy()
        out.fill_(-7.0)
        torch.cuda.synchronize()
        chain()
        ctx.sync()
        assert np.array_equal(got, out.cpu().numpy()) and np.abs(got).max() > 1
    del graph
    ctx.close()
