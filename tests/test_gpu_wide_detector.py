"""A detector far wider than fixed-point positions reach (8 million pixels either
side): the bins around the image give what a narrow detector gives, all others
zero, and the adjoint reads the former alone."""
import pytest

from gpu_util import TOL, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", ["float32", "float64"])
@pytest.mark.parametrize("n1,n2,B,span", [(32, 32, 12_600_001, 2.6), (40, 25, 24_000_000, 1.5)])
def test_centre_bins(n1, n2, B, span, dt):
    torch, api = require_gpu()
    ctx, dtype = api.Context(0), getattr(torch, dt)
    small = 64 + B % 2
    make = lambda bins: api.Operator(ctx, "radon", n1, n2, dtype=dtype, n_angles=2, n_bins=bins, angle_span=span)  # noqa: E731
    wide, narrow = make(B), make(small)
    g = torch.Generator(device="cuda").manual_seed(B)
    x = torch.randn((1, n1, n2), dtype=dtype, device="cuda", generator=g)
    y, ref = api.op_apply(wide, x), api.op_apply(narrow, x)
    lo = (B - small) // 2
    tol = TOL["f32" if dt == "float32" else "f64"] * float(ref.abs().max())
    assert float((y[..., lo:lo + small] - ref).abs().max()) <= tol
    y[..., lo:lo + small] = 0
    assert not y.any()
    s = torch.randn((1, 2, small), dtype=dtype, device="cuda", generator=g)
    y[..., lo:lo + small] = s
    z, zr = api.op_adjoint(wide, y), api.op_adjoint(narrow, s)
    assert float((z - zr).abs().max()) <= TOL["f32" if dt == "float32" else "f64"] * float(zr.abs().max())
    n = api.op_normal(wide, x)
    nr = api.op_normal(narrow, x)
    assert float((n - nr).abs().max()) <= 2 * TOL["f32" if dt == "float32" else "f64"] * float(nr.abs().max())
