"""M_5^-1 on FP32 fields by the lanes of a site is as close to the 64-bit result as by
columns in shared memory, which fields off a 32-byte boundary take. Both round every
element three times (the recursion, p0 y, the sum) and carry the same coefficients, so
their mean square errors are estimates of the same quantity over 5e5 elements or more: 3 %
apart is allowed, ten times the spread of such an estimate."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Ls", [6, 12, 16, 32])
@pytest.mark.parametrize("b,c", [(1.5, 0.5), (1.0, 0.0)])
@pytest.mark.parametrize("dagger", [0, 1])
def test_m5inv_error(Ls, b, c, dagger):
    from paper_1811_08488_gb300 import dwf
    ctx = dwf.Context((8, 8, 8, 16), Ls, b=b, c=c)
    g = torch.Generator(device="cuda").manual_seed(7)
    src = torch.view_as_complex(torch.randn(ctx.canon_shape(1) + (2,), dtype=torch.float32, device="cuda",
                                            generator=g)).to(torch.complex128)

    def apply(prec, off=0):
        n = ctx.field_bytes(prec)
        bufs = [torch.zeros(n + off, dtype=torch.uint8, device="cuda")[off:] for _ in range(2)]
        ctx.field_import(bufs[0], prec, src)
        ctx.m5inv(bufs[1], bufs[0], dagger, prec, [0.03])
        out = torch.zeros_like(src)
        ctx.field_export(out, bufs[1], prec)
        return out

    want = apply("fp64")
    lanes, columns = (float((apply("fp32", off) - want).abs().square().sum().sqrt()) for off in (0, 16))
    assert lanes <= 1.03 * columns
