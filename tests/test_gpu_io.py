"""Import and export at the edges of their tiles (lattices that no tile divides,
smallest and largest Ls) and from canonical fields that start off a 16-byte boundary.
FP64 and FP32 storage of values that fit are exact; FP16 rounds to 2^-11 of the
(site, s) maximum (complex: sqrt(2) times that)."""
import numpy as np
import pytest

from paper_1811_08488_gb300 import synthetic as syn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,Ls", [((2, 2, 2, 2), 2), ((6, 2, 2, 10), 7), ((4, 6, 2, 8), 16),
                                     ((2, 6, 2, 6), 32)])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("canon,off", [("complex128", 0), ("complex64", 0), ("complex64", 1)])
def test_import_export(dims, Ls, prec, canon, off):
    from paper_1811_08488_gb300 import dwf
    ctx = dwf.Context(dims, Ls)
    h = np.stack([syn.half_field(dims, Ls, 31 + r) for r in range(2)]).astype(np.complex64)
    dt = getattr(torch, canon)
    src = torch.zeros(h.size + off, dtype=dt, device="cuda")
    src[off:] = torch.from_numpy(h.reshape(-1)).cuda().to(dt)
    dst = torch.zeros_like(src)
    nat = ctx.new_field(prec, 2)
    ctx.field_import(nat, prec, src[off:], 2)
    ctx.field_export(dst[off:], nat, prec, 2)
    got = dst[off:].cpu().numpy().reshape(h.shape)
    assert (dst[:off] == 0).all()
    if prec != "fp16":
        assert np.array_equal(got, h.astype(got.dtype))
    else:
        m = np.maximum(np.abs(h.real), np.abs(h.imag)).max(axis=(-2, -1), keepdims=True)
        assert (np.abs(got - h) <= 2.0 ** -11 * np.sqrt(2) * 1.01 * m).all()
    # the native layout: chunk k of (h, s) at ((k V + h) Ls + s) 16 bytes
    if prec == "fp32":
        n = ctx.Vh * Ls * 24
        v = nat[: n * 4].view(torch.float32).cpu().numpy().reshape(6, ctx.Vh, Ls, 4)
        want = np.stack([h[0].real, h[0].imag], -1).reshape(Ls, ctx.Vh, 6, 4).transpose(2, 1, 0, 3)
        assert np.array_equal(v, want)
