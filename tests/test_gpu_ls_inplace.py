"""M_5 and M_5^-1 in place (out == in) give the bits that they give out of place, on
lattices of many CTAs: whole warps (Ls = 16), warps with lanes that hold no site
(Ls = 6, 12, 14) and a last CTA that is partly filled, the shared-memory kernel (FP64, odd Ls).
No site is read by a warp that does not own it, so there is nothing to tolerate."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Ls,prec", [(6, "fp32"), (12, "fp32"), (14, "fp32"), (16, "fp32"), (7, "fp32"),
                                     (12, "fp64")])
def test_in_place(Ls, prec):
    from paper_1811_08488_gb300 import dwf
    ctx = dwf.Context((14, 10, 12, 18), Ls, b=1.5, c=0.5)
    masses = [0.02, 0.7, 0.1]
    shape = ctx.canon_shape(3) + (2,)
    g = torch.Generator(device="cuda").manual_seed(5)
    src = torch.view_as_complex(torch.randn(shape, dtype=torch.float64, device="cuda", generator=g))
    nat, out = ctx.new_field(prec, 3), ctx.new_field(prec, 3)
    ctx.field_import(nat, prec, src, 3)
    for fn in (ctx.m5, ctx.m5inv):
        for dagger in (0, 1):
            fn(out, nat, dagger, prec, masses)
            for _ in range(3):
                same = nat.clone()
                fn(same, same, dagger, prec, masses)
                assert torch.equal(same, out), dagger
