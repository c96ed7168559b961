"""M_5 and M_5^-1 on FP32 fields where the lanes of a warp hold whole sites: the
smallest and largest Ls, warps with idle lanes, a last CTA that is partly filled,
in place, and fields off a 32-byte boundary. FP32 against the FP64 oracle, 1e-5 (about
100 roundings along the longest chain); in place and off the boundary against the
plain call: 1e-6 (the same operations up to their order)."""
import numpy as np
import pytest

from oracle import dwf_operator as op
from test_gpu_operator import Setup, relerr

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Ls", [2, 6, 14, 32])
@pytest.mark.parametrize("dagger", [0, 1])
@pytest.mark.parametrize("kw", [dict(), dict(b=1.0, c=0.0)])
def test_m5_m5inv(Ls, dagger, kw):
    S = Setup((2, 6, 2, 10), Ls, seed=3, **kw)
    masses = [0.02, 0.7, 0.1]
    ins = [S.source(41 + r) for r in range(3)]
    nat = S.to_native(ins, "fp32")
    for fn, ref in ((S.ctx.m5, op.m5), (S.ctx.m5inv, op.m5inv)):
        out = S.ctx.new_field("fp32", 3)
        fn(out, nat, dagger, "fp32", masses)
        got = S.from_native(out, "fp32", 3)
        for r in range(3):
            want = op.full_to_half(ref(S.act, op.half_to_full(ins[r], 0), masses[r], bool(dagger)), 0)
            assert relerr(got[r], want) < 1e-5
        same = nat.clone()
        fn(same, same, dagger, "fp32", masses)
        assert torch.equal(same, out)
        n = S.ctx.field_bytes("fp32", 3)
        buf = torch.zeros(n + 16, dtype=torch.uint8, device="cuda")
        buf[16:] = nat
        off = torch.zeros_like(buf)
        fn(off[16:], buf[16:], dagger, "fp32", masses)
        a, b = off[16:].view(torch.float32), out.view(torch.float32)
        assert (a - b).abs().max() <= 1e-6 * b.abs().max()
