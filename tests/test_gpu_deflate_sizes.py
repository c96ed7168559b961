"""The coarse correction V Lambda^-1 V^+ r at the edges of the multi-dot's tiles: 1 to 40
modes (tiles of 8, 16, 24 and 32, the last one partly filled, two tiles), 1 to 4
right-hand sides, vectors shorter than one CTA's segments and longer than all of them.

The dot products are FP32 with compensated sums: an error of 3 2^-24 sum |v_k| |r_k| at
most, 1.8e-7 (2 / pi) N against the |v| |r| / sqrt(N) = sqrt(N) of random vectors, so up to 1.2e-7
sqrt(N) of the result, N = 6144 to 516096 reals; signs differ, and 1e-5 is allowed."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,Ls", [((4, 4, 4, 4), 2), ((6, 4, 14, 16), 8)])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 4])
def test_deflate(dims, Ls, nrhs):
    from paper_1811_08488_gb300 import dwf
    ctx = dwf.Context(dims, Ls, b=1.5, c=0.5)
    n = ctx.Vh * Ls * 24
    g = torch.Generator(device="cuda").manual_seed(9)
    nbytes = ctx.field_bytes("fp32", 1)

    def fields(count):
        f = torch.zeros(count, nbytes, dtype=torch.uint8, device="cuda")
        v = torch.randn(count, n, device="cuda", generator=g)
        f[:, :4 * n] = v.view(torch.uint8)
        return f, torch.view_as_complex(v.double().reshape(count, n // 2, 2))

    r, rc = fields(nrhs)
    for m in (1, 3, 8, 9, 16, 17, 24, 25, 32, 40):
        V, vc = fields(m)
        lam = [0.5 + 0.1 * j for j in range(m)]
        z = torch.zeros_like(r)
        ctx.deflate(z, r.reshape(-1), V.reshape(-1), lam, "fp32", nrhs)
        want = ((rc @ vc.conj().T) / torch.tensor(lam, dtype=torch.float64, device="cuda")) @ vc
        got = torch.view_as_complex(z[:, :4 * n].reshape(nrhs, 4 * n).contiguous().view(torch.float32)
                                    .double().reshape(nrhs, n // 2, 2))
        assert (torch.linalg.vector_norm(got - want) / torch.linalg.vector_norm(want)) < 1e-5, m
