"""The two forms of the two-slice hop against each other: a call with many right-hand
sides fills the waves from which links are staged (hop_staged_sites; checked in
test_hop_staged_sites.py), the same right-hand sides one at a time do not. Last CTAs are
partly filled, Ls = 6, 10, 12 and 14 leave lanes of a warp without a site, the dense CTAs of a
block's hop reach into its ring, and block sites lack neighbours.

Both forms run the same operations on every site, up to the contraction that the
compiler chooses and to zeros that are added: FP32 1e-6 of the largest element (about
ten roundings), block operators in FP32 storage 1e-5 of every element's own maximum (four
hops and M_5), FP16 3e-3 and BF16 2.5e-2 (three roundings to storage), as in
test_gpu_operator.py. Preconditioner applications of two iterations: ten times that."""
import numpy as np
import pytest

from test_gpu_operator import Setup, dwf, elem_relerr, relerr

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-5, "fp16": 3e-3, "bf16": 2.5e-2}


def sources(S, n):
    return [S.source(200 + r) for r in range(n)]


@pytest.mark.parametrize("Ls", [6, 8, 10, 14])
@pytest.mark.parametrize("recon12", [False, True])
def test_whole_lattice_fp32(Ls, recon12):
    S = Setup((6, 6, 14, 14), Ls, seed=12, recon12=recon12)
    n = 16
    masses = [0.02 * (1 + r) for r in range(n)]
    ins = sources(S, n)
    nat, out, one = S.to_native(ins, "fp32"), S.ctx.new_field("fp32", n), S.ctx.new_field("fp32")
    single = [S.to_native([v], "fp32") for v in ins]
    calls = [lambda o, i, m: S.ctx.dslash_eo(o, i, 1, 0, "fp32", m),
             lambda o, i, m: S.ctx.dslash_eo(o, i, 0, 1, "fp32", m),
             lambda o, i, m: S.ctx.mdagm(o, i, "fp32", m),
             lambda o, i, m: S.ctx.mdagm_sym(o, i, "fp32", m)]
    for call in calls:
        call(out, nat, masses)
        got = S.from_native(out, "fp32", n)
        for r in range(n):
            call(one, single[r], masses[r:r + 1])
            assert relerr(got[r], S.from_native(one, "fp32", 1)[0]) < 1e-6, r


@pytest.mark.parametrize("Ls", [6, 10, 14])
def test_nan_stays_with_the_sites_that_use_it(Ls):
    dims, n = (6, 6, 14, 14), 16
    S = Setup(dims, Ls, seed=13)
    ins = sources(S, n)
    # the last site of all: lanes without a site read what it reads
    ins[3][2, -1, -1, -1, -1, 1, 0] = np.nan
    out = S.ctx.new_field("fp32", n)
    for dagger in (0, 1):
        S.ctx.dslash_eo(out, S.to_native(ins, "fp32"), 1, dagger, "fp32", [0.05] * n)
        got = S.from_native(out, "fp32", n)
        assert not any(np.isnan(got[r]).any() for r in range(n) if r != 3)
        bad = np.isnan(got[3]).any(axis=(0, 5, 6))
        t, z, y, xh = np.meshgrid(*(np.arange(k) for k in (dims[3], dims[2], dims[1], dims[0] // 2)),
                                  indexing="ij")
        x = 2 * xh + (1 + y + z + t) % 2
        src = [dims[3] - 1, dims[2] - 1, dims[1] - 1]
        src.append(dims[0] - 2 + sum(src) % 2)
        dist = sum(np.minimum(np.abs(a - b), k - np.abs(a - b))
                   for a, b, k in zip((t, z, y, x), src, dims[::-1]))
        assert (bad == (dist == 1)).all()


# FP16/BF16: hop 1 of the many runs its own sites with staged links, then the ring; FP32: hop 2
# (block sites and first ring, then the second ring), and hops 3 and 4 as a whole
CASES = [("fp16", (8, 8, 8, 16), 12, 9), ("bf16", (8, 8, 8, 16), 12, 9), ("fp16", (8, 8, 16, 16), 6, 9),
         ("fp32", (8, 8, 16, 16), 12, 12), ("fp32", (8, 8, 8, 16), 32, 10), ("fp32", (8, 8, 8, 16), 6, 12)]


@pytest.mark.parametrize("inner,dims,Ls,n", CASES)
@pytest.mark.parametrize("kw,recon12", [(dict(), False), (dict(schur=1), True), (dict(snake=0), False),
                                        (dict(inner_tol=0.3), False)])
def test_blocks(inner, dims, Ls, n, kw, recon12):
    S = Setup(dims, Ls, seed=14, recon12=recon12)
    masses = [0.05 * (1 + r) for r in range(n)]
    ins = sources(S, n)
    nat, single = S.to_native(ins, "fp32"), [S.to_native([v], "fp32") for v in ins]
    prm = dwf().default_params(block=(4, 4, 4, 4), inner=inner, inner_iters=2, **kw)
    out, one = S.ctx.new_field("fp32", n), S.ctx.new_field("fp32")
    for call, tol in ((S.ctx.block_apply, TOL[inner]), (S.ctx.block_precond, 10 * TOL[inner])):
        want = []
        for r in range(n):
            call(one, single[r], prm, masses[r:r + 1])
            want.append(S.from_native(one, "fp32", 1)[0])
        call(out, nat, prm, masses)
        got = S.from_native(out, "fp32", n)
        err = elem_relerr if inner == "fp32" and call == S.ctx.block_apply else relerr
        for r in range(n):
            assert np.isfinite(got[r]).all()
            assert err(got[r], want[r]) < tol, r
        # the plan has its tables by now: one at a time still takes the other form
        call(one, single[0], prm, masses[:1])
        assert np.array_equal(S.from_native(one, "fp32", 1)[0], want[0])
