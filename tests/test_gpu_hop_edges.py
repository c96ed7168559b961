"""The two-slice hop at the edges of its tiles: last CTAs that are partly filled,
the smallest and largest Ls, lanes of a warp without a site, sites of a block with
some of their neighbours, and values that must stay with their own site.

Tolerances as in test_gpu_operator.py: FP32 1e-5 (a few hundred FP32 roundings),
FP16 3e-3 and BF16 2.5e-2 (three roundings to storage), block operator in FP32
storage 1e-5 of every element's own maximum."""
import numpy as np
import pytest

from oracle import dwf_operator as op
from oracle import solvers as sv
from test_gpu_operator import Setup, dwf, elem_relerr, relerr

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-5, "fp16": 3e-3, "bf16": 2.5e-2}


# Vh = 96 and 60 sites; sites per CTA 128, 64, 40, 16, 4 (Ls = 2, 4, 6, 16, 32), so the last CTA is
# partly filled; Ls = 6, 12 and 14 leave lanes of every warp without a site
@pytest.mark.parametrize("Ls", [2, 4, 6, 12, 14, 16, 32])
@pytest.mark.parametrize("recon12", [False, True])
def test_mpc_fp32(Ls, recon12):
    S = Setup((4, 2, 6, 4) if Ls < 14 else (2, 6, 2, 10), Ls, seed=7, recon12=recon12)
    masses = [0.02, 0.4]
    ins = [S.source(91), S.source(92)]
    nat = S.to_native(ins, "fp32")
    for dagger in (0, 1):
        out = S.ctx.new_field("fp32", 2)
        S.ctx.mpc(out, nat, dagger, "fp32", masses)
        got = S.from_native(out, "fp32", 2)
        for r in range(2):
            want = op.full_to_half(op.mpc(S.act, S.U, op.half_to_full(ins[r], 0), masses[r],
                                          bool(dagger)), 0)
            assert relerr(got[r], want) < TOL["fp32"], (dagger, r)


@pytest.mark.parametrize("prec", ["fp16", "bf16"])
@pytest.mark.parametrize("Ls", [2, 6, 14, 32])
def test_dslash_half_storage(prec, Ls):
    S = Setup((2, 6, 2, 10), Ls, seed=8)
    src = S.source(93)
    nat = S.to_native([src], prec)
    for dagger in (0, 1):
        out = S.ctx.new_field(prec)
        S.ctx.dslash_eo(out, nat, 1, dagger, prec, [0.1])
        got = S.from_native(out, prec, 1)[0]
        want = op.full_to_half(op.m4(S.act, S.U, op.half_to_full(src, 0), 0.1, bool(dagger)), 1)
        assert relerr(got, want) < TOL[prec], dagger


# blocks whose own sites all run every direction (8 x 8 x 8 x 4 of a lattice as
# wide, one block a direction periodic), blocks where only some rings do, and
# 2^4 blocks, where none does
@pytest.mark.parametrize("dims,block", [((8, 8, 8, 8), (8, 8, 8, 4)), ((8, 8, 4, 8), (8, 4, 4, 4)),
                                        ((4, 4, 4, 4), (2, 2, 2, 2))])
@pytest.mark.parametrize("snake", [1, 0])
def test_block_apply_fp32(dims, block, snake):
    S = Setup(dims, 6, seed=9)
    src = S.source(94)
    prm = dwf().default_params(block=block, inner="fp32", snake=snake)
    out = S.ctx.new_field("fp32")
    S.ctx.block_apply(out, S.to_native([src], "fp32"), prm, [0.05])
    got = S.from_native(out, "fp32", 1)[0]
    x = op.half_to_full(src, 0)
    want = np.zeros_like(x)
    for o in sv.block_origins(dims, block):
        m = sv.block_mask(S.act, block, o)
        f = sv.a_block if snake else sv.a_block_truncated
        want += f(S.act, S.U, sv.project(x, m), 0.05, m)
    assert elem_relerr(got, op.full_to_half(want, 0)) < 1e-5


@pytest.mark.parametrize("dagger", [0, 1])
def test_nan_stays_with_the_sites_that_use_it(dagger):
    """A NaN in one input element reaches the output sites within two hops of it and
    no other (sites share warps, and their lanes exchange values)."""
    S = Setup((8, 4, 4, 8), 6, seed=10)
    src = S.source(95)
    src[3, 4, 1, 2, 1, 2, 0] = np.nan
    out = S.ctx.new_field("fp32")
    S.ctx.mpc(out, S.to_native([src], "fp32"), dagger, "fp32", [0.05])
    got = S.from_native(out, "fp32", 1)[0]
    bad = np.isnan(got).any(axis=(0, 5, 6))
    t, z, y, xh = np.meshgrid(*(np.arange(n) for n in (8, 4, 4, 4)), indexing="ij")
    x = 2 * xh + (y + z + t) % 2
    def dist(a, b, n):
        d = np.abs(a - b) % n
        return np.minimum(d, n - d)
    far = (dist(t, 4, 8) + dist(z, 1, 4) + dist(y, 2, 4) + dist(x, 2 + (4 + 1 + 2) % 2, 8)) > 2
    assert not bad[far].any()
    assert bad.any()


@pytest.mark.parametrize("inner", ["fp32", "fp16"])
@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("inner_tol", [0.0, 1e-6])
def test_block_solve_starts_from_zero(inner, k, inner_tol):
    """The blocks are solved apart: with the residual of one block set to zero its
    solution is zero, whatever an earlier call left in the plan, and the others'
    is bit for bit what it was."""
    S = Setup((8, 4, 4, 8), 6, seed=11)
    src = S.source(96)
    prm = dwf().default_params(block=(4, 4, 4, 4), inner=inner, inner_iters=k, inner_tol=inner_tol)
    z = S.ctx.new_field("fp32")
    S.ctx.block_precond(z, S.to_native([src], "fp32"), prm, [0.05])
    full = S.from_native(z, "fp32", 1)[0]
    cut = src.copy()
    cut[:, 4:, :, :, 2:] = 0  # x >= 4, t >= 4: the last of the four blocks
    S.ctx.block_precond(z, S.to_native([cut], "fp32"), prm, [0.05])
    got = S.from_native(z, "fp32", 1)[0]
    assert (got[:, 4:, :, :, 2:] == 0).all() and (full != 0).any()
    got[:, 4:, :, :, 2:] = full[:, 4:, :, :, 2:]
    assert np.array_equal(got, full)
