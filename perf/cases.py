"""The work that a user of this library has it do, as timed cases.

Every case goes through `dwf.Context`, the public binding of include/dwf.h. Lattices, actions, block
shapes and masses are those of the workloads in `paper_1811_08488_gb300.synthetic` and of the tests;
the ragged ones are generic. What a case's `op` is:

  hop       dwf_dslash_eo: one application of M^4 or its adjoint, the kernel that all others are made of
  mpc       dwf_mpc: D_PC or its adjoint, which a user applies to sources and residuals
  normal    dwf_mdagm: A = D_PC^+ D_PC, once per CG iteration (FP32) and once per reliable update (FP64)
  m5inv     dwf_m5inv on many right-hand sides, as in source preparation
  precond   dwf_block_precond: the multisplitting preconditioner, k inner CG iterations on every block
  deflate   dwf_deflate: the coarse correction V Lambda^-1 V^+ r of low modes kept by the program
  io        dwf_field_import and dwf_field_export: a canonical field into the library and back
  solve     mspcg_solve: plain CG (k = 0) or MSPCG, right-hand side and solution on the device
"""
import math

import torch

from paper_1811_08488_gb300 import dwf

SIZE = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}
HALF = {"fp16": torch.float16, "bf16": torch.bfloat16}


def _case(op, lx, ly, lz, lt, ls, **more):
    c = dict(op=op, lx=lx, ly=ly, lz=lz, lt=lt, ls=ls, nrhs=1, prec="fp32", dagger=0, b=1.5, c=0.5, eps=0.4,
             mf=0.01)
    c.update(more)
    return c


def listed():
    cases = [
        # the smallest call: one hop of the 8^4 Shamir workload, where the launch and the host path count
        _case("hop", 8, 8, 8, 8, 8, name="hop_small", b=1.0, c=0.0, eps=0.3, mf=0.1),
        # the hop whose bandwidth the benchmark reports, on the lattice it reports it for
        _case("hop", 24, 24, 24, 64, 16, name="hop_fp32", eps=0.45, mf=0.003),
        # the adjoint hop on FP16 fields: the storage and the kernel of the preconditioner's inner solves
        _case("hop", 24, 24, 24, 64, 16, name="hop_fp16_adj", prec="fp16", dagger=1, eps=0.45, mf=0.003),
        # extents that no tile divides and an odd Ls, three masses at once
        _case("mpc", 12, 10, 14, 18, 9, name="mpc_ragged", dagger=1, nrhs=3, mf=0.05),
        # the normal operator on the largest workload, its four sources together
        _case("normal", 32, 32, 32, 64, 12, name="normal_large_4rhs", nrhs=4, eps=0.5, mf=0.0008),
        # the operator of the reliable updates and of FP64 solves
        _case("normal", 16, 16, 16, 32, 12, name="normal_fp64", prec="fp64"),
        # source preparation of the 16-mass workload
        _case("m5inv", 16, 16, 16, 32, 12, name="m5inv_16rhs", nrhs=16),
        # the preconditioner alone, FP32 inner storage, the workload's 8^3 x 16 blocks and k = 6
        _case("precond", 16, 16, 16, 32, 12, name="precond", inner="fp32", k=6, bs=8, bt=16),
        # 24 low modes against four residuals, as in the deflated solves
        _case("deflate", 16, 16, 16, 32, 12, name="deflate", nrhs=4, modes=24),
        # a field of the benchmark's lattice into the library and back, double precision on the user's side
        _case("io", 24, 24, 24, 64, 16, name="io"),
        # the two solvers on the 16^3 x 32 x 12 workload; 1e-12 rather than the default 1e-10, so that the
        # solution itself is settled and can be compared
        _case("solve", 16, 16, 16, 32, 12, name="solve_plain", k=0, tol=1e-12),
        _case("solve", 16, 16, 16, 32, 12, name="solve_mspcg", k=6, inner="fp16", bs=8, bt=16, tol=1e-12),
    ]
    return cases


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _dims(rng, lo, hi):
    """Even extents with a volume near one drawn over the logarithm of [lo, hi]."""
    target = _log_uniform(rng, lo, hi)
    while True:
        d = [rng.choice([4, 6, 8, 10, 12, 14, 16, 18, 20, 24, 28, 32]) for _ in range(3)]
        lt = 2 * round(target / (d[0] * d[1] * d[2]) / 2)
        v = d[0] * d[1] * d[2] * lt
        if 4 <= lt <= 64 and lo <= v <= hi:
            return d + [lt]


def draw(rng):
    """One more case: sizes over the logarithm of the range of the listed cases of the same op."""
    op = rng.choice(["hop", "hop", "hop", "mpc", "normal", "normal", "m5inv", "precond", "deflate", "io", "solve"])
    more = dict(eps=rng.choice([0.3, 0.4, 0.45, 0.5]), mf=_log_uniform(rng, 0.001, 0.1))
    if rng.random() < 0.25:
        more.update(b=1.0, c=0.0)  # Shamir
    ls = rng.choice([4, 6, 7, 8, 9, 10, 12, 12, 14, 16, 16, 20, 24])
    if op == "hop":
        more.update(prec=rng.choice(["fp64", "fp32", "fp32", "fp16", "fp16", "bf16"]), dagger=rng.randrange(2),
                    nrhs=rng.choice([1, 1, 1, 2, 3]))
        hi = 24 ** 3 * 64 // (8 if more["prec"] == "fp64" else 1)
        return _case(op, *_dims(rng, 1024, hi), ls, **more)
    if op == "mpc":
        more.update(dagger=rng.randrange(2), nrhs=rng.choice([1, 1, 2, 3, 4]))
        return _case(op, *_dims(rng, 1024, 24 ** 3 * 64), ls, **more)
    if op == "normal":
        more.update(prec=rng.choice(["fp64", "fp32", "fp32"]), nrhs=rng.choice([1, 1, 2, 4]))
        return _case(op, *_dims(rng, 1024, 16 ** 3 * 32 if more["prec"] == "fp64" else 24 ** 3 * 64), ls, **more)
    if op == "m5inv":
        more.update(dagger=rng.randrange(2), prec=rng.choice(["fp64", "fp32", "fp32"]), nrhs=rng.choice([1, 4, 12, 16]))
        return _case(op, *_dims(rng, 1024, 16 ** 3 * 32), ls, **more)
    if op == "deflate":
        more.update(nrhs=rng.choice([1, 2, 3, 4]), modes=rng.choice([5, 8, 16, 24, 32]))
        return _case(op, *_dims(rng, 1024, 16 ** 3 * 32), min(ls, 12), **more)
    if op == "io":
        more.update(prec=rng.choice(["fp64", "fp32", "fp16"]), nrhs=rng.choice([1, 2]))
        return _case(op, *_dims(rng, 1024, 24 ** 3 * 32), ls, **more)
    # blocks that tile the lattice, two or more of them
    bs, bt = rng.choice([(4, 4), (4, 8), (6, 8), (8, 8), (8, 16)])
    n = [rng.choice([1, 2]) for _ in range(3)] + [rng.choice([2, 3])]
    dims = [bs * n[0], bs * n[1], bs * n[2], min(32, bt * n[3] // bt * bt)]
    if dims[3] < 2 * bt:
        dims[3] = 2 * bt
    ls, more["mf"] = rng.choice([6, 8, 12]), _log_uniform(rng, 0.01, 0.1)
    k = rng.choice([3, 6])
    if op == "precond":
        return _case(op, *dims, ls, bs=bs, bt=bt, k=k, inner="fp32", nrhs=rng.choice([1, 2]), **more)
    if rng.random() < 0.5:
        return _case(op, *dims, ls, k=0, tol=1e-12, nrhs=rng.choice([1, 2]), **more)
    return _case(op, *dims, ls, bs=bs, bt=bt, k=k, inner=rng.choice(["fp32", "fp16", "bf16"]), tol=1e-12, **more)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _volume(case):
    return case["lx"] * case["ly"] * case["lz"] * case["lt"]


def _masses(case):
    """One mass per right-hand side, from the case's own up to twice it."""
    n = case["nrhs"]
    return [case["mf"] * 2 ** (r / n) for r in range(n)]


def _links(case, g):
    """SU(3) links exp(i eps H), H Gaussian traceless Hermitian, as U[t][z][y][x][mu][3][3]."""
    n = _volume(case) * 4
    h = torch.randn(8, n, dtype=torch.float64, device="cuda", generator=g) * (0.5 * case["eps"])
    x = torch.empty(n, 3, 3, dtype=torch.complex128, device="cuda")
    s3 = 1 / math.sqrt(3.0)
    x[:, 0, 0] = 1j * (h[2] + s3 * h[7])
    x[:, 1, 1] = 1j * (s3 * h[7] - h[2])
    x[:, 2, 2] = -2j * s3 * h[7]
    for i, j, k in ((0, 1, 0), (0, 2, 3), (1, 2, 5)):
        x[:, i, j] = torch.complex(h[k + 1], h[k])
        x[:, j, i] = torch.complex(-h[k + 1], h[k])
    del h

    def mul(a, b):
        return sum(a[:, :, i, None] * b[:, None, i, :] for i in range(3))

    x *= 1 / 16  # exp(x) by its series at x / 16, squared four times
    u = torch.eye(3, dtype=torch.complex128, device="cuda").repeat(n, 1, 1)
    for m in range(9, 0, -1):
        u = mul(x, u) / m
        u.diagonal(dim1=1, dim2=2).add_(1.0)
    for _ in range(4):
        u = mul(u, u)
    # the rounding errors of the series out of it again: the first two rows orthonormal, the third their product
    a = u[:, 0] / torch.linalg.vector_norm(u[:, 0], dim=1, keepdim=True)
    b = u[:, 1] - (a.conj() * u[:, 1]).sum(1, keepdim=True) * a
    b = b / torch.linalg.vector_norm(b, dim=1, keepdim=True)
    u = torch.stack([a, b, torch.linalg.cross(a, b, dim=1).conj()], 1)
    return u.reshape(case["lt"], case["lz"], case["ly"], case["lx"], 4, 3, 3)


def _source(case, g, dtype=torch.complex64):
    """Gaussian canonical half fields [rhs][s][t][z][y][xh][4][3]."""
    shape = (case["nrhs"], case["ls"], case["lt"], case["lz"], case["ly"], case["lx"] // 2, 4, 3, 2)
    return torch.view_as_complex(torch.randn(shape, dtype=torch.float32, device="cuda", generator=g)).to(dtype)


def _modes(case, g):
    """Orthonormal vectors in the native FP32 order and their eigenvalues."""
    n = _volume(case) // 2 * case["ls"] * 12
    v = torch.view_as_complex(torch.randn(case["modes"], n, 2, dtype=torch.float32, device="cuda", generator=g))
    v = v.to(torch.complex128)
    for _ in range(2):
        v = torch.linalg.solve_triangular(torch.linalg.cholesky(v.conj() @ v.T).conj(), v, upper=False)
    lam = [0.004 * (1 + 0.02 * j) for j in range(case["modes"])]
    return v.to(torch.complex64), lam


def _params(case):
    p = dict(tol=case.get("tol", 1e-10), inner_iters=case["k"])
    if case["k"]:
        p.update(inner=case["inner"], block=(case["bs"], case["bs"], case["bs"], case["bt"]))
    return dwf.default_params(**p)


def prepare(case, seed):
    g = _generator(seed)
    op, prec, nrhs = case["op"], case["prec"], case["nrhs"]
    ctx = dwf.Context((case["lx"], case["ly"], case["lz"], case["lt"]), case["ls"], b=case["b"], c=case["c"])
    st = dict(case=case, op=op, ctx=ctx, mf=_masses(case))
    if op not in ("io", "m5inv", "deflate"):
        ctx.gauge_load(_links(case, g))
    if op == "deflate":
        v, st["lam"] = _modes(case, g)
        st["V"] = torch.zeros(case["modes"], ctx.field_bytes("fp32", 1), dtype=torch.uint8, device="cuda")
        n = v[0].numel() * 8
        st["V"][:, :n] = v.view(torch.uint8).reshape(case["modes"], n)
    src = _source(case, g, torch.complex128 if op in ("io", "solve") else torch.complex64)
    if op in ("io", "solve"):
        st["src"], st["dst"] = src, torch.zeros_like(src)
    if op == "solve":
        st["params"] = _params(case)
    else:
        st["out"] = ctx.new_field(prec, nrhs)
    if op not in ("io", "solve"):
        st["in"] = ctx.new_field(prec, nrhs)
        ctx.field_import(st["in"], prec, src, nrhs)
        if op == "precond":
            st["params"] = _params(case)
    if op == "hop":
        st["parity"] = int(seed) % 2
    torch.cuda.synchronize()
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _views(case, buf):
    """The native fields of `buf` (see include/dwf.h) as tensors of their own type, one per right-hand side."""
    n = _volume(case) // 2 * case["ls"]
    out = []
    for f in buf.reshape(case["nrhs"], -1):
        prec = case["prec"]
        if prec in HALF:
            data = n * 48
            at = -(-data // 256) * 256
            out.append([f[:data].view(HALF[prec]), f[at:at + 4 * n].view(torch.float32)])
        else:
            out.append(f[:n * 24 * SIZE[prec]].view(torch.float32 if prec == "fp32" else torch.float64))
    return out


def run(st):
    case, ctx, op = st["case"], st["ctx"], st["op"]
    prec, dag, mf = case["prec"], case["dagger"], st["mf"]
    if op == "hop":
        ctx.dslash_eo(st["out"], st["in"], st["parity"], dag, prec, mf)
    elif op == "mpc":
        ctx.mpc(st["out"], st["in"], dag, prec, mf)
    elif op == "normal":
        ctx.mdagm(st["out"], st["in"], prec, mf)
    elif op == "m5inv":
        ctx.m5inv(st["out"], st["in"], dag, prec, mf)
    elif op == "precond":
        ctx.block_precond(st["out"], st["in"], st["params"], mf)
    elif op == "deflate":
        ctx.deflate(st["out"], st["in"], st["V"], st["lam"], "fp32", case["nrhs"])
    elif op == "io":
        ctx.field_import(st["out"], prec, st["src"], case["nrhs"])
        ctx.field_export(st["dst"], st["out"], prec, case["nrhs"])
        return [_views(case, st["out"]), st["dst"]]
    else:
        ctx.solve(st["dst"], st["src"], mf, st["params"])
        return st["dst"]
    return _views(case, st["out"])


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    op, n, prec = case["op"], _volume(case) // 2 * case["ls"], case["prec"]
    vec = n * (24 * SIZE[prec] + (4 if prec in HALF else 0)) * case["nrhs"]
    link = _volume(case) * 4 * 18 * SIZE[prec]
    hop = n * case["nrhs"] * 1320  # Wilson hop: 8 directions on half spinors
    ls_op = n * case["nrhs"] * 24 * 6
    if op == "hop":
        return {"bytes": 2 * vec + link, "flops": hop + ls_op / 2}
    if op == "mpc":  # the even field in and out, both parities' links once
        return {"bytes": 2 * vec + link, "flops": 2 * hop + 3 * ls_op}
    if op == "normal":
        return {"bytes": 2 * vec + link, "flops": 4 * hop + 6 * ls_op}
    if op == "m5inv":
        return {"bytes": 2 * vec, "flops": ls_op}
    if op == "deflate":
        return {"bytes": case["modes"] * n * 96 + 2 * vec, "flops": 2 * case["modes"] * case["nrhs"] * n * 12 * 8}
    if op == "io":
        return {"bytes": 4 * case["nrhs"] * n * 24 * 8 // 2 + 2 * vec, "flops": 0}
    # one application of the operator, the vectors of an iteration read and written once each
    a = {"bytes": 10 * vec + link, "flops": 4 * hop + 6 * ls_op + 12 * n * case["nrhs"] * 24}
    if op == "precond":
        return {k: case["k"] * v for k, v in a.items()}
    iters = 400 if not case["k"] else 140 * (1 + case["k"])  # about what 1e-12 takes
    return {k: iters * v for k, v in a.items()}


# ---------------------------------------------------------------------------
# the same in plain torch, 64 bits: fields as [spin 4][colour 3][s][site of one parity]
# ---------------------------------------------------------------------------
class _Plain:
    def __init__(self, case, links):
        L = [case["lx"], case["ly"], case["lz"], case["lt"]]
        self.case, self.vh = case, _volume(case) // 2
        self.alpha, self.beta = case["b"] * (4 - 1.8) + 1, case["c"] * (4 - 1.8) - 1
        if links is None:
            return
        i = torch.arange(2 * self.vh, device="cuda")
        x, y, z, t = i % L[0], i // L[0] % L[1], i // (L[0] * L[1]) % L[2], i // (L[0] * L[1] * L[2])
        par = (x + y + z + t) % 2
        of = [i[par == 0], i[par == 1]]  # ascending: the half index is the place
        links = links.reshape(-1, 4, 3, 3).clone()
        links[t == L[3] - 1, 3] *= -1  # antiperiodic in t
        self.u, self.nb, self.at = [], [], [[c[o] for c in (x, y, z, t)] for o in of]
        for p in (0, 1):
            nb = []
            for mu in range(4):
                for step in (1, -1):
                    c = [v.clone() for v in self.at[p]]
                    c[mu] = (c[mu] + step) % L[mu]
                    nb.append((((c[3] * L[2] + c[2]) * L[1] + c[1]) * L[0] + c[0]) // 2)
            self.nb.append(nb)
            self.u.append(links[of[p]].permute(1, 2, 3, 0).contiguous())  # [mu][a][b][site]

    @staticmethod
    def _a(mu, v):
        """(A v) of two spins, the upper right block of gamma_mu."""
        return [(-1j * v[1], -1j * v[0]), (-v[1], v[0]), (-1j * v[0], 1j * v[1]), (v[0], v[1])][mu]

    @staticmethod
    def _ad(mu, v):
        return [(1j * v[1], 1j * v[0]), (v[1], -v[0]), (1j * v[0], -1j * v[1]), (v[0], v[1])][mu]

    def hop(self, psi, out_par, dag):
        out = torch.zeros_like(psi)
        for mu in range(4):
            for fwd in (True, False):
                nb = self.nb[out_par][2 * mu + (not fwd)]
                sg = 1 if fwd != bool(dag) else -1
                v = psi[..., nb]
                a = self._a(mu, v[2:])
                h = torch.stack([v[0] - sg * a[0], v[1] - sg * a[1]])
                if fwd:
                    u = self.u[out_par][mu]
                else:
                    u = self.u[1 - out_par][mu][..., nb].conj().transpose(0, 1)
                w = torch.stack([sum(u[r, c] * h[:, c] for c in range(3)) for r in range(3)], 1)
                out[:2] += w
                b = self._ad(mu, w)
                out[2] -= sg * b[0]
                out[3] -= sg * b[1]
        return out

    def ls_matrix(self, p0, p1, mf, inv=False):
        """p0 + p1 C on the upper spins; the lower ones have its transpose."""
        n = self.case["ls"]
        m = p0 * torch.eye(n, dtype=torch.float64)
        for s in range(n):
            m[s, (s - 1) % n] += p1 * (1.0 if s else -mf)
        return (torch.linalg.inv(m) if inv else m).cuda().to(torch.complex128)

    def ls(self, m, psi, dag):
        up, lo = (m.T, m) if dag else (m, m.T)
        return torch.cat([torch.einsum("st,kcth->kcsh", w, v) for w, v in ((up, psi[:2]), (lo, psi[2:]))])

    def m5(self, psi, mf, dag):
        return self.ls(self.ls_matrix(self.alpha, self.beta, mf), psi, dag)

    def m5inv(self, psi, mf, dag):
        return self.ls(self.ls_matrix(self.alpha, self.beta, mf, True), psi, dag)

    def m4(self, psi, out_par, mf, dag):
        phi = self.ls_matrix(self.case["b"], self.case["c"], mf)
        if dag:
            return -0.5 * self.ls(phi, self.hop(psi, out_par, 1), 1)
        return -0.5 * self.hop(self.ls(phi, psi, 0), out_par, 0)

    def mpc(self, psi, mf, dag):
        # the adjoint's factors in reverse order: (M^4_eo M_5^-1 M^4_oe)^+ has the adjoint hop eo <- oe as well
        return self.m5(psi, mf, dag) - self.m4(self.m5inv(self.m4(psi, 1, mf, dag), mf, dag), 0, mf, dag)

    def normal(self, psi, mf):
        return self.mpc(self.mpc(psi, mf, 0), mf, 1)

    def precond(self, r, mf):
        """k CG iterations on the normal operator restricted to each block, from zero."""
        c, z = self.case, torch.zeros_like(r)
        b = [c["bs"], c["bs"], c["bs"], c["bt"]]
        n = [c[d] // v for d, v in zip(("lx", "ly", "lz", "lt"), b)]
        which = sum((x // v) * math.prod(n[:m]) for m, (x, v) in enumerate(zip(self.at[0], b)))
        dot = lambda u, v: (u.conj() * v).sum().real  # noqa: E731
        for blk in range(math.prod(n)):
            mask = which == blk
            res = r * mask
            p, rr = res, dot(res, res)
            for _ in range(c["k"]):
                ap = self.normal(p, mf) * mask
                al = rr / dot(p, ap)
                z += al * p
                res = res - al * ap
                new = dot(res, res)
                p, rr = res + (new / rr) * p, new
        return z

    def to(self, canon):
        return canon.reshape(self.case["ls"], self.vh, 4, 3).permute(2, 3, 0, 1).to(torch.complex128).contiguous()

    def native(self, psi):
        """As `_views` has it."""
        prec = self.case["prec"]
        v = torch.view_as_real(psi.permute(3, 2, 0, 1).contiguous()).reshape(self.vh, self.case["ls"], 24)
        per = 16 // SIZE[prec]
        scale = v.abs().amax(-1) if prec in HALF else None
        if scale is not None:
            v = v / scale[..., None]
        data = v.reshape(self.vh, self.case["ls"], 24 // per, per).permute(2, 0, 1, 3).reshape(-1)
        return data if scale is None else [data, scale.reshape(-1)]


def exact(case, seed):
    op = case["op"]
    if op == "solve":
        return None
    if op == "precond" and _volume(case) * case["ls"] * case["k"] * case["nrhs"] * \
            (_volume(case) // (case["bs"] ** 3 * case["bt"])) > 2 ** 28:
        return None
    g = _generator(seed)
    links = None if op in ("io", "m5inv", "deflate") else _links(case, g)
    if op == "deflate":
        v, lam = _modes(case, g)
        lam = torch.tensor(lam, dtype=torch.float64, device="cuda")
    src = _source(case, g)
    p = _Plain(case, links)
    out = []
    for r, mf in enumerate(_masses(case)):
        psi = p.to(src[r])
        if op == "hop":
            psi = p.m4(psi, int(seed) % 2, mf, case["dagger"])
        elif op == "mpc":
            psi = p.mpc(psi, mf, case["dagger"])
        elif op == "normal":
            psi = p.normal(psi, mf)
        elif op == "m5inv":
            psi = p.m5inv(psi, mf, case["dagger"])
        elif op == "precond":
            psi = p.precond(psi, mf)
        elif op == "deflate":
            x = torch.view_as_complex(p.native(psi).reshape(-1, 2))
            y = torch.zeros_like(x)
            for j in range(case["modes"]):
                w = v[j].to(torch.complex128)
                y += w * ((w.conj() * x).sum() / lam[j])
            out.append(torch.view_as_real(y).reshape(-1))
            continue
        out.append(p.native(psi))
    return [out, src.to(torch.complex128)] if op == "io" else out
