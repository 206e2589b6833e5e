"""What a user of this library has it do, as cases that can be timed and checked.

Each case is one call (or one short sequence of calls) through the public
binding, on seeded synthetic inputs made on the GPU: weak-field SU(3) links,
Gaussian vectors, coarse links of the size Galerkin products have.  `exact`
gives the same results in 64 bits from plain torch.
"""
import math

import numpy as np
import torch

import paper_1612_07873_gb300 as gb

PREC = {"f64": gb.F64, "f32": gb.F32, "bf16": gb.BF16, "f16": gb.F16, "i16": gb.I16}
CSW = 1.0
MASS = -0.40  # the production-shaped workload's mass
EPS = 0.5     # its weak-field strength


def _case(kind, dims, **kw):
    return dict(kind=kind, lx=dims[0], ly=dims[1], lz=dims[2], lt=dims[3], **kw)


def listed():
    return [
        # The coarsest level of the 3-level solve (4^3x8, 64 dofs): the coarsest
        # GCR applies it up to a hundred times per cycle; launch and latency count.
        dict(name="coarse_f32_4x4x4x8_n64", **_case("coarse", (4, 4, 4, 8), n=64, prec="f32", rhs=1)),
        # The level-1 operator of the 32^3x64 workload, the headline benchmark.
        dict(name="coarse_f32_8x8x8x16_n48", **_case("coarse", (8, 8, 8, 16), n=48, prec="f32", rhs=1)),
        # The same operator on eight vectors: FP32 multi-RHS solves and the
        # level-1 setup sweeps.
        dict(name="coarse_f32_8x8x8x16_n48_rhs8",
             **_case("coarse", (8, 8, 8, 16), n=48, prec="f32", rhs=8)),
        # BF16 links on 32 vectors: the batched form as a complex GEMM.
        dict(name="coarse_bf16_8x8x8x16_n48_rhs32",
             **_case("coarse", (8, 8, 8, 16), n=48, prec="bf16", rhs=32)),
        # The fine operator on one vector: every smoothing step of a solve.
        dict(name="wilson_f32_32x32x32x64", **_case("wilson", (32, 32, 32, 64), rhs=1)),
        # The fine operator on eight vectors at a mid-size lattice: batched
        # solves and, in the same kernel, the null-vector sweeps.
        dict(name="wilson_f32_24x24x24x48_rhs8", **_case("wilson", (24, 24, 24, 48), rhs=8)),
        # Red-black preconditioning: the fine Schur operator its smoother applies.
        dict(name="schur_f32_24x24x24x48", **_case("schur", (24, 24, 24, 48), rhs=1)),
        # Restriction and prolongation between the fine and the first coarse level.
        dict(name="transfer_f32_24x24x24x48",
             **_case("transfer", (24, 24, 24, 48), block=4, nvec=24, rhs=1)),
        # Null-vector setup of a level: ten sweeps on 24 vectors and the block QR.
        dict(name="setup_f32_16x16x16x32",
             **_case("setup", (16, 16, 16, 32), block=4, nvec=24, sweeps=10)),
        # The Galerkin product P^dag M P of the fine operator, nine blocks per site.
        dict(name="galerkin_f32_24x24x24x48", **_case("galerkin", (24, 24, 24, 48), block=4, nvec=24)),
        # A whole solve to 1e-10 with the production-shaped 3-level FP32 hierarchy.
        dict(name="solve_f32_32x32x32x64",
             **_case("solve", (32, 32, 32, 64), prec="f32", rhs=1, smoother="f32")),
        # A whole batched solve in the fastest form: BF16 coarse links and BF16
        # fine smoother, eight right-hand sides per call.
        dict(name="solve_bf16_16x16x16x32_rhs8",
             **_case("solve", (16, 16, 16, 32), prec="bf16", rhs=8, smoother="bf16")),
    ]


def _spread(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _extents(rng, lo, hi_s, hi_t, step, most):
    """Four extents (multiples of step) with at most `most` sites."""
    while True:
        d = [max(lo, step * round(_spread(rng, lo, h) / step)) for h in (hi_s, hi_s, hi_s, hi_t)]
        if d[0] * d[1] * d[2] * d[3] <= most:
            return tuple(d)


def draw(rng):
    kind = rng.choice(["coarse", "coarse", "coarse", "wilson", "wilson", "schur", "transfer",
                       "setup", "galerkin", "solve"])
    if kind == "coarse":
        dims = _extents(rng, 2, 12, 20, 1, 8192)
        n = rng.choice([16, 32, 48, 48, 64])
        prec = rng.choice(["f32", "f32", "f32", "bf16", "bf16", "f16", "i16"])
        rhs = 1
        if prec == "f32" and rng.random() < 0.6:
            rhs = round(_spread(rng, 2, 32))
        elif prec in ("bf16", "f16") and rng.random() < 0.7:
            rhs = 4 * round(_spread(rng, 1, 16))
        return _case("coarse", dims, n=n, prec=prec, rhs=rhs)
    if kind in ("wilson", "schur"):
        dims = _extents(rng, 4, 32, 64, 2, 32 ** 3 * 64)
        vol = dims[0] * dims[1] * dims[2] * dims[3]
        most = max(1, min(24 if kind == "wilson" else 8, 8 * 32 ** 3 * 32 // vol))
        rhs = 1 if rng.random() < 0.4 else round(_spread(rng, 1, most))
        return _case(kind, dims, rhs=rhs)
    if kind == "solve":
        while True:
            dims = _extents(rng, 8, 32, 64, 8, 32 ** 3 * 32)
            vol = dims[0] * dims[1] * dims[2] * dims[3]
            rhs = rng.choice([1, 1, 1, 2, 4, 6, 8])
            if vol * rhs <= 32 ** 3 * 32:
                break
        prec, smoother = rng.choice([("f32", "f32"), ("bf16", "f32"), ("bf16", "bf16")])
        return _case("solve", dims, prec=prec, rhs=rhs, smoother=smoother)
    block = rng.choice([2, 4, 4])
    dims = _extents(rng, 2 * block, 24, 48, block, 24 ** 3 * 48)
    nvec = rng.choice([8, 16, 24, 24, 32])
    if kind == "transfer":
        return _case(kind, dims, block=block, nvec=nvec, rhs=1)
    if kind == "galerkin":
        return _case(kind, dims, block=block, nvec=nvec)
    while dims[0] * dims[1] * dims[2] * dims[3] > 16 ** 3 * 32:
        dims = _extents(rng, 2 * block, 24, 48, block, 16 ** 3 * 32)
    return _case("setup", dims, block=block, nvec=nvec, sweeps=rng.choice([4, 10]))


# ------------------------------------------------------------------ inputs
def _dims(case):
    return (case["lx"], case["ly"], case["lz"], case["lt"])


def _vol(case):
    return case["lx"] * case["ly"] * case["lz"] * case["lt"]


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _gauss(g, *shape):
    return torch.view_as_complex(
        torch.randn(*shape, 2, generator=g, device="cuda", dtype=torch.float64))


def _mul3(a, b):
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _gauge(g, vol):
    """Weak-field SU(3) links exp(i EPS H), [4][V][3][3]; H a traceless
    Hermitian Gaussian matrix."""
    out = torch.empty(4, vol, 3, 3, dtype=torch.complex128, device="cuda")
    eye = torch.eye(3, dtype=torch.complex128, device="cuda")
    for mu in range(4):
        a = _gauss(g, vol, 3, 3)
        h = 0.5 * (a + a.mH)
        tr = torch.diagonal(h, dim1=-2, dim2=-1).real.sum(-1) / 3
        h = (1j * EPS / 32) * (h - tr[:, None, None] * eye)
        u = eye + h
        term = h
        for k in range(2, 10):
            term = _mul3(term, h) / k
            u = u + term
        for _ in range(5):
            u = _mul3(u, u)
        r0 = u[:, 0] / torch.linalg.vector_norm(u[:, 0], dim=-1, keepdim=True)
        r1 = u[:, 1] - (r0.conj() * u[:, 1]).sum(-1, keepdim=True) * r0
        r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
        out[mu, :, 0], out[mu, :, 1] = r0, r1
        out[mu, :, 2] = torch.linalg.cross(r0, r1).conj()
    return out


def _links(g, vol, n):
    """Coarse links [V][9][n][n] of the size a Galerkin product has: X near a
    multiple of the identity, the hops a fraction of it."""
    k = _gauss(g, vol, 9, n, n) * (0.25 / math.sqrt(n))
    k[:, 0] += 4.0 * torch.eye(n, dtype=torch.complex128, device="cuda")
    return k


def _context(case, dims, gauge, blocks, nvecs, **kw):
    p = gb.default_params(dims=dims, block=blocks, nvec=nvecs, mass=MASS, csw=CSW,
                          nlevels=len(blocks) + 1, prec_fine=gb.F32, **kw)
    return gb.Multigrid(p, gauge)


def prepare(case, seed):
    g = _gen(seed)
    dims, vol, kind = _dims(case), _vol(case), case["kind"]
    if kind == "coarse":
        n, rhs = case["n"], case["rhs"]
        prec = PREC[case["prec"]]
        fine = tuple(2 * d for d in dims)
        mg = _context(case, fine, _gauge(g, 16 * vol), [(2, 2, 2, 2)], [n // 2], prec_coarse=prec)
        gb.mg_set_coarse_links(mg.ctx, 1, _links(g, vol, n))
        shape = (vol, n) + ((rhs,) if rhs > 1 else ())
        x = _gauss(g, *shape).to(torch.complex64)
        return dict(case=case, mg=mg, x=x, y=torch.empty_like(x))
    gauge = _gauge(g, vol)
    if kind in ("wilson", "schur"):
        blk = tuple(2 if d % 2 == 0 else 1 for d in dims)
        mg = _context(case, dims, gauge, [blk], [4], prec_coarse=gb.F32,
                      red_black=int(kind == "schur"))
        x = _gauss(g, case["rhs"], vol if kind == "wilson" else vol // 2, 12).to(torch.complex64)
        return dict(case=case, mg=mg, x=x, y=torch.empty_like(x))
    if kind == "solve":
        mg = _context(case, dims, gauge, [(4, 4, 4, 4), (2, 2, 2, 2)], [24, 32],
                      prec_coarse=PREC[case["prec"]], prec_smoother=PREC[case["smoother"]],
                      seed=int(seed) % (1 << 31))
        for level in (0, 1):
            gb.mg_setup_nullvecs(mg.ctx, level)
            gb.mg_build_coarse(mg.ctx, level)
        b = _gauss(g, case["rhs"], vol, 12)
        return dict(case=case, mg=mg, b=b, x=torch.empty_like(b))
    block, nvec = case["block"], case["nvec"]
    mg = _context(case, dims, gauge, [(block,) * 4], [nvec], prec_coarse=gb.F32,
                  setup_sweeps=case.get("sweeps", 10))
    v = _gauss(g, nvec, vol, 12)
    cvol = vol // block ** 4
    if kind == "setup":
        return dict(case=case, mg=mg, v=v, out=torch.empty_like(v))
    gb.mg_set_nullvecs(mg.ctx, 0, v)
    if kind == "galerkin":
        return dict(case=case, mg=mg, out=torch.empty(cvol, 9, 2 * nvec, 2 * nvec,
                                                      dtype=torch.complex128, device="cuda"))
    del v
    x = _gauss(g, vol, 12).to(torch.complex64)
    return dict(case=case, mg=mg, x=x, y=torch.empty_like(x),
                c=torch.empty(cvol, 2 * nvec, dtype=torch.complex64, device="cuda"))


# --------------------------------------------------------------------- run
def run(s):
    case, ctx = s["case"], s["mg"].ctx
    kind = case["kind"]
    if kind == "coarse":
        gb.mg_coarse_apply(ctx, 1, s["y"], s["x"], case["rhs"])
        return s["y"]
    if kind == "wilson":
        if case["rhs"] == 1:
            gb.mg_wilson_clover_apply(ctx, s["y"], s["x"])
        else:
            gb.mg_wilson_clover_apply_multi(ctx, s["y"], s["x"], case["rhs"])
        return s["y"]
    if kind == "schur":
        gb.mg_schur_apply(ctx, 0, s["y"], s["x"], case["rhs"])
        return s["y"]
    if kind == "transfer":
        gb.mg_restrict(ctx, 0, s["c"], s["x"])
        gb.mg_prolong(ctx, 0, s["y"], s["c"])
        return s["c"], s["y"]
    if kind == "setup":
        # the vectors of an FP32 level, kept in the level's own precision
        gb.mg_setup_nullvecs(ctx, 0, s["v"])
        return gb.mg_get_nullvecs(ctx, 0, s["out"]).to(s["mg"].levels[0]["dtype"])
    if kind == "galerkin":
        gb.mg_build_coarse(ctx, 0)
        return gb.mg_get_coarse_links(ctx, 1, s["out"]).to(s["mg"].levels[1]["dtype"])
    if case["rhs"] == 1:
        gb.mg_gcr_solve(ctx, s["x"], s["b"], tol=1e-10)
    else:
        gb.mg_gcr_solve_multi(ctx, s["x"], s["b"], case["rhs"], tol=1e-10)
    return s["x"]


# -------------------------------------------------------------------- work
def _wilson_work(vol, rhs, links=1.0):
    # spinor in and out per vector; four links and the clover term per site
    return dict(bytes=vol * (192 * rhs + links * 288 + 288), flops=1824 * vol * rhs)


def work(case):
    vol, kind = _vol(case), case["kind"]
    if kind == "coarse":
        n, rhs = case["n"], case["rhs"]
        elem = 8 if case["prec"] == "f32" else 4
        return dict(bytes=vol * (9 * n * n * elem + 16 * n * rhs), flops=72 * n * n * vol * rhs)
    if kind == "wilson":
        return _wilson_work(vol, case["rhs"])
    if kind == "schur":
        # compact vectors in and out, every link, A_o and A_e^-1
        return dict(bytes=vol * (96 * case["rhs"] + 288 + 288),
                    flops=vol * case["rhs"] * (1320 + 504))
    if kind == "transfer":
        nv = case["nvec"]
        return dict(bytes=2 * vol * 12 * (nv * 8 + 8) + 2 * vol // case["block"] ** 4 * 2 * nv * 8,
                    flops=2 * 8 * vol * 12 * nv)
    if kind == "setup":
        nv, sweeps = case["nvec"], case["sweeps"]
        rows = case["block"] ** 4 * 6
        blocks = 2 * vol // case["block"] ** 4
        # start vectors in, orthonormal vectors out; two applies, the inner
        # products and the update per sweep; one Gram-Schmidt pass
        return dict(bytes=vol * (12 * nv * (16 + 16) + 576),
                    flops=vol * nv * sweeps * (2 * 1824 + 12 * 20)
                    + 8 * nv * (nv - 1) * rows * blocks)
    if kind == "galerkin":
        nv, b = case["nvec"], case["block"]
        faces = 1 + 8 / b
        return dict(bytes=vol * (12 * nv * 8 + 576) + vol // b ** 4 * 9 * (2 * nv) ** 2 * 16,
                    flops=vol * (faces * 8 * 2 * nv * nv * 12 + 2 * nv * (270 + 8 * 204)))
    # right-hand sides in, solutions out, the operator and the hierarchy once;
    # the operator applies a 13-step solve of this hierarchy needs on the fine level
    w = _wilson_work(vol, case["rhs"])
    hier = vol * 12 * 24 * 8 + vol // 256 * 9 * 48 * 48 * (8 if case["prec"] == "f32" else 4)
    return dict(bytes=w["bytes"] + hier + vol * case["rhs"] * 12 * 32, flops=w["flops"] * 130)


# ------------------------------------------------------------------- exact
def _gammas():
    """DeGrand-Rossi gamma matrices; gamma_5 = diag(1, 1, -1, -1)."""
    z = np.zeros((4, 4, 4), dtype=np.complex128)
    z[0, 0, 3] = z[0, 1, 2] = 1j
    z[0, 2, 1] = z[0, 3, 0] = -1j
    z[1, 0, 3] = z[1, 3, 0] = -1
    z[1, 1, 2] = z[1, 2, 1] = 1
    z[2, 0, 2] = z[2, 3, 1] = 1j
    z[2, 1, 3] = z[2, 2, 0] = -1j
    z[3, 0, 2] = z[3, 1, 3] = z[3, 2, 0] = z[3, 3, 1] = 1
    return z


def _shift(dims, mu, step):
    """Index of the neighbour of every site in direction mu."""
    idx = torch.arange(dims[0] * dims[1] * dims[2] * dims[3], device="cuda")
    return torch.roll(idx.view(dims[3], dims[2], dims[1], dims[0]), -step, 3 - mu).reshape(-1)


class _Wilson:
    """The Wilson-clover matrix in complex128 on [V][12] vectors."""

    def __init__(self, dims, U):
        self.dims, self.U = dims, U
        self.vol = U.shape[1]
        self.gam = torch.from_numpy(_gammas()).cuda()
        self.fwd = [_shift(dims, mu, 1) for mu in range(4)]
        self.bwd = [_shift(dims, mu, -1) for mu in range(4)]
        t = torch.arange(self.vol, device="cuda") // (self.vol // dims[3])
        one = torch.ones(self.vol, dtype=torch.float64, device="cuda")
        self.sign_f = torch.where(t == dims[3] - 1, -one, one)  # antiperiodic in t
        self.sign_b = torch.where(t == 0, -one, one)
        A = torch.zeros(self.vol, 4, 3, 4, 3, dtype=torch.complex128, device="cuda")
        for mu in range(4):
            for nu in range(mu + 1, 4):
                sig = 0.5j * (self.gam[mu] @ self.gam[nu] - self.gam[nu] @ self.gam[mu])
                Q = self._leaves(mu, nu)
                F = (Q - Q.mH) / 8
                nz = [(int(a), int(b)) for a, b in torch.nonzero(sig).tolist()]
                for a, b in nz:
                    A[:, a, :, b, :] += (0.5j * CSW * sig[a, b]) * F
        self.A = A.reshape(self.vol, 12, 12)
        self.A += (4.0 + MASS) * torch.eye(12, dtype=torch.complex128, device="cuda")

    def _leaves(self, mu, nu):
        U, f, b = self.U, self.fwd, self.bwd
        Um, Un = U[mu], U[nu]
        mm, mn = b[mu], b[nu]
        q = _mul3(_mul3(Um, Un[f[mu]]), _mul3(Um[f[nu]].mH, Un.mH))
        q += _mul3(_mul3(Un, Um[mm][f[nu]].mH), _mul3(Un[mm].mH, Um[mm]))
        both = mm[mn]
        q += _mul3(_mul3(Um[mm].mH, Un[both].mH), _mul3(Um[both], Un[mn]))
        q += _mul3(_mul3(Un[mn].mH, Um[mn]), _mul3(Un[mn][f[mu]], Um.mH))
        return q

    def diag(self, psi, sites=slice(None)):
        out = torch.empty_like(psi)
        A = self.A[sites]
        for k in range(0, psi.shape[0], 1 << 19):
            out[k:k + (1 << 19)] = (A[k:k + (1 << 19)] * psi[k:k + (1 << 19), None, :]).sum(-1)
        return out

    def term(self, psi, mu, forward, sites=None):
        """The hop term of direction mu (-1/2 included) at `sites` (all)."""
        sites = torch.arange(self.vol, device="cuda") if sites is None else sites
        out = torch.empty(sites.numel(), 12, dtype=torch.complex128, device="cuda")
        eye = torch.eye(4, dtype=torch.complex128, device="cuda")
        for k in range(0, sites.numel(), 1 << 19):
            s = sites[k:k + (1 << 19)]
            nb = (self.fwd if forward else self.bwd)[mu][s]
            p = psi[nb].view(-1, 4, 3)
            P = eye - self.gam[mu] if forward else eye + self.gam[mu]
            h = torch.einsum("st,vtc->vsc", P, p)
            u = self.U[mu][s] if forward else self.U[mu][nb].mH
            w = (u[:, None] * h[:, :, None, :]).sum(-1)
            if mu == 3:
                w = w * (self.sign_f if forward else self.sign_b)[s, None, None]
            out[k:k + (1 << 19)] = -0.5 * w.reshape(-1, 12)
        return out

    def hops(self, psi, sites=None):
        return sum(self.term(psi, mu, f, sites) for mu in range(4) for f in (True, False))

    def apply(self, psi):
        return self.diag(psi) + self.hops(psi)


def _aggregates(dims, block):
    """Sites of every aggregate [coarse site][site in it], both lexicographic."""
    d, c = dims, [x // block for x in dims]
    idx = torch.arange(d[0] * d[1] * d[2] * d[3], device="cuda")
    v = idx.view(c[3], block, c[2], block, c[1], block, c[0], block)
    return v.permute(0, 2, 4, 6, 1, 3, 5, 7).reshape(c[0] * c[1] * c[2] * c[3], block ** 4)


def _orthonormal(v, dims, block):
    """QR (positive diagonal) of every (aggregate, chirality) block: the
    prolongator [V][12][nvec] and the vectors [nvec][V][12]."""
    agg = _aggregates(dims, block)
    nv, vol = v.shape[0], v.shape[1]
    P = torch.empty(vol, 12, nv, dtype=torch.complex128, device="cuda")
    for k in range(0, agg.shape[0], 256):
        a = agg[k:k + 256]
        w = v[:, a].permute(1, 2, 3, 0)  # [aggregate][site][dof][vector]
        for chi in (0, 1):
            m = w[:, :, 6 * chi:6 * chi + 6].reshape(a.shape[0], -1, nv)
            for _ in range(2):  # Cholesky QR, twice
                L = torch.linalg.cholesky(m.mH @ m)
                m = torch.linalg.solve_triangular(L, m.mH, upper=False).mH
            P[a.reshape(-1), 6 * chi:6 * chi + 6] = m.reshape(-1, 6, nv)
    return P, P.permute(2, 0, 1)


def _exact_coarse(case, g):
    vol, n, rhs, dims = _vol(case), case["n"], case["rhs"], _dims(case)
    _gauge(g, 16 * vol)  # drawn before the links
    L = _links(g, vol, n)
    x = _gauss(g, *((vol, n) + ((rhs,) if rhs > 1 else ())))
    x = x.to(torch.complex64).to(torch.complex128).view(vol, n, rhs)
    y = L[:, 0] @ x
    for mu in range(4):
        y += L[:, 1 + 2 * mu] @ x[_shift(dims, mu, 1)]
        y += L[:, 2 + 2 * mu] @ x[_shift(dims, mu, -1)]
    return y if rhs > 1 else y.view(vol, n)


def _exact_schur(case, g, op):
    dims, vol = _dims(case), _vol(case)
    x = _gauss(g, case["rhs"], vol // 2, 12).to(torch.complex64).to(torch.complex128)
    s = torch.arange(vol, device="cuda")
    par = (s % dims[0] + s // dims[0] % dims[1] + s // (dims[0] * dims[1]) % dims[2]
           + s // (dims[0] * dims[1] * dims[2])) % 2
    even, odd = s[par == 0], s[par == 1]
    inv = torch.linalg.inv(op.A[even])
    out = torch.empty_like(x)
    for v in range(case["rhs"]):
        full = torch.zeros(vol, 12, dtype=torch.complex128, device="cuda")
        full[odd] = x[v]
        he = (inv @ op.hops(full, even)[:, :, None])[:, :, 0]
        mid = torch.zeros_like(full)
        mid[even] = he
        out[v] = op.diag(x[v], odd) - op.hops(mid, odd)
    return out


def _exact_galerkin(case, op, P):
    dims, block, nv = _dims(case), case["block"], case["nvec"]
    vol, n = _vol(case), 2 * case["nvec"]
    agg = _aggregates(dims, block)
    cvol = agg.shape[0]
    s = torch.arange(vol, device="cuda")
    coord = [s % dims[0], s // dims[0] % dims[1], s // (dims[0] * dims[1]) % dims[2],
             s // (dims[0] * dims[1] * dims[2])]
    out = torch.zeros(cvol, 9, n, n, dtype=torch.complex128, device="cuda")
    Pa = P[agg.reshape(-1)].view(cvol, -1, 2, 6, nv)  # [aggregate][site][chirality][dof][vector]
    Pa = Pa.permute(0, 2, 4, 1, 3).reshape(cvol, 2, nv, -1).conj()
    for col in range(n):
        chi, j = divmod(col, nv)
        psi = torch.zeros(vol, 12, dtype=torch.complex128, device="cuda")
        psi[:, 6 * chi:6 * chi + 6] = P[:, 6 * chi:6 * chi + 6, j]
        inside = op.diag(psi)
        parts = []
        for mu in range(4):
            for f in (True, False):
                t = op.term(psi, mu, f)
                leaves = (coord[mu] % block == (block - 1 if f else 0))[:, None]
                parts.append(torch.where(leaves, t, 0))
                inside += torch.where(leaves, 0, t)
        for slot, t in enumerate([inside] + parts):
            ta = t[agg.reshape(-1)].view(cvol, -1, 2, 6).permute(0, 2, 1, 3).reshape(cvol, 2, -1, 1)
            out[:, slot, :, col] = (Pa @ ta).reshape(cvol, n)
    return out


def _solve(op, b):
    """BiCGStab to a relative residual of 1e-13, restarted from the true residual."""
    x = torch.zeros_like(b)
    dot = lambda a, c: torch.vdot(a.reshape(-1), c.reshape(-1))  # noqa: E731
    bn = float(torch.linalg.vector_norm(b))
    for _ in range(4):
        r = b - op.apply(x)
        if float(torch.linalg.vector_norm(r)) <= 1e-13 * bn:
            break
        r0, p, rho = r.clone(), r.clone(), dot(r, r)
        for _ in range(150):
            v = op.apply(p)
            alpha = rho / dot(r0, v)
            s = r - alpha * v
            t = op.apply(s)
            om = dot(t, s) / dot(t, t)
            x += alpha * p + om * s
            r = s - om * t
            if float(torch.linalg.vector_norm(r)) <= 3e-14 * bn:
                break
            new = dot(r0, r)
            p = r + (new / rho) * (alpha / om) * (p - om * v)
            rho = new
    return x


def exact(case, seed):
    g = _gen(seed)
    kind, dims, vol = case["kind"], _dims(case), _vol(case)
    if kind == "coarse":
        return _exact_coarse(case, g)
    op = _Wilson(dims, _gauge(g, vol))
    if kind == "wilson":
        x = _gauss(g, case["rhs"], vol, 12).to(torch.complex64).to(torch.complex128)
        return torch.stack([op.apply(v) for v in x])
    if kind == "schur":
        return _exact_schur(case, g, op)
    if kind == "solve":
        b = _gauss(g, case["rhs"], vol, 12)
        return torch.stack([_solve(op, v) for v in b])
    v = _gauss(g, case["nvec"], vol, 12)
    if kind == "setup":
        for i in range(case["nvec"]):
            x = v[i]
            for _ in range(case["sweeps"]):
                t = op.apply(x)
                q = op.apply(t)
                x = x - (torch.vdot(q.reshape(-1), t.reshape(-1))
                         / torch.vdot(q.reshape(-1), q.reshape(-1))) * t
            v[i] = x / torch.linalg.vector_norm(x)
        return _orthonormal(v, dims, case["block"])[1]
    P, _ = _orthonormal(v, dims, case["block"])
    if kind == "galerkin":
        return _exact_galerkin(case, op, P)
    del v
    x = _gauss(g, vol, 12).to(torch.complex64).to(torch.complex128)
    agg = _aggregates(dims, case["block"])
    c = torch.empty(agg.shape[0], 2 * case["nvec"], dtype=torch.complex128, device="cuda")
    y = torch.empty_like(x)
    for k in range(0, agg.shape[0], 256):
        a = agg[k:k + 256]
        for chi in (0, 1):
            q = slice(6 * chi, 6 * chi + 6)
            m = P[a.reshape(-1), q].reshape(a.shape[0], -1, case["nvec"])
            f = x[a.reshape(-1), q].reshape(a.shape[0], -1, 1)
            e = m.mH @ f
            c[k:k + 256, chi * case["nvec"]:(chi + 1) * case["nvec"]] = e[:, :, 0]
            y[a.reshape(-1), q] = (m @ e).reshape(-1, 6)
    return c, y
