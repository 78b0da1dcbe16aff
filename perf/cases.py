"""What the speed of this library is measured on.

Each case is one call (or one short sequence of calls) of a program that uses
the library through its Python binding: the fine domain-wall operator on its
own, one V-cycle (the preconditioner of a caller's own Krylov solver), the
coarsest-level solve, the adaptive setup, and whole solves (multigrid and the
CG it is compared with).  Sizes are those of the repository's benchmark, tests
and plain-method workload, or lie between them.

A case is a dict: "op" (which call), "dims" as "XxYxZxT", "Ls", "mf", "nrhs",
"prec" of the fine fields ("f64" / "f32"), and where a multigrid is involved
"nvec", "block" (as "bxxbyxbzxbt"), "coarse" (link precision of the coarse
stencil), "relax" (CGNR iterations of the setup's start vectors) and the
smoothing and coarsest-solve parameters.

The exact values (`exact`) come from a plain torch FP64 restatement of the
same definitions at the end of this file; it shares no code with the library.
"""
import math

import torch

from paper_1205_2933_gb300 import dwfmg as G

M5 = 1.8
LINK_PREC = {"f64": G.DWF_F64, "f32": G.DWF_F32, "bf16": G.DWF_BF16, "f16": G.DWF_F16}


def _mg(nvec, block, prec, coarse, relax=8, nu=16, ctol=0.03, citer=128):
    """Multigrid part of a case; the defaults are the benchmark's solve parameters.
    The start vectors get a short relaxation: the setup's outputs then still
    are what its definition gives (hundreds of CG steps leave nothing but
    their own rounding to compare)."""
    return {"nvec": nvec, "block": block, "prec": prec, "coarse": coarse, "relax": relax, "nu": nu, "ctol": ctol,
            "citer": citer}


def listed():
    return [
        # the smallest call: one FP32 operator application on the plain-method
        # workload's lattice (a caller's own small solver loop; launch latency)
        {"name": "apply_f32_4x4x4x4", "op": "apply", "dims": "4x4x4x4", "Ls": 8, "mf": 0.1, "nrhs": 1, "prec": "f32",
         "dag": False},
        # the benchmark's lattice, four right-hand sides through D^+ (a batched
        # mixed-precision solver's inner operator)
        {"name": "apply_f32_dag_16x16x16x32", "op": "apply", "dims": "16x16x16x32", "Ls": 16, "mf": 0.001, "nrhs": 4,
         "prec": "f32", "dag": True},
        # ragged extents and a fifth extent that is no power of two, three sources
        {"name": "apply_f32_6x10x6x14_Ls12", "op": "apply", "dims": "6x10x6x14", "Ls": 12, "mf": 0.02, "nrhs": 3,
         "prec": "f32", "dag": False},
        # FP64 operator at the benchmark's lattice: the true residual of every
        # outer cycle, and the whole cost of the plain method
        {"name": "apply_f64_16x16x16x32", "op": "apply", "dims": "16x16x16x32", "Ls": 16, "mf": 0.001, "nrhs": 1,
         "prec": "f64", "dag": False},
        # the production preconditioner: 12 spin-colour sources through one
        # FP32 V-cycle with the BF16 coarse stencil (benchmark parameters)
        dict(_mg(24, "4x4x4x4", "f32", "bf16"), name="vcycle_f32_12rhs_12x12x12x16", op="vcycle", dims="12x12x12x16",
             Ls=16, mf=0.01, nrhs=12),
        # the same V-cycle for one source: a caller's own flexible solver
        dict(_mg(24, "4x4x4x4", "f32", "bf16"), name="vcycle_f32_1rhs_8x8x8x16", op="vcycle", dims="8x8x8x16", Ls=16,
             mf=0.01, nrhs=1),
        # the plain FP64 method's V-cycle (library defaults: 8 steps, 0.1 / 64)
        dict(_mg(16, "2x2x2x2", "f64", "f64", nu=8, ctol=0.1, citer=64), name="vcycle_f64_1rhs_8x8x8x8", op="vcycle",
             dims="8x8x8x8", Ls=8, mf=0.1, nrhs=1),
        # one coarsest-level solve at the benchmark's coarse shape (512 sites x 24)
        dict(_mg(24, "4x4x4x4", "f32", "bf16", relax=4), name="coarse_solve_512x24_bf16", op="coarse_solve",
             dims="16x16x16x32", Ls=4, mf=0.1, nrhs=1),
        # the adaptive setup: relaxation of 12 vectors, block Gram-Schmidt, R D P
        dict(_mg(24, "4x4x4x4", "f32", "f32"), name="setup_f32_12x12x12x16", op="setup", dims="12x12x12x16", Ls=16, mf=0.01,
             nrhs=1),
        # a propagator: 12 sources solved in one call, mixed precision
        dict(_mg(24, "4x4x4x4", "f32", "bf16"), name="solve_f32_12rhs_8x8x8x8", op="solve", dims="8x8x8x8", Ls=16,
             mf=0.05, nrhs=12),
        # one source, mixed precision, small ragged lattice with small blocks
        dict(_mg(8, "2x3x2x2", "f32", "f32", nu=8, ctol=0.1, citer=64), name="solve_f32_1rhs_8x6x4x10", op="solve",
             dims="8x6x4x10", Ls=8, mf=0.1, nrhs=1),
        # the comparison solver: FP32 CG on the normal equations with FP64 updates
        {"name": "cg_f32_8x8x8x16", "op": "cg", "dims": "8x8x8x16", "Ls": 16, "mf": 0.05, "nrhs": 1, "prec": "f32"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges the listed ones stand for: operator
    applications from 2^4-sized to the benchmark's lattice (odd extents, any
    Ls), and multigrid calls from the plain-method workload up to 12 sources
    on 12^3 x 16."""
    op = rng.choice(["apply", "apply", "apply", "vcycle", "vcycle", "coarse_solve", "setup", "solve", "cg"])
    if op in ("apply", "cg"):
        prec = rng.choice(["f32", "f32", "f64"])
        # 5D sites x sources, spread over the logarithm, at most the listed case's
        if op == "cg":
            most, nrhs, prec = _log_int(rng, 2000, 8 * 8 * 8 * 16 * 12), 1, "f32"
        else:
            most = _log_int(rng, 2000, 131072 * 16 * (4 if prec == "f32" else 1))
            nrhs = rng.choice([1, 1, 2, 3, 4, 6, 12])
        Ls = rng.choice([4, 6, 8, 8, 10, 12, 16, 16, 20, 24, 32])
        top = max(16.0, most / (Ls * nrhs))
        dims = [2, 2, 2, 2]
        for _ in range(200):
            i = rng.randrange(4)
            more = dims[i] + rng.choice([1, 1, 2])
            if math.prod(dims) // dims[i] * more <= top and more <= 32:
                dims[i] = more
        c = {"op": op, "dims": "x".join(map(str, dims)), "Ls": Ls, "nrhs": nrhs, "prec": prec,
             "mf": 0.1 if op == "cg" else rng.choice([0.001, 0.01, 0.1])}
        if op == "apply":
            c["dag"] = rng.random() < 0.5
        return c
    plain = op in ("vcycle", "solve") and rng.random() < 0.25
    prec = "f64" if plain else "f32"
    Ls = rng.choice([4, 8, 8, 16]) if plain else rng.choice([4, 8, 12, 16, 16])
    nvec = rng.choice([8, 12, 16]) if plain else rng.choice([8, 16, 24, 24, 32])
    block = rng.choice([(2, 2, 2, 2), (2, 3, 2, 2)]) if nvec <= 16 else rng.choice([(4, 4, 4, 4), (4, 4, 4, 4), (3, 4, 4, 2)])
    nrhs = 1 if op in ("setup", "coarse_solve") else rng.choice([1, 1, 2, 3, 5, 12])
    # 4D sites x Ls x sources, at most what the listed case of this call has
    most = {"vcycle": 12 * 27648 * 16, "solve": 12 * 4096 * 16, "setup": 27648 * 16, "coarse_solve": 131072 * 4}[op]
    if plain:
        most = 4096 * 8 * 2
    top = _log_int(rng, 4096, most) / (Ls * nrhs)
    cd = [2, 2, 2, 2] if nvec <= 16 else [2, 1, 2, 2]
    for _ in range(60):
        i = rng.randrange(4)
        if math.prod(cd) // cd[i] * (cd[i] + 1) * math.prod(block) <= top:
            cd[i] += 1
    coarse = "f64" if plain else rng.choice(["bf16", "bf16", "f32", "f16"])
    nu, ctol, citer = rng.choice([(8, 0.1, 64), (16, 0.03, 128)])
    return dict(_mg(nvec, "x".join(map(str, block)), prec, coarse, relax=4 if op == "coarse_solve" else rng.choice([4, 6, 8]), nu=nu, ctol=ctol,
                    citer=citer), op=op, dims="x".join(str(a * b) for a, b in zip(cd, block)), Ls=Ls,
                mf=rng.choice([0.05, 0.1]), nrhs=nrhs)


# ---- inputs ---------------------------------------------------------------


def _ints(s):
    return [int(v) for v in s.split("x")]


def _volume(case):
    return math.prod(_ints(case["dims"]))


def _inputs(case, seed):
    """Links [V][4][3][3], the sources (internal layout, FP64) and the setup's
    start vectors (canonical layout) or None, on the GPU, from the seed alone.
    Links: exp(i eps H) with H a traceless Hermitian Gaussian, eps = 0.5."""
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * seed + 17)

    def normal(*shape):
        return torch.view_as_complex(torch.randn(*shape, 2, dtype=torch.float64, device="cuda", generator=g))

    V, Ls = _volume(case), case["Ls"]
    A = normal(V * 4, 3, 3) * math.sqrt(0.5)
    H = 0.5 * (A + A.mH)
    H = H - torch.diag_embed((torch.diagonal(H, dim1=1, dim2=2).sum(1) / 3)[:, None].expand(-1, 3))
    X = (0.5j / 8) * H
    U = eye = torch.eye(3, dtype=torch.complex128, device="cuda").expand(V * 4, 3, 3)
    for k in range(14, 0, -1):  # Taylor series of exp(X), then three squarings
        U = eye + (X @ U) / k
    for _ in range(3):
        U = U @ U
    links = U.reshape(V, 4, 3, 3).contiguous()
    b = normal(case["nrhs"] * V * 12 * Ls)
    start = normal(case["nvec"] // 2 * Ls * V * 12) if "nvec" in case else None
    return links, b, start


def _params(case):
    p = G.mg_default_params()
    p.nu_post = case["nu"]
    p.coarsest_tol = case["ctol"]
    p.coarsest_maxiter = case["citer"]
    p.setup_iters0 = case["relax"]
    p.smoother_prec = LINK_PREC[case["prec"]]
    p.coarse_prec[0] = LINK_PREC[case["coarse"]]
    return p


def _coarse_rhs(case, seed, sites):
    """A right-hand side of the coarsest level: [site][Nvec], FP32."""
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * seed + 18)
    return torch.view_as_complex(torch.randn(sites * case["nvec"], 2, dtype=torch.float32, device="cuda", generator=g))


def prepare(case, seed):
    links, b, start = _inputs(case, seed)
    op = case["op"]
    s = {"case": case, "ctx": G.Context(_ints(case["dims"]), case["Ls"], M5, case["mf"], links)}
    if op == "apply":
        s["in"] = b if case["prec"] == "f64" else b.to(torch.complex64)
        s["out"] = torch.empty_like(s["in"])
        return s
    if op == "cg":
        s["b"], s["x"] = b, torch.empty_like(b)
        return s
    s["p"] = _params(case)
    s["shape"] = (2, [case["nvec"]], [_ints(case["block"])])
    if op == "setup":
        n, nv = s["ctx"].field_elems, case["nvec"]
        sites = _volume(case) // math.prod(_ints(case["block"]))
        s["start"] = start
        s["q"] = torch.empty(nv * n, dtype=torch.complex128, device="cuda")
        s["y"] = torch.empty(sites * 9 * nv * nv, dtype=torch.complex128, device="cuda")
        return s
    G.mg_setup(s["ctx"].h, *s["shape"], s["p"], start)
    if op == "coarse_solve":
        s["b"] = _coarse_rhs(case, seed, _volume(case) // math.prod(_ints(case["block"])))
        s["x"] = torch.empty_like(s["b"])
        return s
    s["b"], s["x"] = b, torch.empty_like(b)
    return s


SOLVE_TOL = 1e-12


def run(s):
    case, h = s["case"], s["ctx"].h
    op = case["op"]
    if op == "apply":
        G.dwf_apply(h, s["out"], s["in"], LINK_PREC[case["prec"]], case["dag"], case["nrhs"])
        return s["out"]
    if op == "vcycle":
        if case["nrhs"] == 1:
            G.mg_vcycle(h, s["x"], s["b"])
        else:
            G.mg_vcycle_batch(h, s["x"], s["b"], case["nrhs"])
        # the FP32 V-cycle's result is FP32 numbers in an FP64 buffer; a caller
        # that preconditions a mixed-precision solver keeps them as FP32
        return s["x"] if case["prec"] == "f64" else s["x"].to(torch.complex64)
    if op == "coarse_solve":
        G.mg_coarse_solve(h, 1, s["x"], s["b"])
        return s["x"]
    if op == "setup":
        G.mg_setup(h, *s["shape"], s["p"], s["start"])
        # what the setup leaves behind, read out as a program that stores it
        # would: the block basis and the coarse stencil, both used in FP32
        G.mg_get_vectors(h, 0, s["q"])
        G.mg_get_coarse_links(h, 1, s["y"])
        return {"basis": s["q"].to(torch.complex64), "stencil": s["y"].to(torch.complex64)}
    s["x"].zero_()
    if op == "solve":
        G.mg_solve(h, s["b"], s["x"], SOLVE_TOL, case["nrhs"])
    else:
        G.dwf_cg_solve(h, s["b"], s["x"], SOLVE_TOL, 20000, case["nrhs"], LINK_PREC[case["prec"]])
    return s["x"]


# ---- what a pass cannot do without ------------------------------------------

FLOPS_PER_SITE = 1440  # one 5D site of D: 8 hops (projection, link product, sum) and the fifth-dimension terms


def work(case):
    V, Ls, nrhs = _volume(case), case["Ls"], case["nrhs"]
    n = V * Ls * 12
    if case["op"] == "apply":
        e = 16 if case["prec"] == "f64" else 8
        links = V * 4 * (9 if case["prec"] == "f64" else 6) * e
        return {"bytes": 2 * n * nrhs * e + links, "flops": FLOPS_PER_SITE * V * Ls * nrhs}
    if case["op"] == "cg":
        return {"bytes": 2 * n * 16 + V * 4 * 9 * 16, "flops": 100 * 2 * FLOPS_PER_SITE * V * Ls}
    e = 16 if case["prec"] == "f64" else 8
    nv = case["nvec"]
    sites = V // math.prod(_ints(case["block"]))
    y = {"f64": 16, "f32": 8, "bf16": 4, "f16": 4}[case["coarse"]]
    stencil = sites * 9 * nv * nv * y
    if case["op"] == "coarse_solve":  # the stencil, b and x; about half the allowed iterations
        return {"bytes": stencil + 2 * sites * nv * 8, "flops": case["citer"] // 2 * sites * 9 * nv * nv * 8}
    applies = 2 * case["nu"] + 1
    vflops = nrhs * (applies * FLOPS_PER_SITE * V * Ls + 2 * nv * n * 8 + case["citer"] // 2 * sites * 9 * nv * nv * 8)
    vbytes = 2 * n * nrhs * 16 + nv * n * e + stencil
    if case["op"] == "vcycle":
        return {"bytes": vbytes, "flops": vflops}
    if case["op"] == "solve":  # at least ten V-cycles
        return {"bytes": vbytes, "flops": 10 * vflops}
    # setup: start vectors in, basis and stencil out; relaxation, Gram matrices and basis change (twice), D Q, R D Q
    flops = nv // 2 * 2 * case["relax"] * FLOPS_PER_SITE * V * Ls + nv * FLOPS_PER_SITE * V * Ls + 6 * nv * nv * n * 8
    return {"bytes": nv // 2 * n * 16 + nv * n * 16 + sites * 9 * nv * nv * 16, "flops": flops}


# ---- exact values: the definitions in plain torch, FP64 ----------------------
# Fields are (T, Z, Y, X, 3, 4, Ls, B): colour, spin, fifth dimension, B fields.

# gamma_mu as (source spin, phase) of each row, mu = x, y, z, t
GAMMA = [((3, 1j), (2, 1j), (1, -1j), (0, -1j)), ((3, -1), (2, 1), (1, 1), (0, -1)),
         ((2, 1j), (3, -1j), (0, -1j), (1, 1j)), ((2, 1), (3, 1), (0, 1), (1, 1))]
AXIS = (3, 2, 1, 0)  # of x, y, z, t


class _Fine:
    def __init__(self, case, links):
        X, Y, Z, T = self.dims = _ints(case["dims"])
        self.Ls, self.mf = case["Ls"], case["mf"]
        U = links.reshape(T, Z, Y, X, 4, 3, 3)
        self.U = [U[..., mu, :, :].clone() for mu in range(4)]
        self.U[3][-1] *= -1  # antiperiodic in t

    def spin(self, psi, mu):
        return torch.stack([psi.select(5, k) * ph for k, ph in GAMMA[mu]], 5)

    def links_times(self, M, psi):
        sh = psi.shape
        return (M.reshape(-1, 3, 3) @ psi.reshape(-1, 3, sh[5] * sh[6] * sh[7])).reshape(sh)

    def hop(self, psi, mu, d):
        """-1/2 (1 -+ gamma_mu) U psi of the neighbour at +-mu."""
        if d > 0:
            v = self.links_times(self.U[mu], torch.roll(psi, -1, AXIS[mu]))
            return -0.5 * (v - self.spin(v, mu))
        v = torch.roll(self.links_times(self.U[mu].mH, psi), 1, AXIS[mu])
        return -0.5 * (v + self.spin(v, mu))

    def local(self, psi):
        out = (5 - M5) * psi
        up, dn = torch.roll(psi[:, :, :, :, :, 2:], -1, 6), torch.roll(psi[:, :, :, :, :, :2], 1, 6)
        up[:, :, :, :, :, :, -1] *= -self.mf
        dn[:, :, :, :, :, :, 0] *= -self.mf
        out[:, :, :, :, :, 2:] -= up
        out[:, :, :, :, :, :2] -= dn
        return out

    def D(self, psi):
        out = self.local(psi)
        for mu in range(4):
            out += self.hop(psi, mu, 1)
            out += self.hop(psi, mu, -1)
        return out

    def gamma(self, psi):  # gamma_5 and the reflection of s
        out = psi.flip(6)
        out[:, :, :, :, :, 2:] *= -1
        return out

    def Ddag(self, psi):
        return self.gamma(self.D(self.gamma(psi)))

    def of_internal(self, v, B):
        X, Y, Z, T = self.dims
        return v.to(torch.complex128).reshape(B, T, Z, Y, X, 4, 3, self.Ls).permute(1, 2, 3, 4, 6, 5, 7, 0).contiguous()

    def to_internal(self, psi):
        return psi.permute(7, 0, 1, 2, 3, 5, 4, 6).reshape(-1)

    def of_canonical(self, v, B):
        X, Y, Z, T = self.dims
        return v.reshape(B, self.Ls, T, Z, Y, X, 4, 3).permute(2, 3, 4, 5, 7, 6, 1, 0).contiguous()


def _sq(v):
    """|v_b|^2 of each of the B fields."""
    return (v.real.square() + v.imag.square()).reshape(-1, v.shape[-1]).sum(0)


def _cgnr(fine, b, iters, tol=0.0, x=None):
    """CG on the normal equations for every field at once; until |r| <= tol |b|."""
    r = b if x is None else b - fine.D(x)
    x = torch.zeros_like(b) if x is None else x
    z = fine.Ddag(r)
    p, zz, bb = z.clone(), _sq(z), _sq(b)
    for k in range(iters):
        w = fine.D(p)
        a = zz / _sq(w).clamp_min(1e-300)
        x = x + a * p
        r = r - a * w
        if tol > 0 and k % 8 == 7 and bool((_sq(r) <= tol * tol * bb).all()):
            break
        z = fine.Ddag(r)
        zn = _sq(z)
        p = z + (zn / zz.clamp_min(1e-300)) * p
        zz = zn
    return x


class _Exact:
    """The two-level multigrid of a case in FP64."""

    def __init__(self, case, seed):
        links, b, start = _inputs(case, seed)
        self.case, self.fine, self.b = case, _Fine(case, links), b
        if start is None:
            return
        f, nv = self.fine, case["nvec"]
        self.block = _ints(case["block"])
        self.cd = [a // c for a, c in zip(f.dims, self.block)]
        v = f.of_canonical(start, nv // 2)
        # CGNR on D x = 0 from the start vector, then the whole set orthonormal
        x = _cgnr(f, torch.zeros_like(v), case["relax"], x=v)
        m = (x / _sq(x).sqrt()).reshape(-1, nv // 2)
        for _ in range(2):
            m = m @ torch.linalg.inv(torch.linalg.cholesky(m.mH @ m).mH)
        x = m.reshape(x.shape)
        g = f.gamma(x)
        q = torch.stack([0.5 * (x + g), 0.5 * (x - g)], -1).reshape(x.shape[:-1] + (nv,))
        Q = self.blocks(q)
        for _ in range(2):  # block Gram-Schmidt as two Cholesky QR passes
            Q = Q @ torch.linalg.inv(torch.linalg.cholesky(Q.mH @ Q).mH)
        self.Q = Q
        q = self.unblock(Q, nv)
        rest, Y = f.D(q), [None] * 9
        for mu in range(4):
            c = torch.arange(f.dims[mu], device="cuda")
            for d in (1, -1):
                cross = ((c + d) // self.block[mu] != c // self.block[mu]).to(torch.float64)
                sh = [1] * 8
                sh[AXIS[mu]] = -1
                h = f.hop(q, mu, d) * cross.reshape(sh)
                rest -= h
                Y[1 + 2 * mu + (d < 0)] = Q.mH @ self.blocks(h)
        Y[0] = Q.mH @ self.blocks(rest)
        self.Y = torch.stack(Y, 1)  # (Vc, 9, nv, nv)
        idx = torch.arange(math.prod(self.cd), device="cuda").reshape(self.cd[::-1])
        self.nbr = [idx.reshape(-1)] + [torch.roll(idx, -d, AXIS[mu]).reshape(-1) for mu in range(4) for d in (1, -1)]

    def blocks(self, f):
        X, Y, Z, T = self.cd
        x, y, z, t = self.block
        return f.reshape(T, t, Z, z, Y, y, X, x, -1, f.shape[-1]).permute(0, 2, 4, 6, 1, 3, 5, 7, 8, 9).reshape(
            T * Z * Y * X, -1, f.shape[-1])

    def unblock(self, g, B):
        X, Y, Z, T = self.cd
        x, y, z, t = self.block
        return g.reshape(T, Z, Y, X, t, z, y, x, -1, B).permute(0, 4, 1, 5, 2, 6, 3, 7, 8, 9).reshape(
            T * t, Z * z, Y * y, X * x, 3, 4, self.fine.Ls, B)

    def coarse_apply(self, c):  # (Vc, nv)
        return sum((self.Y[:, d] @ c[self.nbr[d]][:, :, None])[:, :, 0] for d in range(9))

    def coarse_solve(self, b):
        """GCR(16) from x = 0 to the case's tolerance."""
        x, r, bn = torch.zeros_like(b), b, float(torch.linalg.vector_norm(b))
        W, Z, it, rn = [], [], 0, bn
        while it < self.case["citer"] and rn > self.case["ctol"] * bn:
            z, w = r, self.coarse_apply(r)
            if W:
                Wm, Zm = torch.stack(W, 1), torch.stack(Z, 1)
                for _ in range(2):
                    be = Wm.mH @ w.reshape(-1)
                    w = w - (Wm @ be).reshape(w.shape)
                    z = z - (Zm @ be).reshape(z.shape)
            wn = torch.linalg.vector_norm(w)
            w, z = w / wn, z / wn
            a = torch.vdot(w.reshape(-1), r.reshape(-1))
            x, r = x + a * z, r - a * w
            W, Z, it = W + [w.reshape(-1)], Z + [z.reshape(-1)], it + 1
            if len(W) == 16:
                W, Z, r = [], [], b - self.coarse_apply(x)
            rn = float(torch.linalg.vector_norm(r))
        return x

    def vcycle(self, b):  # nu_1 = 0
        rc = self.Q.mH @ self.blocks(b)
        x2 = torch.stack([self.coarse_solve(rc[:, :, k]) for k in range(rc.shape[2])], 2)
        x = self.unblock(self.Q @ x2, b.shape[-1])
        return x + _cgnr(self.fine, b - self.fine.D(x), self.case["nu"])


def exact(case, seed):
    op = case["op"]
    e = _Exact({k: v for k, v in case.items() if op in ("vcycle", "coarse_solve", "setup") or k != "nvec"}, seed)
    f, B = e.fine, case["nrhs"]
    if op == "apply":
        v = e.b if case["prec"] == "f64" else e.b.to(torch.complex64)
        n = v.numel() // B
        return torch.cat([f.to_internal((f.Ddag if case["dag"] else f.D)(f.of_internal(v[k * n:(k + 1) * n], 1)))
                          for k in range(B)])
    if op == "coarse_solve":
        b = _coarse_rhs(case, seed, math.prod(e.cd)).to(torch.complex128).reshape(-1, case["nvec"])
        return e.coarse_solve(b).reshape(-1)
    if op == "setup":
        return {"basis": f.to_internal(e.unblock(e.Q, case["nvec"])), "stencil": e.Y.reshape(-1)}
    b = f.of_internal(e.b, B)
    if op == "vcycle":
        return f.to_internal(e.vcycle(b))
    # solves: D x = b to rounding, CG on the normal equations restarted from the true residual
    x = _cgnr(f, b, 4000, tol=1e-9)
    for _ in range(2):
        x = x + _cgnr(f, b - f.D(x), 4000, tol=1e-6)
    return f.to_internal(x)
