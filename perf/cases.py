"""Performance cases of the domain-decomposed estimate of fermion determinant ratios.

Each case is one call, or the short sequence of calls, that a reweighting program makes through
``paper_1211_1214_gb300.binding.Context``: operator applications, inversions, stochastic estimates,
their adjoint, the exact block determinants and the set-up of a new configuration.  Lattices,
block lengths, masses, precisions and numbers of noise vectors are those of the repository's
benchmark workloads and tests, or lie between them.

``exact`` evaluates the same quantities in 64-bit torch arithmetic with code of its own (dense
gamma matrices, plain shifts of the whole lattice, BiCGStab on the unreduced operator).
"""
import math

import numpy as np
import torch

from paper_1211_1214_gb300 import binding

PRECS = {"fp64": binding.FP64, "fp32": binding.MIXED_FP32, "fp16": binding.MIXED_FP16, "bf16": binding.MIXED_BF16}

#: link width, clover coefficient, ensemble mass and target mass(es) of the repository's workloads
PHYSICS = {
    "tiny": (0.3, 1.0, 0.20, (0.19,)),                     # the test lattices of 4^4 sites
    "coarse": (0.25, 1.5, 0.05, (0.045,)),                 # the 16^4 workload with 4^4 blocks
    "fine": (0.2, 1.9, 0.02, (0.015,)),                    # the 32x16^3 and 48x24^3 workloads
    "sweep": (0.2, 1.9, 0.02, (0.018, 0.015, 0.010)),      # the 64x32^3 mass sweep
}

#: BiCGStab steps to a residual of 1e-10 on these near-unit links (two even-odd operators, that is two
#: applications of D, each): full lattice and inside a block
OUTER_STEPS, BLOCK_STEPS = 80, 18
SITE_FLOPS = 1872.0  # one application of D to one site: hops 1320, clover term 504, diagonal 48


def listed():
    return [
        # the smallest call: one FP64 operator application on the lattice of the first test, where
        # launches and the host path are everything
        dict(name="apply_D 4^4", kind="apply", dims="4x4x4x4", l=2, nrhs=1, prec="fp64", physics="tiny"),
        # an FP64 operator application on the 12 spin-colour columns of a propagator
        dict(name="apply_D 32x16^3 x12", kind="apply", dims="32x16x16x16", l=8, nrhs=12, prec="fp64", physics="fine"),
        # the 12 inversions of a propagator in the production precision
        dict(name="solve_D 32x16^3 x12", kind="solve", dims="32x16x16x16", l=8, nrhs=12, prec="fp16", physics="fine"),
        # a new configuration of a trajectory: links in, clover term and in-block inverses rebuilt,
        # then its first operator application
        dict(name="load 32x16^3", kind="load", dims="32x16x16x16", l=8, nrhs=1, prec="fp64", physics="fine"),
        # the default precision of a new context (everything in FP64) on a small lattice
        dict(name="estimate 8^4 fp64", kind="estimate", dims="8x8x8x8", l=4, nrhs=4, prec="fp64", physics="coarse"),
        # 6^4 blocks, an uneven lattice and an odd number of noise vectors, FP32 inner solves
        dict(name="estimate 24x12^3 fp32", kind="estimate", dims="24x12x12x12", l=6, nrhs=5, prec="fp32", physics="fine"),
        # the 16^4 workload as it stands, in the production precision
        dict(name="estimate 16^4 fp16", kind="estimate", dims="16x16x16x16", l=4, nrhs=16, prec="fp16", physics="coarse"),
        # the sweep over three target masses on a middle-sized lattice
        dict(name="sweep 32x16^3 fp16", kind="masses", dims="32x16x16x16", l=8, nrhs=6, prec="fp16", physics="sweep"),
        # mass interpolation in two steps on 48x24^3 with 6^4 blocks
        dict(name="interp 48x24^3 fp16", kind="interp", dims="48x24x24x24", l=6, nrhs=3, prec="fp16", physics="fine"),
        # the largest lattice, the paper's 64x32^3 with 8^4 blocks
        dict(name="estimate 64x32^3 fp16", kind="estimate", dims="64x32x32x32", l=8, nrhs=4, prec="fp16", physics="fine"),
        # backward: the link force and the mass derivative of four noise vectors (adjoint workload)
        dict(name="force 16^4 fp32", kind="force", dims="16x16x16x16", l=4, nrhs=4, prec="fp32", physics="coarse"),
        # the exact block factor's determinants, one mass, for the 4096 sub-blocks of 2^4 sites
        dict(name="block_logdet 16^4", kind="logdet", dims="16x16x16x16", l=2, nrhs=1, prec="fp64", physics="coarse"),
    ]


# most sites times right-hand sides of a drawn case, by kind and precision (a pass of a second or less)
_MOST = {"apply": 1 << 23, "load": 1 << 21, "solve": 1 << 22, "estimate": 1 << 22, "masses": 1 << 22, "interp": 1 << 22,
         "force": 1 << 18}


def draw(rng):
    kind = rng.choice(["apply", "solve", "load", "estimate", "estimate", "masses", "interp", "force", "logdet"])
    if kind == "logdet":
        dims = "x".join(str(4 * rng.randint(1, 4)) for _ in range(4))
        return dict(kind=kind, dims=dims, l=2, nrhs=1, prec="fp64", physics="coarse", mass=round(rng.uniform(0.02, 0.2), 4))
    prec = "fp64" if kind in ("apply", "load") else rng.choice(["fp64", "fp32", "fp16", "fp16", "bf16"])
    most = _MOST[kind] // (8 if prec == "fp64" and kind not in ("apply", "load") else 1)
    nrhs = 1 if kind == "load" else rng.randint(1, 16)
    slots = {"masses": 3, "interp": 2}.get(kind, 1)
    target = math.exp(rng.uniform(math.log(2048), math.log(most / (nrhs * slots))))
    for _ in range(1000):
        l = rng.choice([2, 4, 4, 6, 8, 8])
        side = target ** 0.25
        dims = [2 * l * max(1, round(side * math.exp(rng.uniform(-0.3, 0.5)) / (2 * l))) for _ in range(4)]
        V = math.prod(dims)
        if target / 2 <= V <= min(2 * target, most / (nrhs * slots)):
            break
    else:
        l, dims, nrhs = 4, [8, 8, 8, 8], 2
    V = math.prod(dims)
    physics = "sweep" if kind == "masses" else "coarse" if V < 80000 else "fine"
    return dict(kind=kind, dims="x".join(map(str, dims)), l=l, nrhs=nrhs, prec=prec, physics=physics)


def _dims(case):
    return tuple(int(d) for d in case["dims"].split("x"))


def _masses(case):
    eps, csw, m1, m2s = PHYSICS[case["physics"]]
    return eps, csw, m1, m2s, case.get("mass", m2s[-1])


# ---- inputs


def _gell_mann_half(device):
    lam = np.zeros((8, 3, 3), dtype=np.complex128)
    lam[0][0, 1] = lam[0][1, 0] = 1
    lam[1][0, 1], lam[1][1, 0] = -1j, 1j
    lam[2][0, 0], lam[2][1, 1] = 1, -1
    lam[3][0, 2] = lam[3][2, 0] = 1
    lam[4][0, 2], lam[4][2, 0] = -1j, 1j
    lam[5][1, 2] = lam[5][2, 1] = 1
    lam[6][1, 2], lam[6][2, 1] = -1j, 1j
    lam[7] = np.diag([1, 1, -2]) / math.sqrt(3)
    return torch.from_numpy(lam / 2).to(device)


def _links(V, eps, seed, device="cuda"):
    """SU(3) links exp(i eps H), H = sum_a w_a lambda_a / 2 with w_a ~ N(0, 1): [V, 4, 3, 3] complex128."""
    g = torch.Generator(device=device).manual_seed(seed)
    lam = _gell_mann_half(device).reshape(8, 9)
    U = torch.empty((V * 4, 3, 3), dtype=torch.complex128, device=device)
    step = 1 << 20
    for lo in range(0, V * 4, step):
        hi = min(V * 4, lo + step)
        w = torch.randn((hi - lo, 8), generator=g, dtype=torch.float64, device=device) * eps
        A = 1j * (w.to(torch.complex128) @ lam).reshape(-1, 3, 3) / 8
        E = torch.eye(3, dtype=torch.complex128, device=device).expand_as(A).clone()
        T = E
        for k in range(1, 14):  # |A| < 1/2: the series ends below 1e-16
            T = (T.unsqueeze(-1) * A.unsqueeze(-3)).sum(-2) / k
            E = E + T
        for _ in range(3):
            E = (E.unsqueeze(-1) * E.unsqueeze(-3)).sum(-2)
        r0 = E[:, 0] / torch.linalg.vector_norm(E[:, 0], dim=-1, keepdim=True)
        r1 = E[:, 1] - (r0.conj() * E[:, 1]).sum(-1, keepdim=True) * r0
        r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
        U[lo:hi] = torch.stack([r0, r1, torch.linalg.cross(r0, r1).conj()], dim=-2)
    return U.reshape(V, 4, 3, 3)


def _gaussian(shape, seed, device="cuda"):
    g = torch.Generator(device=device).manual_seed(seed)
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), generator=g, dtype=torch.float64, device=device) * math.sqrt(0.5))


def _inputs(case, seed):
    """What the case reads besides its parameters: links, source fields or noise, weights."""
    dims = _dims(case)
    V = math.prod(dims)
    U = _links(V, PHYSICS[case["physics"]][0], 2 * seed + 1)
    src = _gaussian((case["nrhs"], V, 4, 3), 2 * seed + 2) if case["kind"] in ("apply", "load", "solve") else None
    w = np.random.RandomState(seed % (1 << 31)).uniform(0.5, 1.5, case["nrhs"]) if case["kind"] == "force" else None
    return U, src, w


def prepare(case, seed):
    dims, kind = _dims(case), case["kind"]
    eps, csw, m1, m2s, m2 = _masses(case)
    U, src, w = _inputs(case, seed)
    ctx = binding.Context(dims, (case["l"],) * 4)
    torch.cuda.synchronize()  # the context has a stream of its own
    ctx.load_gauge(U)
    ctx.set_params(csw, m1, m2)
    prec = PRECS[case["prec"]]
    # solutions and forces, which are used themselves, an order below the exponents' residual
    tol = 1e-11 if kind in ("solve", "force") else 1e-10
    ctx.set_solver(prec, tol_outer=tol, tol_block=1e-13 if prec == binding.FP64 else tol)
    state = dict(case=case, ctx=ctx, seed=seed, m2=m2, m2s=m2s, src=src, weights=w)
    if src is not None:
        state["out"] = torch.empty_like(src)
    if kind == "load":
        state["U"] = U
    if kind == "force":
        state["dU"] = torch.empty((ctx.V, 4, 8), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    return state


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind, n, seed = case["kind"], case["nrhs"], state["seed"]
    if kind == "apply":
        ctx.apply_D(state["m2"], state["src"], state["out"], nrhs=n)
        return state["out"]
    if kind == "load":
        ctx.load_gauge(state["U"])
        ctx.apply_D(state["m2"], state["src"], state["out"], nrhs=n)
        return state["out"]
    if kind == "solve":
        ctx.solve_D(state["m2"], state["src"], state["out"], nrhs=n)
        return state["out"]
    if kind == "estimate":
        e, log_w, _, _ = ctx.estimate(n, seed=seed)
        return e, np.array([log_w])
    if kind == "masses":
        e, log_w, _, _ = ctx.estimate_masses(state["m2s"], n, seed=seed)
        return e, log_w
    if kind == "interp":
        r = ctx.estimate_interp(2, n, seed=seed)
        return r["exponents"], r["exponents_1f"], r["logW_factors"]
    if kind == "force":
        e, dm2, _ = ctx.force(n, seed=seed, weights=state["weights"], dU=state["dU"])
        return e, dm2, state["dU"]
    return ctx.block_logdet(state["m2"])


def work(case):
    V, n, kind = math.prod(_dims(case)), case["nrhs"], case["kind"]
    field, links = 192.0 * V, 576.0 * V
    if kind == "apply":
        return {"bytes": links + 2 * n * field, "flops": SITE_FLOPS * V * n}
    if kind == "load":
        # clover: six planes of four leaves of three 3x3 products; one 6x6 Hermitian inverse per chirality
        return {"bytes": links + 2 * field, "flops": V * (6 * 4 * 3 * 198 + 2 * 2 * 600 + SITE_FLOPS)}
    if kind == "logdet":
        dim = 6 * case["l"] ** 4
        blocks = V // case["l"] ** 4
        return {"bytes": links + 16.0 * blocks, "flops": blocks * 8.0 / 3.0 * dim ** 3}
    slots = {"masses": len(PHYSICS[case["physics"]][3]), "interp": 2}.get(kind, 1)
    outer = 2 * OUTER_STEPS * SITE_FLOPS * V
    blocks = 2 * BLOCK_STEPS * SITE_FLOPS * V  # a solve on each colour is one on the lattice
    if kind == "solve":
        return {"bytes": links + 2 * n * field, "flops": n * outer * 1.2}
    if kind == "force":
        return {"bytes": links + 256.0 * V, "flops": n * (2 * outer * 1.2 + 6 * blocks)}
    return {"bytes": links + 16.0 * n * slots, "flops": n * slots * (outer + 2 * blocks)}


# ---- the same quantities in 64 bits


class _Ref:
    """D(m) on fields [T, X, Y, Z, 3 (colour), 4 (spin), n] by shifts of the whole lattice."""

    def __init__(self, U, dims, l, csw):
        dev = U.device
        self.dims, self.U = dims, U.reshape(dims + (4, 3, 3)).movedim(4, 0)
        x = torch.meshgrid(*[torch.arange(d, device=dev) for d in dims], indexing="ij")
        blk = sum(c // l for c in x) % 2
        self.black = (blk == 0)[..., None, None, None]
        face = torch.zeros_like(blk, dtype=torch.bool)
        for c in x:
            face |= (c % l == 0) | (c % l == l - 1)
        self.P = (face & (blk == 0)).reshape(-1)
        one, z = np.eye(2), np.zeros((2, 2))
        s = [np.array([[0, 1], [1, 0]]), np.array([[0, -1j], [1j, 0]]), np.diag([1.0, -1.0])]
        gam = [np.block([[z, -one], [-one, z]]).astype(complex)] + [np.block([[z, -1j * k], [1j * k, z]]) for k in s]
        self.perm = [torch.tensor([int(np.flatnonzero(g[a])[0]) for a in range(4)], device=dev) for g in gam]
        self.phase = [torch.tensor([g[a, np.flatnonzero(g[a])[0]] for a in range(4)], device=dev)[:, None] for g in gam]
        self.C = None
        for mu in range(4) if csw else ():
            for nu in range(mu + 1, 4):
                sg = torch.from_numpy(0.5j * (gam[mu] @ gam[nu] - gam[nu] @ gam[mu])).to(dev)
                F = self._field_strength(mu, nu)
                t = (0.5j * csw) * torch.einsum("st,...ab->...asbt", sg, F).reshape(dims + (12, 12))
                self.C = t if self.C is None else self.C + t

    def _field_strength(self, mu, nu):
        U, d = self.U, torch.conj
        up = lambda f, m: torch.roll(f, -1, m)
        dn = lambda f, m: torch.roll(f, 1, m)
        dag = lambda f: d(f).transpose(-1, -2)
        loop = U[mu] @ up(U[nu], mu) @ dag(up(U[mu], nu)) @ dag(U[nu])
        # the other three leaves: the plaquettes at x - mu, x - mu - nu and x - nu, started at x
        Un, Um = U[nu], U[mu]
        l2 = Un @ dag(dn(up(Um, nu), mu)) @ dag(dn(Un, mu)) @ dn(Um, mu)
        l3 = dag(dn(Um, mu)) @ dag(dn(dn(Un, mu), nu)) @ dn(dn(Um, mu), nu) @ dn(Un, nu)
        l4 = dag(dn(Un, nu)) @ dn(Um, nu) @ up(dn(Un, nu), mu) @ dag(Um)
        Q = loop + l2 + l3 + l4
        return (Q - dag(Q)) / 8

    def D(self, m, psi):
        out = (4 + m) * psi
        if self.C is not None:
            out = out + (self.C @ psi.reshape(self.dims + (12, -1))).reshape(psi.shape)
        for mu in range(4):
            g = lambda f: f[..., self.perm[mu], :] * self.phase[mu]
            n = psi.shape[-1]
            f = torch.roll(psi, -1, mu)
            f = (self.U[mu] @ (f - g(f)).reshape(self.dims + (3, 4 * n))).reshape(psi.shape)
            b = (self.U[mu].conj().transpose(-1, -2) @ (psi + g(psi)).reshape(self.dims + (3, 4 * n))).reshape(psi.shape)
            out = out - 0.5 * (f + torch.roll(b, 1, mu))
        return out

    def solve(self, m, b, keep=None, tol=1e-13):
        """BiCGStab on D(m), or on its restriction to the sites of `keep`, for every column at once."""
        A = (lambda v: self.D(m, v)) if keep is None else (lambda v: keep * self.D(m, v))
        dot = lambda u, v: (u.conj() * v).reshape(-1, u.shape[-1]).sum(0)
        x, r = torch.zeros_like(b), b.clone()
        rh, p, rho = r.clone(), r.clone(), dot(r, r)
        stop = tol * tol * dot(b, b).real
        safe = lambda u, v: torch.where(v == 0, torch.zeros_like(u), u / torch.where(v == 0, torch.ones_like(v), v))
        for it in range(4000):
            v = A(p)
            alpha = safe(rho, dot(rh, v))
            s = r - alpha * v
            t = A(s)
            omega = safe(dot(t, s), dot(t, t))
            x = x + alpha * p + omega * s
            r = s - omega * t
            new = dot(rh, r)
            p = r + safe(new * alpha, rho * omega) * (p - omega * v)
            rho = new
            if it % 8 == 7:
                live = dot(r, r).real > stop
                if not bool(live.any()):
                    break
                # a column that is done stays as it is
                r, p, rho = r * live, p * live, rho * live
        res = b - A(x)
        if float((dot(res, res).real / dot(b, b).real).max()) > 1e-22 and tol < 1e-12:
            return x + self.solve(m, res, keep, 1e-3)
        return x

    # user layout [n, V, 4, 3] <-> [T, X, Y, Z, 3, 4, n]
    def put(self, f):
        return f.permute(1, 3, 2, 0).reshape(self.dims + (3, 4, -1)).contiguous()

    def take(self, f):
        return f.reshape((-1,) + tuple(f.shape[-3:])).permute(3, 0, 2, 1).contiguous()


def _philox(seed, hits, n):
    """Component k of hit h: Philox4x32-10, counter (k, h, 0, 0), key of the seed; complex Gaussian, E|z|^2 = 1."""
    m = np.uint64(0xFFFFFFFF)
    c = [np.broadcast_to(np.arange(n, dtype=np.uint64), (len(hits), n)).copy(),
         np.broadcast_to(np.array(hits, dtype=np.uint64)[:, None], (len(hits), n)).copy(),
         np.zeros((len(hits), n), np.uint64), np.zeros((len(hits), n), np.uint64)]
    k = [seed & 0xFFFFFFFF, seed >> 32]
    for r in range(10):
        a, b = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        key = [np.uint64((k[0] + r * 0x9E3779B9) & 0xFFFFFFFF), np.uint64((k[1] + r * 0xBB67AE85) & 0xFFFFFFFF)]
        c = [(b >> np.uint64(32)) ^ c[1] ^ key[0], b & m, (a >> np.uint64(32)) ^ c[3] ^ key[1], a & m]
    u1, u2 = (c[0].astype(np.float64) + 1) / 2.0 ** 32, c[1].astype(np.float64) / 2.0 ** 32
    return np.sqrt(-np.log(u1)) * np.exp(2j * np.pi * u2)


class _Chain:
    """One factor 1/det(Mh^dag Mh), Mh = A(mb)^-1 A(ma), for noise on the black face sites."""

    def __init__(self, ref, seed, hits):
        nP = int(ref.P.sum())
        packed = torch.from_numpy(_philox(seed, hits, 12 * nP)).to(ref.P.device).reshape(len(hits), nP, 4, 3)
        full = torch.zeros((len(hits), ref.P.numel(), 4, 3), dtype=torch.complex128, device=ref.P.device)
        full[:, ref.P] = packed
        self.r, self.eta = ref, ref.put(full)
        self.Pm = ref.P.reshape(ref.dims)[..., None, None, None]

    def hop(self, f, to_black):
        """D_bw f (to_black) or D_wb f: the hops from one colour to the other."""
        r = self.r
        src, dst = (~r.black, r.black) if to_black else (r.black, ~r.black)
        return dst * r.D(0.0, src * f)

    def run(self, ma, mb):
        r = self.r
        u = self.hop(self.eta, False)
        a2 = r.solve(mb, u, ~r.black)
        a12 = r.solve(ma, a2, ~r.black)
        t = r.solve(mb, self.hop(a2, True), r.black)
        s = self.Pm * ((ma - mb) * r.solve(ma, self.hop(a12, True) + t, r.black))
        x = r.solve(mb, self.hop(s, False))
        delta = self.Pm * (s - x)
        d = (delta.abs() ** 2).reshape(-1, delta.shape[-1]).sum(0)
        c = (self.eta.conj() * delta).reshape(-1, delta.shape[-1]).sum(0)
        self.delta = delta
        return (d + 2 * c.real).cpu().numpy(), c.cpu().numpy()


def _log_mean(e):
    a = -np.asarray(e)
    return float(a.max() + np.log(np.mean(np.exp(a - a.max()))))


def _exact_force(ref_of, U, case, seed, w, m1, m2):
    """The exponents, de_j/dm2 and sum_j w_j de_j/dU: the solutions of the chain and of its adjoint
    as constants, and the derivative of sum <L, D(U) R> over them by torch's reverse mode."""
    ref = ref_of(U)
    ch = _Chain(ref, seed, list(range(case["nrhs"])))
    e, _ = ch.run(m1, m2)
    g5 = torch.tensor([1.0, 1, -1, -1], device=U.device)[:, None]
    y = ch.eta + ch.delta
    up = ref.solve(m2, g5 * y)
    z = ch.Pm * (y - g5 * ch.hop(up, True))
    pairs = []
    for m, v, sign in ((m1, ch.eta, 1.0), (m2, y, -1.0)):
        a = ref.solve(m, ch.hop(v, False), ~ref.black)
        q = ref.solve(m, ch.hop(a, True), ref.black)
        zt = g5 * ref.solve(m, ref.black * (g5 * z), ref.black)
        wt = g5 * ref.solve(m, ch.hop(g5 * zt, False), ~ref.black)
        pairs += [(zt, q - a, sign), (wt, a - v, sign)]
    dm2 = -2 * sum((L.conj() * R).reshape(-1, L.shape[-1]).sum(0).real for L, R, s in pairs if s < 0).cpu().numpy()
    omega = torch.zeros(U.shape[:2] + (8,), dtype=torch.float64, device=U.device, requires_grad=True)
    X = 1j * torch.einsum("lma,aij->lmij", omega.to(torch.complex128), _gell_mann_half(U.device))
    live = ref_of(U + X @ U)  # exp(X) to first order at omega = 0
    wd = torch.from_numpy(w).to(U.device)
    total = sum(2 * s * (L.conj() * live.D(0.0, R) * wd).sum().real for L, R, s in pairs)
    total.backward()
    return e, dm2, omega.grad


def exact(case, seed):
    dims, kind, l, n = _dims(case), case["kind"], case["l"], case["nrhs"]
    V = math.prod(dims)
    eps, csw, m1, m2s, m2 = _masses(case)
    limit = {"apply": 1 << 23, "load": 1 << 20, "solve": 3 << 19, "estimate": 1 << 20, "masses": 1 << 18, "interp": 1 << 18,
             "force": 1 << 19, "logdet": 1 << 16}[kind]
    if V * n > limit:
        return None
    U, src, w = _inputs(case, seed)
    ref_of = lambda links: _Ref(links, dims, l, csw)
    if kind == "force":
        return _exact_force(ref_of, U, case, seed, w, m1, m2)
    ref = ref_of(U)
    if kind in ("apply", "load"):
        return torch.cat([ref.take(ref.D(m2, ref.put(src[j:j + 1]))) for j in range(n)])
    if kind == "solve":
        return ref.take(ref.solve(m2, ref.put(src)))
    if kind == "estimate":
        e, _ = _Chain(ref, seed, list(range(n))).run(m1, m2)
        return e, np.array([_log_mean(e)])
    if kind == "masses":
        e = np.stack([_Chain(ref, seed, list(range(n))).run(m1, m)[0] for m in m2s])
        return e, np.array([_log_mean(x) for x in e])
    if kind == "interp":
        ms = [m1, 0.5 * (m1 + m2), m2]
        two = [_Chain(ref, seed, list(range(i * n, (i + 1) * n))).run(ms[i], ms[i + 1]) for i in range(2)]
        return np.stack([a for a, _ in two]), np.stack([b for _, b in two]), np.array([_log_mean(a) for a, _ in two])
    # log |det| and sign of every block operator, black blocks first, each colour in lexicographic order
    L4 = l ** 4
    grid = [d // l for d in dims]
    logs = {0: [], 1: []}
    split = lambda f: f.reshape(grid[0], l, grid[1], l, grid[2], l, grid[3], l, 12, -1).permute(0, 2, 4, 6, 1, 3, 5, 7, 8, 9)
    nblk = V // L4
    mats = torch.empty((nblk, 12 * L4, 12 * L4), dtype=torch.complex128, device=U.device)
    cols, per = torch.eye(12 * L4, dtype=torch.complex128, device=U.device), max(1, (1 << 21) // V)
    for j in range(0, 12 * L4, per):
        unit = cols[:, j:j + per].reshape(1, 1, 1, 1, l, l, l, l, 12, -1).expand(*grid, l, l, l, l, 12, -1)
        f = unit.permute(0, 4, 1, 5, 2, 6, 3, 7, 8, 9).reshape(dims + (3, 4, -1))
        out = ref.black * ref.D(m2, ref.black * f) + (~ref.black) * ref.D(m2, (~ref.black) * f)
        mats[:, :, j:j + per] = split(out.reshape(dims + (12, -1))).reshape(nblk, 12 * L4, -1)
    for k in range(nblk):
        b = np.unravel_index(k, grid)
        sign, lg = torch.linalg.slogdet(mats[k])
        logs[int(sum(b)) % 2].append((float(lg), 1.0 if float(sign.real) > 0 else -1.0))
    both = logs[0] + logs[1]
    return np.array([a for a, _ in both]), np.array([b for _, b in both])
