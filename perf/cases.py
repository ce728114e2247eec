"""Representative workloads of the library, from one half-lattice hop to a piece of an RHMC trajectory.

A case is a dict of plain values; prepare() makes the inputs and the context that a user's program
keeps, run() is one pass through the public entry points, exact() the same result in plain torch
complex128, work() the bytes and operations that no implementation can do without.

The lattices, masses and numbers of poles are those of the repository's workloads (4^4, 8^4, 16^3x8,
24^3x6, 32^3x8, 48^3x12 and the mixed-size batch) and ragged ones between them.  Gauge fields and
sources follow the distributions of inputs.py, drawn on the GPU.
"""
import math
import os

# hardware queues for the concurrent solves of the batch case, as the README asks; read at context creation
os.environ.setdefault("CUDA_DEVICE_MAX_CONNECTIONS", "32")

import torch

import paper_1710_09178_gb300 as lq

PRECS = {"fp64": lq.FP64, "df64": lq.DF64, "fp32": lq.FP32, "fp32_r12": lq.FP32_R12, "fp32_r8": lq.FP32_R8,
         "fp32_l16": lq.FP32_L16, "fp16fix": lq.FP16FIX}
LINK_BYTES = {"fp64": 144, "df64": 144, "fp32": 72, "fp32_r12": 48, "fp32_r8": 32, "fp32_l16": 24, "fp16fix": 72}
VEC_BYTES = {"fp64": 48, "df64": 48, "fp32": 24, "fp32_r12": 24, "fp32_r8": 24, "fp32_l16": 24, "fp16fix": 24}
BATCH_SHAPES = [(8, 8, 8, 8), (12, 12, 12, 4), (16, 16, 16, 4), (16, 16, 16, 8)]
MASSES = [0.02, 0.025, 0.05, 0.1]
TOL = 1e-10


def lattice(nx, ny, nz, nt, mass):
    return {"nx": nx, "ny": ny, "nz": nz, "nt": nt, "mass": mass}


def listed():
    return [
        # one hop on a small lattice: what a caller with many small lattices pays per call
        {"name": "hop fp32 8^4", "kind": "hop", "prec": "fp32", "parity": 1, **lattice(8, 8, 8, 8, 0.05)},
        # the hop of the reference workload
        {"name": "hop fp32 32^3x8", "kind": "hop", "prec": "fp32", "parity": 1, **lattice(32, 32, 32, 8, 0.02)},
        # the hop on a lattice far beyond the cache, with the links most such runs would store
        {"name": "hop r12 48^3x12", "kind": "hop", "prec": "fp32_r12", "parity": 0, **lattice(48, 48, 48, 12, 0.02)},
        # the operator A in full precision (eigenvalue bounds, residual checks), with its dot product
        {"name": "apply_A fp64 32^3x8", "kind": "apply", "prec": "fp64", "sigma": 0.3, **lattice(32, 32, 32, 8, 0.02)},
        # the smallest shifted solve, 12 poles
        {"name": "solve fp32 4^4", "kind": "solve", "prec": "fp32", "power": -0.5, "poles": 12,
         **lattice(4, 4, 4, 4, 0.1)},
        # the middle one, 14 poles, in mixed precision and in the paper's all-FP64 form
        {"name": "solve fp32 16^3x8", "kind": "solve", "prec": "fp32", "power": -0.5, "poles": 14,
         **lattice(16, 16, 16, 8, 0.05)},
        {"name": "solve fp64 16^3x8", "kind": "solve", "prec": "fp64", "power": -0.5, "poles": 14,
         **lattice(16, 16, 16, 8, 0.05)},
        # the reference workload's solve, 16 poles
        {"name": "solve fp32 32^3x8", "kind": "solve", "prec": "fp32", "power": -0.5, "poles": 16,
         **lattice(32, 32, 32, 8, 0.02)},
        # the heatbath's x^{1/4} with 12-real links on a ragged lattice
        {"name": "solve r12 24x20x18x10", "kind": "solve", "prec": "fp32_r12", "power": 0.25, "poles": 16,
         **lattice(24, 20, 18, 10, 0.025)},
        # independent lattices of uneven volume, four pseudofermions each, solved concurrently
        {"name": "batch 16x4", "kind": "batch", "prec": "fp32", "power": -0.5, "poles": 12, "lattices": 16, "pick": 7},
        # the gradient of the action in full precision (MD force checks, reversible integration)
        {"name": "force fp64 16^3x8", "kind": "force", "prec": "fp64", "power": -0.5, "poles": 16,
         **lattice(16, 16, 16, 8, 0.025)},
        # a fifth of the 25-step trajectory: heatbath, both Hamiltonians, Omelyan steps with the
        # mixed-precision force
        {"name": "trajectory 24^3x6", "kind": "trajectory", "prec": "fp32", "poles": 16, "steps": 5,
         **lattice(24, 24, 24, 6, 0.025)},
    ]


def draw(rng):
    def extents(most):
        while True:
            d = [2 * round(math.exp(rng.uniform(math.log(2), math.log(20)))) for _ in range(4)]
            if 256 <= math.prod(d) <= most:
                return d

    kind = rng.choice(["hop", "hop", "apply", "solve", "solve", "solve", "batch", "force", "trajectory"])
    mass = rng.choice(MASSES)
    if kind == "hop":
        prec = rng.choice(["fp64", "df64", "fp32", "fp32_r12", "fp32_r8", "fp32_l16"])
        return {"kind": kind, "prec": prec, "parity": rng.randint(0, 1), **lattice(*extents(1 << 20), mass)}
    if kind == "apply":
        prec = rng.choice(["fp64", "df64", "fp32", "fp32_r12"])
        return {"kind": kind, "prec": prec, "sigma": round(rng.uniform(0, 2), 3), **lattice(*extents(1 << 18), mass)}
    if kind == "solve":
        prec = rng.choice(["fp64", "df64", "fp32", "fp32", "fp32_r12", "fp32_l16", "fp16fix"])
        return {"kind": kind, "prec": prec, "power": rng.choice([-0.5, 0.25]), "poles": rng.randint(8, 16),
                **lattice(*extents(1 << 17), mass)}
    if kind == "batch":
        return {"kind": kind, "prec": rng.choice(["fp32", "fp32_r12"]), "power": -0.5, "poles": rng.randint(8, 12),
                "lattices": rng.randint(2, 16), "pick": rng.randint(0, 1 << 20)}
    if kind == "force":
        return {"kind": kind, "prec": "fp64", "power": -0.5, "poles": rng.randint(8, 16),
                **lattice(*extents(1 << 16), mass)}
    return {"kind": kind, "prec": "fp32", "poles": rng.randint(8, 16), "steps": rng.randint(1, 5),
            **lattice(*extents(1 << 16), mass)}


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def dims_of(case):
    return tuple(case[k] for k in ("nx", "ny", "nz", "nt"))


def batch_members(case):
    """(extents, mass) of every lattice of a batch, drawn from the workload's four sizes."""
    out, s = [], case["pick"] * 2654435761 + 12345
    for _ in range(case["lattices"]):
        s = (s * 6364136223846793005 + 1442695040888963407) % (1 << 64)
        out.append((BATCH_SHAPES[(s >> 33) % 4], (0.02, 0.05, 0.1)[(s >> 40) % 3]))
    return out


def generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def matmul3(a, b):
    return sum(a[..., :, k:k + 1] * b[..., k:k + 1, :] for k in range(3))


def hermitian(h):
    """sum_a h_a lambda_a / 2 (Gell-Mann matrices), h: (..., 8) float64."""
    H = torch.zeros(h.shape[:-1] + (3, 3), dtype=torch.complex128, device=h.device)
    t = h[..., 7] / math.sqrt(3)
    H[..., 0, 0] = (h[..., 2] + t) / 2
    H[..., 1, 1] = (t - h[..., 2]) / 2
    H[..., 2, 2] = -t
    for r, c, a in ((0, 1, 0), (0, 2, 3), (1, 2, 5)):
        z = torch.complex(h[..., a], -h[..., a + 1]) / 2
        H[..., r, c] = z
        H[..., c, r] = z.conj()
    return H


def expm3(X):
    """exp of 3x3 matrices by scaling and squaring of the Taylor series."""
    norm = float(X.abs().square().sum((-2, -1)).max().sqrt())
    s = max(0, math.ceil(math.log2(max(norm, 1e-300) / 0.25)))
    X = X / 2.0 ** s
    E = term = torch.eye(3, dtype=X.dtype, device=X.device).expand(X.shape)
    for k in range(1, 15):
        term = matmul3(term, X) / k
        E = E + term
    for _ in range(s):
        E = matmul3(E, E)
    return E


def project_su3(W):
    r0 = W[..., 0, :] / W[..., 0, :].abs().square().sum(-1, keepdim=True).sqrt()
    r1 = W[..., 1, :] - (r0.conj() * W[..., 1, :]).sum(-1, keepdim=True) * r0
    r1 = r1 / r1.abs().square().sum(-1, keepdim=True).sqrt()
    return torch.stack([r0, r1, torch.linalg.cross(r0, r1).conj()], -2).contiguous()


def gauge_field(dims, gen):
    """U = exp(0.5 i H) per link, H with N(0, 1) components; (V, 4, 3, 3)."""
    V, parts = math.prod(dims), []
    for a in range(0, V, 1 << 18):
        n = min(V, a + (1 << 18)) - a
        h = torch.randn((n, 4, 8), dtype=torch.float64, device="cuda", generator=gen)
        parts.append(project_su3(expm3(0.5j * hermitian(h))))
    return torch.cat(parts)


def gaussian(dims, gen):
    """Re, Im ~ N(0, 1/2) on one parity; (V/2, 3)."""
    return torch.randn((math.prod(dims) // 2, 3), dtype=torch.complex128, device="cuda", generator=gen)


def coefficients(power, mass, poles):
    """(c0, residues, poles) of the rational approximation on the spectral interval."""
    return lq.rational_coeffs(power, 4 * mass * mass, 16 + 4 * mass * mass, poles)[:3]


def inputs_of(case, seed):
    gen = generator(seed)
    if case["kind"] == "batch":
        return [{"dims": d, "mass": m, "U": gauge_field(d, gen), "bs": [gaussian(d, gen) for _ in range(4)]}
                for d, m in batch_members(case)]
    dims = dims_of(case)
    x = {"dims": dims, "mass": case["mass"], "U": gauge_field(dims, gen), "b": gaussian(dims, gen)}
    if case["kind"] == "trajectory":
        x["mom"] = torch.randn((math.prod(dims), 4, 8), dtype=torch.float64, device="cuda", generator=gen)
    return x


def context(x):
    ctx = lq.Context(x["dims"], x["mass"])
    ctx.set_gauge(x["U"])
    return ctx


def prepare(case, seed):
    kind, prec, x = case["kind"], PRECS[case["prec"]], inputs_of(case, seed)
    s = {"kind": kind, "prec": prec, "case": case}
    if kind == "batch":
        s["ctxs"], s["problems"], s["ys"] = [], [], []
        for p in x:
            ctx = context(p)
            c0, res, sh = coefficients(case["power"], p["mass"], case["poles"])
            ys = [torch.empty_like(b) for b in p["bs"]]
            s["ctxs"].append(ctx)
            s["ys"].append(ys)
            s["problems"].append({"ctx": ctx, "shifts": sh, "residues": res, "c0": c0, "bs": p["bs"], "ys": ys,
                                  "tol": TOL, "prec": prec})
        return s
    ctx = s["ctx"] = context(x)
    if kind in ("hop", "apply"):
        s["in"], s["out"] = ctx.new_vector(prec), ctx.new_vector(prec)
        ctx.pack(s["in"], prec, x["b"])
        s["canonical"] = torch.empty_like(x["b"])
        return s
    if kind == "trajectory":
        s["act"] = coefficients(-0.5, case["mass"], case["poles"])
        s["heat"] = coefficients(0.25, case["mass"], case["poles"])
        s["U0"], s["mom"], s["xi"] = x["U"], x["mom"], x["b"]
        s["links"], s["mom_out"] = torch.empty_like(x["U"]), torch.empty_like(x["mom"])
        return s
    s["c0"], s["res"], s["sh"] = coefficients(case["power"], case["mass"], case["poles"])
    s["b"] = x["b"]
    if kind == "force":
        s["F"] = torch.empty((ctx.V, 4, 8), dtype=torch.float64, device="cuda")
    else:
        s["x"] = torch.empty((case["poles"],) + tuple(x["b"].shape), dtype=torch.complex128, device="cuda")
        s["xs"] = list(s["x"])
        s["y"] = torch.empty_like(x["b"])
    return s


def result(s):
    """The vector that hop and apply made: its own numbers, (hi, lo) pairs in the canonical layout."""
    if s["prec"] == lq.DF64:
        s["ctx"].unpack(s["canonical"], s["out"], s["prec"])
        return s["canonical"]
    return s["out"].view(torch.float64 if s["prec"] == lq.FP64 else torch.float32)


def run(s):
    kind, prec = s["kind"], s["prec"]
    if kind == "hop":
        lq.dslash_eo(s["ctx"], s["out"], s["in"], s["case"]["parity"], prec)
        return result(s)
    if kind == "apply":
        dot = s["ctx"].apply_A(s["out"], s["in"], s["case"]["sigma"], prec, want_dot=True)
        return {"q": result(s), "dot": dot}
    if kind == "solve":
        lq.mshift_cg(s["ctx"], s["sh"], s["res"], s["c0"], s["b"], s["xs"], s["y"], tol=TOL, prec=prec)
        return {"x": s["x"], "y": s["y"]}
    if kind == "batch":
        lq.mshift_cg_batch(s["problems"])
        return s["ys"]
    if kind == "force":
        _, action, _ = lq.fermion_force(s["ctx"], s["sh"], s["res"], s["c0"], s["b"], Falg=s["F"], tol=TOL, prec=prec)
        return {"F": s["F"], "S": action}
    # every pass starts from the same links (the accepted ones are written over U)
    U = s["U0"].clone()
    n = s["case"]["steps"]
    _, r = lq.rhmc_trajectory(s["ctx"], U, s["mom"], s["xi"], 0.5, 5.4, n / 25, n, s["act"], s["heat"], tol=TOL,
                              prec=prec, mom_out=s["mom_out"], links_out=s["links"])
    return {"links": s["links"], "mom": s["mom_out"], "H0": r["H0"], "H1": r["H1"]}


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------
HOP_FLOPS = 8 * 66 + 7 * 6  # eight 3x3 complex matrix-vector products and their sums, per output site


def iterations(mass):
    """CG iterations to TOL, estimated: the rough fields' smallest eigenvalue of -D_eo D_oe is about 0.07."""
    return 0.5 * math.sqrt(16 / (0.07 + 4 * mass * mass)) * math.log(2 / TOL)


def solve_flops(vh, mass, poles, rhs=1):
    return rhs * vh * iterations(mass) * (2 * HOP_FLOPS + 60 + poles * 24)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        b = f = 0
        for d, m in batch_members(case):
            V = math.prod(d)
            b += V * 4 * 144 + 4 * 2 * V // 2 * 48
            f += solve_flops(V // 2, m, case["poles"], 4)
        return {"bytes": b, "flops": f}
    V = math.prod(dims_of(case))
    vh, lb, vb = V // 2, LINK_BYTES[case["prec"]], VEC_BYTES[case["prec"]]
    if kind == "hop":
        return {"bytes": vh * (8 * lb + 2 * vb), "flops": vh * HOP_FLOPS}
    if kind == "apply":
        return {"bytes": vh * (8 * lb + 2 * vb), "flops": vh * (2 * HOP_FLOPS + 24)}
    if kind == "solve":
        return {"bytes": vh * (8 * lb + 48 * (2 + case["poles"])),
                "flops": solve_flops(vh, case["mass"], case["poles"])}
    force = 8 * vh * (case["poles"] * 90 + 250)
    if kind == "force":
        return {"bytes": V * 4 * (144 + 64) + vh * 48,
                "flops": solve_flops(vh, case["mass"], case["poles"]) + case["poles"] * vh * HOP_FLOPS + force}
    solves = 2 * case["steps"] + 4
    return {"bytes": V * 4 * (2 * 144 + 2 * 64) + vh * 48,
            "flops": solves * solve_flops(vh, case["mass"], case["poles"])
            + (2 * case["steps"] + 1) * (force + 4 * V * 4500)}


# ---------------------------------------------------------------------------------------------
# the same results in plain complex128
# ---------------------------------------------------------------------------------------------
class Operator:
    """D and A on the even and odd half-lattices of canonical links U (V, 4, 3, 3)."""

    def __init__(self, U, dims, mass):
        nx, ny, nz, nt = dims
        self.mass, V = mass, math.prod(dims)
        l = torch.arange(V, device=U.device)
        c = [l % nx, l // nx % ny, l // (nx * ny) % nz, l // (nx * ny * nz)]
        par = (c[0] + c[1] + c[2] + c[3]) % 2
        self.site = [torch.nonzero(par == p)[:, 0] for p in (0, 1)]
        strides, self.fwd, self.nb = (1, nx, nx * ny, nx * ny * nz), [], [[], []]
        W = torch.empty_like(U)
        for mu in range(4):
            up = l + torch.where(c[mu] == dims[mu] - 1, 1 - dims[mu], 1) * strides[mu]
            dn = l + torch.where(c[mu] == 0, dims[mu] - 1, -1) * strides[mu]
            eta = 1 - 2 * (sum(c[:mu]) % 2) if mu else torch.ones_like(l)
            if mu == 3:
                eta = torch.where(c[3] == nt - 1, -eta, eta)
            W[:, mu] = 0.5 * eta[:, None, None] * U[:, mu]
            self.fwd.append(up)
            for p in (0, 1):
                self.nb[p].append((up[self.site[p]], dn[self.site[p]]))
        self.W = W
        self.ahead = [W[s] for s in self.site]
        self.behind = [[W[dn, mu].mH for mu, (_, dn) in enumerate(self.nb[p])] for p in (0, 1)]

    def hop(self, v, p):
        """(D v) on parity p, v on the other one."""
        out = 0
        for mu, (up, dn) in enumerate(self.nb[p]):
            out = out + (self.ahead[p][:, mu] * v[up >> 1][:, None, :]).sum(-1)
            out = out - (self.behind[p][mu] * v[dn >> 1][:, None, :]).sum(-1)
        return out

    def A(self, v, sigma=0.0):
        return (4 * self.mass ** 2 + sigma) * v - self.hop(self.hop(v, 1), 0)

    def solve(self, b, shifts):
        """(A + s) x = b for every s: shifted CG, iterated well below the library's tolerance."""
        shifts = torch.as_tensor([float(v) for v in shifts], dtype=torch.float64, device=b.device)
        base = float(shifts.min())
        s = (shifts - base)[:, None, None]
        n = len(shifts)
        x = torch.zeros((n,) + tuple(b.shape), dtype=b.dtype, device=b.device)
        ps, r, p = b.expand_as(x).clone(), b.clone(), b.clone()
        z = z_old = torch.ones((n, 1, 1), dtype=torch.float64, device=b.device)
        a_old, beta = 1.0, 0.0
        rr = bb = float(torch.vdot(b.flatten(), b.flatten()).real)
        for _ in range(20000):
            q = self.A(p, base)
            a = rr / float(torch.vdot(p.flatten(), q.flatten()).real)
            z_new = z * z_old * a_old / (a * beta * (z_old - z) + z_old * a_old * (1 + s * a))
            live = z.abs() > 1e-60  # a shift far below its own convergence drops out before it underflows
            ratio, z_new = torch.where(live, z_new / z, 0.0), torch.where(live, z_new, 0.0)
            x += (a * ratio) * ps
            r = r - a * q
            rr, old = float(torch.vdot(r.flatten(), r.flatten()).real), rr
            if rr <= 1e-27 * bb:
                return x
            beta = rr / old
            ps = z_new * r + (beta * ratio ** 2) * ps
            p = r + beta * p
            z_old, z, a_old = z, z_new, a
        return x

    def force(self, X, residues):
        """tr(lambda^a F) per link (V, 4, 8) of phi^+ r(A) phi, X_k = (A + d_k)^-1 phi."""
        z = torch.zeros((len(X), self.W.shape[0], 3), dtype=X.dtype, device=X.device)
        z[:, self.site[0]] = X
        z[:, self.site[1]] = torch.stack([self.hop(v, 1) for v in X])
        out = torch.empty((self.W.shape[0], 4, 8), dtype=torch.float64, device=X.device)
        for mu in range(4):
            O = sum(float(c) * v[self.fwd[mu]][:, :, None] * v[:, None, :].conj() for c, v in zip(residues, z))
            M = matmul3(self.W[:, mu], O)
            M[self.site[1]] *= -1
            H = 1j * (M - M.mH)
            out[:, mu] = algebra(H / 2)
        return out


def algebra(F):
    """tr(lambda^a F) of Hermitian F; a trace drops out."""
    re, im = F.real, F.imag
    return torch.stack([2 * re[..., 0, 1], -2 * im[..., 0, 1], re[..., 0, 0] - re[..., 1, 1], 2 * re[..., 0, 2],
                        -2 * im[..., 0, 2], 2 * re[..., 1, 2], -2 * im[..., 1, 2],
                        (re[..., 0, 0] + re[..., 1, 1] - 2 * re[..., 2, 2]) / math.sqrt(3)], -1)


def rational(op, b, coeffs, X=None):
    c0, res, sh = coeffs
    X = op.solve(b, sh) if X is None else X
    return float(c0) * b + sum(float(c) * v for c, v in zip(res, X))


def inner(a, b):
    return float(torch.vdot(a.flatten(), b.flatten()).real)


def gauge_action_and_force(U, op, beta, want):
    """(S_g, None) or (None, dS_g/dw^a)."""
    S, F = 0.0, torch.zeros((U.shape[0], 4, 8), dtype=torch.float64, device=U.device)
    for mu in range(4):
        for nu in range(4):
            if nu == mu:
                continue
            um, un, fm, fn = U[:, mu], U[:, nu], op.fwd[mu], op.fwd[nu]
            # plaquette x -> x+mu -> x+mu+nu -> x+nu -> x
            P = matmul3(matmul3(um, un[fm]), matmul3(un, um[fn]).mH)
            if want == "action":
                if mu < nu:
                    S += float((1 - P.diagonal(dim1=-2, dim2=-1).sum(-1).real / 3).sum())
                continue
            # the plaquette above the link, and the one below it (from x - nu)
            below = torch.empty_like(P)
            below[fn] = matmul3(matmul3(un.mH, um), un[fm])
            W = P + matmul3(um, below.mH)
            F[:, mu] += algebra(-1j * beta / 12 * (W - W.mH))
    return beta * S if want == "action" else F


def trajectory(case, x):
    act, heat = (coefficients(p, case["mass"], case["poles"]) for p in (-0.5, 0.25))
    beta, lam, eps = 5.4, 0.1931833275037836, 1.0 / 25
    U, P = x["U"], x["mom"].clone()
    op = Operator(U, x["dims"], case["mass"])
    phi = rational(op, x["b"], heat)

    def energy():
        return 0.5 * float(P.square().sum()) + gauge_action_and_force(U, op, beta, "action") + inner(
            phi, rational(op, phi, act))

    def force():
        return op.force(op.solve(phi, act[2]), act[1]) + gauge_action_and_force(U, op, beta, "force")

    H0 = energy()
    P -= lam * eps * force()
    for step in range(case["steps"]):
        for kick in (1 - 2 * lam, 2 * lam if step < case["steps"] - 1 else lam):
            U = project_su3(matmul3(expm3(0.5j * eps * hermitian(P)), U))
            op = Operator(U, x["dims"], case["mass"])
            P -= kick * eps * force()
    return {"links": U, "mom": P, "H0": H0, "H1": energy()}


def exact(case, seed):
    kind, x = case["kind"], inputs_of(case, seed)
    if kind == "batch":
        out = []
        for p in x:
            op, co = Operator(p["U"], p["dims"], p["mass"]), coefficients(case["power"], p["mass"], case["poles"])
            out.append([rational(op, b, co) for b in p["bs"]])
        return out
    if kind == "trajectory":
        return trajectory(case, x)
    op = Operator(x["U"], x["dims"], case["mass"])
    if kind in ("hop", "apply"):
        v = op.hop(x["b"], case["parity"]) if kind == "hop" else op.A(x["b"], case["sigma"])
        w = v if case["prec"] == "df64" else torch.view_as_real(v.T.contiguous()).reshape(-1)  # [3][V/2]
        return w if kind == "hop" else {"q": w, "dot": inner(x["b"], v)}
    co = coefficients(case["power"], case["mass"], case["poles"])
    X = op.solve(x["b"], co[2])
    if kind == "force":
        return {"F": op.force(X, co[1]), "S": inner(x["b"], rational(op, x["b"], co, X))}
    return {"x": X, "y": rational(op, x["b"], co, X)}
