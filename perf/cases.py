"""Workloads of the library's hot path, as a program calls it: one entry point per case, on lattices from the
4^4 of the plain method to the 32^4 of a full RMHMC trajectory.

Every case draws its inputs from a seed on the GPU: SU(3) links U = exp(i eps sum_a r_a T_a), r_a ~ N(0,1), and
su(3) fields with N(0,1) coefficients (the recipe of paper_2112_04556_gb300/inputs.py).  A program that uses the
library keeps the lattice context, the imported links and the mass term's coefficients from call to call; prepare()
makes those, run() is the call.

Results of the float32 paths come back as float32, the precision they are computed in (the library stores some of
them in float64 arrays); results with float64 accuracy -- the float64 paths, and mixed-precision solves refined to a
tolerance below float32 -- come back as they are.
"""
import math

import numpy as np
import torch

import paper_2112_04556_gb300 as rm

KAPPA, NPOLE = 0.9, 12            # the mass term of the workloads: 12 poles, kappa = 0.9
BETA, IWASAKI = 6.0, -0.331
LINK_EPS = 0.3
CG_ITERS = 15                     # Krylov iterations that a 3e-7 solve of this mass term needs (13 to 17)


def listed():
    return [
        # the smallest call: one Laplacian on the plain method's 4^4 lattice (launch latency)
        {"name": "laplacian_4^4", "kind": "laplacian", "lattice": "4x4x4x4", "prec": "fp32", "linkfmt": 18, "nfield": 1},
        # the headline Laplacian: one float32 field at 32^4, links and fields far larger than L2
        {"name": "laplacian_32^4", "kind": "laplacian", "lattice": "32x32x32x32", "prec": "fp32", "linkfmt": 18, "nfield": 1},
        # differentiating through the Laplacian: forward, field gradient and link gradient, float64 (16^4 differentiation)
        {"name": "laplacian_grad_16^4", "kind": "laplacian_grad", "lattice": "16x16x16x16", "prec": "fp64"},
        # a kinetic evaluation of a small chain (8^4, the size the strong-coupling chains run at)
        {"name": "kinetic_8^4", "kind": "kinetic", "lattice": "8x8x8x8", "prec": "mixed", "tol": 3e-7},
        # the kinetic evaluation that a 32^4 trajectory makes about 320 times: force, velocity and energy
        {"name": "kinetic_32^4", "kind": "kinetic", "lattice": "32x32x32x32", "prec": "mixed", "tol": 3e-7},
        # the same in float64, as the float64 reference trajectories and the gradient checks run it
        {"name": "kinetic_fp64_16^4", "kind": "kinetic", "lattice": "16x16x16x16", "prec": "fp64", "tol": 1e-10},
        # the rational mass term on a Gaussian field: 12 shifts refined to 1e-10 (24^3 x 48)
        {"name": "mass_solve_24^3x48", "kind": "mass_solve", "lattice": "24x24x24x48", "prec": "mixed", "tol": 1e-10},
        # momentum heatbath on an odd, ragged lattice
        {"name": "heatbath_13x11x9x17", "kind": "heatbath", "lattice": "13x11x9x17", "prec": "mixed", "tol": 1e-11},
        # Iwasaki force, action and plaquette of a configuration (the input of its force spectrum)
        {"name": "gauge_iwasaki_24^3x48", "kind": "gauge", "lattice": "24x24x24x48", "prec": "fp32", "c1": IWASAKI},
        # power spectra of two forces with 16 noise vectors, 64 windows of degree 200, one batched recurrence
        {"name": "spectrum_16^4", "kind": "spectrum", "lattice": "16x16x16x16", "nforce": 2, "nnoise": 16, "degree": 200,
         "nwin": 64},
        # Wilson flow of a configuration, float64, with the flowed energy at every step
        {"name": "flow_16^4", "kind": "flow", "lattice": "16x16x16x16", "nsteps": 8},
        # a whole RMHMC trajectory at the accepting step size (tau = 1 in 40 steps), as a thermalisation runs it
        {"name": "trajectory_16^4", "kind": "trajectory", "lattice": "16x16x16x16", "nsteps": 40},
    ]


def _lattice(rng, lo, hi):
    """Four extents (2 and more, odd ones among them) whose product is spread over lo .. hi in its logarithm."""
    while True:
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        ext = [max(2, round(v ** 0.25 * math.exp(rng.uniform(-0.35, 0.35)))) for _ in range(3)]
        ext.append(max(2, round(v / (ext[0] * ext[1] * ext[2]))))
        if lo <= math.prod(ext) <= hi and ext[3] <= 96:
            return "x".join(map(str, ext))


def draw(rng):
    kind = rng.choice(["laplacian", "laplacian_grad", "kinetic", "mass_solve", "heatbath", "gauge", "spectrum", "flow",
                       "trajectory"])
    v4, v16, v24, v32 = 4 ** 4, 16 ** 4, 24 ** 3 * 48, 32 ** 4
    if kind == "laplacian":
        prec = rng.choice(["fp32", "fp32", "fp64"])
        nfield = rng.choice([1, 1, 1, 2, 4, 8, 18])
        hi = v32 // max(1, nfield // 2) if prec == "fp32" else v16 * 2 // nfield
        return {"kind": kind, "lattice": _lattice(rng, v4, hi), "prec": prec, "linkfmt": rng.choice([18, 18, 12]),
                "nfield": nfield}
    if kind == "laplacian_grad":
        return {"kind": kind, "lattice": _lattice(rng, v4, v16), "prec": rng.choice(["fp64", "fp32"])}
    if kind == "kinetic":
        prec = rng.choice(["mixed", "mixed", "fp64"])
        tol = rng.choice([1e-6, 3e-7]) if prec == "mixed" else 1e-10
        return {"kind": kind, "lattice": _lattice(rng, v4, v32 if prec == "mixed" else v16), "prec": prec, "tol": tol}
    if kind == "mass_solve":
        return {"kind": kind, "lattice": _lattice(rng, v4, v24), "prec": "mixed", "tol": rng.choice([1e-10, 1e-11, 1e-12])}
    if kind == "heatbath":
        return {"kind": kind, "lattice": _lattice(rng, v4, v16), "prec": "mixed", "tol": rng.choice([1e-10, 1e-11, 1e-12])}
    if kind == "gauge":
        prec = rng.choice(["fp32", "fp64"])
        return {"kind": kind, "lattice": _lattice(rng, v4, v24 if prec == "fp32" else v16), "prec": prec,
                "c1": rng.choice([0.0, IWASAKI])}
    if kind == "spectrum":
        return {"kind": kind, "lattice": _lattice(rng, v4, v16), "nforce": rng.choice([1, 2]), "nnoise": rng.choice([8, 16]),
                "degree": rng.choice([64, 128, 200]), "nwin": rng.choice([16, 64])}
    if kind == "flow":
        return {"kind": kind, "lattice": _lattice(rng, v4, v16), "nsteps": rng.randint(2, 8)}
    return {"kind": kind, "lattice": _lattice(rng, v4, v16), "nsteps": rng.randint(2, 10)}


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------
def _dims(case):
    return tuple(int(v) for v in case["lattice"].split("x"))


def _generator(seed, stream):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 16 + stream)


def _gellmann():
    lam = np.zeros((8, 3, 3), dtype=np.complex128)
    for a, (i, j) in ((0, (0, 1)), (3, (0, 2)), (5, (1, 2))):
        lam[a, i, j] = lam[a, j, i] = 1.0
        lam[a + 1, i, j], lam[a + 1, j, i] = -1j, 1j
    lam[2] = np.diag([1.0, -1.0, 0.0])
    lam[7] = np.diag([1.0, 1.0, -2.0]) / np.sqrt(3.0)
    return torch.from_numpy(lam).cuda()


def _mul(a, b):
    """Products of 3x3 matrices (elementwise: batched library products are slow at this size)."""
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _expi(h):
    """exp(i h) of Hermitian 3x3 matrices of norm below 8: the exponential series of h/8, squared three times."""
    m = 0.125j * h
    one = torch.eye(3, dtype=h.dtype, device=h.device).expand_as(h)
    e = one
    for n in range(18, 0, -1):
        e = one + _mul(m, e) / n
    for _ in range(3):
        e = _mul(e, e)
    return e


def _links(dims, seed):
    n = math.prod(dims) * 4
    r = torch.randn((n, 8), dtype=torch.float64, device="cuda", generator=_generator(seed, 1))
    half = 0.5 * LINK_EPS * _gellmann().reshape(8, 9)
    U = torch.empty((n, 3, 3), dtype=torch.complex128, device="cuda")
    for i in range(0, n, 1 << 19):
        U[i:i + (1 << 19)] = _expi((r[i:i + (1 << 19)].to(torch.complex128) @ half).reshape(-1, 3, 3))
    return U.reshape(-1, 4, 3, 3)


def _field(dims, seed, stream, n=None):
    shape = (math.prod(dims), 4, 8) if n is None else (n, math.prod(dims), 4, 8)
    return torch.randn(shape, dtype=torch.float64, device="cuda", generator=_generator(seed, stream))


def _edges(nwin):
    """Equal windows over the band that holds the modes of these links; nearer 0 and 1 a window's trace is down to
    1e-7 of the total, and the power per mode there would be a ratio of rounding errors in float32."""
    return np.linspace(0.125, 0.875, nwin + 1)


def prepare(case, seed):
    dims, kind = _dims(case), case["kind"]
    s = {"case": case, "U": _links(dims, seed), "ctx": rm.Context(dims)}
    if kind in ("laplacian", "laplacian_grad"):
        dt = torch.float64 if case["prec"] == "fp64" else torch.float32
        X = _field(dims, seed, 2, case.get("nfield", 1)).to(dt)
        if kind == "laplacian":
            # repeated applications on one configuration: the links are imported once
            s.update(X=X, Y=torch.empty_like(X))
            rm.set_links(s["ctx"], s["U"])
        else:
            s.update(X=X[0].contiguous(), gY=_field(dims, seed, 3).to(dt))
    elif kind in ("kinetic", "mass_solve", "heatbath"):
        s.update(P=_field(dims, seed, 2), mass=rm.mass_fit(NPOLE, KAPPA))
        rm.set_links(s["ctx"], s["U"])
    elif kind == "spectrum":
        s.update(F=_field(dims, seed, 2, case["nforce"]), noise=_field(dims, seed, 3, case["nnoise"]),
                 edges=_edges(case["nwin"]))
        rm.set_links(s["ctx"], s["U"])
    elif kind == "trajectory":
        s.update(P=torch.empty((math.prod(dims), 4, 8), dtype=torch.float64, device="cuda"),
                 params=rm.make_params(beta=BETA, mass=rm.mass_fit(NPOLE, KAPPA), tau=0.025 * case["nsteps"],
                                       nsteps=case["nsteps"], tol_md=3e-7, tol_h=1e-12, fp_tol=1e-6, fp_extra=4,
                                       maxiter=400, prec=rm.MIXED, seed=int(seed), traj_index=0, metropolis=False))
    return s


def run(state):
    case, ctx, U = state["case"], state["ctx"], state["U"]
    kind = case["kind"]
    if kind == "laplacian":
        prec = rm.FP64 if case["prec"] == "fp64" else rm.FP32
        return rm.lap_apply(ctx, None, state["X"], state["Y"], prec=prec, linkfmt=case["linkfmt"])
    if kind == "laplacian_grad":
        X = state["X"].detach().requires_grad_(True)
        omega = torch.zeros((ctx.V, 4, 8), dtype=torch.float64, device="cuda", requires_grad=True)
        fp64 = case["prec"] == "fp64"
        Y = rm.laplacian(ctx, U, X, omega, prec=rm.FP64 if fp64 else rm.FP32)
        Y.backward(state["gY"])
        return Y.detach(), X.grad, omega.grad if fp64 else omega.grad.float()
    if kind == "kinetic":
        fp64 = case["prec"] == "fp64"
        F, V, T = rm.kinetic_force(ctx, None, state["P"], state["mass"], tol=case["tol"],
                                   prec=rm.FP64 if fp64 else rm.MIXED)
        return (F, V, T) if fp64 else (F.float(), V.float(), np.float32(T))
    if kind == "mass_solve":
        return rm.rat_mass_solve(ctx, None, state["P"], state["mass"], tol=case["tol"], prec=rm.MIXED)[0]
    if kind == "heatbath":
        return rm.heatbath(ctx, None, state["P"], state["mass"], tol=case["tol"], prec=rm.MIXED)
    if kind == "gauge":
        fp64 = case["prec"] == "fp64"
        F, S, plaq = rm.gauge_force(ctx, U, BETA, case["c1"], prec=rm.FP64 if fp64 else rm.FP32)
        return F if fp64 else F.float(), S, plaq
    if kind == "spectrum":
        out = rm.cheb_filter_spectrum(ctx, None, state["F"], state["noise"], case["degree"], state["edges"], prec=rm.MIXED)
        return [a.astype(np.float32) for a in out]
    if kind == "flow":
        V = U.clone()   # the flow works in place, on a copy of the configuration
        E = rm.wilson_flow(ctx, V, 0.01, case["nsteps"])
        return V, E
    V = U.clone()       # the chain's configuration moves in place
    r = rm.rmhmc_trajectory(ctx, V, state["params"], P_out=state["P"])
    return V.to(torch.complex64), state["P"].float(), [r["T0"], r["S0"]], np.float32([r["T1"], r["S1"], r["plaq"]])


# ------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------------
def work(case):
    """Inputs once and outputs once, as they are held, and the operations of the needed applications of the operator (8 hops of 4
    su(3) elements per site and field, 108 multiply-adds each) or of the staples (3x3 complex products)."""
    V, kind = math.prod(_dims(case)), case["kind"]
    hop = 2.0 * 8 * 4 * 108 * V
    links64, field64 = 4 * 144 * V, 256 * V
    if kind == "laplacian":
        real = 8 if case["prec"] == "fp64" else 4
        return {"bytes": V * real * (4 * case["linkfmt"] + 64 * case["nfield"]), "flops": hop * case["nfield"]}
    if kind == "laplacian_grad":
        real = 8 if case["prec"] == "fp64" else 4
        return {"bytes": links64 + V * real * 32 * 4 + field64, "flops": 2 * hop + 2.0 * 4 * 1400 * V}
    if kind == "kinetic":
        fp64 = case["prec"] == "fp64"
        return {"bytes": V * 4 * 18 * (8 if fp64 else 4) + 3 * field64, "flops": hop * CG_ITERS * (1.6 if fp64 else 1.0)}
    if kind in ("mass_solve", "heatbath"):
        return {"bytes": links64 + 2 * field64, "flops": hop * 2 * CG_ITERS}
    if kind == "gauge":
        per_link = 13 if case["c1"] == 0.0 else 43   # 3x3 products of a link's staples
        return {"bytes": links64 + field64, "flops": 2.0 * 108 * 4 * per_link * V}
    if kind == "spectrum":
        nf = case["nforce"] + case["nnoise"]
        return {"bytes": V * 4 * 72 + nf * field64, "flops": hop * nf * ((case["degree"] + 1) // 2)}
    if kind == "flow":
        return {"bytes": 2 * links64, "flops": 2.0 * case["nsteps"] * V * 4 * 3 * (13 * 108 + 450)}
    return {"bytes": 2 * links64 + field64, "flops": hop * CG_ITERS * 8 * 2 * case["nsteps"]}


# ------------------------------------------------------------------------------------------------
# the same in 64 bits, from the definitions
# ------------------------------------------------------------------------------------------------
class _Exact:
    """The adjoint operator A = -Delta/16 and its link derivative as plain torch in float64, from U X U^dag in
    coefficients, U T^b U^dag = sum_a R_ab T^a."""

    def __init__(self, dims, U):
        self.dims, self.U = dims, U
        self.T = 0.5 * _gellmann()
        V = math.prod(dims)
        self.R = torch.empty((4, V, 8, 8), dtype=torch.float64, device="cuda")
        for nu in range(4):
            for i in range(0, V, 1 << 17):
                u = U[i:i + (1 << 17), nu]
                for b in range(8):
                    m = _mul(_mul(u, self.T[b].expand_as(u)), u.conj().transpose(-1, -2))
                    self.R[nu, i:i + (1 << 17), :, b] = 2.0 * torch.einsum("aij,vji->va", self.T, m).real

    def shift(self, x, nu, n):
        """The field at x + n nu (n = +1, -1, ...)."""
        return torch.roll(x.reshape(self.dims[::-1] + x.shape[1:]), -n, 3 - nu).reshape(x.shape)

    def laplacian(self, X):
        h = torch.zeros_like(X)
        for nu in range(4):
            h += self.shift(X, nu, 1) @ self.R[nu].transpose(-1, -2)
            h += self.shift(X @ self.R[nu], nu, -1)
        return 0.5 * X - h / 16

    def link_grad(self, X, Z):
        """d<Z, A X>/dw: the hops across U_nu(y) are z.R x' + x.R z' (primes at y + nu) with
        dR/dw^a = -f_acd R_cb."""
        comm = torch.einsum("aij,cjk->acik", self.T, self.T)
        comm = comm - comm.transpose(0, 1)
        f = (-2j * torch.einsum("acij,dji->acd", comm, self.T)).real
        G = torch.empty_like(X)
        for nu in range(4):
            Rx = self.shift(X, nu, 1) @ self.R[nu].transpose(-1, -2)
            Rz = self.shift(Z, nu, 1) @ self.R[nu].transpose(-1, -2)
            C = torch.einsum("vmc,vmd->vcd", Rx, Z) + torch.einsum("vmc,vmd->vcd", Rz, X)
            G[:, nu] = (C.reshape(-1, 64) @ f.permute(1, 2, 0).reshape(64, 8)) / 16
        return G

    def function(self, b, fun, steps=60):
        """fun(A) b by the Lanczos method."""
        n = min(steps, b.numel())
        beta0 = float(b.norm())
        Q, d, e = torch.empty((n, b.numel()), dtype=torch.float64, device="cuda"), [], []
        Q[0] = b.reshape(-1) / beta0
        for k in range(n):
            w = self.laplacian(Q[k].reshape(b.shape)).reshape(-1)
            d.append(float(w @ Q[k]))
            w = w - Q[:k + 1].T @ (Q[:k + 1] @ w)
            w = w - Q[:k + 1].T @ (Q[:k + 1] @ w)
            nrm = float(w.norm())
            if k + 1 == n or nrm < 1e-13:
                break
            e.append(nrm)
            Q[k + 1] = w / nrm
        lam, S = np.linalg.eigh(np.diag(d) + np.diag(e, 1) + np.diag(e, -1))
        c = torch.from_numpy(S @ (fun(lam) * S[0]) * beta0).cuda()
        return (Q[:len(d)].T @ c).reshape(b.shape)

    def loops(self, mu, c1):
        """Sum of the loops that start with U_mu(x): plaquettes (1 - 8 c1) and 1x2 rectangles (c1)."""
        def path(steps):
            out = None
            at = [0, 0, 0, 0]
            for d, sign in steps:   # move one step along +-d, multiplying by the link passed (or its adjoint)
                if sign < 0:
                    at[d] -= 1
                u = self.U[:, d]
                for q in range(4):
                    if at[q]:
                        u = self.shift(u, q, at[q])
                if sign > 0:
                    at[d] += 1
                else:
                    u = u.conj().transpose(-1, -2)
                out = u if out is None else _mul(out, u)
            return out
        c0 = 1.0 - 8.0 * c1
        total = 0.0
        for nu in range(4):
            if nu == mu:
                continue
            for s in (1, -1):
                m, b = (mu, 1), (mu, -1)
                n, r = (nu, s), (nu, -s)
                rest = [(c0, (n, b, r))]
                if c1:
                    rest += [(c1, (m, n, b, b, r)), (c1, (n, b, b, r, m)), (c1, (n, n, b, r, r))]
                for w, steps in rest:
                    total = total + w * path(((mu, 1),) + steps)
        return total

    def gauge(self, beta, c1):
        """Force, action and average plaquette."""
        F, plaq, rect = [], 0.0, 0.0
        for mu in range(4):
            M = self.loops(mu, 0.0)
            F.append(M)
            plaq += float(torch.einsum("vii->v", M).real.sum()) / 3
        full = [self.loops(mu, c1) for mu in range(4)] if c1 else F
        V = len(self.U)
        nplaq = plaq / 4            # every plaquette holds four links
        if c1:
            for mu in range(4):
                rect += (float(torch.einsum("vii->v", full[mu]).real.sum()) / 3
                         - (1 - 8 * c1) * float(torch.einsum("vii->v", F[mu]).real.sum()) / 3) / c1
        nrect = rect / 6            # every rectangle holds six
        S = beta * ((1 - 8 * c1) * (6 * V - nplaq) + (c1 * (12 * V - nrect) if c1 else 0.0))
        force = torch.stack([beta / 3 * (1j * torch.einsum("aij,vji->va", self.T, m)).real for m in full], 1)
        return force, S, nplaq / (6 * V)


def _windows(edges, degree):
    """Chebyshev coefficients of the windows' indicators with Jackson's damping."""
    k = np.arange(1, degree + 1)
    th = np.arccos(np.clip(2 * np.asarray(edges) - 1, -1, 1))
    C = np.empty((len(edges) - 1, degree + 1))
    C[:, 0] = (th[:-1] - th[1:]) / np.pi
    C[:, 1:] = 2 * (np.sin(np.outer(th[:-1], k)) - np.sin(np.outer(th[1:], k))) / (np.pi * k)
    q, j = np.pi / (degree + 1), np.arange(degree + 1)
    return C * ((degree - j + 1) * np.cos(q * j) + np.sin(q * j) / np.tan(q)) / (degree + 1)


def exact(case, seed):
    dims, kind = _dims(case), case["kind"]
    if kind == "trajectory":
        return None     # the float64 molecular dynamics takes minutes in plain torch
    U = _links(dims, seed)
    if kind == "flow":
        E, t = [], _Exact.__new__(_Exact)
        t.dims, t.T = dims, 0.5 * _gellmann()

        def measure(V):
            t.U = V
            F, _, plaq = t.gauge(1.0, 0.0)
            return 6.0 * F, 36 * (1 - plaq)

        def turn(Z, V):
            h = torch.einsum("vma,aij->vmij", Z.to(torch.complex128), t.T)
            return _mul(_expi(h), V)
        for _ in range(case["nsteps"]):
            Z0, e = measure(U)
            E.append(e)
            W = turn(0.01 / 4 * Z0, U)
            Z1 = measure(W)[0]
            W = turn(0.01 * (8 / 9 * Z1 - 17 / 36 * Z0), W)
            Z2 = measure(W)[0]
            U = turn(0.01 * (0.75 * Z2 - 8 / 9 * Z1 + 17 / 36 * Z0), W)
        return U, np.array(E + [measure(U)[1]])
    if kind == "gauge":
        t = _Exact.__new__(_Exact)
        t.dims, t.U, t.T = dims, U, 0.5 * _gellmann()
        return t.gauge(BETA, case["c1"])
    op = _Exact(dims, U)
    mass = lambda lam: (1 - KAPPA) + KAPPA * lam  # noqa: E731
    if kind == "laplacian":
        dt = torch.float64 if case["prec"] == "fp64" else torch.float32
        X = _field(dims, seed, 2, case["nfield"])
        return torch.stack([op.laplacian(X[f].to(dt).double()) for f in range(case["nfield"])])
    if kind == "laplacian_grad":
        dt = torch.float64 if case["prec"] == "fp64" else torch.float32
        X, gY = (_field(dims, seed, 2, 1)[0].to(dt).double(), _field(dims, seed, 3).to(dt).double())
        return op.laplacian(X), op.laplacian(gY), op.link_grad(X, gY)
    if kind == "spectrum":
        G = torch.cat([_field(dims, seed, 2, case["nforce"]), _field(dims, seed, 3, case["nnoise"])])
        mom = np.empty((len(G), case["degree"] + 1))
        n = len(G)
        g = G.permute(1, 0, 2, 3).reshape(-1, 4 * n, 8).contiguous()   # all fields at once

        def dot(x, y):
            return (x * y).reshape(-1, n, 32).sum((0, 2)).cpu().numpy()
        a, b = g, 2 * op.laplacian(g) - g
        mom[:, 0], mom[:, 1] = dot(g, g), dot(g, b)
        for k in range(2, case["degree"] + 1):
            a, b = b, 2 * (2 * op.laplacian(b) - b) - a
            mom[:, k] = dot(g, b)
        p = mom @ _windows(_edges(case["nwin"]), case["degree"]).T
        num, tr = p[:case["nforce"]], p[case["nforce"]:].mean(0)
        return num / tr, num, tr, mom
    P = _field(dims, seed, 2)
    if kind == "kinetic":
        # R(A)^2 = 1/m(A): V = m(A)^{-1} P, T = <P, V>/2, F = (kappa/2) d<V, A V>/dw
        V = op.function(P, lambda lam: 1 / mass(lam))
        return 0.5 * KAPPA * op.link_grad(V, V), V, 0.5 * float((P * V).sum())
    if kind == "mass_solve":
        return op.function(P, lambda lam: mass(lam) ** -0.5)
    return op.function(P, lambda lam: mass(lam) ** 0.5)
