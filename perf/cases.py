"""The work that a user of this framework has it do, as cases that can be timed.

A case is one call sequence through the public binding: short time-step runs
(state in, a number of steps, state out) of each radial formulation, time scheme
and precision, a batch of uneven runs in one graph, a gradient by the adjoint,
and the explicit terms alone.  Initial states lie on the device; a run starts
from the same state each time, so its outputs do not depend on how often it ran.

``exact`` evaluates the same discrete equations in FP64 with dense torch algebra
(Gastine, pizza, GJI 2019: Sections 2, 3 and 4), independent of the library.
"""
import math
from math import comb

import numpy as np
import torch

from paper_1902_07092_gb300 import binding as B

ETA, PR = 0.35, 1.0
# critical Rayleigh numbers at Pr = 1, radius ratio 0.35 (log E, log Ra_c)
RA_C = [(1e-8, 6.16039e10), (1e-6, 1.69806e8), (1e-5, 9.95658e6), (1e-4, 6.65743e5), (1e-3, 5.48836e4)]


def ra_critical(E):
    x, y = zip(*[(math.log(e), math.log(r)) for e, r in RA_C])
    return math.exp(float(np.interp(math.log(E), x, y)))


def step_case(name, n_r, n_phi, E, scheme, steps, ra=10.0, radial="integration", mixed=False, **kw):
    c = {"name": name, "do": "steps", "n_r": n_r, "n_phi": n_phi, "E": E, "ra": ra, "scheme": scheme,
         "steps": steps, "radial": radial, "mixed": mixed, "pumping": 0.0, "buoyancy": False}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest runs of the tests and of the benchmark: launches and latency count
        step_case("tau_n33_p96_cnab2", 33, 96, 1e-3, "CNAB2", 20, ra=2.0),
        # the collocation formulation, as in the benchmark's small workload and the onset studies
        step_case("coll_n65_p192_cnab2", 65, 192, 1e-4, "CNAB2", 20, radial="collocation"),
        # an ordinary parameter-study run with Ekman pumping, multistep
        step_case("tau_n129_p384_sbdf3_pump", 129, 384, 1e-4, "SBDF3", 16, pumping=3e-3),
        # the medium workload: E = 1e-5, Ra = 10 Ra_c, third-order DIRK
        step_case("tau_n257_p768_ars443", 257, 768, 1e-5, "ARS443", 6),
        # the same in mixed precision
        step_case("mixed_n257_p768_ars443", 257, 768, 1e-5, "ARS443", 6, mixed=True),
        # the same in the Galerkin bases, with the cheaper third-order scheme
        step_case("galerkin_n257_p768_bpr353", 257, 768, 1e-5, "BPR353", 6, radial="galerkin"),
        # implicit buoyancy on a grid with few azimuthal modes
        step_case("tau_n513_p384_sbdf2_buoy", 513, 384, 1e-6, "SBDF2", 8, buoyancy=True),
        # a parameter study: uneven independent runs in one graph
        {"name": "batch_8_runs_cnab2", "do": "batch", "runs": 8, "steps": 10},
        # a gradient of the time-averaged Nusselt number: forward steps and their adjoint
        {"name": "adjoint_n129_p384", "do": "adjoint", "n_r": 129, "n_phi": 384, "E": 1e-4, "ra": 5.0,
         "steps": 10, "every": 5},
        # a high-resolution run
        step_case("tau_n1025_p3072_sbdf2", 1025, 3072, 1e-7, "SBDF2", 4),
        # the explicit terms alone (transforms and products) at the largest size
        {"name": "explicit_n2049_p6144", "do": "explicit", "n_r": 2049, "n_phi": 6144, "E": 1e-8, "ra": 20.0,
         "mixed": False},
        # the largest workload: E = 1e-8, Ra = 20 Ra_c, SBDF3
        step_case("tau_n2049_p6144_sbdf3", 2049, 6144, 1e-8, "SBDF3", 5, ra=20.0),
    ]


def draw(rng):
    do = rng.choice(["steps"] * 7 + ["batch", "adjoint", "explicit"])
    if do == "batch":
        return {"do": "batch", "runs": rng.randint(3, 12), "steps": rng.randint(4, 20)}
    if do == "adjoint":
        return {"do": "adjoint", "n_r": 2 ** rng.randint(4, 7) + 1, "n_phi": 3 * 2 ** rng.randint(4, 7),
                "E": 10 ** rng.uniform(-5, -3), "ra": rng.uniform(1.5, 10.0), "steps": rng.randint(3, 16),
                "every": rng.randint(1, 8)}
    n_r = 2 ** rng.randint(5, 10) + 1
    n_phi = 3 * 2 ** rng.randint(5, 10)
    E = 10 ** rng.uniform(-7, -3)
    ra = rng.uniform(1.5, 20.0)
    if do == "explicit":
        return {"do": "explicit", "n_r": n_r, "n_phi": n_phi, "E": E, "ra": ra, "mixed": False}
    radial = rng.choice(["integration"] * 4 + ["galerkin", "collocation"])
    if radial == "collocation":  # dense systems: the formulation's smaller grids
        n_r, n_phi = min(n_r, 129), min(n_phi, 384)
    elif radial == "galerkin":
        n_r = min(n_r, 257)
    scheme = rng.choice(["CNAB2", "SBDF2", "SBDF3", "ARS443", "BPR353"])
    mixed = radial == "integration" and rng.random() < 0.2
    return {"do": "steps", "n_r": n_r, "n_phi": n_phi, "E": E, "ra": ra, "scheme": scheme,
            "steps": rng.randint(3, 12 if n_r * n_phi < 400000 else 4), "radial": radial, "mixed": mixed,
            "pumping": 3e-3 if radial == "integration" and rng.random() < 0.25 else 0.0,
            "buoyancy": rng.random() < 0.25}


# ---------------------------------------------------------------- inputs -----
def batch_members(case):
    """Uneven members of a parameter study: sizes, E and Ra spread over their ranges."""
    sizes = [(65, 192), (129, 768), (257, 384), (65, 1536), (513, 192), (129, 384), (257, 768), (65, 384),
             (129, 192), (513, 384), (257, 192), (65, 768)]
    out = []
    for i in range(case["runs"]):
        n_r, n_phi = sizes[i % len(sizes)]
        out.append({"n_r": n_r, "n_phi": n_phi, "E": 10 ** (-4.0 - 2.0 * ((5 * i) % 12) / 12),
                    "ra": 1.5 + 1.5 * ((7 * i) % 12), "scheme": "CNAB2", "radial": "integration", "mixed": False,
                    "pumping": 0.0, "buoyancy": False, "steps": case["steps"]})
    return out


def params(c):
    dt = 0.01 * c["E"]
    return {"Ra": c["ra"] * ra_critical(c["E"]), "dt": dt}


def n_coeffs(c):
    return c["n_r"] if c.get("radial") == "collocation" else 2 * (c["n_r"] - 1) // 3


def initial_state(c, seed, member=0):
    """Smooth random fields with decaying Chebyshev and azimuthal spectra that meet
    the wall conditions: theta and u_bar vanish at the walls, the streamfunction
    carries the factor (1 - x^2)^2.  Coefficients f_hat (complex128 [M][n_c])."""
    n_r, M, nc = c["n_r"], c["n_phi"] // 3 + 1, n_coeffs(c)
    g = torch.Generator().manual_seed(1009 * int(seed) + member)
    n = min(nc - 8, 40)
    decay = 1.0 / (1.0 + torch.arange(n, dtype=torch.float64)) ** 2
    modes = 1.0 / (1.0 + torch.arange(M, dtype=torch.float64) / 8.0)

    def field(amp, factor, rows):
        a = torch.randn(rows, n, 2, generator=g, dtype=torch.float64) * decay[:, None]
        a = torch.view_as_complex(a.contiguous()) * (amp * modes[:rows, None])
        out = torch.zeros(rows, nc, dtype=torch.complex128)
        for k, f in enumerate(factor):  # times sum_k f_k T_k, folded into k + n and |k - n|
            if f:
                idx = torch.arange(n)
                out.index_add_(1, idx + k, 0.5 * f * a)
                out.index_add_(1, (idx - k).abs(), 0.5 * f * a)
        C = math.sqrt(2.0 / (n_r - 1))
        w = torch.full((nc,), C, dtype=torch.float64)
        w[0] *= 0.5
        if nc == n_r:
            w[-1] *= 0.5
        return out / w

    theta = field(1e-3, [0.5, 0.0, -0.5], M)                      # 1 - x^2
    psi = field(1e-2, [0.375, 0.0, -0.5, 0.0, 0.125], M)          # (1 - x^2)^2
    u = field(1e-1, [0.5, 0.0, -0.5], 1)[0].real.contiguous()
    theta[0] = theta[0].real.to(torch.complex128)
    psi[0] = 0.0
    return theta, psi, u


class Member:
    """One solver, its initial state and the buffers its results go to."""

    def __init__(self, c, seed, member=0):
        p = params(c)
        self.c = c
        self.s = B.Solver(c["n_r"], c["n_phi"], c["E"], p["Ra"], PR, ETA, c.get("scheme", "CNAB2"), p["dt"],
                          radial=c.get("radial", "integration"), pumping_eps=c.get("pumping") or None,
                          buoy_implicit=c.get("buoyancy", False))
        if c.get("mixed"):
            B.pizza_set_option(self.s.ctx, "precision", 1)
        self.state = [t.cuda() for t in initial_state(c, seed, member)]
        self.out = [torch.zeros_like(t) for t in self.state]

    def begin(self):
        B.pizza_set_state(self.s.ctx, *self.state, self.s.n_c)

    def end(self):
        B.pizza_get_state(self.s.ctx, *self.out)
        return dict(zip(("theta", "psi", "u"), self.out))

    def warm(self):
        """Builds the factored operators (kept by the solver, as in a long run)."""
        self.begin()
        self.s.step(1)
        B.pizza_synchronize(self.s.ctx)


def prepare(case, seed):
    if case["do"] == "batch":
        ms = [Member(c, seed, i) for i, c in enumerate(batch_members(case))]
        for m in ms:
            m.warm()
        return {"case": case, "members": ms, "batch": B.Batch([m.s for m in ms])}
    m = Member(case, seed)
    state = {"case": case, "member": m}
    if case["do"] == "steps":
        m.warm()
    elif case["do"] == "explicit":
        m.begin()
    elif case["do"] == "adjoint":
        m.begin()
        m.s.tape_begin(case["every"])
        w = m.s.nusselt_weights() / case["steps"]
        g = torch.zeros_like(m.state[0])
        g[0] = torch.from_numpy(w).cuda().to(torch.complex128)
        state["g"] = g
        torch.cuda.synchronize()
    return state


# ------------------------------------------------------------------ runs -----
def run(state):
    case = state["case"]
    if case["do"] == "batch":
        for m in state["members"]:
            m.begin()
        state["batch"].step(case["steps"])
        return [m.end() for m in state["members"]]
    m = state["member"]
    if case["do"] == "steps":
        m.begin()
        m.s.step(case["steps"])
        return m.end()
    if case["do"] == "explicit":
        e_theta, e_psi, e_u = m.out
        B.pizza_explicit_terms(m.s.ctx, e_psi, e_theta, e_u)
        return {"e_theta": e_theta, "e_psi": e_psi, "e_u": e_u}
    # gradient of J = (1/K) sum_n (Nu_n - 1) in the initial state and Ra
    K = case["steps"]
    m.begin()
    m.s.tape_begin(case["every"])
    m.s.nusselt_begin()
    m.s.step(K)
    total, _ = m.s.nusselt_end()
    for k in range(K):
        dRa = m.s.adjoint_step(g_theta=state["g"], want_dRa=(k == K - 1))
    theta_bar, psi_bar, u_bar = m.out
    B.pizza_get_adjoint(m.s.ctx, theta_bar, psi_bar, u_bar)
    return {"J": total / K, "dRa": dRa, "theta": theta_bar, "psi": psi_bar, "u": u_bar}


# ------------------------------------------------------------------ work -----
def work(case):
    if case["do"] == "batch":
        ws = [work(dict(c, do="steps")) for c in batch_members(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    n_r, n_phi, nc = case["n_r"], case["n_phi"], n_coeffs(case)
    K, M, coll = n_r - 1, n_phi // 3 + 1, case.get("radial") == "collocation"
    dct, fft = 5.0 * K * math.log2(K), 5.0 * n_phi * math.log2(n_phi)
    band = lambda h: 4.0 * (2 * h + 1) * nc  # noqa: E731
    explicit = M * ((6 if coll else 10) * dct + 70.0 * n_r) + n_r * (4 * fft + 8.0 * n_phi)
    if not coll:
        explicit += M * (band(8) + 2 * band(4))
    state = 32.0 * M * nc + 8.0 * nc
    if case["do"] == "explicit":
        return {"bytes": 2 * state, "flops": explicit}
    if coll:
        solve = M * 20.0 * n_r * (n_r - 2)
        factors = M * 40.0 * n_r * (n_r - 2)
    else:
        solve = M * nc * (8.0 * 33 + 4.0 * 17 + 4.0 * 17 * 2 + 4.0 * 9)  # band sweeps, mass terms
        factors = M * nc * (16.0 * 33 + 8.0 * 17)                         # bordered band LU, read once
    n_exp, n_sol, terms = {"CNAB2": (1, 1, 6), "SBDF2": (1, 1, 6), "SBDF3": (1, 1, 8), "ARS443": (4, 4, 6),
                           "BPR353": (3, 4, 6)}[case.get("scheme", "CNAB2")]
    steps = case["steps"]
    per_flops = n_exp * explicit + n_sol * solve
    per_bytes = n_exp * 2 * state + n_sol * (factors + terms * state)
    if case["do"] == "adjoint":  # each step forward, once more from its checkpoint, and its transpose
        return {"bytes": steps * (3 * per_bytes), "flops": steps * (3 * per_flops + explicit)}
    return {"bytes": steps * per_bytes + 2 * state, "flops": steps * per_flops}


# ----------------------------------------------------------------- exact -----
def rmul(A, X):
    """X A^T for a real matrix A and a complex or real batch X (vectors in the last axis)."""
    if X.is_complex():
        return torch.complex(X.real @ A.T, X.imag @ A.T)
    return X @ A.T


class Dense:
    """The discrete equations with dense FP64 matrices, modes in the first axis."""

    def __init__(self, c):
        self.c, p = c, params(c)
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.Ra, self.dt, self.E = p["Ra"], p["dt"], c["E"]
        self.n_r, self.n_phi, self.nc = c["n_r"], c["n_phi"], n_coeffs(c)
        self.M, self.coll = self.n_phi // 3 + 1, c.get("radial") == "collocation"
        self.buoy, self.eps = c.get("buoyancy", False), c.get("pumping") or 0.0
        n_r, K, nc = self.n_r, self.n_r - 1, self.nc
        self.s_o = 1.0 / (1.0 - ETA)
        a, b = 0.5, 0.5 * (self.s_o + ETA / (1.0 - ETA))
        r = math.sqrt(1.0 - ETA * ETA)
        self.tc = ETA / (1.0 - ETA) * (math.asinh(r / ETA) / r - 1.0) / math.log(ETA)
        cosines = np.cos(np.pi * np.arange(2 * K) / K)
        k = np.arange(n_r)
        T = cosines[np.outer(k, k) % (2 * K)]
        s = a * T[:, 1] + b
        ends = np.ones(n_r)
        ends[[0, -1]] = 0.5
        C = math.sqrt(2.0 / K)
        D = np.triu(2.0 * k[None, :] * ((k[None, :] + k[:, None]) % 2)) / a  # d/ds of plain coefficients
        D[0] *= 0.5
        self.scale = (C * ends)[:nc]
        to = lambda x: torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64, device=self.dev)  # noqa: E731
        self.to = to
        T_, D_ = to(T), to(D)
        TD = T_ @ D_
        self.T0, self.T1, self.T2 = (X[:, :nc] * to(self.scale) for X in (T_, TD, TD @ D_))
        self.icheb = C * T_ * to(ends)
        self.ddr = TD @ (to(C * ends)[:, None] * self.icheb)
        self.s, self.h2 = to(s), to(self.s_o ** 2 - s ** 2)
        self.m = torch.arange(self.M, dtype=torch.float64, device=self.dev)[:, None]
        n = np.arange(nc, dtype=np.float64)
        sg = (-1.0) ** n
        self.bc = {"o": n ** 0, "i": sg, "no": n ** 2, "ni": -sg * n ** 2, "d3": n ** 2 * (n ** 2 - 1) * (n ** 2 - 4)}
        self.bc = {q: to(v * self.scale) for q, v in self.bc.items()}
        self.factors = {}
        if self.coll:
            self.build_collocation()
        else:
            self.build_integration(a, b)

    # ---- Chebyshev integration (Section 3.2): q-fold integrals of polynomial x derivative terms
    def build_integration(self, a, b):
        nc, n = self.nc, self.nc + 40
        X, J = np.zeros((n, n)), np.zeros((n, n))
        for i in range(n):
            if i + 1 < n:
                X[i + 1, i] += 0.5 if i else 1.0
                J[i + 1, i] = (1.0 / (2 * (i + 1)) if i else 1.0) * a
            if i:
                X[i - 1, i] += 0.5
            if i > 1:
                J[i - 1, i] = -a / (2 * (i - 1))
        S, J = self.to(a * X + b * np.eye(n)), self.to(J)
        pows = [torch.eye(n, dtype=torch.float64, device=self.dev)]
        for _ in range(8):
            pows.append(S @ pows[-1])
        Jp = [pows[0]]
        for _ in range(4):
            Jp.append(J @ Jp[-1])
        P = np.polynomial.Polynomial

        def integrated(terms, q):
            out = torch.zeros(n, n, dtype=torch.float64, device=self.dev)
            for p, poly in terms.items():
                for j in range(p + 1):
                    d = poly.deriv(j) if j else poly
                    R = sum(float(x) * pows[i] for i, x in enumerate(d.coef) if x)
                    if not isinstance(R, int):
                        out += (-1) ** j * comb(p, j) * (Jp[q - p + j] @ R)
            out = out[:nc, :nc] * self.to(self.scale)
            out[:q] = 0.0
            return out

        so2, s1 = self.s_o ** 2, P([0.0, 1.0])

        # s^2 L_I = p2 D^2 + p1 D + p00 + m^2 p01
        p2, p1, p00, p01 = P([0, 0, so2, 0, -1.0]), P([0, so2, 0, -6.0]), P([0, 0, -6.0]), P([-so2, 0, 1.0])

        def lap(q2, q1, q0):  # s^4 (d^2/ds^2 + (1/s) d/ds) s^-2 f = s^2 f'' - 3 s f' + 4 f, f = (q2 D^2 + q1 D + q0) Psi
            f0 = {2: q2, 1: q1, 0: q0}
            f1 = {3: q2, 2: q2.deriv() + q1, 1: q1.deriv() + q0, 0: q0.deriv()}
            f2 = {4: q2, 3: 2 * q2.deriv() + q1, 2: q2.deriv(2) + 2 * q1.deriv() + q0,
                  1: q1.deriv(2) + 2 * q0.deriv(), 0: q0.deriv(2)}
            z = P([0.0])
            return {p: s1 ** 2 * f2.get(p, z) - 3 * s1 * f1.get(p, z) + 4 * f0.get(p, z) for p in range(5)}

        self.C = integrated({0: s1 ** 4}, 4)
        self.D = integrated({0: s1 ** 2}, 2)
        self.G = integrated({0: P([so2, 0, -1.0])}, 2)
        if self.c["do"] == "explicit":
            return
        self.A0 = integrated({2: s1 ** 2 * p2, 1: s1 ** 2 * p1, 0: s1 ** 2 * p00}, 4)
        self.A2 = integrated({0: s1 ** 2 * p01}, 4)
        z = P([0.0])
        self.B0 = integrated(lap(p2, p1, p00), 4)
        b2 = lap(z, z, p01)  # and the -m^2 of the Laplacian on the m^0 part
        for p, q in ((2, p2), (1, p1), (0, p00)):
            b2[p] = b2[p] - q
        self.B2 = integrated(b2, 4)
        self.B4 = integrated({0: -1.0 * p01}, 4)
        self.F0 = integrated({2: s1 ** 2, 1: s1}, 2)
        self.F2 = integrated({0: P([-1.0])}, 2)
        self.Ez = integrated({2: s1 ** 2, 1: s1, 0: P([-1.0])}, 2)

    def products(self, v, up, om, th):
        f = [x.clone() for x in (v, up, om, th)]
        for x in f:
            x[0] = x[0].real.to(x.dtype)
        v, up, om, th = (torch.fft.irfft(x, n=self.n_phi, dim=0) * self.n_phi for x in f)
        return (torch.fft.rfft(x, dim=0)[:self.M] / self.n_phi for x in (v * om, up * om, v * th, up * th))

    def explicit(self, y):
        if self.coll:
            return self.explicit_collocation(y)
        psi, th, u = y
        im, s, h2, mu = 1j * self.m, self.s, self.h2, self.m ** 2
        g0, g1, g2 = (rmul(T, psi) for T in (self.T0, self.T1, self.T2))
        ub, dub = rmul(self.T0, u), rmul(self.T1, u)
        first = (self.m == 0)
        v = im * g0
        up = torch.where(first, ub[None].to(g0.dtype), -h2 * g1 + 3 * s * g0)
        om = torch.where(first, (dub + ub / s)[None].to(g0.dtype),
                         -(h2 * g2 + (h2 / s - 5 * s) * g1 - (6 + mu * h2 / s ** 2) * g0))
        vw, uw, vt, ut = self.products(v, up, om, rmul(self.T0, th))
        Nw = (rmul(self.ddr, h2 * vw) + im * uw) / s
        Nt = (rmul(self.ddr, h2 * vt) + im * ut) / s - vt
        Nu = (h2 / s) * vw[0].real
        if self.eps:  # Eq. approx_pump and the zonal-flow terms
            he2 = (self.s_o + self.eps) ** 2 - s ** 2
            ups = math.sqrt(self.s_o / self.E) / he2 ** 0.75
            Nw = Nw - ups * (-om + 0.5 * s * g1 - (1.5 * s ** 2 / he2 + mu + im * 2.5 * self.s_o / he2.sqrt()) * g0)
            Nu = Nu + ups * ub * (1 + 0.5 * self.E * (dub + ub / s))
        nc = self.nc
        hat = rmul(self.icheb, Nw)[:, :nc]
        if not self.buoy:
            hat = hat + (self.Ra / PR / self.s_o) * im * th
        e_psi = torch.where(first, torch.zeros_like(hat), rmul(self.C, hat))
        e_th = -rmul(self.D, rmul(self.icheb, Nt)[:, :nc]) - self.tc * im * rmul(self.G, psi)
        return e_psi, e_th, -rmul(self.D, rmul(self.icheb, Nu)[:nc])

    def mass(self, y):
        if self.coll:
            return tuple(rmul(self.T0, x) for x in y)
        psi, th, u = y
        return rmul(self.A0, psi) + self.m ** 2 * rmul(self.A2, psi), rmul(self.D, th), rmul(self.D, u)

    def buoyancy(self, th):
        return (self.Ra / PR / self.s_o) * 1j * self.m * (rmul(self.T0, th) * -1.0 if self.coll else rmul(self.C, th))

    def imp(self, y):
        if self.coll:
            return self.imp_collocation(y)
        psi, th, u = y
        mu = self.m ** 2
        ip = (rmul(self.B0, psi) + mu * rmul(self.B2, psi) + mu ** 2 * rmul(self.B4, psi)
              + (2j / self.E) * self.m * rmul(self.C, psi))
        if self.buoy:
            ip = ip + self.buoyancy(th)
        return ip, (rmul(self.F0, th) + mu * rmul(self.F2, th)) / PR, rmul(self.Ez, u)

    def solver(self, L):
        """Row-scaled LU with one refinement step."""
        r = 1.0 / L.abs().amax(-1, keepdim=True)
        lu = torch.linalg.lu_factor(L * r)

        def solve(b):
            r1 = r[..., 0] * b
            x = torch.linalg.lu_solve(*lu, r1[..., None])
            res = r1[..., None] - (L * r) @ x
            return (x + torch.linalg.lu_solve(*lu, res))[..., 0]
        return solve

    def solve(self, gamma, rhs):
        if gamma not in self.factors:
            self.factors[gamma] = self.factor_collocation(gamma) if self.coll else self.factor(gamma)
        sp, st, su = self.factors[gamma]
        q = [1, 1, 1] if self.coll else [4, 2, 2]
        rp, rt, ru = (r.clone() for r in rhs)
        for r, n in zip((rp, rt, ru), q):
            r[..., :n] = 0.0
            if self.coll:
                r[..., -1] = 0.0
        th = st(rt)
        if self.buoy:
            add = gamma * self.dt * self.buoyancy(th)
            add[..., :q[0]] = 0.0
            if self.coll:
                add[..., -1] = 0.0
            rp = rp + add
        u = su(ru)
        if self.coll:
            x = sp(torch.cat([rp, torch.zeros_like(rp)], -1))
            w, psi = x[..., :self.nc], x[..., self.nc:]
            return torch.where(self.m == 0, 0 * w, w), torch.where(self.m == 0, 0 * psi, psi), th, u
        psi = sp(rp)
        return torch.where(self.m == 0, torch.zeros_like(psi), psi), th, u

    def factor(self, gamma):
        g, mu = gamma * self.dt, (self.m ** 2)[..., None]
        L = (self.A0 + mu * self.A2) - g * (self.B0 + mu * self.B2 + mu ** 2 * self.B4)
        L = torch.complex(L, -g * (2.0 / self.E) * self.m[..., None] * self.C.expand_as(L))
        L[:, :4] = torch.stack([self.bc[q] for q in ("o", "i", "d3", "ni")]).to(L.dtype)
        Lt = (self.D - g * (self.F0 + mu * self.F2) / PR).to(L.dtype)
        Lu = self.D - g * self.Ez
        d = torch.stack([self.bc["o"], self.bc["i"]])
        Lt[:, :2] = d.to(L.dtype)
        Lu[:2] = d
        return self.solver(L), self.solver(Lt), self.solver(Lu)

    # ---- Chebyshev collocation (Section 3.1): state (omega, psi, theta, u_bar)
    def build_collocation(self):
        s, h2 = self.s, self.h2.clone()
        h2[0] = 1.0
        inner = torch.ones_like(s)
        inner[0] = 0.0
        self.beta = -inner * s / h2
        self.dbeta = -inner * (self.s_o ** 2 + s ** 2) / h2 ** 2
        self.Q = self.T2 + self.T1 / s[:, None]

    def LB(self):  # L_beta psi, per mode
        s, mu = self.s, (self.m ** 2)[..., None]
        base = self.T2 + (self.beta + 1 / s)[:, None] * self.T1 + (self.dbeta + self.beta / s)[:, None] * self.T0
        return base - mu * (self.T0 / (s ** 2)[:, None])

    def vorticity(self, psi):
        g = torch.einsum("mkn,mn->mk", self.LB().to(psi.dtype), psi)
        g[:, 0] = 1.25 * rmul(self.T2, psi)[:, 0]
        w = rmul(self.icheb, -g)
        w[0] = 0.0
        return w

    def explicit_collocation(self, y):
        w, psi, th, u = y
        im, s, first = 1j * self.m, self.s, self.m == 0
        g0, g1, W, TH = rmul(self.T0, psi), rmul(self.T1, psi), rmul(self.T0, w), rmul(self.T0, th)
        ub, dub = rmul(self.T0, u), rmul(self.T1, u)
        up = torch.where(first, ub[None].to(g0.dtype), -g1 - self.beta * g0)
        W = torch.where(first, (dub + ub / s)[None].to(g0.dtype), W)
        vw, uw, vt, ut = self.products(im * g0, up, W, TH)
        Nw = (rmul(self.ddr, vw) + im * uw) / s
        Nt = (rmul(self.ddr, vt) + im * ut) / s + self.beta * vt / s
        ew = -Nw if self.buoy else -Nw - (self.Ra / PR / self.s_o) * im * TH
        et = -im / s * (self.tc / s) * g0 - Nt
        eu = -(vw[0].real / s)
        ew = torch.where(first, torch.zeros_like(ew), ew)
        for e in (ew, et, eu):
            e[..., 0] = 0.0
            e[..., -1] = 0.0
        return ew, et, eu

    def imp_collocation(self, y):
        w, psi, th, u = y
        mu, s = self.m ** 2, self.s
        iw = rmul(self.Q, w) - mu / s ** 2 * rmul(self.T0, w) \
            + (2j / self.E) * self.m * (self.beta / s) * rmul(self.T0, psi)
        if self.buoy:
            iw = iw + self.buoyancy(th)
        iw = torch.where(self.m == 0, torch.zeros_like(iw), iw)
        it = (rmul(self.Q, th) - mu / s ** 2 * rmul(self.T0, th)) / PR
        return iw, it, rmul(self.Q, u) - rmul(self.T0, u) / s ** 2

    def factor_collocation(self, gamma):
        g, mu, N, s = gamma * self.dt, (self.m ** 2)[..., None], self.nc, self.s
        T0 = self.T0
        L = torch.zeros(self.M, 2 * N, 2 * N, dtype=torch.complex128, device=self.dev)
        L[:, :N, :N] = T0 - g * (self.Q - mu * (T0 / (s ** 2)[:, None]))
        L[:, :N, N:] = -g * (2j / self.E) * self.m[..., None] * ((self.beta / s)[:, None] * T0)
        L[:, N:, :N] = T0
        L[:, N:, N:] = self.LB()
        for row, q in ((0, "no"), (N - 1, "ni"), (N, "o"), (2 * N - 1, "i")):
            L[:, row] = 0.0
            L[:, row, N:] = self.bc[q].to(L.dtype)
        Lt = (T0 - g * (self.Q - mu * (T0 / (s ** 2)[:, None])) / PR).to(L.dtype)
        Lu = T0 - g * (self.Q - T0 / (s ** 2)[:, None])
        for X in (Lt, Lu):
            X[..., 0, :] = self.bc["o"].to(X.dtype)
            X[..., -1, :] = self.bc["i"].to(X.dtype)
        return self.solver(L), self.solver(Lt), self.solver(Lu)

    # ---- time schemes (Eqs. multistep1 and dirks), with the lower-order starters
    def steps(self, theta, psi, u, count, each=None):
        y = (psi, theta, u)
        mass_of = (lambda y: self.mass((y[0], y[2], y[3]))) if self.coll else self.mass
        if self.coll:
            y = (self.vorticity(psi),) + y
        ax = lambda acc, c, v: v if acc is None else tuple(p + c * q for p, q in zip(acc, v))  # noqa: E731
        sc = lambda c, v: tuple(c * q for q in v)  # noqa: E731
        scheme, dt = self.c.get("scheme", "CNAB2"), self.dt
        ms, es = [], []
        for n in range(count):
            if scheme in ("ARS443", "BPR353"):
                aI, aE = TABLEAUX[scheme]
                m0, E_, I_ = mass_of(y), [], []
                for i in range(1, 5):
                    E_.append(self.explicit(y))
                    I_.append(self.imp(y))
                    rhs = m0
                    for j in range(i):
                        rhs = ax(ax(rhs, dt * aE[i][j], E_[j]), dt * aI[i][j], I_[j])
                    y = self.solve(aI[i][i], rhs)
            else:
                ms, es = [mass_of(y)] + ms[:2], [self.explicit(y)] + es[:2]
                if scheme == "CNAB2":
                    a, b0, bE = [1.0], 0.5, [1.0] if n == 0 else [1.5, -0.5]
                else:
                    a, b0, bE = SBDF[min(n + 1, 2 if scheme == "SBDF2" else 3)]
                rhs = sc(a[0], ms[0])
                for c, v in zip(a[1:], ms[1:]):
                    rhs = ax(rhs, c, v)
                for c, v in zip(bE, es):
                    rhs = ax(rhs, dt * c, v)
                if scheme == "CNAB2":
                    rhs = ax(rhs, 0.5 * dt, self.imp(y))
                y = self.solve(b0, rhs)
            if each:
                each(y)
        psi, theta, u = y[-3:]
        return {"theta": theta, "psi": psi, "u": u}


SBDF = {1: ([1.0], 1.0, [1.0]), 2: ([4 / 3, -1 / 3], 2 / 3, [4 / 3, -2 / 3]),
        3: ([18 / 11, -9 / 11, 2 / 11], 6 / 11, [18 / 11, -18 / 11, 6 / 11])}
TABLEAUX = {
    "ARS443": ([[0], [0, 1 / 2], [0, 1 / 6, 1 / 2], [0, -1 / 2, 1 / 2, 1 / 2], [0, 3 / 2, -3 / 2, 1 / 2, 1 / 2]],
               [[0], [1 / 2], [11 / 18, 1 / 18], [5 / 6, -5 / 6, 1 / 2], [1 / 4, 7 / 4, 3 / 4, -7 / 4]]),
    "BPR353": ([[0], [1 / 2, 1 / 2], [5 / 18, -1 / 9, 1 / 2], [1 / 2, 0, 0, 1 / 2], [1 / 4, 0, 3 / 4, -1 / 2, 1 / 2]],
               [[0], [1], [4 / 9, 2 / 9], [1 / 4, 0, 3 / 4], [1 / 4, 0, 3 / 4, 0]]),
}


def exact(case, seed):
    if case["do"] == "batch":
        return [exact_steps(c, seed, i) for i, c in enumerate(batch_members(case))]
    if case["do"] == "steps":
        return exact_steps(case, seed)
    d = Dense(case)
    theta, psi, u = (t.to(d.dev) for t in initial_state(case, seed))
    if case["do"] == "explicit":
        e_psi, e_theta, e_u = d.explicit((psi, theta, u))
        return {"e_theta": e_theta, "e_psi": e_psi, "e_u": e_u}
    K, nc = case["steps"], d.nc
    n = torch.arange(nc, dtype=torch.float64, device=d.dev)
    w = n * n * d.to(d.scale) / 0.5 / (d.tc / d.s_o)  # (d theta_0/ds)/(dT_c/ds) at s_o
    leaves = [theta.requires_grad_(), psi.requires_grad_(), u.requires_grad_(),
              torch.tensor(d.Ra, dtype=torch.float64, device=d.dev, requires_grad=True)]
    d.Ra, nu = leaves[3], []
    d.steps(leaves[0], leaves[1], leaves[2], K, each=lambda y: nu.append((w * y[1][0].real).sum()))
    J = sum(nu) / K
    g = torch.autograd.grad(J, leaves)
    return {"J": float(J.detach()), "dRa": float(g[3]), "theta": g[0], "psi": g[1], "u": g[2]}


def exact_steps(c, seed, member=0):
    if c["n_r"] > 513 or (c["n_r"] > 257 and c["n_phi"] > 768):
        return None  # dense factorisations of every mode would take too long
    d = Dense(dict(c, do="steps"))
    theta, psi, u = (t.to(d.dev) for t in initial_state(c, seed, member))
    return d.steps(theta, psi, u, c["steps"])
