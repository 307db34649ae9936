"""The work that a user of this framework has it do, as cases that can be timed and compared.

The method's outer loops are four: time stepping (`step`, `step2`), Newton's method for a rotating
wave (`newton_rw`, alone and as a batch), the Jacobian action on its own (`apply_jacobian`, for
stability analysis) and the implicit solve on its own (`implicit_solve`); a new Ekman number
(continuation in Ek) adds the factorisation.  Each case is one such call on a context that the
program keeps.  Sizes are those of the repository's configurations (seeded_inputs.config: tiny, C1
to C5, M_s as in Table 1), of Table 1's own grids and of the odd truncations that refinement by
20 % produces.  Jacobian actions and solves are called on the FP64 path: on the mixed path they are
the inside of Newton's method, which the Newton cases run.

Shells are kept per case, as a program keeps them: states differ, the context does not.
"""
import cmath
import functools
import math

import numpy as np
import torch

DEV = "cuda"
ETA, PR = 0.35, 1.0


# ---- the cases --------------------------------------------------------------------------------
def _c(name, kind, L, Ms, Nr, Ek, Ra, precision, dt, count=1, tuned=False, coriolis="implicit"):
    return dict(name=name, kind=kind, L=L, Ms=Ms, Nr=Nr, Ek=Ek, Ra=Ra, precision=precision, dt=dt,
                count=count, tuned=tuned, coriolis=coriolis)


def listed():
    return [
        # a first look: one step per call at the smallest configuration (latency, launches)
        _c("tiny_step_mixed", "step", 7, 4, 10, 1e-3, 80.0, "mixed", 1e-4),
        # an interactive run at C1: ten steps, then the energy and Nusselt numbers are read
        _c("c1_monitor_fp64", "monitor", 31, 4, 24, 1e-3, 120.0, "fp64", 1e-4, count=10),
        # the second-order stepper on Table 1's second grid (no size a power of two)
        _c("rw8_step2_mixed", "step2", 52, 8, 60, 1e-4, 130.0, "mixed", 5e-5, count=4),
        # the implicit solve alone, odd sizes (backward-error checks, other explicit terms)
        _c("odd_solve_fp64", "solve", 45, 5, 37, 1e-4, 100.0, "fp64", 200.0),
        # two points of a continuation in Ek: each a new operator, factorised again, and a step
        _c("c2_new_ek_mixed", "new_ek", 63, 8, 48, 1e-4, 130.0, "mixed", 2e-5),
        # four waves of one branch solved together (rsc_batch_newton_rw), small
        _c("c1_batch_newton", "batch", 31, 4, 24, 1e-3, 120.0, "mixed", 2e-3, count=4, tuned=True),
        # time stepping at the benchmark's size, both precisions (a production run is tuned first)
        _c("c3_step_mixed", "step", 127, 12, 64, 1e-5, 140.0, "mixed", 5e-6, count=10, tuned=True),
        _c("c3_step_fp64", "step", 127, 12, 64, 1e-5, 140.0, "fp64", 5e-6, count=2, tuned=True),
        # Jacobian actions about one base state in FP64, as an eigenvalue solver asks for them
        _c("c3_jac_fp64", "jac", 127, 12, 64, 1e-5, 140.0, "fp64", 200.0, count=4, tuned=True),
        # the headline: a rotating wave converged by Newton from a time-stepped guess
        _c("c3_newton_mixed", "newton", 127, 12, 64, 1e-5, 140.0, "mixed", 2e-5, tuned=True),
        # the largest single instance, both precisions
        _c("c5_step_mixed", "step", 255, 8, 96, 3e-6, 241.0, "mixed", 2e-6, count=4, tuned=True),
        _c("c5_step_fp64", "step", 255, 8, 96, 3e-6, 241.0, "fp64", 2e-6, tuned=True),
    ]


def draw(rng):
    """Steps, second-order steps, FP64 Jacobian actions and FP64 solves over the whole range of
    truncations: L = 7..200 and N_r = 8..96 (odd ones among them), 2 to 32 active wavenumbers."""
    kind = rng.choice(["step", "step", "step", "step2", "jac", "jac", "solve", "new_ek"])
    L = int(round(math.exp(rng.uniform(math.log(7), math.log(200)))))
    nr_hi = min(96.0, 16.0 + 0.6 * L)
    Nr = max(8, int(round(math.exp(rng.uniform(math.log(8), math.log(nr_hi))))))
    Ms = rng.randint(max(1, -(-L // 31)), max(2, min(L, 16)))
    Ek = 10.0 ** rng.uniform(-5.0, -3.0)
    precision = "fp64" if kind in ("jac", "solve") else rng.choice(["fp64", "mixed", "mixed"])
    explicit = kind in ("step", "step2", "jac") and rng.random() < 0.15
    dt = 200.0 if kind in ("jac", "solve") else 0.1 * Ek
    count = rng.randint(1, 6) if kind in ("step", "step2", "jac") else 1
    c = _c("", kind, L, Ms, Nr, Ek, 6.0 * Ek ** (-1.0 / 3.0), precision, dt, count, L >= 96,
           "explicit" if explicit else "implicit")
    del c["name"]
    return c


# ---- inputs -----------------------------------------------------------------------------------
def _pairs(L, Ms):
    pl = [l for m in range(0, L + 1, Ms) for l in range(m, L + 1)]
    pm = [m for m in range(0, L + 1, Ms) for l in range(m, L + 1)]
    return pl, pm


def _noise(c, seed, amp, count=1, only_m=None):
    """Decaying Gaussian coefficients [count, n]: amp e^(-l/8) e^(-k/6) N(0, 1), the imaginary
    parts of m = 0 and the absent e_00, f_00 zero (the recipe of seeded_inputs)."""
    pl, pm = _pairs(c["L"], c["Ms"])
    P, Nr = len(pl), c["Nr"]
    g = torch.Generator().manual_seed(int(seed))
    z = torch.randn((count, 3, P, Nr, 2), dtype=torch.float64, generator=g).to(DEV)
    l, m = (torch.tensor(v, dtype=torch.float64, device=DEV) for v in (pl, pm))
    k = torch.arange(Nr, dtype=torch.float64, device=DEV)
    z *= amp * (torch.exp(-l / 8.0)[:, None] * torch.exp(-k / 6.0))[:, :, None]
    z[:, :, m == 0, :, 1] = 0.0
    z[:, 0:2, l == 0] = 0.0
    if only_m is not None:
        z[:, :, m != only_m] = 0.0
    return z.reshape(count, -1)


@functools.lru_cache(maxsize=None)
def _shell(kind, L, Ms, Nr, Ek, Ra, precision, dt, tuned, coriolis):
    """The context a program keeps: created, tuned if it is to run for long, factorised."""
    from paper_2508_16635_gb300 import RotatingShell
    s = RotatingShell(L, Ms, Nr, Ek, Ra, PR, ETA, precision=precision, device=DEV, coriolis=coriolis)
    if tuned:
        s.autotune()
    x = s.conductive_state()
    if kind == "step2":
        s.step2(x, dt)
    else:
        s.step(x, 0.0, dt)
    torch.cuda.synchronize()
    return s


def _shell_of(c, **other):
    d = dict(c, **other)
    return _shell(*(d[k] for k in ("kind", "L", "Ms", "Nr", "Ek", "Ra", "precision", "dt", "tuned",
                                   "coriolis")))


@functools.lru_cache(maxsize=None)
def _guess(L, Ms, Nr, Ek, Ra, dt):
    """A rotating wave by time stepping an m = M_s seed (Sec. 2.2), turned so that its phase slot
    (Im T at l = m = M_s, degree of the largest |Re T|) is exactly zero; (state, drift, slot)."""
    c = dict(L=L, Ms=Ms, Nr=Nr)
    from paper_2508_16635_gb300 import RotatingShell
    s = RotatingShell(L, Ms, Nr, Ek, Ra, PR, ETA, precision="mixed", device=DEV)
    U = s.conductive_state() + _noise(c, 4000, 1e-2, only_m=Ms)[0]
    x, p = U.view(3, s.P, Nr, 2), L + 1      # p: the pair l = m = M_s
    prev = None
    for _ in range(60):
        s.step(U, 0.0, dt, nsteps=500)
        amp = float(torch.linalg.norm(x[2, p]))
        if prev is not None and amp > 1e-3 and abs(amp - prev) < 1e-3 * amp:
            break
        prev = amp
    a0 = torch.view_as_complex(x[2, p].clone())
    s.step(U, 0.0, dt, nsteps=10)
    a1 = torch.view_as_complex(x[2, p].clone())
    k = int(torch.argmax(a0.abs()))
    C0 = -cmath.phase(complex(a1[k]) / complex(a0[k])) / (Ms * 10 * dt)
    k = int(torch.argmax(a1.abs()))
    z = torch.view_as_complex(x.contiguous()).clone()
    m = torch.tensor(_pairs(L, Ms)[1], dtype=torch.float64, device=DEV)
    turn = -cmath.phase(complex(a1[k])) / Ms
    z *= torch.polar(torch.ones_like(m), turn * m)[None, :, None]
    U = torch.view_as_real(z).contiguous()
    U[2, p, k, 1] = 0.0
    J = ((2 * s.P + p) * Nr + k) * 2 + 1
    s.close()
    return U.reshape(-1), C0, J


@functools.lru_cache(maxsize=None)
def _batch(L, Ms, Nr, Ek, Ra, count):
    from paper_2508_16635_gb300 import Batch
    b = Batch([dict(L=L, Ms=Ms, Nr=Nr, Ek=Ek, Ra=Ra + i, Pr=PR, eta=ETA, precision="mixed")
               for i in range(count)], device=DEV)
    b.autotune()
    return b


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind in ("newton", "batch"):
        dims = tuple(case[k] for k in ("L", "Ms", "Nr", "Ek", "Ra"))
        st["guess"], st["C"], st["J"] = _guess(*dims, case["dt"])
        # the next point of a branch: Ra a little away from the guess's
        st["dRa"] = 1.0 * torch.rand(1, generator=torch.Generator().manual_seed(int(seed))).item()
        if kind == "batch":
            st["batch"] = _batch(*dims, case["count"])
        else:
            st["shell"] = _shell_of(case, dt=200.0)
        return st
    st["shell"] = s = _shell_of(case)
    if kind == "solve":
        # a right-hand side as the step forms it: values at the collocation radii, zero boundary
        # rows, nothing in the rows of e_00 and f_00
        b = _noise(case, seed, 1.0)[0].view(3, s.P, case["Nr"], 2)
        b[0][:, [0, -1]] = 0.0
        b[1][:, [0, 1, -2, -1]] = 0.0
        b[2][:, [0, -1]] = 0.0
        st["rhs"] = b.reshape(-1).contiguous()
        return st
    st["U"] = s.conductive_state() + _noise(case, seed, 1e-3)[0]
    if kind == "jac":
        st["u"] = _noise(case, seed + 7919, 1.0, case["count"]).reshape(-1).contiguous()
        st["C"], st["J"] = 0.3, s.phase_slot(case["Ms"], min(2, case["Nr"] - 1))
    elif kind == "new_ek":
        st["Ek"] = _ek_points(case, seed)
    return st


def _ek_points(case, seed):
    a = 0.9 + 0.1 * torch.rand(1, generator=torch.Generator().manual_seed(int(seed))).item()
    return [case["Ek"] * a, case["Ek"] * a * 0.85]


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "batch":
        b, n = state["batch"], c["count"]
        for i, s in enumerate(b.shells):
            s.set_params(Ra=c["Ra"] + i + state["dRa"])
        U = [state["guess"].clone() for _ in range(n)]
        C, _, _ = b.newton_rw(U, [state["C"]] * n, [state["J"]] * n, tol=1e-12, max_newton=12,
                              kmax=300)
        return {"U": U, "C": C}
    s = state["shell"]
    if kind == "newton":
        s.set_params(Ra=c["Ra"] + state["dRa"])
        U = state["guess"].clone()
        C, _, _ = s.newton_rw(U, state["C"], state["J"], tol=1e-12, max_newton=12, kmax=300)
        return {"U": U, "C": C}
    if kind == "solve":
        return s.implicit_solve(state["rhs"], c["dt"])
    U = state["U"]
    if kind == "jac":
        return s.apply_jacobian(U, state["C"], state["J"], state["u"], c["dt"])
    if kind == "step2":
        return s.step2(U, c["dt"], nsteps=c["count"])
    if kind == "new_ek":
        for Ek in state["Ek"]:
            s.set_params(Ek=Ek)
            s.step(U, 0.0, c["dt"])
        return U
    s.step(U, 0.0, c["dt"], nsteps=c["count"])
    if kind == "monitor":
        return {"U": U, "diagnostics": list(s.diagnostics(U))}
    return U


# ---- what a pass cannot do without --------------------------------------------------------------
def _sizes(c):
    L, Ms, Nr = c["L"], c["Ms"], c["Nr"]
    P = len(_pairs(L, Ms)[0])
    need = 3 * (L // Ms) + 1
    nphi = min(2 ** a * 3 ** b for a in range(12) for b in range(8) if 2 ** a * 3 ** b >= need)
    return P, -(-3 * Nr // 2), 2 * ((3 * (L + 1) + 3) // 4), nphi


def work(case):
    """Per step or action: the state read and written once, two complex blocks per diagonal block of
    the chains (a direct solve needs as many entries as its L and U factors), the real temperature
    inverses and the Legendre tables once; the Legendre sums split by parity, an FFT in longitude,
    the radial sums split by parity, the block products."""
    c = case
    P, Nd, nlat, nphi = _sizes(c)
    Nr, K1 = c["Nr"], c["L"] // c["Ms"] + 1
    n = 6 * P * Nr
    fft = 2.5 * nphi * max(1.0, math.log2(nphi))
    blocks = 2.0 * P * Nr * Nr
    solve = {"bytes": 16.0 * n + 2 * 16.0 * blocks + 8.0 * (c["L"] + 1) * Nr * Nr,
             "flops": 2 * 8.0 * blocks + 4.0 * P * Nr * Nr}
    if c["coriolis"] == "explicit":
        solve["bytes"] -= 16.0 * blocks
        solve["flops"] -= 8.0 * blocks
    if c["kind"] == "solve":
        return solve
    lin = c["kind"] in ("jac", "newton", "batch")
    transforms = {"bytes": 6 * 8.0 * P * (nlat // 2) / 2 + 8.0 * n,
                  "flops": (52.0 + 24.0) * P * (nlat // 2) * Nd + (13 * fft + (60 if lin else 30) * nphi) * nlat * Nd
                  + 0.5 * P * (28.0 * Nd * Nr + 16.0 * Nd * Nr + 16.0 * Nr * Nr)}
    one = {k: solve[k] + transforms[k] for k in ("bytes", "flops")}
    times = c["count"] * (2 if c["kind"] == "step2" else 1)
    if c["kind"] == "new_ek":
        # the block LU of every chain: D' and its factors, two solves with N_r right-hand sides
        one["flops"] += 2.0 * P * Nr ** 3 * 8.0 * (2.0 / 3.0 + 2.0) + (c["L"] + 1) * Nr ** 3 * 8.0 / 3.0
        one["bytes"] += 3 * 16.0 * blocks
        times = 2
    elif c["kind"] in ("newton", "batch"):
        # actions of a converged solve (three to four iterations) and the Krylov basis twice per action
        acts = 800 if c["kind"] == "newton" else 450
        times = acts * c["count"]
        one["bytes"] += 2 * 8.0 * n * 100
        one["flops"] += 4 * 2.0 * n * 100
    return {k: float(v) * times for k, v in one.items()}


# ---- the same in 64 bits, by plain torch and numpy ------------------------------------------------
def _lobatto(n):
    return np.cos(np.pi * np.arange(n) / (n - 1))


def _cheb(x, nk, order):
    """d^order T_k / dr^order at the radii of x (the gap has width 1, so dx/dr = 2)."""
    ch = np.polynomial.chebyshev
    return np.stack([ch.chebval(x, ch.chebder(np.eye(nk)[k], order) if order else np.eye(nk)[k])
                     for k in range(nk)], axis=1) * 2.0 ** order


def _gauss(n):
    """Gauss-Legendre nodes, weights and sines, north first, polished in extended precision."""
    x = np.polynomial.legendre.leggauss(n)[0][::-1].astype(np.longdouble)
    one = np.longdouble(1)
    for it in range(4):
        p0, p1 = np.ones_like(x), x.copy()
        for k in range(1, n):
            p0, p1 = p1, ((2 * k + 1) * x * p1 - k * p0) / (k + 1)
        d = n * (p0 - x * p1) / ((one - x) * (one + x))
        if it < 3:
            x = x - p1 / d
    w = 2 * (one - x) * (one + x) / (n * p0) ** 2
    x, w = x.astype(np.float64), w.astype(np.float64)
    return x, w, np.sqrt((1.0 - x) * (1.0 + x))


def _plm(L, m, x, s):
    """sqrt((2l+1)(l-m)!/(l+m)!) P_l^m, rows l = m..L (no Condon-Shortley phase)."""
    out = np.zeros((L - m + 1, x.size))
    if L < m:
        return out
    p = np.ones_like(x)
    for k in range(1, m + 1):
        p = p * s * math.sqrt((2 * k + 1) / (2 * k))
    out[0] = p
    if L > m:
        out[1] = math.sqrt(2 * m + 3) * x * p
    for l in range(m + 2, L + 1):
        a = math.sqrt((4.0 * l * l - 1.0) / (l * l - m * m))
        b = math.sqrt(((l - 1.0) ** 2 - m * m) / (4.0 * (l - 1.0) ** 2 - 1.0))
        out[l - m] = a * (x * out[l - m - 1] - b * out[l - m - 2])
    return out


class _Plain:
    """The discretised model of Secs. 2.1, 3.1-3.4 in FP64 tensors, direct sums throughout."""

    def __init__(self, c, Ek):
        L, Ms, Nr = c["L"], c["Ms"], c["Nr"]
        self.L, self.Ms, self.Nr, self.Ek, self.Ra = L, Ms, Nr, Ek, c["Ra"]
        self.explicit = c["coriolis"] == "explicit"
        self.ri, self.ro = ETA / (1 - ETA), 1 / (1 - ETA)
        P, Nd, nlat, nphi = _sizes(c)
        pl, pm = _pairs(L, Ms)
        T = lambda a: torch.tensor(np.ascontiguousarray(a), device=DEV)  # noqa: E731
        xc, xd = _lobatto(Nr), _lobatto(Nd)
        self.rc, self.rd = T(self.ri + 0.5 * (xc + 1)), T(self.ri + 0.5 * (xd + 1))
        E = [_cheb(xc, Nr, o) for o in range(5)]
        self.E, self.Ed = [T(a) for a in E], [T(_cheb(xd, Nr, o)) for o in range(3)]
        fine = np.linalg.solve(_cheb(xd, Nd, 0), np.eye(Nd))[:Nr]
        self.R0, self.R1 = T(E[0] @ fine), T(E[1] @ fine)
        x, w, s = _gauss(nlat)
        self.ms = list(range(0, L + 1, Ms))
        self.start = [sum(L - q + 1 for q in self.ms[:a]) for a in range(len(self.ms) + 1)]
        self.P_, self.dP, self.sP, self.wt = [], [], [], T(w)
        for m in self.ms:
            f = math.sqrt(2.0) if m else 1.0
            l = np.arange(m, L + 1)[:, None]
            up = np.concatenate([np.zeros((1, x.size)), _plm(L, m + 1, x, s)]) if m < L else np.zeros((1, x.size))
            if m == 0:
                d = -np.sqrt(l * (l + 1.0)) * up
            else:
                d = 0.5 * (np.sqrt((l + m) * (l - m + 1.0)) * _plm(L, m - 1, x, s)[1:]
                           - np.sqrt((l + m + 1.0) * (l - m)) * up)
            p = _plm(L, m, x, s)
            self.P_.append(T(f * p))
            self.dP.append(T(f * d))
            self.sP.append(T(f * p / s))
        a, j = np.arange(len(self.ms))[:, None], np.arange(nphi)[None, :]
        ang = 2 * np.pi * ((a * j) % nphi) / nphi
        self.inv = torch.complex(T(np.cos(ang)), T(np.sin(ang))) * T(np.where(a == 0, 1.0, 2.0))
        self.fwd = torch.complex(T(np.cos(ang)), T(-np.sin(ang))) / nphi
        self.l, self.m = T(np.array(pl, dtype=np.float64)), T(np.array(pm, dtype=np.float64))
        self.lam = (self.l * (self.l + 1))[:, None]
        self.npair = P

    # -- states
    def cplx(self, v):
        return torch.view_as_complex(v.reshape(3, self.npair, self.Nr, 2).contiguous())

    def real(self, z):
        return torch.view_as_real(z.contiguous()).reshape(-1)

    # -- explicit terms
    def _mul(self, z, E):
        return z @ E.T.to(z.dtype)

    def grid(self, z):
        e, f, t = z
        E0, E1, E2 = self.Ed
        r, lam = self.rd[None, :], self.lam
        fv, ev = self._mul(f, E0), self._mul(e, E0)
        S = {"ur": lam * fv / r ** 2, "wr": lam * ev / r ** 2, "Tr": self._mul(t, E1)}
        V = {"u": (self._mul(f, E1) / r, ev / r),
             "w": (self._mul(e, E1) / r, -(self._mul(f, E2) - lam * fv / r ** 2) / r),
             "T": (self._mul(t, E0) / r, None)}
        out = {}

        def to_grid(parts):
            G = torch.stack(parts)                       # [m, lat, Nd]
            G[0] = G[0].real.to(G.dtype)
            G = G.reshape(G.shape[0], -1)
            return (self.inv.T @ G).real.reshape(self.inv.shape[1], -1, self.rd.numel())

        sl = [slice(self.start[a], self.start[a + 1]) for a in range(len(self.ms))]
        for k, q in S.items():
            out[k] = to_grid([self.P_[a].T.to(q.dtype) @ q[sl[a]] for a in range(len(self.ms))])
        for k, (s, t) in V.items():
            th, ph = [], []
            for a, m in enumerate(self.ms):
                d, p = self.dP[a].T.to(s.dtype), self.sP[a].T.to(s.dtype)
                vt, vp = d @ s[sl[a]], 1j * m * (p @ s[sl[a]])
                if t is not None:
                    vt, vp = vt + 1j * m * (p @ t[sl[a]]), vp - d @ t[sl[a]]
                th.append(vt)
                ph.append(vp)
            out[k + "t"], out[k + "p"] = to_grid(th), to_grid(ph)
        return out

    def products(self, A, B=None):
        """U x omega and U.grad T of A, or their linearisation about A in the direction B."""
        def two(a, b):
            return (a["ut"] * b["wp"] - a["up"] * b["wt"], a["up"] * b["wr"] - a["ur"] * b["wp"],
                    a["ur"] * b["wt"] - a["ut"] * b["wr"],
                    a["ur"] * b["Tr"] + a["ut"] * b["Tt"] + a["up"] * b["Tp"])
        q = two(A, A) if B is None else tuple(x + y for x, y in zip(two(A, B), two(B, A)))
        return self.Ek * q[0], self.Ek * q[1], self.Ek * q[2], q[3]

    def project(self, q, T):
        """The rows e_r.curl F, e_r.curl curl F (with the buoyancy of T) and -U.grad T."""
        G = [(self.fwd @ a.reshape(a.shape[0], -1).to(self.fwd.dtype)).reshape(len(self.ms), -1, self.rd.numel())
             for a in q]
        Q, S, To, N = [], [], [], []
        for a, m in enumerate(self.ms):
            w = self.wt[None, :] / (4.0 if m else 2.0)
            p, d, s = ((t * w).to(G[0].dtype) for t in (self.P_[a], self.dP[a], self.sP[a]))
            lam = self.lam[self.start[a]:self.start[a + 1]]
            il = torch.where(lam > 0, 1.0 / lam.clamp(min=1.0), torch.zeros_like(lam))
            Q.append(p @ G[0][a])
            N.append(p @ G[3][a])
            S.append(il * (d @ G[1][a] - 1j * m * (s @ G[2][a])))
            To.append(il * (-1j * m * (s @ G[1][a]) - d @ G[2][a]))
        Q, S, To, N = (torch.cat(v) for v in (Q, S, To, N))
        r, lam = self.rc[None, :], self.lam
        return torch.stack([lam * self._mul(To, self.R0) / r,
                            lam / r ** 2 * (self._mul(Q, self.R0) - self._mul(S * self.rd, self.R1))
                            + lam * self.Ra * self._mul(T, self.E[0]) / (r * self.ro),
                            -self._mul(N, self.R0)])

    def mass(self, z):
        c = self.lam * self.Ek / self.rc ** 2
        f0, f2 = self._mul(z[1], self.E[0]), self._mul(z[1], self.E[2])
        return torch.stack([c * self._mul(z[0], self.E[0]), -c * (f2 - self.lam / self.rc ** 2 * f0),
                            self._mul(z[2], self.E[0])])

    # -- implicit operator: chain blocks [field, pair] as Nr x Nr matrices
    def coupling(self, side):
        """(2/r^2) a ((l/r) E0 - E1) to l - 1, (2/r^2) b (-((l+1)/r) E0 - E1) to l + 1."""
        l, m, r = self.l, self.m, self.rc
        if side < 0:
            a = (l * l - 1) * torch.sqrt((l * l - m * m).clamp(min=0) / (4 * l * l - 1).clamp(min=1))
            g = l
        else:
            a = l * (l + 2) * torch.sqrt(((l + 1) ** 2 - m * m) / (4 * (l + 1) ** 2 - 1))
            g = -(l + 1)
        a = torch.where(l > 0, a, torch.zeros_like(a))
        return (2 * a[:, None] / r ** 2)[:, :, None] * ((g[:, None] / r)[:, :, None] * self.E[0] - self.E[1])

    def diagonal(self, fld, sel, mass, diff, cor):
        """mass M + diff (diffusion) + cor (Coriolis diagonal) of the pairs `sel`, no boundary rows."""
        E = self.E
        l, m, r = self.l[sel, None, None], self.m[sel, None, None], self.rc[None, :, None]
        lam, Ek = l * (l + 1), self.Ek
        Lop = E[2] - lam / r ** 2 * E[0]
        if fld == 0:
            M, D, K = lam * Ek / r ** 2 * E[0], -lam * Ek / r ** 2 * Lop, -2j * m / r ** 2 * E[0]
        elif fld == 1:
            L2 = E[4] - 2 * lam / r ** 2 * E[2] + 4 * lam / r ** 3 * E[1] + (lam * lam - 6 * lam) / r ** 4 * E[0]
            M, D, K = -lam * Ek / r ** 2 * Lop, lam * Ek / r ** 2 * L2, 2j * m / r ** 2 * Lop
        else:
            M, D, K = E[0].expand(l.shape[0], -1, -1), -(1 / PR) * (E[2] + 2 / r * E[1] - lam / r ** 2 * E[0]), 0j
        return mass * M + diff * D + cor * K + 0j

    def bc(self, D, fld):
        E0, E1 = self.E[0], self.E[1]
        rows = ((0, E0[0]), (-1, E0[-1])) if fld != 1 else ((0, E0[0]), (1, E1[0]), (-2, E1[-1]), (-1, E0[-1]))
        for j, v in rows:
            D[:, j] = v.to(D.dtype)
        return D

    def factor(self, dt):
        """Row-equilibrated block LU (partial pivoting inside a block) down every chain, all chains
        of one block index together; LU of every temperature operator."""
        cor = 0.0 if self.explicit else 1.0
        nm, Nr = len(self.ms), self.Nr
        self.chains = []
        low, high = self.coupling(-1), self.coupling(+1)
        prev = None
        for i in range(self.L + 1):
            live = [a for a in range(nm) if self.ms[a] + i <= self.L]
            step = []
            for fld in (0, 1):                    # block i of the chains that hold `fld` there
                sel = torch.tensor([self.start[a] + i for a in live], device=DEV)
                D = self.bc(self.diagonal(fld, sel, 1 / dt, 1.0, cor), fld)
                A, C = (cor * t[sel] + 0j for t in (low, high))
                for j in ((0, -1) if fld == 0 else (0, 1, -2, -1)):
                    A[:, j], C[:, j] = 0, 0
                for q, a in enumerate(live):
                    if self.ms[a] + i == 0:
                        D[q] = torch.eye(Nr, device=DEV, dtype=D.dtype)
                    if i == 0:
                        A[q] = 0
                    if self.ms[a] + i == self.L:
                        C[q] = 0
                sc = 1 / torch.maximum(torch.maximum(D.abs().amax(2), A.abs().amax(2)), C.abs().amax(2))[:, :, None]
                D, A, C = D * sc, A * sc, C * sc
                F = D
                if prev is not None:
                    F = D - A @ prev[1 - fld][4][: len(live)]
                lu, piv = torch.linalg.lu_factor(F)
                step.append((sc[:, :, 0], D, A, C, torch.linalg.lu_solve(lu, piv, C), lu, piv, sel))
            self.chains.append(step)
            prev = step
        l0 = torch.arange(self.L + 1, device=DEV)    # pairs of m = 0: every degree once
        D = self.bc(self.diagonal(2, l0, 1 / dt, 1.0, 0.0), 2).real
        self.tsc = 1 / D.abs().amax(2)
        self.tlu = torch.linalg.lu_factor(D * self.tsc[:, :, None])

    def sweep(self, b):
        """The chains' solution for scaled right-hand sides b[i][fld]."""
        y, x = [], [None] * len(b)
        for i, step in enumerate(self.chains):
            row = []
            for fld in (0, 1):
                sc, D, A, C, W, lu, piv, sel = step[fld]
                r = b[i][fld]
                if i:
                    r = r - (A @ y[i - 1][1 - fld][: r.shape[0], :, None])[:, :, 0]
                row.append(torch.linalg.lu_solve(lu, piv, r[:, :, None])[:, :, 0])
            y.append(row)
        for i in range(len(b) - 1, -1, -1):
            x[i] = [v.clone() for v in y[i]]
            if i + 1 < len(b):
                for fld in (0, 1):
                    n = x[i + 1][1 - fld].shape[0]
                    x[i][fld][:n] -= (self.chains[i][fld][4][:n] @ x[i + 1][1 - fld][:, :, None])[:, :, 0]
        return x

    def solve(self, rhs):
        b = [[rhs[fld, s[fld][7]] * s[fld][0] for fld in (0, 1)] for s in self.chains]
        x = self.sweep(b)
        for _ in range(2):                        # refinement with the residual in FP64
            res = []
            for i, step in enumerate(self.chains):
                row = []
                for fld in (0, 1):
                    sc, D, A, C, *_r = step[fld]
                    q = b[i][fld] - (D @ x[i][fld][:, :, None])[:, :, 0]
                    if i:
                        q = q - (A @ x[i - 1][1 - fld][: q.shape[0], :, None])[:, :, 0]
                    if i + 1 < len(b):
                        n = x[i + 1][1 - fld].shape[0]
                        q[:n] -= (C[:n] @ x[i + 1][1 - fld][:, :, None])[:, :, 0]
                    row.append(q)
                res.append(row)
            d = self.sweep(res)
            x = [[u + v for u, v in zip(p, q)] for p, q in zip(x, d)]
        out = torch.zeros_like(rhs)
        for i, step in enumerate(self.chains):
            for fld in (0, 1):
                out[fld, step[fld][7]] = x[i][fld]
        l = self.l.long()
        t = rhs[2] * self.tsc[l]
        sol = torch.linalg.lu_solve(self.tlu[0][l], self.tlu[1][l], torch.stack([t.real, t.imag], 2))
        out[2] = torch.complex(sol[:, :, 0].contiguous(), sol[:, :, 1].contiguous())
        return out

    def rows(self, rhs, wall):
        rhs[0][:, [0, -1]] = 0
        rhs[1][:, [0, 1, -2, -1]] = 0
        rhs[2][:, [0, -1]] = 0
        rhs[2, 0, -1] = wall
        rhs[0:2, self.l == 0] = 0
        m0 = self.m == 0
        rhs[:, m0] = rhs[:, m0].real.to(rhs.dtype)
        return rhs

    def implicit(self, z, diff, cor):
        """diff (diffusion) + cor (Coriolis) applied to z at the collocation radii."""
        allp = torch.arange(self.npair, device=DEV)
        out = torch.stack([(self.diagonal(f, allp, 0.0, diff, cor if f < 2 else 0.0) @ z[f][:, :, None])[:, :, 0]
                           for f in range(3)])
        if cor:
            low, high = self.coupling(-1) + 0j, self.coupling(+1) + 0j
            for f in (0, 1):
                dn, up = torch.zeros_like(z[f]), torch.zeros_like(z[f])
                for a in range(len(self.ms)):
                    p, q = self.start[a], self.start[a + 1]
                    dn[p + 1:q], up[p:q - 1] = z[1 - f][p:q - 1], z[1 - f][p + 1:q]
                add = cor * ((low @ dn[:, :, None]) + (high @ up[:, :, None]))[:, :, 0]
                add[self.l == 0] = 0
                out[f] += add
        return out

    def explicit_terms(self, z):
        n = self.project(self.products(self.grid(z)), z[2])
        return n - self.implicit(z, 0.0, 1.0) if self.explicit else n

    def conductive(self):
        D = self.bc(self.diagonal(2, torch.tensor([0], device=DEV), 0.0, 1.0, 0.0), 2).real[0]
        b = torch.zeros(self.Nr, dtype=torch.float64, device=DEV)
        b[-1] = 1.0
        z = torch.zeros((3, self.npair, self.Nr), dtype=torch.complex128, device=DEV)
        z[2, 0] = torch.linalg.solve(D, b) + 0j
        return z

    def diagnostics(self, z):
        """Kinetic energy (Parseval for the potentials, Gauss-Legendre in r) and Nusselt numbers."""
        x, w = np.polynomial.legendre.leggauss(2 * self.Nr + 16)
        r = torch.tensor(self.ri + 0.5 * (x + 1), device=DEV)
        w = torch.tensor(0.5 * w, device=DEV)
        E0, E1 = (torch.tensor(_cheb(x, self.Nr, o), device=DEV) for o in (0, 1))
        sq = lambda q: q.abs() ** 2  # noqa: E731
        lam = self.lam
        d = (lam * sq(self._mul(z[0], E0)) / r ** 2 + lam ** 2 * sq(self._mul(z[1], E0)) / r ** 4
             + lam * sq(self._mul(z[1], E1)) / r ** 2)
        wm = 16 * math.pi - 12 * math.pi * (self.m == 0).double()
        V = 4 * math.pi * (self.ro ** 3 - self.ri ** 3) / 3
        ke = 0.5 * float((wm[:, None] * d * (w * r ** 2)).sum()) / V
        g = self._mul(z[2], self.E[1])[0].real
        return [ke, float(g[-1]) * -self.ri / self.ro, float(g[0]) * -self.ro / self.ri]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("newton", "batch"):
        return None           # hundreds of actions and a Krylov solve: minutes in plain tensors
    if kind == "new_ek":
        z = None
        for Ek in _ek_points(case, seed):
            p = _Plain(case, Ek)
            z = p.conductive() + p.cplx(_noise(case, seed, 1e-3)[0]) if z is None else z
            p.factor(case["dt"])
            z = p.solve(p.rows(p.mass(z) / case["dt"] + p.explicit_terms(z), 1.0))
        return p.real(z)
    p = _Plain(case, case["Ek"])
    dt = case["dt"]
    if kind == "solve":
        b = _noise(case, seed, 1.0)[0].view(3, p.npair, case["Nr"], 2)
        z = torch.view_as_complex(b.contiguous())
        p.factor(dt)
        z[0][:, [0, -1]] = 0
        z[1][:, [0, 1, -2, -1]] = 0
        z[2][:, [0, -1]] = 0
        return p.real(p.solve(z))
    z = p.conductive() + p.cplx(_noise(case, seed, 1e-3)[0])
    drift = lambda C: 1j * C * p.m[:, None]  # noqa: E731
    if kind == "step2":
        p.factor(0.5 * dt)
        for _ in range(case["count"]):
            base = p.mass(z) / dt - 0.5 * p.implicit(z, 1.0, 0.0 if p.explicit else 1.0)
            n0 = p.explicit_terms(z)
            s = p.solve(p.rows(2 * (base + n0), 1.0))
            z = p.solve(p.rows(2 * (base + 0.5 * (n0 + p.explicit_terms(s))), 1.0))
        return p.real(z)
    p.factor(dt)
    if kind == "jac":
        n = 6 * p.npair * case["Nr"]
        u = _noise(case, seed + 7919, 1.0, case["count"])
        J = ((2 * p.npair + case["L"] + 1) * case["Nr"] + min(2, case["Nr"] - 1)) * 2 + 1
        gU, MU, out = p.grid(z), p.mass(z), []
        for q in range(case["count"]):
            v = u[q].clone()
            c = v[J].item()
            v[J] = 0.0
            x = p.cplx(v)
            rhs = (1 / dt + drift(0.3)) * p.mass(x) + p.project(p.products(gU, p.grid(x)), x[2])
            if p.explicit:
                rhs = rhs - p.implicit(x, 0.0, 1.0)
            rhs = rhs + c * 1j * p.m[:, None] * MU
            out.append(p.real(p.solve(p.rows(rhs, 0.0))) - v)
        return torch.cat(out).reshape(case["count"] * n)
    for _ in range(case["count"]):
        z = p.solve(p.rows(p.mass(z) / dt + p.explicit_terms(z), 1.0))
    if kind == "monitor":
        return {"U": p.real(z), "diagnostics": p.diagnostics(z)}
    return p.real(z)
