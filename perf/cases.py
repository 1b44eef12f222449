"""The calls whose speed matters to a user of the library, over the range they are made in.

Three kinds of call, each through the public binding (paper_1008_3647_gb300.ufg):
  - one operator or preconditioner application on a vector the caller holds (a caller composing
    its own Krylov solver, a measurement, the backward pass of the pseudofermion action);
  - one solve of M^T M x = b on one lattice, or the HMC force, whose bulk is such a solve;
  - one batch of independent problems.
Lattices are those of the tests and of bench.py: 4^3 x 16, 8^3 x 64, the uneven batch's
N_x in {6, 8, 10, 12}, 16^3 x 256 and 32^3 x 512, plus odd N_tau in between.  The auxiliary field
is i.i.d. uniform on [-pi, pi] and the vectors are i.i.d. N(0, 1), as everywhere in this
repository; tau = 0.05 and g = 5.  The weak-coupling preconditioner is order 2 with the paper's
S_{2k/3,k/3} acceleration unless a case says otherwise.

Solves ask for 1e-10, the residual every solve of this repository is gated on; the two smallest
lattices for 1e-12, the paper's criterion, which FP64 arithmetic reaches there with room to spare.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1008_3647_gb300 import ufg
from paper_1008_3647_gb300.inputs import batch_shapes

TAU, G = 0.05, 5.0
WCE = {"order": 2, "euler": "euler23"}
APPLY = ("M", "Mdag", "Q", "M1", "M1T", "kinetic", "M0inv", "M0invT")
NXS = (4, 6, 8, 10, 12, 16, 32)


def listed():
    return [
        # the smallest call: one FP64 normal-operator application on the 4^3 x 16 lattice
        {"name": "q_f64_4x16", "kind": "apply", "op": "Q", "nx": 4, "ntau": 16, "dtype": "f64"},
        # FP64 transpose on an uneven lattice: N_x without a power of two, odd N_tau
        {"name": "mdag_f64_10x117", "kind": "apply", "op": "Mdag", "nx": 10, "ntau": 117,
         "dtype": "f64"},
        # the ordinary FP32 application, vectors resident in L2
        {"name": "m_f32_16x256", "kind": "apply", "op": "M", "nx": 16, "ntau": 256,
         "dtype": "f32"},
        # the largest FP32 application, from HBM
        {"name": "m_f32_32x512", "kind": "apply", "op": "M", "nx": 32, "ntau": 512,
         "dtype": "f32"},
        # the largest FP64 application: M, then M^T
        {"name": "q_f64_32x512", "kind": "apply", "op": "Q", "nx": 32, "ntau": 512,
         "dtype": "f64"},
        # the preconditioner of the first BiCGStab step, on its own
        {"name": "wce_t_f32_16x256", "kind": "precond", "transpose": 1, "nx": 16, "ntau": 256,
         "dtype": "f32", "order": 2},
        # plain FP64 CG on the smallest lattice: nothing but latency
        {"name": "cg_f64_4x16", "kind": "solve", "method": "cg", "pc": "none", "nx": 4,
         "ntau": 16, "mixed": 0, "tol": 1e-12},
        # FP64 two-step BiCGStab, weak-coupling preconditioner, medium lattice
        {"name": "bicg_f64_8x64", "kind": "solve", "method": "bicgstab", "pc": "wce", "nx": 8,
         "ntau": 64, "mixed": 0, "tol": 1e-12},
        # mixed-precision CG with the Chebyshev preconditioner of degree 16
        {"name": "cg_cheb_mixed_16x256", "kind": "solve", "method": "cg", "pc": "cheb", "nx": 16,
         "ntau": 256, "mixed": 1, "tol": 1e-10},
        # bench.py's headline step: eight configurations solved together in mixed precision
        {"name": "batch_mixed_8x16x256", "kind": "batch", "n": 8, "nx": 16, "ntau": 256,
         "shape_seed": -1, "mixed": 1, "tol": 1e-10},
        # the uneven batch: 96 problems, N_x in {6, 8, 10, 12}, N_tau in {40, 80, 120, 160}
        {"name": "batch_mixed_96", "kind": "batch", "n": 96, "nx": 0, "ntau": 0, "shape_seed": 0,
         "mixed": 1, "tol": 1e-10},
        # the HMC force on the largest lattice: one mixed solve and the adjoint force kernel
        {"name": "force_mixed_32x512", "kind": "force", "nx": 32, "ntau": 512, "mixed": 1,
         "tol": 1e-10},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the same kinds of call, N_x over every extent the library is built for,
    N_tau spread over its logarithm (odd ones included)."""
    kind = rng.choice(("apply", "apply", "apply", "precond", "force_x", "solve", "solve", "batch"))
    dtype = rng.choice(("f64", "f32"))
    if kind in ("apply", "precond", "force_x"):
        c = {"kind": kind, "nx": rng.choice(NXS), "ntau": _log_int(rng, 8, 512),
             "dtype": "f64" if kind == "force_x" else dtype}
        if kind == "apply":
            c["op"] = rng.choice(APPLY)
        elif kind == "precond":
            c["transpose"] = rng.choice((0, 1))
            c["order"] = rng.choice((1, 2, 2, 4))
        return c
    if kind == "solve":
        method, pc = rng.choice((("bicgstab", "wce"), ("bicgstab", "wce"), ("cg", "cheb")))
        c = {"kind": kind, "method": method, "pc": pc, "nx": rng.choice((4, 6, 8, 10, 12, 16)),
             "ntau": _log_int(rng, 16, 200), "mixed": rng.choice((0, 1)), "tol": 1e-10}
        if method == "cg":  # the cost grows with N_tau squared
            c["nx"], c["ntau"] = min(c["nx"], 12), min(c["ntau"], 99)
        return c
    return {"kind": "batch", "n": rng.randint(3, 24), "nx": 0, "ntau": 0,
            "shape_seed": rng.randint(1, 10 ** 6), "mixed": rng.choice((0, 1)), "tol": 1e-10}


def _shapes(case):
    if case["shape_seed"] < 0:
        return [(case["nx"], case["ntau"])] * case["n"]
    return [(nx, nt) for nx, nt, _ in batch_shapes(case["n"], case["shape_seed"])]


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _sigma(g, shape):
    return (2.0 * torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) - 1.0) * math.pi


def _normal(g, shape):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)


def _inputs(case, seed):
    """(sigma, vector) of a single-lattice case, both FP64."""
    g = _generator(seed)
    shape = (case["ntau"],) + (case["nx"],) * 3
    return _sigma(g, shape), _normal(g, shape)


def _batch_inputs(case, seed):
    """The problems of a batch on three flat buffers (sigma, b, x)."""
    g = _generator(seed)
    sizes = [nx ** 3 * nt for nx, nt in _shapes(case)]
    # every problem starts on a 256-byte boundary of its buffer
    starts = np.concatenate([[0], np.cumsum([(s + 31) // 32 * 32 for s in sizes])]).tolist()
    sigma, b = _sigma(g, (starts[-1],)), _normal(g, (starts[-1],))
    x = torch.zeros(starts[-1], device="cuda", dtype=torch.float64)
    probs = []
    for (nx, nt), s, o in zip(_shapes(case), sizes, starts):
        sh = (nt, nx, nx, nx)
        probs.append({"nx": nx, "ntau": nt, "tau": TAU, "g": G, "sigma": sigma[o:o + s].view(sh),
                      "b": b[o:o + s].view(sh), "x": x[o:o + s].view(sh)})
    return probs, x


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        probs, x = _batch_inputs(case, seed)
        return {"case": case, "probs": probs, "x": x}
    sigma, v = _inputs(case, seed)
    lat = ufg.Lattice(case["nx"], case["ntau"], TAU, G)
    st = {"case": case, "lat": lat, "field": ufg.Field(lat, sigma), "sigma": sigma}
    if case.get("dtype") == "f32":
        v = v.float()
    if kind != "apply":
        st["solver"] = ufg.Solver(lat)
    if kind == "precond":
        st["solver"].ufg_set_preconditioner("wce", order=case["order"], euler="euler23")
    elif kind == "force":
        st["solver"].ufg_set_preconditioner("wce", **WCE)
        v = ufg.ufg_apply_Mdag(st["field"], v)  # phi = M^T eta, the pseudofermion heat bath
    elif kind == "solve":
        pc = {"wce": WCE, "cheb": {"degree": 16}, "none": {}}[case["pc"]]
        st["solver"].ufg_set_preconditioner(case["pc"], **pc)
    st["v"] = v
    st["y"] = torch.empty_like(v)
    return st


def _precision(case):
    return ufg.UFG_MIXED if case["mixed"] else ufg.UFG_FP64


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "apply":
        return getattr(ufg, "ufg_apply_" + case["op"])(st["field"], st["v"], st["y"])
    if kind == "precond":
        return st["solver"].ufg_apply_preconditioner(st["field"], st["v"], st["y"],
                                                     transpose=case["transpose"])
    if kind == "force_x":
        return st["solver"].ufg_force_from_solution(st["field"], st["v"], st["y"])
    kw = {"tol": case["tol"], "precision": _precision(case)}
    if kind == "batch":
        ufg.ufg_solve_batch(st["probs"], "wce", WCE, **kw)
        return st["x"]
    if kind == "force":
        dS, X, S, _ = st["solver"].ufg_hmc_force(st["field"], st["v"], **kw)
        return {"dS": dS, "X": X, "S": S}
    solve = (st["solver"].ufg_solve_cg_normal if case["method"] == "cg"
             else st["solver"].ufg_solve_bicgstab_two_step)
    x, _ = solve(st["field"], st["v"], st["y"], **kw)
    return x


# ---- the work a pass cannot do without -------------------------------------------------------

def _line_flops(nx):
    """Multiply-adds of one separable line operator per site and axis, after the reflection x ->
    -x (even and odd part apart) and, where N_x / 2 is even, the reflection x -> N_x/2 - x."""
    h = nx // 2
    if h % 2 == 0 and nx >= 8:
        q = h // 2
        return 2.0 * ((q + 1) ** 2 + 2 * q * q + (q - 1) ** 2) / nx
    return 2.0 * ((h + 1) ** 2 + (h - 1) ** 2) / nx


def _iterations(case, ntau):
    """Typical Krylov iterations of one solve at tol 1e-10 on these fields."""
    if case.get("method") == "cg":
        return 3.0 * ntau if case["pc"] == "cheb" else 24.0 * ntau
    return 9.0 * ntau ** 0.35


def _solve_work(case, nx, ntau):
    """One solve: its iterations' operator applications, each reading its operand and the field
    once and writing its result once (four bytes a value in mixed precision)."""
    sites = nx ** 3 * ntau
    eb = 4.0 if case["mixed"] else 8.0
    it = _iterations(case, ntau)
    kin = 3.0 * _line_flops(nx)
    if case.get("method") == "cg":
        q = 17 if case["pc"] == "cheb" else 1  # Q applications per iteration
        return it * q * 3 * eb * sites, it * q * 2 * (kin + 3) * sites
    # per iteration twice: the operator and the order-2 series (in, out, the field twice)
    d = WCE["order"]
    return (it * 2 * (3 + 2 + d) * eb * sites,
            it * 2 * ((1 + 2 * d) * kin + 4 * (d + 1) + 10) * sites)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = [_solve_work(case, nx, nt) for nx, nt in _shapes(case)]
        return {"bytes": sum(a for a, _ in w), "flops": sum(b for _, b in w)}
    nx, ntau = case["nx"], case["ntau"]
    sites = nx ** 3 * ntau
    kin = 3.0 * _line_flops(nx)
    if kind in ("solve", "force"):
        b, f = _solve_work(case, nx, ntau)
        extra = 4 * 8.0 * sites if kind == "force" else 0.0
        return {"bytes": b + extra, "flops": f + (2 * kin * sites if kind == "force" else 0.0)}
    eb = 4.0 if case["dtype"] == "f32" else 8.0
    if kind == "force_x":  # X, w and c in, dS out; Y = M X and one more kinetic stage
        return {"bytes": 4 * eb * sites, "flops": 2 * (kin + 4) * sites}
    if kind == "precond":  # r and s in, z out; two transforms, d M1 terms of two each
        d = case["order"]
        return {"bytes": 3 * eb * sites, "flops": (2 * (d + 1) * kin + 4 * (d + 1)) * sites}
    op = case["op"]
    vecs = 2 if op in ("kinetic", "M0inv", "M0invT") else 3
    stages = {"Q": 2, "M0inv": 2, "M0invT": 2}.get(op, 1)
    return {"bytes": vecs * eb * sites, "flops": stages * (kin + 3) * sites}


# ---- the same results in 64 bits, by plain torch ---------------------------------------------

class _Plain:
    """M and its relatives written from their definitions, FP64, dense along each axis."""

    def __init__(self, nx, sigma):
        self.A = math.sqrt(2.0 * math.expm1(TAU * G))
        k = 2.0 * math.pi * torch.fft.fftfreq(nx, device="cuda", dtype=torch.float64)
        d = torch.arange(nx, device="cuda", dtype=torch.float64)
        lam = torch.exp(-0.5 * TAU * k * k)
        circ = (lam[None, :] * torch.cos(k[None, :] * d[:, None])).sum(1) / nx
        i = torch.arange(nx, device="cuda")
        self.T = circ[(i[:, None] - i[None, :]) % nx].contiguous()
        self.b = lam[:, None, None] * lam[None, :, None] * lam[None, None, :]
        self.s = torch.sin(sigma)
        self.w = 1.0 + self.A * self.s

    def K(self, x):
        x = x @ self.T
        x = torch.matmul(self.T, x)
        return torch.einsum("ij,tjyx->tiyx", self.T, x)

    @staticmethod
    def up(x):  # t -> t + 1 with the signs of M's off-diagonal blocks
        y = -torch.roll(x, 1, 0)
        y[0] = -y[0]
        return y

    @staticmethod
    def down(x):
        y = -torch.roll(x, -1, 0)
        y[-1] = -y[-1]
        return y

    def M(self, x):
        return x + self.up(self.K(self.w * x))

    def Mdag(self, x):
        return x + self.w * self.K(self.down(x))

    def Q(self, x):
        return self.Mdag(self.M(x))

    def M1(self, x):
        return self.up(self.K(self.s * x))

    def M1T(self, x):
        return self.s * self.K(self.down(x))

    def kinetic(self, x):
        return self.K(x)

    def M0inv(self, x, sign=-1.0):
        nt = x.shape[0]
        t = torch.arange(nt, device="cuda", dtype=torch.float64)
        tw = torch.exp(1j * math.pi * t / nt).view(nt, 1, 1, 1)
        omega = (2.0 * math.pi * torch.fft.fftfreq(nt, device="cuda", dtype=torch.float64)
                 + math.pi / nt).view(nt, 1, 1, 1)
        y = torch.fft.fftn(x * tw.conj())
        y = y / (1.0 - torch.exp(1j * sign * omega) * self.b)
        return (torch.fft.ifftn(y) * tw).real.contiguous()

    def M0invT(self, x):
        return self.M0inv(x, +1.0)

    def wce(self, r, order, transpose):
        inv, one = (self.M0invT, self.M1T) if transpose else (self.M0inv, self.M1)
        term = inv(r)
        sums = [term]
        for _ in range(order):
            term = -self.A * inv(one(term))
            sums.append(sums[-1] + term)
        for _ in range((2 * order + 1) // 3):  # Euler recursion with p = 1/2, 2d/3 levels
            sums = [0.5 * (a + b) for a, b in zip(sums[:-1], sums[1:])]
        return sums[-1]

    def force(self, X, sigma):
        return 2.0 * self.A * torch.cos(sigma) * X * self.K(-self.down(self.M(X)))

    def solve(self, b):
        """CG on Q x = b, restarted from the true residual until it stops falling."""
        x = torch.zeros_like(b)
        last = math.inf
        for _ in range(6):
            r = b - self.Q(x)
            rr = float((r * r).sum())
            if rr >= 0.25 * last or rr == 0.0:
                break
            last, d = rr, torch.zeros_like(b)
            target, p = 1e-28 * rr, r.clone()
            rs = (r * r).sum()
            for it in range(20000):
                q = self.Q(p)
                a = rs / (p * q).sum()
                d += a * p
                r -= a * q
                new = (r * r).sum()
                p = r + (new / rs) * p
                rs = new
                if it % 32 == 31 and float(rs) <= target:
                    break
            x = x + d
        return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch" or kind == "force":
        return None
    sigma, v = _inputs(case, seed)
    if kind == "solve" and v.numel() > 1 << 16:
        return None  # more than a few seconds of plain CG
    if case.get("dtype") == "f32":
        v = v.float().double()
    p = _Plain(case["nx"], sigma)
    if kind == "apply":
        return getattr(p, case["op"])(v)
    if kind == "precond":
        return p.wce(v, case["order"], case["transpose"])
    if kind == "force_x":
        return p.force(v, sigma)
    return p.solve(v)
