"""What this framework is used for, as cases that can be timed and checked.

Every case is one call (or the few calls of one pass) that a CFD or kinetics program makes on cells
it holds on the GPU, through the public binding ``paper_2205_05681_gb300.chem``, on one of the
three mechanisms of the repository's workloads (13, 53 and 111 species):

* ``integrate``  one operator-split step of every cell, in place (any method of the solver table);
* ``switch``     consecutive split steps with quiescent cells moved to the W-method;
* ``gradient``   the autograd function: checkpointed forward, loss on the final temperature,
                 discrete adjoint back to ln A of every reaction and the initial state;
* ``source`` / ``jacobian``  f(y) and df/dy of every cell, for programs that bring their own solver.

The cell states are the recipes of ``synth.make_states``, drawn here for all cells at once.
``exact`` is the same mathematics in plain torch float64: mechanism data in, library operations
only (dense batched linear algebra, no code of the framework's computation).
"""
import functools
import math
import os

import numpy as np
import torch

from paper_2205_05681_gb300 import chem, synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MECH_DIR = os.path.join(ROOT, "paper_2205_05681_gb300", "_cache", "mechs")
RECIPES = ("h2_fresh", "ch4_partial", "ch4_front", "ch4_ign")
FALLOFF = {"LIND", "TROE"}
RU, PATM, RCAL = 8314.462618, 101325.0, 1.987204258640832
EQ_TEMPLATES = 48  # relaxed product states per preparation, tiled over the product cells


# ------------------------------------------------------------------------------ the cases


def _case(op, mech, cells, recipe, **more):
    c = {"op": op, "mech": mech, "cells": cells, "recipe": recipe, "dt": 1e-6, "rtol": 1e-6,
         "atol": 1e-10, "method": chem.ROS4, "splits": 1, "lnA": False}
    c.update(more)
    return c


def listed():
    return [
        # a handful of cells (a 0-D reactor study, one MPI rank's leftovers): all latency
        dict(_case("integrate", "h2_13", 17, "h2_fresh"), name="h2_13_17"),
        # the small forward workload of the repository
        dict(_case("integrate", "h2_13", 1024, "h2_fresh"), name="h2_13_1024"),
        # the same mechanism at a batch that fills the GPU
        dict(_case("integrate", "h2_13", 65536, "h2_fresh"), name="h2_13_65536"),
        # an odd, less than GPU-filling batch of the 53-species mechanism
        dict(_case("integrate", "ch4_53", 333, "ch4_partial"), name="ch4_53_333"),
        # the 53-species forward workload, a quarter of its cells
        dict(_case("integrate", "ch4_53", 16384, "ch4_partial"), name="ch4_53_16384"),
        # a tighter tolerance with RODAS4 and the caller's own ln A (parameter studies)
        dict(_case("integrate", "ch4_53", 1000, "ch4_partial", method=chem.RODAS4, rtol=1e-7,
                   lnA=True), name="ch4_53_rodas4_1000"),
        # one split step of the 111-species flame front: few stiff cells among quiescent ones
        dict(_case("integrate", "ch4_111", 2001, "ch4_front"), name="ch4_111_front_2001"),
        dict(_case("integrate", "ch4_111", 24000, "ch4_front"), name="ch4_111_front_24000"),
        # three split steps of the flame front with quiescent cells on the W-method (cache carried)
        dict(_case("switch", "ch4_111", 6000, "ch4_front", splits=3), name="ch4_111_switch_6000"),
        # f(y) and the Jacobian for a program's own solver
        dict(_case("source", "ch4_53", 50000, "ch4_partial"), name="ch4_53_source_50000"),
        dict(_case("jacobian", "ch4_111", 3000, "ch4_front"), name="ch4_111_jacobian_3000"),
        # gradients through ignition (checkpoint every 16 accepted steps)
        dict(_case("gradient", "ch4_53", 300, "ch4_ign", dt=2e-6), name="ch4_53_gradient_300"),
    ]


def draw(rng):
    """One more case: an operation and mechanism as listed, another size, step and option."""
    def cells(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return max(lo, min(hi, n | 1 if rng.random() < 0.5 else n))

    dt = math.exp(rng.uniform(math.log(5e-7), math.log(1.5e-6)))
    tol = rng.choice([(1e-6, 1e-10), (1e-6, 1e-10), (1e-7, 1e-10)])
    opt = {"dt": dt, "rtol": tol[0], "atol": tol[1], "lnA": rng.random() < 0.3}
    op = rng.choice(["h2", "h2", "ch4_53", "ch4_53", "method", "front", "front", "switch", "source",
                     "jacobian", "gradient"])
    if op == "h2":
        return _case("integrate", "h2_13", cells(5, 65536), "h2_fresh", **opt)
    if op == "ch4_53":
        return _case("integrate", "ch4_53", cells(31, 10000), "ch4_partial", **opt)
    if op == "method":
        m = rng.choice([chem.ROS3, chem.RODAS3, chem.RODAS4])
        return _case("integrate", "ch4_53", cells(100, 2000), "ch4_partial", **dict(opt, method=m))
    if op == "front":
        return _case("integrate", "ch4_111", cells(100, 10000), "ch4_front", **opt)
    if op == "switch":
        return _case("switch", "ch4_111", cells(500, 5000), "ch4_front", splits=rng.choice([2, 3]), **opt)
    if op == "source":
        m, r = rng.choice([("h2_13", "h2_fresh"), ("ch4_53", "ch4_partial"), ("ch4_111", "ch4_front")])
        return _case("source", m, cells(1000, 50000), r, lnA=opt["lnA"])
    if op == "jacobian":
        m, r, top = rng.choice([("h2_13", "h2_fresh", 50000), ("ch4_53", "ch4_partial", 12000),
                                ("ch4_111", "ch4_front", 3000)])
        return _case("jacobian", m, cells(300, top), r, lnA=opt["lnA"])
    return _case("gradient", "ch4_53", cells(50, 300), "ch4_ign",
                 dt=math.exp(rng.uniform(math.log(5e-7), math.log(2e-6))))


# typical step attempts per cell and call of each recipe at 1 us (counted on these states), and the
# algorithmic FP64 operations of one attempt (LU, solves, rates, Jacobian): see work()
ATTEMPTS = {"h2_fresh": 6.0, "ch4_partial": 73.0, "ch4_front": 21.0, "ch4_ign": 80.0}
FLOPS = {"h2_13": 7.7e3, "ch4_53": 1.79e5, "ch4_111": 1.18e6}


def work(case):
    """State in and out once per call; operations of the steps such cells take."""
    ns = synth.MECHS[case["mech"]][0]
    n, op = case["cells"], case["op"]
    flops = n * FLOPS[case["mech"]]
    if op == "source":
        return {"bytes": 8.0 * n * (2 * ns + 1), "flops": 0.1 * flops}
    if op == "jacobian":
        return {"bytes": 8.0 * n * (ns * ns + ns + 1), "flops": 0.25 * flops}
    bytes_ = 8.0 * n * (2 * (ns + 1) + 3) * case["splits"]
    flops *= ATTEMPTS[case["recipe"]] * case["splits"]
    if op == "gradient":
        return {"bytes": 2 * bytes_, "flops": 5 * flops}
    return {"bytes": bytes_, "flops": flops}


# ------------------------------------------------------------------------------ mechanisms, states


@functools.lru_cache(maxsize=None)
def _mech(name):
    return synth.mechanism(name)


@functools.lru_cache(maxsize=None)
def _handle(name):
    """The compiled mechanism: a program loads it once and keeps it."""
    return chem.Mechanism(synth.mechanism_file(name, MECH_DIR))


def _mass(mech, X):
    Y = X * mech.weights()
    return Y / Y.sum(axis=1, keepdims=True)


def _fuel_o2(mech):
    fuel = "CH4" if "CH4" in [s.name for s in mech.species] else "H2"
    return fuel, (2.0 if fuel == "CH4" else 0.5)


def _unburnt(mech, phi):
    fuel, st = _fuel_o2(mech)
    X = np.zeros((len(phi), mech.n_species))
    X[:, mech.index(fuel)] = 1.0
    X[:, mech.index("O2")] = st / phi
    X[:, mech.index("N2")] = 3.76 * st / phi
    return _mass(mech, X)


def _burnt(mech, phi):
    """Complete-combustion products of CH4 and air (CO/H2 split when rich)."""
    X = np.zeros((len(phi), mech.n_species))
    O = 4.0 / phi
    lean = O >= 4.0
    left = np.maximum(O - 1.0, 0.0)
    h2o = np.where(lean, 2.0, np.minimum(2.0, left))
    co2 = np.where(lean, 1.0, np.minimum(1.0, np.maximum(left - h2o, 0.0)))
    X[:, mech.index("N2")] = 3.76 * 2.0 / phi
    X[:, mech.index("CO2")] = co2
    X[:, mech.index("CO")] = 1.0 - co2
    X[:, mech.index("H2O")] = h2o
    X[:, mech.index("H2")] = 2.0 - h2o
    X[:, mech.index("O2")] = np.where(lean, (O - 4.0) / 2.0, 0.0)
    return _mass(mech, X)


def _pool(mech, rng, n, lo, hi):
    Y = np.exp(rng.uniform(math.log(lo), math.log(hi), size=(n, mech.n_species)))
    fuel, _ = _fuel_o2(mech)
    for s in mech.species:
        if s.name in {fuel, "O2", "N2", "H2O", "CO2", "CO", "H2"}:
            Y[:, mech.index(s.name)] = 0.0
    return Y


def _states(mech, n, recipe, seed):
    """T [n], P [n], Y [n, Ns] of the named recipe (see synth.make_states), numpy float64."""
    rng = np.random.default_rng([seed, RECIPES.index(recipe)])
    U = rng.uniform
    if recipe == "h2_fresh":
        T, P = U(1000.0, 1600.0, n), U(1.0, 25.0, n) * PATM
        d = rng.dirichlet(np.ones(3), size=n)
        Y = _pool(mech, rng, n, 1e-8, 1e-5)
        Y[:, mech.index("H2")] += 0.5 * d[:, 0]
        Y[:, mech.index("O2")] += 0.5 * d[:, 1]
        Y[:, mech.index("N2")] += 0.5 + 0.5 * d[:, 2]
    elif recipe == "ch4_partial":
        T, P = U(800.0, 2200.0, n), U(1.0, 50.0, n) * PATM
        phi, xi = U(0.5, 2.0, n), U(0.0, 1.0, n)[:, None]
        Y = (1 - xi) * _unburnt(mech, phi) + xi * _burnt(mech, phi) + _pool(mech, rng, n, 1e-8, 1e-3)
    elif recipe == "ch4_ign":
        T, P, phi = U(900.0, 1400.0, n), U(1.0, 40.0, n) * PATM, U(0.5, 2.0, n)
        Y = _unburnt(mech, phi) + _pool(mech, rng, n, 1e-4, 3e-2)
    else:
        # flame front: 10% radical-rich front cells among relaxed product cells
        front = rng.random(n) < 0.10
        P = U(1.0, 50.0, n) * PATM
        xi = U(0.0, 0.5, n)[:, None]
        phi = U(0.5, 1.5, n)
        T = U(1000.0, 1300.0, n)
        Y = (1 - xi) * _unburnt(mech, phi) + xi * _burnt(mech, phi) + _pool(mech, rng, n, 1e-6, 1e-2)
        t = EQ_TEMPLATES
        Tq, Pq = U(1800.0, 2400.0, t), U(1.0, 50.0, t) * PATM
        Yq = _burnt(mech, U(0.7, 1.3, t)) + _pool(mech, rng, t, 1e-6, 1e-4)
        Yq /= Yq.sum(axis=1, keepdims=True)
        Tq, Yq = _relax(mech.name, Tq, Pq, Yq)
        k = rng.integers(0, t, n)
        noise = 1.0 + 1e-9 * rng.standard_normal((n, mech.n_species))
        T, P = np.where(front, T, Tq[k]), np.where(front, P, Pq[k])
        Y = np.where(front[:, None], Y, Yq[k] * noise)
    return T, P, Y / Y.sum(axis=1, keepdims=True)


def _relax(name, T, P, Y):
    """Product states near chemical equilibrium: implicit Euler steps of growing size up to 1e-3 s."""
    r = _ref(name)
    P = _dev(P)
    y = r.state(_dev(T), _dev(Y))
    eye = torch.eye(r.ns, dtype=torch.float64, device=y.device)
    h = 1e-10
    while h < 1e-3:
        for _ in range(2):
            f, J = r.source(y, P, jac=True)
            y = y + torch.linalg.solve(eye / h - J, f.unsqueeze(-1)).squeeze(-1)
            y[:, 1:].clamp_(min=0.0)
        h *= 2.0
    T, Y = r.mass(y)
    return T.cpu().numpy(), Y.cpu().numpy()


def _dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype).cuda()


def prepare(case, seed):
    mech, m = _mech(case["mech"]), _handle(case["mech"])
    n, op = case["cells"], case["op"]
    T, P, Y = _states(mech, n, case["recipe"], seed)
    s = {"case": case, "m": m, "T": _dev(T), "P": _dev(P), "Y": _dev(Y.T)}
    if case["lnA"]:
        d = np.random.default_rng([seed, 77]).uniform(-0.2, 0.2, m.nr)
        s["lnA"] = _dev(m.lnA() + d)
    if op in ("source", "jacobian"):
        s["n"] = (s["Y"][:-1] / _dev(mech.weights()[:-1])[:, None]).contiguous()
    elif op == "gradient":
        s["target"] = _dev(np.random.default_rng([seed, 78]).uniform(1500.0, 2500.0, n))
        s["lnA"] = _dev(m.lnA())
        s["fn"] = chem.chem_integrate_fn()
    else:
        o = m.opts(tableau=case["method"], lnA=s.get("lnA"))
        s["status"] = torch.empty(n, dtype=torch.int32, device="cuda")
        s["h"] = torch.zeros(n, dtype=torch.float64, device="cuda")
        if op == "switch":
            s["meth"] = torch.zeros(n, dtype=torch.int32, device="cuda")
            s["jc"] = m.jac_cache(n)
            o = m.opts(tableau=case["method"], lnA=s.get("lnA"), cell_method=s["meth"],
                       jac_cache=s["jc"], alt_tableau=chem.ROS2W)
        s["opts"], s["ws"] = o, m.workspace(n, o)
    return s


def run(s):
    case, m = s["case"], s["m"]
    op = case["op"]
    if op == "source":
        return {"f": m.eval_source(s["T"], s["P"], s["n"], lnA=s.get("lnA"))}
    if op == "jacobian":
        return {"J": m.eval_jacobian(s["T"], s["P"], s["n"], lnA=s.get("lnA"))}
    if op == "gradient":
        T0 = s["T"].detach().clone().requires_grad_(True)
        Y0 = s["Y"].detach().clone().requires_grad_(True)
        lnA = s["lnA"].detach().clone().requires_grad_(True)
        T, Y = s["fn"].apply(T0, Y0, lnA, m, s["P"], case["dt"], case["rtol"], case["atol"], 2048, 16)
        ((T - s["target"]) ** 2).sum().backward()
        return {"T": T.detach(), "Y": Y.detach(), "gT0": T0.grad, "gY0": Y0.grad, "glnA": lnA.grad}
    # a split step starts from the flow solver's new T and Y; h < = 0 stands for "no step size yet"
    T, Y = s["T"].clone(), s["Y"].clone()
    s["h"].zero_()
    if op == "switch":
        s["meth"].zero_()
    for _ in range(case["splits"]):
        m.integrate(T, s["P"], Y, case["dt"], rtol=case["rtol"], atol=case["atol"], h=s["h"],
                    status=s["status"], opts=s["opts"], workspace=s["ws"])
    return {"T": T, "Y": Y, "h": s["h"].clone(), "status": s["status"].clone()}


# ------------------------------------------------------------------------------ 64-bit reference

# transformed coefficients from the methods' publications: order, gamma, a, c, m, e
_A4 = [1.221224509226641, 6.019134481288629, 12.53708332932087, -0.6878860361058950]
_G2 = 1.0 + 1.0 / math.sqrt(2.0)
METHODS = {
    chem.ROS4: (4, 0.57282, [[], [2.0], [1.867943637803922, 0.2344449711399156],
                             [1.867943637803922, 0.2344449711399156, 0.0]],
                [[], [-7.137615036412310], [2.580708087951457, 0.6515950076447975],
                 [-2.137148994382534, -0.3214669691237626, -0.6949742501781779]],
                [2.255570073418735, 0.2870493262186792, 0.4353179431840180, 1.093502252409163],
                [-0.2815431932141155, -0.07276199124938920, -0.1082196201495311, -1.093502252409163]),
    chem.ROS3: (3, 0.43586652150845899941601945119356, [[], [1.0], [1.0, 0.0]],
                [[], [-1.0156171083877702091975600115545],
                 [4.0759956452537699824805835358067, 9.2076794298330791242156818474003]],
                [1.0, 6.1697947043828245592553615689730, -0.42772256543218573326237383806514],
                [0.5, -2.9079558716805469821718236208017, 0.22354069897811569627360909276199]),
    chem.RODAS3: (3, 0.5, [[], [0.0], [2.0, 0.0], [2.0, 0.0, 1.0]],
                  [[], [4.0], [1.0, -1.0], [1.0, -1.0, -8.0 / 3.0]], [2.0, 0.0, 1.0, 1.0],
                  [0.0, 0.0, 0.0, 1.0]),
    chem.RODAS4: (4, 0.25, [[], [1.544], [0.9466785280815826, 0.2557011698983284],
                            [3.314825187068521, 2.896124015972201, 0.9986419139977817],
                            _A4, _A4 + [1.0]],
                  [[], [-5.6688], [-2.430093356833875, -0.2063599157091915],
                   [-0.1073529058151375, -9.594562251023355, -20.47028614809616],
                   [7.496443313967647, -10.24680431464352, -33.99990352819905, 11.70890893206160],
                   [8.083246795921522, -7.981132988064893, -31.52159432874371, 16.31930543123136,
                    -6.058818238834054]], _A4 + [1.0, 1.0], [0.0, 0.0, 0.0, 0.0, 0.0, 1.0]),
    chem.ROS2W: (2, _G2, [[], [1.0 / _G2]], [[], [-2.0 / _G2]], [1.5 / _G2, 0.5 / _G2],
                 [0.5 / _G2, 0.5 / _G2]),
}


class _Ref:
    """Rates, source, Jacobian and integrators of one mechanism in plain batched torch float64."""

    def __init__(self, mech):
        ns, nr = mech.n_species, mech.n_reactions
        d = _dev
        self.ns, self.nr = ns, nr
        self.W = d(mech.weights())
        self.lo = d(np.array([s.lo for s in mech.species], dtype=float))
        self.hi = d(np.array([s.hi for s in mech.species], dtype=float))
        self.Tmid = d(np.array([s.Tmid for s in mech.species], dtype=float))
        nu = np.zeros((nr, ns))
        slots = np.full((2, nr, 3), ns)  # species of each unit of reaction order; ns: none
        self.kinds = [rx.kind for rx in mech.reactions]
        eff = np.ones((nr, ns))
        p = np.zeros((nr, 10))
        for r, rx in enumerate(mech.reactions):
            for side, (lst, sg) in enumerate(((rx.reac, -1.0), (rx.prod, 1.0))):
                ids = [k for k, v in lst for _ in range(v)]
                slots[side, r, : len(ids)] = ids
                for k in ids:
                    nu[r, k] += sg
            order = sum(v for _, v in rx.reac) + (rx.kind == "THIRD")
            p[r, :3] = math.log(rx.A) + (order - 1) * math.log(1e-3), rx.b, rx.Ea / RCAL
            for k, e in rx.eff:
                eff[r, k] = e
            if rx.kind in FALLOFF:
                order = sum(v for _, v in rx.reac) + 1
                p[r, 3:6] = math.log(rx.low[0]) + (order - 1) * math.log(1e-3), rx.low[1], rx.low[2] / RCAL
            if rx.kind == "TROE":
                p[r, 6:10] = rx.troe
        self.p, self.nu, self.eff = d(p), d(nu), d(eff)
        self.dnu = self.nu.sum(1)
        self.slots = torch.as_tensor(slots).cuda()
        self.onehot = torch.nn.functional.one_hot(self.slots, ns + 1)[..., :ns].to(torch.float64)
        is_ = lambda *ks: torch.tensor([k in ks for k in self.kinds], device="cuda")  # noqa: E731
        self.third, self.fall, self.troe = is_("THIRD"), is_("LIND", "TROE"), is_("TROE")
        self.lnA = self.p[:, 0]
        self.E = torch.cat([torch.eye(ns - 1, dtype=torch.float64, device="cuda"),
                            -(self.W[:-1] / self.W[-1])[None, :]])  # d n_k / d n_j with the bath closure

    # y = [T, n_1 .. n_{ns-1}] per cell
    def state(self, T, Y):
        return torch.cat([T[:, None], (Y / self.W)[:, :-1]], 1)

    def mass(self, y):
        Y = y[:, 1:] * self.W[:-1]
        return y[:, 0], torch.cat([Y, 1.0 - Y.sum(1, keepdim=True)], 1)

    def thermo(self, T):
        a = torch.where((T[:, None] < self.Tmid)[..., None], self.lo, self.hi)
        t = T[:, None]
        a1, a2, a3, a4, a5, a6, a7 = a.unbind(-1)
        cp = a1 + t * (a2 + t * (a3 + t * (a4 + t * a5)))
        h = a1 + t * (a2 / 2 + t * (a3 / 3 + t * (a4 / 4 + t * a5 / 5))) + a6 / t
        s = a1 * torch.log(t) + t * (a2 + t * (a3 / 2 + t * (a4 / 3 + t * a5 / 4))) + a7
        dcp = a2 + t * (2 * a3 + t * (3 * a4 + t * 4 * a5))
        return cp, h, s, dcp

    def source(self, y, P, lnA=None, jac=False):
        """f [C, N] and, asked for, J [C, N, N]."""
        lnA = self.lnA if lnA is None else lnA
        T = y[:, 0]
        t = T[:, None]
        n = y[:, 1:] @ self.E.T
        n = torch.cat([n[:, :-1], n[:, -1:] + 1.0 / self.W[-1]], 1)
        V = n.sum(1) * RU * T / P
        C = n / V[:, None]
        cp, h, s, dcp = self.thermo(T)
        cpm = (n * cp).sum(1)
        p = self.p
        lt, it = torch.log(t), 1.0 / t
        kinf = torch.exp(lnA + p[:, 1] * lt - p[:, 2] * it)
        M = C @ self.eff.T
        dlk = (p[:, 1] + p[:, 2] * it) * it  # d ln k / dT
        dlM = torch.zeros_like(M)            # d ln k / d[M]
        fall = self.fall
        k, g = kinf, None
        if bool(fall.any()):
            Mf = torch.where(fall, M, 1.0)
            Pr = torch.exp(p[:, 3] + p[:, 4] * lt - p[:, 5] * it) * Mf / kinf
            floored = Pr < 1e-300
            Pr = torch.where(floored, 1e-300, Pr)
            a, T3, T1, T2 = (torch.where(self.troe, p[:, 6 + i], 1.0) for i in range(4))
            e3, e1 = (1 - a) * torch.exp(-t / T3), a * torch.exp(-t / T1)
            e2 = torch.where(T2 > 0, torch.exp(-T2 * it), torch.zeros_like(e1))
            Fc = e3 + e1 + e2
            L10 = math.log(10.0)
            lF = torch.log(Fc) / L10
            nn = 0.75 - 1.27 * lF
            x = torch.log(Pr) / L10 - 0.4 - 0.67 * lF
            dd = nn - 0.14 * x
            f1 = x / dd
            q = 1.0 + f1 * f1
            F = torch.where(self.troe, torch.exp(L10 * lF / q), 1.0)
            k = torch.where(fall, kinf * (Pr / (1.0 + Pr)) * F, kinf)
            if jac:
                dPr = torch.where(floored, 0.0, (p[:, 4] + p[:, 5] * it) * it - dlk)  # d ln Pr / dT
                dPrM = torch.where(floored, 0.0, 1.0 / Mf)
                dFc = (-e3 / T3 - e1 / T1 + e2 * T2 * it * it) / (Fc * L10)  # d lF / dT

                def dlnF(dlnPr, dlF):
                    dx = dlnPr / L10 - 0.67 * dlF
                    df1 = (dx * dd - x * (-1.27 * dlF - 0.14 * dx)) / (dd * dd)
                    r = L10 * (dlF / q - lF * 2.0 * f1 * df1 / (q * q))
                    return torch.where(self.troe, r, 0.0)

                dlk = torch.where(fall, dlk + dPr / (1.0 + Pr) + dlnF(dPr, dFc), dlk)
                dlM = torch.where(fall, dPrM / (1.0 + Pr) + dlnF(dPrM, torch.zeros_like(dFc)), dlM)
        lnKc = (s - h) @ self.nu.T + self.dnu * torch.log(PATM / (RU * t))
        kr = k * torch.exp(-lnKc)
        pad = torch.cat([C, torch.ones_like(C[:, :1])], 1)
        c = [[pad[:, self.slots[i, :, j]] for j in range(3)] for i in range(2)]
        fwd, rev = k * c[0][0] * c[0][1] * c[0][2], kr * c[1][0] * c[1][1] * c[1][2]
        m = torch.where(self.third, M, 1.0)
        qn = fwd - rev
        om = (m * qn) @ self.nu
        f = torch.cat([(-T * V * (h * om).sum(1) / cpm)[:, None], V[:, None] * om[:, :-1]], 1)
        if not jac:
            return f
        D = (torch.where(self.third, qn, qn * dlM))[..., None] * self.eff * (~(self.plain))[:, None]
        for i, kk in ((0, m * k), (1, -m * kr)):
            for j in range(3):
                a, b = c[i][(j + 1) % 3], c[i][(j + 2) % 3]
                D = D + (kk * a * b)[..., None] * self.onehot[i, :, j]
        JC = self.nu.T @ D  # d omega / dC at constant T
        dlKc = (h @ self.nu.T - self.dnu) * it
        omT = (m * (fwd * dlk - rev * (dlk - dlKc))) @ self.nu  # d omega / dT at constant C
        gV = self.E.sum(0)  # d n_tot / d n_j
        dV = (RU * T / P)[:, None] * gV
        dC = self.E / V[:, None, None] - n[..., None] * dV[:, None, :] / (V * V)[:, None, None]
        dom = JC @ dC
        domT = omT - (JC @ C[..., None])[..., 0] / t
        # f_k = V omega_k; f_T = -T V sum_k h_k omega_k / cpm
        J = torch.empty((y.shape[0], self.ns, self.ns), dtype=torch.float64, device=y.device)
        Jn = V[:, None, None] * dom[:, :-1] + om[:, :-1, None] * dV[:, None, :]
        JT = V[:, None] * domT[:, :-1] + om[:, :-1] * (V / T)[:, None]
        Q = (h * om).sum(1)
        dh = (cp - h) * it
        dQT = (dh * om + h * domT).sum(1)
        dQn = (h[:, None, :] @ dom)[:, 0]
        dcn = cp @ self.E
        dcT = (n * dcp).sum(1)
        row = torch.cat([(-(2 * V * Q + T * V * dQT - T * V * Q * dcT / cpm) / cpm)[:, None],
                         -(T[:, None] * (dV * Q[:, None] + V[:, None] * dQn)
                           - (T * V * Q / cpm)[:, None] * dcn) / cpm[:, None]], 1)
        J = torch.cat([row[:, None, :], torch.cat([JT[..., None], Jn], 2)], 1)
        return f, J

    @functools.cached_property
    def plain(self):
        return torch.tensor([k == "ELEM" for k in self.kinds], device="cuda")

    def step(self, method, y, P, h, lnA=None, W=None):
        """One step of size h [C] from y: (y_new, error vector, Jacobian used).  `W`: (J, hW) to use."""
        order, gam, a, c, m, e = METHODS[method]
        if W is None:
            f, J = self.source(y, P, lnA, jac=True)
        else:
            f, J = self.source(y, P, lnA), W
        eye = torch.eye(self.ns, dtype=torch.float64, device=y.device)
        lu, piv = torch.linalg.lu_factor(eye / (gam * h)[:, None, None] - J)
        u, prev = [], None
        for i in range(len(m)):
            if i and any(a[i]) and not (i > 1 and a[i] == a[i - 1] + [0.0]):
                g = y + sum(a[i][j] * u[j] for j in range(i) if a[i][j] != 0.0)
                fi = self.source(g, P, lnA)
            elif i and not any(a[i]):
                fi = f
            else:
                fi = f if prev is None else prev
            prev = fi
            b = fi + sum(c[i][j] * u[j] for j in range(i)) / h[:, None] if i else fi
            u.append(torch.linalg.lu_solve(lu, piv, b.unsqueeze(-1)).squeeze(-1))
        return (y + sum(x * v for x, v in zip(m, u) if x), sum(x * v for x, v in zip(e, u) if x), J)

    def integrate(self, y, P, dt, rtol, atol, h, method, lnA=None, budget=None, cache=None, tape=None):
        """Adaptive integration of every cell to dt; status 1 where a cell's attempt budget ran out."""
        order = METHODS[method][0]
        y, h = y.clone(), torch.where(h > 0, h, torch.full_like(h, dt))
        C = y.shape[0]
        t, rej = torch.zeros_like(h), torch.zeros(C, dtype=torch.bool, device=y.device)
        att = torch.zeros(C, dtype=torch.int64, device=y.device)
        status = torch.zeros(C, dtype=torch.int32, device=y.device)
        live = torch.arange(C, device=y.device)
        block = max(16, int(1.5e9 / (8.0 * self.nr * self.ns)))
        while True:
            if budget is not None:
                out = att[live] >= budget[live]
                status[live[out]] = 1
                live = live[~out]
            if not live.numel():
                return y, h, status, att
            keep = []
            for i in live.split(block):
                hi, ti, yi = h[i], t[i], y[i]
                last = ti + 1.0001 * hi >= dt
                hh = torch.where(last, dt - ti, hi)
                W = None
                if cache is not None:
                    new = (cache["h"][i] != hh) | (cache["age"][i] >= 32)
                    j = i[new]
                    if j.numel():
                        cache["J"][j] = self.source(y[j], P[j], lnA, jac=True)[1]
                        cache["h"][j], cache["age"][j] = hh[new], 0
                    W = cache["J"][i]
                yn, ev, _ = self.step(method, yi, P[i], hh, lnA, W)
                att[i] += 1
                sc = atol + rtol * torch.maximum(yi.abs(), yn.abs())
                err = ((ev / sc) ** 2).mean(1).sqrt()
                fin = torch.isfinite(err) & torch.isfinite(yn).all(1)
                fac = (0.9 * torch.clamp(err, min=1e-10) ** (-1.0 / order)).clamp(0.2, 6.0)
                fac = torch.where(fin, fac, torch.full_like(fac, 0.2))
                ok = fin & (err <= 1.0)
                fac = torch.where(ok & rej[i], fac.clamp(max=1.0), fac)
                y[i] = torch.where(ok[:, None], yn, yi)
                rej[i] = ~ok
                if tape is not None:
                    tape.append((i[ok], yi[ok], hh[ok]))
                if cache is not None:
                    cache["age"][i] += ok.to(torch.int64)
                t[i] = torch.where(ok & ~last, ti + hh, ti)
                h[i] = torch.where(ok & last & (hh < hi), hi, hh * fac)
                keep.append(i[~(ok & last)])
            live = torch.cat(keep)

    def gradient(self, y, P, tape, lam, lnA):
        """dL/dy0 and dL/dlnA through the accepted steps (step sizes frozen), from dL/dy_end `lam`."""
        gA = torch.zeros_like(lnA)
        for i, yi, hh in reversed(tape):
            if not i.numel():
                continue
            yi = yi.detach().requires_grad_(True)
            A = lnA.detach().clone().requires_grad_(True)
            yn, _, _ = self.step(chem.ROS4, yi, P[i], hh, A)
            gy, ga = torch.autograd.grad(yn, (yi, A), lam[i])
            lam[i] = gy
            gA += ga
        return lam, gA


@functools.lru_cache(maxsize=None)
def _ref(name):
    return _Ref(_mech(name))


def exact(case, seed):
    mech, r = _mech(case["mech"]), _ref(case["mech"])
    T, P, Y = (_dev(a) for a in _states(mech, case["cells"], case["recipe"], seed))
    lnA = r.lnA
    if case["lnA"]:
        lnA = lnA + _dev(np.random.default_rng([seed, 77]).uniform(-0.2, 0.2, r.nr))
    op, C = case["op"], case["cells"]
    y = r.state(T, Y)
    parts = torch.arange(C, device=y.device).split(max(16, int(1.5e9 / (8.0 * r.nr * r.ns))))
    if op == "source":
        return {"f": torch.cat([r.source(y[i], P[i], lnA) for i in parts]).T.contiguous()}
    if op == "jacobian":
        J = torch.cat([r.source(y[i], P[i], lnA, jac=True)[1] for i in parts])
        return {"J": J.reshape(C, -1).T.contiguous()}
    h = torch.zeros_like(T)
    args = (case["dt"], case["rtol"], case["atol"])
    if op == "gradient":
        tape = []
        ye, h, status, _ = r.integrate(y, P, *args, h, chem.ROS4, lnA, tape=tape)
        T1, Y1 = r.mass(ye)
        target = _dev(np.random.default_rng([seed, 78]).uniform(1500.0, 2500.0, C))
        lam = torch.zeros_like(ye)
        lam[:, 0] = 2.0 * (T1 - target)
        lam, gA = r.gradient(y, P, tape, lam, lnA)
        gY = torch.cat([lam[:, 1:] / r.W[:-1], torch.zeros_like(T)[:, None]], 1)
        return {"T": T1, "Y": Y1.T.contiguous(), "gT0": lam[:, 0].clone(), "gY0": gY.T.contiguous(), "glnA": gA}
    if op == "integrate":
        y, h, status, _ = r.integrate(y, P, *args, h, case["method"], lnA)
    else:
        # quiescent cells (one attempt, next proposal at least 2 dt) take the W-method next time
        meth = torch.zeros(C, dtype=torch.int64, device=y.device)
        cache = {"J": torch.zeros((C, r.ns, r.ns), dtype=torch.float64, device=y.device),
                 "h": torch.zeros_like(T), "age": torch.zeros(C, dtype=torch.int64, device=y.device)}
        for _ in range(case["splits"]):
            w = torch.nonzero(meth > 0)[:, 0]
            part = {k: v[w] for k, v in cache.items()}
            yw, hw, sw, aw = r.integrate(y[w], P[w], *args, h[w], chem.ROS2W, lnA, budget=meth[w], cache=part)
            for k in cache:
                cache[k][w] = part[k]
            done = sw == 0
            y[w[done]], h[w[done]], meth[w[done]] = yw[done], hw[done], 4 * aw[done] + 8
            rest = torch.ones(C, dtype=torch.bool, device=y.device)
            rest[w[done]] = False
            i = torch.nonzero(rest)[:, 0]
            yi, hi, _, ai = r.integrate(y[i], P[i], *args, h[i], case["method"], lnA)
            y[i], h[i] = yi, hi
            meth[i] = torch.where((ai == 1) & (hi >= 2.0 * case["dt"]), 12, 0)
            cache["h"][i] = 0.0
        status = torch.zeros(C, dtype=torch.int32, device=y.device)
    T1, Y1 = r.mass(y)
    return {"T": T1, "Y": Y1.T.contiguous(), "h": h, "status": status}
