"""The calls whose speed is measured, with their inputs and their values in 64 bits.

A case is a solve that a program of this library makes through the public Python API:
an evolution, a gate fidelity, a fidelity with its gradient, an optimiser's step through
autograd, a burst of requests to the server, a batch of small systems, an open-system gate.
``listed`` has one case for each kind of use; ``draw`` gives others of the same ranges.

Energies and amplitudes are rad/ns, times ns; a case holds the step count and dt.

Solves in mixed precision compute their stages in FP32, so the programs here keep what
these return in single precision (complex64 columns, float32 fidelities and gradients);
FP64 solves keep double precision.
"""
import math

import numpy as np
import torch

from paper_2406_18155_gb300 import workloads as W
from paper_2406_18155_gb300 import api
from paper_2406_18155_gb300 import autograd as diff

DEV = "cuda:0"


def listed():
    return [
        # Two coupled transmons, a Gaussian pulse over 50 ns at dt = 5 ps: the whole D = 16
        # propagator and its fidelity, in FP64, as a gate is characterised.
        {"name": "pair_fidelity_fp64", "use": "fidelity", "system": "transmon_pair", "nq": 2, "levels": 4,
         "steps": 10000, "dt": 0.005, "precision": "fp64"},
        # Cross-resonance gate of two fluxoniums, 20 segments over 100 ns: fidelity and the
        # gradient of every pulse and device parameter, the usual step of gate design.
        {"name": "cr_gradient", "use": "gradient", "system": "cr_pair", "nq": 2, "levels": 5,
         "steps": 10000, "dt": 0.01, "precision": "mixed"},
        # Two fluxoniums through a transmon coupler (D = 64), gradient in FP64: the precision
        # asked for when a design converges.
        {"name": "coupler_gradient_fp64", "use": "gradient", "system": "coupler", "nq": 3, "levels": 4,
         "steps": 4000, "dt": 0.01, "precision": "fp64"},
        # The smallest call: one optimiser step on a D = 9 pair over 2 ns, parameters set,
        # eigensystems rebuilt, F and its gradient; latency and launches are all of it.
        {"name": "optimiser_step", "use": "optimise", "system": "multipath_pair", "nq": 2, "levels": 3,
         "steps": 200, "dt": 0.01, "precision": "mixed"},
        # The largest request of the serving stream (five modes of five levels, D = 3125, 32
        # columns), solved alone over 10 ns.
        {"name": "request_d3125", "use": "gradient", "system": "request_fluxonium", "nq": 5, "levels": 5,
         "steps": 1000, "dt": 0.01, "precision": "mixed"},
        # Twelve requests of the serving stream (2-5 modes, 3-5 levels, durations from 20 ns),
        # submitted together and awaited.
        {"name": "serving_burst", "use": "serve", "requests": 12, "slots": 16, "steps_min": 2000,
         "steps_max": 5000, "dt": 0.01, "precision": "mixed"},
        # A chain of six fluxoniums (D = 4096), all 64 computational columns over 60 ns.
        {"name": "chain6_evolve", "use": "evolve", "system": "chain", "nq": 6, "levels": 4, "cols": 64,
         "steps": 6000, "dt": 0.01, "precision": "mixed"},
        # The same chain with the second-order Suzuki-Trotter solver and its pulse gradient.
        {"name": "chain6_trotter_gradient", "use": "gradient", "system": "chain", "nq": 6, "levels": 4, "cols": 64,
         "steps": 300, "dt": 0.01, "precision": "mixed", "solver": "q2", "ham": False},
        # Ring of ten fluxoniums (D = 1,048,576), 16 columns: the large-state workload, forward
        # and pulse gradient in mixed precision (a short piece of its 40 ns).
        {"name": "ring10_gradient", "use": "gradient", "system": "ring", "nq": 10, "levels": 4, "cols": 16,
         "steps": 24, "dt": 0.01, "precision": "mixed", "ham": False},
        # A chain of eight (D = 65,536), 16 columns, every gradient in FP64.
        {"name": "chain8_gradient_fp64", "use": "gradient", "system": "chain", "nq": 8, "levels": 4, "cols": 16,
         "steps": 40, "dt": 0.01, "precision": "fp64"},
        # 512 transmon pairs of different parameters evolved together (a parameter scan).
        {"name": "pairs_batch", "use": "batch", "system": "transmon_pair", "nq": 2, "levels": 4, "count": 512,
         "steps": 2000, "dt": 0.005, "precision": "mixed"},
        # The cross-resonance pair at three levels with damping and dephasing: the open gate's
        # average fidelity and its gradient (16 columns of a D^2 = 81 density operator).
        {"name": "open_gradient", "use": "open", "system": "cr_pair", "nq": 2, "levels": 3,
         "steps": 1000, "dt": 0.01, "precision": "mixed"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    use = rng.choice(["fidelity", "gradient", "gradient", "optimise", "serve", "evolve", "trotter", "tiled", "tiled",
                      "batch", "open"])
    prec = rng.choice(["mixed", "mixed", "fp64"])
    if use == "fidelity":
        return {"use": "fidelity", "system": "transmon_pair", "nq": 2, "levels": rng.choice([3, 4, 5]),
                "steps": _log_int(rng, 100, 10000), "dt": 0.005, "precision": prec}
    if use == "gradient":
        system = rng.choice(["cr_pair", "coupler", "multipath_pair", "request_transmon", "request_fluxonium"])
        nq = {"cr_pair": 2, "coupler": 3, "multipath_pair": 2}.get(system) or rng.choice([2, 3, 4, 5])
        levels = rng.choice([3, 4, 5])
        most = 5000 if levels ** nq <= 125 else 1000
        return {"use": "gradient", "system": system, "nq": nq, "levels": levels, "steps": _log_int(rng, 100, most),
                "dt": 0.01, "precision": prec if levels ** nq <= 125 else "mixed"}
    if use == "optimise":
        return {"use": "optimise", "system": rng.choice(["multipath_pair", "cr_pair"]), "nq": 2,
                "levels": rng.choice([3, 4, 5]), "steps": _log_int(rng, 50, 1000), "dt": 0.01, "precision": prec}
    if use == "serve":
        lo = _log_int(rng, 500, 2000)
        return {"use": "serve", "requests": rng.randint(3, 12), "slots": rng.choice([4, 8, 16]), "steps_min": lo,
                "steps_max": lo + rng.randint(200, 2500), "dt": 0.01, "precision": "mixed"}
    if use == "evolve":
        nq = rng.choice([4, 5, 6])
        return {"use": "evolve", "system": rng.choice(["chain", "ring"]), "nq": nq, "levels": rng.choice([3, 4]),
                "cols": rng.randint(1, 2 ** nq), "steps": _log_int(rng, 100, 3000), "dt": 0.01, "precision": "mixed"}
    if use == "trotter":
        nq = rng.choice([2, 3, 4, 5, 6])
        return {"use": "gradient", "system": "chain", "nq": nq, "levels": rng.choice([3, 4]),
                "cols": rng.randint(1, 2 ** nq), "steps": _log_int(rng, 50, 300), "dt": 0.01, "precision": "mixed",
                "solver": "q2", "ham": False}
    if use == "tiled":
        nq = rng.choice([7, 8, 9])
        return {"use": rng.choice(["evolve", "gradient"]), "system": rng.choice(["chain", "ring"]), "nq": nq,
                "levels": 4, "cols": rng.randint(1, 16), "steps": _log_int(rng, 8, 40), "dt": 0.01,
                "precision": prec, "ham": rng.choice([False, False, True])}
    if use == "batch":
        return {"use": "batch", "system": "transmon_pair", "nq": 2, "levels": 4, "count": _log_int(rng, 16, 512),
                "steps": _log_int(rng, 100, 2000), "dt": 0.005, "precision": "mixed"}
    return {"use": "open", "system": "cr_pair", "nq": 2, "levels": rng.choice([2, 3]),
            "steps": _log_int(rng, 100, 1000), "dt": 0.01, "precision": prec}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _local_rotations(nq, rng):
    """A simultaneous single-qubit gate: on every qubit a rotation by up to pi/4 about a
    random axis of the equator."""
    t = np.ones((1, 1), dtype=np.complex128)
    for _ in range(nq):
        th, al = rng.uniform(0.0, np.pi / 4), rng.uniform(0.0, 2 * np.pi)
        c, s = math.cos(th / 2), math.sin(th / 2)
        t = np.kron(t, np.array([[c, -1j * s * np.exp(-1j * al)], [-1j * s * np.exp(1j * al), c]]))
    return t


def _length(wl, steps, dt):
    wl["T"], wl["dt"] = steps * dt, dt
    for d in wl["drives"]:
        d["length"] = wl["T"]
        if d["env"] == "gaussian":
            d["sigma"], d["t0"] = wl["T"] / 4, wl["T"] / 2
    return wl


def _workload(case, seed):
    rng = np.random.Generator(np.random.PCG64([int(seed), 77]))
    nq, lv, steps, dt = case["nq"], case["levels"], case["steps"], case["dt"]
    T = steps * dt
    system = case["system"]
    seed = int(rng.integers(0, 2 ** 31))
    if system == "transmon_pair":
        wl = W.transmon_pair(seed, T=T, dt=dt)
    elif system == "cr_pair":
        wl = W.fluxonium_pair_cr(seed, T=T, dt=dt)
    elif system == "multipath_pair":
        wl = W.fluxonium_pair_multipath(seed, T=T, dt=dt, levels=lv)
    elif system == "coupler":
        wl = W.coupler_scheme(seed, T=T, dt=dt, levels=(lv, lv, lv))
    elif system in ("request_transmon", "request_fluxonium"):
        wl = W.serving_request(rng, dt=dt, nq=nq, kind=system[8:], levels=lv)
    else:
        wl = W.fluxonium_chain(seed, nq=nq, levels=lv, T=T, dt=dt, ring=system == "ring", ncols=case["cols"])
        wl["target"] = _local_rotations(nq, rng)
    if system in ("transmon_pair", "cr_pair"):
        for m in wl["modes"]:
            m["levels"] = lv
        wl["col_index"] = list(range(lv * lv)) if system == "transmon_pair" else W.comp_states([lv, lv])
    _length(wl, steps, dt)
    if case["use"] == "open":
        # damping (level k -> k - 1) and dephasing on both modes, at T1 and T2 of tens of microseconds
        lower = np.diag(np.sqrt(np.arange(1.0, lv)), 1).astype(np.complex128)
        level = np.diag(np.arange(float(lv))).astype(np.complex128)
        wl["collapse"] = [c for i in range(2) for c in (
            {"mode": i, "L": lower, "rate": float(rng.uniform(1e-5, 1e-4))},
            {"mode": i, "L": level, "rate": float(rng.uniform(1e-5, 1e-4))})]
    return wl


def _requests(case, seed):
    rng = np.random.Generator(np.random.PCG64([int(seed), 78]))
    # every seed gives other devices, pulses, targets and durations of the same mix of shapes
    shapes = [(2 + i % 4, ("transmon", "fluxonium")[(i // 2) % 2], 3 + (i * 2) % 3) for i in range(case["requests"])]
    out = []
    for i, (nq, kind, lv) in enumerate(shapes):
        wl = W.serving_request(rng, dt=case["dt"], nq=nq, kind=kind, levels=lv)
        lo, hi = case["steps_min"], case["steps_max"]
        out.append(_length(wl, lo + (hi - lo) * ((i * 5) % 12) // 11 + int(rng.integers(0, 20)), case["dt"]))
    return out


def _batch(case, seed):
    return [_workload(case, 1000003 * int(seed) + i) for i in range(case["count"])]


def prepare(case, seed):
    st = {"case": dict(case)}
    ctx = st["ctx"] = api.Context(0)
    use = case["use"]
    if use == "serve":
        st["wls"] = _requests(case, seed)
    elif use == "batch":
        st["wls"] = _batch(case, seed)
    else:
        st["wls"] = [_workload(case, seed)]
    st["systems"] = [api.System.from_workload(ctx, wl) for wl in st["wls"]]
    for s in st["systems"]:
        s.prepare()
    if use == "serve":
        st["server"] = api.Server(ctx, mem_budget_bytes=64 << 30, max_slots=case["slots"])
    if use == "optimise":
        # a program's own parameters, a little off the values that the system was built with
        rng = np.random.Generator(np.random.PCG64([int(seed), 79]))
        pulse, ham = st["systems"][0].get_params()
        st["pulse"] = torch.tensor(pulse * (1 + 0.01 * rng.standard_normal(pulse.size)), requires_grad=True)
        st["ham"] = torch.tensor(ham * (1 + 0.001 * rng.standard_normal(ham.size)), requires_grad=True)
    return st


def _single(case, v):
    """A mixed-precision result in single precision, an FP64 one as it is."""
    if case["precision"] != "mixed":
        return v
    if isinstance(v, torch.Tensor):
        return v.to(torch.complex64 if v.is_complex() else torch.float32)
    v = np.asarray(v)
    return v.astype(np.complex64 if v.dtype.kind == "c" else np.float32)


def run(st):
    case, wl, s = st["case"], st["wls"][0], st["systems"][0]
    prec = case["precision"]
    use = case["use"]
    if use == "evolve":
        return {"psi": _single(case, s.evolve(wl["T"], wl["dt"], precision=prec, col_index=wl["col_index"]))}
    if use == "batch":
        return {"psi": _single(case, api.evolve_batch(st["systems"], wl["T"], wl["dt"], wl["col_index"]))}
    if use == "fidelity":
        Fa, Fs, U = s.fidelity(wl["T"], wl["dt"], wl["target"], wl["col_index"], precision=prec)
        return {"F_avg": _single(case, Fa), "F_state": _single(case, Fs), "U": _single(case, U)}
    if use == "gradient":
        F, gp, gh = s.fidelity_grad(wl["T"], wl["dt"], wl["target"], wl["col_index"], kind=wl["fid_kind"],
                                    precision=prec, ham=case.get("ham", True), solver=case.get("solver", "rk4"))
        return _gradient(case, F[1 if wl["fid_kind"] == "state" else 0], gp, gh)
    if use == "optimise":
        F = diff.fidelity(s, st["pulse"], st["ham"], wl["T"], wl["dt"], wl["target"], wl["col_index"],
                          kind=wl["fid_kind"], precision=prec)
        gp, gh = torch.autograd.grad(F, [st["pulse"], st["ham"]])
        return _gradient(case, F.detach(), gp, gh)
    if use == "open":
        F, gp, gh = s.gate_fidelity_open_grad(wl["T"], wl["dt"], wl["target"], precision=prec, ham=True)
        return _gradient(case, F[0], gp, gh)
    srv = st["server"]
    tickets = [srv.submit(sy, w["T"], w["dt"], w["target"], w["col_index"], kind=w["fid_kind"], precision=prec)
               for sy, w in zip(st["systems"], st["wls"])]
    out = []
    for t in tickets:
        r = srv.wait(t)
        if r["status"] != 0:
            raise RuntimeError(r["error"])
        out.append(_gradient(case, r["F"][0], r["grad_pulse"], r["grad_ham"]))
    return out


def _gradient(case, F, gp, gh):
    return {"F": _single(case, F), "pulse": _single(case, gp), "ham": None if gh is None else _single(case, gh)}


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _solve_work(nq, nterm1, nterm2, levels, cols, steps, grad, size=8):
    """Flops of one solve: four stages a step, each a contraction per one-body term and two
    per coupling over the column entries (the operators couple every second level, a real
    number by a complex one is two multiply-adds), and the stage update (four); a gradient
    needs the states, the co-states (as much again) and a complex product per term."""
    d = levels
    D = d ** nq
    apply = 4 * D * cols * (4 * ((d // 2) * (nterm1 + 2 * nterm2) + 4))
    flops = steps * apply * (2 if grad else 1)
    if grad:
        flops += steps * 4 * D * cols * 8 * (nterm1 + nterm2)
    return flops


def work(case):
    use, c16 = case["use"], 8 if case["precision"] == "mixed" else 16
    if use == "serve":
        flops = moved = 0
        for i in range(case["requests"]):
            nq, lv = 2 + i % 4, 3 + (i * 2) % 3
            steps = case["steps_min"] + (case["steps_max"] - case["steps_min"]) * ((i * 5) % 12) // 11 + 10
            flops += _solve_work(nq, nq, nq - 1, lv, 2 ** nq, steps, True)
            moved += 16 * 4 ** nq + 8 * 2 * (10 * nq + 4 * nq)
        return {"bytes": moved, "flops": flops}
    nq, lv, steps = case["nq"], case["levels"], case["steps"]
    edges = {"coupler": 3, "multipath_pair": 2, "ring": nq}.get(case["system"], nq - 1)
    drives = {"transmon_pair": 1, "cr_pair": 1, "coupler": 2}.get(case["system"], nq)
    cols = case.get("cols") or {"transmon_pair": lv * lv, "coupler": 4}.get(case["system"], 2 ** nq)
    if use == "open":
        # density operators: twice the modes, couplings and drives, jumps, D_c^2 columns
        return {"bytes": 16 * 16 + 800,
                "flops": _solve_work(4, 2 * drives + 4, 2 * edges + 4, lv, 16, steps, True)}
    grad = use in ("gradient", "optimise")
    flops = _solve_work(nq, drives, edges, lv, cols, steps, grad)
    if use in ("evolve", "batch"):
        n = case.get("count", 1)
        return {"bytes": n * (c16 * lv ** nq * cols + 200), "flops": n * flops}
    return {"bytes": 16 * 4 ** nq + 8 * 2 * (10 * drives + 3 * nq + edges), "flops": flops}


# ---------------------------------------------------------------------------
# the same values in 64 bits: plain numpy and torch
# ---------------------------------------------------------------------------
def _mode_exact(m):
    """Lowest levels of one mode and their first derivatives in (E_J, E_C, E_L):
    E, n, phi and dE, dn, dphi as numpy arrays (perturbation theory over the full basis)."""
    if m["kind"] == "transmon":
        q = np.arange(-m["ncut"], m["ncut"] + 1.0) - m["ng"]
        M = q.size
        cos = 0.5 * (np.eye(M, k=1) + np.eye(M, k=-1))
        H = 4 * m["ec"] * np.diag(q * q) - m["ej"] * cos
        zero = np.zeros((M, M), complex)
        ops, dH = [np.diag(q) + 0j, zero], [-cos, 4 * np.diag(q * q), 0 * cos]
        dops = [[zero] * 3, [zero] * 3]
    else:
        M, ec, el = m["n_osc"], m["ec"], m["el"]
        low = np.diag(np.sqrt(np.arange(1.0, M)), 1)
        x, p = (low + low.T) / math.sqrt(2), 1j * (low.T - low) / math.sqrt(2)
        node, vec = np.linalg.eigh(x)
        z = (8 * ec / el) ** 0.25
        w = math.sqrt(8 * ec * el)
        ladder = np.diag(np.arange(M) + 0.5)
        arg = z * node - m["phi_ext"]
        cos = (vec * np.cos(arg)) @ vec.T
        slope = -(vec * (node * np.sin(arg))) @ vec.T          # d cos / dz
        dz, dw = [0.0, z / (4 * ec), -z / (4 * el)], [0.0, w / (2 * ec), w / (2 * el)]
        H = w * ladder - m["ej"] * cos
        dH = [dw[k] * ladder - m["ej"] * dz[k] * slope - (cos if k == 0 else 0) for k in range(3)]
        ops = [p / z, z * x + 0j]
        dops = [[-p * dz[k] / z ** 2 for k in range(3)], [dz[k] * x + 0j for k in range(3)]]
    e, v = np.linalg.eigh(H)
    for j in range(M):
        first = np.flatnonzero(np.abs(v[:, j]) >= 1e-3 * np.abs(v[:, j]).max())[0]
        v[:, j] *= np.sign(v[first, j])
    d = m["levels"]
    kept = v[:, :d]
    dE, dO = [], [[], []]
    for k in range(3):
        h = v.T @ dH[k] @ v
        gap = e[None, :d] - e[:, None]
        np.fill_diagonal(gap, np.inf)
        dv = v @ (h[:, :d] / gap)
        dE.append(np.diag(h)[:d] - h[0, 0])
        for o in range(2):
            dO[o].append(dv.T @ ops[o] @ kept + kept.T @ ops[o] @ dv + kept.T @ dops[o][k] @ kept)
    return {"E": e[:d] - e[0], "n": kept.T @ ops[0] @ kept, "phi": kept.T @ ops[1] @ kept,
            "dE": np.array(dE), "dn": np.array(dO[0]), "dphi": np.array(dO[1])}


class _Exact:
    """One workload in complex128 on the GPU: its parameters as leaves, its operators and
    drive coefficients as differentiable tensors of them (first order at these values)."""

    def __init__(self, wl):
        self.wl, self.dims = wl, [m["levels"] for m in wl["modes"]]
        self.nq, self.D = len(self.dims), int(np.prod(self.dims))
        self.dt, self.N = wl["dt"], int(round(wl["T"] / wl["dt"]))
        t = lambda v: torch.tensor(v, device=DEV)  # noqa: E731
        self.dev, self.modes = [], []
        for m in wl["modes"]:
            x = _mode_exact(m)
            at = t(np.zeros(3)).requires_grad_()              # offsets of (E_J, E_C, E_L)
            lin = lambda v, dv: t(v) + torch.einsum("k,k...->...", at.to(t(dv).dtype), t(dv))  # noqa: E731,B023
            self.dev.append(at)
            self.modes.append({"E": lin(x["E"], x["dE"]), "n": lin(x["n"], x["dn"]), "phi": lin(x["phi"], x["dphi"])})
        self.J = [t(np.float64(c["J"])).requires_grad_() for c in wl["couplings"]]
        self.amps = [t(np.array(d["amps"] if d["env"] == "pwc" else [d["amp"]], float)).requires_grad_()
                     for d in wl["drives"]]
        # RK4 stage times (step start, middle, end) x steps
        n = torch.arange(self.N, device=DEV, dtype=torch.float64)
        self.t = torch.stack([n * self.dt, (n + 0.5) * self.dt, (n + 1) * self.dt], 1)

    def leaves(self):
        return self.amps + self.dev + self.J

    def drive(self, k, t):
        """f_k at times t (steps, any): the segment is the one that holds the step's middle."""
        d = self.wl["drives"][k]
        if d["env"] == "pwc":
            seg = ((2 * torch.arange(self.N, device=DEV) + 1) * len(d["amps"])) // (2 * self.N)
            env = self.amps[k][seg][:, None]
        else:
            env = self.amps[k] * torch.exp(-((t - d["t0"]) / d["sigma"]) ** 2 / 2)
        return env * torch.cos(self.modes[d["omega_mode"]]["E"][1] * t + d["phase"])

    def turned(self, op, i, t):
        """op of mode i in the interaction frame at times t."""
        ph = torch.polar(torch.ones_like(t)[..., None], t[..., None] * self.modes[i]["E"])
        return op * ph[..., :, None] * ph[..., None, :].conj()

    def rows(self):
        """Matrices of every term at every stage time: [(modes, matrices (steps, 3, d, d) each)]."""
        out = []
        for k, d in enumerate(self.wl["drives"]):
            f = self.drive(k, self.t)[..., None, None]
            out.append(((d["mode"],), [f * self.turned(self.modes[d["mode"]][d["op"]], d["mode"], self.t)]))
        for c, J in zip(self.wl["couplings"], self.J):
            a, b = c["a"], c["b"]
            out.append(((a, b), [J * self.turned(self.modes[a][c["op_a"]], a, self.t),
                                 self.turned(self.modes[b][c["op_b"]], b, self.t)]))
        return out

    def total_energy(self):
        e = torch.zeros(1, device=DEV, dtype=torch.float64)
        for m in self.modes:
            e = (e[:, None] + m["E"][None, :]).reshape(-1)
        return e

    def lab(self):
        return torch.polar(torch.ones_like(self.total_energy()), -self.total_energy() * self.N * self.dt)

    def comp(self):
        """Flat indices of the computational states (couplers in their lowest level)."""
        at = [0]
        for m, d in zip(self.wl["modes"], self.dims):
            at = [x * d + b for x in at for b in ((0,) if m.get("coupler") else (0, 1))]
        return at

    def loss(self, psi):
        """The workload's fidelity of lab-frame columns psi (D, columns), and the block."""
        comp = self.comp()
        tgt = torch.tensor(np.asarray(self.wl["target"]), device=DEV)
        U = psi[comp]
        cols = [comp.index(c) if c in comp else -1 for c in self.wl["col_index"]]
        on = [s for s, j in enumerate(cols) if j >= 0]
        z = (tgt[:, [cols[s] for s in on]].conj() * U[:, on]).sum()
        n = len(comp)
        Fa = ((tgt.conj().T @ U[:, on]).abs().square().sum() + z.abs() ** 2) / (n * (n + 1))
        return Fa, (z / len(on)).abs() ** 2, U

    def grads(self, F, extra=()):
        """dF/d(pulse), dF/d(device and couplings) from F, or from table co-gradients `extra`."""
        heads, seeds = ([F], [None]) if F is not None else zip(*extra)
        g = torch.autograd.grad(list(heads), self.leaves(), list(seeds), allow_unused=True)
        g = [torch.zeros_like(v) if x is None else x for v, x in zip(self.leaves(), g)]
        na, nm = len(self.amps), len(self.dev)
        for m, x in zip(self.wl["modes"], g[na:na + nm]):
            if m["kind"] == "transmon":
                x[2] = 0.0
        return torch.cat(g[:na]), torch.cat(g[na:na + nm] + [x.reshape(1) for x in g[na + nm:]])


def _rk4_maps(A1, A2, A3, h):
    """RK4 step maps of y' = A(t) y for stacks of dense generators."""
    eye = torch.eye(A1.shape[-1], device=DEV, dtype=A1.dtype)
    k2 = A2 + h / 2 * (A2 @ A1)
    k3 = A2 + h / 2 * (A2 @ k2)
    k4 = A3 + h * (A3 @ k3)
    return eye + h / 6 * (A1 + 2 * k2 + 2 * k3 + k4)


def _product(R):
    """R[-1] ... R[1] R[0] by halves."""
    while R.shape[0] > 1:
        pair = R[1::2] @ R[0:R.shape[0] - R.shape[0] % 2:2]
        R = torch.cat([pair, R[-1:]]) if R.shape[0] % 2 else pair
    return R[0]


def _embed(dims, mats):
    """Kronecker product over the modes of stacks of matrices {mode: (..., d, d)}."""
    out = torch.ones((1, 1), device=DEV, dtype=torch.complex128)
    for i, d in enumerate(dims):
        m = mats.get(i, torch.eye(d, device=DEV, dtype=torch.complex128))
        out = torch.einsum("...ab,...cd->...acbd", out, m)
        out = out.reshape(out.shape[:-4] + (out.shape[-4] * d, out.shape[-2] * d))
    return out


def _dense_hamiltonian(x):
    return sum(_embed(x.dims, dict(zip(at, m))) for at, m in x.rows())


def _dense_columns(x):
    A = -1j * _dense_hamiltonian(x)
    U = _product(_rk4_maps(A[:, 0], A[:, 1], A[:, 2], x.dt))
    return x.lab()[:, None] * U[:, x.wl["col_index"]]


def _act(m, i, y, dims):
    """m on mode i of columns y (D, S)."""
    left, d = int(np.prod(dims[:i])), dims[i]
    return torch.matmul(m, y.reshape(left, d, -1)).reshape(y.shape)


def _apply(terms, j, y, dims):
    out = None
    for at, ms in terms:
        v = y
        for i, m in zip(reversed(at), reversed(ms)):
            v = _act(m[j], i, v, dims)
        out = v if out is None else out + v
    return -1j * out


def _step(terms, y, h, dims):
    k1 = _apply(terms, 0, y, dims)
    k2 = _apply(terms, 1, y + h / 2 * k1, dims)
    k3 = _apply(terms, 1, y + h / 2 * k2, dims)
    k4 = _apply(terms, 2, y + h * k3, dims)
    return y + h / 6 * (k1 + 2 * k2 + 2 * k3 + k4)


def _start(x):
    y = torch.zeros((x.D, len(x.wl["col_index"])), device=DEV, dtype=torch.complex128)
    y[x.wl["col_index"], range(y.shape[1])] = 1.0
    return y


def _by_steps(x, tables, step, y, grad):
    """Columns after all steps of y' = step(tables at n, y) and, with grad, a function that
    pulls a co-state back and returns the tables' co-gradients."""
    past = []
    with torch.no_grad():
        for n in range(x.N):
            if grad:
                past.append(y)
            y = step([t[n] for t in tables], y)

    def back(bar):
        g = [torch.zeros_like(t) for t in tables]
        for n in reversed(range(x.N)):
            at = [t[n].detach().requires_grad_() for t in tables]
            yn = past.pop().requires_grad_()
            out = step(at, yn)
            got = torch.autograd.grad(out, [yn] + at, bar)
            bar = got[0]
            for a, v in zip(g, got[1:]):
                a[n] += v
        return g

    return y, back


def _rk4_by_steps(x, grad):
    rows = x.rows()
    shape = [(at, len(ms)) for at, ms in rows]
    tables = [m for _, ms in rows for m in ms]

    def step(ts, y):
        it = iter(ts)
        return _step([(at, [next(it) for _ in range(c)]) for at, c in shape], y, x.dt, x.dims)

    y, back = _by_steps(x, tables, step, _start(x), grad)
    return tables, y, back


def _q2_by_steps(x, grad):
    """Second-order Suzuki-Trotter: one-body terms in mode order, couplings in order, each
    over half a step, then all in reverse; lab frame, drives at the step's middle."""
    h = x.dt
    mid = x.t[:, 1:2]
    one = []
    for i in range(x.nq):
        H = torch.diag(x.modes[i]["E"]).to(torch.complex128)[None].expand(x.N, -1, -1)
        for k, d in enumerate(x.wl["drives"]):
            if d["mode"] == i:
                H = H + x.drive(k, mid)[:, :, None] * x.modes[i][d["op"]]
        one.append(torch.linalg.matrix_exp(-0.5j * h * H))
    two = []
    for c, J in zip(x.wl["couplings"], x.J):
        ab = J * torch.kron(x.modes[c["a"]][c["op_a"]], x.modes[c["b"]][c["op_b"]])
        two.append(((c["a"], c["b"]), torch.linalg.matrix_exp(-0.5j * h * ab).detach()))

    def pair(at, u, y):
        a, b = at
        v = y.reshape(x.dims + [-1]).movedim((a, b), (0, 1))
        full = v.shape
        v = (u @ v.reshape(u.shape[0], -1)).reshape(full)
        return v.movedim((0, 1), (a, b)).reshape(y.shape)

    def step(us, y):
        for i, u in enumerate(us):
            y = _act(u, i, y, x.dims)
        for at, u in two + two[::-1]:
            y = pair(at, u, y)
        for i, u in reversed(list(enumerate(us))):
            y = _act(u, i, y, x.dims)
        return y

    y, back = _by_steps(x, one, step, _start(x), grad)
    return one, y, back


def _open_gate(x):
    """Average fidelity of the open gate: the channel on the computational block from the
    vectorised master equation (row-major), damping in the interaction frame."""
    H = _dense_hamiltonian(x)
    eye = torch.eye(x.D, device=DEV, dtype=torch.complex128)

    def kron(a, b):
        v = torch.einsum("...ab,...cd->...acbd", a, b)
        return v.reshape(v.shape[:-4] + (x.D ** 2, x.D ** 2))

    A = -1j * (kron(H, eye) - kron(eye, H.transpose(-1, -2)))
    for c in x.wl["collapse"]:
        L = _embed(x.dims, {c["mode"]: x.turned(torch.tensor(c["L"], device=DEV), c["mode"], x.t)})
        LL = L.mH @ L
        A = A + c["rate"] * (kron(L, L.conj()) - kron(LL, eye) / 2 - kron(eye, LL.transpose(-1, -2)) / 2)
    U = _product(_rk4_maps(A[:, 0], A[:, 1], A[:, 2], x.dt))
    lab = x.lab()
    U = (lab[:, None] * lab.conj()[None, :]).reshape(-1, 1) * U
    comp = x.comp()
    n = len(comp)
    at = [a * x.D + b for a in comp for b in comp]
    S = U[at][:, at]
    tgt = torch.tensor(np.asarray(x.wl["target"]), device=DEV)
    pro = (torch.kron(tgt, tgt.conj()).conj() * S).sum().real / n ** 2
    diag = [a * n + a for a in range(n)]
    kept = S[diag][:, diag].sum().real
    return (n * n * pro + kept) / (n * (n + 1))


def _solve_exact(case, wl, use):
    x = _Exact(wl)
    grad = use in ("gradient", "optimise")
    if use == "open":
        F = _open_gate(x)
        gp, gh = x.grads(F)
        return {"F": F.detach(), "pulse": gp, "ham": gh}
    q2 = case.get("solver") == "q2"
    if not q2 and x.D <= 128:
        with torch.set_grad_enabled(grad):
            psi = _dense_columns(x)
        if grad:
            F = x.loss(psi)[1 if wl["fid_kind"] == "state" else 0]
            gp, gh = x.grads(F)
    else:
        tables, psi, back = (_q2_by_steps if q2 else _rk4_by_steps)(x, grad)
        lab = torch.ones(x.D, device=DEV, dtype=torch.complex128) if q2 else x.lab()
        if not grad:
            psi = lab[:, None] * psi
        else:
            leaf = psi.requires_grad_()
            F = x.loss(lab[:, None] * leaf)[1 if wl["fid_kind"] == "state" else 0]
            (bar,) = torch.autograd.grad(F, [leaf], retain_graph=True)
            g = back(bar)
            extra = list(zip(tables, g)) + ([(F, torch.ones_like(F))] if not q2 else [])
            gp, gh = x.grads(None, extra)
    if grad:
        return {"F": F.detach(), "pulse": gp, "ham": gh if case.get("ham", True) else None}
    if use == "fidelity":
        Fa, Fs, U = x.loss(psi)
        return {"F_avg": Fa, "F_state": Fs, "U": U}
    return {"psi": psi}


def exact(case, seed):
    use = case["use"]
    if use == "serve":
        wls = _requests(case, seed)
        # the dense form covers the requests up to D = 125; the larger ones take too long here
        return [_solve_exact(case, wl, "gradient") if np.prod([m["levels"] for m in wl["modes"]]) <= 128 else
                {"F": None, "pulse": None, "ham": None} for wl in wls]
    if use == "batch":
        wls = _batch(case, seed)
        with torch.no_grad():
            return {"psi": torch.stack([_solve_exact(case, wl, "evolve")["psi"] for wl in wls])}
    wl = _workload(case, seed)
    if use == "optimise":
        # the parameters that prepare() moved off the workload's values
        rng = np.random.Generator(np.random.PCG64([int(seed), 79]))
        amps = np.concatenate([np.atleast_1d(d["amps"] if d["env"] == "pwc" else d["amp"]) for d in wl["drives"]])
        amps = amps * (1 + 0.01 * rng.standard_normal(amps.size))
        ham = np.array([v for m in wl["modes"] for v in (m["ej"], m["ec"], m.get("el", 0.0))] +
                       [c["J"] for c in wl["couplings"]])
        ham = ham * (1 + 0.001 * rng.standard_normal(ham.size))
        for d in wl["drives"]:
            d["amps"], amps = list(amps[:len(d["amps"])]), amps[len(d["amps"]):]
        for i, m in enumerate(wl["modes"]):
            m["ej"], m["ec"] = ham[3 * i], ham[3 * i + 1]
            if m["kind"] == "fluxonium":
                m["el"] = ham[3 * i + 2]
        for c, J in zip(wl["couplings"], ham[3 * len(wl["modes"]):]):
            c["J"] = float(J)
    return _solve_exact(case, wl, use)
