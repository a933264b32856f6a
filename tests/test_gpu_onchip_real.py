"""Real-operator on-chip kernels, forward and gradient: every routing of couplings through the pairs of
modes (own pair, two on one pair, images between phases from either digit, several images at
once, odd mode counts), level counts and column counts, against the general gather kernels;
and plans that they do not take.  Amplitudes and F within 1e-10 (FP64) and 1e-5 (mixed),
gradients within 1e-8 and 1e-3 of the largest component, as for the other kernel families."""
import numpy as np
import pytest

from paper_2406_18155_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# name: modes, levels, couplings (a, op_a, b, op_b), modes driven, columns
PLANS = {
    "pair_l2": (2, 2, [(0, "n", 1, "n")], [0, 1], 3),
    "pair_reversed_l5": (2, 5, [(1, "n", 0, "n")], [1], 4),
    "multipath_l3": (2, 3, [(0, "n", 1, "n"), (0, "phi", 1, "phi")], [0, 1], 4),
    "no_coupling_l4": (3, 4, [], [0, 2], 5),
    "no_drive_l3": (3, 3, [(0, "n", 1, "n"), (1, "n", 2, "n")], [], 8),
    "triangle_l4": (3, 4, [(0, "n", 1, "n"), (1, "n", 2, "n"), (0, "n", 2, "n")], [0, 1, 2], 8),
    "chain4_l5": (4, 5, [(0, "n", 1, "n"), (1, "n", 2, "n"), (2, "n", 3, "n")], [0, 1, 2, 3], 3),
    "ring4_l3": (4, 3, [(0, "n", 1, "n"), (1, "n", 2, "n"), (2, "n", 3, "n"), (3, "n", 0, "n")], [0, 1, 2, 3], 16),
    "ring5_l4": (5, 4, [(i, "n", (i + 1) % 5, "n") for i in range(5)], [0, 1, 2, 3, 4], 7),
    "chain5_l5": (5, 5, [(i, "n", i + 1, "n") for i in range(4)], [0, 1, 2, 3, 4], 2),
    "ring6_l3": (6, 3, [(i, "n", (i + 1) % 6, "n") for i in range(6)], [0, 1, 2, 3, 4, 5], 9),
    "chain6_l4": (6, 4, [(i, "n", i + 1, "n") for i in range(5)], [0, 1, 2, 3, 4, 5], 2),
    "star5_l3": (5, 3, [(2, "n", k, "phi" if k == 9 else "n") for k in (0, 1, 3, 4)], [2], 5),
    "mixed_ops_l4": (4, 4, [(0, "n", 2, "n"), (1, "phi", 3, "phi"), (0, "phi", 3, "phi")], [1, 2], 6),
    "two_drives_l3": (3, 3, [(0, "n", 1, "n"), (2, "n", 1, "n")], [1, 1, 2], 8),
}


def _workload(name, steps=13, dt=0.01):
    nq, lv, edges, driven, cols = PLANS[name]
    wl = W.fluxonium_chain(seed=len(name), nq=nq, levels=lv, T=steps * dt, dt=dt, nseg=3, ncols=min(cols, 2 ** nq))
    wl["couplings"] = [{"a": a, "op_a": oa, "b": b, "op_b": ob, "J": W.MHZ * (12.0 + 3 * i)}
                       for i, (a, oa, b, ob) in enumerate(edges)]
    base = wl["drives"]
    wl["target"] = W.haar_unitary(2 ** nq, np.random.Generator(np.random.PCG64(5)))
    wl["drives"] = [dict(base[m], amps=[x * (1 + 0.3 * i) for x in base[m]["amps"]], phase=0.2 * i)
                    for i, m in enumerate(driven)]
    return wl


@pytest.mark.parametrize("name", sorted(PLANS))
def test_real_forward_matches_the_general_kernels(sgctx, monkeypatch, name):
    from paper_2406_18155_gb300.api import System
    wl = _workload(name)
    s = System.from_workload(sgctx, wl)
    s.prepare()
    kw = dict(col_index=wl["col_index"])
    psi = {p: s.evolve(wl["T"], wl["dt"], precision=p, **kw).cpu().numpy() for p in ("fp64", "mixed")}
    start = W.random_columns(s.dims()[0], 3, seed=1)
    import torch
    own = s.evolve(wl["T"], wl["dt"], precision="fp64", psi=torch.tensor(start, device="cuda:0")).cpu().numpy()
    monkeypatch.setenv("SG_PATH", "gather")
    ref = s.evolve(wl["T"], wl["dt"], precision="fp64", **kw).cpu().numpy()
    ref_own = s.evolve(wl["T"], wl["dt"], precision="fp64", psi=torch.tensor(start, device="cuda:0")).cpu().numpy()
    assert np.max(np.abs(psi["fp64"] - ref)) <= 1e-10
    assert np.max(np.abs(psi["mixed"] - ref)) <= 1e-5
    assert np.max(np.abs(own - ref_own)) <= 1e-10


@pytest.mark.parametrize("name", sorted(PLANS))
def test_real_gradient_matches_the_general_kernels(sgctx, monkeypatch, name):
    from paper_2406_18155_gb300.api import System
    wl = _workload(name, steps=9)
    s = System.from_workload(sgctx, wl)
    s.prepare()
    args = (wl["T"], wl["dt"], wl["target"], wl["col_index"])
    got = {(p, k): s.fidelity_grad(*args, kind="state", precision=p, ckpt=k)
           for p in ("fp64", "mixed") for k in (0, 4)}
    pulse = s.fidelity_grad(*args, kind="state", precision="fp64", ham=False)
    monkeypatch.setenv("SG_PATH", "gather")
    F, gp, gh = s.fidelity_grad(*args, kind="state", precision="fp64")
    g = np.concatenate([gp, gh])
    scale = np.max(np.abs(g))
    for (p, _), (f, a, b) in got.items():
        ta, tg = (1e-10, 1e-8) if p == "fp64" else (1e-5, 1e-3)
        assert abs(f[1] - F[1]) <= ta
        assert np.max(np.abs(np.concatenate([a, b]) - g)) <= tg * scale, p
    if gp.size:
        assert np.max(np.abs(pulse[1] - gp)) <= 1e-8 * scale


def _charge_driven():
    # charge drives (imaginary on a fluxonium) on two of three modes, n (x) n and n (x) phi couplings
    wl = _workload("triangle_l4", steps=9)
    wl["couplings"][1]["op_b"] = "phi"
    wl["couplings"] = wl["couplings"][:2]
    for d in wl["drives"][:2]:
        d["op"] = "n"
    wl["drives"] = wl["drives"][:2]
    return wl


@pytest.mark.parametrize("make", [lambda: W.coupler_scheme(seed=2, kind="ftf", T=0.09),
                                  lambda: W.coupler_scheme(seed=3, kind="ftf", T=0.09, levels=(3, 3, 3)),
                                  _charge_driven])
def test_turned_modes_match_the_general_kernels(sgctx, monkeypatch, make):
    # a real factor against an imaginary one: a mode's odd levels are turned by i
    from paper_2406_18155_gb300.api import System
    wl = make()
    s = System.from_workload(sgctx, wl)
    s.prepare()
    args = (wl["T"], wl["dt"], wl["target"], wl["col_index"])
    got = {p: (s.evolve(wl["T"], wl["dt"], precision=p, col_index=wl["col_index"]).cpu().numpy(),
               s.fidelity_grad(*args, kind="state", precision=p)) for p in ("fp64", "mixed")}
    monkeypatch.setenv("SG_PATH", "gather")
    ref = s.evolve(wl["T"], wl["dt"], precision="fp64", col_index=wl["col_index"]).cpu().numpy()
    F, gp, gh = s.fidelity_grad(*args, kind="state", precision="fp64")
    g = np.concatenate([gp, gh])
    for p, (psi, (f, a, b)) in got.items():
        ta, tg = (1e-10, 1e-8) if p == "fp64" else (1e-5, 1e-3)
        assert np.max(np.abs(psi - ref)) <= ta and abs(f[1] - F[1]) <= ta, p
        assert np.max(np.abs(np.concatenate([a, b]) - g)) <= tg * np.max(np.abs(g)), p


@pytest.mark.parametrize("make", [
    lambda: W.local_op_pair(seed=3, T=0.2),                           # complex operators without parity
    lambda: dict(W.transmon_pair(seed=4, T=0.2), modes=[dict(m, ng=0.2) for m in W.transmon_pair(seed=4)["modes"]]),
])
def test_other_terms_keep_their_kernels(sgctx, monkeypatch, make):
    from paper_2406_18155_gb300.api import System
    wl = make()
    s = System.from_workload(sgctx, wl)
    s.prepare()
    psi = s.evolve(wl["T"], wl["dt"], precision="fp64", col_index=wl["col_index"]).cpu().numpy()
    monkeypatch.setenv("SG_PATH", "gather")
    ref = s.evolve(wl["T"], wl["dt"], precision="fp64", col_index=wl["col_index"]).cpu().numpy()
    assert np.max(np.abs(psi - ref)) <= 1e-10


@pytest.mark.parametrize("odd_one_out", [False, True])
def test_batch_of_pairs(sgctx, odd_one_out):
    # one structure: the on-chip kernel, a warp per system; a system with its coupling written
    # the other way round: the tensor-core kernel for all
    from paper_2406_18155_gb300.api import System, evolve_batch
    wls = [W.fluxonium_pair_multipath(seed=s, T=0.3, levels=4) for s in range(3)]
    if odd_one_out:
        c = wls[1]["couplings"][0]
        c["a"], c["b"] = c["b"], c["a"]
    cols = [3, 0, 15, 1, 4, 5, 2, 7, 8, 14, 6, 9, 10, 13, 12, 11]
    systems = [System.from_workload(sgctx, wl) for wl in wls]
    for s in systems:
        s.prepare()
    psi = evolve_batch(systems, 0.3, 0.01, cols).cpu().numpy()
    for p, s in zip(psi, systems):
        ref = s.evolve(0.3, 0.01, precision="fp64", col_index=cols).cpu().numpy()
        assert np.max(np.abs(p - ref)) <= 1e-5
