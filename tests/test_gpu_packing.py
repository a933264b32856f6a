"""Solves that share a batched on-chip launch: what differs between them although their shapes are alike."""
import numpy as np
import pytest

from paper_2406_18155_gb300 import workloads as W

pytestmark = pytest.mark.gpu

X = np.array([[0, 1, 0], [1, 0, 1.3], [0, 1.3, 0]], complex)
Y = np.array([[0, -1j, 0], [1j, 0, -1.3j], [0, 1.3j, 0]], complex)


def _system(ctx, op, seed):
    """Two uncoupled transmons, each driven through a local operator: same shape for X and Y, but the
    real-operator kernels turn the basis of a mode whose drive is imaginary."""
    from paper_2406_18155_gb300.api import System
    rng = np.random.Generator(np.random.PCG64(seed))
    s = System(ctx)
    for m in range(2):
        s.add_transmon(2 * np.pi * (12 + m), 2 * np.pi * 0.3, levels=3)
    for m in range(2):
        k = s.add_local_op(m, op)
        s.add_drive(m, k, "pwc", amps=rng.uniform(0.2, 0.6, 3), length=0.6, omega_mode=m)
    s.prepare()
    return s


def test_packed_solves_keep_their_own_gauge(sgctx):
    from paper_2406_18155_gb300.api import Server, System
    T, dt, cols = 0.6, 0.01, W.comp_states([3, 3])
    target = W.haar_unitary(4, np.random.Generator(np.random.PCG64(2)))
    ops = [X, Y, Y, X]
    alone = [_system(sgctx, op, i).fidelity_grad(T, dt, target, cols, precision="mixed") for i, op in enumerate(ops)]
    srv = Server(sgctx, mem_budget_bytes=8 << 30, max_slots=1, max_batch=4)
    # a first request holds the slot while the others queue up behind it
    wl = W.fluxonium_chain(seed=1, nq=4, levels=4, T=10.0, dt=dt)
    first = System.from_workload(sgctx, wl)
    first.prepare()
    systems = [_system(sgctx, op, i) for i, op in enumerate(ops)]
    tickets = [srv.submit(first, wl["T"], dt, wl["target"], wl["col_index"], kind="state", precision="fp64")]
    tickets += [srv.submit(s, T, dt, target, cols) for s in systems]
    res = [srv.wait(t) for t in tickets][1:]
    assert srv.stats()["batched_requests"] >= 2
    srv.close()
    # a packed solve does the arithmetic of the lone one
    for (F, gp, gh), r in zip(alone, res):
        assert r["status"] == 0, r["error"]
        assert abs(r["F"][0] - F[0]) <= 1e-12
        assert np.max(np.abs(r["grad_pulse"] - gp)) <= 1e-12 * max(1.0, np.max(np.abs(gp)))
        assert np.max(np.abs(r["grad_ham"] - gh)) <= 1e-12 * max(1.0, np.max(np.abs(gh)))


def test_packed_serial_passes_share_one_launch(sgctx):
    """Beyond D = 256 the states and the basis of co-states are serial passes that do not wait for one
    another: a pack issues them together, so each batch is one round of launches."""
    from paper_2406_18155_gb300.api import Server, System
    wls = []
    for i in range(4):
        wl = W.serving_request(np.random.Generator(np.random.PCG64(i)), nq=4, kind="fluxonium", levels=5)
        wl["T"] = 3000 * wl["dt"] if i == 0 else 12 * wl["dt"]
        for d in wl["drives"]:
            d["length"] = wl["T"]
        wls.append(wl)

    def system(wl):
        s = System.from_workload(sgctx, wl)
        s.prepare()
        return s

    args = lambda wl: (wl["T"], wl["dt"], wl["target"], wl["col_index"])  # noqa: E731
    alone = [system(wl).fidelity_grad(*args(wl), kind=wl["fid_kind"], precision="mixed") for wl in wls[1:]]
    srv = Server(sgctx, mem_budget_bytes=32 << 30, max_slots=1, max_batch=4)
    systems = [system(wl) for wl in wls]
    # the first request holds the slot while the others queue up behind it
    tickets = [srv.submit(s, *args(wl), kind=wl["fid_kind"], precision="mixed") for s, wl in zip(systems, wls)]
    res = [srv.wait(t) for t in tickets][1:]
    st = srv.stats()
    srv.close()
    assert st["batches"] == 1 and st["batched_requests"] == 3
    assert st["batched_launches"] == 1 and st["batched_launch_members"] == 6
    for (F, gp, gh), r in zip(alone, res):
        assert r["status"] == 0, r["error"]
        assert abs(r["F"][0] - F[0]) <= 1e-12
        assert np.max(np.abs(r["grad_pulse"] - gp)) <= 1e-12 * max(1.0, np.max(np.abs(gp)))
        assert np.max(np.abs(r["grad_ham"] - gh)) <= 1e-12 * max(1.0, np.max(np.abs(gh)))


@pytest.mark.parametrize("slots,batch", [(1, 4), (4, 1)])
def test_small_budget_still_runs_requests_together(sgctx, slots, batch):
    """64 MiB hold the needs of many D = 27 requests: what each may take to run its chunks side by side
    must not fill the budget."""
    from paper_2406_18155_gb300.api import Server, System
    wls = []
    for i in range(5):
        wl = W.serving_request(np.random.Generator(np.random.PCG64(i)), nq=3, kind="fluxonium", levels=3)
        # the first request of one slot holds it while the others queue up
        wl["T"] = (1000 if i == 0 or slots > 1 else 60) * wl["dt"]
        for d in wl["drives"]:
            d["length"] = wl["T"]
        wls.append(wl)

    def system(wl):
        s = System.from_workload(sgctx, wl)
        s.prepare()
        return s

    args = lambda wl: (wl["T"], wl["dt"], wl["target"], wl["col_index"])  # noqa: E731
    alone = [system(wl).fidelity_grad(*args(wl), kind=wl["fid_kind"], precision="fp64") for wl in wls]
    srv = Server(sgctx, mem_budget_bytes=64 << 20, max_slots=slots, max_batch=batch)
    systems = [system(wl) for wl in wls]
    tickets = [srv.submit(s, *args(wl), kind=wl["fid_kind"], precision="fp64") for s, wl in zip(systems, wls)]
    res = [srv.wait(t) for t in tickets]
    st = srv.stats()
    srv.close()
    for (F, gp, gh), r in zip(alone, res):
        assert r["status"] == 0, r["error"]
        assert abs(r["F"][0] - F[0]) <= 1e-10
        g = np.concatenate([gp, gh])
        assert np.max(np.abs(np.concatenate([r["grad_pulse"], r["grad_ham"]]) - g)) <= 1e-8 * np.max(np.abs(g))
    if slots == 1:
        assert st["batched_requests"] == 4
    else:
        assert sorted(r["start_s"] for r in res)[1] < min(r["done_s"] for r in res)
