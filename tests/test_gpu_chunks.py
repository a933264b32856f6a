"""On-chip solves in chunks of steps that run side by side: chunk counts at their edges
(one step either side of the shortest chunked solve, a ragged last chunk, one and two
levels of products), propagators of every size they are computed for and the serial
boundary states beyond, against the general gather kernels, FP64 and mixed.

Tolerances are those of the kernel families' comparisons: FP64 1e-10 on amplitudes and F
and 1e-8 of the largest gradient component (a product of short propagators rounds like
the steps it replaces), mixed 1e-5 and 1e-3."""
import numpy as np
import pytest

from paper_2406_18155_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _chain(nq, levels, steps, ring=False, ncols=None, dt=0.01):
    return W.fluxonium_chain(seed=nq * 10 + levels, nq=nq, levels=levels, T=steps * dt, dt=dt, nseg=3, ring=ring,
                             ncols=ncols)


def _system(sgctx, wl):
    from paper_2406_18155_gb300.api import System
    s = System.from_workload(sgctx, wl)
    s.prepare()
    return s


def _solve(s, wl, precision, ckpt=0):
    psi = s.evolve(wl["T"], wl["dt"], precision=precision, col_index=wl["col_index"]).cpu().numpy()
    F, gp, gh = s.fidelity_grad(wl["T"], wl["dt"], wl["target"], wl["col_index"], kind="state",
                                precision=precision, ckpt=ckpt)
    return psi, F[1], np.concatenate([gp, gh])


def _agree(monkeypatch, s, wl, ckpt=0):
    monkeypatch.setenv("SG_PATH", "gather")
    psi, F, g = _solve(s, wl, "fp64")
    monkeypatch.delenv("SG_PATH")
    scale = np.max(np.abs(g))
    for prec, ta, tg in (("fp64", 1e-10, 1e-8), ("mixed", 1e-5, 1e-3)):
        p, f, h = _solve(s, wl, prec, ckpt)
        assert np.max(np.abs(p - psi)) <= ta and abs(f - F) <= ta, prec
        assert np.max(np.abs(h - g)) <= tg * scale, prec


@pytest.mark.parametrize("steps", [1, 7, 8, 9, 13, 605, 1301])
def test_chunk_counts(sgctx, monkeypatch, steps):
    wl = _chain(2, 3, steps)
    _agree(monkeypatch, _system(sgctx, wl), wl)


@pytest.mark.parametrize("ckpt", [1, 3, 29, 1000])
def test_requested_chunk_lengths(sgctx, monkeypatch, ckpt):
    wl = _chain(2, 4, 30)
    _agree(monkeypatch, _system(sgctx, wl), wl, ckpt)


@pytest.mark.parametrize("nq,levels,ring", [(2, 2, False), (2, 5, False), (4, 3, True), (3, 5, False), (5, 3, False),
                                            (4, 4, False), (8, 2, False), (4, 5, False), (5, 4, True)])
def test_chunks_of_every_dimension(sgctx, monkeypatch, nq, levels, ring):
    # D = 4, 25, 81, 125, 243, 256, 256 by propagators; 625, 1024 by serial boundary states
    wl = _chain(nq, levels, 41, ring=ring, ncols=min(2 ** nq, 12))
    _agree(monkeypatch, _system(sgctx, wl), wl)


def test_chunks_one_after_the_other_when_memory_is_short(sgctx):
    # a server whose budget holds the solve but not its chunks side by side
    from paper_2406_18155_gb300.api import Server
    wl = _chain(3, 3, 60)
    s = _system(sgctx, wl)
    _, F, g = _solve(s, wl, "fp64")
    srv = Server(sgctx, mem_budget_bytes=3 << 20, max_slots=1)
    r = srv.wait(srv.submit(s, wl["T"], wl["dt"], wl["target"], wl["col_index"], kind="state", precision="fp64"))
    srv.close()
    assert r["status"] == 0, r["error"]
    assert abs(r["F"][1] - F) <= 1e-10
    got = np.concatenate([r["grad_pulse"], r["grad_ham"]])
    assert np.max(np.abs(got - g)) <= 1e-8 * np.max(np.abs(g))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_an_unstable_level_stays_out_of_columns_that_never_reach_it(sgctx, monkeypatch, precision):
    # lab frame, no coupling and no drive, dt E_3 = 4.7: RK4 blows level 3 up to infinity, which
    # columns with at most one excitation (dt E = 1.6, stable) never occupy
    wl = W.transmon_pair(seed=3, T=3000.0, dt=0.05)
    wl["couplings"], wl["drives"], wl["col_index"] = [], [], [0, 1, 4]
    s = _system(sgctx, wl)
    kw = dict(precision=precision, frame="lab", col_index=wl["col_index"])
    psi = s.evolve(wl["T"], wl["dt"], **kw).cpu().numpy()
    monkeypatch.setenv("SG_PATH", "gather")
    ref = s.evolve(wl["T"], wl["dt"], precision="fp64", frame="lab", col_index=wl["col_index"]).cpu().numpy()
    assert np.all(np.isfinite(ref)) and np.all(np.isfinite(psi))
    scale = np.max(np.abs(ref))
    assert np.max(np.abs(psi - ref)) <= (1e-9 if precision == "fp64" else 1e-2) * scale
