"""Rings of six, and a chain of eight modes of three levels, with as many drives as leave them on the kernels that
the other tests of these sizes are about (a plan has 16 cross-density slots: a drive takes one, a
coupling two), against the general gather kernels, and that they run there: launches that do not grow
with the steps on chip, other than the gather kernels' on tiles."""
import numpy as np
import pytest

from paper_2406_18155_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _workload(nq, levels, ring, driven, steps, cols):
    wl = W.fluxonium_chain(seed=nq, nq=nq, levels=levels, T=steps * 0.01, dt=0.01, nseg=3, ring=ring, ncols=cols)
    wl["drives"] = [wl["drives"][m] for m in driven]
    return wl


def _solve(s, wl, precision):
    psi = s.evolve(wl["T"], wl["dt"], precision=precision, col_index=wl["col_index"]).cpu().numpy()
    F, gp, gh = s.fidelity_grad(wl["T"], wl["dt"], wl["target"], wl["col_index"], kind="state", precision=precision)
    return psi, F[1], np.concatenate([gp, gh]), s.last_stats()["launches"]


@pytest.mark.parametrize("nq,levels,ring,driven,on_chip", [
    (6, 3, True, [0, 1, 3, 4], True), (6, 2, True, [0, 2, 3, 5], True), (8, 3, False, [0, 2, 4, 6], False)])
def test_sizes_at_the_slot_limit(sgctx, monkeypatch, nq, levels, ring, driven, on_chip):
    from paper_2406_18155_gb300.api import System
    out, ref = {}, {}
    for steps in (9, 21):
        wl = _workload(nq, levels, ring, driven, steps, 9)
        s = System.from_workload(sgctx, wl)
        s.prepare()
        out[steps] = {p: _solve(s, wl, p) for p in ("fp64", "mixed")}
        monkeypatch.setenv("SG_PATH", "gather")
        ref[steps] = _solve(s, wl, "fp64")
        monkeypatch.delenv("SG_PATH")
    for steps, (psi, F, g, n) in ref.items():
        for p, (a, f, b, m) in out[steps].items():
            ta, tg = (1e-10, 1e-8) if p == "fp64" else (1e-5, 1e-3)
            assert np.max(np.abs(a - psi)) <= ta and abs(f - F) <= ta, (steps, p)
            assert np.max(np.abs(b - g)) <= tg * np.max(np.abs(g)), (steps, p)
            assert m != n, (steps, p, m, n)
    if on_chip:
        for p in ("fp64", "mixed"):
            assert out[21][p][3] < out[9][p][3] + 12, (out[9][p][3], out[21][p][3])     # a launch a step
