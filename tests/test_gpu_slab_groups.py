"""Two-pass tiled plans whose second group would hold few modes (chains just beyond one tile):
both groups filled up to the tile budget, against the general gather kernels, every level
count and both gradients.  FP64 1e-10 on amplitudes, 1e-8 of the largest gradient component;
mixed 1e-5 and 1e-3, as for the other kernel families."""
import numpy as np
import pytest

from paper_2406_18155_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq,levels,ring,ncols", [(7, 4, False, 3), (8, 4, True, 1), (8, 3, False, 2), (6, 5, False, 2),
                                                  (13, 2, False, 2)])
@pytest.mark.parametrize("ham", [True, False])
def test_filled_groups_match_the_general_kernels(sgctx, monkeypatch, nq, levels, ring, ncols, ham):
    from paper_2406_18155_gb300.api import System
    wl = W.fluxonium_chain(seed=nq, nq=nq, levels=levels, T=0.05, dt=0.01, nseg=5, ring=ring, ncols=ncols)
    rng = np.random.Generator(np.random.PCG64(nq))
    wl["target"] = np.diag(np.exp(1j * rng.uniform(0, 2 * np.pi, 2 ** nq)))
    if nq > 12:                                      # the fidelity takes 12 qubit modes at most
        for i in range(12, nq):
            wl["modes"][i]["coupler"] = True
        wl["col_index"] = W.comp_states([levels] * nq, couplers=range(12, nq))[:ncols]
        wl["target"] = wl["target"][:4096, :4096]
    s = System.from_workload(sgctx, wl)
    s.prepare()

    def solve(precision):
        psi = s.evolve(wl["T"], wl["dt"], precision=precision, col_index=wl["col_index"]).cpu().numpy()
        F, gp, gh = s.fidelity_grad(wl["T"], wl["dt"], wl["target"], wl["col_index"], kind="state",
                                    precision=precision, ham=ham)
        return psi, F[1], np.concatenate([gp, gh]) if ham else gp
    got = {p: solve(p) for p in ("fp64", "mixed")}
    monkeypatch.setenv("SG_PATH", "gather")
    psi, F, g = solve("fp64")
    for p, (a, f, b) in got.items():
        ta, tg = (1e-10, 1e-8) if p == "fp64" else (1e-5, 1e-3)
        assert np.max(np.abs(a - psi)) <= ta and abs(f - F) <= ta, p
        assert np.max(np.abs(b - g)) <= tg * np.max(np.abs(g)), p
