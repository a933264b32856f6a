"""Gradients whose stage inputs pass the store of one round (1 GiB): several rounds of chunks side by
side, the first of them ragged, against the same solve in one chunk that keeps all of them.

Both do the same steps from the same states up to rounding (FP64 1e-10 on F and 1e-8 of the
largest gradient component, mixed 1e-5 and 1e-3, as for the kernel families)."""
import numpy as np
import pytest

from paper_2406_18155_gb300 import workloads as W

pytestmark = pytest.mark.gpu

GIB = 1 << 30


@pytest.mark.parametrize("nq,levels,cols,steps,precision,images", [
    (5, 3, 32, 3001, "mixed", 2),      # propagators, real operators (which keep states and co-states)
    (5, 5, 32, 1403, "mixed", 2),      # serial passes side by side (more than 8 GiB in all, so not kept)
    (6, 3, 70, 2703, "mixed", 2),      # serial passes one after the other (more columns than the basis takes)
    (3, 4, 8, 17003, "fp64", 2),       # propagators, FP64
    (5, 4, 32, 1203, "fp64", 1),       # complex rows
])
def test_rounds_of_chunks(sgctx, nq, levels, cols, steps, precision, images):
    from paper_2406_18155_gb300.api import System
    D, n, cs = levels ** nq, 2 ** nq, 8 if precision == "mixed" else 16
    assert images * 4 * steps * D * cols * cs > GIB
    wl = W.fluxonium_chain(seed=nq + levels, nq=nq, levels=levels, T=steps * 0.01, dt=0.01, nseg=7, ncols=min(cols, n))
    wl["col_index"] += [j for j in range(D) if j not in wl["col_index"]][:cols - n if cols > n else 0]
    s = System.from_workload(sgctx, wl)
    s.prepare()
    got = [s.fidelity_grad(wl["T"], wl["dt"], wl["target"], wl["col_index"], kind="state", precision=precision,
                           ckpt=k) for k in (0, steps)]
    (F, gp, gh), (f, p, h) = got[1], got[0]
    ta, tg = (1e-10, 1e-8) if precision == "fp64" else (1e-5, 1e-3)
    g = np.concatenate([gp, gh])
    assert abs(f[1] - F[1]) <= ta
    assert np.max(np.abs(np.concatenate([p, h]) - g)) <= tg * np.max(np.abs(g))
