"""Solves beside other users of the GPU's memory: what only makes a solve faster is left out when
it does not fit, and the results stay those of the solve with room."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# a process of its own: the library's pool must not hold memory of earlier solves
_SOLVE = """
import sys
import numpy as np, torch
from paper_2406_18155_gb300 import workloads as W
from paper_2406_18155_gb300.api import Context, System
nq, levels, cols, steps, ckpt, left = map(int, sys.argv[1:])
wl = W.fluxonium_chain(seed=3, nq=nq, levels=levels, T=steps * 0.01, dt=0.01, nseg=3, ncols=cols)
s = System.from_workload(Context(0), wl)
s.prepare()
s.fidelity_grad(0.04, 0.01, wl["target"], wl["col_index"], kind="state", precision="mixed")   # kernels loaded
torch.zeros(1, device="cuda")
other = torch.empty(torch.cuda.mem_get_info()[0] - (left << 20), dtype=torch.uint8, device="cuda")
out = []
for _ in range(2):
    F, gp, gh = s.fidelity_grad(wl["T"], wl["dt"], wl["target"], wl["col_index"], kind="state", precision="mixed",
                                ckpt=ckpt)
    out.append((F[1], np.concatenate([gp, gh]), s.last_stats()["peak_bytes"]))
    del other
    torch.cuda.empty_cache()
    other = None
(f, g, b), (F, G, B) = out
print("bytes", b, B)
assert b < (left << 20) < B, (b, B)
assert abs(f - F) < 1e-6 and np.max(np.abs(g - G)) < 1e-4 * np.max(np.abs(G))
"""


@pytest.mark.parametrize("nq,levels,cols,steps,ckpt,left", [
    (5, 5, 32, 1000, 0, 3000),      # 6.4 GB of stage inputs with room, segments of them without
    (3, 4, 8, 40000, 1, 1500),      # a propagator of 64 kB per requested chunk of one step
])
def test_gradient_fits_beside_another_user(sgctx, nq, levels, cols, steps, ckpt, left):
    r = subprocess.run([sys.executable, "-c", _SOLVE] + [str(v) for v in (nq, levels, cols, steps, ckpt, left)],
                       cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr[-2000:]


_BATCH = """
import numpy as np, torch
from paper_2406_18155_gb300 import workloads as W
from paper_2406_18155_gb300.api import Context, System, evolve_batch
ctx, dt, steps = Context(0), 0.005, 4000
systems = []
for i in range(512):
    s = System.from_workload(ctx, W.transmon_pair(seed=i, T=steps * dt, dt=dt))
    s.prepare()
    systems.append(s)
cols = list(range(16))
evolve_batch(systems[:2], 4 * dt, dt, cols)                     # kernels loaded
other = torch.empty(torch.cuda.mem_get_info()[0] - (110 << 20), dtype=torch.uint8, device="cuda")
out = []
for _ in range(2):
    out.append((evolve_batch(systems, steps * dt, dt, cols).cpu().numpy(), systems[0].last_stats()["launches"]))
    del other
    torch.cuda.empty_cache()
    other = None
(a, n), (b, m) = out
print("launches", n, m)
assert n < m and np.max(np.abs(a - b)) < 1e-5
"""


def test_batch_fits_beside_another_user(sgctx):
    # 512 pairs of 4000 steps: 131 MB of frame phases with room, the dense kernel without
    r = subprocess.run([sys.executable, "-c", _BATCH], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr[-2000:]
