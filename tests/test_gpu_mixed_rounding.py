"""What is constant for a whole solve is not rounded to FP32 on the real-operator on-chip kernels.

A constant relative error e of H (of the step's weights h/6, of the modulus of the phases) adds up over
the steps to e times the angle that H turns the state by, where rounding that changes from step to
step grows with their square root.
"""
import numpy as np
import pytest

from paper_2406_18155_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STEPS = 10000


# fl(h/6) is off by -7.5e-8 at the first step, by +7.7e-8 at the second
@pytest.mark.parametrize("dt", [0.009174, 0.009081])
def test_resonant_drive_turns_by_its_angle(sgctx, dt):
    """A two-level resonance turned by A T / 2 = 180 rad: the error stays below 2^-26 of the
    angle, plus four standard deviations of a rounding of the increment h A per step."""
    from paper_2406_18155_gb300.api import System
    A, T = 4.0, STEPS * dt
    s = System(sgctx)
    for _ in range(2):
        s.add_transmon(12.0 * 2 * np.pi, 0.3 * 2 * np.pi, levels=2)
    x = s.add_local_op(0, np.array([[0, 1], [1, 0]], complex))
    s.add_drive(0, x, "pwc", amps=[A], length=T, omega_mode=0)
    s.prepare()
    a, b = (s.evolve(T, dt, precision=p, col_index=[0, 1, 2, 3]).cpu().numpy() for p in ("fp64", "mixed"))
    err = np.linalg.norm(a - b) / np.linalg.norm(a)
    assert err < 2.0 ** -26 * A * T / 2 + 4 * 2.0 ** -24 * A * dt * STEPS ** 0.5


@pytest.mark.parametrize("seed", [1, 4])
def test_long_gradient_keeps_single_precision(sgctx, seed):
    """Cross-resonance pair, 10,000 steps, turned by 30 to 40 rad: 2^-26 of that, 5e-7."""
    from paper_2406_18155_gb300.api import System
    rng = np.random.Generator(np.random.PCG64([seed, 77]))
    wl = W.fluxonium_pair_cr(int(rng.integers(0, 2 ** 31)), T=STEPS * 0.01, dt=0.01)
    s = System.from_workload(sgctx, wl)
    s.prepare()
    g = [s.fidelity_grad(wl["T"], wl["dt"], wl["target"], wl["col_index"], kind=wl["fid_kind"], precision=p)
         for p in ("fp64", "mixed")]
    for ref, got in zip(g[0][1:], g[1][1:]):
        assert np.linalg.norm(np.asarray(got) - ref) < 5e-7 * np.linalg.norm(ref)
