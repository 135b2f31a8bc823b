"""Whole steps with the options that the per-axis passes and the split particle
step serve, against the float64 oracle, within the parity tolerances."""

import dataclasses

import numpy as np
import pytest

from oracle import sipf_oracle as O
from paper_2605_20140_gb300 import sipf
from sipf_inputs import uniform_positions, workload

from parity_helpers import compare, oracle_state

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _needs_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _run(wl, plan, steps):
    stream = torch.cuda.Stream()
    with sipf.Simulation(wl.H, wl.L, wl.origin, wl.N, wl.params,
                         stream=stream.cuda_stream) as sim:
        if plan is not None:
            t = sipf.sipf_get_tuning(sim.ctx)
            t["radix_plan"] = plan
            sipf.sipf_set_tuning(sim.ctx, **t)
        sim.set_state(wl.x, wl.mass, wl.ids, wl.v, wl.m, wl.w)
        sim.step(wl.dt, steps)
        compare(sim, O.run(oracle_state(wl), wl.dt, steps), wl)


# above 128 rows of m* and of w* are paired apart; plan 2 packs m* + i w*
@pytest.mark.parametrize("H,plan,steps,filtered,smoothed,v_update,diffusion", [
    (144, 0, 2, True, False, 0, 0), (144, 1, 3, True, True, 1, 1), (216, 0, 2, False, True, 1, 0),
    (64, 2, 3, False, True, 0, 0), (64, 2, 4, True, True, 1, 1), (128, 2, 2, True, False, 1, 0),
    (32, 0, 3, False, False, 1, 0), (72, 1, 3, True, True, 1, 1)])
def test_options_on_each_spectral_path(H, plan, steps, filtered, smoothed, v_update, diffusion):
    wl = workload("small", H=H, N=1 << 16)
    wl.params = dataclasses.replace(
        wl.params, v_update=v_update, diffusion=diffusion, H0=H ** (8 / 13) if filtered else 0.0,
        sigma=(1.5 * wl.L / H) ** 2 if smoothed else 0.0)
    _run(wl, plan, steps)


# few particles in all, many per tile: the split form; evenly spread, so that the
# negative weights of R^(4) leave u_bar above 0 and eta(u_bar) w can be compared
@pytest.mark.parametrize("H,N", [(8, 20011), (16, 200000)])
def test_fourth_order_split_step_with_w(H, N):
    wl = workload("small", H=H, N=N)
    wl.x = uniform_positions(N, wl.L, wl.origin, np.random.default_rng(H))
    wl.params = dataclasses.replace(wl.params, p2g_order=4)
    assert O.density(oracle_state(wl)).min() > 0.0
    _run(wl, None, 3)
