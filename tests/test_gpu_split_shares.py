"""The split form of the particle step against the dense one, which a run beside
others takes: the same state gives the same bits.  Sizes at both ends of the split
form's range (a chunk for each block, fourth order three) and just beyond."""

import dataclasses

import numpy as np
import pytest

from paper_2605_20140_gb300 import sipf
from sipf_inputs import uniform_positions, workload

from parity_helpers import by_id

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


# blocks per GPU: 760, fourth order 608
@pytest.mark.parametrize("H,N,order,uniform", [
    (8, 512, 2, False), (8, 194304, 2, True), (8, 194305, 2, False), (8, 466688, 4, True),
    (16, 131072, 2, False), (24, 187648, 2, True), (32, 262144, 4, False), (32, 178177, 2, False),
    (48, 110592, 2, True), (48, 411648, 4, False), (64, 262144, 4, True), (72, 373249, 4, False)])
def test_split_and_dense_steps_have_the_same_bits(H, N, order, uniform):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = workload("small", H=H, N=N)
    wl.params = dataclasses.replace(wl.params, p2g_order=order)
    if uniform:
        wl.x = uniform_positions(N, wl.L, wl.origin, np.random.default_rng(H))
    if order == 4:      # negative weights: eta(u_bar) may be singular, so w = 0
        wl.params = dataclasses.replace(wl.params, gamma=0.0)
        wl.w = np.zeros_like(wl.w)
    got = []

    def run(sim, step):
        sim.set_state(wl.x, wl.mass, wl.ids, wl.v, wl.m, wl.w)
        step()
        got.append((sim.fields(), by_id(*sim.particle_state())))

    stream = torch.cuda.Stream()
    with sipf.Simulation(H, wl.L, wl.origin, N, wl.params, stream=stream.cuda_stream) as sim:
        run(sim, lambda: sim.step(wl.dt, 3))
    with sipf.Ensemble([(H, wl.L, wl.origin, N, wl.params)],
                       mode=sipf.SIPF_ENSEMBLE_STREAMS) as ens:
        run(ens.members[0], lambda: ens.step([wl.dt], 3))
    for k in got[0][0]:
        np.testing.assert_array_equal(got[0][0][k], got[1][0][k], err_msg=k)
    for a, b in zip(got[0][1], got[1][1]):
        np.testing.assert_array_equal(a, b)
