"""The plan of large grids by one block (a batched ensemble's) and by a cluster of
blocks (a run of its own): the steps that follow have the same bits."""

import numpy as np
import pytest

from paper_2605_20140_gb300 import sipf
from sipf_inputs import uniform_positions, workload

from parity_helpers import by_id

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def test_one_block_plans_as_a_cluster_does():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wls = []
    for H, N in ((96, 20011), (128, 200003)):      # 1728 and 4096 tiles, thin and thick ones
        wl = workload("small", H=H, N=N)
        wl.x[: N // 3] = uniform_positions(N // 3, wl.L, wl.origin, np.random.default_rng(H))
        wls.append(wl)
    got = [[], []]
    with sipf.Ensemble([(w.H, w.L, w.origin, w.N, w.params) for w in wls],
                       mode=sipf.SIPF_ENSEMBLE_BATCHED) as ens:
        for sim, w in zip(ens.members, wls):
            sim.set_state(w.x, w.mass, w.ids, w.v, w.m, w.w)
        ens.step([w.dt for w in wls], 5)
        ens.sync()
        assert ens.last_path() == sipf.SIPF_ENSEMBLE_BATCHED
        got[0] = [(sim.fields(), by_id(*sim.particle_state())) for sim in ens.members]
    for w in wls:
        with sipf.Simulation(w.H, w.L, w.origin, w.N, w.params) as sim:
            sim.set_state(w.x, w.mass, w.ids, w.v, w.m, w.w)
            sim.step(w.dt, 5)
            got[1].append((sim.fields(), by_id(*sim.particle_state())))
    for a, b in zip(*got):
        for k in a[0]:
            np.testing.assert_array_equal(a[0][k], b[0][k], err_msg=k)
        for p, q in zip(a[1], b[1]):
            np.testing.assert_array_equal(p, q)
