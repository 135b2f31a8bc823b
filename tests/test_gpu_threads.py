"""Contexts of different sizes set up on host threads of their own at the same
time: distinct contexts are independent."""

import threading

import numpy as np
import pytest

from paper_2605_20140_gb300 import sipf
from sipf_inputs import workload

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def test_states_set_on_several_threads():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    # 216: the tile counts take 77 KB of shared memory, 8: four bytes
    sizes = [(216, 4099), (216, 4099)] + [(8, 64)] * 4
    sims, states, errors = [], [], []
    for k, (H, N) in enumerate(sizes):
        wl = workload("small", H=H, N=N, seed=k)
        stream = torch.cuda.Stream()
        sims.append(sipf.Simulation(wl.H, wl.L, wl.origin, wl.N, wl.params,
                                    stream=stream.cuda_stream))
        sims[-1].torch_stream = stream
        states.append([torch.from_numpy(np.ascontiguousarray(a)).cuda()
                       for a in (wl.x.T, wl.mass, wl.v, wl.m, wl.w)])
    torch.cuda.synchronize()
    stop = threading.Event()

    def loop(sim, t, count):
        try:
            n = 0
            while n < count if count else not stop.is_set():
                sipf.sipf_set_state(sim.ctx, t[0], t[1], None, t[2], t[3], t[4],
                                    sipf.SIPF_DEVICE)
                n += 1
        except sipf.SipfError as e:
            errors.append(e)

    large = [threading.Thread(target=loop, args=(sims[k], states[k], 100)) for k in (0, 1)]
    small = [threading.Thread(target=loop, args=(sims[k], states[k], 0)) for k in (2, 3, 4, 5)]
    for th in large + small:
        th.start()
    for th in large:
        th.join()
    stop.set()
    for th in small:
        th.join()
    for sim in sims:
        sim.close()
    assert not errors, errors[0]
