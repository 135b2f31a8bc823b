"""A context or an ensemble that is given another state after it has stepped:
what the captured step graphs hold may not outlive the state they were
captured with."""

import numpy as np
import pytest

from paper_2605_20140_gb300 import sipf
from sipf_inputs import workload

from parity_helpers import by_id

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _needs_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _set(sim, wl):
    sim.set_state(wl.x, wl.mass, wl.ids, wl.v, wl.m, wl.w)


def _other_masses(wl):
    """The same workload with three times the total mass, spread over a factor of a
    thousand: another reference mass and another deposit scale."""
    wl.mass = wl.mass * 10.0 ** np.random.default_rng(7).uniform(-2.0, 1.0, wl.N)
    wl.mass *= 3.0 / wl.mass.sum()
    return wl


def _snapshot(sim):
    return sim.fields(), by_id(*sim.particle_state())


def _assert_same(a, b):
    for k in a[0]:
        np.testing.assert_array_equal(a[0][k], b[0][k], err_msg=k)
    for p, q in zip(a[1], b[1]):
        np.testing.assert_array_equal(p, q)


def test_steps_from_a_second_state_equal_those_of_a_fresh_context():
    first = workload("small", H=32, N=20011)
    second = _other_masses(workload("small", H=32, N=20011, seed=1))
    got = []
    for states in ((first, second), (second,)):
        stream = torch.cuda.Stream()         # pairs of steps replay a captured graph
        with sipf.Simulation(second.H, second.L, second.origin, second.N, second.params,
                             stream=stream.cuda_stream) as sim:
            for wl in states:
                _set(sim, wl)
                sim.step(second.dt, 4)
            got.append(_snapshot(sim))
    _assert_same(*got)


def test_batched_steps_from_a_second_state_equal_those_of_a_fresh_ensemble():
    sizes = ((32, 20011), (48, 9001))
    first = [workload("small", H=H, N=N) for H, N in sizes]
    second = [_other_masses(workload("small", H=H, N=N, seed=1)) for H, N in sizes]
    specs = [(w.H, w.L, w.origin, w.N, w.params) for w in second]
    got = []
    for rounds in ((first, second), (second,)):
        with sipf.Ensemble(specs, mode=sipf.SIPF_ENSEMBLE_BATCHED) as ens:
            for wls in rounds:
                for sim, wl in zip(ens.members, wls):
                    _set(sim, wl)
                ens.step([w.dt for w in second], 4)
                ens.sync()
                assert ens.last_path() == sipf.SIPF_ENSEMBLE_BATCHED
            got.append([_snapshot(sim) for sim in ens.members])
    for a, b in zip(*got):
        _assert_same(a, b)


def test_steps_after_a_state_with_a_non_finite_position():
    """Such a state is reported with the position reset to 0; a context that already
    had a state goes on from the one that it was given, with its reference mass."""
    first = workload("small", H=32, N=20011)
    second = _other_masses(workload("small", H=32, N=20011, seed=1))
    reset = _other_masses(workload("small", H=32, N=20011, seed=1))
    second.x[77, 1] = np.nan
    reset.x[77, 1] = 0.0
    got = []
    for before in (True, False):
        with sipf.Simulation(reset.H, reset.L, reset.origin, reset.N, reset.params) as sim:
            if before:
                _set(sim, first)
                sim.step(first.dt, 3)
                with pytest.raises(sipf.SipfError) as e:
                    _set(sim, second)
                assert e.value.code == sipf.SIPF_ENONFINITE
            else:
                _set(sim, reset)
            sim.step(reset.dt, 3)
            got.append(_snapshot(sim))
    _assert_same(*got)
