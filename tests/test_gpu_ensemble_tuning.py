"""A member's tuning changed after the ensemble has stepped takes effect in the
batched steps that follow."""

import numpy as np
import pytest

from paper_2605_20140_gb300 import sipf
from sipf_inputs import workload

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def test_tuning_set_between_batched_steps_is_used():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wls = [workload("small", H=H, N=20011) for H in (48, 48, 32)]
    specs = [(w.H, w.L, w.origin, w.N, w.params) for w in wls]

    def run(ens, tuned):
        for sim, w in zip(ens.members, wls):
            if tuned:
                t = sipf.sipf_get_tuning(sim.ctx)
                t["radix_plan"] = 1 - t["radix_plan"]       # another rounding of m and w
                sipf.sipf_set_tuning(sim.ctx, **t)
            sim.set_state(w.x, w.mass, w.ids, w.v, w.m, w.w)
        ens.step([w.dt for w in wls], 4)
        ens.sync()
        assert ens.last_path() == sipf.SIPF_ENSEMBLE_BATCHED
        return [sim.fields() for sim in ens.members]

    with sipf.Ensemble(specs, mode=sipf.SIPF_ENSEMBLE_BATCHED) as ens:
        plain = run(ens, False)
        retuned = run(ens, True)
    with sipf.Ensemble(specs, mode=sipf.SIPF_ENSEMBLE_BATCHED) as ens:
        fresh = run(ens, True)
    assert any(not np.array_equal(a["m"], b["m"]) for a, b in zip(plain, fresh))
    for a, b in zip(retuned, fresh):
        for k in a:
            np.testing.assert_array_equal(a[k], b[k], err_msg=k)
