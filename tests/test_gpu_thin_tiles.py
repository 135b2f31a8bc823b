"""Readouts of states whose tiles hold few particles, many, or some of each: the
FP64 diagnostics and the cell orders walk the buckets item by item."""

import math

import numpy as np
import pytest

from oracle import sipf_oracle as O
from paper_2605_20140_gb300 import sipf
from sipf_inputs import uniform_positions, workload

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


# evenly spread: a few particles per tile; "both": half of them, the others in one cell
@pytest.mark.parametrize("H,N,cloud", [
    (8, 1, "even"), (8, 31, "even"), (96, 20011, "even"), (256, 100003, "even"),
    (48, 27648, "even"), (48, 27649, "both"), (72, 300007, "even"), (64, 200003, "both")])
def test_diagnostics_and_cell_orders(H, N, cloud):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = workload("small", H=H, N=N)
    rng = np.random.default_rng(N)
    wl.x = uniform_positions(N, wl.L, wl.origin, rng)
    if cloud == "both":
        wl.x[: N // 2] = np.float32(0.5 + 0.25 / H)
    wl.ids = rng.permutation(N).astype(np.uint32)
    wl.mass = wl.mass * rng.uniform(0.5, 2.0, N)
    with sipf.Simulation(H, wl.L, wl.origin, N, wl.params) as sim:
        sim.set_state(wl.x, wl.mass, wl.ids, wl.v, wl.m, wl.w)
        d = sim.diagnostics()
        cs, canon = sim.canonical_order()
        starts = sim.cell_start()
        s, _, ids = sim.particle_state()
    # every mass exp(log a) within a few ulp, their sum exact
    assert abs(d["mass_particles"] - math.fsum(wl.mass)) <= 1e-14 * math.fsum(wl.mass)
    assert d["nonfinite"] == 0
    assert abs(d["mass_grid"] - d["mass_particles"]) <= 1e-5 * d["mass_particles"]
    keys = O.cell_keys(s.astype(np.float64), H)
    np.testing.assert_array_equal(cs.astype(np.int64), O.cell_start(keys, H))
    np.testing.assert_array_equal(starts, cs)
    np.testing.assert_array_equal(canon, ids[O.canonical_order(keys, ids)])
