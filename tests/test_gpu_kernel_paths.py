"""The kernel that a size or an input selects, at the edges of each rule: forms
of the particle step, set-up of a state from device and from host memory,
initial binning and cell orders with and without shared-memory counts, the
slab path of the allocation-free deposit."""

import dataclasses

import numpy as np
import pytest

from oracle import sipf_oracle as O
from paper_2605_20140_gb300 import sipf
from sipf_inputs import workload

from parity_helpers import by_id, compare, oracle_state, rel_l2

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _needs_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# tiles (H/8)^3: dense from 256 particles per tile on, split from 512 on (few
# particles in all), sparse below; chunks of 256 and items of 1024 particles
@pytest.mark.parametrize("H,N,order", [
    (8, 511, 2), (8, 512, 2), (8, 513, 2), (8, 1025, 4), (16, 4095, 2), (16, 4096, 4),
    (16, 9001, 2), (24, 9001, 2), (24, 13824, 4), (32, 3001, 2), (32, 16385, 4), (32, 32769, 2)])
def test_particle_step_forms_match_oracle(H, N, order):
    wl = workload("small", H=H, N=N)
    wl.params = dataclasses.replace(wl.params, p2g_order=order)
    if order == 4:
        # R^(4) has negative weights; at these counts u_bar goes below -1, where eta(u) =
        # 2u/(1 + u) is singular and w has no comparable value.  With w = 0 eta plays no part.
        wl.params = dataclasses.replace(wl.params, gamma=0.0)
        wl.w = np.zeros_like(wl.w)
    stream = torch.cuda.Stream()
    with sipf.Simulation(wl.H, wl.L, wl.origin, wl.N, wl.params,
                         stream=stream.cuda_stream) as sim:
        sim.set_state(wl.x, wl.mass, wl.ids, wl.v, wl.m, wl.w)
        sim.step(wl.dt, 3)
        st = O.run(oracle_state(wl), wl.dt, 3)
        if order == 4:
            # w = 0 up to what the transform it shares with m leaves there (float32
            # rounding of values below 1); a relative error of zero says nothing
            w = sim.fields(sipf.FIELD_W)["w"].astype(np.float64)
            assert np.max(np.abs(w)) <= 1e-6
            st.w = w
        compare(sim, st, wl)


def _device_state(sim, wl):
    t = [torch.from_numpy(np.ascontiguousarray(a)).cuda()
         for a in (wl.x.T, wl.mass, wl.v, wl.m, wl.w)]
    torch.cuda.synchronize()
    sipf.sipf_set_state(sim.ctx, t[0], t[1], None, t[2], t[3], t[4], sipf.SIPF_DEVICE)


@pytest.mark.parametrize("N,masses,v", [
    (1 << 15, "equal", "plain"), (20011, "equal", "plain"), (20011, "unequal", "plain"),
    (65537, "unequal", "tiny"), (131073, "unequal", "plain"), (20011, "zeros", "tiny"),
    (20011, "all zero", "zero")])
def test_state_from_device_and_host_memory_has_the_same_bits(N, masses, v):
    """The masses' sum and the mean of v come from a kernel's statistics or from
    the host's loop; everything after depends on their last bit."""
    wl = workload("small", H=32, N=N)
    rng = np.random.default_rng(3)
    if masses == "unequal":
        wl.mass = wl.mass * rng.uniform(0.5, 2.0, N)
    elif masses == "zeros":
        wl.mass = np.where(rng.random(N) < 0.5, 0.0, wl.mass)
    elif masses == "all zero":
        wl.mass = np.zeros(N)
    if v == "tiny":       # not exact in every order
        wl.v = (wl.v * 10.0 ** rng.uniform(-20.0, 0.0, wl.v.shape)).astype(np.float32)
    elif v == "zero":
        wl.v = np.zeros_like(wl.v)
    got = []
    for device in (False, True):
        with sipf.Simulation(wl.H, wl.L, wl.origin, wl.N, wl.params) as sim:
            if device:
                _device_state(sim, wl)
            else:
                sim.set_state(wl.x, wl.mass, wl.ids, wl.v, wl.m, wl.w)
            sim.step(wl.dt, 2)
            got.append((sim.fields(), by_id(*sim.particle_state())))
    for k in got[0][0]:
        np.testing.assert_array_equal(got[0][0][k], got[1][0][k], err_msg=k)
    for a, b in zip(got[0][1], got[1][1]):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -1.0])
def test_bad_masses_on_the_device_are_refused_and_leave_the_state(bad):
    wl = workload("small", H=16, N=4099)
    with sipf.Simulation(wl.H, wl.L, wl.origin, wl.N, wl.params) as sim:
        _device_state(sim, wl)
        before = sim.fields()
        good = wl.mass
        wl.mass = good.copy()
        wl.mass[4097] = bad
        with pytest.raises(sipf.SipfError) as e:
            _device_state(sim, wl)
        assert e.value.code == sipf.SIPF_EINVAL
        after = sim.fields()
    for k in before:
        np.testing.assert_array_equal(before[k], after[k])


# 32768 tiles (H = 256) are the most that are binned in shared memory
@pytest.mark.parametrize("H,N", [(8, 1), (8, 1025), (96, 20011), (256, 20011), (288, 20011)])
def test_binning_and_cell_orders(H, N):
    wl = workload("small", H=H, N=N)
    with sipf.Simulation(wl.H, wl.L, wl.origin, wl.N, wl.params) as sim:
        sim.set_state(wl.x, wl.mass, wl.ids, wl.v, wl.m, wl.w)
        s, _, ids = sim.particle_state()
        cs, canon = sim.canonical_order()
        starts = sim.cell_start()
    keys = O.cell_keys(s.astype(np.float64), H)
    np.testing.assert_array_equal(np.sort(ids), wl.ids)
    np.testing.assert_array_equal(cs.astype(np.int64), O.cell_start(keys, H))
    np.testing.assert_array_equal(starts, cs)
    np.testing.assert_array_equal(canon, ids[O.canonical_order(keys, ids)])


# slab path from 2^18 particles up to H = 32, from 2^19 above; one slab, several, a
# last one cut short
@pytest.mark.parametrize("H,N", [(1, 1 << 18), (16, 1 << 18), (32, (1 << 18) + 1),
                                 (33, (1 << 19) + 5), (48, 1 << 19), (64, (1 << 19) + 1)])
def test_slab_deposit_matches_float64_sums(H, N):
    rng = np.random.default_rng(H)
    x = rng.uniform(-0.3, 1.4, (3, N))                       # outside the box too
    x[:, : N // 2] = 0.97 + 0.02 * rng.standard_normal((3, N // 2))
    x = x.astype(np.float32)
    mass = rng.uniform(0.1, 1.0, N) / N
    bad = rng.integers(0, N, 9)
    with_bad = mass.copy()
    with_bad[bad] = [np.nan, np.inf, -np.inf] * 3
    mass[bad] = 0.0
    out = []
    for a in (mass, with_bad):
        xd, ad = torch.from_numpy(x).cuda(), torch.from_numpy(a).cuda()
        u = torch.full((H ** 3,), -1.0, device="cuda")
        sipf.sipf_deposit_noalloc(sipf.make_grid(H, 1.0), xd, ad, N, u)
        torch.cuda.synchronize()
        out.append(u.cpu().numpy())
    np.testing.assert_array_equal(out[0], out[1])
    s = np.mod(x.T.astype(np.float64) * H, H)
    ref = O.deposit(s, mass, H, 1.0 / H).reshape(-1)
    # float32 grid positions (4 sqrt 3 H 2^-24: their rounding moves the weights) and
    # three float32 products per weight
    assert rel_l2(out[0], ref) <= max(1e-6, 4.0 * np.sqrt(3.0) * H * 2.0 ** -24)
    assert abs(out[0].astype(np.float64).sum() / H ** 3 - mass.sum()) <= 1e-6 * mass.sum()
