"""The work a user of the library has it do, as cases to be timed.

Kinds of case:

* ``deposit``  -- one allocation-free particle-to-grid deposit
                  (``sipf_deposit_noalloc``): the smallest call.
* ``run``      -- one simulation through the C ABI: initial state from device
                  arrays, ``steps`` steps, all seven fields back to device
                  arrays.
* ``readout``  -- what a monitoring loop reads between steps: canonical
                  particle order, cell offsets, FP64 diagnostics, fields.
* ``resample`` -- residual resampling of unequal weights (state set, resampled,
                  particles read back).
* ``ensemble`` -- independent uneven runs advanced together.
* ``serve``    -- requests submitted, advanced and collected through the
                  continuous-batching server (host arrays in and out).

Inputs are seeded, of the shapes of ``sipf_inputs``: Gaussian particle clouds
(or uniform ones), the v, m, w fields that go with them.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_2605_20140_gb300 import sipf
from sipf_inputs import Params

DEV = "cuda"

# ------------------------------------------------------------------ cases

_RUN = {"kind": "run", "diffusion": 0, "v_update": 0, "order": 2, "H0": 0.0, "sigma": 0.0,
        "chi": 0.01, "spread": "seeds"}


def listed():
    return [
        # a density on demand for a small plug-in grid: launches and latency count
        {"name": "deposit-32", "kind": "deposit", "H": 32, "N": 2 ** 15, "masses": "equal"},
        # the same at the largest grid this call takes, unequal weights, an odd count
        {"name": "deposit-64", "kind": "deposit", "H": 64, "N": 1000003, "masses": "unequal"},
        # the small workload: one cloud on a 32^3 grid, its 100 steps
        {"name": "run-32", **_RUN, "H": 32, "N": 2 ** 15, "dt": 1e-3, "steps": 100},
        # a radix-3 grid with an odd, spread-out particle count, the exponential
        # multiplier and the explicit v update
        {"name": "run-72", **_RUN, "H": 72, "N": 200003, "dt": 1e-3, "steps": 100,
         "diffusion": 1, "v_update": 1, "spread": "uniform"},
        # fourth-order assignment with the low-pass filter (H0 = H^(8/13)) and the
        # regularised m source, as the convergence analysis configures it
        {"name": "run-64-order4", **_RUN, "H": 64, "N": 2 ** 18, "dt": 1e-3, "steps": 100,
         "order": 4, "H0": 64 ** (8 / 13), "sigma": 1e-3},
        # the benchmark workload: 128^3 nodes, 2^22 particles
        {"name": "run-128", **_RUN, "H": 128, "N": 2 ** 22, "dt": 5e-4, "steps": 100},
        # the largest production run: 256^3 nodes, 2^25 particles
        {"name": "run-256", **_RUN, "H": 256, "N": 2 ** 25, "dt": 2.5e-4, "steps": 200,
         "chi": 0.02},
        # a fine grid that is not a power of two with fewer particles than nodes
        {"name": "run-384", **_RUN, "H": 384, "N": 2 ** 22, "dt": 2.5e-4, "steps": 40},
        # readouts between the steps of the benchmark workload
        {"name": "readout-128", "kind": "readout", "H": 128, "N": 2 ** 22},
        # weights spread by growth and decay made equal again
        {"name": "resample-64", "kind": "resample", "H": 64, "N": 2 ** 20},
        # a parameter study: uneven independent runs
        {"name": "ensemble-9", "kind": "ensemble", "members": 9, "steps": 100},
        # requests of a service, sizes drawn like the ensemble's
        {"name": "serve-8", "kind": "serve", "members": 8, "steps": 100},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["deposit", "run", "run", "run", "run", "run", "readout", "resample",
                       "ensemble", "serve"])
    if kind == "deposit":
        return {"kind": kind, "H": rng.choice([8, 16, 24, 32, 40, 48, 64]),
                "N": _log_int(rng, 1000, 2 ** 21), "masses": rng.choice(["equal", "unequal"])}
    if kind == "readout":
        return {"kind": kind, "H": rng.choice([32, 48, 64, 96, 128, 144]),
                "N": _log_int(rng, 10000, 2 ** 22)}
    if kind == "resample":
        return {"kind": kind, "H": rng.choice([32, 64, 72, 128]), "N": _log_int(rng, 5000, 2 ** 21)}
    if kind in ("ensemble", "serve"):
        return {"kind": kind, "members": rng.randint(2, 9), "steps": rng.randint(21, 100)}
    H = rng.choice([16, 24, 32, 48, 64, 72, 96, 128, 128, 144, 192, 216, 256, 256, 288, 384])
    option = rng.choice(["plain", "plain", "plain", "exp", "order4", "filter", "sigma"])
    return {**_RUN, "H": H, "N": _log_int(rng, 5000, 2 ** 22 if H < 256 else 2 ** 24),
            "dt": 1e-3 if H <= 96 else 5e-4 if H <= 216 else 2.5e-4,
            "steps": rng.randint(41, 120) if H <= 144 else rng.randint(15, 40),
            "diffusion": int(option == "exp"), "v_update": int(option == "exp"),
            "order": 4 if option == "order4" else 2,
            "H0": round(H ** (8 / 13), 6) if option == "filter" else 0.0,
            "sigma": 1e-3 if option == "sigma" else 0.0,
            "chi": rng.choice([0.005, 0.01, 0.02]),
            "spread": rng.choice(["seeds", "seeds", "uniform"])}


# ------------------------------------------------------------------ inputs


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 13)
    return g


def _cloud(N, centres, sigma, g):
    """N positions of an equal-weight Gaussian mixture in the unit box, (3, N) float32."""
    pick = torch.randint(0, centres.shape[0], (N,), generator=g, device=DEV)
    x = centres[pick].T + sigma * torch.randn((3, N), generator=g, device=DEV,
                                              dtype=torch.float64)
    x = torch.remainder(x, 1.0).float()
    return torch.where(x >= 1.0, torch.zeros_like(x), x).contiguous()


def _fields(H, centres):
    q = torch.arange(H, device=DEV, dtype=torch.float64) / H
    v = torch.ones((H, H, H), device=DEV, dtype=torch.float64)
    m = torch.zeros_like(v)
    for c in centres:
        r2 = 0.0
        for d, shape in ((0, (1, 1, H)), (1, (1, H, 1)), (2, (H, 1, 1))):
            t = q - c[d]
            r2 = r2 + ((t - torch.round(t)) ** 2).reshape(shape)
        gs = torch.exp(-r2 / 0.01)
        v *= 1.0 - 0.5 * gs
        m += 0.5 * gs
    w = torch.full((H, H, H), 0.5, device=DEV)
    return v.float(), m.float(), w


def _inputs(H, N, seed, spread="seeds", masses="equal"):
    """Initial state in the unit box: positions (3, N), masses, v, m, w."""
    g = _generator(seed)
    k = 3 if spread == "seeds" else 1
    centres = 0.2 + 0.6 * torch.rand((k, 3), generator=g, device=DEV, dtype=torch.float64)
    if spread == "uniform":
        x = torch.rand((3, N), generator=g, device=DEV)
    else:
        x = _cloud(N, centres, 0.04, g)
    mass = torch.full((N,), 1.0 / N, device=DEV, dtype=torch.float64)
    if masses == "unequal":
        mass = mass * torch.exp(torch.randn((N,), generator=g, device=DEV, dtype=torch.float64))
    v, m, w = _fields(H, centres)
    return {"x": x, "mass": mass, "v": v, "m": m, "w": w}


def _params(case, seed):
    return Params(chi=case["chi"], diffusion=case["diffusion"], v_update=case["v_update"],
                  H0=case["H0"], seed=int(seed), p2g_order=case["order"], sigma=case["sigma"])


def _members(case, seed):
    """The members of an ensemble (or requests of a service): grids and counts
    spread over the study's range (the same for every seed, so that a pass is
    the same work), parameters and initial states from the seed."""
    out = []
    rng = np.random.default_rng(int(seed))
    n = case["members"]
    for i in range(n):
        H = (32, 48, 64, 96)[i % 4]
        N = int(round(2.0 ** (14.0 + 6.0 * ((7 * i + 3) % n + 0.5) / n)))
        p = Params(chi=rng.uniform(0.005, 0.03), alpha=rng.uniform(5.0, 20.0),
                   Du=rng.uniform(5e-4, 2e-3), seed=(int(seed) << 16) | i)
        g = _generator(int(seed) * 64 + i)
        centre = torch.full((1, 3), 0.5, device=DEV, dtype=torch.float64)
        v, m, w = _fields(H, centre)
        mass = torch.full((N,), 1.0 / N, device=DEV, dtype=torch.float64)
        out.append({"H": H, "N": N, "params": p, "x": _cloud(N, centre, 0.05, g), "mass": mass,
                    "v": v, "m": m, "w": w, "dt": 1e-3, "steps": case["steps"]})
    return out


class _Owner:
    """Closes a handle of the library when the state that holds it goes."""

    def __init__(self, handle, close):
        self.handle, self._close = handle, close

    def __del__(self):
        if self.handle is not None:
            self._close(self.handle)
            self.handle = None


def _context(H, N, params):
    stream = torch.cuda.Stream()
    ctx = sipf.sipf_create(sipf.make_grid(H, 1.0), N, sipf.make_params(params),
                           stream.cuda_stream)
    return stream, _Owner(ctx, sipf.sipf_destroy)


def _set(ctx, s):
    sipf.sipf_set_state(ctx, s["x"], s["mass"], None, s["v"], s["m"], s["w"], sipf.SIPF_DEVICE)


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "deposit":
        st |= _inputs(case["H"], case["N"], seed, masses=case["masses"])
        st["grid"] = sipf.make_grid(case["H"], 1.0)
        st["u"] = torch.empty((case["H"],) * 3, device=DEV)
    elif kind in ("run", "readout", "resample"):
        H, N = case["H"], case["N"]
        st |= _inputs(H, N, seed, case.get("spread", "seeds"),
                      "unequal" if kind == "resample" else "equal")
        p = _params(case, seed) if kind == "run" else Params(seed=int(seed))
        st["stream"], st["owner"] = _context(H, N, p)
        st["params"] = p
        torch.cuda.synchronize()
        if kind == "run":
            st["out"] = torch.empty((7, H, H, H), device=DEV)
        elif kind == "readout":
            st["out"] = torch.empty((7, H, H, H), device=DEV)
            st["cells"] = torch.empty(H ** 3 + 1, device=DEV, dtype=torch.int32)
            st["ids"] = torch.empty(N, device=DEV, dtype=torch.int32)
            st["starts"] = torch.empty(H ** 3 + 1, device=DEV, dtype=torch.int32)
            _set(st["owner"].handle, st)
        else:
            st["px"] = torch.empty((3, N), device=DEV)
            st["pm"] = torch.empty(N, device=DEV, dtype=torch.float64)
            st["pid"] = torch.empty(N, device=DEV, dtype=torch.int32)
    elif kind == "ensemble":
        st["members"] = _members(case, seed)
        ens = sipf.Ensemble([(s["H"], 1.0, (0.0, 0.0, 0.0), s["N"], s["params"])
                             for s in st["members"]])
        st["owner"] = _Owner(ens, lambda e: e.close())
        st["dts"] = np.array([s["dt"] for s in st["members"]])
        st["outs"] = [torch.empty((7,) + (s["H"],) * 3, device=DEV) for s in st["members"]]
    else:
        st["requests"] = [{k: a.cpu().numpy() if isinstance(a, torch.Tensor) else a
                           for k, a in s.items()} for s in _members(case, seed)]
        for s in st["requests"]:
            s["x"] = np.ascontiguousarray(s["x"].T)      # (N, 3), as the server takes it
        st["owner"] = _Owner(sipf.Server(20 << 30), lambda srv: srv.close())
    torch.cuda.synchronize()
    return st


# ------------------------------------------------------------------ passes


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "deposit":
        sipf.sipf_deposit_noalloc(st["grid"], st["x"], st["mass"], case["N"], st["u"],
                                  torch.cuda.current_stream().cuda_stream)
        return st["u"]
    if kind == "ensemble":
        ens = st["owner"].handle
        for sim, s in zip(ens.members, st["members"]):
            _set(sim.ctx, s)
        ens.step(st["dts"], case["steps"])
        for sim, out in zip(ens.members, st["outs"]):
            sipf.sipf_fields(sim.ctx, 127, out, sipf.SIPF_DEVICE)
        return [dict(zip(sipf.FIELD_NAMES, out)) for out in st["outs"]]
    if kind == "serve":
        srv = st["owner"].handle
        rids = [srv.submit(s["H"], 1.0, (0.0, 0.0, 0.0), s["N"], s["params"], s["x"], s["mass"],
                           s["v"], s["m"], s["w"], s["dt"], s["steps"]) for s in st["requests"]]
        done = {}
        while len(done) < len(rids):
            srv.advance()
            for rid in srv.poll():
                done[rid] = srv.collect(rid)
        return [done[rid] for rid in rids]
    ctx = st["owner"].handle
    if kind == "run":
        _set(ctx, st)
        sipf.sipf_step(ctx, case["dt"], case["steps"])
        sipf.sipf_fields(ctx, 127, st["out"], sipf.SIPF_DEVICE)
        return dict(zip(sipf.FIELD_NAMES, st["out"]))
    if kind == "readout":
        sipf.sipf_canonical_order(ctx, st["cells"], st["ids"], sipf.SIPF_DEVICE)
        sipf.sipf_cell_start(ctx, st["starts"], sipf.SIPF_DEVICE)
        d = sipf.sipf_diagnostics(ctx)
        sipf.sipf_fields(ctx, 127, st["out"], sipf.SIPF_DEVICE)
        return {"cells": st["cells"], "ids": st["ids"], "starts": st["starts"],
                "diagnostics": {k: d[k] for k in ("mass_particles", "mass_grid", "min_u", "min_v",
                                                  "min_m", "min_w", "nonfinite")},
                **dict(zip(sipf.FIELD_NAMES, st["out"]))}
    _set(ctx, st)
    sipf.sipf_resample(ctx, 0.0)
    sipf.sipf_particles(ctx, st["px"], st["pm"], st["pid"], sipf.SIPF_DEVICE)
    # the storage order within a tile is not specified: by id
    order = torch.argsort(st["pid"])
    return {"x": st["px"][:, order], "mass": st["pm"][order], "id": st["pid"][order]}


# ------------------------------------------------------------------ work

def _run_work(H, N, steps, order=2):
    """Initial state in, steps, seven fields out.  Per particle and step: read
    and write position (12 B) and log-mass (8 B); per node and step: read v, m,
    w, u, write v, m, w, grad v, and the gather and the deposit (60 B)."""
    H3 = H ** 3
    bytes_ = 20 * N + 12 * H3 + steps * (40 * N + 60 * H3) + 28 * H3
    # gather 64, deposit 24 (R^(4): 160), noise and push about 120 per particle;
    # three complex transforms of each of three fields, 5 log2 H per node and axis
    flops = steps * (N * (208 if order == 2 else 344) + 3 * 2 * 3 * 2.5 * math.log2(H) * H3)
    return bytes_, flops


def work(case):
    kind = case["kind"]
    if kind == "deposit":
        b, f = 20 * case["N"] + 4 * case["H"] ** 3, 40 * case["N"]
    elif kind == "readout":
        H3, N = case["H"] ** 3, case["N"]
        b, f = 28 * N + 8 * H3 + 28 * H3, 60 * N
    elif kind == "resample":
        b, f = (20 + 24) * case["N"] + 12 * case["H"] ** 3, 20 * case["N"]
    elif kind == "run":
        b, f = _run_work(case["H"], case["N"], case["steps"], case["order"])
    else:
        b = f = 0
        for i in range(case["members"]):
            H = (32, 48, 64, 96)[i % 4]
            N = 2.0 ** (14.0 + 6.0 * ((7 * i + 3) % case["members"] + 0.5) / case["members"])
            db, df = _run_work(H, N, case["steps"])
            b, f = b + db, f + df
    return {"bytes": float(b), "flops": float(f)}


# ------------------------------------------------------------------ 64 bits

_U32 = 0xFFFFFFFF


def _philox_normals(N, n, seed):
    """Three standard normals per particle id 0..N-1 in step n: Box-Muller on
    the Philox4x32-10 words of counter (n, 0, id, 0)."""
    c0 = torch.full((N,), n & _U32, device=DEV, dtype=torch.int64)
    c2 = torch.arange(N, device=DEV, dtype=torch.int64)
    c1, c3 = torch.zeros_like(c0), torch.zeros_like(c0)
    k0, k1 = seed & _U32, (seed >> 32) & _U32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((p1 >> 32) & _U32) ^ c1 ^ k0, p1 & _U32,
                          ((p0 >> 32) & _U32) ^ c3 ^ k1, p0 & _U32)
        k0, k1 = (k0 + 0x9E3779B9) & _U32, (k1 + 0xBB67AE85) & _U32
    u0, u1, u2, u3 = ((2 * (c >> 9) + 1).double() * 2.0 ** -24 for c in (c0, c1, c2, c3))
    r0, r2 = torch.sqrt(-2.0 * torch.log(u0)), torch.sqrt(-2.0 * torch.log(u2))
    return torch.stack([r0 * torch.cos(2 * math.pi * u1), r0 * torch.sin(2 * math.pi * u1),
                        r2 * torch.cos(2 * math.pi * u3)])


def _cells(s, H):
    c = torch.floor(s)
    f = s - c
    c = c.long().clamp_(0, H - 1)
    return c, f


def _corners(s, H):
    """(flat node index, trilinear weight) of the eight corners of each particle's cell."""
    c, f = _cells(s, H)
    c1 = torch.where(c + 1 < H, c + 1, torch.zeros_like(c))
    for k in range(8):
        d = (k & 1, (k >> 1) & 1, k >> 2)
        n = [c1[j] if d[j] else c[j] for j in range(3)]
        w = 1.0
        for j in range(3):
            w = w * (f[j] if d[j] else 1.0 - f[j])
        yield (n[2] * H + n[1]) * H + n[0], w


def _density(s, a, H, order):
    u = torch.zeros(H ** 3, device=DEV, dtype=torch.float64)
    if order == 2:
        for node, w in _corners(s, H):
            u.index_add_(0, node, a * w)
    else:
        c, f = _cells(s, H)
        for ox in range(-1, 3):
            for oy in range(-1, 3):
                for oz in range(-1, 3):
                    o = (ox, oy, oz)
                    outer = [j for j in range(3) if o[j] in (-1, 2)]
                    if len(outer) > 1:
                        continue
                    p = [(f[j] - o[j]).abs() for j in range(3)]
                    if not outer:
                        w = (1 - p[0]) * (1 - p[1]) * (1 - p[2])
                        w = w * (1 + sum(t * (1 - t) for t in p) / 2)
                    else:
                        t = p[outer[0]]
                        w = -(t - 1) * (2 - t) * (3 - t) / 6
                        for j in range(3):
                            if j != outer[0]:
                                w = w * (1 - p[j])
                    n = [torch.remainder(c[j] + o[j], H) for j in range(3)]
                    u.index_add_(0, (n[2] * H + n[1]) * H + n[0], a * w)
    return u.reshape(H, H, H) * float(H) ** 3


class _Exact:
    """The scheme in 64 bits on the unit box (ids 0..N-1)."""

    def __init__(self, H, s, p):
        self.H, self.p, self.n = H, p, 0
        self.s = torch.remainder(s["x"].double() * H, float(H))
        self.loga = torch.log(s["mass"])
        self.v, self.m, self.w = (s[k].double() for k in "vmw")
        q = torch.fft.fftfreq(H, 1.0 / H, device=DEV, dtype=torch.float64)
        qr = torch.arange(H // 2 + 1, device=DEV, dtype=torch.float64)
        self.q = (qr.reshape(1, 1, -1), q.reshape(1, -1, 1), q.reshape(-1, 1, 1))
        self.q2 = self.q[0] ** 2 + self.q[1] ** 2 + self.q[2] ** 2
        on = 0.0 < p.H0 < H
        self.filter = torch.exp(-2 * math.pi ** 2 * self.q2 / p.H0 ** 2) if on else 1.0
        self.grad = self._gradient()

    def _back(self, F):
        return torch.fft.irfftn(F, s=(self.H,) * 3)

    def _gradient(self):
        V = torch.fft.rfftn(self.v) * self.filter
        out = []
        for q in self.q:
            k = torch.where(q.abs() == self.H / 2, torch.zeros_like(q), q)
            out.append(self._back(2j * math.pi * k * V))
        return out

    def density(self):
        return _density(self.s, torch.exp(self.loga), self.H, self.p.p2g_order)

    def _diffuse(self, f, D, R, tau):
        k2 = (2 * math.pi) ** 2 * self.q2
        g = torch.exp(-tau * D * k2 - tau * R) if self.p.diffusion else 1 / (1 + tau * R + tau * D * k2)
        return self._back(torch.fft.rfftn(f) * g * self.filter)

    def step(self, tau):
        p, H = self.p, self.H
        self.n += 1
        u = self.density()
        um = u
        if p.sigma > 0:
            um = self._back(torch.fft.rfftn(u)
                            * torch.exp(-p.sigma * (2 * math.pi) ** 2 * self.q2 / 2))
        got = [torch.zeros_like(self.loga) for _ in range(4)]
        at = [f.reshape(-1) for f in (*self.grad, self.w)]
        for node, wt in _corners(self.s, H):
            for g, f in zip(got, at):
                g += wt * f[node]
        z = _philox_normals(self.loga.numel(), self.n, p.seed)
        noise = math.sqrt(2 * p.Du * tau) * H
        s = self.s + p.chi * tau * H * torch.stack(got[:3]) + noise * z
        s = s - H * torch.floor(s / H)
        self.s = torch.where(s >= H, torch.zeros_like(s), s)
        self.loga = self.loga + torch.log1p(tau * (2 * got[3] / (1 + got[3]) - 1))
        ms = self.m + tau * um
        ws = self.w + tau * (p.gamma * self.v - 2 * u / (1 + u) * self.w)
        self.v = (self.v * (1 - p.alpha * tau * self.m) if p.v_update
                  else self.v / (1 + p.alpha * tau * self.m))
        self.m = self._diffuse(ms, p.Dm, p.beta, tau)
        self.w = self._diffuse(ws, p.Dw, 1.0, tau)
        self.grad = self._gradient()

    def fields(self):
        return {"u": self.density(), "v": self.v, "m": self.m, "w": self.w, "gx": self.grad[0],
                "gy": self.grad[1], "gz": self.grad[2]}


def _exact_run(H, s, p, dt, steps):
    e = _Exact(H, s, p)
    for _ in range(steps):
        e.step(dt)
    return e.fields()


def exact(case, seed):
    kind = case["kind"]
    if kind == "deposit":
        s = _inputs(case["H"], case["N"], seed, masses=case["masses"])
        H = case["H"]
        return _density(torch.remainder(s["x"].double() * H, float(H)), s["mass"], H, 2)
    if kind == "run":
        # about 20 seconds of 64-bit steps at most
        if case["steps"] * (case["N"] * (4 if case["order"] == 4 else 1) + 4 * case["H"] ** 3) > 2e9:
            return None
        s = _inputs(case["H"], case["N"], seed, case["spread"])
        return _exact_run(case["H"], s, _params(case, seed), case["dt"], case["steps"])
    if kind == "readout":
        H, N = case["H"], case["N"]
        s = _inputs(H, N, seed)
        e = _Exact(H, s, Params())
        T = H // 8
        sf = torch.clamp(torch.floor(s["x"] * float(H)), 0, H - 1).long()
        tile = ((sf[2] >> 3) * T + (sf[1] >> 3)) * T + (sf[0] >> 3)
        key = (tile << 9) | ((sf[2] & 7) << 6) | ((sf[1] & 7) << 3) | (sf[0] & 7)
        ids = torch.argsort(key, stable=True).int()
        cells = torch.zeros(H ** 3 + 1, device=DEV, dtype=torch.int64)
        cells[1:] = torch.cumsum(torch.bincount(key, minlength=H ** 3), 0)
        f = e.fields()
        return {"cells": cells.int(), "ids": ids, "starts": cells.int(),
                "diagnostics": {"mass_particles": float(s["mass"].sum()),
                                "mass_grid": float(f["u"].sum()) / H ** 3, "min_u": None,
                                "min_v": float(f["v"].min()), "min_m": float(f["m"].min()),
                                "min_w": float(f["w"].min()), "nonfinite": 0}, **f}
    if kind == "resample":
        N = case["N"]
        s = _inputs(case["H"], N, seed, masses="unequal")
        mean = torch.full((N,), float(s["mass"].sum()) / N, device=DEV, dtype=torch.float64)
        return {"x": None, "mass": mean, "id": torch.arange(N, device=DEV, dtype=torch.int32)}
    return [_exact_run(s["H"], s, s["params"], s["dt"], s["steps"])
            for s in _members(case, seed)]
