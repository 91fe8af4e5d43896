"""What the simulator's performance is measured on.

A case is a dict of plain values.  Six kinds of work stand for what a program
does with the simulator, each through its public calls:

* ``run``      one network advanced by ``Network.run`` and its new spikes and
               state read, as an interactive program or a long run in pieces does;
* ``pair``     two large networks of one grid (slow waves and awake-like firing)
               advanced side by side by ``run_concurrent``;
* ``batch``    a parameter sweep of small networks advanced by ``run_batch``;
* ``request``  a whole simulation: build, run, read everything, free;
* ``serve``    a stream of requests of mixed sizes through ``serve.Server``;
* ``build``    the synapse rows of a network built into the caller's own memory.

Networks are those of the repository's workloads: modules of 1250 neurons on a
grid, 1125 synapses per neuron, delays of 1..20 steps of 0.1 ms, 80% of the
excitatory synapses kept in the module, the slow-wave (SWA) and awake-like (AW)
regimes, or the Table S1 efficacies with the pure Eq. 1 kernel (S1).  Records
are f32 or i16.  Networks that are advanced have left the volley of their
initial state behind before the first pass.
"""
from __future__ import annotations

import ctypes
import math
import random

import numpy as np
import torch

import paper_1902_08410_gb300 as snn
from paper_1902_08410_gb300 import serve

K = 1250                      # neurons per module
REGIMES = {"SWA": (0.02, 1.6), "AW": (0.005, 4.5)}   # adaptation conductance (nS), external rate per train (Hz)
RATE_HZ = {"SWA": 4.0, "AW": 8.7, "S1": 8.0}         # mean firing, for the work done by a pass
RECORD_BYTES = {"f32": 8, "i16": 6}


def _params(gx, gy, lam, regime, fmt, n_delay=20, min_delay=1, out_degree=1125, g_c=None, nu_ext=None):
    exc = 0.5
    p = {
        "gx": gx, "gy": gy, "lambda": lam, "p_local": 0.8, "out_degree": out_degree,
        "n_delay": n_delay, "min_delay": min_delay, "dt_ms": 0.1,
        "record_format": snn.REC_I16 if fmt == "i16" else snn.REC_F32, "bin_steps": 50,
        "dJ_frac": 0.25, "dJ_ext_frac": 0.25,
        "J": [[exc, exc, -2.0] for _ in range(3)],
        "J_ext": [0.858, 0.858, 1.120], "N_ext": [400.0, 400.0, 400.0],
        "tau_m": [20.0, 20.0, 10.0], "C_m": [1.0, 1.0, 1.0], "E_L": [0.0, 0.0, 0.0],
        "V_th": [20.0, 20.0, 20.0], "V_r": [15.0, 15.0, 15.0], "tau_arp": [2.0, 2.0, 1.0],
        "alpha_c": [1.0, 1.0, 0.0], "tau_c": [1000.0, 1000.0, 1000.0],
    }
    if regime == "S1":        # Table S1, state AW 8.8 Hz: three populations, pure Eq. 1 kernel
        p["p_local"] = -1.0
        p["J"] = [[0.515, 0.412, -1.5], [0.412, 0.429, -1.5], [0.560, 0.560, -1.5]]
        p["J_ext"] = [1.416, 1.416, 1.120]
        p["nu_ext"] = [3.17, 3.17, 3.0]
        p["g_c"] = [0.02, 0.02, 0.0]
    else:
        g, nu = REGIMES[regime]
        g, nu = (g if g_c is None else g_c), (nu if nu_ext is None else nu_ext)
        p["g_c"] = [g, g, 0.0]
        p["nu_ext"] = [nu, nu, nu]
    return p


def listed():
    return [
        # Closed loop on a small patch of cortex: the program looks at the spikes and the state after every
        # step of 0.1 ms.  The smallest call: latency and launches are all there is.
        {"name": "run_2x2_one_step", "kind": "run", "gx": 2, "gy": 2, "lam": 0.4, "regime": "AW", "fmt": "f32",
         "n_delay": 20, "min_delay": 1, "out_degree": 1125, "steps": 1},
        # The 4x4 slow-wave network over its whole second, in one call: many cheap steps.
        {"name": "run_4x4_swa_1s", "kind": "run", "gx": 4, "gy": 4, "lam": 0.4, "regime": "SWA", "fmt": "f32",
         "n_delay": 20, "min_delay": 1, "out_degree": 1125, "steps": 10000},
        # The repository's headline grid on its own (720k neurons, 0.81G synapses), 0.1 s a call.
        {"name": "run_24x24_aw", "kind": "run", "gx": 24, "gy": 24, "lam": 1.0, "regime": "AW", "fmt": "f32",
         "n_delay": 20, "min_delay": 1, "out_degree": 1125, "steps": 1000},
        # The largest grid of the benchmark (5.12M neurons, 5.76G synapses), packed records.
        {"name": "run_64x64_aw_i16", "kind": "run", "gx": 64, "gy": 64, "lam": 1.0, "regime": "AW", "fmt": "i16",
         "n_delay": 20, "min_delay": 1, "out_degree": 1125, "steps": 500},
        # The paper's own exchange step: no delay below 1 ms, spikes of ten steps delivered together.
        {"name": "run_16x16_exchange_1ms", "kind": "run", "gx": 16, "gy": 16, "lam": 1.0, "regime": "AW",
         "fmt": "i16", "n_delay": 20, "min_delay": 10, "out_degree": 1125, "steps": 1000},
        # Table S1 on a ragged grid with slow fibres (delays to 6 ms) and a short call.
        {"name": "run_13x7_table_s1", "kind": "run", "gx": 13, "gy": 7, "lam": 0.6, "regime": "S1", "fmt": "f32",
         "n_delay": 60, "min_delay": 1, "out_degree": 1125, "steps": 250},
        # The benchmark's default workload: the 24x24 slow-wave and awake-like networks side by side.
        {"name": "pair_24x24", "kind": "pair", "gx": 24, "gy": 24, "lam": 1.0, "fmt": "f32", "steps": 1000},
        # A sweep from slow waves to awake-like firing: 64 networks of sides 2..8 in one call.
        {"name": "batch_64_sweep", "kind": "batch", "nets": 64, "min_side": 2, "max_side": 8, "fmt": "i16",
         "steps": 1000},
        # One small simulation from its parameters to its spikes, rates and state.
        {"name": "request_6x6", "kind": "request", "gx": 6, "gy": 6, "lam": 1.0, "regime": "SWA", "fmt": "i16",
         "steps": 2000},
        # Twelve requests of sides 2..16 through the server: builds, batched chunks, reads and releases.
        {"name": "serve_12", "kind": "serve", "nets": 12, "min_side": 2, "max_side": 16, "fmt": "i16",
         "min_steps": 500, "max_steps": 3000},
        # Construction of a small network's rows (20k rows, 22.5M synapses).
        {"name": "build_4x4", "kind": "build", "gx": 4, "gy": 4, "lam": 0.4, "fmt": "f32", "out_degree": 1125},
        # Construction of the headline grid's rows, packed (720k rows, 0.81G synapses).
        {"name": "build_24x24_i16", "kind": "build", "gx": 24, "gy": 24, "lam": 1.0, "fmt": "i16",
         "out_degree": 1125},
    ]


def draw(rng):
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))

    def grid(most):
        gx = int(min(most, log(1, most)))
        return gx, max(1, min(most, int(round(gx * rng.uniform(0.5, 2.0)))))

    fmt = rng.choice(["f32", "i16"])
    lam = round(rng.choice([0.4, 0.6, 1.0, 2.0]) * rng.uniform(0.9, 1.1), 3)
    kind = rng.choice(["run", "run", "run", "run", "pair", "batch", "request", "serve", "build", "build"])
    if kind == "run":
        gx, gy = grid(56)
        n_delay = rng.choice([20, 20, 20, rng.randint(2, 32), rng.randint(33, 200)])
        min_delay = rng.choice([1, 1, min(n_delay, 10), rng.randint(1, n_delay)])
        most = 4096 * 500 * 0.7 / (gx * gy)        # module-steps of the largest listed case
        return {"kind": "run", "gx": gx, "gy": gy, "lam": lam, "regime": rng.choice(["SWA", "AW", "AW", "S1"]),
                "fmt": fmt, "n_delay": n_delay, "min_delay": min_delay,
                "out_degree": rng.choice([1125, 1125, rng.randint(100, 1300)]),
                "steps": max(1, int(log(1, min(5000.0, most))))}
    if kind == "pair":
        gx, gy = rng.randint(6, 28), rng.randint(6, 28)
        return {"kind": "pair", "gx": gx, "gy": gy, "lam": lam, "fmt": fmt, "steps": int(log(100, 1200))}
    if kind == "batch":
        lo = rng.randint(1, 4)
        return {"kind": "batch", "nets": int(log(2, 64)), "min_side": lo, "max_side": rng.randint(lo, 8),
                "fmt": fmt, "steps": int(log(50, 1500))}
    if kind == "request":
        gx, gy = grid(16)
        return {"kind": "request", "gx": gx, "gy": gy, "lam": lam, "regime": rng.choice(["SWA", "AW"]), "fmt": fmt,
                "steps": int(log(100, 4000))}
    if kind == "serve":
        lo = rng.randint(100, 1000)
        return {"kind": "serve", "nets": rng.randint(3, 12), "min_side": 2, "max_side": rng.randint(3, 16),
                "fmt": fmt, "min_steps": lo, "max_steps": lo + rng.randint(1, 2000)}
    gx, gy = grid(23)
    return {"kind": "build", "gx": gx, "gy": gy, "lam": lam, "fmt": fmt,
            "out_degree": rng.choice([1125, 1125, rng.randint(100, 1300)])}


def _sweep(case, rng):
    """Parameters of a sweep's networks: sides, adaptation and external rate as the batched workload draws them."""
    out = []
    for _ in range(case["nets"]):
        side = rng.randint(case["min_side"], case["max_side"])
        g = 0.02 + (0.005 - 0.02) * rng.randrange(16) / 15.0
        out.append(_params(side, side, 1.0, "SWA", case["fmt"], g_c=g, nu_ext=rng.uniform(2.0, 8.0)))
    return out


def _sides(case, rng):
    """Grid side, steps and regime of every request of a stream."""
    lo, hi = math.log2(case["min_side"]), math.log2(case["max_side"])
    return [(int(round(2.0 ** rng.uniform(lo, hi))), rng.randint(case["min_steps"], case["max_steps"]),
             rng.choice(["SWA", "AW"])) for _ in range(case["nets"])]


def _case_rng(case):
    # sizes belong to the case, not to the seed of its inputs: every seed is the same amount of work
    return random.Random(",".join("%s=%s" % (k, case[k]) for k in sorted(case) if k != "name"))


class Buffers:
    """Host arrays a program keeps for what it reads: spikes, counted in `n` and zero behind, and the state of
    `neurons` neurons.  Room for `steps` steps at 60 Hz and `volley` spikes of each neuron."""

    def __init__(self, neurons, steps, volley):
        cap = int(neurons * (steps * 1e-4 * 60.0 + volley)) + 64
        self.steps, self.ids = np.zeros(cap, np.int32), np.zeros(cap, np.int32)    # both below 2^31
        self.V, self.c, self.ref = (np.zeros(neurons, d) for d in (np.float32, np.float32, np.int32))
        self.n = self.at = self.last = 0

    def start(self):
        self.last, self.n, self.at = self.n, 0, 0

    def read(self, net, t0, t1):
        """The spikes of [t0, t1) and the state of a network, behind what was read before."""
        lib, got = snn.lib(), ctypes.c_size_t(0)
        _ok(lib.snn_read_spikes(net.handle, t0, t1, ctypes.c_void_p(self.steps[self.n:].ctypes.data),
                                ctypes.c_void_p(self.ids[self.n:].ctypes.data), len(self.ids) - self.n,
                                ctypes.byref(got)))
        to = [ctypes.c_void_p(a[self.at:].ctypes.data) for a in (self.V, self.c, self.ref)]
        _ok(lib.snn_read_state(net.handle, *to, net.N))
        self.n += got.value
        self.at += net.N

    def done(self):
        self.steps[self.n:self.last] = 0
        self.ids[self.n:self.last] = 0
        return {"n": self.n, "steps": self.steps, "ids": self.ids, "V": self.V, "c": self.c, "ref": self.ref}


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "t": 0}
    if kind == "run":
        p = _params(case["gx"], case["gy"], case["lam"], case["regime"], case["fmt"], case["n_delay"],
                    case["min_delay"], case["out_degree"])
        s["nets"] = [snn.Network(p, 1000 + seed)]
        s["nets"][0].run(1000)
    elif kind == "pair":
        s["streams"] = [torch.cuda.Stream() for _ in range(2)]
        s["nets"] = [snn.Network(_params(case["gx"], case["gy"], case["lam"], regime, case["fmt"]), 1000 + seed + i,
                                 stream=s["streams"][i].cuda_stream) for i, regime in enumerate(("SWA", "AW"))]
        snn.run_concurrent(s["nets"], 1000)
    elif kind == "batch":
        s["nets"] = [snn.Network(p, 1000 * seed + i) for i, p in enumerate(_sweep(case, _case_rng(case)))]
        snn.run_batch(s["nets"], 1000)
    elif kind == "request":
        s["params"] = _params(case["gx"], case["gy"], case["lam"], case["regime"], case["fmt"])
        s["seed"] = 1000 + seed
        s["read"] = Buffers(case["gx"] * case["gy"] * K, case["steps"], 4)
    elif kind == "serve":
        sides = _sides(case, _case_rng(case))
        s["requests"] = [(_params(side, side, 1.0, regime, case["fmt"]), 1000 * seed + i, steps)
                         for i, (side, steps, regime) in enumerate(sides)]
        s["read"] = Buffers(sum(side * side * K for side, _, _ in sides), case["max_steps"], 4)
    else:
        p = _params(case["gx"], case["gy"], case["lam"], "AW", case["fmt"], out_degree=case["out_degree"])
        s["params"], s["seed"] = snn.make_params(p), 1000 + seed
        need = ctypes.c_size_t(0)
        _ok(snn.lib().snn_build_rows_static(ctypes.byref(s["params"]), s["seed"], None, ctypes.byref(need), None))
        s["rows"] = torch.empty(need.value, dtype=torch.uint8, device="cuda")
    if "nets" in s:
        s["t"] = 1000
        s["read"] = Buffers(sum(net.N for net in s["nets"]), case["steps"], 0.5)
    return s


def _ok(rc):
    if rc != snn.SNN_OK:
        raise snn.SnnError(rc, snn.lib().snn_last_error().decode())


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind != "build":
        read = state["read"]
        read.start()
    if kind in ("run", "pair", "batch"):
        nets, n = state["nets"], case["steps"]
        if kind == "run":
            nets[0].run(n)
        elif kind == "pair":
            snn.run_concurrent(nets, n)
        else:
            snn.run_batch(nets, n)
        t0 = state["t"]
        state["t"] = t0 + n
        for net in nets:
            read.read(net, t0, t0 + n)
        return read.done()
    if kind == "request":
        net = snn.Network(state["params"], state["seed"])
        net.run(case["steps"])
        read.read(net, 0, case["steps"])
        rates = net.rates()
        net.close()
        return dict(read.done(), rates=rates.view(np.int32))
    if kind == "serve":
        server = serve.Server(memory_budget=64 << 30, realtime=False, keep_state=True)
        for params, seed, steps in state["requests"]:
            server.submit(params, seed, steps)
        results = server.run()["results"]
        for r in results:
            k, m = len(r.spike_ids), len(r.state[0])
            read.steps[read.n:read.n + k], read.ids[read.n:read.n + k] = r.spike_steps, r.spike_ids
            for a, b in zip((read.V, read.c, read.ref), r.state):
                a[read.at:read.at + m] = b
            read.n += k
            read.at += m
        return dict(read.done(), rates=np.concatenate([r.rates.reshape(-1) for r in results]).view(np.int32))
    rows = state["rows"]
    have = ctypes.c_size_t(rows.numel())
    _ok(snn.lib().snn_build_rows_static(ctypes.byref(state["params"]), state["seed"],
                                        ctypes.c_void_p(rows.data_ptr()), ctypes.byref(have),
                                        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    N, m_pad = case["gx"] * case["gy"] * K, (case["out_degree"] + 7) // 8 * 8
    rows = rows.view(N, -1)
    weight = torch.int16 if case["fmt"] == "i16" else torch.float32
    return {"keys": rows[:, :4 * m_pad].view(torch.int32), "weights": rows[:, 4 * m_pad:].view(weight)}


def work(case):
    """Of an advance: the state read and written once, the records of every spike read once (at the regime's mean
    rate), the spikes written once, about 30 integer and floating operations per neuron and step for the drive and the
    integration, and an addition per delivered record.  Of a construction: the rows written once, about 70 operations
    per synapse."""
    kind = case["kind"]

    def advance(modules, steps, regime, fmt, M=1125):
        n = modules * K
        spikes = n * steps * 1e-4 * RATE_HZ[regime]
        return np.array([n * 18 + spikes * (M * RECORD_BYTES[fmt] + 8), n * steps * 30.0 + spikes * M])

    def rows(modules, fmt, M=1125):
        n = modules * K
        return np.array([n * ((M + 7) // 8 * 8) * RECORD_BYTES[fmt], n * M * 70.0])

    if kind == "run":
        w = advance(case["gx"] * case["gy"], case["steps"], case["regime"], case["fmt"], case["out_degree"])
    elif kind == "pair":
        w = sum(advance(case["gx"] * case["gy"], case["steps"], r, case["fmt"]) for r in ("SWA", "AW"))
    elif kind == "batch":
        w = sum(advance(p["gx"] * p["gy"], case["steps"], "AW", case["fmt"]) for p in _sweep(case, _case_rng(case)))
    elif kind == "request":
        m = case["gx"] * case["gy"]
        w = rows(m, case["fmt"]) + advance(m, case["steps"], case["regime"], case["fmt"])
    elif kind == "serve":
        w = sum(rows(side * side, case["fmt"]) + advance(side * side, steps, regime, case["fmt"])
                for side, steps, regime in _sides(case, _case_rng(case)))
    else:
        w = rows(case["gx"] * case["gy"], case["fmt"], case["out_degree"])
    return {"bytes": float(w[0]), "flops": float(w[1])}


# ---------------------------------------------------------------------------
# 64-bit values.  Weights of constructed rows have them.  The state after an
# advance has none: a spike is a comparison of the rounded potential with the
# threshold, so any other rounding gives another raster within a few steps,
# and V and c follow it.  (i16 weights, keys and spikes are whole numbers.)
# ---------------------------------------------------------------------------
def _philox(c, key):
    """Philox4x32-10 of counter words c (int64 tensors holding 32-bit values)."""
    mask = 0xFFFFFFFF
    k0, k1 = key & mask, key >> 32
    c0, c1, c2, c3 = c
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57      # low 64 bits: the arithmetic wraps
        c0, c1, c2, c3 = ((p1 >> 32) & mask) ^ c1 ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c3 ^ k1, p0 & mask
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c0, c1, c2, c3


def exact(case, seed):
    if case["kind"] != "build" or case["fmt"] != "f32" or case["gx"] * case["gy"] * case["out_degree"] > 40 * 1125:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    gx, gy, M = case["gx"], case["gy"], case["out_degree"]
    G = gx * gy
    p = _params(gx, gy, case["lam"], "AW", "f32", out_degree=M)
    lam, p_local = float(np.float32(p["lambda"])), float(np.float32(p["p_local"]))
    # cumulative probability of the target module of every source module, in units of 2^-32
    y, x = np.divmod(np.arange(G), gx)
    kern = np.exp(-np.sqrt((x[:, None] - x) ** 2.0 + (y[:, None] - y) ** 2.0) / lam)
    np.fill_diagonal(kern, 0.0)
    prob = np.zeros((G, G))
    if G > 1:
        prob = (1.0 - p_local) * kern / np.cumsum(kern, 1)[:, -1:]
    np.fill_diagonal(prob, p_local)
    edges = np.minimum(np.floor(np.cumsum(prob, 1)[:, :-1] * 2.0 ** 32), 2.0 ** 32 - 1).astype(np.int64)
    z = torch.special.ndtri((torch.arange(4096, dtype=torch.float64, device=dev) + 0.5) / 4096.0)
    m_pad = (M + 7) // 8 * 8
    out = torch.zeros((G * K, m_pad), dtype=torch.float64, device=dev)
    j = torch.arange(M, device=dev)
    for m in range(G):
        src = torch.arange(m * K, (m + 1) * K, device=dev)[:, None]
        zero = torch.zeros((K, M), dtype=torch.int64, device=dev)
        r0, r1, r2, r3 = _philox((zero + src, zero + j, zero, zero), 1000 + seed)
        module = torch.full_like(r0, m)
        if G > 1:
            module = torch.searchsorted(torch.from_numpy(edges[m]).to(dev), r0, right=True)
        inhibitory = torch.arange(K, device=dev)[:, None] >= 1000
        module = torch.where(inhibitory, torch.full_like(module, m), module)     # inhibitory targets stay local
        target = module * K + ((r1 * K) >> 32)
        delay = 1 + ((r2 * p["n_delay"]) >> 32)
        J = torch.where(inhibitory, -2.0, 0.5).double()
        w = J + 0.25 * J.abs() * z[r3 >> 20]
        w = torch.where(J > 0, w.clamp(min=0.0), w.clamp(max=0.0))
        order = torch.sort((delay << 24) | target, dim=1, stable=True).indices
        out[m * K:(m + 1) * K, :M] = torch.gather(w, 1, order)
    return {"keys": None, "weights": out.cpu().numpy()}
