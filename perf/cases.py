"""The work that users of this library have it do, as timed cases.

A case is a dict of plain values. Three kinds:
  transport  whole transport jobs through a context: the event's rows reset,
             its primaries queued (from host arrays, as an offloading
             application holds them, or from device memory), the step loop
             run to the end, the tallies of every event read;
  serve      a burst of requests through the continuous-batching loop;
  partition  the allocation-free partition of slot indices by key.
Energies in MeV, lengths in cm, fields in tesla.
"""
import math

import numpy as np
import torch

from paper_2503_17608_gb300 import binding, workloads as wl

POLICIES = {"none": wl.SORT_NONE, "action": wl.SORT_ACTION, "action_type": wl.SORT_ACTION_TYPE,
            "local": wl.SORT_LOCAL, "data": wl.SORT_DATA}
LOOPS = dict(binding.LOOP_NAMES)

# Mean track-steps of one primary in the Pb/LAr calorimeter by energy, and of
# a photon in the water cube; FP64 operations of one track-step (interpolated
# cross sections, distances, the interaction's kinematics, spread over steps).
STEP_E = [10.0, 30.0, 100.0, 300.0, 1000.0, 3000.0, 10000.0]
STEPS_ELECTRON = [37.0, 92.0, 187.0, 301.0, 451.0, 607.0, 802.0]
STEPS_PHOTON = 16.0
STEPS_WATER = 18.0
FLOPS_PER_STEP = 90.0


def transport(name, **kw):
    c = dict(name=name, kind="transport", world="calorimeter", bz=0.0, half=50.0, cap=0, source="electrons", e_min=1000.0,
             e_max=1000.0, patch=0.0, oblique=False, n=1000, events=1, slots=65536, policy="local", loop="async",
             entry="host", blocks=0, hits=0)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest request of an offloading application: one event of a
        # dozen particles, alone on the GPU (launches and chains of steps)
        transport("event_small", bz=4.0, source="mix", e_min=100.0, e_max=10000.0, patch=50.0, n=12, slots=1 << 18),
        # photon-only job in the plain step loop: no reordering, the whole
        # loop in one CUDA graph (the API's default loop and policy)
        transport("water_graph_none", world="water", source="photons", e_min=10.0, e_max=10.0, n=2000, slots=4096,
                  policy="none", loop="graph"),
        # the sampling calorimeter with the tracks sorted by action and
        # particle type before every step, in the persistent loop
        transport("calo_1gev_sorted", policy="action_type", loop="persistent"),
        # the same job in the asynchronous loop, the one a user picks for speed
        transport("calo_1gev_async"),
        # the full-size job of the benchmark: 10 GeV showers in 4 T, primaries
        # made on the device, asynchronous loop
        transport("field_10gev_async", bz=4.0, e_min=10000.0, e_max=10000.0, patch=5.0, n=10000, slots=1 << 20,
                  entry="device"),
        # the same job with the tracks partitioned by charge, persistent loop
        transport("field_10gev_data", bz=4.0, e_min=10000.0, e_max=10000.0, patch=5.0, n=10000, slots=1 << 20,
                  policy="data", loop="persistent", entry="device"),
        # a production-size batch in one array: ten times the full-size job
        transport("field_10gev_large", bz=4.0, e_min=10000.0, e_max=10000.0, patch=5.0, n=100000, slots=1 << 20,
                  entry="device"),
        # offloaded events of uneven size stepped together, each event's tally
        # returned to the host
        transport("offload_batch", bz=4.0, source="mix", e_min=100.0, e_max=10000.0, patch=50.0, n=200, events=64,
                  slots=1 << 20),
        # narrow world, oblique tracks leaving through the sides, Runge-Kutta
        # substeps with a cap: the field propagation options, ragged sizes
        transport("narrow_substeps", bz=4.0, half=2.0, cap=10, source="mix", e_min=20.0, e_max=2000.0, patch=1.5,
                  oblique=True, n=5003, slots=50001, policy="local", loop="persistent"),
        # one event of the event-per-stream mode: host-issued iterations on a
        # quarter of the GPU with a hit copy after each
        transport("event_host_loop", bz=4.0, source="mix", e_min=100.0, e_max=10000.0, patch=50.0, n=200, slots=1 << 16,
                  loop="host", blocks=38, hits=1),
        # a burst of requests served by continuous batching
        dict(name="serve_burst", kind="serve", n=200, events=32, slots=1 << 19, loop="async", chunk=8),
        # the key partition as a call of its own, at its largest
        dict(name="partition_full", kind="partition", n=1 << 20, keys=9, skip=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["async", "async", "async", "sync", "sync", "batch", "water", "narrow", "host", "serve", "partition"])
    energy = math.exp(rng.uniform(math.log(100.0), math.log(10000.0)))
    bz = rng.choice([0.0, 1.0, 3.8, 4.0])
    if kind == "async":
        n = _log_int(rng, 10, 60000)
        c = transport("", bz=bz, e_min=energy, e_max=energy, patch=5.0, n=n, policy=rng.choice(["local", "local", "data"]),
                      slots=_log_int(rng, 1 << 15, 1 << 20), entry=rng.choice(["host", "device"]))
    elif kind == "sync":
        c = transport("", bz=bz, e_min=energy, e_max=energy, patch=5.0, n=_log_int(rng, 10, 12000),
                      policy=rng.choice(sorted(POLICIES)), loop=rng.choice(["persistent", "graph"]),
                      slots=_log_int(rng, 1 << 15, 1 << 20))
    elif kind == "batch":
        c = transport("", bz=bz, source="mix", e_min=100.0, e_max=10000.0, patch=50.0, n=_log_int(rng, 20, 400),
                      events=_log_int(rng, 2, 100), slots=_log_int(rng, 1 << 18, 1 << 20))
    elif kind == "water":
        c = transport("", world="water", source="photons", e_min=energy / 100.0, e_max=energy / 100.0,
                      n=_log_int(rng, 50, 50000), slots=_log_int(rng, 1000, 1 << 17), policy=rng.choice(sorted(POLICIES)),
                      loop=rng.choice(["persistent", "graph", "host"]))
    elif kind == "narrow":
        c = transport("", bz=rng.choice([1.0, 4.0]), half=rng.uniform(1.0, 5.0), cap=rng.choice([0, 10, 1000]), source="mix",
                      e_min=20.0, e_max=2000.0, patch=0.9, oblique=True, n=_log_int(rng, 100, 10000),
                      slots=_log_int(rng, 1 << 13, 1 << 17), policy=rng.choice(["local", "data", "action_type"]),
                      loop="persistent")
    elif kind == "host":
        c = transport("", bz=bz, source="mix", e_min=100.0, e_max=10000.0, patch=50.0, n=_log_int(rng, 5, 500),
                      slots=_log_int(rng, 1 << 15, 1 << 18), policy=rng.choice(["local", "action"]), loop="host",
                      blocks=rng.choice([19, 38, 152]), hits=1)
    elif kind == "serve":
        return dict(kind="serve", n=_log_int(rng, 20, 400), events=_log_int(rng, 1, 48), slots=_log_int(rng, 1 << 17, 1 << 20),
                    loop=rng.choice(["async", "persistent"]), chunk=rng.choice([8, 16, 32]))
    else:
        keys = rng.randint(2, 16)
        return dict(kind="partition", n=_log_int(rng, 100, 1 << 20), keys=keys, skip=rng.choice([-1, keys - 1]))
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _event_sizes(case, rng):
    if case["events"] == 1:
        return [case["n"]]
    # lognormal sizes around n, as the offload mix has them, with the total kept
    w = rng.lognormal(0.0, 1.0, case["events"])
    sizes = np.maximum(1, np.floor(w * (case["n"] * case["events"] / w.sum()))).astype(int)
    return sizes.tolist()


def _primaries(case, seed):
    rng = np.random.default_rng([int(seed), case["n"]])
    events = []
    for e, n in enumerate(_event_sizes(case, rng)):
        energy = np.exp(rng.uniform(math.log(case["e_min"]), math.log(case["e_max"]), n)) if case["e_max"] > case["e_min"] \
            else np.full(n, case["e_min"])
        pos = np.zeros((n, 3))
        if case["patch"] > 0.0:
            pos[:, :2] = rng.uniform(-case["patch"], case["patch"], (n, 2))
        d = np.tile([0.0, 0.0, 1.0], (n, 1))
        if case["oblique"]:
            cost, phi = rng.uniform(0.3, 1.0, n), rng.uniform(0.0, 2.0 * math.pi, n)
            sint = np.sqrt(1.0 - cost * cost)
            d = np.stack([sint * np.cos(phi), sint * np.sin(phi), cost], 1)
            d /= np.linalg.norm(d, axis=1, keepdims=True)
        if case["source"] == "mix":
            ptype = np.where(rng.uniform(size=n) < 0.5, wl.GAMMA, wl.ELECTRON)
        else:
            ptype = np.full(n, wl.GAMMA if case["source"] == "photons" else wl.ELECTRON)
        events.append(wl.make_primaries(energy, pos, d, ptype.astype(np.int32), np.full(n, e, np.uint32)))
    return events


def _problem(case, seed):
    kw = dict(seed=int(seed) & 0x7FFFFFFF, max_events=case["events"], sort_policy=POLICIES[case["policy"]])
    if case["world"] == "water":
        return wl.water_cube_problem(case["slots"], init_capacity=max(4 * case["slots"], 4 * case["n"]), **kw)
    cap = max(8 * case["slots"], 16 * case["n"] * case["events"])
    return wl.calorimeter_problem(case["slots"], Bz=case["bz"], half_x=case["half"], half_y=case["half"],
                                  field_substep_cap=case["cap"], init_capacity=cap, **kw)


def _serve_as_transport(case):
    return transport("", bz=4.0, source="mix", e_min=100.0, e_max=10000.0, patch=50.0, n=case["n"], events=case["events"],
                     slots=case["slots"], loop=case["loop"])


def prepare(case, seed):
    if case["kind"] == "partition":
        g = torch.Generator(device="cuda").manual_seed(int(seed))
        # most slots vacant (the last key), live keys in runs of a few, as a
        # slot store looks between steps
        keys = torch.randint(0, case["keys"], (case["n"],), generator=g, device="cuda", dtype=torch.uint8)
        vacant = torch.rand((case["n"] + 31) // 32, generator=g, device="cuda") < 0.6
        keys[vacant.repeat_interleave(32)[: case["n"]]] = case["keys"] - 1
        return dict(kind="partition", keys=keys, n=case["n"], n_keys=case["keys"], skip=case["skip"],
                    perm=torch.zeros(case["n"], dtype=torch.int32, device="cuda"),
                    offsets=torch.zeros(case["keys"] + 1, dtype=torch.int32, device="cuda"))
    serve = case["kind"] == "serve"
    full = _serve_as_transport(case) if serve else case
    ctx = binding.Context(_problem(full, seed))
    events = _primaries(full, seed)
    s = dict(kind=case["kind"], ctx=ctx, mode=LOOPS[case["loop"]])
    if serve:
        s["requests"] = [(0.0, e, prim) for e, prim in enumerate(events)]
        s["chunk"] = case["chunk"]
        return s
    records = [binding.to_c_primaries(prim) for prim in events]
    s["n"] = [len(r) for r in records]
    s["device"] = case["entry"] == "device"
    s["records"] = [torch.from_numpy(r.view(np.uint8)).cuda() for r in records] if s["device"] else records
    if case["blocks"]:
        ctx.set_grid_blocks(case["blocks"])
    if case["hits"]:
        s["hits"] = torch.zeros(ctx.prob.max_events * ctx.n_bins, dtype=torch.float64).pin_memory()
        ctx.set_hit_readout(case["hits"], s["hits"])
    s["steps"] = ctx.stats()["steps_total"]
    return s


# ---------------------------------------------------------------- one pass
def run(state):
    if state["kind"] == "partition":
        binding.partition_keys_noalloc(state["keys"].data_ptr(), state["n"], state["n_keys"], state["skip"],
                                       state["perm"].data_ptr(), state["offsets"].data_ptr(),
                                       torch.cuda.current_stream().cuda_stream)
        return state["perm"], state["offsets"]
    ctx = state["ctx"]
    if state["kind"] == "serve":
        results, summary, tallies = ctx.serve(state["requests"], mode=state["mode"], chunk_iterations=state["chunk"],
                                              with_tallies=True)
        return tallies, results["escaped"], int(summary["track_steps"])
    for event, record in enumerate(state["records"]):
        ctx.reset_event(event)
        if state["device"]:
            ctx.add_primaries_device(event, record.data_ptr(), state["n"][event])
        else:
            ctx.add_primaries(event, record)
    ctx.run_events(state["mode"])
    rows = [ctx.read_tallies(event) for event in range(len(state["records"]))]
    total = ctx.stats()["steps_total"]
    steps, state["steps"] = total - state["steps"], total
    return np.stack([r[0] for r in rows]), np.array([r[1] for r in rows]), int(steps)


def work(case):
    if case["kind"] == "partition":
        return dict(bytes=5.0 * case["n"], flops=0.0)
    c = _serve_as_transport(case) if case["kind"] == "serve" else case
    if c["world"] == "water":
        steps, bins = STEPS_WATER, 100
    else:
        x = np.linspace(math.log(c["e_min"]), math.log(c["e_max"]), 9)
        e = float(np.mean(np.interp(x, np.log(STEP_E), STEPS_ELECTRON)))
        steps, bins = {"electrons": e, "photons": STEPS_PHOTON, "mix": 0.5 * (e + STEPS_PHOTON)}[c["source"]], 80
    n = c["n"] * c["events"]
    return dict(bytes=64.0 * n + 8.0 * (bins + 1) * c["events"], flops=FLOPS_PER_STEP * steps * n)


# -------------------------------------------------- the same in plain torch
# Every track of the job steps once per round, in 64-bit torch operations: the
# definitions of the transport (cross-section tables linear in ln E, straight
# lines or the helix, continuous loss by the inverse range table, the five
# interactions, Philox draws keyed by seed, event, track id and draw index).
ME = 0.51099895
RE = 2.8179403262e-13
FIELD_K = 2.99792458
GRID = 200
LN_EMIN = math.log(1e-3)
DL = math.log(1e4 / 1e-3) / (GRID - 1)
GAMMA, ELECTRON = 0, 1
NO_ACT, ZUP, ZDOWN, SIDE, RANGE, TRAPPED, INTERACT, FIELD = range(8)
INF = math.inf


def _kn(E):
    k = E / ME
    a = 1 + 2 * k
    L = np.log(a)
    return 2 * math.pi * RE**2 * ((1 + k) / k**2 * (2 * (1 + k) / a - L / k) + L / (2 * k) - (1 + 3 * k) / a**2)


def _moller(T, cut):
    T = np.maximum(T, 2 * cut * (1 + 1e-15))
    x, g = cut / T, T / ME + 1
    br = (g - 1) ** 2 / g**2 * (0.5 - x) + 1 / x - 1 / (1 - x) - (2 * g - 1) / g**2 * np.log((1 - x) / x)
    return 2 * math.pi * RE**2 / ((1 - 1 / g**2) * (g - 1)) * br


def _stopping(T, m, ne, cut_m, cut_b):
    tau = T / ME
    g2 = (tau + 1) ** 2
    b2 = tau * (tau + 2) / g2
    d = np.minimum(cut_m / ME, 0.5 * tau)
    F = -1 - b2 + np.log((tau - d) * d) + tau / (tau - d) + (0.5 * d * d + (2 * tau + 1) * np.log(1 - d / tau)) / g2
    col = 2 * math.pi * RE**2 * ME * ne / b2 * (np.log(2 * (tau + 2) / (m.I / ME) ** 2) + F)
    return col + np.minimum(T, cut_b) / m.X0


def _tables(p):
    gx, gw = np.polynomial.legendre.leggauss(16)
    out = np.zeros((len(p.materials), 6, GRID))
    lnE = LN_EMIN + np.arange(GRID) * DL
    E = np.exp(lnE)
    for i, m in enumerate(p.materials):
        ne = m.ne if m.ne > 0 else 6.02214076e23 * m.rho * m.Z / m.A
        zr = m.Z / 7.42
        on = lambda bit, v: v if p.processes & bit else np.zeros(GRID)  # noqa: E731
        out[i, 0] = on(wl.PROC_COMPTON, ne * _kn(E))
        out[i, 1] = on(wl.PROC_PHOTOELECTRIC, ne / 3.343e23 * zr**3 * 0.15 * (E / 0.030) ** -3.5)
        out[i, 2] = on(wl.PROC_PAIR, np.where(E > 1.022, ne / 3.343e23 * zr * 0.0096 * np.log(np.maximum(E, 1.022) / 1.022), 0.0))
        out[i, 3] = on(wl.PROC_MOLLER, np.where(E > 2 * p.cut_moller, ne * _moller(E, p.cut_moller), 0.0))
        out[i, 4] = on(wl.PROC_BREMS, np.where(E > p.cut_brems, np.log(np.maximum(E, p.cut_brems) / p.cut_brems) / m.X0, 0.0))
        if p.processes & wl.PROC_ELOSS:
            t = np.exp(lnE[:-1, None] + 0.5 * (1 + gx) * DL)
            seg = 0.5 * DL * (gw * t / _stopping(t, m, ne, p.cut_moller, p.cut_brems)).sum(1)
            out[i, 5, 0] = E[0] / (2 * _stopping(E[:1], m, ne, p.cut_moller, p.cut_brems)[0])
            out[i, 5, 1:] = out[i, 5, 0] + np.cumsum(seg)
    return out


class _Job:
    """One job's tracks as torch columns, and its tallies."""

    def __init__(self, p, events):
        self.p = p
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.f = lambda v: torch.tensor(np.asarray(v), dtype=torch.float64, device=self.dev)  # noqa: E731
        self.tab = self.f(_tables(p))
        thick = [0.0] + [p.layer_thickness[i % len(p.layer_thickness)] for i in range(p.n_layers_total)]
        self.zb = self.f(np.cumsum(thick))
        self.lmat = torch.tensor([p.layer_material[i % len(p.layer_material)] for i in range(p.n_layers_total)], device=self.dev)
        self.L = p.n_layers_total
        self.tally = torch.zeros(len(events), p.n_bins, dtype=torch.float64, device=self.dev)
        self.escaped = torch.zeros(len(events), dtype=torch.float64, device=self.dev)
        self.steps = 0
        q = np.concatenate(events)
        i64 = lambda v: torch.tensor(np.asarray(v, np.int64), device=self.dev)  # noqa: E731
        n = len(q)
        self.t = dict(E=self.f(q["E"]), x=self.f(q["pos"][:, 0]), y=self.f(q["pos"][:, 1]), z=self.f(q["pos"][:, 2]),
                      ux=self.f(q["dir"][:, 0]), uy=self.f(q["dir"][:, 1]), uz=self.f(q["dir"][:, 2]),
                      nmfp=self.f(np.full(n, -1.0)), ptype=i64(q["ptype"]), event=i64(q["event"]), layer=i64(np.zeros(n)),
                      tid=i64(np.concatenate([np.arange(len(e)) for e in events])), ctr=i64(np.zeros(n)))

    # ---- draws: key (seed, event), counter (track id, index / 2)
    def words(self, t, at):
        M = 0xFFFFFFFF
        tid, ctr = t["tid"][at], t["ctr"][at]
        c = [tid & M, (tid >> 32) & M, ctr >> 1, torch.zeros_like(ctr)]
        key0, key1 = torch.full_like(ctr, self.p.seed & M), t["event"][at] & M

        def mul(a, b):  # 32 x 32 bits -> high and low words
            lo = a * (b & 0xFFFF)
            hi = a * (b >> 16) + (lo >> 16)
            return hi >> 16, ((hi & 0xFFFF) << 16) | (lo & 0xFFFF)

        for _ in range(10):
            h0, l0 = mul(c[0], torch.full_like(ctr, 0xD2511F53))
            h1, l1 = mul(c[2], torch.full_like(ctr, 0xCD9E8D57))
            c = [h1 ^ c[1] ^ key0, l1, h0 ^ c[3] ^ key1, l0]
            key0, key1 = (key0 + 0x9E3779B9) & M, (key1 + 0xBB67AE85) & M
        odd = (ctr & 1) == 1
        lo, hi = torch.where(odd, c[2], c[0]), torch.where(odd, c[3], c[1])
        t["ctr"][at] = ctr + 1
        return hi, lo

    def uniform(self, t, at):
        hi, lo = self.words(t, at)
        return (((hi << 20) | (lo >> 12)).double() + 0.5) * 2.0**-52

    def raw(self, t, at):
        hi, lo = self.words(t, at)
        return (hi << 32) | lo

    # ---- tallies
    def deposit(self, event, layer, z, e):
        if self.p.tally_mode == wl.TALLY_LAYERS:
            b = layer
        else:
            span = self.zb[-1] - self.zb[0]
            b = torch.floor((z - self.zb[0]) * (self.p.n_bins / span)).long().clamp(0, self.p.n_bins - 1)
        self.tally.view(-1).index_add_(0, event * self.p.n_bins + b, e)

    def interp(self, mat, col, b, f):
        v = self.tab[mat, col, b]
        return v + f * (self.tab[mat, col, b + 1] - v)

    # ---- the helix
    def kappa(self, E):
        return -self.p.Bz * FIELD_K / torch.sqrt(E * (E + 2 * ME))

    def helix_side(self, k, x, y, ux, uy):
        hx, hy = self.p.half_x, self.p.half_y
        A = torch.sqrt(ux * ux + uy * uy)
        none = A == 0
        A = torch.where(none, 1.0, A)
        xc, yc, rho, sg = x + uy / k, y - ux / k, A / k.abs(), torch.sign(k)
        best = torch.full_like(x, INF)
        for plane, c, beta in ((hx, xc, torch.atan2(-uy, ux)), (-hx, xc, torch.atan2(-uy, ux)), (hy, yc, torch.atan2(ux, uy)),
                               (-hy, yc, torch.atan2(ux, uy))):
            d = k * (plane - c) / A
            a = torch.asin(d.clamp(-1, 1))
            for cand in (a, math.pi - a):
                turn = torch.fmod(sg * (cand - beta), 2 * math.pi)
                turn = torch.where(turn < 0, turn + 2 * math.pi, turn)
                best = torch.where((d.abs() <= 1) & (turn < best), turn, best)
        inside = (xc + rho < hx) & (xc - rho > -hx) & (yc + rho < hy) & (yc - rho > -hy)
        return torch.where(none | inside, INF, best / k.abs())

    def helix_move(self, t, k, s, n_rk):
        x, y, ux, uy = t["x"], t["y"], t["ux"], t["uy"]
        if self.p.field_substep_cap <= 0:
            hs, hc = torch.sin(0.5 * k * s), torch.cos(0.5 * k * s)
            sp, om = 2 * hs * hc, 2 * hs * hs
            return (x + (ux * sp + uy * om) / k, y + (uy * sp - ux * om) / k, ux * (1 - om) + uy * sp, uy * (1 - om) - ux * sp)
        h, X, Y, U, V = s / n_rk, x, y, ux, uy
        for i in range(int(n_rk.max())):
            on = i < n_rk
            k1 = (U, V, k * V, -k * U)
            u2, v2 = U + 0.5 * h * k1[2], V + 0.5 * h * k1[3]
            u3, v3 = U + 0.5 * h * (k * v2), V + 0.5 * h * (-k * u2)
            u4, v4 = U + h * (k * v3), V + h * (-k * u3)
            X = torch.where(on, X + h / 6 * (U + 2 * u2 + 2 * u3 + u4), X)
            Y = torch.where(on, Y + h / 6 * (V + 2 * v2 + 2 * v3 + v4), Y)
            du, dv = h / 6 * k * (V + 2 * v2 + 2 * v3 + v4), -h / 6 * k * (U + 2 * u2 + 2 * u3 + u4)
            U, V = torch.where(on, U + du, U), torch.where(on, V + dv, V)
        q = U * U + V * V
        f = torch.where(q > 0, torch.sqrt((ux * ux + uy * uy) / torch.where(q > 0, q, 1.0)), 1.0)
        return X, Y, U * f, V * f

    # ---- one step of every track
    def step(self):
        t, p, dev = self.t, self.p, self.dev
        n = len(t["E"])
        self.steps += n
        every = torch.arange(n, device=dev)
        at = every[t["nmfp"] < 0]
        t["nmfp"][at] = -torch.log(self.uniform(t, at))
        E, layer, ev = t["E"], t["layer"], t["event"]
        charged = t["ptype"] != GAMMA
        eloss = charged & bool(p.processes & wl.PROC_ELOSS)
        mat = self.lmat[layer]
        g = (torch.log(E) - LN_EMIN) * (1.0 / DL)
        b = torch.floor(g).long().clamp(0, GRID - 2)
        f = g - b
        mu = [torch.where(charged, self.interp(mat, 3, b, f), self.interp(mat, 0, b, f)),
              torch.where(charged, self.interp(mat, 4, b, f), self.interp(mat, 1, b, f)),
              torch.where(~charged & (E > 1.022), self.interp(mat, 2, b, f), 0.0)]
        tot = mu[0] + mu[1] + mu[2]
        s_int = torch.where(tot > 0, t["nmfp"] / torch.where(tot > 0, tot, 1.0), INF)
        R = self.interp(mat, 5, b, f)
        s_rng = torch.where(R <= 0.1, R, 0.2 * R + 0.08 * (2 - 0.1 / R.clamp(min=1e-300)))
        s_rng = torch.where(eloss, s_rng, INF)
        x, y, z, ux, uy, uz = (t[k] for k in ("x", "y", "z", "ux", "uy", "uz"))
        up, down = uz > 0, uz < 0
        plane = torch.where(up, self.zb[layer + 1], self.zb[layer])
        s = torch.where(up | down, (plane - z) / torch.where(uz == 0, 1.0, uz), INF)
        act = torch.where(up, ZUP, torch.where(down, ZDOWN, NO_ACT))
        far = lambda c, u, h: torch.where(u != 0, (torch.where(u > 0, h, -h) - c) / torch.where(u == 0, 1.0, u), INF)  # noqa: E731
        side = torch.minimum(far(x, ux, p.half_x), far(y, uy, p.half_y))
        k = None
        if p.Bz != 0.0:
            k = self.kappa(E)
            side = torch.where(charged, self.helix_side(k, x, y, ux, uy), side)
        act = torch.where(side < s, SIDE, act)
        s = torch.minimum(s, side).clamp(min=0.0)
        act = torch.where(s_rng < s, RANGE, act)
        s = torch.minimum(s, s_rng)
        act = torch.where(s_int < s, INTERACT, act)
        s = torch.minimum(s, s_int)
        act = torch.where(s == INF, TRAPPED, act)
        cap = p.field_substep_cap
        n_rk = None
        if k is not None and cap > 0:
            cut = charged & (act != TRAPPED) & (s * k.abs() > 0.1 * cap)
            s = torch.where(cut, 0.1 * cap / k.abs(), s)
            act = torch.where(cut, FIELD, act)
            n_rk = torch.where(cut, float(cap), torch.ceil(s * k.abs() / 0.1).clamp(1, cap + 1))
        trapped = act == TRAPPED
        s = torch.where(trapped, 0.0, s)
        t["nmfp"] = t["nmfp"] - s * tot

        # propagation and continuous loss
        nx, ny, nz, nux, nuy = x + s * ux, y + s * uy, z + s * uz, ux, uy
        if k is not None:
            c = self.helix_move(t, k, s, n_rk)
            nx, ny, nux, nuy = (torch.where(charged, a, d) for a, d in zip(c, (nx, ny, nux, nuy)))
        t["x"], t["y"], t["z"], t["ux"], t["uy"] = nx, ny, nz, nux, nuy
        at = every[eloss & ~trapped]
        if len(at):
            m, r = mat[at], (R - s)[at]
            tr = self.tab[:, 5]
            i = torch.zeros_like(at)
            for j in range(len(p.materials)):
                i = torch.where(m == j, torch.searchsorted(tr[j].contiguous(), r, right=True) - 1, i)
            stopped = r <= tr[m, 0]
            i = i.clamp(0, GRID - 2)
            lnE = LN_EMIN + i.double() * DL + (r - tr[m, i]) / (tr[m, i + 1] - tr[m, i]) * DL
            Ep = torch.where(stopped, 0.0, torch.exp(lnE))
            self.deposit(ev[at], layer[at], nz[at], E[at] - Ep)
            E = E.clone()
            E[at] = Ep
        # planes, escape, tracking cut
        layer = layer + (act == ZUP).long() - (act == ZDOWN).long()
        out = (act == SIDE) | (layer >= self.L) | (layer < 0)
        self.escaped.index_add_(0, ev[out], E[out])
        layer = layer.clamp(0, self.L - 1)
        cross = ((act == ZUP) | (act == ZDOWN)) & ~out
        # a crossing ends on the plane: the lower plane of the layer above, the upper plane of the layer below
        t["z"] = torch.where(cross, torch.where(act == ZUP, self.zb[layer], self.zb[layer + 1]), t["z"])
        t["layer"], t["E"] = layer, E
        low = ~out & ((E < p.cut_track) | trapped)
        self.deposit(ev[low], layer[low], t["z"][low], E[low])
        alive = ~out & ~low
        born = []

        # interactions
        at = every[alive & (act == INTERACT)]
        if len(at):
            target = self.uniform(t, at) * tot[at]
            m0, m1, m2 = (v[at] for v in mu)
            last = torch.where(m2 > 0, 2, torch.where(m1 > 0, 1, 0))
            sel = torch.where(target < m0, 0, torch.where(target < m0 + m1, 1, torch.where(target < m0 + m1 + m2, 2, last)))
            ch = charged[at]
            self.compton(at[~ch & (sel == 0)], alive)
            self.absorb(at[~ch & (sel == 1)], alive)
            born.append(self.pair(at[~ch & (sel == 2)], alive))
            born.append(self.moller(at[ch & (sel == 0)], alive))
            born.append(self.brems(at[ch & (sel == 1)], alive))
            t["nmfp"][at] = -1.0
        born = [c for c in born if c is not None]
        self.t = {key: torch.cat([t[key][alive]] + [c[key] for c in born]) for key in t}

    def end_low(self, at, alive):
        t = self.t
        at = at[t["E"][at] < self.p.cut_track]
        self.deposit(t["event"][at], t["layer"][at], t["z"][at], t["E"][at])
        alive[at] = False

    def rotated(self, t, at, cost, u_phi):
        ux, uy, uz = t["ux"][at], t["uy"][at], t["uz"][at]
        phi = 2 * math.pi * u_phi
        sint = torch.sqrt((1 - cost * cost).clamp(min=0.0))
        pole = uz.abs() >= 1.0 - 1e-10
        n1 = torch.sqrt(ux * ux + uy * uy)
        n1 = torch.where(pole, 1.0, n1)
        n2 = torch.sqrt(uz * uz + uy * uy)
        n2 = torch.where(n2 == 0, 1.0, n2)
        zero, one = torch.zeros_like(ux), torch.ones_like(ux)
        e1 = [torch.where(pole, a, c) for a, c in zip((one, zero, zero), (uy / n1, -ux / n1, zero))]
        e2 = [torch.where(pole, a, c) for a, c in zip((zero, uz / n2, -uy / n2), (uz * ux / n1, uz * uy / n1, -n1))]
        v = [cost * u + sint * (torch.cos(phi) * a + torch.sin(phi) * c) for u, a, c in zip((ux, uy, uz), e1, e2)]
        norm = torch.sqrt(v[0] ** 2 + v[1] ** 2 + v[2] ** 2)
        return [c / norm for c in v]

    def compton(self, at, alive):
        if not len(at):
            return
        t = self.t
        E = t["E"][at]
        k = E / ME
        e0 = 1 / (1 + 2 * k)
        a1, a2 = -torch.log(e0), 0.5 * (1 - e0 * e0)
        eps, todo = torch.ones_like(E), torch.arange(len(at), device=self.dev)
        while len(todo):
            u1, u2, u3 = (self.uniform(t, at[todo]) for _ in range(3))
            kk, ee, b1, b2 = k[todo], e0[todo], a1[todo], a2[todo]
            e = torch.where(u1 * (b1 + b2) < b1, torch.exp(-b1 * u2), torch.sqrt(ee * ee + (1 - ee * ee) * u2))
            c = (1 - e) / (kk * e)
            ok = u3 <= 1 - e * c * (2 - c) / (1 + e * e)
            eps[todo[ok]] = e[ok]
            todo = todo[~ok]
        cost = 1 - (1 - eps) / (k * eps)
        d = self.rotated(t, at, cost, self.uniform(t, at))
        self.deposit(t["event"][at], t["layer"][at], t["z"][at], E - eps * E)
        t["E"][at] = eps * E
        t["ux"][at], t["uy"][at], t["uz"][at] = d
        self.end_low(at, alive)

    def absorb(self, at, alive):
        t = self.t
        self.deposit(t["event"][at], t["layer"][at], t["z"][at], t["E"][at])
        alive[at] = False

    def child(self, at, ptype, E, d):
        """Secondaries of the tracks `at`; those below the cut are deposited and draw no id."""
        t = self.t
        low = E < self.p.cut_track
        self.deposit(t["event"][at][low], t["layer"][at][low], t["z"][at][low], E[low])
        keep, at = ~low, at[~low]
        c = {key: v[at].clone() for key, v in t.items()}
        c["tid"] = self.raw(t, at)
        c["E"], c["ux"], c["uy"], c["uz"] = E[keep], d[0][keep], d[1][keep], d[2][keep]
        c["nmfp"], c["ctr"], c["ptype"] = torch.full_like(c["E"], -1.0), torch.zeros_like(c["ctr"]), torch.full_like(c["ptype"], ptype)
        return c

    def pair(self, at, alive):
        if not len(at):
            return None
        t = self.t
        self.deposit(t["event"][at], t["layer"][at], t["z"][at], t["E"][at] - 2 * ME)
        cost = 2 * self.uniform(t, at) - 1
        phi = 2 * math.pi * self.uniform(t, at)
        sint = torch.sqrt((1 - cost * cost).clamp(min=0.0))
        d = [sint * torch.cos(phi), sint * torch.sin(phi), cost]
        e = torch.full_like(cost, ME)
        first, second = self.child(at, GAMMA, e, d), self.child(at, GAMMA, e, [-v for v in d])
        alive[at] = False
        return {key: torch.cat([first[key], second[key]]) for key in first}

    def moller(self, at, alive):
        cut = self.p.cut_moller
        at = at[self.t["E"][at] > 2 * cut]  # closed below: a null collision
        if not len(at):
            return None
        t = self.t
        T = t["E"][at]
        x, g = cut / T, T / ME + 1
        g2 = g * g
        norm = 4 / (9 * g2 - 10 * g + 5)
        eps, todo = torch.full_like(T, 0.5), torch.arange(len(at), device=self.dev)
        while len(todo):
            u1, u2 = self.uniform(t, at[todo]), self.uniform(t, at[todo])
            xx, gg, gg2 = x[todo], g[todo], g2[todo]
            e = xx / (1 - u1 * (1 - 2 * xx))
            om = 1 - e
            ok = u2 <= norm[todo] * ((gg - 1) ** 2 * e * e - (2 * gg2 + 2 * gg - 1) * e / om + gg2 / (om * om))
            eps[todo[ok]] = e[ok]
            todo = todo[~ok]
        Td = eps * T
        cost = torch.sqrt(Td * (T + 2 * ME) / (T * (Td + 2 * ME))).clamp(max=1.0)
        d = self.rotated(t, at, cost, self.uniform(t, at))
        pp, pd = torch.sqrt(T * (T + 2 * ME)), torch.sqrt(Td * (Td + 2 * ME))
        v = [pp * u - pd * c for u, c in zip((t["ux"][at], t["uy"][at], t["uz"][at]), d)]
        norm = torch.sqrt(v[0] ** 2 + v[1] ** 2 + v[2] ** 2)
        c = self.child(at, ELECTRON, Td, d)
        t["E"][at] = T - Td
        t["ux"][at], t["uy"][at], t["uz"][at] = [w / norm for w in v]
        self.end_low(at, alive)
        return c

    def brems(self, at, alive):
        cut = self.p.cut_brems
        at = at[self.t["E"][at] > cut]
        if not len(at):
            return None
        t = self.t
        T = t["E"][at]
        k = torch.minimum(cut * torch.exp(self.uniform(t, at) * torch.log(T / cut)), T)
        c = self.child(at, GAMMA, k, (t["ux"][at], t["uy"][at], t["uz"][at]))
        t["E"][at] = T - k
        self.end_low(at, alive)
        return c


def exact(case, seed):
    if case["kind"] == "partition":
        s = prepare(case, seed)
        keys = s["keys"].cpu().numpy()
        perm = np.zeros(case["n"], np.int32)
        order = np.argsort(keys, kind="stable").astype(np.int32)
        counts = np.bincount(keys, minlength=case["keys"])
        offsets = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
        end = offsets[-2] if case["skip"] == case["keys"] - 1 else offsets[-1]
        perm[:end] = order[:end]
        return perm, offsets
    c = _serve_as_transport(case) if case["kind"] == "serve" else case
    job = _Job(_problem(c, seed), _primaries(c, seed))
    while len(job.t["E"]):
        job.step()
    return job.tally.cpu().numpy(), job.escaped.cpu().numpy(), job.steps
