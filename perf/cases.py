"""What the speed of this framework is measured on: calls that a user's program makes, over the sizes it makes them at.

A case is one of
  push     PIC steps of one ensemble (qed_push_and_generate / qed_push_async), the framework's main path:
           photon emission in a fixed field, or a cascade of electrons, positrons and photons with global leveling
  batch    many independent ensembles through all their steps in one call (qed_batch_push)
  train    training of the surrogate sampler (qed_train_surrogate)
  context  a context with its rate and inverse-CDF tables, as every program makes at least one (qed_init_tables),
           then the rates and energy fractions at the program's own points (qed_eval_rate, qed_sample)

A pass puts the ensemble back to the state of `prepare` (a program that goes on would not; the copy is a few
percent), calls the framework, and hands all particles back.  Appended particles land in an order that differs
from run to run, so species that grow are handed back in the order of their ids, as a restart file holds them, in
arrays of a fixed length (the unused end is zero).
"""
import math

import numpy as np
import torch

import paper_2409_17299_gb300 as q
from paper_2409_17299_gb300 import workloads as W

COLUMNS = ("x", "y", "z", "px", "py", "pz", "w")
KINDS = {"uniform_b": W.FIELD_UNIFORM, "rotating_e": W.FIELD_ROTATING_E, "standing_cp": W.FIELD_STANDING_CP,
         "grid": W.FIELD_GRID}


def _push(name, field, precision, n, warm, steps, cap=0, strength=1000.0, period=100, calls="one",
          method="substep", sampler="table", photons=1, restore=0):
    c = {"kind": "push", "field": field, "precision": precision, "n": n, "warm": warm, "steps": steps, "cap": cap,
         "strength": strength, "period": period, "calls": calls, "method": method, "sampler": sampler,
         "photons": photons, "restore": restore}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one PIC step of a small bunch in a magnet, photons recorded; all latency and launches
        _push("emission_one_step", "uniform_b", "fp32", 1000, 0, 1, strength=1.0, period=200, photons=0, restore=1),
        # the benchmark's emission workload: 16384 electrons at chi = 1 in a uniform field, 200 steps, in FP64
        _push("emission_uniform_b", "uniform_b", "fp64", 16384, 0, 200, strength=1.0, period=200, photons=0, restore=1),
        # the start of the benchmark's cascade: 1e5 leptons, steps enqueued one by one, each a handful of small launches
        _push("cascade_growth", "rotating_e", "fp32", 100000, 5, 20, cap=50_000_000, calls="enqueue"),
        # the benchmark's headline: the cascade at its cap of 5e7 photons, leveled every step
        _push("cascade_at_cap", "rotating_e", "fp32", 100000, 280, 40, cap=50_000_000),
        # the paper's test problem in FP64 (standing wave, a0 = 1557, dt = T / 200), a quarter of its seeds and cap
        _push("test_problem_fp64", "standing_cp", "fp64", 62500, 500, 20, cap=500_000, strength=1557.0, period=200),
        # the standing-wave cascade at a twentieth of its size, all species at their cap: leptons dominate
        _push("standing_wave", "standing_cp", "fp32", 50000, 300, 40, cap=10_000_000, strength=2000.0),
        # the same wave given on the 128 x 4 x 4 grid of a PIC code that hands over new fields each step
        _push("standing_wave_grid", "grid", "fp32", 5000, 300, 20, cap=1_000_000, strength=2000.0, calls="each"),
        # the accumulated-optical-depth method that other PIC codes use, on the rotating-field cascade
        _push("optical_depth", "rotating_e", "fp32", 20000, 280, 40, cap=10_000_000, method="optical_depth"),
        # the cascade with photon energies drawn from the network
        _push("network_sampler", "rotating_e", "fp32", 20000, 280, 40, cap=10_000_000, sampler="network"),
        # 64 bunches of uneven size, each in its own field, through 50 steps in one call
        {"kind": "batch", "name": "batched_bunches", "precision": "fp32", "ensembles": 64, "size_lo": 250.0,
         "size_hi": 250000.0, "steps": 50},
        # the first stretch of training the network sampler
        {"kind": "train", "name": "train_network", "samples": 32 * 8192, "batch": 8192},
        # a context of its own and a scan of rates and energies with it
        {"kind": "context", "name": "context_tables", "precision": "fp64", "points": 100000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["emission", "growth", "cap", "cap", "fp64", "wave", "grid", "depth", "network", "batch",
                       "train", "context"])
    if kind == "emission":
        return _push("", "uniform_b", rng.choice(["fp32", "fp64"]), _log(rng, 500, 200000), 0, _log(rng, 1, 200),
                     strength=round(10.0 ** rng.uniform(-1, 0.5), 3), period=rng.choice([100, 200]), photons=0, restore=1)
    if kind == "growth":
        return _push("", "rotating_e", "fp32", _log(rng, 1000, 200000), rng.randint(0, 60), rng.randint(3, 25),
                     cap=50_000_000, calls=rng.choice(["one", "each", "enqueue"]), strength=rng.choice([800.0, 1000.0]))
    if kind in ("cap", "depth", "network"):
        cap = _log(rng, 500_000, 20_000_000)
        return _push("", "rotating_e", "fp32", max(500, cap // 500 + rng.randint(0, 99)), rng.randint(270, 300),
                     rng.randint(10, 40), cap=cap, calls=rng.choice(["one", "enqueue"]),
                     method="optical_depth" if kind == "depth" else "substep",
                     sampler="network" if kind == "network" else "table")
    if kind == "fp64":
        cap = _log(rng, 100_000, 600_000)
        return _push("", rng.choice(["standing_cp", "rotating_e"]), "fp64", cap // 8, rng.randint(150, 300),
                     rng.randint(5, 20), cap=cap, strength=1557.0, period=rng.choice([100, 200]))
    if kind in ("wave", "grid"):
        cap = _log(rng, 200_000, 10_000_000 if kind == "wave" else 2_000_000)
        return _push("", "standing_cp" if kind == "wave" else "grid", "fp32", cap // 200 + rng.randint(1, 99),
                     rng.randint(280, 400), rng.randint(10, 40), cap=cap, strength=2000.0,
                     calls="one" if kind == "wave" else "each")
    if kind == "batch":
        hi = _log(rng, 20_000, 250_000)
        return {"kind": "batch", "precision": "fp32", "ensembles": rng.randint(3, 64), "size_lo": hi / 1000.0,
                "size_hi": float(hi), "steps": rng.randint(10, 50)}
    if kind == "train":
        batch = 128 * rng.randint(8, 152)
        return {"kind": "train", "samples": batch * rng.randint(8, 32), "batch": batch}
    return {"kind": "context", "precision": rng.choice(["fp32", "fp64"]), "points": _log(rng, 1000, 1_000_000)}


# ---------------------------------------------------------------- inputs
def _precision(case):
    return q.QED_FP32 if case["precision"] == "fp32" else q.QED_FP64


def _ensemble(species, capacity, precision, optical_depth=False):
    """A DeviceEnsemble whose columns are rows of one array per species."""
    ens = q.DeviceEnsemble([0, 0, 0], precision, optical_depth=optical_depth)
    columns = COLUMNS + (("od",) if optical_depth else ())
    for s in range(3):
        cap = (max(int(capacity[s]), 1) + 3) // 4 * 4            # every row starts on 16 bytes
        room = cap + 4                                           # a place past the capacity stays zero
        rows = torch.zeros((len(columns), room), dtype=ens.fdtype, device="cuda")
        ens.arr[s] = {c: rows[i] for i, c in enumerate(columns)}
        ens.arr[s]["id"] = torch.zeros(room, dtype=torch.int64, device="cuda")
        ens.arr[s]["nevents"] = torch.zeros(room, dtype=torch.int32, device="cuda")
        ens.arr[s]["rows"] = rows
        ens.capacity[s] = cap
        n = len(species[s]["id"])
        if n:
            host = np.stack([np.asarray(species[s][c], dtype=np.float64) for c in COLUMNS])
            rows[:len(COLUMNS), :n].copy_(torch.from_numpy(host))
            ens.arr[s]["id"][:n].copy_(torch.from_numpy(species[s]["id"].view(np.int64)))
        ens.count[s] = n
    return ens


def _network(ctx, seed):
    """A network for the sampler: seeded hidden layers, the last layer fitted to the context's emission table."""
    em = np.zeros((121, 257))
    q.qed_get_tables(ctx, None, None, em.ctypes.data, None)
    r = np.random.default_rng(seed)
    w1, b1 = r.normal(0, 2.0, (64, 2)), r.normal(0, 1.0, 64)
    w2, b2 = r.normal(0, 0.25, (64, 64)), r.normal(0, 0.3, 64)
    w3, b3 = r.normal(0, 0.25, (64, 64)), r.normal(0, 0.3, 64)
    i, j = r.integers(0, 121, 6000), r.integers(8, 249, 6000)
    f = np.stack([(i / 20.0 - 3.0) / 3.0, (j / 8.0 - 16.0) / 16.0])
    silu = lambda z: z / (1.0 + np.exp(-z))  # noqa: E731
    h = silu(w3 @ silu(w2 @ silu(w1 @ f + b1[:, None]) + b2[:, None]) + b3[:, None])
    a = np.vstack([h, np.ones(h.shape[1])])
    gram = a @ a.T + 1e-3 * h.shape[1] * np.eye(65)              # ridge: coefficients of moderate size
    last = np.linalg.solve(gram, a @ (em[i, j] / 16.0 + 0.5))
    return np.concatenate([w1.ravel(), b1, w2.ravel(), b2, w3.ravel(), b3, last]).astype(np.float32)


def _workload(case, seed):
    n, period = case["n"], case["period"]
    if case["field"] == "uniform_b":
        return W.uniform_b_emission(n=n, seed=seed, chi0=case["strength"], steps_per_period=period, nsteps=case["steps"])
    if case["field"] == "rotating_e":
        return W.rotating_e_cascade(n=n, seed=seed, a0=case["strength"], steps_per_period=period)
    if case["period"] == 200:
        return W.paper_test_problem(n=n, seed=seed, a0=case["strength"])
    make = W.standing_wave_grid if case["field"] == "grid" else W.standing_wave_cascade
    return make(n=n, seed=seed, a0=case["strength"], steps_per_period=period)


def _emissions(chi, gamma, dt, steps):
    """At most how often a lepton emits in these steps (the classical rate)."""
    return W.R_SCHWINGER / 137.036 / gamma * 5.0 / (2.0 * math.sqrt(3.0)) * chi * dt * steps


def _room(case):
    """Places for each species in what is handed back: more than any seed's particles take."""
    n, cap, t = case["n"], case["cap"], case["warm"] + case["steps"]
    if not case["photons"]:
        dt = 2.0 * math.pi / case["period"]
        return n, 0, int(1.1 * n * _emissions(case["strength"], 1000.0, dt, case["steps"])) + 2048
    full = cap + 10 * int(math.sqrt(cap)) + 64                   # leveling leaves the cap, give or take a few sigma
    if cap > 200 * n and t < 120:                                # the start of a cascade
        lepton, photon = n * (1.3 + 0.0005 * t * t), n * (2.0 + 0.1 * t ** 1.45)
    elif case["field"] == "rotating_e" and case["precision"] == "fp32":
        lepton, photon = 0.2 * cap, full
    else:
        lepton, photon = full, full
    return min(full, int(lepton)), min(full, int(lepton)), min(full, int(photon))


def _prepare_push(case, seed):
    w = _workload(case, seed)
    precision, cap = _precision(case), case["cap"]
    config = q.make_config(precision=precision, seed=seed, push_photons=case["photons"], thin_cap=cap,
                           restore_on_overflow=case["restore"],
                           event_method=q.QED_METHOD_OPTICAL_DEPTH if case["method"] == "optical_depth" else q.QED_METHOD_SUBSTEP,
                           sampler=q.QED_SAMPLER_MLP if case["sampler"] == "network" else q.QED_SAMPLER_TABLE)
    gen = q.Generator(config)
    if case["sampler"] == "network":
        q.qed_mlp_set_params(gen.ctx, _network(gen.ctx, seed))
    n = case["n"]
    room = _room(case)
    if cap:                                                      # and what one step emits
        burst = 3.0 if case["field"] in ("standing_cp", "grid") else 1.6
        capacity = [int(1.6 * room[0]) + 4 * n, int(1.6 * room[1]) + 4 * n, int(burst * room[2]) + 4 * n]
    else:
        capacity = room
    ens = _ensemble(w.species, capacity, precision, case["method"] == "optical_depth")
    grids = None
    if case["field"] == "grid":                                  # the fields of each step, as a PIC code holds them
        nx, ny, nz = W.GRID_SHAPE
        t = torch.arange(case["warm"] + case["steps"], device="cuda", dtype=torch.float64) * w.dt
        x = torch.arange(nx, device="cuda", dtype=torch.float64) * (W.TWO_PI / nx)
        e, b = case["strength"] * torch.cos(x), case["strength"] * torch.sin(x)
        zero = torch.zeros(len(t), nx, device="cuda", dtype=torch.float64)
        g = torch.stack([zero, torch.outer(torch.cos(t), e), torch.outer(torch.sin(t), e),
                         zero, torch.outer(torch.cos(t), b), torch.outer(torch.sin(t), b)], 1)
        grids = g[:, :, None, None, :].expand(-1, -1, nz, ny, -1).to(ens.fdtype).contiguous()
    state = {"case": case, "gen": gen, "ens": ens, "field": q.make_field(KINDS[case["field"]], w.field_prm),
             "dt": w.dt, "grids": grids}
    if case["warm"]:
        _advance(state, 0, case["warm"], "each" if grids is not None else "one")
    state["count"] = list(ens.count)
    state["init"] = [[ens.arr[s][k][..., :ens.count[s]].clone() for k in ("rows", "id", "nevents")] for s in range(3)]
    state["index"] = [torch.full((m,), ens.capacity[s], device="cuda") for s, m in enumerate(room)]
    return state


def _advance(state, step0, steps, calls):
    gen, ens, field, dt = state["gen"], state["ens"], state["field"], state["dt"]
    if calls == "one":
        gen.push(ens, field, dt, steps, step0, auto_grow=False)
    elif calls == "each":                                        # a PIC loop: the counts are needed after every step
        for k in range(step0, step0 + steps):
            if state["grids"] is not None:
                q.qed_set_field_grid(gen.ctx, state["grids"][k].data_ptr())
            gen.push(ens, field, dt, 1, k, auto_grow=False)
    else:                                                        # steps enqueued one by one, one wait
        for k in range(step0, step0 + steps):
            gen.push_async(ens, field, dt, 1, k)
        gen.wait(ens)


def _prepare_batch(case, seed):
    ws = W.batched_uniform_b(n_ens=case["ensembles"], seed=2, size_lo=case["size_lo"], size_hi=case["size_hi"],
                             nsteps=case["steps"])
    precision = _precision(case)
    gen = q.Generator(q.make_config(precision=precision, seed=seed, push_photons=0))
    dtype = torch.float32 if precision == q.QED_FP32 else torch.float64
    arr, fields = (q.QedParticles * len(ws))(), (q.QedFieldDesc * len(ws))()
    for i, w in enumerate(ws):
        fields[i] = q.make_field(w.field_kind, w.field_prm)
    state = {"case": case, "gen": gen, "arr": arr, "fields": fields, "dt": ws[0].dt, "rows": [0] * 3, "ids": [0] * 3,
             "events": [0] * 3}

    def allocate(s, sizes):                                      # one species of all ensembles, side by side
        m = sum(sizes)
        state["rows"][s] = torch.zeros((7, m), dtype=dtype, device="cuda")
        state["ids"][s] = torch.zeros(m, dtype=torch.int64, device="cuda")
        state["events"][s] = torch.zeros(m, dtype=torch.int32, device="cuda")
        at = 0
        for i, cap in enumerate(sizes):
            S = arr[i].s[s]
            for c, name in enumerate(COLUMNS):
                setattr(S, name, state["rows"][s][c, at:].data_ptr())
            S.id, S.nevents = state["ids"][s][at:].data_ptr(), state["events"][s][at:].data_ptr()
            S.count, S.capacity = 0, cap
            at += cap

    allocate(0, [(int(w.notes["n"]) + 3) // 4 * 4 for w in ws])
    at = 0
    for i, w in enumerate(ws):
        e, n = w.species[0], int(w.notes["n"])
        state["rows"][0][:, at:at + n].copy_(torch.from_numpy(np.stack([e[c] for c in COLUMNS])))
        state["ids"][0][at:at + n].copy_(torch.from_numpy(e["id"].view(np.int64)))
        arr[i].s[0].count = n
        at += arr[i].s[0].capacity
    state["init"] = state["rows"][0].clone()
    sizes = [w.notes["n"] * _emissions(w.notes["chi0"], 2000.0, w.dt, case["steps"]) / 4 + 4096 for w in ws]
    # the bunches: an energy spread of one percent, and ids of their own
    r = torch.Generator(device="cuda").manual_seed(seed)
    state["init"][3] *= 1.0 + 0.01 * torch.randn(len(state["ids"][0]), generator=r, device="cuda", dtype=dtype).clamp_(-3, 3)
    state["ids"][0] += (seed & 0xFFFF) << 32
    need = None
    while need is None:                                          # sizing passes, as for any recorded photons
        allocate(2, [int(m) // 4 * 4 for m in sizes])
        need = _push_batch(state)
        sizes = [2 * m for m in sizes]
    allocate(2, [(int(1.25 * m) + 8192) // 4 * 4 for m in need])
    return state


def _push_batch(state):
    arr = state["arr"]
    state["rows"][0].copy_(state["init"])
    state["events"][0].zero_()
    for i in range(len(arr)):
        arr[i].s[2].count = 0
    rc, _ = q.qed_batch_push(state["gen"].ctx, arr, state["fields"], state["dt"], state["case"]["steps"], 0)
    if rc != q.QED_OK:
        return None                                              # the photons need more room
    return np.array([arr[i].s[2].count for i in range(len(arr))])


def prepare(case, seed):
    if case["kind"] == "push":
        return _prepare_push(case, seed)
    if case["kind"] == "batch":
        return _prepare_batch(case, seed)
    if case["kind"] == "train":
        gen = q.Generator(q.make_config(precision=q.QED_FP32, seed=seed, sampler=q.QED_SAMPLER_MLP))
        return {"case": case, "gen": gen, "seed": seed}
    r = torch.Generator(device="cuda").manual_seed(seed)
    n = case["points"]
    chi = 10.0 ** (torch.rand(n, generator=r, device="cuda", dtype=torch.float64) * 5.0 - 2.0)
    u = torch.rand(n, generator=r, device="cuda", dtype=torch.float64).clamp_(1e-12, 1.0 - 1e-12)
    return {"case": case, "seed": seed, "chi": chi, "u": u}


# ---------------------------------------------------------------- one pass
def _in_order(rows, ids, events, n, index):
    """The first n particles in the order of their ids; index holds the place of a zero past n."""
    index[:n] = torch.argsort(ids[:n])
    return {"rows": rows.index_select(1, index), "id": ids[index], "nevents": events[index]}


def run(state):
    case = state["case"]
    if case["kind"] == "push":
        ens, gen = state["ens"], state["gen"]
        for s in range(3):
            n = state["count"][s]
            if n:
                for k, v in zip(("rows", "id", "nevents"), state["init"][s]):
                    ens.arr[s][k][..., :n].copy_(v)
            ens.count[s] = n
        _advance(state, case["warm"], case["steps"], case["calls"])
        out = {}
        for s in range(3):
            d, n = ens.arr[s], ens.count[s]
            if not case["photons"] and s < 2:                    # leptons stay in their places
                if n:
                    out[W.SPECIES[s]] = {"rows": d["rows"][:, :n], "id": d["id"][:n], "nevents": d["nevents"][:n]}
            else:
                out[W.SPECIES[s]] = _in_order(d["rows"], d["id"], d["nevents"], n, state["index"][s])
        return out
    if case["kind"] == "batch":
        # the bunches as they leave, and how many photons they gave (which stay in the recorder's arrays: a tile of
        # two bunches shares them out differently from run to run)
        photons = int(_push_batch(state).sum())
        return {"electron": {"rows": state["rows"][0], "id": state["ids"][0], "nevents": state["events"][0]},
                "photons": photons}
    if case["kind"] == "train":
        ctx = state["gen"].ctx
        loss = q.qed_train_surrogate(ctx, case["samples"], case["batch"], 4e-3, state["seed"])
        return {"parameters": q.qed_mlp_get_params(ctx), "loss": loss}
    ctx = q.qed_init_tables(q.make_config(precision=_precision(case), seed=state["seed"]),
                            torch.cuda.current_stream().cuda_stream)
    cheb_em, cheb_pair = np.zeros((6, 11)), np.zeros((5, 11))
    icdf_em, icdf_pair = np.zeros((121, 257)), np.zeros((101, 129))
    q.qed_get_tables(ctx, *(a.ctypes.data for a in (cheb_em, cheb_pair, icdf_em, icdf_pair)))
    chi, u = state["chi"], state["u"]
    n = len(chi)
    out = {"cheb_em": cheb_em, "cheb_pair": cheb_pair, "icdf_em": icdf_em, "icdf_pair": icdf_pair}
    for photon, name in ((False, "emission"), (True, "pair")):
        rate, delta, rest = (torch.empty_like(chi) for _ in range(3))
        q.qed_eval_rate(ctx, photon, chi.data_ptr(), n, rate.data_ptr())
        q.qed_sample(ctx, photon, chi.data_ptr(), u.data_ptr(), n, delta.data_ptr(), rest.data_ptr())
        out[name] = {"rate": rate, "delta": delta, "rest": rest}
    q.qed_destroy(ctx)
    return out


# ---------------------------------------------------------------- what a pass cannot do without
def _population(case):
    """About how many leptons and photons are pushed per step."""
    n, cap, t = case["n"], case["cap"], case["warm"] + 0.5 * case["steps"]
    if not case["photons"]:
        return n, 0.0
    if cap > 200 * n and t < 120:                                # the start of a cascade
        return 1.05 * n, 0.05 * n * t ** 1.45
    if case["field"] == "rotating_e":
        return (0.23 * cap if n < cap // 100 else min(2.0, 0.1 + 0.0036 * t) * cap), cap
    return (min(2.0, 0.15 + 0.00165 * t) * cap if case["period"] == 200 else 2.0 * cap), cap


def work(case):
    """Bytes: every particle read and written once a step where leveling couples the particles of a step, once a
    call where nothing does; appended particles written once.  Operations: as counted on the FP64 passes."""
    kind = case["kind"]
    if kind == "train":
        return {"bytes": 8 * 8577, "flops": 49920 * case["samples"]}
    if kind == "context":
        nodes = 121 * 257 + 101 * 129                            # each the root of a 16-point panel
        return {"bytes": 8 * (nodes + 121) + 8 * 8 * case["points"], "flops": nodes * 16 * 200 + 200 * case["points"]}
    e = 4 if case["precision"] == "fp32" else 8
    lepton, photon, record = 13 * e + 8, 10 * e + 8, 7 * e + 12
    if kind == "batch":
        lo, hi, steps = case["size_lo"], case["size_hi"], case["steps"]
        n = case["ensembles"] * (hi - lo) / math.log(hi / lo)
        chi = [1e-2 * 1e4 ** ((i + 0.5) / 20) for i in range(20)]
        events = n * sum(_emissions(c, 2000.0, 2.0 * math.pi / 100, steps) for c in chi) / 20
        return {"bytes": n * (lepton + 4) + events * record, "flops": 480 * n * steps + 300 * events}          # events: the classical rate, energy loss left out
    leptons, photons = _population(case)
    steps = case["steps"]
    if not case["photons"]:
        events = leptons * _emissions(case["strength"], 1000.0, 2.0 * math.pi / case["period"], steps)
        return {"bytes": leptons * (lepton + 4) + events * record, "flops": 480 * leptons * steps + 300 * events}
    od = 2 * e if case["method"] == "optical_depth" else 0
    flops = 480 * leptons + 193 * photons + (2 * 8384 * 0.3 * leptons if case["sampler"] == "network" else 0)
    return {"bytes": steps * (leptons * (lepton + od + 0.3 * record) + photons * (photon + od)), "flops": steps * flops}


# ---------------------------------------------------------------- the same in 64 bits, in plain torch
def _bessel(y):
    """K_2/3(y) and the integral of K_1/3 from y on, by the trapezoid rule on their integral representations."""
    k23, k13 = torch.empty_like(y), torch.empty_like(y)
    j = torch.arange(1200, device=y.device, dtype=y.dtype)
    weight = torch.where(j == 0, 0.5, 1.0)
    for a in range(0, len(y), 1 << 15):
        v = y[a:a + (1 << 15), None]
        h = torch.clamp(0.4 / torch.sqrt(v), max=0.1)
        t = j * h
        f = torch.exp(-v * torch.cosh(t)) * weight * h
        k23[a:a + (1 << 15)] = (f * torch.cosh(t * (2.0 / 3.0))).sum(1)
        k13[a:a + (1 << 15)] = (f * torch.cosh(t * (1.0 / 3.0)) / torch.cosh(t)).sum(1)
    return k23, k13


def _density(pair, z, chi):
    """The LCFA spectrum in z: emission z = ln y, y = 2 d / (3 chi (1 - d)); pairs d = 1 / (1 + e^-z)."""
    if pair:
        d, rest = 1.0 / (1.0 + torch.exp(-z)), 1.0 / (1.0 + torch.exp(z))
        y, jacobian, sign = 2.0 / (3.0 * chi * d * rest), d * rest, 1.0
    else:
        y = torch.exp(z)
        a = 3.0 * chi * y
        d, rest, sign = a / (2.0 + a), 2.0 / (2.0 + a), -1.0
        jacobian = y * 6.0 * chi / (2.0 + a) ** 2
    shape = torch.broadcast_shapes(z.shape, chi.shape)
    k23, k13 = (v.reshape(shape) for v in _bessel(y.expand(shape).reshape(-1)))
    first = (d / rest + rest / d) if pair else (rest + 1.0 / rest)
    return (first * k23 + sign * k13) * jacobian


def _panels(pair, chi):
    """Edges of the panels in z, and the spectrum's integral over each for every chi."""
    x, w = (torch.from_numpy(v).cuda() for v in np.polynomial.legendre.leggauss(16))
    lo, width, count = (-38.0, 0.1, 380) if pair else (-110.0, 0.25, 472)
    edges = lo + width * torch.arange(count + 1, device="cuda", dtype=torch.float64)
    z = edges[:-1, None] + 0.5 * width * (x + 1.0)
    mass = torch.stack([(_density(pair, z, c.reshape(1, 1)) * w).sum(1) * 0.5 * width for c in chi])
    tail = torch.zeros_like(chi) if pair else 3.0 * _density(False, edges[:1].expand(len(chi)), chi)
    return x, w, edges, mass, tail


def _exact_tables():
    out = []
    for pair in (False, True):
        lo, decades, rows, columns = (-2.0, 5, 101, 129) if pair else (-3.0, 6, 121, 257)
        node = math.pi * (torch.arange(11, device="cuda", dtype=torch.float64) + 0.5) / 11
        chi = 10.0 ** (lo + torch.arange(decades, device="cuda", dtype=torch.float64)[:, None] + 0.5 + 0.5 * torch.cos(node))
        _, _, _, mass, tail = _panels(pair, chi.reshape(-1))
        rate = ((mass.sum(1) + tail) * (2.0 if pair else 1.0) / (math.sqrt(3.0) * math.pi)).reshape(chi.shape)
        f = torch.log(rate) + 8.0 / (3.0 * chi) if pair else rate / chi
        dct = torch.cos(torch.arange(11, device="cuda", dtype=torch.float64)[:, None] * node)
        coefficients = 2.0 / 11 * f @ dct.T

        chi = 10.0 ** (lo + torch.arange(rows, device="cuda", dtype=torch.float64) / 20)
        x, w, edges, mass, tail = _panels(pair, chi)
        s = torch.linspace(-16.0, 0.0 if pair else 16.0, columns, device="cuda", dtype=torch.float64).expand(rows, -1)
        below = torch.cat([tail[:, None], tail[:, None] + torch.cumsum(mass, 1)], 1)
        above = torch.cat([torch.flip(torch.cumsum(torch.flip(mass, [1]), 1), [1]), torch.zeros_like(tail)[:, None]], 1)
        total = (below[:, -1] * (2.0 if pair else 1.0))[:, None]
        low, high = total / (1.0 + torch.exp(-s)), total / (1.0 + torch.exp(s))
        up = s <= 0                                              # from the nearer end, so that both tails stay exact
        p = torch.where(up, torch.searchsorted(below[:, 1:].contiguous(), low.contiguous()),
                        mass.shape[1] - 1 - torch.searchsorted(torch.flip(above[:, :-1], [1]).contiguous(), high.contiguous()))
        p = p.clamp(0, mass.shape[1] - 1)
        za, zb = edges[p], edges[p + 1]
        goal = torch.where(up, low - torch.gather(below, 1, p), torch.gather(mass, 1, p) - (high - torch.gather(above, 1, p + 1)))
        z, c = 0.5 * (za + zb), chi[:, None].expand_as(za)
        for _ in range(9):                                       # Newton's method inside the panel
            nodes = za[..., None] + (z - za)[..., None] * 0.5 * (x + 1.0)
            integral = (_density(pair, nodes, c[..., None]) * w).sum(-1) * 0.5 * (z - za)
            z = torch.minimum(torch.maximum(z - (integral - goal) / _density(pair, z, c), za + 1e-3 * (z - za)), zb)
        z = torch.where(low <= tail[:, None], edges[0] + 3.0 * torch.log(low / tail[:, None].clamp(min=1e-300)), z)
        out += [coefficients, -torch.log1p(torch.exp(-z)) if pair else z]
    return out


def _exact_rate(pair, coefficients, chi):
    lo, decades = (-2.0, 5) if pair else (-3.0, 6)
    s = torch.log10(chi)
    d = torch.clamp(torch.floor(s - lo).long(), 0, decades - 1)
    x = 2.0 * (s - lo - d) - 1.0
    k = torch.arange(11, device="cuda", dtype=torch.float64)
    terms = torch.cos(k * torch.arccos(x.clamp(-1.0, 1.0))[:, None]) * coefficients[d]
    f = terms.sum(1) - 0.5 * coefficients[d][:, 0]
    return torch.where(chi >= 0.01, torch.exp(f - 8.0 / (3.0 * chi)), 0.0) if pair else chi * f


def _exact_sample(pair, table, chi, u):
    s = torch.log(u) - torch.log1p(-u)
    if pair:
        s = -s.abs()
    rows, columns = table.shape
    c = ((torch.log10(chi) + (2.0 if pair else 3.0)) * 20.0).clamp(0.0, rows - 1.0)
    t = (s + 16.0) * 8.0
    i, j = c.long().clamp(0, rows - 2), torch.floor(t).long().clamp(0, columns - 2)
    a, b = c - i, t - j
    v = (1 - a) * ((1 - b) * table[i, j] + b * table[i, j + 1]) + a * ((1 - b) * table[i + 1, j] + b * table[i + 1, j + 1])
    if pair:
        d = torch.exp(v)
        return torch.where(u > 0.5, 1.0 - d, d), torch.where(u > 0.5, d, 1.0 - d)
    y = 3.0 * chi * torch.exp(v)
    return y / (2.0 + y), 2.0 / (2.0 + y)


def exact(case, seed):
    """Only the tables and what is read from them: the other outputs are histories of random draws, or of thousands
    of rounded updates."""
    if case["kind"] != "context":
        return None
    r = torch.Generator(device="cuda").manual_seed(seed)
    n = case["points"]
    chi = 10.0 ** (torch.rand(n, generator=r, device="cuda", dtype=torch.float64) * 5.0 - 2.0)
    u = torch.rand(n, generator=r, device="cuda", dtype=torch.float64).clamp_(1e-12, 1.0 - 1e-12)
    cheb_em, icdf_em, cheb_pair, icdf_pair = _exact_tables()
    out = {"cheb_em": cheb_em, "cheb_pair": cheb_pair, "icdf_em": icdf_em, "icdf_pair": icdf_pair}
    for pair, name, cheb, icdf in ((False, "emission", cheb_em, icdf_em), (True, "pair", cheb_pair, icdf_pair)):
        delta, rest = _exact_sample(pair, icdf, chi, u)
        out[name] = {"rate": _exact_rate(pair, cheb, chi), "delta": delta, "rest": rest}
    return out
