"""The work that users of this framework have it do, as cases to be timed.

A case is a dict of plain values; prepare(case, seed) builds what a user's
program holds before the call (discharges loaded on the GPU, a captured batch,
a network, particle arrays), run(state) makes one pass through the public
entry points, and work(case) says what a pass cannot do without.

Kinds of case:
  step     Discharge.step on the library's own stream, then the state read back
  graph    the same discharge as a Batch of one (one CUDA graph per launch)
  sweep    several discharges in one Batch
  reload   host particles loaded, a stretch of steps, particles read to the host
  forward, gradients, train    the warm-start network
  compact  stable removal of dead particles from a caller's arrays
"""
import math

import numpy as np
import torch

from paper_0705_0497_gb300 import api, inputs, xsec

N0 = 1.0e15                  # m^-3, the density that the workloads are loaded at
BYTES_PER_PUSH = 16          # x and v_x, read and written, for each particle pushed
FLOPS_PER_PUSH = 24          # gather, leapfrog, deposit
HIDDEN = 256


def listed():
    return [
        # The network asked for the profiles of 32 new discharges (the warm
        # start's held-out set): a few launches, the smallest call.
        dict(name="mlp_forward_32", kind="forward", rows=32, hidden=HIDDEN, outputs=864),
        # Training as the warm start does it: full batch (81 converged runs),
        # 25 Adam steps, then the parameters for a checkpoint.
        dict(name="mlp_train_81", kind="train", rows=81, hidden=HIDDEN, outputs=864, steps=25),
        # The gradient over the training set that the batched sweep is meant
        # to give (2000 runs): the network's large contraction.
        dict(name="mlp_gradients_2000", kind="gradients", rows=2000, hidden=HIDDEN, outputs=864),
        # Removal of the absorbed and consumed particles from a caller's own
        # arrays, ragged length, a few per cent dead.
        dict(name="compact_20m", kind="compact", n=20_000_003, dead=0.05, noalloc=True),
        # The small discharge of the parity tests, one RF cycle launch by
        # launch: 2e4 particles, so launches and latency count.  (Counts as
        # the discharge has them after its first cycles.)
        dict(name="step_128", kind="step", cells=128, L=0.02, U=200.0, p=10.0, C=0.05, S=1, spc=400, weight=2.0e9,
             ne=3600, nm=1700, np=6900, cap=8.0, cap_extra=65536, steps=400, settle=400, caps=False, rec=False,
             edet=False, coulomb=0),
        # Every reaction of Table 1 on: Coulomb collisions (1)-(6), (16), (17)
        # and (22), launch by launch, an odd number of cells.
        dict(name="step_table1_301", kind="step", cells=301, L=0.025, U=250.0, p=13.8, C=1.0 / 6.0, S=5, spc=1000,
             weight=N0 * 0.025 / 400_000, ne=400_000, nm=400_000, np=800_000, cap=2.0, cap_extra=1 << 20, steps=100,
             settle=100, caps=False, rec=True, edet=True, coulomb=63),
        # The benchmark's discharge at its periodic state (512 cells, ions
        # every tenth step), one RF cycle as a replay of its step graph.
        dict(name="graph_512", kind="graph", cells=512, L=0.025, U=300.0, p=20.0, C=0.05, S=10, spc=1000,
             weight=6.25e6, ne=1_400_000, nm=3_730_000, np=5_700_000, cap=1.7, cap_extra=1 << 22, steps=1000,
             launch=1000, settle=4000, caps=True, rec=False, edet=False, coulomb=0),
        # The largest discharge (2048 cells, ions pushed every step): the
        # particle arrays stream from HBM.
        dict(name="graph_2048", kind="graph", cells=2048, L=0.03, U=500.0, p=50.0, C=0.10, S=1, spc=2000,
             weight=1.0e6, ne=52_000_000, nm=30_000_000, np=93_000_000, cap=1.5, cap_extra=1 << 22, steps=20,
             launch=20, settle=60, caps=True, rec=False, edet=False, coulomb=0),
        # The paper's discharge without and with metastables, the two in one
        # batch as the demonstration runs them.
        dict(name="sweep_paper_2", kind="sweep", n=2, cells=256, U_lo=250.0, U_hi=250.0, p_lo=13.8, p_hi=13.8,
             C_lo=0.0, C_hi=1.0 / 6.0, N_lo=100_000, N_hi=100_000, S=10, launch=200, steps=1000, settle=0, cap=6.0,
             cap_extra=1 << 20, tune=True, check=20),
        # The warm start's held-out discharges in one batch: equal, small
        # particle numbers.
        dict(name="sweep_study_32", kind="sweep", n=32, cells=256, U_lo=100.0, U_hi=300.0, p_lo=30.0, p_hi=50.0,
             C_lo=0.1, C_hi=1.0 / 6.0, N_lo=100_000, N_hi=100_000, S=10, launch=200, steps=400, settle=0, cap=8.0,
             cap_extra=65536, tune=True, check=200),
        # A parameter sweep with particle numbers over a factor of twenty
        # between its discharges.
        dict(name="sweep_mixed_24", kind="sweep", n=24, cells=256, U_lo=100.0, U_hi=500.0, p_lo=5.0, p_hi=50.0,
             C_lo=0.05, C_hi=0.05, N_lo=100_000, N_hi=2_000_000, S=10, launch=100, steps=200, settle=0, cap=1.5,
             cap_extra=1 << 20, tune=True, check=20),
        # A program that keeps the particles in pinned host memory between
        # stretches: load, a tenth of an RF cycle, read everything back.
        dict(name="reload_512", kind="reload", cells=512, L=0.025, U=300.0, p=20.0, C=0.05, S=10, spc=1000,
             weight=2.5e7, ne=350_001, nm=932_503, np=1_425_007, cap=1.5, cap_extra=1 << 20, steps=100, caps=True,
             rec=False, edet=False, coulomb=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "graph", "graph", "graph", "sweep", "sweep", "reload", "forward", "gradients",
                       "train", "compact"])
    if kind in ("forward", "gradients", "train"):
        c = dict(kind=kind, rows=_log(rng, 1 if kind == "forward" else 8, 2000 if kind != "train" else 300),
                 hidden=rng.randint(64, 384), outputs=rng.randint(96, 1000))
        if kind == "train":
            c["steps"] = rng.randint(5, 25)
        return c
    if kind == "compact":
        return dict(kind=kind, n=_log(rng, 1000, 20_000_000), dead=rng.uniform(0.0, 0.5), noalloc=rng.random() < 0.5)
    S = rng.choice([1, 2, 5, 10])
    U, p, C = rng.uniform(100.0, 500.0), math.exp(rng.uniform(math.log(5.0), math.log(50.0))), rng.uniform(0.0, 1 / 6)
    if kind == "sweep":
        n = rng.randint(2, 24)
        lo = _log(rng, 20_000, 200_000)
        hi = min(400_000, _log(rng, lo, 10 * lo))
        return dict(kind=kind, n=n, cells=rng.randint(128, 512), U_lo=100.0, U_hi=U + 1.0, p_lo=5.0, p_hi=max(p, 5.5),
                    C_lo=0.0, C_hi=C, N_lo=lo, N_hi=max(lo, hi), S=S, launch=100, steps=200, settle=0, cap=4.0,
                    cap_extra=1 << 18, tune=rng.random() < 0.7, check=20)
    cells = _log(rng, 64, 2048)
    ne = _log(rng, 4000, 1_000_000 if kind != "graph" else 8_000_000)
    nm = int(ne * rng.uniform(0.2, 2.5))
    np_ = int((ne + nm) * rng.uniform(1.02, 1.15))
    L = rng.uniform(0.02, 0.03)
    every = kind == "step" and rng.random() < 0.4
    c = dict(kind=kind, cells=cells, L=L, U=U, p=p, C=C, S=S, spc=1000, weight=N0 * L / ne, ne=ne, nm=nm, np=np_,
             cap=3.0, cap_extra=1 << 20, steps=100 if kind != "graph" else 200, caps=rng.random() < 0.5, rec=every,
             edet=every, coulomb=rng.choice([0, 63]) if every else 0)
    if kind != "reload":
        c["settle"] = 100
    if kind == "graph":
        c["launch"] = 200
    return c


# ---------------------------------------------------------------- inputs

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _particles(cfg, counts, seed):
    """Particles of a discharge near its periodic state: electrons and O- in
    the bulk (densities falling towards the sheath edges), O2+ neutralising
    them there and, for the rest, in the sheaths; Maxwellian velocities."""
    g = _generator(seed)
    L = cfg["L"]
    edge = 0.1 * L
    rand = lambda n: torch.rand(n, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    below = float(np.nextafter(np.float32(L), np.float32(0)))
    out = []
    for s, (n, T) in enumerate(zip(counts, (3.0, 0.026, 0.05))):
        x = edge + (L - 2 * edge) * torch.acos(1.0 - 2.0 * rand(n)) / math.pi
        if s == inputs.OP:
            m = min(n, counts[0] + counts[1])
            x[m:] = torch.remainder(L - edge + 2 * edge * rand(n - m), L)
            x = x[torch.randperm(n, generator=g, device="cuda")]
        sig = math.sqrt(T * inputs.QE / inputs.species_mass(cfg, s))
        v = torch.randn(3, n, generator=g, device="cuda") * sig
        out.append(dict(x=x.to(torch.float32).clamp_(max=below), vx=v[0], vy=v[1], vz=v[2],
                        id=torch.arange(n, device="cuda", dtype=torch.int32)))
    return out


def _discharge(c, seed, compact_check):
    cfg = inputs.base_config(L=c["L"], n_cells=c["cells"], steps_per_cycle=c["spc"], U=c["U"], p=c["p"],
                             C_meta=c["C"], ion_subcycle=c["S"], weight=c["weight"], seed=seed & 0xFFFFFFFF)
    counts = (c["ne"], c["nm"], c["np"])
    d = api.Discharge(cfg, tuple(int(c["cap"] * n) + c["cap_extra"] for n in counts), compact_check=compact_check)
    if c["caps"]:
        d.set_majorant_cap(inputs.majorant_caps(cfg))
    d.set_processes(xsec.oxygen_set(include_rec=c["rec"], include_edet=c["edet"]))
    if c["coulomb"]:
        d.set_coulomb(c["coulomb"])
    return d, cfg, _particles(cfg, counts, seed)


def _room(n):
    """Caller tensors x, vx, vy, vz, id for about n particles."""
    n = int(1.3 * n) + 16384
    return [torch.zeros(n, device="cuda") for _ in range(4)] + [torch.zeros(n, device="cuda", dtype=torch.int32)]


def _widths(c):
    return [4, c["hidden"], c["hidden"], c["hidden"], c["outputs"]]


def _network(c, seed):
    """Normalised (U, log p, L, C) and log-density profiles: smooth functions
    of them, of order one."""
    rng = np.random.Generator(np.random.PCG64(seed))
    X = rng.uniform(-1.0, 1.0, (c["rows"], 4)).astype(np.float32)
    A = rng.standard_normal((4, 8))
    B = rng.standard_normal((8, c["outputs"])) / 3.0
    T = (np.tanh(X @ A) @ B - 1.0).astype(np.float32)
    return X, T


def _caller_arrays(c, seed):
    g = _generator(seed)
    n = c["n"]
    x = 0.025 * torch.rand(n, generator=g, device="cuda")
    x[torch.rand(n, generator=g, device="cuda") < c["dead"]] = math.nan
    v = [torch.randn(n, generator=g, device="cuda") * 4.0e5 for _ in range(3)]
    ids = torch.randperm(n, generator=g, device="cuda", dtype=torch.int32)
    return [x, *v, ids]


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind in ("forward", "gradients", "train"):
        X, T = _network(c, seed)
        return dict(case=c, mlp=api.MLP(_widths(c), seed=seed), X=torch.from_numpy(X).cuda(),
                    T=torch.from_numpy(T).cuda(), loss=torch.empty(1, device="cuda"))
    if kind == "compact":
        a = _caller_arrays(c, seed)
        return dict(case=c, arrays=a, out=[torch.zeros_like(t) for t in a])
    if kind == "sweep":
        rng = np.random.Generator(np.random.PCG64(seed))
        ds = []
        for i in range(c["n"]):
            f = i / max(1, c["n"] - 1)
            N = int(round(math.exp(rng.uniform(math.log(c["N_lo"]), math.log(c["N_hi"] + 1e-9)))))
            cfg = inputs.base_config(L=0.025, n_cells=c["cells"], U=float(rng.uniform(c["U_lo"], c["U_hi"])),
                                     p=float(math.exp(rng.uniform(math.log(c["p_lo"]), math.log(c["p_hi"])))),
                                     C_meta=c["C_lo"] + f * (c["C_hi"] - c["C_lo"]), ion_subcycle=c["S"],
                                     weight=N0 * 0.025 / N, seed=(seed + i) & 0xFFFFFFFF)
            counts = (N, N, 2 * N)
            d = api.Discharge(cfg, tuple(int(c["cap"] * n) + c["cap_extra"] for n in counts),
                              compact_check=c["check"])
            d.set_processes(xsec.oxygen_set())
            d.load_state(_particles(cfg, counts, seed + 7919 * i))
            ds.append(d)
        b = api.Batch(ds, c["launch"])
        if c["tune"]:
            b.autotune()
        b.step(1)
        b.synchronize()
        for d in ds:
            d.moments(reset=True)
        room = [_room(c["n"] * k * c["N_hi"]) for k in (1, 1, 2)]
        return dict(case=c, batch=b, discharges=ds, room=room)
    if kind == "reload":
        d, cfg, st = _discharge(c, seed, 20)
        host = []
        for p in st:
            n = len(p["x"])
            room = int(1.2 * n) + 65536
            h = {}
            for k, t in p.items():
                pinned = torch.empty(room, dtype=t.dtype).pin_memory()
                pinned[:n] = t.cpu()
                h[k] = pinned.numpy() if k != "id" else pinned.numpy().view(np.uint32)
            host.append((n, h, {k: torch.zeros(room, dtype=p[k].dtype).pin_memory() for k in p}))
        return dict(case=c, discharge=d, host=host)
    d, cfg, st = _discharge(c, seed, 20 if kind == "graph" else 0)
    d.load_state(st)
    state = dict(case=c, discharge=d)
    if kind == "graph":
        state["batch"] = api.Batch([d], c["launch"])
        state["batch"].step(max(1, c["settle"] // c["launch"]))
        state["batch"].synchronize()
    else:
        d.step(c["settle"])
    d.moments(reset=True)
    state["room"] = [_room(c[k]) for k in ("ne", "nm", "np")]
    return state


# ------------------------------------------------------------------ a pass

def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "forward":
        return state["mlp"].forward(state["X"])
    if kind == "gradients":
        return state["mlp"].gradients(state["X"], state["T"])
    if kind == "train":
        for _ in range(c["steps"]):
            state["mlp"].train_step(state["X"], state["T"], 2e-4, loss=state["loss"])
        return state["loss"], state["mlp"].params()
    if kind == "compact":
        kept = api.compact_particles(*state["arrays"], out=state["out"], noalloc=c["noalloc"])
        return state["out"], len(kept[0])
    if kind == "sweep":
        b, ds = state["batch"], state["discharges"]
        b.step(c["steps"] // c["launch"])
        b.synchronize()
        # the particles of all discharges, one after the other in one array
        live, per = [], [len(r[0]) // c["n"] for r in state["room"]]
        for i, d in enumerate(ds):
            live.append([d.particles_into(s, *(t[i * m:(i + 1) * m] for t in room))
                         for s, (m, room) in enumerate(zip(per, state["room"]))])
        return (state["room"], np.array(live), np.stack([d.field()[1] for d in ds]),
                np.stack([d.moments(reset=True)[0] for d in ds]))
    d = state["discharge"]
    if kind == "reload":
        out = []
        for s, (n, h, _) in enumerate(state["host"]):
            d.load(s, *(h[k][:n] for k in ("x", "vx", "vy", "vz", "id")))
        d.set_step(0)
        d.step(c["steps"])
        for s, (_, _, back) in enumerate(state["host"]):
            into = {k: t.numpy() if k != "id" else t.numpy().view(np.uint32) for k, t in back.items()}
            out.append([d.read_into(s, into), *back.values()])
        return out, d.moments(reset=True)[0]
    if kind == "graph":
        state["batch"].step(c["steps"] // c["launch"])
        state["batch"].synchronize()
    else:
        d.step(c["steps"])
    live = [d.particles_into(s, *room) for s, room in enumerate(state["room"])]
    phi, E = d.field()
    return state["room"], live, phi, E, d.moments(reset=True)[0]


# ------------------------------------------------- what a pass cannot do without

def work(case):
    c, kind = case, case["kind"]
    if kind in ("forward", "gradients", "train"):
        w = _widths(c)
        B = c["rows"]
        weights = sum(a * b for a, b in zip(w[:-1], w[1:]))
        params = weights + sum(w[1:])
        if kind == "forward":
            return dict(bytes=2 * weights + 4 * (B * (w[0] + w[-1]) + sum(w[1:])), flops=2 * B * weights)
        flops = B * (6 * weights - 2 * w[0] * w[1])
        if kind == "gradients":
            return dict(bytes=2 * weights + 4 * (B * (w[0] + w[-1]) + params), flops=flops)
        return dict(bytes=c["steps"] * (24 * params + 4 * B * (w[0] + w[-1])), flops=c["steps"] * (flops + 12 * params))
    if kind == "compact":
        return dict(bytes=4 * c["n"] + (16 + 20) * c["n"] * (1 - c["dead"]), flops=0)
    if kind == "sweep":
        # N is log-uniform on [N_lo, N_hi]
        N = c["N_lo"] if c["N_hi"] <= c["N_lo"] else (c["N_hi"] - c["N_lo"]) / math.log(c["N_hi"] / c["N_lo"])
        pushes = c["n"] * c["steps"] * (N + 3 * N / c["S"])
        # and the particles read out at the end
        return dict(bytes=BYTES_PER_PUSH * pushes + 40 * c["n"] * 4 * N, flops=FLOPS_PER_PUSH * pushes)
    total = c["ne"] + c["nm"] + c["np"]
    pushes = c["steps"] * (c["ne"] + (c["nm"] + c["np"]) / c["S"])
    # the particles read out at the end (and, on reload, in at the start)
    moved = (20 if kind == "reload" else 40) * total + (20 * total if kind == "reload" else 0)
    return dict(bytes=BYTES_PER_PUSH * pushes + moved, flops=FLOPS_PER_PUSH * pushes)


# --------------------------------------------------------- values in 64 bits

def _bf16(w):
    """float32 values rounded to bfloat16 (to nearest, ties to even)."""
    u = np.asarray(w, np.float32).view(np.uint32).astype(np.uint64)
    u = (u + 0x7FFF + ((u >> 16) & 1)) & 0xFFFF0000
    return u.astype(np.uint32).view(np.float32).astype(np.float64)


def _initial_parameters(w, seed):
    """Glorot-uniform weights from SplitMix64, zero biases: [W0, b0, W1, ...]."""
    n = sum(a * b for a, b in zip(w[:-1], w[1:]))
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + np.arange(1, n + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    u = (z >> np.uint64(11)).astype(np.float64) / 9007199254740992.0
    out, k = [], 0
    for a, b in zip(w[:-1], w[1:]):
        lim = math.sqrt(6.0 / (a + b))
        out += [((2.0 * u[k:k + a * b] - 1.0) * lim).astype(np.float32).astype(np.float64).reshape(a, b), np.zeros(b)]
        k += a * b
    return out


def _forward64(P, X):
    H = [X]
    layers = len(P) // 2
    for i in range(layers):
        Z = H[-1] @ _bf16(P[2 * i]) + P[2 * i + 1]
        H.append(Z if i == layers - 1 else np.tanh(Z))
    return H


def _gradients64(P, X, T):
    H = _forward64(P, X)
    d = H[-1] - T
    loss, dZ, G = np.mean(d * d), 2.0 * d / d.size, []
    for i in reversed(range(len(P) // 2)):
        G = [H[i].T @ dZ, dZ.sum(0)] + G
        if i:
            dZ = (dZ @ _bf16(P[2 * i]).T) * (1.0 - H[i] ** 2)
    return G, loss


def exact(case, seed):
    """The network's results and the compaction in 64 bits.  A discharge has no
    such value: its collisions are random events decided by comparisons in
    single precision, and another rounding gives another, equally valid run."""
    c, kind = case, case["kind"]
    if kind == "compact":
        a = [t.cpu().numpy() for t in _caller_arrays(c, seed)]
        keep = ~np.isnan(a[0])
        m = int(keep.sum())
        out = [np.zeros(len(t), np.float64 if t.dtype == np.float32 else t.dtype) for t in a]
        for o, t in zip(out, a):
            o[:m] = t[keep]
        return out, m
    if kind not in ("forward", "gradients", "train"):
        return None
    X, T = (v.astype(np.float64) for v in _network(c, seed))
    P = _initial_parameters(_widths(c), seed)
    if kind == "forward":
        return _forward64(P, X)[-1]
    if kind == "gradients":
        G, loss = _gradients64(P, X, T)
        return np.concatenate([g.ravel() for g in G]), np.array([loss])
    m, v = [np.zeros_like(p) for p in P], [np.zeros_like(p) for p in P]
    for t in range(1, c["steps"] + 1):
        G, loss = _gradients64(P, X, T)
        for p, g, a, b in zip(P, G, m, v):
            a += 0.1 * (g - a)
            b += 0.001 * (g * g - b)
            p -= 2e-4 * (a / (1 - 0.9 ** t)) / (np.sqrt(b / (1 - 0.999 ** t)) + 1e-8)
    return np.array([loss]), np.concatenate([p.ravel() for p in P])
