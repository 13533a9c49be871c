"""The engine's measured cases: what a user's program has it do, through its public entry points.

Each case is a dict of plain values.  ``prepare`` makes the inputs and the
handle of one case from a seed, ``run`` makes one pass, ``work`` counts the
bytes and operations a pass cannot do without, ``exact`` gives the computed
numbers in 64 bits from the models' definitions alone (torch), ``draw`` gives
further cases of the same ranges.

The engine has two layers and both are used here: model handles (``Model``:
simulate and reduce, with intervals) and the stage entry points on tensors the
caller owns.
"""
import math

import numpy as np
import torch

import paper_1501_01405_gb300 as mrip

MAPPINGS = {"auto": mrip.MRIP_MAP_AUTO, "thread": mrip.MRIP_MAP_THREAD, "warp": mrip.MRIP_MAP_WARP_COOP,
            "cta": mrip.MRIP_MAP_CTA}
DEV = "cuda"


def listed():
    return [
        # The smallest experiment: 32 replications of 1,000 customers, the mean wait and its 95 %
        # interval through a handle.  A user who explores parameters makes this call by the hundred;
        # launches, copies and latency are all of it.
        dict(name="mm1_interval_32", kind="mm1_model", n_dp=1, n_reps=32, n_clients=1000, mapping="cta"),
        # Throughput of the same model: 2^16 replications, one thread each, three outputs.
        dict(name="mm1_64k", kind="mm1", n_dp=1, n_reps=65536, n_clients=1000, mapping="auto"),
        # An experimental plan on the 3-station tandem: 4,096 design points x 256 replications x
        # 10,000 customers, outputs, early-window features and per-design-point moments.
        dict(name="tandem_plan", kind="tandem_model", n_dp=4096, n_reps=256, n_clients=10000, window=100,
             mapping="auto"),
        # Few replications of a long horizon: 16 x 100,000 customers, a block per replication.
        dict(name="tandem_long_16", kind="tandem", n_dp=1, n_reps=16, n_clients=100000, window=100, mapping="cta"),
        # Forest fire 128 x 128, 1,000 steps, 1,024 replications: the count of every step.
        dict(name="ff128", kind="ff", n_dp=1, n_reps=1024, L=128, n_steps=1000),
        # The control-variate experiment on the 256 x 256 forest fire: 64 design points x 128
        # replications x 2,000 steps, intervals, network training and the decision: one whole call.
        dict(name="ff256_cv", kind="ff_cv", n_dp=64, n_reps=128, L=256, n_steps=2000, window=100),
        # The skip-sampled variant at the size of ff128.
        dict(name="ff128_skip", kind="ff_skip", n_dp=1, n_reps=1024, L=128, n_steps=1000),
        # Uneven stopping times: the L1-exit walk, 8 radii x 2^17 replications, through a handle.
        dict(name="walk8", kind="walk_model", n_dp=8, r_min=16, r_max=256, n_reps=131072),
        # The paper's 30-area walk of 1,000 moves, 2^16 replications.
        dict(name="area_walk_64k", kind="area", n_reps=65536, n_steps=1000, mapping="auto"),
        # The paper's Monte Carlo pi: 10^7 draws per replication.
        dict(name="pi_64", kind="pi", n_reps=64, n_draws=10000000),
        # Training of the control variate's network: the tandem plan's 4,096 x 23 fit samples, one epoch of
        # minibatches of 1,024, and its 4,096 x 3 validation samples.
        dict(name="mlp_train_94k", kind="mlp_train", d_in=8, n=94208, n_val=12288, batch=1024, epochs=1),
        # Prediction for the plan's 4,096 x 230 held-out replications.
        dict(name="mlp_predict_942k", kind="mlp_forward", d_in=8, n=942080),
    ]


def _log_int(rng, lo, hi):
    """An integer of [lo, hi], spread evenly over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["mm1_model", "mm1", "tandem_model", "tandem", "ff", "ff", "ff_cv", "ff_skip", "walk_model",
                       "area", "pi", "mlp_train", "mlp_forward"])
    if kind in ("mm1_model", "mm1", "tandem_model", "tandem"):
        n_clients = _log_int(rng, 200, 100000)
        few = rng.random() < 0.5
        n_reps = _log_int(rng, 30, 1500) if few else _log_int(rng, 2000, 200000)
        n_reps = max(30, min(n_reps, 3 * 10 ** 9 // n_clients))
        n_dp = max(1, min(_log_int(rng, 1, 4096), 200000 // n_reps, 3 * 10 ** 9 // (n_clients * n_reps)))
        # a block or a warp per replication is meant for a few thousand replications at most
        mapping = rng.choice(["cta", "cta", "warp", "thread"]) if n_dp * n_reps <= 1500 else "auto"
        c = dict(kind=kind, n_dp=n_dp, n_reps=n_reps, n_clients=n_clients, mapping=mapping)
        if kind in ("tandem_model", "tandem"):
            c["window"] = rng.choice([50, 75, 100, 100])
        return c
    if kind in ("ff", "ff_skip", "ff_cv"):
        L = rng.choice([32, 64, 128, 128, 256, 256, 512])
        # (the control variate's window is an early one: 100 steps of many more)
        n_steps = _log_int(rng, 800 if kind == "ff_cv" else 120, 2500)
        n_dp = _log_int(rng, 1, 64)
        n_reps = _log_int(rng, 40, 4000)
        limit = 4 * 10 ** 11 // (L * L * n_steps)
        n_dp = max(1, min(n_dp, limit // 40))
        n_reps = max(40, min(n_reps, limit // n_dp))
        c = dict(kind=kind, n_dp=n_dp, n_reps=n_reps, L=L, n_steps=n_steps)
        if kind == "ff_cv":
            c["window"] = 100
        return c
    if kind == "walk_model":
        r_min = _log_int(rng, 4, 64)
        n_dp = _log_int(rng, 1, 12)
        return dict(kind=kind, n_dp=n_dp, r_min=r_min, r_max=_log_int(rng, r_min + n_dp, 300),
                    n_reps=_log_int(rng, 500, 300000))
    if kind == "area":
        n_reps = _log_int(rng, 30, 300000)
        return dict(kind=kind, n_reps=n_reps, n_steps=_log_int(rng, 300, 10000),
                    mapping="warp" if n_reps < 16000 else "auto")
    if kind == "pi":
        n_draws = _log_int(rng, 100000, 20000000)
        return dict(kind=kind, n_reps=max(1, min(_log_int(rng, 1, 300), 4 * 10 ** 9 // n_draws)), n_draws=n_draws)
    if kind == "mlp_train":
        n = _log_int(rng, 600, 100000)
        return dict(kind=kind, d_in=rng.choice([6, 8]), n=n, n_val=max(64, n // 9),
                    batch=rng.choice([256, 512, 1024, 1024, 2048]), epochs=rng.choice([1, 2, 3]))
    return dict(kind="mlp_forward", d_in=rng.choice([6, 8]), n=_log_int(rng, 5000, 2000000))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _queue_points(case, rng):
    """(lambda, mu) or (lambda, mu1..3); one M/M/1 design point is the paper's kind of loaded queue."""
    n = case["n_dp"]
    if case["kind"].startswith("mm1"):
        lam = rng.uniform(0.85, 0.95, size=n) if n == 1 else rng.uniform(0.3, 0.95, size=n)
        return np.ascontiguousarray(np.column_stack([lam, np.ones(n)]))
    return np.ascontiguousarray(np.column_stack([rng.uniform(0.5, 0.95, size=n), rng.uniform(1.0, 1.5, size=(n, 3))]))


def _fire_points(case, rng):
    """(p_grow, p_lightning): growth from 1e-3 to 5e-2 over the design points, 0.01 for one."""
    n = case["n_dp"]
    i = np.arange(n)
    p = 1e-3 * 50.0 ** (i / (n - 1)) if n > 1 else np.array([0.01])
    return np.ascontiguousarray(np.column_stack([p * rng.uniform(0.97, 1.0, size=n), np.full(n, 1e-5)]))


def _radii(case):
    if (case["n_dp"], case["r_min"], case["r_max"]) == (8, 16, 256):
        return np.array([16, 32, 48, 64, 96, 128, 192, 256], dtype=np.float64)
    n = case["n_dp"]
    if n == 1:
        return np.array([float(case["r_max"])])
    return np.round(case["r_min"] * (case["r_max"] / case["r_min"]) ** (np.arange(n) / (n - 1)))


def _samples(case, seed):
    """Standardised inputs (d_in planes) and a smooth target with noise, as the engine's own features give."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    d = case["d_in"]

    def some(n):
        x = torch.randn((d, n), generator=g, device=DEV)
        y = 0.7 * x[0] - 0.4 * x[1] + 0.25 * x[0] * x[2] + 0.2 * torch.tanh(x[3] + x[4])
        y = y + 0.3 * torch.randn(n, generator=g, device=DEV)
        return x.contiguous(), ((y - y.mean()) / y.std()).contiguous()

    return some


def _empty(n, dtype=torch.float64):
    return torch.empty(n, dtype=dtype, device=DEV)


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng(int(seed))
    s = dict(case=case, seed=int(rng.integers(1, 2 ** 62)))
    if kind in ("mm1", "mm1_model", "tandem", "tandem_model"):
        dps = _queue_points(case, rng)
        items = case["n_dp"] * case["n_reps"]
        s["dps"] = dps
        if kind == "mm1":
            s["d_dps"] = torch.tensor(dps, device=DEV)
            s["out"] = [_empty(items) for _ in range(3)]
        elif kind == "tandem":
            s["d_dps"] = torch.tensor(dps, device=DEV)
            s["y"], s["feat"] = _empty(items), _empty(8 * items)
        else:
            if kind == "mm1_model":
                s["model"] = mrip.Model(mrip.MRIP_MM1, n_clients=case["n_clients"])
            else:
                s["model"] = mrip.Model(mrip.MRIP_TANDEM3, n_clients=case["n_clients"], window=case["window"])
                s["y"], s["feat"] = _empty(items), _empty(8 * items)
            if case["mapping"] != "auto":
                s["model"].set_plan('{"mapping": %d}' % MAPPINGS[case["mapping"]])
    elif kind in ("ff", "ff_skip"):
        items = case["n_dp"] * case["n_reps"]
        s["d_dps"] = torch.tensor(_fire_points(case, rng), device=DEV)
        s["counts"] = torch.empty((items, case["n_steps"]), dtype=torch.int32, device=DEV)
        s["scalar"] = _empty(items)
    elif kind == "ff_cv":
        s["dps"] = _fire_points(case, rng)
        s["model"] = mrip.Model(mrip.MRIP_FOREST_FIRE, L=case["L"], n_steps=case["n_steps"], density=0.5,
                                window=case["window"])
        items = case["n_dp"] * case["n_reps"]
        s["counts"], s["scalar"] = torch.empty((items, case["n_steps"]), dtype=torch.int32, device=DEV), _empty(items)
    elif kind == "walk_model":
        s["dps"] = _radii(case)[:, None]
        s["model"] = mrip.Model(mrip.MRIP_WALK_L1_EXIT, max_steps=1 << 38)
        s["tau"] = _empty(case["n_dp"] * case["n_reps"], torch.int64)
    elif kind == "area":
        s["final"] = _empty(case["n_reps"], torch.int32)
        s["visits"] = torch.empty((30, case["n_reps"]), dtype=torch.int32, device=DEV)
    elif kind == "pi":
        s["hits"] = _empty(case["n_reps"], torch.int64)
    elif kind == "mlp_train":
        some = _samples(case, seed)
        (s["x"], s["y"]), (s["xv"], s["yv"]) = some(case["n"]), some(case["n_val"])
        P = mrip.mrip_mlp_param_count(case["d_in"])
        steps = case["epochs"] * -(-case["n"] // case["batch"])
        s["theta"], s["m"], s["v"] = (_empty(P, torch.float32) for _ in range(3))
        s["losses"], s["val_losses"] = _empty(steps, torch.float32), _empty(case["epochs"], torch.float32)
    else:
        s["x"] = _samples(case, seed)(case["n"])[0]
        s["theta"] = _empty(mrip.mrip_mlp_param_count(case["d_in"]), torch.float32)
        mrip.mrip_mlp_init(case["d_in"], s["seed"], s["theta"])
        s["yhat"] = _empty(case["n"], torch.float32)
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "mm1":
        mrip.mrip_mm1_simulate(s["d_dps"], case["n_reps"], case["n_clients"], s["seed"], MAPPINGS[case["mapping"]],
                               *s["out"])
        return {"wait": s["out"][0], "idle": s["out"][1], "system": s["out"][2]}
    if kind == "tandem":
        mrip.mrip_tandem3_simulate(s["d_dps"], 0, case["n_reps"], case["n_clients"], case["window"], s["seed"], 0,
                                   MAPPINGS[case["mapping"]], s["y"], s["feat"])
        return {"y": s["y"], "features": s["feat"]}
    if kind == "mm1_model":
        m = s["model"]
        m.run(s["dps"], case["n_reps"], s["seed"])
        stats = m.stats(0.95)
        return {"mean": np.array([d["mean"] for d in stats]), "var": np.array([d["var"] for d in stats]),
                "half_width": np.array([d["half_width"] for d in stats]), "wait": m.outputs(0)}
    if kind == "tandem_model":
        m = s["model"]
        m.run(s["dps"], case["n_reps"], s["seed"])
        moments = m.moments()
        mrip.mrip_outputs(m.h, 0, s["y"])
        mrip.mrip_outputs(m.h, 1, s["feat"])
        return {"moments": moments, "y": s["y"], "features": s["feat"]}
    if kind in ("ff", "ff_skip"):
        simulate = mrip.mrip_forest_fire_simulate if kind == "ff" else mrip.mrip_forest_fire_skip_simulate
        simulate(s["d_dps"], case["n_reps"], case["L"], case["n_steps"], 0.5, s["seed"], counts=s["counts"],
                 scalar=s["scalar"])
        return {"counts": s["counts"], "scalar": s["scalar"]}
    if kind == "ff_cv":
        plain, cv, report = s["model"].run_cv(s["dps"], case["n_reps"], s["seed"])
        theta, norm = s["model"].cv_network()
        mrip.mrip_outputs(s["model"].h, 0, s["counts"])
        mrip.mrip_outputs(s["model"].h, 1, s["scalar"])
        return {"plain": np.array([[d["mean"], d["var"], d["half_width"]] for d in plain]),
                "cv": np.array([[d["beta"], d["mean"], d["var"], d["half_width"]] for d in cv]),
                "declined": report["declined"], "epochs": report["epochs_run"], "m_ctrl": report["m_ctrl"],
                "theta": theta, "norm": norm, "counts": s["counts"], "scalar": s["scalar"]}
    if kind == "walk_model":
        m = s["model"]
        m.run(s["dps"], case["n_reps"], s["seed"])
        moments = m.moments()
        mrip.mrip_outputs(m.h, 0, s["tau"])
        return {"moments": moments, "tau": s["tau"]}
    if kind == "area":
        mrip.mrip_area_walk_simulate(case["n_reps"], case["n_steps"], s["seed"], MAPPINGS[case["mapping"]],
                                     s["final"], s["visits"])
        return {"final": s["final"], "visits": s["visits"]}
    if kind == "pi":
        mrip.mrip_pi_simulate(case["n_reps"], case["n_draws"], s["seed"], s["hits"])
        return {"hits": s["hits"]}
    if kind == "mlp_train":
        mrip.mrip_mlp_init(case["d_in"], s["seed"], s["theta"])
        info = mrip.mrip_mlp_train(case["d_in"], s["x"], s["y"], s["theta"], case["batch"], case["epochs"], s["seed"],
                                   xv=s["xv"], yv=s["yv"], losses=s["losses"], m=s["m"], v=s["v"],
                                   val_losses=s["val_losses"])
        return {"theta": s["theta"], "m": s["m"], "v": s["v"], "losses": s["losses"], "val_losses": s["val_losses"],
                "epochs": info[0], "kept": info[1], "steps": info[2]}
    mrip.mrip_mlp_forward(s["theta"], case["d_in"], s["x"], s["yhat"])
    return {"yhat": s["yhat"]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
BLOCK_OPS = 60   # one Philox4x32-10 block: 10 rounds of 2 widening multiplies and 4 exclusive ors
LOG_OPS = 12     # one logarithm: normalise, one table entry, a cubic and the scaling


def work(case):
    kind = case["kind"]
    items = case.get("n_dp", 1) * case.get("n_reps", 1)
    if kind in ("mm1", "mm1_model"):
        out = 3 if kind == "mm1" else 1
        return {"bytes": 8.0 * (out * items + 2 * case["n_dp"]),
                "flops": float(items) * case["n_clients"] * (BLOCK_OPS + 2 * LOG_OPS + 6)}
    if kind in ("tandem", "tandem_model"):
        return {"bytes": 8.0 * (9 * items + 4 * case["n_dp"]),
                "flops": float(items) * case["n_clients"] * (2 * BLOCK_OPS + 4 * LOG_OPS + 10)}
    if kind in ("ff", "ff_cv"):
        cells = float(items) * case["n_steps"] * case["L"] ** 2
        return {"bytes": 4.0 * items * case["n_steps"] + 8.0 * items, "flops": cells * (BLOCK_OPS / 4 + 1)}
    if kind == "ff_skip":
        p = float(np.mean(_fire_points(case, np.random.default_rng(0))[:, 0]))
        events = p * case["L"] ** 2 + 2
        return {"bytes": 4.0 * items * case["n_steps"] + 8.0 * items,
                "flops": float(items) * case["n_steps"] * (events * (BLOCK_OPS / 2 + LOG_OPS) + case["L"] ** 2 / 2)}
    if kind == "walk_model":
        moves = float(np.sum(_radii(case) ** 2)) * 2 / 3 * case["n_reps"]  # E[tau] is near 2 R^2 / 3
        return {"bytes": 8.0 * items, "flops": moves * (BLOCK_OPS / 64 + 0.5)}
    if kind == "area":
        return {"bytes": 4.0 * 31 * items, "flops": float(items) * case["n_steps"] * (BLOCK_OPS / 64 + 3)}
    if kind == "pi":
        return {"bytes": 8.0 * items, "flops": float(items) * case["n_draws"] * (BLOCK_OPS / 2 + 4)}
    d = case["d_in"]
    macs = 64 * d + 64 * 64 + 64
    if kind == "mlp_train":
        n, e = case["n"], case["epochs"]
        return {"bytes": 4.0 * ((d + 1) * (n + case["n_val"]) * e + 3 * (macs + 129)),
                "flops": 2.0 * e * (3 * n + case["n_val"]) * macs}
    return {"bytes": 4.0 * (d + 1) * case["n"], "flops": 2.0 * case["n"] * macs}


# ---------------------------------------------------------------------------
# the computed numbers in 64 bits, from the definitions
# ---------------------------------------------------------------------------
M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    k0, k1 = seed & M32, (seed >> 32) & M32
    x = [c0, c1, c2, c3]
    for _ in range(10):
        p0, p1 = x[0] * 0xD2511F53, x[2] * 0xCD9E8D57
        x = [((p1 >> 32) & M32) ^ x[1] ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ x[3] ^ k1, p0 & M32]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return x


def _expo(lo, hi):
    """-log(1 - u), u the top 53 bits of hi:lo times 2^-53 (1 - u is exact in 64 bits)."""
    u = ((hi << 21) | (lo >> 11)).double() * 2.0 ** -53
    return -torch.log(1.0 - u)


def _variates(c0, n0, n_clients, rep, dp, seed):
    """The two exponentials of block (c0, client) for clients n0 .. of every item: (items, clients) each."""
    n = torch.arange(n0, n0 + n_clients, device=DEV)[None, :].expand(rep.numel(), n_clients)
    w = _philox(torch.full_like(n, c0), n, rep[:, None].expand_as(n), dp[:, None].expand_as(n), seed)
    return _expo(w[0], w[1]), _expo(w[2], w[3])


def _chunks(items, per):
    step = max(1, (1 << 23) // per)
    return [(a, min(a + step, items)) for a in range(0, items, step)]


def _exact_mm1(case, dps, seed):
    n, items = case["n_clients"], case["n_dp"] * case["n_reps"]
    dps = torch.tensor(dps, device=DEV)
    out = [_empty(items) for _ in range(3)]
    for a, b in _chunks(items, n):
        i = torch.arange(a, b, device=DEV)
        dp = i // case["n_reps"]
        S, A = _variates(0, 0, n, i % case["n_reps"], dp, seed)
        S, A = S / dps[dp, 1:2], A / dps[dp, 0:1]
        P = torch.cumsum(S - A, 1)
        P = torch.cat([torch.zeros_like(P[:, :1]), P], 1)
        W = P - torch.cummin(P, 1).values  # W_n = P_n - min over k <= n of P_k
        out[0][a:b] = W[:, :n].mean(1)
        out[1][a:b] = torch.relu(A - W[:, :n] - S).mean(1)
        out[2][a:b] = (W[:, :n] + S).mean(1)
    return out


def _exact_tandem(case, dps, seed):
    n, items = case["n_clients"], case["n_dp"] * case["n_reps"]
    dps = torch.tensor(dps, device=DEV)
    y, feat = _empty(items), torch.empty((8, items), dtype=torch.float64, device=DEV)
    w = min(case["window"], n)
    for a, b in _chunks(items, 2 * n):
        i = torch.arange(a, b, device=DEV)
        dp = i // case["n_reps"]
        gap, s1 = _variates(0, 0, n, i % case["n_reps"], dp, seed)
        s2, s3 = _variates(1, 0, n, i % case["n_reps"], dp, seed)
        v = [t / dps[dp, k:k + 1] for k, t in enumerate((gap, s1, s2, s3))]
        arrive = torch.cumsum(v[0], 1)
        D = arrive
        for S in v[1:]:  # D_{n,j} = max(D_{n-1,j}, D_{n,j-1}) + S_{n,j}
            C = torch.cumsum(S, 1)
            D = C + torch.cummax(D - (C - S), 1).values
        y[a:b] = (D - arrive).mean(1)
        feat[:4, a:b] = dps[dp].T
        for k in range(4):
            feat[4 + k, a:b] = v[k][:, :w].mean(1)
    return y, feat.reshape(-1)


def _exact_fire(case, dps, seed):
    """The mean burning fraction of every replication."""
    L, items = case["L"], case["n_dp"] * case["n_reps"]
    item = torch.arange(items, device=DEV)
    dp, rep = (item // case["n_reps"])[:, None], (item % case["n_reps"])[:, None]
    block = torch.arange(L * L // 4, device=DEV)[None, :]
    grow, light = (torch.floor(torch.tensor(dps, device=DEV) * 2.0 ** 32).long()[dp[:, 0], k] for k in (0, 1))

    def words(t, tag):
        c1 = torch.full_like(block, t)
        w = torch.broadcast_tensors(*_philox(block, c1, rep, dp + (tag << 24), seed))
        return torch.stack(w, 2).reshape(items, L, L)

    tree = words(0, 1) < 2 ** 31
    burning = torch.zeros_like(tree)
    total = torch.zeros(items, dtype=torch.int64, device=DEV)
    for t in range(1, case["n_steps"] + 1):
        w = words(t, 0)
        near = burning.roll(1, 1) | burning.roll(-1, 1) | burning.roll(1, 2) | burning.roll(-1, 2)
        ignite = tree & (near | (w < light[:, None, None]))
        tree = (tree & ~ignite) | (~tree & ~burning & (w < grow[:, None, None]))
        burning = ignite
        total += burning.sum((1, 2))
    return total.double() / (float(case["n_steps"]) * L * L)


def _bf16(x):
    return x.float().bfloat16().double()


def _unpack(theta, d):
    """W1, b1, W2, b2, W3, b3 of a flat parameter vector."""
    at = np.cumsum([0, 64 * d, 64, 64 * 64, 64, 64, 1])
    p = [theta[a:b] for a, b in zip(at[:-1], at[1:])]
    return p[0].view(64, d), p[1], p[2].view(64, 64), p[3], p[4], p[5]


def _initial(d, seed):
    """He-uniform weights from stream tag 3, zero biases."""
    e = torch.arange(64 * d + 64 * 64 + 64, device=DEV)
    z = torch.zeros_like(e)
    w = _philox(e >> 1, z, z, z + (3 << 24), seed)
    lo, hi = torch.where(e % 2 == 1, w[2], w[0]), torch.where(e % 2 == 1, w[3], w[1])
    u = ((hi << 21) | (lo >> 11)).double() * 2.0 ** -53
    fan = torch.where(e < 64 * d, float(d), 64.0)
    v = ((2.0 * u - 1.0) * torch.sqrt(6.0 / fan)).float().double()
    zero = torch.zeros(64, dtype=torch.float64, device=DEV)
    return torch.cat([v[:64 * d], zero, v[64 * d:64 * d + 4096], zero, v[64 * d + 4096:], zero[:1]])


def _forward(theta, d, x):
    W1, b1, W2, b2, W3, b3 = _unpack(theta, d)
    h1 = torch.relu(_bf16(x).T @ _bf16(W1).T + b1)
    h2 = torch.relu(_bf16(h1) @ _bf16(W2).T + b2)
    return h1, h2, _bf16(h2) @ _bf16(W3) + b3


def _exact_train(case, s):
    d, n, B = case["d_in"], case["n"], case["batch"]
    x, y, xv, yv = (s[k].double() for k in ("x", "y", "xv", "yv"))
    theta = _initial(d, s["seed"])
    m, v = torch.zeros_like(theta), torch.zeros_like(theta)
    losses, val, best, t = [], [], None, 0
    zero = torch.zeros(1, dtype=torch.int64, device=DEV)
    lr, b1, b2, eps = (float(np.float32(k)) for k in (1e-3, 0.9, 0.999, 1e-8))
    for epoch in range(case["epochs"]):
        w = _philox(zero, zero + epoch, zero, zero + (4 << 24), s["seed"])
        a = 1 + int(w[0]) % (n - 1)
        while math.gcd(a, n) != 1:
            a = a + 1 if a + 1 < n else 1
        order = (torch.arange(n, device=DEV) * a + int(w[1]) % n) % n
        for k in range(0, n, B):
            i = order[k:k + B]
            xb, nb = x[:, i], i.numel()
            h1, h2, out = _forward(theta, d, xb)
            W1, _, W2, _, W3, _ = _unpack(theta, d)
            r = out - y[i]
            losses.append((r * r).mean())
            dy = 2.0 * r / nb
            dz2 = dy[:, None] * _bf16(W3) * (h2 > 0)
            dz1 = (_bf16(dz2) @ _bf16(W2)) * (h1 > 0)
            g = torch.cat([(_bf16(dz1).T @ _bf16(xb).T).reshape(-1), dz1.sum(0), (_bf16(dz2).T @ _bf16(h1)).reshape(-1),
                           dz2.sum(0), _bf16(h2).T @ dy, dy.sum()[None]])
            t += 1
            m = b1 * m + (1 - b1) * g
            v = b2 * v + (1 - b2) * g * g
            theta = theta - lr * (m / (1 - b1 ** t)) / (torch.sqrt(v / (1 - b2 ** t)) + eps)
        val.append(((_forward(theta, d, xv)[2] - yv) ** 2).mean())
        if best is None or val[-1] < best[0]:
            best = (val[-1], theta)
    return {"theta": best[1], "m": m, "v": v, "losses": torch.stack(losses), "val_losses": torch.stack(val),
            "epochs": None, "kept": None, "steps": None}


def exact(case, seed):
    kind = case["kind"]
    items = case.get("n_dp", 1) * case.get("n_reps", 1)
    if kind in ("mm1", "mm1_model") and items * case["n_clients"] <= 3 * 10 ** 9:
        s = prepare(case, seed)
        wait, idle, system = _exact_mm1(case, s["dps"], s["seed"])
        if kind == "mm1":
            return {"wait": wait, "idle": idle, "system": system}
        w = wait.view(case["n_dp"], case["n_reps"])
        return {"mean": w.mean(1), "var": w.var(1), "half_width": None, "wait": wait}
    if kind in ("tandem", "tandem_model") and items * case["n_clients"] <= 3 * 10 ** 9:
        s = prepare(case, seed)
        y, feat = _exact_tandem(case, s["dps"], s["seed"])
        if kind == "tandem":
            return {"y": y, "features": feat}
        w = y.view(case["n_dp"], case["n_reps"])
        mean = w.mean(1)
        m2 = ((w - mean[:, None]) ** 2).sum(1)
        return {"moments": torch.stack([torch.full_like(mean, case["n_reps"]), mean, m2], 1), "y": y, "features": feat}
    if kind == "ff" and items * case["n_steps"] * case["L"] ** 2 <= 2 * 10 ** 10 and items * case["L"] ** 2 <= 2 ** 26:
        s = prepare(case, seed)
        return {"counts": None, "scalar": _exact_fire(case, s["d_dps"].cpu().numpy(), s["seed"])}
    if kind == "mlp_train":
        return _exact_train(case, prepare(case, seed))
    if kind == "mlp_forward":
        s = prepare(case, seed)
        d = case["d_in"]
        theta = _initial(d, s["seed"])
        return {"yhat": torch.cat([_forward(theta, d, part.double())[2] for part in s["x"].split(1 << 18, 1)])}
    return None
