"""Performance cases: the work that a user of this library has it do.

Every case goes through the public entry points of the Python binding
(``paper_2609_21803_gb300``), on seeded synthetic inputs of the sizes that the
tests, the benchmark and the examples use.  Kinds of work:

  push     score mode orders of pushing instances (``Problem.eval``): one
           persistent launch that solves one trajectory optimisation per order,
           with the trajectories returned.  Families: ``l2`` (2 segments of 8
           intervals), ``l4`` (4 of 20), ``mixed`` (rectangles, 1..6 segments of
           10..30 intervals by the instance's number, ragged lengths in one call),
           ``free`` (the pushing grammar with free motion, up to 8 segments of
           10).  Cold starts, or warm starts from a record per order.
  timed    the same with the interval durations among the controls
           (``comet_eval_modes_timed``), under a duration bound with room or one
           that binds.
  bim      score mode orders of the bimanual box flip (507 modes).
  predict  the learned proposal on a batch of orders: predicted merits and warm
           starts (``comet_proposal_predict``), for pushing and the box flip.
  train    one optimiser step of the learned proposal on a batch held by the
           caller, gradients and updated parameters returned.
  expand   one expansion round of Algorithm 1 on an evaluated set: top-k,
           neighbourhood, deduplication, the next batch (``comet_expand``).
  plan     whole calls: Algorithm 1 for many instances (``comet_plan_batch``).
"""
import math

import numpy as np
import torch

import paper_2609_21803_gb300 as P

# typical solver iterations per order, for work(): the counts that the
# evaluators report on these families (they differ from seed to seed)
_ITERS = {"l2": 60, "l4": 110, "mixed": 110, "free": 120, "bim1": 120, "bim": 170, "timed": 340}
# FP32 operations of the method per stage and iteration (the oracle's count)
_FLOPS = {"push": 1989.2, "timed": 3555.3, "bim": 8185.0}
_WIDTH = 256


def listed():
    return [
        # a single small call: every 2-segment order of one instance (144
        # solves of 16 intervals); its time is the latency of the longest solve
        {"name": "push_l2_enum", "kind": "push", "family": "l2", "n": 144, "instances": 1, "warm": False},
        # the benchmark's step: every 4-segment order of one instance, 80 intervals
        {"name": "push_l4_enum", "kind": "push", "family": "l4", "n": 20736, "instances": 1, "warm": False},
        # many instances of different shapes and lengths scored in one call
        {"name": "push_mixed", "kind": "push", "family": "mixed", "n": 16384, "instances": 64, "warm": False},
        # the paper's box experiment: every admissible order of at most 8
        # segments, free motion among the modes
        {"name": "push_free_enum", "kind": "push", "family": "free", "n": 6297, "instances": 1, "warm": False},
        # orders refined with their durations free, under a bound that binds
        {"name": "timed_l4", "kind": "timed", "family": "l4", "n": 4096, "instances": 1, "bound": "binding"},
        # the seed batch of a box-flip plan: the 507 one-segment orders
        {"name": "bim_seeds", "kind": "bim", "n": 507, "instances": 1, "segments": 1},
        # box-flip orders of 1..6 segments over several instances in one call
        {"name": "bim_mixed", "kind": "bim", "n": 2048, "instances": 8, "segments": 6},
        # ranking and warm-starting a whole enumeration with the proposal
        {"name": "predict_push", "kind": "predict", "family": "l4", "n": 20736, "instances": 1},
        # ranking and warm-starting a box-flip beam's neighbourhood
        {"name": "predict_bim", "kind": "predict", "family": "bim", "n": 8192, "instances": 1},
        # one training step of the proposal at the training batch size
        {"name": "train_push", "kind": "train", "family": "l4", "n": 4096, "instances": 16},
        # one expansion round: beam 64, two-edit neighbourhoods under the
        # pushing grammar, the next batch of at most 1,024 orders
        {"name": "expand_free", "kind": "expand", "family": "free", "n": 3000, "k": 64, "batch": 1024, "radius": 2},
        # a whole planning call: 32 instances at once, three expansion rounds,
        # refinement of the best
        {"name": "plan_mixed", "kind": "plan", "family": "mixed", "instances": 32, "k": 16, "batch": 256,
         "rounds": 3, "k_ref": 16, "ref_iters": 600},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["push", "push", "push", "timed", "bim", "predict", "train", "expand", "plan"])
    if kind == "push":
        fam = rng.choice(["l2", "l4", "mixed", "free"])
        n = _log_int(rng, 32, {"l2": 16384, "l4": 20736, "mixed": 16384, "free": 12288}[fam])
        inst = rng.randint(1, max(1, min(64, n // 32)))
        return {"kind": "push", "family": fam, "n": n, "instances": inst, "warm": rng.random() < 0.3}
    if kind == "timed":
        fam = rng.choice(["l2", "l4"])
        n = _log_int(rng, 64, 4096)
        return {"kind": "timed", "family": fam, "n": n, "instances": rng.randint(1, 4),
                "bound": rng.choice(["room", "binding"])}
    if kind == "bim":
        return {"kind": "bim", "n": _log_int(rng, 64, 2048), "instances": rng.randint(1, 8),
                "segments": rng.randint(1, 6)}
    if kind == "predict":
        fam = rng.choice(["l4", "mixed", "bim"])
        n = _log_int(rng, 256, {"l4": 20736, "mixed": 16384, "bim": 8192}[fam])
        return {"kind": "predict", "family": fam, "n": n, "instances": rng.randint(1, 16)}
    if kind == "train":
        fam = rng.choice(["l4", "mixed", "bim"])
        return {"kind": "train", "family": fam, "n": _log_int(rng, 256, 4096), "instances": rng.randint(1, 16)}
    if kind == "expand":
        fam = rng.choice(["l4", "free", "bim"])
        n = _log_int(rng, 300, 6000 if fam == "free" else 16384)
        return {"kind": "expand", "family": fam, "n": n, "k": rng.choice([16, 32, 64]),
                "batch": _log_int(rng, 128, 4096), "radius": rng.choice([1, 2]) if fam == "free" else 1}
    return {"kind": "plan", "family": rng.choice(["l4", "mixed"]), "instances": _log_int(rng, 2, 32),
            "k": rng.choice([8, 16]), "batch": rng.choice([64, 128, 256]), "rounds": rng.randint(1, 3),
            "k_ref": rng.choice([8, 16]), "ref_iters": 600}


# ------------------------------------------------------------------ inputs


def _mean_radius(a, b):
    """Mean distance from the centre of an a x b rectangle (midpoint rule)."""
    xs = (np.arange(200) + 0.5) / 200 * a - a / 2
    ys = (np.arange(200) + 0.5) / 200 * b - b / 2
    return float(np.mean(np.hypot(*np.meshgrid(xs, ys))))


def _instance(family, rng, i):
    if family == "bim":
        w, h = rng.uniform(0.1, 0.3, 2)
        mass, sgn, off = rng.uniform(0.5, 2.0), rng.choice([-1.0, 1.0]), rng.uniform(0.0, 0.3)
        ax, az, th = 0.5 * w, 0.5 * h, math.pi / 2 + sgn * off
        goal = [-ax + ax * math.cos(th) - az * math.sin(th), ax * math.sin(th) + az * math.cos(th), th]
        return {"task": 1, "side_x": w, "side_y": h, "c_ls": 0.0, "mu": 0.5, "dt": 0.05, "kappa": 1.0,
                "knots_per_segment": 15, "max_segments": 6, "n_modes": 507, "start": [0.0, az, 0.0], "goal": goal,
                "w_terminal": 10.0, "w_control": 0.1, "mass": mass, "ground_mu": 0.5}
    d = {"task": 0, "side_x": 0.09, "side_y": 0.09, "c_ls": 0.04, "mu": 0.3, "dt": 0.1, "kappa": 1.0, "n_modes": 12,
         "w_terminal": 10.0, "w_control": 0.1}
    pose = lambda p, t: [float(v) for v in (rng.uniform(-p, p), rng.uniform(-p, p), rng.uniform(-t, t))]  # noqa: E731
    if family == "l2":
        d.update(knots_per_segment=8, max_segments=2, start=[0.0, 0.0, 0.0], goal=pose(0.2, math.pi / 2))
    elif family == "l4":
        d.update(knots_per_segment=20, max_segments=4, start=pose(0.3, math.pi), goal=pose(0.3, math.pi))
    elif family == "free":
        d.update(knots_per_segment=10, max_segments=8, n_modes=13, start=pose(0.3, math.pi), goal=pose(0.3, math.pi))
    else:
        a, asp = rng.uniform(0.05, 0.15), rng.uniform(1.0, 3.0)
        d.update(side_x=float(a), side_y=float(a / asp), c_ls=_mean_radius(a, a / asp), mu=float(rng.uniform(0.2, 0.6)),
                 knots_per_segment=10 + (7 * i + 12) % 21, max_segments=1 + (i + 3) % 6,
                 start=pose(0.3, math.pi), goal=pose(0.3, math.pi))
    return d


def _admissible(cap):
    """Orders of the pushing grammar: free motion (12) first, no repeats,
    direct contact switches only between adjacent faces."""
    out, level = [], [(12,)]
    for _ in range(cap):
        out += level
        level = [s + (m,) for s in level for m in (0, 3, 6, 9, 12)
                 if m != s[-1] and (s[-1] == 12 or m == 12 or (s[-1] // 3 - m // 3) % 4 in (1, 3))]
    return out


def _orders(family, n, insts, rng, segments=0):
    """n packed orders; orders of one instance are distinct where they can be."""
    idx = np.sort(np.arange(n, dtype=np.int32) % len(insts))
    if family == "free":
        every = _admissible(8)
        per = [rng.permutation(len(every)) for _ in insts]
        seen = [0] * len(insts)
        seqs = []
        for i in idx:
            seqs.append(every[per[i][seen[i] % len(every)]])
            seen[i] += 1
        return P.pack_mode_seqs(seqs, idx)
    if family in ("l2", "l4"):
        L = 2 if family == "l2" else 4
        codes = np.concatenate([rng.permutation(np.resize(np.arange(12 ** L), c)) if c >= 12 ** L
                                else rng.choice(12 ** L, c, replace=False)
                                for c in np.bincount(idx, minlength=len(insts))])
        modes = np.stack([codes // 12 ** (L - 1 - j) % 12 for j in range(L)], axis=1)
        return P.pack_mode_seqs(modes.astype(np.uint16), idx)
    if family == "bim":
        if segments == 1 and n == 507 * len(insts):
            return P.pack_mode_seqs(np.tile(np.arange(507, dtype=np.uint16), len(insts))[:, None], idx)
        lens = rng.integers(1, segments + 1, n)
        modes = rng.integers(0, 507, (n, 6))
    else:
        lens = np.array([rng.integers(1, insts[i]["max_segments"] + 1) for i in idx])
        modes = rng.integers(0, 12, (n, 6))
    modes = np.where(np.arange(6)[None, :] < lens[:, None], modes, 0).astype(np.uint16)
    return P.pack_mode_seqs(modes, idx, lens)


def _device(packed):
    return torch.from_numpy(packed.view(np.uint8).reshape(len(packed), P.MODE_SEQ_BYTES)).cuda()


def _warm(insts, packed, n_max, rng):
    """Warm-start records: the poses interpolated, small random controls (the
    form that the proposal predicts)."""
    n = len(packed)
    w = np.zeros((n, 7 * n_max + 4), np.float32)
    K = np.array([d["knots_per_segment"] for d in insts])[packed["instance"]]
    N = K * packed["len"]
    k = np.arange(n_max + 1)[None, :]
    al = k / N[:, None]
    s = np.array([d["start"] for d in insts])[packed["instance"]]
    g = np.array([d["goal"] for d in insts])[packed["instance"]]
    for c in range(3):
        w[:, c * (n_max + 1):(c + 1) * (n_max + 1)] = np.where(k <= N[:, None],
                                                               (1 - al) * s[:, c:c + 1] + al * g[:, c:c + 1], 0.0)
    u = rng.normal(0.0, 0.05, (n, 3, n_max)) * (np.arange(n_max)[None, None, :] < N[:, None, None])
    u[:, 0] = np.abs(u[:, 0])
    w[:, 4 * (n_max + 1):] = u.reshape(n, -1)
    return torch.from_numpy(w).cuda()


def _params(dims, rng):
    """Network weights as a trained proposal has them: U(-a, a) with a few
    times the initial scale, small biases."""
    flat = []
    for i, o in zip(dims[:-1], dims[1:]):
        flat += [rng.uniform(-2.0, 2.0, o * i) / math.sqrt(i), rng.uniform(-0.05, 0.05, o)]
    return np.concatenate(flat).astype(np.float32)


def _make(case, seed):
    """Everything of a case that is numbers: instances, orders, weights."""
    rng = np.random.default_rng([int(seed), 77])
    fam = "bim" if case["kind"] == "bim" else case["family"]
    n_inst = 1 if case["kind"] == "expand" else case["instances"]
    insts = [_instance(fam, rng, i) for i in range(n_inst)]
    m = {"rng": rng, "family": fam, "insts": insts,
         "n_max": max(d["knots_per_segment"] * d["max_segments"] for d in insts),
         "l_max": max(d["max_segments"] for d in insts)}
    if case["kind"] != "plan":
        segments = case.get("segments", 6)
        if case["kind"] == "expand" and fam != "free":
            segments = 2
        m["packed"] = _orders(fam, case["n"], insts, rng, segments)
    if case["kind"] in ("predict", "train"):
        bim = fam == "bim"
        i_dim = -(-(12 + (30 if bim else 13) * m["l_max"]) // 64) * 64
        o_dim = -(-(1 + (12 if bim else 3) * m["n_max"]) // 16) * 16
        m["dims"] = [i_dim, _WIDTH, _WIDTH, _WIDTH, o_dim]
        m["flat"] = _params(m["dims"], rng)
    if case["kind"] == "train":
        n, o_dim = case["n"], m["dims"][-1]
        m["target"] = rng.normal(0.0, 0.3, (n, o_dim)).astype(np.float32)
        # weights as the training set has them: 1 on the log merit, a share on
        # each control of a converged solve, 0 elsewhere
        N = np.array([d["knots_per_segment"] for d in insts])[m["packed"]["instance"]] * m["packed"]["len"]
        nc = 12 if fam == "bim" else 3
        om = np.zeros((n, o_dim), np.float32)
        om[:, 0] = 1.0
        conv = rng.random(n) < 0.85
        ctrl = np.tile(np.arange(m["n_max"]), nc)[None, :] < N[:, None]
        om[:, 1:1 + nc * m["n_max"]] = np.where(ctrl & conv[:, None], 1.0 / (nc * N[:, None]), 0.0)
        m["omega"] = om
    if case["kind"] == "expand":
        m["cost"] = rng.uniform(0.01, 5.0, case["n"]).astype(np.float32)
        m["viol"] = (10.0 ** rng.uniform(-8.0, -1.0, case["n"])).astype(np.float32)
    if case["kind"] == "plan":
        m["seeds"] = [[(a,) for a in range(12)] + ([(a, b) for a in range(12) for b in range(12)][i % 5::5]
                                                   if d["max_segments"] > 1 else []) for i, d in enumerate(insts)]
    return m


def _features(m):
    """The proposal's input rows (float64 values of the BF16 features)."""
    bim = m["family"] == "bim"
    q, n = m["packed"], len(m["packed"])
    f = np.zeros((len(m["insts"]), 12), np.float32)
    for i, d in enumerate(m["insts"]):
        s, g = d["start"], d["goal"]
        dx, dy, c, sn = g[0] - s[0], g[1] - s[1], math.cos(s[2]), math.sin(s[2])
        rel = [3 * dx, 3 * dy, g[2] - s[2], d["mass"]] if bim else [3 * (c * dx + sn * dy), 3 * (-sn * dx + c * dy),
                                                                    g[2] - s[2], 0.0]
        f[i] = [*s, *g, 10 * d["side_x"], 10 * d["side_y"], *rel]
    x = np.zeros((n, m["dims"][0]), np.float32)
    x[:, :12] = f[q["instance"]]
    rows = np.arange(n)
    slot = 30 if bim else 13
    for j in range(m["l_max"]):
        on, mo, at = j < q["len"], q["modes"][:, j].astype(np.int64), 12 + slot * j
        if bim:
            for e in (mo // 169, 3 + mo // 13 % 13, 16 + mo % 13):
                x[rows[on], at + e[on]] = 1.0
            x[rows[~on], at + 29] = 1.0
        else:
            x[rows, at + np.where(on, mo, 12)] = 1.0
    return torch.from_numpy(x).to(torch.bfloat16)


# ----------------------------------------------------------------- the calls


def prepare(case, seed):
    m = _make(case, seed)
    kind, insts = case["kind"], m["insts"]
    prob = P.Problem(insts)
    s = {"kind": kind, "prob": prob}
    if kind in ("push", "bim", "timed"):
        s["orders"], n = _device(m["packed"]), case["n"]
        if kind == "push":
            s["warm"] = _warm(insts, m["packed"], m["n_max"], m["rng"]) if case["warm"] else None
        if kind == "timed":
            dt, N = insts[0]["dt"], m["n_max"]
            s["bounds"] = (dict(h_min=0.5 * dt, h_max=2.0 * dt, T_max=2.0 * N * dt) if case["bound"] == "room"
                           else dict(h_min=0.2 * dt, h_max=3.0 * dt, T_max=0.75 * N * dt))
            f32 = dict(dtype=torch.float32, device="cuda")
            i32 = dict(dtype=torch.int32, device="cuda")
            s["out"] = {"cost": torch.empty(n, **f32), "status": torch.empty(n, **i32),
                        "traj": torch.empty((n, 9 * N + 5), **f32), "viol": torch.empty(n, **f32),
                        "merit": torch.empty(n, **f32), "iters": torch.empty(n, **i32), "stat": torch.empty(n, **f32)}
    elif kind in ("predict", "train"):
        q = s["q"] = P.comet_proposal_create(prob.handle, dict(width=_WIDTH, rows_cap=case["n"]))
        i_dim, _, o_dim, n_params = P.comet_proposal_dims(q)
        assert [i_dim, o_dim, n_params] == [m["dims"][0], m["dims"][-1], len(m["flat"])]
        P.comet_proposal_set_params(q, m["flat"])
        f32 = dict(dtype=torch.float32, device="cuda")
        if kind == "predict":
            s["orders"] = _device(m["packed"])
            s["merit"], s["warm"] = torch.empty(case["n"], **f32), torch.empty((case["n"], prob.stride), **f32)
        else:
            s["x"] = _features(m).cuda().view(torch.int16)
            s["target"], s["omega"] = torch.from_numpy(m["target"]).cuda(), torch.from_numpy(m["omega"]).cuda()
            s["params"], s["grad"] = torch.empty(n_params, **f32), torch.empty(n_params, **f32)
    elif kind == "expand":
        grammar = P.GRAMMAR_PUSH if m["family"] == "free" else P.GRAMMAR_NONE
        cap = case["n"] + 4 * case["batch"]
        s["f"] = P.comet_frontier_create(prob.handle, 0, cap, case["batch"], case["k"], case["radius"], grammar)
        P.comet_frontier_add(s["f"], _device(m["packed"]), case["n"], torch.from_numpy(m["cost"]).cuda(),
                             torch.from_numpy(m["viol"]).cuda())
        s["k"], s["batch"] = case["k"], case["batch"]
        s["next"] = torch.zeros((case["batch"], P.MODE_SEQ_BYTES), dtype=torch.uint8, device="cuda")
    else:
        s["seeds"] = m["seeds"]
        s["opts"] = dict(k=case["k"], batch=case["batch"], rounds=case["rounds"], k_ref=case["k_ref"],
                         ref_iters=case["ref_iters"])
    return _State(s)


class _State:
    """What the caller's program holds; handles go with it."""

    def __init__(self, s):
        self.s = s

    def __del__(self):
        try:
            if "q" in self.s:
                P.comet_proposal_destroy(self.s["q"])
            if "f" in self.s:
                P.comet_frontier_destroy(self.s["f"])
            self.s["prob"].close()
        except Exception:
            pass


def run(state):
    s = state.s
    kind, prob = s["kind"], s["prob"]
    if kind in ("push", "bim"):
        return prob.eval(s["orders"], warm=s.get("warm"), want_traj=True)
    if kind == "timed":
        o = s["out"]
        P.comet_eval_modes_timed(prob.handle, s["bounds"], s["orders"], len(s["orders"]), None, 1500, o["cost"],
                                 o["traj"], o["status"])
        P.comet_eval_stats(prob.handle, o["viol"], o["merit"], o["iters"], o["stat"])
        return o
    if kind == "predict":
        P.comet_proposal_predict(s["q"], s["orders"], len(s["orders"]), s["merit"], s["warm"])
        return {"merit": s["merit"], "warm": s["warm"]}
    if kind == "train":
        loss = P.comet_proposal_train_batch(s["q"], s["x"], s["target"], s["omega"], len(s["x"]))
        P.comet_proposal_get_params(s["q"], s["params"], s["grad"])
        return {"loss": np.float32(loss), "params": s["params"], "grad": s["grad"]}
    if kind == "expand":
        P.comet_expand(prob.handle, s["f"], s["k"])
        n = P.comet_frontier_copy_next(s["f"], s["next"], s["batch"])
        return {"n": n, "next": s["next"]}
    res = P.comet_plan_batch(prob.handle, list(range(len(s["seeds"]))), s["seeds"], s["opts"])
    best = np.full((len(res), 16), -1, np.int32)
    for i, r in enumerate(res):
        best[i, :len(r["best"])] = r["best"]
    return {"best": best, "cost": np.array([r["best_cost"] for r in res], np.float32),
            "viol": np.array([r["best_viol"] for r in res], np.float32),
            "status": np.array([r["best_status"] for r in res], np.int32),
            "evaluations": np.array([r["evaluations"] for r in res], np.int64)}


# ----------------------------------------------------------- work and truth


def work(case):
    kind, n = case["kind"], case.get("n", 0)
    if kind in ("push", "bim", "timed"):
        fam = "bim" if kind == "bim" else case["family"]
        N = {"l2": 16, "l4": 80, "mixed": 60, "free": 75, "bim": 7.5 * (case.get("segments", 1) + 1)}[fam]
        it = _ITERS["timed" if kind == "timed" else "bim1" if kind == "bim" and case["segments"] == 1 else fam]
        # the trajectory records are as long as the longest order allows
        stride = {"l2": 116, "l4": 564, "mixed": 1264, "free": 564, "bim": 1535}[fam]
        stride = {"l2": 149, "l4": 725}[fam] if kind == "timed" else stride
        return {"bytes": n * (64.0 + 4 * stride * (2 if case.get("warm") else 1)), "flops": _FLOPS[kind] * n * N * it}
    if kind in ("predict", "train"):
        i, o, stride = {"l4": (64, 256, 564), "mixed": (128, 544, 1264), "bim": (192, 1088, 1535)}[case["family"]]
        macs = i * _WIDTH + 2 * _WIDTH * _WIDTH + _WIDTH * o
        if kind == "predict":
            return {"bytes": n * (44.0 + 4 * stride) + 2 * macs, "flops": 2.0 * n * macs}
        # the batch read once; parameters and both moments read and written,
        # gradients written, parameters and gradients returned
        return {"bytes": n * (2.0 * i + 8 * o) + 36.0 * macs, "flops": 2.0 * n * (3 * macs - i * _WIDTH)}
    if kind == "expand":
        slots1 = {"l4": 112, "free": 93, "bim": 6597}[case["family"]]
        slots = slots1 * (1 + (slots1 if case["radius"] == 2 else 0))
        # the evaluated set read, a probe of its table per neighbour, the batch written
        return {"bytes": 12.0 * n + 8.0 * case["k"] * slots + 40.0 * case["batch"], "flops": 0}
    i, N = case["instances"], {"l4": 60, "mixed": 45}[case["family"]]
    solves = i * (40 + case["batch"] * case["rounds"])
    return {"bytes": 64.0 * solves, "flops": _FLOPS["push"] * N * (110 * solves + 300 * i * case["k_ref"])}


def _gelu(z):
    t = torch.tanh(math.sqrt(2 / math.pi) * (z + 0.044715 * z ** 3))
    return 0.5 * z * (1 + t), 0.5 * (1 + t) + 0.5 * z * (1 - t * t) * math.sqrt(2 / math.pi) * (1 + 0.134145 * z * z)


def exact(case, seed):
    """The network's calls in 64 bits, on the BF16 features and weights that
    the proposal holds.  The evaluators are local solvers of non-convex
    problems: their results have no closed value (None)."""
    if case["kind"] not in ("predict", "train"):
        return None
    m = _make(case, seed)
    x = _features(m).double().cuda()
    W, b, off = [], [], 0
    flat = torch.from_numpy(m["flat"]).cuda()
    for i, o in zip(m["dims"][:-1], m["dims"][1:]):
        W.append(flat[off:off + o * i].reshape(o, i).to(torch.bfloat16).double())
        b.append(flat[off + o * i:off + o * i + o].double())
        off += o * i + o
    H, D = [x], []
    for j in range(3):
        h, d = _gelu(H[-1] @ W[j].T + b[j])
        H.append(h)
        D.append(d)
    y = H[3] @ W[3].T + b[3]
    q, n_max = m["packed"], m["n_max"]
    if case["kind"] == "predict":
        bim = m["family"] == "bim"
        nx, nc = (5, 12) if bim else (4, 3)
        N = torch.from_numpy(np.array([d["knots_per_segment"] for d in m["insts"]])[q["instance"]] * q["len"]).cuda()
        per = lambda key: torch.tensor([d[key] for d in m["insts"]], dtype=torch.float64).cuda()[  # noqa: E731
            torch.from_numpy(q["instance"].astype(np.int64)).cuda()]
        start, goal = per("start"), per("goal")
        k = torch.arange(n_max + 1, device="cuda", dtype=torch.float64)[None, :]
        al = k / N[:, None]
        w = torch.zeros((len(q), nx * (n_max + 1) + nc * n_max), dtype=torch.float64, device="cuda")
        for c in range(3):
            w[:, c * (n_max + 1):(c + 1) * (n_max + 1)] = torch.where(
                k <= N[:, None], (1 - al) * start[:, c:c + 1] + al * goal[:, c:c + 1], 0.0)
        u = y[:, 1:1 + nc * n_max].reshape(len(q), nc, n_max).clone()
        if bim:
            u[:, [3, 4, 6, 7, 9, 10]] *= (per("mass") * 9.81)[:, None, None]
        u *= (torch.arange(n_max, device="cuda")[None, :] < N[:, None])[:, None, :]
        w[:, nx * (n_max + 1):] = u.reshape(len(q), -1)
        return {"merit": torch.exp(y[:, 0]), "warm": w}
    n = case["n"]
    t, om = torch.from_numpy(m["target"]).double().cuda(), torch.from_numpy(m["omega"]).double().cuda()
    loss = (om * (y - t) ** 2).sum() / n
    g = 2 * om * (y - t) / n
    grads = []
    for j in (3, 2, 1, 0):
        grads = [(g.T @ H[j]).reshape(-1), g.sum(0)] + grads
        if j:
            g = (g @ W[j]) * D[j - 1]
    grad = torch.cat(grads)
    # the first AdamW step at the default options: the bias-corrected moments
    # are the gradient and its square
    params = flat.double() - 1e-3 * grad / (grad.abs() + 1e-8)
    return {"loss": float(loss), "params": params, "grad": grad}
