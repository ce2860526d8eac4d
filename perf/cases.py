"""Performance cases: the calls that a user of this planner makes, at the sizes its
configurations, tests and benchmark use, through the public entry points.

A case is a dict of plain values.  `listed()` names the fixed ones, `draw(rng)` gives one
more of the same ranges, `prepare` builds what a program has in hand before the call,
`run` makes one pass, `work` counts what a pass cannot do without, and `exact` gives the
computed floating-point outputs in 64 bits from the mathematics alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_22608_gb300 import ops, planner, surrogate, synth

FLOP_TORQUE = 1379        # one evaluation of the inverse dynamics
FLOP_IK_START = 28267     # one start of the goal chart's inverse kinematics
FLOP_PAIR = 44            # one (query, node) distance
FLOP_END = 116            # both end samples of one duration from the end-sample split
DEV = "cuda"


def listed():
    return [
        # the smallest timing call: one small batch of random edges on the coarse grid (the
        # plain-timing configuration); launch, latency and the host's share count here
        dict(name="edges_small", kind="edges", E=256, K=64, S=32, cap=False, arm=0),
        # the bulk exact scan: labelling training edges, or a whole planner's edges at once
        dict(name="edges_large", kind="edges", E=65536, K=128, S=64, cap=False, arm=0),
        # goal candidates of one planning round: one fixed duration per edge (the goal branch)
        dict(name="edges_fixed", kind="fixed", E=9104, K=128, S=64, arm=0),
        # durations refined to a continuous T* (odd size: the edges that survived a filter)
        dict(name="edges_refined", kind="nary", E=20011, K=128, S=64, eps=1e-4, cap=False, arm=0),
        # surrogate-windowed timing: the network's prediction, then the verified window scan
        dict(name="surrogate_window", kind="window", E=65536, K=128, S=64, W=16, arm=0),
        # one gradient of the surrogate's training (forward and backward, the loss read back)
        dict(name="surrogate_gradient", kind="gradient", E=8192, K=128, S=64, arm=0),
        # nearest parents of one planning batch in a tree of uniformly drawn states
        dict(name="parents_batch", kind="knn", B=2048, N=4096, k=8, first=1, grown=False, arm=0),
        # nearest parents in the largest tree, whose states were grown along chords to goals
        dict(name="parents_large", kind="knn", B=8192, N=65536, k=16, first=1, grown=True, arm=0),
        # one 50 Hz control tick of a fleet: a controller cycle per instance and the
        # full-resolution recheck of one incumbent plan with obstacles
        dict(name="control_tick", kind="control", B=64, E=16, S=256, S_clear=64, n_obs=5, arm=0),
        # one planning cycle of a single problem: tree in from the host, two rounds, tree out
        dict(name="plan_cycle", kind="plan", N=4096, B=2048, k=8, K=128, S=64, rounds=2, n_obs=0,
             arm=0),
        # a planning service: 64 uneven problems in one captured iteration, four rounds after
        # their trees came in
        dict(name="plan_batched", kind="batched", P=64, n_lo=256, n_hi=16384, b_lo=128, b_hi=4096,
             k=8, K=128, S=64, rounds=4, arm=0),
        # one toss of the anytime loop from an empty tree: 48 cycles of 20 ms with pruning,
        # obstacles and the learned goal density (the tree grows past 24k nodes); the scene is
        # the stress workload's, the seed its sampling stream
        dict(name="plan_anytime", kind="anytime", cap=65536, B=8192, k=16, K=128, S=64, cycles=48,
             n_obs=5, scene=5, arm=0),
    ]


def _log_int(rng, lo, hi):
    """An integer whose logarithm is uniform, odd or even as it falls."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["edges", "edges", "fixed", "nary", "window", "gradient", "knn", "knn",
                       "control", "plan", "batched", "anytime"])
    arm = rng.randrange(4)
    K, S = rng.choice([64, 96, 128]), rng.choice([32, 48, 64])
    if kind == "edges":
        return dict(kind=kind, E=_log_int(rng, 256, 65536), K=K, S=S, cap=rng.random() < 0.5,
                    arm=arm)
    if kind == "fixed":
        return dict(kind=kind, E=_log_int(rng, 256, 65536), K=K, S=S, arm=arm)
    if kind == "nary":
        return dict(kind=kind, E=_log_int(rng, 256, 40000), K=K, S=S,
                    eps=rng.choice([1e-3, 1e-4]), cap=rng.random() < 0.5, arm=arm)
    if kind == "window":
        return dict(kind=kind, E=_log_int(rng, 4096, 65536), K=K, S=S, W=rng.choice([8, 16]),
                    arm=arm)
    if kind == "gradient":
        return dict(kind=kind, E=_log_int(rng, 1024, 32768), K=K, S=S, arm=arm)
    if kind == "knn":
        return dict(kind=kind, B=_log_int(rng, 128, 8192), N=_log_int(rng, 256, 65536),
                    k=rng.choice([4, 7, 8, 15, 16]), first=rng.choice([0, 1]),
                    grown=rng.random() < 0.5, arm=arm)
    if kind == "control":
        return dict(kind=kind, B=_log_int(rng, 1, 65536), E=_log_int(rng, 2, 64), S=256, S_clear=64,
                    n_obs=rng.choice([0, 5]), arm=arm)
    if kind == "plan":
        return dict(kind=kind, N=_log_int(rng, 256, 16384), B=_log_int(rng, 128, 4096),
                    k=rng.choice([4, 8, 16]), K=K, S=S, rounds=rng.choice([1, 2, 4]),
                    n_obs=rng.choice([0, 5]), arm=arm)
    if kind == "batched":
        return dict(kind=kind, P=_log_int(rng, 4, 64), n_lo=256, n_hi=_log_int(rng, 1024, 16384),
                    b_lo=128, b_hi=_log_int(rng, 512, 4096), k=8, K=K, S=S, rounds=4, arm=arm)
    # scenes whose object this arm can reach at once, late, or hardly
    return dict(kind=kind, cap=65536, B=_log_int(rng, 1024, 8192), k=rng.choice([8, 16]), K=128,
                S=64, cycles=rng.randrange(8, 40), n_obs=rng.choice([0, 5]),
                scene=rng.choice([1, 4, 5, 5, 7]), arm=0)


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _edges(case, seed):
    arm = synth.make_arm(case["arm"])
    s0, s1 = synth.random_edges(arm, case["E"], seed)
    return arm, s0, s1, synth.duration_grid(case["K"])


def _caps(case, seed):
    """Admissible durations left by a planner's arrival time: t_best - t(parent)."""
    if not case.get("cap"):
        return None
    rng = np.random.default_rng([0xCA9, seed])
    return rng.uniform(0.1, 1.5, case["E"]).astype(np.float32)


def _knn_states(case, seed):
    arm = synth.make_arm(case["arm"])
    N, B = case["N"], case["B"]
    if not case["grown"]:
        return synth.random_states(arm, N, seed), synth.random_states(arm, B, seed + 500_009)
    # a grown tree: states near the chords from the root to a handful of goals
    rng = np.random.default_rng([0x6012, seed])
    root, goals = synth.random_states(arm, 1, seed)[0], synth.random_states(arm, 32, seed + 7)
    half = 0.5 * (arm["q_hi"] - arm["q_lo"]).astype(np.float64)

    def near_chords(n):
        lam = rng.uniform(0.0, 1.0, (n, 1))
        g = goals[rng.integers(0, len(goals), n)].astype(np.float64)
        x = root.astype(np.float64) + lam * (g - root)
        q = np.clip(x[:, :7] + 0.1 * half * rng.standard_normal((n, 7)), arm["q_lo"], arm["q_hi"])
        qd = x[:, 8:15] + 0.1 * arm["qd_max"] * rng.standard_normal((n, 7))
        return synth.pack_states(q, qd)

    return near_chords(N), near_chords(B)


def _control_inputs(case, seed):
    arm = synth.make_arm(case["arm"])
    rng = np.random.default_rng([0xC0, seed])
    B, E = case["B"], case["E"]
    d = dict(x=synth.random_states(arm, B, 11 + seed), g=synth.random_states(arm, B, 12 + seed),
             T=rng.uniform(0.1, 1.0, B).astype(np.float32),
             prev=rng.uniform(-5.0, 5.0, (B, 7)).astype(np.float32),
             Te=rng.uniform(0.4, 1.6, E).astype(np.float32))
    d["s0"], d["s1"] = synth.random_edges(arm, E, seed)
    obs = synth.obstacles(case["n_obs"], seed) if case["n_obs"] else None
    return arm, d, obs


RATE = np.full(7, 1000.0, np.float32)   # slew limit of the controller, N m / s


def _features(arm, s0, s1):
    """The network's 28 inputs: positions scaled by the joint box, velocities by their limit."""
    lo, hi, vm = (torch.as_tensor(arm[n], dtype=s0.dtype, device=s0.device)
                  for n in ("q_lo", "q_hi", "qd_max"))
    c, h = 0.5 * (lo + hi), 0.5 * (hi - lo)
    return torch.cat([(s0[:, :7] - c) / h, s0[:, 8:15] / vm, (s1[:, :7] - c) / h, s1[:, 8:15] / vm],
                     1)


def _train_network(arm, grid, S, seed, n=131072, steps=400, batch=8192):
    """Weights of a trained duration network, as a program loads them: a few hundred Adam steps
    in plain torch on edges labelled by the exact scan."""
    a, b = synth.random_edges(arm, n, 3_000_017 + seed)
    a, b = _gpu(a), _gpu(b)
    k = ops.time_edges(arm, a, b, grid, S)["k_star"].long()
    X, f = _features(arm, a, b), (k >= 0).float()
    logT = torch.log(_gpu(grid))[k.clamp(min=0)]
    g = torch.Generator(device=DEV).manual_seed(seed)
    dims = (28, 256, 256, 256, 2)
    Ws = [((torch.rand(i, o, generator=g, device=DEV) * 2 - 1) * math.sqrt(6.0 / i))
          for i, o in zip(dims, dims[1:])]
    Ws[-1].mul_(0.1)
    bs = [torch.zeros(o, device=DEV) for o in dims[1:]]
    ps = [p.requires_grad_() for p in Ws + bs]
    opt = torch.optim.Adam(ps, lr=2e-3)
    for i in range(steps):
        for grp in opt.param_groups:
            grp["lr"] = 2e-3 * (0.02 + 0.98 * 0.5 * (1 + math.cos(math.pi * i / steps)))
        lo = (i * batch) % (n - batch + 1)
        h = X[lo:lo + batch]
        for l in range(4):
            h = h @ Ws[l] + bs[l]
            if l < 3:
                h = torch.relu(h)
        ft = f[lo:lo + batch]
        loss = (ft * (h[:, 0] - logT[lo:lo + batch]) ** 2).mean() + \
            torch.nn.functional.binary_cross_entropy_with_logits(h[:, 1], ft)
        opt.zero_grad()
        loss.backward()
        opt.step()
    out = []
    for l in range(4):
        W = Ws[l].detach().cpu().numpy()
        if l == 0:
            W = np.concatenate([W, np.zeros((4, 256), np.float32)])
        out.append((W, bs[l].detach().cpu().numpy()))
    return out


def _problem(arm, seed, batch, n_obs):
    toss = synth.random_toss(arm, seed)
    root = synth.random_states(arm, 1, 7000 + seed)[0]
    pr = synth.make_problem(toss, root=root)
    obs = synth.obstacles(n_obs, seed) if n_obs else None
    return pr, root, planner.problem_struct(pr, batch, batch // 2, root=root, obstacles=obs,
                                            seed=1000 + seed)


def _batched_sizes(case):
    """Log-uniform tree and batch sizes, fixed by the case (seeds change the states)."""
    rng = np.random.default_rng([0xC3, case["P"], case["n_hi"], case["b_hi"]])
    N = np.exp(rng.uniform(np.log(case["n_lo"]), np.log(case["n_hi"]), case["P"])).astype(int)
    B = np.exp(rng.uniform(np.log(case["b_lo"]), np.log(case["b_hi"]), case["P"])).astype(int)
    return N, B


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind in ("edges", "fixed", "nary", "window", "gradient"):
        arm, s0, s1, grid = _edges(case, seed)
        st.update(arm=arm, s0=_gpu(s0), s1=_gpu(s1), grid=grid)
        cap = _caps(case, seed)
        st["cap"] = None if cap is None else _gpu(cap)
        if kind == "fixed":
            rng = np.random.default_rng([0xF1, seed])
            st["T"] = _gpu(rng.uniform(0.1, 1.6, case["E"]).astype(np.float32))
        elif kind == "window":
            st["mlp"] = surrogate.MLP(max_batch=case["E"], seed=0)
            for l, (W, b) in enumerate(_train_network(arm, grid, case["S"], seed)):
                st["mlp"].set_params(l, W, b)
        elif kind == "gradient":
            st["mlp"] = surrogate.MLP(max_batch=case["E"], seed=seed & 0xFFFF)
            st["k_star"] = surrogate.label_edges(arm, st["s0"], st["s1"], grid, case["S"])
    elif kind == "knn":
        tree, q = _knn_states(case, seed)
        st.update(tree=_gpu(tree), q=_gpu(q))
    elif kind == "control":
        arm, d, obs = _control_inputs(case, seed)
        st.update(arm=arm, obs=obs, **{n: _gpu(v) for n, v in d.items()})
    elif kind == "plan":
        arm = synth.make_arm(case["arm"])
        pr, root, prob = _problem(arm, seed % 100_003, case["B"], case["n_obs"])
        tree, parent, t = synth.random_tree(arm, case["N"], seed, root=root, t_max=pr["t_fall"])
        pl = planner.Planner(arm, P=1, n_cap=case["N"] + (case["rounds"] + 1) * case["B"],
                             b_max=case["B"], k=case["k"], K=case["K"], S=case["S"])
        s = torch.cuda.Stream()
        pl.reset([prob], stream=s)
        pl.load_tree(0, tree, t, parent, stream=s)
        pl.capture(0, stream=s)
        st.update(pl=pl, probs=[prob], trees=[(tree, t, parent)], stream=s)
    elif kind == "batched":
        arm = synth.make_arm(case["arm"])
        N, B = _batched_sizes(case)
        trees, probs = [], []
        for p in range(case["P"]):
            pr, root, prob = _problem(arm, (seed * 64 + p) % 100_003, int(B[p]), 0)
            tree, parent, t = synth.random_tree(arm, int(N[p]), seed * 64 + p, root=root,
                                                t_max=pr["t_fall"])
            trees.append((tree, t, parent))
            probs.append(prob)
        b_max = int(B.max())
        pl = planner.Planner(arm, P=case["P"], n_cap=int(N.max()) + (case["rounds"] + 1) * b_max,
                             b_max=b_max, k=case["k"], K=case["K"], S=case["S"])
        s = torch.cuda.Stream()
        pl.reset(probs, stream=s)
        pl.capture(0, stream=s)
        st.update(pl=pl, probs=probs, trees=trees, stream=s)
    else:
        arm = synth.make_arm(case["arm"])
        scene = case["scene"]
        root = synth.random_states(arm, 1, 9000 + scene)[0]
        pr = synth.make_problem(synth.random_toss(arm, scene), root=root, sigma_linear=(0.01, 0.05))
        obs = synth.obstacles(case["n_obs"], 3) if case["n_obs"] else None
        prob = planner.problem_struct(pr, case["B"], case["B"] // 2, root=root, obstacles=obs,
                                      seed=77 + seed)
        pl = planner.Planner(arm, P=1, n_cap=case["cap"], b_max=case["B"], k=case["k"],
                             K=case["K"], S=case["S"])
        pl.set_sampler()
        s = torch.cuda.Stream()
        pl.reset([prob], stream=s)
        pl.capture(planner.FN_PLAN_PRUNE | planner.FN_PLAN_DENSITY | planner.FN_PLAN_CHORD |
                   planner.FN_PLAN_REFIT, stream=s)
        st.update(pl=pl, probs=[prob], stream=s)
    return st


# ----------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------
def _rendezvous(rounds):
    """The rendezvous records of every round and problem, field by field."""
    return {f: np.array([[r[f] for r in rs] for rs in rounds])
            for f in ("q_g", "qd_g", "T", "J", "t_best", "incumbent", "n_nodes", "n_added",
                      "status")}


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "edges":
        return ops.time_edges(st["arm"], st["s0"], st["s1"], st["grid"], case["S"],
                              T_cap=st["cap"])
    if kind == "fixed":
        return ops.time_edges(st["arm"], st["s0"], st["s1"], S=case["S"], mode=ops.FN_MODE_FIXED,
                              T_fixed=st["T"])
    if kind == "nary":
        return ops.time_edges_nary(st["arm"], st["s0"], st["s1"], st["grid"], case["S"],
                                   case["eps"], T_cap=st["cap"])
    if kind == "window":
        Y = st["mlp"].predict(st["arm"], st["s0"], st["s1"])
        out = surrogate.time_edges_window(st["arm"], st["s0"], st["s1"], st["grid"], case["S"], Y,
                                          W=case["W"])
        return dict(out, Y=Y)
    if kind == "gradient":
        loss = st["mlp"].backward(st["arm"], st["s0"], st["s1"], st["k_star"], st["grid"])
        return dict(loss=loss, grads=[st["mlp"].get_grads(l) for l in range(4)])
    if kind == "knn":
        idx, d2 = ops.knn_tree(st["tree"], st["q"], case["k"], 0.1, first=case["first"])
        return dict(idx=idx, d2=d2)
    if kind == "control":
        tau = ops.controller_torque(st["arm"], st["x"], st["g"], st["T"], 1e-3,
                                    tau_prev=st["prev"], tau_rate_max=RATE)
        chk = ops.check_edges_full(st["arm"], st["s0"], st["s1"], st["Te"], case["S"],
                                   case["S_clear"], st["obs"], 0.02)
        return dict(controller=tau, recheck=chk)
    pl, probs, s = st["pl"], st["probs"], st["stream"]
    pl.reset(probs, stream=s)
    for p, tree in enumerate(st.get("trees", ())):
        pl.load_tree(p, *tree, stream=s)
    rounds = [pl.replay(probs, it, stream=s) for it in range(case.get("cycles") or case["rounds"])]
    out = dict(rendezvous=_rendezvous(rounds))
    if kind != "batched":
        # the tree as the binding reads it: the arrays of n_cap rows under its views of n rows
        tree = pl.get_tree(0)
        out["tree"] = {f: a.base if isinstance(a, np.ndarray) else a for f, a in tree.items()}
    return out


# ----------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind in ("edges", "window", "nary"):
        # the end-sample split (6 evaluations), the end samples of every duration, and the full
        # check at the answer; refined: at least the two ends of the last bracket too
        E, S = case["E"], case["S"]
        f = E * (FLOP_TORQUE * (6 + S) + FLOP_END * case["K"])
        b = E * (128 + 21)
        if kind == "nary":
            f += E * FLOP_TORQUE * S
            b += E * 8
        if kind == "window":
            f += E * 2 * (28 * 256 + 2 * 256 * 256 + 512)
            b += E * 9
        return dict(bytes=b, flops=f)
    if kind == "fixed":
        return dict(bytes=case["E"] * (128 + 4 + 21), flops=case["E"] * FLOP_TORQUE * case["S"])
    if kind == "gradient":
        n_w = 28 * 256 + 2 * 256 * 256 + 512
        return dict(bytes=case["E"] * 132 + 8 * n_w, flops=case["E"] * 6 * n_w)
    if kind == "knn":
        return dict(bytes=64 * (case["B"] + case["N"]) + 8 * case["B"] * case["k"],
                    flops=FLOP_PAIR * case["B"] * case["N"])
    if kind == "control":
        return dict(bytes=case["B"] * (128 + 4 + 28 + 57) + case["E"] * 149,
                    flops=FLOP_TORQUE * (case["B"] + case["E"] * case["S"]))
    if kind == "batched":
        N, B = _batched_sizes(case)
    elif kind == "plan":
        N, B = np.array([case["N"]]), np.array([case["B"]])
    else:   # the tree grows from one node; take a few hundred new nodes per cycle
        N, B = np.array([min(case["cap"], 250 * case["cycles"])]), np.array([case["B"]])
    rounds = case.get("cycles") or case["rounds"]
    # per round: the distance of every candidate to every node, the goal draws' inverse
    # kinematics (one start), the split of every free edge and the check of one edge in eight
    f = rounds * float((FLOP_PAIR * N * B + FLOP_IK_START * (B // 2) +
                        FLOP_TORQUE * (B - B // 2) * case["k"] * (6 + case["S"] / 8)).sum())
    b = float((rounds * 64 * (N + B) + 72 * N).sum())
    return dict(bytes=b, flops=f)


# ----------------------------------------------------------------------------
# the same outputs in 64 bits, from the mathematics alone
# ----------------------------------------------------------------------------
class _Arm64:
    def __init__(self, arm):
        g = {k: np.asarray(v, np.float64) for k, v in arm.items()}
        self.ca, self.sa = np.cos(g["dh_alpha"]), np.sin(g["dh_alpha"])
        self.p = np.stack([g["dh_a"], -self.sa * g["dh_d"], self.ca * g["dh_d"]], 1)
        self.th0, self.m, self.c, self.I = g["dh_theta0"], g["mass"], g["com"], g["inertia"]
        self.arma, self.fr, self.grav = g["armature"], g["fric"], g["gravity"]
        self.off = self.fr[:, 0] / (1 + np.exp(-self.fr[:, 1] * self.fr[:, 2]))
        self.tau_max, self.w_max = g["tau_max"], float(g["w_max"])
        self.lo, self.hi, self.vm, self.a = g["q_lo"], g["q_hi"], g["qd_max"], g["qd_taper_a"]
        self.flange, self.rad = float(g["flange_d"]), g["link_radius"]


def _cross(a, b):
    return (a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0])


def _add(*vs):
    return tuple(sum(x) for x in zip(*vs))


def _torque(A, q, qd, qdd):
    """Recursive Newton-Euler with rotor inertia and sigmoid friction; [n, 7] float64 tensors."""
    z = torch.zeros_like(q[:, 0])
    w, dw = (z, z, z), (z, z, z)
    dv = tuple(z - x for x in A.grav)
    F, N, cs = [], [], []

    def down(j, v):       # R^T v
        c, s = cs[j]
        y = A.ca[j] * v[1] + A.sa[j] * v[2]
        return (c * v[0] + s * y, c * y - s * v[0], A.ca[j] * v[2] - A.sa[j] * v[1])

    def up(j, v):         # R v
        c, s = cs[j]
        x, y = c * v[0] - s * v[1], s * v[0] + c * v[1]
        return (x, A.ca[j] * y - A.sa[j] * v[2], A.sa[j] * y + A.ca[j] * v[2])

    for j in range(7):
        th = q[:, j] + A.th0[j]
        cs.append((torch.cos(th), torch.sin(th)))
        p, c, v, a = A.p[j], A.c[j], qd[:, j], qdd[:, j]
        dv = down(j, _add(_cross(dw, p), _cross(w, _cross(w, p)), dv))
        rw, rdw = down(j, w), down(j, dw)
        w = (rw[0], rw[1], rw[2] + v)
        dw = (rdw[0] + rw[1] * v, rdw[1] - rw[0] * v, rdw[2] + a)
        ac = _add(_cross(dw, c), _cross(w, _cross(w, c)), dv)
        F.append(tuple(A.m[j] * x for x in ac))
        Iw = tuple(A.I[j][i] * w[i] for i in range(3))
        N.append(_add(tuple(A.I[j][i] * dw[i] for i in range(3)), _cross(w, Iw)))
    tau = [None] * 7
    f, n = (z, z, z), (z, z, z)
    for j in range(6, -1, -1):
        if j < 6:
            Rf, Rn = up(j + 1, f), up(j + 1, n)
            pRf = tuple(x if torch.is_tensor(x) else z + x for x in _cross(A.p[j + 1], Rf))
        else:
            Rf, Rn, pRf = (z, z, z), (z, z, z), (z, z, z)
        n = _add(N[j], Rn, _cross(A.c[j], F[j]), pRf)
        f = _add(F[j], Rf)
        fr = A.fr[j]
        tau[j] = n[2] + A.arma[j] * qdd[:, j] + \
            fr[0] / (1 + torch.exp(-fr[1] * (qd[:, j] + fr[2]))) - A.off[j]
    return torch.stack(tau, 1)


def _cubic(s0, s1, T):
    """Coefficients of the cubic in u = t / T; [n, 7] each."""
    q0, v0, q1, v1 = s0[:, :7], s0[:, 8:15], s1[:, :7], s1[:, 8:15]
    T = T[:, None]
    d1, d2 = q1 - q0 - v0 * T, v1 - v0
    return q0, v0 * T, 3 * d1 - d2 * T, d2 * T - 2 * d1, T


def _ratios(A, s0, s1, T, u):
    """rho_tau and rho_P of the samples at normalised times u of edges at durations T."""
    q0, b1, b2, b3, T = _cubic(s0, s1, T)
    u = u[:, None]
    q = q0 + u * (b1 + u * (b2 + u * b3))
    v = (b1 + u * (2 * b2 + 3 * u * b3)) / T
    tau = _torque(A, q, v, (2 * b2 + 6 * u * b3) / T ** 2)
    tm = torch.as_tensor(A.tau_max, device=tau.device)
    return (tau.abs() / tm).amax(1), (tau * v).sum(1).abs() / A.w_max


def _taper(A, q):
    lo, hi, vm, a = (torch.as_tensor(x, device=q.device) for x in (A.lo, A.hi, A.vm, A.a))
    m = torch.minimum(q - lo, hi - q).clamp(min=0.0)
    return torch.minimum(vm.expand_as(q), torch.sqrt(2 * a * m))


def _rho_v(A, s0, s1, T):
    q0, b1, b2, b3, T = _cubic(s0, s1, T)
    us = torch.where(b3 != 0, -b2 / (3 * b3), torch.zeros_like(b3))
    us = torch.where((us > 0) & (us < 1), us, torch.zeros_like(us))
    best = torch.zeros_like(T[:, 0])
    for u in (torch.zeros_like(us), torch.ones_like(us), us):
        v = ((b1 + u * (2 * b2 + 3 * u * b3)) / T).abs()
        bd = _taper(A, q0 + u * (b1 + u * (b2 + u * b3)))
        r = torch.where(bd > 0, v / bd, torch.where(v != 0, math.inf, 0.0))
        best = torch.maximum(best, r.amax(1))
    return best


CHUNK = 1 << 20


def _check_all(A, s0, s1, T, S):
    """Both ratios over all S samples of each edge at its duration."""
    u = torch.arange(S, dtype=torch.float64, device=DEV) / (S - 1)
    rt, rp = [], []
    step = max(1, CHUNK // S)
    for i in range(0, len(T), step):
        n = len(T[i:i + step])
        a, b = _ratios(A, s0[i:i + step].repeat_interleave(S, 0),
                       s1[i:i + step].repeat_interleave(S, 0),
                       T[i:i + step].repeat_interleave(S), u.repeat(n))
        rt.append(a.view(n, S).amax(1))
        rp.append(b.view(n, S).amax(1))
    return torch.cat(rt), torch.cat(rp)


def _first_feasible(A, s0, s1, D, ok, S):
    """Per edge the first column of durations D [E, n] (admissible where ok) whose S samples all
    pass, -1 if none: single samples first (they rule most durations out), then full checks of
    the lowest durations left."""
    u = torch.arange(S, dtype=torch.float64, device=DEV) / (S - 1)
    ok = ok.clone()
    for s in sorted({0, S - 1, S // 2, S // 4, 3 * S // 4, S // 8, 7 * S // 8}):
        e, k = ok.nonzero(as_tuple=True)
        for i in range(0, len(e), CHUNK):
            ee, kk = e[i:i + CHUNK], k[i:i + CHUNK]
            a, b = _ratios(A, s0[ee], s1[ee], D[ee, kk], u[s].expand(len(ee)))
            ok[ee, kk] = (a <= 1) & (b <= 1)
    res = torch.full((len(s0),), -1, dtype=torch.long, device=DEV)
    left = ok.any(1).nonzero(as_tuple=True)[0]
    while len(left):
        k = ok[left].int().argmax(1)
        a, b = _check_all(A, s0[left], s1[left], D[left, k], S)
        good = (a <= 1) & (b <= 1)
        res[left[good]] = k[good]
        ok[left[~good], k[~good]] = False
        left = left[~good]
        left = left[ok[left].any(1)]
    return res


def _at(A, s0, s1, T, S, hit):
    """rho3 at durations T where hit, NaN elsewhere."""
    r3 = torch.full((len(T), 3), math.nan, dtype=torch.float64, device=DEV)
    if hit.any():
        a, b = _check_all(A, s0[hit], s1[hit], T[hit], S)
        r3[hit] = torch.stack([a, b, _rho_v(A, s0[hit], s1[hit], T[hit])], 1)
    return r3


def _exact_edges(case, seed):
    arm, s0, s1, grid = _edges(case, seed)
    A, S = _Arm64(arm), case["S"]
    s0, s1 = _gpu(s0).double(), _gpu(s1).double()
    if case["kind"] == "fixed":
        rng = np.random.default_rng([0xF1, seed])
        T = _gpu(rng.uniform(0.1, 1.6, case["E"]).astype(np.float32)).double()
        r3 = _at(A, s0, s1, T, S, torch.ones(len(T), dtype=torch.bool, device=DEV))
        return dict(k_star=None, T_star=T, rho3=r3, ok=None)
    cap = _caps(case, seed)
    g = _gpu(grid).double()
    D = g.expand(len(s0), -1)
    adm = torch.ones_like(D, dtype=torch.bool) if cap is None else D <= _gpu(cap).double()[:, None]
    k = _first_feasible(A, s0, s1, D, adm, S)
    hit = k >= 0
    T = torch.where(hit, g[k.clamp(min=0)], math.inf)
    out = dict(k_star=None, ok=None)
    if case["kind"] == "nary":
        # the bracket's points are formed in single precision, as the method states them
        lo = torch.where(k > 0, g[(k - 1).clamp(min=0)], 0.0).float()
        hi = T.float()
        for _ in range(8):
            act = (hit & (hi - lo > np.float32(case["eps"]))).nonzero(as_tuple=True)[0]
            if not len(act):
                break
            a, b = lo[act], hi[act]
            w = (b - a) * np.float32(1 / 32)
            j = torch.arange(1, 32, device=DEV)
            pts = (j.double() * w.double()[:, None] + a.double()[:, None]).float()
            i = _first_feasible(A, s0[act], s1[act], pts.double(),
                                torch.ones_like(pts, dtype=torch.bool), S)
            r = torch.arange(len(act), device=DEV)
            low = torch.where(i < 0, 30, i - 1)
            lo[act] = torch.where(low >= 0, pts[r, low.clamp(min=0)], a)
            hi[act] = torch.where(i >= 0, pts[r, i.clamp(min=0)], b)
        T = torch.where(hit, hi.double(), math.inf)
        out.update(T_lo=torch.where(hit, lo.double(), math.nan), rounds=None)
    out.update(T_star=T, rho3=_at(A, s0, s1, T, S, hit))
    if case["kind"] == "window":
        h = _features({n: np.asarray(arm[n], np.float64) for n in ("q_lo", "q_hi", "qd_max")}, s0,
                      s1)
        for l, (W, b) in enumerate(_train_network(arm, grid, S, seed)):
            W, b = _gpu(W).double(), _gpu(b).double()
            h = h @ W[:h.shape[1]] + b
            h = torch.relu(h) if l < 3 else h
        out.update(path=None, Y=h)
    return out


def _exact_gradient(case, seed):
    st = prepare(case, seed)
    arm, k = st["arm"], st["k_star"].long()
    ps = []
    for l in range(4):
        W, b = st["mlp"].get_params(l)
        ps.append((_gpu(W).double().requires_grad_(), _gpu(b).double().requires_grad_()))
    h = _features(arm, st["s0"].double(), st["s1"].double())
    h = torch.cat([h, torch.zeros(len(h), 4, dtype=h.dtype, device=DEV)], 1)
    for l, (W, b) in enumerate(ps):
        h = h @ W + b
        h = torch.relu(h) if l < 3 else h
    f = (k >= 0).double()
    logT = torch.log(_gpu(st["grid"]).double())[k.clamp(min=0)]
    loss = (f * (h[:, 0] - logT) ** 2).mean() + \
        torch.nn.functional.binary_cross_entropy_with_logits(h[:, 1], f)
    loss.backward()
    return dict(loss=float(loss), grads=[(W.grad, b.grad) for W, b in ps])


def _exact_knn(case, seed):
    tree, q = (_gpu(x).double() for x in _knn_states(case, seed))
    w = torch.cat([torch.ones(7), torch.tensor([0.0]), torch.full((7,), float(np.float32(0.1))),
                   torch.tensor([0.0])]).double().to(DEV)
    t, out = tree[case["first"]:], []
    step = max(1, (1 << 24) // max(1, len(t)))
    for i in range(0, len(q), step):
        x = q[i:i + step]
        d = (x * x * w).sum(1)[:, None] + (t * t * w).sum(1) - 2 * (x * w) @ t.T
        j = d.topk(min(case["k"], len(t)), largest=False).indices
        d = ((x[:, None] - t[j]) ** 2 * w).sum(2).sort(1).values     # without the cancellation
        out.append(torch.nn.functional.pad(d, (0, case["k"] - d.shape[1]), value=math.inf))
    return dict(idx=None, d2=torch.cat(out))


def _clearance(A, q, obs):
    """Least distance between the links' capsules and the spheres at configurations q [n, 7]."""
    n = len(q)
    R = torch.eye(3, dtype=torch.float64, device=DEV).expand(n, 3, 3)
    o = torch.zeros(n, 3, dtype=torch.float64, device=DEV)
    pts = []
    for j in range(7):
        o = o + R @ torch.as_tensor(A.p[j], device=DEV)
        c, s = torch.cos(q[:, j] + A.th0[j]), torch.sin(q[:, j] + A.th0[j])
        z, ca, sa = torch.zeros_like(c), float(A.ca[j]), float(A.sa[j])
        R = R @ torch.stack([c, -s, z, ca * s, ca * c, z - sa, sa * s, sa * c, z + ca],
                            1).view(n, 3, 3)
        pts.append(o)
    pts.append(o + R[:, :, 2] * A.flange)
    best = torch.full((n,), math.inf, dtype=torch.float64, device=DEV)
    for j in range(7):
        a, d = pts[j], pts[j + 1] - pts[j]
        dd = (d * d).sum(1)
        for b in obs:
            cc = torch.as_tensor(b[:3], dtype=torch.float64, device=DEV)
            t = torch.where(dd > 0, ((cc - a) * d).sum(1) / dd, 0.0).clamp(0, 1)
            dist = (cc - a - t[:, None] * d).norm(dim=1) - A.rad[j] - float(b[3])
            best = torch.minimum(best, dist)
    return best


def _exact_control(case, seed):
    arm, d, obs = _control_inputs(case, seed)
    A = _Arm64(arm)
    g = {n: _gpu(v).double() for n, v in d.items()}
    dt = float(np.float32(1e-3))
    q, v = g["x"][:, :7], g["x"][:, 8:15]
    T = g["T"][:, None]
    acc = 6 * (g["g"][:, :7] - q) / T ** 2 - (4 * v + 2 * g["g"][:, 8:15]) / T
    bd = _taper(A, q)
    acc = torch.minimum(torch.maximum(acc, (-bd - v) / dt), (bd - v) / dt)
    tm = torch.as_tensor(A.tau_max, device=DEV)
    tau = _torque(A, q, v, acc)
    tau = torch.minimum(torch.maximum(tau, -tm), tm)
    pw = (tau * v).sum(1).abs()[:, None]
    tau = torch.where(pw > A.w_max, tau * (A.w_max / pw), tau)
    sl = torch.as_tensor((RATE * np.float32(1e-3)).astype(np.float64), device=DEV)
    tau = torch.minimum(torch.maximum(tau, g["prev"] - sl), g["prev"] + sl)
    r3 = _at(A, g["s0"], g["s1"], g["Te"], case["S"],
             torch.ones(case["E"], dtype=torch.bool, device=DEV))
    cl = torch.full((case["E"],), math.inf, dtype=torch.float64, device=DEV)
    if obs is not None:
        n, E = case["S_clear"], case["E"]
        u = (torch.arange(n, dtype=torch.float64, device=DEV) / (n - 1)).repeat(E)[:, None]
        q0, b1, b2, b3, _ = (x.repeat_interleave(n, 0) for x in _cubic(g["s0"], g["s1"], g["Te"]))
        cl = _clearance(A, q0 + u * (b1 + u * (b2 + u * b3)), obs).view(E, n).amin(1)
    return dict(controller=dict(tau=tau, qdd=acc, flags=None),
                recheck=dict(rho3=r3, clearance=cl, ok=None))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("edges", "fixed", "nary", "window"):
        return _exact_edges(case, seed)
    if kind == "gradient":
        return _exact_gradient(case, seed)
    if kind == "knn":
        return _exact_knn(case, seed)
    if kind == "control":
        return _exact_control(case, seed)
    return None   # whole planning rounds: minutes of plain arithmetic
