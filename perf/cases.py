"""What this library is timed on: passes through its public entry points, as a program that uses it makes them.

A program builds a run (RelayRun on the GPU, HostRelayRun for a state in pinned host memory), binds its
objective, and then makes one call per iteration (step), one call for many iterations (steps), or asks for
the convergence metrics.  The state here is that of a run some way in: models close to one another, messages
holding the sums of the models behind them, counters at their steady values, optimiser moments that have
built up.  Sizes are those of workloads.py (the paper's worker counts, topologies and model sizes) and odd
ones between them.

A case: entry ("step", "steps", "metrics" or "host"), tree, n workers, d parameters, and
  k          iterations per call (entry "steps"; entry "host": 1 is step(), more is steps(k))
  objective  "stored" centres (an array read at each step) or "generated" (formed in the kernel)
  mix        the generated centres' mixture: "identity" (one Gaussian per worker) or "dirichlet" (10 shared)
  opt        local step: "sgd", "nesterov" or "adam"
  algo       "relaysgd", "grad" (the updates are relayed) or "dme" (mean estimation)
  lost       share of the messages lost in transit on the call's iterations
  mode       rebuild: 0 divides by the models received, 1 fills the missing ones
"""
import functools
import math

import numpy as np
import torch

import paper_2110_04175_gb300 as rs
from paper_2110_04175_gb300 import host_stream
from paper_2110_04175_gb300 import workloads as wl

DEV = "cuda"
T0 = 100          # the iteration that the state stands at
X0_STD = 0.1
MU_SCALE = 1.0
CENTRES = 10      # Gaussian centres of the Dirichlet mixture
BETA1, BETA2, EPS = 0.9, 0.999, 1e-8


def _case(name, entry, tree, n, d, k=1, objective="stored", mix="identity", opt="sgd", algo="relaysgd", lost=0.0,
          mode=1, lr=0.05, sigma=0.05):
    c = dict(entry=entry, tree=tree, n=n, d=d, k=k, objective=objective, mix=mix, opt=opt, algo=algo, lost=lost,
             mode=mode, lr=lr, sigma=sigma)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest run: a toy problem or a unit test of somebody's training loop, one call per iteration;
        # latency and launches are all there is
        _case("step_chain8_d4096", "step", "chain", 8, 4_096, lr=0.1, sigma=0.1),
        # a small vision model on a binary tree, one call per iteration (d is not a multiple of 4)
        _case("step_binary16_d272474", "step", "binary", 16, 272_474),
        # a mid-size model on a chain whose workers' data is a Dirichlet mixture; the centres take no memory
        _case("step_chain16_dirichlet", "step", "chain", 16, 9_231_114, objective="generated", mix="dirichlet"),
        # the same model on the data-centre topology of double binary trees (two column windows per step)
        _case("step_double16_d9231114", "step", "double", 16, 9_231_114),
        # a hub with 63 neighbours: every message of the step passes one worker
        _case("step_star64_d25000000", "step", "star", 64, 25_000_000),
        # an unreliable network on an irregular tree: Adam, a tenth of the messages lost, odd length
        _case("step_torus64_adam_lost", "step", "torus", 64, 1_000_003, opt="adam", lost=0.1, lr=0.001),
        # the largest: a language model's 1.1e8 parameters on 32 workers, one call per iteration
        _case("step_binary32_d110000000", "step", "binary", 32, 110_000_000, lr=0.01, sigma=0.01),
        # many iterations per call, for a program that looks at the state only now and then: smallest,
        # small and mid-size models
        _case("steps64_chain8_d4096", "steps", "chain", 8, 4_096, k=64, lr=0.1, sigma=0.1),
        _case("steps64_binary16_d272474", "steps", "binary", 16, 272_474, k=64),
        _case("steps64_binary32_d9231114", "steps", "binary", 32, 9_231_114, k=64, lr=0.01, sigma=0.01),
        # how far the workers are apart and from the optimum, asked between iterations
        _case("metrics_torus64_d9231114", "metrics", "torus", 64, 9_231_114),
        # a state that stays in pinned host memory and passes through the GPU in chunks
        _case("host_binary16_d2000003", "host", "binary", 16, 2_000_003, objective="generated"),
    ]


def draw(rng):
    entry = rng.choice(["step", "step", "step", "steps", "steps", "metrics", "host"])
    tree = rng.choice(["chain", "binary", "star", "random", "double", "torus"])
    if entry == "host" and tree == "double":
        tree = "binary"  # a host run takes one tree
    n = rng.choice([16, 36, 64]) if tree == "torus" else int(round(math.exp(rng.uniform(math.log(4), math.log(64)))))
    # worker-coordinates of the call at most, per entry: a step's worth of the larger listed ones
    most = {"step": 8e8, "steps": 1.5e8, "metrics": 6e8, "host": 3.2e7}[entry]
    d = int(math.exp(rng.uniform(math.log(1_000), math.log(most / n))))
    k = {"step": 1, "metrics": 1, "steps": rng.choice([2, 8, 33, 64, 100]), "host": rng.choice([1, 1, 8])}[entry]
    objective = "generated" if entry == "host" else rng.choice(["stored", "stored", "generated"])
    mix = rng.choice(["identity", "dirichlet"])
    opt = "sgd" if entry == "host" else rng.choice(["sgd", "sgd", "nesterov", "adam"])
    algo = "relaysgd" if opt != "sgd" or entry == "host" else rng.choice(["relaysgd", "relaysgd", "grad", "dme"])
    lost = rng.choice([0.0, 0.0, 0.1]) if entry in ("step", "steps") else 0.0
    lr = 0.001 if opt == "adam" else rng.choice([0.01, 0.05])
    return _case(None, entry, tree, n, d, k, objective, mix, opt, algo, lost, rng.choice([0, 1, 1]), lr,
                 rng.choice([0.01, 0.05]))


# ------------------------------------------------------------------ inputs


@functools.lru_cache(maxsize=64)
def _edges(tree, n):
    if tree == "double":
        return [np.asarray(t, np.int32) for t in wl.double_binary_trees(n)]
    side = int(round(math.sqrt(n)))
    make = {"chain": wl.chain, "binary": wl.binary_tree, "star": wl.star,
            "random": lambda m: wl.random_tree(m, seed=1),
            "torus": lambda m: wl.torus_spanning_tree(side, side, seed=0)}
    return [np.asarray(make[tree](n), np.int32)]


def _windows(case):
    """(first column, columns) of each tree: the trees split the coordinates at whole quads."""
    trees, nq = len(_edges(case["tree"], case["n"])), (case["d"] + 3) // 4
    cut = [min(4 * (nq * k // trees), case["d"]) for k in range(trees + 1)]
    return [(a, b - a) for a, b in zip(cut, cut[1:])]


def _directed(edges):
    """(src, dst) of the directed edges: 2u is edges[u][0] -> edges[u][1], 2u + 1 its reverse."""
    src, dst = np.empty(2 * len(edges), np.int64), np.empty(2 * len(edges), np.int64)
    src[0::2], src[1::2], dst[0::2], dst[1::2] = edges[:, 0], edges[:, 1], edges[:, 1], edges[:, 0]
    return src, dst


def _next_counts(src, dst, n, c, lost=None):
    arriving = np.zeros(n, np.int64)
    np.add.at(arriving, dst, c)
    new = 1 + arriving[src] - c[np.arange(len(c)) ^ 1]
    return new if lost is None else np.where(lost, 0, new)


def _steady(edges, n):
    src, dst = _directed(edges)
    c = np.zeros(len(src), np.int64)
    while True:
        new = _next_counts(src, dst, n, c)
        if np.array_equal(new, c):
            return c
        c = new


def _lost(case, seed, k):
    """Lost messages of tree k on the call's iterations, or None."""
    E = 2 * (case["n"] - 1)
    if not case["lost"]:
        return None
    return np.random.Generator(np.random.PCG64(seed * 2 + k)).random(E) < case["lost"]


def _mix(case):
    n = case["n"]
    return wl.identity_mix(n) if case["mix"] == "identity" else wl.dirichlet_mix(n, CENTRES, 0.1, seed=0)


def _wide(edges, n):
    """Workers with more than 4 neighbours: their received sums follow the messages of a device run."""
    deg = np.bincount(np.asarray(edges).ravel(), minlength=n)
    return [i for i in range(n) if deg[i] > 4]


def _fill(case, seed, x, mu, state, msgs):
    """The state of a run at iteration T0 in the given tensors, from the seed alone."""
    n, d, algo = case["n"], case["d"], case["algo"]
    g = torch.Generator(device=x.device)
    g.manual_seed(seed)
    base = torch.empty(d, device=x.device).normal_(generator=g)
    if mu is not None:
        for i in range(n):
            mu[i, :d].normal_(generator=g)
    for s, t in enumerate(state):
        for i in range(n):
            row = t[i, :d].normal_(generator=g)
            if s == 0:
                row.mul_(0.3)
            else:
                row.square_().mul_(0.1).add_(0.01)
    spread = {"relaysgd": 0.05, "grad": 0.05, "dme": 10.0}[algo]
    for i in range(n):
        x[i, :d].normal_(generator=g).mul_(spread).add_(base)
    for (col, w), m, edges in zip(_windows(case), msgs, _edges(case["tree"], n)):
        src, dst = _directed(edges)
        for e, c in enumerate(_steady(edges, n)):
            row = m[e, :w].normal_(generator=g)
            if algo == "relaysgd":      # the sum of c models
                row.mul_(0.05 * math.sqrt(c)).add_(base[col:col + w], alpha=float(c))
            elif algo == "grad":        # the sum of c updates
                row.mul_(case["lr"] * math.sqrt(c))
            else:                       # the sum of c samples
                row.mul_(math.sqrt(c))
        if m.shape[0] > len(src):       # the received sums of the workers with more than 4 neighbours
            for r, i in enumerate(_wide(edges, n)):
                total = m[len(src) + r, :w].zero_()
                for e in np.flatnonzero(dst == i):
                    total += m[e, :w]


def _optimizer(case):
    return {"sgd": None, "nesterov": ("nesterov", BETA1), "adam": ("adam", BETA1, BETA2, EPS)}[case["opt"]]


def prepare(case, seed):
    n, d = case["n"], case["d"]
    trees = _edges(case["tree"], n)
    if case["entry"] == "host":
        run = host_stream.HostRelayRun(n, d, trees[0], chunk=1 << 19, mode=case["mode"], full_output=True, device=DEV)
        run.init(X0_STD, seed, _mix(case), MU_SCALE, seed + 1, case["sigma"])
        x = torch.zeros(run.x_h.shape, device=DEV)
        m = torch.zeros(run.msg_h[0].shape, device=DEV)
        _fill(case, seed, x, None, [], [m])
        run.x_h.copy_(x)
        run.msg_h[run.cur].copy_(m)
        run.counts_h[:run.E].copy_(torch.from_numpy(_steady(trees[0], n)))
        run.t = T0
        return {"case": case, "seed": seed, "run": run}
    run = rs.RelayRun(n, d, trees if len(trees) > 1 else trees[0], device=DEV, mode=case["mode"],
                      objective=case["objective"], optimizer=_optimizer(case), algorithm=case["algo"])
    run.init(X0_STD, seed, _mix(case), MU_SCALE, seed + 1, case["sigma"])
    _fill(case, seed, run.x, run.mu, run.state, [tr.msg[tr.cur] for tr in run.trees])
    for k, (tr, edges) in enumerate(zip(run.trees, trees)):
        tr.counts[:tr.E].copy_(torch.from_numpy(_steady(edges, n)))
        if case["lost"]:
            run.set_lost(_lost(case, seed, k), k)
    run.t = T0
    return {"case": case, "seed": seed, "run": run}


def run(state):
    case, seed, r = state["case"], state["seed"], state["run"]
    d = case["d"]
    if case["entry"] == "metrics":
        return r.metrics()
    if case["entry"] == "host":
        if case["k"] == 1:
            r.step(case["lr"], seed)
        else:
            r.steps(case["k"], case["lr"], seed)
        return {"x": r.x_h[:, :d], "messages": [r.msg_h[r.cur][:, :d]], "counts": [r.counts_h[:r.E]]}
    if case["entry"] == "step":
        r.step(case["lr"], seed)
    else:
        r.steps(case["k"], case["lr"], seed)
    out = {"x": r.x[:, :d], "messages": [tr.msg[tr.cur][:, :tr.d] for tr in r.trees],
           "counts": [tr.counts[:tr.E] for tr in r.trees]}
    if case["entry"] == "steps":  # the messages of the iteration before the last
        out["before"] = [tr.msg[1 - tr.cur][:, :tr.d] for tr in r.trees]
    if r.state:
        out["state"] = [s[:, :d] for s in r.state]
    if case["algo"] == "dme":
        out["received"] = [tr.dme_count for tr in r.trees]
    return out


# ---------------------------------------------------------- work, tolerance


def work(case):
    """Bytes: each array that the call needs read once, each that it leaves written once, 4 bytes a value
    (a message that arrives at a worker with one neighbour is written and never read again).  Operations per
    worker-coordinate and iteration: about 25 integer ones for a quarter of a Philox block, 10 for
    Box-Muller, 6 for the local step (14 with Adam) and 3 for each message."""
    n, d, k = case["n"], case["d"], case["k"]
    E = 2 * (n - 1)
    trees = _edges(case["tree"], n)
    leaves = sum(int((np.bincount(np.asarray(t).ravel(), minlength=n) == 1).sum()) for t in trees) / len(trees)
    centres = {"identity": n, "dirichlet": CENTRES}[case["mix"]] if case["objective"] == "generated" else 0
    mixed = 2 * n * CENTRES if case["mix"] == "dirichlet" and centres else 0
    if case["entry"] == "metrics":
        return {"bytes": 4.0 * d * (n + (0 if centres else n)), "flops": d * (8.0 * n + 35 * centres + mixed)}
    slots = {"sgd": 0, "nesterov": 1, "adam": 2}[case["opt"]]
    rows = 2 * n + (0 if centres else n) + 2 * slots * n + (E - leaves) + E * (2 if case["entry"] == "steps" else 1)
    step = n * (35 + (14 if case["opt"] == "adam" else 6)) + 3 * E
    once = 35 * centres + mixed
    return {"bytes": 4.0 * d * rows, "flops": float(d) * (k * step + once)}


def tolerance(case):
    """32-bit sums and normals: up to 2.3e-7 off the 64-bit result was measured (100 iterations, Adam); the
    metrics are summed in 64 bits, 7e-16 off."""
    return {"rel": 1e-12} if case["entry"] == "metrics" else {"rel": 1e-6}


# ------------------------------------------------------------------- exact

_M0, _M1, _W0, _W1 = 0xD2511F53, 0xCD9E8D57, 0x9E3779B9, 0xBB67AE85
_LOW = 0xFFFFFFFF


def _normals(quads, rows, step, stream, key):
    """Philox4x32-10 (Salmon et al., SC'11) at counters (quad, row, step, stream), and Box-Muller in 64 bits
    on u = ((word >> 8) + 1) 2^-24: normals [rows][4 * quads]."""
    q, r = torch.meshgrid(quads, rows, indexing="xy")  # [rows][quads]
    c = [q, r, torch.full_like(q, step), torch.full_like(q, stream)]
    k0, k1 = key & _LOW, (key >> 32) & _LOW
    for _ in range(10):
        p0, p1 = c[0] * _M0, c[2] * _M1  # 64-bit products that wrap; shift and mask give the halves
        c = [((p1 >> 32) & _LOW) ^ c[1] ^ k0, p1 & _LOW, ((p0 >> 32) & _LOW) ^ c[3] ^ k1, p0 & _LOW]
        k0, k1 = (k0 + _W0) & _LOW, (k1 + _W1) & _LOW
    u = [((w >> 8) + 1).double() * 2.0 ** -24 for w in c]
    z = []
    for a, b in ((u[0], u[1]), (u[2], u[3])):
        rad = (-2.0 * a.log()).sqrt()
        z += [rad * (2 * math.pi * b).cos(), rad * (2 * math.pi * b).sin()]
    return torch.stack(z, dim=-1).reshape(len(rows), -1)


def _f(v):
    return float(np.float32(v))  # what a 32-bit argument holds


def _centres(case, quads, seed):
    """The generated centres in 64 bits, [n][4 * quads]."""
    mix = torch.from_numpy(_mix(case).astype(np.float64)).to(quads.device)
    rows = torch.arange(mix.shape[1], device=quads.device)
    return MU_SCALE * (mix @ _normals(quads, rows, 0, 1, seed + 1))


def _exact_window(case, seed, k, lo, hi, x, mu, state, m, c):
    """k iterations on the columns [lo, hi) of tree k's window, in 64 bits, in place; returns the messages of
    the last two iterations, the counters and the models received."""
    n, algo, opt = case["n"], case["algo"], case["opt"]
    src, dst = _directed(_edges(case["tree"], n)[k])
    lost = _lost(case, seed, k)
    lr, sigma, b1, b2, eps = (_f(v) for v in (case["lr"], case["sigma"], BETA1, BETA2, EPS))
    dev = x.device
    quads = torch.arange(lo // 4, (hi + 3) // 4, device=dev)
    rows = torch.arange(n, device=dev)
    if mu is None:
        mu = _centres(case, quads, seed)[:, :hi - lo]
    s_src, s_dst = torch.from_numpy(src).to(dev), torch.from_numpy(dst).to(dev)
    rev = torch.arange(len(src), device=dev) ^ 1
    received = np.zeros(n, np.int64)
    before = m
    for j in range(case["k"]):
        xi = _normals(quads, rows, T0 + j, 0, seed)[:, :hi - lo]
        c = _next_counts(src, dst, n, c, lost)
        nbar = np.ones(n, np.int64)
        np.add.at(nbar, dst, c)
        received += nbar
        if algo == "dme":
            rel = mu + sigma * xi
        else:
            g = (x - mu) + sigma * xi
            if opt == "sgd":
                u = -lr * g
            elif opt == "nesterov":
                state[0] = b1 * state[0] + g
                u = -lr * (g + b1 * state[0])
            else:
                t = T0 + j + 1
                state[0] = b1 * state[0] + (1 - b1) * g
                state[1] = b2 * state[1] + (1 - b2) * g * g
                u = -lr / (1 - b1 ** t) * state[0] / (state[1].sqrt() / math.sqrt(1 - b2 ** t) + eps)
            rel = u if algo == "grad" else x + u
        arriving = torch.zeros_like(x).index_add_(0, s_dst, m)
        before, m = m, rel[s_src] + arriving[s_src] - m[rev]
        if lost is not None:
            m[torch.from_numpy(np.flatnonzero(lost)).to(dev)] = 0.0
        total = torch.zeros_like(x).index_add_(0, s_dst, m)
        nb = torch.from_numpy(nbar).to(dev).double()[:, None]
        if algo == "grad":
            x = x + (rel + total) / n
        elif algo == "dme":
            x = x + rel + total
        elif case["mode"] == 0:
            x = (rel + total) / nb
        else:
            x = (rel + total + (n - nb) * x) / n
    return x, state, m, before, c, received


def exact(case, seed):
    n, d = case["n"], case["d"]
    trees, windows = _edges(case["tree"], n), _windows(case)
    E = 2 * (n - 1)
    if n * d > 2e9:
        return None  # over 20 seconds in 64 bits
    host = case["entry"] == "host"
    x = torch.zeros(n, d, device=DEV)
    mu = torch.zeros(n, d, device=DEV) if case["objective"] == "stored" else None
    state = [torch.zeros(n, d, device=DEV) for _ in range({"sgd": 0, "nesterov": 1, "adam": 2}[case["opt"]])]
    rows = [E + len(_wide(t, n)) for t in trees]
    msgs = [torch.zeros(r, w, device=DEV) for r, (_, w) in zip(rows, windows)]
    _fill(case, seed, x, mu, state, msgs)
    part = max(4, int(1.5e8 / (n * (3 if case["entry"] == "metrics" else 4))) // 4 * 4)
    if case["entry"] == "metrics":
        out = torch.zeros(len(trees), 2, dtype=torch.float64, device=DEV)
        for k, (col, w) in enumerate(windows):
            for lo in range(col, col + w, part):
                hi = min(lo + part, col + w)
                xs = x[:, lo:hi].double()
                cs = (mu[:, lo:hi].double() if mu is not None else
                      _centres(case, torch.arange(lo // 4, (hi + 3) // 4, device=DEV), seed)[:, :hi - lo])
                mean = xs.mean(0)
                out[k, 0] += (xs - mean).square().sum() / (n * w)
                out[k, 1] += (mean - cs.mean(0)).square().sum() / w
        return out
    f64 = dict(dtype=torch.float64, device=DEV)
    new_x, new_state = torch.empty(n, d, **f64), [torch.empty(n, d, **f64) for _ in state]
    out = {"x": new_x, "messages": [], "counts": []}
    befores, received = [], []
    for k, ((col, w), edges) in enumerate(zip(windows, trees)):
        new, bef = torch.empty(rows[k], w, **f64), torch.empty(rows[k], w, **f64)
        src, dst = _directed(edges)
        c, got = _steady(edges, n), np.zeros(n, np.int64)
        for lo in range(col, col + w, part):
            hi = min(lo + part, col + w)
            cut = [t[:, lo:hi].double() for t in state]
            xs, st, ms, bs, c, got = _exact_window(
                case, seed, k, lo, hi, x[:, lo:hi].double(), None if mu is None else mu[:, lo:hi].double(), cut,
                msgs[k][:E, lo - col:hi - col].double(), _steady(edges, n))
            new_x[:, lo:hi] = xs
            for a, b in zip(new_state, st):
                a[:, lo:hi] = b
            for a, b in ((new, ms), (bef, bs)):
                a[:E, lo - col:hi - col] = b
                for r, i in enumerate(_wide(edges, n)):
                    a[E + r, lo - col:hi - col] = b[torch.from_numpy(np.flatnonzero(dst == i)).to(DEV)].sum(0)
        out["messages"].append(new)
        out["counts"].append(torch.from_numpy(c).to(torch.int32))
        befores.append(bef)
        received.append(torch.from_numpy(got))
    if case["entry"] == "steps":
        out["before"] = befores
    if state:
        out["state"] = new_state
    if case["algo"] == "dme":
        out["received"] = received
    return out
