"""The calls whose speed counts, as a program that uses this library makes them.

listed() gives a fixed set over the real range, draw() more of the same ranges.  A case names its kind:

  sweep   PTHandle.sweep + state      stepping runs and reading them back (with or without walk statistics)
  tts     PTHandle.tts_eval           one PT-TTS evaluation of one instance
  many    PTHandle.tts_eval_many      candidates of an engineering step, evaluated in one batch
  rao     engineer_begin + engineer_run   an RAO loop (Algorithm 1)
  lao     lao_begin + lao_run         an LAO loop on a planted instance (Algorithm 2)
  batch   PTBatch.reset + run + tts   many instances of uneven size and temperature count
  rank    Surrogate.forward           predictions that rank an engineering step's proposals
  grad    Surrogate.grad              loss and gradient of a training batch

Sizes: C_L with L = 1..16, N_T = 2..64 temperatures, R = 1..1024 runs; beta ladders are geometric.  Handles and
batches keep the library's own schedule unless `tuned` is set, where the program tunes it once as bench.py does
(a single instance with an odd L above 5, or L = 14, has to be tuned or given a mapping).
"""
import math

import numpy as np
import torch

import paper_1605_03607_gb300 as P

# integer operations of one spin-flip attempt: a quarter of a Philox4x32-10 call (15), the local field (6),
# the spin's sign (1), the acceptance test (5), the updates (3) and the spin loads and store (1.25)
OPS_PER_ATTEMPT = 31.25
HIDDEN, LAYERS = 64, 4


def listed():
    return [
        # a monitored run of the tiny configuration: ten sweeps and one exchange, then a look at the state
        dict(name="step_c4", kind="sweep", L=4, NT=16, R=8, sweeps=10, x=10, walk=False, tuned=False, lo=0.1,
             hi=3.0),
        # the tiny configuration's evaluation, 8 runs of 2048 sweeps
        dict(name="tts_c4", kind="tts", L=4, NT=16, R=8, S=2048, mult=1, x=1, tuned=False, lo=0.1, hi=3.0),
        # the tiny configuration's loop: 20 RAO steps, four candidates at a time
        dict(name="rao_c4", kind="rao", L=4, NT=16, R=8, S=1024, mult=1, x=1, steps=20, spec=4, tuned=False, lo=0.1,
             hi=3.0),
        # one C_8 instance with the 4x target pass and 64 runs (an engineering loop's starting point)
        dict(name="tts_c8", kind="tts", L=8, NT=32, R=64, S=1024, mult=4, x=1, tuned=False, lo=0.1, hi=4.0),
        # the C_8 loop's speculative batch: 16 candidates of 64 runs, schedule tuned once
        dict(name="many_c8", kind="many", L=8, NT=32, R=64, k=16, S=512, mult=4, top=0, x=1, tuned=True, lo=0.1, hi=4.0),
        # the C_16 loop's step: the 4 best-ranked candidates of 32 runs under the doubling budget
        dict(name="many_c16", kind="many", L=16, NT=48, R=32, k=4, S=256, mult=1, top=1024, x=1, tuned=False, lo=0.05,
             hi=5.0),
        # odd sizes: mixing of an instance without a round size, walk statistics on, exchange every 10 sweeps
        dict(name="walk_c7", kind="sweep", L=7, NT=30, R=100, sweeps=1000, x=10, walk=True, tuned=True, lo=0.1,
             hi=4.0),
        # a planted C_8 instance: 16 LAO steps evaluated together (couplers above 3, longer threshold tables)
        dict(name="lao_c8", kind="lao", L=8, NT=32, R=64, S=1024, x=1, loops=350, wmax=5, steps=16, spec=16,
             tuned=False, lo=0.1, hi=4.0),
        # 256 instances over C_4, C_8, C_12, C_16 with 24..48 temperatures, tuned once
        dict(name="batch_256", kind="batch", n=256, Lmin=4, Lstep=4, Ls=4, NTmin=24, NTspan=25, R=32, sweeps=64, x=1,
             tuned=True, lo=0.1, hi=4.0),
        # ranking the 64 proposals of a guided step on C_8
        dict(name="rank_c8", kind="rank", L=8, B=64),
        # a training batch: 256 C_8 graphs
        dict(name="grad_c8", kind="grad", L=8, B=256),
        # a training batch of the online loop: 64 evaluated candidates and the 64 instances they were drawn from, on C_4
        dict(name="grad_c4", kind="grad", L=4, B=128),
    ]


def _log_int(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["tts", "tts", "many", "many", "sweep", "sweep", "batch", "rao", "lao", "rank", "grad"])
    if kind in ("rank", "grad"):
        L = rng.randint(2, 16)
        most = 256 * 64 // (L * L)              # no more nodes than the largest listed batch
        B = max(2, min(1024, _log_int(rng, 8, max(9, most))))
        return dict(kind=kind, L=L, B=B)
    ladder = dict(lo=round(rng.uniform(0.05, 0.2), 3), hi=round(rng.uniform(2.0, 5.0), 2))
    if kind == "batch":
        step, Ls = rng.choice([(1, 5), (2, 4), (3, 3), (4, 4)])
        Lmin = rng.randint(2, 16 - step * (Ls - 1))
        n = _log_int(rng, 12, 256)
        return dict(kind=kind, n=n, Lmin=Lmin, Lstep=step, Ls=Ls, NTmin=rng.randint(8, 24), NTspan=rng.randint(1, 25),
                    R=_log_int(rng, 2, 32), sweeps=_log_int(rng, 16, 64), x=rng.choice([1, 1, 2, 10]),
                    tuned=rng.random() < 0.5, **ladder)
    L = rng.choice([2, 3, 4, 4, 5, 6, 7, 8, 8, 8, 9, 10, 11, 12, 13, 14, 15, 16, 16])
    NT = rng.randint(4, 64)
    tuned = L in (7, 9, 11, 13, 14, 15) or rng.random() < 0.25
    if kind in ("rao", "lao"):
        L = min(L, 10)
        NT = min(NT, 40)
        c = dict(kind=kind, L=L, NT=NT, R=_log_int(rng, 4, 64), S=_log_int(rng, 128, 1024), x=rng.choice([1, 1, 2]),
                 tuned=tuned, steps=rng.randint(4, 20), spec=rng.choice([1, 4, 16]), **ladder)
        per = 8 * L * L * NT * c["R"] * c["spec"] * c["steps"]    # at most a batch for every step
        if kind == "rao":
            c["mult"] = rng.choice([1, 4])
        c["S"] = max(16, min(c["S"], int(3.2e10 / (per * c.get("mult", 1)))))
        if kind == "rao":
            return c
        return dict(c, loops=max(4, int(5.5 * L * L)), wmax=rng.choice([3, 5]))
    k = rng.randint(2, 16) if kind == "many" else 1
    spins = 8 * L * L * NT * k                   # attempts of one sweep of one run of every instance
    R = _log_int(rng, 1, 1024 if kind == "sweep" else 128)
    R = max(1, min(R, int((1.2e7 if kind == "sweep" else 2e8) / spins)))
    most = max(64, min(4096, int(1.5e10 / (spins * R))))
    total = _log_int(rng, 16 if kind == "sweep" else 64, most)
    if kind == "sweep":
        return dict(kind=kind, L=L, NT=NT, R=R, sweeps=total, x=rng.choice([1, 1, 3, 10]), walk=rng.random() < 0.3,
                    tuned=tuned, **ladder)
    mult = rng.choice([1, 4])
    c = dict(kind=kind, L=L, NT=NT, R=R, x=rng.choice([1, 1, 2]), tuned=tuned, **ladder)
    if kind == "tts":
        return dict(c, S=max(1, total // mult), mult=mult)
    if rng.random() < 0.5:
        return dict(c, k=k, S=max(1, total // mult), mult=mult, top=0)
    return dict(c, k=k, S=max(1, total // 4), mult=1, top=max(1, total // 4) * 4)


def _edges(L):
    return 16 * L * L + 8 * L * (L - 1)


def _couplers(rng, L, *lead):
    return np.array([-3, -2, -1, 1, 2, 3], np.int8)[rng.integers(0, 6, size=(*lead, _edges(L)))]


def _ladder(NT, lo, hi):
    return hi * np.power(lo / hi, np.arange(NT) / max(NT - 1, 1))


def _neighbours(rng, J, k):
    """k candidates of J, each with one coupler redrawn."""
    out = np.repeat(J[None, :], k, axis=0)
    for j in range(k):
        e = rng.integers(0, len(J))
        out[j, e] = rng.choice([v for v in (-3, -2, -1, 1, 2, 3) if v != J[e]])
    return out


def _params(rng):
    """Parameters as a training run starts with: weights uniform in +-1/sqrt(fan-in), embeddings in +-1, biases small.
    The layer matrices are BF16 values, as in a checkpoint of the weights that the network multiplies with."""
    out = []
    for name, shape in _shapes():
        if name in ("X", "Jt"):
            w = rng.uniform(-1, 1, shape)
        elif len(shape) == 2:
            w = rng.uniform(-1, 1, shape) / math.sqrt(shape[1])
        elif name == "w2":
            w = rng.uniform(-1, 1, shape) / math.sqrt(HIDDEN)
        elif name == "b2":
            w = np.full(shape, 3.0)
        else:
            w = rng.uniform(-0.05, 0.05, shape)
        w = torch.from_numpy(w).float()
        if name[:2] in ("Wm", "Wu", "We"):
            w = w.bfloat16().float()
        out.append(w.reshape(-1))
    return torch.cat(out).numpy()


def _shapes():
    H = HIDDEN
    s = [("X", (2, H)), ("Jt", (6, H))]
    for l in range(LAYERS):
        for n in ("m", "u", "e"):
            s += [("W%s%d" % (n, l), (H, 2 * H)), ("b%s%d" % (n, l), (H,))]
    return s + [("W1", (H, H)), ("b1", (H,)), ("w2", (H,)), ("b2", (1,))]


def _graphs(case, rng):
    """Graphs and targets of a surrogate case: proposals around one instance, or candidates and the instances they were
    drawn from, with their log10 TTS."""
    L, B = case["L"], case["B"]
    if case["kind"] == "rank":
        return _neighbours(rng, _couplers(rng, L), B), None
    base = _couplers(rng, L, (B + 1) // 2)
    cand = np.concatenate([_neighbours(rng, b, 1) for b in base])
    return np.concatenate([cand, base])[:B], rng.normal(3.0, 0.2, B).astype(np.float32)


def prepare(case, seed):
    rng = np.random.default_rng([int(seed), 20160511])
    kind = case["kind"]
    uid = int(rng.integers(0, 2 ** 31))
    if kind in ("rank", "grad"):
        J, t = _graphs(case, rng)
        m = P.Surrogate(hidden=HIDDEN, layers=LAYERS)
        m.set_params(_params(rng))
        return dict(case=case, m=m, J=J, t=t)
    if kind == "batch":
        inst = []
        for i in range(case["n"]):
            L = case["Lmin"] + case["Lstep"] * (i * case["Ls"] // case["n"])
            NT = case["NTmin"] + (7 * i) % case["NTspan"]
            inst.append(dict(L=L, J=_couplers(rng, L), betas=_ladder(NT, case["lo"], case["hi"]), uid=uid + i))
        b = P.PTBatch(inst, case["R"], seed=int(seed) & 0x7FFFFFFF)
        if case["tuned"]:
            b.autotune(trial_sweeps=8)
        return dict(case=case, b=b)
    L, betas = case["L"], _ladder(case["NT"], case["lo"], case["hi"])
    J = _couplers(rng, L)
    h = P.PTHandle(L, J, betas, case["R"], seed=int(seed) & 0x7FFFFFFF, uid=uid)
    s = dict(case=case, h=h, uid=uid)
    if kind == "many":
        s["Js"] = _neighbours(rng, J, case["k"])
        s["uids"] = uid + 1 + np.arange(case["k"])
    if case["tuned"]:
        h.autotune(n_inst=case.get("k", case.get("spec", 1)), trial_sweeps=32)
    if kind == "sweep" and case["walk"]:
        h.set_walk_stats(True)
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "sweep":
        h = state["h"]
        h.sweep(case["sweeps"], case["x"])
        out = h.state()
        if case["walk"]:
            out["hot"], out["trips"], out["passes"] = h.walk_stats()
        return {k: v.view(np.int64) if isinstance(v, np.ndarray) and v.dtype == np.uint64 else v for k, v in out.items()}
    if kind == "tts":
        return state["h"].tts_eval(state["uid"], case["S"], case["mult"], case["x"])
    if kind == "many":
        return state["h"].tts_eval_many(state["Js"], state["uids"], case["S"], case["mult"], case["top"], case["x"])
    if kind == "rao":
        h = state["h"]
        t0 = h.engineer_begin(case["S"], case["mult"], case["x"], base_uid=state["uid"])
        res = h.engineer_run(0, case["steps"], case["spec"])
        J = h.couplers()
        for i in reversed(np.nonzero(res["accepted"])[0]):       # back to the instance the loop started from
            h.set_coupler(res["edge"][i], res["old_value"][i])
        return dict(t0=t0, J=J, **res)
    if kind == "lao":
        h = state["h"]
        t0 = h.lao_begin(case["S"], state["uid"], case["loops"], case["wmax"], case["x"])
        res = h.lao_run(1, case["steps"], case["spec"])
        return dict(t0=t0, **res, **{"now_" + k: v for k, v in h.lao_state().items()})
    if kind == "batch":
        b = state["b"]
        b.reset()
        b.run(case["sweeps"], case["x"])
        return b.tts(case["sweeps"])
    m, L, J, t = state["m"], case["L"], state["J"], state["t"]
    if kind == "rank":
        return m.forward(L, J)
    return m.grad(L, J, t)


def _attempts(case):
    if case["kind"] == "batch":
        n = 0
        for i in range(case["n"]):
            L = case["Lmin"] + case["Lstep"] * (i * case["Ls"] // case["n"])
            n += 8 * L * L * (case["NTmin"] + (7 * i) % case["NTspan"]) * case["R"]
        return n * case["sweeps"], n
    per = 8 * case["L"] ** 2 * case["NT"] * case["R"]
    if case["kind"] == "sweep":
        return per * case["sweeps"], per
    if case["kind"] == "tts":
        return per * case["S"] * case["mult"], per
    if case["kind"] == "many":                   # the doubling budget's last level is the most that it can take
        return per * case["k"] * (case["top"] or case["S"] * case["mult"]), per * case["k"]
    evals = 1 + case["steps"]                    # the start and one candidate a step
    return per * evals * case["S"] * case.get("mult", 1), per * case["spec"]


def work(case):
    if case["kind"] not in ("rank", "grad"):
        attempts, spins = _attempts(case)
        return dict(bytes=spins * (2 if case["kind"] == "sweep" else 1), flops=OPS_PER_ATTEMPT * attempts)
    L, B = case["L"], case["B"]
    N, E = 8 * L * L, _edges(L)
    gemm = 2 * (2 * HIDDEN) * HIDDEN * LAYERS * B * (2 * E + N + E)
    params = 4 * sum(int(np.prod(s)) for _, s in _shapes())
    passes = {"rank": 1, "grad": 3}[case["kind"]]
    # the couplers and parameters; a gradient also keeps every layer's node and edge rows (BF16) for the backward
    keep = 0 if case["kind"] == "rank" else 2 * 2 * HIDDEN * LAYERS * B * (N + E) + params
    return dict(bytes=B * E + 4 * B + params + keep, flops=gemm * passes)


def exact(case, seed):
    """The surrogate's outputs in 64 bits; the Monte Carlo's are whole numbers."""
    if case["kind"] not in ("rank", "grad"):
        return None
    rng = np.random.default_rng([int(seed), 20160511])
    rng.integers(0, 2 ** 31)
    J, t = _graphs(case, rng)
    theta = torch.from_numpy(_params(rng)).double().cuda().requires_grad_(case["kind"] != "rank")
    L, B = case["L"], case["B"]
    y = _net(theta, L, torch.from_numpy(J).cuda())
    if case["kind"] == "rank":
        return y.detach()
    loss = ((y - torch.from_numpy(t).double().cuda()) ** 2).mean()
    loss.backward()
    return float(loss.detach()), theta.grad


def _topology(L):
    """Endpoints of C_L's couplers in the library's order: in-cell, vertical, horizontal."""
    ei, ej = [], []
    at = lambda r, c, u, k: 8 * (r * L + c) + 4 * u + k  # noqa: E731
    for r in range(L):
        for c in range(L):
            for k in range(4):
                for q in range(4):
                    ei.append(at(r, c, 0, k))
                    ej.append(at(r, c, 1, q))
    for r in range(L - 1):
        for c in range(L):
            for k in range(4):
                ei.append(at(r, c, 0, k))
                ej.append(at(r + 1, c, 0, k))
    for r in range(L):
        for c in range(L - 1):
            for k in range(4):
                ei.append(at(r, c, 1, k))
                ej.append(at(r, c + 1, 1, k))
    return torch.tensor(ei).cuda(), torch.tensor(ej).cuda()


def _net(theta, L, J):
    """Predictions of the message-passing network (include/pt.h) for the coupler vectors J [B, E]."""
    p, o = {}, 0
    for name, shape in _shapes():
        n = int(np.prod(shape))
        p[name] = theta[o:o + n].reshape(shape)
        o += n
    B, N = J.shape[0], 8 * L * L
    ei, ej = _topology(L)
    u = (torch.arange(N, device="cuda") >> 2) & 1
    j = J.long()
    h = p["X"][u].expand(B, N, HIDDEN)
    e = p["Jt"][torch.where(j < 0, j + 3, j + 2)]
    lin = lambda n, a, b: torch.relu(a @ p["W" + n][:, :HIDDEN].T + b @ p["W" + n][:, HIDDEN:].T + p["b" + n])  # noqa: E731
    for l in range(LAYERS):
        m = torch.zeros(B, N, HIDDEN, dtype=torch.float64, device="cuda")
        m = m.index_add(1, ei, lin("m%d" % l, h[:, ej], e)).index_add(1, ej, lin("m%d" % l, h[:, ei], e))
        h = h + lin("u%d" % l, h, m)
        e = e + lin("e%d" % l, e, h[:, ei] + h[:, ej])
    g = h.mean(1)
    return torch.relu(g @ p["W1"].T + p["b1"]) @ p["w2"] + p["b2"]
