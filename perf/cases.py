"""The framework's work as its users run it, one pass per case, through the
public binding (paper_2407_11523_gb300).

  decode       syndromes on the device -> estimates, convergence flags and
               iteration counts (decode; parallel or serial schedule)
  host         the same from page-locked host buffers (decode_host)
  montecarlo   one point of a logical-error-rate curve: sample errors and
               syndromes, decode, classify the residuals
  batch        a planned launch over many codes and channels (BatchPlan)
  serve        a burst of single-shot requests through the slot server
  train        loss and gradients of an unrolled decoder (unrolled_loss)
"""
import math

import numpy as np
import torch

import paper_2407_11523_gb300 as bpq

# Ten of the mixed-size workload's codes (bench.py --workload mixed).
MIXED = [("planar", 5), ("toric", 8), ("xzzx", 7), ("planar", 25), ("toric", 12), ("xzzx", 11), ("planar", 9),
         ("toric", 16), ("xzzx", 15), ("planar", 17)]
SERVED = [(k, d) for k in ("planar", "xzzx") for d in (5, 7, 9, 11, 13)]


def listed():
    return [
        # one syndrome at a time, as a real-time decoder gets them: latency and launches
        {"name": "one_shot_toric15", "kind": "decode", "code": "toric", "d": 15, "p": 0.08, "eta": 0.5,
         "variant": "ewainit", "schedule": "parallel", "shots": 1, "max_iter": 100},
        # a small batch (a few syndromes per SM) of a small code, Momentum-BP
        {"name": "small_momentum_planar9", "kind": "decode", "code": "planar", "d": 9, "p": 0.05, "eta": 0.5,
         "variant": "momentum", "schedule": "parallel", "shots": 1000, "max_iter": 50},
        # the headline: one p of the toric d = 15 sweep, 10^6 shots
        {"name": "sweep_toric15", "kind": "decode", "code": "toric", "d": 15, "p": 0.08, "eta": 0.5,
         "variant": "ewainit", "schedule": "parallel", "shots": 1000000, "max_iter": 100},
        # plain BP, the comparison decoder of every experiment, on a large planar code; odd shot count
        {"name": "plain_planar25", "kind": "decode", "code": "planar", "d": 25, "p": 0.06, "eta": 0.5,
         "variant": "plain", "schedule": "parallel", "shots": 30001, "max_iter": 100},
        # AdaGrad-BP on the XZZX code under Z-biased noise
        {"name": "adagrad_xzzx7", "kind": "decode", "code": "xzzx", "d": 7, "p": 0.06, "eta": 10.0,
         "variant": "adagrad", "schedule": "parallel", "shots": 200000, "max_iter": 100},
        # Algorithm 1's serial schedule, one point of the schedule comparison
        {"name": "serial_toric15", "kind": "decode", "code": "toric", "d": 15, "p": 0.04, "eta": 0.5,
         "variant": "ewainit", "schedule": "serial", "shots": 100000, "max_iter": 100},
        # Appendix C's adaptive decoder, one point of its comparison
        {"name": "aewa_planar11", "kind": "decode", "code": "planar", "d": 11, "p": 0.06, "eta": 0.5,
         "variant": "aewa", "schedule": "parallel", "shots": 100000, "max_iter": 100},
        # syndromes that arrive in host memory, copies included
        {"name": "host_toric15", "kind": "host", "code": "toric", "d": 15, "p": 0.06, "eta": 0.5,
         "variant": "ewainit", "shots": 262144, "max_iter": 100},
        # a logical-error-rate point: sampling and classification beside the decode
        {"name": "montecarlo_planar7", "kind": "montecarlo", "code": "planar", "d": 7, "p": 0.05, "eta": 0.5,
         "variant": "ewainit", "shots": 1000000, "max_iter": 100},
        # ten codes x two channels with uneven shot counts in one planned launch
        {"name": "batch_mixed20", "kind": "batch", "codes": 10, "p": 0.06, "variant": "ewainit", "shots": 262144,
         "max_iter": 100},
        # a burst of single-shot requests over ten codes
        {"name": "serve_burst", "kind": "serve", "codes": 10, "p": 0.05, "variant": "ewainit", "shots": 4096,
         "max_iter": 100},
        # a training step of the unrolled decoder: loss and gradients of every parameter
        {"name": "train_planar9", "kind": "train", "d": 9, "T": 25, "every": 5, "model": "momentum", "loss": "coset",
         "shots": 4096},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "decode", "host", "montecarlo", "batch", "serve", "train",
                       "train"])
    p = round(math.exp(rng.uniform(math.log(0.02), math.log(0.12))), 4)
    if kind == "train":
        # The unrolled EWAInit decoder's gradients are ill-conditioned over many iterations (in 32 bits 1e-4 off at
        # T = 25) and under the coset loss (its probabilities get tiny): it is drawn with the posterior loss, T <= 10.
        model = rng.choice(["ewainit", "momentum"])
        return {"kind": kind, "d": rng.randint(3, 11), "T": rng.randint(4, 25 if model == "momentum" else 10),
                "every": rng.randint(3, 6), "model": model,
                "loss": rng.choice(["coset", "posterior"]) if model == "momentum" else "posterior",
                "shots": _log_int(rng, 32, 4096)}
    if kind == "batch":
        return {"kind": kind, "codes": rng.randint(2, 10), "p": p, "variant": rng.choice(["plain", "momentum",
                "adagrad", "ewainit"]), "shots": _log_int(rng, 1024, 262144), "max_iter": rng.choice([50, 100])}
    if kind == "serve":
        return {"kind": kind, "codes": rng.randint(1, 10), "p": min(p, 0.06), "variant": "ewainit",
                "shots": _log_int(rng, 64, 4096), "max_iter": rng.choice([50, 100])}
    code = rng.choice(["planar", "toric", "xzzx"])
    d = rng.randint(3, 25 if kind == "decode" else 15)
    nodes = _nodes(code, d)
    case = {"kind": kind, "code": code, "d": d, "p": p, "eta": rng.choice([0.5, 0.5, 2.0, 10.0]),
            "variant": rng.choice(["plain", "momentum", "adagrad", "ewainit"]),
            # as much work as the largest listed cases of the kind at most
            "shots": _log_int(rng, 1 if kind == "decode" else 1000, min(1000000, 60000000 // nodes)),
            "max_iter": rng.choice([50, 100])}
    if kind == "decode":
        case["schedule"] = rng.choice(["parallel", "parallel", "serial"])
        if case["schedule"] == "parallel" and rng.random() < 0.15:
            case["variant"], case["shots"] = "aewa", min(case["shots"], 20000000 // nodes)
        if case["schedule"] == "serial":
            case["shots"] = min(case["shots"], 30000000 // nodes)
    return case


def _nodes(code, d):
    return 2 * d * d if code == "toric" else 2 * d * d - 2 * d + 1


def _channel(p, eta):
    """Pauli probabilities of total rate p and bias eta = p_z / (p_x + p_y); eta = 0.5 is depolarising."""
    return (p / (2 * (1 + eta)), p / (2 * (1 + eta)), p * eta / (1 + eta))


def _buffers(shots, n, pinned=False):
    where = {"pin_memory": True} if pinned else {"device": "cuda"}
    return (torch.empty((shots, n), dtype=torch.uint8, **where), torch.empty(shots, dtype=torch.uint8, **where),
            torch.empty(shots, dtype=torch.uint8, **where))


def _split(total, parts, rng):
    """Uneven shot counts, as a user's mix of codes has them."""
    return [int(n) for n in rng.multinomial(total, rng.dirichlet(np.ones(parts)))]


def prepare(case, seed):
    kind, B = case["kind"], case["shots"]
    if kind == "train":
        return _prepare_train(case, seed)
    params = bpq.make_params(case["variant"])
    rng = np.random.default_rng(seed)
    if kind == "batch":
        channels = [_channel(case["p"], 0.5), _channel(case["p"], 10.0)]
        counts = _split(B, 2 * case["codes"], np.random.default_rng(7))
        items = []
        for k, (code, d) in enumerate(MIXED[:case["codes"]]):
            t = bpq.Tanner(code, d).upload()
            for c, ch in enumerate(channels):
                _, syn = bpq.sample(t, *ch, seed=seed + 1000 * (2 * k + c), shot0=0, B=counts[2 * k + c])
                items.append((t, syn, bpq.prior_tensor(t, *ch)))
        return {"kind": kind, "plan": bpq.BatchPlan(items, case["variant"], params=params,
                                                    max_iter=case["max_iter"])}
    if kind == "serve":
        ch = _channel(case["p"], 0.5)
        codes = [bpq.Tanner(c, d).upload() for c, d in SERVED[:case["codes"]]]
        code = rng.permutation(np.arange(B) % len(codes))
        pool = []
        for k, t in enumerate(codes):
            _, syn = bpq.sample(t, *ch, seed=seed + 1000 * k, shot0=0, B=B)
            pool.append(syn.cpu().numpy().view(np.uint32))
        return {"kind": kind, "code": code, "arrival": np.zeros(B), "syn": [pool[c][r] for r, c in enumerate(code)],
                "server": bpq.Server(codes, [bpq.prior_tensor(t, *ch) for t in codes], case["variant"],
                                     params=params, max_iter=case["max_iter"], mode="slots", slots_per_code=1024)}
    t = bpq.Tanner(case["code"], case["d"]).upload()
    ch = _channel(case["p"], case["eta"])
    prior = bpq.prior_tensor(t, *ch)
    state = {"kind": kind, "t": t, "prior": prior, "variant": case["variant"], "params": params,
             "max_iter": case["max_iter"], "schedule": case.get("schedule", "parallel")}
    err, syn = bpq.sample(t, *ch, seed=seed, shot0=0, B=B)
    if kind == "host":
        state.update(syn=syn.cpu().pin_memory(), prior=prior.cpu().pin_memory(), out=_buffers(B, t.N, pinned=True),
                     buf=torch.empty(bpq.decode_host_bytes(t, B), dtype=torch.uint8, device="cuda"))
        return state
    state.update(syn=syn, out=_buffers(B, t.N), work=bpq.workspace())
    if kind == "montecarlo":
        state.update(ch=ch, seed=seed, shots=B, err=err, fail=torch.empty(B, dtype=torch.uint8, device="cuda"))
    return state


def run(s):
    kind = s["kind"]
    if kind == "decode":
        return bpq.decode(s["t"], s["syn"], s["prior"], s["variant"], params=s["params"], max_iter=s["max_iter"],
                          out=s["out"], work=s["work"], schedule=s["schedule"])
    if kind == "host":
        return bpq.decode_host(s["t"], s["syn"], s["prior"], s["variant"], params=s["params"],
                               max_iter=s["max_iter"], out=s["out"], dev_buf=s["buf"])
    if kind == "montecarlo":
        err, syn = bpq.sample(s["t"], *s["ch"], seed=s["seed"], shot0=0, B=s["shots"], err=s["err"], syn=s["syn"])
        est, conv, iters = bpq.decode(s["t"], syn, s["prior"], s["variant"], params=s["params"],
                                      max_iter=s["max_iter"], out=s["out"], work=s["work"])
        fail = bpq.check_logical(s["t"], err, est, out=s["fail"])
        return err, syn, est, conv, iters, fail
    if kind == "batch":
        return s["plan"].run()
    if kind == "serve":
        ests, conv, iters, _, _ = s["server"].replay(s["code"], s["arrival"], s["syn"])
        return np.concatenate(ests), conv, iters
    leaves = [x for x in (s["alpha"], s["beta"], s["w"], s["gamma"]) if x is not None]
    loss = bpq.unrolled_loss(s["t"], s["syn"], s["err"], s["prior"], s["alpha"], s["beta"], s["w"], T=s["T"],
                             ckpt_every=s["every"], model=s["model"], gamma=s["gamma"], loss=s["loss"])
    grads = torch.autograd.grad(loss, leaves)
    return {"loss": loss.detach(), **dict(zip(("alpha", "beta", "w", "gamma"), grads))}


# ------------------------------------------------------------------ training inputs (no library code)

def _planar(d):
    """Check matrix (M, N) and logical operators (2, N) of the planar code as Pauli codes (0 I, 1 X, 2 Y, 3 Z):
    hypergraph product of two repetition codes, X checks first."""
    h = np.zeros((d - 1, d), dtype=np.uint8)
    for i in range(d - 1):
        h[i, i] = h[i, i + 1] = 1
    hx = np.concatenate([np.kron(h, np.eye(d, dtype=np.uint8)), np.kron(np.eye(d - 1, dtype=np.uint8), h.T)], 1)
    hz = np.concatenate([np.kron(np.eye(d, dtype=np.uint8), h), np.kron(h.T, np.eye(d - 1, dtype=np.uint8))], 1)
    H = np.concatenate([hx, 3 * hz], 0)
    L = np.zeros((2, H.shape[1]), dtype=np.uint8)
    L[0, :d] = 1
    L[1, 0:d * d:d] = 3
    return H, L


def _anti(a, b):
    return (a != 0) & (b != 0) & (a != b)


def _train_inputs(case, seed):
    """Errors, syndrome bits and parameters in numpy: error rates 0.03 .. 0.10 (the training workload's), parameters
    around the paper's, as a run has them after some steps."""
    rng = np.random.default_rng(seed)
    H, L = _planar(case["d"])
    B, T, N, E = case["shots"], case["T"], H.shape[1], int((H != 0).sum())
    p = np.linspace(0.03, 0.10, 8)[np.arange(B) % 8][:, None]
    u = rng.random((B, N))
    err = np.where(u < p / 3, 1, np.where(u < 2 * p / 3, 2, np.where(u < p, 3, 0))).astype(np.uint8)
    syn = np.stack([_anti(err, row[None, :]).sum(1) & 1 for row in H], 1).astype(np.uint8)
    par = {"alpha": 0.5 + 0.05 * rng.standard_normal(T), "beta": 0.05 * np.abs(rng.standard_normal(T)),
           "w": 1.0 + 0.05 * rng.standard_normal(E)}
    if case["model"] == "momentum":
        par["gamma"] = 0.2 + 0.05 * rng.standard_normal(T)
    return H, L, err, syn, {k: v.astype(np.float32) for k, v in par.items()}


TRAIN_RATE = float(np.linspace(0.03, 0.10, 8).mean())


def _prepare_train(case, seed):
    H, _, err, syn, par = _train_inputs(case, seed)
    t = bpq.Tanner("planar", case["d"]).upload()
    bits = np.zeros((syn.shape[0], t.W * 32), dtype=np.uint8)
    bits[:, :syn.shape[1]] = syn
    words = np.packbits(bits, axis=1, bitorder="little").view(np.uint32).view(np.int32)
    state = {"kind": "train", "t": t, "T": case["T"], "every": case["every"], "model": case["model"],
             "loss": case["loss"], "syn": torch.from_numpy(words.copy()).cuda(), "err": torch.from_numpy(err).cuda(),
             "prior": bpq.prior_tensor(t, *_channel(TRAIN_RATE, 0.5)), "gamma": None}
    for k, v in par.items():
        state[k] = torch.from_numpy(v).cuda().requires_grad_(True)
    return state


def exact(case, seed):
    """The training step in float64 torch and autograd; every other case returns whole numbers only."""
    if case["kind"] != "train":
        return None
    H, L, err, syn, par = _train_inputs(case, seed)
    dev, f64 = "cuda", torch.float64
    par = {k: torch.tensor(v, dtype=f64, device=dev, requires_grad=True) for k, v in par.items()}
    total, B = 0.0, err.shape[0]
    for b in range(0, B, 512):  # autograd keeps every iteration: in slices of the batch
        part = _unrolled(case, H, L, err[b:b + 512], syn[b:b + 512], par) * (min(512, B - b) / B)
        part.backward()
        total += float(part.detach())
    return {"loss": torch.tensor(total, dtype=f64), **{k: v.grad for k, v in par.items()}}


def _unrolled(case, H, L, err, syn, par, clip=30.0):
    dev, f64 = "cuda", torch.float64
    T, N = case["T"], H.shape[1]
    ii, jj = np.nonzero(H)
    E = ii.size
    anti = torch.tensor(np.stack([_anti(np.full(E, w), H[ii, jj]) for w in (1, 2, 3)], 1), dtype=f64, device=dev)
    others = np.full((E, 3), E)
    for e in range(E):
        o = [f for f in np.nonzero(ii == ii[e])[0] if f != e]
        others[e, :len(o)] = o
    others, var = torch.tensor(others, device=dev), torch.tensor(jj, device=dev)
    rate = np.float32(np.asarray(_channel(TRAIN_RATE, 0.5))).astype(np.float64)
    pi0 = torch.tensor(np.log((1 - rate.sum()) / rate), dtype=f64, device=dev).expand(len(err), N, 3)
    sign = torch.tensor(1.0 - 2.0 * syn[:, ii], dtype=f64, device=dev)

    def lam(q):  # ln (1 + e^-q_H) / (e^-q_a + e^-q_b), H the edge's Pauli
        z = torch.zeros_like(q[..., :1])
        neg = torch.cat([z, -q], -1)
        none = torch.full_like(neg, -math.inf)
        on = torch.cat([torch.zeros_like(anti[:, :1]), anti], 1).bool()
        return torch.logsumexp(torch.where(on, none, neg), -1) - torch.logsumexp(torch.where(on, neg, none), -1)

    def phi(x):
        return torch.log1p(2.0 / torch.expm1(x))

    m = lam(pi0[:, var]).clamp(-clip, clip)
    Q, g, Qs = pi0, torch.zeros_like(pi0), []
    for t in range(T):
        mag = torch.cat([phi(m.abs()), torch.zeros_like(m[:, :1])], 1)
        sgn = torch.cat([torch.sign(m), torch.ones_like(m[:, :1])], 1)
        c = (par["w"] * sign * sgn[:, others].prod(-1) * phi(mag[:, others].sum(-1))).clamp(-clip, clip)
        S = torch.zeros_like(pi0).index_add(1, var, c[..., None] * anti)
        if case["model"] == "momentum":
            g = par["gamma"][t] * g + (1 - par["gamma"][t]) * (Q - pi0 - S)
            Q = Q - par["alpha"][t] * g
        else:
            Q = (pi0 if t == 0 else par["alpha"][t] * pi0 + (1 - par["alpha"][t]) * Q) + S
        m = (1 - par["beta"][t]) * lam(Q[:, var] - c[..., None] * anti).clamp(-clip, clip) + par["beta"][t] * m
        Qs.append(Q)
    if case["loss"] == "posterior":
        logp = torch.log_softmax(torch.cat([torch.zeros_like(Q[..., :1]), -Q], -1), -1)
        return -logp.gather(-1, torch.tensor(err, dtype=torch.long, device=dev)[..., None]).mean()
    loss = 0.0
    for Q in Qs:
        pr = torch.softmax(torch.cat([torch.zeros_like(Q[..., :1]), -Q], -1), -1)
        for rows, target in ((H, syn), (L, np.stack([_anti(err, row[None, :]).sum(1) & 1 for row in L], 1))):
            width = int((rows != 0).sum(1).max())
            at, pauli = np.zeros((len(rows), width), dtype=np.int64), np.zeros((len(rows), width), dtype=np.int64)
            for r, row in enumerate(rows):
                on = np.nonzero(row)[0]
                at[r, :len(on)], pauli[r, :len(on)] = on, row[on]
            even, odd = 1.0, 0.0
            for k in range(width):
                a = torch.tensor(np.stack([_anti(np.full(len(rows), w), pauli[:, k]) for w in (0, 1, 2, 3)], 1),
                                 dtype=f64, device=dev)
                x = pr[:, torch.tensor(at[:, k], device=dev)]
                yes, no = (x * a).sum(-1), (x * (1 - a)).sum(-1)
                even, odd = even * no + odd * yes, even * yes + odd * no
            P = torch.where(torch.tensor(target, device=dev).bool(), odd, even)
            loss = loss - torch.log(P.clamp_min(1e-30)).mean(-1)
    return (loss / T).mean()


# ------------------------------------------------------------------ what a pass cannot do without

def _iterations(p, max_iter):
    """About the mean iterations per shot (toric d = 15, EWAInit-BP: 12 at p = 0.04, 22 at 0.08, over 90 at 0.16)."""
    return min(max_iter, 3 + 3800 * p * p)


def _decode_work(code, d, shots, p, max_iter, runs=1.0):
    n = _nodes(code, d)
    edges = (4 if code == "toric" else 4 * (1 - 1 / d)) * n
    # per edge and iteration about 20 operations, the transcendental ones counted once
    return {"bytes": shots * (n / 8 + n + 2) + 12 * n, "flops": shots * runs * _iterations(p, max_iter) * edges * 20}


def work(case):
    kind = case["kind"]
    if kind == "train":
        n = _nodes("planar", case["d"])
        edges = 4 * (1 - 1 / case["d"]) * n
        # forward and adjoint: about 100 operations per edge and iteration
        return {"bytes": case["shots"] * (n + n / 8) + 8 * (edges + 3 * case["T"]),
                "flops": case["shots"] * case["T"] * edges * 100}
    if kind in ("batch", "serve"):
        codes = (MIXED if kind == "batch" else SERVED)[:case["codes"]]
        total = {"bytes": 0.0, "flops": 0.0}
        for code, d in codes:
            for k, v in _decode_work(code, d, case["shots"] / len(codes), case["p"], case["max_iter"]).items():
                total[k] += v
        return total
    # AEWA-BP runs EWAInit-BP with eleven weights at most, most shots with one
    w = _decode_work(case["code"], case["d"], case["shots"], case["p"], case["max_iter"],
                     2.0 if case["variant"] == "aewa" else 1.0)
    if kind == "montecarlo":
        n = _nodes(case["code"], case["d"])
        # the errors written and read, the flag; Philox: about 60 operations per qubit
        w = {"bytes": w["bytes"] + case["shots"] * (2 * n + n / 8 + 1), "flops": w["flops"] + case["shots"] * n * 60}
    return w
