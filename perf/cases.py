"""The work that users of this library have it do, as measurable cases.

Every case goes through the public binding (``paper_2406_01821_gb300.rs``). Data and rule sets follow
the library's own workloads (``synth.py``, ``bench.py``): Gaussian classes, conditions that are pairs
with probability 0.2, thresholds at empirical quantiles; sizes span the ranges of the plain, ragged,
fine-tuning, evolution, serving and categorical workloads. The kinds:

  hard      exact counts of a population (rs_eval_hard), arrays on the device or on the host
  preds     the same with every set's predictions, on a stream of the caller's own
  soft      sigmoid-relaxed loss and its adjoint (rs_eval_soft_bwd): one gradient of fine-tuning
  autograd  the same through rs.rule_soft_loss(...).sum().backward()
  probs     soft forward with class probabilities
  evolve    generations of the device-resident evolution loop
  serve     requests of several runs submitted together and polled
  register  a dataset registered, one population evaluated on it, the dataset dropped

Fine-tuning inside evolution is stood for by ``soft`` and ``autograd``: its integer results would
turn on the last bits of the gradients.
"""
import math

import numpy as np
import torch

from paper_2406_01821_gb300 import rs, synth

TAU = 0.1


def _case(name, kind, **sizes):
    return dict(name=name, kind=kind, **sizes)


def listed():
    return [
        # the paper's experiment: 64 candidates on 569 x 30, counts and predictions, one blocking call
        _case("plain_preds", "preds", N=569, F=30, K=2, P=64, rlo=8, rhi=8, chi=3),
        # predictions of a mid-size population on a larger table (ensembles, error analysis)
        _case("preds_mid", "preds", N=100_000, F=64, K=5, P=200, rlo=1, rhi=32, chi=6),
        # a population that the caller's own evolution keeps in host arrays
        _case("hard_host", "hard", N=100_000, F=32, K=3, P=512, rlo=1, rhi=32, chi=6, host=True, ncat=0),
        # the headline workload: a ragged population on a million samples
        _case("hard_ragged", "hard", N=1 << 20, F=128, K=10, P=4096, rlo=1, rhi=64, chi=8, host=False, ncat=0),
        # wide tables: the upper part of the serving workload's feature range
        _case("hard_wide", "hard", N=150_001, F=233, K=7, P=600, rlo=1, rhi=64, chi=8, host=False, ncat=0),
        # a quarter of the features categorical
        _case("hard_categorical", "hard", N=262_144, F=128, K=10, P=1024, rlo=1, rhi=64, chi=8, host=False, ncat=32),
        # back-propagation fine-tuning of a whole population: one gradient
        _case("soft_tune", "soft", N=262_144, F=64, K=2, P=1024, rlo=32, rhi=32, chi=-4),
        # fine-tuning of the best few of an evolution run, through autograd
        _case("soft_few", "autograd", N=100_000, F=32, K=2, P=64, rlo=2, rhi=32, chi=6),
        # class probabilities of the candidates that a user looks at
        _case("soft_probs", "probs", N=20_000, F=30, K=3, P=48, rlo=3, rhi=24, chi=5),
        # generations of the device-resident loop at its full population
        _case("evolve", "evolve", N=100_000, F=32, K=2, P=10_000, rlo=1, rhi=32, chi=6, gens=10),
        # a server's mix: requests of uneven size over several resident datasets
        _case("serve_mix", "serve", nlo=500, nhi=300_000, flo=8, fhi=256, runs=16, requests=72, plo=16, phi=2048,
              rhi=64, chi=8),
        # a new dataset: registered from device memory, evaluated once, dropped
        _case("register", "register", N=300_007, F=96, K=4, P=100, rlo=1, rhi=16, chi=5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


HARD_MOST, SOFT_MOST = 3.0e11, 2.0e10      # nominal condition-samples of a drawn case


def draw(rng):
    kind = rng.choice(["preds", "preds", "hard", "hard", "hard", "hard", "soft", "autograd", "probs", "evolve",
                       "serve", "register"])
    if kind == "serve":
        return dict(kind=kind, nlo=500, nhi=_log(rng, 5_000, 300_000), flo=8, fhi=rng.choice([64, 160, 256]),
                    runs=rng.randint(4, 16), requests=rng.randint(16, 64), plo=16, phi=_log(rng, 128, 2048),
                    rhi=rng.randint(8, 64), chi=rng.randint(2, 8))
    if kind == "evolve":
        return dict(kind=kind, N=_log(rng, 2_000, 100_000), F=rng.randint(8, 64), K=rng.randint(2, 4),
                    P=_log(rng, 300, 8_000), rlo=1, rhi=rng.randint(8, 32), chi=rng.randint(2, 6),
                    gens=rng.randint(2, 10))
    K = rng.randint(2, 10)
    c = dict(kind=kind, N=_log(rng, 500, 1 << 20), F=rng.randint(8, 160), K=K, P=_log(rng, 16, 4096), rlo=1,
             rhi=rng.randint(8, 64), chi=rng.randint(2, 8))
    most = HARD_MOST
    if kind == "hard":
        form = rng.choice(["", "", "host", "cat", "wide"])
        c["host"], c["ncat"] = form == "host", 0
        if form == "wide":
            c["F"] = rng.randint(161, 256)
        if form == "cat":
            c["F"] = rng.randint(8, 128)
            c["ncat"] = max(1, c["F"] // rng.randint(2, 6))
    elif kind == "preds":
        c["P"] = _log(rng, 16, 512)
        while c["P"] * c["N"] > 40_000_000:
            c["N"] = max(500, c["N"] // 2 + rng.randint(0, 99))
    elif kind == "register":
        c["P"] = _log(rng, 16, 256)
    else:
        c["K"] = rng.randint(2, 4)
        c["rlo"], c["rhi"] = c["K"], rng.randint(8, 32)
        c["F"] = rng.randint(8, 128)
        c["N"], c["P"] = _log(rng, 500, 262_144), _log(rng, 16, 1024)
        most = SOFT_MOST
        if kind == "probs":
            c["N"], c["P"] = _log(rng, 500, 50_000), _log(rng, 4, 128)
    while _conds(c) * c["N"] > most:
        c["N"] = max(500, c["N"] // 2 + rng.randint(0, 99))
    return c


def _conds(c):
    """Expected number of conditions of the case's rule sets."""
    per_rule = -c["chi"] if c["chi"] < 0 else (1 + c["chi"]) / 2
    return c["P"] * (c["rlo"] + c["rhi"]) / 2 * per_rule


# ------------------------------------------------------------------------------------- inputs

def _gen(seed, *more):
    g = torch.Generator(device="cuda")
    s = seed & 0xFFFFFFFF
    for m in more:
        s = (s * 1_000_003 + m) & 0x7FFFFFFFFFFF
    g.manual_seed(s)
    return g


def _data(N, F, K, ncat, g):
    """Features and labels on the device: two classes 37/63 with a mean shift of 1, or a K-class
    Gaussian mixture; the last ncat features hold category codes 0..47 that depend on the class."""
    if K == 2:
        y = (torch.rand(N, generator=g, device="cuda") >= 0.37).to(torch.int32)
        mu = torch.stack([torch.zeros(F, device="cuda"), torch.ones(F, device="cuda")])
    else:
        y = torch.randint(0, K, (N,), generator=g, device="cuda", dtype=torch.int32)
        mu = torch.randn(K, F, generator=g, device="cuda")
    X = torch.randn(N, F, generator=g, device="cuda")
    X += mu[y.long()]
    if ncat:
        codes = torch.rand(N, ncat, generator=g, device="cuda") ** (0.5 + 0.3 * y[:, None].float())
        X[:, F - ncat:] = torch.floor(codes * 48).clamp_(0, 47)
    return X, y


def _rules(c, X, K, seed, P=None, default=None):
    m = min(len(X), 8192)
    qtab = torch.sort(X[:m], dim=0).values.t().contiguous().cpu().numpy()
    F = X.shape[1]
    ncat = c.get("ncat", 0)
    # the rule and condition counts belong to the case, so that outputs keep their shapes from seed to seed
    P = P or c["P"]
    form = synth.random_rulesets(qtab, K, P, (c["rlo"], c["rhi"]), -c["chi"] if c["chi"] < 0 else (1, c["chi"]),
                                 P * 131 + c["rhi"])
    b = synth.random_rulesets(qtab, K, 1, 1, form.C, seed, cat_from=F - ncat if ncat else None, n_codes=48)
    r = np.random.default_rng([seed, 5])
    b.set_rule_off, b.rule_cond_off = form.set_rule_off, form.rule_cond_off
    b.rule_class = r.integers(0, K, size=form.R, dtype=np.int32)
    b.set_default = r.integers(0, K, size=P, dtype=np.int32) if default is None else np.full(P, default, np.int32)
    if c["kind"] in ("soft", "autograd", "probs"):
        # every class has a path (a label without one has loss +inf): the first K rules name them all
        first = b.set_rule_off[:-1]
        for k in range(K):
            b.rule_class[first + k] = k
    return b


def _population(b, RMAX, CMAX):
    """The fixed-slot arrays of a batch (unused slots zero, cg -1)."""
    P = b.P
    rp, cr = np.diff(b.set_rule_off), np.diff(b.rule_cond_off)
    set_of_rule = np.repeat(np.arange(P), rp)
    r_in_set = np.arange(b.R) - np.repeat(b.set_rule_off[:-1], rp)
    at = np.repeat(set_of_rule, cr), np.repeat(r_in_set, cr), np.arange(b.C) - np.repeat(b.rule_cond_off[:-1], cr)
    pop = {"nrule": rp.astype(np.int32), "deflt": b.set_default.copy(), "rcls": np.zeros((P, RMAX), np.int32),
           "ncond": np.zeros((P, RMAX), np.int32)}
    pop["rcls"][set_of_rule, r_in_set] = b.rule_class
    pop["ncond"][set_of_rule, r_in_set] = cr
    for k, src, t, fill in (("cf", b.cond_f, np.int32, 0), ("cg", b.cond_g, np.int32, -1), ("cop", b.cond_op, np.int8, 0),
                            ("ca", b.cond_a, np.float32, 0), ("cb", b.cond_b, np.float32, 0),
                            ("ct", b.cond_t, np.float32, 0)):
        pop[k] = np.full((P, RMAX, CMAX), fill, t)
        pop[k][at] = src
    return pop


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"kind": kind, "ctx": rs.Context(0)}
    if kind == "serve":
        r = np.random.default_rng([c["runs"], c["requests"], c["nhi"]])        # the mix belongs to the case
        runs = []
        for i in range(c["runs"]):
            N = int(np.exp(r.uniform(np.log(c["nlo"]), np.log(c["nhi"]))))
            F, K = int(r.integers(c["flo"], c["fhi"] + 1)), int(r.integers(2, 11))
            X, y = _data(N, F, K, 0, _gen(seed, 3, i))
            runs.append((s["ctx"].dataset(X, y, K), K, X))
        s["requests"] = []
        for j in range(c["requests"]):
            ds, K, X = runs[j % len(runs)]
            P = int(np.exp(r.uniform(np.log(c["plo"]), np.log(c["phi"]))))
            b = _rules(dict(c, rlo=1), X, K, seed * 64 + j, P=P)
            s["requests"].append((ds, K, P, rs.HostBatch(b)))
        return s
    N, F, K = c["N"], c["F"], c["K"]
    X, y = _data(N, F, K, c.get("ncat", 0), _gen(seed, 1))
    default = None if kind == "hard" and K > 2 else int(torch.bincount(y, minlength=K).argmax())
    b = _rules(c, X, K, seed, default=default)
    s.update(N=N, K=K)
    if kind == "register":
        s.update(X=X, y=y, batch=rs.DeviceBatch.from_host(b))
        return s
    s["ds"] = s["ctx"].dataset(X, y, K)
    if kind == "evolve":
        s.update(pop=_population(b, c["rhi"], c["chi"]), gens=c["gens"], seed=seed, elite=max(1, c["P"] // 100))
    elif c.get("host"):
        s["batch"] = rs.HostBatch(b)
    else:
        s["batch"] = rs.DeviceBatch.from_host(b)
    if kind == "preds":
        s["stream"] = torch.cuda.Stream()
        i32 = dict(dtype=torch.int32, device="cuda")
        s["out"] = (torch.empty(b.P, **i32), torch.empty((b.P, K), **i32), torch.empty((b.P, N), **i32))
    elif kind == "soft":
        s["dloss"] = torch.rand(b.P, generator=_gen(seed, 2), device="cuda") + 0.5
    elif kind == "autograd":
        s["params"] = [s["batch"].t[k].clone().requires_grad_(True) for k in ("cond_a", "cond_b", "cond_t")]
    torch.cuda.synchronize()
    return s


def run(s):
    ctx, kind = s["ctx"], s["kind"]
    if kind == "hard":
        correct, per_class, _ = ctx.eval_hard(s["ds"], s["batch"], s["K"])
        return [correct, per_class]
    if kind == "preds":
        return list(ctx.eval_hard(s["ds"], s["batch"], s["K"], s["N"], preds=True, out=s["out"], stream=s["stream"]))
    if kind == "soft":
        ga, gb, gt, loss = ctx.soft_bwd(s["ds"], s["batch"], TAU, s["dloss"])
        return [loss, ga, gb, gt]
    if kind == "autograd":
        for p in s["params"]:
            p.grad = None
        loss = rs.rule_soft_loss(*s["params"], ctx, s["ds"], s["batch"], TAU)
        loss.sum().backward()
        return [loss.detach(), *[p.grad for p in s["params"]]]
    if kind == "probs":
        return list(ctx.soft_fwd(s["ds"], s["batch"], TAU, N=s["N"], K=s["K"], probs=True))
    if kind == "evolve":
        pop, fitness, best, mean = ctx.evolve(s["ds"], s["pop"], s["gens"], s["elite"], s["seed"])
        return [pop, fitness, best, mean]
    if kind == "serve":
        tickets = [ctx.submit(ds, b) for ds, _, _, b in s["requests"]]
        done = [ctx.poll(t, P, K, timeout_us=60_000_000) for t, (_, K, P, _) in zip(tickets, s["requests"])]
        return [np.concatenate([d[i].ravel() for d in done]) for i in (0, 1)]       # every request's counts
    ds = ctx.dataset(s["X"], s["y"], s["K"])
    correct, per_class, _ = ctx.eval_hard(ds, s["batch"], s["K"])
    counts = ctx.dataset_info(ds)[3]
    ctx.dataset_destroy(ds)
    return [correct, per_class, counts]


def work(case):
    """One pass's input and output bytes, and its nominal operations: a threshold test is one compare,
    a pair test two products and a compare (1.4 on average); a soft condition a margin (3), an
    exponential and its use in the product (4), and in the adjoint the same with the two sums (8)."""
    c, kind = case, case["kind"]
    if kind == "serve":
        n = (c["nhi"] - c["nlo"]) / math.log(c["nhi"] / c["nlo"])
        p = (c["phi"] - c["plo"]) / math.log(c["phi"] / c["plo"])
        conds = p * (1 + c["rhi"]) / 2 * (1 + c["chi"]) / 2
        return {"bytes": int(c["runs"] * n * (c["flo"] + c["fhi"]) / 2 * 4 + c["requests"] * conds * 25),
                "flops": int(c["requests"] * conds * n * 1.4)}
    N, F, K, P = c["N"], c["F"], c["K"], c["P"]
    conds = _conds(c)
    data, rules = 4 * N * F + 4 * N, 25 * conds + 4 * P * (c["rlo"] + c["rhi"])
    if kind in ("hard", "preds", "register"):
        out = 4 * P * (K + 1) + (4 * P * N if kind == "preds" else 0)
        return {"bytes": int(data + rules + out), "flops": int(1.4 * conds * N)}
    if kind == "evolve":
        return {"bytes": int(data + 2 * rules), "flops": int(1.4 * conds * N * (c["gens"] + 1))}
    out = 4 * P + (4 * P * N * K if kind == "probs" else 12 * conds)
    return {"bytes": int(data + rules + out), "flops": int(conds * N * (7 if kind == "probs" else 15))}


# ------------------------------------------------------------------------- the soft path in 64 bits

EXACT_MOST = 6.0e9                 # padded condition-samples
_BLOCK = 1.2e7                     # padded condition-samples of one step


def exact(case, seed):
    """Losses, gradients and class probabilities of the soft path in float64; the other kinds return
    whole numbers (None)."""
    c, kind = case, case["kind"]
    if kind not in ("soft", "autograd", "probs"):
        return None
    N, F, K = c["N"], c["F"], c["K"]
    X, y = _data(N, F, K, 0, _gen(seed, 1))
    b = _rules(c, X, K, seed, default=int(torch.bincount(y, minlength=K).argmax()))
    P = b.P
    rp, cr = np.diff(b.set_rule_off), np.diff(b.rule_cond_off)
    R, C = int(rp.max()), int(cr.max())
    if float(P) * R * C * N > EXACT_MOST:
        return None
    f64 = dict(dtype=torch.float64, device="cuda")
    set_of_rule = np.repeat(np.arange(P), rp)
    r_in_set = np.arange(b.R) - np.repeat(b.set_rule_off[:-1], rp)
    at = tuple(torch.as_tensor(i, device="cuda") for i in
               (np.repeat(set_of_rule, cr), np.repeat(r_in_set, cr), np.arange(b.C) - np.repeat(b.rule_cond_off[:-1], cr)))
    rule_at = tuple(torch.as_tensor(i, device="cuda") for i in (set_of_rule, r_in_set))

    def slots(v, fill, dtype):
        t = torch.full((P, R, C), fill, dtype=dtype, device="cuda")
        t[at] = torch.as_tensor(v, device="cuda").to(dtype)
        return t

    f = slots(b.cond_f, 0, torch.int64)
    g = slots(b.cond_g, -1, torch.int64)
    live = slots(np.ones(b.C), False, torch.bool)
    sign = slots(np.where(b.cond_op == 1, -1.0, 1.0), 1.0, torch.float64)
    par = [slots(v, 0.0, torch.float64) for v in (b.cond_a, b.cond_b, b.cond_t)]
    pair = g >= 0
    cls = torch.full((P, R), -1, dtype=torch.int64, device="cuda")
    cls[rule_at] = torch.as_tensor(b.rule_class, device="cuda").long()
    deflt = torch.as_tensor(b.set_default, device="cuda").long()
    Xt = X.t().double().contiguous()
    y = y.long()
    tau = float(np.float32(TAU))
    weight = torch.ones(P, **f64)
    if kind == "soft":
        weight = (torch.rand(P, generator=_gen(seed, 2), device="cuda") + 0.5).double()
    loss = torch.zeros(P, **f64)
    grads = [torch.zeros((P, R, C), **f64) for _ in range(3)]
    probs = torch.zeros((P, N, K), **f64) if kind == "probs" else None
    step_n = min(N, 16384)
    step_p = max(1, int(_BLOCK / (R * C * step_n)))
    for p0 in range(0, P, step_p):
        sl = slice(p0, min(P, p0 + step_p))
        a_, b_, t_ = (v[sl].clone().requires_grad_(kind != "probs") for v in par)
        for n0 in range(0, N, step_n):
            x = Xt[:, n0:n0 + step_n]
            yy = y[n0:n0 + step_n]
            rhs = torch.where(pair[sl][..., None], b_[..., None] * x[g[sl].clamp(min=0)], t_[..., None])
            u = sign[sl][..., None] * (a_[..., None] * x[f[sl]] - rhs) / tau
            lq = torch.where(live[sl][..., None], torch.nn.functional.logsigmoid(u), 0.0).sum(2)     # [p, R, n]
            real = (cls[sl] >= 0)[..., None]
            lq = torch.where(real, lq, -1e4)                     # padding rules never fire
            l1q = torch.log(-torch.expm1(lq))
            lu = torch.cumsum(l1q, 1)
            before = lu - l1q
            last = lu[:, -1]
            if kind == "probs":
                w = torch.exp(lq + before)
                for k in range(K):
                    pk = (w * (cls[sl] == k)[..., None]).sum(1) + torch.exp(last) * (deflt[sl] == k)[:, None]
                    probs[sl, n0:n0 + step_n, k] = pk
                    loss[sl] -= (torch.log(pk) * (yy == k)).sum(1)
                continue
            hit = cls[sl][:, :, None] == yy
            terms = torch.where(hit, lq + before, -math.inf)
            terms = torch.cat([terms, torch.where(deflt[sl][:, None] == yy, last, -math.inf)[:, None]], 1)
            part = -torch.logsumexp(terms, 1).sum(1)
            got = torch.autograd.grad((part * weight[sl]).sum() / N, (a_, b_, t_))
            loss[sl] += part.detach()
            for dst, src in zip(grads, got):
                dst[sl] += src
    loss /= N
    if kind == "probs":
        return [loss, probs]
    return [loss, *[v[at] for v in grads]]
