"""The work a user of this library has it do, as timed cases.

Every case goes through the public entry points of ``capi``.  Three kinds:

* ``run``: one optimisation (or a batch of them, or an island model) from its
  initial population: ``de_reset``, ``de_run`` and the final population, fitness
  and result records read back, as a program does that keeps a handle and
  restarts it;
* ``eval``: ``de_eval`` of device rows with a handle's objective (a caller that
  scores its own candidate points);
* ``mlp``: the surrogate network on its own: parameters in, Adam steps on an
  archive, parameters out, predictions of a batch of candidate rows.

Sizes are those of the benchmark's workloads (NP = 64, D = 10; NP = 1024,
D = 100; 512 uneven runs; NP = 8192, D = 1000; 30 trials of NP = 250, D = 100 on
the proposed benchmark; 16 islands of NP = 64, D = 30; the ODE fit at NP = 256)
and of the tests around them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2405_16551_gb300 import capi, problems

FP64, BF16X3, TF32X3 = capi.DE_PREC_FP64, capi.DE_PREC_BF16X3, capi.DE_PREC_TF32X3
F, CR = 0.5, 0.9


def _run(**kw):
    c = dict(kind="run", np=64, d=10, objective=0, precision=FP64, runs=1, gens=100, jde=False, strategy=0,
             islands=0, interval=20, surrogate_k=0, uneven=False, rotate=True)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest run in use: shifted sphere to 1e-8, where launches and barriers count
        _run(name="run_sphere_np64_d10_fp64", np=64, d=10, objective=0, gens=1000, rotate=False),
        # the paper's comparison size in the plain FP64 form
        _run(name="run_rastrigin_np1024_d100_fp64", np=1024, d=100, objective=1, gens=500),
        # the same problem on the tensor cores: the headline workload, whole
        _run(name="run_rastrigin_np1024_d100_bf16", np=1024, d=100, objective=1, precision=BF16X3, gens=3000),
        # adaptive parameters and the wider split type, odd sizes
        _run(name="run_ackley_np501_d50_tf32_jde", np=501, d=50, objective=3, precision=TF32X3, gens=1000, jde=True),
        # many independent small runs in one handle (a parameter study)
        _run(name="run_batch512_bf16", runs=512, uneven=True, precision=BF16X3, gens=200),
        # the large dense problem
        _run(name="run_rastrigin_np8192_d1000_bf16", np=8192, d=1000, objective=1, precision=BF16X3, gens=200),
        # the proposed benchmark's protocol: 30 trials of one composition function
        _run(name="run_suite_f09_30x250_d100_fp64", np=250, d=100, objective=19, runs=30, gens=40),
        # the island model with ring migration
        _run(name="run_islands16_np64_d30_fp64", np=64, d=30, objective=1, islands=16, gens=1000),
        # a costly objective with surrogate screening (trains after 5 and 15 generations)
        _run(name="run_ode_np256_surrogate8", np=256, d=20, objective=4, gens=20, surrogate_k=8, rotate=False),
        # a caller scoring a few of its own points: one small launch
        dict(kind="eval", name="eval_ackley_n250_d30_fp64", n=250, d=30, objective=3, precision=FP64),
        # ... and many of them
        dict(kind="eval", name="eval_rastrigin_n16384_d100_fp64", n=16384, d=100, objective=1, precision=FP64),
        # the network by itself: one retraining and one generation's predictions
        dict(kind="mlp", name="mlp_train25_n20000", n=20000, steps=25, rows=2048),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    k = rng.choice(["fp64", "split", "split", "batch", "suite", "islands", "eval", "eval_split", "mlp"])
    if k == "mlp":
        return dict(kind="mlp", n=_logint(rng, 300, 20000), steps=rng.randint(5, 100), rows=_logint(rng, 100, 8000))
    if k == "eval":
        return dict(kind="eval", n=_logint(rng, 50, 16000), d=_logint(rng, 2, 200),
                    objective=rng.choice([0, 1, 2, 3, 5, 6, 18, 19]), precision=FP64)
    if k == "eval_split":
        return dict(kind="eval", n=_logint(rng, 200, 30000), d=_logint(rng, 10, 250),
                    objective=rng.randint(0, 3), precision=rng.choice([BF16X3, TF32X3]))
    if k == "batch":
        prec = rng.choice([FP64, BF16X3, TF32X3])
        return _run(runs=_logint(rng, 16, 100 if prec == FP64 else 500), uneven=True, precision=prec,
                    gens=rng.randint(20, 100))
    if k == "suite":
        return _run(np=rng.randint(50, 250), d=rng.choice([10, 30, 50, 100]), runs=rng.randint(1, 30),
                    objective=rng.choice([5, 2, 1, 6, 18, 19]), gens=rng.randint(20, 100))
    if k == "islands":
        return _run(np=_logint(rng, 20, 128), d=_logint(rng, 5, 60), objective=rng.randint(0, 3),
                    islands=rng.randint(2, 16), interval=rng.randint(5, 40), gens=rng.randint(100, 500))
    if k == "fp64":
        n, d = _logint(rng, 20, 2000), _logint(rng, 2, 128)
        return _run(np=n, d=d, objective=rng.randint(0, 3), gens=rng.randint(50, 400),
                    jde=rng.random() < 0.3, strategy=rng.choice([0, 0, 1, 2]))
    # split precisions: the whole range of D, fewer generations for the large ones
    d = _logint(rng, 10, 1000)
    n = _logint(rng, 50, 4000)
    return _run(np=n, d=d, objective=rng.choice([0, 1, 3] if d > 256 else [0, 1, 2, 3]),
                precision=rng.choice([BF16X3, TF32X3]), gens=rng.randint(100, 1000) if n * d < 200000 else 50)


# ----------------------------------------------------------------------------- inputs
def _stream():
    return torch.cuda.current_stream().cuda_stream


class _Handle:
    """What a user's program keeps: the library's handle, freed with it."""

    def __init__(self, h, free):
        self.h, self._free = h, free

    def __del__(self):
        self._free(self.h)


def _problem(objective, d, seed, run_id=0, rotate=True):
    if objective == capi.DE_OBJ_ODE:
        return dict(shift=problems.ode_hidden(seed), rot=None, scale=1.0)
    if objective >= problems.ZAKHAROV:
        s = problems.suite(objective, d, seed=seed)
        return dict(shift=s["shift"], rot=s["rot"], scale=s["scale"])
    return dict(shift=problems.shift(d, seed=seed, run_id=run_id),
                rot=problems.rotation(d, seed=seed, run_id=run_id) if rotate else None, scale=1.0)


def _runs(case, seed):
    """(np, d, objective, run_id, problem) of every run of the case."""
    if case["uneven"]:
        return [(n, d, obj, r, _problem(obj, d, seed, r))
                for r, (n, d, obj) in enumerate(problems.batch_shapes(case["runs"], seed=1))]
    p = _problem(case["objective"], case["d"], seed, 0, case["rotate"])
    return [(case["np"], case["d"], case["objective"], r, p) for r in range(case["islands"] or case["runs"])]


def _mlp_params(seed):
    r = np.random.default_rng(seed)
    fan = dict(W1=20, W2=256, w3=256)
    return np.concatenate([r.uniform(-1, 1, shape).ravel() * math.sqrt(6 / fan[k]) if k in fan else np.zeros(shape)
                           for k, shape in capi.MLP_SHAPES]).astype(np.float32)


def prepare(case, seed):
    if case["kind"] == "mlp":
        g = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.rand(case["n"], 20, dtype=torch.float64, device="cuda", generator=g) * 200 - 100
        # standardised log of a sum of squares: what the network is trained on in a run
        t = torch.log((x - 10.0).square().sum(1))
        t = ((t - t.mean()) / t.std()).float()
        q = torch.rand(case["rows"], 20, dtype=torch.float64, device="cuda", generator=g) * 200 - 100
        m = capi.de_mlp_create(seed, _stream())
        return dict(kind="mlp", m=_Handle(m, capi.de_mlp_destroy), params=_mlp_params(seed), x=x, t=t, q=q,
                    y=torch.empty(case["rows"], dtype=torch.float32, device="cuda"), steps=case["steps"])
    if case["kind"] == "eval":
        p = _problem(case["objective"], case["d"], seed)
        cfg = capi.make_config(64, case["d"], f=F, cr=CR, objective=case["objective"], seed=seed,
                               precision=case["precision"], **p)
        g = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.rand(case["n"], case["d"], dtype=torch.float64, device="cuda", generator=g) * 200 - 100
        return dict(kind="eval", h=_Handle(capi.de_init(cfg, _stream()), capi.de_destroy), x=x,
                    f=torch.empty(case["n"], dtype=torch.float64, device="cuda"))
    cfgs = [capi.make_config(n, d, f=F, cr=CR, objective=obj, seed=seed, run_id=rid, precision=case["precision"],
                             max_generations=case["gens"], strategy=case["strategy"], jde=case["jde"],
                             surrogate_k=case["surrogate_k"], **p) for n, d, obj, rid, p in _runs(case, seed)]
    if case["islands"]:
        h = capi.de_init_islands(cfgs[0], case["islands"], case["interval"], 2, _stream())
    elif len(cfgs) > 1:
        h = capi.de_init_batch(cfgs, _stream())
    else:
        h = capi.de_init(cfgs[0], _stream())
    return dict(kind="run", h=_Handle(h, capi.de_destroy), runs=len(cfgs))


def run(state):
    if state["kind"] == "mlp":
        m = state["m"].h
        capi.de_mlp_set_params(m, state["params"])
        loss = capi.de_mlp_train(m, state["x"].data_ptr(), 20, state["t"].data_ptr(), state["x"].shape[0],
                                 state["steps"])
        capi.de_mlp_forward(m, state["q"].data_ptr(), 20, state["q"].shape[0], state["y"].data_ptr())
        return dict(loss=loss, params=capi.de_mlp_get_params(m), y=state["y"])
    if state["kind"] == "eval":
        x, f = state["x"], state["f"]
        capi.de_eval(state["h"].h, 0, x.data_ptr(), x.shape[1], x.shape[0], f.data_ptr())
        return f
    h, n = state["h"].h, state["runs"]
    capi.de_reset(h)
    res = capi.de_run(h, n)
    pops = [capi.de_get_population(h, r) for r in range(n)]
    x, f = pops[0] if n == 1 else (np.concatenate([x.ravel() for x, _ in pops]), np.concatenate([f for _, f in pops]))
    return dict(best_f=np.array([r["best_f"] for r in res]),
                best_index=np.array([r["best_index"] for r in res]),
                generations=np.array([r["generations"] for r in res]),
                evals=np.array([r["evals"] for r in res]),
                stop=np.array([r["stop_reason"] for r in res]),
                x=x, f=f)


# ----------------------------------------------------------------------------- work
def _eval_flops(objective, d, rotate=True):
    if objective == capi.DE_OBJ_ODE:
        return 2000 * 10 * 60.0  # RK4 steps x masses x operations
    comps = {18: 3, 19: 4, 20: 5}.get(objective, 1)
    return comps * ((2.0 * d * d if rotate else 0.0) + 9.0 * d)


def work(case):
    if case["kind"] == "mlp":
        n = 71425
        fwd = 2.0 * (20 * 256 + 256 * 256 + 256)
        return dict(bytes=case["n"] * 164.0 + 8.0 * n + case["rows"] * 164.0,
                    flops=case["steps"] * 256 * 3 * fwd + case["rows"] * fwd)
    if case["kind"] == "eval":
        comps = {18: 3, 19: 4, 20: 5}.get(case["objective"], 1)
        return dict(bytes=case["n"] * (case["d"] + 1) * 8.0 + comps * case["d"] ** 2 * 8.0,
                    flops=case["n"] * _eval_flops(case["objective"], case["d"]))
    b = f = 0.0
    for n, d, obj in (problems.batch_shapes(case["runs"], seed=1) if case["uneven"] else
                      [(case["np"], case["d"], case["objective"])] * (case["islands"] or case["runs"])):
        # a generation reads the target row and writes the next one; the draws cost no memory
        b += (case["gens"] + 1) * n * (16.0 * d + 16)
        f += (case["gens"] + 1) * n * _eval_flops(obj, d, case["rotate"])
    return dict(bytes=b, flops=f)


# ----------------------------------------------------------------------------- the same in plain numpy, 64 bits
def _philox(seed, c0, c1, c2, c3):
    """Philox4x32-10 (Salmon et al., SC'11), vectorised; counters broadcast."""
    m32 = np.uint64(0xFFFFFFFF)
    c = [np.asarray(v, dtype=np.uint64) for v in (c0, c1, c2, c3)]
    c = [np.ascontiguousarray(v) for v in np.broadcast_arrays(*c)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1),
             p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _range(w, n):
    return ((w * np.uint64(n)) >> np.uint64(32)).astype(np.int64)


def _basic(fn, z):
    n = z.shape[1]
    i = np.arange(1, n + 1)
    if fn == 0:
        return (z * z).sum(1)
    if fn == 1:
        return (z * z - 10 * np.cos(2 * np.pi * z) + 10).sum(1)
    if fn == 2:
        t = z + 1
        return (100 * (t[:, 1:] - t[:, :-1] ** 2) ** 2 + (t[:, :-1] - 1) ** 2).sum(1)
    if fn == 3:
        return (20 + math.e - 20 * np.exp(-0.2 * np.sqrt((z * z).mean(1))) - np.exp(np.cos(2 * np.pi * z).mean(1)))
    if fn == 5:
        b = (0.5 * i * z).sum(1)
        return (z * z).sum(1) + b ** 2 + b ** 4
    if fn == 6:
        t = z + 420.9687462275036
        m = np.fmod(np.abs(t), 500.0)
        out = np.sign(t) * (500 - m) * np.sin(np.sqrt(500 - m)) - (np.abs(t) - 500) ** 2 / (1e4 * n)
        g = np.where(np.abs(t) > 500, out, t * np.sin(np.sqrt(np.abs(t))))
        return 418.9828872724338 * n - g.sum(1)
    if fn == 13:
        return (1e6 ** ((i - 1) / max(n - 1, 1)) * z * z).sum(1)
    if fn == 14:
        return (z * z).sum(1) / 4000 - np.prod(np.cos(z / np.sqrt(i)), 1) + 1
    raise KeyError(fn)


_DOMAIN = {1: 0.0512, 2: 0.02048, 6: 10.0, 14: 6.0}
_COMPOSED = {18: ((1, 14, 6), (10, 20, 30), (1, 10, 1), (0, 100, 200)),
             19: ((3, 13, 14, 1), (10, 20, 30, 40), (10, 1e-6, 10, 1), (0, 100, 200, 300))}


def _objective(objective, p, x):
    o, M = p["shift"], p["rot"]
    if objective not in _COMPOSED:
        y = (x - o) * p["scale"]
        return _basic(objective, y if M is None else y @ M.T)
    fns, sigma, lam, bias = _COMPOSED[objective]
    D = np.stack([((x - o[c]) ** 2).sum(1) for c in range(len(fns))], 1)
    lw = -D / (2 * x.shape[1] * np.square(sigma, dtype=np.float64)) - 0.5 * np.log(D)
    w = np.exp(lw - lw.max(1, keepdims=True))
    w /= w.sum(1, keepdims=True)
    return sum(w[:, c] * (lam[c] * _basic(fn, ((x - o[c]) * _DOMAIN.get(fn, 1.0)) @ M[c].T) + bias[c])
               for c, fn in enumerate(fns))


def _init(n, d, seed, run_id):
    nb = (d + 1) // 2
    w = _philox(seed, np.arange(nb)[None, :], np.arange(n)[:, None], 0, (run_id << 12) | 1)
    u = np.stack([((w[0] << np.uint64(32)) | w[1]) >> np.uint64(11),
                  ((w[2] << np.uint64(32)) | w[3]) >> np.uint64(11)], 2).reshape(n, 2 * nb)[:, :d]
    return u.astype(np.float64) * 2.0 ** -53 * 200.0 - 100.0


def _generation(x, f, objective, p, seed, run_id, g):
    """DE/rand/1/bin, the bound repair and greedy selection of one generation."""
    n, d = x.shape
    i = np.arange(n)
    w = _philox(seed, np.arange(1 + (d + 3) // 4)[None, :], i[:, None], g, (run_id << 12) | 2)
    w0 = [v[:, 0] for v in w]
    r1 = _range(w0[0], n - 1)
    r1 += r1 >= i
    taken = np.sort(np.stack([i, r1], 1), 1)
    r2 = _range(w0[1], n - 2)
    for c in range(2):
        r2 += r2 >= taken[:, c]
    taken = np.sort(np.stack([i, r1, r2], 1), 1)
    r3 = _range(w0[2], n - 3)
    for c in range(3):
        r3 += r3 >= taken[:, c]
    u = np.stack([v[:, 1:] for v in w], 2).reshape(n, -1)[:, :d]
    cross = (u <= np.uint64(int(CR * 2.0 ** 32))) | (np.arange(d)[None, :] == _range(w0[3], d)[:, None])
    v = x[r1] + F * (x[r2] - x[r3])
    v = np.where(v < -100, 0.5 * (x - 100), np.where(v > 100, 0.5 * (x + 100), v))
    t = np.where(cross, v, x)
    ft = _objective(objective, p, t)
    keep = ft <= f
    return np.where(keep[:, None], t, x), np.where(keep, ft, f)


def _exact_run(case, seed):
    todo = _runs(case, seed)
    size = sum(n * (d * (d + 600) * {18: 3, 19: 4}.get(obj, 1)) for n, d, obj, _, _ in todo) * case["gens"]
    if case["precision"] != FP64 or case["jde"] or case["strategy"] or case["surrogate_k"] or size > 1e11:
        return None  # split decisions may differ inside the stated bound; the others take too long
    pop = []
    for n, d, obj, rid, p in todo:
        x = _init(n, d, seed, rid)
        pop.append([x, _objective(obj, p, x)])
    gens = [0] * len(pop)
    stop = [0] * len(pop)
    for g in range(1, case["gens"] + 1):
        done = [f.min() < 1e-8 for _, f in pop]
        if case["islands"] and any(done):
            done = [True] * len(pop)
        for r, (n, d, obj, rid, p) in enumerate(todo):
            if done[r]:
                stop[r] = 1
            else:
                pop[r] = list(_generation(*pop[r], obj, p, seed, rid, g))
                gens[r] = g
        if all(done):
            break
        if case["islands"] and g % case["interval"] == 0:
            if any(f.min() < 1e-8 for _, f in pop):
                return None  # the stop falls on a migration: not worked out here
            gone = [(x[b].copy(), f[b].copy()) for x, f in pop for b in [np.argsort(f, kind="stable")[:2]]]
            for r, (x, f) in enumerate(pop):
                worst = np.lexsort((-np.arange(len(f)), -f))[:2]  # the higher index first on ties
                x[worst], f[worst] = gone[r - 1]
    best = [int(np.argmin(f)) for _, f in pop]
    return dict(best_f=np.array([f[b] for (_, f), b in zip(pop, best)]), best_index=None, generations=None,
                evals=None, stop=None, x=np.concatenate([x.ravel() for x, _ in pop]) if len(pop) > 1 else pop[0][0],
                f=np.concatenate([f for _, f in pop]))


def _exact_mlp(case, seed):
    s = prepare(case, seed)
    P = {k: v for k, v in capi.mlp_unpack(s["params"]).items()}
    x, t, q = (s[k].double().cpu().numpy() for k in ("x", "t", "q"))

    def forward(a):
        h1 = np.maximum(a / 100 @ P["W1"].T + P["b1"], 0)
        h2 = np.maximum(h1 @ P["W2"].T + P["b2"], 0)
        return h1, h2, h2 @ P["w3"] + P["b3"]

    m = {k: np.zeros_like(v) for k, v in P.items()}
    v = {k: np.zeros_like(a) for k, a in P.items()}
    loss = 0.0
    for step in range(case["steps"]):
        w = _philox(seed, 0, np.arange(64), step, 5)
        rows = _range(np.stack(w, 1).ravel(), case["n"])
        h1, h2, y = forward(x[rows])
        r = y - t[rows]
        loss = (r * r).mean()
        d2 = (2 * r / 256)[:, None] * P["w3"] * (h2 > 0)
        d1 = d2 @ P["W2"] * (h1 > 0)
        G = dict(W1=d1.T @ (x[rows] / 100), b1=d1.sum(0), W2=d2.T @ h1, b2=d2.sum(0), w3=(2 * r / 256) @ h2,
                 b3=np.array([(2 * r / 256).sum()]))
        for k in P:
            m[k] = 0.9 * m[k] + 0.1 * G[k]
            v[k] = 0.999 * v[k] + 0.001 * G[k] ** 2
            P[k] = P[k] - 1e-3 * (m[k] / (1 - 0.9 ** (step + 1))) / (np.sqrt(v[k] / (1 - 0.999 ** (step + 1))) + 1e-8)
    return dict(loss=float(loss), params=np.concatenate([P[k].ravel() for k, _ in capi.MLP_SHAPES]),
                y=forward(q)[2])


def exact(case, seed):
    if case["kind"] == "mlp":
        return _exact_mlp(case, seed)
    if case["kind"] == "eval":
        g = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.rand(case["n"], case["d"], dtype=torch.float64, device="cuda", generator=g) * 200 - 100
        return _objective(case["objective"], _problem(case["objective"], case["d"], seed), x.cpu().numpy())
    return _exact_run(case, seed)
