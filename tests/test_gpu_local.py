"""The FP64 generation loop with a cluster per run and the population in shared
memory, against the other forms of the same loop: the numbers are the same."""
import numpy as np
import pytest

import oracle
from paper_2405_16551_gb300 import capi, problems

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu(monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    monkeypatch.setenv("DE_GB300_AUTOTUNE", "0")


def _cfg(np_, d, obj, rot, **kw):
    kw.setdefault("target_error", 0.0)
    kw.setdefault("max_generations", 10**6)
    M = None if rot == "none" else problems.rotation(d, seed=d)
    if rot == "sparse":  # rows with few entries are not sliced: the DFMA chain
        M = np.eye(d)[np.random.default_rng(d).permutation(d)]
    return capi.make_config(np_, d, objective=obj, shift=problems.shift(d, seed=np_), rot=M, seed=np_ + d, **kw)


def _result(h, runs=1):
    return [(capi.de_get_population(h, k), capi.de_get_best(h, k)) for k in range(runs)]


def _equal(a, b):
    for ((xa, fa), ba), ((xb, fb), bb) in zip(a, b):
        assert np.array_equal(xa, xb) and np.array_equal(fa, fb)
        for key in ("generations", "evals", "best_index", "best_f", "stop_reason"):
            assert ba[key] == bb[key], key


def _both(make, use, monkeypatch, csize, want=3):
    out = []
    for mode in ("3", "1"):
        monkeypatch.setenv("DE_GB300_FP64_PERSIST", mode)
        h = make()
        try:
            plan = capi.de_get_plan(h)
            assert plan == {"kernel_path": 3, "cluster_size": csize if mode == "3" else 0}
            out.append(use(h))
        finally:
            capi.de_destroy(h)
    _equal(*out)
    return out[0]


@pytest.mark.parametrize("np_,d,obj,rot", [
    (64, 10, 0, "none"), (4, 1, 1, "none"), (9, 32, 3, "none"), (63, 31, 2, "none"), (57, 2, 2, "none"),
    (64, 15, 1, "full"), (8, 30, 3, "sparse"), (33, 32, 0, "sparse"),
    (64, 30, 1, "full"), (5, 16, 3, "full"), (41, 33, 2, "full"), (64, 64, 0, "full"), (64, 63, 1, "full"),
])
def test_same_run(np_, d, obj, rot, monkeypatch):
    def use(h):
        for n in (1, 2, 37):  # buffers of either parity across launches
            capi.de_step(h, n)
        return _result(h)

    _both(lambda: capi.de_init(_cfg(np_, d, obj, rot)), use, monkeypatch, -(-np_ // 8))


@pytest.mark.parametrize("kw", [dict(target_error=1e-3, max_generations=20000),
                                dict(max_evals=64 * 100 + 5), dict(max_generations=77)])
def test_same_stop_of_every_run_of_a_batch(kw, monkeypatch):
    def use(h):
        capi.de_run(h, 3)
        return _result(h, 3)

    cfgs = [_cfg(n, d, 0, "none", **kw) for n, d in ((64, 6), (20, 3), (30, 9))]
    _both(lambda: capi.de_init_batch(cfgs), use, monkeypatch, 8)


@pytest.mark.parametrize("rot", ["none", "full"])
@pytest.mark.parametrize("asynchronous", [False, True])
@pytest.mark.parametrize("m,interval,nmig,target", [(4, 5, 2, 0.0), (3, 1, 1, 0.0), (7, 1000, 3, 150.0),
                                                    (5, 7, 2, 150.0)])
def test_same_islands(m, interval, nmig, target, asynchronous, rot, monkeypatch):
    """Migrations, and the common stop at the first generation below the target
    (which each island learns of a generation late and takes one back for)."""
    kind = capi.DE_MIGRATE_ASYNC if asynchronous else capi.DE_MIGRATE_SYNC

    def use(h):
        for n in (3, 11):
            capi.de_step(h, n)
        capi.de_run(h, m)
        return _result(h, m)

    cfg = _cfg(24, 20, 0, rot, target_error=target, max_generations=400)
    out = _both(lambda: capi.de_init_islands_ex(cfg, m, interval, nmig, kind), use, monkeypatch, 3)
    assert {b["stop_reason"] for _, b in out} == {capi.DE_STOP_TARGET if target else capi.DE_STOP_GENERATIONS}


def test_islands_set_apart_use_the_other_form(monkeypatch):
    def use(h):
        capi.de_step(h, 6)
        capi.de_reset(h, 1)
        capi.de_step(h, 4)
        capi.de_reset(h, -1)
        capi.de_step(h, 9)
        return _result(h, 2)

    _both(lambda: capi.de_init_islands(_cfg(16, 8, 1, "none"), 2, 1000, 1), use, monkeypatch, 2)


def test_an_island_that_never_arrives_ends_the_launch(monkeypatch):
    monkeypatch.setenv("DE_GB300_FP64_PERSIST", "3")
    monkeypatch.setenv("DE_GB300_TEST_GRID_TIMEOUT", "2")
    cfg = _cfg(16, 8, 1, "none", max_generations=50)
    h = capi.de_init_islands(cfg, 3, 5, 1)
    try:
        with pytest.raises(capi.DEError) as e:
            capi.de_run(h, 3)
        assert "timed out" in str(e.value)
    finally:
        capi.de_destroy(h)


def test_matches_the_oracle(monkeypatch):
    monkeypatch.setenv("DE_GB300_FP64_PERSIST", "3")
    o = problems.shift(10, seed=4)
    Xo, fo, go, evo, _ = oracle.run(64, 10, 0.5, 0.9, -100, 100, 0, o, None, seed=4, max_generations=60,
                                    target_error=0.0)
    h = capi.de_init(capi.make_config(64, 10, objective=0, shift=o, seed=4, max_generations=60, target_error=0.0))
    try:
        assert capi.de_run(h)[0]["generations"] == go
        assert np.array_equal(capi.de_get_population(h)[0], Xo)
    finally:
        capi.de_destroy(h)


@pytest.mark.parametrize("obj", [0, 1, 2, 3])
@pytest.mark.parametrize("d,n,ld", [(16, 1, 16), (17, 9, 20), (30, 153, 30), (31, 1217, 31), (32, 5000, 33)])
def test_evaluation_of_rows(obj, d, n, ld):
    """Rows of every kind (ordinary, one coordinate far above the rest, zero,
    huge, not finite) at the edges of a tile and of a round over the device,
    against the oracle, and against the fitness of the generation loop."""
    import torch

    o, M = problems.shift(d, seed=d), problems.rotation(d, seed=d)
    x = problems.population(n, d, seed=n)
    for r in range(0, n, 7):
        x[r, r % d] *= 1e9
    if n > 8:
        x[3] = o
        x[5] *= 1e-300
        x[6, 1] = np.nan
        x[8, 0] = np.inf
    buf = np.full((n, ld), 1e30)
    buf[:, :d] = x
    xd = torch.from_numpy(buf).cuda()
    f = torch.full((n + 2,), -7.0, dtype=torch.float64, device="cuda")
    h = capi.de_init(capi.make_config(16, d, objective=obj, shift=o, rot=M, seed=3, max_generations=10**6,
                                      target_error=0.0))
    try:
        capi.de_eval(h, 0, xd.data_ptr(), ld, n, f.data_ptr())
        capi.de_step(h, 5)
        xp, fp = capi.de_get_population(h)
        xg = torch.from_numpy(xp).cuda()
        g = torch.zeros(16, dtype=torch.float64, device="cuda")
        capi.de_eval(h, 0, xg.data_ptr(), d, 16, g.data_ptr())
        torch.cuda.synchronize()
    finally:
        capi.de_destroy(h)
    assert np.array_equal(g.cpu().numpy(), fp)
    f = f.cpu().numpy()
    assert np.all(f[n:] == -7.0)
    ok = np.isfinite(x).all(1)
    assert not np.isfinite(f[:n][~ok]).any()
    fo, S = oracle.evaluate(obj, x[ok], o, M)
    # the oracle's own bound (its rows' rounding enters the cosines of z = 2^30 as well)
    big = np.abs(x[ok]).max(1) > 1e6
    assert np.all((np.abs(f[:n][ok] - fo) <= 1e-12 * (np.abs(fo) + S))[~big])
    assert np.all((np.abs(f[:n][ok] - fo) <= (1e-12 if obj in (0, 2) else 1e-9) * (np.abs(fo) + S) + 100 * d)[big])
