"""Composition functions whose components run on CTAs of their own (few tiles), one
after another in a CTA (many), and in groups of rows (a generation per launch):
the numbers are the same."""
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


def _run(np_, d, obj, runs, **kw):
    s = problems.suite(obj, d, seed=obj)
    cfgs = [capi.make_config(np_, d, objective=obj, shift=s["shift"], rot=s["rot"], seed=3, run_id=r,
                             max_generations=9 + r, target_error=0.0, **kw) for r in range(runs)]
    h = capi.de_init_batch(cfgs) if runs > 1 else capi.de_init(cfgs[0])
    try:
        capi.de_step(h, 3)
        res = capi.de_run(h, runs)
        return capi.de_get_plan(h)["kernel_path"], [capi.de_get_population(h, r) for r in range(runs)], res
    finally:
        capi.de_destroy(h)


@pytest.mark.parametrize("np_,d,obj,runs,kw", [
    (8, 16, 18, 1, {}), (50, 33, 20, 1, {}), (250, 30, 19, 1, dict(jde=True)), (61, 64, 18, 3, {}),
    (40, 65, 19, 1, dict(strategy=capi.DE_BEST1BIN)), (250, 100, 18, 1, {}), (9, 128, 20, 2, {}),
    (400, 20, 20, 1, {}), (300, 50, 19, 4, {}),
])
def test_every_form_agrees(np_, d, obj, runs, kw, monkeypatch):
    out = []
    for mode in ("0", "1"):
        monkeypatch.setenv("DE_GB300_FP64_PERSIST", mode)
        out.append(_run(np_, d, obj, runs, **kw))
    for (xa, fa), (xb, fb) in zip(out[0][1], out[1][1]):
        assert np.array_equal(xa, xb) and np.array_equal(fa, fb)
    for a, b in zip(out[0][2], out[1][2]):
        assert all(a[k] == b[k] for k in ("best_f", "best_index", "generations", "evals", "stop_reason"))
    s = problems.suite(obj, d, seed=obj)
    for x, f in out[1][1]:
        fo, S = oracle.evaluate(obj, x, s["shift"], s["rot"])
        assert np.all(np.abs(f - fo) <= 1e-12 * (np.abs(fo) + S))


@pytest.mark.parametrize("env", ["2", "9"])
def test_a_cta_that_never_arrives_ends_the_launch(env, monkeypatch):
    """... a component's CTA as well as one that mixes."""
    monkeypatch.setenv("DE_GB300_FP64_PERSIST", "1")
    monkeypatch.setenv("DE_GB300_TEST_GRID_TIMEOUT", env)
    s = problems.suite(18, 20, seed=18)
    h = capi.de_init(capi.make_config(40, 20, objective=18, shift=s["shift"], rot=s["rot"], seed=3,
                                      max_generations=50, target_error=0.0))
    try:
        with pytest.raises(capi.DEError) as e:
            capi.de_run(h)
        assert "timed out" in str(e.value)
    finally:
        capi.de_destroy(h)


@pytest.mark.parametrize("obj", [5, 6, 15, 18, 20])
@pytest.mark.parametrize("d", [30, 64, 100])
def test_a_few_rows(obj, d):
    """One and two rows go another way than more."""
    import torch

    s = problems.suite(obj, d, seed=obj)
    x = problems.population(5, d, seed=8)
    xd = torch.from_numpy(x).cuda()
    fo, S = oracle.evaluate(obj, x, s["shift"], s["rot"], scale=s["scale"], perm=s["perm"])
    h = capi.de_init(capi.make_config(8, d, objective=obj, shift=s["shift"], rot=s["rot"], perm=s["perm"],
                                      scale=s["scale"], seed=1))
    try:
        for n in (1, 2, 3, 5):
            f = torch.full((6,), -7.0, dtype=torch.float64, device="cuda")
            capi.de_eval(h, 0, xd.data_ptr(), d, n, f.data_ptr())
            f = f.cpu().numpy()
            assert np.all(np.abs(f[:n] - fo[:n]) <= 1e-12 * (np.abs(fo[:n]) + S[:n])) and np.all(f[n:] == -7.0)
    finally:
        capi.de_destroy(h)
