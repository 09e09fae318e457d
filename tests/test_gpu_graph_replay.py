"""A caller that captures de_step on its own stream and launches the graph: the
library is not called, and what it reads afterwards is the new state."""
import numpy as np
import pytest

from paper_2405_16551_gb300 import capi, problems

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu(monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    monkeypatch.setenv("DE_GB300_AUTOTUNE", "0")


def _cfg(np_, d, prec, **kw):
    return capi.make_config(np_, d, objective=1, shift=problems.shift(d, seed=2), rot=problems.rotation(d, seed=3),
                            seed=7, precision=prec, target_error=0.0, max_generations=10**6, **kw)


def _captured(stream, work):
    import torch

    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
        work()
    return g


@pytest.mark.parametrize("prec,persist,np_,d,gens", [
    (capi.DE_PREC_FP64, "0", 40, 12, 1), (capi.DE_PREC_FP64, "0", 150, 40, 3), (capi.DE_PREC_FP64, "1", 40, 12, 1),
    (capi.DE_PREC_FP64, "1", 150, 40, 3), (capi.DE_PREC_FP64, "3", 40, 24, 1), (capi.DE_PREC_BF16X3, "", 150, 40, 1),
])
def test_population_after_each_replay(prec, persist, np_, d, gens, monkeypatch):
    import torch

    if persist:
        monkeypatch.setenv("DE_GB300_FP64_PERSIST", persist)
    s = torch.cuda.Stream()
    h, ref = capi.de_init(_cfg(np_, d, prec), s.cuda_stream), capi.de_init(_cfg(np_, d, prec))
    try:
        capi.de_step(h, 2)
        capi.de_step(ref, 2)
        g = _captured(s, lambda: capi.de_step(h, gens))
        for _ in range(4):
            with torch.cuda.stream(s):
                g.replay()
            capi.de_step(ref, gens)
            (x, f), (xr, fr) = capi.de_get_population(h), capi.de_get_population(ref)
            assert np.array_equal(x, xr) and np.array_equal(f, fr)
            assert capi.de_get_best(h)["generations"] == capi.de_get_best(ref)["generations"]
        del g
    finally:
        capi.de_destroy(h)
        capi.de_destroy(ref)


def _islands(stream, monkeypatch, mode):
    monkeypatch.setenv("DE_GB300_FP64_PERSIST", mode)
    cfg = capi.make_config(16, 8, objective=1, shift=problems.shift(8, seed=2), seed=7, target_error=0.0,
                           max_generations=10**6)
    return capi.de_init_islands(cfg, 3, 5, 1, stream)


def test_an_island_reset_by_a_graph(monkeypatch):
    """Its generations are no longer those of the other islands, which the
    cluster-per-run loop would take for granted."""
    import torch

    s = torch.cuda.Stream()
    h, ref = _islands(s.cuda_stream, monkeypatch, "3"), _islands(None, monkeypatch, "1")
    try:
        g = _captured(s, lambda: capi.de_reset(h, 1))
        for n in (7, 4):
            capi.de_step(h, n)
            capi.de_step(ref, n)
            with torch.cuda.stream(s):
                g.replay()
            capi.de_reset(ref, 1)
        capi.de_step(h, 6)
        capi.de_step(ref, 6)
        for r in range(3):
            (x, f), (xr, fr) = capi.de_get_population(h, r), capi.de_get_population(ref, r)
            assert np.array_equal(x, xr) and np.array_equal(f, fr), r
        del g
    finally:
        capi.de_destroy(h)
        capi.de_destroy(ref)


def test_step_after_one_islands_reset_only_enqueues(monkeypatch):
    import torch

    s = torch.cuda.Stream()
    h = _islands(s.cuda_stream, monkeypatch, "3")
    try:
        capi.de_step(h, 3)
        capi.de_reset(h, 1)
        torch.cuda.synchronize()
        before = torch.cuda.Event()
        with torch.cuda.stream(s):
            torch.cuda._sleep(1_000_000_000)  # about half a second
            before.record()
        capi.de_step(h, 4)
        assert not before.query()
        assert capi.de_get_best(h, 0)["generations"] == 7
    finally:
        capi.de_destroy(h)
