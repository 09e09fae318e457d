"""Handles beside one another: what one meets or needs does not reach the others."""
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


def _init(np_, d, prec, rot):
    return capi.de_init(capi.make_config(np_, d, objective=1, shift=problems.shift(d, seed=2),
                                         rot=problems.rotation(d, seed=3) if rot else None, seed=7, precision=prec,
                                         target_error=0.0, max_generations=10**6))


def test_a_handle_that_cannot_be_created_leaves_no_error_behind(monkeypatch):
    monkeypatch.setenv("DE_GB300_FP64_PERSIST", "0")
    h = _init(24, 6, capi.DE_PREC_FP64, False)
    try:
        # five runs of the largest accepted shape: more than the device holds
        with pytest.raises(capi.DEError) as e:
            capi.de_init_batch([capi.make_config(1 << 20, 4096, run_id=r) for r in range(5)])
        assert e.value.status == capi.DE_ERR_OOM
        capi.de_step(h, 3)
        assert capi.de_get_best(h)["generations"] == 3
    finally:
        capi.de_destroy(h)


@pytest.mark.parametrize("env,prec,rot,np_,d_large,d_small", [
    (("DE_GB300_FP64_PERSIST", "3"), capi.DE_PREC_FP64, True, 24, 30, 20),
    (("DE_GB300_FP64_PERSIST", "0"), capi.DE_PREC_FP64, False, 24, 1500, 6),
    (("DE_GB300_FP64_PERSIST", "1"), capi.DE_PREC_FP64, False, 24, 1500, 6),
    (("DE_GB300_PERSIST", "0"), capi.DE_PREC_BF16X3, True, 40, 600, 10),
    (("DE_GB300_PERSIST", "0"), capi.DE_PREC_TF32X3, True, 40, 100, 10),
    (("DE_GB300_PERSIST", "1"), capi.DE_PREC_BF16X3, True, 40, 100, 10),
])
def test_the_larger_handle_goes_on(env, prec, rot, np_, d_large, d_small, monkeypatch):
    """A kernel's limit of shared memory belongs to the process, not to a handle."""
    monkeypatch.setenv(*env)
    alone = _init(np_, d_large, prec, rot)
    capi.de_step(alone, 5)
    x0, f0 = capi.de_get_population(alone)
    capi.de_destroy(alone)
    a = _init(np_, d_large, prec, rot)
    b = _init(np_, d_small, prec, rot)
    try:
        capi.de_step(a, 5)
        capi.de_step(b, 5)
        x, f = capi.de_get_population(a)
        assert np.array_equal(x, x0) and np.array_equal(f, f0)
        capi.de_get_population(b)
    finally:
        capi.de_destroy(b)
        capi.de_destroy(a)
