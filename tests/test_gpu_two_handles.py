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
