"""FP64 batches whose runs differ widely: rotations that run as digit products
beside rows too long for them, against the same runs one handle at a time."""
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


def _runs(handle, n):
    try:
        capi.de_run(handle, n)
        return [capi.de_get_population(handle, r) for r in range(n)]
    finally:
        capi.de_destroy(handle)


@pytest.mark.parametrize("shapes", [
    [(40, 128, 1, True), (9, 1500, 0, False)],  # (np, d, objective, rotated)
    [(17, 16, 3, True), (64, 100, 1, True), (8, 2200, 1, False)],
])
def test_long_rows_beside_a_sliced_rotation(shapes):
    cfgs = [capi.make_config(n, d, objective=obj, shift=problems.shift(d, seed=r),
                             rot=problems.rotation(d, seed=r) if rot else None, seed=5, run_id=r, max_generations=4,
                             target_error=0.0) for r, (n, d, obj, rot) in enumerate(shapes)]
    batch = _runs(capi.de_init_batch(cfgs), len(cfgs))
    for (xb, fb), c in zip(batch, cfgs):
        x, f = _runs(capi.de_init(c), 1)[0]
        assert np.array_equal(x, xb) and np.array_equal(f, fb)
