"""Islands that a call has set apart go on by themselves, the same in every form
of the loop, and exchange migrants again once they are together."""
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


@pytest.mark.parametrize("kind", [capi.DE_MIGRATE_SYNC, capi.DE_MIGRATE_ASYNC])
@pytest.mark.parametrize("np_,d,rot", [(16, 8, False), (70, 20, True)])
def test_every_form_of_the_loop_agrees(np_, d, rot, kind, monkeypatch):
    cfg = capi.make_config(np_, d, objective=1, shift=problems.shift(d, seed=2),
                           rot=problems.rotation(d, seed=3) if rot else None, seed=7, target_error=0.0,
                           max_generations=10**6)
    out = []
    for mode in ("0", "1", "3"):
        monkeypatch.setenv("DE_GB300_FP64_PERSIST", mode)
        h = capi.de_init_islands_ex(cfg, 3, 5, 2, kind)
        try:
            seen = []
            for step, apart in ((6, 1), (13, None), (4, -1), (17, 0), (3, None)):
                capi.de_step(h, step)
                seen += [capi.de_get_population(h, r) for r in range(3)]
                seen += [capi.de_get_best(h, r) for r in range(3)]
                if apart is not None:
                    capi.de_reset(h, apart)
            out.append(seen)
        finally:
            capi.de_destroy(h)
    gens = [b["generations"] for b in out[0] if isinstance(b, dict)]
    assert gens == [6, 6, 6, 19, 13, 19, 23, 17, 23, 17, 17, 17, 3, 20, 20]
    for other in out[1:]:
        for a, b in zip(out[0], other):
            if isinstance(a, dict):
                assert all(np.array_equal(a[k], b[k]) for k in a)
            else:
                assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
