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


def _cfgs(shapes, gens, **kw):
    return [capi.make_config(n, d, objective=obj, shift=problems.shift(d, seed=r),
                             rot=problems.rotation(d, seed=r) if rot else None, seed=5, run_id=r,
                             max_generations=gens + 3 * r, target_error=0.0, **kw)
            for r, (n, d, obj, rot) in enumerate(shapes)]


def _populations(shapes):
    """Rows of every kind: ordinary, one coordinate far above the rest (they take
    the chain), at the optimum."""
    out = []
    for r, (n, d, _, _) in enumerate(shapes):
        x = problems.population(n, d, seed=r)
        x[::5] *= 1e-7
        x[::5, r % d] = 90.0
        x[-1] = problems.shift(d, seed=r)
        out.append(x)
    return out


# every width of the operands and the edges of each, whole and partial tiles,
# more tiles of a width than one CTA takes, and runs that are not sliced
_SHAPES = [(64, 16, 1, True), (9, 17, 3, True), (130, 32, 2, True), (4, 33, 1, True), (71, 48, 0, True),
           (40, 49, 2, True), (150, 64, 3, True), (33, 65, 1, True), (64, 128, 3, True), (50, 10, 1, True),
           (20, 40, 0, False)]


@pytest.mark.parametrize("persist", ["0", "1"])
@pytest.mark.parametrize("copies", [1, 4])
@pytest.mark.parametrize("kw", [{}, dict(jde=True), dict(strategy=capi.DE_BEST1BIN)])
def test_every_width_in_one_batch(kw, copies, persist, monkeypatch):
    """The digit products on mma.sync (several CTAs per SM), on tcgen05 and the
    chain side by side give each run what it gets by itself."""
    monkeypatch.setenv("DE_GB300_FP64_PERSIST", persist)
    shapes = _SHAPES * copies
    cfgs, pops = _cfgs(shapes, 6, **kw), _populations(shapes)
    h = capi.de_init_batch(cfgs)
    for r, x in enumerate(pops):
        capi.de_set_population(h, r, x)
    batch = _runs(h, len(cfgs))
    monkeypatch.setenv("DE_GB300_FP64_PERSIST", "1")
    for r in range(len(shapes) - len(_SHAPES), len(shapes)):
        h = capi.de_init(cfgs[r])
        capi.de_set_population(h, 0, pops[r])
        x, f = _runs(h, 1)[0]
        assert np.array_equal(x, batch[r][0]) and np.array_equal(f, batch[r][1]), shapes[r]


@pytest.mark.parametrize("shapes,csize", [
    ([(64, 16, 1, True), (20, 30, 3, True), (5, 32, 0, True)], 8),
    ([(64, 64, 1, True), (9, 17, 3, True), (33, 40, 2, True)], 8),
])
def test_widths_of_the_cluster_per_run_loop(shapes, csize, monkeypatch):
    out = []
    for mode in ("3", "1"):
        monkeypatch.setenv("DE_GB300_FP64_PERSIST", mode)
        h = capi.de_init_batch(_cfgs(shapes, 20))
        assert capi.de_get_plan(h) == {"kernel_path": 3, "cluster_size": csize if mode == "3" else 0}
        out.append(_runs(h, len(shapes)))
    for (xa, fa), (xb, fb) in zip(*out):
        assert np.array_equal(xa, xb) and np.array_equal(fa, fb)


@pytest.mark.parametrize("m,np_,d", [(16, 128, 30), (12, 120, 50), (3, 500, 20)])
def test_islands_of_more_tiles_than_the_device_has_sms(m, np_, d, monkeypatch):
    out = []
    for mode in ("1", "0"):
        monkeypatch.setenv("DE_GB300_FP64_PERSIST", mode)
        cfg = capi.make_config(np_, d, objective=1, shift=problems.shift(d), rot=problems.rotation(d), seed=3,
                               max_generations=25, target_error=0.0)
        h = capi.de_init_islands(cfg, m, 4, 2)
        out.append(_runs(h, m))
    for (xa, fa), (xb, fb) in zip(*out):
        assert np.array_equal(xa, xb) and np.array_equal(fa, fb)
