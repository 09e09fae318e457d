"""The fitness kernel's two-tile form (k_fit_tc<., 2>: several N tiles, more
one-tile CTAs than SMs): one generation against the oracle, with odd tile
counts, ragged rows and ragged N tiles."""
import numpy as np
import pytest

import oracle
from paper_2405_16551_gb300 import capi, problems

pytestmark = pytest.mark.gpu
# the bounds of tests/test_gpu_split.py
REL = {capi.DE_PREC_BF16X3: 1e-5, capi.DE_PREC_TF32X3: 1e-6}


@pytest.mark.parametrize("np_,d,obj,prec,band", [
    (9800, 300, 1, capi.DE_PREC_BF16X3, capi.DE_BAND_NEAR),   # 77 tiles x 2: the last pair has one tile
    (9985, 257, 0, capi.DE_PREC_TF32X3, capi.DE_BAND_NEAR),   # ... of one row
    (6700, 700, 3, capi.DE_PREC_BF16X3, capi.DE_BAND_ALL),    # 53 tiles x 3
    (5120, 1000, 1, capi.DE_PREC_TF32X3, capi.DE_BAND_NEAR),  # 40 tiles x 4
])
def test_pair_generation_matches_oracle(np_, d, obj, prec, band):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    o, M = problems.shift(d, seed=7), problems.rotation(d, seed=7)
    X = problems.population(np_, d, seed=7)
    fX, _ = oracle.evaluate(obj, X, o, M, threads=8)
    h = capi.de_init(capi.make_config(np_, d, objective=obj, shift=o, rot=M, seed=7, precision=prec, fp64_band=band,
                                      max_generations=10**6, target_error=0.0, debug_capture=True))
    try:
        capi.de_set_population(h, 0, X, fX)
        capi.de_set_generation(h, 0, 4)
        capi.de_step(h, 1)
        g = capi.de_get_debug(h)
        xn, fn = capi.de_get_population(h)
        best = capi.de_get_best(h)
        st = capi.de_get_stats(h)
    finally:
        capi.de_destroy(h)
    r = oracle.step(X, fX, 0.5, 0.9, -100, 100, obj, o, M, seed=7, generation=5, threads=8)
    assert np.array_equal(g["trial"], r["trial"])
    scale = np.abs(r["f_trial"]) + r["sabs_trial"]
    fp64 = g["fp64_checked"].astype(bool)
    assert np.all(np.abs(g["f_trial"] - r["f_trial"]) <= np.where(fp64, 1e-12, REL[prec]) * scale)
    rel = 1e-12 if band == capi.DE_BAND_ALL else REL[prec]
    inband = np.abs(r["f_trial"] - fX) <= rel * scale
    assert np.array_equal(g["accept"][~inband], r["accept"][~inband])
    acc = g["accept"].astype(bool)
    assert np.array_equal(xn[acc], r["trial"][acc]) and np.array_equal(xn[~acc], X[~acc])
    assert st["trials"] == np_ and best["best_index"] == int(np.argmin(fn))
