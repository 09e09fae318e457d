"""The FP64 rotation as digit products on the tensor cores (de_slice.cuh),
against the same objective in extended precision and against the oracle: tile
and K-step edges, rows that take the DFMA chain, non-finite rows, matrices that
are not sliced, and row groups of a composition function."""
import numpy as np
import pytest

import oracle
from paper_2405_16551_gb300 import capi, problems

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _eval(obj, x, o, M, ld=None, **kw):
    torch = _torch()
    n, d = x.shape
    ld = ld or d
    buf = np.full((n, ld), 1e30)
    buf[:, :d] = x
    xd = torch.from_numpy(buf).cuda()
    f = torch.full((n + 3,), -7.0, dtype=torch.float64, device="cuda")
    h = capi.de_init(capi.make_config(8, d, objective=obj, shift=o, rot=M, **kw))
    try:
        capi.de_eval(h, 0, xd.data_ptr(), ld, n, f.data_ptr())
        torch.cuda.synchronize()
    finally:
        capi.de_destroy(h)
    f = f.cpu().numpy()
    assert np.all(f[n:] == -7.0), "written past the last row"
    return f[:n]


def _z(x, o, M):
    L = np.longdouble
    return (x.astype(L) - o.astype(L)).astype(np.float64).astype(L) @ M.astype(L).T


def _sphere_bound(z):
    """Rounding of sum z^2: 1 per z (2 in the square), 1 per fma of a lane's at
    most 4 terms, 5 in the tree; doubled."""
    return 24 * U * (z * z).sum(1)


@pytest.mark.parametrize("d,n", [(16, 1), (17, 7), (31, 8), (33, 9), (48, 300), (64, 65), (100, 1217), (112, 8),
                                 (113, 40), (127, 17), (128, 2433)])
def test_sphere_rotation_to_a_few_ulps(d, n):
    o, M = problems.shift(d, seed=d), problems.rotation(d, seed=d)
    x = problems.population(n, d, seed=n)
    z = _z(x, o, M)
    f = _eval(0, x, o, M, ld=d + 3)
    assert np.all(np.abs(f - (z * z).sum(1)) <= _sphere_bound(z))


@pytest.mark.parametrize("scale", [1e-290, 1e-30, 1e30, 1e140])
def test_row_exponents(scale):
    """Row sizes over the exponent range (the extreme ones take the chain)."""
    d, n = 40, 24
    M = problems.rotation(d, seed=3)
    x = problems.population(n, d, seed=4) * scale
    z = _z(x, np.zeros(d), M)
    f = _eval(0, x, np.zeros(d), M)
    ref = (z * z).sum(1)
    assert np.all(np.abs(f - ref) <= _sphere_bound(z) + 2 * d * d * U * ref + 1e-323)


def test_rows_with_few_large_coordinates_are_as_exact_as_the_chain():
    """One coordinate far above the rest, in some rows of a tile: z_j is one
    product and small terms, which the splitting would lose."""
    d, n = 100, 21
    M = problems.rotation(d, seed=5)
    x = problems.population(n, d, seed=6)
    for r in range(0, n, 3):
        x[r] *= 1e-9
        x[r, r] = 1e9
    x[20] = 0.0
    z = _z(x, np.zeros(d), M)
    f = _eval(0, x, np.zeros(d), M)
    ref = (z * z).sum(1)
    # the chain's d roundings on sums without cancellation
    assert np.all(np.abs(f - ref) <= _sphere_bound(z) + 2 * d * U * ref)
    assert f[20] == 0.0


def test_matrices_that_are_not_sliced():
    """A block matrix on coordinates of very different size: the large ones
    cancel to exactly 0 in their block, and the small ones keep their precision."""
    d = 48
    M = np.zeros((d, d))
    M[:4, :4] = [[1, -1, 0, 0], [0, 1, -1, 0], [0, 0, 1, -1], [1, 0, 0, -1]]
    for b in range(4, d, 4):
        M[b:b + 4, b:b + 4] = problems.rotation(4, seed=b + 1)
    x = np.full((9, d), 1e-6)
    x[:, :4] = 1e9
    z = _z(x, np.zeros(d), M)
    assert np.all(z[:, :4] == 0)
    f = _eval(0, x, np.zeros(d), M)
    assert np.all(np.abs(f - (z * z).sum(1)) <= 2 * _sphere_bound(z))
    w = np.linspace(1, 2, d)
    f = _eval(0, x, np.zeros(d), np.diag(w))
    ref = ((x * w) ** 2).sum(1)
    assert np.all(np.abs(f - ref) <= 64 * U * ref)


def test_non_finite_rows():
    d, n = 50, 16
    o, M = problems.shift(d, seed=7), problems.rotation(d, seed=7)
    x = problems.population(n, d, seed=8)
    x[1, 3], x[2, 7], x[9, 0], x[10, :] = np.inf, np.nan, -np.inf, np.inf
    f = _eval(0, x, o, M)
    with np.errstate(all="ignore"):
        z = (x - o) @ M.T
    ok = np.isfinite(x).all(1)
    ref = _z(x[ok], o, M)
    assert np.all(np.abs(f[ok] - (ref * ref).sum(1)) <= _sphere_bound(ref))
    assert np.all(np.isinf(f[[1, 9]])) and np.all(np.isnan(f[[2, 10]])), (f[[1, 2, 9, 10]], z.shape)


@pytest.mark.parametrize("obj,d,n", [(18, 17, 20001), (19, 100, 777), (20, 33, 64), (16, 60, 130), (9, 25, 9)])
def test_suite_rows_match_the_oracle(obj, d, n):
    s = problems.suite(obj, d, seed=obj)
    x = problems.population(n, d, seed=9)
    f = _eval(obj, x, s["shift"], s["rot"], perm=s["perm"], scale=s["scale"])
    fo, S = oracle.evaluate(obj, x, s["shift"], s["rot"], scale=s["scale"], perm=s["perm"])
    assert np.all(np.abs(f - fo) <= 1e-12 * (np.abs(fo) + S))


@pytest.mark.parametrize("persist", ["0", "1"])
@pytest.mark.parametrize("obj,d,np_,jde", [(18, 16, 10100, False), (1, 128, 700, True), (3, 90, 1216, False)])
def test_generation_matches_the_oracle(obj, d, np_, jde, persist, monkeypatch):
    """One generation: shares of several tiles (and of more than one row group
    of a composition function) per CTA, and the persistent kernel."""
    _torch()
    monkeypatch.setenv("DE_GB300_FP64_PERSIST", persist)
    monkeypatch.setenv("DE_GB300_AUTOTUNE", "0")
    s = problems.suite(obj, d, seed=2) if obj > 4 else dict(shift=problems.shift(d), rot=problems.rotation(d))
    X = problems.population(np_, d, seed=11)
    fX, _ = oracle.evaluate(obj, X, s["shift"], s["rot"])
    h = capi.de_init(capi.make_config(np_, d, objective=obj, shift=s["shift"], rot=s["rot"], seed=3, jde=jde,
                                      max_generations=50, target_error=0.0, debug_capture=True))
    try:
        capi.de_set_population(h, 0, X, fX)
        capi.de_step(h, 1)
        g = capi.de_get_debug(h)
        best = capi.de_get_best(h)
        x1, f1 = capi.de_get_population(h)
    finally:
        capi.de_destroy(h)
    kw = dict(jde=True, jF=np.full(np_, 0.5), jCR=np.full(np_, 0.9)) if jde else {}
    r = oracle.step(X, fX, 0.5, 0.9, -100, 100, obj, s["shift"], s["rot"], seed=3, generation=1, **kw)
    assert np.array_equal(g["trial"], r["trial"]) and np.array_equal(g["mask"], r["mask"])
    tol = 1e-12 * (np.abs(r["f_trial"]) + r["sabs_trial"])
    assert np.all(np.abs(g["f_trial"] - r["f_trial"]) <= tol)
    band = np.abs(r["f_trial"] - fX) <= tol
    assert np.array_equal(g["accept"][~band], r["accept"][~band])
    assert best["best_index"] == int(np.argmin(f1)) and best["best_f"] == f1.min() and best["generations"] == 1
