"""Griewank's cosine from a 117-bit product, Elliptic's weights from a table, and
composition rows finished and mixed across a row group: against extended
precision and the oracle, at the edges of a row group and at the optima."""
import numpy as np
import pytest

import oracle
from paper_2405_16551_gb300 import capi, problems

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _eval(obj, x, o, M=None):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n, d = x.shape
    xd = torch.from_numpy(x).cuda()
    f = torch.zeros(n, dtype=torch.float64, device="cuda")
    h = capi.de_init(capi.make_config(8, d, objective=obj, shift=o, rot=M, lo=-1e9, hi=1e9))
    try:
        capi.de_eval(h, 0, xd.data_ptr(), d, n, f.data_ptr())
        torch.cuda.synchronize()
    finally:
        capi.de_destroy(h)
    return f.cpu().numpy()


@pytest.mark.parametrize("d", [1, 2, 33, 128, 700])
@pytest.mark.parametrize("size", [1e-300, 1e-9, 1e-3, 1.0, 30.0, 600.0, 1e6])
def test_griewank_terms(d, size):
    L = np.longdouble
    w = np.random.default_rng(d).uniform(-1, 1, (16, d)) * size
    w[0] = 0.0
    s = (w.astype(L) ** 2).sum(1) / 4000
    p = np.cos(w.astype(L) / np.sqrt(np.arange(1, d + 1, dtype=L))).prod(1)
    f = _eval(14, w, np.zeros(d))
    # 1 rounding per square and per sum step of a lane's ceil(d / 32) terms, 5 in
    # the tree, 3 in the result; a factor of the product is off by its
    # rounding and its argument's size 2^-63 (the constant's 2^-59 relative, and
    # extended precision's own 2^-64 of the argument)
    steps = -(-d // 32) + 5 + 3
    arg = np.abs(w) / np.sqrt(np.arange(1, d + 1))
    tol = steps * U * (s + 2.0) + (U * steps + (arg * 2.0 ** -58).sum(1)) + d * U
    assert np.all(np.abs(f - (s - p + 1)) <= tol)
    w[3, d // 2] = np.inf
    assert not np.isfinite(_eval(14, w, np.zeros(d))[3])


@pytest.mark.parametrize("d", [1, 2, 40])
def test_elliptic_weights(d):
    L = np.longdouble
    w = np.random.default_rng(d).uniform(-100, 100, (9, d))
    c = L(10) ** (L(6) * np.arange(d, dtype=L) / max(d - 1, 1))
    ref = (c * w.astype(L) ** 2).sum(1)
    # pow within 2 ulp of a quotient that is within half an ulp (times 6 ln 10), 2
    # roundings per term, 2 per lane, 5 in the tree
    assert np.all(np.abs(_eval(13, w, np.zeros(d)) - ref) <= (2 + 14 + 2 + 2 + 5) * 2 * U * ref)


@pytest.mark.parametrize("obj,d,n", [(18, 16, 64), (19, 100, 65), (20, 33, 130), (19, 10, 9), (20, 128, 7)])
def test_composition_rows(obj, d, n):
    s = problems.suite(obj, d, seed=3)
    x = problems.population(n, d, seed=4)
    nc = s["shift"].shape[0]
    for c in range(nc):  # weight 1 for the component whose optimum it is
        x[(c * 37 + 5) % n] = s["shift"][c]
    f = _eval(obj, x, s["shift"], s["rot"])
    fo, S = oracle.evaluate(obj, x, s["shift"], s["rot"])
    assert np.all(np.abs(f - fo) <= 1e-12 * (np.abs(fo) + S))
