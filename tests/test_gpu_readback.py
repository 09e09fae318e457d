"""de_get_population into buffers of every kind: kept and never touched, aligned to
nothing, at the sizes where the copy changes its way."""
import ctypes
import mmap

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


# (up to 256 KB staged, 2 MB in untouched pages; above, rows of another stride are
# mapped first, by several threads from 16 MB on)
@pytest.mark.parametrize("np_,d", [(4, 1), (320, 100), (324, 100), (1000, 99), (3000, 100), (5000, 101), (21000, 100),
                                  (23000, 99), (55000, 100)])
def test_the_same_rows_in_every_buffer(np_, d):
    h = capi.de_init(capi.make_config(np_, d, objective=1, shift=problems.shift(d), seed=3, target_error=0.0))
    try:
        capi.de_step(h, 1)
        x, f = capi.de_get_population(h)
        n = 8 * np_ * d
        untouched = mmap.mmap(-1, n + 16384)  # pages that nobody has written
        kept = bytearray(b"\x5a" * (n + 16384))
        dp = ctypes.POINTER(ctypes.c_double)
        for buf, off in ((untouched, 4096 + 24), (kept, 40), (untouched, 4096 + 24)):
            at = ctypes.addressof(ctypes.c_char.from_buffer(buf, off))
            before, after = bytes(buf[:off]), bytes(buf[off + n:])
            fb = np.full(np_ + 2, -3.0)
            status = capi.load().de_get_population(ctypes.c_void_p(h), 0, ctypes.cast(at, dp),
                                                   fb[1:].ctypes.data_as(dp))
            assert status == capi.DE_OK
            assert buf[off:off + n] == x.tobytes() and np.array_equal(fb[1:-1], f)
            assert buf[:off] == before and buf[off + n:] == after and fb[0] == fb[-1] == -3.0
    finally:
        capi.de_destroy(h)
