"""Which kernel a b = 1 product runs (``gather_form`` of the plan's info): X in
shared memory where that is clearly the faster one, the row items where few
non-zeros, a heavy band of rows, a band of columns per row or short pieces of
X would leave it waiting.  Each case was timed with both kernels; the faster
one is at least 1.3 times as fast.  Host-only plans: no GPU.
"""
import numpy as np
import pytest

from paper_2303_16999_gb300 import spmm as S


def _form(m, k, n, mask, dt=S.F16, **kw):
    r, c = np.nonzero(mask)
    p = S.Plan(m, k, n, 1, w_dtype=dt, brow=r, bcol=c, kernel="gather", host_only=True, **kw)
    return p.info()["gather_form"]


def _uniform(m, k, d, seed=0):
    return np.random.default_rng(seed).random((m, k), dtype=np.float32) < d


@pytest.mark.parametrize("m,d,n,dt,form", [
    (4096, 1 / 8, 9, S.F16, 1), (4096, 1 / 8, 64, S.F16, 1), (4096, 1 / 8, 64, S.F32, 1),
    (4096, 1 / 16, 32, S.BF16, 1),
    (8192, 1 / 1024, 100, S.F16, 0), (4096, 1 / 1024, 100, S.F32, 0), (4096, 1 / 256, 64, S.F32, 0),
    (2048, 1 / 64, 20, S.F16, 0), (256, 1 / 32, 9, S.F16, 0), (512, 1 / 32, 16, S.F32, 0)])
def test_uniform(m, d, n, dt, form):
    assert _form(m, m, n, _uniform(m, m, d), dt) == form


def test_uneven_patterns():
    m = 4096
    i, j = np.arange(m)[:, None], np.arange(m)[None]
    assert _form(m, m, 64, np.abs(i - j) < m // 32, S.F32) == 0     # near the diagonal
    rows = _uniform(2048, 2048, 1 / 64)
    rows[512:576] = True                                            # 64 full rows in one place
    assert _form(2048, 2048, 64, rows, S.F32) == 0


def test_items_of_a_given_length_run_the_items():
    mask = _uniform(2048, 2048, 1 / 8)
    assert _form(2048, 2048, 32, mask) == 1
    assert _form(2048, 2048, 32, mask, max_per_item=64) == 0


def test_host_only_plans_leave_the_device_alone():
    """A process that plans on the host and asks for the plan's info holds no
    device context afterwards (a pool may fork from it)."""
    import subprocess
    import sys
    code = """
import ctypes
import numpy as np
from paper_2303_16999_gb300 import spmm as S
r, c = np.nonzero(np.random.default_rng(0).random((900, 900)) < 0.25)
S.Plan(900, 900, 32, 1, brow=r, bcol=c, kernel="gather", host_only=True).info()
try:
    cu = ctypes.CDLL("libcuda.so.1")
except OSError:
    raise SystemExit(0)              # no driver here
flags, active = ctypes.c_uint(), ctypes.c_int()
st = cu.cuDevicePrimaryCtxGetState(0, ctypes.byref(flags), ctypes.byref(active))
assert st != 0 or not active.value, (st, active.value)
"""
    p = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True,
                       cwd=S.os.path.dirname(S.HERE))
    assert p.returncode == 0, p.stderr[-2000:]
