"""The b = 1 gather with X in shared memory (static plans), on integer-valued
operands: sums of products are exact in FP32, so Y must equal the 64-bit
product rounded once to the output type.  n sits on the edges of the column
groups (8, 16, 32 and 64 columns of 16-bit values, 4 to 32 of FP32), k on
those of the parts and clusters, rows on those of the 32-non-zero loads.
"""
import numpy as np
import pytest

from paper_2303_16999_gb300 import spmm as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _case(seed, m, k, counts):
    rng = np.random.default_rng(seed)
    brow = np.repeat(np.arange(m, dtype=np.int32), counts)
    bcol = np.concatenate([rng.choice(k, c, replace=False) for c in counts] or [[]]).astype(np.int32)
    order = rng.permutation(len(brow))
    vals = torch.from_numpy(rng.integers(-2, 3, len(brow)).astype(np.float32)).cuda()
    return brow[order], bcol[order], vals


def _check(m, k, n, dt, case, ld=None, off=0, **kw):
    brow, bcol, vals = case
    rng = np.random.default_rng(n)
    rows, cols = (k, m) if kw.get("transposed") else (m, k)
    ld = ld or n
    buf = torch.full((cols * ld + off,), float("nan"), dtype=dt, device="cuda")
    x = buf[off:].view(cols, ld)[:, :n]
    x.copy_(torch.from_numpy(rng.integers(-1, 2, (cols, n))))
    w = torch.sparse_coo_tensor(torch.from_numpy(np.stack([brow, bcol]).astype(np.int64)),
                                vals.double().cpu(), (m, k)).to_dense().cuda()
    w = w.t() if kw.get("transposed") else w
    if "rows" in kw:
        w, rows = w[slice(*kw["rows"])], kw["rows"][1] - kw["rows"][0]
    p = S.Plan(m, k, n, 1, w_dtype=S.dtype_code(dt), brow=brow, bcol=bcol, kernel="gather", **kw)
    p.pack(vals.to(dt).view(-1, 1, 1))
    y = torch.full((rows, n + 3), float("nan"), dtype=dt, device="cuda")
    p.run(x, y[:, :n])
    torch.cuda.synchronize()
    assert p.status() == 0
    p.close()
    assert torch.equal(y[:, :n], (w @ x.double()).to(dt))
    assert torch.isnan(y[:, n:]).all()


COUNTS = (0, 1, 7, 31, 32, 33, 64, 127, 128, 129, 160, 255, 256, 257, 300)


@pytest.mark.parametrize("dt", [torch.float16, torch.bfloat16, torch.float32])
@pytest.mark.parametrize("n", [3, 5, 7, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 100, 130])
def test_columns(n, dt):
    m, k = 45, 601
    case = _case(n, m, k, [COUNTS[r % len(COUNTS)] for r in range(m)])
    _check(m, k, n, dt, case)                                  # rows of X unaligned for odd n
    _check(m, k, n, dt, case, ld=(n + 7) // 8 * 8)             # 16-byte rows
    _check(m, k, n, dt, case, ld=n + 1, off=1)                 # unaligned base


@pytest.mark.parametrize("m,k,n,dt", [
    (5, 1, 9, torch.float16), (3, 7, 12, torch.float32), (40, 8, 33, torch.bfloat16),
    (30, 13900, 8, torch.float16),       # one vector per row, too large for the ring kernel
    (300, 6000, 32, torch.float16),      # two CTAs per cluster
    (700, 12000, 30, torch.bfloat16),    # four
    (200, 20000, 40, torch.float16),     # four, in chunks of 16 columns
    (64, 65536, 9, torch.bfloat16), (64, 65537, 9, torch.float16),
    (50, 6000, 20, torch.float32), (50, 9000, 64, torch.float32)])
def test_sizes(m, k, n, dt):
    rng = np.random.default_rng(m + k)
    _check(m, k, n, dt, _case(m, m, k, rng.integers(0, min(k, 700) + 1, m)))


def test_more_rows_than_partials_fit():
    m, k, n = 150000, 64, 64
    rng = np.random.default_rng(0)
    brow = np.repeat(np.arange(m, dtype=np.int32), 2)
    bcol = np.stack([rng.integers(0, 32, m), rng.integers(32, 64, m)], 1).reshape(-1).astype(np.int32)
    vals = torch.from_numpy(rng.integers(-2, 3, 2 * m).astype(np.float32)).cuda()
    _check(m, k, n, torch.float16, (brow, bcol, vals))


def test_transposed_slices_and_infinities():
    m, k, n = 200, 500, 24
    rng = np.random.default_rng(4)
    case = _case(4, m, k, rng.integers(0, 200, m))
    _check(m, k, n, torch.bfloat16, case, transposed=True)
    _check(m, k, n, torch.float16, case, rows=(33, 160))
    brow, bcol, vals = case
    x = torch.ones((k, n), dtype=torch.float16, device="cuda")
    x[7, 5] = float("inf")
    p = S.Plan(m, k, n, 1, w_dtype=S.F16, brow=brow, bcol=bcol, kernel="gather")
    y = p.run(x, values=torch.ones_like(vals).half())
    used = torch.from_numpy(np.isin(np.arange(m), brow[bcol == 7])).cuda()
    assert torch.isfinite(y[:, :5]).all() and torch.isfinite(y[:, 6:]).all()
    assert torch.equal(torch.isinf(y[:, 5]), used)
    p.close()
