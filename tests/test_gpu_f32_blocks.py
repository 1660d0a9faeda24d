"""The FP32 block kernel that AUTO plans run (b >= 4), against the product in
64 bits.  Sizes sit on the edges of the kernel's column chunks (16, 32, 64
and 128 columns per CTA), of its 16-byte pieces and of its blocks per warp,
with aligned and unaligned rows of X and Y.

Bar: an FP32 sum of s products is off by at most s 2^-24 / (1 - s 2^-24) of
the sum of the products' magnitudes, in any order.
"""
import numpy as np
import pytest

from paper_2303_16999_gb300 import spmm as S
from paper_2303_16999_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b", [4, 8, 16])
@pytest.mark.parametrize("n,pad", [(1, 0), (3, 2), (16, 0), (17, 3), (32, 0), (33, 0), (64, 4),
                                   (65, 0), (127, 1), (128, 0), (129, 3), (300, 1)])
def test_f32_blocks(b, n, pad):
    mb, kb = 15, 165                 # rows of 0, 1, 2, ... blocks and one full row
    rng = np.random.default_rng(8100 + b + n)
    counts = [kb if r == 9 else (0, 1, 2, 3, 4, 5, 7, 8, 9)[r % 9] for r in range(mb)]
    brow = np.concatenate([np.full(c, r, np.int32) for r, c in enumerate(counts)])
    bcol = np.concatenate([rng.choice(kb, c, replace=False).astype(np.int32) for c in counts])
    order = rng.permutation(len(brow))
    brow, bcol = brow[order], bcol[order]
    vals = torch.from_numpy(rng.standard_normal((len(brow), b, b), dtype=np.float32)).cuda()
    dense = torch.zeros((mb, kb, b, b), dtype=torch.float64, device="cuda")
    dense[torch.from_numpy(brow).long(), torch.from_numpy(bcol).long()] = vals.double()
    dense = dense.transpose(1, 2).reshape(mb * b, kb * b)
    for tr in (False, True):
        w = dense.t() if tr else dense
        rows, cols = w.shape
        x = torch.full((cols, n + pad), float("nan"), device="cuda")
        x[:, :n] = torch.from_numpy(rng.standard_normal((cols, n), dtype=np.float32)).cuda()
        p = S.Plan(mb * b, kb * b, n, b, w_dtype=S.F32, brow=brow, bcol=bcol, transposed=tr)
        p.pack(vals)
        y = torch.full((rows, n + pad), float("nan"), device="cuda")
        p.run(x[:, :n], y[:, :n])
        torch.cuda.synchronize()
        assert p.status() == 0 and p.info()["kernel"] == S.KERNEL_PLAIN
        p.close()
        assert torch.isnan(y[:, n:]).all()
        want, size = w @ x[:, :n].double(), w.abs() @ x[:, :n].double().abs()
        s = (w != 0).sum(1, keepdim=True) * 2.0 ** -24
        assert ((y[:, :n].double() - want).abs() <= s / (1 - s) * size).all()
        assert (y[:, :n][(w != 0).sum(1) == 0] == 0).all()


def test_f32_blocks_row_slices_and_infinities():
    """A row slice equals those rows of the whole product, and an infinity in
    X reaches only the columns and rows that use it."""
    b, mb, kb, n = 8, 12, 20, 70
    c = wl.problem(8200, mb * b, kb * b, n, b, mb * kb // 3)
    vals, x = torch.from_numpy(c["vals"]).cuda(), torch.from_numpy(c["X"]).cuda()
    x[5, 3] = float("inf")
    out = []
    for rows in (None, (16, 56)):
        p = S.Plan(mb * b, kb * b, n, b, w_dtype=S.F32, brow=c["brow"], bcol=c["bcol"], rows=rows)
        p.pack(vals)
        out.append(p.run(x))
        torch.cuda.synchronize()
        p.close()
    assert torch.equal(out[0][16:56].nan_to_num(7.0), out[1].nan_to_num(7.0))
    used = np.isin(np.arange(mb), c["brow"][c["bcol"] == 0]).repeat(b)
    finite = torch.isfinite(out[0]).cpu().numpy()
    assert finite[:, :3].all() and finite[:, 4:].all()
    assert (finite[:, 3] == ~used).all()
