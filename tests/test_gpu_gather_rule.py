"""The b = 1 gather with X in shared memory on products that take it
(``gather_form``), integer-valued: sums of products are exact in FP32, so Y must
equal the 64-bit product rounded once.  n sits on the edges of the column
groups and chunks, k on those of the slices (1, 2 and 4 CTAs per cluster), m on
those of the row ranges and passes; X and Y with aligned and unaligned rows.
And calls that fall to the row items: pieces of X that the ring kernel cannot
take, items of a given length.
"""
import numpy as np
import pytest

from paper_2303_16999_gb300 import spmm as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _problem(m, k, d, dt, seed=1):
    g = torch.Generator(device="cuda").manual_seed(seed)
    w = torch.randint(1, 3, (m, k), generator=g, device="cuda").to(dt)
    w[torch.rand((m, k), generator=g, device="cuda") >= d] = 0
    r, c = w.nonzero(as_tuple=True)
    return w, r.int().cpu().numpy(), c.int().cpu().numpy()


def _run(w, r, c, n, ld=None, off=0, ypad=0, form=None, **kw):
    m, k = w.shape
    dt = w.dtype
    g = torch.Generator(device="cuda").manual_seed(n)
    ld = ld or (n + 7) // 8 * 8
    buf = torch.full((k * ld + off,), float("nan"), dtype=dt, device="cuda")
    x = buf[off:].view(k, ld)[:, :n]
    x.copy_(torch.randint(-1, 2, (k, n), generator=g, device="cuda"))
    p = S.Plan(m, k, n, 1, w_dtype=S.dtype_code(dt), brow=r, bcol=c, **kw)
    assert p.info()["kernel"] == S.KERNEL_GATHER
    if form is not None:
        assert p.info()["gather_form"] == form
    p.pack(w[w != 0].view(-1, 1, 1).contiguous())
    y = torch.full((m, n + ypad), float("nan"), dtype=dt, device="cuda")
    p.run(x, y[:, :n])
    torch.cuda.synchronize()
    assert p.status() == 0
    p.close()
    assert torch.equal(y[:, :n], (w.double() @ x.double()).to(dt))
    assert torch.isnan(y[:, n:]).all()


@pytest.mark.parametrize("dt", [torch.float16, torch.bfloat16, torch.float32])
def test_columns(dt):
    w, r, c = _problem(1501, 2001, 1 / 3, dt)
    for n in (9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 100):
        _run(w, r, c, n, form=1)
        _run(w, r, c, n, ld=n, ypad=3)             # rows unaligned for odd n
        _run(w, r, c, n, ld=n + 1, off=1)          # unaligned base


@pytest.mark.parametrize("m,k,d,n,dt,form", [
    (1200, 6001, 1 / 5, 33, torch.float16, 1), (900, 12001, 1 / 6, 30, torch.bfloat16, 1),
    (700, 20001, 1 / 6, 40, torch.float16, 1), (600, 50001, 1 / 8, 9, torch.bfloat16, 1),
    (600, 65535, 1 / 16, 9, torch.bfloat16, 0),          # a slice of k is too long
    (500, 6001, 1 / 3, 20, torch.float32, 1), (153, 3001, 1 / 2, 24, torch.float16, 1),
    (40000, 65, 1 / 2, 64, torch.float16, 1)])
def test_sizes(m, k, d, n, dt, form):
    w, r, c = _problem(m, k, d, dt)
    _run(w, r, c, n, form=form)


@pytest.mark.parametrize("n,ld", [(1, 1), (2, 3), (4, 7), (8, 9), (8, 15), (8, 8)])
def test_few_columns_and_items(n, ld):
    w, r, c = _problem(700, 1500, 1 / 8, torch.float16)
    _run(w, r, c, n, ld=ld)
    _run(w, r, c, n, ld=ld, max_per_item=33)
    _run(w, r, c, 40, max_per_item=33, form=0)
