"""More split groups than one reduction launch has blocks in y (65535): the
per-product reduction adds them.  Integer-valued, so Y must equal the 64-bit
product rounded once."""
import numpy as np
import pytest

from paper_2303_16999_gb300 import spmm as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [False, True])
def test_more_split_groups_than_grid_rows(batch):
    groups, kt, n = 65600, 4, 8
    g = torch.Generator(device="cuda").manual_seed(3)
    vals = torch.randint(-2, 3, (groups * kt, 16, 16), generator=g, device="cuda").half()
    x = torch.randint(-1, 2, (16 * kt, n), generator=g, device="cuda").half()
    brow = np.repeat(np.arange(groups, dtype=np.int32), kt)
    bcol = np.tile(np.arange(kt, dtype=np.int32), groups)
    p = S.Plan(16 * groups, 16 * kt, n, 16, w_dtype=S.F16, brow=brow, bcol=bcol, kernel="tc",
               rows_per_group=1, k_splits=2)
    assert p.info()["n_reductions"] == groups
    p.pack(vals)
    y = torch.full((16 * groups, n), float("nan"), dtype=torch.float16, device="cuda")
    if batch:
        S.spmm_batch_run([p], [x], [y])
    else:
        p.run(x, y)
    torch.cuda.synchronize()
    assert p.status() == 0
    p.close()
    w = vals.view(groups, kt, 16, 16).transpose(1, 2).reshape(16 * groups, 16 * kt)
    assert torch.equal(y, (w.double() @ x.double()).half())
