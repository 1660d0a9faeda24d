"""How the planner cuts static tensor-core plans into work items, on host-only
plans: groups far above the mean length are cut, others are not, and the
length follows from the groups' entries."""
import numpy as np
import pytest

from paper_2303_16999_gb300 import spmm as S


def _plan(mask, b, n, **kw):
    r, c = np.nonzero(mask)
    return S.Plan(mask.shape[0] * b, mask.shape[1] * b, n, b, w_dtype=S.F16, brow=r, bcol=c,
                  kernel="tc", host_only=True, **kw)


def _mask(rng, mb, kb, kind, d):
    p = np.full((mb, kb), d)
    if kind == "band":
        p[mb // 4: mb // 4 + max(1, mb // 32)] = 1
    elif kind == "rows":
        p[::mb // 8] = 1
    elif kind == "falling":
        w = 1 / (1 + np.arange(mb)) ** .7
        p = np.repeat(np.minimum(1, w / w.mean() * d)[:, None], kb, 1)
    return rng.random((mb, kb)) < p


@pytest.mark.parametrize("kind", ["uniform", "band", "rows", "falling"])
@pytest.mark.parametrize("m,k,b,d,kw", [
    (2048, 2048, 8, 1 / 32, dict(rows_per_group=1)), (1024, 4096, 16, 1 / 8, dict(rows_per_group=1)),
    (4096, 4096, 16, 1 / 32, dict(rows_per_group=4)), (4080, 1040, 4, 1 / 32, dict(groups=19)),
    (4080, 1040, 4, 1 / 4, dict(rows_per_group=16)), (48, 8192, 16, 1 / 4, dict(rows_per_group=2))])
def test_item_length(m, k, b, d, kw, kind):
    """1.25 times the mean group's entries where the longest group is more
    than 32 above that, else whole groups; at least 16."""
    if kind != "uniform" and m < 128:
        kind = "falling"
    p = _plan(_mask(np.random.default_rng(m + b), m // b, k // b, kind, d), b, 24, **kw)
    i, ebeg = p.info(), p.array("grp_ebeg")
    length, total, groups = np.diff(ebeg), int(ebeg[-1]), len(ebeg) - 1
    head = max(16, -(-5 * total // (4 * groups)))
    cut = length.max() - head > 32
    assert i["max_per_item"] == (head if cut else max(head, length.max()))
    assert i["n_reductions"] == (int((length > head).sum()) if cut else 0)
    if kind == "uniform":
        assert not cut


def test_a_full_band_is_cut():
    """4 of 128 groups hold every column: their items stay near the others'
    length (whole or cut to 67 entries they took 1.2 times as long)."""
    p = _plan(_mask(np.random.default_rng(3), 256, 256, "band", 1 / 32), 8, 24)
    items = p.array("items").reshape(-1, 6)
    length = np.diff(p.array("grp_ebeg"))
    assert length.max() == 128 and (items[:, 2] - items[:, 1]).max() <= 32
    assert p.info()["n_reductions"] >= 4
