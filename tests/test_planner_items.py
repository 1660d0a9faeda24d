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


def test_automatic_splits_stay_in_one_wave():
    """Plans that the planner splits along k make no more units (items x
    column tiles) than run at once on 152 SMs: two per SM, or one that covers
    two column tiles."""
    rng = np.random.default_rng(5)
    split = 0
    sizes = [(624, 9056, 45, 8, 16), (592, 3936, 217, 4, 32), (1952, 3024, 51, 4, 16),
             (976, 3568, 120, 8, 8), (640, 15888, 122, 8, 8), (384, 7936, 245, 4, 32),
             (272, 10640, 66, 8, 8), (1936, 15120, 25, 16, 8), (256, 6160, 147, 4, 16),
             (672, 10592, 369, 4, 64), (608, 14112, 70, 16, 8)]
    sizes += [(16 * int(2 ** rng.uniform(4, 7)), 16 * int(2 ** rng.uniform(6, 9.5)),
               int(2 ** rng.uniform(4, 9)), int(rng.choice([4, 8, 16])),
               int(rng.choice([8, 16, 32]))) for _ in range(60)]
    for m, k, n, b, d in sizes:
        i = _plan(_mask(rng, m // b, k // b, "uniform", 1 / d), b, n).info()
        if i["n_items"] < 1.9 * i["n_groups"]:
            continue
        split += 1
        cols, slots = (256, 152) if i["auto_col_tiles"] == 2 else (128, 304)
        assert i["n_items"] * -(-n // cols) <= slots, (m, k, n, b, d, i)
    assert split >= 30


@pytest.mark.parametrize("m,k,n,b,d,kind", [
    (4096, 16384, 24, 8, 1 / 8, "split"), (4096, 16384, 200, 8, 1 / 8, "wide split"),
    (4096, 4096, 100, 4, 1 / 8, "split"), (4096, 4096, 1000, 4, 1 / 8, "one wave"),
    (4096, 4096, 1000, 16, 1 / 4, "one wave"), (1024, 1024, 24, 16, 1 / 16, "rule"),
    (4096, 4096, 2048, 16, 1 / 16, "one wave")])
def test_shapes_by_kind(m, k, n, b, d, kind):
    """Which shape AUTO plans take: groups split along k (over two column
    tiles per CTA), near-equal groups that fill the SMs once, or the
    rows-per-group rule."""
    i = _plan(_mask(np.random.default_rng(1), m // b, k // b, "uniform", d), b, n).info()
    split = i["n_reductions"] == i["n_groups"]
    assert split == ("split" in kind) and (i["auto_col_tiles"] == 2) == ("wide" in kind)
    if kind == "one wave":       # one unit per SM, or one per CTA slot
        assert i["rows_per_group"] == 0 and i["n_items"] * -(-n // 128) in (152, 304)
    if kind == "rule":
        assert (i["rows_per_group"], i["n_items"]) == (1, m // 16)
