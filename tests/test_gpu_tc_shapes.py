"""Launch shapes of the static tensor-core plans, on integer-valued operands:
sums of products are exact in FP32, so Y must equal the 64-bit product rounded
once to the output type, whatever the groups, splits and column tiles.
"""
import numpy as np
import pytest

from paper_2303_16999_gb300 import spmm as S
from paper_2303_16999_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _problem(seed, m, k, n, b, nnzb, dt):
    c = wl.integer_problem(seed, m, k, n, b, nnzb)
    vals = torch.from_numpy(c["vals"]).to(dt).cuda()
    x = torch.full((k, (n + 7) // 8 * 8), float("nan"), dtype=dt, device="cuda")
    x[:, :n] = torch.from_numpy(c["X"]).to(dt)
    w = torch.zeros((m // b, k // b, b, b), dtype=torch.float64, device="cuda")
    w[torch.from_numpy(c["brow"]).long(), torch.from_numpy(c["bcol"]).long()] = vals.double()
    want = w.transpose(1, 2).reshape(m, k) @ x[:, :n].double()
    return c, vals, x[:, :n], want.to(dt)


def _run(c, vals, x, want, pad=0, **kw):
    m, n = want.shape
    p = S.Plan(c["m"], c["k"], n, c["b"], w_dtype=S.dtype_code(vals.dtype), brow=c["brow"],
               bcol=c["bcol"], kernel="tc", **kw)
    p.pack(vals)
    y = torch.full((m, n + pad), float("nan"), dtype=want.dtype, device="cuda")
    p.run(x, y[:, :n])
    torch.cuda.synchronize()
    info = p.info()
    assert p.status() == 0
    p.close()
    assert torch.equal(y[:, :n], want)
    assert torch.isnan(y[:, n:]).all()
    return info


@pytest.mark.parametrize("n", [1, 8, 63, 65, 72, 100, 127, 129, 191, 200, 257, 450])
@pytest.mark.parametrize("geo,ct", [(1, 1), (2, 1), (1, 2), (2, 2)])
def test_joint_boxes_with_2d_maps(n, geo, ct):
    """Stages of consecutive tile columns (every tile present) with n not a
    multiple of 64: one box of slabs per 64-column half, the upper half
    absent where it lies past n; k ends inside a box (31 tile columns)."""
    case = _problem(300 + n, 272, 496, n, 4, 68 * 124 // 2, torch.bfloat16)
    _run(*case, rows_per_group=16, stage_geometry=geo, col_tiles=ct)


@pytest.mark.parametrize("n,pad", [(1, 0), (3, 1), (4, 0), (5, 3), (64, 4), (100, 2), (131, 0)])
@pytest.mark.parametrize("splits", [2, 7, 8, 9, 20])
def test_split_groups_reduction(n, pad, splits):
    """The reduction of groups split along k: values a thread adds run over
    row ends (n not a multiple of 4), rows of Y aligned and not, and more
    partials than one pass of loads (8)."""
    case = _problem(500 + n, 400, 1600, n, 8, 50 * 200 // 4, torch.float16)
    info = _run(*case, pad=pad, rows_per_group=16, k_splits=splits)
    assert info["n_reductions"] == 2 and info["n_items"] > 2 * (splits - 1)


@pytest.mark.parametrize("m,k,n,b,d,dt", [
    (4096, 16384, 24, 8, 1 / 8, torch.bfloat16), (4096, 16384, 200, 8, 1 / 8, torch.float16),
    (4096, 4096, 100, 4, 1 / 8, torch.bfloat16), (1024, 4096, 33, 8, 1 / 4, torch.float16),
    (1024, 1024, 128, 8, 1 / 8, torch.bfloat16), (48, 8192, 300, 16, 1 / 2, torch.float16),
    (16, 65536, 9, 16, 1.0, torch.bfloat16), (2048, 32, 64, 4, 1 / 2, torch.float16)])
def test_planner_shapes_exact(m, k, n, b, d, dt):
    """Plans whose shape the planner chooses, against the 64-bit product; a
    col_tiles option changes neither groups nor splits."""
    case = _problem(m + n, m, k, n, b, int((m // b) * (k // b) * d), dt)
    infos = [_run(*case, col_tiles=ct) for ct in (0, 1, 2)]
    for f in ("rows_per_group", "max_per_item", "n_items", "n_reductions"):
        assert len({i[f] for i in infos}) == 1, f


def test_batch_of_split_plans_one_reduction():
    """Several split plans of one batch share a reduction launch (odd and even
    n, padded Y); each equals its exact product."""
    plans, xs, ys, wants = [], [], [], []
    for i, n in enumerate((3, 40, 129, 64, 20)):
        c, vals, x, want = _problem(700 + i, 320 + 16 * i, 2048, n, 8, (40 + 2 * i) * 64,
                                    torch.bfloat16)
        p = S.Plan(c["m"], c["k"], n, 8, w_dtype=S.BF16, brow=c["brow"], bcol=c["bcol"],
                   kernel="tc", **({} if i == 3 else dict(rows_per_group=16, k_splits=3 + i)))
        p.pack(vals)
        plans.append(p)
        xs.append(x)
        ys.append(torch.full((c["m"], n + i), float("nan"), dtype=torch.bfloat16,
                             device="cuda")[:, :n])
        wants.append(want)
    S.spmm_batch_run(plans, xs, ys)
    torch.cuda.synchronize()
    for p, y, want in zip(plans, ys, wants):
        assert p.status() == 0 and torch.equal(y, want)
        p.close()


@pytest.mark.parametrize("dt", ["f16", "bf16", "e4m3"])
@pytest.mark.parametrize("geo", [1, 2])
@pytest.mark.parametrize("extra", [-1, 0, 1])
def test_deep_ring_units(dt, geo, extra):
    """One work unit per SM or fewer takes the deep ring, one more unit does
    not; 40 entries per unit, so every ring wraps."""
    g = torch.cuda.get_device_properties(0).multi_processor_count + extra
    xdt = torch.float16 if dt == "f16" else torch.bfloat16
    c, vals, x, want = _problem(40 + g, 16 * g, 640, 72, 8, g * 2 * 80 // 2, xdt)
    if dt != "e4m3":
        _run(c, vals, x, want, rows_per_group=1, stage_geometry=geo)
        return
    p = S.Plan(16 * g, 640, 72, 8, w_dtype=S.E4M3, x_dtype=S.BF16, brow=c["brow"], bcol=c["bcol"],
               kernel="tc", rows_per_group=1, stage_geometry=geo)
    p.pack(vals.to(torch.float8_e4m3fn), torch.ones(len(c["brow"]), device="cuda"))
    y = p.run(x)
    torch.cuda.synchronize()
    assert p.status() == 0 and torch.equal(y, want)
    p.close()
