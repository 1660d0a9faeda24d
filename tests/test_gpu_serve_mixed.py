"""Serving weights that differ in stage geometry, in type and in whether their
plans split rows, on several
launches in flight at a time.  Operands are integer-valued, so every Y must equal the
64-bit product rounded once, whatever shares a launch with it.
"""
import pytest

from paper_2303_16999_gb300 import spmm as S
from paper_2303_16999_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _weight(seed, m, k, n_max, b, d, wt="f16", **kw):
    """A packed plan and its 64-bit dense weight; wt: f16, bf16 or e4m3 (unit
    scales; small integers are exact in all three)."""
    xdt = torch.float16 if wt == "f16" else torch.bfloat16
    c = wl.integer_problem(seed, m, k, 1, b, int((m // b) * (k // b) * d))
    vals = torch.from_numpy(c["vals"]).cuda()
    w = torch.zeros((m // b, k // b, b, b), dtype=torch.float64, device="cuda")
    w[torch.from_numpy(c["brow"]).long(), torch.from_numpy(c["bcol"]).long()] = vals.double()
    code = S.E4M3 if wt == "e4m3" else S.dtype_code(xdt)
    p = S.Plan(m, k, n_max, b, w_dtype=code, x_dtype=S.dtype_code(xdt), brow=c["brow"],
               bcol=c["bcol"], kernel="tc", **kw)
    if wt == "e4m3":
        p.pack(vals.to(torch.float8_e4m3fn), torch.ones(len(c["brow"]), device="cuda"))
    else:
        p.pack(vals.to(xdt))
    return dict(plan=p, w=w.transpose(1, 2).reshape(m, k), dt=xdt, m=m, k=k)


def _requests(ws, ids, seq):
    """(weight id, X, Y, wanted Y) of each (weight, n)."""
    g = torch.Generator().manual_seed(len(seq))
    out = []
    for i, n in seq:
        x = torch.randint(-1, 2, (ws[i]["k"], n), generator=g).to(ws[i]["dt"])
        y = torch.full((ws[i]["m"], n), float("nan"), dtype=ws[i]["dt"]).pin_memory()
        out.append((ids[i], x.pin_memory(), y, (ws[i]["w"] @ x.double().cuda()).to(ws[i]["dt"]).cpu()))
    return out


def _serve(srv, reqs):
    tickets = [srv.submit(w, x, y) for w, x, y, _ in reqs]
    for t in tickets:
        srv.wait(t)
    for _, _, y, want in reqs:
        assert torch.equal(y, want)


def test_both_geometries_on_four_launches():
    """New weights of either stage geometry, first requests of all of them at
    once: launches of two requests, four in flight, whose other-geometry
    records do not exist yet."""
    for rnd in range(6):
        ws = [_weight(20 * rnd + i, 512, 1024, 64, 8, 1 / 4, stage_geometry=1 + i % 2)
              for i in range(6)]
        assert {w["plan"].info()["stage_geometry"] for w in ws} == {0, 1}
        assert all(w["plan"].info()["n_reductions"] == 0 for w in ws)
        torch.cuda.synchronize()
        srv = S.Server(hbm_budget_bytes=64 << 20, max_inflight=4, max_batch=2)
        ids = [srv.register(w["plan"]) for w in ws]
        pairs = [(0, 1), (1, 2), (3, 0), (2, 5), (4, 1), (5, 4), (1, 0), (3, 2)]
        reqs = _requests(ws, ids, [(i, 8 + 5 * q) for q, p in enumerate(pairs) for i in p])
        _serve(srv, reqs)
        assert srv.stats()["failed"] == 0
        srv.close()
        for w in ws:
            assert w["plan"].status() == 0
            w["plan"].close()


def test_types_do_not_share_a_launch():
    """F16, BF16 and E4M3 weights in one queue, all of it there before the
    second launch: neighbours of one type may share one, others never do."""
    ws = [_weight(200 + i, 256, 512, 64, 8, 1 / 4, wt=t)
          for i, t in enumerate(("f16", "bf16", "e4m3", "f16"))]
    torch.cuda.synchronize()
    srv = S.Server(hbm_budget_bytes=64 << 20, max_inflight=2, inject_delay_us=100000)
    ids = [srv.register(w["plan"]) for w in ws]
    seq = [0, 0, 1, 2, 2, 1, 3, 0, 2, 0]
    _serve(srv, _requests(ws, ids, [(i, 5 + 6 * q) for q, i in enumerate(seq)]))
    st = srv.stats()
    srv.close()
    assert st["completed"] == len(seq) and st["failed"] == 0
    assert st["launches"] >= 7        # runs of one type: 0 0 | 1 | 2 2 | 1 | 3 0 | 2 | 0
    for w in ws:
        assert w["plan"].status() == 0
        w["plan"].close()


def _split_weight(seed):
    """A wide weight that the planner splits along k."""
    w = _weight(seed, 512, 4096, 64, 8, 1 / 8)
    assert w["plan"].info()["n_reductions"] > 0
    return w


def test_burst_to_a_split_weight_is_one_launch():
    """The first request goes out alone; the others are all there when the
    next launch is made, and share it."""
    ws = [_split_weight(300), _weight(301, 512, 512, 64, 8, 1 / 4)]
    torch.cuda.synchronize()
    srv = S.Server(hbm_budget_bytes=256 << 20, max_inflight=2, inject_delay_us=100000)
    ids = [srv.register(w["plan"]) for w in ws]
    _serve(srv, _requests(ws, ids, [(1 if q % 5 == 3 else 0, 1 + 3 * q) for q in range(17)]))
    st = srv.stats()
    srv.close()
    assert st["failed"] == 0 and st["launches"] == 2
    assert all(w["plan"].status() == 0 for w in ws)


def test_split_weight_on_four_launches():
    """Launches of two requests, four in flight, all to one split weight and
    one other: each has partials of its own."""
    ws = [_split_weight(310), _weight(311, 512, 1024, 64, 8, 1 / 4)]
    torch.cuda.synchronize()
    srv = S.Server(hbm_budget_bytes=256 << 20, max_inflight=4, max_batch=2)
    ids = [srv.register(w["plan"]) for w in ws]
    for rnd in range(4):
        _serve(srv, _requests(ws, ids, [(int(q % 3 == rnd), 1 + (7 * q + rnd) % 64)
                                        for q in range(32)]))
    assert srv.stats()["failed"] == 0
    srv.close()
    assert all(w["plan"].status() == 0 for w in ws)


def test_split_weight_on_a_small_budget():
    """A budget of one request's X and Y: partials fit nowhere but in the
    plan, and requests follow one another."""
    ws = [_split_weight(320)]
    torch.cuda.synchronize()
    srv = S.Server(hbm_budget_bytes=(4096 + 512) * 64 * 2, max_inflight=4)
    ids = [srv.register(w["plan"]) for w in ws]
    _serve(srv, _requests(ws, ids, [(0, n) for n in (64, 8, 40, 64, 3, 64, 64)]))
    assert srv.stats()["failed"] == 0
    srv.close()


def test_a_plan_under_two_ids():
    """One split plan registered twice has one workspace: requests to both
    ids, four launches in flight."""
    ws = [_split_weight(330)] * 2
    torch.cuda.synchronize()
    srv = S.Server(hbm_budget_bytes=256 << 20, max_inflight=4, max_batch=1)
    ids = [srv.register(w["plan"]) for w in ws]
    for rnd in range(4):
        _serve(srv, _requests(ws, ids, [(q % 2, 1 + (5 * q + rnd) % 64) for q in range(24)]))
    assert srv.stats()["failed"] == 0
    srv.close()
    assert ws[0]["plan"].status() == 0
