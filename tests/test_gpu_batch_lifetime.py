"""Batches of plans that came after others: a batch's launch schedule belongs
to the plans it was made for, so a plan that takes a destroyed one's address
(and number of columns) gets a schedule of its own.  Operands are
integer-valued, so Y must equal the 64-bit product rounded once.
"""
import numpy as np
import pytest

from paper_2303_16999_gb300 import spmm as S
from paper_2303_16999_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _plan(seed, m, k, n, b, d, dt=torch.float16):
    c = wl.integer_problem(seed, m, k, n, b, int((m // b) * (k // b) * d))
    vals = torch.from_numpy(c["vals"]).to(dt).cuda()
    x = torch.from_numpy(c["X"]).to(dt).cuda()
    w = torch.zeros((m // b, k // b, b, b), dtype=torch.float64, device="cuda")
    w[torch.from_numpy(c["brow"]).long(), torch.from_numpy(c["bcol"]).long()] = vals.double()
    want = (w.transpose(1, 2).reshape(m, k) @ x.double()).to(dt)
    p = S.Plan(m, k, n, b, w_dtype=S.dtype_code(dt), brow=c["brow"], bcol=c["bcol"], kernel="tc")
    p.pack(vals)
    return p, x, want


def test_batches_of_recreated_plans():
    """Sets of two plans of the same n, alternately of many and of few work
    items, each run as a batch and destroyed before the next is made."""
    n, reused, seen = 64, 0, set()
    for rnd in range(8):
        big = rnd % 2 == 0
        shapes = [(2048, 1024), (1024, 2048)] if big else [(64, 256), (48, 512)]
        made = [_plan(10 * rnd + i, m, k, n, 8, 1 / 4) for i, (m, k) in enumerate(shapes)]
        reused += sum(p.h.value in seen for p, _, _ in made)
        seen |= {p.h.value for p, _, _ in made}
        ys = [torch.full((p.m, n), float("nan"), dtype=torch.float16, device="cuda")
              for p, _, _ in made]
        for _ in range(2):
            S.spmm_batch_run([p for p, _, _ in made], [x for _, x, _ in made], ys)
        torch.cuda.synchronize()
        for (p, _, want), y in zip(made, ys):
            assert p.status() == 0 and torch.equal(y, want)
        for p, _, _ in made:
            p.close()
    assert reused > 0, "no address was used twice: the case was not reached"
