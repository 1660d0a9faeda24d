"""Workloads of the block-sparse products, as a program that uses the library has them run.

Each case is one pass through the public entry points of
``paper_2303_16999_gb300.spmm``: a product on a static plan, a training step
of a sparse layer, a dynamic call, a batch of products, or a burst of served
requests.  Sizes are those of the library's own workloads (the 4096 x 4096
sweep, the 16384 x 16384 element-sparse gather, the 8192 x 8192 dynamic call,
the FFN-like 4096 x 16384 batch, the served 2048 to 8192 weights) and ragged
ones between them.
"""
import math
import random

import torch

from paper_2303_16999_gb300 import spmm as S

DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
DEV = "cuda"
# a batch's weights stay loaded for the life of the program: the library keeps
# the launch schedule of a set of plans from their first batched call on
_RESIDENT = []


def listed():
    return [
        # the smallest layer: one FP32 product of a 256 x 256 weight, bound by
        # the call itself
        dict(name="f32_small", kind="static", m=256, k=256, n=64, b=4, d=1 / 8, w="f32", x="f32"),
        # an FP32 layer on a ragged batch of columns
        dict(name="f32_layer", kind="static", m=2048, k=4096, n=500, b=8, d=1 / 8, w="f32",
             x="f32"),
        # the static sweep's native block size, FP16: forward over a prompt
        dict(name="b16_n2048", kind="static", m=4096, k=4096, n=2048, b=16, d=1 / 16, w="f16",
             x="f16"),
        # the sweep's element-sparse weight over the same prompt (16 x 16
        # tiles all occupied)
        dict(name="b1_n2048", kind="static", m=4096, k=4096, n=2048, b=1, d=1 / 8, w="f16",
             x="f16"),
        # small blocks, BF16, a number of columns that no tile divides
        dict(name="b4_n1000", kind="static", m=4096, k=4096, n=1000, b=4, d=1 / 8, w="bf16",
             x="bf16"),
        # an FFN weight over a short chunk of columns
        dict(name="ffn_n200", kind="static", m=4096, k=16384, n=200, b=8, d=1 / 8, w="bf16",
             x="bf16"),
        # decoding one token with an element-sparse weight: indices and
        # values streamed once
        dict(name="b1_n1", kind="static", m=16384, k=16384, n=1, b=1, d=1 / 16, w="f16", x="f16"),
        # decoding 32 sequences at once with an element-sparse weight
        dict(name="b1_n32", kind="static", m=8192, k=8192, n=32, b=1, d=1 / 16, w="f16", x="f16"),
        # one training step of a sparse layer: forward and dX with this step's
        # values, and the weight gradient on the mask
        dict(name="train_b8", kind="train", m=4096, k=4096, n=2048, b=8, d=1 / 16, w="bf16",
             x="bf16"),
        # a dynamic call: pattern and values arrive on the device
        dict(name="dynamic_b16", kind="dynamic", m=8192, k=8192, n=1024, b=16, d=1 / 16,
             fill=0.75, layout="coo", w="bf16", x="bf16"),
        # uneven FFN-like E4M3 products in one batched call
        dict(name="batch_e4m3", kind="batch", count=12, m=4096, k=16384, n_max=512, mix=3,
             w="e4m3", x="bf16"),
        # a burst of requests to a server that holds six weights
        dict(name="serve_burst", kind="serve", m_max=8192, requests=32, n_max=256, mix=4,
             w="f16", x="f16"),
    ]


def _log(rng, lo, hi, step=1):
    """Log-uniform in [lo, hi], a multiple of step."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return int(min(hi // step * step, max(step, round(v / step) * step)))


def draw(rng):
    kind = rng.choice(["static", "static", "static", "gather", "f32", "train", "dynamic", "batch",
                       "serve"])
    d = rng.choice([1 / 32, 1 / 16, 1 / 8, 1 / 4])
    x = rng.choice(["f16", "bf16"])
    if kind == "static":
        # a prompt, a chunk or a few columns against a layer or an FFN weight
        return dict(kind="static", m=_log(rng, 256, 8192, 16), k=_log(rng, 256, 8192, 16),
                    n=_log(rng, 1, 2048), b=rng.choice([4, 8, 16]), d=d,
                    w=rng.choice([x, x, "e4m3"]), x=x)
    if kind == "gather":
        x = rng.choice(["f16", "bf16", "f32"])
        return dict(kind="static", m=_log(rng, 256, 8192), k=_log(rng, 256, 8192),
                    n=_log(rng, 1, 256), b=1, d=d, w=x, x=x)
    if kind == "f32":
        b = rng.choice([4, 8, 16])
        return dict(kind="static", m=_log(rng, 256, 4096, b), k=_log(rng, 256, 4096, b),
                    n=_log(rng, 1, 1024), b=b, d=d, w="f32", x="f32")
    if kind == "train":
        return dict(kind="train", m=_log(rng, 256, 4096, 16), k=_log(rng, 256, 4096, 16),
                    n=_log(rng, 16, 2048, 8), b=rng.choice([4, 8, 16]), d=d, w=x, x=x)
    if kind == "dynamic":
        b = rng.choice([1, 4, 8, 16, 16])
        return dict(kind="dynamic", m=_log(rng, 256, 8192 if b > 4 else 2048, 16),
                    k=_log(rng, 256, 8192 if b > 4 else 2048, 16), n=_log(rng, 16, 1024, 8), b=b,
                    d=rng.choice([1 / 32, 1 / 16]), fill=round(rng.uniform(0.5, 1.0), 3),
                    layout=rng.choice(["coo", "ell"]) if b == 16 else "coo", w=x, x=x)
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(4, 12), m=_log(rng, 512, 4096, 16),
                    k=_log(rng, 1024, 16384, 16), n_max=rng.choice([128, 256, 512]),
                    mix=rng.randint(0, 999), w=rng.choice(["e4m3", x]), x=x)
    return dict(kind="serve", m_max=rng.choice([2048, 4096, 8192]), requests=rng.randint(8, 32),
                n_max=rng.choice([64, 128, 256]), mix=rng.randint(0, 999), w=x, x=x)


# ------------------------------------------------------------------ problems
def _problems(case):
    """The weights of a case: (m, k, b, d) each; with the products or requests
    made of them, (weight, n) each."""
    if case["kind"] == "batch":
        # W m x k and k x m in turn, b in {8, 16}, d in {1/16, 1/8}, n
        # log-uniform; every n another one
        rng = random.Random(case["mix"])
        ws, calls, seen = [], [], set()
        for i in range(case["count"]):
            m, k = (case["m"], case["k"]) if i % 2 == 0 else (case["k"], case["m"])
            n = _log(rng, 1, case["n_max"])
            while n in seen:
                n = n + 1 if n < case["n_max"] else 1
            seen.add(n)
            ws.append((m, k, (8, 16)[(i >> 1) & 1], (1 / 16, 1 / 8)[(i >> 2) & 1]))
            calls.append((i, n))
        return ws, calls
    if case["kind"] == "serve":
        rng = random.Random(case["mix"])
        ws = [(m, m, b, 1 / 16) for m in (2048, 4096, 8192) if m <= case["m_max"]
              for b in (8, 16)]
        return ws, [(rng.randrange(len(ws)), _log(rng, 1, case["n_max"]))
                    for _ in range(case["requests"])]
    return [(case["m"], case["k"], case["b"], case["d"])], [(0, case["n"])]


def _nnzb(m, k, b, d):
    return max(1, round(d * (m // b) * (k // b)))


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _pattern(g, m, k, b, nnzb):
    """nnzb distinct blocks, uniform over the grid (in random order; by rows
    for element-sparse weights, as a mask's non-zeros come)."""
    mb, kb = m // b, k // b
    if b == 1 and mb * kb > 1 << 22:
        # the mask is drawn element by element, so the count is d * m * k on
        # average
        rows, cols = (torch.rand((mb, kb), generator=g, device=DEV) < nnzb / (mb * kb)).nonzero(
            as_tuple=True)
        return rows.int(), cols.int()
    idx = torch.randperm(mb * kb, generator=g, device=DEV)[:nnzb]
    if b == 1:
        idx = idx.sort().values
    return (idx // kb).int(), (idx % kb).int()


def _weight(g, case, m, k, b, nnzb):
    """Pattern, values and (E4M3) one scale per block, max|w| / 448."""
    brow, bcol = _pattern(g, m, k, b, nnzb)
    v = torch.randn((brow.numel(), b, b), generator=g, device=DEV)
    if case["w"] != "e4m3":
        return brow, bcol, v.to(DTYPES[case["w"]]), None
    scale = v.abs().amax(dim=(1, 2)).clamp_min(1e-30) / 448
    return brow, bcol, (v / scale[:, None, None]).to(torch.float8_e4m3fn), scale


def _dense(g, rows, n, dt):
    """rows x n values N(0, 1), rows padded to a multiple of 8 values."""
    x = torch.zeros((rows, (n + 7) // 8 * 8), dtype=DTYPES[dt], device=DEV)
    x[:, :n] = torch.randn((rows, n), generator=g, device=DEV)
    return x[:, :n]


def _inputs(case, seed):
    """Everything a pass reads: the weights, then the dense operands."""
    g = _gen(seed)
    ws, calls = _problems(case)
    weights = []
    for m, k, b, d in ws:
        nnzb = _nnzb(m, k, b, d)
        if case["kind"] == "dynamic":
            nnzb = max(1, int(nnzb * case["fill"]))
        weights.append(_weight(g, case, m, k, b, nnzb))
    xs = [_dense(g, ws[w][1], n, case["x"]) for w, n in calls]
    dy = _dense(g, case["m"], case["n"], case["x"]) if case["kind"] == "train" else None
    return ws, calls, weights, xs, dy


def _code(name):
    return S.E4M3 if name == "e4m3" else S.dtype_code(DTYPES[name])


def _plan(case, shape, weight, n_max, **kw):
    m, k, b, _ = shape
    return S.Plan(m, k, n_max, b, w_dtype=_code(case["w"]), x_dtype=_code(case["x"]),
                  brow=weight[0].cpu().numpy(), bcol=weight[1].cpu().numpy(), **kw)


def _ell(brow, bcol, vals, mb):
    """Blocked-ELL layout of the blocks: columns ascending, -1 padding."""
    order = torch.argsort(brow.long() * (1 << 31) + bcol.long())
    r, c, v = brow[order].long(), bcol[order], vals[order]
    counts = torch.bincount(r, minlength=mb)
    slot = torch.arange(r.numel(), device=DEV) - (counts.cumsum(0) - counts)[r]
    width = int(counts.max())
    cols = torch.full((mb, width), -1, dtype=torch.int32, device=DEV)
    cols[r, slot] = c
    blocks = torch.zeros((mb, width) + v.shape[1:], dtype=v.dtype, device=DEV)
    blocks[r, slot] = v
    return cols, blocks


# ------------------------------------------------------------------- a pass
def prepare(case, seed):
    ws, calls, weights, xs, dy = _inputs(case, seed)
    kind = case["kind"]
    st = dict(kind=kind, xs=xs)
    if kind == "static":
        plan = _plan(case, ws[0], weights[0], case["n"])
        plan.pack(weights[0][2], weights[0][3])
        st.update(plan=plan)
    elif kind == "train":
        st.update(fwd=_plan(case, ws[0], weights[0], case["n"]),
                  bwd=_plan(case, ws[0], weights[0], case["n"], transposed=True),
                  vals=weights[0][2], dy=dy)
    elif kind == "dynamic":
        m, k, b, d = ws[0]
        brow, bcol, vals, _ = weights[0]
        cap = max(_nnzb(m, k, b, d), brow.numel())
        plan = S.Plan(m, k, case["n"], b, w_dtype=_code(case["w"]), mode=S.DYNAMIC, nnzb_max=cap)
        st.update(plan=plan)
        if case["layout"] == "ell":
            st.update(ell=_ell(brow, bcol, vals, m // b))
        else:
            pad = cap - brow.numel()
            grow = torch.nn.functional.pad
            st.update(pattern=(torch.tensor([brow.numel()], dtype=torch.int32, device=DEV),
                               grow(brow, (0, pad)), grow(bcol, (0, pad))),
                      vals=grow(vals, (0, 0, 0, 0, 0, pad)))
    elif kind == "batch":
        plans = []
        for (w, n), weight in zip(calls, weights):
            plans.append(_plan(case, ws[w], weight, n))
            plans[-1].pack(weight[2], weight[3])
        _RESIDENT.extend(plans)
        st.update(plans=plans, ys=[torch.empty((p.m, n), dtype=x.dtype, device=DEV)
                                   for p, (_, n), x in zip(plans, calls, xs)])
    else:
        plans = []
        for shape, weight in zip(ws, weights):
            plans.append(_plan(case, shape, weight, case["n_max"]))
            plans[-1].pack(weight[2], weight[3])
        server = S.Server(hbm_budget_bytes=256 << 20, max_inflight=4, max_batch=16)
        ids = [server.register(p) for p in plans]
        hx = [x.contiguous().cpu().pin_memory() for x in xs]
        hy = [torch.empty((ws[w][0], n), dtype=xs[0].dtype).pin_memory() for w, n in calls]
        st.update(server=server, requests=[(ids[w], x, y) for (w, _), x, y in zip(calls, hx, hy)],
                  xs=None)
    torch.cuda.synchronize()
    return st


def run(st):
    kind = st["kind"]
    if kind == "static":
        return st["plan"].run(st["xs"][0])
    if kind == "train":
        x = st["xs"][0]
        y = st["fwd"].run(x, values=st["vals"])
        dx = st["bwd"].run(st["dy"], values=st["vals"])
        return y, dx, st["fwd"].sddmm(st["dy"], x)
    if kind == "dynamic":
        if "ell" in st:
            return st["plan"].run_ell(*st["ell"], st["xs"][0])
        return st["plan"].run(st["xs"][0], values=st["vals"], pattern=st["pattern"])
    if kind == "batch":
        S.spmm_batch_run(st["plans"], st["xs"], st["ys"])
        return st["ys"]
    tickets = [st["server"].submit(w, x, y) for w, x, y in st["requests"]]
    for t in tickets:
        st["server"].wait(t)
    return [y for _, _, y in st["requests"]]


def work(case):
    """Non-zero FLOPs; values, indices and dense operands each once (16-bit
    block columns wherever a column fits them, as a plan may hold them)."""
    ws, calls = _problems(case)
    xb = 4 if case["x"] == "f32" else 2
    wb = {"f32": 4, "e4m3": 1}.get(case["w"], 2)
    nbytes = flops = 0
    for i in sorted({w for w, _ in calls}):
        m, k, b, d = ws[i]
        nnzb = _nnzb(m, k, b, d)
        ib = 2 + 4 * (m // b) / nnzb
        if case["kind"] == "dynamic":
            nnzb, ib = max(1, int(nnzb * case["fill"])), 8
        nbytes += nnzb * (b * b * wb + ib + (4 if case["w"] == "e4m3" else 0))
    for w, n in calls:
        m, k, b, d = ws[w]
        nnzb = _nnzb(m, k, b, d)
        if case["kind"] == "dynamic":
            nnzb = max(1, int(nnzb * case["fill"]))
        one = 2 * nnzb * b * b * n
        if case["kind"] == "train":
            # X, dY in; Y, dX, and dW (FP32) out; three products
            nbytes += 2 * (m + k) * n * xb + nnzb * b * b * 4
            flops += 3 * one
        else:
            nbytes += (m + k) * n * xb
            flops += one
    return dict(bytes=int(nbytes), flops=int(flops))


# ------------------------------------------------------------------- 64 bits
def _to_dense(shape, weight):
    """The m x k weight in 64 bits."""
    m, k, b, _ = shape
    brow, bcol, vals, scale = weight
    v = vals.to(torch.float32).double()
    if scale is not None:
        v = v * scale.double()[:, None, None]
    w = torch.zeros((m // b, k // b, b, b), dtype=torch.float64, device=DEV)
    w[brow.long(), bcol.long()] = v
    return w.transpose(1, 2).reshape(m, k)


def exact(case, seed):
    ws, calls, weights, xs, dy = _inputs(case, seed)
    if case["kind"] == "train":
        m, k, b, _ = ws[0]
        w, x, g = _to_dense(ws[0], weights[0]), xs[0].double(), dy.double()
        full = (g @ x.t()).reshape(m // b, b, k // b, b).transpose(1, 2)
        return w @ x, w.t() @ g, full[weights[0][0].long(), weights[0][1].long()]
    outs = [None] * len(calls)
    for i, weight in enumerate(weights):
        dense = _to_dense(ws[i], weight)
        for j, (w, _) in enumerate(calls):
            if w == i:
                y = dense @ xs[j].double()
                outs[j] = y.cpu() if case["kind"] == "serve" else y
    return outs if case["kind"] in ("batch", "serve") else outs[0]
