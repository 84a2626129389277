"""The calls that a calibration run, a folding pass or a serving process makes into this framework, as cases that can
be timed and compared with 64-bit arithmetic.

Kinds of case (``kind``):

  step      statistics of one streamed batch at a fixed rotation, on top of resumed statistics: ``set_M``, ``step``,
            ``get_objective``, ``get_M`` (what a token-sharded rank does around its all-reduce)
  update    the polar update of given statistics: ``set_M``, ``update``, ``get_R``
  cycle     a short calibration from a given rotation: ``set_R``, the batches, ``update``, ``get_R``
  heads     the per-head form of ``step`` (``update`` = False) or ``cycle`` (``update`` = True) on many d = 128 problems
  hadamard  the online Walsh-Hadamard rotation of activation rows
  fold      a rotation absorbed into a weight matrix

Sizes are those of ``paper_2605_10793_b200/inputs.py``, ``bench.py`` and ``bench_extra.py`` or generic; activations follow
the recipe of ``inputs.py`` (Student-t(3) values, outlier channels, a scale per token, a few massive tokens), drawn on
the GPU.  The rotation of a state is a dense orthogonal matrix, as every rotation after the first update is.
"""
from __future__ import annotations

import math

import torch

from paper_2605_10793_b200 import binding as B

_DT = {"f32": torch.float32, "bf16": torch.bfloat16}


def _case(kind, name=None, **kw):
    base = {
        "step": dict(d=4096, n=2048, mode="tc", dtype="bf16", quant_bits=0, quant_mode="sym", clip=0.0),
        "update": dict(d=4096, rows=16384, mode="tc", prior=0.0),
        "cycle": dict(d=3072, n=2048, batches=1, mode="tc", dtype="bf16", quant_bits=0, quant_mode="sym", clip=0.0, prior=0.01),
        "heads": dict(problems=1024, d=128, n=4096, dtype="bf16", interleaved=False, quant_bits=0, quant_mode="sym", clip=0.0,
                      update=True),
        "hadamard": dict(d=4096, n=32768, dtype="bf16", out="bf16", pad=0),
        "fold": dict(rows=4096, cols=14336, block=4096, side="output", mode="tc"),
    }[kind]
    out = dict(kind=kind, **base)
    out.update(kw)
    if name:
        out["name"] = name
    return out


def listed():
    return [
        # the d = 128 alternation on fp32 rows, fp32 arithmetic: the smallest calibration, bound by latency
        _case("cycle", "cycle_exact_d128", d=128, n=2048, mode="exact", dtype="f32", prior=0.0),
        # a ragged fp32 batch at a 3B-class width in fp32 arithmetic (the parity anchor, also the choice for tiny runs)
        _case("step", "step_exact_d3072_ragged", d=3072, n=1000, mode="exact", dtype="f32"),
        # one 2048-token sequence at a 7B/8B-class width, tensor cores
        _case("step", "step_tc_d4096"),
        # a ragged batch at a 70B-class width with the zero-point INT4 target of the paper's evaluation
        _case("step", "step_tc_d8192_zp4", d=8192, n=4093, quant_bits=4, quant_mode="zp", clip=0.9),
        # the update of a 7B/8B-class shared rotation from eight 2048-token sequences
        _case("update", "update_tc_d4096"),
        # a 3B-class width updated after every batch (fewer tokens than dimensions: proximal)
        _case("cycle", "cycle_tc_d3072_prior"),
        # all per-head rotations of a 32-block, 32-head model: one batch and one update
        _case("heads", "heads_1024"),
        # one block's 32 heads from the head-interleaved o_proj input, ragged, with the symmetric INT4 target
        _case("heads", "heads_block_int4", problems=32, n=4001, interleaved=True, quant_bits=4, update=False),
        # online rotation in prefill
        _case("hadamard", "hadamard_prefill"),
        # online rotation of a few fp32 rows inside a wider buffer (decode)
        _case("hadamard", "hadamard_decode", d=8192, n=33, dtype="f32", out="bf16", pad=64),
        # the down projection of an 8B-class block takes the shared rotation
        _case("fold", "fold_down"),
        # the value projection takes its per-head rotations
        _case("fold", "fold_heads", rows=4096, cols=4096, block=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step_exact", "update", "cycle", "heads", "heads", "hadamard", "hadamard", "fold"])
    quant = rng.choice([dict(), dict(), dict(quant_bits=4), dict(quant_bits=rng.choice([3, 8])),
                        dict(quant_bits=4, quant_mode="zp", clip=0.9)])
    if kind == "step":
        return _case("step", d=128 * _log_int(rng, 2, 64), n=_log_int(rng, 64, 4096), dtype=rng.choice(["bf16", "bf16", "f32"]), **quant)
    if kind == "step_exact":
        return _case("step", mode="exact", d=_log_int(rng, 2, 3072), n=_log_int(rng, 16, 2048), dtype=rng.choice(["bf16", "f32"]), **quant)
    if kind == "update":
        d = 128 * _log_int(rng, 4, 32)
        return _case("update", d=d, rows=rng.choice([4, 16, 64]) * d + rng.randrange(1000), prior=rng.choice([0.0, 0.01]))
    if kind == "cycle":
        if rng.random() < 0.4:
            d = _log_int(rng, 16, 512)
            return _case("cycle", mode="exact", dtype="f32", d=d, n=_log_int(rng, 16, 2048), prior=0.01)
        d = 128 * _log_int(rng, 2, 32)
        return _case("cycle", d=d, n=_log_int(rng, 256, 2048), batches=rng.choice([1, 2, 8]), prior=0.01, **quant)
    if kind == "heads":
        return _case("heads", problems=_log_int(rng, 2, 1024), n=_log_int(rng, 128, 4096), dtype="bf16", interleaved=rng.random() < 0.5,
                     update=rng.random() < 0.4, **quant)
    if kind == "hadamard":
        d = 1 << rng.randrange(2, 14)
        return _case("hadamard", d=d, n=max(1, _log_int(rng, 4096, 1 << 27) // d), dtype=rng.choice(["bf16", "bf16", "f32"]),
                     out=rng.choice(["bf16", "f32"]), pad=rng.choice([0, 0, 8, 20]))
    block = rng.choice([64, 128, 1024, 2048, 4096])
    side = rng.choice(["input", "output"])
    k = 1 if block >= 1024 else rng.choice([4, 20, 32])
    other = 32 * _log_int(rng, 8, 448)
    rows, cols = (other, k * block) if side == "input" else (k * block, other)
    return _case("fold", rows=rows, cols=cols, block=block, side=side, mode=rng.choice(["tc", "exact"]))


# ---- inputs -------------------------------------------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1009 + 17)
    return g


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32)


def _student_t3(g, *shape):
    c = _randn(g, *shape).square_()
    c += _randn(g, *shape).square_()
    c += _randn(g, *shape).square_()
    c *= 1.0 / 3.0
    return _randn(g, *shape).mul_(c.rsqrt_())


def _activations(g, n, d, massive=4, outliers=None, scale=100.0):
    """n rows of the residual-stream recipe, fp32."""
    x = _student_t3(g, n, d)
    ch = torch.randperm(d, generator=g, device="cuda")[: (max(1, d // 256) if outliers is None else outliers)]
    x[:, ch] *= scale
    x *= torch.exp(0.5 * _randn(g, n, 1))
    if massive and n > massive:
        rows = torch.randperm(n, generator=g, device="cuda")[:massive]
        dims = torch.randperm(d, generator=g, device="cuda")[: min(4, d)]
        x[rows[:, None], dims[None, :]] *= 1000.0
    return x


def _rotation(g, d):
    q, r = torch.linalg.qr(_randn(g, d, d))
    q = q * torch.sign(torch.diagonal(r))[None, :]
    return q.contiguous()


def _head_rotations(g, problems, d):
    q, r = torch.linalg.qr(_randn(g, problems, d, d))
    return (q * torch.sign(torch.diagonal(r, dim1=1, dim2=2))[:, None, :]).contiguous()


def _head_rows(case, g):
    """(n, P, d) if interleaved, else (P, n, d), in the storage type; the per-head recipe."""
    p, n, d = case["problems"], case["n"], case["d"]
    x = torch.empty((n, p, d) if case["interleaved"] else (p, n, d), dtype=_DT[case["dtype"]], device="cuda")
    v = x.transpose(0, 1) if case["interleaved"] else x
    step = max(1, (1 << 26) // (n * d))
    for a in range(0, p, step):
        b = min(p, a + step)
        t = _student_t3(g, b - a, n, d)
        ch = torch.rand(b - a, d, generator=g, device="cuda").argsort(dim=1)[:, :2]
        t.mul_(torch.ones(b - a, d, device="cuda").scatter_(1, ch, 30.0)[:, None, :])
        t.mul_(torch.exp(0.5 * _randn(g, b - a, n, 1)))
        v[a:b] = t.to(x.dtype)
    return x


def _statistics(g, d, rows):
    """The cross-covariance of `rows` rows at a dense rotation, with that rotation."""
    r = _rotation(g, d)
    m = torch.zeros(d, d, device="cuda")
    for a in range(0, rows, 16384):
        x = _activations(g, min(16384, rows - a), d)
        x /= x.norm(dim=1, keepdim=True)
        m += x.T @ torch.sign(x @ r)
    return r, m / math.sqrt(d)


def prepare(case, seed):
    g = _gen(seed)
    k = case["kind"]
    s = {"case": case}
    if k in ("step", "cycle"):
        d, n, nb = case["d"], case["n"], case.get("batches", 1)
        s["x"] = [_activations(g, n, d).to(_DT[case["dtype"]]) for _ in range(nb)]
        s["r"] = _rotation(g, d)
        s["ctx"] = B.Context(d, n, in_dtype=case["dtype"], mode=case["mode"], quant_bits=case["quant_bits"],
                             quant_mode=case["quant_mode"], clip_ratio=case["clip"], prior_rel=case.get("prior", 0.0),
                             defer_batches=nb if nb > 1 else 0)
        if k == "step":
            s["ctx"].set_R(s["r"])
            s["m"] = torch.zeros(d, d, device="cuda")
    elif k == "update":
        d = case["d"]
        s["r"], s["m"] = _statistics(g, d, case["rows"])
        s["ctx"] = B.Context(d, 2048, mode=case["mode"], prior_rel=case["prior"])
        if case["prior"] == 0:
            s["ctx"].set_R(s["r"])
    elif k == "heads":
        p, d, n = case["problems"], case["d"], case["n"]
        s["x"] = _head_rows(case, g)
        s["r"] = _head_rotations(g, p, d)
        s["ctx"] = B.Context(d, n, in_dtype=case["dtype"], batch=p, quant_bits=case["quant_bits"], quant_mode=case["quant_mode"],
                             clip_ratio=case["clip"], prior_rel=0.01 if case["update"] else 0.0)
        if not case["update"]:
            s["ctx"].set_R(s["r"])
            s["m"] = torch.zeros(p, d, d, device="cuda")
    elif k == "hadamard":
        n, d, pad = case["n"], case["d"], case["pad"]
        x = torch.empty(n, d + pad, dtype=_DT[case["dtype"]], device="cuda")
        step = max(1, (1 << 26) // (d + pad))
        for a in range(0, n, step):
            x[a:a + step] = _student_t3(g, min(step, n - a), d + pad).to(x.dtype)
        s["x"] = x[:, :d]
        s["y"] = torch.empty(n, d + pad, dtype=_DT[case["out"]], device="cuda")[:, :d]
    else:
        rows, cols, block = case["rows"], case["cols"], case["block"]
        s["w"] = _randn(g, rows, cols) / math.sqrt(cols)
        k_blocks = (cols if case["side"] == "input" else rows) // block
        s["r"] = _rotation(g, block) if k_blocks == 1 else _head_rotations(g, k_blocks, block)
    return s


# ---- one pass -----------------------------------------------------------------------------------------------------


def run(s):
    case = s["case"]
    k = case["kind"]
    if k == "step":
        c = s["ctx"]
        c.set_M(s["m"], 0.0, 0)
        for x in s["x"]:
            c.step(x)
        j, n = c.get_objective()
        return {"J": j, "M": c.get_M(), "N": n}
    if k == "update":
        c = s["ctx"]
        if case["prior"] > 0:
            c.set_R(s["r"])
        c.set_M(s["m"], 0.0, case["rows"])
        c.update()
        return c.get_R()
    if k == "cycle":
        c = s["ctx"]
        c.set_R(s["r"])
        for x in s["x"]:
            c.step(x)
        j, n = c.get_objective()
        c.update()
        return {"J": j, "N": n, "R": c.get_R()}
    if k == "heads":
        c, p, d, n = s["ctx"], case["problems"], case["d"], case["n"]
        if case["update"]:
            c.set_R(s["r"])
        else:
            c.set_M(s["m"], [0.0] * p, [0] * p)
        if case["interleaved"]:
            c.step_batched(s["x"], n, p * d, d)
        else:
            c.step_batched(s["x"], n, d, n * d)
        j, cnt = c.get_objective()
        if case["update"]:
            c.update()
            return {"J": j, "N": cnt, "R": c.get_R()}
        return {"J": j, "M": c.get_M(), "N": cnt}
    if k == "hadamard":
        return B.conqur_hadamard_rows(s["x"], out=s["y"])
    return B.conqur_fold_weight(s["w"], s["r"], case["side"], case["mode"])


# ---- what a pass cannot do without --------------------------------------------------------------------------------

# The polar factor by odd polynomials: about ten steps, each two symmetric products (d^3 flops) and a full one (2 d^3).
_POLAR_FLOPS = 40.0


def work(case):
    k = case["kind"]
    size = {"f32": 4, "bf16": 2}
    if k in ("step", "cycle", "heads"):
        d, p = case["d"], case.get("problems", 1)
        rows = case["n"] * case.get("batches", 1) * p
        flops, nbytes = 4.0 * rows * d * d, rows * d * size[case["dtype"]] + 8.0 * p * d * d
        if k == "cycle" or (k == "heads" and case["update"]):
            flops += _POLAR_FLOPS * p * d ** 3
        else:
            nbytes += 4.0 * p * d * d                       # the resumed statistics
        return {"bytes": nbytes, "flops": flops}
    if k == "update":
        return {"bytes": 8.0 * case["d"] ** 2, "flops": _POLAR_FLOPS * case["d"] ** 3}
    if k == "hadamard":
        n, d = case["n"], case["d"]
        return {"bytes": float(n * d * (size[case["dtype"]] + size[case["out"]])), "flops": n * d * math.log2(d)}
    rows, cols, block = case["rows"], case["cols"], case["block"]
    nblk = (cols if case["side"] == "input" else rows) // block
    return {"bytes": 8.0 * rows * cols + 4.0 * nblk * block * block, "flops": 2.0 * rows * cols * block}


def tolerance(case):
    k = case["kind"]
    # One sign that falls the other way (a rotated coordinate within rounding of zero) moves a single entry of M by far more
    # than rounding does, and with it the rotation: hence the wide "max".  Measured against 64 bits: fp32 arithmetic M 5e-7
    # (7e-5 with one flipped sign in ten million), R 1.3e-6; bf16 operands M 1e-3 .. 5e-3 (few rows: 1.4e-2), R 5e-3 from
    # given statistics and 1e-2 .. 4e-2 from rows; a repeated update of the same statistics differs from the first by 5e-3.
    if k in ("step", "cycle") and case["mode"] == "exact":
        return {"rel": 3e-4 if k == "step" else 1e-3, "max": 0.5}
    if k == "update":
        return {"rel": 0.02, "max": 0.3}
    if k in ("step", "cycle", "heads"):
        return {"rel": 0.02 if k == "step" else 0.03, "max": 0.99}
    if k == "hadamard":
        return {"rel": 1e-2 if case["out"] == "bf16" else 2e-6, "max": 1e-2 if case["out"] == "bf16" else 1e-4}
    return {"rel": 4e-5 if case["mode"] == "tc" else 5e-6}


# ---- the same in 64 bits, plain torch -----------------------------------------------------------------------------


def _polar64(m):
    """Polar factor by Newton's iteration with norm scaling; m: (..., d, d) float64."""
    x = m / m.flatten(-2).norm(dim=-1)[..., None, None]
    for it in range(60):
        y = torch.linalg.inv(x).mT
        g = torch.ones_like(x[..., :1, :1])
        if it < 16:
            g = (y.flatten(-2).norm(dim=-1) / x.flatten(-2).norm(dim=-1)).sqrt()[..., None, None]
        new = 0.5 * (g * x + y / g)
        delta = ((new - x).flatten(-2).norm(dim=-1) / math.sqrt(x.shape[-1])).max().item()
        x = new
        if it >= 3 and delta < 1e-12:
            break
    return x


def _targets64(y, case):
    """(signs, objective terms) of rotated normalised rows, fake-quantised first where the case says so."""
    b = case["quant_bits"]
    if not b:
        return torch.sign(y), y.abs()
    if case["quant_mode"] == "sym":
        lev = 2 ** (b - 1) - 1
        delta = y.abs().amax(dim=-1, keepdim=True) / lev
        k = torch.round(y / delta).clamp_(-lev, lev)
    else:
        lev = 2 ** b - 1
        lo, hi = case["clip"] * y.amin(dim=-1, keepdim=True), case["clip"] * y.amax(dim=-1, keepdim=True)
        delta = (hi - lo) / lev
        zeta = -torch.round(lo / delta)
        k = torch.minimum(torch.maximum(torch.round(y / delta), -zeta), lev - zeta)
    return torch.sign(k), delta * k.abs()


def _step64(x, r, case):
    """(J, M, N) of rows x (..., n, d) in float64."""
    x = x.double()
    x = x / x.norm(dim=-1, keepdim=True)
    s, o = _targets64(x @ r, case)
    root = math.sqrt(x.shape[-1])
    return o.sum(dim=(-2, -1)) / root, x.mT @ s / root, x.shape[-2]


def exact(case, seed):
    s = prepare(case, seed)
    s.pop("ctx", None)
    k = case["kind"]
    if k in ("step", "cycle"):
        r = s["r"].double()
        j, m, n = 0.0, 0.0, 0
        for x in s["x"]:
            j1, m1, n1 = _step64(x, r, case)
            j, m, n = j + float(j1), m + m1, n + n1
        if k == "step":
            return {"J": j, "M": m, "N": n}
        return {"J": j, "N": n, "R": _proximal64(m, r, case["prior"])}
    if k == "update":
        return _proximal64(s["m"].double(), s["r"].double(), case["prior"])
    if k == "heads":
        p, n = case["problems"], case["n"]
        x = s["x"].transpose(0, 1) if case["interleaved"] else s["x"]
        js, out = [], []
        for a in range(0, p, 128):
            r = s["r"][a:a + 128].double()
            j, m, _ = _step64(x[a:a + 128], r, case)
            js.append(j)
            out.append(_proximal64(m, r, 0.01) if case["update"] else m)
        j = torch.cat(js).cpu().numpy()
        cnt = torch.full((p,), n, dtype=torch.int64).numpy()
        return {"J": j, "N": cnt, "R" if case["update"] else "M": torch.cat(out)}
    if k == "hadamard":
        y = s["x"].double()
        n, d = y.shape
        h = 1
        while h < d:
            v = y.view(n, d // (2 * h), 2, h)
            y = torch.stack((v[:, :, 0] + v[:, :, 1], v[:, :, 0] - v[:, :, 1]), dim=2).reshape(n, d)
            h *= 2
        return y / math.sqrt(d)
    w, r = s["w"].double(), s["r"].double()
    rows, cols, block = case["rows"], case["cols"], case["block"]
    if r.dim() == 2:
        return w @ r if case["side"] == "input" else r.T @ w
    if case["side"] == "input":
        return torch.einsum("akb,kbc->akc", w.view(rows, cols // block, block), r).reshape(rows, cols)
    return torch.einsum("kba,kbc->kac", r, w.view(rows // block, block, cols)).reshape(rows, cols)


def _proximal64(m, r, prior):
    if prior > 0:
        lam = prior * m.flatten(-2).norm(dim=-1)[..., None, None] / math.sqrt(m.shape[-1])
        m = m + lam * r
    return _polar64(m)
