"""The per-head step without fake-quantisation (tensor cores, d = 128): edges of its 256-row double tiles, layouts, token
splits, many short problems per thread block, rows that take no part."""
import pytest
import torch

from paper_2605_10793_b200 import binding as B

pytestmark = pytest.mark.gpu
D = 128


def _setup(P, n, interleaved, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.randn(P, n, D, generator=g, device="cuda") * torch.exp(torch.randn(P, n, 1, generator=g, device="cuda"))
    x = x.to(torch.bfloat16)
    r = torch.linalg.qr(torch.randn(P, D, D, generator=g, device="cuda"))[0].contiguous()
    return x, r, (x.transpose(0, 1).contiguous() if interleaved else x)


@pytest.mark.parametrize("P,n,interleaved", [
    (2, 1, False), (2, 127, True), (3, 128, False), (2, 129, True), (5, 255, False), (4, 256, True), (3, 257, False),
    (2, 1000, True), (7, 511, False), (33, 513, True), (150, 300, False), (700, 40, False), (460, 257, True), (300, 640, False)])
def test_statistics_against_fp64(P, n, interleaved):
    x, r, xin = _setup(P, n, interleaved, 7 * P + n)
    xv = xin.transpose(0, 1) if interleaved else xin               # (P, n, D) view of what the kernel reads
    bad = []
    if n >= 3:                                                     # zero row, NaN, Inf in different problems
        xv[0, 0] = 0.0
        xv[P // 2, n // 2, 5] = float("nan")
        xv[P - 1, n - 1, 127] = float("inf")
        bad = [(0, 0), (P // 2, n // 2), (P - 1, n - 1)]
    c = B.Context(D, n, batch=P)
    c.set_R(r)
    signs = torch.full((P * n, D), 9, dtype=torch.int8, device="cuda")
    c.debug_capture_signs(signs)
    for rep in range(2):                                           # the second step adds to what the first one left
        c.step_batched(xin, n, *((P * D, D) if interleaved else (D, n * D)))
    m = c.get_M(check=False).double()
    j, cnt = c.get_objective(check=False)
    s = signs.view(P, n, D).double()
    keep = torch.ones(P, n, dtype=torch.bool, device="cuda")
    for p, i in bad:
        keep[p, i] = False
    assert (s[~keep] == 0).all() and (signs.abs() <= 1).all()
    xd = torch.where(keep[..., None], xv, torch.zeros((), dtype=xv.dtype, device="cuda")).double()
    norm = xd.norm(dim=-1, keepdim=True).clamp_min(1e-300)
    y = xd @ r.to(torch.bfloat16).double()
    # decisions: wrong only within fp32 accumulation of zero (128 products of exact bf16 operands)
    size = xd.abs() @ r.to(torch.bfloat16).double().abs()
    assert ((torch.sign(y) == s) | (y.abs() <= 128 * 2.0 ** -23 * size)).all()
    # M: the scale enters as bf16 (8 significant bits: rounding up to 2^-8), everything else in fp32
    rn = torch.where(keep[..., None], 1.0 / norm, torch.zeros_like(norm))
    ref = 2 * (xd.mT @ (s * rn)) / D ** 0.5
    slack = 2 * (xd.abs().mT @ (s.abs() * rn)) / D ** 0.5
    assert ((m - ref).abs() <= (2.0 ** -8 + 2 * n * 2.0 ** -23 + 2.0 ** -12) * slack + 1e-7).all()
    jd = torch.from_numpy(j).cuda()
    assert torch.equal(torch.from_numpy(cnt).cuda(), 2 * keep.sum(dim=1))
    assert ((jd - (r.double() * m).sum(dim=(1, 2))).abs() <= 1e-5 * (r.double() * m).abs().sum(dim=(1, 2)) + 1e-9).all()


def test_reruns_are_bit_identical_and_quantised_neighbours_unaffected():
    P, n = 20, 900
    x, r, xin = _setup(P, n, True, 3)
    out = []
    for _ in range(2):
        c = B.Context(D, n, batch=P)
        c.set_R(r)
        c.step_batched(xin, n, P * D, D)
        c.step_batched_range(xin[:, 4:9], 300, P * D, D, 4, 5)
        out.append(c.get_M())
    assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("P,n", [(700, 100), (310, 129), (301, 385)])
def test_short_quantised_problems(P, n):
    """Several short problems per thread block in the fake-quantised kernel: each accumulator is its own problem's."""
    x, r, xin = _setup(P, n, False, P + n)
    c = B.Context(D, n, batch=P, quant_bits=4)
    c.set_R(r)
    signs = torch.zeros((P * n, D), dtype=torch.int8, device="cuda")
    c.debug_capture_signs(signs)
    c.step_batched(xin, n, D, n * D)
    m = c.get_M().double()
    xd = xin.double()
    s = signs.view(P, n, D).double()
    rn = 1.0 / xd.norm(dim=-1, keepdim=True)
    ref = (xd.mT @ (s * rn)) / D ** 0.5
    slack = (xd.abs().mT @ (s.abs() * rn)) / D ** 0.5
    assert ((m - ref).abs() <= (2.0 ** -8 + n * 2.0 ** -23) * slack + 1e-7).all()
