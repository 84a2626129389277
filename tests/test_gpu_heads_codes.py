"""Codes of the per-head fake-quantised step where rounding and clamping show: ties, range ends, codes too large to round by an addition."""
import math

import pytest
import torch

from paper_2605_10793_b200 import binding as B

pytestmark = pytest.mark.gpu


def _step(x, r, bits, mode, clip):
    p, n, d = x.shape
    c = B.Context(d, n, in_dtype="bf16", batch=p, quant_bits=bits, quant_mode=mode, clip_ratio=clip)
    c.set_R(r)
    signs = torch.zeros(p * n, d, dtype=torch.int8, device="cuda")
    c.debug_capture_signs(signs)
    c.step_batched(x, n, d, n * d)
    j, cnt = c.get_objective()
    assert (cnt == n).all()
    return signs.view(p, n, d), torch.from_numpy(j).cuda(), c.get_M().double()


# rows whose codes are exact (R = I, a scale that is a power of two): halves round to even, both signs, whole tiles and a remainder
@pytest.mark.parametrize("bits,mode", [(4, "sym"), (8, "sym"), (3, "sym"), (4, "zp"), (3, "zp"), (8, "zp")])
@pytest.mark.parametrize("n", [128, 300])
def test_halves_round_to_even(bits, mode, n):
    d, p = 128, 2
    top = 2 ** (bits - 1) - 1 if mode == "sym" else 2 ** bits - 1
    g = torch.Generator(device="cuda").manual_seed(bits + n)
    span = top if mode == "sym" else top / 2.0
    k = torch.randint(0, 2 * int(2 * span) + 1, (p, n, d), generator=g, device="cuda").float() / 2 - span        # multiples of a half
    k[..., 0], k[..., 1] = span, -span
    x = (k * torch.exp2(torch.randint(-3, 4, (p, n, 1), generator=g, device="cuda").float())).to(torch.bfloat16)
    keep = x.float().reshape(p, n, d)
    r = torch.eye(d, device="cuda").expand(p, d, d).contiguous()
    signs, j, m = _step(x, r, bits, mode, 1.0 if mode == "zp" else 0.0)
    y = keep.double()
    hi, lo = y.amax(-1, keepdim=True), y.amin(-1, keepdim=True)
    if mode == "sym":
        delta = torch.maximum(hi, -lo) / top
        code = torch.round(y / delta).clamp(-top, top)
    else:
        delta = (hi - lo) / top
        zeta = -torch.round(lo / delta)
        code = torch.minimum(torch.maximum(torch.round(y / delta), -zeta), top - zeta)
    assert torch.equal(signs.double(), torch.sign(code))
    rn = 1.0 / y.norm(dim=-1, keepdim=True)
    ref = (delta * code.abs() * rn).sum((1, 2)) / math.sqrt(d)
    assert ((j - ref).abs() <= 1e-6 * ref).all()                                    # (fp32 sums of a row, double beyond)
    # targets carry the row's scale in bf16 (2^-9)
    ta, size = (y.mT @ (torch.sign(code) * rn)) / math.sqrt(d), (y.abs().mT @ rn.expand_as(y)) / math.sqrt(d)
    assert ((m - ta).abs() <= 2.0 ** -8 * size).all()


def test_codes_beyond_what_an_addition_rounds():
    """A zero-point row whose range is 2^-20 of its values: codes of 2^24 and beyond, all of one sign."""
    d, p, n = 128, 2, 130
    r = torch.eye(d, device="cuda").repeat(p, 1, 1)
    r[:, 5, 0] = 2.0 ** -20
    x = torch.ones(p, n, d, device="cuda")
    x[:, ::2] = -2.0
    signs, j, _ = _step(x.to(torch.bfloat16), r.contiguous(), 4, "zp", 1.0)
    assert torch.equal(signs.float(), torch.sign(x))
    # every coordinate is quantised to within half a step of 2^-20 / 15: sum |y| / (||y|| sqrt(d)) = 1
    assert ((j - n).abs() <= 1e-5 * n).all()


# rows counted and skipped (zero, NaN) over three steps: a problem of one tile or more on one CTA, or shared out over several; more problems
# than a read's results fit in page-locked memory
@pytest.mark.parametrize("bits", [0, 4])
@pytest.mark.parametrize("problems,n", [(2, 1), (3, 200), (3, 700), (150, 300), (2100, 2)])
def test_rows_counted(problems, n, bits):
    d = 128
    g = torch.Generator(device="cuda").manual_seed(problems + n)
    x = torch.randn(problems, n, d, generator=g, device="cuda").bfloat16()
    bad = torch.zeros(problems, n, dtype=torch.bool, device="cuda")
    bad[0, 0] = bad[-1, n // 2] = bad[-1, n - 1] = True
    x[0, 0] = 0
    x[-1, n // 2] = float("nan")
    x[-1, n - 1] = 0
    c = B.Context(d, n, in_dtype="bf16", batch=problems, quant_bits=bits)
    for _ in range(3):
        c.step_batched(x, n, d, n * d)
    for _ in range(2):                                   # a second read finds the same, and the same status
        j, cnt = c.get_objective(check=False)
        assert cnt.tolist() == (3 * (n - bad.sum(dim=1))).tolist()
        if bool(x.isnan().any()):
            with pytest.raises(RuntimeError):
                c.get_objective()
    if bits == 0:                                        # <R, M> in double, M as read out (rounded to fp32 once more)
        part = c.get_R(check=False).double() * c.get_M(check=False).double()
        assert ((torch.from_numpy(j).cuda() - part.sum(dim=(1, 2))).abs() <= 2.0 ** -23 * part.abs().sum(dim=(1, 2))).all()
    assert c.get_stats().n_skipped == 3 * int(bad.sum())
