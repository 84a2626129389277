"""Row norms and the staged copy of a tensor-core step: row lengths around a warp's share, both types, odd alignments."""
import pytest
import torch

from paper_2605_10793_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [128, 384, 2176, 4096, 4224, 8192, 8320])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("offset", [0, 4])
def test_rows_that_take_no_part_and_alignment(d, dtype, offset):
    """offset 4: rows that do not start on 16-byte boundaries (bf16) or whose first one does not (fp32)."""
    n = 19
    g = torch.Generator(device="cuda")
    g.manual_seed(d + offset)
    tt = torch.float32 if dtype == "f32" else torch.bfloat16
    if dtype == "f32" and offset:
        offset = 1
    wide = torch.randn(n, d + 8, generator=g, device="cuda").to(tt)
    x = wide[:, offset:offset + d]
    x[3] = 0.0
    x[7, d - 1] = float("nan")
    x[n - 1, 0] = float("-inf")
    c = B.Context(d, n, in_dtype=dtype, mode="tc", prior_rel=0.01)
    c.step(x)
    m = c.get_M(check=False).double()
    signs = c_signs = torch.empty(n, d, dtype=torch.int8, device="cuda")
    assert B.conqur_debug_get_signs(c.h, signs.data_ptr(), n) in (0, -7)       # (the latched non-finite status)
    j, cnt = c.get_objective(check=False)
    keep = torch.ones(n, dtype=torch.bool, device="cuda")
    keep[[3, 7, n - 1]] = False
    assert cnt == n - 3 and (c_signs[~keep] == 0).all()
    xb = torch.where(keep[:, None], x.to(torch.bfloat16), torch.zeros((), dtype=torch.bfloat16, device="cuda")).double()
    # R = I: the rotated row is the row, and every decision its sign
    assert torch.equal(c_signs.double(), torch.sign(xb))
    rn = torch.where(keep, 1.0 / xb.norm(dim=1).clamp_min(1e-30), torch.zeros_like(keep, dtype=torch.float64))
    ref = xb.T @ (torch.sign(xb) * rn[:, None]) / d ** 0.5
    slack = xb.abs().T @ ((xb != 0).double() * rn[:, None]) / d ** 0.5
    # the scale enters as bf16 (2^-8); sums of n terms in fp32
    assert ((m - ref).abs() <= (2.0 ** -8 + n * 2.0 ** -23) * slack + 1e-9).all()
    jr = float((xb.abs().sum(dim=1) * rn).sum()) / d ** 0.5
    assert abs(j - jr) <= 1e-5 * jr                    # fp32 sums of squares and of d magnitudes


@pytest.mark.parametrize("d", [128, 2176, 4224, 8192])
@pytest.mark.parametrize("dtype,offset,pad", [("bf16", 0, 4), ("bf16", 4, 8), ("bf16", 2, 8), ("bf16", 1, 1), ("f32", 1, 4), ("f32", 2, 3)])
def test_rows_off_16_byte_boundaries_match_the_same_rows_on_them(d, dtype, offset, pad):
    """Some rows on 16-byte boundaries and some not (odd paddings), all of them or none: copied and normed alike."""
    n = 37
    g = torch.Generator(device="cuda")
    g.manual_seed(d + 10 * offset + pad)
    tt = torch.float32 if dtype == "f32" else torch.bfloat16
    wide = torch.randn(n, d + pad, generator=g, device="cuda").to(tt)
    x = torch.as_strided(wide, (n, d), (d + pad, 1), min(offset, pad))
    x[5] = 0.0
    out = []
    for rows in (x, x.contiguous()):
        c = B.Context(d, n, in_dtype=dtype, mode="tc", prior_rel=0.01)
        c.step(rows)
        out.append((c.get_M().double(), c.get_objective(), c.debug_get_signs(n)))
    (ma, (ja, na), sa), (mb, (jb, nb), sb) = out
    assert na == nb == n - 1 and torch.equal(sa, sb)
    xd = x.to(torch.bfloat16).double()
    rn = torch.where(xd.abs().sum(dim=1) > 0, 1.0 / xd.norm(dim=1).clamp_min(1e-30), torch.zeros((), dtype=torch.float64, device="cuda"))
    # sums of squares in another order: a scale may round to the next bf16 (2^-7 at most)
    assert ((ma - mb).abs() <= 2.0 ** -7 * (xd.abs().T @ (rn[:, None] * (xd != 0).double())) / d ** 0.5 + 1e-9).all()
    assert abs(ja - jb) <= 1e-6 * jb
