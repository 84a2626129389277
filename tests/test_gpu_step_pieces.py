"""Exact steps whose products run on the tensor cores over bf16 pieces: signs, statistics and objective against float64."""
import math

import pytest
import torch

from paper_2605_10793_b200 import binding as B

pytestmark = pytest.mark.gpu


def _rand(seed, *shape):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(*shape, generator=g, device="cuda")


def _rows(seed, n, d, dtype):
    """Heavy-tailed rows with outlier channels and tokens, a zero row, and rows that are not finite."""
    x = _rand(seed, n, d) * torch.exp(1.5 * _rand(seed + 1, n, d)) * torch.exp(8.0 * _rand(seed + 2, n, 1))
    x[:, ::97] *= 300.0
    x[n // 2] = 0.0
    x[n // 3, d // 2] = float("nan")
    x[0, 0] = float("-inf")
    return x.to(dtype)


# sums of K terms, 64 at a time: at most 24 + 4 instructions' cuts of 16 2^-25 + 2^-23 of the terms' sizes, of which all but four
# act on sums 2^-7 smaller, the pieces' remainder (2^-25), then K / 64 fp32 additions of 2^-24
def _unit(k):
    return (4 * 10 + 4 + k / 64 + 1) * 2.0 ** -24


# edges of the 128 / 192 / 256 wide tiles, of 64-long k blocks and of 256-row tiles; odd widths; one row of tiles and many
SHAPES = [(512, 512), (513, 600), (575, 577), (640, 511), (767, 1025), (769, 513), (1001, 900), (1027, 129), (1536, 1280), (2050, 2049)]


@pytest.mark.parametrize("d,n", SHAPES)
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_signs_statistics_and_objective(d, n, dtype):
    x = _rows(d + n, n, d, dtype)
    r = torch.linalg.qr(_rand(7, d, d).double())[0].float().contiguous()
    c = B.Context(d, n, in_dtype="f32" if dtype == torch.float32 else "bf16", mode="exact")
    c.set_R(r)
    c.step(x)
    j, cnt = c.get_objective(check=False)
    s = c.debug_get_signs(n) if c.get_stats().status == -7 else None
    m = c.get_M().double()
    xd = x.double()
    norm = xd.norm(dim=1, keepdim=True)
    live = torch.isfinite(norm) & (norm > 0)
    xt = torch.where(live, torch.nan_to_num(xd) / torch.where(live, norm, 1.0), 0.0)
    assert cnt == int(live.sum())
    y, size = xt @ r.double(), xt.abs() @ r.abs().double()
    sd = s.double()
    wrong = (sd != torch.sign(y)) & live
    assert (y.abs()[wrong] <= _unit(d) * size[wrong]).all() and (sd[~live[:, 0]] == 0).all()
    ta = xt.T @ sd / math.sqrt(d)                         # with the signs taken
    # (1 / ||x|| in fp32: a sum of d squares and two roundings, of which a warp's 32 partial sums leave d / 32 + 7 in a chain)
    assert ((m - ta).abs() <= (_unit(n) + (d / 32 + 9) * 2.0 ** -24) * (xt.abs().T @ sd.abs()) / math.sqrt(d) + 1e-30).all()
    ref = float(y.abs().sum()) / math.sqrt(d)
    assert abs(j - ref) <= (_unit(d) * float(size.sum()) / math.sqrt(d)) + (d / 32 + 9) * 2.0 ** -24 * ref


@pytest.mark.parametrize("d,n", [(513, 600), (768, 1025)])
@pytest.mark.parametrize("mode,bits,clip", [("sym", 4, 0.0), ("zp", 3, 0.9)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_quantised_targets_and_strided_rows(d, n, mode, bits, clip, dtype):
    t = torch.float32 if dtype == "f32" else torch.bfloat16
    x = torch.zeros(n, d + 5, dtype=t, device="cuda")[:, 3:d + 3]
    x.copy_(_rand(d + n, n, d))
    r = torch.linalg.qr(_rand(9, d, d).double())[0].float().contiguous()
    c = B.Context(d, n, in_dtype=dtype, mode="exact", quant_bits=bits, quant_mode=mode, clip_ratio=clip, diagnostics=True)
    c.set_R(r)
    c.step(x)
    j, cnt = c.get_objective()
    s = c.debug_get_signs(n).double()
    m = c.get_M().double()
    xt = x.double() / x.double().norm(dim=1, keepdim=True)
    y, size = xt @ r.double(), xt.abs() @ r.abs().double()
    if mode == "sym":
        lev = 2 ** (bits - 1) - 1
        delta = y.abs().amax(1, keepdim=True) / lev
        lo, hi, z = -lev, lev, 0.0
        k = torch.round(y / delta).clamp(lo, hi)
    else:
        lev = 2 ** bits - 1
        a, b = clip * y.amin(1, keepdim=True), clip * y.amax(1, keepdim=True)
        delta = (b - a) / lev
        z = -torch.round(a / delta)
        k = torch.minimum(torch.maximum(torch.round(y / delta), -z), lev - z)
    q = y / delta
    # a code may fall the other way where y / delta lies within the rounding of y (and of the row's range) of a half
    near = ((q - torch.floor(q)) - 0.5).abs() * delta <= 4 * _unit(d) * size
    wrong = s != torch.sign(k)
    assert cnt == n and not (wrong & ~near).any()
    ta = xt.T @ s / math.sqrt(d)
    assert ((m - ta).abs() <= (_unit(n) + (d / 32 + 9) * 2.0 ** -24) * (xt.abs().T @ s.abs()) / math.sqrt(d) + 1e-30).all()
    ref = float((delta * k.abs()).sum()) / math.sqrt(d)
    slack = float((delta * near).sum()) / math.sqrt(d)
    assert abs(j - ref) <= 4 * (_unit(d) * float(size.sum()) / math.sqrt(d)) + (d / 32 + 9) * 2.0 ** -24 * ref + slack
    dg = c.get_diagnostics()[0]
    pr = float((y.pow(2).sum(1) ** 2 / (d * y.pow(4).sum(1))).sum())
    assert abs(dg["sum_pr_over_d"] - pr) <= 1e-4 * pr
    den = float(x.double().pow(2).sum())
    assert abs(dg["qerr_den"] - den) <= 1e-4 * den


def test_rows_accumulate_and_rotation_follows():
    """Two batches of different lengths, an update, and a batch at the rotation it returned."""
    d = 520
    c = B.Context(d, 1500, in_dtype="f32", mode="exact")
    r = torch.linalg.qr(_rand(3, d, d).double())[0].float().contiguous()
    c.set_R(r)
    a, b = _rand(4, 1500, d), _rand(5, 700, d)
    ref = 0.0
    for x in (a, b):
        c.step(x)
        xt = x.double() / x.double().norm(dim=1, keepdim=True)
        ref += float((xt @ r.double()).abs().sum()) / math.sqrt(d)
    j, n = c.get_objective()
    assert n == 2200 and abs(j - ref) <= 2e-6 * ref
    c.update()
    r1 = c.get_R()
    c.step(b)
    xt = b.double() / b.double().norm(dim=1, keepdim=True)
    ref = float((xt @ r1.double()).abs().sum()) / math.sqrt(d)
    j, n = c.get_objective()
    assert n == 700 and abs(j - ref) <= 2e-6 * ref


# the smallest steps that take the pieces, by row type and width: one row of tiles of which the second CTA's half is empty or nearly so
@pytest.mark.parametrize("d,n,dtype", [(768, 64, torch.bfloat16), (769, 65, torch.bfloat16), (1023, 100, torch.bfloat16),
                                       (2050, 64, torch.bfloat16), (768, 342, torch.float32), (1024, 128, torch.float32),
                                       (1030, 130, torch.float32), (2050, 64, torch.float32)])
def test_smallest_steps_over_pieces(d, n, dtype):
    test_signs_statistics_and_objective(d, n, dtype)


# one chunk of 512 terms and a part of another, whole chunks, one k block more; rows of one size and rows that one number rules
@pytest.mark.parametrize("d,n", [(768, 700), (1024, 1024), (1088, 513), (2560, 300)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("massive", [False, True])
def test_objective_is_not_biased(d, n, dtype, massive):
    """What the tensor cores cut off has the sign of the sum: an objective of sums that lose any of it comes out below 64 bits."""
    off = []
    for seed in range(3):
        x = _rand(d + seed, n, d)
        if massive:
            x[torch.arange(n, device="cuda"), torch.randint(0, d, (n,), generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")] *= 300.0
        x = x.to(dtype)
        r = torch.linalg.qr(_rand(70 + seed, d, d).double())[0].float().contiguous()
        c = B.Context(d, n, in_dtype="f32" if dtype == torch.float32 else "bf16", mode="exact")
        c.set_R(r)
        c.step(x)
        xt = x.double() / x.double().norm(dim=1, keepdim=True)
        y = xt @ r.double()
        off.append((c.get_objective()[0] * math.sqrt(d) - float(y.abs().sum())) / float(y.abs().sum()))
        s = c.debug_get_signs(n).double()
        # a rotated number is off by a few 2^-24 of its row's norm over sqrt(d), whatever the number
        assert (y.abs()[s != torch.sign(y)] <= 12.0 * 2.0 ** -24 / math.sqrt(768.0)).all()
    # rows' norms in fp32: d squares in chains of d / 128 and three more sums, a root and a division, each to nearest, the same for a row's
    # numbers and averaged over n rows; sums in one accumulator each of 64 terms left -6e-8 .. -1.2e-7 at any n
    assert max(abs(o) for o in off) <= 2.5e-8, off


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_a_feature_of_tiny_values(dtype):
    """Low pieces of values below 2^-110 or so are subnormal: a feature that small everywhere loses up to 2^-126 a row, absolutely."""
    d, n = 800, 1000
    x = _rand(1, n, d)
    x[:, 7] *= 1e-36
    x = x.to(dtype)
    r = torch.linalg.qr(_rand(7, d, d).double())[0].float().contiguous()
    c = B.Context(d, n, in_dtype="f32" if dtype == torch.float32 else "bf16", mode="exact")
    c.set_R(r)
    c.step(x)
    m, s = c.get_M().double(), c.debug_get_signs(n).double()
    xt = x.double() / x.double().norm(dim=1, keepdim=True)
    err = (m - xt.T @ s / math.sqrt(d)).abs()
    bound = (_unit(n) + (d / 32 + 9) * 2.0 ** -24) * (xt.abs().T @ s.abs()) / math.sqrt(d)
    assert (err <= bound + n * 2.0 ** -126 / math.sqrt(d)).all() and float(m[7].abs().max()) > 0.0


# tiles of the last round shared out over k: all of them (fewer tiles than pairs) in parts of one accumulator, and in runs that straddle two
# tiles; those behind a round of whole tiles; odd widths; a row of tiles that is mostly past the end; quantised targets
@pytest.mark.parametrize("d,n,bits", [(1024, 300, 0), (1100, 257, 0), (2560, 1100, 0), (3072, 512, 0), (3001, 900, 0), (3072, 1000, 4), (4096, 70, 4)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_tiles_shared_out_over_k(d, n, bits, dtype):
    if bits == 0:
        test_signs_statistics_and_objective(d, n, torch.float32 if dtype == "f32" else torch.bfloat16)
    else:
        test_quantised_targets_and_strided_rows(d, n, "sym", bits, 0.0, dtype)
    # the parts are added in their order, whichever comes last
    x = _rand(d + n, n, d).to(torch.float32 if dtype == "f32" else torch.bfloat16)
    r = torch.linalg.qr(_rand(7, d, d).double())[0].float().contiguous()
    c = B.Context(d, n, in_dtype=dtype, mode="exact", quant_bits=bits)
    c.set_R(r)
    runs = []
    for _ in range(6):
        c.set_M(torch.zeros(d, d, device="cuda"), 0.0, 0)
        c.step(x)
        runs.append((c.get_objective(), c.get_M()))
    assert all(j == runs[0][0] and torch.equal(m, runs[0][1]) for j, m in runs[1:])
