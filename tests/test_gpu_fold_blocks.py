"""Block-diagonal weight folds over bf16 pieces on the tensor cores against float64, and the values that pieces cannot hold."""
import pytest
import torch

from paper_2605_10793_b200 import binding as B

pytestmark = pytest.mark.gpu


def _rand(seed, *shape):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(*shape, generator=g, device="cuda")


def _reference(w, r, side):
    k, b = r.shape[0], r.shape[1]
    w, r = w.double(), r.double()
    if side == "input":
        return torch.einsum("akb,kbc->akc", w.view(-1, k, b), r).reshape(w.shape)
    return torch.einsum("kba,kbc->kac", r, w.view(k, b, -1)).reshape(w.shape)


# (blocks, block, other side): odd numbers of 64-blocks, fewest tiles and more than one a block of threads, remainders of a tile
# and of 16-byte pieces; the first two and some of the next three stay on the CUDA cores, the last four are the smallest that do not
SHAPES = [(2, 64, 32), (3, 128, 127), (65, 64, 993), (2, 128, 4065), (3, 128, 2690), (32, 128, 1003), (127, 64, 640), (4, 128, 9000),
          (3, 128, 2560), (80, 128, 96), (241, 64, 512), (129, 64, 1030)]


@pytest.mark.parametrize("k,b,other", SHAPES)
@pytest.mark.parametrize("side", ["input", "output"])
@pytest.mark.parametrize("mode", ["exact", "tc"])
def test_fold_of_several_blocks(k, b, other, side, mode):
    shape = (other, k * b) if side == "input" else (k * b, other)
    r = _rand(k + b, k, b, b) / b ** 0.5
    wide = _rand(other, shape[0], shape[1] + 3) * torch.exp(3.0 * _rand(other + 1, shape[0], 1))
    for w in (wide[:, : shape[1]].contiguous(), wide[:, 1: shape[1] + 1]):           # (the second off 16-byte boundaries)
        got = B.conqur_fold_weight(w, r, side, mode).double()
        ref, size = _reference(w.contiguous(), r, side), _reference(w.abs().contiguous(), r.abs(), side)
        # two sums of 64 terms: per sum 4 instructions' cuts of 16 2^-25 + 2^-23, the smaller pieces' twenty at 2^-7 of that,
        # the pieces' remainder 2^-25; one fp32 addition
        assert ((got - ref).abs() <= (4 * 10 + 4 + 2) * 2.0 ** -24 * size).all()
        assert float((got - ref).norm() / ref.norm()) <= 4.0 * 2.0 ** -24           # an fp32 chain of 64 leaves 2.4 .. 2.9, of 128 3.4 .. 3.7


@pytest.mark.parametrize("side", ["input", "output"])
@pytest.mark.parametrize("b", [64, 128])
def test_values_that_pieces_cannot_hold(side, b):
    """Infinities, NaN, the largest and tiny values give what a fold of the one block by itself gives."""
    k, other = 4, 16500
    r = _rand(1, k, b, b) / b ** 0.5
    w = _rand(2, *((other, k * b) if side == "input" else (k * b, other)))
    v = w if side == "input" else w.T                   # (other, folded)
    v[3, b + 5] = float("inf")
    v[4, 5] = float("nan")
    v[140, 2 * b + 1] = 3.4e38
    v[290, : k * b] *= 1e-36
    r[3, 2, 2] = float("-inf")
    got = B.conqur_fold_weight(w, r, side, "exact")
    for i in range(k):
        part = w[:, i * b:(i + 1) * b] if side == "input" else w[i * b:(i + 1) * b]
        ref = B.conqur_fold_weight(part, r[i], side, "exact")
        out = got[:, i * b:(i + 1) * b] if side == "input" else got[i * b:(i + 1) * b]
        assert torch.equal(torch.isnan(out), torch.isnan(ref))
        assert torch.equal(torch.isinf(out), torch.isinf(ref))
        assert torch.equal(out[torch.isinf(out)], ref[torch.isinf(ref)])
        fine = torch.isfinite(ref)
        p, q = out.double(), ref.double()
        sz = _reference(torch.nan_to_num(part, 0.0, 0.0, 0.0).abs(), torch.nan_to_num(r[i:i + 1], 0.0, 0.0, 0.0).abs(), side)
        assert ((p - q).abs()[fine] <= (b + 46) * 2.0 ** -24 * sz[fine]).all()


def _median_us(call, n=21):
    for _ in range(3):
        call()
    times = []
    for _ in range(n):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        call()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b) * 1e3)
    return sorted(times)[n // 2]


# (blocks, block, other side): whole tiles and remainders, an odd number of 64-blocks; W off 16-byte boundaries in the last two
@pytest.mark.parametrize("k,b,other,pad", [(32, 128, 2048, 0), (65, 64, 4100, 1), (5, 128, 2690, 1)])
@pytest.mark.parametrize("side", ["input", "output"])
@pytest.mark.parametrize("where", ["one a tile", "every row", "rotation", "all"])
def test_tiny_values_change_no_other_element_and_cost_nothing(k, b, other, pad, side, where):
    """Values whose low pieces would be subnormal, and subnormal ones: held exactly, at the speed of any others."""
    r = _rand(k, k, b, b) / b ** 0.5
    w = _rand(other, *((other, k * b + pad) if side == "input" else (k * b, other + pad)))
    w = w[:, : w.shape[1] - pad]
    v, q = w.clone(), r.clone()
    if pad:
        v = torch.nn.functional.pad(v, (0, 1))[:, :-1]
    vo = v if side == "input" else v.T                                   # (other, folded)
    touched = torch.zeros(other, k, b, dtype=torch.bool, device="cuda")  # element (o, block, column of its rotation)
    if where == "one a tile":
        vo[5::128, 7::128] = 1e-35
        touched[5::128, 0::(128 // b)] = True
    elif where == "every row":
        vo[:, 3::b] = 3e-39
        touched[:] = True
    elif where == "rotation":
        q[:, 3, 9::32] = -2e-41
        touched[:, :, 9::32] = True
    else:
        vo *= 1e-33
        q *= 1e-3
        touched[:] = True
    clean, got = (B.conqur_fold_weight(a, c, side, "exact") for a, c in ((w, r), (v, q)))
    back = lambda t: (t if side == "input" else t.T).reshape(other, k, b)
    assert torch.equal(back(got)[~touched], back(clean)[~touched])
    ref = torch.einsum("okb,kbc->okc", vo.double().reshape(other, k, b), q.double())
    size = torch.einsum("okb,kbc->okc", vo.double().abs().reshape(other, k, b), q.double().abs())
    # (the bound of the first test; a subnormal result is rounded to a multiple of 2^-149)
    assert ((back(got) - ref).abs() <= (4 * 10 + 4 + 2) * 2.0 ** -24 * size + 2.0 ** -150).all()
    t = [_median_us(lambda a=a, c=c: B.conqur_fold_weight(a, c, side, "exact")) for a, c in ((w, r), (v, q))]
    assert t[1] <= 2.0 * t[0] + 20.0, t                                  # (element by element it took 5 .. 11 ms for 70 us)


@pytest.mark.parametrize("k,b,other", [(32, 128, 2048), (65, 64, 4100)])
@pytest.mark.parametrize("side", ["input", "output"])
def test_large_values_cost_one_more_fold(side, k, b, other):
    """Infinities, NaN and values whose scaled sums could overflow: the fold is done again on the CUDA cores, and once is enough."""
    r = _rand(1, k, b, b) / b ** 0.5
    w = _rand(2, *((other, k * b) if side == "input" else (k * b, other)))
    clean = _median_us(lambda: B.conqur_fold_weight(w, r, side, "exact"))
    for bad in (float("nan"), float("inf"), 6e11):
        v = w.clone()
        v[7::128, 5::128] = bad
        assert _median_us(lambda: B.conqur_fold_weight(v, r, side, "exact")) <= 6.0 * clean + 100.0
    # the limits themselves: |W| < 2^39 and |R| < 2^16 stay on the pieces, beyond them a chain of fp32 multiply-adds gives the same
    for scale_w, scale_r in ((2.0 ** 36, 2.0 ** 14), (2.0 ** 60, 2.0 ** 40)):
        got = B.conqur_fold_weight(w * scale_w, r * scale_r, side, "exact").double() / (scale_w * scale_r)
        ref, size = _reference(w, r, side), _reference(w.abs(), r.abs(), side)
        assert ((got - ref).abs() <= (b + 2) * 2.0 ** -24 * size).all()


# many blocks and a short other side, and just below each size from which the pieces are taken
@pytest.mark.parametrize("k,b,other,side", [(1024, 64, 1, "input"), (512, 64, 32, "output"), (1024, 128, 17, "input"), (130, 128, 95, "output"),
                                            (2, 128, 3839, "input"), (2, 128, 3839, "output"), (257, 64, 255, "input"),
                                            (64, 64, 959, "input"), (257, 64, 511, "output"), (64, 64, 1919, "output")])
def test_short_and_small_folds_stay_on_the_cuda_cores(k, b, other, side):
    """Their tiles would be mostly empty: the same bits as block by block (one block is always folded there)."""
    r = _rand(k, k, b, b) / b ** 0.5
    w = _rand(other, *((other, k * b) if side == "input" else (k * b, other)))
    got = B.conqur_fold_weight(w, r, side, "exact")
    for i in range(0, k, max(1, k // 16)):
        cut = (slice(None), slice(i * b, (i + 1) * b)) if side == "input" else (slice(i * b, (i + 1) * b), slice(None))
        assert torch.equal(got[cut], B.conqur_fold_weight(w[cut], r[i], side, "exact"))


# one group of blocks and several a block of threads, an odd number of 64-blocks, remainders of a tile
@pytest.mark.parametrize("k,b,other", [(3, 128, 2690), (241, 64, 512), (256, 128, 97)])
@pytest.mark.parametrize("side", ["input", "output"])
def test_rotations_and_results_off_16_byte_boundaries(k, b, other, side):
    """R that the copy engine does not take, and out whose rows 16-byte stores do not: the same bits."""
    w = _rand(other, *((other, k * b) if side == "input" else (k * b, other)))
    r = _rand(k, k, b, b) / b ** 0.5
    odd = torch.empty(r.numel() + 1, device="cuda")[1:].view(k, b, b)
    odd.copy_(r)
    ref = B.conqur_fold_weight(w, r, side, "exact")
    assert torch.equal(B.conqur_fold_weight(w, odd, side, "exact"), ref)
    rows, cols = w.shape
    wide = torch.full((rows, cols + 1), 7.0, device="cuda")
    scratch = torch.empty(4096, dtype=torch.uint8, device="cuda")
    code = B.CONQUR_FOLD_INPUT if side == "input" else B.CONQUR_FOLD_OUTPUT
    rc = B.load().conqur_fold_weight(w.data_ptr(), w.stride(0), rows, cols, r.data_ptr(), b, code, B.CONQUR_EXACT_F32, wide.data_ptr(),
                                     wide.stride(0), scratch.data_ptr(), 4096, torch.cuda.current_stream().cuda_stream)
    assert rc == 0 and torch.equal(wide[:, :cols], ref) and bool((wide[:, cols] == 7.0).all())
