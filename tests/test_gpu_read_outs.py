"""Read-outs and set_M: small results go through page-locked memory, those of many problems by a copy."""
import numpy as np
import pytest
import torch

from paper_2605_10793_b200 import binding as B

pytestmark = pytest.mark.gpu


# 16 bytes a problem and the status: 2047 problems fill the 32 KB they go through, 2048 do not; odd widths leave the 16-byte pieces
@pytest.mark.parametrize("batch,d", [(1, 3), (1, 640), (2, 5), (2047, 2), (2048, 2), (2500, 3)])
def test_statistics_round_trip(batch, d):
    g = torch.Generator(device="cuda").manual_seed(batch + d)
    contexts = [B.Context(d, 4, in_dtype="f32", mode="exact", batch=batch) for _ in range(3)]      # (more than one at a time)
    kept = []
    for i, c in enumerate(contexts):
        m = torch.randn(batch, d, d, generator=g, device="cuda")
        j, n = np.arange(batch) * 0.5 + i, np.arange(batch) + 7 * i
        c.set_M(m if batch > 1 else m[0], j, n)
        kept.append((m, j, n))
    for c, (m, j, n) in zip(contexts, kept):
        got_j, got_n = c.get_objective()
        assert np.array_equal(np.atleast_1d(got_j), j) and np.array_equal(np.atleast_1d(got_n), n)
        # scaled by sqrt(d) and back, each factor and product rounded to fp32
        assert torch.allclose(c.get_M().view(batch, d, d), m, rtol=4 * 2.0 ** -24, atol=0.0)
        eye = torch.eye(d, device="cuda").expand(batch, d, d)
        assert torch.equal(c.get_R().view(batch, d, d), eye)
    contexts[0].close()
    again = B.Context(d, 4, in_dtype="f32", mode="exact", batch=batch)                             # (takes the freed slot)
    assert np.array_equal(np.atleast_1d(again.get_objective()[0]), np.zeros(batch))
    assert np.array_equal(np.atleast_1d(contexts[1].get_objective()[0]), kept[1][1])


def test_status_of_any_problem_is_reported():
    c = B.Context(2, 4, in_dtype="f32", mode="exact", batch=300)
    x = torch.randn(300, 4, 2, device="cuda")
    x[299, 1, 0] = float("nan")
    c.step_batched(x, 4, 2, 8)
    for call in (c.get_R, c.get_M, c.get_objective):
        with pytest.raises(B.ConqurError) as e:
            call()
        assert e.value.status == -7
    assert c.get_stats().status == -7
    c.get_R()


@pytest.mark.parametrize("mode,d,batch", [("exact", 33, 1), ("tc", 256, 1), ("tc", 128, 3)])
def test_rotation_into_memory_that_is_not_this_gpus(mode, d, batch):
    """conqur_get_R into page-locked host memory and at an odd device address: what a device-to-device copy reaches."""
    c = B.Context(d, 64, in_dtype="bf16", mode=mode, batch=batch)
    r = torch.linalg.qr(torch.randn(batch, d, d, device="cuda", dtype=torch.float64))[0].float().contiguous()
    c.set_R(r if batch > 1 else r[0])
    host = torch.zeros(batch, d, d, dtype=torch.float32).pin_memory()
    assert B.conqur_get_R(c.h, host.data_ptr()) == 0
    assert torch.equal(host, r.cpu())
    odd = torch.zeros(batch * d * d + 1, device="cuda")
    assert B.conqur_get_R(c.h, odd.data_ptr() + 4) == 0
    assert torch.equal(odd[1:].view(batch, d, d), r)


def test_objective_behind_long_and_short_work():
    """The word that says the results are there is the call's own, whatever it waited for: sums of every step as it is read, in turn from contexts
    that each use their slot, and from one that takes over a closed one's."""
    d = 700
    rows = torch.randn(16384, d, device="cuda")
    work = [rows, rows[:3]]                                  # steps of over 1 ms and of some 40 us; a call looks out for its word for 200 us
    contexts = [B.Context(d, 16384, in_dtype="f32", mode="exact") for _ in range(3)]
    alone = []                                               # what either batch adds to J
    for x in work:
        contexts[0].step(x)
        torch.cuda.synchronize()
        alone.append(contexts[0].get_objective()[0])
        contexts[0].set_M(torch.zeros(d, d, device="cuda"), 0.0, 0)
    sums = [[0.0, 0] for _ in contexts]
    order = [(i, w) for w in (0, 1, 1, 0, 0, 1) for i in range(3)] * 8
    for k, (i, w) in enumerate(order):
        if k % 17 == 16:                                     # another context, in the slot this one leaves
            contexts[i].close()
            contexts[i], sums[i] = B.Context(d, 16384, in_dtype="f32", mode="exact"), [0.0, 0]
        contexts[i].step(work[w])
        sums[i][0] += alone[w]
        sums[i][1] += work[w].shape[0]
        j, got = contexts[i].get_objective()
        assert got == sums[i][1]
        assert abs(j - sums[i][0]) <= 1e-12 * sums[i][0]     # (the same doubles, added in another order at most)


@pytest.mark.parametrize("mode,d,batch", [("exact", 16, 1), ("exact", 778, 1), ("tc", 128, 32), ("tc", 1024, 1)])
def test_cross_covariance_into_page_locked_memory(mode, d, batch):
    """conqur_get_M where the host reads: what it has left is there when it returns, behind long and short work."""
    c = B.Context(d, 4096, in_dtype="f32", mode=mode, batch=batch)
    g = torch.Generator(device="cuda").manual_seed(d)
    host = torch.zeros(batch, d, d).pin_memory()
    filler = torch.empty(1 << 27, device="cuda")
    for k in range(40):
        m = torch.randn(batch, d, d, generator=g, device="cuda")
        c.set_M(m if batch > 1 else m[0], [0.0] * batch if batch > 1 else 0.0, [1] * batch if batch > 1 else 1)
        want = c.get_M().cpu().view(batch, d, d)
        host.zero_()
        for _ in range(k % 3):
            filler.fill_(float(k))                           # (some 80 us each)
        assert B.conqur_get_M(c.h, host.data_ptr()) == 0
        assert torch.equal(host, want)


@pytest.mark.parametrize("d", [33, 160, 640])
def test_rotations_refused_and_taken_in_turn(d):
    """conqur_set_R reads its decision from the same place, behind long and short work."""
    c = B.Context(d, 4096, in_dtype="f32", mode="exact")
    x = torch.randn(4096, d, device="cuda")
    q = [torch.linalg.qr(torch.randn(d, d, device="cuda", dtype=torch.float64))[0].float().contiguous() for _ in range(2)]
    for k in range(24):
        if k % 2:
            for _ in range(4):
                c.step(x)
        c.set_R(q[k % 2])
        with pytest.raises(B.ConqurError):
            c.set_R(1.01 * q[1 - k % 2])
        assert torch.equal(c.get_R(), q[k % 2])
