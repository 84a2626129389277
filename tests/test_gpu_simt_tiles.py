"""The fp32 CUDA-core product runs on one of three tiles, chosen from the output's size: every tile gives the same sums."""
import numpy as np
import pytest
import torch

from paper_2605_10793_b200 import binding as B

pytestmark = pytest.mark.gpu


def _rand(seed, *shape):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(*shape, generator=g, device="cuda")


# (rows, cols) of the weight, block = the folded side; edges of the 32, 64 and 128 tiles and of their k pieces (16, 32)
SIZES = [(33, 31), (32, 65), (127, 129), (130, 100), (200, 1003), (1000, 1537), (2049, 640), (4096, 260)]


@pytest.mark.parametrize("rows,cols", SIZES)
@pytest.mark.parametrize("side", ["input", "output"])
def test_fold_edges_and_tile_independence(rows, cols, side):
    w = _rand(rows * 7 + cols, rows, cols)
    k = cols if side == "input" else rows
    r = _rand(3, k, k) / k ** 0.5
    out = B.conqur_fold_weight(w, r, side, "exact")
    ref = w.double() @ r.double() if side == "input" else r.double().T @ w.double()
    # k fused multiply-adds: error at most k 2^-24 of the sum of the terms' sizes
    size = w.abs().double() @ r.abs().double() if side == "input" else r.abs().double().T @ w.abs().double()
    assert ((out.double() - ref).abs() <= k * 2.0 ** -24 * size + 1e-30).all()
    # a slice that a smaller tile serves, with rows that are not 16-byte aligned, adds the same terms in the same order
    if side == "input":
        part = B.conqur_fold_weight(w[1:34], r, side, "exact")
        assert torch.equal(part, out[1:34])
    else:
        part = B.conqur_fold_weight(w[:, 1:30], r, side, "exact")
        assert torch.equal(part, out[:, 1:30])


@pytest.mark.parametrize("d,n", [(2, 5), (31, 64), (33, 300), (129, 1000), (640, 777), (1100, 130)])
def test_step_and_update_over_tiles(d, n):
    """Statistics with skipped rows (zero, NaN, Inf) and the symmetric Newton-Schulz products, against float64."""
    x = _rand(d + n, n, d)
    x[0] = 0.0
    x[n // 2, d // 2] = float("nan")
    x[n - 1, 0] = float("inf")
    q, _ = torch.linalg.qr(_rand(d, d, d).double())
    r = q.float().contiguous()
    c = B.Context(d, n, in_dtype="f32", mode="exact", prior_rel=0.05)
    c.set_R(r)
    c.step(x)
    m = c.get_M(check=False).double()
    keep = [i for i in range(n) if i not in (0, n // 2, n - 1)]
    xt = x[keep].double()
    xt = xt / xt.norm(dim=1, keepdim=True)
    y = xt @ r.double()
    ref = xt.T @ torch.sign(y) / d ** 0.5
    # signs within rounding of zero may differ: sqrt(d) 2^-23 of a row of unit norm, each worth 2 |x| / sqrt(d)
    near = (y.abs() < d ** 0.5 * 2.0 ** -23).double()
    slack = 2.0 * xt.abs().T @ near / d ** 0.5
    assert ((m - ref).abs() <= n * 2.0 ** -24 * (xt.abs().T @ torch.ones_like(y)) / d ** 0.5 + slack + 1e-7).all()
    j, cnt = c.get_objective(check=False)
    assert cnt == len(keep)
    assert abs(j - float(y.abs().sum()) / d ** 0.5) <= 1e-5 * abs(j)
    c.get_stats()                                    # clears the latched non-finite status
    c.update()
    got = c.get_R().double()
    me = m + 0.05 * m.norm() / d ** 0.5 * r.double()
    u, s, vt = torch.linalg.svd(me)
    gap = 1.0 - float((got * me).sum() / s.sum())
    assert gap <= 2e-5
    assert float((got.T @ got - torch.eye(d, device="cuda", dtype=torch.float64)).abs().max()) <= 1e-4


def test_set_R_refuses_in_every_tile_size():
    for d in (2, 33, 200, 1100, 3072):
        c = B.Context(d, 4, in_dtype="f32", mode="exact")
        r = torch.eye(d, device="cuda")
        r[0, d - 1] = 0.01                           # seen only in the corner of R^T R
        with pytest.raises(B.ConqurError):
            c.set_R(r)
        c.set_R(torch.eye(d, device="cuda"))
        assert np.allclose(c.get_R().cpu().numpy(), np.eye(d))


@pytest.mark.parametrize("batch", [1, 3, 40])
def test_exact_update_graph_equals_direct_launches(batch):
    """From a context's second update on, the fp32 iteration is replayed as a graph with a device-side loop: the same bits
    as the launches enqueued one by one, problems that converge after different numbers of steps among them."""
    d, n = 48, 200
    out = []
    for flags in (0, B.CONQUR_DEBUG_NO_GRAPH):
        c = B.Context(d, n, in_dtype="f32", mode="exact", batch=batch, debug_flags=flags)
        for rep in range(3):
            x = _rand(rep, batch, n, d)
            x *= torch.logspace(0, -2, batch, device="cuda")[:, None, None] ** torch.linspace(0, 1, d, device="cuda")
            if batch == 1:
                c.step(x[0])
            else:
                c.step_batched(x, n, d, n * d)
            c.update()
        st = c.get_stats()
        assert st.status == 0 and st.updates == 3
        out.append((c.get_R(), st.ns_steps_used))
    assert torch.equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]


def test_exact_update_inside_a_callers_capture():
    d, n = 64, 256
    x = _rand(1, n, d)
    ref = B.Context(d, n, in_dtype="f32", mode="exact")
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        c = B.Context(d, n, in_dtype="f32", mode="exact")
        for _ in range(2):
            c.step(x)
            c.update()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        c.step(x)
        c.update()
    g.replay()
    torch.cuda.synchronize()
    for _ in range(3):
        ref.step(x)
        ref.update()
    assert torch.equal(c.get_R(), ref.get_R())


@pytest.mark.parametrize("d", [128, 512, 640, 1024])
def test_set_R_decides_alike_in_both_modes(d):
    """The tensor-core contexts decide on a bf16-pair product and go to the fp32 one near the limit of 1e-3: the same
    rotations pass, on both sides of the limit, close to it, and with infinities in them."""
    q = torch.linalg.qr(_rand(d, d, d).double())[0]
    tc = B.Context(d, 8, mode="tc")
    ex = B.Context(d, 8, in_dtype="f32", mode="exact")

    def takes(ctx, r):
        try:
            ctx.set_R(r)
            return True
        except B.ConqurError as e:
            assert e.status == -3
            return False

    cases = []
    for err in (0.0, 2e-4, 8e-4, 9.7e-4, 9.97e-4, 9.997e-4, 1.0003e-3, 1.003e-3, 1.03e-3, 1.3e-3, 0.1):
        r = q.clone()
        r[:, d // 3] *= (1.0 + err) ** 0.5                 # one diagonal element of R^T R off by err
        # (fp32 sums of d terms of size up to 1: within 1e-6 of the limit either answer is right, but the same one)
        want = err < 1e-3 if abs(err - 1e-3) > 2e-6 else None
        cases.append((r.float().contiguous(), want))
        r = q.clone()
        r[:, 1] = (r[:, 1] + err * r[:, d - 1])            # one off-diagonal pair
        cases.append((r.float().contiguous(), want))
    for bad in (float("inf"), 1e30):
        r = q.float().contiguous()
        r[d // 2, 3] = bad
        cases.append((r, False))
    for r, want in cases:
        got = takes(tc, r)
        assert got == takes(ex, r) and want in (None, got)
    big = torch.zeros(d * d + 1, device="cuda")
    big[1:] = q.float().flatten()                          # not 16-byte aligned
    assert takes(tc, big[1:].view(d, d))
    assert torch.equal(tc.get_R(), q.float())


@pytest.mark.parametrize("P", [2, 5, 500])
def test_set_R_of_many_heads_refuses_when_one_is_off(P):
    d = 128
    q = torch.linalg.qr(_rand(P, P, d, d).double())[0]
    tc = B.Context(d, 8, mode="tc", batch=P)
    ex = B.Context(d, 8, in_dtype="f32", mode="exact", batch=P)
    for err, want in ((0.0, True), (9.0e-4, True), (9.95e-4, True), (1.005e-3, False), (1.1e-3, False), (float("inf"), False)):
        for p in sorted({0, P // 2, P - 1}):
            r = q.clone()
            r[p, :, 77] *= (1.0 + err) ** 0.5
            if err == float("inf"):
                r[p] = q[p]
                r[p, 3, 4] = err
            r = r.float().contiguous()
            got = []
            for c in (tc, ex):
                try:
                    c.set_R(r)
                    got.append(True)
                except B.ConqurError as e:
                    assert e.status == -3
                    got.append(False)
            assert got == [want, want], (err, p)
            if want:
                assert torch.equal(tc.get_R(), r)


@pytest.mark.parametrize("n,d", [(2097120, 2), (2097121, 2), (4194240, 33), (4194241, 2), (8388480, 2)])
def test_more_rows_than_a_launch_has_blocks_of_the_smaller_tiles(n, d):
    """65535 rows of tiles at most: 2097120 rows of the 32-row tile, 4194240 of the 64-row one, 8388480 of the 128-row one."""
    x = _rand(n, n, d)
    c = B.Context(d, n, in_dtype="f32", mode="exact")
    r = torch.linalg.qr(_rand(1, d, d))[0].contiguous()
    c.set_R(r)
    c.step(x)
    j, cnt = c.get_objective()
    assert cnt == n
    ref = 0.0
    for part in x.split(1 << 20):
        y = part.double() / part.double().norm(dim=1, keepdim=True)
        ref += float((y @ r.double()).abs().sum()) / d ** 0.5
    # per row of norm 1: fp32 errors of the d sums of d products and of the norm, against a sum of at least 1
    assert abs(j - ref) <= d * (d + 4) * 2.0 ** -24 * ref
    out = B.conqur_fold_weight(x, r, "input", "exact")
    for a in (0, n // 2, n - 1000):                  # first, middle and last tiles
        want = x[a:a + 1000].double() @ r.double()
        assert ((out[a:a + 1000].double() - want).abs() <= d * 2.0 ** -24 * (x[a:a + 1000].abs() @ r.abs()).double() + 1e-30).all()


@pytest.mark.parametrize("mode,d,P", [("exact", 33, 1), ("exact", 600, 1), ("exact", 48, 3), ("tc", 256, 1), ("tc", 640, 1), ("tc", 128, 2),
                                      ("tc", 128, 200)])
def test_set_R_refuses_nan(mode, d, P):
    """A NaN reaches one row and one column of R^T R only; the rotation in place stays."""
    q = torch.linalg.qr(_rand(d, P, d, d).double())[0].float().contiguous()
    c = B.Context(d, 8, in_dtype="f32" if mode == "exact" else "bf16", mode=mode, batch=P)
    c.set_R(q[0] if P == 1 else q)
    for p, i, j in ((0, 0, 0), (P - 1, d - 1, 3), (P // 2, d // 2, d - 1)):
        r = q.clone()
        r[p, i, j] = float("nan")
        with pytest.raises(B.ConqurError) as e:
            c.set_R(r[0] if P == 1 else r)
        assert e.value.status == -3
        assert torch.equal(c.get_R(), q[0] if P == 1 else q)


@pytest.mark.parametrize("d", [512, 1024, 2048, 4096, 8192])
def test_set_R_decides_alike_where_every_term_is_rounded_the_same_way(d):
    """One column of a large entry and small ones whose squares lie just above half a unit of its sum in fp32: the fp32
    product adds a whole unit for each, the tensor cores half of one."""
    tc = B.Context(d, 8, mode="tc")
    ex = B.Context(d, 8, in_dtype="f32", mode="exact")
    eps = 2.0 ** -12 * (1.0 + 2.0 ** -10)
    r = torch.eye(d, device="cuda")
    r[1:, 0] = eps
    fp32 = (d - 1) * 2.0 ** -23
    seen = set()
    for delta in np.linspace(0.0, 1.1e-3, 45):
        r[0, 0] = (1.0 + delta) ** 0.5
        got = []
        for c in (tc, ex):
            try:
                c.set_R(r)
                got.append(True)
            except B.ConqurError as e:
                assert e.status == -3
                got.append(False)
        assert got[0] == got[1], (delta, got)
        if abs(delta + fp32 - 1e-3) > 1e-6:              # (the entry's own rounding)
            assert got[1] == (delta + fp32 < 1e-3), delta
        seen.add(got[0])
    assert seen == {True, False}
