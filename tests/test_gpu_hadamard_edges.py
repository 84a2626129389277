"""The tensor-core transform's bf16 write-out at the ends of its 32-chunk groups and 256-chunk tiles."""
import pytest
import torch

from paper_2605_10793_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n", [(128, 1), (128, 31), (128, 33), (128, 255), (128, 257), (256, 17), (64, 66), (4, 96), (1024, 5),
                                 (4096, 9), (8192, 3), (8192, 150), (4096, 1201)])
def test_bf16_rows_match_fp64_and_leave_the_rest_alone(d, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(d + n)
    x = torch.randn(n, d, generator=g, device="cuda").to(torch.bfloat16)
    buf = torch.full((n + 2, d), 7.0, dtype=torch.bfloat16, device="cuda")
    B.conqur_hadamard_rows(x, out=buf[1:n + 1])
    assert B.conqur_hadamard_status() == 0
    y = x.double()
    h = 1
    while h < d:
        v = y.view(n, d // (2 * h), 2, h)
        y = torch.stack((v[:, :, 0] + v[:, :, 1], v[:, :, 0] - v[:, :, 1]), dim=2).reshape(n, d)
        h *= 2
    ref = y / d ** 0.5
    # log2(d) levels of fp32 additions of partial sums bounded by ||x||_2, then one rounding to bf16
    bound = max(d.bit_length() - 1, 1) * 2.0 ** -24 * x.double().norm(dim=1, keepdim=True) + 2.0 ** -8 * ref.abs()
    assert ((buf[1:n + 1].double() - ref).abs() <= bound).all()
    assert (buf[0] == 7.0).all() and (buf[n + 1] == 7.0).all()


@pytest.mark.parametrize("d,n,padx,pady,out", [(128, 300, 8, 8, "bf16"), (128, 5, 16, 0, "f32"), (256, 129, 0, 24, "bf16"), (512, 70, 40, 4, "f32"),
                                               (4096, 21, 8, 8, "bf16"), (4096, 8, 8, 20, "f32"), (8192, 7, 64, 8, "bf16"), (64, 40, 8, 8, "bf16"),
                                               (1024, 33, 20, 20, "bf16")])
def test_strided_rows_agree_with_the_cuda_core_kernel(d, n, padx, pady, out):
    """Rows inside wider buffers, on both routes: both sum in fp32, each partial sum bounded by ||x||_2."""
    g = torch.Generator(device="cuda")
    g.manual_seed(d + n + padx)
    x = torch.randn(n, d + padx, generator=g, device="cuda").to(torch.bfloat16)[:, :d]
    dt = torch.float32 if out == "f32" else torch.bfloat16
    bufs = [torch.full((n, d + pady), 7.0, dtype=dt, device="cuda") for _ in range(2)]
    B.conqur_hadamard_rows(x, out=bufs[0][:, :d])
    B.conqur_hadamard_rows(x, out=bufs[1][:, :d], cuda_cores_only=True)
    assert B.conqur_hadamard_status() == 0
    a, b = bufs[0][:, :d].double(), bufs[1][:, :d].double()
    bound = 2 * (d.bit_length() - 1) * 2.0 ** -24 * x.double().norm(dim=1, keepdim=True)
    if out == "bf16":
        bound = bound + 2.0 ** -7 * b.abs()            # both rounded to bf16, one apart at most
    assert ((a - b).abs() <= bound).all()
    assert (bufs[0][:, d:] == 7.0).all()
    if padx == pady and out == "bf16":                 # in place
        y = torch.full((n, d + padx), 7.0, dtype=dt, device="cuda")
        y[:, :d] = x
        B.conqur_hadamard_rows(y[:, :d], out=y[:, :d])
        assert torch.equal(y[:, :d], bufs[0][:, :d]) and (y[:, d:] == 7.0).all()


@pytest.mark.parametrize("d,n", [(128, 300), (256, 129), (1024, 65), (8192, 20)])
def test_strided_fp32_results_keep_the_cuda_cores_rounding(d, n):
    """fp32 results show what the tensor cores' sums drop: rows inside wider buffers have theirs from fp32 additions."""
    g = torch.Generator(device="cuda")
    g.manual_seed(d + n)
    x = torch.randn(n, d + 8, generator=g, device="cuda").to(torch.bfloat16)[:, :d]
    a, b = (torch.full((n, d + 8), 7.0, device="cuda") for _ in range(2))
    B.conqur_hadamard_rows(x, out=a[:, :d])
    B.conqur_hadamard_rows(x, out=b[:, :d], cuda_cores_only=True)
    assert B.conqur_hadamard_status() == 0
    assert torch.equal(a, b)
