"""The per-head update's rotation against the polar factor in 64 bits."""
import pytest
import torch

from paper_2605_10793_b200 import binding as B

pytestmark = pytest.mark.gpu


def _polar(m):
    u, _, vt = torch.linalg.svd(m)
    return u @ vt


# given spectra, and rows that lie far below the others; one problem more than fit the chip at once, and two
@pytest.mark.parametrize("problems", [2, 297])
@pytest.mark.parametrize("kind", [1e-1, 1e-4, 1e-6, "rows 1e-3", "rows 1e-6"])
def test_rotation_of_given_statistics(problems, kind):
    d = 128
    g = torch.Generator(device="cuda").manual_seed(problems)
    m = torch.randn(problems, d, d, generator=g, device="cuda", dtype=torch.float64)
    low = 0.0
    if isinstance(kind, str):
        m[:, ::3] *= float(kind.split()[1])
    else:
        s = torch.logspace(0, torch.log10(torch.tensor(kind)).item(), d, device="cuda", dtype=torch.float64)
        low = 2.0 ** -23 * float((1.0 / s).square().mean().sqrt())
        m = (_polar(m) * s) @ _polar(torch.randn(problems, d, d, generator=g, device="cuda", dtype=torch.float64))
    m = m.float().contiguous()
    c = B.Context(d, 4096, in_dtype="bf16", batch=problems)
    for _ in range(3):                                       # (the planned number of lifting steps, then learnt ones)
        c.set_M(m, [0.0] * problems, [4096] * problems)
        c.update()
    r = c.get_R().double()
    assert c.get_stats().status == 0
    eye = torch.eye(d, device="cuda", dtype=torch.float64)
    assert float((r.mT @ r - eye).abs().max()) <= 1e-4
    err = (r - _polar(m.double())).flatten(1).norm(dim=1) / d ** 0.5
    # each of up to 20 steps rounds the iterate's upper half, the residual and the polynomial to 2^-12 of their size; the pair is good to 2^-24 of
    # an entry, which turns a direction of singular value s by that over s, and so is what a product adds up (low: the mean over directions)
    assert float(err.max()) <= 20 * 2.0 ** -12 + low, float(err.max())
