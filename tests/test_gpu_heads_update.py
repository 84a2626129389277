"""The per-head update's rotation against the polar factor in 64 bits."""
import pytest
import torch

from paper_2605_10793_b200 import binding as B

pytestmark = pytest.mark.gpu
D = 128


def _polar(m):
    u, _, vt = torch.linalg.svd(m)
    return u @ vt


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _updated(m, updates=3):
    """R after so many updates (the first with the planned number of lifting steps, the others with learnt ones) and the steps taken."""
    problems = m.shape[0]
    c = B.Context(D, 4096, in_dtype="bf16", batch=problems)
    for _ in range(updates):
        c.set_M(m, [0.0] * problems, [4096] * problems)
        c.update()
    st = c.get_stats()
    assert st.status == 0
    r = c.get_R().double()
    eye = torch.eye(D, device="cuda", dtype=torch.float64)
    assert float((r.mT @ r - eye).abs().max()) <= 1e-4
    return r, st.ns_steps_used


def _error(r, m):
    return (r - _polar(m.double())).flatten(1).norm(dim=1) / D ** 0.5


# A step rounds the iterate's upper half, the residual and the polynomial to at most 2^-9 of their size, 2^-9 / sqrt(3) each on average: 2^-9 a step,
# sqrt(steps) of that in all where they are independent, and two and a half times that at the worst of some hundred problems.
def _roundings(steps):
    return 2.5 * steps ** 0.5 * 2.0 ** -9


# given spectra; two problems, and one more than fit the chip at once
@pytest.mark.parametrize("problems", [2, 297])
@pytest.mark.parametrize("smallest", [1e-1, 1e-4, 1e-6])
def test_rotation_of_given_spectra(problems, smallest):
    g = torch.Generator(device="cuda").manual_seed(problems)
    s = smallest ** (torch.arange(D, device="cuda", dtype=torch.float64) / (D - 1))
    m = ((_polar(_randn(g, problems, D, D)) * s) @ _polar(_randn(g, problems, D, D))).float().contiguous()
    r, steps = _updated(m)
    # the pair holds an entry to 2^-18 of itself, on average to half of that: a singular direction turns by that share of the norm, which its 128
    # neighbours divide among them, over its own singular value
    pair = 2.0 ** -19 * float(s.norm()) / D ** 0.5 * float((1.0 / s).square().mean().sqrt())
    assert float(_error(r, m).max()) <= _roundings(steps) + pair


# rows or columns far below the others, alone or a third of them, in some problems of several: the iterate keeps fp32's range
@pytest.mark.parametrize("axis", ["rows", "columns"])
@pytest.mark.parametrize("part", ["one", "a third"])
@pytest.mark.parametrize("scale", [1e-3, 1e-6, 1e-8, 1e-10, 1e-11, 1e-12, 1e-13])
def test_rotation_of_rows_and_columns_far_below_the_others(axis, part, scale):
    g = torch.Generator(device="cuda").manual_seed(7)
    s = torch.linspace(1.0, 0.3, D, device="cuda", dtype=torch.float64)      # (no singular value is small by chance)
    m = (_polar(_randn(g, 10, D, D)) * s) @ _polar(_randn(g, 10, D, D))
    where = slice(5, 6) if part == "one" else slice(None, None, 3)
    if axis == "rows":
        m[::3, where] *= scale
    else:
        m[::3, :, where] *= scale
    m = m.float().contiguous()
    r, steps = _updated(m, updates=1)
    assert float(_error(r, m).max()) <= _roundings(steps)


@pytest.mark.parametrize("n", [128, 160, 512])
@pytest.mark.parametrize("quant", [dict(), dict(quant_bits=4), dict(quant_bits=4, quant_mode="zp", clip_ratio=0.9)])
def test_singular_directions_keep_their_sign(n, quant):
    """Fresh rows with two loud channels, few of them: statistics whose least singular values lie far below the largest.  The pair turns a direction
    of singular value s by about 3e-7 / s of the largest (see above), so its sign is safe well above that."""
    problems = 512
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randn(problems, n, D, generator=g, device="cuda")
    x[:, :, [5, 77]] *= 100.0
    r0 = _polar(_randn(g, problems, D, D)).float().contiguous()
    c = B.Context(D, n, in_dtype="bf16", batch=problems, prior_rel=0.01, **quant)
    c.set_R(r0)
    c.step_batched(x.to(torch.bfloat16), n, D, n * D)
    m = c.get_M().double()
    c.update()
    r = c.get_R().double()
    assert c.get_stats().status == 0
    lam = 0.01 * m.flatten(1).norm(dim=1) / D ** 0.5
    u, s, vt = torch.linalg.svd(m + lam[:, None, None] * r0.double())
    along = torch.einsum("pki,pkl,pil->pi", u, r, vt)                        # 1 where a direction is the polar factor's, -1 with the other sign
    assert not bool(((along < 0) & (s > 1e-6 * s[:, :1])).any())
