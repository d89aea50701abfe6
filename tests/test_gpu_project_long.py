"""The l1-ball projection of vectors long enough for the sampled search, and of
those short enough for one CTA, against torch in float64: lengths at the edges of its blocks, unaligned vectors, values
whose sample says little (a period, a few large outliers, ties, all in the
ball), and NaN.  Tolerances: those of the projection's other tests for tau (1e-6
relative); an output is one float32 subtraction of tau rounded to float32, 2^-23
relative to the largest value."""
import pytest
import torch

from paper_2510_00562_gb300.solver import project_l1ball

pytestmark = pytest.mark.gpu
N = 1 << 21


def exact(x, r):
    a = x.double().abs()
    if float(a.sum()) <= r:
        return 0.0
    s = a.sort(descending=True).values
    c = s.cumsum(0) - r
    k = torch.arange(1, len(s) + 1, device=x.device, dtype=torch.float64)
    rho = int((s * k > c).sum())
    return float(c[rho - 1] / rho)


def vector(kind, n):
    g = torch.Generator(device="cuda").manual_seed(n)
    x = 0.1 * torch.randn(n, device="cuda", generator=g)
    if kind == "period":
        x = torch.where(torch.arange(n, device="cuda") % 1024 < 32, 50.0 * x, x)
    if kind == "outliers":
        x[:: n // 3] = 1e4
    if kind == "ties":
        x = (x * 8).round() / 8
    return x


@pytest.mark.parametrize("kind", ["normal", "period", "outliers", "ties"])
@pytest.mark.parametrize("n", [N - 1, N, N + 1023, 3 * N + 5])
@pytest.mark.parametrize("frac", [0.02, 0.6, 0.9999, 2.0])
def test_long_vectors(kind, n, frac):
    x = vector(kind, n)
    for y in (x, x[1:]):
        r = frac * float(y.abs().sum(dtype=torch.float64))
        out, tau = project_l1ball(y, r)
        ref = exact(y, r)
        assert tau == pytest.approx(ref, rel=1e-6, abs=1e-12)
        want = y.double().sign() * (y.double().abs() - ref).clamp(min=0.0)
        assert float((out.double() - want).abs().max()) <= 2.0 ** -23 * float(y.abs().max())


@pytest.mark.parametrize("n", [1, 31, 1024, 8191, 8192, 8193])
@pytest.mark.parametrize("frac", [0.0, 0.02, 0.6, 0.9999, 2.0])
def test_short_vectors(n, frac):
    for x in (vector("normal", n), vector("ties", n)):
        r = frac * float(x.abs().sum(dtype=torch.float64))
        out, tau = project_l1ball(x, r)
        if r == 0.0:
            assert torch.equal(out, torch.zeros_like(x))
            continue
        ref = exact(x, r)
        assert tau == pytest.approx(ref, rel=1e-6, abs=1e-12)
        want = x.double().sign() * (x.double().abs() - ref).clamp(min=0.0)
        assert float((out.double() - want).abs().max()) <= 2.0 ** -23 * float(x.abs().max())


@pytest.mark.parametrize("n", [100, 10000, N])
def test_nan_leaves_the_vector(n):
    x = vector("normal", n)
    x[77] = float("nan")
    out, tau = project_l1ball(x, 10.0)
    assert tau == 0.0 and torch.equal(out.nan_to_num(7.0), x.nan_to_num(7.0))


@pytest.mark.parametrize("n", [64, 4096, 8192, 8193, N + 5])
@pytest.mark.parametrize("top", [2e37, 1e36, 3e38])
@pytest.mark.parametrize("frac", [0.02, 0.6, 2.0])
def test_a_norm_above_the_largest_float(n, top, frac):
    """Finite values whose sum of absolute values float32 cannot hold."""
    g = torch.Generator(device="cuda").manual_seed(n)
    x = top * (2.0 * torch.rand(n, device="cuda", generator=g) - 1.0)
    r = frac * float(x.abs().sum(dtype=torch.float64))
    out, tau = project_l1ball(x, r)
    ref = exact(x, r)
    assert tau == pytest.approx(ref, rel=1e-6)
    want = x.double().sign() * (x.double().abs() - ref).clamp(min=0.0)
    assert float((out.double() - want).abs().max()) <= 2.0 ** -23 * float(x.double().abs().max())
