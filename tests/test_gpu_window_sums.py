"""Thresholds of a pass whose sums above the l1 windows pass the largest float32:
s and t of +-1e37 that cancel in y4, so that every other sum of the pass is an
ordinary number.  Against the soft threshold in float64; tolerance as for the
projection: one float32 subtraction of tau rounded to float32, 2^-23 relative to
the largest value."""
import contextlib

import pytest
import torch

from paper_2510_00562_gb300.solver import STATE_KEYS, STATE_LEAD, GeoSSTVSolver, make_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fixed", [False, True])
@pytest.mark.parametrize("shape", [(16, 32, 2), (48, 65, 40), (157, 203, 21)])
def test_thresholds_of_sums_above_the_largest_float(shape, fixed):
    n1, n2, n3 = shape
    g = torch.Generator(device="cuda").manual_seed(n1)
    a = 1e37 * (2.0 * torch.rand((n3, n1, n2), device="cuda", generator=g) - 1.0)
    x = {k: torch.zeros(STATE_LEAD[k] + (n3, n1, n2), device="cuda") for k in STATE_KEYS}
    x["s"], x["t"] = a, -a
    mag = a.double().abs().flatten().sort(descending=True).values
    r = 0.4 * float(mag.sum())
    excess = mag * torch.arange(1, len(mag) + 1, device="cuda") - (mag.cumsum(0) - r)
    m = int((excess > 0).sum())
    tau = float((mag[:m].sum() - r) / m)
    want = a.double().sign() * (a.double().abs() - tau).clamp(min=0.0)
    with GeoSSTVSolver(n1, n2, n3, make_params(eps=1.0, alpha=r, beta=r, omega=0.03, graph_iters=0)) as sol:
        sol.load(torch.zeros_like(a))
        sol.set_state(x)
        with sol.fixed_sums() if fixed else contextlib.nullcontext():
            sol.iterate(1)
        got = sol.get_state()
    for k, sign in (("s", 1.0), ("t", -1.0)):
        assert float((got[k].double() - sign * want).abs().max()) <= 2.0 ** -23 * float(mag[0]), k
