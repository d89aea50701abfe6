"""The FP64 adjoints of an unrolled run, to 1e-9 of recorded ones.

A threshold or an l2-ball scale that rounds to the neighbouring float32 moves
these adjoints by 1e-8 to 1e-5, so the sums behind them keep one order and
rounding in the passes of a differentiated run (gsstv_set_fixed_sums).  The
problems are exact in float32 (multiples of 1/1024), so that they are the same on
every machine.  tests/golden/gradient_sums.json holds the adjoints that these sums
gave on a GB300 when they were fixed; those of one run differ from the next by the
order of FP64 atomics, about 1e-15."""
import json
import os

import numpy as np
import pytest
import torch

from paper_2510_00562_gb300.autograd import unrolled_geosstv
from paper_2510_00562_gb300.solver import GRAD_PARAMS, GeoSSTVSolver, make_params

pytestmark = pytest.mark.gpu
GOLDEN = json.load(open(os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "gradient_sums.json")))


def problem(n1, n2, n3, seed):
    """Blocks, noise, stripes and salt and pepper, in multiples of 1/1024; the
    clean cube and the radii that bind."""
    rng = np.random.default_rng(seed)
    blocks = rng.integers(0, 1024, (n3, 4, 4))
    clean = blocks[:, np.arange(n1)[:, None] * 4 // n1, np.arange(n2)[None, :] * 4 // n2]
    noise = rng.integers(-88, 89, (4, n3, n1, n2)).sum(0)
    stripe = np.where(rng.integers(0, 20, (n3, 1, n2)) == 0, rng.integers(-256, 257, (n3, 1, n2)), 0)
    hit, val = rng.integers(0, 20, (n3, n1, n2)) == 0, 1024 * rng.integers(0, 2, (n3, n1, n2))
    v = np.where(hit, val, clean + noise + stripe)
    radii = dict(eps=0.95 * float(np.square(noise * ~hit).sum()) ** 0.5 / 1024,
                 alpha=0.9 * float((np.abs(val - clean - stripe) * hit).sum()) / 1024,
                 beta=0.9 * float(n1 * np.abs(stripe).sum()) / 1024, omega=0.03)
    return (v / 1024).astype(np.float32), (clean / 1024).astype(np.float32), radii


def adjoints(case, solve=unrolled_geosstv, solver=GeoSSTVSolver, params=make_params):
    n1, n2, n3 = case["shape"]
    v, clean, radii = problem(n1, n2, n3, case["seed"])
    r = {k: torch.tensor(x, dtype=torch.float64, requires_grad=True) for k, x in radii.items()}
    sol = solver(n1, n2, n3, params(max_iter=case["iters"], **radii))
    u = solve(torch.from_numpy(v).cuda(), *(r[k] for k in GRAD_PARAMS), iters=case["iters"], solver=sol,
              ckpt_every=case["ckpt"])
    ((u - torch.from_numpy(clean).cuda()) ** 2).sum().backward()
    sol.close()
    return {k: float(r[k].grad) for k in GRAD_PARAMS}


@pytest.mark.parametrize("case", GOLDEN, ids=lambda c: "x".join(map(str, c["shape"])) + "-%d" % c["seed"])
def test_adjoints_are_the_recorded_ones(case):
    got = adjoints(case)
    for k in GRAD_PARAMS:
        assert got[k] == pytest.approx(case[k], rel=1e-9), k


def test_an_autotuned_or_solving_handle_gives_the_same():
    """Neither the run length that the autotuner keeps nor a solve in between
    changes the sums of a differentiated run."""
    case = GOLDEN[0]
    n1, n2, n3 = case["shape"]
    v, _, radii = problem(n1, n2, n3, case["seed"])
    v = torch.from_numpy(v).cuda()
    bar = torch.ones_like(v)
    with GeoSSTVSolver(n1, n2, n3, make_params(max_iter=case["iters"], **radii)) as sol:
        sol.load(v)
        a = sol.unrolled_vjp(case["iters"], bar)
        sol.autotune(v, passes=2)
        sol.solve(v)
        sol.load(v)
        b = sol.unrolled_vjp(case["iters"], bar)
    assert torch.equal(a[0], b[0])
    for k in GRAD_PARAMS:
        assert b[1][k] == pytest.approx(a[1][k], rel=1e-12), k
