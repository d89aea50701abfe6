"""The single transposed pass (gsstv_vjp_step) against the FP64 reverse mode at
the edges of its tiles (32 x 16, runs of bands), in place and not.  Tolerance as
for one pass elsewhere: float32 arithmetic on float32 inputs, a few roundings of
6e-8 per term amplified by the stencil sums: 1e-5 relative."""
import numpy as np
import pytest
import torch

from oracle import adjoint as A
from oracle import ppds as o
from paper_2510_00562_gb300 import synth
from paper_2510_00562_gb300.solver import GRAD_PARAMS, STATE_KEYS, STATE_LEAD, GeoSSTVSolver, make_params

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("shape", [(16, 32, 2), (17, 33, 5), (15, 31, 3), (48, 65, 4), (33, 1, 2)])
def test_one_pass_at_tile_edges(shape, in_place):
    n1, n2, n3 = shape
    rs = synth.random_state(n1, n2, n3, seed=n2, scale=0.1)
    rng = np.random.default_rng(5)
    v = rng.uniform(0, 1, (n3, n1, n2)).astype(np.float32)
    kw = dict(eps=0.02 * v.size ** 0.5, alpha=0.4 * np.abs(rs["s"]).sum(dtype=np.float64),
              beta=0.4 * np.abs(rs["t"]).sum(dtype=np.float64), omega=0.05)
    bn = {k: rng.standard_normal(rs[k].shape).astype(np.float32) for k in STATE_KEYS}
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()  # noqa: E731
    with GeoSSTVSolver(n1, n2, n3, make_params(graph_iters=0, **kw)) as sol:
        sol.load(dev(v))
        x = {k: dev(rs[k]) for k in STATE_KEYS}
        sol.set_state(x)
        sol.iterate(1)
        bar, vbar, pbar = sol.vjp_step(x, sol.get_state(), {k: dev(bn[k]) for k in STATE_KEYS}, in_place=in_place)
        got = {k: t.cpu().numpy().astype(np.float64) for k, t in bar.items()}
        vbar = vbar.cpu().numpy().astype(np.float64)
    ref, vref, pref = A.step_vjp(o.State(**{k: rs[k].astype(np.float64) for k in STATE_KEYS}), v.astype(np.float64),
                                 o.Params(**kw), o.State(**{k: bn[k].astype(np.float64) for k in STATE_KEYS}))
    for k in STATE_KEYS:
        assert rel(got[k], getattr(ref, k)) < 1e-5, k
    assert rel(vbar, vref) < 1e-5
    for k in GRAD_PARAMS:
        assert pbar[k] == pytest.approx(pref[k], rel=1e-5, abs=1e-9 * np.linalg.norm(vref)), k


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("shape", [(33, 65, 5)])
def test_one_pass_whose_sums_pass_the_largest_float(shape, in_place):
    """y4 of 4e18: a square is an ordinary float32, a block's sum of them is not."""
    n1, n2, n3 = shape
    rs = synth.random_state(n1, n2, n3, seed=n2, scale=0.1)
    rng = np.random.default_rng(6)
    rs["y4"] = (4e18 * rng.standard_normal((n3, n1, n2))).astype(np.float32)
    v = rng.uniform(0, 1, (n3, n1, n2)).astype(np.float32)
    big = np.abs(rs["y4"]).sum(dtype=np.float64)
    kw = dict(eps=0.02 * v.size ** 0.5, alpha=1e-4 * big, beta=1e-4 * big, omega=0.05)
    bn = {k: rng.standard_normal(rs[k].shape).astype(np.float32) for k in STATE_KEYS}
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()  # noqa: E731
    with GeoSSTVSolver(n1, n2, n3, make_params(graph_iters=0, **kw)) as sol:
        sol.load(dev(v))
        x = {k: dev(rs[k]) for k in STATE_KEYS}
        sol.set_state(x)
        sol.iterate(1)
        bar, vbar, pbar = sol.vjp_step(x, sol.get_state(), {k: dev(bn[k]) for k in STATE_KEYS}, in_place=in_place)
        got = {k: t.cpu().numpy().astype(np.float64) for k, t in bar.items()}
        vbar = vbar.cpu().numpy().astype(np.float64)
    ref, vref, pref = A.step_vjp(o.State(**{k: rs[k].astype(np.float64) for k in STATE_KEYS}), v.astype(np.float64),
                                 o.Params(**kw), o.State(**{k: bn[k].astype(np.float64) for k in STATE_KEYS}))
    for k in STATE_KEYS:
        assert rel(got[k], getattr(ref, k)) < 1e-5, k
    assert rel(vbar, vref) < 1e-5
    for k in GRAD_PARAMS:
        assert pbar[k] == pytest.approx(pref[k], rel=1e-5, abs=1e-9 * np.linalg.norm(vref)), k


def test_workspace_follows_the_form():
    """A call that writes to buffers of its own takes 2 N floats; the spare set of
    8 N is taken by the first call in place, and both forms agree after it."""
    n1, n2, n3 = 48, 65, 4
    n = n1 * n2 * n3
    rs = synth.random_state(n1, n2, n3, seed=3, scale=0.1)
    x = {k: torch.from_numpy(rs[k].astype(np.float32)).cuda() for k in STATE_KEYS}
    with GeoSSTVSolver(n1, n2, n3, make_params(eps=1.0, alpha=10.0, beta=10.0, omega=0.05, graph_iters=0)) as sol:
        sol.load(torch.zeros((n3, n1, n2), device="cuda"))
        sol.set_state(x)
        sol.iterate(1)
        nxt = sol.get_state()
        held, got = [sol.device_bytes()], []
        for in_place in (False, True, False):
            bar = {k: torch.full_like(v, 0.5) for k, v in x.items()}
            got.append(sol.vjp_step(x, nxt, bar, in_place=in_place)[0])
            held.append(sol.device_bytes())
    grown = [b - a for a, b in zip(held, held[1:])]
    assert 8 * n <= grown[0] <= 8 * n + 2048 and 32 * n <= grown[1] <= 32 * n + 4096 and grown[2] == 0
    for k in STATE_KEYS:
        for g in got[1:]:
            assert rel(g[k].double().cpu().numpy(), got[0][k].double().cpu().numpy()) < 1e-6, k


def test_omega_sum_of_long_runs_does_not_drift():
    """w = (2, 0), y = 0 and an adjoint of (1.3, 0) everywhere make every radial part
    1.3 exactly, so the adjoint of omega is -g_w1 3 N 1.3 and what is left is the
    rounding of the sum: one of three terms a band (2^-24 relative) and pairs."""
    n1, n2, n3 = 192, 384, 32                       # blocks that march over all the bands
    zero = {k: torch.zeros(STATE_LEAD[k] + (n3, n1, n2), device="cuda") for k in STATE_KEYS}
    x = dict(zero, w1=zero["w1"].clone())
    bar = dict(zero, w1=zero["w1"].clone())
    x["w1"][:, 0], bar["w1"][:, 0] = 2.0, 1.3
    p = make_params(eps=1.0, alpha=1.0, beta=1.0, omega=0.05, graph_iters=0)
    with GeoSSTVSolver(n1, n2, n3, p) as sol:
        sol.load(zero["u"])
        _, _, pbar = sol.vjp_step(x, zero, bar)
    want = -p.gamma_w1 * 3 * n1 * n2 * n3 * float(np.float32(1.3))
    assert pbar["omega"] == pytest.approx(want, rel=2.0 ** -23)
