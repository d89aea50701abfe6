"""A batch of as many cubes as one launch takes, of very uneven sizes, so that its
launches have several CTAs per SM: every cube equals its single solve.  Tolerance
as for the other batches: the order of the global sums, 1e-6 relative."""
import numpy as np
import pytest
import torch

import bench
from paper_2510_00562_gb300 import synth
from paper_2510_00562_gb300.solver import GeoSSTVBatch, GeoSSTVSolver, make_params

pytestmark = pytest.mark.gpu


def rel(a, b):
    a, b = a.double(), b.double()
    return float((a - b).norm() / b.norm()) if b.any() else float(a.norm())


@pytest.mark.parametrize("count", [2, 24, 64])
def test_every_cube_equals_its_single_solve(count):
    shapes, params, vs = [], [], []
    for k, (n1, n2, n3, sigma, sp, st) in enumerate(bench.batch_workload(count)):
        n1, n2, n3 = n1 // 2 + k % 3, n2 // 2 + k % 5, n3 // 2       # (odd sides among them)
        pb = synth.make_problem(n1, n2, n3, seed=k, noise=synth.NoiseSpec(sigma=sigma, sp_rate=sp, stripe_rate=st,
                                                                            stripe_amp=0.25))
        shapes.append((n1, n2, n3))
        params.append(make_params(eps=pb["eps"], alpha=pb["alpha"], beta=pb["beta"], omega=0.03,
                                  max_iter=int(np.random.default_rng(k).integers(24, 49))))
        vs.append(torch.from_numpy(pb["v"]).cuda())
    with GeoSSTVBatch(shapes, params) as bt:
        us, ss, ts, done = bt.solve(vs)
    for k, (n1, n2, n3) in enumerate(shapes):
        with GeoSSTVSolver(n1, n2, n3, params[k]) as sol:
            u, s, t, n = sol.solve(vs[k])
        assert done[k] == n == params[k].max_iter
        for got, want in ((us[k], u), (ss[k], s), (ts[k], t)):
            assert rel(got, want) < 1e-6, (k, shapes[k])
