"""16-bit storage: the persistent K1 gives the cooperative K1's iterates bit
for bit (same arithmetic, same rounding streams, and sums above the l1 windows
taken in the same order and pieces), at tile edges, ragged sides and band
counts that leave a short last piece."""
import pytest
import torch

from paper_2510_00562_gb300 import synth
from paper_2510_00562_gb300.solver import GeoSSTVSolver, make_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(16, 32, 1), (33, 65, 17), (96, 70, 40), (157, 203, 21)])
@pytest.mark.parametrize("storage", ["bf16", "fp16"])
def test_equals_the_cooperative_kernel(shape, storage, monkeypatch):
    n1, n2, n3 = shape
    pb = synth.make_problem(n1, n2, n3, seed=n1)
    v = torch.from_numpy(pb["v"]).cuda()
    got = []
    for k1 in ("tma", "coop"):
        monkeypatch.setenv("GSSTV_K1", k1)
        p = make_params(eps=pb["eps"], alpha=0.1 * pb["alpha"], beta=0.1 * pb["beta"], omega=0.03, max_iter=40,
                        storage=storage)
        with GeoSSTVSolver(n1, n2, n3, p) as sol:
            got.append([x.clone() for x in sol.solve(v)[:3]])
    for a, b in zip(*got):
        assert torch.equal(a, b)
