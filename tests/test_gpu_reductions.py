"""Inner products summed across threads and row bands (FP64 path): one band,
bands at and past the 256 that one reduction batch holds, and magnitudes whose
squares come near both ends of the binary64 range; in the oracle's operation
order the decisions are the oracle's, an overflowing flip included."""
import numpy as np
import pytest

import oracle
from paper_2103_07210_gb300 import ftgcr, inputs
from tests.gpu_util import rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [0, -380, 380])
@pytest.mark.parametrize("nlon,nlat,tiles", [(16, 12, 1), (24, 256, 256), (24, 257, 257), (20, 600, 600)])
def test_sums_over_bands_match_oracle(nlon, nlat, tiles, scale):
    p = inputs.hill_problem(nlon, nlat, rhs="random", seed=nlat)
    R = np.ldexp(p.R, scale)
    faults = [(3, "r", (nlon * nlat) // 2, 62)]
    o = oracle.ftgcr(p.D, R, p.mu, 4, 1e-10, faults=faults)
    with ftgcr.Solver(p.D, p.mu, k=4, tol=1e-10, precision="fp64", tiles=tiles, oracle_order=True) as s:
        Rt = torch.from_numpy(R).cuda()
        x = torch.zeros_like(Rt)
        s.solve(Rt, x, faults=faults)
        st = s.stats()
    assert st["tiles"] == tiles
    assert st["steps"] == o["steps"] and st["detect_steps"] == o["detect_steps"] and st["converged"] == o["converged"]
    assert rel_err(x.cpu().numpy(), o["x"]) <= 1e-10
