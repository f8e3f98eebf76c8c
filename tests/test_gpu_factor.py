"""The mixed path's line-preconditioner constants (pivots from ratios of
minors, the bordering solve from running products) at the edges of their
layout: rows shorter and longer than a block of columns loaded ahead, rows of
one piece a thread and of many, widths around both, one latitude row, and a
coefficient scaled near both ends of the FP32 range.  A solve whose
preconditioner were wrong would need more steps than the FP64 path's, which
factorises by the serial chains: with a first-order perturbation of the
preconditioner by FP32 rounding the inner solves take the same steps within
the restarts of the refinement (at most three cycles of k more), and the
solution is the FP64 path's within 1e-7 (both at tol 1e-10; wide grids among them)."""
import numpy as np
import pytest

from paper_2103_07210_gb300 import ftgcr, inputs
from tests.gpu_util import rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 2.0 ** 40, 2.0 ** -40])
@pytest.mark.parametrize("nlon,nlat", [(8, 6), (9, 7), (17, 9), (18, 1), (33, 31), (34, 33), (255, 20), (258, 65), (770, 12)])
def test_mixed_factors_precondition_like_the_chains(nlon, nlat, scale):
    p = inputs.hill_problem(nlon, nlat, rhs="random", seed=nlon)
    D, mu, out = p.D * scale, p.mu * scale, {}
    for precision in ("fp64", "mixed"):
        with ftgcr.Solver(D, mu, k=4, tol=1e-10, precision=precision) as s:
            R = torch.from_numpy(np.ascontiguousarray(p.R)).cuda()
            x = torch.zeros_like(R)
            s.set_coeffs(D)  # once more, through the rebuild
            s.solve(R, x)
            st = s.stats()
        assert st["converged"], (precision, st)
        out[precision] = (x.cpu().numpy(), st["steps"])
    assert out["mixed"][1] <= out["fp64"][1] + 15
    assert rel_err(out["mixed"][0], out["fp64"][0]) <= 1e-7
