"""A handle's solve number is ten bits of the tags by which banded rounds tell
new edge rows from old: 1024 solves later the number repeats.  Here the rows
of the earlier solve are then still where its last round left them, because
every solve between starts converged and sends rows in at most one round; a
solve that took them for new would use old neighbour rows in its first step.
The last solve must be bitwise that of a new handle."""
import numpy as np
import pytest

from paper_2103_07210_gb300 import ftgcr, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NLON, NLAT, TOL = 128, 24, 1e-8


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_solve_number_repeats_without_meeting_old_rows(precision):
    p = inputs.hill_problem(NLON, NLAT, rhs="random", seed=3)
    q = inputs.hill_problem(NLON, NLAT, rhs="random", seed=4)
    R, R2 = torch.from_numpy(p.R).cuda(), torch.from_numpy(q.R).cuda()
    opts = dict(k=4, precision=precision)
    with ftgcr.Solver(p.D, p.mu, tol=1e-14 if precision == "fp64" else 1e-13, **opts) as s:
        exact = torch.zeros_like(R)
        s.solve(R, exact)
    with ftgcr.Solver(p.D, p.mu, tol=TOL, **opts) as s:
        # one step away: a smooth error whose residual is a little above the tolerance
        err = torch.from_numpy(np.ascontiguousarray(np.broadcast_to(np.sin(np.arange(NLAT))[:, None], p.R.shape))).cuda()
        lerr = torch.zeros_like(err)
        s.apply_operator(err, lerr)
        x = exact + err * (1.2 * TOL * R.norm() / lerr.norm())
        s.solve(R, x)
        first = s.stats()
        assert first["steps"] == 1 and first["converged"], first
        for _ in range(1023):
            x.copy_(exact)
            s.solve_async(R, x)
        assert s.stats()["steps"] == 0
        x.zero_()
        s.solve(R2, x)  # the first solve's number again
        with ftgcr.Solver(p.D, p.mu, tol=TOL, **opts) as t:
            y = torch.zeros_like(R2)
            t.solve(R2, y)
            assert s.stats()["steps"] == t.stats()["steps"]
        assert torch.equal(x, y)
