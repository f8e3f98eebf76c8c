"""Banded solves whose CTAs hold several bands: teams smaller than the solves'
bands (a batch of more large solves than the GPU has places for), and a solve of
more bands than SMs.  Pass 1 (the rows) then runs over all of a CTA's bands
before pass 2 (operator and dots), several bands at a time where they are
small, and e comes back from memory; flips of the first step fall into pass 2 of
INIT.  Every result is bitwise the solve's alone.  Last, large solves whose most
bands belong to the smaller grid."""
import pytest

from paper_2103_07210_gb300 import ftgcr, inputs
from tests.gpu_util import rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KEYS = ("steps", "detect_steps", "faults_injected", "outer", "res_final_true", "converged")


def _alone_and_together(precision, specs):
    """specs: (nlon, nlat, k, faults, losses); (x alone, x in the batch, stats of both) of each."""
    solvers, Rs, alone = [], [], []
    for q, (nlon, nlat, k, faults, losses) in enumerate(specs):
        p = inputs.hill_problem(nlon, nlat, rhs="random", seed=40 + q)
        solvers.append(ftgcr.Solver(p.D, p.mu, k=k, tol=1e-10, precision=precision))
        Rs.append(torch.from_numpy(p.R).cuda())
        x = torch.zeros_like(Rs[-1])
        solvers[-1].solve(Rs[-1], x, faults=faults, losses=losses)
        alone.append((x, solvers[-1].stats()))
    xs = [torch.zeros_like(R) for R in Rs]
    ftgcr.solve_batch(solvers, Rs, xs, faults=[s[3] for s in specs], losses=[s[4] for s in specs])
    torch.cuda.synchronize()
    for (nlon, nlat, *_), s, x, (xa, info) in zip(specs, solvers, xs, alone):
        assert info["converged"] and torch.equal(x, xa), (nlon, nlat)
        st = s.stats()
        for key in KEYS:
            assert st[key] == info[key], (nlon, nlat, key)
        s.close()
    return alone


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_several_bands_a_cta_are_bitwise_one(precision):
    bit = 62 if precision == "fp64" else 30
    shapes = [(33, 61, 3), (255, 150, 4), (1023, 100, 4), (64, 152, 8), (20, 300, 2), (256, 128, 4)]
    specs = []
    for q in range(24):  # 19 teams of eight CTAs on 152 SMs
        nlon, nlat, k = shapes[q % len(shapes)]
        N = nlon * nlat
        faults, losses = (), ()
        if 6 <= q < 12:  # the first step's flips, at both edges of the grid and inside
            faults = [(1, ("x", "r", "p", "ap")[q % 4], (3, N // 2, N - 2)[q % 3], bit - 6 if q % 2 else 3)]
        elif 12 <= q < 18:
            faults = [(2 + q % 3, ("r", "e", "ap")[q % 3], N // 3 + q, bit)]
        elif q >= 22:
            losses = [(3, 1, 4, 40, 77 + q)]
        specs.append((nlon, nlat, k, faults, losses))
    _alone_and_together(precision, specs)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_more_bands_than_sms_alone(precision):
    """400 one-row bands against 100 of four rows: the same solution to the
    tolerance (other sums, other rounding), and the FP64 path's steps."""
    p = inputs.hill_problem(121, 400, rhs="random", seed=8)
    R, out = torch.from_numpy(p.R).cuda(), []
    for tiles in (400, 100):
        with ftgcr.Solver(p.D, p.mu, k=4, tol=1e-12, precision=precision, tiles=tiles) as s:
            x = torch.zeros_like(R)
            s.solve(R, x, faults=[(1, "r", 121 * 200, 5)])
            st = s.stats()
        assert st["converged"] and st["tiles"] == tiles
        out.append((x.cpu().numpy(), st["steps"]))
    assert rel_err(out[0][0], out[1][0]) <= 1e-9
    if precision == "fp64":
        assert out[0][1] == out[1][1]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_the_widest_team_need_not_be_the_largest_solves(precision):
    flip = [(4, "r", 1000, 62 if precision == "fp64" else 30)]
    _alone_and_together(precision, [(1024, 512, 4, (), ()), (700, 700, 4, flip, ()), (700, 700, 4, (), ()), (512, 512, 2, (), ())])
