"""Streamed rounds at two edges of their bands, against split rounds of the same
solve stopped after a few steps: the true residual then holds every row of
every round.  (The layouts differ by FP32 rounding, 1e-6 of the residual or so
after so few steps; a row left out or taken from the wrong round changes it in
the first digits: 1e-4.)

The last band of exactly two rows: its last row has no row north of it, and its
stencil would come straight after its axpy, whose r' the stencil's copies, issued
ahead, must not miss.  Flips of step 1: INIT of a band they fall into runs as
split rounds beside streamed ones, and the two exchange edge rows."""
import pytest

from paper_2103_07210_gb300 import ftgcr, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _residual(p, k, tiles, rounds, steps, faults=()):
    with ftgcr.Solver(p.D, p.mu, k=k, tol=1e-13, precision="mixed", tiles=tiles, rounds=rounds, max_steps=steps) as s:
        R = torch.from_numpy(p.R).cuda()
        x = torch.zeros_like(R)
        s.solve(R, x, faults=faults)
        st = s.stats()
    assert st["steps"] == steps and st["tiles"] == tiles and st["faults_detected"] == 0, st
    assert st["streamed_rounds"] == (rounds == "streamed")
    return st["res_final_true"] / st["norm_R"]


@pytest.mark.parametrize("steps", [1, 2, 3, 5])
@pytest.mark.parametrize("nlon,nlat,tiles", [(1024, 8, 4), (1024, 11, 5), (2048, 8, 4), (1024, 5, 2)])
def test_last_band_of_two_rows(nlon, nlat, tiles, steps):
    p = inputs.hill_problem(nlon, nlat, rhs="random", seed=nlat)
    a, b = (_residual(p, 4, tiles, r, steps) for r in ("streamed", "split"))
    assert abs(a - b) <= 1e-4 * b, (a, b)


@pytest.mark.parametrize("vec", ["x", "r", "p", "ap"])
@pytest.mark.parametrize("row", [0, 7, 8, 11, 15, 16, 31])  # bands of eight rows: both edges and inside
def test_first_step_flips_beside_streamed_bands(vec, row):
    nlon, nlat, tiles = 1024, 32, 4
    p = inputs.hill_problem(nlon, nlat, rhs="random", seed=6)
    fault = [(1, vec, row * nlon + 513, 2)]  # a low bit: the flip itself changes nothing in the fourth digit
    for steps in (1, 2):
        a, b = _residual(p, 4, tiles, "streamed", steps, fault), _residual(p, 4, tiles, "streamed", steps)
        assert abs(a - b) <= 1e-4 * b, (steps, a, b)
