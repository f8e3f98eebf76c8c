"""Banded rounds (a CTA of 512 threads per row band, neighbours' edge rows
sent as packets) at the edges of their layout: one row in all, one-row bands,
a ragged last band, widths around a piece of 8 or 16 elements and around a
warp of pieces, more directions than a band keeps on chip, every vector on
chip (mixed, narrow bands) and edge rows of e exchanged.  FP64: the oracle's
decisions, solution within 1e-10; mixed at tol 1e-10: a true residual below
it and a solution within 1e-7 of the oracle's at tol 1e-12 (the wide grids
among them keep any true residual near 1e-12).  In a batch, where a CTA takes several bands
one after another, every result is bitwise the one found alone."""
import numpy as np
import pytest

import oracle
from paper_2103_07210_gb300 import ftgcr, inputs
from tests.gpu_util import rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [  # nlon, nlat, k, tiles
    (16, 1, 2, 0), (8, 7, 1, 7), (31, 10, 4, 4), (33, 12, 3, 0), (255, 40, 8, 6), (257, 39, 4, 13),
    (264, 20, 16, 3), (513, 24, 4, 8), (1023, 30, 4, 6), (1025, 31, 5, 10),
]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_banded_rounds_match_oracle_alone_and_in_a_batch(precision):
    fp64 = precision == "fp64"
    problems, faults, solvers, alone = [], [], [], []
    for nlon, nlat, k, tiles in SIZES:
        p = inputs.hill_problem(nlon, nlat, rhs="random", seed=nlon + nlat)
        f = [(3, "r", nlon * nlat // 2, 62 if fp64 else 30)] if nlat > 8 else []
        o = oracle.ftgcr(p.D, p.R, p.mu, k, 1e-10 if fp64 else 1e-12, faults=f if fp64 else [])
        s = ftgcr.Solver(p.D, p.mu, k=k, tol=1e-10, precision=precision, tiles=tiles)
        R = torch.from_numpy(p.R).cuda()
        x = torch.zeros_like(R)
        s.solve(R, x, faults=f)
        info = s.stats()
        assert info["converged"] and info["split_rounds"] == 0 and (not tiles or info["tiles"] == tiles), info
        if fp64:
            assert info["steps"] == o["steps"] and info["detect_steps"] == o["detect_steps"], (nlon, nlat)
        else:
            assert info["res_final_true"] <= 1e-10 * info["norm_R"], (nlon, nlat)
        assert rel_err(x.cpu().numpy(), o["x"]) <= (1e-10 if fp64 else 1e-7), (nlon, nlat)
        problems.append(R), faults.append(f), solvers.append(s), alone.append((x.cpu().numpy(), info["steps"]))
    xs = [torch.zeros_like(R) for R in problems]
    ftgcr.solve_batch(solvers, problems, xs, faults=faults)
    torch.cuda.synchronize()
    for s, x, (xa, steps) in zip(solvers, xs, alone):
        assert np.array_equal(x.cpu().numpy(), xa) and s.stats()["steps"] == steps
    for s in solvers:
        s.close()
