"""The shortest launches a server may ask for: every solve then leaves the
device and resumes from its record after one, two or three rounds, with teams
of CTAs that have no band in the smaller solves, flips pending across
launches, and solves whose last transition falls on the first round of a
launch.  Every result is bitwise the same request's solved alone."""
import pytest

from paper_2103_07210_gb300 import ftgcr, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# nlon, nlat, precision, (vector, bit) of a flip of step 3
REQUESTS = [
    (2048, 1024, "mixed", None), (1024, 512, "mixed", None), (1024, 512, "mixed", ("r", 30)), (700, 700, "mixed", None),
    (64, 32, "mixed", None), (255, 150, "mixed", ("e", 27)), (128, 64, "mixed", None),
    (1024, 512, "fp64", None), (512, 256, "fp64", ("ap", 62)), (64, 32, "fp64", None), (33, 61, "fp64", ("x", 50)),
]


@pytest.mark.parametrize("epoch_rounds", [1, 2, 3])
def test_short_epochs_resume_bitwise(epoch_rounds):
    probs, faults = [], []
    for q, (nlon, nlat, precision, flip) in enumerate(REQUESTS):
        probs.append(inputs.hill_problem(nlon, nlat, **inputs.random_hill(700 + q)))
        faults.append([(3, flip[0], nlon * nlat // 2, flip[1])] if flip else ())
    Rs = [torch.from_numpy(p.R).cuda() for p in probs]
    xs = [torch.zeros_like(R) for R in Rs]
    with ftgcr.Server(max_slots=16, epoch_rounds=epoch_rounds) as srv:
        tickets = [srv.submit(torch.from_numpy(p.D).cuda(), p.mu, R, x, precision=prec, faults=f)
                   for p, R, x, (_, _, prec, _), f in zip(probs, Rs, xs, REQUESTS, faults)]
        results = [srv.wait(t, timeout=120) for t in tickets]
    for p, R, x, (nlon, nlat, prec, _), f, (status, served) in zip(probs, Rs, xs, REQUESTS, faults, results):
        with ftgcr.Solver(p.D, p.mu, precision=prec, tiles=served["tiles"]) as s:
            alone = torch.zeros_like(R)
            s.solve(R, alone, faults=f)
            info = s.stats()
        assert status == ftgcr.OK and served["converged"], (nlon, nlat, prec, served)
        assert torch.equal(x, alone), (nlon, nlat, prec)
        for key in ("steps", "detect_steps", "faults_injected", "outer", "res_final_true"):
            assert served[key] == info[key], (nlon, nlat, prec, key)
