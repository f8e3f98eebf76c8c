"""Calls from two threads on handles of different widths, on a stream each: a
kernel's shared-memory limit is the process's, and what one thread needs must
not fall below it because the other needs less."""
import threading

import pytest

from paper_2103_07210_gb300 import ftgcr, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _in_two_threads(calls, repeat):
    errors, start = [], threading.Barrier(len(calls))

    def work(call):
        stream = torch.cuda.Stream()
        start.wait()
        try:
            for _ in range(repeat):
                call(stream)
        except Exception as e:  # noqa: BLE001 (reported below)
            errors.append(e)
        stream.synchronize()

    threads = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def test_rebuilds_of_two_widths_in_two_threads():
    # both rows need more than a kernel's default shared memory in the mixed factorisation
    solvers, calls = [], []
    for nlon in (2600, 8000):
        p = inputs.hill_problem(nlon, 2)
        solvers.append(ftgcr.Solver(p.D, p.mu, precision="mixed"))
        D = torch.from_numpy(p.D).cuda()
        calls.append(lambda stream, s=solvers[-1], D=D: s.set_coeffs(D, stream=stream))
    torch.cuda.synchronize()
    _in_two_threads(calls, 1500)
    for s in solvers:
        s.close()


def test_preconditioners_of_two_widths_in_two_threads():
    solvers, calls = [], []
    for nlon in (64, 4000):
        p = inputs.hill_problem(nlon, 4)
        solvers.append(ftgcr.Solver(p.D, p.mu))
        inp = torch.from_numpy(p.R).cuda()
        calls.append(lambda stream, s=solvers[-1], i=inp, o=torch.zeros_like(inp): s.apply_precond(i, o, stream=stream))
    torch.cuda.synchronize()
    _in_two_threads(calls, 3000)
    for s in solvers:
        s.close()
