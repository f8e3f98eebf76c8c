"""The schedule of a launch of several banded solves (csrc/ftgcr_teams.h):
every solve is in one team's list, the teams' CTAs are as many as the launch
may have at most, and no CTA is left over while a team has fewer CTAs than a
solve of its list has bands (such a solve takes several bands a CTA and loses
its place on chip)."""
import ctypes
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2103_07210_gb300", "csrc")
SOURCE = """
#include "ftgcr_teams.h"
extern "C" int band_class(long long points, int nt, int sms) { return ftgcr::band_class(points, nt, sms); }
extern "C" int plan(int n, const long long* points, const int* nt, int sms, int most, int* cta, int* order) {
  ftgcr::TeamPlan p;
  ftgcr::plan_teams(std::vector<long long>(points, points + n), std::vector<int>(nt, nt + n), sms, most, &p);
  for (size_t i = 0; i < p.cta.size(); ++i) {
    const ftgcr::TeamCta& c = p.cta[i];
    const int v[5] = {c.team, c.rank, c.size, c.q0, c.q1};
    std::copy(v, v + 5, cta + 5 * i);
  }
  std::copy(p.order.begin(), p.order.end(), order);
  return (int)p.cta.size();
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("teams")
    (d / "t.cpp").write_text(SOURCE)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "t.so"), str(d / "t.cpp")])
    lib = ctypes.CDLL(str(d / "t.so"))

    def call(solves, sms, most):
        """[(CTAs, [solve, ...])] of the teams"""
        n = len(solves)
        points, nt = (ctypes.c_longlong * n)(*[s[0] for s in solves]), (ctypes.c_int * n)(*[s[1] for s in solves])
        cta, order = (ctypes.c_int * (5 * 1024))(), (ctypes.c_int * n)()
        grid = lib.plan(n, points, nt, sms, most, cta, order)
        rows = [tuple(cta[5 * i:5 * i + 5]) for i in range(grid)]
        teams = []
        for team, rank, size, q0, q1 in rows:
            if rank == 0:
                assert team == len(teams)
                teams.append((size, list(order[q0:q1])))
            assert teams[team] == (size, list(order[q0:q1])) and 0 <= rank < size
        assert sum(t[0] for t in teams) == grid
        return teams

    call.band_class = lambda points, nt, sms: lib.band_class(ctypes.c_longlong(points), nt, sms)

    return call


def _bands(nlat, sms=152):
    h = -(-nlat // sms)
    return -(-nlat // h)


def _check(solves, sms, most, teams):
    assert sorted(i for _, order in teams for i in order) == list(range(len(solves)))
    used = sum(size for size, _ in teams)
    assert len(teams) <= most and used <= sms and all(order for _, order in teams)
    short = [size for size, order in teams if size < max(solves[i][1] for i in order)]
    assert not short or used == sms, (short, used)


@pytest.mark.parametrize("sizes", [[(1024, 512), (700, 700)], [(700, 700), (1024, 512), (2048, 1024)],
                                   [(1024, 512)] * 3 + [(700, 700)] * 2, [(4000, 66), (512, 600)]])
def test_one_team_has_a_cta_for_each_band_of_every_solve(plan, sizes):
    solves = [(a * b, _bands(b)) for a, b in sizes]
    teams = plan(solves, 152, 1)
    _check(solves, 152, 1, teams)
    assert len(teams) == 1 and teams[0][0] == max(nt for _, nt in solves)


@pytest.mark.parametrize("seed", range(6))
def test_no_cta_is_left_over_while_a_solve_lacks_one(plan, seed):
    rng = random.Random(seed)
    for _ in range(100):
        solves = []
        for _ in range(rng.randint(1, 40)):
            nlon, nlat = round(2 ** rng.uniform(4, 12)), round(2 ** rng.uniform(0, 11))
            solves.append((nlon * nlat, _bands(nlat) if rng.random() < 0.7 else rng.randint(1, nlat)))
        sms, most = rng.choice([(152, 256), (152, 1), (20, 256), (4, 256)])
        _check(solves, sms, most, plan(solves, sms, most))


def test_a_solve_takes_all_ctas_only_with_bands_for_most_of_them(plan):
    """Large solves of few bands (asked for, or few rows) run side by side: one
    after another they would leave the other CTAs idle."""
    whole = [(1024 * 512, 128), (700 * 700, 140), (2048 * 1024, 147), (2048 * 1024, 1024)]
    side_by_side = [(1024 * 512, 32), (1024 * 512, 16), (4000 * 66, 66), (512 * 512, 38), (2048 * 1024, 64), (512 * 256, 128)]
    assert [plan.band_class(*s, 152) for s in whole] == [2] * len(whole)
    assert [plan.band_class(*s, 152) for s in side_by_side] == [1] * len(side_by_side)
