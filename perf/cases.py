"""Workloads of the FT-GCR(k) library, each one call (or one short sequence of calls) a user's program
makes through the Python binding: single solves from a coarse grid to an HBM-resident one, in both
precisions, on regular and ragged grids, from a zero and from a warm initial guess; a solve of host
arrays; a coefficient update followed by a solve; a batch of uneven solves in one launch; a burst of
requests to the server.

Fields of a case:
  call       "solve" (device arrays, enqueued), "host" (blocking, pinned host arrays), "update" (new
             coefficients, solve, operator applied to the result), "batch", "serve"
  precision  "fp64" or "mixed"
  nlon, nlat, k, tol
  rhs        "flow" (divergence of the zonal flow over the hill), "random" (uniform noise) or "smooth"
             (the operator of a smooth field)
  warm       the initial guess is a nearby smooth field (the previous time step), else zero
  flip       one exponent-bit flip of the residual at that step, detected and recovered from (0: none)
  n, mix     number of solves of a batch or burst, and the seed of their sizes
"""
import math
import random

import numpy as np
import torch

from paper_2103_07210_gb300 import ftgcr

MU_HAT = 0.3  # mu = MU_HAT / dtheta^2, the repository's Helmholtz coefficient on every grid
BATCH_SIZES = ((128, 64), (256, 128), (512, 256), (1024, 512))
SERVE_SIZES = ((256, 128), (512, 256), (1024, 512), (2048, 1024))


def _case(name, call, precision, nlon, nlat, k=4, tol=1e-10, rhs="flow", warm=False, flip=0, n=1, mix=0):
    c = dict(call=call, precision=precision, nlon=nlon, nlat=nlat, k=k, tol=tol, rhs=rhs, warm=warm, flip=flip, n=n, mix=mix)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest grid in use: a coarse model or a unit of a fault study, one flip detected and redone
        _case("fp64_64x32_flip", "solve", "fp64", 64, 32, rhs="random", flip=5),
        # one solve of the fault studies (k = 4, plain FP64)
        _case("fp64_512x256", "solve", "fp64", 512, 256),
        # the quarter-degree grid in plain FP64: ragged, rows wider than one staged band allows
        _case("fp64_1440x721", "solve", "fp64", 1440, 721, rhs="random"),
        # the one-degree grid with both poles: odd number of rows, columns no multiple of 32
        _case("mixed_360x181", "solve", "mixed", 360, 181, rhs="random"),
        # the headline solve
        _case("mixed_1024x512", "solve", "mixed", 1024, 512),
        # a model's time step at the parity tolerance: longer cycles, the last step's field as first guess
        _case("mixed_1024x512_k8_warm", "solve", "mixed", 1024, 512, k=8, tol=1e-13, rhs="smooth", warm=True),
        # a single solve whose vectors outgrow the L2 cache
        _case("mixed_2048x1024", "solve", "mixed", 2048, 1024),
        # the largest single solve: vectors streamed from HBM
        _case("mixed_4096x2048", "solve", "mixed", 4096, 2048),
        # a program that keeps its fields on the host
        _case("host_mixed_1024x512", "host", "mixed", 1024, 512),
        # a time step with moving coefficients: rebuild the operator, solve, form the residual's operand
        _case("update_mixed_512x256", "update", "mixed", 512, 256, rhs="random"),
        # an ensemble: uneven independent solves in one launch
        _case("batch_mixed_128", "batch", "mixed", 0, 0, n=128, mix=42),
        # a burst of uneven requests with host right-hand sides
        _case("serve_mixed_32", "serve", "mixed", 0, 0, n=32, mix=7),
    ]


def draw(rng):
    call = rng.choices(("solve", "host", "update", "batch", "serve"), (12, 2, 2, 2, 2))[0]
    precision = "fp64" if rng.random() < 0.35 else "mixed"
    if call in ("batch", "serve"):
        most = 32 if call == "serve" or precision == "fp64" else 128
        n = round(math.exp(rng.uniform(math.log(6), math.log(most))))
        return _case("", call, precision, 0, 0, n=n, mix=rng.randrange(1, 1 << 20))
    widest = {"solve": 4096, "host": 2048, "update": 2048}[call]
    if precision == "fp64":
        widest = 2048
    nlon = round(math.exp(rng.uniform(math.log(64), math.log(widest))))
    if rng.random() < 0.5:
        nlon -= nlon % 8
    nlat = max(24, round(nlon * rng.uniform(0.4, 0.52)))
    rhs = rng.choice(("flow", "random", "smooth"))
    flip = rng.randrange(2, 7) if call == "solve" and precision == "fp64" and rng.random() < 0.3 else 0
    return _case("", call, precision, nlon, nlat, k=rng.choice((2, 4, 4, 4, 5, 8)), tol=rng.choice((1e-10, 1e-10, 1e-12)), rhs=rhs,
                 warm=rhs == "smooth" and rng.random() < 0.5, flip=flip)


# ---------------------------------------------------------------- the problem, in plain torch
def _sizes(case):
    if case["call"] not in ("batch", "serve"):
        return [(case["nlon"], case["nlat"])]
    rng = random.Random(case["mix"])
    return [rng.choice(BATCH_SIZES if case["call"] == "batch" else SERVE_SIZES) for _ in range(case["n"])]


def _mu(nlat):
    return MU_HAT * (nlat / math.pi) ** 2


def _angles(nlon, nlat):
    lam = (torch.arange(nlon, device="cuda", dtype=torch.float64) + 0.5) * (2 * math.pi / nlon)
    th = (torch.arange(nlat, device="cuda", dtype=torch.float64) + 0.5) * (math.pi / nlat) - math.pi / 2
    return lam, th


def _depth(rng, nlon, nlat):
    """D = 1 - a Gaussian hill with a random place, height and width."""
    lam, th = _angles(nlon, nlat)
    lc, tc = rng.uniform(0, 2 * math.pi), math.asin(rng.uniform(-1, 1))
    h0, w = rng.uniform(0.05, 0.2), math.radians(rng.uniform(10, 30))
    s = torch.sin(0.5 * (th - tc))[:, None] ** 2 + (torch.cos(th) * math.cos(tc))[:, None] * torch.sin(0.5 * (lam - lc))[None, :] ** 2
    return 1.0 - h0 * torch.exp(-((2.0 * torch.asin(torch.sqrt(s.clamp(0, 1)))) / w) ** 2)


def _smooth(rng, nlon, nlat):
    lam, th = _angles(nlon, nlat)
    u = torch.zeros(nlat, nlon, device="cuda", dtype=torch.float64)
    for m in range(4):
        z = rng.uniform(-1, 1) * torch.cos(th) ** m * torch.sin((m + 1) * th + rng.uniform(0, 6))
        u += z[:, None] * torch.cos(m * lam + rng.uniform(0, 6))[None, :]
    return u


class _Operator:
    """L of the problem: faces Tx, Ty and mu * cell areas."""

    def __init__(self, D):
        nlat, nlon = D.shape
        dlam, dth = 2 * math.pi / nlon, math.pi / nlat
        _, th = _angles(nlon, nlat)
        edge = torch.arange(1, nlat, device="cuda", dtype=torch.float64) * dth - math.pi / 2
        self.tx = 0.5 * (D + torch.roll(D, -1, 1)) * (dth / (torch.cos(th) * dlam))[:, None]
        self.ty = 0.5 * (D[:-1] + D[1:]) * (torch.cos(edge) * dlam / dth)[:, None]
        self.mua = (_mu(nlat) * dlam * (torch.sin(th + dth / 2) - torch.sin(th - dth / 2)))[:, None]

    def __call__(self, x):
        fx = self.tx * (torch.roll(x, -1, 1) - x)
        y = fx - torch.roll(fx, 1, 1) - self.mua * x
        if x.shape[0] > 1:
            fy = self.ty * (x[1:] - x[:-1])
            y[:-1] += fy
            y[1:] -= fy
        return y

    def solve(self, R):
        """x with L(x) = R: conjugate gradients on -L, preconditioned by the rows' mean operator
        (diagonal in longitude's Fourier modes), each sweep restarted from the true residual."""
        nlat, nlon = R.shape
        m = torch.arange(nlon // 2 + 1, device="cuda", dtype=torch.float64)
        c = self.mua.clone()
        c[:-1] += self.ty.mean(1, keepdim=True)
        c[1:] += self.ty.mean(1, keepdim=True)
        lam = c + self.tx.mean(1, keepdim=True) * (2 - 2 * torch.cos(2 * math.pi * m / nlon))[None, :]
        x, end = torch.zeros_like(R), 1e-15 * R.norm()
        for _ in range(3):
            r = self(x) - R  # the residual of (-L) x = -R
            if not bool(r.norm() > end):
                break
            d, p, rz = torch.zeros_like(R), None, None
            for i in range(400):
                z = torch.fft.irfft(torch.fft.rfft(r) / lam, n=nlon)
                new = (r * z).sum()
                p = z if p is None else z + (new / rz) * p
                rz = new
                q = -self(p)
                a = rz / (p * q).sum()
                d += a * p
                r = r - a * q
                if i % 8 == 7 and not bool(r.norm() > end):
                    break
            x = x + d
        return x


def _problem(case, seed, i, nlon, nlat):
    """(D, rhs, first guess or None) of solve i."""
    rng = random.Random("%d %d" % (seed, i))
    D = _depth(rng, nlon, nlat)
    x0 = None
    if case["rhs"] == "random":
        g = torch.Generator(device="cuda").manual_seed(rng.randrange(1 << 40))
        R = 2 * torch.rand(nlat, nlon, generator=g, device="cuda", dtype=torch.float64) - 1
    elif case["rhs"] == "smooth":
        u = _smooth(rng, nlon, nlat)
        R = _Operator(D)(u)
        if case["warm"]:
            x0 = u + 0.02 * _smooth(rng, nlon, nlat)
    else:
        lam, th = _angles(nlon, nlat)
        f = 0.5 * (D + torch.roll(D, -1, 1)) * (torch.cos(th) * (math.pi / nlat))[:, None]
        # the zonal wind's strength differs from one solve to the next
        R = rng.uniform(0.5, 2.0) * (f - torch.roll(f, 1, 1))
    return D, R.contiguous(), x0


# ---------------------------------------------------------------- the calls
def prepare(case, seed):
    sizes, call = _sizes(case), case["call"]
    opts = dict(k=case["k"], tol=case["tol"], precision=case["precision"], zero_guess=not case["warm"])
    out = torch.zeros(sum(a * b for a, b in sizes), dtype=torch.float64, device="cpu" if call in ("host", "serve") else "cuda",
                      pin_memory=call in ("host", "serve"))
    s, at = dict(case=case, opts=opts, D=[], R=[], x=[], out=out), 0
    for i, (nlon, nlat) in enumerate(sizes):
        D, R, x0 = _problem(case, seed, i, nlon, nlat)
        if call in ("host", "serve"):
            R = R.cpu().pin_memory()
            x0 = None if x0 is None else x0.cpu().pin_memory()
        s["D"].append(D)
        s["R"].append(R)
        s["x"].append(out[at:at + nlon * nlat].view(nlat, nlon))
        s["x0"] = x0
        at += nlon * nlat
    if call == "serve":
        s["server"] = ftgcr.Server(budget_bytes=24 << 30)
        return s
    s["solvers"] = []
    for (nlon, nlat), D in zip(sizes, s["D"]):
        first = torch.ones_like(D) if call == "update" else D  # an update starts from other coefficients
        s["solvers"].append(ftgcr.Solver(first, _mu(nlat), **opts))
    s["faults"] = ()
    if case["flip"]:
        rng = random.Random("flip %d" % seed)
        s["faults"] = ((case["flip"], "r", rng.randrange(case["nlon"] * case["nlat"]), 62),)
    if call == "update":
        s["lx"] = torch.zeros_like(s["x"][0])
    return s


def run(s):
    call = s["case"]["call"]
    if call == "serve":
        todo = [s["server"].submit(D, _mu(D.shape[0]), R, x, coeff_key=i + 1, **s["opts"])
                for i, (D, R, x) in enumerate(zip(s["D"], s["R"], s["x"]))]
        for t in todo:
            s["server"].wait(t)
        return s["out"]
    if call == "batch":
        ftgcr.solve_batch(s["solvers"], s["R"], s["x"])
        return s["out"]
    h, R, x = s["solvers"][0], s["R"][0], s["x"][0]
    if s["case"]["warm"]:
        x.copy_(s["x0"])
    if call == "host":
        h.solve(R, x)
        return x
    if call == "update":
        h.set_coeffs(s["D"][0])
        h.solve_async(R, x)
        h.apply_operator(x, s["lx"])
        return {"x": x, "lx": s["lx"]}
    h.solve_async(R, x, faults=s["faults"])
    return x


def work(case):
    """Bytes: the right-hand side, the faces in both directions and the solution (and the guess, the
    coefficients), each once.  Flops: the preconditioned step's, times the steps that the tolerance
    takes a solve in FP64 (1.3 a digit)."""
    N = sum(a * b for a, b in _sizes(case))
    arrays = 4 + (1 if case["warm"] else 0) + (3 if case["call"] == "update" else 0)
    steps = round(-1.3 * math.log10(case["tol"]))
    return {"bytes": 8.0 * arrays * N, "flops": float(steps * (32 + 3 * (case["k"] + 1)) * N)}


def exact(case, seed):
    xs, R = [], None
    for i, (nlon, nlat) in enumerate(_sizes(case)):
        D, R, _ = _problem(case, seed, i, nlon, nlat)
        xs.append(_Operator(D).solve(R))
    if case["call"] in ("batch", "serve"):
        return torch.cat([x.reshape(-1) for x in xs])
    return {"x": xs[0], "lx": R} if case["call"] == "update" else xs[0]
