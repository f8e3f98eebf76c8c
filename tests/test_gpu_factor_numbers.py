"""The mixed path's factorisation by minors against the serial chains, number
by number: both run on the same operator in FP64.  What is kept of it is
rounded to FP32 (2^-24), so 1/w, the multipliers and the row constants must
agree to 2^-30, and the bordering vector to 2^-30 of its row's largest entry:
a change of a sixty-fourth of that rounding.  Widths: the shortest, around the
16 columns loaded ahead and the 256 threads of a row, rows that need more than
the default shared memory, and the longest; one latitude row; coefficients near
both ends of the FP32 range."""
import ctypes

import numpy as np
import pytest

from paper_2103_07210_gb300 import inputs
from tests.cuda_unit import compile_cuda

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "ftgcr_factor.cuh"
// l, w, u, z: [N], row: [nlat][4]; row32: null for the chains
extern "C" int factor(int nlon, int nlat, const double* Tx, const double* Ty, const double* muA, double* l, double* w,
                      double* u, double* z, double* row, float* row32) {
  const int rc = ftgcr::launch_line_factor(nlon, nlat, ftgcr::chunk_len(nlon), ftgcr::PC_LINE, Tx, Ty, muA, l, w, u, z, row,
                                           nullptr, nullptr, nullptr, row32, nullptr);
  return rc ? rc : (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def unit(tmp_path_factory):
    return compile_cuda(SOURCE, tmp_path_factory.mktemp("factor"))


def _operator(nlon, nlat, scale):
    """Faces of the finite-volume operator on the sphere and mu * cell area."""
    p = inputs.hill_problem(nlon, nlat, **inputs.random_hill(nlon))
    D = p.D * scale
    dlam, dth = 2 * np.pi / nlon, np.pi / nlat
    th = -np.pi / 2 + (np.arange(nlat) + 0.5) * dth
    Tx = 0.5 * (D + np.roll(D, -1, 1)) * (dth / (np.cos(th) * dlam))[:, None]
    Ty = np.zeros_like(D)
    Ty[:-1] = 0.5 * (D[:-1] + D[1:]) * (np.cos(th[:-1] + dth / 2) * dlam / dth)[:, None]
    muA = p.mu * scale * dlam * (np.sin(th + dth / 2) - np.sin(th - dth / 2))
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (Tx, Ty, muA)]


def _factor(unit, nlon, nlat, op, minors):
    out = [torch.zeros(nlat, nlon, dtype=torch.float64, device="cuda") for _ in range(4)]
    row = torch.zeros(nlat, 4, dtype=torch.float64, device="cuda")
    row32 = torch.zeros(nlat, 4, dtype=torch.float32, device="cuda")
    ptr = [ctypes.c_void_p(t.data_ptr()) for t in op + out + [row]]
    assert unit.factor(nlon, nlat, *ptr, ctypes.c_void_p(row32.data_ptr() if minors else None)) == 0
    return [t.cpu().numpy() for t in out[1:] + [row]], row32.cpu().numpy()


@pytest.mark.parametrize("scale", [1.0, 2.0 ** 110, 2.0 ** -110])
@pytest.mark.parametrize("nlon,nlat", [(8, 5), (16, 6), (17, 7), (18, 1), (33, 40), (255, 9), (257, 9), (513, 33), (1024, 512),
                                       (2560, 3), (2561, 3), (8000, 2), (12800, 2)])
def test_minors_agree_with_the_chains(unit, nlon, nlat, scale):
    op = _operator(nlon, nlat, scale)
    (w, u, z, row), row32 = _factor(unit, nlon, nlat, op, True)
    (wc, uc, zc, rowc), _ = _factor(unit, nlon, nlat, op, False)
    bound = 2.0 ** -30
    assert np.all(np.abs(w - wc) <= bound * np.abs(wc))
    assert np.all(np.abs(u - uc) <= bound * np.abs(uc))
    assert np.all(np.abs(z - zc) <= bound * np.abs(zc).max(1, keepdims=True))
    assert np.all(np.abs(row - rowc) <= bound * np.abs(rowc))
    assert np.array_equal(row32[:, :3], row[:, 1:].astype(np.float32)) and not row32[:, 3].any()
    assert not (w[:, -1].any() or u[:, -2:].any() or z[:, -1].any())  # past the leading block
