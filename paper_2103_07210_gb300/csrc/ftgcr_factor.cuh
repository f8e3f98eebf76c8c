// The line preconditioner's factorisation: set-up kernels, run when a handle is
// created and whenever its coefficients change.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <map>
#include <mutex>

#include "../../include/ftgcr.h"
#include "ftgcr_device.cuh"

namespace ftgcr {

// Line-preconditioner factorisation, one thread per latitude row (setup
// only).  Row system M x = b, M_ii = d_i = Tx_i + Tx_{i-1} + sigma_i,
// M_{i,i+1} = -Tx_i (periodic).  Thomas factorisation of the leading
// (n-1) x (n-1) block, operation for operation the CPU oracle's:
// w_0 = d_0, l_i = -Tx_{i-1} / w_{i-1}, w_i = d_i - l_i (-Tx_{i-1}),
// winv_i = 1 / w_i, u_i = -Tx_i winv_i; bordering vector z = A0^-1 c,
// c = (-Tx_{n-1}, 0, ..., 0, -Tx_{n-2}) by the same substitution; delta =
// d_{n-1} + Tx_{n-1} z_0 + Tx_{n-2} z_{n-2}.
// FP64 outputs (natural layout): l, winv, u, z, delta.  FP32 outputs (chunk
// layout, element i -> [row][i % C][i / C]): c = -u, winv, z, and per row
// 1/delta, Tx_{n-1}/delta, Tx_{n-2}/delta.  Jacobi: d_i (FP64) or 1/d_i (FP32).
static __global__ void k_line_factor(int nlon, int nlat, int C, int precond, const double* __restrict__ Tx,
                              const double* __restrict__ Ty, const double* __restrict__ muA, double* l64,
                              double* w64, double* u64, double* z64, double* lrow64, float* lc32, float* lw32,
                              float* lz32, float* lrow32) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= nlat) return;
  const int n = nlon, m = n - 1;
  const long long rb = (long long)j * n;
  const double* tx = Tx + rb;
  auto diag = [&](int i) {
    const long long c = rb + i;
    double s = 0.0;
    if (j < nlat - 1) s = s + Ty[c];
    if (j > 0) s = s + Ty[c - n];
    s = s + muA[j];
    return tx[i] + tx[(i + n - 1) % n] + s;
  };
  if (precond == PC_JACOBI) {
    for (int i = 0; i < n; ++i) {
      const double d = diag(i);
      if (w64) w64[rb + i] = d;
      if (lw32) lw32[rb + i] = (float)(1.0 / d);
    }
    return;
  }
  if (precond != PC_LINE) return;
  double* l = l64 + rb;
  double* winv = w64 + rb;
  double* u = u64 + rb;
  double* z = z64 + rb;
  double w = diag(0);
  winv[0] = 1.0 / w;
  l[0] = 0.0;
  for (int i = 1; i < m; ++i) {
    l[i] = -tx[i - 1] / w;
    w = diag(i) - l[i] * -tx[i - 1];
    winv[i] = 1.0 / w;
  }
  for (int i = 0; i < m; ++i) u[i] = (i < m - 1) ? -tx[i] * winv[i] : 0.0;
  u[m] = 0.0;
  l[m] = 0.0;
  winv[m] = 0.0;
  // z = A0^-1 c
  for (int i = 0; i < m; ++i) z[i] = 0.0;
  z[0] = -tx[n - 1];
  z[m - 1] = z[m - 1] + -tx[n - 2];
  for (int i = 1; i < m; ++i) z[i] = fma(-l[i], z[i - 1], z[i]);
  z[m - 1] = z[m - 1] * winv[m - 1];
  for (int i = m - 2; i >= 0; --i) z[i] = fma(-u[i], z[i + 1], z[i] * winv[i]);
  z[m] = 0.0;
  const double delta = diag(n - 1) + tx[n - 1] * z[0] + tx[n - 2] * z[m - 1];
  lrow64[(long long)j * 4 + 0] = delta;
  lrow64[(long long)j * 4 + 1] = 0.0;
  lrow64[(long long)j * 4 + 2] = 0.0;
  lrow64[(long long)j * 4 + 3] = 0.0;
  if (lc32) {
    const long long cb = (long long)j * 32 * C;
    for (int i = 0; i < 32 * C; ++i) {
      const int lane = i / C, k = i % C;
      const long long pos = cb + (long long)k * 32 + lane;
      const bool in = i < m;
      lc32[pos] = in ? (float)(-u[i]) : 0.f;
      lw32[pos] = in ? (float)winv[i] : 0.f;
      lz32[pos] = in ? (float)z[i] : 0.f;
    }
    const double dinv = 1.0 / delta;
    lrow32[(long long)j * 4 + 0] = (float)dinv;
    lrow32[(long long)j * 4 + 1] = (float)(tx[n - 1] * dinv);
    lrow32[(long long)j * 4 + 2] = (float)(tx[n - 2] * dinv);
    lrow32[(long long)j * 4 + 3] = 0.f;
  }
}

// The same factorisation as k_line_factor, split into its three dependent
// chains and the elementwise work between them.  The chains run one lane per
// latitude row, 32 rows to a warp, because GB300's FP64 unit costs the same
// per warp instruction for 1 or 32 active lanes.  Each lane loads a block of
// inputs ahead while it steps through the current one.  The off-chain work
// runs one thread per element: the diagonal, the reciprocal pivots, u, the
// products of the backward substitution and the FP32 layout.  Every value is
// formed by the same operations in the same order as in k_line_factor and the
// CPU oracle, so the factors are bitwise the same.
constexpr int kLfBlock = 8;  // inputs loaded ahead per lane

// d_i of every element (the diagonal of the row systems).
static __global__ void k_lf_diag(int nlon, int nlat, const double* __restrict__ Tx, const double* __restrict__ Ty,
                          const double* __restrict__ muA, double* dg) {
  const long long N = (long long)nlon * nlat;
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < N; g += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(g / nlon), i = (int)(g - (long long)j * nlon);
    double s = 0.0;
    if (j < nlat - 1) s = s + Ty[g];
    if (j > 0) s = s + Ty[g - nlon];
    s = s + muA[j];
    dg[g] = Tx[g] + Tx[(long long)j * nlon + (i + nlon - 1) % nlon] + s;
  }
}

// Chain 1: w_0 = d_0, l_i = -Tx_{i-1} / w_{i-1}, w_i = d_i - l_i (-Tx_{i-1}),
// i < m; l and the pivots w (not yet inverted) stored.
static __global__ void k_lf_chain_lw(int nlon, int nlat, const double* __restrict__ Tx, const double* __restrict__ dg,
                              double* __restrict__ l, double* __restrict__ wout) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= nlat) return;
  const int m = nlon - 1;
  const long long rb = (long long)j * nlon;
  const double* tx = Tx + rb;
  const double* d = dg + rb;
  double w = d[0];
  wout[rb] = w;
  l[rb] = 0.0;
  double ta[kLfBlock], da[kLfBlock], tb[kLfBlock], db[kLfBlock];
  auto load = [&](int i0, double* t, double* dd) {
#pragma unroll
    for (int q = 0; q < kLfBlock; ++q)
      if (i0 + q < m) {
        t[q] = tx[i0 + q - 1];
        dd[q] = d[i0 + q];
      }
  };
  auto step = [&](int i0, const double* t, const double* dd) {
#pragma unroll
    for (int q = 0; q < kLfBlock; ++q)
      if (i0 + q < m) {
        const double li = -t[q] / w;
        w = dd[q] - li * -t[q];
        l[rb + i0 + q] = li;
        wout[rb + i0 + q] = w;
      }
  };
  load(1, ta, da);
  for (int i0 = 1; i0 < m; i0 += 2 * kLfBlock) {
    load(i0 + kLfBlock, tb, db);
    step(i0, ta, da);
    load(i0 + 2 * kLfBlock, ta, da);
    step(i0 + kLfBlock, tb, db);
  }
}

// winv_i = 1 / w_i, u_i = -Tx_i winv_i (u_{m-1} = 0), the padding l_m = winv_m
// = u_m = 0, and the bordering right-hand side c into z:
// c = (-Tx_{n-1}, 0, ..., 0, 0 + -Tx_{n-2}), z_m = 0.
static __global__ void k_lf_recip(int nlon, int nlat, const double* __restrict__ Tx, double* l, double* winv, double* u,
                           double* z) {
  const long long N = (long long)nlon * nlat;
  const int m = nlon - 1;
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < N; g += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(g / nlon), i = (int)(g - (long long)j * nlon);
    const long long rb = (long long)j * nlon;
    if (i < m) {
      const double wi = 1.0 / winv[g];
      winv[g] = wi;
      u[g] = (i < m - 1) ? -Tx[g] * wi : 0.0;
      double c = 0.0;
      if (i == 0) c = -Tx[rb + nlon - 1];
      if (i == m - 1) c = c + -Tx[rb + nlon - 2];
      z[g] = c;
    } else {
      winv[g] = 0.0;
      u[g] = 0.0;
      l[g] = 0.0;
      z[g] = 0.0;
    }
  }
}

// Chain 2: forward substitution of c, z_i = fma(-l_i, z_{i-1}, z_i), i < m.
static __global__ void k_lf_chain_fwd(int nlon, int nlat, const double* __restrict__ l, double* __restrict__ z) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= nlat) return;
  const int m = nlon - 1;
  const long long rb = (long long)j * nlon;
  double y = z[rb];
  double la[kLfBlock], ca[kLfBlock], lb[kLfBlock], cb[kLfBlock];
  auto load = [&](int i0, double* ll, double* cc) {
#pragma unroll
    for (int q = 0; q < kLfBlock; ++q)
      if (i0 + q < m) {
        ll[q] = l[rb + i0 + q];
        cc[q] = z[rb + i0 + q];
      }
  };
  auto step = [&](int i0, const double* ll, const double* cc) {
#pragma unroll
    for (int q = 0; q < kLfBlock; ++q)
      if (i0 + q < m) {
        y = fma(-ll[q], y, cc[q]);
        z[rb + i0 + q] = y;
      }
  };
  load(1, la, ca);
  for (int i0 = 1; i0 < m; i0 += 2 * kLfBlock) {
    load(i0 + kLfBlock, lb, cb);
    step(i0, la, ca);
    load(i0 + 2 * kLfBlock, la, ca);
    step(i0 + kLfBlock, lb, cb);
  }
}

// The backward step's products z_i winv_i, i < m (z_{m-1} winv_{m-1} is also
// the first value of the backward substitution).
static __global__ void k_lf_products(int nlon, int nlat, const double* __restrict__ winv, double* z) {
  const long long N = (long long)nlon * nlat;
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < N; g += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(g % nlon);
    if (i < nlon - 1) z[g] = z[g] * winv[g];
  }
}

// Chain 3: backward substitution z_i = fma(-u_i, z_{i+1}, z_i winv_i),
// i = m-2 .. 0, then delta = d_{n-1} + Tx_{n-1} z_0 + Tx_{n-2} z_{m-1} and the
// row constants (FP64: delta, then 1/delta, Tx_{n-1}/delta, Tx_{n-2}/delta;
// FP32: the last three).
static __global__ void k_lf_chain_bwd(int nlon, int nlat, const double* __restrict__ Tx, const double* __restrict__ Ty,
                               const double* __restrict__ muA, const double* __restrict__ u, double* __restrict__ z,
                               double* lrow64, float* lrow32) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= nlat) return;
  const int n = nlon, m = n - 1;
  const long long rb = (long long)j * n;
  double y = z[rb + m - 1];
  double ua[kLfBlock], pa[kLfBlock], ub[kLfBlock], pb[kLfBlock];
  auto load = [&](int i1, double* uu, double* pp) {  // elements i1, i1 - 1, ...
#pragma unroll
    for (int q = 0; q < kLfBlock; ++q)
      if (i1 - q >= 0) {
        uu[q] = u[rb + i1 - q];
        pp[q] = z[rb + i1 - q];
      }
  };
  auto step = [&](int i1, const double* uu, const double* pp) {
#pragma unroll
    for (int q = 0; q < kLfBlock; ++q)
      if (i1 - q >= 0) {
        y = fma(-uu[q], y, pp[q]);
        z[rb + i1 - q] = y;
      }
  };
  load(m - 2, ua, pa);
  for (int i1 = m - 2; i1 >= 0; i1 -= 2 * kLfBlock) {
    load(i1 - kLfBlock, ub, pb);
    step(i1, ua, pa);
    load(i1 - 2 * kLfBlock, ua, pa);
    step(i1 - kLfBlock, ub, pb);
  }
  const double* tx = Tx + rb;
  double s = 0.0;
  if (j < nlat - 1) s = s + Ty[rb + n - 1];
  if (j > 0) s = s + Ty[rb + n - 1 - n];
  s = s + muA[j];
  const double d_last = tx[n - 1] + tx[n - 2] + s;
  const double delta = d_last + tx[n - 1] * z[rb] + tx[n - 2] * z[rb + m - 1];
  const double dinv = 1.0 / delta;
  lrow64[(long long)j * 4 + 0] = delta;
  lrow64[(long long)j * 4 + 1] = dinv;
  lrow64[(long long)j * 4 + 2] = tx[n - 1] * dinv;
  lrow64[(long long)j * 4 + 3] = tx[n - 2] * dinv;
  if (lrow32) {
    lrow32[(long long)j * 4 + 0] = (float)dinv;
    lrow32[(long long)j * 4 + 1] = (float)(tx[n - 1] * dinv);
    lrow32[(long long)j * 4 + 2] = (float)(tx[n - 2] * dinv);
    lrow32[(long long)j * 4 + 3] = 0.f;
  }
}

// Constants in the per-lane chunk layout (FP32, or FP64 for the FP64 path's
// chunked row solve): position k*32 + lane of row j holds element
// i = lane*C + k (c = -u, winv, z; zero past the block).
template <typename O>
static __global__ void k_lf_chunks(int nlon, int nlat, int C, const double* __restrict__ u, const double* __restrict__ winv,
                            const double* __restrict__ z, O* lc32, O* lw32, O* lz32) {
  const long long per = 32LL * C, total = per * nlat;
  const int m = nlon - 1;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < total; q += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(q / per);
    const int pos = (int)(q - (long long)j * per), k = pos >> 5, lane = pos & 31;
    const int i = lane * C + k;
    const bool in = i < m;
    const long long g = (long long)j * nlon + i;
    lc32[q] = in ? (O)(-u[g]) : O(0);
    lw32[q] = in ? (O)winv[g] : O(0);
    lz32[q] = in ? (O)z[g] : O(0);
  }
}

// FP32 constants in the piece-major layout of the streamed rounds: position
// L (C + 4) + kk of row j holds element i = L C + kk (c = -u, winv, z; zero
// past the leading block and in the padding).
static __global__ void k_lf_pieces(int nlon, int nlat, int C, const double* __restrict__ u, const double* __restrict__ winv,
                            const double* __restrict__ z, float* lc, float* lw, float* lz) {
  const int P = C + 4;
  const long long per = 32LL * P, total = per * nlat;
  const int m = nlon - 1;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < total; q += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(q / per);
    const int pos = (int)(q - (long long)j * per), L = pos / P, kk = pos - L * P;
    const int i = L * C + kk;
    const bool in = kk < C && i < m;
    const long long g = (long long)j * nlon + i;
    lc[q] = in ? (float)(-u[g]) : 0.f;
    lw[q] = in ? (float)winv[g] : 0.f;
    lz[q] = in ? (float)z[g] : 0.f;
  }
}

// Constants in the layout of the banded rounds: row j, plane q, piece p holds
// the W elements p CQ + q W .. of c = -u, winv, z (zero past the leading block
// and in the padding), CQ = W 2^lq.
template <typename O>
static __global__ void k_lf_band(int nlon, int nlat, int lq, int PC, const double* __restrict__ u,
                          const double* __restrict__ winv, const double* __restrict__ z, O* lc, O* lw, O* lz) {
  constexpr int W = 16 / sizeof(O);
  const int Q = 1 << lq, per = Q * PC * W, m = nlon - 1;
  const long long total = (long long)per * nlat;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < total; q += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(q / per), pos = (int)(q - (long long)j * per);
    const int un = pos / W, plane = un / PC, p = un - plane * PC;
    const int i = (p << lq) * W + plane * W + (pos - un * W);
    const bool in = i < m;
    const long long g = (long long)j * nlon + i;
    lc[q] = in ? (O)(-u[g]) : O(0);
    lw[q] = in ? (O)winv[g] : O(0);
    lz[q] = in ? (O)z[g] : O(0);
  }
}

// The mixed path's factorisation, whose constants are kept in FP32: FP64
// throughout, without the division in the serial chain (some 13 dependent
// FP64 instructions of 64 cycles a column: 512 x 256 took 444 us in
// all with the rebuild's other kernels, now 224; 4096 x 2048 3.70 ms, now 2.00).  The pivots of the leading block are ratios of consecutive minors,
// w_i = p_i / p_{i-1} with p_i = d_i p_{i-1} - Tx_{i-1}^2 p_{i-2}: one dependent
// multiply-add a column, every fourth followed by a scaling by a power of two.
// The same from the other end gives w'_i, and the bordering solve A0 z = c
// needs no substitution: column m-1 of A0^-1 is g_i = (Tx_i / w_i) g_{i+1} from
// g_{m-1} = 1 / w_{m-1}, column 0 is h_i = (Tx_{i-1} / w'_i) h_{i-1} from h_0 =
// 1 / w'_0, both running products.  Against 80-bit arithmetic on the rows of
// 64 x 32 to 4096 x 2048 the relative errors are those of k_line_factor's order
// within a small factor (at most 5e-15 in 1/w, 1e-12 in z and delta): far below
// the FP32 rounding of what is stored.
constexpr int kLfMinBlock = 16;    // inputs loaded ahead per lane
constexpr int kLfRowThreads = 256;

// 2^(1023 - e) for a normal number of biased exponent e: its reciprocal scale.
__device__ __forceinline__ double lf_scale(double p) {
  const unsigned e = ((unsigned)__double2hiint(p) >> 20) & 0x7ffu;
  return e - 1u < 2045u ? __hiloint2double((int)((2046u - e) << 20), 0) : 1.0;
}
// The minors from the west (even blocks) and from the east (odd), one lane a
// row; p as formed, before the scaling that follows every fourth.
static __global__ void k_lf_minors(int nlon, int nlat, const double* __restrict__ Tx, const double* __restrict__ dg,
                            double* __restrict__ pf, double* __restrict__ pb) {
  const bool back = blockIdx.x & 1;
  const int j = (int)(blockIdx.x >> 1) * 32 + (int)threadIdx.x, m = nlon - 1, s = back ? -1 : 1;
  if (j >= nlat) return;
  const long long rb = (long long)j * nlon, o = rb + (back ? m - 1 : 0);
  const double *t = Tx + (back ? o : o - 1), *d = dg + o;  // column k: Tx at s k, d at s k
  double* out = (back ? pb : pf) + o;
  double p = d[0], q = 1.0;
  out[0] = p;
  double ta[kLfMinBlock], da[kLfMinBlock], tb[kLfMinBlock], db[kLfMinBlock];
  auto load = [&](int k0, double* tt, double* dd) {
#pragma unroll
    for (int w = 0; w < kLfMinBlock; ++w)
      if (k0 + w < m) {
        tt[w] = t[s * (k0 + w)];
        dd[w] = d[s * (k0 + w)];
      }
  };
  auto step = [&](int k0, const double* tt, const double* dd) {  // k0 = 1 modulo 4
#pragma unroll
    for (int w = 0; w < kLfMinBlock; ++w)
      if (k0 + w < m) {
        const double pn = fma(dd[w], p, -(tt[w] * tt[w]) * q);
        q = p;
        p = pn;
        out[s * (k0 + w)] = p;
        if ((w & 3) == 3) {
          const double e = lf_scale(p);
          p = p * e;
          q = q * e;
        }
      }
  };
  load(1, ta, da);
  for (int k0 = 1; k0 < m; k0 += 2 * kLfMinBlock) {
    load(k0 + kLfMinBlock, tb, db);
    step(k0, ta, da);
    load(k0 + 2 * kLfMinBlock, ta, da);
    step(k0 + kLfMinBlock, tb, db);
  }
}
// One block a row: 1/w, u = -Tx / w, z and the row constants from the minors
// (w, l: the minors on entry; z: the diagonal).  Shared memory: two rows.
static __global__ void __launch_bounds__(kLfRowThreads) k_lf_rows(int nlon, int nlat, const double* __restrict__ Tx, double* w,
                                                           const double* l, double* u, double* z, double* lrow64,
                                                           float* lrow32) {
  extern __shared__ double lf_sm[];
  __shared__ double wa[kLfRowThreads / 32], wb[kLfRowThreads / 32];
  const int n = nlon, m = n - 1, j = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const long long rb = (long long)j * n;
  const double *t = Tx + rb, *pf = w + rb, *pb = l + rb;
  double *A = lf_sm, *B = lf_sm + n, *zr = z + rb;
  for (int i = tid; i < m; i += kLfRowThreads) {
    double qf = 1.0, qb = 1.0;
    if (i > 0) {
      qf = pf[i - 1];
      if (i - 1 > 0 && ((i - 1) & 3) == 0) qf = qf * lf_scale(qf);
    }
    if (i < m - 1) {
      qb = pb[i + 1];
      const int k = m - 2 - i;
      if (k > 0 && (k & 3) == 0) qb = qb * lf_scale(qb);
    }
    const double wi = qf / pf[i], wbi = qb / pb[i];
    const double a = i < m - 1 ? t[i] * wi : 0.0;
    A[i] = i < m - 1 ? a : wi;
    B[i] = i > 0 ? t[i - 1] * wbi : wbi;
    u[rb + i] = -a;
    zr[i] = wi;
  }
  __syncthreads();
  // running products, west to east of B and east to west of A: a piece a
  // thread (an odd length: no bank conflicts)
  const int L = ((m + kLfRowThreads - 1) / kLfRowThreads) | 1, lo = min(tid * L, m), hi = min(lo + L, m);
  double pa = 1.0, pr = 1.0;
  for (int i = lo; i < hi; ++i) {
    pa = pa * A[i];
    pr = pr * B[i];
  }
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double ya = __shfl_down_sync(0xffffffffu, pa, o), yb = __shfl_up_sync(0xffffffffu, pr, o);
    if (lane + o < 32) pa = pa * ya;
    if (lane >= o) pr = pr * yb;
  }
  if (lane == 0) wa[wp] = pa;
  if (lane == 31) wb[wp] = pr;
  double ga = __shfl_down_sync(0xffffffffu, pa, 1), hb = __shfl_up_sync(0xffffffffu, pr, 1);
  if (lane == 31) ga = 1.0;
  if (lane == 0) hb = 1.0;
  __syncthreads();
  for (int v = kLfRowThreads / 32 - 1; v > wp; --v) ga = ga * wa[v];
  for (int v = 0; v < wp; ++v) hb = hb * wb[v];
  for (int i = hi - 1; i >= lo; --i) A[i] = ga = ga * A[i];
  for (int i = lo; i < hi; ++i) B[i] = hb = hb * B[i];
  __syncthreads();
  const double tl = t[n - 1], tp = t[n - 2], dl = zr[m];
  auto zv = [&](int i) { return fma(-tl, B[i], -tp * A[i]); };
  for (int i = tid; i < m; i += kLfRowThreads) {
    w[rb + i] = zr[i];
    zr[i] = zv(i);
  }
  __syncthreads();  // zr[m] is read
  if (tid == 0) {
    w[rb + m] = 0.0;
    u[rb + m] = 0.0;
    zr[m] = 0.0;
    const double delta = dl + tl * zv(0) + tp * zv(m - 1), dinv = 1.0 / delta;
    const double row[4] = {delta, dinv, tl * dinv, tp * dinv};
    for (int q = 0; q < 4; ++q) lrow64[(long long)j * 4 + q] = row[q];
    for (int q = 0; q < 3; ++q) lrow32[(long long)j * 4 + q] = (float)row[q + 1];
    lrow32[(long long)j * 4 + 3] = 0.f;
  }
}

// The dynamic shared memory attribute of a kernel is process-wide: only ever
// raise it, so that a launch of another thread never finds it below what that
// thread has asked for.
static cudaError_t raise_dynamic_smem(const void* f, size_t bytes) {
  static std::mutex mu;
  static std::map<const void*, size_t> set;
  std::lock_guard<std::mutex> lk(mu);
  size_t& at = set[f];
  if (at >= bytes) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) at = bytes;
  return e;
}

// The line preconditioner's factorisation (Jacobi: its diagonal), enqueued
// on st.  FP64 outputs l, winv, u, z (z doubles as scratch for the diagonal)
// and the row constants; FP32 chunk-layout constants when lc32 is given.
static int launch_line_factor(int nlon, int nlat, int C, int precond, const double* Tx, const double* Ty,
                       const double* muA, double* l64, double* w64, double* u64, double* z64, double* r64,
                       float* lc32, float* lw32, float* lz32, float* lrow32, cudaStream_t st, double* lcc = nullptr,
                       double* lwc = nullptr, double* lzc = nullptr, float* lcp = nullptr, float* lwp = nullptr,
                       float* lzp = nullptr) {
  if (precond != PC_LINE) {
    k_line_factor<<<(nlat + 63) / 64, 64, 0, st>>>(nlon, nlat, C, precond, Tx, Ty, muA, l64, w64, u64, z64, r64, lc32,
                                                   lw32, lz32, lrow32);
    return cudaGetLastError() == cudaSuccess ? FTGCR_OK : FTGCR_ERR_CUDA;
  }
  const long long N = (long long)nlon * nlat;
  const int eb = 256, eg = (int)std::min<long long>((N + eb - 1) / eb, 8192);
  const int rg = (nlat + 31) / 32;  // one lane per row, one warp per block
  k_lf_diag<<<eg, eb, 0, st>>>(nlon, nlat, Tx, Ty, muA, z64);
  // FP32 constants: no serial divisions (rows that its two shared-memory rows
  // do not hold, and the shortest, keep the chains)
  const size_t rows2 = 2 * sizeof(double) * (size_t)nlon;
  if (lrow32 && nlon >= 8 && rows2 <= 200 * 1024) {
    if (rows2 > 40 * 1024 && raise_dynamic_smem((const void*)k_lf_rows, rows2) != cudaSuccess) {
      cudaGetLastError();
      return FTGCR_ERR_CUDA;
    }
    k_lf_minors<<<2 * rg, 32, 0, st>>>(nlon, nlat, Tx, z64, w64, l64);
    k_lf_rows<<<nlat, kLfRowThreads, rows2, st>>>(nlon, nlat, Tx, w64, l64, u64, z64, r64, lrow32);
  } else {
    k_lf_chain_lw<<<rg, 32, 0, st>>>(nlon, nlat, Tx, z64, l64, w64);
    k_lf_recip<<<eg, eb, 0, st>>>(nlon, nlat, Tx, l64, w64, u64, z64);
    k_lf_chain_fwd<<<rg, 32, 0, st>>>(nlon, nlat, l64, z64);
    k_lf_products<<<eg, eb, 0, st>>>(nlon, nlat, w64, z64);
    k_lf_chain_bwd<<<rg, 32, 0, st>>>(nlon, nlat, Tx, Ty, muA, u64, z64, r64, lrow32);
  }
  const long long nc = 32LL * C * nlat;
  const int cgrid = (int)std::min<long long>((nc + eb - 1) / eb, 8192);
  if (lc32) k_lf_chunks<float><<<cgrid, eb, 0, st>>>(nlon, nlat, C, u64, w64, z64, lc32, lw32, lz32);
  if (lcc) k_lf_chunks<double><<<cgrid, eb, 0, st>>>(nlon, nlat, C, u64, w64, z64, lcc, lwc, lzc);
  if (lcp) {
    const long long np = 32LL * (C + 4) * nlat;
    k_lf_pieces<<<(int)std::min<long long>((np + eb - 1) / eb, 8192), eb, 0, st>>>(nlon, nlat, C, u64, w64, z64, lcp,
                                                                                 lwp, lzp);
  }
  return cudaGetLastError() == cudaSuccess ? FTGCR_OK : FTGCR_ERR_CUDA;
}

}  // namespace ftgcr
