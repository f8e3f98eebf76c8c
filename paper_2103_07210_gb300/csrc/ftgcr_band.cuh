// Banded rounds: the line-preconditioned solves of both precisions on rows of
// up to kBandMaxLon columns (FTGCR_FLAG_ORACLE_ORDER, Jacobi, identity, split
// and streamed solves keep the kernels of ftgcr_phases.cuh).
//
// A solve belongs to a team of CTAs, each holding one band of latitude rows
// (or a few).  A step round forms r' on the band's own rows only, solves the
// rows, sends its edge rows to the two neighbouring bands, does the
// step's off-path work (the recurrences of p and phi) while
// the neighbours' rows arrive, then forms L(e) and the dots.  Nothing is
// recomputed for halo rows, and a band's vectors are private to its CTA: the
// operands of the critical path (r, L(e), the L(p^l)) stay in shared memory
// from one round to the next where they fit, so a round of a grid that the
// chip holds waits for no operand load.  Everything is also written through
// to global memory, so that any round can start from there.
//
// What a round costs on such grids is latency, not bytes: 512 threads (against
// 256 in the one-pass rounds) halve the trips of every loop, and a row's line
// solve spreads over up to 16 warps in pieces of 8 or 16 elements held in
// registers.  Measured on a GB300, one-pass rounds of 256 threads / banded, us a
// solve (k = 4, tol 1e-10, zero initial guess, random right-hand sides): FP64
// 64 x 32 1464 / 1088 (a detected flip), 1440 x 721 6297 / 4981; mixed 360 x 181
// 743 / 554, 1024 x 512 1172 / 1085, 2048 x 1024 4226 / 3386 (bound by L2).  The
// hill's flow takes fewer steps: FP64 512 x 256 1152 / 660, mixed 1024 x 512 742
// / 701; a batch of 128 such mixed solves 60.6 / 37.7 ms.  Tried and slower: 256 threads; larger bands on fewer CTAs (360 x
// 181 with 5 rows a band 671 against 545); the line solve's constants all
// loaded at its start, or the face coefficients one group ahead (registers
// spill); halo packets of several groups polled together; the step out of line.
//
// Every wait on a neighbour is bounded; one that runs out raises the launch's
// error flag and the CTA goes on to its next barrier, where every CTA of the
// team leaves.
#pragma once
#include "ftgcr_instances.h"
#include "ftgcr_phases.cuh"
#include "ftgcr_teams.h"

namespace ftgcr {

constexpr int kBandMaxBuf = kMaxK + 2;

template <typename T>
struct BandArgs {
  SolveDev<T>* const* solves;  // [n]
  int* active;                 // [n] 1 while a solve has rounds to run
  const TeamCta* cta;          // [gridDim.x], or null: one team, one solve
  const int* order;
  unsigned int* counter;       // [teams] barrier counters, zeroed before the launch
  LaunchCtl* ctl;
  int max_rounds;              // per solve
  TraceEnt* trace;
  int trace_rounds;
  int* diag;                   // [gridDim][4]
};

// ------------------------------------------------------------ groups of four columns
template <typename T>
struct G4 {
  T v[4];
};
// Columns [i, i + 4) of a row in global memory at p.  AL: rows are a multiple
// of four columns, so every group is 16-byte aligned and whole; otherwise nv
// columns are left in the row.
template <bool AL, bool NC = false, typename T>
__device__ __forceinline__ G4<T> ldg4(const T* p, int nv) {
  G4<T> r;
  if constexpr (AL) {
    constexpr int W = V16<T>::W;
#pragma unroll
    for (int h = 0; h < 4; h += W) {
      const V16<T> x = NC ? ldv_nc(p + h) : ldv(p + h);
#pragma unroll
      for (int w = 0; w < W; ++w) r.v[h + w] = x.v[w];
    }
  } else {
#pragma unroll
    for (int w = 0; w < 4; ++w) r.v[w] = w < nv ? (NC ? __ldg(p + w) : ldcg(p + w)) : T(0);
  }
  return r;
}
template <bool AL, typename T>
__device__ __forceinline__ void stg4(T* p, const G4<T>& x, int nv) {
  if constexpr (AL) {
    constexpr int W = V16<T>::W;
#pragma unroll
    for (int h = 0; h < 4; h += W) {
      V16<T> y;
#pragma unroll
      for (int w = 0; w < W; ++w) y.v[w] = x.v[h + w];
      stv(p + h, y);
    }
  } else {
#pragma unroll
    for (int w = 0; w < 4; ++w)
      if (w < nv) p[w] = x.v[w];
  }
}
// A 16-byte unit by a generic pointer (constants: shared or global memory).
template <typename T>
__device__ __forceinline__ V16<T> ld16(const T* p) {
  const uint4 u = *reinterpret_cast<const uint4*>(p);
  V16<T> r;
  memcpy(&r, &u, 16);
  return r;
}
// 16-byte units of shared memory.
template <typename T>
__device__ __forceinline__ V16<T> lds16(unsigned a) {
  unsigned x, y, z, w;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(x), "=r"(y), "=r"(z), "=r"(w) : "r"(a));
  const uint4 u = make_uint4(x, y, z, w);
  V16<T> r;
  memcpy(&r, &u, 16);
  return r;
}
template <typename T>
__device__ __forceinline__ void sts16(unsigned a, const V16<T>& v) {
  uint4 u;
  memcpy(&u, &v, 16);
  asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(u.x), "r"(u.y), "r"(u.z), "r"(u.w) : "memory");
}
// Group `idx` of a band's vector buffer (dense: 4 elements per group).  Only
// the thread that takes the group in every loop reads or writes it.
template <typename T>
__device__ __forceinline__ G4<T> lds4g(unsigned buf, int idx) {
  constexpr int W = V16<T>::W;
  G4<T> r;
#pragma unroll
  for (int h = 0; h < 4; h += W) {
    const V16<T> x = lds16<T>(buf + (unsigned)(idx * (4 * (int)sizeof(T)) + h * (int)sizeof(T)));
#pragma unroll
    for (int w = 0; w < W; ++w) r.v[h + w] = x.v[w];
  }
  return r;
}
template <typename T>
__device__ __forceinline__ void sts4g(unsigned buf, int idx, const G4<T>& x) {
  constexpr int W = V16<T>::W;
#pragma unroll
  for (int h = 0; h < 4; h += W) {
    V16<T> y;
#pragma unroll
    for (int w = 0; w < W; ++w) y.v[w] = x.v[h + w];
    sts16<T>(buf + (unsigned)(idx * (4 * (int)sizeof(T)) + h * (int)sizeof(T)), y);
  }
}

// ------------------------------------------------------------ rows
// A row in shared memory is split into pieces of Q 16-byte units (8 or 16
// elements), one per thread of its line solve; unit q of every piece lies in
// plane q, so the solve's threads (consecutive pieces) read consecutive units,
// and so, nearly, do the elementwise loops (consecutive units): plane pitches
// NP of 4 mod 8 units (Q = 2) or 2 mod 8 (Q = 4) keep both free of bank
// conflicts.
struct BandRow {
  int lq, NP;
  __device__ __forceinline__ unsigned unit(int u) const { return 16u * (unsigned)((u & ((1 << lq) - 1)) * NP + (u >> lq)); }
  template <typename T>
  __device__ __forceinline__ unsigned elem(int i) const {
    constexpr int W = V16<T>::W;
    return unit(i / W) + (unsigned)((i % W) * (int)sizeof(T));
  }
};
template <typename T>
__device__ __forceinline__ G4<T> lds_row4(const BandRow& g, unsigned row, int g4) {
  constexpr int W = V16<T>::W, U = 4 / W;
  G4<T> r;
#pragma unroll
  for (int h = 0; h < U; ++h) {
    const V16<T> x = lds16<T>(row + g.unit(g4 * U + h));
#pragma unroll
    for (int w = 0; w < W; ++w) r.v[h * W + w] = x.v[w];
  }
  return r;
}
template <typename T>
__device__ __forceinline__ void sts_row4(const BandRow& g, unsigned row, int g4, const G4<T>& x) {
  constexpr int W = V16<T>::W, U = 4 / W;
#pragma unroll
  for (int h = 0; h < U; ++h) {
    V16<T> y;
#pragma unroll
    for (int w = 0; w < W; ++w) y.v[w] = x.v[h * W + w];
    sts16<T>(row + g.unit(g4 * U + h), y);
  }
}

// ------------------------------------------------------------ line solve
// M e = -r of row j in place in shared memory (the factorisation and the
// bordering of line_solve_row), by the 32 G threads of a group, thread p on
// piece p: the piece's affine map, a warp scan of the maps and G totals
// through shared memory give each piece its exact carry-in, then the piece is
// replayed in registers, forward and backward.  c, w, z: the row's constants
// in planes of PC units (shared or global memory).  tot: 4 G + 2 values of
// shared memory per group; bar: the group's named barrier.
template <typename T, int CQ>
__device__ __noinline__ void band_line_solve(const SolveDev<T>& sd, int j, unsigned row, const T* c, const T* w,
                                             const T* z, T* tot, int bar, int p) {
  constexpr int W = V16<T>::W, Q = CQ / W;
  const int lane = threadIdx.x & 31, G = 1 << sd.lG, gw = p >> 5;
  const int n = sd.nlon, m = n - 1, PC = sd.PC;
  const BandRow g{sd.lq, sd.NP};
  const bool on = p < sd.NPc;
  const T* lr = sd.lrow + (long long)j * 4 + (sizeof(T) == 8 ? 1 : 0);
  const T lr0 = __ldg(lr + 0), lr1 = __ldg(lr + 1), lr2 = __ldg(lr + 2);
  T r[CQ], cv[CQ];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    V16<T> x, y;
#pragma unroll
    for (int u = 0; u < W; ++u) x.v[u] = y.v[u] = T(0);
    if (on) {
      x = lds16<T>(row + 16u * (unsigned)(q * g.NP + p));
      y = ld16(c + (q * PC + p) * W);
    }
#pragma unroll
    for (int u = 0; u < W; ++u) {
      // positions past the row hold no data (their factors are zero)
      r[q * W + u] = p * CQ + q * W + u < n ? x.v[u] : T(0);
      cv[q * W + u] = y.v[u];
    }
  }
  const T bl = -lds<T>(row + g.elem<T>(n - 1));
  // the forward multiplier of the piece's first element: c of the element before
  T a0 = __shfl_up_sync(0xffffffffu, cv[CQ - 1], 1);
  if (lane == 0) a0 = gw > 0 && on ? c[((Q - 1) * PC + p - 1) * W + W - 1] : T(0);
  auto sync = [&] {
    if (G > 1) group_sync(bar, 32 * G);
    else __syncwarp();
  };
  // forward: the piece's map g_out = F g_in + S
  T F = T(1), S = T(0);
  {
    T a = a0;
#pragma unroll
    for (int q = 0; q < CQ; ++q) {
      S = tfma(a, S, -r[q]);
      F = F * a;
      a = cv[q];
    }
  }
#pragma unroll 1
  for (int d = 1; d < 32; d <<= 1) {
    const T Fo = __shfl_up_sync(0xffffffffu, F, d), So = __shfl_up_sync(0xffffffffu, S, d);
    if (lane >= d) {
      S = tfma(F, So, S);
      F = F * Fo;
    }
  }
  T carry = T(0);
  if (G > 1) {
    if (lane == 31) {
      tot[gw] = F;
      tot[G + gw] = S;
    }
    sync();
#pragma unroll 1
    for (int q = 0; q < gw; ++q) carry = tfma(tot[q], carry, tot[G + q]);
  }
  {
    const T Fe = __shfl_up_sync(0xffffffffu, F, 1), Se = __shfl_up_sync(0xffffffffu, S, 1);
    if (lane > 0) carry = tfma(Fe, carry, Se);
  }
  T wv[CQ];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    V16<T> y;
#pragma unroll
    for (int u = 0; u < W; ++u) y.v[u] = T(0);
    if (on) y = ld16(w + (q * PC + p) * W);
#pragma unroll
    for (int u = 0; u < W; ++u) wv[q * W + u] = y.v[u];
  }
  {
    T a = a0, x = carry;
#pragma unroll
    for (int q = 0; q < CQ; ++q) {
      x = tfma(a, x, -r[q]);
      r[q] = x * wv[q];  // the backward step's product
      a = cv[q];
    }
  }
  // backward: the piece's map y_in = F y_out + S
  F = T(1), S = T(0);
#pragma unroll
  for (int q = CQ - 1; q >= 0; --q) {
    S = tfma(cv[q], S, r[q]);
    F = F * cv[q];
  }
#pragma unroll 1
  for (int d = 1; d < 32; d <<= 1) {
    const T Fo = __shfl_down_sync(0xffffffffu, F, d), So = __shfl_down_sync(0xffffffffu, S, d);
    if (lane + d < 32) {
      S = tfma(F, So, S);
      F = F * Fo;
    }
  }
  carry = T(0);
  if (G > 1) {
    if (lane == 0) {
      tot[2 * G + gw] = F;
      tot[3 * G + gw] = S;
    }
    sync();
#pragma unroll 1
    for (int q = G - 1; q > gw; --q) carry = tfma(tot[2 * G + q], carry, tot[3 * G + q]);
  }
  {
    const T Fe = __shfl_down_sync(0xffffffffu, F, 1), Se = __shfl_down_sync(0xffffffffu, S, 1);
    if (lane < 31) carry = tfma(Fe, carry, Se);
  }
#pragma unroll
  for (int q = CQ - 1; q >= 0; --q) {
    carry = tfma(cv[q], carry, r[q]);
    r[q] = carry;
  }
  // bordering: x_{n-1} = (b_{n-1} + Tx_{n-1} y_0 + Tx_{n-2} y_{m-1}) / delta
  if (p == 0) tot[4 * G] = r[0];
#pragma unroll
  for (int q = 0; q < CQ; ++q)
    if (p * CQ + q == m - 1) tot[4 * G + 1] = r[q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    V16<T> y;
#pragma unroll
    for (int u = 0; u < W; ++u) y.v[u] = T(0);
    if (on) y = ld16(z + (q * PC + p) * W);
#pragma unroll
    for (int u = 0; u < W; ++u) wv[q * W + u] = y.v[u];
  }
  sync();
  const T xl = tfma(lr2, tot[4 * G + 1], tfma(lr1, tot[4 * G], bl * lr0));
  if (on) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      V16<T> o;
#pragma unroll
      for (int u = 0; u < W; ++u) {
        const int i = p * CQ + q * W + u;
        o.v[u] = i == n - 1 ? xl : tfma(-xl, wv[q * W + u], r[q * W + u]);
      }
      sts16<T>(row + 16u * (unsigned)(q * g.NP + p), o);
    }
  }
  sync();  // the totals are read before the group's next row rewrites them
}

// ------------------------------------------------------------ vector buffers
// Where a step's operands are: shared-memory buffer number, or -1 (global
// memory).
struct BandPlan {
  int le, r, oR, oLp, oLe;  // inputs L(e) (PA: L(p^nu)) and r; outputs r', L(p') (PA: L(p^nu) kept), L(e)
  int lo[kMaxK];            // PF: L(p^l) of the recurrences
  int lp[kMaxK];            // L(p^l) of the dots
};
// One warp, after the context c is complete; tag: the global vector each
// buffer mirrors.  kind INIT, PA, PF; any other kind writes the vectors by
// other loops: every mirror is dropped.
template <typename T>
__device__ __noinline__ void band_plan(const SolveDev<T>& sd, const Ctx<T>& c, BandPlan& bp, const void** tag, int lane) {
  const int kind = c.kind;
  const bool step = kind == K_PA || kind == K_PF;
  const bool have = lane < sd.nbuf;
  const void* t = have && step ? tag[lane] : nullptr;
  auto find = [&](const void* q) { return __ffs(__ballot_sync(0xffffffffu, have && t == q && q)) - 1; };
  unsigned busy = 0u;
  int le = -1, r = -1, oR = -1, oLp = -1, oLe = -1;
  // output q in buffer b, or in a free one (stale mirrors of it dropped)
  auto out = [&](int b, const void* q) {
    if (t == q) t = nullptr;
    const unsigned fr = ~busy & ((1u << sd.nbuf) - 1u);
    if (b < 0) b = __ffs(fr) - 1;
    if (b >= 0) {
      busy |= 1u << b;
      if (lane == b) t = q;
    }
    return b;
  };
  if (step || kind == K_INIT) {
    const void* outLp = kind == K_PA ? (const void*)c.lpnu : (const void*)c.lpnew;
    if (step) {
      le = find(kind == K_PF ? (const void*)c.LeR : (const void*)c.lpnu);
      r = find(c.rC);
      if (kind == K_PF) {
#pragma unroll 1
        for (int l = 0; l <= c.nuo; ++l) {
          const int b = find(c.lo[l]);
          if (lane == 0) bp.lo[l] = b;
        }
      }
      // the dots' older directions stay where they are
#pragma unroll 1
      for (int l = 0; l <= c.nu; ++l)
        if ((const void*)c.lp[l] != outLp) {
          const int b = find(c.lp[l]);
          if (b >= 0) busy |= 1u << b;
        }
    }
    if (le >= 0) busy |= 1u << le;
    oR = out(r, c.rW);
    oLp = out(le, outLp);
    if (step) {
      oLe = out(-1, c.LeW);
#pragma unroll 1
      for (int l = 0; l <= c.nu; ++l) {
        const int b = find(c.lp[l]);
        if (lane == 0) bp.lp[l] = b;
      }
    }
  } else {
    t = nullptr;
  }
  if (have) tag[lane] = t;
  if (lane == 0) {
    bp.le = le;
    bp.r = r;
    bp.oR = oR;
    bp.oLp = oLp;
    bp.oLe = oLe;
  }
}

// ------------------------------------------------------------ neighbours
// A failed wait: the launch's error flag, and the top bit of the team's barrier
// counter, which every CTA of the team sees at its next barrier and leaves.
constexpr unsigned kTeamFailed = 0x80000000u;
struct TeamFail {
  unsigned int* counter;
  int* err;
  __device__ __forceinline__ void raise(int code) const {
    atomicExch(err, code);
    atomicOr(counter, kTeamFailed);
  }
};
// The edge rows of e travel as packets: each 32-bit word of a value beside a
// 32-bit tag of the round, written and read as one 8-byte word, two packets to
// a 16-byte access (the scheme of NCCL's LL protocol).  A reader polls the
// packets themselves, so an exchange costs one trip through L2 and no fence,
// where rows under a flag cost a release, the flag's trip and the rows' trip.
// A tag is ten bits of the solve's number and 22 of the round's (solve_id,
// round + 1): old packets are cleared before one repeats (k_begin_solve).
// Two sets, by the round's parity: a neighbour may read a round's packets as
// late as its own next round.
template <typename T>
__device__ __forceinline__ uint4* band_edges(const SolveDev<T>& sd, unsigned round, int tau) {  // first row, last row
  return sd.hrow + ((size_t)(round & 1u) * sd.nt + tau) * (size_t)(sd.NG * (int)sizeof(T));
}
__device__ __forceinline__ void put_packets(uint4* p, unsigned a, unsigned b, unsigned tag) {
  asm volatile("st.relaxed.gpu.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(a), "r"(tag), "r"(b), "r"(tag)
               : "memory");
}
__device__ __forceinline__ void put_group(uint4* p, const G4<float>& x, unsigned tag) {
  put_packets(p, __float_as_uint(x.v[0]), __float_as_uint(x.v[1]), tag);
  put_packets(p + 1, __float_as_uint(x.v[2]), __float_as_uint(x.v[3]), tag);
}
__device__ __forceinline__ void put_group(uint4* p, const G4<double>& x, unsigned tag) {
#pragma unroll
  for (int w = 0; w < 4; ++w) put_packets(p + w, (unsigned)__double2loint(x.v[w]), (unsigned)__double2hiint(x.v[w]), tag);
}
__device__ __forceinline__ uint4 ld_packets(const uint4* p) {
  uint4 u;
  asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(u.x), "=r"(u.y), "=r"(u.z), "=r"(u.w)
               : "l"(p)
               : "memory");
  return u;
}
// The group's packets (2 or 4 accesses), polled (bounded) until all carry tag.
template <typename T>
__device__ __forceinline__ G4<T> get_group(const uint4* p, unsigned tag, const TeamFail& tf) {
  constexpr int U = sizeof(T) / 2;
  uint4 u[U];
  unsigned long long t0 = 0ull;
#pragma unroll 1
  for (unsigned it = 1;; ++it) {
    bool all = true;
#pragma unroll
    for (int q = 0; q < U; ++q) u[q] = ld_packets(p + q);
#pragma unroll
    for (int q = 0; q < U; ++q) all = all && u[q].y == tag && u[q].w == tag;
    if (all) break;
    if ((it & 63u) == 0u) {
      const unsigned long long t = globaltimer();
      if (t0 == 0ull) t0 = t;
      if (t - t0 > kBarrierTimeoutNs) {
        tf.raise(4);
        break;
      }
      if (ld_relaxed_u32(tf.counter) & kTeamFailed) break;
    }
  }
  G4<T> r;
  if constexpr (sizeof(T) == 4) {
    r.v[0] = __uint_as_float(u[0].x), r.v[1] = __uint_as_float(u[0].z);
    r.v[2] = __uint_as_float(u[1].x), r.v[3] = __uint_as_float(u[1].z);
  } else {
#pragma unroll
    for (int w = 0; w < 4; ++w) r.v[w] = __hiloint2double((int)u[w].z, (int)u[w].x);
  }
  return r;
}
// Wait (bounded) until `target` CTAs of the team have arrived; false: give up.
static __device__ __noinline__ bool team_wait(unsigned target, const TeamFail& tf) {
  unsigned long long t0 = 0ull;
#pragma unroll 1
  for (unsigned it = 1;; ++it) {
    const unsigned v = ld_acquire_u32(tf.counter);
    if (v & kTeamFailed) return false;
    if (v >= target) return true;
    if ((it & 63u) == 0u) {
      const unsigned long long t = globaltimer();
      if (t0 == 0ull) t0 = t;
      if (t - t0 > kBarrierTimeoutNs) {
        tf.raise(1);
        return false;
      }
    }
  }
}

// The CTA's records, at the start of the dynamic shared memory, so that every
// function reaches them by constant shared addresses.
template <typename T>
struct BandSmem {
  SolveDev<T> sd;
  SolveState S;
  SolveState N;
  Ctx<T> c[2];      // this round's, and the next one's while it is formed
  BandPlan bp[2];
  PhaseSmem ps;
  const void* tag[kBandMaxBuf];
  double red[kNPart];
  double qd[32];
  T tot[kWarps * 6];
  TeamFail tf;
  int bail;
  int met;  // the team has met at a barrier since its CTAs loaded the solve's record
  int expected;
  int events;  // the plan holds flips or data-loss events of the round's step
  int cs_ok;  // the band's static data are staged
};
template <typename T>
__device__ __forceinline__ BandSmem<T>& band_smem() {
  extern __shared__ __align__(128) unsigned char dsm[];
  static_assert(sizeof(BandSmem<T>) <= (size_t)kBandFixed, "the records' room in shared memory");
  return *reinterpret_cast<BandSmem<T>*>(dsm);
}
// The rest of it: rows, sums, constants, buffers.
__device__ __forceinline__ unsigned char* band_rest() {
  extern __shared__ __align__(128) unsigned char dsm[];
  return dsm + kBandFixed;
}

// ------------------------------------------------------------ sums
// A step's sums: every thread leaves its accumulators in shared memory (value
// v at red + v * kRedPitch), and after a block barrier one warp per value adds
// them up and writes the band's partial sum, so that the work of a sum is done
// once instead of once per warp (with a warp sum in every warp it took 2 us of
// a round).  The last warp takes no part: it forms the next transition
// meanwhile.
constexpr unsigned kRedPitch = 8u * kThreads;
constexpr int kSumWarps = kWarps - 1;
__device__ __forceinline__ void red_leave(unsigned red, int v, const Acc<float>& a) {
  asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(red + (unsigned)v * kRedPitch + 8u * threadIdx.x), "f"(a.hi),
               "f"(a.lo)
               : "memory");
}
__device__ __forceinline__ void red_leave(unsigned red, int v, double x) {
  sts(red + (unsigned)v * kRedPitch + 8u * threadIdx.x, x);
}
__device__ __forceinline__ void red_leave(unsigned red, int v, const Acc<double>& a) { red_leave(red, v, a.p); }
// Values [v0, nv), of each of ntile bands side by side (band i: threads from
// its first row's first group on; a band's sum takes them in the same order
// wherever it lies).  Those with their bit in dbl are doubles whatever T.
template <typename T>
__device__ __noinline__ void band_sums(unsigned red, int v0, int nv, unsigned dbl, int tau, int ntile, double* out,
                                       int stride) {
  __syncthreads();
  const SolveDev<T>& sd = band_smem<T>().sd;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nval = nv - v0;
  if (w >= kSumWarps) return;
  int i = 0, v = v0 + w, at = 0;
#pragma unroll 1
  for (;; v += kSumWarps) {
#pragma unroll 1
    while (v >= nv && i < ntile) {  // the next band
      at += (sd.rb + (tau + i < sd.rx ? 1 : 0)) * sd.NG;
      v -= nval;
      ++i;
    }
    if (i >= ntile) break;
    const int na = min((sd.rb + (tau + i < sd.rx ? 1 : 0)) * sd.NG, kThreads);
    const unsigned a = red + (unsigned)v * kRedPitch + 8u * (unsigned)(at + lane);
    double* o = out + 2 * i + (long long)v * stride;
    if (sizeof(T) == 4 && !((dbl >> v) & 1u)) {
      float h = 0.f, l = 0.f;
#pragma unroll 2
      for (int q = lane; q < na; q += 32) {
        float h2, l2;
        asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(h2), "=f"(l2) : "r"(a + 8u * (unsigned)(q - lane)));
        const float t = h + h2, z = t - h, e = (h - (t - z)) + (h2 - z);
        h = t;
        l = (l + l2) + e;
      }
      __syncwarp();
      const double y = fx_float_sum(h, l);
      if (lane == 0) {
        o[0] = y;
        o[1] = 0.0;
      }
    } else {
      Fx x{0ull, 0ll, 1};
      int E = 1;
#pragma unroll 2
      for (int q = lane; q < na; q += 32) E = max(E, fx_exp(lds<double>(a + 8u * (unsigned)(q - lane))));
      __syncwarp();
      x.e = (int)__reduce_max_sync(0xffffffffu, (unsigned)E);
      if (x.e < 0x7ff) {
#pragma unroll 1
        for (int q = lane; q < na; q += 32) fx_add(x, lds<double>(a + 8u * (unsigned)(q - lane)), x.e);
        __syncwarp();
        x = fx_warp_sum(x);
      } else {
        x.e = kFxNaN;
      }
      const DD d = fx_dd(x);
      if (lane == 0) {
        o[0] = d.hi;
        o[1] = d.lo;
      }
    }
  }
}
// The bands' partial sums of value v added up (one warp; the pairs of a value
// lie side by side; FP32 vectors: the second of each is zero).
template <typename T>
__device__ __noinline__ double band_total(const double* part, int nt) {
  const int lane = threadIdx.x & 31;
  constexpr int B = 5;  // 160 bands in one batch
  Fx sum{0ull, 0ll, 1};
#pragma unroll 1
  for (int t0 = 0; t0 < nt; t0 += 32 * B) {
    double hi[B], lo[B];
    int E = 1;
#pragma unroll
    for (int q = 0; q < B; ++q) {
      hi[q] = lo[q] = 0.0;
      const int tau = t0 + lane + 32 * q;
      if (tau < nt) {
        if constexpr (sizeof(T) == 8) {
          const V16<double> x = ldv(part + 2 * (long long)tau);
          hi[q] = x.v[0], lo[q] = x.v[1];
        } else {
          hi[q] = ldcg(part + 2 * (long long)tau);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < B; ++q) {
      E = max(E, fx_exp(hi[q]));
      if constexpr (sizeof(T) == 8) E = max(E, fx_exp(lo[q]));
    }
    E = (int)__reduce_max_sync(0xffffffffu, (unsigned)E);
    Fx x{0ull, 0ll, E < 0x7ff ? E : kFxNaN};
    if (E < 0x7ff) {
      // shifting the batch down keeps the loop rolled (code size)
#pragma unroll 1
      for (int q = 0; q < B && t0 + 32 * q < nt; ++q) {
        fx_add(x, hi[0], E);
        if constexpr (sizeof(T) == 8) fx_add(x, lo[0], E);
#pragma unroll
        for (int u = 0; u + 1 < B; ++u) {
          hi[u] = hi[u + 1];
          if constexpr (sizeof(T) == 8) lo[u] = lo[u + 1];
        }
      }
      x = fx_warp_sum(x);
    }
    if (nt <= 32 * B) return fx_double(x);
    // room for the carries of up to 8192 batches (2^20 bands): 13 bits
    if (x.e < kFxNaN) {
      x.lo = (x.lo >> 13) | ((unsigned long long)x.hi << 51);
      x.hi >>= 13;
      x.e += 13;
    }
    const int e = max(x.e, sum.e);
    fx_down(x, e);
    fx_down(sum, e);
    sum.lo += x.lo;
    sum.hi += x.hi + (sum.lo < x.lo ? 1ll : 0ll);
  }
  return fx_double(sum);
}

// ------------------------------------------------------------ scalars
// a / b for the step's scalars: the reciprocal of b from the hardware's 20-bit
// estimate by one Newton-Raphson iteration, the quotient corrected by its
// residual (Markstein): five dependent operations (64 cycles each) where the
// division takes some 650.  Far from the range where every intermediate is
// normal the division itself.
__device__ __forceinline__ double quick_div(double a, double b) {
  const int ea = (__double2hiint(a) >> 20) & 0x7ff, eb = (__double2hiint(b) >> 20) & 0x7ff;
  double q;
  if ((a == 0.0 || (ea > 600 && ea < 1447)) && eb > 600 && eb < 1447) {
    double x;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(b));
    x = fma(x, fma(-b, x, 1.0), x);
    q = a * x;
    q = fma(fma(-b, q, a), x, q);
  } else {
    q = a / b;
  }
  return q;
}
// The quotients a transition may need (alpha_l, the next beta, <L(p'), L(p')>):
// precompute_divisions with quick_div.  One warp.
static __device__ __noinline__ void band_scalars(int pending, int nu, const double* lpn2, const double* red, double* qd) {
  const int lane = threadIdx.x & 31;
  const bool step = pending == K_PA || pending == K_PF;
  double num = 0.0, den = 1.0;
  if (step) {
    if (lane <= nu) num = -red[1 + lane], den = lpn2[lane];
  } else if (lane == kMaxK) {
    if (pending == K_INIT) num = -red[2], den = red[3];
    if (pending == K_PB || pending == K_RESTORE) num = -red[0], den = red[1];
  }
  double q = quick_div(num, den);
  if (step) {
    // see precompute_divisions
    double sum = lane <= nu ? q * num : 0.0;  // -alpha_l d_l
#pragma unroll 1
    for (int o = nu < 4 ? 2 : 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    sum = __shfl_sync(0xffffffffu, sum, 0);
    const double h = red[2 + nu], qq = red[3 + nu];
    const double d = qq - sum;
    const bool ok = d > 1e-3 * qq && isfinite(d) && isfinite(h);
    if (lane == kMaxK + 1) q = ok ? quick_div(-h, d) : 0.0;  // next beta
    if (lane == kMaxK + 2) q = ok ? d : -1.0;                // <L(p'), L(p')>, or -1: form p' (PB)
  }
  qd[lane] = q;
}

// ------------------------------------------------------------ planned flips (cold)
// The flips of vector `vec` among the nfl planned ones that hit columns of the
// group at g; keep: their clean values into patchval (the first step's flips).
template <typename T>
__device__ __noinline__ G4<T> flip4(G4<T> x, long long g, int vec, int nv, int nfl, const FlipEnt* fl, double* patchval) {
#pragma unroll 1
  for (int q = 0; q < nfl; ++q) {
    if (fl[q].vec != vec || fl[q].g < g || fl[q].g >= g + min(nv, 4)) continue;
    const int w = (int)(fl[q].g - g);
    bool first = patchval != nullptr;
    for (int u = 0; u < q; ++u) first = first && !(fl[u].vec == vec && fl[u].g == fl[q].g);
    T y = w == 0 ? x.v[0] : w == 1 ? x.v[1] : w == 2 ? x.v[2] : x.v[3];
    if (patchval) {
      // every flip of one element keeps the same clean value
      if (first)
        for (int u = q; u < nfl; ++u)
          if (fl[u].vec == vec && fl[u].g == fl[q].g) patchval[fl[u].q] = (double)y;
    }
    y = flip_bits(y, fl[q].bit);
    x.v[0] = w == 0 ? y : x.v[0];
    x.v[1] = w == 1 ? y : x.v[1];
    x.v[2] = w == 2 ? y : x.v[2];
    x.v[3] = w == 3 ? y : x.v[3];
  }
  return x;
}
// Whether the plan holds flips or data-loss events of step t (every lane of a
// warp, the same answer in all).
template <typename T>
__device__ __noinline__ bool band_events(const SolveDev<T>& sd, long long t) {
  const int lane = threadIdx.x & 31;
  bool hit = false;
  for (int q = lane; q < sd.nfaults; q += 32) hit = hit || sd.faults[q].step == t;
  for (int q = lane; q < sd.nlosses; q += 32) hit = hit || sd.losses[q].step == t;
  return __any_sync(0xffffffffu, hit);
}
// The e-site flips and data-loss events (Section 3) of step t on rows [j0, j1),
// the first at `rows`.
template <typename T>
__device__ __noinline__ void band_e_faults(const SolveDev<T>& sd, long long t, int j0, int j1, unsigned char* rows,
                                           int nfl, const FlipEnt* fl) {
  using U = typename std::conditional<sizeof(T) == 8, unsigned long long, unsigned int>::type;
  const BandRow g{sd.lq, sd.NP};
  const int n = sd.nlon;
  auto at = [&](long long f) {
    const int j = (int)(f / n), i = (int)(f - (long long)j * n);
    return reinterpret_cast<U*>(rows + (size_t)(j - j0) * sd.rowb + g.elem<T>(i));
  };
  if (threadIdx.x == 0) {
#pragma unroll 1
    for (int q = 0; q < nfl; ++q)
      if (fl[q].vec == V_E) {
        U* w = at(fl[q].g);
        *w ^= (U)1 << (unsigned)(fl[q].bit & (8 * (int)sizeof(T) - 1));
      }
  }
  __syncthreads();
  const long long b0 = (long long)j0 * n, b1 = (long long)j1 * n;
#pragma unroll 1
  for (int q = 0; q < sd.nlosses; ++q) {
    const LossEv ev = sd.losses[q];
    if (ev.step != t) continue;
    const long long l0 = (long long)ev.rank * sd.N / ev.nranks, l1 = (long long)(ev.rank + 1) * sd.N / ev.nranks;
    const long long len = l1 - l0;
    if (len <= 0 || l1 <= b0 || l0 >= b1) continue;
#pragma unroll 1
    for (long long i = 1 + threadIdx.x; i <= ev.count; i += kThreads) {
      const unsigned long long z = splitmix64_at(ev.seed, (unsigned long long)i);
      const long long f = l0 + (long long)(z % (unsigned long long)len);
      if (f >= b0 && f < b1) atomicXor(at(f), (U)1 << (unsigned)((z >> 32) % (8u * sizeof(T))));
    }
  }
  __syncthreads();
}
// r0 of a group (INIT) with the sums of R: L(x0) - R, or -R, or -R_in.
template <bool AL, typename T>
__device__ __noinline__ G4<T> init_r0(const SolveDev<T>& sd, int rin_R, int zero_guess, int j, int i, int nv, double* sumR) {
  const int n = sd.nlon;
  const long long gi = (long long)j * n + i;
  G4<T> rn;
  if (sizeof(T) == 4 && !rin_R) {
    rn = ldg4<AL>((const T*)sd.Rin + gi, nv);
#pragma unroll
    for (int w = 0; w < 4; ++w) rn.v[w] = -rn.v[w];
    return rn;
  }
  double Rv[4];
#pragma unroll
  for (int w = 0; w < 4; ++w) Rv[w] = w < nv ? ldcg(sd.R + gi + w) : 0.0;
#pragma unroll 1
  for (int w = 0; w < 4; ++w) {
    T v = T(0);
    if (w < nv) {
      const double R = w == 0 ? Rv[0] : w == 1 ? Rv[1] : w == 2 ? Rv[2] : Rv[3];
      if constexpr (sizeof(T) == 8) {
        T Lx = T(0);
        if (!zero_guess) Lx = stencil_global<double>(sd.x0, sd.Tx64, sd.Ty64, sd.muA64, n, sd.nlat, j, i + w, 0);
        v = Lx - R;
      } else {
        v = -(T)R;
      }
      if (sumR) *sumR = fma(R, R, *sumR);
    }
    rn.v[0] = w == 0 ? v : rn.v[0];
    rn.v[1] = w == 1 ? v : rn.v[1];
    rn.v[2] = w == 2 ? v : rn.v[2];
    rn.v[3] = w == 3 ? v : rn.v[3];
  }
  return rn;
}

// ------------------------------------------------------------ the step
// The band's static data into shared memory, once per solve: the line-solve
// constants of its rows (local: and of its halo rows) and (ts_staged) its face
// coefficients as dense groups, Tx of the own rows, Ty from the row below the
// band on.
template <typename T, bool AL>
__device__ __noinline__ void band_stage(int j0, int H) {
  const SolveDev<T>& sd = band_smem<T>().sd;
  unsigned char* rest = band_rest();
  if (sd.cs_staged) {
    const int co = sd.local, a0 = max(0, j0 - co), a1 = min(sd.nlat, j0 + H + co);
    const size_t arr = (size_t)(sd.nt_hmax + 2 * co) * sd.conb;
    unsigned char* cs = rest + sd.con_off + (size_t)(a0 - (j0 - co)) * sd.conb;
    const int u16 = (a1 - a0) * (sd.conb >> 4);
#pragma unroll 1
    for (int a = 0; a < 3; ++a) {
      const unsigned char* s =
          reinterpret_cast<const unsigned char*>(a == 0 ? sd.lcp : a == 1 ? sd.lwp : sd.lzp) + (size_t)a0 * sd.conb;
#pragma unroll 1
      for (int q = threadIdx.x; q < u16; q += kThreads) cp_async16(cs + a * arr + 16 * q, s + 16 * q);
    }
    cp_async_commit();
    cp_async_wait_all();
  }
  if (sd.ts_staged) {
    const int n = sd.nlon, NG = sd.NG;
    const unsigned tx = smem_addr(rest) + (unsigned)sd.ts_off, ty = tx + (unsigned)sd.faceb;
#pragma unroll 1
    for (int idx = threadIdx.x; idx < (H + 1) * NG; idx += kThreads) {
      const int jr = idx / NG, g4 = idx - jr * NG, nv = AL ? 4 : n - 4 * g4;
      const long long gi = (long long)(j0 + jr) * n + 4 * g4;
      if (jr < H) sts4g<T>(tx, idx, ldg4<AL, true>(sd.Tx + gi, nv));
      sts4g<T>(ty, idx, ldg4<AL, true>(sd.Ty + gi - (j0 + jr > 0 ? n : 0), nv));  // row j0 - 1 + jr (the first row's is masked)
    }
  }
}

// group idx: row jr of the band, group g4 of the row, element gi of a vector
#define FTGCR_GROUP(idx)                                      \
  const int jr = __float2int_rz(((float)(idx) + 0.5f) * rng); \
  const int g4 = (idx) - jr * NG, nv = AL ? 4 : n - 4 * g4;   \
  const long long gi = base + (jr * n + 4 * g4);

// The recurrences that no dot needs, p' = e + sum_l alpha_l p^l (PF) and phi' =
// phi + beta p', and the write-through of the step's vectors (rows of e; r',
// L(p') and, late, L(e) from their buffers), by threads t of nth.
template <typename T, int KB, bool kFused, bool AL, bool FLT>
__device__ __forceinline__ void band_window(int j0, int H, bool keep, int cur, int nfl, int t, int nth, bool late) {
  BandSmem<T>& ks = band_smem<T>();
  const SolveDev<T>& sd = ks.sd;
  const Ctx<T>& c = ks.c[cur];
  const BandPlan& bp = ks.bp[cur];
  const int n = sd.nlon, NG = sd.NG;
  const float rng = sd.rng;
  const BandRow g{sd.lq, sd.NP};
  const unsigned rowb = (unsigned)sd.rowb, sm0 = smem_addr(band_rest()), rows = sm0 + rowb;
  const unsigned buf0 = sm0 + (unsigned)sd.buf_off, bufb = (unsigned)sd.bufb;
  const int total = H * NG;
  const long long base = (long long)j0 * n;
  const T beta = c.beta;
  const int nuo = c.nuo, oR = keep ? bp.oR : -1, oLp = keep && kFused ? bp.oLp : -1, oLe = late ? bp.oLe : -1;
#pragma unroll 1
  for (int idx = t; idx < total; idx += nth) {
    FTGCR_GROUP(idx)
    G4<T> pn = ldg4<AL>((kFused ? c.eR : c.pnu) + gi, nv);
    G4<T> ph = ldg4<AL>(c.phiC + gi, nv);
    constexpr int LB = sizeof(T) == 8 ? 2 : 4;  // loads in flight together
    if constexpr (kFused) {
#pragma unroll
      for (int l0 = 0; l0 < KB; l0 += LB) {
        G4<T> pl[LB];
#pragma unroll
        for (int l = 0; l < LB; ++l)
          if (l0 + l <= nuo) pl[l] = ldg4<AL>(c.pp[l0 + l] + gi, nv);
        if (l0 == 0) {
          if (oR >= 0) stg4<AL>(c.rW + gi, lds4g<T>(buf0 + (unsigned)oR * bufb, idx), nv);
          if (oLp >= 0) stg4<AL>(c.lpnew + gi, lds4g<T>(buf0 + (unsigned)oLp * bufb, idx), nv);
          if (oLe >= 0) stg4<AL>(c.LeW + gi, lds4g<T>(buf0 + (unsigned)oLe * bufb, idx), nv);
          stg4<AL>(c.eW + gi, lds_row4<T>(g, rows + (unsigned)jr * rowb, g4), nv);
        }
#pragma unroll
        for (int l = 0; l < LB; ++l)
          if (l0 + l <= nuo) {
            const T a = c.alpha[l0 + l];
#pragma unroll
            for (int w = 0; w < 4; ++w) pn.v[w] = tfma(a, pl[l].v[w], pn.v[w]);
          }
      }
      if (FLT && nfl) {
        ph = flip4(ph, gi, V_X, nv, nfl, ks.ps.fl, (double*)nullptr);
        pn = flip4(pn, gi, V_P, nv, nfl, ks.ps.fl, (double*)nullptr);
      }
      stg4<AL>(c.pnew + gi, pn, nv);
    } else {
      if (oR >= 0) stg4<AL>(c.rW + gi, lds4g<T>(buf0 + (unsigned)oR * bufb, idx), nv);
      if (oLe >= 0) stg4<AL>(c.LeW + gi, lds4g<T>(buf0 + (unsigned)oLe * bufb, idx), nv);
      stg4<AL>(c.eW + gi, lds_row4<T>(g, rows + (unsigned)jr * rowb, g4), nv);
    }
#pragma unroll
    for (int w = 0; w < 4; ++w) ph.v[w] = tfma(beta, pn.v[w], ph.v[w]);
    stg4<AL>(c.phiW + gi, ph, nv);
  }
}
// After a local round's arrival, by threads t of nth: the halo rows of L(e)
// (INIT: L(p0)) from the neighbours' packets, into buffer b.
template <typename T>
__device__ __noinline__ void band_halo(int tau, int b, unsigned round, int t, int nth) {
  const BandSmem<T>& ks = band_smem<T>();
  const SolveDev<T>& sd = ks.sd;
  constexpr int U = sizeof(T) / 2;
  const int NG = sd.NG, H = sd.rb + (tau < sd.rx ? 1 : 0), j0 = tau * sd.rb + min(tau, sd.rx);
  const unsigned tag = (sd.solve_id << 22) + round + 1u;
  const unsigned buf = smem_addr(band_rest()) + (unsigned)(sd.buf_off + b * sd.bufb);
  const uint4* edges = band_edges(sd, round, tau);
#pragma unroll 1
  for (int q = t; q < 2 * NG; q += nth) {
    const bool up = q >= NG;
    if (up ? j0 + H < sd.nlat : j0 > 0)
      sts4g<T>(buf, H * NG + q, get_group<T>(up ? edges + (size_t)(NG + q) * U : edges + (size_t)q * U - (size_t)NG * U, tag, ks.tf));
  }
}
// ... and band_window.
template <typename T, int KB, bool AL, bool FLT>
__device__ __noinline__ void band_after(int kind, int tau, int cur, int t, int nth) {
  const BandSmem<T>& ks = band_smem<T>();
  const int nfl = FLT && ks.sd.nfaults ? ks.ps.nfl : 0;
  const int j0 = tau * ks.sd.rb + min(tau, ks.sd.rx), H = ks.sd.rb + (tau < ks.sd.rx ? 1 : 0);
  if (kind == K_PF)
    band_window<T, KB, true, AL, FLT>(j0, H, true, cur, nfl, t, nth, true);
  else
    band_window<T, KB, false, AL, FLT>(j0, H, true, cur, nfl, t, nth, true);
}

// A round of band tau.  Pass bits: 1 forms r' (INIT: r0) and solves the rows,
// 2 forms L(e) (INIT: L(p0)) and the dots.  A CTA with one band runs both at
// once with its vectors in the buffers; a CTA with several runs pass 1 over
// all of them, then pass 2, ntile bands at a time where they hold at most one
// group per thread together (their rows then make one taller band; only the
// sums stay apart).  The halo rows of e:
//   local (FP32, one band, all vectors in buffers): formed here as well.  The
//   buffers hold the halo rows of r and the L(p^l) too, so all that comes from
//   a neighbour is its edge rows of L(e), which travel while the sums, the
//   barrier and the scalars of the round run.  Nothing but these packets and
//   the sums leaves the CTA before it arrives at the barrier: p', phi' and the
//   write-through of the vectors follow while the barrier is waited for
//   (band_window).
//   else: the neighbours' edge rows of e, sent once the rows are solved; what
//   band_window does is done while they travel.
// Either way every value is formed by the same operations, so a solve's result
// does not depend on which is taken.
// FLT: the instance for the rounds of steps with planned faults (a call in a
// loop makes the compiler keep the loop's values in local memory, and with
// shared memory taking the L1 cache every such access costs an L2 trip).  Only
// those rounds take it: on every round of a solve with a fault plan it made a
// mixed 1024 x 512 solve 26 % slower.  (Which rounds these are is asked of the
// plan here, by one warp; counted in the state machine, it moved the compiler's
// allocation and cost solves without a plan 1 to 3 %.)
template <typename T, int KB, int KIND, bool AL, bool FLT>
__device__ __forceinline__ void band_step(int tau, int ntile, int pass, int cur, double* part_out) {
  BandSmem<T>& ks = band_smem<T>();
  const SolveDev<T>& sd = ks.sd;
  const Ctx<T>& c = ks.c[cur];
  const BandPlan& bp = ks.bp[cur];
  PhaseSmem& ps = ks.ps;
  constexpr bool kInit = KIND == K_INIT, kFused = KIND == K_PF;
  constexpr int U = sizeof(T) / 2;  // 16-byte packet pairs of a group
  const int n = sd.nlon, nlat = sd.nlat, NG = sd.NG;
  const int j0 = tau * sd.rb + min(tau, sd.rx), H = ntile * sd.rb + max(0, min(sd.rx - tau, ntile)), j1 = j0 + H;
  const bool keep = pass == 3;
  const bool local = sizeof(T) == 4 && keep && sd.local;
  const float rng = sd.rng;
  const BandRow g{sd.lq, sd.NP};
  const unsigned rowb = (unsigned)sd.rowb, sm0 = smem_addr(band_rest());
  const unsigned rows = sm0 + rowb;  // row j at rows + (j - j0) rowb; one halo row below
  const unsigned buf0 = sm0 + (unsigned)sd.buf_off, bufb = (unsigned)sd.bufb;
  auto buf = [&](int b) { return buf0 + (unsigned)b * bufb; };
  const unsigned red = sm0 + (unsigned)sd.red_off;
  const int total = H * NG;
  const long long base = (long long)j0 * n;
  const unsigned tag = (sd.solve_id << 22) + (unsigned)ks.S.round + 1u;
  uint4* const edges = band_edges(sd, (unsigned)ks.S.round, tau);  // first row, last row: of band tau
  const size_t lastband = (size_t)(ntile - 1) * 2 * NG * U;
  T* const eout = kInit ? sd.e[0] : c.eW;  // INIT: scratch for the unflipped p0
  Acc<T> an;
  an.mode(0);
  if (pass & 1) {
    double sumR = 0.0;
    int nfl = 0;
    if (FLT && sd.nfaults) {
      if (threadIdx.x == 0)
        ps.nfl = collect_flips(sd, c.t, kInit ? kStateVecs : (kFused ? (kStateVecs | (1u << V_E)) : (1u << V_E)),
                               (long long)(j0 - local) * n, (long long)(j1 + local) * n, ps.fl);
      __syncthreads();
      nfl = ps.nfl;
    }
    // (1) r' of the own rows, then (local) of the halo rows
    {
      const T beta = c.beta;
      const int nuo = c.nuo;
      const int bLe = keep ? bp.le : -1, bR = keep ? bp.r : -1, oR = keep ? bp.oR : -1, oLp = keep ? bp.oLp : -1;
      const int all = local ? total + 2 * NG : total;
#pragma unroll 1
      for (int idx = threadIdx.x; idx < all; idx += kThreads) {
        const bool own = idx < total;
        int jr, g4;
        if (own) {
          jr = __float2int_rz(((float)idx + 0.5f) * rng);
          g4 = idx - jr * NG;
        } else {
          const bool up = idx >= total + NG;
          jr = up ? H : -1;
          g4 = idx - total - (up ? NG : 0);
          if (up ? j1 >= nlat : j0 == 0) continue;
        }
        const int nv = AL ? 4 : n - 4 * g4;
        const long long gi = base + (jr * n + 4 * g4);
        const unsigned row = rows + (unsigned)(jr * (int)rowb);
        G4<T> rn;
        if constexpr (kInit) {
          rn = init_r0<AL>(sd, c.rin_R, c.zero_guess, j0 + jr, 4 * g4, nv, own ? &sumR : nullptr);
          sts_row4(g, row, g4, rn);
          if (own) {
#pragma unroll
            for (int w = 0; w < 4; ++w)
              if (w < nv) an.add(rn.v[w], rn.v[w]);
          }
          G4<T> xv;
#pragma unroll
          for (int w = 0; w < 4; ++w) {
            xv.v[w] = T(0);
            if constexpr (sizeof(T) == 8)
              if (!c.zero_guess && w < nv) xv.v[w] = ldcg(sd.x0 + gi + w);
          }
          if (FLT && nfl) {
            xv = flip4(xv, gi, V_X, nv, nfl, ps.fl, own ? sd.patchval : nullptr);
            rn = flip4(rn, gi, V_R, nv, nfl, ps.fl, own ? sd.patchval : nullptr);
          }
          if (own) stg4<AL>(c.phiW + gi, xv, nv);
        } else {
          G4<T> ln, rr;
          if (bLe >= 0) ln = lds4g<T>(buf(bLe), idx);
          else ln = ldg4<AL>((kFused ? c.LeR : c.lpnu) + gi, nv);
          if (bR >= 0) rr = lds4g<T>(buf(bR), idx);
          else rr = ldg4<AL>(c.rC + gi, nv);
          if constexpr (kFused) {
#pragma unroll
            for (int l = 0; l < KB; ++l)
              if (l <= nuo) {
                const int b = keep ? bp.lo[l] : -1;
                G4<T> ll;
                if (b >= 0) ll = lds4g<T>(buf(b), idx);
                else ll = ldg4<AL>(c.lo[l] + gi, nv);
                const T a = c.alpha[l];
#pragma unroll
                for (int w = 0; w < 4; ++w) ln.v[w] = tfma(a, ll.v[w], ln.v[w]);
              }
            if (FLT && nfl) {
              rr = flip4(rr, gi, V_R, nv, nfl, ps.fl, (double*)nullptr);
              ln = flip4(ln, gi, V_AP, nv, nfl, ps.fl, (double*)nullptr);
            }
            if (oLp < 0) stg4<AL>(c.lpnew + gi, ln, nv);
          }
          if (oLp >= 0) sts4g<T>(buf(oLp), idx, ln);
#pragma unroll
          for (int w = 0; w < 4; ++w) rn.v[w] = tfma(beta, ln.v[w], rr.v[w]);
          sts_row4(g, row, g4, rn);
        }
        if (oR >= 0) sts4g<T>(buf(oR), idx, rn);
        if (oR < 0 || (kInit && own)) stg4<AL>(c.rW + gi, rn, nv);
      }
    }
    if constexpr (kInit) {
      red_leave(red, 0, an);
      red_leave(red, 1, sumR);
    }
    // (2) e = P^-1 r'
    {
      if (keep && !ks.cs_ok) band_stage<T, AL>(j0, H);
      __syncthreads();
      sub_mark(ps, 0);
      if (keep && threadIdx.x == 0) ks.cs_ok = 1;
      const int lG = sd.lG, grp = (int)(threadIdx.x >> 5) >> lG, ngrp = kWarps >> lG;
      const int p = (int)threadIdx.x - (grp << (5 + lG));
      T* tot = ks.tot + grp * ((4 << lG) + 2);
      const int first = local && j0 > 0 ? -1 : 0, last = local && j1 < nlat ? H : H - 1;
#pragma unroll 1
      for (int jr = first + grp; jr <= last; jr += ngrp) {
        const unsigned char *pc, *pw, *pz;
        if (keep && sd.cs_staged) {
          const size_t arr = (size_t)(sd.nt_hmax + 2 * sd.local) * sd.conb;
          pc = band_rest() + sd.con_off + (jr + sd.local) * sd.conb;
          pw = pc + arr;
          pz = pw + arr;
        } else {
          const size_t o = (size_t)(j0 + jr) * sd.conb;
          pc = reinterpret_cast<const unsigned char*>(sd.lcp) + o;
          pw = reinterpret_cast<const unsigned char*>(sd.lwp) + o;
          pz = reinterpret_cast<const unsigned char*>(sd.lzp) + o;
        }
        const T *tc = reinterpret_cast<const T*>(pc), *tw = reinterpret_cast<const T*>(pw),
                *tz = reinterpret_cast<const T*>(pz);
        const unsigned row = rows + (unsigned)(jr * (int)rowb);
        if (sizeof(T) == 8 || sd.lq == 1) {
          band_line_solve<T, 8>(sd, j0 + jr, row, tc, tw, tz, tot, 1 + grp, p);
        } else {
          if constexpr (sizeof(T) == 4) band_line_solve<T, 16>(sd, j0 + jr, row, tc, tw, tz, tot, 1 + grp, p);
        }
      }
      __syncthreads();
      sub_mark(ps, 1);
    }
    if constexpr (!kInit)
      if (FLT && (nfl || sd.nlosses)) {
        const int lo = max(0, j0 - local), hi = min(nlat, j1 + local);
        band_e_faults(sd, c.t, lo, hi, band_rest() + (size_t)(1 + lo - j0) * sd.rowb, nfl, ps.fl);
      }
    if (!local) {
      // (3) the edge rows of e to the neighbours
#pragma unroll 1
      for (int q = threadIdx.x; q < 2 * NG; q += kThreads) {
        const int up = q >= NG ? 1 : 0, g4 = q - up * NG;
        if (up ? j1 < nlat : j0 > 0)
          put_group(edges + (up ? lastband : 0) + (size_t)q * U, lds_row4<T>(g, rows + (up ? (unsigned)(H - 1) * rowb : 0u), g4), tag);
      }
      // (4) while they travel: e written out, and the work of band_window
      if constexpr (kInit) {
#pragma unroll 1
        for (int idx = threadIdx.x; idx < total; idx += kThreads) {
          FTGCR_GROUP(idx)
          stg4<AL>(eout + gi, lds_row4<T>(g, rows + (unsigned)jr * rowb, g4), nv);
        }
      } else {
        band_window<T, KB, kFused, AL, FLT>(j0, H, keep, cur, nfl, threadIdx.x, kThreads, false);
      }
    }
    if (!(pass & 2)) {
      if constexpr (kInit) band_sums<T>(red, 0, 2, 2u, tau, ntile, part_out, ps.cr.stride);
      return;
    }
  }
  if (!local) {
    // (5) the halo rows (pass 2 alone: the own rows too): two halves of the
    // block, one per neighbour
    const int half = threadIdx.x >= kThreads / 2 ? 1 : 0;
    if (half ? j1 < nlat : j0 > 0) {
      // the north neighbour's first row, the south neighbour's last
      const uint4* src = half ? edges + lastband + (size_t)2 * NG * U : edges - (size_t)NG * U;
      const unsigned dst = half ? rows + (unsigned)H * rowb : rows - rowb;
#pragma unroll 1
      for (int g4 = (int)threadIdx.x - half * (kThreads / 2); g4 < NG; g4 += kThreads / 2)
        sts_row4(g, dst, g4, get_group<T>(src + (size_t)g4 * U, tag, ks.tf));
    }
    if (!(pass & 1)) {
      if (FLT && kInit && sd.nfaults && threadIdx.x == 0)
        ps.nfl = collect_flips(sd, c.t, kStateVecs, (long long)j0 * n, (long long)j1 * n, ps.fl);
#pragma unroll 1
      for (int idx = threadIdx.x; idx < total; idx += kThreads) {
        FTGCR_GROUP(idx)
        sts_row4(g, rows + (unsigned)jr * rowb, g4, ldg4<AL>((const T*)eout + gi, nv));
      }
    }
    __syncthreads();
  }
  // (6) L(e) of the own rows, the norm and the dots
  constexpr int ND = kInit ? 1 : KB;
  Acc<T> ad[ND], ah, aq;
  ah.mode(0), aq.mode(0);
#pragma unroll
  for (int l = 0; l < ND; ++l) ad[l].mode(0);
  const int bRn = keep ? bp.oR : -1, oLe = keep ? (kInit ? bp.oLp : bp.oLe) : -1, nu = c.nu;
  const bool ts = keep && sd.ts_staged;
  const unsigned sTx = sm0 + (unsigned)sd.ts_off, sTy = sTx + (unsigned)sd.faceb;
#pragma unroll 1
  for (int idx = threadIdx.x; idx < total; idx += kThreads) {
    FTGCR_GROUP(idx)
    const int j = j0 + jr, i = 4 * g4;
    const bool hasN = j < nlat - 1, hasS = j > 0;
    G4<T> tx, ty, tys, rn;
    T txw0;
    if (ts) {
      tx = lds4g<T>(sTx, idx);
      tys = lds4g<T>(sTy, idx);
      ty = lds4g<T>(sTy, idx + NG);
      txw0 = lds<T>(sTx + (unsigned)sizeof(T) * (unsigned)(g4 == 0 ? 4 * jr * NG + n - 1 : 4 * idx - 1));
    } else {
      // (the last row's Ty is zero; the first row's south face is masked)
      tx = ldg4<AL, true>(sd.Tx + gi, nv);
      ty = ldg4<AL, true>(sd.Ty + gi, nv);
      tys = ldg4<AL, true>(sd.Ty + gi - (hasS ? n : 0), nv);
      txw0 = __ldg(sd.Tx + gi + (i == 0 ? n - 1 : -1));
    }
    if (bRn >= 0) rn = lds4g<T>(buf(bRn), idx);
    else rn = ldg4<AL>((const T*)c.rW + gi, nv);
    const T muA = __ldg(sd.muA + j);
    const unsigned row = rows + (unsigned)jr * rowb;
    const G4<T> ec = lds_row4<T>(g, row, g4);
    G4<T> le;
    {
      const G4<T> en = lds_row4<T>(g, hasN ? row + rowb : row, g4), es = lds_row4<T>(g, hasS ? row - rowb : row, g4);
      const T ew = lds<T>(row + g.elem<T>(i == 0 ? n - 1 : i - 1));
      const T ee = lds<T>(row + g.elem<T>(i + 4 >= n ? 0 : i + 4));
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        T ve = ee;
        if (w < 3 && (AL || w + 1 < nv)) ve = ec.v[w < 3 ? w + 1 : 3];
        const T vw = w > 0 ? ec.v[w > 0 ? w - 1 : 0] : ew;
        le.v[w] = stencil_op<T>(0, ec.v[w], ve, vw, en.v[w], es.v[w], tx.v[w],
                                w == 0 ? txw0 : tx.v[w > 0 ? w - 1 : 0], ty.v[w], tys.v[w], muA, hasN, hasS);
        if (!AL && w >= nv) le.v[w] = T(0);
      }
    }
    if constexpr (kInit) {
      G4<T> pv = ec;
      if (FLT && sd.nfaults && ps.nfl) {
        pv = flip4(pv, gi, V_P, nv, ps.nfl, ps.fl, sd.patchval);
        le = flip4(le, gi, V_AP, nv, ps.nfl, ps.fl, sd.patchval);
      }
      stg4<AL>(c.pnew + gi, pv, nv);
      stg4<AL>(c.lpnew + gi, le, nv);
    }
    if (local) {
      if (jr == 0 && j0 > 0) put_group(edges + (size_t)g4 * U, le, tag);
      if (jr == H - 1 && j1 < nlat) put_group(edges + (size_t)(NG + g4) * U, le, tag);
    } else if constexpr (!kInit) {
      stg4<AL>(c.LeW + gi, le, nv);
    }
    if (oLe >= 0) sts4g<T>(buf(oLe), idx, le);
    if constexpr (!kInit) {
#pragma unroll
      for (int l = 0; l < ND; ++l)
        if (l <= nu) {
          const int b = keep ? bp.lp[l] : -1;
          G4<T> lp;
          if (b >= 0) lp = lds4g<T>(buf(b), idx);
          else lp = ldg4<AL>((const T*)c.lp[l] + gi, nv);
#pragma unroll
          for (int w = 0; w < 4; ++w) ad[l].add(le.v[w], AL || w < nv ? lp.v[w] : T(0));
        }
    }
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const T r = AL || w < nv ? rn.v[w] : T(0);
      if constexpr (!kInit) an.add(r, r);
      ah.add(r, le.v[w]);
      aq.add(le.v[w], le.v[w]);
    }
  }
  sub_mark(ps, 2);
  // (7) the band's partial sums
  const int vh = kInit ? 2 : 2 + nu;
  if constexpr (!kInit) {
    red_leave(red, 0, an);
#pragma unroll
    for (int l = 0; l < ND; ++l)
      if (l <= nu) red_leave(red, 1 + l, ad[l]);
  }
  red_leave(red, vh, ah);
  red_leave(red, vh + 1, aq);
  band_sums<T>(red, kInit && pass == 2 ? 2 : 0, vh + 2, kInit ? 2u : 0u, tau, ntile, part_out, ps.cr.stride);
}
// The rounds a solve takes but a few times, out of line; the PF round of a
// step without planned faults is inlined into the kernel, where it saves no
// registers at entry (a function of its size saves some 80, which go through
// L2).
template <typename T, int KB, int KIND, bool AL, bool FLT>
__device__ __noinline__ void band_step_out(int tau, int ntile, int pass, int cur, double* part_out) {
  band_step<T, KB, KIND, AL, FLT>(tau, ntile, pass, cur, part_out);
}
template <typename T, int KB>
__device__ __forceinline__ void band_step_any(int kind, int tau, int ntile, int pass, int cur, double* part_out) {
  const SolveDev<T>& sd = band_smem<T>().sd;
  const bool al = (sd.nlon & 3) == 0;
  if (band_smem<T>().events) {  // the unaligned form serves every row width
    if (kind == K_INIT)
      band_step_out<T, KB, K_INIT, false, true>(tau, ntile, pass, cur, part_out);
    else if (kind == K_PA)
      band_step_out<T, KB, K_PA, false, true>(tau, ntile, pass, cur, part_out);
    else
      band_step_out<T, KB, K_PF, false, true>(tau, ntile, pass, cur, part_out);
  } else if (kind == K_PF) {
    if (al)
      band_step<T, KB, K_PF, true, false>(tau, ntile, pass, cur, part_out);
    else
      band_step<T, KB, K_PF, false, false>(tau, ntile, pass, cur, part_out);
  } else if (kind == K_INIT) {
    if (al)
      band_step_out<T, KB, K_INIT, true, false>(tau, ntile, pass, cur, part_out);
    else
      band_step_out<T, KB, K_INIT, false, false>(tau, ntile, pass, cur, part_out);
  } else {
    if (al)
      band_step_out<T, KB, K_PA, true, false>(tau, ntile, pass, cur, part_out);
    else
      band_step_out<T, KB, K_PA, false, false>(tau, ntile, pass, cur, part_out);
  }
}

// The usual next transition (see can_expect) of a solve without planned
// faults, and with steps left, in few instructions: the outcome of
// transition(..., expect) on the same record.  One thread; N a copy of S.
template <typename T>
__device__ __noinline__ void usual_transition(const SolveDev<T>& sd, const SolveState& S, SolveState& N, Ctx<T>& c) {
  const int nu = S.nu;
  int phiC = S.phiC, rC = S.rC, phiS = S.phiS, rS = S.rS, slotS = S.slotS;
  int nun = nu, ns = 0;
  const bool step = S.pending == K_PA || S.pending == K_PF;
  if (step) {
    N.step = S.step + 1;
    N.stag = 0;
    if (nu == 0) {  // ^* <- ^0
      phiS = phiC;
      rS = rC;
      slotS = S.slot[0];
      N.phiS = phiS;
      N.rS = rS;
      N.slotS = slotS;
      N.nrm2_S = S.nrm2_prev;
      N.patched = 0;
    }
    phiC = S.phiW;
    rC = S.rW;
    N.phiC = phiC;
    N.rC = rC;
    unsigned used = 1u << slotS;
#pragma unroll 1
    for (int l = 0; l <= nu; ++l) used |= 1u << S.slot[l];
    ns = __ffs(~used) - 1;
    N.slot[nu + 1] = ns;
    nun = nu + 1;
    if (nun == sd.k) {
      N.slot[0] = ns;
      nun = 0;
      N.cycles = S.cycles + 1;
    }
    N.nu = nun;
    c.kind = K_PF;
    c.nuo = nu;
    c.pnew = sd.p[ns];
    c.lpnew = sd.Lp[ns];
    c.eR = sd.e[S.ecur];
    c.LeR = sd.Le[S.ecur];
  } else {
    ns = S.slot[nu];
    c.kind = K_PA;
  }
  auto other = [](int a, int b) { return a == b ? (a == 0 ? 1 : 0) : 3 - a - b; };
  const int phiW = other(phiC, phiS), rW = other(rC, rS), ec = S.ecur ^ 1;
  N.phiW = phiW;
  N.rW = rW;
  N.ecur = ec;
  N.pending = c.kind;
  c.nu = nun;
  c.t = S.step + (step ? 2 : 1);
  c.phiC = sd.phi[phiC];
  c.phiW = sd.phi[phiW];
  c.rC = sd.r[rC];
  c.rW = sd.r[rW];
  c.pnu = sd.p[ns];
  c.lpnu = sd.Lp[ns];
  c.eW = sd.e[ec];
  c.LeW = sd.Le[ec];
}

// ------------------------------------------------------------ the kernel
// Cooperative launch, one CTA per SM.  Each team runs its solves one after
// another, each for at most max_rounds rounds; a solve that is not done then
// resumes in a later launch from its record and its vectors.
template <typename T, int KB>
__global__ void __launch_bounds__(kThreads, 1) k_ftgcr_band(BandArgs<T> a) {
  BandSmem<T>& ks = band_smem<T>();
  TeamCta me;
  if (a.cta)
    me = a.cta[blockIdx.x];
  else
    me = TeamCta{0, (int)blockIdx.x, (int)gridDim.x, 0, 1};
  unsigned int* counter = a.counter + 32 * me.team;
  const unsigned long long t_start = globaltimer();
  const int warp = threadIdx.x >> 5;
  // after a round's arrival the lower warps wait for the barrier, fetch the
  // halo rows and add up the partial sums; the others do the late work
  constexpr int kTotWarps = kWarps / 2;
  unsigned int nbar = 0;
  int tr = 0;
  auto arrive = [&] {
    if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(counter), "r"(1u) : "memory");
  };
#pragma unroll 1
  for (int q = me.q0; q < me.q1; ++q) {
    const int s = a.order ? a.order[q] : q;
    if (threadIdx.x == 0) {
      ks.tf = TeamFail{counter, &a.ctl->err};
      ks.bail = 0;
      ks.cs_ok = 0;
    }
    cta_load_cg(&ks.sd, a.solves[s]);
    __syncthreads();
    cta_load_cg(&ks.S, ks.sd.st);
    if (threadIdx.x < kBandMaxBuf) ks.tag[threadIdx.x] = nullptr;
    __syncthreads();
    if (!ks.S.active) {
      __syncthreads();
      continue;
    }
    const int nt = ks.sd.nt;
    const int ta = (int)((long long)me.rank * nt / me.size), tb = (int)((long long)(me.rank + 1) * nt / me.size);
    const bool single = me.size >= nt;  // every CTA of the team holds one band
    const bool local = sizeof(T) == 4 && single && ks.sd.local;
    if (threadIdx.x == 0) ks.ps.cr.stride = 2 * nt;
    bool expected = false, done = false, late = false;
    long long round = ks.S.round;  // of ks.S, which the last warp rewrites while the others go on
    int pending = ks.S.pending, cur = 0, halo = -1;
    __syncthreads();
    // (ks.S: the record the last round left; expected: ks.N and c, bp [cur ^ 1]
    // hold the usual transition from it)
#pragma unroll 1
    for (int it = 0; it < a.max_rounds; ++it) {
      unsigned long long tr0 = 0ull, tr1 = 0ull;
      cur ^= 1;
      if (threadIdx.x == 0) {
        tr0 = globaltimer();
        if (tr0 - t_start > kKernelTimeoutNs) ks.tf.raise(2);
        ks.met = it;
        ks.ps.tracing = a.trace != nullptr;
      }
      const int par = (int)(round & 1);
      // the last round's partial sums, once every band has written its own
      // (the first round of a launch: written by an earlier launch)
      if (warp < kTotWarps && pending != K_NONE) {
        if (it > 0) {
          // one thread waits: more of them polling one word hold up the arrivals
          if (threadIdx.x == 0 && !team_wait(nbar * (unsigned)me.size, ks.tf)) ks.bail = 1;
          if (sizeof(T) == 4 && warp > 0 && halo >= 0)
            band_halo<T>(ta, halo, (unsigned)round - 1u, (int)threadIdx.x - 32, 32 * kTotWarps - 32);
          asm volatile("bar.sync 13, %0;" ::"n"(32 * kTotWarps) : "memory");
        }
        const bool ok = ks.bail == 0;
        const double* part = ks.sd.part + (long long)(par ^ 1) * nt * kPartStride;
        const int nv = part_values(ks.sd);
#pragma unroll 1
        for (int v = warp; ok && v < nv; v += kTotWarps) {
          const double x = band_total<T>(part + (long long)v * 2 * nt, nt);
          if ((threadIdx.x & 31) == 0) ks.red[v] = x;
        }
      }
      if (a.trace && threadIdx.x == 0) {
        tr1 = globaltimer();
        if (it > 0 && tr > 0 && tr <= a.trace_rounds) a.trace[(long long)(tr - 1) * gridDim.x + blockIdx.x].t3 = tr1;
        ks.ps.sub[0] = ks.ps.sub[1] = ks.ps.sub[2] = 0ull;
        tr0 = tr1;
      }
      __syncthreads();
      if (ks.bail) return;
      if (warp == 0) {
        band_scalars(pending, ks.S.nu, ks.S.lpn2, ks.red, ks.qd);
        __syncwarp();
        const bool holds = expected && expectation_holds(ks.sd, ks.S, ks.red, ks.qd, ks.N, ks.c[cur]);
        const bool events = (ks.sd.nfaults | ks.sd.nlosses) && band_events(ks.sd, ks.c[cur].t);
        if (threadIdx.x == 0) ks.expected = holds, ks.events = events;
      }
      __syncthreads();
      if (!ks.expected) {
        if (expected) {
          // the buffers' mirrors were planned for another step: drop them
          if (threadIdx.x < kBandMaxBuf) ks.tag[threadIdx.x] = nullptr;
          __syncthreads();
        }
        cta_store(&ks.N, &ks.S);
        cta_zero(&ks.c[cur]);
        __syncthreads();
        if (threadIdx.x == 0) {
          transition(ks.sd, ks.S, ks.red, ks.qd, ks.N, ks.c[cur]);
          ks.N.round = ks.S.round + 1;
        }
        __syncthreads();
        if (warp == 0) {
          fill_directions(ks.sd, ks.S, ks.N, ks.qd, ks.c[cur], threadIdx.x);
          __syncwarp();
          band_plan(ks.sd, ks.c[cur], ks.bp[cur], ks.tag, threadIdx.x);
          if (ks.sd.nfaults | ks.sd.nlosses) {
            const bool events = band_events(ks.sd, ks.c[cur].t);
            if (threadIdx.x == 0) ks.events = events;
          }
        }
        __syncthreads();
      }
      const int kind = ks.c[cur].kind;
      expected = can_expect(ks.N);
      pending = ks.N.pending;
      ++round;
      if (a.trace && threadIdx.x == 0) tr1 = globaltimer();
      if (threadIdx.x == 0 && a.diag) {
        a.diag[blockIdx.x * 4 + 0] = it;
        a.diag[blockIdx.x * 4 + 1] = kind;
      }
      if (kind == K_NONE) {
        done = true;
        break;
      }
      const bool step = kind == K_INIT || kind == K_PA || kind == K_PF;
      if (!step) {
        if (threadIdx.x == 0) ks.cs_ok = 0;  // shared memory reused
        if (late) {
          // the late work of the last step round is read by other CTAs now
          ++nbar;
          arrive();  // (behind the block barriers above)
          if (threadIdx.x == 0 && !team_wait(nbar * (unsigned)me.size, ks.tf)) ks.bail = 1;
          __syncthreads();
          if (ks.bail) return;
        }
      }
      late = local && (kind == K_PA || kind == K_PF);
      halo = !local || !step || ta == tb ? -1 : kind == K_INIT ? ks.bp[cur].oLp : ks.bp[cur].oLe;
      const int first = step && single ? 3 : 1, last = step && !single ? 2 : 1;
      const int mt = step && !single ? ks.sd.mega : 1;
#pragma unroll 1
      for (int pass = first; pass == first || pass <= last; ++pass) {
#pragma unroll 1
        for (int tau = ta; tau < tb; tau += mt) {
          double* part_out = ks.sd.part + (long long)par * nt * kPartStride + 2 * tau;
          if (step) {
            band_step_any<T, KB>(kind, tau, min(mt, tb - tau), pass, cur, part_out);
          } else {
            switch (kind) {
              case K_PB: phase_pb<T, KB>(ks.sd, ks.c[cur], tau, ks.ps, part_out); break;
              case K_RESTORE: phase_restore(ks.sd, ks.c[cur], tau, ks.ps, part_out); break;
              case K_OUT:
                phase_out(ks.sd, ks.c[cur], tau, reinterpret_cast<double*>(band_rest()), ks.ps, part_out);
                break;
              default: phase_fin(ks.sd, ks.c[cur], tau, ks.ps, part_out); break;
            }
          }
          if (!single) __syncthreads();
        }
      }
      if (a.trace && threadIdx.x == 0 && tr < a.trace_rounds) {
        TraceEnt e;
        e.t0 = tr0;
        e.t1 = tr1;
        e.t2 = e.t3 = globaltimer();
        e.s0 = ks.ps.sub[0];
        e.s1 = ks.ps.sub[1];
        e.s2 = ks.ps.sub[2];
        e.kind = kind;
        e.items = tb - ta;
        a.trace[(long long)tr * gridDim.x + blockIdx.x] = e;
      }
      ++tr;
      ++nbar;
      if (ta == tb) __syncthreads();  // no band, no block barrier in the phase: nobody is still reading ks.N
      // the phase's last block barrier is behind every warp, and the sums'
      // warps alone have written since: they arrive, the last warp forms the
      // usual next transition and the upper warps do a local round's late work
      // (the block barrier at the top of the loop joins them)
      if (warp < kSumWarps) {
        asm volatile("bar.sync 14, %0;" ::"n"(32 * kSumWarps) : "memory");
        arrive();
        if (sizeof(T) == 4 && late && ta < tb && warp >= kTotWarps) {
          const int t = (int)threadIdx.x - 32 * kTotWarps, nth = 32 * (kSumWarps - kTotWarps);
          if (ks.events)
            band_after<T, KB, false, true>(kind, ta, cur, t, nth);
          else if ((ks.sd.nlon & 3) == 0)
            band_after<T, KB, true, false>(kind, ta, cur, t, nth);
          else
            band_after<T, KB, false, false>(kind, ta, cur, t, nth);
        }
      } else {
        const int t = threadIdx.x & 31;
        Ctx<T>& c = ks.c[cur ^ 1];
#pragma unroll 1
        for (int i = t; i < (int)(sizeof(SolveState) / 8); i += 32)
          reinterpret_cast<long long*>(&ks.S)[i] = reinterpret_cast<const long long*>(&ks.N)[i];
        if (expected) {
          const bool plain = ks.sd.nfaults == 0 && ks.sd.nlosses == 0 && ks.N.step + 1 < ks.sd.max_steps;
          if (!plain)
            for (int i = t; i < (int)(sizeof(Ctx<T>) / 8); i += 32) reinterpret_cast<long long*>(&c)[i] = 0;
          __syncwarp();
          if (t == 0) {
            if (plain)
              usual_transition(ks.sd, ks.S, ks.N, c);
            else
              transition(ks.sd, ks.S, ks.red, ks.qd, ks.N, c, true);
            ks.N.round = ks.S.round + 1;
          }
          __syncwarp();
          fill_directions(ks.sd, ks.S, ks.N, ks.qd, c, t);
          __syncwarp();
          band_plan(ks.sd, c, ks.bp[cur ^ 1], ks.tag, t);
        }
      }
    }
    __syncthreads();
    if (ks.met == 0) {
      // a launch of one round, or a solve with nothing left but its end: the
      // record may be rewritten only once every CTA of the team has loaded it
      if (done) {
        ++nbar;
        arrive();
      }
      if (me.rank == 0) {
        if (threadIdx.x == 0 && !team_wait(nbar * (unsigned)me.size, ks.tf)) ks.bail = 1;
        __syncthreads();
        if (ks.bail) return;
      }
    }
    if (me.rank == 0) {
      // the record: finished (with K_NONE's transition in ks.N), or to be resumed
      if (done) {
        cta_store(ks.sd.result, &ks.N);
        cta_store(ks.sd.st, &ks.N);
        if (threadIdx.x == 0) a.active[s] = 0;
      } else {
        cta_store(ks.sd.st, &ks.S);
      }
    }
    __syncthreads();
  }
}

#undef FTGCR_GROUP
}  // namespace ftgcr
