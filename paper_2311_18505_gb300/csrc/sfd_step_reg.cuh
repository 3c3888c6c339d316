// Register-resident transverse path of the step kernel (included by
// sfd_kernel.cu).  Same scheme and stages as the shared-memory path
// (acceleration form of Eq. 4, partitioned tridiagonal solve, block
// Gauss-Seidel with the longitudinal grid, scalar hammer / bow
// elimination); the MU transverse rows of each lane live in registers with
// fully unrolled loops and neighbours come from shuffles.
//
// A step is one long chain of dependent operations, so what bounds it is the
// number of instructions on that chain and how many warps an SM holds to
// overlap the chains of different strings, not arithmetic or memory.  Hence
// one instance per kind of string (step_string): rows per lane of both
// grids, excitation, linear or not, are compile-time constants, which drops
// the flag tests, the unused stages and the registers they held.  Measured
// alone, microseconds a step, before (one loop for all kinds) and now:
// linear 1.04 / 0.41 (100 rows), one row per lane plucked 3.04 / 1.91 and
// bowed 3.92 / 2.82, three rows 3.01 / 1.88 and 4.05 / 2.68, five rows 4.76 /
// 2.51 and 6.07 / 3.28; 1186 instructions a step became 768 (one row,
// plucked, 2 sweeps).
#pragma once

#include "sfd_device.cuh"

namespace sfd {

// Pad rows (i >= n_u) of every transverse array are zero and the last row of
// lane 31 is always one, so the left neighbour comes by rotation: lane 0
// reads lane 31's pad, the fixed end's zero, without a select.  The right
// neighbour of lane 31 (its own value by __shfl_down) only enters pad rows.
__device__ __forceinline__ float rot_up(float x, int lane) {
  return __shfl_sync(SFD_FULL, x, (lane + kWarp - 1) & (kWarp - 1));
}

// Row values of x at offsets -2..+2 around the lane's chunk:
// e[0] = row base-2, e[1] = base-1, e[2 + r] = x[r], e[MU+2] = base+MU, e[MU+3].
template <int MU>
__device__ __forceinline__ void extend(const float (&x)[MU], float (&e)[MU + 4], int lane) {
  const float l1 = rot_up(x[MU - 1], lane);
  float r1 = __shfl_down_sync(SFD_FULL, x[0], 1);
  float l2, r2;
  if (MU >= 2) {
    l2 = __shfl_up_sync(SFD_FULL, x[MU >= 2 ? MU - 2 : 0], 1);
    r2 = __shfl_down_sync(SFD_FULL, x[MU >= 2 ? 1 : 0], 1);
    if (lane == 0) l2 = 0.f;
    if (lane == kWarp - 1) r1 = 0.f;   // row 32 MU - 2 may be real: its second neighbour is the end
  } else {
    l2 = __shfl_up_sync(SFD_FULL, x[0], 2);
    r2 = __shfl_down_sync(SFD_FULL, x[0], 2);
    if (lane < 2) l2 = 0.f;
    if (lane >= kWarp - 2) r2 = 0.f;
  }
  e[0] = l2;
  e[1] = l1;
#pragma unroll
  for (int r = 0; r < MU; ++r) e[r + 2] = x[r];
  e[MU + 2] = r1;
  e[MU + 3] = r2;
}

// Left/right neighbours only.
template <int MU>
__device__ __forceinline__ void extend1(const float (&x)[MU], float (&e)[MU + 2], int lane) {
  const float l1 = rot_up(x[MU - 1], lane);
  const float r1 = __shfl_down_sync(SFD_FULL, x[0], 1);
  e[0] = l1;
#pragma unroll
  for (int r = 0; r < MU; ++r) e[r + 1] = x[r];
  e[MU + 1] = r1;
}

// Shared-memory accesses at a register plus an immediate (both addresses in
// bytes), and a loop over compile-time indices for them.
template <int OFF>
__device__ __forceinline__ float lds(unsigned a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1+%2];" : "=f"(v) : "r"(a), "n"(OFF) : "memory");
  return v;
}
template <int OFF>
__device__ __forceinline__ void sts(unsigned a, float v) {
  asm volatile("st.shared.f32 [%0+%1], %2;" ::"r"(a), "n"(OFF), "f"(v) : "memory");
}
template <int V>
struct IntC {
  static constexpr int value = V;
};
template <int N, int K = 0, class F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (K < N) {
    f(IntC<K>{});
    static_for<N, K + 1>(f);
  }
}

// The step's sums of products, each with its rounding written out (which
// product is fused into the sum, which is rounded first): left to the
// compiler, that choice depends on the code around the expression, and a
// string's samples would differ in the last bit from one instance to another.
__device__ __forceinline__ float lerp_rn(float w0, float a, float w1, float b) {   // w0 a + w1 b
  return fmaf(w0, a, __fmul_rn(w1, b));
}
__device__ __forceinline__ float div_rn(float gr, float dr, float gl, float dl) {   // gr dr - gl dl
  return fmaf(gr, dr, -__fmul_rn(gl, dl));
}

// A transverse node of the grid, where the warp reads it: row q as (lane,
// row within the lane); a fixed end reads the last pad row.
struct NodePos {
  int src, r;
};
template <int MU>
__device__ __forceinline__ NodePos node_pos(int q, int n_u) {
  const int qq = (q < 0 || q >= n_u) ? kWarp * MU - 1 : q;
  NodePos p;
  p.src = qq / MU;
  p.r = qq - p.src * MU;
  return p;
}
template <int MU>
__device__ __forceinline__ float row_value(const float (&x)[MU], NodePos p) {
  float t = x[0];
#pragma unroll
  for (int k = 1; k < MU; ++k)
    if (k == p.r) t = x[k];
  return __shfl_sync(SFD_FULL, t, p.src);
}
// linear interpolation between two neighbouring nodes, weight w on the second
template <int MU>
__device__ __forceinline__ float node_interp(const float (&x)[MU], NodePos a, NodePos b, float w) {
  return lerp_rn(1.f - w, row_value<MU>(x, a), w, row_value<MU>(x, b));
}

// Partition factorisation of the lane's MU rows (register version of
// tri_factor): on entry iv = diagonal, cp = super-diagonal, sb = sub-diagonal;
// on exit iv = 1/pivot, cp = c', ff/gg = back-substitution weights.  In the
// cyclic reduction a lane without a neighbour 2^l below (above) reads its own
// values: its coupling A (C) to that side is exactly zero by then, since row
// 0 has no sub-diagonal and the last row no super-diagonal, so no select is
// needed.  The reciprocal of each pivot is taken once, before the shuffles.
// On entry rd.nlev is the last step's number of reduction levels, a guess:
// that many run without a vote after each, and two votes at the end correct
// it, so the chain of an ordinary step is the shuffles alone (with the
// intervals' terms formed once, 256 mixed strings 4.51 -> 4.32 ms a block of
// 1024 samples).
template <int MU>
__device__ __forceinline__ void tri_factor_r(const float (&sb)[MU], float (&iv)[MU], float (&cp)[MU],
                                             float (&ff)[MU], float (&gg)[MU], Red& rd) {
  float al[MU];
  float cprev = 0.f, alprev = 0.f;
#pragma unroll
  for (int r = 0; r < MU; ++r) {
    float inv;
    if (r == 0) {
      inv = fast_rcp(iv[r]);
      al[r] = sb[r] * inv;
    } else {
      inv = fast_rcp(fmaf(-sb[r], cprev, iv[r]));
      al[r] = -sb[r] * alprev * inv;
    }
    cp[r] = cp[r] * inv;
    iv[r] = inv;
    cprev = cp[r];
    alprev = al[r];
  }
  ff[MU - 1] = 1.f;
  gg[MU - 1] = 0.f;
#pragma unroll
  for (int r = MU - 2; r >= 0; --r) {
    ff[r] = -cp[r] * ff[r + 1];
    gg[r] = fmaf(-cp[r], gg[r + 1], -al[r]);
  }
  float f0n = 1.f, g0n = 0.f;   // one row per lane: every lane's ff = 1, gg = 0
  if (MU > 1) {
    f0n = __shfl_down_sync(SFD_FULL, ff[0], 1);
    g0n = __shfl_down_sync(SFD_FULL, gg[0], 1);
  }
  const float cl = cp[MU - 1];   // (lane 31's is a pad row's: zero)
  const float A0 = al[MU - 1], B0 = fmaf(cl, g0n, 1.f), C0 = cl * f0n;
  rd.cl = cl;
  // The reduction stops at the first level whose couplings have all dropped
  // below kPcrDrop (at most 5).  That level hardly changes from step to step,
  // so the levels of the last step are run without looking, and two votes
  // tell whether it was the first: not dropped one level before, dropped at
  // it.  (A vote and a branch at every level cost some 45 cycles each on the
  // step's chain.)
  for (;;) {
    float A = A0, B = B0, C = C0;
    bool before = false;    // dropped one level before the last
#pragma unroll
    for (int l = 0; l < 5; ++l) {
      if (l >= rd.nlev) break;
      before = fabsf(A) + fabsf(C) <= kPcrDrop * fabsf(B);
      const int s = 1 << l;
      const float rB = fast_rcp(B);
      const float Am = __shfl_up_sync(SFD_FULL, A, s), Cm = __shfl_up_sync(SFD_FULL, C, s);
      const float Ap = __shfl_down_sync(SFD_FULL, A, s), Cp = __shfl_down_sync(SFD_FULL, C, s);
      const float k1 = A * __shfl_up_sync(SFD_FULL, rB, s), k2 = C * __shfl_down_sync(SFD_FULL, rB, s);
      A = -Am * k1;
      C = -Cp * k2;
      B = fmaf(-Ap, k2, fmaf(-Cm, k1, B));
      rd.k1[l] = k1;
      rd.k2[l] = k2;
    }
    rd.binv = fast_rcp(B);
    if (__all_sync(SFD_FULL, before) && rd.nlev > 0) --rd.nlev;
    else if (rd.nlev < 5 && !__all_sync(SFD_FULL, fabsf(A) + fabsf(C) <= kPcrDrop * fabsf(B))) ++rd.nlev;
    else break;
  }
}

// Solve one (NR = 1) or two (NR = 2) right-hand sides in place, interleaved.
// (Missing neighbours read the lane's own value: their weights are zero.)
template <int MU, int NR>
__device__ __forceinline__ void tri_solve_r(const float (&sb)[MU], const float (&iv)[MU], const float (&cp)[MU],
                                            const float (&ff)[MU], const float (&gg)[MU], float (&x1)[MU],
                                            float (&x2)[MU], const Red& rd) {
  float p1 = 0.f, p2 = 0.f, y1 = 0.f, y2 = 0.f;
#pragma unroll
  for (int r = 0; r < MU; ++r) {
    if (r == 0) {
      p1 = x1[r] * iv[r];
      if (NR == 2) p2 = x2[r] * iv[r];
    } else {
      y1 = fmaf(-sb[r], p1, x1[r]);
      p1 = y1 * iv[r];
      if (NR == 2) { y2 = fmaf(-sb[r], p2, x2[r]); p2 = y2 * iv[r]; }
    }
    x1[r] = p1;
    if (NR == 2) x2[r] = p2;
  }
  const float pl1 = p1, pl2 = p2;
  x1[MU - 1] = 0.f;
  if (NR == 2) x2[MU - 1] = 0.f;
#pragma unroll
  for (int r = MU - 2; r >= 0; --r) {
    x1[r] = fmaf(-cp[r], x1[r + 1], x1[r]);
    if (NR == 2) x2[r] = fmaf(-cp[r], x2[r + 1], x2[r]);
  }
  // (one row per lane: the row just cleared is the neighbour's first, so
  // e1 = e2 = 0 and the shuffles are skipped)
  float e1 = 0.f, e2 = 0.f;
  if (MU > 1) {
    e1 = __shfl_down_sync(SFD_FULL, x1[0], 1);
    e2 = NR == 2 ? __shfl_down_sync(SFD_FULL, x2[0], 1) : 0.f;
  }
  float D1 = MU > 1 ? fmaf(y1, iv[MU - 1], -__fmul_rn(rd.cl, e1)) : pl1;
  float D2 = MU > 1 ? fmaf(y2, iv[MU - 1], -__fmul_rn(rd.cl, e2)) : pl2;
#pragma unroll
  for (int l = 0; l < 5; ++l) {
    if (l >= rd.nlev) break;      // the factorisation dropped the remaining levels (warp-uniform)
    const int s = 1 << l;
    const float m1 = __shfl_up_sync(SFD_FULL, D1, s), q1 = __shfl_down_sync(SFD_FULL, D1, s);
    float m2 = 0.f, q2 = 0.f;
    if (NR == 2) {
      m2 = __shfl_up_sync(SFD_FULL, D2, s);
      q2 = __shfl_down_sync(SFD_FULL, D2, s);
    }
    D1 = fmaf(-rd.k2[l], q1, fmaf(-rd.k1[l], m1, D1));
    if (NR == 2) D2 = fmaf(-rd.k2[l], q2, fmaf(-rd.k1[l], m2, D2));
  }
  const float X1 = D1 * rd.binv, X2 = D2 * rd.binv;
  // (one row per lane: gg = 0, so the previous lane's unknown is not needed;
  // lane 0: gg = 0, no sub-diagonal)
  float Xp1 = 0.f, Xp2 = 0.f;
  if (MU > 1) {
    Xp1 = __shfl_up_sync(SFD_FULL, X1, 1);
    Xp2 = NR == 2 ? __shfl_up_sync(SFD_FULL, X2, 1) : 0.f;
  }
#pragma unroll
  for (int r = 0; r < MU; ++r) {
    x1[r] = fmaf(gg[r], Xp1, fmaf(ff[r], X1, x1[r]));
    if (NR == 2) x2[r] = fmaf(gg[r], Xp2, fmaf(ff[r], X2, x2[r]));
  }
}

// Barrier of the ng = 4 or 8 warps stepping one string together (named
// barrier 1).  Id and counts are immediates, so the kernel reserves only that
// barrier.
__device__ __forceinline__ void group_sync(int ng) {
  if (ng == 8) asm volatile("bar.sync 1, 256;" ::: "memory");
  else asm volatile("bar.sync 1, 128;" ::: "memory");
}

// A string may be stepped by one warp or by a group of ng = 4 or 8 warps, all
// of one CTA (this one is warp pw; they share the string's shared-memory
// region and the exchange cells xcell, 256 floats per warp).  Every warp of a
// group does the whole transverse side identically (same data, same
// operations, so the same bits), and the group splits the longitudinal rows
// by k mod ng; the warps meet at a barrier once the state is loaded, once the
// longitudinal right-hand side is formed (its transfer slots are written
// again in the sweeps), once per Gauss-Seidel sweep (where they also take the
// maximum of each lane's convergence measures, so all see exactly what one
// warp over all rows would) and once per step after the longitudinal update.
// Every barrier sits in control flow that depends only on that shared data.
// Only strings whose longitudinal grid is folded into the sweeps (z_jacobi)
// and gives every warp a row take a group; in a CTA launched for groups
// another string is stepped by warp 0 while the others return at once.
// Warp 0 of a group writes the output, the trajectory record and the state.
constexpr uint32_t kSweepFlush = 1u << 30;

struct WarpGroup {
  int pw = 0, ng = 1;            // this warp's place in the group stepping the string
  float* xcell = nullptr;
};

// One job of one string that is not unstable yet.  MZ: longitudinal rows per
// lane held in registers (0: no longitudinal grid; 1 or 3, folded into the
// sweeps, one warp; 403, 803: up to 12 or 24, three in the registers of each
// of a group's 4 or 8 warps), -1 for any number kept in shared memory (folded,
// one warp or a group), -2 for a factored longitudinal matrix (shared memory,
// one warp).
// Not inlined: each instance gets its own registers (inlined side by side in
// one kernel, the descriptor loads of all of them were hoisted together).
// The region is passed as an offset into the CTA's shared memory, so that
// the accesses stay shared-memory instructions.
template <int MU, int MZ, int EXC, bool LIN>
__device__ __noinline__ void step_string(const Job& job, int region, int lane, const WarpGroup g) {
  extern __shared__ float smem[];
  float* __restrict__ const wbase = smem + region;
  constexpr bool kHasZ = MZ != 0, kReg = MZ > 0, kRows = MZ == -1, kFact = MZ == -2;
  constexpr int kNG = MZ > 100 ? MZ / 100 : 1;        // warps of a register instance
  constexpr int NZ = MZ > 0 ? MZ % 100 : 1;           // register rows (dummy when unused)
  constexpr bool kRecs = kRows || kNG > 1;            // longitudinal rows as records (below)
  constexpr bool kForced = EXC != kPluck;
  const Desc* __restrict__ Dp = job.desc;
  const int n_t = Dp->n_t, n_l = Dp->n_l, n_u = Dp->n_u, n_z = Dp->n_z;
  const int m_z = kReg && kNG == 1 ? NZ : Dp->m_z;
  const bool paired = kNG > 1 || (kRows && g.ng > 1);
  const int kz0 = kRecs ? g.pw : 0, kzs = kRows ? g.ng : kNG;   // this warp's longitudinal rows: k = pw, pw + ng, ...
  const int n_mine = kRows ? (m_z - kz0 + kzs - 1) / kzs : 0;   // ... how many
  const bool writer = !kRecs || g.pw == 0;
  int xpar = 0;                                             // exchange buffer in use
  const int RU = kWarp * MU + 4, RZ = kWarp * m_z + 4;
  // Byte address of longitudinal row 0's first field, and the fields' offsets
  // from a row's address.  Register instances: one array per field, so that
  // row i is at 4 i and every access a register plus an immediate.  Rows in
  // shared memory: one record of 11 words per row (odd: no bank conflicts
  // between lanes), for the same reason with any number of rows.
  constexpr int kRec = 44;
  constexpr int kRowBytes = kRecs ? kRec : 4, kFld = kRecs ? 4 : 4 * (kWarp * NZ + 4);
  constexpr int kStep = kRowBytes * kWarp;             // ... of row i + 32
  constexpr int oZ = 0, oDZ = kFld, oAZ = 2 * kFld, oXZ = 3 * kFld, oSF0 = 4 * kFld, oSF1 = 5 * kFld;
  constexpr int oSX0 = 6 * kFld, oSX1 = 7 * kFld, oSV0 = kRecs ? oSF0 : 8 * kFld, oSV1 = kRecs ? oSF1 : 9 * kFld;
  constexpr int oRZ = 8 * kFld, oE2 = 9 * kFld, oE3 = 10 * kFld;   // (records only)
  constexpr int rb = kRowBytes;
  const unsigned sbase = static_cast<unsigned>(__cvta_generic_to_shared(smem)) + 4u * (region + 2 * RU) +
                         2 * kRowBytes;
  const unsigned zrow = sbase + kRowBytes * lane;      // longitudinal row `lane`; row lane + 32 k at + 32 k rows
  unsigned fA = oAZ, fX = oXZ;                         // records: where the current accelerations are
  const float dg = Dp->dg, og = Dp->og, s1l = Dp->s1l;
  const float bsgn = Dp->boundary == 1 ? -1.f : 1.f;
  const int mod_kind = Dp->mod_kind;
  const int sweep_cap = job.sweep_cap > 0 ? job.sweep_cap : kMaxSweeps;

  // ---- shared memory: the longitudinal grid and the transfer slots, after
  // two transverse slots (kept free) ----
  float* p = wbase + 2 * RU;
  float *Z = nullptr, *DZ = nullptr, *AZ = nullptr, *XZ = nullptr, *RZ_ = nullptr, *E1Z = nullptr;
  float *SUBZ = nullptr, *INVZ = nullptr, *CPZ = nullptr, *ALZ = nullptr, *FFZ = nullptr, *GGZ = nullptr;
  float *SF0 = nullptr, *SF1 = nullptr, *SX0 = nullptr, *SX1 = nullptr;   // scatter slots
  if (kFact) {   // factored longitudinal matrix: one array per field
    auto Z_ = [&]() { float* a = p + 2; p += RZ; return a; };
    Z = Z_(); DZ = Z_(); AZ = Z_(); XZ = Z_(); RZ_ = Z_(); E1Z = Z_(); SF0 = Z_(); SF1 = Z_(); SX0 = Z_();
    SX1 = Z_(); SUBZ = Z_(); INVZ = Z_(); CPZ = Z_(); ALZ = Z_(); FFZ = Z_(); GGZ = Z_();
  } else if (kHasZ) {
    p += (kRecs ? 11 : 10) * RZ;
  }
  if (kHasZ) {
    const int total = static_cast<int>(p - wbase);
    for (int k = 2 * RU + lane + kWarp * kz0; k < total; k += kWarp * kzs) wbase[k] = 0.f;
    __syncwarp();
    if (paired) group_sync(g.ng);   // the region is zero before either warp writes to it
  }
  // value of a field at longitudinal row i
  auto zat = [&](int field, const float* A, int i) {
    return kFact ? A[i] : lds<0>(sbase + kRowBytes * i + field);
  };
  // Register instances: address and number of the warp's row k.  In a group a
  // warp may have fewer rows than registers: a missing row reads the first
  // one's neighbours, is never real and stores nothing.
  unsigned za[NZ];
  int zn[NZ];
#pragma unroll
  for (int k = 0; k < NZ; ++k) {
    const int kk = kz0 + kNG * k;
    const bool have = kNG == 1 || kk < m_z;
    za[k] = zrow + kStep * (have ? kk : kz0);
    zn[k] = have ? lane + kWarp * kk : 0x7fffffff;
  }
  auto zget = [&](auto kc, auto off_c) {
    constexpr int k = decltype(kc)::value, off = decltype(off_c)::value;
    if constexpr (kNG == 1) return lds<off + kStep * k>(zrow);
    else return lds<off>(za[k]);
  };
  auto zput = [&](auto kc, auto off_c, float v) {
    constexpr int k = decltype(kc)::value, off = decltype(off_c)::value;
    if constexpr (kNG == 1) sts<off + kStep * k>(zrow, v);
    else if (k == 0 || zn[k] != 0x7fffffff) sts<off>(za[k], v);
  };
  // this warp's rows in batches of up to four, whose loads overlap: fn(batch
  // size, row addresses, row numbers).  A short last batch repeats its last
  // row (the same values are computed and stored again).
  auto my_rows = [&](auto fn) {
    int t = 0;
    auto batch = [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      unsigned a[R];
      int i[R];
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const int k = kz0 + kzs * min(t + q, n_mine - 1);
        i[q] = lane + kWarp * k;
        a[q] = zrow + kStep * k;
      }
      fn(rc, a, i);
    };
    for (; t + 4 <= n_mine; t += 4) batch(IntC<4>{});
    if (n_mine - t == 1) batch(IntC<1>{});
    else if (n_mine > t) batch(IntC<4>{});
  };

  // ---- registers: the lane's transverse rows i = lane*MU + r, and its
  // longitudinal rows i = lane + 32 k ----
  const int ub = lane * MU;
  float U[MU], DU[MU];
#pragma unroll
  for (int r = 0; r < MU; ++r) {
    const int i = ub + r;
    U[r] = i < n_u ? Dp->u[i] : 0.f;
    DU[r] = i < n_u ? Dp->du[i] : 0.f;
  }
  float zr[NZ], dzr[NZ], azr[NZ], xzr[NZ], rzr[NZ];
  if (kHasZ) {
    if (kFact) {
      for (int i = lane; i < n_z; i += kWarp) {
        Z[i] = Dp->z[i]; DZ[i] = Dp->dz[i]; XZ[i] = Dp->xz[i]; AZ[i] = Dp->az[i];
      }
    } else if (kRows) {
      for (int i = lane + kWarp * kz0; i < n_z; i += kWarp * kzs) {
        const unsigned a = sbase + kRowBytes * i;
        sts<oZ>(a, Dp->z[i]);
        sts<oDZ>(a, Dp->dz[i]);
        sts<oAZ>(a, Dp->az[i]);
        if (kForced) sts<oXZ>(a, Dp->xz[i]);
      }
    } else {
      static_for<NZ>([&](auto kc) {
        constexpr int k = decltype(kc)::value;
        const int i = zn[k];
        const bool real = i < n_z;
        zr[k] = real ? Dp->z[i] : 0.f;
        dzr[k] = real ? Dp->dz[i] : 0.f;
        azr[k] = real ? Dp->az[i] : 0.f;
        xzr[k] = real && kForced ? Dp->xz[i] : 0.f;
        zput(kc, IntC<oZ>{}, zr[k]);
        zput(kc, IntC<oDZ>{}, dzr[k]);
        zput(kc, IntC<oAZ>{}, azr[k]);
        if (kForced) zput(kc, IntC<oXZ>{}, xzr[k]);
      });
    }
  }
  const Scalars* scp = Dp->sc;
  int64_t n = scp->n, jnext = scp->next_out;
  const int64_t n_first = n;
  float uh = scp->uh, duh = scp->duh, bow_w = scp->bow_w, scz = scp->scale_z, scx = scp->scale_x;
  int status = scp->status;
  int max_sweeps = scp->max_sweeps;
  // (32 bits while stepping: at most kMaxSweepCap per step, added to the
  // string's total every kSweepFlush steps and at the end)
  uint32_t sweeps_sum = 0;
  __syncwarp();
  if (paired) group_sync(g.ng);   // both halves of the longitudinal state are loaded

  // (P^T F) at longitudinal node m = sum over the transverse nodes l of
  // P[l, m] F_l, P the linear interpolation from the longitudinal to the
  // transverse nodes.  Transverse node l (row l - 1) lies in the longitudinal
  // interval [m_l, m_l + 1) and gives (1 - w_l) F_l to node m_l and w_l F_l
  // to node m_l + 1.  The rows of one interval are consecutive, and each
  // lane owns consecutive rows, so emit() sums every interval by a segmented
  // scan (within the lane's rows, then across lanes by shuffles) and the
  // interval's last row stores the two sums: S0[m] = sum of (1 - w) F over
  // interval m, S1[m + 1] = sum of w F over it.  Node m then reads
  // S0[m] + S1[m] (spreadS).  Which slots are written is fixed by the grid,
  // so the others keep the zeros they were given; pad rows form their own
  // interval N_l + 1 with weight 0.
  //
  // mme / we: the map of rows -1 .. MU of the lane (exact integer positions;
  // row -1 of lane 0 is the fixed end: node 0 with weight 0, pad rows point
  // at node N_l + 1, a zero cell), so each lane interpolates its neighbours'
  // rows itself rather than waiting for a shuffle.
  int mme[MU + 2];
  float we[MU + 2];
  int mmr[MU];
  float wr[MU];
  unsigned lastm = 0;          // bit r: row r is the last row of its interval
  bool carry_ok = false;       // the lane's first interval began in an earlier lane
  int scan_lv = 0;             // shuffle levels that close every interval
  unsigned scan_add = 0;       // bit l: the lane adds the sum from lane - 2^l at scan level l
  if (kHasZ) {
#pragma unroll
    for (int q = 0; q < MU + 2; ++q) {
      const int i = ub + q - 1;
      const int pos = (i + 1) * n_l;
      mme[q] = i < n_u ? pos / n_t : n_l + 1;
      we[q] = i < n_u ? static_cast<float>(pos - mme[q] * n_t) / static_cast<float>(n_t) : 0.f;
    }
#pragma unroll
    for (int r = 0; r < MU; ++r) { mmr[r] = mme[r + 1]; wr[r] = we[r + 1]; }
    const int nxt = __shfl_down_sync(SFD_FULL, mmr[0], 1);
    const int prv = __shfl_up_sync(SFD_FULL, mmr[MU - 1], 1);
#pragma unroll
    for (int r = 0; r < MU - 1; ++r)
      if (mmr[r + 1] != mmr[r]) lastm |= 1u << r;
    if (lane == kWarp - 1 || nxt != mmr[MU - 1]) lastm |= 1u << (MU - 1);
#pragma unroll
    for (int r = 0; r < MU; ++r)
      if (ub + r >= n_u) lastm &= ~(1u << r);   // pad rows store nothing
    carry_ok = lane > 0 && prv == mmr[0];
    bool f = !(lane > 0 && prv == mmr[MU - 1]);   // the lane's last interval begins in this lane
    for (int l = 0; l < 5 && !__all_sync(SFD_FULL, f); ++l) {
      const int sh = 1 << l;
      const bool fu = __shfl_up_sync(SFD_FULL, f ? 1 : 0, sh) != 0;
      if (lane >= sh) {
        if (!f) scan_add |= 1u << l;
        f = f || fu;
      }
      scan_lv = l + 1;
    }
  }
  // A longitudinal field interpolated to rows -1 .. MU of the lane.
  unsigned mmo[MU + 2];             // address of row mm - 1, the node left of transverse row q - 1
#pragma unroll
  for (int q = 0; q < MU + 2; ++q) mmo[q] = sbase + kRowBytes * (mme[q] - 1);
  auto interp_z = [&](const float* A, unsigned field, float (&e)[MU + 2]) {
#pragma unroll
    for (int q = 0; q < MU + 2; ++q) {
      const float w = we[q];
      if (kFact) {
        e[q] = lerp_rn(1.f - w, A[mme[q] - 1], w, A[mme[q]]);
      } else {
        const unsigned a = mmo[q] + field;
        e[q] = lerp_rn(1.f - w, lds<0>(a), w, lds<kRowBytes>(a));
      }
    }
  };
  // Interval sums of (1 - w) f and w f for one or two fields at once
  // (independent chains interleaved), stored into their slot pairs.
  auto emit2 = [&](const float (&f)[MU], float* S0, float* S1, const float (&h)[MU], float* T0, float* T1,
                   auto two_c, auto off_c) {
    constexpr bool two = decltype(two_c)::value;
    constexpr int o0 = decltype(off_c)::value, o1 = o0 + kFld, o2 = oSX0, o3 = oSX1;   // slots of node mm: row mm
    float a0[MU], a1[MU], b0[MU], b1[MU];
#pragma unroll
    for (int r = 0; r < MU; ++r) {
      const bool cont = r > 0 && mmo[r + 1] == mmo[r > 0 ? r : 1];
      const int rp = r > 0 ? r - 1 : 0;
      const float p0 = __fmul_rn(1.f - wr[r], f[r]), p1 = __fmul_rn(wr[r], f[r]);
      const float q0 = __fmul_rn(1.f - wr[r], h[r]), q1 = __fmul_rn(wr[r], h[r]);
      a0[r] = cont ? __fadd_rn(a0[rp], p0) : p0;
      a1[r] = cont ? __fadd_rn(a1[rp], p1) : p1;
      b0[r] = cont ? __fadd_rn(b0[rp], q0) : q0;
      b1[r] = cont ? __fadd_rn(b1[rp], q1) : q1;
    }
    float v0 = a0[MU - 1], v1 = a1[MU - 1], x0 = b0[MU - 1], x1 = b1[MU - 1];
#pragma unroll
    for (int l = 0; l < 5; ++l) {
      if (l >= scan_lv) break;
      const int sh = 1 << l;
      const float u0 = __shfl_up_sync(SFD_FULL, v0, sh), u1 = __shfl_up_sync(SFD_FULL, v1, sh);
      float y0 = 0.f, y1 = 0.f;
      if (two) {
        y0 = __shfl_up_sync(SFD_FULL, x0, sh);
        y1 = __shfl_up_sync(SFD_FULL, x1, sh);
      }
      if ((scan_add >> l) & 1u) { v0 += u0; v1 += u1; x0 += y0; x1 += y1; }
    }
    float c0 = __shfl_up_sync(SFD_FULL, v0, 1), c1 = __shfl_up_sync(SFD_FULL, v1, 1);
    float d0 = 0.f, d1 = 0.f;
    if (two) {
      d0 = __shfl_up_sync(SFD_FULL, x0, 1);
      d1 = __shfl_up_sync(SFD_FULL, x1, 1);
    }
#pragma unroll
    for (int r = 0; r < MU; ++r) {
      if (!((lastm >> r) & 1u)) continue;
      const bool add = carry_ok && mmo[r + 1] == mmo[1];
      const float t0 = add ? a0[r] + c0 : a0[r], t1 = add ? a1[r] + c1 : a1[r];
      if (kFact) {
        S0[mmr[r]] = t0;
        S1[mmr[r] + 1] = t1;
      } else {
        sts<o0 + kRowBytes>(mmo[r + 1], t0);
        sts<o1 + 2 * kRowBytes>(mmo[r + 1], t1);
      }
      if (two) {
        const float s0x = add ? b0[r] + d0 : b0[r], s1x = add ? b1[r] + d1 : b1[r];
        if (kFact) {
          T0[mmr[r]] = s0x;
          T1[mmr[r] + 1] = s1x;
        } else {
          sts<o2 + kRowBytes>(mmo[r + 1], s0x);
          sts<o3 + 2 * kRowBytes>(mmo[r + 1], s1x);
        }
      }
    }
  };
  auto spreadS = [&](const float* S0, const float* S1, int i) { return S0[i + 1] + S1[i + 1]; };

  // ---- constant matrices ----
  Red rdu, rdz;
  rdu.nlev = 3;
#pragma unroll
  for (int l = 0; l < 5; ++l) { rdu.k1[l] = 0.f; rdu.k2[l] = 0.f; }
  const float dz_diag = 1.f + Dp->s0 + 2.f * s1l;
  const float dz_inv = fast_rcp(dz_diag);
  if (kFact) {
    for (int r = 0; r < m_z; ++r) {
      const int i = lane * m_z + r;
      if (i < n_z) {
        SUBZ[i] = i > 0 ? -s1l : 0.f;
        INVZ[i] = dz_diag;
        CPZ[i] = i < n_z - 1 ? -s1l : 0.f;
      } else {
        SUBZ[i] = 0.f; INVZ[i] = 1.f; CPZ[i] = 0.f;
      }
    }
    tri_factor(SUBZ, INVZ, CPZ, ALZ, FFZ, GGZ, m_z, lane, rdz);
  }
  float SB[MU], IV[MU], CPr[MU], FFr[MU], GGr[MU];
  // unfactored diagonal and superdiagonal, kept for the refinement residual
  // (single-row lanes only: the strings that refine have at most 31 rows)
  float DG0[MU], CP0[MU];
  const bool refine = MU == 1 && Dp->refine != 0;
#pragma unroll
  for (int r = 0; r < MU; ++r) {
    const int i = ub + r;
    if (i < n_u) {
      SB[r] = i > 0 ? og : 0.f;
      IV[r] = dg;
      CPr[r] = i < n_u - 1 ? og : 0.f;
    } else {
      SB[r] = 0.f; IV[r] = 1.f; CPr[r] = 0.f;
    }
    DG0[r] = IV[r];
    CP0[r] = CPr[r];
  }
  int en = Dp->e_node;              // excitation point (a bow envelope moves it per step)
  float ew = Dp->e_w;
  NodePos e0 = node_pos<MU>(en - 1, n_u), e1 = node_pos<MU>(en, n_u);
  const float js = Dp->jscale;
  float XP[MU];
  auto load_J = [&](float (&E)[MU]) {
#pragma unroll
    for (int r = 0; r < MU; ++r) {
      const int i = ub + r;
      float v = 0.f;
      if (i == en - 1) v += (1.f - ew) * js;
      if (i == en) v += ew * js;
      E[r] = (i < n_u) ? v : 0.f;
    }
  };
#pragma unroll
  for (int r = 0; r < MU; ++r) XP[r] = 0.f;
  if (LIN) {
    tri_factor_r<MU>(SB, IV, CPr, FFr, GGr, rdu);
    if (kForced) {
      load_J(XP);
      tri_solve_r<MU, 1>(SB, IV, CPr, FFr, GGr, XP, XP, rdu);
    }
  }
  __syncwarp();

  // One step of iterative refinement of the transverse solve A x = b: the
  // residual against the unfactored entries (exact floats for a linear
  // string) is solved with the same factors and added, which removes the
  // lasting error of the FP32 factorisation from the solution.
  auto refine_solve = [&](const float (&b)[MU], float (&x)[MU]) {
    float xe[MU + 2], rr[MU];
    extend1<MU>(x, xe, lane);
#pragma unroll
    for (int r = 0; r < MU; ++r)
      rr[r] = b[r] - fmaf(CP0[r], xe[r + 2], fmaf(DG0[r], xe[r + 1], __fmul_rn(SB[r], xe[r])));
    tri_solve_r<MU, 1>(SB, IV, CPr, FFr, GGr, rr, rr, rdu);
#pragma unroll
    for (int r = 0; r < MU; ++r) x[r] += rr[r];
  };

  const int on = Dp->o_node, oln = Dp->ol_node;
  const NodePos o0 = node_pos<MU>(on - 1, n_u), o1 = node_pos<MU>(on, n_u);
  const float ow = Dp->o_w, olw = Dp->ol_w, oscale = Dp->out_scale;
  const bool zout = Dp->out_ch == 1;
  const int64_t j_end = jnext + job.n_samples;
  const bool recorded = job.traj != nullptr;
  float outbuf = 0.f;
  int opos = 0;                     // samples in outbuf
  float* out = job.out;
  float AC[MU];

  // sample of the current level, or of the one before
  auto sample = [&](bool before) {
    float y;
    if (zout) {   // L zeta^j at the pickup (zero without a longitudinal grid)
      y = 0.f;
      if (kHasZ) {
        // between longitudinal nodes oln and oln + 1; the fixed ends read zero
        auto at = [&](int field, const float* A) {
          const float a = (oln >= 1 && oln - 1 < n_z) ? zat(field, A, oln - 1) : 0.f;
          const float b = (oln >= 0 && oln < n_z) ? zat(field, A, oln) : 0.f;
          return lerp_rn(1.f - olw, a, olw, b);
        };
        y = at(oZ, Z);
        if (before) y -= at(oDZ, DZ);
      }
    } else if (before) {
      y = node_interp<MU>(U, o0, o1, ow) - node_interp<MU>(DU, o0, o1, ow);
    } else {
      y = node_interp<MU>(U, o0, o1, ow);
    }
    return y * oscale;
  };
  auto put = [&](float y) {
    if (opos == lane) outbuf = y;
    if (++opos == kWarp) {
      if (writer) out[lane] = outbuf;
      out += kWarp;
      opos = 0;
    }
  };

  // the levels already reached (at most two samples)
  while (jnext < j_end && jnext <= n) {
    put(sample(jnext == n - 1));
    ++jnext;
  }

  // gamma^2 coefficients of the step (constant without f0 modulation)
  float lam2 = Dp->lam2, lam2_lo = Dp->lam2_lo, lam2l = Dp->lam2l, ca = Dp->ca, cb = Dp->cb, cz = Dp->cz;

  // jnext = n + 1 from here: each step reaches the level of one sample
  const int64_t n_end = j_end - 1;
  while (n < n_end) {
    // ======================= one step n -> n+1 =======================
    if (mod_kind != 0) {
      const Desc* Dm = reread(Dp);
      const float rm = mod_factor_at(mod_kind, static_cast<uint64_t>(n) * Dm->mod_inc_fx + Dm->mod_phase_fx,
                                     Dm->mod_depth2, Dm->mod_inc, Dm->mod_hold, Dm->mod_n_end, n);
      const float lam2_0 = Dm->lam2;
      lam2 = lam2_0 * rm;
      // low part of lam2_0 * rm (exact product residual plus the stored low part)
      lam2_lo = fmaf(lam2_0, rm, -lam2) + Dm->lam2_lo * rm;
      if (!LIN) { ca = Dm->ca * rm; }
      if (kHasZ) { lam2l = Dm->lam2l * rm; cb = Dm->cb * rm; cz = Dm->cz * rm; }
    }
    const Desc* De = kForced ? reread(Dp) : Dp;   // constants read once a step (forced: not held in registers)
    const float s0u = De->s0u, s1 = De->s1, mu2 = De->mu2;

    float eta = 0.f, k2G = 0.f, FB = 0.f, bv = 0.f;
    float vrec = 0.f;   // bow: relative velocity of the step (0 while sticking), for the adjoint
    if (EXC == kHammer) {
      eta = __fsub_rn(uh, node_interp<MU>(U, e0, e1, ew));
      if (eta > 0.f) k2G = De->ham_k2w * powf(eta, De->ham_expo);
    } else if (EXC == kBow) {
      float bf = De->bow_F;
      bv = De->bow_v;
      if (De->bow_env_n > 0) {
        const int en0 = en;
        const float ew0 = ew;
        bow_env_eval(Dp, n, bv, bf, en, ew);
        if (en != en0) { e0 = node_pos<MU>(en - 1, n_u); e1 = node_pos<MU>(en, n_u); }
        if (LIN && (en != en0 || ew != ew0)) {   // the fixed-matrix response A^-1 J follows x_B
          load_J(XP);
          tri_solve_r<MU, 1>(SB, IV, CPr, FFr, GGr, XP, XP, rdu);
        }
      }
      FB = (n < De->bow_release_n) ? bf : 0.f;
    }
    const bool need_resp = !LIN && ((EXC == kHammer && k2G > 0.f) || (EXC == kBow && FB > 0.f));

    // ---- stage 1: transverse right-hand side and matrix (registers) ----
    float Ue[MU + 4], DUe[MU + 2], GL[MU], GR[MU], gi[MU + 1], yi[MU + 1], gi2[MU + 1];
    extend<MU>(U, Ue, lane);
    extend1<MU>(DU, DUe, lane);
#pragma unroll
    for (int r = 0; r < MU + 1; ++r) gi[r] = Ue[r + 2] - Ue[r + 1];   // interval left of row r
#pragma unroll
    for (int r = 0; r < MU; ++r) {   // interval differences; zero on pad rows
      const bool real = ub + r < n_u;
      GL[r] = real ? gi[r] : 0.f;
      GR[r] = real ? gi[r + 1] : 0.f;
    }
    float ZTe[MU + 2];
    if (kHasZ) interp_z(Z, oZ, ZTe);
    // the strain's and the coupling's terms of every interval (each serves the
    // rows on both sides)
    if (!LIN) {
#pragma unroll
      for (int r = 0; r < MU + 1; ++r) {
        const float gk = gi[r];
        gi2[r] = __fmul_rn(gk, gk);
        yi[r] = __fmul_rn(2.f * ca * gi2[r], gk);
        if (kHasZ) {
          const float zk = ZTe[r + 1] - ZTe[r];
          // (the two forms differ in the last bit; each class keeps the one
          // its samples have had)
          if (MU >= 5) yi[r] = fmaf(2.f * ca * gi2[r], gk, __fmul_rn(4.f * cb * gk, zk));
          else yi[r] = fmaf(4.f * cb * gk, zk, yi[r]);
        }
      }
    }
    float RA[MU], fv[MU];
#pragma unroll
    for (int r = 0; r < MU; ++r) {
      const int i = ub + r;
      const bool real = i < n_u;
      fv[r] = 0.f;
      const float u0 = Ue[r + 2], um1 = Ue[r + 1], up1 = Ue[r + 3], um2 = Ue[r], up2 = Ue[r + 4];
      const float gl = gi[r], gr = gi[r + 1];
      const float d2 = gr - gl;
      float d4 = ((up2 - up1) - gr) - 2.f * d2 + (gl - (um1 - um2));
      if (i == 0) d4 += bsgn * u0;
      if (i == n_u - 1) d4 += bsgn * u0;
      const float du0 = DUe[r + 1];
      const float d2du = (DUe[r + 2] - du0) - (du0 - DUe[r]);
      float rhs = fmaf(2.f * s1, d2du, fmaf(-2.f * s0u, du0, fmaf(-mu2, d4, fmaf(lam2, d2, __fmul_rn(lam2_lo, d2)))));
      if (!LIN) {
        // (fv of a pad row goes to no slot)
        if (kHasZ) fv[r] = gi2[r + 1] - gi2[r];
        rhs = __fadd_rn(rhs, __fsub_rn(yi[r + 1], yi[r]));
        SB[r] = (real && i > 0) ? fmaf(-ca, gi2[r], og) : 0.f;
        IV[r] = real ? fmaf(ca, __fadd_rn(gi2[r], gi2[r + 1]), dg) : 1.f;
        CPr[r] = i < n_u - 1 ? fmaf(-ca, gi2[r + 1], og) : 0.f;
        DG0[r] = IV[r];
        CP0[r] = CPr[r];
      }
      RA[r] = i < n_u ? rhs : 0.f;
    }
    if (kHasZ) emit2(fv, SF0, SF1, fv, SF0, SF1, BoolC<false>{}, IntC<oSV0>{});
    if (!LIN) tri_factor_r<MU>(SB, IV, CPr, FFr, GGr, rdu);
    if (kHasZ) __syncwarp();

    if (!kHasZ) {
#pragma unroll
      for (int r = 0; r < MU; ++r) AC[r] = RA[r];
      if (need_resp) {
        load_J(XP);
        tri_solve_r<MU, 2>(SB, IV, CPr, FFr, GGr, AC, XP, rdu);
      } else {
        tri_solve_r<MU, 1>(SB, IV, CPr, FFr, GGr, AC, AC, rdu);
      }
      if (refine) refine_solve(RA, AC);
    } else {
      // ---- stage 2: longitudinal right-hand side ----
      float dzmax = 0.f;   // lane's largest |Dz|: scale of the longitudinal increments
      auto rhs_row = [&](int i, float zm, float z0, float zp, float dzm, float dz0, float dzp, float sv) {
        const float d2z = (zp - z0) - (z0 - zm);
        const float d2dz = (dzp - dz0) - (dz0 - dzm);
        dzmax = fmaxf(dzmax, fabsf(dz0));
        const float s0 = De->s0;
        const float v = fmaf(2.f * cz, sv,
                             fmaf(2.f * s1l, d2dz, fmaf(lam2l, d2z, -__fmul_rn(2.f * s0, dz0))));
        return i < n_z ? v : 0.f;
      };
      if (kFact) {
        for (int i = lane; i < kWarp * m_z; i += kWarp)
          RZ_[i] = rhs_row(i, Z[i - 1], Z[i], Z[i + 1], DZ[i - 1], DZ[i], DZ[i + 1], spreadS(SF0, SF1, i));
        __syncwarp();
      } else if (kRows) {
        my_rows([&](auto rc, const unsigned (&a)[decltype(rc)::value], const int (&i)[decltype(rc)::value]) {
          constexpr int R = decltype(rc)::value;
          float v[R];
#pragma unroll
          for (int q = 0; q < R; ++q)
            v[q] = rhs_row(i[q], lds<oZ - kRec>(a[q]), lds<oZ>(a[q]), lds<oZ + kRec>(a[q]), lds<oDZ - kRec>(a[q]),
                           lds<oDZ>(a[q]), lds<oDZ + kRec>(a[q]),
                           lds<oSF0 + kRec>(a[q]) + lds<oSF1 + kRec>(a[q]));
#pragma unroll
          for (int q = 0; q < R; ++q) sts<oRZ>(a[q], v[q]);
        });
        __syncwarp();
        if (paired) group_sync(g.ng);   // every warp has read the slots that the sweeps rewrite
      } else {
        static_for<NZ>([&](auto kc) {
          constexpr int k = decltype(kc)::value;
          rzr[k] = rhs_row(zn[k], zget(kc, IntC<oZ - rb>{}), zr[k], zget(kc, IntC<oZ + rb>{}),
                           zget(kc, IntC<oDZ - rb>{}), dzr[k], zget(kc, IntC<oDZ + rb>{}),
                           zget(kc, IntC<oSV0 + rb>{}) + zget(kc, IntC<oSV1 + rb>{}));
        });
        if (paired) {
          __syncwarp();
          group_sync(g.ng);
        }
      }
      // ---- stage 3: block Gauss-Seidel on (a, az) [and the response] ----
      auto gauss_seidel = [&](auto resp_c) {
        constexpr bool resp = decltype(resp_c)::value;
        int sweep = 0;
        float e_prev = 0.f, mag_all = 0.f, mgx_all = 0.f;
        for (;;) {
          float AZe[MU + 2], azs[NZ], xzs[NZ];
          interp_z(AZ, kRecs ? fA : oAZ, AZe);
          if (kReg) {
            static_for<NZ>([&](auto kc) {   // neighbours of the old field, before it is overwritten
              constexpr int k = decltype(kc)::value;
              if constexpr (kNG == 1) {
                azs[k] = zget(kc, IntC<oAZ - rb>{}) + zget(kc, IntC<oAZ + rb>{});
                if (resp) xzs[k] = zget(kc, IntC<oXZ - rb>{}) + zget(kc, IntC<oXZ + rb>{});
              } else {
                azs[k] = lds<-rb>(za[k] + fA) + lds<rb>(za[k] + fA);
                if (resp) xzs[k] = lds<-rb>(za[k] + fX) + lds<rb>(za[k] + fX);
              }
            });
          }
#pragma unroll
          for (int r = 0; r < MU; ++r)
            AC[r] = fmaf(cb, div_rn(GR[r], AZe[r + 2] - AZe[r + 1], GL[r], AZe[r + 1] - AZe[r]), RA[r]);
          float BC[MU];
#pragma unroll
          for (int r = 0; r < MU; ++r) BC[r] = AC[r];
          if (resp) {
            float XZe[MU + 2];
            interp_z(XZ, kRecs ? fX : oXZ, XZe);
            load_J(XP);
#pragma unroll
            for (int r = 0; r < MU; ++r)
              XP[r] = fmaf(cb, div_rn(GR[r], XZe[r + 2] - XZe[r + 1], GL[r], XZe[r + 1] - XZe[r]), XP[r]);
            tri_solve_r<MU, 2>(SB, IV, CPr, FFr, GGr, AC, XP, rdu);
          } else {
            tri_solve_r<MU, 1>(SB, IV, CPr, FFr, GGr, AC, AC, rdu);
          }
          if (refine) refine_solve(BC, AC);
          // nodal d_+[g d(.)] of the new accelerations for the longitudinal rows
          {
            float ACe[MU + 2], fc[MU], fx[MU];
            extend1<MU>(AC, ACe, lane);
#pragma unroll
            for (int r = 0; r < MU; ++r)
              fc[r] = div_rn(GR[r], ACe[r + 2] - ACe[r + 1], GL[r], ACe[r + 1] - ACe[r]);
            if (resp) {
              float XPe[MU + 2];
              extend1<MU>(XP, XPe, lane);
#pragma unroll
              for (int r = 0; r < MU; ++r)
                fx[r] = div_rn(GR[r], XPe[r + 2] - XPe[r + 1], GL[r], XPe[r + 1] - XPe[r]);
              emit2(fc, SF0, SF1, fx, SX0, SX1, BoolC<true>{}, IntC<oSF0>{});
            } else {
              emit2(fc, SF0, SF1, fc, SF0, SF1, BoolC<false>{}, IntC<oSF0>{});
            }
          }
          __syncwarp();
          float chg = 0.f, mag = 0.f, chx = 0.f, mgx = 0.f;
          if (kReg) {
            // one Jacobi update of each field
            // (a group's other warps may still read the old field: it goes
            // to the spare, and the two swap)
            const unsigned eA = kNG > 1 ? oAZ + oE2 - fA : 0, eX = kNG > 1 ? oXZ + oE3 - fX : 0;
            static_for<NZ>([&](auto kc) {
              constexpr int k = decltype(kc)::value;
              const bool real = zn[k] < n_z;
              const float sf = zget(kc, IntC<oSF0 + rb>{}) + zget(kc, IntC<oSF1 + rb>{});
              float v = fmaf(s1l, azs[k], fmaf(cz, sf, rzr[k])) * dz_inv;
              v = real ? v : 0.f;
              chg = fmaxf(chg, fabsf(v - azr[k]));
              mag = fmaxf(mag, fabsf(v));
              azr[k] = v;
              if constexpr (kNG == 1) zput(kc, IntC<oAZ>{}, v);
              else if (k == 0 || zn[k] != 0x7fffffff) sts<0>(za[k] + eA, v);
              if (resp) {
                const float sx = zget(kc, IntC<oSX0 + rb>{}) + zget(kc, IntC<oSX1 + rb>{});
                float x = fmaf(cz, sx, __fmul_rn(s1l, xzs[k])) * dz_inv;
                x = real ? x : 0.f;
                chx = fmaxf(chx, fabsf(x - xzr[k]));
                mgx = fmaxf(mgx, fabsf(x));
                xzr[k] = x;
                if constexpr (kNG == 1) zput(kc, IntC<oXZ>{}, x);
                else if (k == 0 || zn[k] != 0x7fffffff) sts<0>(za[k] + eX, x);
              }
            });
            if (kNG > 1) {
              fA = eA;
              if (resp) fX = eX;
            }
            __syncwarp();
          } else if (kRows) {
            // one Jacobi update of each field into its spare, then swap
            const unsigned eA = oAZ + oE2 - fA, eX = oXZ + oE3 - fX;
            my_rows([&](auto rc, const unsigned (&a)[decltype(rc)::value], const int (&i)[decltype(rc)::value]) {
              constexpr int R = decltype(rc)::value;
              float v[R], x[R];
#pragma unroll
              for (int q = 0; q < R; ++q) {
                const bool real = i[q] < n_z;
                const unsigned b = a[q] + fA;
                v[q] = fmaf(s1l, lds<-kRec>(b) + lds<kRec>(b),
                            fmaf(cz, lds<oSF0 + kRec>(a[q]) + lds<oSF1 + kRec>(a[q]), lds<oRZ>(a[q]))) * dz_inv;
                v[q] = real ? v[q] : 0.f;
                chg = fmaxf(chg, fabsf(v[q] - lds<0>(b)));
                mag = fmaxf(mag, fabsf(v[q]));
                if (resp) {
                  const unsigned c = a[q] + fX;
                  x[q] = fmaf(cz, lds<oSX0 + kRec>(a[q]) + lds<oSX1 + kRec>(a[q]),
                              __fmul_rn(s1l, lds<-kRec>(c) + lds<kRec>(c))) * dz_inv;
                  x[q] = real ? x[q] : 0.f;
                  chx = fmaxf(chx, fabsf(x[q] - lds<0>(c)));
                  mgx = fmaxf(mgx, fabsf(x[q]));
                }
              }
#pragma unroll
              for (int q = 0; q < R; ++q) {
                sts<0>(a[q] + eA, v[q]);
                if (resp) sts<0>(a[q] + eX, x[q]);
              }
            });
            __syncwarp();
            fA = eA;
            if (resp) fX = eX;
          } else {
            for (int r = 0; r < m_z; ++r) {
              const int i = lane * m_z + r;
              E1Z[i] = i < n_z ? fmaf(cz, spreadS(SF0, SF1, i), RZ_[i]) : 0.f;
            }
            tri_solve(SUBZ, INVZ, CPZ, FFZ, GGZ, E1Z, m_z, lane, rdz);
            for (int r = 0; r < m_z; ++r) {
              const int i = lane * m_z + r;
              const float v = E1Z[i];
              chg = fmaxf(chg, fabsf(v - AZ[i]));
              mag = fmaxf(mag, fmaxf(fabsf(v), fabsf(DZ[i])));
              AZ[i] = v;
            }
            if (resp) {
              for (int r = 0; r < m_z; ++r) {
                const int i = lane * m_z + r;
                E1Z[i] = i < n_z ? cz * spreadS(SX0, SX1, i) : 0.f;
              }
              tri_solve(SUBZ, INVZ, CPZ, FFZ, GGZ, E1Z, m_z, lane, rdz);
              for (int r = 0; r < m_z; ++r) {
                const int i = lane * m_z + r;
                const float v = E1Z[i];
                chx = fmaxf(chx, fabsf(v - XZ[i]));
                mgx = fmaxf(mgx, fabsf(v));
                XZ[i] = v;
              }
            }
            __syncwarp();
          }
          // relative change: each field against the larger of its magnitude
          // in this lane and its string-wide scale from the previous step,
          // so one warp reduction per sweep suffices
          mag = fmaxf(mag, dzmax);
          if (paired) {
            // each lane's maxima over the group's rows: the other warps'
            // updates are in shared memory once all pass the barrier
            float4* xc = reinterpret_cast<float4*>(g.xcell) + xpar * (kNG > 1 ? 32 * kNG : 32 * g.ng) + lane;
            xc[g.pw * 32] = make_float4(chg, mag, chx, mgx);
            group_sync(g.ng);
#pragma unroll
            for (int w = 0; w < 8; ++w) {
              if (w >= (kNG > 1 ? kNG : g.ng)) break;
              const float4 o = xc[w * 32];
              chg = fmaxf(chg, o.x);
              mag = fmaxf(mag, o.y);
              chx = fmaxf(chx, o.z);
              mgx = fmaxf(mgx, o.w);
            }
            xpar ^= 1;
          }
          // (a measure compared with thresholds: the fast divide suffices)
          float el = chg > 0.f ? __fdividef(chg, fmaxf(mag, scz)) : 0.f;
          if (resp) el = fmaxf(el, chx > 0.f ? __fdividef(chx, fmaxf(mgx, scx)) : 0.f);
          mag_all = fmaxf(mag_all, mag);
          mgx_all = fmaxf(mgx_all, mgx);
          const float e = warp_max_nonneg(el);
          ++sweep;
          if (sweep_converged(e, e_prev, sweep)) break;
          if (sweep >= sweep_cap) { status |= kStNoConv; break; }
          e_prev = e;
        }
        sweeps_sum += sweep;
        if (sweep > max_sweeps) max_sweeps = sweep;
        // string-wide scales for the next step's convergence test
        scz = warp_max_nonneg(mag_all);
        if (resp) scx = warp_max_nonneg(mgx_all);
      };
      if constexpr (EXC == kPluck) {
        gauss_seidel(BoolC<false>{});
      } else {
        if (need_resp) gauss_seidel(BoolC<true>{});
        else gauss_seidel(BoolC<false>{});
      }
    }

    // ---- stage 4: excitation force (scalar elimination) ----
    auto add_response = [&](float s) {
#pragma unroll
      for (int r = 0; r < MU; ++r) AC[r] = fmaf(s, XP[r], AC[r]);
      if (kFact) {
        for (int i = lane; i < kWarp * m_z; i += kWarp) AZ[i] = fmaf(s, XZ[i], AZ[i]);
      } else if (kRows) {
        my_rows([&](auto rc, const unsigned (&a)[decltype(rc)::value], const int (&)[decltype(rc)::value]) {
          constexpr int R = decltype(rc)::value;
          float v[R];
#pragma unroll
          for (int q = 0; q < R; ++q) v[q] = fmaf(s, lds<0>(a[q] + fX), lds<0>(a[q] + fA));
#pragma unroll
          for (int q = 0; q < R; ++q) sts<0>(a[q] + fA, v[q]);
        });
      } else if (kHasZ) {
        static_for<NZ>([&](auto kc) {
          constexpr int k = decltype(kc)::value;
          azr[k] = fmaf(s, xzr[k], azr[k]);
          if constexpr (kNG == 1) zput(kc, IntC<oAZ>{}, azr[k]);
          else if (k == 0 || zn[k] != 0x7fffffff) sts<0>(za[k] + fA, azr[k]);
        });
      }
    };
    if (EXC == kHammer) {
      float s = 0.f;
      if (k2G > 0.f) {
        const float ham_M = De->ham_M;
        const float cm = 0.5f * ham_M * k2G;
        s = __fmul_rn(cm, fmaf(2.f, eta, -node_interp<MU>(AC, e0, e1, ew))) /
            fmaf(cm, node_interp<MU>(XP, e0, e1, ew), fmaf(0.5f, k2G, 1.f));
        duh -= s / ham_M;
      }
      uh += duh;
      if (s != 0.f) add_response(s);
    } else if (EXC == kBow) {
      if (FB > 0.f) {
        const float kk = De->k;
        const float inv2k = 0.5f / kk;   // 1 / 2k: the bow's velocity I(a + 2D) / 2k
        const float b = fmaf(fmaf(2.f, node_interp<MU>(DU, e0, e1, ew), node_interp<MU>(AC, e0, e1, ew)), inv2k, -bv);
        const float c = 0.5f * kk * FB * node_interp<MU>(XP, e0, e1, ew);
        const float phi = bow_phi(b, c, De->bow_a, De->bow_eps, bow_w);
        vrec = !(c > 0.f) ? b : (fabsf(b) <= c ? 0.f : b - c * phi);
        add_response(-De->k2 * FB * phi);
      }
    }

    // ---- stage 5: advance the time level ----
    bool bad = false;
#pragma unroll
    for (int r = 0; r < MU; ++r) {   // pad rows stay zero (their accelerations are zero)
      DU[r] = DU[r] + AC[r];
      U[r] = U[r] + DU[r];
      bad |= !isfinite(U[r]);
    }
    if (kFact) {
      for (int i = lane; i < kWarp * m_z; i += kWarp) {
        const float d = DZ[i] + AZ[i];
        DZ[i] = d;
        Z[i] = Z[i] + d;
      }
    } else if (kRows) {
      my_rows([&](auto rc, const unsigned (&a)[decltype(rc)::value], const int (&)[decltype(rc)::value]) {
        constexpr int R = decltype(rc)::value;
        float d[R], z[R];
#pragma unroll
        for (int q = 0; q < R; ++q) {
          d[q] = lds<oDZ>(a[q]) + lds<0>(a[q] + fA);
          z[q] = lds<oZ>(a[q]) + d[q];
        }
#pragma unroll
        for (int q = 0; q < R; ++q) {
          sts<oDZ>(a[q], d[q]);
          sts<oZ>(a[q], z[q]);
        }
      });
    } else if (kHasZ) {
      static_for<NZ>([&](auto kc) {
        constexpr int k = decltype(kc)::value;
        dzr[k] = dzr[k] + azr[k];
        zr[k] = zr[k] + dzr[k];
        zput(kc, IntC<oDZ>{}, dzr[k]);
        zput(kc, IntC<oZ>{}, zr[k]);
      });
    }
    const bool unstable = __any_sync(SFD_FULL, bad);
    if (kHasZ) __syncwarp();
    if (paired) group_sync(g.ng);   // the new level is complete in shared memory
    ++n;
    if (recorded && writer) {   // record for the adjoint: the new level
      const Job* J = reread(&job);
      const int nu = reread(Dp)->n_u, nz = kHasZ ? n_z : 0;
      float* rec = J->traj + (n - n_first - 1) * J->traj_stride;
#pragma unroll
      for (int r = 0; r < MU; ++r) {
        const int i = ub + r;
        if (i < nu) { rec[i] = U[r]; rec[nu + i] = DU[r]; }
      }
      if (kHasZ)
        for (int i = lane; i < nz; i += kWarp) {
          rec[2 * nu + i] = zat(oZ, Z, i);
          rec[2 * nu + nz + i] = zat(oDZ, DZ, i);
        }
      // (a bowed string has no hammer state: its slot holds the step's bow velocity)
      if (lane == 0) { rec[2 * nu + 2 * nz] = EXC == kBow ? vrec : uh; rec[2 * nu + 2 * nz + 1] = duh; }
    }
    if (unstable) {
      status |= kStUnstable;
      break;
    }
    put(sample(false));
    if (kHasZ && sweeps_sum >= kSweepFlush) {
      if (lane == 0 && writer) Dp->sc->sweeps_total += sweeps_sum;
      sweeps_sum = 0;
    }
  }
  if (jnext < j_end) {
    jnext = j_end;
    // unstable: this sample (of level n) and the remaining ones are zero
    if (status & kStUnstable)
      for (int64_t j = n; j < j_end; ++j) put(0.f);
  }
  if (lane < opos && writer) out[lane] = outbuf;

  // ---- store the state ----
  __syncwarp();
  if (!writer) return;
#pragma unroll
  for (int r = 0; r < MU; ++r) {
    const int i = ub + r;
    if (i < n_u) { Dp->u[i] = U[r]; Dp->du[i] = DU[r]; }
  }
  if (kHasZ) {
    for (int i = lane; i < n_z; i += kWarp) {
      Dp->z[i] = zat(oZ, Z, i);
      Dp->dz[i] = zat(oDZ, DZ, i);
      Dp->az[i] = zat(kRecs ? fA : oAZ, AZ, i);
      if (kForced) Dp->xz[i] = zat(kRecs ? fX : oXZ, XZ, i);
    }
  }
  if (lane == 0) {
    Scalars* so = Dp->sc;
    so->n = n;
    so->next_out = jnext;
    so->uh = uh;
    so->duh = duh;
    so->bow_w = bow_w;
    so->scale_z = scz;
    so->scale_x = scx;
    so->status = status;
    so->max_sweeps = max_sweeps;
    so->sweeps_total += sweeps_sum;
  }
  __syncwarp();
}

// The instance of a string's excitation and longitudinal grid.
template <int MU, int EXC>
__device__ __forceinline__ void run_job_exc(const Job& job, int region, int lane, WarpGroup g, int npw) {
  const Desc* __restrict__ Dp = job.desc;
  const int m_z = Dp->m_z;
  const bool zjac = Dp->z_jacobi != 0;
  if (npw > 1 && zjac && m_z >= npw) g.ng = npw;   // (a row for every warp)
  if (g.pw >= g.ng) return;                       // the group's other warps step it
  if (Dp->linear) step_string<MU, 0, EXC, true>(job, region, lane, g);
  else if (m_z == 0) step_string<MU, 0, EXC, false>(job, region, lane, g);
  else if (!zjac) step_string<MU, -2, EXC, false>(job, region, lane, g);
  else if (m_z == 1) step_string<MU, 1, EXC, false>(job, region, lane, g);
  else if (m_z == 3) step_string<MU, 3, EXC, false>(job, region, lane, g);
  else if (g.ng == 4 && m_z <= 12) step_string<MU, 403, EXC, false>(job, region, lane, g);
  else if (g.ng == 8 && m_z > 8 && m_z <= 24) step_string<MU, 803, EXC, false>(job, region, lane, g);
  else step_string<MU, -1, EXC, false>(job, region, lane, g);
}

template <int MU>
__device__ __forceinline__ void run_job_reg(const Job& job, int region, int lane, int pw, int npw, float* xcell) {
  WarpGroup g;
  g.pw = pw;
  g.xcell = xcell;
  const int exc = job.desc->exc;
  if (exc == kPluck) run_job_exc<MU, kPluck>(job, region, lane, g, npw);
  else if (exc == kHammer) run_job_exc<MU, kHammer>(job, region, lane, g, npw);
  else run_job_exc<MU, kBow>(job, region, lane, g, npw);
}

}  // namespace sfd
