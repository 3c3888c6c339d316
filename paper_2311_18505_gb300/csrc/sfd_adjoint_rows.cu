// Adjoint sweep with one thread per transverse row (the reverse step itself is
// described in sfd_adjoint.cu, whose kernel takes the strings this one does
// not: more than 255 rows, or a longitudinal matrix that is not folded).
//
// A reverse step is a chain of two or more solves whose every operation takes
// some 50 cycles in double-floats, so what bounds it is the length of that
// chain.  Here every row is a thread's: the transverse system is reduced
// cyclically over all rows at once (5 levels; the partition method's chain is
// a lane's rows forward and back, then the same 5 levels over the lanes, on
// one warp of four), the longitudinal one, nearly diagonal, in the 1 to 3
// levels its coupling needs, the two right-hand sides of a struck or bowed
// step go through the sweeps together, P^T is a sum over the rows of two
// intervals (split over idle threads) of products formed in parallel, and the
// next level of the trajectory is copied to shared memory while a step runs.
// 64 plucked and struck strings of 40-1000 Hz take 20.7 us a step (one of 87 x
// 143 rows alone 14.0), against 41 us (27) with four warps per string and the
// solves on one of them; 12 bowed ones 22 against 45.
#include <cuda_runtime.h>

#include <mutex>

#include "sfd_device.cuh"

namespace sfd {

namespace {

using R = df64;
constexpr float kTol = 1e-13f;   // relative change that ends a block Gauss-Seidel solve
constexpr int kSweeps = 40;
constexpr int kLev = kAdjRowsLev;
constexpr int kZLev = kAdjRowsZLev;
constexpr int kThreads = kAdjRowsMax + 1;

__device__ __forceinline__ R get(const float2* a) { return R(a->x, a->y); }
__device__ __forceinline__ void put(float2* a, R v) { *a = make_float2(v.hi, v.lo); }

__device__ __forceinline__ bool converged(float e, float e_prev, int sweep) {
  if (e <= kTol) return true;
  if (sweep >= 2 && e < e_prev && e * e <= kTol * e_prev) return true;
  if (sweep >= 3 && e >= 0.5f * e_prev && e <= 64.f * kTol) return true;
  return sweep >= kSweeps;
}

// 16 bytes from global to shared memory, completing at wait_copies()
__device__ __forceinline__ void copy16(float* dst, const float* src) {
  const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void wait_copies() { asm volatile("cp.async.wait_all;" ::: "memory"); }

}  // namespace

__global__ void __launch_bounds__(kThreads, 1) adjoint_rows_kernel(const AdjJob* __restrict__ jobs) {
  extern __shared__ float4 smem4[];
  __shared__ float red[2][4][kThreads / kWarp];
  __shared__ float2 gsum[kThreads / kWarp][kGradSlots];
  __shared__ float2 scal;          // a step's FP64 function value
  const int tid = threadIdx.x, T = blockDim.x, lane = tid & (kWarp - 1), warp = tid >> 5, n_warps = T >> 5;
  const AdjJob J = jobs[blockIdx.x];
  const Desc* __restrict__ Dp = J.desc;
  const int n_t = Dp->n_t, n_l = Dp->n_l, n_u = Dp->n_u, n_z = Dp->n_z;
  const bool has_z = n_z > 0, linear = Dp->linear != 0;
  const bool hammer = Dp->exc == kHammer, bow = Dp->exc == kBow;
  const R dg = Dp->dg, og = Dp->og, s0 = Dp->s0, s0u = Dp->s0u, s1 = Dp->s1, s1l = Dp->s1l, mu2 = Dp->mu2;
  const float lam2_0f = Dp->lam2, lam2lo_0f = Dp->lam2_lo, lam2l_0f = Dp->lam2l;
  const float ca_0f = Dp->ca, cb_0f = Dp->cb, cz_0f = Dp->cz;
  const int mod_kind = Dp->mod_kind;
  R lam2 = static_cast<R>(lam2_0f) + static_cast<R>(lam2lo_0f), lam2l = lam2l_0f;
  R ca = ca_0f, cb = cb_0f, cz = cz_0f, rmd = 1.0f;
  const R bsgn = Dp->boundary == 1 ? -1.0f : 1.0f;
  const int en = Dp->e_node, on = Dp->o_node, oln = Dp->ol_node;
  const R ew = Dp->e_w, js = Dp->jscale, ow = Dp->o_w, olw = Dp->ol_w, oscale = Dp->out_scale;
  const bool zout = Dp->out_ch == 1;
  const R hM = Dp->ham_M, hk2w = Dp->ham_k2w, hexpo = Dp->ham_expo;
  const R bF = Dp->bow_F, ba = Dp->bow_a, beps = Dp->bow_eps, kk = Dp->k;
  const int64_t brel = Dp->bow_release_n;

  // ---- shared memory (adj_rows_smem_bytes): three trajectory records, then
  // the double-float arrays (two zero cells at both ends), floats and ints ----
  const int rec_n = (2 * n_u + 2 * n_z + 2 + 3) & ~3;
  float* recs = reinterpret_cast<float*>(smem4);
  float2* pd = reinterpret_cast<float2*>(recs + 3 * rec_n);
  auto du = [&]() { float2* a = pd + 2; pd += n_u + 4; return a; };
  auto dz = [&]() { float2* a = pd + 2; pd += n_z + 4; return a; };
  float2 *FA[2], *FC[2], *FR[2], *X = nullptr, *XP = nullptr, *P0 = nullptr, *P1 = nullptr, *Q0 = nullptr, *Q1 = nullptr;
  float2 *TN = nullptr, *TX = nullptr;
  FA[0] = du(); FA[1] = du(); FC[0] = du(); FC[1] = du(); FR[0] = du(); FR[1] = du();
  X = du(); XP = du(); P0 = du(); P1 = du(); Q0 = du(); Q1 = du(); TN = du(); TX = du();
  float2 *NZ = nullptr, *XZ = nullptr, *RZ = nullptr, *LZ = nullptr, *LDZ = nullptr, *BZ = nullptr;
  float2 *NZP = nullptr, *XZP = nullptr;
  float2 *E[2] = {nullptr, nullptr}, *G[2] = {nullptr, nullptr}, *KA = nullptr, *KC = nullptr;
  const int zl = n_z + 4;          // one level of KA, KC
  if (has_z) {
    NZ = dz(); XZ = dz(); RZ = dz(); LZ = dz(); LDZ = dz(); BZ = dz(); NZP = dz(); XZP = dz(); E[0] = dz(); E[1] = dz(); G[0] = dz();
    G[1] = dz();
    KA = dz(); pd += (kZLev - 1) * zl;
    KC = dz(); pd += (kZLev - 1) * zl;
  }
  float2 *KU = pd, *KL = pd + kLev * n_u;   // transverse reduction weights, level by level
  pd += 2 * kLev * n_u;
  float* pf = reinterpret_cast<float*>(pd);
  float *A = pf + 2, *AZ = nullptr;
  pf += n_u + 4;
  int* ROW0 = nullptr;             // first transverse row of longitudinal interval m
  if (has_z) {
    AZ = pf + 2; pf += n_z + 4;
    ROW0 = reinterpret_cast<int*>(pf); pf += n_z + 4;
  }
  {
    const int n = static_cast<int>(pf - recs);
#pragma unroll 1
    for (int k = tid; k < n; k += T) recs[k] = 0.f;
  }
  __syncthreads();

  // ---- this thread's transverse row, and its longitudinal rows zi, zi + zs, ...
  // (parts: threads per longitudinal row in the sums of P^T) ----
  const int i = tid;
  const bool act = i < n_u;
  int parts = 1;
  if (has_z) while (parts < 8 && 2 * parts * n_z <= T) parts *= 2;
  const int zi = tid / parts, zs = T / parts, part = tid & (parts - 1);
  const bool zown = part == 0;
  // grid transfer: maps of rows i - 1, i, i + 1 (row -1: the fixed end, node 0)
  int mm[3] = {0, 0, 0};
  R wm[3], w1m[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int r = i + q - 1, pos = (r + 1) * n_l;
    const bool in = has_z && r < n_u;
    mm[q] = in ? pos / n_t : n_l;
    const float w = in ? static_cast<float>(pos - mm[q] * n_t) / static_cast<float>(n_t) : 0.f;
    wm[q] = w;
    w1m[q] = 1.0f - wm[q];
  }
  // the row's weights in P^T, in double-floats as in sfd_adjoint.cu (wm, w1m
  // are the forward's own floats; with those the gradients of plucked and
  // bowed strings were up to 5e-6 from that kernel's, with these 2e-9)
  dfl::NodeWeights wt = {1.0f, 0.0f};
  if (has_z && act) wt = dfl::node_weights((i + 1) * n_l - mm[1] * n_t, n_t, 1.0f / static_cast<R>(n_t));
  if (has_z)
#pragma unroll 1
    for (int m = tid; m <= n_l + 1; m += T) {   // n_z + 3 entries
      const int l = static_cast<int>((static_cast<int64_t>(m) * n_t + n_l - 1) / n_l);   // first node l with m_l >= m
      ROW0[m] = min(max(l, 1) - 1, n_u);
    }
  // fields of longitudinal nodes interpolated to row i - 1 + q
  auto to_t = [&](const float2* F, int q) -> R { return w1m[q] * get(F + mm[q] - 1) + wm[q] * get(F + mm[q]); };
  auto to_tf = [&](const float* F, int q) -> R { return w1m[q] * F[mm[q] - 1] + wm[q] * F[mm[q]]; };
  // (P^T f) at longitudinal row z from the products P0 = (1 - w) f, P1 = w f
  auto spread = [&](const float2* a0, const float2* a1, int z) -> R {
    const int r0 = ROW0[z], r1 = ROW0[z + 1], r2 = ROW0[z + 2];
    R s0a = 0.0f, s1a = 0.0f;
#pragma unroll 1
    for (int r = r0 + part; r < r1; r += parts) s0a += get(a1 + r);
#pragma unroll 1
    for (int r = r1 + part; r < r2; r += parts) s1a += get(a0 + r);
    R s = s0a + s1a;
#pragma unroll 1
    for (int o = 1; o < parts; o <<= 1) s += shfl_xor(s, o);
    return s;
  };
  auto zrows = [&](auto fn) {   // every thread of a row's group calls fn (its shuffles are theirs together)
#pragma unroll 1
    for (int z = zi; z < ((n_z + zs - 1) / zs) * zs; z += zs) fn(z, z < n_z);
  };
  // block-wide maxima of four non-negative floats (one barrier, two buffers)
  int rbuf = 0;
  auto block_max4 = [&](float (&v)[4]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = warp_max_nonneg(v[k]);
    if (lane < 4) red[rbuf][lane][warp] = lane == 0 ? v[0] : lane == 1 ? v[1] : lane == 2 ? v[2] : v[3];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float o = lane < n_warps ? red[rbuf][k][lane] : 0.f;
      v[k] = warp_max_nonneg(o);
    }
    rbuf ^= 1;
  };

  // ---- longitudinal matrix: reduced once, as many levels as its coupling needs ----
  int zlev = 0;
  if (has_z) {
    const R d = 1.0f + s0 + 2.0f * s1l;
    // rows in E (sub), G (super), BZ (diagonal), ping-pong; the reciprocal is taken where it is read
#pragma unroll 1
    for (int z = tid; z < n_z; z += T) {
      put(E[0] + z, z > 0 ? -s1l : R(0.0f));
      put(G[0] + z, z < n_z - 1 ? -s1l : R(0.0f));
      put(BZ + z, d);
    }
    __syncthreads();
#pragma unroll 1
    for (int l = 0; l < kZLev; ++l) {
      bool ok = true;
#pragma unroll 1
      for (int z = tid; z < n_z; z += T)
        ok = ok && ::fabsf(E[l & 1][z].x) + ::fabsf(G[l & 1][z].x) <= pcr_drop(R(0.0f)) * ::fabsf(BZ[z].x);
      if (__syncthreads_and(ok)) break;
      const int s = 1 << l;
      // (the new diagonal goes to RZ until every thread has read the old one)
#pragma unroll 1
      for (int z = tid; z < n_z; z += T) {
        const int a = z >= s ? z - s : z, b = z + s < n_z ? z + s : z;
        const R k1 = get(E[l & 1] + z) * rcp_df(get(BZ + a)), k2 = get(G[l & 1] + z) * rcp_df(get(BZ + b));
        put(KA + l * zl + z, k1);
        put(KC + l * zl + z, k2);
        put(RZ + z, get(BZ + z) - get(G[l & 1] + a) * k1 - get(E[l & 1] + b) * k2);
        put(E[(l + 1) & 1] + z, -(get(E[l & 1] + a) * k1));
        put(G[(l + 1) & 1] + z, -(get(G[l & 1] + b) * k2));
      }
      __syncthreads();
#pragma unroll 1
      for (int z = tid; z < n_z; z += T) BZ[z] = RZ[z];
      zlev = l + 1;
      __syncthreads();
    }
#pragma unroll 1
    for (int z = tid; z < n_z; z += T) put(BZ + z, rcp_df(get(BZ + z)));
    for (int k = 0; k < 2; ++k)
#pragma unroll 1
      for (int z = tid; z < n_z; z += T) { put(E[k] + z, R(0.0f)); put(G[k] + z, R(0.0f)); }
  }

  // ---- transverse system: cyclic reduction over all rows.  (The level loops
  // stay rolled, their weights in shared memory: unrolled with the weights in
  // registers the kernel was 338 KB of code and waited for instructions 1.9
  // cycles of every 5.1 per issue.) ----
  R binv = 1.0f;
  int nlev = 0;
  auto assemble = [&](float gl, float gr) {
    const R gl2 = linear ? R(0.0f) : dfl::mul_ff(gl, gl), gr2 = linear ? R(0.0f) : dfl::mul_ff(gr, gr);
    R a = act && i > 0 ? og - ca * gl2 : R(0.0f), c = act && i < n_u - 1 ? og - ca * gr2 : R(0.0f);
    R b = act ? dg + ca * (gl2 + gr2) : R(1.0f), r = 1.0f;
#pragma unroll 1
    for (nlev = 0;; ++nlev) {
      const bool ok = !act || ::fabsf(a.hi) + ::fabsf(c.hi) <= pcr_drop(R(0.0f)) * ::fabsf(b.hi);
      r = rcp_df(b);
      float2 *fa = FA[nlev & 1], *fc = FC[nlev & 1], *fr = FR[nlev & 1];
      if (act) { put(fa + i, a); put(fc + i, c); put(fr + i, r); }
      if (__syncthreads_and(ok) || nlev == kLev) break;
      if (act) {
        // (a row without a neighbour 2^l away reads its own values: its
        // coupling to that side is zero)
        const int s = 1 << nlev, m = i >= s ? i - s : i, p = i + s < n_u ? i + s : i;
        const R k1 = a * get(fr + m), k2 = c * get(fr + p);
        b = b - (get(fc + m) * k1 + get(fa + p) * k2);
        a = -(get(fa + m) * k1);
        c = -(get(fc + p) * k2);
        put(KU + nlev * n_u + i, k1);
        put(KL + nlev * n_u + i, k2);
      }
    }
    binv = r;
    __syncthreads();
  };
  // solve in place one or two right-hand sides (row i's entries)
  auto solve = [&](R& d, R& e, bool two) {
#pragma unroll 1
    for (int l = 0; l < nlev; ++l) {
      float2 *fd = FA[l & 1], *fe = FC[l & 1];
      if (act) { put(fd + i, d); if (two) put(fe + i, e); }
      __syncthreads();
      if (act) {
        const int s = 1 << l, m = i >= s ? i - s : i, p = i + s < n_u ? i + s : i;
        const R k1 = get(KU + l * n_u + i), k2 = get(KL + l * n_u + i);
        d = d - (k1 * get(fd + m) + k2 * get(fd + p));
        if (two) e = e - (k1 * get(fe + m) + k2 * get(fe + p));
      }
    }
    d = d * binv;
    if (two) e = e * binv;
  };

  // Solve M (x, NZ) = (ra, RZ) and, with two, M (y, XZ) = (J, 0), by block
  // Gauss-Seidel from the warm starts in NZ, XZ; x, y are left in X, XP too.
  auto coupled = [&](R ra, R rj, float gl, float gr, R& x, R& y, bool two) {
    if (!has_z) {
      x = ra;
      y = rj;
      solve(x, y, two);
      if (act) { put(X + i, x); if (two) put(XP + i, y); }
      __syncthreads();
      return;
    }
    float e_prev = 0.f;
#pragma unroll 1
    for (int sweep = 1;; ++sweep) {
      {
        const R t1 = to_t(NZ, 1), v1 = two ? to_t(XZ, 1) : R(0.0f);
        if (act) { put(TN + i, t1); if (two) put(TX + i, v1); }
        __syncthreads();
        if (act) x = ra + cb * ((get(TN + i + 1) - t1) * gr - (t1 - get(TN + i - 1)) * gl);
        if (act && two) y = rj + cb * ((get(TX + i + 1) - v1) * gr - (v1 - get(TX + i - 1)) * gl);
      }
      solve(x, y, two);
      if (act) { put(X + i, x); if (two) put(XP + i, y); }
      __syncthreads();
      if (act) {   // d_+[g d_- x] at the row, times the row's weights
        const R f = (get(X + i + 1) - x) * gr - (x - get(X + i - 1)) * gl;
        put(P0 + i, wt.left * f);
        put(P1 + i, wt.right * f);
        if (two) {
          const R h = (get(XP + i + 1) - y) * gr - (y - get(XP + i - 1)) * gl;
          put(Q0 + i, wt.left * h);
          put(Q1 + i, wt.right * h);
        }
      }
      __syncthreads();
      zrows([&](int z, bool in) {
        const int zz = in ? z : n_z - 1;
        const R s = spread(P0, P1, zz);
        R h = 0.0f;
        if (two) h = spread(Q0, Q1, zz);
        if (in && zown) {
          put(E[0] + z, get(RZ + z) + cz * s);
          if (two) put(G[0] + z, cz * h);
        }
      });
      __syncthreads();
#pragma unroll 1
      for (int l = 0; l + 1 < zlev; ++l) {
        const int s = 1 << l;
#pragma unroll 1
        for (int z = tid; z < n_z; z += T) {
          const int a = z >= s ? z - s : z, b = z + s < n_z ? z + s : z;
          const R k1 = get(KA + l * zl + z), k2 = get(KC + l * zl + z);
          put(E[(l + 1) & 1] + z, get(E[l & 1] + z) - (k1 * get(E[l & 1] + a) + k2 * get(E[l & 1] + b)));
          if (two) put(G[(l + 1) & 1] + z, get(G[l & 1] + z) - (k1 * get(G[l & 1] + a) + k2 * get(G[l & 1] + b)));
        }
        __syncthreads();
      }
      float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
      for (int z = tid; z < n_z; z += T) {
        const int l = zlev > 0 ? zlev - 1 : 0, s = 1 << l;
        const int a = z >= s ? z - s : z, b = z + s < n_z ? z + s : z;
        R f = get(E[l & 1] + z), h = two ? get(G[l & 1] + z) : R(0.0f);
        if (zlev > 0) {
          const R k1 = get(KA + l * zl + z), k2 = get(KC + l * zl + z);
          f = f - (k1 * get(E[l & 1] + a) + k2 * get(E[l & 1] + b));
          if (two) h = h - (k1 * get(G[l & 1] + a) + k2 * get(G[l & 1] + b));
        }
        f = f * get(BZ + z);
        v[0] = fmaxf(v[0], ::fabsf((f - get(NZ + z)).hi));
        v[1] = fmaxf(v[1], ::fabsf(f.hi));
        put(NZ + z, f);
        if (two) {
          h = h * get(BZ + z);
          v[2] = fmaxf(v[2], ::fabsf((h - get(XZ + z)).hi));
          v[3] = fmaxf(v[3], ::fabsf(h.hi));
          put(XZ + z, h);
        }
      }
      block_max4(v);   // (its barrier also orders the updates)
      const float e = fmaxf(v[0] > 0.f ? __fdividef(v[0], v[1]) : 0.f, v[2] > 0.f ? __fdividef(v[2], v[3]) : 0.f);
      if (converged(e, e_prev, sweep)) break;
      e_prev = e;
    }
  };

  // ---- adjoint state at level m_end, warm starts ----
  double* adj = J.adj;
  R LU = 0.0f, LD = 0.0f;
  if (act) { LU = df_from_double(adj[i]); LD = df_from_double(adj[n_u + i]); }
#pragma unroll 1
  for (int z = tid; z < n_z; z += T) {
    put(LZ + z, df_from_double(adj[2 * n_u + z]));
    put(LDZ + z, df_from_double(adj[2 * n_u + n_z + z]));
    put(NZ + z, df_from_double(adj[2 * n_u + 2 * n_z + 2 + z]));
    put(XZ + z, df_from_double(adj[2 * n_u + 3 * n_z + 2 + z]));
  }
  R luh = df_from_double(adj[2 * n_u + 2 * n_z]), ldh = df_from_double(adj[2 * n_u + 2 * n_z + 1]);
  R acc[kGradSlots];
#pragma unroll
  for (int k = 0; k < kGradSlots; ++k) acc[k] = 0.0f;
  // dJ/du of an output sample y = L I(x_o) u, or dJ/dz of y = L I_l(x_o) z
  // (D, Dz also take -c w for the first sample, which reads level 1 - D)
  auto add_output = [&](float dyv, bool first_level) {
    const R c = dyv * oscale;
    if (zout) {
#pragma unroll 1
      for (int z = tid; z < n_z; z += T) {
        if (z != oln - 1 && z != oln) continue;
        const R w = z == oln ? olw : 1.0f - olw;
        put(LZ + z, get(LZ + z) + c * w);
        if (first_level) put(LDZ + z, get(LDZ + z) - c * w);
      }
    } else if (act && (i == on - 1 || i == on)) {
      const R w = i == on ? ow : 1.0f - ow;
      LU += c * w;
      if (first_level) LD -= c * w;
    }
  };

  // levels: m_start from the checkpoint, later ones from the trajectory
  auto fetch = [&](int64_t lev, float* dst) {
    if (lev > J.m_start) {
      const float* src = J.traj + (lev - J.m_start - 1) * J.traj_stride;
#pragma unroll 1
      for (int k = 4 * tid; k < rec_n; k += 4 * T) copy16(dst + k, src + k);
    } else if (lev == J.m_start) {
#pragma unroll 1
      for (int k = tid; k < n_u; k += T) { dst[k] = J.u0[k]; dst[n_u + k] = J.du0[k]; }
#pragma unroll 1
      for (int k = tid; k < n_z; k += T) { dst[2 * n_u + k] = J.z0[k]; dst[2 * n_u + n_z + k] = J.dz0[k]; }
      if (tid == 0) { dst[2 * n_u + 2 * n_z] = J.sc0->uh; dst[2 * n_u + 2 * n_z + 1] = J.sc0->duh; }
    }
  };
  float *r1 = recs, *rn = recs + rec_n, *rp = recs + 2 * rec_n;   // levels n + 1, n and n - 1 of the step
  fetch(J.m_end, r1);
  if (J.m_end > J.m_start) fetch(J.m_end - 1, rn);
  wait_copies();
  __syncthreads();

  int steps = 0, steps_two = 0;   // steps whose solutions NZ, XZ hold in a row
  float dy_next = J.m_end > J.m_start ? J.dy[J.m_end] : 0.f;
  for (int64_t m = J.m_end; m > J.m_start; --m) {
    const int64_t n = m - 1;
    const float dy_m = dy_next;
    if (n > J.m_start) { fetch(n - 1, rp); dy_next = J.dy[n]; }   // used by the next step
    if (mod_kind != 0) {   // the step n -> n + 1 as the forward took it
      const float rm = mod_factor(mod_kind, Dp->mod_inc_fx, Dp->mod_phase_fx, Dp->mod_depth2, Dp->mod_inc,
                                  Dp->mod_hold, Dp->mod_n_end, n);
      const float l2 = lam2_0f * rm;
      lam2 = static_cast<R>(l2) + static_cast<R>(fmaf(lam2_0f, rm, -l2) + lam2lo_0f * rm);
      lam2l = static_cast<R>(lam2l_0f * rm);
      ca = static_cast<R>(ca_0f * rm);
      cb = static_cast<R>(cb_0f * rm);
      cz = static_cast<R>(cz_0f * rm);
      rmd = static_cast<R>(rm);
    }
    add_output(dy_m, false);
    const float *U = rn, *DU = rn + n_u, *Z = rn + 2 * n_u, *DZ = Z + n_z, *DN1 = r1 + n_u, *DZN1 = r1 + 2 * n_u + n_z;
    const float uh = rn[2 * n_u + 2 * n_z], dh = rn[2 * n_u + 2 * n_z + 1];
    const float uh1 = r1[2 * n_u + 2 * n_z], dh1 = r1[2 * n_u + 2 * n_z + 1];
    auto zr = [&](const float* F, int z) { return z >= 0 && z < n_z ? F[z] : 0.f; };
    const float ui = act ? U[i] : 0.f, um = i > 0 && i <= n_u ? U[i - 1] : 0.f, up = i < n_u - 1 ? U[i + 1] : 0.f;
    const float gl = i <= n_u ? ui - um : 0.f, gr = act ? up - ui : 0.f;   // intervals i and i + 1
    if (act) A[i] = DN1[i] - DU[i];
#pragma unroll 1
    for (int z = tid; z < n_z; z += T) AZ[z] = DZN1[z] - DZ[z];
    const R s_h = -hM * (static_cast<R>(dh1) - dh);   // hammer force of the step (k^2-scaled)
    // Z at rows i - 1 and i (the nearest floats, as the forward read them)
    float zt0 = 0.f, zt1 = 0.f;
    if (has_z) {
      auto zt = [&](int q) { return (w1m[q] * zr(Z, mm[q] - 1) + wm[q] * zr(Z, mm[q])).hi; };
      zt0 = i <= n_u && i > 0 ? zt(0) : 0.f;
      zt1 = act ? zt(1) : 0.f;
    }
    if (!linear || m == J.m_end) assemble(gl, gr);   // (a linear string's matrix is constant)
    else __syncthreads();
    R eta = 0.0f, k2G = 0.0f;
    if (hammer) {
      const float ua = en >= 1 ? U[en - 1] : 0.f, ub = en < n_u ? U[en] : 0.f;
      eta = static_cast<R>(uh) - ((1.0f - ew) * ua + ew * ub);
    }
    // ---- transposed solve ----
    const R mus = hammer ? -(ldh + luh) / hM : 0.0f;
    const bool bow_on = bow && n < brel && bF > 0.0f;
    const bool contact = hammer && eta > 0.0f, two = contact || bow_on;
    const R vb = uh1;
    // (FP64 functions, in contact or while bowing: one warp's work, since the
    // SM's FP64 rate is a 74th of its FP32 rate)
    if (warp == 0 && two) {
      const double f = contact ? pow(to_double(eta), to_double(hexpo))
                               : exp(-to_double(ba) * ::fabs(static_cast<double>(uh1)));
      if (lane == 0) put(&scal, df_from_double(f));
    }
    const R zsc = has_z ? cz / cb : 0.0f;
#pragma unroll 1
    // (the warm starts move on linearly with the last two steps)
    for (int z = tid; z < n_z; z += T) {
      put(RZ + z, zsc * (get(LDZ + z) + get(LZ + z)));
      const R f = get(NZ + z);
      if (steps > 1) put(NZ + z, f + (f - get(NZP + z)));
      put(NZP + z, f);
      if (two) {
        const R h = get(XZ + z);
        if (steps_two > 1) put(XZ + z, h + (h - get(XZP + z)));
        put(XZP + z, h);
      }
    }
    ++steps;
    steps_two = two ? steps_two + 1 : 0;
    R rj = 0.0f;
    if (i == en - 1) rj += (1.0f - ew) * js;
    if (i == en) rj += ew * js;
    if (!act) rj = 0.0f;
    R x = 0.0f, y = 0.0f;
    __syncthreads();
    coupled(act ? LD + LU : R(0.0f), rj, gl, gr, x, y, two);
    R nus = mus;
    R phid = 0.0f;
    if (contact) k2G = hk2w * get(&scal);
    if (bow_on) phid = -ba * (1.0f - beps) * get(&scal);
    if (two) {
      const R ia = (1.0f - ew) * get(X + en - 1) + ew * get(X + en);
      const R ix = (1.0f - ew) * get(XP + en - 1) + ew * get(XP + en);
      R st;
      if (contact && !(k2G > 0.0f)) {   // (eta underflowed)
        st = 0.0f;
      } else if (contact) {
        const R rs = -(hM * k2G / (2.0f * js)) * mus, cm = 0.5f * hM * k2G;
        st = (rs - cm * ia) / (1.0f + 0.5f * k2G + cm * ix);
        nus = -(2.0f * js / (hM * k2G)) * st;
      } else if (vb == 0.0f) {   // sticking: I nu_a = 0
        st = -ia / ix;
        nus = 2.0f * kk * js * st;
      } else {                   // sliding
        const R bj = 0.5f * kk * bF * phid;
        st = -bj * ia / (1.0f + bj * ix);
        nus = -js * (ia + st * ix);
      }
      __syncthreads();   // every thread has read X at the force
      x = fma(st, y, x);
      if (act) put(X + i, x);
#pragma unroll 1
      for (int z = tid; z < n_z; z += T) put(NZ + z, fma(st, get(XZ + z), get(NZ + z)));
      __syncthreads();
    }
    // nu_z = (cb / cz) nz; the warm start of the next step keeps nz
    const R zrr = has_z ? cb / cz : 0.0f;

    // ---- (dR/dx)^T nu and (dR/dc)^T nu: interval i (left of row i) ----
    // (the coefficients of the step carry the modulation factor rm)
    auto add = [&](int slot, R v, bool scaled) { acc[slot] += scaled && mod_kind != 0 ? v * rmd : v; };
    const float ai = act ? A[i] : 0.f, am = i <= n_u ? A[i - 1] : 0.f, ap = act ? A[i + 1] : 0.f;
    const R xm = get(X + min(i, n_u) - 1), xi = act ? x : R(0.0f);
    if (i <= n_u) {
      const R psi = xi - xm, sa = static_cast<R>(ai) - am;
      R e = 0.0f, q = 0.0f, chi = 0.0f;
      if (has_z) {
        e = static_cast<R>(zt1) - zt0;
        const float a1 = act ? to_tf(AZ, 1).hi : 0.f, a0 = i > 0 ? to_tf(AZ, 0).hi : 0.f;
        q = static_cast<R>(a1) - a0;
        const R n1 = act ? to_t(NZ, 1) : R(0.0f), n0 = i > 0 ? to_t(NZ, 0) : R(0.0f);
        chi = zrr * (n1 - n0);
      }
      const R g = gl;
      // GAM in P0, PSG = psi g in P1 (read by rows i - 1 and i)
      put(P0 + i, -psi * (6.0f * ca * g * g + 4.0f * cb * e + cb * q + 2.0f * ca * g * sa) -
                      chi * (4.0f * cz * g + cz * sa));
      put(P1 + i, psi * g);
      add(kGCa, -psi * (2.0f * g * g * g + g * g * sa), true);
      add(kGCb, -psi * (4.0f * g * e + g * q), true);
      add(kGCz, -chi * (2.0f * g * g + g * sa), true);
    }
    __syncthreads();
    if (act) {
      const R xp = get(X + i + 1), xmm = get(X + i - 2), xpp = get(X + i + 2);
      const R dl = xi - xm, dr = xp - xi;
      const R d2na = dr - dl;
      R d4na = ((xpp - xp) - dr) - 2.0f * d2na + (dl - (xm - xmm));
      if (i == 0) d4na += bsgn * xi;
      if (i == n_u - 1) d4na += bsgn * xi;
      const R d2u = (static_cast<R>(up) - ui) - (static_cast<R>(ui) - um);
      const float d0 = DU[i], dm = i > 0 ? DU[i - 1] : 0.f, dp = i < n_u - 1 ? DU[i + 1] : 0.f;
      const R d2du = (static_cast<R>(dp) - d0) - (static_cast<R>(d0) - dm);
      const R d2a = (static_cast<R>(ap) - ai) - (static_cast<R>(ai) - am);
      R lun = LU + lam2 * d2na - mu2 * d4na;
      if (!linear) lun += get(P0 + i) - get(P0 + i + 1);
      LD = LD + LU - 2.0f * s0u * xi + 2.0f * s1 * d2na;
      LU = lun;
      add(kGLam2, xi * d2u, true);
      // nu . d4 u summed by parts: (d2 nu) . (d2 u) plus the ghost's corner terms
      R nd4u = d2na * d2u;
      if (i == 0 || i == n_u - 1) nd4u += (1.0f + bsgn) * xi * static_cast<R>(ui);
      add(kGMu2, -nd4u, false);
      add(kGS0u, xi * (-2.0f * static_cast<R>(d0) - static_cast<R>(ai)), false);
      add(kGS1, xi * (2.0f * d2du + d2a), false);
      if (has_z) {
        const R f = get(P1 + i + 1) - get(P1 + i);   // d_+[psi g] at the row
        put(Q0 + i, wt.left * f);
        put(Q1 + i, wt.right * f);
      }
    }
    if (has_z) {
      __syncthreads();
      zrows([&](int z, bool in) {
        const R sp = spread(Q0, Q1, in ? z : n_z - 1);
        if (!in || !zown) return;
        const R nz = zrr * get(NZ + z);
        auto d2f = [&](const float* F) {
          return (static_cast<R>(zr(F, z + 1)) - F[z]) - (static_cast<R>(F[z]) - zr(F, z - 1));
        };
        const R d2n = zrr * ((get(NZ + z + 1) - get(NZ + z)) - (get(NZ + z) - get(NZ + z - 1)));
        const R d2z = d2f(Z), d2dz = d2f(DZ), d2az = d2f(AZ);
        const R lz = get(LZ + z);
        put(LDZ + z, get(LDZ + z) + lz - 2.0f * s0 * nz + 2.0f * s1l * d2n);
        put(LZ + z, lz + lam2l * d2n + 4.0f * cb * sp);
        add(kGLam2l, nz * d2z, true);
        add(kGS0, nz * (-2.0f * static_cast<R>(DZ[z]) - static_cast<R>(AZ[z])), false);
        add(kGS1l, nz * (2.0f * d2dz + d2az), false);
      });
    }
    if (hammer) {
      R psi_eta = 0.0f;
      if (k2G > 0.0f) {
        const R dG = hexpo * k2G / eta;
        const R ia = (1.0f - ew) * (en >= 1 ? A[en - 1] : 0.f) + ew * (en < n_u ? A[en] : 0.f);
        psi_eta = nus * (hM * k2G + (hM * eta - 0.5f * hM * ia - 0.5f * s_h) * dG);
        if (act && i == en - 1) LU -= psi_eta * (1.0f - ew);
        if (act && i == en) LU -= psi_eta * ew;
      }
      ldh = ldh + luh;
      luh = luh + psi_eta;
    }
    if (bow_on) {
      // (dR3/dD)^T nu_s and dR3/dv_B (the amplitude slot of a bowed string)
      const R cd = vb == 0.0f ? 1.0f / kk : kk * bF * phid;
      if (act && i == en - 1) LD += cd * (1.0f - ew) * nus;
      if (act && i == en) LD += cd * ew * nus;
      if (tid == 0) add(kGAmp, vb == 0.0f ? -nus : -kk * kk * bF * phid * nus, false);
    }
    wait_copies();      // the level of the next step is in shared memory
    __syncthreads();
    { float* t = r1; r1 = rn; rn = rp; rp = t; }
  }

  if (J.first) {
    // level 1 output, level 0 output y^0 = L I(u^1 - D^1), initial-state terms
    add_output(J.dy[1], false);
    add_output(J.dy[0], true);
    R pa = 0.0f;
    if (J.pluck_pos >= 0.f) {   // u^0 = u^1 = c0 tri(x), D^1 = 0
      const R xp = J.pluck_pos, x = static_cast<R>(i + 1) * (1.0f / static_cast<R>(n_t));
      if (act) pa = LU * (x <= xp ? x / xp : (1.0f - x) / (1.0f - xp));
    } else if (hammer && tid == 0) {   // u_H^1 = D_H^1 = v k
      pa = static_cast<R>(Dp->k) * (luh + ldh);
    }
    acc[kGAmp] += pa;
  }

  // ---- store the adjoint state, the warm starts and the gradients ----
  __syncthreads();
  if (act) { adj[i] = to_double(LU); adj[n_u + i] = to_double(LD); }
#pragma unroll 1
  for (int z = tid; z < n_z; z += T) {
    adj[2 * n_u + z] = to_double(get(LZ + z));
    adj[2 * n_u + n_z + z] = to_double(get(LDZ + z));
    adj[2 * n_u + 2 * n_z + 2 + z] = to_double(get(NZ + z));
    adj[2 * n_u + 3 * n_z + 2 + z] = to_double(get(XZ + z));
  }
  if (tid == 0) { adj[2 * n_u + 2 * n_z] = to_double(luh); adj[2 * n_u + 2 * n_z + 1] = to_double(ldh); }
#pragma unroll
  for (int k = 0; k < kGradSlots; ++k) {
    R v = acc[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += shfl_xor(v, o);
    if (lane == 0) put(&gsum[warp][k], v);
  }
  __syncthreads();
  if (tid < kGradSlots) {
    R v = get(&gsum[0][tid]);
#pragma unroll 1
    for (int w = 1; w < n_warps; ++w) v += get(&gsum[w][tid]);
    J.grad[tid] += to_double(v);
  }
}

namespace {
// (as for the other kernels: raised once per device, never lowered)
std::mutex g_rows_mu;
bool g_rows_done[64] = {};
}  // namespace

cudaError_t adjoint_rows_static_smem(size_t* bytes) {
  cudaFuncAttributes fa;
  const cudaError_t e = cudaFuncGetAttributes(&fa, adjoint_rows_kernel);
  if (e == cudaSuccess) *bytes = fa.sharedSizeBytes;
  return e;
}

// One block per job, `threads` of them (a multiple of 32, more than any
// job's transverse rows).
cudaError_t launch_adjoint_rows(const AdjJob* d_jobs, int n_jobs, int threads, int smem_bytes, cudaStream_t stream) {
  if (n_jobs <= 0) return cudaSuccess;
  if (threads < kWarp || threads > kThreads || threads % kWarp) return cudaErrorInvalidValue;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  {
    std::lock_guard<std::mutex> lock(g_rows_mu);
    if (!g_rows_done[dev]) {
      int optin = 0;
      size_t fixed = 0;
      if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
      if ((e = adjoint_rows_static_smem(&fixed)) != cudaSuccess) return e;
      e = cudaFuncSetAttribute(adjoint_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               optin - static_cast<int>(fixed));
      if (e != cudaSuccess) return e;
      e = cudaFuncSetAttribute(adjoint_rows_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, kSmemCarveout);
      if (e != cudaSuccess) return e;
      g_rows_done[dev] = true;
    }
  }
  adjoint_rows_kernel<<<n_jobs, threads, static_cast<size_t>(smem_bytes), stream>>>(d_jobs);
  return cudaGetLastError();
}

}  // namespace sfd
