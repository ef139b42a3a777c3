// Register-blocked tile sweep (see qsweep.h for the descriptor).
//
// One CTA evolves tiles of 2^T amplitudes of one state through every op of the
// sweep:
//   1. the tile is copied from HBM into shared memory with 16-byte cp.async
//      copies (chunk c of the tile lands at the swizzled chunk swz(c));
//   2. each thread reads its 2^B rows for the first register layout into
//      registers and applies the ops: a factor whose flips lie in the
//      register bits touches only registers; a LAYOUT op writes the rows back
//      and reads them again for the next set of register bits;
//   3. the rows go straight from registers to HBM in the last layout.
// With T = 13 and B = 5 the tile is 64 KiB, the CTA has 256 threads, and a
// step of the 24-qubit MaxCut instance (24 factors) takes one sweep.
//
// What bounds it: HBM (2 * s * N * R bytes per sweep) for few ops per
// amplitude, the FP32 pipe and the shared-memory path of the layout changes
// for many.  A MaxCut sweep over 22 qubits and 16 states moves 1.01 GB at 2.4
// TB/s with its issue slots 45% busy; per instruction issued 1.8 warps wait for
// shared memory, 1.5 for a fixed latency, 0.8 for the FP32 pipe, 0.6 for the
// memory queue, 0.5 at barriers, 0.4 each for HBM and for instructions.
// Instructions came first before: the kernel is an interpreter of fully
// unrolled op bodies, and with scalar complex arithmetic, a phase body with a
// sincospi per register pattern and four store bodies 2.3 warps per issue waited
// for them (instruction-cache hit rate 78%, 24-qubit sweep 2.09 ms).  So the
// executed footprint is kept small: complex64 rows are held as pairs
// (re0, re1), (im0, im1) of the two rows that differ in register bit 0, and
// every op works on pairs with the two-element FP32 instructions (half the
// instructions of the scalar form for the same operations), and the phase
// factors are produced by one loop with one sincospi.  On the 24-qubit MaxCut
// instance with 16 states a sweep went from 2.09 to 1.46 ms; a periodic
// 22-qubit Heisenberg chain with 2 states (BOND ops) from 3.85 to 1.67 ms for
// 20 steps.  Registers matter as much: the tiles leave little L1, so a spilled
// register costs an L2 round trip (52 local loads per warp and tile made the
// 1.51 ms sweep a 6.2 ms one).
//
// PHASE ops generate a diagonal run's values from (z_j, theta_j): with the
// tile's fixed bits folded in, phi(r) = C0 + sum_m C_m chi_m(l), where m runs
// over the distinct local parts of the z_j, chi_m(l) = (-1)^popcount(m & l)
// and C_m sums +-theta_j (units of pi, once per tile).  A thread's rows differ
// only in their register bits, so phi over its 2^B rows is the Walsh-Hadamard
// transform of the per-thread coefficients E[mu] = sum over classes with
// register part mu of +-C_m; each row takes a product of exp(-+ i pi E[mu]).
// They do not depend on the state: a CTA runs up to kMaxRhsChunk states of a
// tile back to back and computes them for the first one only.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <mutex>
#include <type_traits>

#include "counters.h"
#include "hs_internal.h"
#include "qsweep.h"
#include "sweep_core.cuh"

namespace hs {
namespace q {
namespace {

using sweep::C2;
using sweep::cp_async16;
using sweep::cp_async_commit;
using sweep::cp_async_wait;
using sweep::deposit_runs;
using sweep::global_of;
using sweep::grid_dependency_wait;
using sweep::grid_launch_dependents;
using sweep::pattern_fast;

__device__ __forceinline__ int parity(uint32_t v) { return __popc(v) & 1; }

__host__ __device__ constexpr int highest_bit(int v) {
  int h = 0;
  while (v >> (h + 1)) ++h;
  return v ? (1 << h) : 0;
}

// (re, im) * (bx, by).
template <typename T2, typename R>
__device__ __forceinline__ T2 cmul(T2 a, R bx, R by) {
  return T2{fma(a.x, bx, -a.y * by), fma(a.x, by, a.y * bx)};
}

// v with its sign flipped where the lowest bit of s is set.
__device__ __forceinline__ float flip_sign(float v, uint32_t s) {
  return __uint_as_float(__float_as_uint(v) ^ (s << 31));
}
__device__ __forceinline__ double flip_sign(double v, uint32_t s) { return (s & 1u) ? -v : v; }

// ---------------------------------------------------------------------------
// A thread's 2^B rows.  complex64: rows 2j and 2j + 1 share the pairs re[j]
// and im[j]; complex128: row by row.
// ---------------------------------------------------------------------------
template <typename R, int B>
struct Rows;

template <int B>
struct Rows<float, B> {
  static constexpr int NP = 1 << (B - 1);
  float2 re[NP], im[NP];
  __device__ __forceinline__ float2 get(int k) const {
    return (k & 1) ? make_float2(re[k >> 1].y, im[k >> 1].y) : make_float2(re[k >> 1].x, im[k >> 1].x);
  }
  __device__ __forceinline__ void set(int k, float2 v) {
    if (k & 1) {
      re[k >> 1].y = v.x;
      im[k >> 1].y = v.y;
    } else {
      re[k >> 1].x = v.x;
      im[k >> 1].x = v.y;
    }
  }
};

template <int B>
struct Rows<double, B> {
  double2 x[1 << B];
  __device__ __forceinline__ double2 get(int k) const { return x[k]; }
  __device__ __forceinline__ void set(int k, double2 v) { x[k] = v; }
};

__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 neg2(float2 v) { return make_float2(-v.x, -v.y); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// ---------------------------------------------------------------------------
// ROT: x <- (cos I - i sin P_j) x for one term whose flips are the register
// coordinates KU.  Row k's partner is k ^ KU; the off-diagonal coefficient of
// row k is sin * i^q * (-1)^popcount(z & r_{k ^ KU}), r_k the global row.
//
// A term with y = 0 and z = 0 (P = X on the flipped qubits) takes the factor
// build's split exp(-i theta P) = cos(theta') (I - i t P) (-i P)^k, t =
// tan(theta'), |theta'| <= pi / 4: rot_tan applies I - i t P with two fused
// multiply-adds per amplitude, cos(theta') and (-i)^k go into the sweep's
// scale, and an odd k swaps the partner rows (flip_pairs) at the end of the
// op, so the rotation itself has no data-dependent branch.
// ---------------------------------------------------------------------------
template <int KU, int B>
__device__ __forceinline__ void rot_tan(Rows<float, B>& x, float t) {
  constexpr int NP = Rows<float, B>::NP;
  constexpr int JU = KU >> 1, HB = highest_bit(JU);
  if constexpr ((KU & 1) == 0) {
    const float2 tp = dup(t), tn = dup(-t);
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      if (j & HB) continue;
      const int j2 = j ^ JU;
      const float2 r1 = x.re[j], m1 = x.im[j], r2 = x.re[j2], m2 = x.im[j2];
      x.re[j] = fma2(tp, m2, r1);
      x.im[j] = fma2(tn, r2, m1);
      x.re[j2] = fma2(tp, m1, r2);
      x.im[j2] = fma2(tn, r1, m2);
    }
  } else {
    // The partner sits in the other half of a pair.
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      if (j & HB) continue;
      const int j2 = j ^ JU;
      const float2 r1 = x.re[j], m1 = x.im[j], r2 = x.re[j2], m2 = x.im[j2];
      x.re[j] = make_float2(fmaf(t, m2.y, r1.x), fmaf(t, m2.x, r1.y));
      x.im[j] = make_float2(fmaf(-t, r2.y, m1.x), fmaf(-t, r2.x, m1.y));
      if constexpr (JU != 0) {
        x.re[j2] = make_float2(fmaf(t, m1.y, r2.x), fmaf(t, m1.x, r2.y));
        x.im[j2] = make_float2(fmaf(-t, r1.y, m2.x), fmaf(-t, r1.x, m2.y));
      }
    }
  }
}

template <int KU, int B>
__device__ __forceinline__ void rot_tan(Rows<double, B>& x, double t) {
  constexpr int HB = highest_bit(KU);
#pragma unroll
  for (int k = 0; k < (1 << B); ++k) {
    if (k & HB) continue;
    const int k2 = k ^ KU;
    const double2 b1 = x.x[k], b2 = x.x[k2];
    x.x[k] = make_double2(fma(t, b2.y, b1.x), fma(-t, b2.x, b1.y));
    x.x[k2] = make_double2(fma(t, b1.y, b2.x), fma(-t, b1.x, b2.y));
  }
}

template <typename R, int KU, int B>
__device__ __forceinline__ void flip_pairs(Rows<R, B>& x) {
  constexpr int HB = highest_bit(KU);
#pragma unroll
  for (int k = 0; k < (1 << B); ++k) {
    if (k & HB) continue;
    const auto b = x.get(k);
    x.set(k, x.get(k ^ KU));
    x.set(k ^ KU, b);
  }
}

template <typename R, int KU, int B>
__device__ __forceinline__ void rot_ku(Rows<R, B>& x, R c, R s, bool fast, int q, uint32_t zk, int sb, bool flip) {
  using T2 = typename C2<R>::T;
  constexpr int HB = highest_bit(KU);
  if (fast) {
    rot_tan<KU>(x, c);
    if (flip) flip_pairs<R, KU>(x);
    return;
  }
  // (i^q s as one component, real or imaginary; a row's sign from z's bits by
  // XOR with one mask per bit, so that no table of signs fills the registers)
  const bool imag = q & 1;
  uint32_t zm[B];
#pragma unroll
  for (int i = 0; i < B; ++i) zm[i] = (zk >> i) & 1u;
  const R s0 = flip_sign(s, uint32_t(sb) ^ uint32_t(q >> 1));
  auto coef = [&](int k) {  // of a row whose partner is row k
    uint32_t p = 0;
#pragma unroll
    for (int i = 0; i < B; ++i)
      if ((k >> i) & 1) p ^= zm[i];
    return flip_sign(s0, p);
  };
#pragma unroll
  for (int k = 0; k < (1 << B); ++k) {
    if (k & HB) continue;
    const int k2 = k ^ KU;
    const T2 b1 = x.get(k), b2 = x.get(k2);
    const R c1 = coef(k2), c2 = coef(k);
    // (x, y) i = (-y, x)
    const R u1 = imag ? -b2.y : b2.x, v1 = imag ? b2.x : b2.y, u2 = imag ? -b1.y : b1.x, v2 = imag ? b1.x : b1.y;
    x.set(k, T2{fma(c1, u1, c * b1.x), fma(c1, v1, c * b1.y)});
    x.set(k2, T2{fma(c2, u2, c * b2.x), fma(c2, v2, c * b2.y)});
  }
}

// ---------------------------------------------------------------------------
// BOND: rows (.., 0 1, ..) and (.., 1 0, ..) on the two register bits of KU
// become a + w (b - a) and b - w (b - a); the other rows stay.
// ---------------------------------------------------------------------------
template <typename R, int KU, int B>
__device__ __forceinline__ void bond_rows(Rows<R, B>& x, typename C2<R>::T w) {
  using T2 = typename C2<R>::T;
  constexpr int HB = highest_bit(KU), LB = KU ^ HB;
  if constexpr (sizeof(R) == 4 && (KU & 1) == 0) {
    constexpr int NP = 1 << (B - 1);
    const float2 wx = dup(w.x), wy = dup(w.y), nx = dup(-w.x), ny = dup(-w.y), m1 = dup(-1.0f);
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      if ((j & (HB >> 1)) || !(j & (LB >> 1))) continue;
      const int j2 = j ^ (KU >> 1);
      const float2 dr = fma2(m1, x.re[j], x.re[j2]), di = fma2(m1, x.im[j], x.im[j2]);
      x.re[j] = fma2(wx, dr, fma2(ny, di, x.re[j]));
      x.im[j] = fma2(wx, di, fma2(wy, dr, x.im[j]));
      x.re[j2] = fma2(nx, dr, fma2(wy, di, x.re[j2]));
      x.im[j2] = fma2(nx, di, fma2(ny, dr, x.im[j2]));
    }
  } else {
#pragma unroll
    for (int k = 0; k < (1 << B); ++k) {
      if ((k & HB) || !(k & LB)) continue;
      const T2 a = x.get(k), b = x.get(k ^ KU);
      const R dx = b.x - a.x, dy = b.y - a.y;
      x.set(k, T2{fma(w.x, dx, fma(-w.y, dy, a.x)), fma(w.x, dy, fma(w.y, dx, a.y))});
      x.set(k ^ KU, T2{fma(-w.x, dx, fma(w.y, dy, b.x)), fma(-w.x, dy, fma(-w.y, dx, b.y))});
    }
  }
}

// ---------------------------------------------------------------------------
// TAB: x[k] <- v(p_k, 0) x[k] + v(p_k, 1) x[k ^ KU] with p_k the pattern of
// row k's global index at the factor's support (p_k = pt ^ XOR of pr[i] over
// the set bits i of k: the pattern map is linear over XOR).
// ---------------------------------------------------------------------------
template <typename R, int B, int KU>
__device__ __forceinline__ void tab_ku(Rows<R, B>& x, const typename C2<R>::T* tb, int ns, uint32_t pt,
                                       const uint32_t (&pr)[B]) {
  using T2 = typename C2<R>::T;
  constexpr int NR = 1 << B;
  constexpr int HB = KU ? highest_bit(KU) : 0;
  // Pattern of register row k: pt ^ XOR of pr[i] over the set bits i of k.
  auto pat = [&](int k) {
    uint32_t p = pt;
#pragma unroll
    for (int i = 0; i < B; ++i)
      if ((k >> i) & 1) p ^= pr[i];
    return p;
  };
  if constexpr (KU == 0) {
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      const T2 v0 = tb[pat(k) * uint32_t(ns)];
      x.set(k, cmul<T2, R>(x.get(k), v0.x, v0.y));
    }
  } else {
    // Two slots: a row's entries (r, r) and (r, r ^ u) sit side by side in the
    // table, one 2 * sizeof(T2)-byte load.
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      if (k & HB) continue;
      const int k2 = k ^ KU;
      T2 a0, a1, c0, c1;
      if constexpr (sizeof(T2) == 8) {
        const float4 va = *reinterpret_cast<const float4*>(tb + pat(k) * 2u);
        const float4 vc = *reinterpret_cast<const float4*>(tb + pat(k2) * 2u);
        a0 = T2{va.x, va.y};
        a1 = T2{va.z, va.w};
        c0 = T2{vc.x, vc.y};
        c1 = T2{vc.z, vc.w};
      } else {
        const T2* va = tb + pat(k) * 2u;
        const T2* vc = tb + pat(k2) * 2u;
        a0 = va[0];
        a1 = va[1];
        c0 = vc[0];
        c1 = vc[1];
      }
      const T2 b1 = x.get(k), b2 = x.get(k2);
      T2 r1, r2;
      r1.x = fma(a0.x, b1.x, fma(-a0.y, b1.y, fma(a1.x, b2.x, -a1.y * b2.y)));
      r1.y = fma(a0.x, b1.y, fma(a0.y, b1.x, fma(a1.x, b2.y, a1.y * b2.x)));
      r2.x = fma(c0.x, b2.x, fma(-c0.y, b2.y, fma(c1.x, b1.x, -c1.y * b1.y)));
      r2.y = fma(c0.x, b2.y, fma(c0.y, b2.x, fma(c1.x, b1.y, c1.y * b1.x)));
      x.set(k, r1);
      x.set(k2, r2);
      // (keeps the loads of later rows below: hoisted, they take more registers
      // than there are)
      asm volatile("" ::: "memory");
    }
  }
}

// ROTN: commuting X rotations on distinct single register bits (tan form, see
// ROT), the slot of register bit i in byte i of (zthr, zrest).  The rows of
// one rotation change register in pairs, so a body that ends in a branch pays
// a move per row; the run over all bits above bit 0 (a full layout of single
// flips) is therefore one straight-line body (24-qubit MaxCut: 87.5 ms with a
// branch per bit).  The odd-k swaps follow the whole run (every factor of the
// run is a function of its own X, so they commute).
template <typename R, int B, int I, bool ALL>
__device__ __forceinline__ void rotn_bits(Rows<R, B>& x, uint32_t ku, const R (&t)[5]) {
  if constexpr (I < B) {
    if (ALL || ((ku >> I) & 1)) rot_tan<(1 << I)>(x, t[I]);
    rotn_bits<R, B, I + 1, ALL>(x, ku, t);
  }
}

template <typename R, int B>
__device__ __forceinline__ void rotn(Rows<R, B>& x, uint32_t ku, const R (&t)[5]) {
  constexpr uint32_t kUpper = ((1u << B) - 1u) & ~1u;
  if (sizeof(R) == 4 && (ku & kUpper) == kUpper) {
    if (ku & 1u) rot_tan<1>(x, t[0]);
    rotn_bits<R, B, 1, true>(x, ku, t);
  } else {
    rotn_bits<R, B, 0, false>(x, ku, t);
  }
}

template <typename R, int B, int I>
__device__ __forceinline__ void flip_run(Rows<R, B>& x, uint32_t fl) {
  if constexpr (I < B) {
    if ((fl >> I) & 1) flip_pairs<R, (1 << I)>(x);
    flip_run<R, B, I + 1>(x, fl);
  }
}

// DROT: x[k] <- (cos - i sin (-1)^popcount(z & r_k)) x[k], the rotation of one
// diagonal term; sb is the parity of z over the row's fixed bits.
template <typename R, int B>
__device__ __forceinline__ void diag_rot(Rows<R, B>& x, R c, R s, uint32_t zk, int sb) {
  using T2 = typename C2<R>::T;
#pragma unroll
  for (int k = 0; k < (1 << B); ++k) {
    const R ss = (sb ^ parity(zk & uint32_t(k))) ? -s : s;
    const T2 v = x.get(k);
    x.set(k, T2{fma(ss, v.y, c * v.x), fma(-ss, v.x, c * v.y)});
  }
}

// Register flips the planner may emit: one or two register bits.
#define HS_Q_KU2_LIST(X) X(3) X(5) X(6) X(9) X(10) X(12) X(17) X(18) X(20) X(24)
#define HS_Q_KU_LIST(X) X(1) X(2) X(4) X(8) X(16) HS_Q_KU2_LIST(X)

template <typename R, int B>
__device__ __forceinline__ void rot_dispatch(Rows<R, B>& x, int ku, R c, R s, bool fast, int q, uint32_t zk, int sb,
                                             bool flip) {
  switch (ku) {
#define HS_Q_ROT_CASE(K) \
  case K:                \
    if constexpr (K < (1 << B)) rot_ku<R, K>(x, c, s, fast, q, zk, sb, flip); \
    break;
    HS_Q_KU_LIST(HS_Q_ROT_CASE)
#undef HS_Q_ROT_CASE
    default: break;
  }
}

template <typename R, int B>
__device__ __forceinline__ void tan_dispatch(Rows<R, B>& x, int ku, R t, bool flip) {
  switch (ku) {
#define HS_Q_TAN_CASE(K)                \
  case K:                               \
    if constexpr (K < (1 << B)) {       \
      rot_tan<K>(x, t);                 \
      if (flip) flip_pairs<R, K>(x);    \
    }                                   \
    break;
    HS_Q_KU_LIST(HS_Q_TAN_CASE)
#undef HS_Q_TAN_CASE
    default: break;
  }
}

template <typename R, int B>
__device__ __forceinline__ void bond_dispatch(Rows<R, B>& x, int ku, typename C2<R>::T w) {
  switch (ku) {
#define HS_Q_BOND_CASE(K) \
  case K:                 \
    if constexpr (K < (1 << B)) bond_rows<R, K>(x, w); \
    break;
    HS_Q_KU2_LIST(HS_Q_BOND_CASE)
#undef HS_Q_BOND_CASE
    default: break;
  }
}

template <typename R, int B>
__device__ __forceinline__ void tab_dispatch(Rows<R, B>& x, int ku, const typename C2<R>::T* tb, int ns, uint32_t pt,
                                             const uint32_t (&pr)[B]) {
  switch (ku) {
    case 0: tab_ku<R, B, 0>(x, tb, ns, pt, pr); break;
#define HS_Q_TAB_CASE(K) \
  case K:                \
    if constexpr (K < (1 << B)) tab_ku<R, B, K>(x, tb, ns, pt, pr); \
    break;
    HS_Q_KU_LIST(HS_Q_TAB_CASE)
#undef HS_Q_TAB_CASE
    default: break;
  }
}

// ---------------------------------------------------------------------------
// PHASE: x[k] <- exp(-i phi(r_k)) x[k].  With the tile's fixed bits folded
// into the per-tile class constants (units of pi) and the thread's bits into
// E[mu] = sum over the classes with register part mu of +-C_c, the phase of
// register row k is e0 * prod_mu exp(-i pi E[mu] chi_mu(k)), chi_mu(k) =
// (-1)^popcount(mu & k).  The factors of mu = 0 and of the single register
// bits are multiplied out in two small groups of bits (all rows' values from a
// few products), with the patterns of two or more bits inside a group; a
// pattern across the groups multiplies every row.
//
// A thread's factors go through its own slots of shared memory: slot 0 the
// product of e0 and mu = 0, slots 1 .. B (cos, sin) of the single register
// bits, then one (cos, sin) per pattern inside a group and per pattern across
// the groups, ascending (Args::fac_keep; otherwise those across take turns in
// one slot).  One sincospi per slot, not per row, in one loop.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void sincospi_r(float x, float* s, float* c) { sincospif(x, s, c); }
__device__ __forceinline__ void sincospi_r(double x, double* s, double* c) { sincospi(x, s, c); }

template <typename R>
struct ClassC {
  R c;           // the class constant of the tile
  uint32_t thr;  // local part on thread positions
};

template <typename R>
__device__ __forceinline__ void phase_factor(const Phase& P, const ClassC<R>* cw, int mu, uint32_t lt, R* sn, R* cn) {
  R e = R(0);
  const int c1 = P.cls0 + P.mu_beg[mu + 1];
#pragma unroll 1
  for (int cc = P.cls0 + P.mu_beg[mu]; cc < c1; ++cc) {
    const ClassC<R> C = cw[cc];
    e += flip_sign(C.c, uint32_t(__popc(C.thr & lt)));
  }
  sincospi_r(e, sn, cn);
}

// A[k], k over N register bits, from A[0] and the bits' (cos, sin) in the slots
// at cs (read one at a time: few registers are left beside the rows): f_i(0) =
// cos - i sin, f_i(1) = cos + i sin; then the patterns (in coordinates of the
// N bits) listed in `pats`, from the slots at `f`.
template <typename T2, typename R, int N>
__device__ __forceinline__ void group_values(T2 (&A)[1 << N], const T2* cs, uint32_t pats, const T2*& f, int nt) {
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const T2 c = cs[i * nt];
#pragma unroll
    for (int k = 0; k < (1 << i); ++k) {
      const T2 p = A[k];
      const R ac = p.x * c.x, bs = p.y * c.y, bc = p.y * c.x, as = p.x * c.y;
      A[k] = T2{ac + bs, bc - as};
      A[k + (1 << i)] = T2{ac - bs, bc + as};
    }
  }
#pragma unroll 1
  for (uint32_t r = pats; r; r &= r - 1u, f += nt) {
    const int mu = __ffs(r) - 1;
    const T2 v = *f;
#pragma unroll
    for (int k = 0; k < (1 << N); ++k) A[k] = cmul<T2, R>(A[k], v.x, parity(uint32_t(mu) & uint32_t(k)) ? v.y : -v.y);
  }
}

// Register bits 0 .. B1 - 1 form the lower group, the others the upper one.
__host__ __device__ constexpr int lower_bits(int B) { return (B + 1) / 2; }

template <int B>
__device__ __forceinline__ void phase_apply(Rows<float, B>& x, uint32_t mu_mask, const float2* fac, int nt) {
  constexpr int B1 = lower_bits(B), B2 = B - B1;
  const float2* f = fac + (1 + B) * nt;
  {
    float2 A[1 << B1];
    A[0] = fac[0];
    group_values<float2, float, B1>(A, fac + nt, lower_patterns<B>(mu_mask), f, nt);
#pragma unroll
    for (int a = 0; a < (1 << (B1 - 1)); ++a) {
      const float2 c = make_float2(A[2 * a].x, A[2 * a + 1].x), s = make_float2(A[2 * a].y, A[2 * a + 1].y), ns = neg2(s);
#pragma unroll
      for (int b = 0; b < (1 << B2); ++b) {
        const int j = a + (b << (B1 - 1));
        const float2 r = x.re[j], m = x.im[j];
        x.re[j] = fma2(r, c, __fmul2_rn(m, ns));
        x.im[j] = fma2(r, s, __fmul2_rn(m, c));
      }
    }
  }
  {
    float2 A[1 << B2];
    A[0] = make_float2(1.0f, 0.0f);
    group_values<float2, float, B2>(A, fac + (1 + B1) * nt, upper_patterns<B>(mu_mask), f, nt);
#pragma unroll
    for (int b = 0; b < (1 << B2); ++b) {
      const float2 c = dup(A[b].x), s = dup(A[b].y), ns = dup(-A[b].y);
#pragma unroll
      for (int a = 0; a < (1 << (B1 - 1)); ++a) {
        const int j = a + (b << (B1 - 1));
        const float2 r = x.re[j], m = x.im[j];
        x.re[j] = fma2(r, c, __fmul2_rn(m, ns));
        x.im[j] = fma2(r, s, __fmul2_rn(m, c));
      }
    }
  }
}

template <int B>
__device__ __forceinline__ void pattern_apply(Rows<float, B>& x, int mu, float2 v) {
  constexpr int NP = 1 << (B - 1);
  const float2 c = dup(v.x);
  // row 2j + h takes cos - i sin (-1)^popcount(mu & (2j + h))
  const float2 s0 = make_float2(v.y, flip_sign(v.y, uint32_t(mu)));
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    const uint32_t sg = uint32_t(__popc(mu & (2 * j)));
    const float2 s = make_float2(flip_sign(s0.x, sg), flip_sign(s0.y, sg)), ns = neg2(s);
    const float2 r = x.re[j], m = x.im[j];
    x.re[j] = fma2(r, c, __fmul2_rn(m, s));
    x.im[j] = fma2(r, ns, __fmul2_rn(m, c));
  }
}

template <int B>
__device__ __forceinline__ void phase_apply(Rows<double, B>& x, uint32_t mu_mask, const double2* fac, int nt) {
  constexpr int B1 = lower_bits(B), B2 = B - B1;
  const double2* f = fac + (1 + B) * nt;
  double2 A[1 << B1], C[1 << B2];
  A[0] = fac[0];
  group_values<double2, double, B1>(A, fac + nt, lower_patterns<B>(mu_mask), f, nt);
  C[0] = make_double2(1.0, 0.0);
  group_values<double2, double, B2>(C, fac + (1 + B1) * nt, upper_patterns<B>(mu_mask), f, nt);
#pragma unroll
  for (int k = 0; k < (1 << B); ++k) x.x[k] = cmul<double2, double>(x.x[k], A[k & ((1 << B1) - 1)].x, A[k & ((1 << B1) - 1)].y);
#pragma unroll
  for (int k = 0; k < (1 << B); ++k) x.x[k] = cmul<double2, double>(x.x[k], C[k >> B1].x, C[k >> B1].y);
}

template <int B>
__device__ __forceinline__ void pattern_apply(Rows<double, B>& x, int mu, double2 v) {
#pragma unroll
  for (int k = 0; k < (1 << B); ++k) x.x[k] = cmul<double2, double>(x.x[k], v.x, parity(mu & k) ? v.y : -v.y);
}

// The whole op; `fresh`: the factors are not in the slots yet.
template <typename R, int B>
__device__ __forceinline__ void phase_op(Rows<R, B>& x, const Phase& P, const ClassC<R>* cw, typename C2<R>::T e0,
                                         uint32_t lt, typename C2<R>::T* fac, int nt, bool fresh, bool keep) {
  using T2 = typename C2<R>::T;
  const uint32_t mu_mask = P.mu_mask;
  // Patterns in the order of their slots: inside the groups, then across.
  uint32_t inside = inside_patterns<B>(mu_mask), across = across_patterns<B>(mu_mask);
  const int n_in = B + __popc(inside);  // last slot of the first round
  int slot = 0, last = n_in, mu = 0;
#pragma unroll 1
  while (true) {
    if (fresh) {
#pragma unroll 1
      for (int k = slot; k <= last; ++k) {
        if (k <= B) {
          mu = k == 0 ? 0 : 1 << (k - 1);
        } else if (k <= n_in) {
          mu = __ffs(inside) - 1;
          inside &= inside - 1u;
        }
        R sn, cn;
        phase_factor<R>(P, cw, mu, lt, &sn, &cn);
        fac[k * nt] = mu == 0 ? cmul<T2, R>(e0, cn, -sn) : T2{cn, sn};
      }
    }
    if (slot == 0)
      phase_apply<B>(x, mu_mask, fac, nt);
    else
      pattern_apply<B>(x, mu, fac[slot * nt]);
    if (!across) break;
    mu = __ffs(across) - 1;
    across &= across - 1u;
    slot = (slot == 0 || !keep) ? n_in + 1 : slot + 1;
    last = slot;
  }
}

// ---------------------------------------------------------------------------
// Coefficients.  rec: the term records of the op (ROTN: one per register bit).
// m, kq and ph collect the sweep's scale: the product of the fast rotations'
// cos(theta') and quarter turns (-i)^k and of the bonds' phases e^{-i theta}.
// ---------------------------------------------------------------------------
struct Records {
  const double* rq;
  const double* cs;
  int n;
};

template <typename R>
__device__ __forceinline__ Coef<R> coef_of(const Op& op, const int32_t* rec, const Records& t, double& m, double& ph,
                                           int& kq, bool exact = false) {
  Coef<R> c{};
  // A fast rotation (y = 0, z = 0): tan(theta') of the factor build's record.
  auto take = [&](int e, R& v) {
    const double* q = t.rq + 4 * HS_BCHK(e, t.n, BS_REG_TERM);
    v = R(q[0]);
    m *= q[2];
    const int k = int(q[1]);
    kq += k;
    return uint32_t(k & 1);
  };
  if (op.type == OP_ROTN) {
#pragma unroll
    for (int i = 0; i < 5; ++i)
      if ((op.ku >> i) & 1) c.swap |= take(rec[i], c.v[i]) << i;
  } else if (op.type == OP_ROT && (op.flags & 1)) {
    c.swap = take(rec[0], c.v[0]);
  } else if (op.type == OP_ROT || op.type == OP_DROT) {
    const double* p = t.cs + 2 * HS_BCHK(rec[0], t.n, BS_REG_TERM);
    c.v[0] = R(p[0]);
    c.v[1] = R(p[1]);
  } else if (op.type == OP_BOND) {
    // w = (1 - e^{4 i theta}) / 2 = sin(2 theta) (sin(2 theta) - i cos(2 theta))
    const int64_t e = HS_BCHK(rec[0], t.n, BS_REG_TERM);
    const double cs = t.cs[2 * e], sn = t.cs[2 * e + 1];
    const double s2 = 2.0 * cs * sn, c2 = fma(-2.0 * sn, sn, 1.0);
    c.v[0] = R(s2 * s2);
    c.v[1] = R(-s2 * c2);
    ph += t.rq[4 * e + 3];  // theta / pi
    if constexpr (sizeof(R) == 4) {
      // The norm of what the bond stands for, whose coefficients are rounded: the
      // factor's value table (half the rows e^{-i theta}, half e^{i theta}
      // (cos 2 theta, -i sin 2 theta)), or the rotations of YY and ZZ.  Over some
      // fifty to a hundred steps that norm drifts by up to 2e-5 (5e-5 for the worst
      // chain seen); with it results are within 2e-6 to 8e-6 of those forms', without
      // it 5e-5.
      auto sq = [](double a) { return double(R(a)) * double(R(a)); };
      const double r2 = sq(cs) + sq(sn);
      if (op.flags & 1) {
        const double s2r = sq(cs * c2) + sq(sn * c2) + sq(sn * s2) + sq(cs * s2);
        m *= 1.0 + 0.5 * (0.5 * (r2 + s2r) - 1.0);
      } else if (!exact) {
        m *= r2;
      }
    }
  }
  return c;
}

__device__ __forceinline__ void sum_scale(double& m, double& ph, int& kq) {
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) {
    m *= __shfl_xor_sync(0xffffffffu, m, o);
    ph += __shfl_xor_sync(0xffffffffu, ph, o);
    kq += __shfl_xor_sync(0xffffffffu, kq, o);
  }
}

// The sweep's scale rounded to R; lost: what the rounding took off.
template <typename R>
__device__ __forceinline__ typename C2<R>::T scale_of(double m, double ph, int kq,
                                                      typename C2<R>::T* lost = nullptr) {
  using T2 = typename C2<R>::T;
  const double u0 = ph + 0.5 * double(kq & 3), u = u0 - 2.0 * rint(0.5 * u0);
  double sn, cn;
  sincospi(u, &sn, &cn);
  const T2 c{R(m * cn), R(-m * sn)};
  if (lost) *lost = T2{R(m * cn - double(c.x)), R(-m * sn - double(c.y))};
  return c;
}

// The records of op oi of a descriptor.
__host__ __device__ __forceinline__ void records_of(const Args& a, const Op& op, int32_t (&rec)[5]) {
  for (int i = 0; i < 5; ++i) rec[i] = 0;
  if (op.type == OP_ROTN) {
    for (int i = 0; i < 5; ++i)
      if ((op.ku >> i) & 1) rec[i] = a.rot[rotn_slot(op, i)].cs;
  } else if (op.type == OP_ROT || op.type == OP_DROT) {
    rec[0] = a.rot[op.idx].cs;
  } else if (op.type == OP_BOND) {
    rec[0] = a.bond[op.idx];
  }
}

// A descriptor's tables, by the whole CTA (complete after the next barrier).
template <typename R, int B>
__device__ __forceinline__ void make_tables(const Args& a, const SmemMap& sm, unsigned char* smem_raw) {
  using T2 = typename C2<R>::T;
  constexpr int VB = sizeof(T2) == 8 ? 1 : 0;  // register bits inside a 16-byte chunk
  const int NT = blockDim.x;
  const uint32_t tid = threadIdx.x;
  OpRec<R>* ops = reinterpret_cast<OpRec<R>*>(smem_raw + sm.ops);
  LayRec* lays = reinterpret_cast<LayRec*>(smem_raw + sm.lays);
  auto copy_words = [&](void* dst, const void* src, size_t bytes) {
    const uint32_t* s4 = static_cast<const uint32_t*>(src);
    uint32_t* d4 = static_cast<uint32_t*>(dst);
    for (uint32_t w = tid; w < bytes / 4; w += NT) d4[w] = s4[w];
  };
  for (int i = 0; i < a.n_lay; ++i) copy_words(&lays[i].L, a.lay + i, sizeof(Layout));
  copy_words(smem_raw + sm.tabs, a.tab, sizeof(Tab) * a.n_tab);
  copy_words(smem_raw + sm.ph, a.ph, sizeof(Phase) * a.n_phase);
  copy_words(smem_raw + sm.cls, a.cls, sizeof(PClass) * a.n_cls);
  copy_words(smem_raw + sm.pt, a.pt, sizeof(PTerm) * a.n_pterm);
  for (int e = tid; e < 48 * a.n_lay; e += NT) {
    const int li = e / 48, j = e - 48 * li;
    const uint32_t d = deposit_index(a.lay[li], j);
    lays[li].dep[j] = make_uint2(d, swz(d >> VB));
  }
  uint32_t* clane = reinterpret_cast<uint32_t*>(smem_raw + sm.clane);
  for (int j = tid; j < 48; j += NT) clane[j] = copy_index(a.lay[a.ops[0].idx], j, VB);
  R* thpi = reinterpret_cast<R*>(smem_raw + sm.thpi);
  for (int t = tid; t < a.n_pterm; t += NT) thpi[t] = R(a.rq[4 * HS_BCHK(a.pt[t].th, a.n_terms_g, BS_REG_TERM) + 3]);
  T2* vts = reinterpret_cast<T2*>(smem_raw + sm.vts);
  for (int t = 0; t < a.n_tab; ++t) {
    const T2* g = reinterpret_cast<const T2*>(a.vt) + a.tab[t].vt0;
    const int s0 = a.tab[t].s0, n = a.tab[t].n;
    for (int e = tid; e < n; e += NT) vts[s0 + e] = g[HS_BCHK(a.tab[t].vt0 + e, a.n_vt_g, BS_REG_VT) - a.tab[t].vt0];
  }
  // One warp makes the coefficients and the scale, in FP64: the FP64 pipe takes
  // tens of cycles per warp instruction, so the others stay off it.
  if (tid < 32) {
    double m = 1.0, ph = 0.0;
    int kq = 0;
    const Records t{a.rq, a.cs, a.n_terms_g};
    for (int oi = tid; oi < a.n_ops; oi += 32) {
      const Op op = a.ops[oi];
      int32_t rec[5];
      records_of(a, op, rec);
      ops[oi].op = op;
      ops[oi].c = coef_of<R>(op, rec, t, m, ph, kq, a.exact_scale != 0);
    }
    sum_scale(m, ph, kq);
    if (tid == 0) {
      T2* out = reinterpret_cast<T2*>(smem_raw + sm.scale);
      out[0] = scale_of<R>(m, ph, kq, sizeof(T2) == 8 && a.exact_scale ? out + 1 : nullptr);
    }
  }
}

// ---------------------------------------------------------------------------
// The sweep of chunks q0, q0 + stride, ... < q1 of one descriptor (single
// launch: the kernel parameter; batched launch: a descriptor in global
// memory).  NT = 2^(T - B) threads; NR = 2^B rows per thread.
//
// A state's tile moves HBM -> shared memory -> registers by warp-cooperative
// copies (each warp copies exactly the rows its threads hold in the first
// layout, in address order), so the first read needs only a warp barrier.
// Once its last layout has been read, the tile buffer is free: every warp
// starts copying its rows of the CTA's next state or tile, which land while
// the current one finishes in registers and goes straight back to HBM.
// ---------------------------------------------------------------------------
// Slots of one PHASE run whose patterns across the groups take turns: 0, the
// register bits, the patterns inside the groups, one across.
template <int B>
constexpr int kMaxFac = 2 + B + ((1 << lower_bits(B)) - 1 - lower_bits(B)) + ((1 << (B - lower_bits(B))) - 1 - (B - lower_bits(B)));

// D: Args (the tables are made here) or Hdr (they are copied from the image).
// LEAN: a thread's phase factors in local memory instead of shared-memory slots,
// computed on each use, and one copy of the class constants for all warps: the
// same arithmetic in less shared memory.
template <typename R, int B, bool FULL, bool EXACT, bool LEAN, typename D>
__device__ __forceinline__ void qsweep_core(const D& a, uint32_t q0, uint32_t q1, uint32_t stride,
                                            unsigned char* smem_raw) {
  using T2 = typename C2<R>::T;
  constexpr bool kImage = std::is_same_v<D, Hdr>;
  constexpr int NR = 1 << B;
  constexpr int V = 16 / int(sizeof(T2));  // rows per 16-byte chunk (2 for complex64)
  constexpr int VB = V == 2 ? 1 : 0;       // register bits inside a chunk
  constexpr int NJ = NR / V;               // chunks per thread
  const int NT = blockDim.x;
  const uint32_t tid = threadIdx.x;
  const uint32_t m0 = a.m0, m1 = a.m1;
  const int sh = a.sh;
  const int warp = tid >> 5, lane = tid & 31;

  SmemMap sm;
  int first_lay;
  if constexpr (kImage) {
    sm = a.sm;
    first_lay = a.first_lay;
  } else {
    sm = smem_map(a, sizeof(T2), NT);
    first_lay = a.ops[0].idx;  // the first op is always a layout
  }
  auto at = [&](uint32_t SmemMap::* field) -> unsigned char* { return smem_raw + sm.*field; };
  T2* tile = reinterpret_cast<T2*>(smem_raw);
  OpRec<R>* ops = reinterpret_cast<OpRec<R>*>(at(&SmemMap::ops));
  LayRec* lays = reinterpret_cast<LayRec*>(at(&SmemMap::lays));
  T2* fac = reinterpret_cast<T2*>(at(&SmemMap::fac)) + tid;
  T2 fac_local[LEAN ? kMaxFac<B> : 1];
  const int cwarp = LEAN ? 0 : warp;  // whose copy of the class constants

  // Per-CTA tables (written before the launch before this one began, or an ordinary
  // launch: see enqueue_evolve).
  if constexpr (kImage) {
    for (uint32_t w = tid * 16; w < a.img_bytes; w += NT * 16) cp_async16(smem_raw + sm.ops + w, a.img + w);
    cp_async_commit();
    cp_async_wait(0);
  } else {
    make_tables<R, B>(a, sm, smem_raw);
  }
  const int n_ops = a.n_ops, n_cls = a.n_cls;
  const int last_lay = a.last_lay;

  // Warp-cooperative copy of this warp's rows of a tile in the first layout of
  // the sweep into the tile buffer: chunk mm of the thread lies at swizzled
  // chunk s0 ^ mswz(mm) and global row g0 ^ mglob(mm), both maps linear over
  // XOR, so four basis values each give all of them.
  constexpr int NJB = B - VB;  // log2 NJ
  const Layout* L0 = &lays[first_lay].L;
  auto copy_in = [&](uint32_t base, int state) {
    const T2* src = reinterpret_cast<const T2*>(a.src) + HS_BCHK(state, a.n_rhs, BS_REG_STATE) * a.N;
    const uint4 ms4 = *reinterpret_cast<const uint4*>(L0->mswz), mg4 = *reinterpret_cast<const uint4*>(L0->mglob);
    const uint32_t ms[4] = {ms4.x, ms4.y, ms4.z, ms4.w}, mg[4] = {mg4.x, mg4.y, mg4.z, mg4.w};
    const uint32_t* clane = reinterpret_cast<const uint32_t*>(at(&SmemMap::clane));
    const uint32_t l0 = clane[lane] | clane[32 + warp];
    const uint32_t s0 = swz(l0 >> VB), g0 = global_of(l0, m0, m1, sh) | base;
#pragma unroll
    for (int mm = 0; mm < NJ; ++mm) {
      uint32_t sx = s0, gx = g0;
#pragma unroll
      for (int k = 0; k < NJB; ++k)
        if ((mm >> k) & 1) {
          sx ^= ms[k];
          gx ^= mg[k];
        }
      cp_async16(tile + sx * V, src + HS_BCHK(gx, a.N - (V - 1), BS_REG_STATE));
    }
    cp_async_commit();
  };

  grid_dependency_wait();  // the state written by the previous launch is visible after this
  __syncthreads();         // the tables are in shared memory

  // Chunk q: tile index and its states [state, state_end).
  uint32_t q = q0, base = 0;
  int state = 0, state_end = 0;
  auto chunk = [&](uint32_t c, uint32_t& b, int& s0, int& s1) {
    const uint32_t t = c / uint32_t(a.rhs_chunks);
    b = deposit_runs(t, a.rest);
    s0 = int(c - t * uint32_t(a.rhs_chunks)) * a.rhs_chunk;
    s1 = min(s0 + a.rhs_chunk, a.n_rhs);
  };
  chunk(q, base, state, state_end);
  copy_in(base, state);
  grid_launch_dependents();  // the next sweep may load its tables meanwhile

  bool new_tile = true;
  uint32_t have = 0;  // PHASE runs whose factors are in shared memory for this tile
  while (true) {
    // Per-tile phase constants, in this warp's copy: class sums of +-theta_j
    // (units of pi, each term reduced mod 2 in FP64 by the factor build) with
    // the signs of the tile's fixed bits, reduced mod 2 again; a constant class
    // becomes its phase op's e0.  (The first barrier keeps a lane from writing
    // them while another lane still reads the previous tile's.)
    if (new_tile) {
      have = 0;
      const PClass* scls = reinterpret_cast<const PClass*>(at(&SmemMap::cls));
      const PTerm* spt = reinterpret_cast<const PTerm*>(at(&SmemMap::pt));
      const R* thpi = reinterpret_cast<const R*>(at(&SmemMap::thpi));
      T2* e0s = reinterpret_cast<T2*>(at(&SmemMap::e0s)) + cwarp * a.n_phase;
      ClassC<R>* cw = reinterpret_cast<ClassC<R>*>(at(&SmemMap::cw)) + cwarp * n_cls;
      if constexpr (LEAN) __syncthreads(); else __syncwarp();
      for (int cc = LEAN ? int(tid) : lane; cc < n_cls; cc += LEAN ? NT : 32) {
        const PClass C = scls[cc];
        R acc = R(0);
        for (int t = C.t0; t < C.t0 + C.nt; ++t) acc += flip_sign(thpi[t], uint32_t(__popc(spt[t].rest & base)));
        const R ur = acc - R(2) * rint(R(0.5) * acc);
        if (C.c0p >= 0) {
          R sn, cn;
          sincospi_r(ur, &sn, &cn);
          e0s[C.c0p] = T2{cn, -sn};
          cw[cc].c = R(0);
        } else {
          cw[cc].c = ur;
        }
        cw[cc].thr = C.thr;
      }
      if constexpr (LEAN) __syncthreads(); else __syncwarp();
    }

    const int cur_state = state;
    const uint32_t cur_base = base;
    // What this CTA runs next.
    bool more;
    {
      if (state + 1 < state_end) {
        ++state;
        more = true;
        new_tile = false;
      } else {
        more = q1 - q > stride;
        if (more) {
          q += stride;
          chunk(q, base, state, state_end);
        }
        new_tile = true;
      }
    }

    Rows<R, B> x;
    int cur = -1;  // the register layout in effect
    // Local row of this thread's register row 0 in that layout.
    auto local_row = [&]() { return lays[cur].dep[lane].x | lays[cur].dep[32 + warp].x; };
    // Its chunk j in the tile buffer: st ^ XOR of qo over the set bits of j.
    auto chunk_of = [&](uint32_t& st, uint32_t (&qo)[4]) {
      st = lays[cur].dep[lane].y ^ lays[cur].dep[32 + warp].y;
      const uint4 v = *reinterpret_cast<const uint4*>(lays[cur].L.qoff);
      qo[0] = v.x;
      qo[1] = v.y;
      qo[2] = v.z;
      qo[3] = v.w;
    };
    for (int oi = 0; oi < n_ops; ++oi) {
      const Op op = ops[oi].op;
      if (op.type == OP_LAYOUT) {
        uint32_t st, qo[4];
        // A thread writes back exactly the rows it read in the layout so far;
        // the new layout reads rows of its own warp only (flag 1: the warp bits
        // are the previous layout's) or of all warps.
        if (cur >= 0) {
          chunk_of(st, qo);
#pragma unroll
          for (int j = 0; j < NJ; ++j) {
            uint32_t pc = st;
#pragma unroll
            for (int i = 0; i < NJB; ++i)
              if ((j >> i) & 1) pc ^= qo[i];
            if constexpr (V == 2)
              *reinterpret_cast<float4*>(tile + pc * 2) = make_float4(x.re[j].x, x.re[j].y, x.im[j].x, x.im[j].y);
            else
              tile[pc] = x.x[j];
          }
          if (op.flags & 1)
            __syncwarp();
          else
            __syncthreads();
        } else {
          cp_async_wait(0);  // this tile's rows, copied by this warp
          __syncwarp();
        }
        const bool first = cur < 0;
        cur = op.idx;
        chunk_of(st, qo);
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
          uint32_t pc = st;
#pragma unroll
          for (int i = 0; i < NJB; ++i)
            if ((j >> i) & 1) pc ^= qo[i];
          if constexpr (V == 2) {
            const float4 w = *reinterpret_cast<const float4*>(tile + pc * 2);
            x.re[j] = make_float2(w.x, w.y);
            x.im[j] = make_float2(w.z, w.w);
          } else {
            x.x[j] = tile[pc];
          }
        }
        if constexpr (V == 2) {
          // The copied tile holds (re, im) row by row, a written-back one pairs.
          // (Selected, not branched on: with a branch here the compiler ran out of
          // registers; without its four spilled words 77.5 -> 74.4 ms.)
#pragma unroll
          for (int j = 0; j < NJ; ++j) {
            const float t = first ? x.im[j].x : x.re[j].y;
            x.im[j].x = first ? x.re[j].y : x.im[j].x;
            x.re[j].y = t;
          }
        }
        if (oi == last_lay && more) {
          // The tile buffer is free once every warp (the warp itself where it
          // copies the rows it has just read) has read its rows.
          if (a.free_local)
            __syncwarp();
          else
            __syncthreads();
          copy_in(base, state);
        }
      } else if (op.type == OP_ROTN) {
        const Coef<R> c = ops[oi].c;
        rotn<R, B>(x, op.ku, c.v);
        if (c.swap) flip_run<R, B, 0>(x, c.swap);
      } else if (op.type == OP_PHASE) {
        const Phase& P = reinterpret_cast<const Phase*>(at(&SmemMap::ph))[op.idx];
        const ClassC<R>* cw = reinterpret_cast<const ClassC<R>*>(at(&SmemMap::cw)) + cwarp * n_cls;
        const T2 e0 = reinterpret_cast<const T2*>(at(&SmemMap::e0s))[cwarp * a.n_phase + op.idx];
        if constexpr (LEAN) {
          phase_op<R, B>(x, P, cw, e0, local_row(), fac_local, 1, true, false);
        } else {
          phase_op<R, B>(x, P, cw, e0, local_row(), fac + P.fac0 * NT, NT, !((have >> op.idx) & 1u), a.fac_keep != 0);
          if (a.fac_keep) have |= 1u << op.idx;
        }
      } else if (op.type == OP_BOND) {
        bond_dispatch<R, B>(x, op.ku, T2{ops[oi].c.v[0], ops[oi].c.v[1]});
      } else if (op.type == OP_ROT) {
        const R c = ops[oi].c.v[0];
        const bool swap = ops[oi].c.swap != 0;
        if constexpr (FULL) {
          const bool fast = op.flags & 1;
          const int sbit = fast ? 0 : (parity(op.zrest & cur_base) ^ parity(op.zthr & local_row()));
          rot_dispatch<R, B>(x, op.ku, c, ops[oi].c.v[1], fast, (op.flags >> 1) & 3, op.zk, sbit, swap);
        } else {
          tan_dispatch<R, B>(x, op.ku, c, swap);  // the planner sends only tan-form rotations here
        }
      } else if (op.type == OP_DROT) {
        diag_rot<R, B>(x, ops[oi].c.v[0], ops[oi].c.v[1], op.zk, parity(op.zrest & cur_base) ^ parity(op.zthr & local_row()));
      } else {
        if constexpr (FULL) {
          const Tab& tb = reinterpret_cast<const Tab*>(at(&SmemMap::tabs))[op.idx];
          const uint32_t smask = tb.sm;
          const int tsh = tb.sh;
          uint32_t pr[B];
#pragma unroll
          for (int i = 0; i < B; ++i)
            pr[i] = pattern_fast(i < VB ? lays[cur].L.g0 : lays[cur].L.goff[i - VB], smask, tsh);
          tab_dispatch<R, B>(x, op.ku, reinterpret_cast<const T2*>(at(&SmemMap::vts)) + tb.s0, tb.ns, pattern_fast(global_of(local_row(), m0, m1, sh) | cur_base, smask, tsh), pr);
        }
      }
    }
    // The sweep's scale (real unless a rotation made an odd number of quarter
    // turns or a bond left its phase), then the rows straight to HBM: chunk j
    // of the thread sits at global row gt ^ XOR of the layout's global offsets
    // of the set bits of j.
    const T2 out_scale = *reinterpret_cast<const T2*>(at(&SmemMap::scale));
    if (out_scale.y != R(0)) {
      if constexpr (V == 2) {
        const float2 c = dup(out_scale.x), s = dup(out_scale.y), ns = dup(-out_scale.y);
        if constexpr (EXACT) {
          const float2 lost = reinterpret_cast<const float2*>(at(&SmemMap::scale))[1];
          const float2 cl = dup(lost.x), sl = dup(lost.y), nsl = dup(-lost.y);
#pragma unroll
          for (int j = 0; j < NJ; ++j) {
            const float2 r = x.re[j], m = x.im[j];
            x.re[j] = fma2(r, c, fma2(m, ns, fma2(r, cl, __fmul2_rn(m, nsl))));
            x.im[j] = fma2(r, s, fma2(m, c, fma2(r, sl, __fmul2_rn(m, cl))));
          }
        } else {
#pragma unroll
          for (int j = 0; j < NJ; ++j) {
            const float2 r = x.re[j], m = x.im[j];
            x.re[j] = fma2(r, c, __fmul2_rn(m, ns));
            x.im[j] = fma2(r, s, __fmul2_rn(m, c));
          }
        }
      } else {
#pragma unroll
        for (int k = 0; k < NR; ++k) x.x[k] = cmul<T2, R>(x.x[k], out_scale.x, out_scale.y);
      }
    } else if (out_scale.x != R(1)) {
      if constexpr (V == 2) {
        const float2 c = dup(out_scale.x);
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
          x.re[j] = __fmul2_rn(x.re[j], c);
          x.im[j] = __fmul2_rn(x.im[j], c);
        }
      } else {
#pragma unroll
        for (int k = 0; k < NR; ++k) x.x[k] = T2{x.x[k].x * out_scale.x, x.x[k].y * out_scale.x};
      }
    }
    T2* dst = reinterpret_cast<T2*>(a.dst) + HS_BCHK(cur_state, a.n_rhs, BS_REG_STATE) * a.N;
    const uint4 go4 = *reinterpret_cast<const uint4*>(lays[cur].L.goff);
    const uint32_t go[4] = {go4.x, go4.y, go4.z, go4.w};
    const uint32_t gt = global_of(local_row(), m0, m1, sh) | cur_base;
    // When the two lowest register bits are local bits 0 and 1 (complex64;
    // for complex128 register bit 0 is local bit 0) and the tile keeps those
    // bits contiguous, a thread's registers 4q .. 4q + 3 (2q, 2q + 1) are 32
    // consecutive bytes: one 32-byte store fills a whole sector.
    constexpr int WB = V == 2 ? 2 : 1;  // register bits inside a 32-byte store
    const uint32_t wide_bits = (1u << WB) - 1u;  // local bits that must be the lowest register bits
    const bool wide = (lays[cur].L.reg & wide_bits) == wide_bits && (m0 & wide_bits) == wide_bits &&
                      (reinterpret_cast<uintptr_t>(a.dst) & 31u) == 0;  // (states may be only 16-byte aligned)
    if (wide) {
#pragma unroll
      for (int w = 0; w < (NR >> WB); ++w) {
        uint32_t g = gt;
#pragma unroll
        for (int i = WB; i < B; ++i)
          if (((w << WB) >> i) & 1) g ^= go[i - VB];
        T2* p = dst + HS_BCHK(g, a.N - (1 << WB) + 1, BS_REG_STATE);
        if constexpr (V == 2) {
          const float2 r0 = x.re[2 * w], i0 = x.im[2 * w], r1 = x.re[2 * w + 1], i1 = x.im[2 * w + 1];
          asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"l"(p), "f"(r0.x), "f"(i0.x),
                       "f"(r0.y), "f"(i0.y), "f"(r1.x), "f"(i1.x), "f"(r1.y), "f"(i1.y)
                       : "memory");
        } else {
          const T2 v0 = x.x[2 * w], v1 = x.x[2 * w + 1];
          asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};\n" ::"l"(p), "d"(v0.x), "d"(v0.y), "d"(v1.x), "d"(v1.y)
                       : "memory");
        }
      }
    } else {
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        uint32_t g = gt;
#pragma unroll
        for (int i = 0; i < NJB; ++i)
          if ((j >> i) & 1) g ^= go[i];
        if constexpr (V == 2)
          *reinterpret_cast<float4*>(dst + HS_BCHK(g, a.N - 1, BS_REG_STATE)) =
              make_float4(x.re[j].x, x.im[j].x, x.re[j].y, x.im[j].y);
        else
          dst[HS_BCHK(g, a.N, BS_REG_STATE)] = x.x[j];
      }
    }
    if (!more) break;
  }
}

// FULL: the kernel with the TAB and general-rotation paths; sweeps without
// them run the lighter instantiation.  NT: threads per CTA the instantiation
// is built for (2^(tile_bits - B); 512 for 2^14-row complex64 tiles with five
// register bits, one CTA per SM).  EXACT: a bond sweep applies its scale to more
// than R's precision.  Rounded, a scale shifts the norm by up to 6e-8 a sweep, all
// one way: 1.1e-5 over 200 steps of a 20-qubit Heisenberg chain, 1e-8 with it.  (An
// instantiation of its own: as a branch it cost the MaxCut sweeps 0.5%.)  LEAN:
// see qsweep_core.
template <typename R, int B, bool FULL, int NT = (B == 5 ? 256 : 512), bool EXACT = false, bool LEAN = false>
__global__ void __launch_bounds__(NT, NT == 256 ? 2 : 1) qsweep_kernel(const __grid_constant__ Args a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  qsweep_core<R, B, FULL, EXACT, LEAN>(a, blockIdx.x, uint32_t(a.n_chunks), gridDim.x, smem_raw);
}

template <typename R, int B, bool FULL, bool LEAN = false>
__global__ void __launch_bounds__(B == 5 ? 256 : 512, B == 5 ? 2 : 1) qlevel_kernel(const __grid_constant__ LevelArgs p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Hdr& a = *reinterpret_cast<Hdr*>(smem_raw + p.prefix_smem);  // the job's header
  int* pref = reinterpret_cast<int*>(smem_raw + p.prefix_smem + kHdrSmem);
  for (int i = threadIdx.x; i < p.count; i += blockDim.x) pref[i] = p.lvl_prefix[p.off + i];
  __syncthreads();
  int lo = 0, hi = p.count - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (pref[mid] <= int(blockIdx.x)) lo = mid; else hi = mid - 1;
  }
  const uint32_t* hd = reinterpret_cast<const uint32_t*>(p.descs + p.lvl_desc[p.off + lo]);
  static_assert(sizeof(Hdr) % 4 == 0, "copied by words");
  for (uint32_t w = threadIdx.x; w < sizeof(Hdr) / 4; w += blockDim.x) reinterpret_cast<uint32_t*>(&a)[w] = hd[w];
  __syncthreads();
  const uint32_t u = uint32_t(HS_BCHK(blockIdx.x - uint32_t(pref[lo]), a.n_chunks, BS_BATCH_JOB));
  qsweep_core<R, B, FULL, false, LEAN>(a, u, u + 1, 1u, smem_raw);
}

// One block per image: the template's bytes, then the coefficients of every op
// from the term records, the phase terms' angles, the value tables and the
// sweep's scale.
template <typename R>
__global__ void __launch_bounds__(128) qfill_kernel(const FillRec* recs) {
  using T2 = typename C2<R>::T;
  const FillRec f = recs[blockIdx.x];
  const int tid = threadIdx.x;
  for (uint32_t w = tid; w < f.bytes / 16; w += 128)
    reinterpret_cast<uint4*>(f.img)[w] = reinterpret_cast<const uint4*>(f.tmpl)[w];
  __syncthreads();
  const PTerm* pt = reinterpret_cast<const PTerm*>(f.tmpl + f.pt);
  R* thpi = reinterpret_cast<R*>(f.img + f.thpi);
  for (int t = tid; t < f.n_pterm; t += 128) thpi[t] = R(f.rq[4 * HS_BCHK(pt[t].th, f.n_terms_g, BS_REG_TERM) + 3]);
  const Tab* tabs = reinterpret_cast<const Tab*>(f.tmpl + f.tabs);
  T2* vts = reinterpret_cast<T2*>(f.img + f.vts);
  for (int t = 0; t < f.n_tab; ++t)
    for (int e = tid; e < tabs[t].n; e += 128)
      vts[tabs[t].s0 + e] = reinterpret_cast<const T2*>(f.vt)[HS_BCHK(tabs[t].vt0 + e, f.n_vt_g, BS_REG_VT)];
  // One warp, as in make_tables: the scale's factors then meet in the same order,
  // and a batch gives the bits of its jobs alone.
  if (tid >= 32) return;
  double m = 1.0, ph = 0.0;
  int kq = 0;
  const Records rec{f.rq, f.cs, f.n_terms_g};
  const OpRec<R>* src = reinterpret_cast<const OpRec<R>*>(f.tmpl + f.ops);
  OpRec<R>* dst = reinterpret_cast<OpRec<R>*>(f.img + f.ops);
  for (int oi = tid; oi < f.n_ops; oi += 32) {
    const Op op = src[oi].op;
    dst[oi].c = coef_of<R>(op, reinterpret_cast<const int32_t*>(src[oi].c.v), rec, m, ph, kq);
  }
  sum_scale(m, ph, kq);
  if (tid == 0) *reinterpret_cast<T2*>(f.img + f.scale) = scale_of<R>(m, ph, kq);
}

using LFn = void (*)(LevelArgs);

using QFn = void (*)(Args);

// The instantiation for (precision, register bits, tile bits): 2^(T - B)
// threads, at most 256 for five register bits (512 with T = 14), at most 512
// for four; nullptr otherwise.
template <bool FULL>
QFn qsweep_fn_t(hs_dtype dt, int B, int tile_bits) {
  const int tb = tile_bits - B;
  if (tb < 5) return nullptr;
  if (dt == HS_C64 && B == 5)
    return tb <= 8 ? qsweep_kernel<float, 5, FULL> : (tb == 9 ? qsweep_kernel<float, 5, FULL, 512> : nullptr);
  if (B == 4 && tb <= 9) return dt == HS_C64 ? qsweep_kernel<float, 4, FULL> : qsweep_kernel<double, 4, FULL>;
  return nullptr;
}
QFn lean_fn(hs_dtype dt, int B, int tile_bits) {
  const int tb = tile_bits - B;
  if (tb < 5 || tb > 9) return nullptr;
  if (dt == HS_C64 && B == 5) return qsweep_kernel<float, 5, true, 512, false, true>;
  if (B != 4) return nullptr;
  return dt == HS_C64 ? qsweep_kernel<float, 4, true, 512, false, true> : qsweep_kernel<double, 4, true, 512, false, true>;
}
QFn qsweep_fn(hs_dtype dt, int B, bool full, int tile_bits, bool exact = false, bool lean = false) {
  if (lean) return lean_fn(dt, B, tile_bits);
  if (exact && !full && dt == HS_C64 && B == 5 && tile_bits >= 10 && tile_bits <= 13)
    return qsweep_kernel<float, 5, false, 256, true>;
  return full ? qsweep_fn_t<true>(dt, B, tile_bits) : qsweep_fn_t<false>(dt, B, tile_bits);
}

template <bool FULL>
LFn qlevel_fn_t(hs_dtype dt, int B) {
  if (dt == HS_C64)
    return B == 5 ? qlevel_kernel<float, 5, FULL> : (B == 4 ? qlevel_kernel<float, 4, FULL> : nullptr);
  return B == 4 ? qlevel_kernel<double, 4, FULL> : nullptr;
}
LFn qlevel_fn(hs_dtype dt, int B, bool full, bool lean) {
  if (!lean) return full ? qlevel_fn_t<true>(dt, B) : qlevel_fn_t<false>(dt, B);
  if (dt == HS_C64 && B == 5) return qlevel_kernel<float, 5, true, true>;
  if (B != 4) return nullptr;
  return dt == HS_C64 ? qlevel_kernel<float, 4, true, true> : qlevel_kernel<double, 4, true, true>;
}

}  // namespace

cudaError_t prepare_qsweep() {
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(mu);
  if (dev < 64 && done[dev]) return cudaSuccess;
  const hs_dtype dts[3] = {HS_C64, HS_C64, HS_C128};
  const int Bs[3] = {5, 4, 4};
  for (int v = 0; v < 3; ++v)
    for (bool full : {false, true}) {
      e = cudaFuncSetAttribute((const void*)qsweep_fn(dts[v], Bs[v], full, Bs[v] + 8),
                               cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSweepSmemMax));
      if (e == cudaSuccess && v == 0)
        e = cudaFuncSetAttribute((const void*)qsweep_fn(dts[v], Bs[v], full, 14),
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSweepSmemMax));
      if (e == cudaSuccess && v == 0)
        e = cudaFuncSetAttribute((const void*)qsweep_fn(dts[v], Bs[v], full, 13, true),
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSweepSmemMax));
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute((const void*)qlevel_fn(dts[v], Bs[v], full, false),
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSweepSmemMax));
      if (e == cudaSuccess && full)
        e = cudaFuncSetAttribute((const void*)qsweep_fn(dts[v], Bs[v], true, Bs[v] + 8, false, true),
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSweepSmemMax));
      if (e == cudaSuccess && full)
        e = cudaFuncSetAttribute((const void*)qlevel_fn(dts[v], Bs[v], true, true),
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSweepSmemMax));
      if (e != cudaSuccess) return e;
    }
  if (dev < 64) done[dev] = true;
  return cudaSuccess;
}

cudaError_t launch_fill(hs_dtype dt, const unsigned char* dev, int n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const FillRec* r = reinterpret_cast<const FillRec*>(dev);
  if (dt == HS_C64)
    qfill_kernel<float><<<unsigned(n), 128, 0, s>>>(r);
  else
    qfill_kernel<double><<<unsigned(n), 128, 0, s>>>(r);
  note_launches();
  return cudaGetLastError();
}

void op_records(const Args& a, int oi, int32_t (&rec)[5]) { records_of(a, a.ops[oi], rec); }

size_t qsweep_smem_bytes(const Args& a, hs_dtype dt, int B) {
  return smem_map(a, uint32_t(elem_bytes(dt)), 1u << (a.tile_bits - B)).total;
}

// The most states of a tile a CTA runs back to back (a PHASE run's factors are
// computed for the first only) that does not lengthen the longest CTA by more
// than a fiftieth.
int pick_rhs_chunk(int64_t tiles, int n_rhs, int slots) {
  int best = 1;
  int64_t best_len = 0;
  for (int k = 1; k <= std::min(n_rhs, kMaxRhsChunk); k *= 2) {
    const int64_t chunks = tiles * ((n_rhs + k - 1) / k);
    const int64_t len = (chunks + slots - 1) / slots * k;
    if (best_len == 0 || len * 50 <= best_len * 51) {
      best = k;
      best_len = best_len == 0 ? len : std::min(len, best_len);
    }
  }
  return best;
}

void fill_job(const hs_factors* f, Args& a, void* psi, int n_rhs, int rhs_chunk) {
  const Plan& p = f->plan;
  a.src = psi;
  a.dst = psi;
  a.cs = f->bin.cs;
  a.th = f->bin.th;
  a.rq = f->bin.rq;
  a.vt = f->d_vt;
  a.N = p.N;
  a.n_vt_g = p.total_vt;
  a.n_terms_g = int(p.x.size()) * p.n_kinds;
  a.n_rhs = n_rhs;
  a.n_tiles_log2 = p.n_qubits - a.tile_bits;
  a.rhs_chunk = rhs_chunk;
  a.rhs_chunks = (n_rhs + rhs_chunk - 1) / rhs_chunk;
  a.n_chunks = (1 << a.n_tiles_log2) * a.rhs_chunks;
}

cudaError_t launch_qlevel(hs_dtype dt, int B, bool full, bool lean, int tile_bits, const LevelArgs& L, int64_t ctas,
                          size_t smem, bool pdl, cudaStream_t s) {
  LFn fn = qlevel_fn(dt, B, full, lean);
  if (!fn || tile_bits - B < 5 || smem > kSweepSmemMax || ctas <= 0 || ctas >= (int64_t(1) << 31))
    return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(ctas), 1u, 1u);
  cfg.blockDim = dim3(unsigned(1u << (tile_bits - B)), 1u, 1u);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, fn, L);
  if (e == cudaSuccess) note_launches();
  return e;
}

cudaError_t launch_qsweep(const hs_factors* f, Args& a, const void* src, void* dst, int n_rhs, int B, bool pdl,
                          cudaStream_t s, const double* rq, const double* cs, int n_terms) {
  const Plan& p = f->plan;
  QFn fn = qsweep_fn(f->dtype, B, a.full != 0, a.tile_bits, a.exact_scale != 0, a.lean != 0);
  if (!fn || a.tile_bits - B < 5 || a.tile_bits > p.n_qubits) return cudaErrorInvalidValue;
  const size_t smem = qsweep_smem_bytes(a, f->dtype, B);
  if (smem > kSweepSmemMax) return cudaErrorInvalidValue;
  // One resident CTA per slot of the chip runs its share of the chunks back to
  // back (its tables are loaded once).
  const int threads = 1 << (a.tile_bits - B);
  const int per_sm = std::max(1, std::min({32, 65536 / (128 * threads), int((kSmemPerSm) / (smem + 1024))}));
  const int slots = kSMs * per_sm;
  fill_job(f, a, const_cast<void*>(src), n_rhs, pick_rhs_chunk(int64_t(1) << (p.n_qubits - a.tile_bits), n_rhs, slots));
  a.dst = dst;
  if (rq) {
    a.rq = rq;
    a.cs = cs;
    a.n_terms_g = n_terms;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(std::min(a.n_chunks, slots)), 1u, 1u);
  cfg.blockDim = dim3(unsigned(threads), 1u, 1u);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, fn, a);
  if (e == cudaSuccess) note_launches();
  return e;
}

}  // namespace q
}  // namespace hs
