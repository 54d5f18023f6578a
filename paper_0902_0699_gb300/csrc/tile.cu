// Fused shared-memory tile passes.
//
// One-qubit operators on distinct pairs are independent (sec. 3, after
// Eq. resmat1), and operators on different qubits commute, so every gate
// acting on a contiguous group of qubits [lo, lo+k) can be applied in one
// pass: a CTA stages a tile -- all 2^k values of the group bits, times the
// 2^c lowest index bits kept contiguous for 128-byte rows -- in shared
// memory, applies the group's gates there, and writes the tile back.
// HALL (Eq. HALL) and layers of one-qubit operators take a few passes
// instead of n.  Hadamards are applied as unnormalised butterflies
// (a0 + a1, a0 - a1) and the pass multiplies by 2^{-p/2} once at the end.
//
// The QFT circuit of Appendix A processes qubits from the most significant
// down: Hadamard on t, then CPHASEK(t, t') for every lower t' with phase
// e^{2 pi i / 2^{t-t'+1}}.  For a group [lo, hi] the phases with t' inside
// the group are applied right after the group's Hadamard on t (a diagonal
// "ladder" e^{2 pi i x / 2^{j+1}}, x = group bits below group qubit j);
// those with t' < lo commute with the rest of the group's gates and are
// applied at the end of the pass as one twiddle factor
//   Omega_{hi+1}^{L f},  Omega_m = e^{2 pi i / 2^m},
//   L = index bits below lo, f = the group bits in reversed order.
// With L = Ltile + l (Ltile fixed per tile, l the c contiguous low bits)
// the twiddle is V[f] * Omega^{l f}: V is built once per tile from global
// root tables, Omega^{l f} (l f < 2^{c+k}) comes from a two-level table in
// shared memory, the ladder phases from a direct table.  The final SWAPs
// are one in-place blocked bit-reversal pass (complex64: with the lowest five
// levels; a transform of one tile reverses on its store).
//
// complex64 tiles compute in FP32.  complex128 tiles compute in double-float
// (ff.cuh) on the FP32 pipe: the FP64 pipe of GB300 (0.5 Top/s) would
// otherwise bound every pass many times over the memory time.
#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"
#include "ff.cuh"
#include "fixpt.cuh"

namespace qc {

enum TileOpKind { TOP_U2 = 0, TOP_QFTLEVEL = 1, TOP_HB = 2 };
#define QC_TILE_MAXOPS 36

// ------------------------------------------------ arithmetic policies ----
template <typename R> struct TA;

template <> struct TA<float> {
  using E = Cx<float>;
  using V2 = float2;
  using M = Mat2<float>;
  static M mat(const double* U) { return mat_from_host<float>(U); }
  __device__ static E from(V2 v) { return cmake<float>(v.x, v.y); }
  __device__ static V2 to(E z) { return make_float2(z.re, z.im); }
  __device__ static E add(E a, E b) { return cmake<float>(a.re + b.re, a.im + b.im); }
  __device__ static E sub(E a, E b) { return cmake<float>(a.re - b.re, a.im - b.im); }
  // first level of a radix-4 step (no renormalisation to skip in FP32)
  __device__ static E add_u(E a, E b) { return add(a, b); }
  __device__ static E sub_u(E a, E b) { return sub(a, b); }
  __device__ static E norm(E a) { return a; }
  __device__ static E mul(E a, E b) { return cmul(a, b); }
  __device__ static E times_i(E a) { return cmake<float>(-a.im, a.re); }
  __device__ static E neg(E a) { return cmake<float>(-a.re, -a.im); }
  __device__ static E root(uint64_t num, int m) {  // e^{2 pi i num / 2^m}
    double s, c;
    sincospi(ldexp((double)num, 1 - m), &s, &c);
    return cmake<float>((float)c, (float)s);
  }
  __device__ static E fromd(double re, double im) { return cmake<float>((float)re, (float)im); }
  // 2^{-p/2}, computed once per thread, and the multiplication by it
  using S = float;
  __device__ static S scale_const(int p) { return (float)exp2(-0.5 * p); }
  __device__ static E scale_by(E a, S s) { return cmake<float>(a.re * s, a.im * s); }
  __device__ static void u2(int kind, const M& U, E& a0, E& a1) {
    switch (kind) {
      case MK_GENERAL: apply2<float, MK_GENERAL>(U, a0, a1); break;
      case MK_REAL: apply2<float, MK_REAL>(U, a0, a1); break;
      case MK_DIAG: apply2<float, MK_DIAG>(U, a0, a1); break;
      case MK_PHASE1: apply2<float, MK_PHASE1>(U, a0, a1); break;
      case MK_PH_NEG: apply2<float, MK_PH_NEG>(U, a0, a1); break;
      case MK_PH_I: apply2<float, MK_PH_I>(U, a0, a1); break;
      case MK_PH_MI: apply2<float, MK_PH_MI>(U, a0, a1); break;
      case MK_ANTI: apply2<float, MK_ANTI>(U, a0, a1); break;
      case MK_SWAPX: apply2<float, MK_SWAPX>(U, a0, a1); break;
      case MK_HAD: apply2<float, MK_HAD>(U, a0, a1); break;
      default: break;
    }
  }
};

template <> struct TA<double> {
  using E = ffc;
  using V2 = double2;
  using M = Mat2ff;
  static M mat(const double* U) { return mat2ff_from_host(U); }
  // the tile passes are arithmetic bound: the integer-lean conversions
  __device__ static E from(V2 v) { return ffc_make(ff_from_d_fast(v.x), ff_from_d_fast(v.y)); }
  __device__ static V2 to(E z) { return make_double2(ff_to_d_fast(z.re), ff_to_d_fast(z.im)); }
  __device__ static E add(E a, E b) { return ffc_add(a, b); }
  __device__ static E sub(E a, E b) { return ffc_sub(a, b); }
  // first level of a radix-4 step: its sums feed the second level's adds
  // directly, so their renormalisation is left to those
  __device__ static E add_u(E a, E b) { return ffc_add_u(a, b); }
  __device__ static E sub_u(E a, E b) { return ffc_sub_u(a, b); }
  // the closing renormalisation of an unnormalised sum (fast two-sum per
  // component), for a value stored without passing through a product
  __device__ static E norm(E a) {
    float h, l;
    ffc r;
    fast_two_sum(a.re.hi, a.re.lo, h, l);
    r.re = ff_make(h, l);
    fast_two_sum(a.im.hi, a.im.lo, h, l);
    r.im = ff_make(h, l);
    return r;
  }
  __device__ static E mul(E a, E b) { return ffc_mul(a, b); }
  __device__ static E times_i(E a) { return ffc_make(ff_neg(a.im), a.re); }
  __device__ static E neg(E a) { return ffc_make(ff_neg(a.re), ff_neg(a.im)); }
  __device__ static E root(uint64_t num, int m) {
    double s, c;
    sincospi(ldexp((double)num, 1 - m), &s, &c);
    return ffc_from_d(c, s);
  }
  __device__ static E fromd(double re, double im) { return ffc_from_d(re, im); }
  // 2^{-p/2} = 2^{-floor(p/2)} (exact) times 1/sqrt(2) when p is odd
  using S = ff;
  __device__ static S scale_const(int p) {
    ff s = ff_make(ff_bitsf((uint32_t)(127 - p / 2) << 23), 0.f);
    if (p & 1) s = ff_mul(s, ff_from_d(0.70710678118654752440));
    return s;
  }
  __device__ static E scale_by(E a, S s) { return ffc_scale(a, s); }
  __device__ static void u2(int kind, const M& U, E& a0, E& a1) {
    switch (kind) {
      case MK_GENERAL: apply2_ff<MK_GENERAL>(U, a0, a1); break;
      case MK_REAL: apply2_ff<MK_REAL>(U, a0, a1); break;
      case MK_DIAG: apply2_ff<MK_DIAG>(U, a0, a1); break;
      case MK_PHASE1: apply2_ff<MK_PHASE1>(U, a0, a1); break;
      case MK_ANTI: apply2_ff<MK_ANTI>(U, a0, a1); break;
      case MK_HAD: apply2_ff<MK_HAD>(U, a0, a1); break;
      case MK_PH_NEG: a1 = ffc_make(ff_neg(a1.re), ff_neg(a1.im)); break;
      case MK_PH_I: a1 = ffc_make(ff_neg(a1.im), a1.re); break;
      case MK_PH_MI: a1 = ffc_make(a1.im, ff_neg(a1.re)); break;
      case MK_SWAPX: {
        const E t = a0;
        a0 = a1;
        a1 = t;
        break;
      }
      default: break;
    }
  }
};

template <typename R> struct TileProg {
  int nops;
  int lo, k, c;     // group [lo, lo+k), c low contiguous bits (c <= lo)
  int n;            // bits of the QFT's root tables (the transformed register's width)
  int base;         // the register's lowest qubit: the QFT's phases use the index bits from here up
  int rev;          // store the lowest `rev` group bits in reversed order (a register of one group)
  int twiddle;      // apply the QFT cross phase with the register bits below lo
  int qft;          // QFT levels, on the lowest `qft` group bits (the ladder table has as many)
  int nl;           // global root table split: low table has 2^nl entries
  int scale_p;      // unnormalised butterflies: multiply by 2^{-scale_p/2} at the end
  int8_t kind[QC_TILE_MAXOPS];
  int8_t q[QC_TILE_MAXOPS];   // group-relative qubit
  int8_t mk[QC_TILE_MAXOPS];  // MatKind of a TOP_U2 operator
  typename TA<R>::M U[QC_TILE_MAXOPS];
};

// Shared memory after the tile: V[2^k] (twiddle passes), LAD[lad_entries(k)]
// (QFT passes: level j's 2^j ladder phases e^{2 pi i x / 2^{j+1}} at
// LAD[2^j - 1 + x], so a warp reads consecutive entries), TWA[128], TWB[128].
#define TS_TWA 128
#define TS_TWB 128  // x < 2^{c+k} <= 2^14

// Ladder levels kept in the table.  complex128 stops at level 10 (2047
// double-float entries, 32 KiB), so the 12-qubit lowest group's pass fits
// two CTAs per SM; its level 11 phase is L_11(y) = L_10(y >> 1) times
// e^{2 pi i / 2^12} for odd y, the latter stored after the table.
template <typename R>
__host__ __device__ constexpr int lad_levels(int k) {
  return sizeof(R) == 8 ? (k < 11 ? k : 11) : k;
}
template <typename R>
__host__ __device__ constexpr int lad_entries(int k) {
  return (1 << lad_levels<R>(k)) - 1 + (k > lad_levels<R>(k) ? 1 : 0);
}

__device__ __forceinline__ uint64_t tile_global(uint64_t e, uint64_t T, int lo, int k, int c) {
  const uint64_t cm = (1ull << c) - 1ull;
  const uint64_t tmid = T & ((1ull << (lo - c)) - 1ull);
  const uint64_t thi = T >> (lo - c);
  return (e & cm) | (tmid << c) | ((e >> c) << lo) | (thi << (lo + k));
}

// Root of unity Omega_n^r from the two global tables.
template <typename R>
__device__ __forceinline__ typename TA<R>::E omega(const typename CT<R>::V2* __restrict__ tlo,
                                                   const typename CT<R>::V2* __restrict__ thi, uint64_t r, int nl) {
  const auto a = tlo[r & ((1ull << nl) - 1ull)];
  const auto b = thi[r >> nl];
  return TA<R>::mul(TA<R>::from(a), TA<R>::from(b));
}

// L_j(y) = e^{2 pi i y / 2^{j+1}}, y < 2^j, from the ladder table (levels
// below kl) or, for level kl, from level kl - 1 and the extra entry.
template <typename R>
__device__ __forceinline__ typename TA<R>::E ladder_at(const typename TA<R>::E* LAD, int kl, int j, int y) {
  if (j < kl) return LAD[(1 << j) - 1 + y];
  const typename TA<R>::E m = LAD[(1 << (j - 1)) - 1 + (y >> 1)];
  return (y & 1) ? TA<R>::mul(m, LAD[(1 << kl) - 1]) : m;
}

// A ladder table entry in global memory (16 bytes for double-float).
template <typename R> struct LadIO;
template <> struct LadIO<float> {
  __device__ static Cx<float> ld(const float2* p) { return cmake<float>(p->x, p->y); }
  __device__ static void st(float2* p, Cx<float> z) { *p = make_float2(z.re, z.im); }
};
template <> struct LadIO<double> {
  __device__ static ffc ld(const double2* p) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    return ffc_make(ff_make(v.x, v.y), ff_make(v.z, v.w));
  }
  __device__ static void st(double2* p, ffc z) {
    *reinterpret_cast<float4*>(p) = make_float4(z.re.hi, z.re.lo, z.im.hi, z.im.lo);
  }
};

// Shared tables of a pass: the ladders (QFT programs, copied from the
// transform's table: one FP64 sincospi per entry and block costs more than
// the pass itself on states of up to 2^20 amplitudes) and the twiddle
// remainder tables TWA, TWB (QFT programs with a twiddle whose contiguous
// bits belong to the register).
template <typename R>
__device__ __forceinline__ void tile_tables(const TileProg<R>& P, const typename CT<R>::V2* __restrict__ lad,
                                            typename TA<R>::E* LAD, typename TA<R>::E* TWA, typename TA<R>::E* TWB) {
  using A = TA<R>;
  const int hi = P.lo + P.k - 1 - P.base;
  if (!P.qft) return;
  for (int a = threadIdx.x; a < lad_entries<R>(P.qft); a += blockDim.x) LAD[a] = LadIO<R>::ld(lad + a);
  // twiddle remainder: Omega_{hi+1}^x = TWA[x & 127] * TWB[x >> 7], x < 2^{c+k}
  if (P.twiddle && P.base < P.c)
    for (int i = threadIdx.x; i < TS_TWA + TS_TWB; i += blockDim.x) {
      if (i < TS_TWA) TWA[i] = A::root((uint64_t)i, hi + 1);
      else TWB[i - TS_TWA] = A::root((uint64_t)(i - TS_TWA) << 7, hi + 1);
    }
}

// V[f] = 2^{-p/2} Omega_{hi+1}^{Ltile f} for tile T (Ltile = the tile's
// register bits between c and lo; hi counted within the register).
template <typename R>
__device__ __forceinline__ void tile_twiddle_v(const TileProg<R>& P, uint64_t T, typename TA<R>::E* V,
                                               const typename CT<R>::V2* __restrict__ tlo,
                                               const typename CT<R>::V2* __restrict__ thi, typename TA<R>::S sc) {
  const int lo = P.lo, k = P.k, c = P.c, hi = lo + k - 1 - P.base;
  const uint64_t Lt = ((T & ((1ull << (lo - c)) - 1ull)) << c) >> P.base;
  for (int f = threadIdx.x; f < (1 << k); f += blockDim.x) {
    const uint64_t r = (Lt * (uint64_t)f) & ((2ull << hi) - 1ull);
    V[f] = TA<R>::scale_by(omega<R>(tlo, thi, r << (P.n - hi - 1), P.nl), sc);
  }
}

// The program's operators on the staged tile sm (2^{k+c} elements), with a
// barrier after each shared-memory round trip.
template <typename R>
__device__ __forceinline__ void tile_ops(typename TA<R>::E* sm, const TileProg<R>& P, const typename TA<R>::E* LAD,
                                         int kl) {
  using A = TA<R>;
  using E = typename A::E;
  const int c = P.c;
  const int NE = 1 << (P.k + c);
  for (int o = 0; o < P.nops; ++o) {
    const int b = c + P.q[o];
    const int kind = P.kind[o];
    // two butterfly levels on neighbouring qubits: one shared-memory round
    // trip (radix 4).  QFT levels come in descending order j, j-1; plain
    // Hadamard butterflies commute, so any neighbouring pair qualifies.
    if (kind != TOP_U2 && o + 1 < P.nops && P.kind[o + 1] == kind &&
        (P.q[o + 1] == P.q[o] - 1 || (kind == TOP_HB && P.q[o + 1] == P.q[o] + 1))) {
      const int jh = max(P.q[o], P.q[o + 1]), jl = jh - 1;  // levels jh then jl
      const int bh = c + jh, bl = c + jl;
      const bool lad = (kind == TOP_QFTLEVEL);
      for (int p = threadIdx.x; p < (NE >> 2); p += blockDim.x) {
        const int e00 = (int)insert0(insert0((uint64_t)p, bl), bh);
        const int e01 = e00 | (1 << bl), e10 = e00 | (1 << bh), e11 = e01 | (1 << bh);
        const E a00 = sm[e00], a01 = sm[e01], a10 = sm[e10], a11 = sm[e11];
        // level jh on bit bh: pairs (e00, e10), (e01, e11)
        const E s0 = A::add_u(a00, a10), d0 = A::sub_u(a00, a10);
        const E s1 = A::add_u(a01, a11), d1 = A::sub_u(a01, a11);
        E t0, u0, t1, u1;
        if (lad) {
          // With L(y) = e^{2 pi i y / 2^{jh+1}} and x = group bits below jl:
          // level jh multiplies d0 by L(x) and d1 by L(x + 2^jl) = i L(x);
          // level jl multiplies its bit-1 outputs by L(2x).  So
          //   t0 = s0 + s1,  u0 = L(2x) (s0 - s1),
          //   t1 = L(x) (d0 + i d1),  u1 = L(3x) (d0 - i d1):
          // three multiplications per four amplitudes instead of four.
          const int x = (e00 >> c) & ((1 << jl) - 1);
          const E id1 = A::times_i(d1);
          t0 = A::add(s0, s1);
          // the products renormalise u0, t1, u1; without one (x = 0) the
          // closing fast two-sum does
          u0 = A::sub_u(s0, s1);
          t1 = A::add_u(d0, id1);
          u1 = A::sub_u(d0, id1);
          if (x) {
            u0 = A::mul(ladder_at<R>(LAD, kl, jh, 2 * x), u0);
            t1 = A::mul(ladder_at<R>(LAD, kl, jh, x), t1);
            const int x3 = 3 * x;  // < 1.5 2^jh; L(y + 2^jh) = -L(y)
            u1 = A::mul(ladder_at<R>(LAD, kl, jh, x3 & ((1 << jh) - 1)), u1);
            if (x3 >> jh) u1 = A::neg(u1);
          } else {
            u0 = A::norm(u0);
            t1 = A::norm(t1);
            u1 = A::norm(u1);
          }
        } else {  // plain butterflies on both bits
          t0 = A::add(s0, s1);
          u0 = A::sub(s0, s1);
          t1 = A::add(d0, d1);
          u1 = A::sub(d0, d1);
        }
        sm[e00] = t0;
        sm[e01] = u0;
        sm[e10] = t1;
        sm[e11] = u1;
      }
      __syncthreads();
      ++o;
      continue;
    }
    if (kind == TOP_U2) {
      const int mk = P.mk[o];
      for (int p = threadIdx.x; p < (NE >> 1); p += blockDim.x) {
        const int e0 = (int)insert0((uint64_t)p, b), e1 = e0 | (1 << b);
        E a0 = sm[e0], a1 = sm[e1];
        A::u2(mk, P.U[o], a0, a1);
        sm[e0] = a0;
        sm[e1] = a1;
      }
    } else {
      // unnormalised butterfly (a0 + a1, a0 - a1); for a QFT level the
      // bit-1 half then takes the ladder phase e^{2 pi i x / 2^{j+1}}
      // = omega_k^{x 2^{k-j-1}}, x = group bits below group qubit j
      const int j = P.q[o];
      const bool lad = (kind == TOP_QFTLEVEL);
      for (int p = threadIdx.x; p < (NE >> 1); p += blockDim.x) {
        const int e0 = (int)insert0((uint64_t)p, b), e1 = e0 | (1 << b);
        const E a0 = sm[e0], a1 = sm[e1];
        sm[e0] = A::add(a0, a1);
        E d = A::sub(a0, a1);
        if (lad) {
          const int x = (e0 >> c) & ((1 << j) - 1);
          if (x) d = A::mul(ladder_at<R>(LAD, kl, j, x), d);
        }
        sm[e1] = d;
      }
    }
    __syncthreads();
  }
}

// The tile back to the state: twiddle (which carries the 2^{-p/2} scale) or
// the bare scale.
template <typename R>
__device__ __forceinline__ void tile_store(typename CT<R>::V2* __restrict__ s, uint64_t T, const typename TA<R>::E* sm,
                                           const TileProg<R>& P, const typename TA<R>::E* V,
                                           const typename TA<R>::E* TWA, const typename TA<R>::E* TWB,
                                           typename TA<R>::S sc) {
  using A = TA<R>;
  using E = typename A::E;
  using V2 = typename CT<R>::V2;
  const int lo = P.lo, k = P.k, c = P.c;
  const int NE = 1 << (k + c), cm = (1 << c) - 1;
  const bool own = P.base < c;  // contiguous bits of the register's
  // the staged element that goes to place e
  const int keep = cm | ~0 << (c + P.rev);
  auto from = [&](int e) {
    return P.rev ? (int)((__brev((unsigned)(e >> c)) >> (32 - P.rev)) << c) | (e & keep) : e;
  };
  auto twiddled = [&](int e, E z) {
    const int f = (int)(__brev((unsigned)(e >> c)) >> (32 - k));
    E w = V[f];
    if (own) {
      const int x = ((e & cm) >> P.base) * f;  // < 2^{c+k}
      w = A::mul(w, A::mul(TWA[x & 127], TWB[x >> 7]));
    }
    return A::mul(w, z);
  };
  if (sizeof(R) == 8) {
    for (int e = threadIdx.x; e < NE; e += blockDim.x) {
      E z = sm[from(e)];
      if (P.twiddle) z = twiddled(e, z);
      else if (P.scale_p) z = A::scale_by(z, sc);
      s[tile_global(e, T, lo, k, c)] = A::to(z);
    }
  } else {
    for (int e = 2 * threadIdx.x; e < NE; e += 2 * blockDim.x) {
      E z0 = sm[from(e)], z1 = sm[from(e + 1)];
      if (P.twiddle) {
        z0 = twiddled(e, z0);
        z1 = twiddled(e + 1, z1);
      } else if (P.scale_p) {
        z0 = A::scale_by(z0, sc);
        z1 = A::scale_by(z1, sc);
      }
      const V2 w0 = A::to(z0), w1 = A::to(z1);
      *reinterpret_cast<float4*>(s + tile_global(e, T, lo, k, c)) = make_float4(w0.x, w0.y, w1.x, w1.y);
    }
  }
}

// Two CTAs per SM (64 registers): every layer program and the complex128 QFT.
template <typename R>
__global__ void __launch_bounds__(512, 2) k_tile(typename CT<R>::V2* __restrict__ s, uint64_t ntiles,
                                                 const TileProg<R> P, const typename CT<R>::V2* __restrict__ tlo,
                                                 const typename CT<R>::V2* __restrict__ thi,
                                                 const typename CT<R>::V2* __restrict__ lad) {
  using A = TA<R>;
  using E = typename A::E;
  using V2 = typename CT<R>::V2;
  extern __shared__ __align__(16) unsigned char smraw[];
  E* sm = reinterpret_cast<E*>(smraw);
  const int lo = P.lo, k = P.k, c = P.c;
  const int NE = 1 << (k + c);
  E* V = sm + NE;
  E* LAD = V + (P.twiddle ? (1 << k) : 0);
  const int kl = lad_levels<R>(P.qft);  // levels in the table
  E* TWA = LAD + (P.qft ? lad_entries<R>(P.qft) : 0);
  E* TWB = TWA + TS_TWA;
  const typename A::S sc = A::scale_const(P.scale_p);
  tile_tables<R>(P, lad, LAD, TWA, TWB);
  for (uint64_t T = blockIdx.x; T < ntiles; T += gridDim.x) {
    if (P.twiddle) tile_twiddle_v<R>(P, T, V, tlo, thi, sc);
    // load: 16-byte vectors; for complex64 two neighbouring elements (c >= 1
    // or a fully contiguous tile, so e and e+1 are neighbours in memory);
    // four 16-byte loads in flight per thread before the first shared-memory
    // store (the tile is read once; with two CTAs per SM the load phase is
    // otherwise latency bound)
    constexpr int LU = 4;
    if (sizeof(R) == 8) {
      for (int e0 = threadIdx.x; e0 < NE; e0 += LU * blockDim.x) {
        V2 v[LU];
#pragma unroll
        for (int u = 0; u < LU; ++u) {
          const int e = e0 + u * blockDim.x;
          if (e < NE) v[u] = s[tile_global(e, T, lo, k, c)];
        }
#pragma unroll
        for (int u = 0; u < LU; ++u) {
          const int e = e0 + u * blockDim.x;
          if (e < NE) sm[e] = A::from(v[u]);
        }
      }
    } else {
      for (int e0 = 2 * threadIdx.x; e0 < NE; e0 += 2 * LU * blockDim.x) {
        float4 v[LU];
#pragma unroll
        for (int u = 0; u < LU; ++u) {
          const int e = e0 + 2 * u * blockDim.x;
          if (e < NE) v[u] = *reinterpret_cast<const float4*>(s + tile_global(e, T, lo, k, c));
        }
#pragma unroll
        for (int u = 0; u < LU; ++u) {
          const int e = e0 + 2 * u * blockDim.x;
          if (e < NE) {
            sm[e] = A::from(CT<R>::make(v[u].x, v[u].y));
            sm[e + 1] = A::from(CT<R>::make(v[u].z, v[u].w));
          }
        }
      }
    }
    __syncthreads();
    tile_ops<R>(sm, P, LAD, kl);
    tile_store<R>(s, T, sm, P, V, TWA, TWB, sc);
    __syncthreads();
  }
}

// ------------------------------------------------ complex128 QFT passes --
// For states of at least 12 qubits every complex128 QFT pass has k + c = 12,
// so the pass is compiled per group size K: the radix-4 level pairs' bit
// positions are constants, the tile is XOR-swizzled in 16-byte elements
// (bits 0..2 take bits 3..5, which is linear over XOR, so every element of a
// radix-4 quad is one XOR away from the thread's base and the low-bit
// stages are free of bank conflicts), and a thread's eight load / store
// addresses are one base plus multiples of a per-pass stride.  The
// arithmetic is that of k_tile's QFT programs.
__device__ __forceinline__ int tsw(int e) { return e ^ ((e >> 3) & 7); }

template <int BH, int BL, int JH, int C>
__device__ __forceinline__ void qft_quad_c128(ffc* sm, const ffc* LAD, int kl) {
  using A = TA<double>;
  constexpr int NE = 1 << 12, JL = JH - 1;
  static_assert(BH == BL + 1, "neighbouring levels");
#pragma unroll
  for (int r = 0; r < (NE >> 2) / 512; ++r) {
    const int p = threadIdx.x + 512 * r;
    const int e00 = ((p >> BL) << (BL + 2)) | (p & ((1 << BL) - 1));
    const int b = tsw(e00);
    const int o01 = tsw(1 << BL), o10 = tsw(1 << BH), o11 = tsw(3 << BL);
    const ffc a00 = sm[b], a01 = sm[b ^ o01], a10 = sm[b ^ o10], a11 = sm[b ^ o11];
    const ffc s0 = A::add_u(a00, a10), d0 = A::sub_u(a00, a10);
    const ffc s1 = A::add_u(a01, a11), d1 = A::sub_u(a01, a11);
    // as in k_tile: t0 = s0 + s1, u0 = L(2x)(s0 - s1), t1 = L(x)(d0 + i d1),
    // u1 = L(3x)(d0 - i d1), L(y) = e^{2 pi i y / 2^{JH+1}}, x = group bits below JL
    const int x = (e00 >> C) & ((1 << JL) - 1);
    const ffc id1 = A::times_i(d1);
    const ffc t0 = A::add(s0, s1);
    ffc u0 = A::sub_u(s0, s1), t1 = A::add_u(d0, id1), u1 = A::sub_u(d0, id1);
    if (x) {
      u0 = A::mul(ladder_at<double>(LAD, kl, JH, 2 * x), u0);
      t1 = A::mul(ladder_at<double>(LAD, kl, JH, x), t1);
      const int x3 = 3 * x;
      u1 = A::mul(ladder_at<double>(LAD, kl, JH, x3 & ((1 << JH) - 1)), u1);
      if (x3 >> JH) u1 = A::neg(u1);
    } else {
      u0 = A::norm(u0);
      t1 = A::norm(t1);
      u1 = A::norm(u1);
    }
    sm[b] = t0;
    sm[b ^ o01] = u0;
    sm[b ^ o10] = t1;
    sm[b ^ o11] = u1;
  }
}

// level 0 alone (odd K): plain butterflies on tile bit C (no ladder below it)
template <int C>
__device__ __forceinline__ void qft_single0_c128(ffc* sm) {
  using A = TA<double>;
  constexpr int NE = 1 << 12;
#pragma unroll
  for (int r = 0; r < (NE >> 1) / 512; ++r) {
    const int p = threadIdx.x + 512 * r;
    const int e0 = ((p >> C) << (C + 1)) | (p & ((1 << C) - 1));
    const int b = tsw(e0), o = tsw(1 << C);
    const ffc a0 = sm[b], a1 = sm[b ^ o];
    sm[b] = A::add(a0, a1);
    sm[b ^ o] = A::sub(a0, a1);
  }
}

// levels JH, JH-1 as one quad stage, then the rest
template <int K, int JH>
__device__ __forceinline__ void qft_stages_c128(ffc* sm, const ffc* LAD, int kl) {
  constexpr int C = 12 - K;
  if constexpr (JH >= 1) {
    qft_quad_c128<C + JH, C + JH - 1, JH, C>(sm, LAD, kl);
    __syncthreads();
    qft_stages_c128<K, JH - 2>(sm, LAD, kl);
  } else if constexpr (JH == 0) {
    qft_single0_c128<C>(sm);
    __syncthreads();
  }
}

// Between the passes of one transform the state holds each amplitude's
// double-float parts (re.hi, re.lo, im.hi, im.lo: the same 16 bytes), so
// only the first pass converts from IEEE double, and the bit reversal that
// ends the transform converts back.
__device__ __forceinline__ ffc ffc_unpack(double2 v) {
  return ffc_make(ff_make(__int_as_float(__double2loint(v.x)), __int_as_float(__double2hiint(v.x))),
                  ff_make(__int_as_float(__double2loint(v.y)), __int_as_float(__double2hiint(v.y))));
}
__device__ __forceinline__ double2 ffc_pack(ffc z) {
  return make_double2(__hiloint2double(__float_as_int(z.re.lo), __float_as_int(z.re.hi)),
                      __hiloint2double(__float_as_int(z.im.lo), __float_as_int(z.im.hi)));
}

template <int K>
__global__ void __launch_bounds__(512, 2) k_qft_c128_k(double2* __restrict__ s, uint64_t ntiles, const TileProg<double> P,
                                                       const double2* __restrict__ tlo,
                                                       const double2* __restrict__ thi,
                                                       const double2* __restrict__ lad, int ld_ff, int st_ff) {
  using A = TA<double>;
  constexpr int C = 12 - K, NE = 1 << 12, PER = NE / 512;
  static_assert(C <= 9, "512-element strides stay inside the group bits");
  static_assert(PER == 8, "eight elements per thread");
  extern __shared__ __align__(16) unsigned char smraw[];
  ffc* sm = reinterpret_cast<ffc*>(smraw);
  const int lo = P.lo, hi = lo + K - 1, sh = P.n - hi - 1, nl = P.nl;
  const bool tw = P.twiddle != 0;
  ffc* LAD = sm + NE;
  constexpr int kl = lad_levels<double>(K);
#pragma unroll 1
  for (int a = threadIdx.x; a < lad_entries<double>(K); a += blockDim.x) LAD[a] = LadIO<double>::ld(lad + a);
  const typename A::S sc = A::scale_const(K);
  const int tid = threadIdx.x;
  const int st = tsw(tid);
  const uint64_t gstep = (uint64_t)(512 >> C) << lo;
  const uint64_t hm = (2ull << hi) - 1ull;
  // twiddle of element e = tid + 512 u: 2^{-K/2} Omega_{hi+1}^{m f} with
  // m = its bits below lo (the tile's bits between C and lo, then the C low
  // bits of tid: the same for all eight elements of a thread) and
  // f = brev_K(e >> C) = F + brev_3(u), F = brev_K(tid >> C) (a multiple of
  // 8).  So the eight twiddles are B g^v, v = brev_3(u), with
  // B = 2^{-K/2} Omega^{m F} and g = Omega^m: two root-table lookups and a
  // chain of seven products per thread instead of two products per element.
  const int F = (int)(__brev((unsigned)(tid >> C)) >> (32 - K));
  for (uint64_t T = blockIdx.x; T < ntiles; T += gridDim.x) {
    const uint64_t g0 = tile_global((uint64_t)tid, T, lo, K, C);
    // four 16-byte loads in flight per thread, twice
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      double2 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = s[g0 + (4 * h + u) * gstep];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        sm[st ^ tsw(512 * (4 * h + u))] =
            ld_ff ? ffc_unpack(v[u]) : ffc_make(ff_from_d_fast(v[u].x), ff_from_d_fast(v[u].y));
    }
    __syncthreads();
    qft_stages_c128<K, K - 1>(sm, LAD, kl);
    // store: the twiddle (which carries the 2^{-K/2} scale), or the scale
    if (tw) {
      const uint64_t m = ((T & ((1ull << (lo - C)) - 1ull)) << C) | (uint64_t)(tid & ((1 << C) - 1));
      ffc W = A::scale_by(omega<double>(tlo, thi, ((m * (uint64_t)F) & hm) << sh, nl), sc);
      const ffc g = omega<double>(tlo, thi, (m & hm) << sh, nl);
#pragma unroll
      for (int v = 0; v < PER; ++v) {
        const int u = ((v & 1) << 2) | (v & 2) | (v >> 2);  // brev_3(v)
        const ffc z = A::mul(W, sm[st ^ tsw(512 * u)]);
        s[g0 + u * gstep] = st_ff ? ffc_pack(z) : A::to(z);
        if (v + 1 < PER) W = A::mul(W, g);
      }
    } else {
#pragma unroll
      for (int u = 0; u < PER; ++u) {
        const ffc z = A::scale_by(sm[st ^ tsw(512 * u)], sc);
        s[g0 + u * gstep] = st_ff ? ffc_pack(z) : A::to(z);
      }
    }
    __syncthreads();
  }
}

// ------------------------------------------------- complex64 QFT passes --
// Bound by memory latency and shared-memory round trips.  On a 2^13-amplitude
// tile (k_qft_c64_k) two CTAs share an SM, each with one 64 KiB tile: while
// one waits at its barriers or for its loads, the other computes.  What is the
// same for every tile (the twiddles W, the ladders) is built once per
// transform and read through L1, which is what makes room for the second tile.
// 29 qubits, an 8-level pass above the lowest group: 2.16 ms with one CTA of two
// buffers; 1.39 ms (0.91 of the copy bandwidth) with two CTAs, the first levels
// straight from the state and the last straight to it.
// The group's levels run in register blocks
// of up to four levels (one shared-memory round trip each).  Within a block
// on group qubits jlo .. jlo+QR-1, level j = jlo + lv multiplies the
// difference of the pair with local low bits m by
//   L_j(x) = e^{2 pi i x / 2^{j+1}},  x = m 2^jlo + xlow,
// read from the ladder table (one rounding; a constant root times L_j(xlow)
// has two).  The lowest block's are constants.  The shared tile is swizzled in
// 16-byte units:
// strided register blocks then hit at most twice the minimum number of
// shared-memory wavefronts instead of up to 16x.
__device__ __forceinline__ int qsw(int e) { return e ^ (((e >> 4) & 7) << 1); }

__device__ __forceinline__ float2 c2mul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// e^{2 pi i m / 2^{lv+1}} for m < 2^lv, lv <= 3 (constants)
__device__ __forceinline__ float2 qroot(int lv, int m) {
  const float r = 0.70710678118654752f, c1 = 0.92387953251128676f, s1 = 0.38268343236508977f;
  if (lv <= 0 || m == 0) return make_float2(1.f, 0.f);
  if (lv == 1) return make_float2(0.f, 1.f);
  if (lv == 2) {
    switch (m) {
      case 1: return make_float2(r, r);
      case 2: return make_float2(0.f, 1.f);
      default: return make_float2(-r, r);
    }
  }
  switch (m) {  // lv == 3: sixteenth roots e^{2 pi i m / 16}
    case 1: return make_float2(c1, s1);
    case 2: return make_float2(r, r);
    case 3: return make_float2(s1, c1);
    case 4: return make_float2(0.f, 1.f);
    case 5: return make_float2(-s1, c1);
    case 6: return make_float2(-r, r);
    default: return make_float2(-c1, s1);
  }
}

// States of at least 13 qubits (smaller ones: the general tile program).
// Every tile holds 2^13 amplitudes (k + c = 13): the register blocks' bit
// positions, the swizzled offsets of a block's elements and a thread's
// copy and store offsets are constants, so the index arithmetic is one XOR
// per element.  qsw is linear over XOR, qsw(x ^ y) = qsw(x) ^ qsw(y).
template <int QR, int JLO>
__device__ __forceinline__ void qft_butterflies_c64(float2* a, const float2* LAD, int xlow) {
  constexpr int NR = 1 << QR;
#pragma unroll
  for (int lv = QR - 1; lv >= 0; --lv) {
    const int j = JLO + lv;
#pragma unroll
    for (int i = 0; i < NR; ++i) {
      if ((i >> lv) & 1) continue;
      const int i1 = i | (1 << lv);
      const float2 x0 = a[i], x1 = a[i1];
      a[i] = make_float2(x0.x + x1.x, x0.y + x1.y);
      const int m = i & ((1 << lv) - 1);
      const float2 d = make_float2(x0.x - x1.x, x0.y - x1.y);
      if (JLO) a[i1] = c2mul(d, LAD[(1 << j) - 1 + (m << JLO) + xlow]);  // L_j(m 2^jlo + xlow)
      else a[i1] = m ? c2mul(d, qroot(lv, m)) : d;
    }
  }
}

template <int QR, int BL, int JLO>
__device__ __forceinline__ void qft_block_c64_ct(float2* sm, const float2* LAD) {
  constexpr int NR = 1 << QR, NE = 1 << 13;
  constexpr int C = BL - JLO;
#pragma unroll
  for (int r = 0; r < (NE >> QR) / 512; ++r) {
    const int p = threadIdx.x + 512 * r;
    const int base = ((p >> BL) << (BL + QR)) | (p & ((1 << BL) - 1));
    const int sb = qsw(base);
    float2 a[NR];
#pragma unroll
    for (int i = 0; i < NR; ++i) a[i] = sm[sb ^ qsw(i << BL)];
    qft_butterflies_c64<QR, JLO>(a, LAD, (base >> C) & ((1 << JLO) - 1));
#pragma unroll
    for (int i = 0; i < NR; ++i) sm[sb ^ qsw(i << BL)] = a[i];
  }
}

// The first block (the group's top QR levels, tile bits 13 - QR ..) straight
// from the state: a warp's elements are rows of 2^C consecutive amplitudes,
// and a thread's 2^QR loads are in flight together.  A round trip through
// shared memory and its barrier fewer.
template <int K, int QR>
__device__ __forceinline__ void qft_first_block_load_c64(float2* sm, const float2* LAD, const float2* __restrict__ s,
                                                         uint64_t T, int lo) {
  constexpr int NR = 1 << QR, NE = 1 << 13, C = 13 - K, BL = 13 - QR, JLO = K - QR;
#pragma unroll
  for (int r = 0; r < (NE >> QR) / 512; ++r) {
    const int base = threadIdx.x + 512 * r;
    const uint64_t g = tile_global((uint64_t)base, T, lo, K, C), step = (uint64_t)(1 << JLO) << lo;
    float2 a[NR];
#pragma unroll
    for (int i = 0; i < NR; ++i) a[i] = s[g + i * step];
    qft_butterflies_c64<QR, JLO>(a, LAD, (base >> C) & ((1 << JLO) - 1));
    const int sb = qsw(base);
#pragma unroll
    for (int i = 0; i < NR; ++i) sm[sb ^ qsw(i << BL)] = a[i];
  }
}

// block b of the K levels: ceil(K/4) blocks, balanced, the larger first
__host__ __device__ constexpr int qft_nblocks(int K) { return (K + 3) >> 2; }
__host__ __device__ constexpr int qft_block_size(int K, int b) {
  int j = K - 1, qr = 0;
  for (int i = 0; i <= b; ++i) {
    const int nb = qft_nblocks(K);
    qr = (j + 1 + (nb - i) - 1) / (nb - i);
    if (i < b) j -= qr;
  }
  return qr;
}
__host__ __device__ constexpr int qft_block_jlo(int K, int b) {
  int j = K - 1;
  for (int i = 0; i <= b; ++i) j -= qft_block_size(K, i);
  return j + 1;
}

// blocks B .. END-1 of the K levels, a barrier after each
template <int K, int B, int END>
__device__ __forceinline__ void qft_levels_c64_ct(float2* sm, const float2* LAD) {
  if constexpr (B < END) {
    constexpr int QR = qft_block_size(K, B), JLO = qft_block_jlo(K, B), C = 13 - K;
    qft_block_c64_ct<QR, C + JLO, JLO>(sm, LAD);
    __syncthreads();
    qft_levels_c64_ct<K, B + 1, END>(sm, LAD);
  }
}

// The last block (levels QR-1 .. 0, on tile bits C .. C+QR-1) of a twiddle
// pass, written straight to the state: element i of a thread's block has
// group bits (base >> C) | i, so its state index is the block base's plus
// i << lo, and its twiddle is W[e] V[f] with f = brev(base >> C) | brev(i).
// Consecutive threads hold consecutive low bits (2^C >= 16 amplitudes, at
// least 128 contiguous bytes per warp and element).
template <int K, int QR>
__device__ __forceinline__ void qft_last_block_store_c64(const float2* sm, const float2* LAD, const float2* __restrict__ W,
                                                         const float2* V, float2* __restrict__ s, uint64_t T,
                                                         int lo) {
  constexpr int NR = 1 << QR, NE = 1 << 13, C = 13 - K, BL = C;
#pragma unroll
  for (int r = 0; r < (NE >> QR) / 512; ++r) {
    const int p = threadIdx.x + 512 * r;
    const int base = ((p >> BL) << (BL + QR)) | (p & ((1 << BL) - 1));
    const int sb = qsw(base);
    float2 a[NR];
#pragma unroll
    for (int i = 0; i < NR; ++i) a[i] = sm[sb ^ qsw(i << BL)];
    qft_butterflies_c64<QR, 0>(a, LAD, 0);  // every level's ladder phase is a constant root
    const uint64_t g = tile_global((uint64_t)base, T, lo, K, C);
    const int fb = (int)(__brev((unsigned)(base >> C)) >> (32 - K));
#pragma unroll
    for (int i = 0; i < NR; ++i) {
      const int f = fb | (int)(__brev((unsigned)i) >> (32 - K));
      s[g + ((uint64_t)i << lo)] = c2mul(c2mul(a[i], W[base | (i << BL)]), V[f]);
    }
  }
}

template <int K>
__global__ void __launch_bounds__(512, 2) k_qft_c64_k(float2* __restrict__ s, uint64_t ntiles, int lo,
                                                      const float2* __restrict__ W,
                                                      const float2* __restrict__ lad) {
  constexpr int C = 13 - K, NE = 1 << 13;
  static_assert(C <= 10, "1024-element copy strides stay inside the group bits");
  extern __shared__ __align__(16) unsigned char smraw[];
  const int hi = lo + K - 1;
  float2* cur = reinterpret_cast<float2*>(smraw);
  float2* V = cur + NE;
  float2* LAD = V + (1 << K);
  const float sc = (float)exp2(-0.5 * K);
  const int e0 = 2 * threadIdx.x;
  const int se0 = qsw(e0);
  const uint64_t gstep = (uint64_t)(1024 >> C) << lo;
  // this thread's copy / store elements e0 + 1024 u share the group bits'
  // low part; their reversed group bits are f0 | brev(u) at the top
  const int f0 = (int)(__brev((unsigned)(e0 >> C)) >> (32 - K));
  for (int a = threadIdx.x; a < (1 << K) - 1; a += blockDim.x) LAD[a] = lad[a];
  __syncthreads();
  constexpr int NB = qft_nblocks(K);
  for (uint64_t T = blockIdx.x; T < ntiles; T += gridDim.x) {
    // V[f] = Omega_{hi+1}^{Lt f} sc: the angle in two floats, the low one a
    // small rotation (closer than a product of two rounded table entries)
    const uint64_t Lt = (T & ((1ull << (lo - C)) - 1ull)) << C;
    for (int f = threadIdx.x; f < (1 << K); f += blockDim.x) {
      const uint64_t r = (Lt * (uint64_t)f) & ((2ull << hi) - 1ull);
      const float ah = (float)r, al = (float)((int64_t)r - (int64_t)ah);
      float vr, vi;
      sincospif(ldexpf(ah, -hi), &vi, &vr);
      const float d = ldexpf(al * 3.14159265358979f, -hi);
      V[f] = make_float2(fmaf(-vi, d, vr) * sc, fmaf(vr, d, vi) * sc);
    }
    qft_first_block_load_c64<K, qft_block_size(K, 0)>(cur, LAD, s, T, lo);
    __syncthreads();
    if constexpr (NB >= 2) {  // the last block goes straight to the state
      qft_levels_c64_ct<K, 1, NB - 1>(cur, LAD);
      qft_last_block_store_c64<K, qft_block_size(K, NB - 1)>(cur, LAD, W, V, s, T, lo);
    } else {
      const uint64_t g = tile_global((uint64_t)e0, T, lo, K, C);
#pragma unroll
      for (int u = 0; u < NE / 1024; ++u) {
        const float4 z = *reinterpret_cast<const float4*>(cur + (se0 ^ qsw(1024 * u)));
        // the group bits of e0 + 1024 u are (e0 >> C) + (1024 u >> C): reversed,
        // brev(u) lands below f0's bits
        const int f = f0 | (int)(__brev((unsigned)((1024 * u) >> C)) >> (32 - K));
        const float2 v = V[f];
        const float4 w = *reinterpret_cast<const float4*>(W + e0 + 1024 * u);
        const float2 z0 = c2mul(c2mul(make_float2(z.x, z.y), make_float2(w.x, w.y)), v);
        const float2 z1 = c2mul(c2mul(make_float2(z.z, z.w), make_float2(w.z, w.w)), v);
        *reinterpret_cast<float4*>(s + g + u * gstep) = make_float4(z0.x, z0.y, z1.x, z1.y);
      }
    }
    __syncthreads();
  }
}

// The lowest QFTR_B levels with the reversal of all n index bits (see the bit
// reversal below for its tiles).  Index = (h, m, l), h and l of QFTR_B bits:
// the transform of a row (the 2^QFTR_B values of l) gives, at position p,
// frequency rev(p), whose place is (rev p, rev m, rev h).  The block for m
// (m <= rev m) reads the tiles of m and rev m, one level on its loads' way
// into shared memory and four on the way out, so that the levels cost no pass.
// 29 qubits: a 13-level lowest group took 2.07 ms and the reversal 1.72;
// an 8-level group and this kernel take 1.39 each (0.91 of the copy
// bandwidth), the whole QFT 6.76 -> 5.60 (8.16 with one CTA an SM).
constexpr int QFTR_B = 5;
constexpr int QFTR_T = 128;
__global__ void __launch_bounds__(QFTR_T, 8) k_qft_rev_c64(float2* __restrict__ s, int n, const float2* __restrict__ lad) {
  constexpr int B = QFTR_B, W = 1 << B, WP = W + 1;
  static_assert(B == 5 && QFTR_T == 128, "two warps a tile, sixteen amplitudes a thread");
  __shared__ float2 A[2][W * WP];
  const int lane = threadIdx.x & 31, w = (threadIdx.x >> 5) & 1, t = threadIdx.x >> 6;
  const int nm = n - 2 * B;
  const uint64_t M = 1ull << nm;
  const float sc = (float)exp2(-0.5 * B);
  // loads: l = 2j, 2j + 1 and 16 above them, of rows r0 + 8 u; a half-warp's
  // two rows are neighbours, so that its stores to the padded tile hit every bank
  const int j = lane & 7, r0 = (lane >> 3) | (w << 2);
  const float2 c0 = lad[(1 << (B - 1)) - 1 + 2 * j], c1 = lad[(1 << (B - 1)) + 2 * j];
  // stores: positions 16 w + i, i < 16, of row rev(lane)
  const int rr = (int)(__brev((unsigned)lane) >> (32 - B));
  for (uint64_t m = blockIdx.x; m < M; m += gridDim.x) {
    const uint64_t mr = nm ? (__brevll((unsigned long long)m) >> (64 - nm)) : 0ull;
    if (mr < m) continue;
    const bool act = t == 0 || mr != m;
    if (act) {
      const float2* g = s + (((uint64_t)r0 << (n - B)) | ((t ? mr : m) << B) | (uint64_t)(2 * j));
      float4 x[4], y[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        x[u] = *reinterpret_cast<const float4*>(g + ((uint64_t)(8 * u) << (n - B)));
        y[u] = *reinterpret_cast<const float4*>(g + ((uint64_t)(8 * u) << (n - B)) + 16);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {  // the top level
        float2* o = A[t] + (r0 + 8 * u) * WP + 2 * j;
        o[0] = make_float2(x[u].x + y[u].x, x[u].y + y[u].y);
        o[1] = make_float2(x[u].z + y[u].z, x[u].w + y[u].w);
        o[16] = c2mul(make_float2(x[u].x - y[u].x, x[u].y - y[u].y), c0);
        o[17] = c2mul(make_float2(x[u].z - y[u].z, x[u].w - y[u].w), c1);
      }
    }
    __syncthreads();
    if (act) {
      float2 a[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) a[i] = A[t][rr * WP + 16 * w + i];
      qft_butterflies_c64<4, 0>(a, lad, 0);
      float2* g = s + (((uint64_t)w << (n - B)) | ((t ? m : mr) << B) | (uint64_t)lane);
#pragma unroll
      for (int i = 0; i < 16; ++i)
        g[(uint64_t)(__brev((unsigned)i) >> (32 - 4)) << (n - B + 1)] = make_float2(a[i].x * sc, a[i].y * sc);
    }
    __syncthreads();
  }
}

// Tables of Omega^a (a < 2^nl) and Omega^{a 2^nl} (a < 2^{n-nl}),
// Omega = e^{2 pi i / 2^n}, from sincospi in double precision, and the first
// nlad entries of the ladder table: level j's e^{2 pi i x / 2^{j+1}} at
// 2^j - 1 + x (complex128: e^{2 pi i / 2^12} at 2047).
template <typename R>
__global__ void k_roots(typename CT<R>::V2* tlo, typename CT<R>::V2* thi, int n, int nl, typename CT<R>::V2* lad,
                        int nlad) {
  const uint64_t nlo = 1ull << nl, nhi = 1ull << (n - nl);
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nlo + nhi + (uint64_t)nlad;
       i += (uint64_t)gridDim.x * blockDim.x) {
    if (i >= nlo + nhi) {
      const int a = (int)(i - nlo - nhi), j = 31 - __clz(a + 1);
      const bool extra = sizeof(R) == 8 && a == 2047;
      LadIO<R>::st(lad + a, extra ? TA<R>::root(1, 12) : TA<R>::root((uint64_t)(a + 1 - (1 << j)), j + 1));
      continue;
    }
    const bool low = i < nlo;
    const uint64_t a = low ? i : (i - nlo);
    // angle / pi = 2 a 2^{shift} / 2^n, reduced mod 2 exactly in integers
    const int shift = low ? 0 : nl;
    const uint64_t num = (a << (shift + 1)) & ((2ull << n) - 1ull);  // mod 2^{n+1}
    const double x = ldexp((double)num, -n);
    double sn, cs;
    sincospi(x, &sn, &cs);
    if (low) tlo[a] = CT<R>::make((R)cs, (R)sn);
    else thi[a] = CT<R>::make((R)cs, (R)sn);
  }
}

// --------------------------------------------------------------------------
// Tile-size choices: c low contiguous bits give 128-byte rows; k group bits;
// the tile holds 2^{k+c} amplitudes (64 KiB: 2^12 complex128 or 2^13
// complex64 amplitudes, 128 KiB for complex64 layer groups of 10): 30
// complex128 qubits in three QFT passes, 12 + 9 + 9, 32 complex64 qubits in
// four, 5 + 9 + 9 + 9 (the lowest five with the bit reversal).
template <typename R> struct TileCfg;
template <> struct TileCfg<double> { static constexpr int C = 3, K = 9, BOT = 12; };
// the ladder helper reaches one level past the table (levels 0..10)
static_assert(TileCfg<double>::BOT <= 12 && TileCfg<double>::K <= 12, "complex128 groups of at most 12 qubits");
// complex64 layers: 128 KiB tiles for groups of 10 (c = 4, one CTA per SM),
// 64 KiB for smaller ones; the complex64 QFT of 13 qubits and more has groups of
// its own (qft_groups_c64)
template <> struct TileCfg<float> { static constexpr int C = 4, K = 10, BOT = 13; };

struct Group {
  int lo, k;
};

// Groups covering qubits [0, n): the lowest group up to bot qubits (no
// separate contiguous bits needed), the others up to K, balanced.
static std::vector<Group> plan_groups_k(int n, int bot, int K) {
  std::vector<Group> g;
  const int g0 = std::min(n, bot);
  g.push_back({0, g0});
  int rest = n - g0;
  if (rest > 0) {
    const int np = (rest + K - 1) / K;
    int lo = g0;
    for (int i = 0; i < np; ++i) {
      const int k = (rest + (np - i) - 1) / (np - i);  // balanced
      g.push_back({lo, k});
      lo += k;
      rest -= k;
    }
  }
  return g;
}

template <typename R>
static std::vector<Group> plan_groups(int n) {
  return plan_groups_k(n, TileCfg<R>::BOT, TileCfg<R>::K);
}

template <typename R>
static size_t tile_smem(int k, int c, bool twiddle, int qft) {
  using E = typename TA<R>::E;
  return sizeof(E) * (((size_t)1 << (k + c)) + (twiddle ? ((size_t)1 << k) : 0) +
                      (qft ? (size_t)lad_entries<R>(qft) : 0) + TS_TWA + TS_TWB);
}

template <typename R>
static qc_status run_tile(qc_state* s, TileProg<R>& P, const typename CT<R>::V2* tlo = nullptr,
                          const typename CT<R>::V2* thi = nullptr, const typename CT<R>::V2* lad = nullptr) {
  using V2 = typename CT<R>::V2;
  if (P.nops == 0 && !P.twiddle) return QC_OK;
  const int tb = P.k + P.c;
  const uint64_t ntiles = 1ull << (s->n - tb);
  const size_t smem = tile_smem<R>(P.k, P.c, P.twiddle != 0, P.qft);
  const int threads = std::max(64, std::min(512, (1 << tb) >> 2));  // four amplitudes a thread
  allow_smem(k_tile<R>, 200 * 1024);
  const unsigned grid = resident_grid(k_tile<R>, threads, (int64_t)ntiles, 1, smem);
  k_tile<R><<<grid, threads, smem, s->stream>>>(reinterpret_cast<V2*>(s->data), ntiles, P, tlo, thi, lad);
  return check_launch("tile pass");
}

// complex128 QFT pass: the compiled kernel for 2^12-amplitude tiles, else
// the general tile program.
static bool qft_c128_compiled(const TileProg<double>& P) {
  return P.k + P.c == 12 && P.scale_p == P.k && P.nops == P.k && ((P.k >= 3 && P.k <= 9) || P.k == 12);
}

// ld_ff / st_ff: the pass reads / leaves the double-float form (compiled
// passes only; the transform's first pass reads IEEE doubles, and the bit
// reversal after its last pass converts back).
static qc_status run_qft_c128(qc_state* s, TileProg<double>& P, const double2* tlo, const double2* thi,
                              const double2* lad, bool ld_ff, bool st_ff) {
  if (qft_c128_compiled(P)) {
    const uint64_t ntiles = 1ull << (s->n - 12);
    const size_t smem = sizeof(ffc) * (((size_t)1 << 12) + (size_t)lad_entries<double>(P.k));
    double2* d = reinterpret_cast<double2*>(s->data);
    switch (P.k) {
#define QC_QFT_C128(KK)                                                                             \
  case KK: {                                                                                        \
    allow_smem(k_qft_c128_k<KK>, 200 * 1024);                                                       \
    const unsigned g = resident_grid(k_qft_c128_k<KK>, 512, (int64_t)ntiles, 1, smem);             \
    k_qft_c128_k<KK><<<g, 512, smem, s->stream>>>(d, ntiles, P, tlo, thi, lad, ld_ff, st_ff);       \
    return check_launch("qft pass");                                                                \
  }
      QC_QFT_C128(3) QC_QFT_C128(4) QC_QFT_C128(5) QC_QFT_C128(6) QC_QFT_C128(7) QC_QFT_C128(8)
      QC_QFT_C128(9) QC_QFT_C128(12)
#undef QC_QFT_C128
      default: break;
    }
  }
  if (ld_ff || st_ff) return QC_EINVAL;
  return run_tile<double>(s, P, tlo, thi, lad);
}

// complex64 QFT pass on a group of three to ten qubits (2^13-amplitude tiles).
static qc_status run_qft_c64(qc_state* s, const Group& g, const float2* W, const float2* lad) {
  const int64_t ntiles = (int64_t)1 << (s->n - 13);
  switch (g.k) {
#define QC_QFT_C64(KK)                                                                                  \
  case KK: {                                                                                            \
    const size_t smem = sizeof(float2) * ((1 << 13) + 2 * (1 << KK));                                   \
    allow_smem(k_qft_c64_k<KK>, smem);                                                                  \
    const unsigned grid = resident_grid(k_qft_c64_k<KK>, 512, ntiles, 1, smem);                         \
    k_qft_c64_k<KK><<<grid, 512, smem, s->stream>>>(reinterpret_cast<float2*>(s->data), (uint64_t)ntiles, g.lo, W, lad); \
    return check_launch("qft pass");                                                                    \
  }
    QC_QFT_C64(3) QC_QFT_C64(4) QC_QFT_C64(5) QC_QFT_C64(6) QC_QFT_C64(7) QC_QFT_C64(8) QC_QFT_C64(9) QC_QFT_C64(10)
#undef QC_QFT_C64
    default: return QC_EINVAL;
  }
}

// Contiguous low bits of a group's tile: at least C (128-byte rows) and, for
// small groups, enough to fill the tile to 2^TB amplitudes, so that a pass
// has few large tiles with long rows rather than many small ones (each tile
// costs a DRAM round trip before its compute).  TB: 64 KiB tiles (two CTAs
// per SM).  The QFT
// twiddle tables need c + k <= 14.
template <typename R>
static int tile_c(const Group& g) {
  const int TB = sizeof(R) == 8 ? 12 : 13;
  return std::min(g.lo, std::max(TileCfg<R>::C, TB - g.k));
}

template <typename R>
static void prog_init(TileProg<R>& P, const Group& g, int n) {
  P.nops = 0;
  P.lo = g.lo;
  P.k = g.k;
  P.c = tile_c<R>(g);
  P.n = n;
  P.base = 0;
  P.rev = 0;
  P.twiddle = 0;
  P.qft = 0;
  P.nl = 0;
  P.scale_p = 0;
}

// Hadamards (operators that are exactly h [[1,1],[1,-1]] with h = 1/sqrt 2)
// become unnormalised butterflies with the scale deferred to the store.
static bool is_exact_hadamard(const double* u) {
  const double h = 1.0 / sqrt(2.0);
  return u[0] == h && u[2] == h && u[4] == h && u[6] == -h && u[1] == 0 && u[3] == 0 && u[5] == 0 && u[7] == 0;
}

template <typename R>
static qc_status layer_impl(qc_state* s, const double* U, uint64_t mask) {
  for (const Group& g : plan_groups<R>(s->n)) {
    TileProg<R> P;
    prog_init(P, g, s->n);
    for (int j = 0; j < g.k; ++j) {
      const int q = g.lo + j;
      if (!((mask >> q) & 1)) continue;
      const MatKind mk = classify(U + 8 * q);
      if (mk == MK_IDENT) continue;
      P.q[P.nops] = (int8_t)j;
      if (is_exact_hadamard(U + 8 * q)) {
        P.kind[P.nops] = TOP_HB;
        P.mk[P.nops] = 0;
        ++P.scale_p;
      } else {
        P.kind[P.nops] = TOP_U2;
        P.mk[P.nops] = (int8_t)mk;
        P.U[P.nops] = TA<R>::mat(U + 8 * q);
      }
      ++P.nops;
    }
    qc_status st = run_tile<R>(s, P);
    if (st) return st;
  }
  return QC_OK;
}

qc_status launch_layer(qc_state* s, const double* U, uint64_t mask) {
  s->sum_valid = false;
  // a layer of Hadamards only (HALL among them): Walsh-Hadamard passes
  bool all_h = mask != 0;
  for (int q = 0; q < s->n && all_h; ++q)
    if ((mask >> q) & 1) all_h = is_exact_hadamard(U + 8 * q);
  if (all_h && s->n >= hadamard_layer_min_qubits(s->dt)) return launch_hadamard_layer(s, mask);
  return s->dt == QC_C128 ? layer_impl<double>(s, U, mask) : layer_impl<float>(s, U, mask);
}

qc_status launch_hall(qc_state* s) {
  std::vector<double> U(8 * (size_t)s->n);
  const double h = 1.0 / sqrt(2.0);
  for (int q = 0; q < s->n; ++q) {
    double* u = U.data() + 8 * q;
    const double v[8] = {h, 0, h, 0, h, 0, -h, 0};
    for (int i = 0; i < 8; ++i) u[i] = v[i];
  }
  const uint64_t mask = (s->n >= 64) ? ~0ull : ((1ull << s->n) - 1ull);
  return launch_layer(s, U.data(), mask);
}

// ------------------------------------------------------- bit reversal ----
// In-place reversal of all n index bits (complex128).  Index = (h, m, l) with h, l of B
// bits: rev(h, m, l) = (rev l, rev m, rev h).  The block for middle value m
// (with m <= rev m) exchanges the 2^B x 2^B tiles of m and rev m through
// shared memory (rows of 2^B contiguous amplitudes, padded against bank
// conflicts).  The pass is latency bound (load both tiles, synchronise,
// store), so many small blocks beat few large ones: B = 4
// with 128 threads (twelve blocks per SM; 0.89 of copy bandwidth on GB300
// at 30 qubits).  complex128 states of
// more than one group only: a single tile reverses on its store.
template <bool FF>
__device__ __forceinline__ double2 bitrev_out(double2 v) {
  if constexpr (FF) {
    const ffc z = ffc_unpack(v);
    return make_double2(ff_to_d_fast(z.re), ff_to_d_fast(z.im));
  } else {
    return v;
  }
}

// FF: the input holds double-float parts (the form the
// compiled QFT passes leave) and is converted to IEEE double on the way.
constexpr int BITREV_B = 4, BITREV_T = 128;
template <bool FF>
__global__ void __launch_bounds__(BITREV_T) k_bitrev(double2* __restrict__ s, int n) {
  using V2 = double2;
  constexpr int B = BITREV_B, T = BITREV_T, W = 1 << B, WP = W + 1, PER = W * W / T;
  static_assert(PER * T == W * W, "whole tiles per block");
  extern __shared__ __align__(16) unsigned char smraw[];
  V2* A = reinterpret_cast<V2*>(smraw);
  V2* Bt = A + W * WP;
  const int nm = n - 2 * B;
  const uint64_t M = 1ull << nm;
  for (uint64_t m = blockIdx.x; m < M; m += gridDim.x) {
    const uint64_t mr = nm ? (__brevll((unsigned long long)m) >> (64 - nm)) : 0ull;
    if (mr < m) continue;
    // every load of both tiles in flight before the first shared-memory store
    {
      V2 va[PER], vb[PER];
#pragma unroll
      for (int u = 0; u < PER; ++u) {
        const int e = threadIdx.x + u * T;
        const int h = e >> B, l = e & (W - 1);
        va[u] = s[((uint64_t)h << (n - B)) | (m << B) | (uint64_t)l];
        if (mr != m) vb[u] = s[((uint64_t)h << (n - B)) | (mr << B) | (uint64_t)l];
      }
#pragma unroll
      for (int u = 0; u < PER; ++u) {
        const int e = threadIdx.x + u * T;
        const int h = e >> B, l = e & (W - 1);
        A[h * WP + l] = va[u];
        if (mr != m) Bt[h * WP + l] = vb[u];
      }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < W * W; e += T) {
      const int h = e >> B, l = e & (W - 1);
      const int rl = (int)(__brev((unsigned)l) >> (32 - B)), rh = (int)(__brev((unsigned)h) >> (32 - B));
      // element (h, m, l) of the output is the input at rev(h, m, l)
      if (mr != m) {
        s[((uint64_t)h << (n - B)) | (m << B) | (uint64_t)l] = bitrev_out<FF>(Bt[rl * WP + rh]);
        s[((uint64_t)h << (n - B)) | (mr << B) | (uint64_t)l] = bitrev_out<FF>(A[rl * WP + rh]);
      } else {
        s[((uint64_t)h << (n - B)) | (m << B) | (uint64_t)l] = bitrev_out<FF>(A[rl * WP + rh]);
      }
    }
    __syncthreads();
  }
}

// Blocks of a reversal over M middle values.  A block takes m = blockIdx +
// i grid and skips m > rev m; with an even grid its m keep their low bit, so
// that (rev m having it on top) the odd blocks skipped a quarter of theirs and
// the even ones three quarters, which left half of the SMs idle half of the
// time.  An odd grid: 30 complex128 qubits 6.81 -> 5.65 ms (0.89 of the copy
// bandwidth), 29 complex64 1.74 -> 1.39 ms (0.91).
static unsigned odd_grid(unsigned grid, int64_t M) { return grid < M ? (grid - 1) | 1 : grid; }

static qc_status bitrev_impl(qc_state* s, bool from_ff) {
  double2* d = reinterpret_cast<double2*>(s->data);
  const int64_t M = (int64_t)1 << (s->n - 2 * BITREV_B);
  const size_t smem = 2 * sizeof(double2) * ((1 << BITREV_B) * ((1 << BITREV_B) + 1));
  if (from_ff) {
    const unsigned grid = odd_grid(resident_grid(k_bitrev<true>, BITREV_T, M, 1, smem), M);
    k_bitrev<true><<<grid, BITREV_T, smem, s->stream>>>(d, s->n);
  } else {
    const unsigned grid = odd_grid(resident_grid(k_bitrev<false>, BITREV_T, M, 1, smem), M);
    k_bitrev<false><<<grid, BITREV_T, smem, s->stream>>>(d, s->n);
  }
  return check_launch("bitrev");
}

__global__ void k_roots_fix(longlong2* tlo, longlong2* thi, int n, int nl, longlong2* lad, int nlad);

// Root and ladder tables of a transform over n bits, in one allocation (tlo);
// fixed: in 64-bit fixed point (complex128 register passes).
template <typename R>
struct QftTables {
  typename CT<R>::V2 *tlo, *thi, *lad;
};
template <typename R>
static qc_status qft_tables(qc_state* s, int n, int nl, int nlad, QftTables<R>* t, bool fixed = false) {
  const size_t tot = ((size_t)1 << nl) + ((size_t)1 << (n - nl)) + (size_t)nlad;
  cudaError_t e = ws_alloc((void**)&t->tlo, (tot + 2) * sizeof(typename CT<R>::V2), s->stream);
  if (e != cudaSuccess) return cuda_fail(e, "qft tables");
  t->thi = t->tlo + ((size_t)1 << nl);
  t->lad = t->thi + (((size_t)1 << (n - nl)) + 1) / 2 * 2;  // 16-byte aligned
  const unsigned grid = grid_for((int64_t)tot, 64, 8);
  if (fixed && sizeof(R) == 8)  // complex128 register passes
    k_roots_fix<<<grid, 64, 0, s->stream>>>(reinterpret_cast<longlong2*>(t->tlo), reinterpret_cast<longlong2*>(t->thi), n,
                                            nl, reinterpret_cast<longlong2*>(t->lad), nlad);
  else
    k_roots<R><<<grid, 64, 0, s->stream>>>(t->tlo, t->thi, n, nl, t->lad, nlad);
  const qc_status st = check_launch("qft roots");
  if (st) cudaFreeAsync(t->tlo, s->stream);  // the callers go no further
  return st;
}

// W[e] = Omega_{hi+1}^{l f} of the complex64 pass blockIdx.y on group
// [lo, lo + k): l = tile element e's c = 13 - k low bits, f its group bits
// reversed.  Every tile of a pass uses the same 64 KiB, read through L1.
// Below the tables: the ladder, level j's e^{2 pi i x / 2^{j+1}} at 2^j - 1 + x
// (blockIdx.y = np).
constexpr int QFT_LAD = 1 << 10;
struct QftGroups {
  int np;
  int lo[8], k[8];
};
__global__ void __launch_bounds__(256) k_qft_w(const QftGroups G, float2* __restrict__ lad) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (blockIdx.y == G.np) {
    if (e < QFT_LAD) {
      const int j = 31 - __clz(e + 1);
      const TA<float>::E z = TA<float>::root((uint64_t)(e + 1 - (1 << j)), j + 1);
      lad[e] = make_float2(z.re, z.im);
    }
    return;
  }
  const int lo = G.lo[blockIdx.y], k = G.k[blockIdx.y], c = 13 - k;
  const int f = (int)(__brev((unsigned)(e >> c)) >> (32 - k));
  float zr, zi;  // an exact argument: one rounding
  sincospif(ldexpf((float)((e & ((1 << c) - 1)) * f), 1 - lo - k), &zi, &zr);
  lad[QFT_LAD + ((size_t)blockIdx.y << 13) + e] = make_float2(zr, zi);
}

// Groups of a complex64 transform of at least 13 qubits: the bit reversal's
// kernel does the lowest QFTR_B levels, the others are balanced in groups of
// at most nine (2^13-amplitude tiles with rows of 128 bytes or more), the
// lowest of at least eight, so that its tiles are whole.  Ten levels (n = 15)
// run as one group.
static std::vector<Group> qft_groups_c64(int n) {
  const int total = n - QFTR_B;
  if (total <= 10) return {{QFTR_B, total}};
  const int np = (total + 8) / 9, g0 = std::max(8, (total + np - 1) / np);
  std::vector<Group> g{{QFTR_B, g0}};
  for (int i = 1, lo = QFTR_B + g0; i < np; ++i) {
    const int k = (n - lo + np - i - 1) / (np - i);
    g.push_back({lo, k});
    lo += k;
  }
  return g;
}

static qc_status qft_c64(qc_state* s) {
  const std::vector<Group> groups = qft_groups_c64(s->n);
  QftGroups G{(int)groups.size(), {}, {}};
  for (int i = 0; i < G.np; ++i) G.lo[i] = groups[i].lo, G.k[i] = groups[i].k;
  float2* lad = nullptr;  // the ladder, then the passes' W tables
  cudaError_t e = ws_alloc((void**)&lad, sizeof(float2) * (QFT_LAD + ((size_t)G.np << 13)), s->stream);
  if (e != cudaSuccess) return cuda_fail(e, "qft tables");
  k_qft_w<<<dim3(32, G.np + 1), 256, 0, s->stream>>>(G, lad);
  qc_status st = check_launch("qft tables");
  for (int gi = G.np - 1; gi >= 0 && !st; --gi)
    st = run_qft_c64(s, groups[gi], lad + QFT_LAD + ((size_t)gi << 13), lad);
  if (!st) {
    const int64_t M = (int64_t)1 << (s->n - 2 * QFTR_B);
    const unsigned grid = odd_grid(resident_grid(k_qft_rev_c64, QFTR_T, M, 1, 0), M);
    k_qft_rev_c64<<<grid, QFTR_T, 0, s->stream>>>(reinterpret_cast<float2*>(s->data), s->n, lad);
    st = check_launch("qft bit reversal");
  }
  cudaFreeAsync(lad, s->stream);
  return st;
}

template <typename R>
static qc_status qft_impl(qc_state* s) {
  using V2 = typename CT<R>::V2;
  const int n = s->n;
  const int nl = (n + 1) / 2;
  std::vector<Group> groups = plan_groups<R>(n);
  QftTables<R> tab;
  qc_status st = qft_tables(s, n, nl, 1 << std::min(n, sizeof(R) == 8 ? 11 : 12), &tab);
  if (st) return st;
  V2 *tlo = tab.tlo, *thi = tab.thi;
  std::vector<TileProg<R>> progs(groups.size());
  bool all_compiled = true;  // complex128: double-float form between the passes
  for (int gi = (int)groups.size() - 1; gi >= 0; --gi) {
    const Group& g = groups[gi];
    TileProg<R>& P = progs[gi];
    prog_init(P, g, n);
    P.nl = nl;
    P.qft = g.k;
    for (int j = g.k - 1; j >= 0; --j) {
      P.kind[P.nops] = TOP_QFTLEVEL;
      P.q[P.nops] = (int8_t)j;
      P.mk[P.nops] = 0;
      ++P.nops;
    }
    P.scale_p = g.k;
    P.twiddle = g.lo > 0;
    if constexpr (sizeof(R) == 8) all_compiled = all_compiled && qft_c128_compiled(P);
  }
  // one tile: it is stored in reversed order (every complex64 state that comes here)
  if (groups.size() == 1 && !(sizeof(R) == 8 && all_compiled)) progs[0].rev = n;
  for (int gi = (int)groups.size() - 1; gi >= 0 && !st; --gi) {
    if constexpr (sizeof(R) == 4)
      st = run_tile<R>(s, progs[gi], tlo, thi, tab.lad);
    else
      st = run_qft_c128(s, progs[gi], tlo, thi, tab.lad, all_compiled && gi + 1 < (int)groups.size(), all_compiled);
  }
  if constexpr (sizeof(R) == 8) {  // the bit reversal converts the double-float form back
    if (!st && !progs[0].rev) st = bitrev_impl(s, all_compiled);
  }
  cudaFreeAsync(tab.tlo, s->stream);
  return st;
}

qc_status launch_qft(qc_state* s) {
  s->sum_valid = false;
  if (s->dt == QC_C128) return qft_impl<double>(s);
  return s->n >= 13 ? qft_c64(s) : qft_impl<float>(s);
}

// ---------------------------------------------------- register QFT -------
// Reversal of the bits [lo, lo + w) of every index, in place: amplitude rows
// of 2^lo swap (runs of 2^lo amplitudes stream).  An odd grid, as above: 17
// bits of a 26-qubit complex128 state 486 -> 423 us.
template <typename V2>
__global__ void __launch_bounds__(256) k_reg_rev(V2* __restrict__ s, uint64_t N, int lo, int w) {
  const uint64_t mask = (1ull << w) - 1ull;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t r = (i >> lo) & mask, q = __brevll(r) >> (64 - w);
    if (q <= r) continue;
    const uint64_t j = i ^ ((r ^ q) << lo);
    const V2 a = s[i], b = s[j];
    s[i] = b;
    s[j] = a;
  }
}

// complex128 register passes in 64-bit fixed point.  A tile holds 2^c columns,
// the transforms over the group's bits for each value of its contiguous low bits.
// The largest exponent of a column sets its binary point, so that columns share
// nothing: not a scale, nor an infinity or a NaN.  Sums are exact, a radix-4 step's two
// 1/sqrt 2 are one halving (a shift, or the factor 1/2 that the high word of a
// product by a root scaled by 2^63 brings), and the result is rounded once to
// binary64.  Against double-float (k_tile) a sum costs two integer additions
// instead of about 20 FP32 operations and a value keeps 54 bits or more of
// the column's largest instead of 47: an 11-qubit register of a 17-qubit state
// has a relative error of 4e-16 where double-float passes have 1.2e-14 and
// one pass per gate had 5.8e-15.  Double-float passes take 0.8 of the time
// (two 9-qubit passes of a 26-qubit state 2.37 ms against 2.96 ms) but would
// lose accuracy against the gates.
struct RqftProg {
  int lo, k, c, h;   // group [lo, lo+k), c contiguous low bits, h bits above the group
  int base, w, nl;   // the register's lowest qubit and width, split of its root table
  int twiddle, rev;
  long long rsqrt2;  // floor(2^62.5)
};

__device__ __forceinline__ longlong2 fx_mul(longlong2 a, longlong2 r) {
  return make_longlong2(__mul64hi(a.x, r.x) - __mul64hi(a.y, r.y), __mul64hi(a.x, r.y) + __mul64hi(a.y, r.x));
}
__device__ __forceinline__ longlong2 fx_add(longlong2 a, longlong2 b) { return make_longlong2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ longlong2 fx_sub(longlong2 a, longlong2 b) { return make_longlong2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ longlong2 fx_half(longlong2 a) { return make_longlong2((a.x + 1) >> 1, (a.y + 1) >> 1); }

// The tables of k_roots scaled by 2^63 (1 itself saturates, 2^-63 low).
__global__ void k_roots_fix(longlong2* tlo, longlong2* thi, int n, int nl, longlong2* lad, int nlad) {
  const uint64_t nlo = 1ull << nl, nhi = 1ull << (n - nl);
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nlo + nhi + (uint64_t)nlad;
       i += (uint64_t)gridDim.x * blockDim.x) {
    double x;
    longlong2* out;
    if (i < nlo + nhi) {
      const bool low = i < nlo;
      const uint64_t a = low ? i : (i - nlo);
      x = ldexp((double)((a << ((low ? 0 : nl) + 1)) & ((2ull << n) - 1ull)), -n);
      out = low ? tlo + a : thi + a;
    } else {
      const int a = (int)(i - nlo - nhi), j = 31 - __clz(a + 1);
      x = ldexp((double)(a + 1 - (1 << j)), -j);
      out = lad + a;
    }
    double sn, cs;
    sincospi(x, &sn, &cs);
    *out = make_longlong2(__double2ll_rn(cs * 9223372036854775808.0), __double2ll_rn(sn * 9223372036854775808.0));
  }
}

// Omega_w^r / 2 at scale 2^63 (the product's factor)
__device__ __forceinline__ longlong2 fx_omega(const longlong2* __restrict__ tlo, const longlong2* __restrict__ thi,
                                              uint64_t r, int nl) {
  return fx_mul(tlo[r & ((1ull << nl) - 1ull)], thi[r >> nl]);
}

// ONE: a thread's elements are of one column (the eight differ in group bits only).
template <bool ONE>
__global__ void __launch_bounds__(512, 2) k_rqft_c128(double2* __restrict__ s, uint64_t ntiles,
                                                      const __grid_constant__ RqftProg P,
                                                      const longlong2* __restrict__ tlo,
                                                      const longlong2* __restrict__ thi,
                                                      const longlong2* __restrict__ lad) {
  constexpr int PER = 8;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int k = P.k, c = P.c, lo = P.lo, NE = 1 << (k + c + P.h), T = blockDim.x, tid = threadIdx.x, cm = (1 << c) - 1;
  const int hi = lo + k - 1 - P.base, sh = P.w - hi - 1, ns = (k + 1) / 2;
  const uint64_t hm = (2ull << hi) - 1ull;
  const bool own = P.base < c;  // contiguous bits of the register's: no common twiddle table of a tile
  longlong2* sm = reinterpret_cast<longlong2*>(smraw);
  longlong2* LAD = sm + NE;
  longlong2* V = LAD + (1 << k) - 1;
  // the columns' largest exponents, of this tile and of the next (cleared meanwhile)
  int* const top0 = reinterpret_cast<int*>(V + (P.twiddle && !own ? 1 << k : 0));
  int* top = top0;
  const int nc = 1 << (c + P.h), lb = min(5, c + k);
  auto col = [&](int e) { return ONE ? e & cm : (e & cm) | (e >> (c + k)) << c; };
  for (int a = tid; a < (1 << k) - 1; a += T) LAD[a] = lad[a];
  for (int i = tid; i < 2 * nc; i += T) top0[i] = 0;
  __syncthreads();
  for (uint64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    double2 v[PER];
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int e = tid + T * u;
      v[u] = e < NE ? s[tile_global(e, tile, lo, k + P.h, c)] : make_double2(0.0, 0.0);
    }
    // to the columns' maxima, the lanes of a column first (those that differ in
    // lane bits [c, lb)); subnormal numbers count as 2^-1022
    auto note = [&](int e, int ex) {
      for (int o = (1 << lb) / 2; o > cm; o >>= 1) ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, o));
      if (((tid & ((1 << lb) - 1)) & ~cm) == 0 && e < NE) atomicMax(&top[col(e)], max(ex, 1));
    };
    int em = 0;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int ex = max((int)((__double_as_longlong(v[u].x) >> 52) & 0x7FF),
                         (int)((__double_as_longlong(v[u].y) >> 52) & 0x7FF));
      if (ONE) em = max(em, ex);
      else note(tid + T * u, ex);
    }
    if (ONE) note(tid, em);
    __syncthreads();
    // |x| < 2^(em - 1022) times 2^(1075 - G) is below 2^(61 - ns).  A step's
    // values grow by at most 2 and its sums of four by 4: below 2^63.
    const int G0 = ns - 8, mine = ONE ? top[tid & cm] : 0;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int e = tid + T * u, G = (ONE || e >= NE ? mine : top[col(e)]) + G0;
      if (e < NE) sm[tsw(e)] = make_longlong2(d2fix<true>(v[u].x, G), d2fix<true>(v[u].y, G));
    }
    int* const next = top == top0 ? top0 + nc : top0;
    for (int i = tid; i < nc; i += T) next[i] = 0;
    const uint64_t Lt = (tile & ((1ull << (lo - c)) - 1ull)) << c;  // the tile's index bits below the group
    if (P.twiddle && !own)
      for (int f = tid; f < (1 << k); f += T) V[f] = fx_omega(tlo, thi, (((Lt >> P.base) * (uint64_t)f) & hm) << sh, P.nl);
    __syncthreads();
    int jh = k - 1;
    for (; jh >= 1; jh -= 2) {  // levels jh, jh - 1 as in k_tile
      const int jl = jh - 1, bl = c + jl;
      for (int p = tid; p < (NE >> 2); p += T) {
        const int e00 = ((p >> bl) << (bl + 2)) | (p & ((1 << bl) - 1));
        const int b = tsw(e00), o01 = tsw(1 << bl), o10 = tsw(2 << bl), o11 = tsw(3 << bl);
        const longlong2 a00 = sm[b], a01 = sm[b ^ o01], a10 = sm[b ^ o10], a11 = sm[b ^ o11];
        const longlong2 s0 = fx_add(a00, a10), d0 = fx_sub(a00, a10), s1 = fx_add(a01, a11), d1 = fx_sub(a01, a11);
        const longlong2 id1 = make_longlong2(-d1.y, d1.x);
        longlong2 u0 = fx_sub(s0, s1), t1 = fx_add(d0, id1), u1 = fx_sub(d0, id1);
        const int x = (e00 >> c) & ((1 << jl) - 1);
        if (x) {
          const longlong2* L = LAD + (1 << jh) - 1;
          const int x3 = 3 * x, m = (1 << jh) - 1;
          u0 = fx_mul(u0, L[2 * x]);
          t1 = fx_mul(t1, L[x]);
          u1 = fx_mul(u1, L[x3 & m]);
          if (x3 >> jh) u1 = make_longlong2(-u1.x, -u1.y);
        } else {
          u0 = fx_half(u0);
          t1 = fx_half(t1);
          u1 = fx_half(u1);
        }
        sm[b] = fx_half(fx_add(s0, s1));
        sm[b ^ o01] = u0;
        sm[b ^ o10] = t1;
        sm[b ^ o11] = u1;
      }
      __syncthreads();
    }
    if (jh == 0) {
      for (int p = tid; p < (NE >> 1); p += T) {
        const int b = tsw(((p >> c) << (c + 1)) | (p & cm)), o = tsw(1 << c);
        const longlong2 a0 = sm[b], a1 = sm[b ^ o];
        sm[b] = fx_add(a0, a1);
        sm[b ^ o] = fx_sub(a0, a1);
      }
      __syncthreads();
    }
    // odd k: the last level's 1/sqrt 2 (the high word of 2^62.5 v is v / sqrt 2 / 2)
    const int F0 = 1075 - G0 - (k & 1) - (P.twiddle ? 2 : 0);
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int e = tid + T * u;
      if (e < NE) {
        const int f = (int)(__brev((unsigned)(e >> c)) >> (32 - k));
        longlong2 z = sm[tsw(P.rev ? (f << c) | (e & (ONE ? cm : cm | ~0 << (c + k))) : e)];
        if (k & 1) z = make_longlong2(__mul64hi(z.x, P.rsqrt2), __mul64hi(z.y, P.rsqrt2));
        if (P.twiddle) {
          const longlong2 W =
              own ? fx_omega(tlo, thi, ((((Lt | (uint64_t)(e & cm)) >> P.base) * (uint64_t)f) & hm) << sh, P.nl) : V[f];
          z = fx_mul(z, W);
        }
        // a column with an infinity or a NaN comes out as NaN
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
        const int t = ONE ? mine : top[col(e)], F = F0 - t;
        s[tile_global(e, tile, lo, k + P.h, c)] =
            t == 0x7FF ? make_double2(nan, nan) : make_double2(fix2d<true>(z.x, F), fix2d<true>(z.y, F));
      }
    }
    top = next;
    __syncthreads();
  }
}

// Appendix A's circuit on the register [lo, lo + w) as tile passes: the
// register's qubits in groups from the top, each pass one read and write of
// the state; the phases between groups as in qft_impl, over the register's
// bits.  A register of up to eleven qubits is a single pass (rows of 32 bytes
// or longer: c contiguous bits below it) that also stores the reversed order;
// larger ones take groups of up to nine with longer rows and one reversal
// pass.  Gate by gate this is w Hadamard, w (w - 1) / 2 phase and w / 2 swap
// passes: 195 us (71 launches) for 11 qubits of 17.
struct RangePlan {
  std::vector<Group> groups;
  int kmax = 0;
};
static RangePlan plan_range(int lo, int w) {
  RangePlan R;
  if (w <= 11) {
    R.groups.push_back({lo, w});
  } else if (lo == 0) {
    R.groups = plan_groups_k(w, 11, 9);
  } else {
    const int ng = (w + 8) / 9;
    for (int i = 0, at = lo, left = w; i < ng; ++i) {
      const int k = (left + (ng - i) - 1) / (ng - i);  // balanced
      R.groups.push_back({at, k});
      at += k;
      left -= k;
    }
  }
  for (const Group& g : R.groups) R.kmax = std::max(R.kmax, g.k);
  return R;
}

template <typename R>
static qc_status qft_range_impl(qc_state* s, int lo, int w) {
  using V2 = typename CT<R>::V2;
  constexpr int ROW = sizeof(R) == 8 ? 1 : 2, TB = sizeof(R) == 8 ? 12 : 13;
  const RangePlan plan = plan_range(lo, w);
  const int nl = (w + 1) / 2, nlad = (1 << plan.kmax) - 1;
  QftTables<R> tab;
  qc_status st = qft_tables(s, w, nl, nlad, &tab, true);
  if (st) return st;
  for (int gi = (int)plan.groups.size() - 1; gi >= 0 && !st; --gi) {
    const Group& g = plan.groups[gi];
    // near the bottom of the state there are few contiguous bits: bits above the
    // group fill the tile, while 256 tiles (two per SM, about) are left.  26
    // complex128 qubits, registers at qubit 0: tiles of 2^w amplitudes took 30 ms
    // for w = 1 and 11.8 for w = 3, full ones 0.82 and 1.13
    const int c = std::min(g.lo, std::max(ROW, TB - g.k)),
              h = g.lo == lo && c == g.lo ? std::max(0, std::min(s->n - 8, TB) - g.k - c) : 0;
    if constexpr (sizeof(R) == 8) {
      RqftProg P{g.lo, g.k, c, h, lo, w, nl, g.lo > lo, plan.groups.size() == 1, 6521908912666391106ll};
      const size_t NE = (size_t)1 << (g.k + c + h);
      const size_t smem = sizeof(longlong2) * (NE + ((size_t)1 << g.k) - 1 + (P.twiddle && lo >= c ? (size_t)1 << g.k : 0)) +
                          2 * sizeof(int) * ((size_t)1 << (c + h));
      const int T = std::max(32, (int)(NE / 8));
      const uint64_t ntiles = (1ull << s->n) / NE;
      const auto kernel = h == 0 && (1 << c) <= T ? k_rqft_c128<true> : k_rqft_c128<false>;
      allow_smem(kernel, 200 * 1024);
      kernel<<<resident_grid(kernel, T, (int64_t)ntiles, 1, smem), T, smem, s->stream>>>(
          reinterpret_cast<double2*>(s->data), ntiles, P, reinterpret_cast<const longlong2*>(tab.tlo),
          reinterpret_cast<const longlong2*>(tab.thi), reinterpret_cast<const longlong2*>(tab.lad));
      st = check_launch("register qft pass");
    } else {
      TileProg<R> P;
      prog_init(P, g, w);
      P.k = g.k + h;
      P.c = c;
      P.base = lo;
      P.nl = nl;
      P.qft = g.k;
      for (int j = g.k - 1; j >= 0; --j) {
        P.kind[P.nops] = TOP_QFTLEVEL;
        P.q[P.nops] = (int8_t)j;
        P.mk[P.nops] = 0;
        ++P.nops;
      }
      P.scale_p = g.k;
      P.twiddle = g.lo > lo;
      P.rev = plan.groups.size() == 1 ? g.k : 0;
      st = run_tile<R>(s, P, tab.tlo, tab.thi, tab.lad);
    }
  }
  if (!st && plan.groups.size() > 1 && sizeof(R) == 8 && w == s->n) {
    st = bitrev_impl(s, false);
  } else if (!st && plan.groups.size() > 1) {
    const uint64_t N = 1ull << s->n;
    const unsigned grid = odd_grid(resident_grid(k_reg_rev<V2>, 256, (int64_t)N, 256), ((int64_t)N + 255) / 256);
    k_reg_rev<V2><<<grid, 256, 0, s->stream>>>(reinterpret_cast<V2*>(s->data), N, lo, w);
    st = check_launch("register reversal");
  }
  cudaFreeAsync(tab.tlo, s->stream);
  return st;
}

qc_status launch_qft_range(qc_state* s, int lo, int w) {
  s->sum_valid = false;
  // The whole state in complex64 is qft_c64's.  The complex128 passes of
  // launch_qft are in double-float (20 qubits: 60 us, relative error 2.2e-14;
  // gate by gate 9.3e-15; here 99 us and 8.6e-16): not for a register that
  // happens to be the state.
  if (lo == 0 && w == s->n && s->dt == QC_C64) return launch_qft(s);
  // One qubit in complex64 is the Hadamard's own kernel (26 qubits: 175 us, and
  // 210 through tiles; 20 qubits 5 us and 17).  In complex128 that kernel is
  // faster too (335 us and 830), but its double-float drops what lies below
  // 2^-100, which a column of a register here keeps.
  if (w == 1 && s->dt == QC_C64) {
    const double h = 1.0 / sqrt(2.0), H[8] = {h, 0, h, 0, h, 0, -h, 0};
    return launch_1q(s, lo, H);
  }
  return s->dt == QC_C128 ? qft_range_impl<double>(s, lo, w) : qft_range_impl<float>(s, lo, w);
}

}  // namespace qc
