// Parameterised circuits on a batch of states and the adjoint gradient of
// E = <psi|H|psi> (not part of the QCMPI paper).
//
// The gate list is compiled into passes over shared-memory tiles
// (circuit_passes.cuh).
//
// Forward: psi_b = U_G .. U_1 |0..0>.  Backward: lambda = H psi (one gather
// pass over the Pauli terms), E = Re <psi|lambda>, then the passes are
// walked in reverse; a rotation accumulates Im <lambda_j|P_j|psi_j> -- the
// derivative of U_j = exp(-i theta P_j / 2) gives
// dE/dtheta_j = 2 Re <lambda_j|(-i/2) P_j|psi_j> = Im <lambda_j|P_j|psi_j>
// -- and U_j^dagger is applied to both.  No intermediate state is stored: psi
// is uncomputed instead of checkpointed.
//
// Accumulation: complex128 with FMA in double.  complex64: the energy's
// products are exact float pairs (two-product), summed as float pairs over
// short runs and then in double; a derivative's products are summed in float
// pairs with a common high binade (Acc) and then in 64-bit fixed point.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "circuit_passes.cuh"
#include "common.cuh"
#include "fixpt.cuh"

namespace qc {

#define ADJ_T 256
#define ADJ_GX_MAX 256

// Rotation matrices exp(-i theta P / 2) for P = X, Y, Z; H.
template <typename R>
__device__ __forceinline__ Mat2<R> gate_matrix(int kind, double theta) {
  Mat2<R> U;
  double s, c;
  sincos(0.5 * theta, &s, &c);
  const R cr = (R)c, sr = (R)s;
  const R z = (R)0;
  if (kind == QC_G_RX) {
    U.m[0] = cmake<R>(cr, z);
    U.m[1] = cmake<R>(z, -sr);
    U.m[2] = cmake<R>(z, -sr);
    U.m[3] = cmake<R>(cr, z);
  } else if (kind == QC_G_RY) {
    U.m[0] = cmake<R>(cr, z);
    U.m[1] = cmake<R>(-sr, z);
    U.m[2] = cmake<R>(sr, z);
    U.m[3] = cmake<R>(cr, z);
  } else if (kind == QC_G_RZ) {
    U.m[0] = cmake<R>(cr, -sr);
    U.m[1] = cmake<R>(z, z);
    U.m[2] = cmake<R>(z, z);
    U.m[3] = cmake<R>(cr, sr);
  } else {  // H
    const R h = (R)0.70710678118654752440;
    U.m[0] = cmake<R>(h, z);
    U.m[1] = cmake<R>(h, z);
    U.m[2] = cmake<R>(h, z);
    U.m[3] = cmake<R>(-h, z);
  }
  return U;
}

// ----------------------------------------------------- accumulators ------
// The energy's sum.  complex64: products exact as float pairs (two-product),
// summed as a float pair with two-sum (relative error ~ terms * 2^-48),
// converted to double every few terms.
template <typename R> struct SumE;
template <> struct SumE<double> {
  double a = 0.0;
  __device__ void add(double x, double y) { a = fma(x, y, a); }
  __device__ void flush() {}
  __device__ double value() const { return a; }
};
template <> struct SumE<float> {
  double a = 0.0;
  float s = 0.f, c = 0.f;
  __device__ void add(float x, float y) {
    const float p = x * y, e = fmaf(x, y, -p);
    const float t = s + p;
    const float bp = t - s;
    c += ((s - (t - bp)) + (p - bp)) + e;
    s = t;
  }
  __device__ void flush() {
    a += (double)s + (double)c;
    s = c = 0.f;
  }
  __device__ double value() const { return a; }
};

// The derivatives' sums.
template <typename R> struct Acc;
template <> struct Acc<double> {
  double a = 0.0;
  __device__ void add(double x, double y) { a = fma(x, y, a); }
  __device__ void sub(double x, double y) { a = fma(-x, y, a); }
  __device__ void start(double) {}
  __device__ void settle(double) {}
  __device__ double value() const { return a; }
  __device__ void merge(const Acc& o) { a += o.a; }
  __device__ void merge_neg(const Acc& o) { a -= o.a; }
  __device__ void into(double& z) const { z += a; }
  __device__ bool finite() const { return isfinite(a); }
};
// complex64: a float pair, no FP64 instruction.  The high word starts at
// C = 1.5 2^e with every partial sum below 2^{e-1}: it stays in one binade, so
// that s' - s is the multiple of its unit that a product was rounded to,
// exactly, and fma(x, y, -(s' - s)) what that left out.  Four instructions a
// product; a two-product and a two-sum take ten (20 qubits, 64 states: the
// backward passes 28.5 -> 24.9 ms; what is left waits: issue slots 0.53
// busy, barriers, shared memory and the tile's loads in turn).
// Error: 2^-24 units a term, a unit being at most 2^-16 of the product of the
// thread's largest |p| and |l| where C was set, and at most 2^-13 of it up to
// ACC_SPAN operators later.
template <> struct Acc<float> {
  float s = 0.f, c = 0.f;
  __device__ void start(float C) { s = C; }
  __device__ void settle(float C) { s -= C; }
  __device__ void add(float x, float y) {
    const float t = fmaf(x, y, s);
    c += fmaf(x, y, s - t);
    s = t;
  }
  __device__ void sub(float x, float y) { add(-x, y); }
  // sums with a common C, settled: the high words are multiples of one unit
  __device__ void merge(const Acc& o) { s += o.s; c += o.c; }
  __device__ void merge_neg(const Acc& o) { s -= o.s; c -= o.c; }
  __device__ void into(float2& z) const {  // two-sum
    const float t = z.x + s, bp = t - z.x;
    z = make_float2(t, z.y + (((z.x - (t - bp)) + (s - bp)) + c));
  }
  __device__ bool finite() const { return isfinite(s); }
  // (s + c) 2^k as hi 2^26 + lo, to a unit (k may exceed a float's range of
  // exponents; no 64-bit conversion, which would run on the FP64 pipe)
  __device__ int2 fixed(int k) const {
    const int e = k - 26;
    const float f0 = __int_as_float((127 + e / 2) << 23), f1 = __int_as_float((127 + e - e / 2) << 23);
    const float t = s + c, b = t - s;  // two-sum: the low word below half a unit of the high one
    const float x = t * f0 * f1, y = ((s - (t - b)) + (c - b)) * f0 * f1;
    const int hi = __float2int_rn(x);
    return make_int2(hi, __float2int_rn(((x - (float)hi) + y) * 67108864.f));
  }
};

__device__ __forceinline__ double block_reduce(double v) {
  __shared__ double sh[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
  __syncthreads();
  return t;
}

// ------------------------------------------------------------ forward ----
// What a pass's operators are on one batch element, prepared once per call
// in FP64 by k_prep (the sines and cosines of GB300's slow FP64 pipe stay out
// of the tile kernels).
//
// A rotation is applied without its factor: RY as b0 = a0 + t a1,
// b1 = a1 - t a0 with t = s/c when |s| <= |c|, else b0 = t a0 + a1,
// b1 = t a1 - a0 with t = c/s (RX likewise with i t), two multiply-adds an
// amplitude and component instead of a 2x2 product; the factors c or s of all
// of a pass's operators go into its one phase per amplitude.
enum OpMode { OM_RY0, OM_RY1, OM_RX0, OM_RX1, OM_RZ, OM_H };
template <typename R>
struct OpRec {
  R t, u;
  int mode;
  int eq;    // backward: the sum's value is f times the one accumulated, eq = floor(log2 f)
  double f;
};
// tab: phase of a thread's lane bits [0, 32), its warp bits [32, 48), of the
// register bits [48, 56); the phase times the pass's factor is their product.
template <typename R>
struct PassRec {
  typename CT<R>::V2 tab[56];
  OpRec<R> op[TP_MAXOP];
};

// 1 / sqrt(1 + t^2) as an unevaluated sum (the rounded root and its first
// correction): the product of a pass's factors is then good to one rounding,
// so the state's norm does not drift by it.
__device__ __forceinline__ double2 inv_norm(double t) {
  const double s = fma(t, t, 1.0), sl = fma(t, t, 1.0 - s), r = 1.0 / sqrt(s);
  const double q = s * r, ql = fma(s, r, -q);
  const double res = fma(-q, r, 1.0) - ql * r - sl * r * r;  // 1 - (1 + t^2) r^2
  return make_double2(r, 0.5 * r * res);
}

// Per pass and batch element (grid.x, grid.y).  dir = +1: the operators as
// they are, the phase in the last round; -1: their inverses, the phase in the
// first round.
template <typename R>
__global__ void __launch_bounds__(128) k_prep(const TilePass* __restrict__ passes, PassRec<R>* __restrict__ recs, int B,
                                              const double* __restrict__ theta, int64_t stride, int dir) {
  __shared__ double2 ph[TP_MAXK + 3];  // e^{-i dir theta / 2}
  __shared__ double2 fac[TP_MAXOP];  // factor as an unevaluated sum
  const TilePass& P = passes[blockIdx.x];
  const int b = blockIdx.y, tid = threadIdx.x;
  PassRec<R>& rec = recs[(int64_t)blockIdx.x * B + b];
  const double* th = theta + (int64_t)b * stride;
  if (tid < P.nop) {
    const TileOp o = P.op[tid];
    OpRec<R> r{};
    double2 f = make_double2(1.0, 0.0);
    if (o.ka == QC_G_H) {
      r.mode = OM_H;
      f = inv_norm(1.0);
    } else {
      double s, c;
      sincos(-0.5 * dir * th[o.pa], &s, &c);  // b0 = c a0 + s a1 undoes RY(theta)
      if (o.ka == QC_G_RZ) {
        r.mode = OM_RZ;
        r.t = (R)c;
        r.u = (R)s;
      } else {
        const bool small = fabs(s) <= fabs(c);
        r.mode = (o.ka == QC_G_RY ? OM_RY0 : OM_RX0) + (small ? 0 : 1);
        r.t = (R)(small ? s / c : c / s);
        f = inv_norm((double)r.t);  // of the t in use: the operator is unitary to rounding
        if ((small ? c : s) < 0.0) f = make_double2(-f.x, -f.y);
      }
    }
    rec.op[tid] = r;
    fac[tid] = f;
  } else if (tid >= 64 && tid < 64 + P.kt) {
    const int p = tid - 64;
    double s = 0.0, c = 1.0;
    if (P.dp[p] >= 0) sincos(-0.5 * dir * th[P.dp[p]], &s, &c);
    ph[p] = make_double2(c, s);
  }
  __syncthreads();
  if (dir < 0 && tid < P.nop) {  // operator `tid` still has the factors from itself on in psi and in lambda
    double f = 1.0;
    for (int k = tid; k < P.nop; ++k) f *= fac[k].x;
    f = 1.0 / (f * f);
    rec.op[tid].f = f;
    rec.op[tid].eq = ilogb(f);
  }
  if (tid < 56) {
    const TileRound& rd = P.rd[dir > 0 ? P.nround - 1 : 0];
    constexpr int rb = 3;
    double re = 1.0, im = 0.0;
    // thread bit i is the i-th tile position outside the round's registers
    int i = 0;
    for (int p = 0; p < P.kt; ++p) {
      int reg = -1;
      for (int x = 0; x < rb; ++x)
        if (rd.r[x] == p) reg = x;
      int bit;
      bool mine;
      if (reg >= 0) {
        mine = tid >= 48;
        bit = (tid - 48) >> reg;
      } else {
        mine = i < 5 ? tid < 32 : (tid >= 32 && tid < 48);
        bit = i < 5 ? tid >> i : (tid - 32) >> (i - 5);
        ++i;
      }
      if (!mine || P.dp[p] < 0) continue;
      const double c = ph[p].x, s = (bit & 1) ? -ph[p].y : ph[p].y;
      const double nr = re * c - im * s;
      im = re * s + im * c;
      re = nr;
    }
    // products of rounded phases: back to modulus 1, then the factor
    const double m = 0.5 * (fma(re, re, -1.0) + im * im);
    re = fma(-m, re, re);
    im = fma(-m, im, im);
    if (tid >= 48) {
      double h = 1.0, l = 0.0;
      for (int k = 0; k < P.nop; ++k) {
        const double p = h * fac[k].x;
        l = fma(h, fac[k].x, -p) + fma(h, fac[k].y, l * fac[k].x);
        h = p;
      }
      re = fma(re, l, re * h);
      im = fma(im, l, im * h);
    }
    rec.tab[tid] = CT<R>::make((R)re, (R)im);
  }
}

// The merged operators of the complex64 forward passes as 2x2 matrices.
__global__ void __launch_bounds__(64) k_prep_mats(const TilePass* __restrict__ passes, Mat2<float>* __restrict__ mats, int B,
                                                  const double* __restrict__ theta, int64_t stride) {
  const TilePass& P = passes[blockIdx.x];
  const int b = blockIdx.y;
  if ((int)threadIdx.x >= P.nop) return;
  const TileOp o = P.op[threadIdx.x];
  const double* th = theta + (int64_t)b * stride;
  Mat2<double> M = gate_matrix<double>(o.ka, o.pa >= 0 ? th[o.pa] : 0.0);
  if (o.kb >= 0) {
    const Mat2<double> A = M, Bm = gate_matrix<double>(o.kb, th[o.pb]);
    for (int r = 0; r < 2; ++r)
      for (int c = 0; c < 2; ++c) M.m[2 * r + c] = cmul2(Bm.m[2 * r], A.m[c], Bm.m[2 * r + 1], A.m[2 + c]);
  }
  Mat2<float> F;
  for (int k = 0; k < 4; ++k) F.m[k] = cmake<float>((float)M.m[k].re, (float)M.m[k].im);
  mats[((int64_t)blockIdx.x * B + b) * TP_MAXOP + threadIdx.x] = F;
}

// One operator on a thread's 2^RB amplitudes along register bit BIT.
template <int MODE, int BIT, int RB, typename R>
__device__ __forceinline__ void op_mode(const R t, const R u, Cx<R>* v) {
#pragma unroll
  for (int m = 0; m < (1 << (RB - 1)); ++m) {
    const int j0 = ((m >> BIT) << (BIT + 1)) | (m & ((1 << BIT) - 1)), j1 = j0 | (1 << BIT);
    const Cx<R> a = v[j0], c = v[j1];
    if (MODE == OM_RY0) {  // a + t c, c - t a
      v[j0] = cmake<R>(fma(t, c.re, a.re), fma(t, c.im, a.im));
      v[j1] = cmake<R>(fma(-t, a.re, c.re), fma(-t, a.im, c.im));
    } else if (MODE == OM_RY1) {  // t a + c, t c - a
      v[j0] = cmake<R>(fma(t, a.re, c.re), fma(t, a.im, c.im));
      v[j1] = cmake<R>(fma(t, c.re, -a.re), fma(t, c.im, -a.im));
    } else if (MODE == OM_RX0) {  // a + i t c, c + i t a
      v[j0] = cmake<R>(fma(-t, c.im, a.re), fma(t, c.re, a.im));
      v[j1] = cmake<R>(fma(-t, a.im, c.re), fma(t, a.re, c.im));
    } else if (MODE == OM_RX1) {  // t a + i c, t c + i a
      v[j0] = cmake<R>(fma(t, a.re, -c.im), fma(t, a.im, c.re));
      v[j1] = cmake<R>(fma(t, c.re, -a.im), fma(t, c.im, a.re));
    } else if (MODE == OM_RZ) {  // (t + i u) a, (t - i u) c
      v[j0] = cmake<R>(fma(-u, a.im, t * a.re), fma(u, a.re, t * a.im));
      v[j1] = cmake<R>(fma(u, c.im, t * c.re), fma(-u, c.re, t * c.im));
    } else {  // a + c, a - c
      v[j0] = cmake<R>(a.re + c.re, a.im + c.im);
      v[j1] = cmake<R>(a.re - c.re, a.im - c.im);
    }
  }
}
template <int BIT, int RB, typename R>
__device__ __forceinline__ void op_bit(const OpRec<R>& o, Cx<R>* v) {
  switch (o.mode) {
    case OM_RY0: op_mode<OM_RY0, BIT, RB>(o.t, o.u, v); break;
    case OM_RY1: op_mode<OM_RY1, BIT, RB>(o.t, o.u, v); break;
    case OM_RX0: op_mode<OM_RX0, BIT, RB>(o.t, o.u, v); break;
    case OM_RX1: op_mode<OM_RX1, BIT, RB>(o.t, o.u, v); break;
    case OM_RZ: op_mode<OM_RZ, BIT, RB>(o.t, o.u, v); break;
    default: op_mode<OM_H, BIT, RB>(o.t, o.u, v); break;
  }
}
template <int BIT, int RB>
__device__ __forceinline__ void mat_bit(const Mat2<float>& M, Cx<float>* v) {
#pragma unroll
  for (int m = 0; m < (1 << (RB - 1)); ++m) {
    const int j0 = ((m >> BIT) << (BIT + 1)) | (m & ((1 << BIT) - 1));
    apply2<float, MK_GENERAL>(M, v[j0], v[j0 | (1 << BIT)]);
  }
}

template <typename V2>
__device__ __forceinline__ V2* sm_at(V2* sm, int byte) {
  return reinterpret_cast<V2*>(reinterpret_cast<unsigned char*>(sm) + byte);
}

// The register rounds of a pass on the tile in `sm`, each closed by a barrier.
template <typename R> struct Fwd;
template <> struct Fwd<float> {
  static constexpr int KT = 13, C0 = 4, RB = 4, VE = 2;
  using Ops = Mat2<float>;
};
template <> struct Fwd<double> {
  static constexpr int KT = 12, C0 = 3, RB = 3, VE = 1;
  using Ops = PassRec<double>;
};

template <typename R>
__device__ __forceinline__ void fwd_rounds(const TilePass& P, typename CT<R>::V2* sm, const typename Fwd<R>::Ops* ops) {
  constexpr int RB = Fwd<R>::RB, NA = 1 << RB;
  const int tid = threadIdx.x;
  const bool active = tid < (1 << (P.kt - RB));
#pragma unroll 1
  for (int r = 0; r < P.nround; ++r) {
    const TileRound& rd = P.rd[r];
    if (active) {
      const int base = tp_round_base<R, RB>(rd);
      int bas[RB];
#pragma unroll
      for (int x = 0; x < RB; ++x) bas[x] = rd.bas[x];
      Cx<R> v[NA];
#pragma unroll
      for (int j = 0; j < NA; ++j) v[j] = AmpIO<R>::ld(sm_at(sm, tp_round_at<RB>(base, bas, j)));
#pragma unroll 1
      for (int k = rd.op0; k < rd.op1; ++k) {
        if constexpr (sizeof(R) == 4) {
          const Mat2<float> M = ops[k];
          switch (P.op[k].bit) {
            case 0: mat_bit<0, RB>(M, v); break;
            case 1: mat_bit<1, RB>(M, v); break;
            case 2: mat_bit<2, RB>(M, v); break;
            default: mat_bit<3, RB>(M, v); break;
          }
        } else {
          const OpRec<R> o = ops->op[k];
          switch (P.op[k].bit) {
            case 0: op_bit<0, RB, R>(o, v); break;
            case 1: op_bit<1, RB, R>(o, v); break;
            default: op_bit<2, RB, R>(o, v); break;
          }
        }
      }
      if constexpr (sizeof(R) == 8) {
        if (r == P.nround - 1 && !P.has_diag && P.has_fac) {  // the factor alone
          const R f = ops->tab[48].x;
#pragma unroll
          for (int j = 0; j < NA; ++j) v[j] = cmake<R>(v[j].re * f, v[j].im * f);
        } else if (r == P.nround - 1 && P.has_diag) {
          const auto A = ops->tab[tid & 31], Bw = ops->tab[32 + (tid >> 5)];
          const Cx<R> d = cmul(cmake<R>(A.x, A.y), cmake<R>(Bw.x, Bw.y));
#pragma unroll
          for (int j = 0; j < NA; ++j) {
            const auto J = ops->tab[48 + j];
            v[j] = cmul(v[j], cmul(d, cmake<R>(J.x, J.y)));
          }
        }
      }
#pragma unroll
      for (int j = 0; j < NA; ++j) AmpIO<R>::st(sm_at(sm, tp_round_at<RB>(base, bas, j)), v[j]);
    }
    __syncthreads();
  }
}

// 16-byte vectors of a tile (TileShare), to and from shared memory at byte
// offsets i0 and i1 of their amplitudes.
template <typename R> struct Vec;
template <> struct Vec<float> {
  using T = float4;
  __device__ static void to_sm(float2* sm, int i0, int i1, const float4& v) {
    *sm_at(sm, i0) = make_float2(v.x, v.y);
    *sm_at(sm, i1) = make_float2(v.z, v.w);
  }
  __device__ static float4 from_sm(float2* sm, int i0, int i1) {
    const float2 a = *sm_at(sm, i0), b = *sm_at(sm, i1);
    return make_float4(a.x, a.y, b.x, b.y);
  }
  // al: the state starts on a 16-byte boundary (8 bytes suffice for the caller)
  __device__ static float4 ld(const float2* g, bool al) {
    if (al) return *reinterpret_cast<const float4*>(g);
    const float2 a = g[0], b = g[1];
    return make_float4(a.x, a.y, b.x, b.y);
  }
  __device__ static void st(float2* g, const float4& v, bool al) {
    if (al) {
      *reinterpret_cast<float4*>(g) = v;
    } else {
      g[0] = make_float2(v.x, v.y);
      g[1] = make_float2(v.z, v.w);
    }
  }
  __device__ static float4 zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
  __device__ static float4 one() { return make_float4(1.f, 0.f, 0.f, 0.f); }
};
template <> struct Vec<double> {
  using T = double2;
  __device__ static void to_sm(double2* sm, int i0, int, const double2& v) { *sm_at(sm, i0) = v; }
  __device__ static double2 from_sm(double2* sm, int i0, int) { return *sm_at(sm, i0); }
  __device__ static double2 ld(const double2* g, bool) { return *g; }
  __device__ static void st(double2* g, const double2& v, bool) { *g = v; }
  __device__ static double2 zero() { return make_double2(0.0, 0.0); }
  __device__ static double2 one() { return make_double2(1.0, 0.0); }
};

constexpr int FWD_T = 512, FWD_LV = 3, FWD_NV = 1 << FWD_LV;  // threads of a full tile, vectors of each

// One pass over the batch: tile blockIdx.x of state blockIdx.y (first: the
// state is |0..0>, nothing is read).
template <typename R>
__global__ void __launch_bounds__(FWD_T, 2) k_fwd_tile(typename CT<R>::V2* __restrict__ psi, int n,
                                                       const __grid_constant__ TilePass P,
                                                       const typename Fwd<R>::Ops* __restrict__ recs, int nrec, int first) {
  using V2 = typename CT<R>::V2;
  using V = typename Vec<R>::T;
  extern __shared__ __align__(16) unsigned char dynsm[];
  V2* sm = reinterpret_cast<V2*>(dynsm);
  auto* ops = reinterpret_cast<typename Fwd<R>::Ops*>(dynsm + (sizeof(V2) << P.kt));
  const int tid = threadIdx.x, T = blockDim.x;
  const uint64_t base = tp_tile_base(P, blockIdx.x);
  V2* g = psi + ((uint64_t)blockIdx.y << n) + base;
  const bool al = (reinterpret_cast<uintptr_t>(psi) & 15) == 0;
  {  // this element's operators
    const int words = (int)(sizeof(typename Fwd<R>::Ops) * nrec / 16);
    const uint4* src = reinterpret_cast<const uint4*>(recs + (size_t)blockIdx.y * nrec);
    for (int i = tid; i < words; i += T) reinterpret_cast<uint4*>(ops)[i] = src[i];
  }
  TileShare<R, FWD_LV> sh;
  sh.init(P, T);
  V v[FWD_NV];
#pragma unroll
  for (int u = 0; u < FWD_NV; ++u) {
    if (first) v[u] = (tid + u == 0 && base == 0) ? Vec<R>::one() : Vec<R>::zero();
    else v[u] = Vec<R>::ld(g + sh.g(u), al);
  }
#pragma unroll
  for (int u = 0; u < FWD_NV; ++u) Vec<R>::to_sm(sm, sh.a(u), sh.a(u) ^ tp_at<R>(1), v[u]);
  __syncthreads();
  fwd_rounds<R>(P, sm, ops);
  const int cst = tp_cst(P, base);
#pragma unroll
  for (int u = 0; u < FWD_NV; ++u) {
    const int s = sh.s(u) ^ cst;
    Vec<R>::st(g + sh.g(u), Vec<R>::from_sm(sm, s, s ^ sh.s1), al);
  }
}

// The whole circuit of states that fit one tile: one block a state, all
// passes in shared memory, one store at the end.
template <typename R>
__global__ void __launch_bounds__(FWD_T, 2) k_fwd_whole(typename CT<R>::V2* __restrict__ psi, int n,
                                                        const TilePass* __restrict__ passes, int npass,
                                                        const typename Fwd<R>::Ops* __restrict__ recs, int nrec, int B) {
  using V2 = typename CT<R>::V2;
  using V = typename Vec<R>::T;
  constexpr int VE = Fwd<R>::VE;
  extern __shared__ __align__(16) unsigned char dynsm[];
  __shared__ TilePass P;
  const int tid = threadIdx.x, T = blockDim.x, kt = passes[0].kt, ne = 1 << n, b = blockIdx.x;
  V2* sm = reinterpret_cast<V2*>(dynsm);
  auto* ops = reinterpret_cast<typename Fwd<R>::Ops*>(dynsm + (sizeof(V2) << kt));
  for (int e = tid; e < (1 << kt); e += T) sm[tp_swz<R>(e)] = CT<R>::make((R)(e == 0), (R)0);
  V v[FWD_NV];
#pragma unroll 1
  for (int k = 0; k < npass; ++k) {
    static_assert(sizeof(TilePass) % 4 == 0, "copied in words");
    for (int i = tid; i < (int)sizeof(TilePass) / 4; i += T)
      reinterpret_cast<uint32_t*>(&P)[i] = reinterpret_cast<const uint32_t*>(passes + k)[i];
    const int words = (int)(sizeof(typename Fwd<R>::Ops) * nrec / 16);
    const uint4* src = reinterpret_cast<const uint4*>(recs + ((size_t)k * B + b) * nrec);
    for (int i = tid; i < words; i += T) reinterpret_cast<uint4*>(ops)[i] = src[i];
    __syncthreads();
    fwd_rounds<R>(P, sm, ops);
    // P, through registers (the last pass's goes with the store)
    TileShare<R, FWD_LV> sh;
    sh.init(P, T);
#pragma unroll
    for (int u = 0; u < FWD_NV; ++u)
      if ((tid + T * u) * VE < (1 << kt)) v[u] = Vec<R>::from_sm(sm, sh.s(u), sh.s(u) ^ sh.s1);
    __syncthreads();
    if (k + 1 < npass) {
#pragma unroll
      for (int u = 0; u < FWD_NV; ++u)
        if ((tid + T * u) * VE < (1 << kt)) Vec<R>::to_sm(sm, sh.a(u), sh.a(u) ^ tp_at<R>(1), v[u]);
    }
  }
  V2* g = psi + ((uint64_t)b << n);
  const bool al = (reinterpret_cast<uintptr_t>(psi) & 15) == 0;
#pragma unroll
  for (int u = 0; u < FWD_NV; ++u) {
    const int e = (tid + T * u) * VE;
    if (e < ne) Vec<R>::st(g + e, v[u], al);
  }
}

template <typename R>
__global__ void k_zero_state_batch(typename CT<R>::V2* __restrict__ psi, int n, int B) {
  const uint64_t N = 1ull << n, tot = N * (uint64_t)B;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < tot; i += (uint64_t)gridDim.x * blockDim.x)
    psi[i] = CT<R>::make((R)((i & (N - 1)) == 0 ? 1 : 0), (R)0);
}

// Sum partial[b][0..gx) in order into out[b * ostride + ooff].
__global__ void k_final_batch(const double* __restrict__ part, int gx, double* __restrict__ out, int64_t ostride,
                              int64_t ooff) {
  const int b = blockIdx.x;
  double t = 0.0;
  for (int i = threadIdx.x; i < gx; i += blockDim.x) t += part[(int64_t)b * gx + i];
  t = block_reduce(t);
  if (threadIdx.x == 0) out[(int64_t)b * ostride + ooff] = t;
}

// ------------------------------------------------------------ backward ---
// A pass of the backward sweep undoes P (address map of the tile's load),
// then D, then the operators of S last to first, on psi and lambda together.
// The derivative of each rotation is taken where its own qubit has been
// undone up to it: what other qubits' operators did meanwhile is unitary and
// commutes with the generator, so it does not change Im <lambda|P|psi>.
//
//  - The derivatives of all of D's RZ come from one product
//    w_j = Im(conj(lambda_j) psi_j) per amplitude and its signed sums: over a
//    thread's register bits on the spot, over its other tile bits when the
//    block is done (the sign is the thread's).
//  - Those of S (RX, RY, inner RZ) are four products a pair.
//
// Sums: complex64 products and a thread's sums in float
// pairs (Acc), then 64-bit fixed point; complex128 in FP64 per thread, then
// two 64-bit words of fixed point.  Every sum is bounded by ||psi|| ||lambda||
// <= sum_k |c_k|, which sets the point (accumulated integers do not depend on
// the order of the blocks).
template <typename R> struct Bwd;
template <> struct Bwd<float> {
  static constexpr int KT = 12, C0 = 4, T = 512, OCC = 2, LV = 2, VE = 2;
  using Z = float2;  // a thread's running sum
};
template <> struct Bwd<double> {
  static constexpr int KT = 11, C0 = 3, T = 256, OCC = 2, LV = 3, VE = 1;
  using Z = double;
};
constexpr int BWD_SLOTS = TP_MAXOP + TP_MAXK + 3;  // sums of a pass: operators, then tile positions of D

// An operator's derivative term Im <l|P|p>, P its generator, over the pairs of
// register bit BIT; then the operator on both states.
template <int MODE, int BIT, typename R>
__device__ __forceinline__ void bwd_mode(const R t, const R u, Acc<R>& acc, Cx<R>* p, Cx<R>* l) {
  // Im(conj(a) b) = a.re b.im - a.im b.re
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const int j0 = ((m >> BIT) << (BIT + 1)) | (m & ((1 << BIT) - 1)), j1 = j0 | (1 << BIT);
    if (MODE == OM_RZ) {  // Z: conj(l0) p0 - conj(l1) p1
      acc.add(l[j0].re, p[j0].im); acc.sub(l[j0].im, p[j0].re);
      acc.sub(l[j1].re, p[j1].im); acc.add(l[j1].im, p[j1].re);
    } else if (MODE == OM_RX0 || MODE == OM_RX1) {  // X: conj(l0) p1 + conj(l1) p0
      acc.add(l[j0].re, p[j1].im); acc.sub(l[j0].im, p[j1].re);
      acc.add(l[j1].re, p[j0].im); acc.sub(l[j1].im, p[j0].re);
    } else if (MODE != OM_H) {  // Y: conj(l0)(-i p1) + conj(l1)(i p0); Im(conj(a)(-i b)) = -Re(conj(a) b)
      acc.sub(l[j0].re, p[j1].re); acc.sub(l[j0].im, p[j1].im);
      acc.add(l[j1].re, p[j0].re); acc.add(l[j1].im, p[j0].im);
    }
  }
  op_mode<MODE, BIT, 3>(t, u, p);
  op_mode<MODE, BIT, 3>(t, u, l);
}
template <int BIT, typename R>
__device__ __forceinline__ void bwd_bit(const OpRec<R>& o, Acc<R>& acc, Cx<R>* p, Cx<R>* l) {
  switch (o.mode) {
    case OM_RY0: bwd_mode<OM_RY0, BIT>(o.t, o.u, acc, p, l); break;
    case OM_RY1: bwd_mode<OM_RY1, BIT>(o.t, o.u, acc, p, l); break;
    case OM_RX0: bwd_mode<OM_RX0, BIT>(o.t, o.u, acc, p, l); break;
    case OM_RX1: bwd_mode<OM_RX1, BIT>(o.t, o.u, acc, p, l); break;
    case OM_RZ: bwd_mode<OM_RZ, BIT>(o.t, o.u, acc, p, l); break;
    default: bwd_mode<OM_H, BIT>(o.t, o.u, acc, p, l); break;
  }
}

// value * 2^k, k up to twice an exponent's range
__device__ __forceinline__ double scale2(double v, int k) { return ldexp(ldexp(v, k / 2), k - k / 2); }

// Sum of fixed-point values over the warp (in every lane); |sum| < 2^56.
__device__ __forceinline__ long long warp_sum(int2 v) {
  return ((long long)__reduce_add_sync(0xffffffffu, v.x) << 26) + __reduce_add_sync(0xffffffffu, v.y);
}

// A block's sums: shared memory behind the two tiles.
//   complex64: z[4][T] float pairs, y[nwarp][nop] integers
//   complex128: z[4][T], y[nop][T] doubles
template <typename R>
struct BwdSums {
  typename Bwd<R>::Z* z;
  void* y;
  int bad;  // this thread saw a non-finite sum
};
template <typename R>
__host__ __device__ inline size_t bwd_sum_bytes(int T, int nop) {
  return sizeof(typename Bwd<R>::Z) * 4 * T + (sizeof(R) == 4 ? (size_t)8 * (T / 32) * nop : (size_t)8 * T * nop);
}

template <typename R>
__device__ __forceinline__ void bwd_zero_sums(BwdSums<R>& S, int nop) {
  const int T = blockDim.x, words = (int)(bwd_sum_bytes<R>(T, nop) / 8);
  for (int i = threadIdx.x; i < words; i += T) reinterpret_cast<unsigned long long*>(S.z)[i] = 0ull;
}

// The C of complex64 sums of products of a thread's p and l, each component
// taken once: they stay below |p| |l| < 2^ex.  (At the ends of the range the
// sums lose the low word, not the high one.)
constexpr float ACC_TOP = 0x1.8p126f;
// Operators of a round between two looks at the amplitudes: C doubles with
// every operator, since one without its factor can double a product, but most
// do not, and after some seventeen the high word would hold nothing of a
// product.  Rounds of up to four operators (an ansatz's have three) look once.
constexpr int ACC_SPAN = 4;
template <typename R>
__device__ __forceinline__ R acc_point(const Cx<R>* p, const Cx<R>* l) {
  if constexpr (sizeof(R) == 8) {
    return 0.0;
  } else {
    float a = 0.f, b = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      a = fmaxf(a, fmaxf(fabsf(p[j].re), fabsf(p[j].im)));
      b = fmaxf(b, fmaxf(fabsf(l[j].re), fabsf(l[j].im)));
    }
    const int ex = (__float_as_int(a * b) >> 23) + 1 + 4 + 1;
    return __int_as_float((min(ex, 253) << 23) | 0x400000);
  }
}

// kq: the fixed point of complex64 sums (k_prep adds each operator's own part)
template <typename R>
__device__ __forceinline__ void bwd_rounds(const TilePass& P, typename CT<R>::V2* sp, typename CT<R>::V2* sl,
                                           const PassRec<R>* rec, BwdSums<R>& S, int kq) {
  constexpr int RB = 3, NA = 8;
  const int tid = threadIdx.x, T = blockDim.x;
  const bool active = tid < (1 << (P.kt - RB));
#pragma unroll 1
  for (int r = 0; r < P.nround; ++r) {
    const TileRound& rd = P.rd[r];
    const int base = active ? tp_round_base<R, RB>(rd) : 0;
    int bas[RB];
#pragma unroll
    for (int x = 0; x < RB; ++x) bas[x] = rd.bas[x];
    Cx<R> p[NA], l[NA];
#pragma unroll
    for (int j = 0; j < NA; ++j) {
      const int at = tp_round_at<RB>(base, bas, j);
      p[j] = AmpIO<R>::ld(sm_at(sp, at));
      l[j] = AmpIO<R>::ld(sm_at(sl, at));
    }
    if (!active) {  // lanes past a small tile take part in the warp sums only
#pragma unroll
      for (int j = 0; j < NA; ++j) p[j] = l[j] = cmake<R>((R)0, (R)0);
    }
    if (r == 0 && P.has_diag) {
      const R C = acc_point<R>(p, l);
      Acc<R> z[RB], s[RB], w;  // s: the sum of the lower half of each bit's block
#pragma unroll
      for (int j = 0; j < NA; ++j) {
        w = Acc<R>();
        w.start(C);
        w.add(l[j].re, p[j].im);
        w.sub(l[j].im, p[j].re);
        w.settle(C);
#pragma unroll
        for (int x = 0; x < RB; ++x) {  // bit x: lower half less upper half; their sum goes on to bit x + 1
          if ((j >> x) & 1) {
            z[x].merge(s[x]);
            z[x].merge_neg(w);
            w.merge(s[x]);
          } else {
            s[x] = w;
            break;
          }
        }
      }
      w.into(S.z[tid]);
#pragma unroll
      for (int x = 0; x < RB; ++x) z[x].into(S.z[(1 + x) * T + tid]);
      S.bad |= !w.finite();
    }
    if (r == 0 && (P.has_diag || P.nop)) {
      const auto A = rec->tab[tid & 31], Bw = rec->tab[32 + (tid >> 5)];
      const Cx<R> d = cmul(cmake<R>(A.x, A.y), cmake<R>(Bw.x, Bw.y));
#pragma unroll
      for (int j = 0; j < NA; ++j) {
        const auto J = rec->tab[48 + j];
        const Cx<R> f = cmul(d, cmake<R>(J.x, J.y));
        p[j] = cmul(p[j], f);
        l[j] = cmul(l[j], f);
      }
    }
    R C = 0;
#pragma unroll 1
    for (int k = rd.op0; k < rd.op1; ++k) {
      if ((k - rd.op0) % ACC_SPAN == 0) C = acc_point<R>(p, l);
      const OpRec<R> o = rec->op[k];
      Acc<R> acc;
      acc.start(C);
      switch (P.op[k].bit) {
        case 0: bwd_bit<0>(o, acc, p, l); break;
        case 1: bwd_bit<1>(o, acc, p, l); break;
        default: bwd_bit<2>(o, acc, p, l); break;
      }
      acc.settle(C);
      S.bad |= !acc.finite();
      if constexpr (sizeof(R) == 4) {
        C = fminf(2.f * C, ACC_TOP);  // an operator without its factor at most doubles a product
        const long long v = warp_sum(acc.fixed(kq + o.eq));
        long long* y = reinterpret_cast<long long*>(S.y) + (tid >> 5) * P.nop + k;
        if ((tid & 31) == 0) *y += v;
      } else {
        reinterpret_cast<double*>(S.y)[k * T + tid] += acc.value();
      }
    }
    if (active) {
#pragma unroll
      for (int j = 0; j < NA; ++j) {
        const int at = tp_round_at<RB>(base, bas, j);
        AmpIO<R>::st(sm_at(sp, at), p[j]);
        AmpIO<R>::st(sm_at(sl, at), l[j]);
      }
    }
    __syncthreads();
  }
}

// acc[2 slot + word] of one batch element; a non-finite sum sets the flag.
__device__ __forceinline__ void bwd_add(unsigned long long* acc, int slot, double v, int k) {
  const double x = scale2(v, k);
  if (!isfinite(x)) return;
  long long hi, lo;
  fx_split(x, hi, lo);
  atomicAdd(acc + 2 * slot, (unsigned long long)hi);
  atomicAdd(acc + 2 * slot + 1, (unsigned long long)lo);
}
template <typename R>
__device__ __forceinline__ void bwd_flush(const TilePass& P, const PassRec<R>* rec, BwdSums<R>& S, int kq,
                                          unsigned long long* __restrict__ acc, int* __restrict__ flag) {
  const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, wp = tid >> 5, nw = T >> 5;
  if (S.bad) *flag = 1;
  __syncthreads();
  if constexpr (sizeof(R) == 4) {
    const long long* y = reinterpret_cast<const long long*>(S.y);
    for (int k = tid; k < P.nop; k += T) {
      long long v = 0;
      for (int w = 0; w < nw; ++w) v += y[w * P.nop + k];
      if (v) atomicAdd(acc + 2 * k, (unsigned long long)v);
    }
  } else {
    const double* y = reinterpret_cast<const double*>(S.y);
    for (int k = wp; k < P.nop; k += nw) {
      double v = 0.0;
      for (int i = lane; i < T; i += 32) v += y[k * T + i];
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) bwd_add(acc, k, v, kq + rec->op[k].eq);
    }
  }
  if (!P.has_diag) return;
  int i = 0, x = 0;
  for (int p = 0; p < P.kt; ++p) {
    const bool reg = x < 3 && P.rd[0].r[x] == p;
    const int slot = reg ? 1 + x : 0, bit = reg ? -1 : i;
    if (reg) ++x;
    else ++i;
    if (P.dp[p] < 0 || (p % nw) != wp) continue;
    if constexpr (sizeof(R) == 4) {
      long long v = 0;
      for (int t = lane; t < T; t += 32) {
        Acc<float> a;
        a.s = S.z[slot * T + t].x;
        a.c = S.z[slot * T + t].y;
        const int2 f = a.fixed(kq);
        const long long w = warp_sum((bit >= 0 && ((t >> bit) & 1)) ? make_int2(-f.x, -f.y) : f);
        v += w;
      }
      if (lane == 0 && v) atomicAdd(acc + 2 * (TP_MAXOP + p), (unsigned long long)v);
    } else {
      double v = 0.0;
      for (int t = lane; t < T; t += 32) {
        const double f = S.z[slot * T + t];
        v += (bit >= 0 && ((t >> bit) & 1)) ? -f : f;
      }
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) bwd_add(acc, TP_MAXOP + p, v, kq);
    }
  }
}

// One pass over the batch: tiles blockIdx.x + gridDim.x i of state blockIdx.y.
template <typename R>
__global__ void __launch_bounds__(Bwd<R>::T, Bwd<R>::OCC) k_bwd_tile(typename CT<R>::V2* __restrict__ psi,
                                                           typename CT<R>::V2* __restrict__ lam, int n, int ntiles,
                                                           const __grid_constant__ TilePass P,
                                                           const PassRec<R>* __restrict__ recs, int kq,
                                                           unsigned long long* __restrict__ acc, int* __restrict__ flag) {
  using V2 = typename CT<R>::V2;
  using V = typename Vec<R>::T;
  constexpr int NV = 1 << Bwd<R>::LV;
  extern __shared__ __align__(16) unsigned char dynsm[];
  V2* sp = reinterpret_cast<V2*>(dynsm);
  V2* sl = sp + (1 << P.kt);
  PassRec<R>* rec = reinterpret_cast<PassRec<R>*>(sl + (1 << P.kt));
  BwdSums<R> S{reinterpret_cast<typename Bwd<R>::Z*>(rec + 1), nullptr, 0};
  S.y = S.z + 4 * blockDim.x;
  const int tid = threadIdx.x, T = blockDim.x;
  const bool al = ((reinterpret_cast<uintptr_t>(psi) | reinterpret_cast<uintptr_t>(lam)) & 15) == 0;
  {
    const uint4* src = reinterpret_cast<const uint4*>(recs + blockIdx.y);
    for (int i = tid; i < (int)(sizeof(PassRec<R>) / 16); i += T) reinterpret_cast<uint4*>(rec)[i] = src[i];
  }
  bwd_zero_sums<R>(S, P.nop);
  TileShare<R, Bwd<R>::LV> sh;
  sh.init(P, T);
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const uint64_t base = tp_tile_base(P, tile);
    V2* gp = psi + ((uint64_t)blockIdx.y << n) + base;
    V2* gl = lam + ((uint64_t)blockIdx.y << n) + base;
    const int cst = tp_cst(P, base);
    V vp[NV], vl[NV];
#pragma unroll
    for (int u = 0; u < NV; ++u) vp[u] = Vec<R>::ld(gp + sh.g(u), al);
#pragma unroll
    for (int u = 0; u < NV; ++u) vl[u] = Vec<R>::ld(gl + sh.g(u), al);
#pragma unroll
    for (int u = 0; u < NV; ++u) {
      const int s = sh.s(u) ^ cst;
      Vec<R>::to_sm(sp, s, s ^ sh.s1, vp[u]);
      Vec<R>::to_sm(sl, s, s ^ sh.s1, vl[u]);
    }
    __syncthreads();
    bwd_rounds<R>(P, sp, sl, rec, S, kq);
#pragma unroll
    for (int u = 0; u < NV; ++u) {
      const int a = sh.a(u), a1 = a ^ tp_at<R>(1);
      Vec<R>::st(gp + sh.g(u), Vec<R>::from_sm(sp, a, a1), al);
      Vec<R>::st(gl + sh.g(u), Vec<R>::from_sm(sl, a, a1), al);
    }
    __syncthreads();
  }
  bwd_flush<R>(P, rec, S, kq, acc + (size_t)blockIdx.y * BWD_SLOTS * 2, flag + blockIdx.y);
}

// The whole backward sweep of states that fit one tile, one block a state.
template <typename R>
__global__ void __launch_bounds__(Bwd<R>::T, Bwd<R>::OCC) k_bwd_whole(const typename CT<R>::V2* __restrict__ psi,
                                                            const typename CT<R>::V2* __restrict__ lam, int n,
                                                            const TilePass* __restrict__ passes, int npass,
                                                            const PassRec<R>* __restrict__ recs, int kq,
                                                            unsigned long long* __restrict__ acc, int* __restrict__ flag,
                                                            int B) {
  using V2 = typename CT<R>::V2;
  using V = typename Vec<R>::T;
  constexpr int NV = 1 << Bwd<R>::LV, VE = Bwd<R>::VE;
  extern __shared__ __align__(16) unsigned char dynsm[];
  __shared__ TilePass P;
  const int tid = threadIdx.x, T = blockDim.x, kt = passes[0].kt, b = blockIdx.x;
  V2* sp = reinterpret_cast<V2*>(dynsm);
  V2* sl = sp + (1 << kt);
  PassRec<R>* rec = reinterpret_cast<PassRec<R>*>(sl + (1 << kt));
  BwdSums<R> S{reinterpret_cast<typename Bwd<R>::Z*>(rec + 1), nullptr, 0};
  S.y = S.z + 4 * T;
  const V2 zero = CT<R>::make((R)0, (R)0);
  for (int e = tid; e < (1 << kt); e += T) {
    *sm_at(sp, tp_at<R>(e)) = e < (1 << n) ? psi[((uint64_t)b << n) + e] : zero;
    *sm_at(sl, tp_at<R>(e)) = e < (1 << n) ? lam[((uint64_t)b << n) + e] : zero;
  }
  __syncthreads();
#pragma unroll 1
  for (int k = npass - 1; k >= 0; --k) {
    for (int i = tid; i < (int)sizeof(TilePass) / 4; i += T)
      reinterpret_cast<uint32_t*>(&P)[i] = reinterpret_cast<const uint32_t*>(passes + k)[i];
    const uint4* src = reinterpret_cast<const uint4*>(recs + (size_t)k * B + b);
    for (int i = tid; i < (int)(sizeof(PassRec<R>) / 16); i += T) reinterpret_cast<uint4*>(rec)[i] = src[i];
    __syncthreads();
    bwd_zero_sums<R>(S, P.nop);
    if (P.has_perm) {
      TileShare<R, Bwd<R>::LV> sh;
      sh.init(P, T);
      V vp[NV], vl[NV];
#pragma unroll
      for (int u = 0; u < NV; ++u)
        if ((tid + T * u) * VE < (1 << kt)) {
          const int a = sh.a(u), a1 = a ^ tp_at<R>(1);
          vp[u] = Vec<R>::from_sm(sp, a, a1);
          vl[u] = Vec<R>::from_sm(sl, a, a1);
        }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < NV; ++u)
        if ((tid + T * u) * VE < (1 << kt)) {
          const int s = sh.s(u);
          Vec<R>::to_sm(sp, s, s ^ sh.s1, vp[u]);
          Vec<R>::to_sm(sl, s, s ^ sh.s1, vl[u]);
        }
    }
    __syncthreads();
    bwd_rounds<R>(P, sp, sl, rec, S, kq);
    bwd_flush<R>(P, rec, S, kq, acc + ((size_t)k * B + b) * BWD_SLOTS * 2, flag + b);
    __syncthreads();
  }
}

// The sums of pass blockIdx.x, element blockIdx.y, into the gradient.
template <typename R>
__global__ void __launch_bounds__(64) k_bwd_finish(const TilePass* __restrict__ passes, const PassRec<R>* __restrict__ recs,
                                                   const unsigned long long* __restrict__ acc,
                                                   const int* __restrict__ flag, int B, int kq, double* __restrict__ grad,
                                                   int64_t stride) {
  const TilePass& P = passes[blockIdx.x];
  const int64_t pb = (int64_t)blockIdx.x * B + blockIdx.y;
  for (int slot = threadIdx.x; slot < BWD_SLOTS; slot += blockDim.x) {
    const bool op = slot < TP_MAXOP;
    if (op ? slot >= P.nop : P.dp[slot - TP_MAXOP] < 0) continue;
    const int par = op ? P.op[slot].pa : P.dp[slot - TP_MAXOP];
    if (par < 0) continue;  // H
    const OpRec<R>* o = op ? &recs[pb].op[slot] : nullptr;
    const unsigned long long* a = acc + (pb * BWD_SLOTS + slot) * 2;
    double v = fx_join((long long)a[0], (long long)a[1]);
    v = scale2(v, -(kq + (op ? o->eq : 0)));
    if (op) v *= o->f;
    if (flag[blockIdx.y]) v = __longlong_as_double(0x7ff8000000000000ll);
    grad[(int64_t)blockIdx.y * stride + par] = v;
  }
}

// lam = H psi = sum_k c_k P_k psi, P_k = i^{|x&z|} X^x Z^z:
// (P psi)[j] = i^{|x&z|} (-1)^{|(j^x)&z|} psi[j^x],
// and Re <psi|lam> per batch element (block partials).  The factor of i and
// (-1)^{|x&z|} are folded into the coefficient on the host; what is left of a
// term is a load, the parity of j & z if z is not zero, and two multiply-adds.
// A thread takes four amplitudes a term, and a block a contiguous chunk, so
// that partners across the low index bits come from its L1.  64 states of 20
// qubits, 21 terms: 3.55 ms with one amplitude a thread and a pass of its own
// for the energy.
template <typename R>
struct TermsDev {
  int nt;
  uint32_t x[64], z[64];
  R c[64];
  uint8_t imag[64];  // the coefficient is i c
};
constexpr int AH_UNR = 4, AH_CHUNK = 4096;

template <typename R>
__global__ void __launch_bounds__(ADJ_T) k_apply_h(const typename CT<R>::V2* __restrict__ psi,
                                                   typename CT<R>::V2* __restrict__ lam, int n,
                                                   const __grid_constant__ TermsDev<R> T, double* __restrict__ part) {
  using V2 = typename CT<R>::V2;
  const int b = blockIdx.y;
  const V2* s = psi + ((uint64_t)b << n);
  V2* l = lam + ((uint64_t)b << n);
  const uint32_t N = 1u << n;
  double e = 0.0;
  for (uint64_t c0 = (uint64_t)blockIdx.x * AH_CHUNK; c0 < N; c0 += (uint64_t)gridDim.x * AH_CHUNK) {
    SumE<R> acc;
    for (uint32_t j0 = (uint32_t)c0 + threadIdx.x; j0 < (uint32_t)min((uint64_t)N, c0 + AH_CHUNK); j0 += AH_UNR * ADJ_T) {
      R ar[AH_UNR], ai[AH_UNR];
#pragma unroll
      for (int u = 0; u < AH_UNR; ++u) ar[u] = ai[u] = 0;
      for (int k = 0; k < T.nt; ++k) {
        const uint32_t x = T.x[k], z = T.z[k];
        const R c = T.c[k];
        const bool imag = T.imag[k];
        V2 v[AH_UNR];
#pragma unroll
        for (int u = 0; u < AH_UNR; ++u) {
          const uint32_t j = j0 + u * ADJ_T;
          if (j < N) v[u] = s[j ^ x];
        }
#pragma unroll
        for (int u = 0; u < AH_UNR; ++u) {
          const uint32_t j = j0 + u * ADJ_T;
          if (j < N) {
            const R cj = z && (__popc(j & z) & 1) ? -c : c;
            if (imag) {
              ar[u] = fma(-cj, v[u].y, ar[u]);
              ai[u] = fma(cj, v[u].x, ai[u]);
            } else {
              ar[u] = fma(cj, v[u].x, ar[u]);
              ai[u] = fma(cj, v[u].y, ai[u]);
            }
          }
        }
      }
#pragma unroll
      for (int u = 0; u < AH_UNR; ++u) {
        const uint32_t j = j0 + u * ADJ_T;
        if (j < N) {
          const V2 v = s[j];
          l[j] = CT<R>::make(ar[u], ai[u]);
          acc.add(v.x, ar[u]);
          acc.add(v.y, ai[u]);
        }
      }
    }
    acc.flush();
    e += acc.value();
  }
  const double t = block_reduce(e);
  if (threadIdx.x == 0) part[(int64_t)b * gridDim.x + blockIdx.x] = t;
}

// ------------------------------------------------------------ host side --
static qc_status check_circuit(int n, qc_dtype dt, int B, const qc_gate* gates, int n_gates, int64_t stride,
                               int n_params) {
  if (n < 2 || n > 30) {
    set_error("n = %d out of range [2, 30]", n);
    return QC_EINVAL;
  }
  if (dt != QC_C128 && dt != QC_C64) {
    set_error("unknown dtype %d", (int)dt);
    return QC_EINVAL;
  }
  if (B < 1 || B > 65535) {
    set_error("batch B = %d out of range [1, 65535]", B);
    return QC_EINVAL;
  }
  if (n_gates < 0 || (n_gates > 0 && !gates)) {
    set_error("bad gate list");
    return QC_EINVAL;
  }
  for (int i = 0; i < n_gates; ++i) {
    const qc_gate& g = gates[i];
    if (g.kind < QC_G_RX || g.kind > QC_G_H || g.q0 < 0 || g.q0 >= n) {
      set_error("gate %d: bad kind %d or qubit %d", i, g.kind, g.q0);
      return QC_EINVAL;
    }
    if (g.kind == QC_G_CNOT && (g.q1 < 0 || g.q1 >= n || g.q1 == g.q0)) {
      set_error("gate %d: bad CNOT target %d", i, g.q1);
      return QC_EINVAL;
    }
    if (g.kind <= QC_G_RZ && (g.param < 0 || g.param >= stride || (n_params > 0 && g.param >= n_params))) {
      set_error("gate %d: parameter index %d out of range", i, g.param);
      return QC_EINVAL;
    }
  }
  return QC_OK;
}

// Blocks per batch element of the H psi pass.
template <typename R>
static unsigned gx_for(int n, int B) {
  const uint64_t chunks = std::max<uint64_t>(1, (1ull << n) / AH_CHUNK);
  const uint64_t cap = std::max<uint64_t>(
      1, 4ull * sm_count() * resident_blocks((const void*)k_apply_h<R>, ADJ_T, 0) / (uint64_t)B);
  return (unsigned)std::min<uint64_t>({chunks, cap, ADJ_GX_MAX});
}

// Passes of a forward sweep on the device, with room for the operators of as
// many batch elements at a time as fit PREP_BYTES.
constexpr size_t PREP_BYTES = 64u << 20;
template <typename R>
struct FwdPlan {
  std::vector<TilePass> passes;
  TilePass* dpass = nullptr;
  typename Fwd<R>::Ops* recs = nullptr;
  int chunk = 0;  // batch elements at a time
  static constexpr int nrec = sizeof(R) == 4 ? TP_MAXOP : 1;
};

template <typename R>
static cudaError_t fwd_plan(FwdPlan<R>& F, const qc_gate* gates, int ng, int n, int B, cudaStream_t st) {
  // complex128: an SM's FP64 pipe bounds a tile (2^12 amplitudes under two
  // operators: 12 us), so that tiles shrink down to 2^10 until there are 256 of
  // them.  60 x (RX, RY, CNOT) on three of 14 qubits: 888 us gate by gate, 855
  // with tiles of 2^12, 514 of 2^10, 511 of 2^9 (whose lists get longer: over
  // circuits of 5 to 20 qubits 1.01 times the time).
  const int few = n - 8 + 31 - __builtin_clz((unsigned)B);
  const int kt = sizeof(R) == 8 ? std::max(10, std::min<int>(Fwd<R>::KT, few)) : Fwd<R>::KT;
  const PassCfg cfg{kt, Fwd<R>::C0, Fwd<R>::RB, sizeof(R) == 4, false};
  F.passes = build_passes<R>(gates, ng, n, cfg);
  if (F.passes.empty()) return cudaSuccess;
  const size_t per = F.passes.size() * F.nrec * sizeof(typename Fwd<R>::Ops);
  F.chunk = (int)std::max<size_t>(1, std::min<size_t>(B, PREP_BYTES / per));
  cudaError_t e = ws_alloc((void**)&F.dpass, (F.passes.size() * sizeof(TilePass) + 15) / 16 * 16, st);
  if (e == cudaSuccess) e = ws_alloc((void**)&F.recs, per * F.chunk, st);
  return e;
}
template <typename R>
static void fwd_plan_free(FwdPlan<R>& F, cudaStream_t st) {
  if (F.dpass) cudaFreeAsync(F.dpass, st);
  if (F.recs) cudaFreeAsync(F.recs, st);
}

// psi_b = U_G .. U_1 |0..0>; returns the launches made.
template <typename R>
static int forward_passes(const FwdPlan<R>& F, int n, int B, const double* theta, int64_t stride,
                          typename CT<R>::V2* psi, cudaStream_t st) {
  if (F.passes.empty()) {
    k_zero_state_batch<R><<<grid_for((int64_t)B << n, ADJ_T, 8), ADJ_T, 0, st>>>(psi, n, B);
    return 1;
  }
  const int np = (int)F.passes.size();
  int nk = put_bytes(F.dpass, F.passes.data(), np * sizeof(TilePass), st);
  const int kt = F.passes[0].kt, T = std::max(32, 1 << (kt - Fwd<R>::RB));
  const size_t ops = sizeof(typename Fwd<R>::Ops) * F.nrec, smem = (sizeof(typename CT<R>::V2) << kt) + ops;
  constexpr size_t most = sizeof(typename CT<R>::V2) << Fwd<R>::KT;
  allow_smem(k_fwd_tile<R>, most + ops);
  allow_smem(k_fwd_whole<R>, most + ops);
  for (int b0 = 0; b0 < B; b0 += F.chunk) {
    const int nb = std::min(F.chunk, B - b0);
    const double* th = theta + (int64_t)b0 * stride;
    typename CT<R>::V2* s = psi + ((uint64_t)b0 << n);
    if constexpr (sizeof(R) == 4)
      k_prep_mats<<<dim3(np, nb), 64, 0, st>>>(F.dpass, F.recs, nb, th, stride);
    else
      k_prep<R><<<dim3(np, nb), 128, 0, st>>>(F.dpass, F.recs, nb, th, stride, 1);
    ++nk;
    if (n <= kt) {
      k_fwd_whole<R><<<nb, T, smem, st>>>(s, n, F.dpass, np, F.recs, F.nrec, nb);
      ++nk;
    } else {
      for (int k = 0; k < np; ++k, ++nk)
        k_fwd_tile<R><<<dim3(1u << (n - kt), nb), T, smem, st>>>(s, n, F.passes[k], F.recs + (size_t)k * nb * F.nrec,
                                                                 F.nrec, k == 0);
    }
  }
  return nk;
}

template <typename R>
static qc_status forward_impl(int n, int B, const qc_gate* gates, int n_gates, const double* theta,
                              int64_t stride, void* psi, cudaStream_t st) {
  FwdPlan<R> F;
  const cudaError_t e = fwd_plan(F, gates, n_gates, n, B, st);
  if (e != cudaSuccess) {
    fwd_plan_free(F, st);
    return cuda_fail(e, "forward workspace");
  }
  const int nk = forward_passes<R>(F, n, B, theta, stride, reinterpret_cast<typename CT<R>::V2*>(psi), st);
  fwd_plan_free(F, st);
  return check_launch("circuit forward", nk);
}

// The backward sweep on the device: passes, and the operators and sums of as
// many batch elements at a time as fit PREP_BYTES.
template <typename R>
struct BwdPlan {
  std::vector<TilePass> passes;
  TilePass* dpass = nullptr;
  PassRec<R>* recs = nullptr;
  unsigned long long* acc = nullptr;  // sums, then a flag per element
  int chunk = 0;
  size_t acc_bytes(int nb) const { return passes.size() * nb * BWD_SLOTS * 16 + sizeof(int) * (size_t)nb; }
};
template <typename R>
static cudaError_t bwd_plan(BwdPlan<R>& W, const qc_gate* gates, int ng, int n, int B, cudaStream_t st) {
  W.passes = build_passes<R>(gates, ng, n, PassCfg{Bwd<R>::KT, Bwd<R>::C0, 3, false, true});
  if (W.passes.empty()) return cudaSuccess;
  const size_t np = W.passes.size();
  W.chunk = (int)std::max<size_t>(1, std::min<size_t>(B, PREP_BYTES / (np * (sizeof(PassRec<R>) + BWD_SLOTS * 16))));
  cudaError_t e = ws_alloc((void**)&W.dpass, (np * sizeof(TilePass) + 15) / 16 * 16, st);
  if (e == cudaSuccess) e = ws_alloc((void**)&W.recs, np * W.chunk * sizeof(PassRec<R>), st);
  if (e == cudaSuccess) e = ws_alloc((void**)&W.acc, W.acc_bytes(W.chunk), st);
  return e;
}
template <typename R>
static void bwd_plan_free(BwdPlan<R>& W, cudaStream_t st) {
  if (W.dpass) cudaFreeAsync(W.dpass, st);
  if (W.recs) cudaFreeAsync(W.recs, st);
  if (W.acc) cudaFreeAsync(W.acc, st);
}

// Walks the circuit back from psi and lambda; kq: fixed point of the sums.
template <typename R>
static int backward_passes(const BwdPlan<R>& W, int n, int B, const double* theta, int64_t stride, int kq,
                           typename CT<R>::V2* psi, typename CT<R>::V2* lam, double* grad, cudaStream_t st) {
  if (W.passes.empty()) return 0;
  const int np = (int)W.passes.size();
  int nk = put_bytes(W.dpass, W.passes.data(), np * sizeof(TilePass), st), maxop = 0;
  for (const TilePass& P : W.passes) maxop = std::max<int>(maxop, P.nop);
  const int kt = W.passes[0].kt, T = std::max(32, 1 << (kt - 3));
  const size_t tiles2 = 2 * (sizeof(typename CT<R>::V2) << kt) + sizeof(PassRec<R>);
  const size_t most = 2 * (sizeof(typename CT<R>::V2) << Bwd<R>::KT) + sizeof(PassRec<R>) +
                      bwd_sum_bytes<R>(Bwd<R>::T, TP_MAXOP);
  allow_smem(k_bwd_tile<R>, most);
  allow_smem(k_bwd_whole<R>, most);
  for (int b0 = 0; b0 < B; b0 += W.chunk) {
    const int nb = std::min(W.chunk, B - b0);
    const double* th = theta + (int64_t)b0 * stride;
    typename CT<R>::V2 *p = psi + ((uint64_t)b0 << n), *l = lam + ((uint64_t)b0 << n);
    cudaMemsetAsync(W.acc, 0, W.acc_bytes(nb), st);
    int* flag = reinterpret_cast<int*>(W.acc + (size_t)np * nb * BWD_SLOTS * 2);
    k_prep<R><<<dim3(np, nb), 128, 0, st>>>(W.dpass, W.recs, nb, th, stride, -1);
    ++nk;
    if (n <= kt) {
      k_bwd_whole<R><<<nb, T, tiles2 + bwd_sum_bytes<R>(T, maxop), st>>>(p, l, n, W.dpass, np, W.recs, kq, W.acc, flag,
                                                                        nb);
      ++nk;
    } else {
      // a block takes up to eight tiles of a state (its sums then cost
      // little), as long as six waves of blocks remain
      const int64_t tiles = 1ll << (n - kt), all = tiles * nb;
      const int64_t per = std::max<int64_t>(1, std::min<int64_t>({8, tiles, all / (12ll * sm_count())}));
      const dim3 grid((unsigned)((tiles + per - 1) / per), nb);
      for (int k = np - 1; k >= 0; --k, ++nk)
        k_bwd_tile<R><<<grid, T, tiles2 + bwd_sum_bytes<R>(T, W.passes[k].nop), st>>>(
            p, l, n, (int)tiles, W.passes[k], W.recs + (size_t)k * nb, kq, W.acc + (size_t)k * nb * BWD_SLOTS * 2,
            flag);
    }
    k_bwd_finish<R><<<dim3(np, nb), 64, 0, st>>>(W.dpass, W.recs, W.acc, flag, nb, kq, grad + (int64_t)b0 * stride,
                                                 stride);
    ++nk;
  }
  return nk;
}

template <typename R>
static qc_status adjoint_impl(int n, int B, const qc_gate* gates, int n_gates, const double* theta,
                              int64_t stride, const qc_pauli_term* H, int n_terms, void* psi, void* lam,
                              double* energy, double* grad, cudaStream_t st) {
  using V2 = typename CT<R>::V2;
  const unsigned gx = gx_for<R>(n, B);
  const dim3 grid(gx, B);
  V2 *p = reinterpret_cast<V2*>(psi), *l = reinterpret_cast<V2*>(lam);
  double* part = nullptr;
  FwdPlan<R> F;
  BwdPlan<R> W;
  cudaError_t e = ws_alloc((void**)&part, sizeof(double) * (size_t)gx * B, st);
  if (e == cudaSuccess) e = fwd_plan(F, gates, n_gates, n, B, st);
  qc_status s = QC_OK;
  if (e == cudaSuccess) {
    TermsDev<R> T;
    double bound = 0.0;  // ||H|| <= sum |c_k|
    T.nt = n_terms;
    for (int k = 0; k < n_terms; ++k) {
      const uint64_t x = H[k].xmask, z = H[k].zmask;
      const int ny = __builtin_popcountll(x & z);  // i^ny (-1)^ny = (-i)^ny
      T.x[k] = (uint32_t)x;
      T.z[k] = (uint32_t)z;
      T.imag[k] = ny & 1;
      T.c[k] = (R)(((ny & 3) == 1 || (ny & 3) == 2) ? -H[k].coeff : H[k].coeff);
      bound += std::fabs(H[k].coeff) / 64.0;
    }
    // sums stay below 2^55 units: bound * 64 < 2^(ilogb + 7)
    int kq = 55 - (bound > 0.0 ? std::ilogb(bound) + 7 : 0);
    if (sizeof(R) == 4) kq = std::min(160, std::max(-160, kq));  // past this H is 0 or infinite in complex64
    e = cudaMemsetAsync(grad, 0, sizeof(double) * (size_t)B * stride, st);
    if (e != cudaSuccess) s = cuda_fail(e, "adjoint setup");
    if (!s) {
      int nk = forward_passes<R>(F, n, B, theta, stride, p, st);
      k_apply_h<R><<<grid, ADJ_T, 0, st>>>(p, l, n, T, part);
      k_final_batch<<<B, ADJ_T, 0, st>>>(part, gx, energy, 1, 0);
      nk += 2;
      // the backward passes are planned while the forward ones run
      e = bwd_plan(W, gates, n_gates, n, B, st);
      if (e != cudaSuccess) s = cuda_fail(e, "adjoint workspace");
      else nk += backward_passes<R>(W, n, B, theta, stride, kq, p, l, grad, st);
      const qc_status sl = check_launch("adjoint", nk);
      if (!s) s = sl;
    }
  } else {
    s = cuda_fail(e, "adjoint workspace");
  }
  e = cudaStreamSynchronize(st);
  if (part) cudaFreeAsync(part, st);
  fwd_plan_free(F, st);
  bwd_plan_free(W, st);
  if (!s && e != cudaSuccess) s = cuda_fail(e, "adjoint");
  return s;
}

static qc_status check_param_once(const qc_gate* gates, int n_gates) {
  // each angle may drive at most one gate (the gradient slot is written,
  // not accumulated)
  std::vector<int> seen;
  for (int i = 0; i < n_gates; ++i)
    if (gates[i].kind <= QC_G_RZ) seen.push_back(gates[i].param);
  std::sort(seen.begin(), seen.end());
  for (size_t i = 1; i < seen.size(); ++i)
    if (seen[i] == seen[i - 1]) {
      set_error("parameter %d drives more than one gate", seen[i]);
      return QC_EINVAL;
    }
  return QC_OK;
}

}  // namespace qc

using namespace qc;

QC_API qc_status qc_circuit_forward(int n, qc_dtype dt, int B, const qc_gate* gates, int n_gates,
                                    const double* theta_dev, int64_t theta_stride, void* psi_dev, void* stream) {
  clear_error();
  qc_status s = check_circuit(n, dt, B, gates, n_gates, theta_stride, 0);
  if (s) return s;
  if (!psi_dev || (!theta_dev && n_gates > 0)) {
    set_error("NULL device buffer");
    return QC_EINVAL;
  }
  cudaStream_t st = (cudaStream_t)stream;
  return dt == QC_C128 ? forward_impl<double>(n, B, gates, n_gates, theta_dev, theta_stride, psi_dev, st)
                       : forward_impl<float>(n, B, gates, n_gates, theta_dev, theta_stride, psi_dev, st);
}

QC_API qc_status qc_adjoint_grad(int n, qc_dtype dt, int B, const qc_gate* gates, int n_gates,
                                 const double* theta_dev, int64_t theta_stride, int n_params,
                                 const qc_pauli_term* H, int n_terms, void* psi_dev, void* lam_dev,
                                 double* energy_dev, double* grad_dev, void* stream) {
  clear_error();
  qc_status s = check_circuit(n, dt, B, gates, n_gates, theta_stride, n_params);
  if (!s) s = check_param_once(gates, n_gates);
  if (s) return s;
  if (n_params < 0 || n_params > theta_stride) {
    set_error("n_params = %d out of range [0, theta_stride]", n_params);
    return QC_EINVAL;
  }
  if (!H || n_terms < 1 || n_terms > 64) {
    set_error("need 1..64 Hamiltonian terms");
    return QC_EINVAL;
  }
  for (int k = 0; k < n_terms; ++k)
    if ((n < 64 && ((H[k].xmask | H[k].zmask) >> n)) || !std::isfinite(H[k].coeff)) {
      set_error("Hamiltonian term %d has bits at or above n or a non-finite coefficient", k);
      return QC_EINVAL;
    }
  if (!psi_dev || !lam_dev || !energy_dev || !grad_dev || (!theta_dev && n_gates > 0)) {
    set_error("NULL device buffer");
    return QC_EINVAL;
  }
  cudaStream_t st = (cudaStream_t)stream;
  return dt == QC_C128 ? adjoint_impl<double>(n, B, gates, n_gates, theta_dev, theta_stride, H, n_terms,
                                              psi_dev, lam_dev, energy_dev, grad_dev, st)
                       : adjoint_impl<float>(n, B, gates, n_gates, theta_dev, theta_stride, H, n_terms,
                                             psi_dev, lam_dev, energy_dev, grad_dev, st);
}
