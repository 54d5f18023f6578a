// The paper's noise intrusions and the ensemble density matrix (sec. 6.1-6.3).
//
// * qc_wigner_d: the Wigner rotation D^j(alpha, beta, gamma) for j = 1/2
//   (D2, a one-qubit intrusion) and j = 3/2 (D4, a two-qubit one), rows and
//   columns ordered m = j .. -j, D_{m'm} = e^{-i m' alpha} d^j_{m'm}(beta)
//   e^{-i m gamma}; host arithmetic, applied with qc_apply_1q / qc_apply_2q.
// * qc_density_matrix: <n|rho|n'> = sum_a P_a C_a(n) C_a(n')^* over a batch
//   of B states ("multiverses"), written out for small n.
// * qc_mixed_spectrum: the eigenvalues of rho without forming it.  rho has
//   rank <= B, and its nonzero eigenvalues are those of the B x B Gram
//   matrix G_ab = sqrt(P_a P_b) <psi_a|psi_b>, which one streaming pass over
//   the batch builds; a cluster reduces G to tridiagonal form (Householder)
//   and one CTA an eigenvalue finds it by multisection.  Trace,
//   purity Tr rho^2 and the entropy -sum l ln l follow.
//
// Inner products run in double-float on the FP32 pipe (GB300's FP64 rate is
// ~1/70 of FP32); the eigenvalue solver works in FP64 on a matrix of at
// most 64 x 64.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "common.cuh"

namespace qc {

// ------------------------------------------------ amplitudes as ff pairs --
// A non-finite amplitude becomes a NaN pair (the double-float split would
// turn it into a finite value), so that it reaches the Gram matrix.
__device__ __forceinline__ ffc load_ffc(const double2* p, uint64_t i) {
  const double2 v = p[i];
  if (!isfinite(v.x) || !isfinite(v.y)) return ffc_make(ff_make(NAN, 0.f), ff_make(NAN, 0.f));
  return ffc_make(ff_from_d(v.x), ff_from_d(v.y));
}
__device__ __forceinline__ ffc load_ffc(const float2* p, uint64_t i) {
  const float2 v = p[i];
  return ffc_make(ff_make(v.x, 0.f), ff_make(v.y, 0.f));
}
template <typename V2> __device__ __forceinline__ V2 ffc_to_v2(const ffc& z);
template <> __device__ __forceinline__ double2 ffc_to_v2<double2>(const ffc& z) {
  if (!isfinite(z.re.hi) || !isfinite(z.im.hi)) return make_double2(NAN, NAN);  // the join would make it finite
  return make_double2(ff_to_d(z.re), ff_to_d(z.im));
}
template <> __device__ __forceinline__ float2 ffc_to_v2<float2>(const ffc& z) {
  return make_float2(z.re.hi + z.re.lo, z.im.hi + z.im.lo);
}
__device__ __forceinline__ double2 conj_v(double2 v) { return make_double2(v.x, -v.y); }
__device__ __forceinline__ float2 conj_v(float2 v) { return make_float2(v.x, -v.y); }

// rho is Hermitian: only tiles on and above the diagonal are formed, and an
// off-diagonal tile's conjugate transpose goes through shared memory (Tm) to
// the mirrored tile in coalesced rows.
template <typename V2>
__device__ __forceinline__ void rho_mirror(V2 (*Tm)[33], V2* __restrict__ rho, uint64_t N, uint64_t r0, uint64_t c0) {
  __syncthreads();
  for (int e = threadIdx.x; e < 32 * 32; e += blockDim.x) {
    const int rr = e >> 5, cc = e & 31;
    if (c0 + rr < N && r0 + cc < N) rho[(c0 + rr) * N + r0 + cc] = Tm[rr][cc];
  }
}

// acc += a * conj(b)
__device__ __forceinline__ void mac_conj_b(ffc& acc, const ffc& a, const ffc& b) {
  acc.re = ff_add(acc.re, ff_dot2p(a.re, b.re, a.im, b.im));
  acc.im = ff_add(acc.im, ff_dot2m(a.im, b.re, a.re, b.im));
}

// ------------------------------------------------------------- rho -------
#define RHO_TILE 32
#define RHO_KC 16

// A thread's 2 x 2 entries of the 32 x 32 tile (rows r0 + 2 ty + i, columns
// c0 + 2 tx + j) in double-float.  SIZES: also the sums of the terms' sizes
// (|re| + |im| of each factor).
template <bool SIZES>
__device__ __forceinline__ void rho_tile_c128(const double2* __restrict__ psi, uint64_t N, int B,
                                              const double* __restrict__ P, uint64_t r0, uint64_t c0,
                                              ffc (*Ar)[RHO_TILE], ffc (*Ac)[RHO_TILE], ffc (*acc)[2],
                                              float (*size)[2]) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  for (int i = 0; i < 2; ++i)
    for (int j = 0; j < 2; ++j) {
      acc[i][j] = ffc_make(ff_make(0.f, 0.f), ff_make(0.f, 0.f));
      if (SIZES) size[i][j] = 0.f;
    }
  for (int a0 = 0; a0 < B; a0 += RHO_KC) {
    const int kc = min(RHO_KC, B - a0);
    for (int e = threadIdx.x; e < kc * RHO_TILE; e += blockDim.x) {
      const int k = e / RHO_TILE, x = e % RHO_TILE;
      const int a = a0 + k;
      ffc vr = ffc_make(ff_make(0.f, 0.f), ff_make(0.f, 0.f)), vc = vr;
      const ff w = ff_from_d(P[a]);
      if (r0 + x < N) {
        vr = load_ffc(psi, (uint64_t)a * N + r0 + x);
        vr = ffc_make(ff_mul(vr.re, w), ff_mul(vr.im, w));
      }
      if (c0 + x < N) vc = load_ffc(psi, (uint64_t)a * N + c0 + x);
      Ar[k][x] = vr;
      Ac[k][x] = vc;
    }
    __syncthreads();
#pragma unroll 4
    for (int k = 0; k < kc; ++k) {
      const ffc r[2] = {Ar[k][2 * ty], Ar[k][2 * ty + 1]}, c[2] = {Ac[k][2 * tx], Ac[k][2 * tx + 1]};
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          mac_conj_b(acc[i][j], r[i], c[j]);
          if (SIZES)
            size[i][j] = fmaf(fabsf(r[i].re.hi) + fabsf(r[i].im.hi), fabsf(c[j].re.hi) + fabsf(c[j].im.hi), size[i][j]);
        }
    }
    __syncthreads();
  }
}

// One CTA: a 32 x 32 tile of rho (rows r0.., columns c0..); each of the 256
// threads owns 2 x 2 entries.  The weights P_a scale the row operands.
template <typename V2>
__global__ void __launch_bounds__(256) k_rho(const V2* __restrict__ psi, uint64_t N, int B,
                                             const double* __restrict__ P, V2* __restrict__ rho) {
  static_assert(RHO_TILE == 32, "the mirror tile is 32 x 32");
  if (blockIdx.y > blockIdx.x) return;  // the mirror of a tile above the diagonal
  const bool mirror = blockIdx.y != blockIdx.x;
  __shared__ ffc Ar[RHO_KC][RHO_TILE], Ac[RHO_KC][RHO_TILE];
  __shared__ V2 Tm[RHO_TILE][RHO_TILE + 1];
  const uint64_t r0 = (uint64_t)blockIdx.y * RHO_TILE, c0 = (uint64_t)blockIdx.x * RHO_TILE;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  if constexpr (std::is_same<V2, float2>::value) {
    // complex64: plain FP32 (B terms per entry, the dtype's own precision)
    __shared__ float2 Fr[RHO_KC][RHO_TILE], Fc[RHO_KC][RHO_TILE];
    float2 f[2][2] = {{{0.f, 0.f}, {0.f, 0.f}}, {{0.f, 0.f}, {0.f, 0.f}}};
    for (int a0 = 0; a0 < B; a0 += RHO_KC) {
      for (int e = threadIdx.x; e < RHO_KC * RHO_TILE; e += blockDim.x) {
        const int k = e / RHO_TILE, x = e % RHO_TILE, a = a0 + k;
        float2 vr = make_float2(0.f, 0.f), vc = vr;
        if (a < B) {
          const float w = (float)P[a];
          if (r0 + x < N) {
            vr = psi[(uint64_t)a * N + r0 + x];
            vr.x *= w;
            vr.y *= w;
          }
          if (c0 + x < N) vc = psi[(uint64_t)a * N + c0 + x];
        }
        Fr[k][x] = vr;
        Fc[k][x] = vc;
      }
      __syncthreads();
#pragma unroll
      for (int k = 0; k < RHO_KC; ++k) {
        const float2 r[2] = {Fr[k][2 * ty], Fr[k][2 * ty + 1]}, c[2] = {Fc[k][2 * tx], Fc[k][2 * tx + 1]};
        for (int i = 0; i < 2; ++i)
          for (int j = 0; j < 2; ++j) {  // r conj(c)
            f[i][j].x = fmaf(r[i].x, c[j].x, fmaf(r[i].y, c[j].y, f[i][j].x));
            f[i][j].y = fmaf(r[i].y, c[j].x, fmaf(-r[i].x, c[j].y, f[i][j].y));
          }
      }
      __syncthreads();
    }
    for (int i = 0; i < 2; ++i)
      for (int j = 0; j < 2; ++j) {
        const uint64_t r = r0 + 2 * ty + i, c = c0 + 2 * tx + j;
        if (r < N && c < N) rho[r * N + c] = f[i][j];
        Tm[2 * tx + j][2 * ty + i] = conj_v(f[i][j]);
      }
    if (mirror) rho_mirror<V2>(Tm, rho, N, r0, c0);
  } else {
  ffc acc[2][2];
  rho_tile_c128<false>(psi, N, B, P, r0, c0, Ar, Ac, acc, nullptr);
  for (int i = 0; i < 2; ++i)
    for (int j = 0; j < 2; ++j) {
      const uint64_t r = r0 + 2 * ty + i, c = c0 + 2 * tx + j;
      const V2 v = ffc_to_v2<V2>(acc[i][j]);
      if (r < N && c < N) rho[r * N + c] = v;
      Tm[2 * tx + j][2 * ty + i] = conj_v(v);
    }
  if (mirror) rho_mirror<V2>(Tm, rho, N, r0, c0);
  }
}

#define RHO_FEW 96

// Entries of the digit products (rho_tc128.cu) that double-float products give
// better, replaced by those; a CTA (or four, or sixteen, for few blocks) per
// 128 x 128 block on or above the diagonal (the lower triangle gets the
// conjugates).
//
// The digits' error is about 2^-52.3 sqrt(2 B) of the product of the rows'
// scales 2^(E - 1023), that of the double-float products 2^-47.6 of the terms'
// own sizes (both from sums of random rows against exact ones) and 2^-98 a
// factor.  So an entry is replaced if its terms come to less than
// sqrt(2 B) / 26 of the scales' product, and of that by its terms' sizes, summed
// in FP32.  More than RHO_EXACT states: the sums are formed only for 32 x 32 tiles
// that may hold such an entry.  A state that is at least a quarter (an eighth) of
// the scale in both rows has a term of 1/16 (1/64) of it or more, so K16 =
// ceil(16 sqrt(2 B) / 26) (K64 likewise) of those rule an entry out; so does one
// state of the full scale in one row and half of it in the other (sqrt(2 B) / 26
// is below 1/2), and having no state in common, which makes the entry exactly
// zero.  Two rows of c1 and c2 such states share at least c1 + c2 - B: for some
// thirty states and more of an ordinary ensemble the block's smallest counts
// decide without a look at its pairs.
// A tile with few entries to replace takes them one by one (a warp an entry, two
// states a lane), one with more is formed whole as k_rho does.
// The call without and with it, 13 qubits: ordinary batches of 64 states 830 ->
// 837 us, of 2 states 410 -> 445 (no entry is replaced, bound by the sums); 64
// Grover runs that noise strikes at different steps 830 -> 905 us, of 14 qubits
// 3.17 -> 3.36 ms (a few rows dominated by one run, 0.001% replaced); states
// that are each large on amplitudes of their own and 1e-9 elsewhere 6.4 ms, two
// of them 0.98 (every tile whole; k_rho alone 4.64 ms).
__global__ void __launch_bounds__(256) k_rho_fix(const double2* __restrict__ psi, uint64_t N, int B,
                                                 const double* __restrict__ P, const int16_t* __restrict__ E,
                                                 const void* __restrict__ rows, int K16, int K64, float lim,
                                                 const unsigned char* __restrict__ redo, double2* __restrict__ rho) {
  // the upper triangle's blocks column by column: column J's rows are 0 .. J
  int J = (int)(0.5f * (sqrtf(8.f * (float)blockIdx.x + 1.f) - 1.f));
  while ((J + 1) * (J + 2) / 2 <= (int)blockIdx.x) ++J;
  while (J * (J + 1) / 2 > (int)blockIdx.x) --J;
  const int I = (int)blockIdx.x - J * (J + 1) / 2;
  // |re| + |im| of sqrt(P_a) C_a, of the row's scale: all 128 + 128 rows (up to RHO_EXACT states) or a
  // tile's 32 + 32; padded rows, whose 16-byte loads hit every bank
  constexpr int W16 = RHO_EXACT + 4, W64 = 64 + 4;
  __shared__ union {
    float all[2][128][W16];
    struct {
      RhoBig mask[2][128];
      union {
        float size[2][32][W64];
        ffc op[2][RHO_KC][RHO_TILE];
      } t;
    } m;
    struct {
      float all[2][128][W16];
      ffc op[2][RHO_KC][RHO_TILE];
    } x;
  } S;
  __shared__ float scale[2][128];  // of the rows; 0: none of its entries is replaced
  __shared__ float wt[64];
  __shared__ int least[2], listed;
  __shared__ uint16_t list[RHO_FEW];  // entries of a tile: row << 5 | column
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, tx = tid & 15, ty = tid >> 4;
  const bool redo_all = redo[I * (int)((N + 127) / 128) + J] != 0, exact = B <= RHO_EXACT;
  const int nh = (B + 3) / 4;
  const uint64_t R0 = (uint64_t)I * 128, C0 = (uint64_t)J * 128;
  const int side = tid >> 7, x = tid & 127;
  const uint64_t row = (side ? C0 : R0) + x;
  scale[side][x] = rho_scale(E[row]);
  if (tid < 64) wt[tid] = tid < B ? sqrtf((float)P[tid]) : 0.f;
  if (tid < 2) least[tid] = 64;
  __syncthreads();
  // the sizes of a row (index i of the block's, side s), states 4 h .. 4 h + 3, from the amplitudes
  auto sizes = [&](int s, int i, int h, float* to) {
    const float sc = scale[s][i], inv = sc > 0.f ? 1.f / sc : 0.f;
    const uint64_t at = (s ? C0 : R0) + i;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int a = 4 * h + k;
      double2 v = make_double2(0.0, 0.0);
      if (a < B && at < N) v = psi[(uint64_t)a * N + at];
      to[k] = (mag_f(v.x) + mag_f(v.y)) * (wt[a] * inv);
    }
  };
  if (exact) {
    const float4* mine = reinterpret_cast<const float4*>(rows) + row * (RHO_EXACT / 4);
#pragma unroll
    for (int h = 0; h < RHO_EXACT / 4; ++h)
      if (h < nh) *reinterpret_cast<float4*>(&S.all[side][x][4 * h]) = mine[h];
  } else {
    const RhoBig mine = reinterpret_cast<const RhoBig*>(rows)[row];
    S.m.mask[side][x] = mine;
    const int cnt = __reduce_min_sync(0xffffffffu, mine.any ? __popcll(mine.eighth) : 64);
    if (lane == 0) atomicMin(&least[side], cnt);
  }
  __syncthreads();
  if (!exact && !redo_all && least[0] + least[1] - B >= K64) return;
  ffc(*op)[RHO_KC][RHO_TILE] = exact ? S.x.op : S.m.t.op;
  auto put = [&](uint64_t r, uint64_t c, const ffc& z) {
    // joined in FP64: such an entry may be below 2^-75, where ff_to_d keeps 24 bits
    const double2 v = make_double2((double)z.re.hi + (double)z.re.lo, (double)z.im.hi + (double)z.im.lo);
    rho[r * N + c] = r < c || !isfinite(v.x) ? v : make_double2(v.x, 0.0);
    if (r < c) rho[c * N + r] = make_double2(v.x, -v.y);
  };
  auto smaller = [&](float size, int r, int c) {  // size: of the scales' product
    const float er = scale[0][r], ec = scale[1][c];
    return fmaf(0x1p-48f, er + ec, size * er * ec) < lim * er * ec;
  };
  // of this thread's entries (rl + warp + 8 q, cl + lane) of a tile, those to replace: bit q
  auto small = [&](int rl, int cl) {
    float z[4] = {0.f, 0.f, 0.f, 0.f};
    const float* pr = exact ? S.all[0][rl + warp] : S.m.t.size[0][warp];
    const float* pc = exact ? S.all[1][cl + lane] : S.m.t.size[1][lane];
    const int ld = exact ? W16 : W64;
#pragma unroll 4
    for (int h = 0; h < nh; ++h) {
      const float4 y = *reinterpret_cast<const float4*>(pc + 4 * h);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 w = *reinterpret_cast<const float4*>(pr + 8 * q * ld + 4 * h);
        z[q] = fmaf(w.x, y.x, fmaf(w.y, y.y, fmaf(w.z, y.z, fmaf(w.w, y.w, z[q]))));
      }
    }
    unsigned mine = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = rl + warp + 8 * q, c = cl + lane;
      mine |= (unsigned)(z[q] > 0.f && R0 + r < C0 + c && smaller(z[q], r, c)) << q;
    }
    return mine;
  };
  if (exact && !redo_all) {  // most blocks have none: one barrier for all of a block's tiles
    unsigned any = 0;
    for (int t = blockIdx.y; t < 16; t += gridDim.y) any |= small(32 * (t >> 2), 32 * (t & 3));
    if (!__syncthreads_or(any)) return;
  }
  for (int t = blockIdx.y; t < 16; t += gridDim.y) {
    const int rl = 32 * (t >> 2), cl = 32 * (t & 3);
    const uint64_t r0 = R0 + rl, c0 = C0 + cl;
    if (r0 > c0 || c0 >= N) continue;
    int n = 1024;  // entries to replace
    if (!redo_all) {
      if (!exact) {  // does the tile need its sizes?
        bool hit = false;
        const RhoBig b = S.m.mask[1][cl + lane];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const RhoBig a = S.m.mask[0][rl + warp + 8 * q];
          hit |= (a.any & b.any) && !((a.full & b.half) | (a.half & b.full)) &&
                 __popcll(a.quarter & b.quarter) < K16 && __popcll(a.eighth & b.eighth) < K64 &&
                 r0 + warp + 8 * q < c0 + lane;
        }
        if (!__syncthreads_or(hit)) continue;
        for (int i = tid; i < 64 * nh; i += blockDim.x)
          sizes((i >> 5) & 1, ((i >> 5) & 1 ? cl : rl) + (i & 31), i >> 6, &S.m.t.size[(i >> 5) & 1][i & 31][4 * (i >> 6)]);
        __syncthreads();
      }
      unsigned mine = small(rl, cl);
      if (tid == 0) listed = 0;
      if (!__syncthreads_or(mine)) continue;
      for (; mine; mine &= mine - 1) {
        const int at = atomicAdd(&listed, 1);
        if (at < RHO_FEW) list[at] = (uint16_t)((warp + 8 * (__ffs(mine) - 1)) << 5 | lane);
      }
      __syncthreads();
      n = listed;
    }
    if (n <= RHO_FEW) {
      for (int i = warp; i < n; i += 8) {
        const uint64_t r = r0 + (list[i] >> 5), c = c0 + (list[i] & 31);
        ffc z = ffc_make(ff_make(0.f, 0.f), ff_make(0.f, 0.f));
        for (int a = lane; a < B; a += 32) {
          const ff w = ff_from_d(P[a]);
          const ffc u = load_ffc(psi, (uint64_t)a * N + r);
          mac_conj_b(z, ffc_make(ff_mul(u.re, w), ff_mul(u.im, w)), load_ffc(psi, (uint64_t)a * N + c));
        }
        for (int o = 16; o; o >>= 1)
          z = ffc_add(z, ffc_make(ff_make(__shfl_xor_sync(0xffffffffu, z.re.hi, o), __shfl_xor_sync(0xffffffffu, z.re.lo, o)),
                                  ff_make(__shfl_xor_sync(0xffffffffu, z.im.hi, o), __shfl_xor_sync(0xffffffffu, z.im.lo, o))));
        if (lane == 0) put(r, c, z);
      }
    } else {
      ffc acc[2][2];
      float size[2][2];
      rho_tile_c128<true>(psi, N, B, P, r0, c0, op[0], op[1], acc, size);
      for (int i = 0; i < 2; ++i)
        for (int j = 0; j < 2; ++j) {
          const int rr = 2 * ty + i, cc = 2 * tx + j;
          const uint64_t r = r0 + rr, c = c0 + cc;
          if (r > c || c >= N) continue;
          const float er = scale[0][rl + rr], ec = scale[1][cl + cc];
          if (redo_all || (r < c && fmaf(0x1p-48f, er + ec, size[i][j]) < lim * er * ec)) put(r, c, acc[i][j]);
        }
    }
    __syncthreads();  // listed and list are read
  }
}
int launch_rho_fix(const double2* psi, int n, int B, const double* P, const int16_t* E, const void* rows,
                   const unsigned char* redo, double2* rho, cudaStream_t s) {
  const unsigned nb = (unsigned)(((1ull << n) + 127) / 128);
  const double unit = std::sqrt(2.0 * B) / 26.0;
  // sizes are sums of |re| + |im| of both factors: twice the terms' moduli at most
  k_rho_fix<<<dim3(nb * (nb + 1) / 2, nb <= 8 ? 16 : nb <= 16 ? 4 : 1), 256, 0, s>>>(
      psi, 1ull << n, B, P, E, rows, (int)std::ceil(16.0 * unit), (int)std::ceil(64.0 * unit), (float)(2.0 * unit), redo,
      rho);
  return 1;
}

// ------------------------------------------------------------ Gram -------
#define GRAM_K 32

// Partial Gram sums over one slice of the amplitude axis per CTA:
// part[blk][a][b] = sum_n conj(C_a(n)) C_b(n) (float pairs: re hi, re lo,
// im hi, im lo).  Thread t owns the 4 x 4 block a = 4 (t/16).., b = 4 (t%16)..
template <typename V2>
__global__ void __launch_bounds__(256) k_gram(const V2* __restrict__ psi, uint64_t N, int B, uint64_t per_blk,
                                              float4* __restrict__ part) {
  __shared__ ffc X[QC_SPECTRUM_MAX_UNIVERSES][GRAM_K];
  const int ta = (threadIdx.x >> 4) * 4, tb = (threadIdx.x & 15) * 4;
  ffc acc[4][4];
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < 4; ++j) acc[i][j] = ffc_make(ff_make(0.f, 0.f), ff_make(0.f, 0.f));
  const uint64_t lo = (uint64_t)blockIdx.x * per_blk, hi = min(N, lo + per_blk);
  for (uint64_t k0 = lo; k0 < hi; k0 += GRAM_K) {
    for (int e = threadIdx.x; e < B * GRAM_K; e += blockDim.x) {
      const int a = e / GRAM_K, x = e % GRAM_K;
      X[a][x] = (k0 + x < hi) ? load_ffc(psi, (uint64_t)a * N + k0 + x)
                              : ffc_make(ff_make(0.f, 0.f), ff_make(0.f, 0.f));
    }
    __syncthreads();
    if (std::is_same<V2, float2>::value && ta < B && tb < B) {
      // complex64: exact-enough FP32 sums over the 32 amplitudes of a tile,
      // added into the float pairs once per tile
      float2 f[4][4];
      for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) f[i][j] = make_float2(0.f, 0.f);
      for (int x = 0; x < GRAM_K; ++x) {
        float2 va[4], vb[4];
        for (int i = 0; i < 4; ++i) {
          va[i] = (ta + i < B) ? make_float2(X[ta + i][x].re.hi, X[ta + i][x].im.hi) : make_float2(0.f, 0.f);
          vb[i] = (tb + i < B) ? make_float2(X[tb + i][x].re.hi, X[tb + i][x].im.hi) : make_float2(0.f, 0.f);
        }
        for (int i = 0; i < 4; ++i)
          for (int j = 0; j < 4; ++j) {  // conj(C_a) C_b
            f[i][j].x = fmaf(va[i].x, vb[j].x, fmaf(va[i].y, vb[j].y, f[i][j].x));
            f[i][j].y = fmaf(va[i].x, vb[j].y, fmaf(-va[i].y, vb[j].x, f[i][j].y));
          }
      }
      for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) {
          acc[i][j].re = ff_add(acc[i][j].re, ff_make(f[i][j].x, 0.f));
          acc[i][j].im = ff_add(acc[i][j].im, ff_make(f[i][j].y, 0.f));
        }
    } else if (ta < B && tb < B) {
      for (int x = 0; x < GRAM_K; ++x) {
        ffc va[4], vb[4];
        for (int i = 0; i < 4; ++i) {
          va[i] = (ta + i < B) ? X[ta + i][x] : ffc_make(ff_make(0.f, 0.f), ff_make(0.f, 0.f));
          vb[i] = (tb + i < B) ? X[tb + i][x] : ffc_make(ff_make(0.f, 0.f), ff_make(0.f, 0.f));
        }
        // conj(C_a) C_b = C_b conj(C_a)
        for (int i = 0; i < 4; ++i)
          for (int j = 0; j < 4; ++j) mac_conj_b(acc[i][j], vb[j], va[i]);
      }
    }
    __syncthreads();
  }
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < 4; ++j) {
      const int a = ta + i, b = tb + j;
      if (a < B && b < B)
        part[((uint64_t)blockIdx.x * B + a) * B + b] =
            make_float4(acc[i][j].re.hi, acc[i][j].re.lo, acc[i][j].im.hi, acc[i][j].im.lo);
    }
}

// G[a][b] = sqrt(P_a P_b) * sum over blocks: 32 entries a block of 256
// threads, eight threads an entry (each every eighth block's partial, their
// sums added in order; one thread an entry was a chain of 304 additions,
// 57 us).  G is made exactly Hermitian: the entries with a > b are the
// conjugates of their mirrors and the diagonal is real (the two triangles'
// separately rounded sums differ by ~1e-14; the solver assumes a Hermitian G).
__global__ void __launch_bounds__(256) k_gram_final(const float4* __restrict__ part, int nblk, int B,
                                                    const double* __restrict__ sqrtP, double2* __restrict__ G) {
  __shared__ ffc sh[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + lane;
  ffc z = ffc_make(ff_make(0.f, 0.f), ff_make(0.f, 0.f));
  const int a = e / B, b = e % B;
  if (e < B * B) {
    const int u = min(a, b) * B + max(a, b);  // the upper-triangle entry
    for (int k = w; k < nblk; k += 8) {
      const float4 v = part[(uint64_t)k * B * B + u];
      z = ffc_add(z, ffc_make(ff_make(v.x, v.y), ff_make(v.z, v.w)));
    }
  }
  sh[w][lane] = z;
  __syncthreads();
  if (w || e >= B * B) return;
  for (int k = 1; k < 8; ++k) z = ffc_add(z, sh[k][lane]);
  if (!isfinite(z.re.hi) || !isfinite(z.im.hi)) {  // kept non-finite (the join would not)
    G[e] = make_double2(NAN, NAN);
    return;
  }
  const double wt = sqrtP[a] * sqrtP[b];
  const double gi = (a == b) ? 0.0 : ff_to_d(z.im) * wt;
  G[e] = make_double2(ff_to_d(z.re) * wt, a > b ? -gi : gi);
}

// ------------------------------------------------------- eigenvalues ----
// Eigenvalues of the Hermitian B x B matrix G (FP64, B <= 64):
//  1. k_tridiag: Householder reduction to a real symmetric tridiagonal matrix.
//     Step k reflects x = A[k+1.., k] onto alpha e_1 with
//     alpha = -(x_0/|x_0|) |x| (no cancellation in v = x - alpha e_1):
//     tau = 2 / |v|^2 = 1 / (|x| (|x| + |x_0|)), p = tau A22 v,
//     q = p - (tau/2) (v^H p) v, A22 -= v q^H + q v^H.  The off-diagonal
//     entries' phases are removed by a diagonal unitary similarity, so T has
//     diagonal Re A_kk and off-diagonal |x|.
//  2. k_sturm: each eigenvalue by 129-section on Sturm counts of T, one CTA
//     (and SM) an eigenvalue, from the Gershgorin interval down to a width of
//     2^-52 of its magnitude.
// One SM's FP64 pipe completes under two operations a clock, a warp's
// operation takes its quarter of the pipe about 70 clocks, and roots and
// quotients are ten operations each: one CTA whose threads all repeated the
// step's scalars took 2.92 ms for 64 x 64.  The rows are spread over a cluster
// of eight CTAs (16 threads a row, the row in registers, all four quarters
// busy), x and p go to every CTA through distributed shared memory, one warp
// takes the step's scalars (both roots at once, in two lanes), and the counts
// need no division and run 128 points at a time.
constexpr int EIG_CTAS = 8;

__device__ __forceinline__ double warp_add(double x) {
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// de: d[0..64), then e2[0..64) (squared off-diagonal)
__global__ void __cluster_dims__(EIG_CTAS, 1, 1) __launch_bounds__(128) k_tridiag(const double2* __restrict__ G, int B,
                                                                               double* __restrict__ de) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  __shared__ double2 sx[2][64], sp[64], sv[64], sq[64];
  __shared__ double sc[2];  // tau, |x|^2
  const int rank = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, row = tid >> 4, sub = tid & 15;
  const int i = row * EIG_CTAS + rank;  // this thread's matrix row; its columns are sub, sub + 16, ..
  double2 A[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int c = sub + 16 * j;
    A[j] = i < B && c < B ? G[i * B + c] : make_double2(0.0, 0.0);
  }
  cl.sync();  // every CTA runs before another writes its shared memory
  for (int k = 0; k + 2 < B; ++k) {
    const int o = k + 1;
    double2* x = sx[k & 1];
    // column k: each row's element to every CTA
    if (sub == (k & 15) && i < B) {
      double2 a = A[0];
#pragma unroll
      for (int j = 1; j < 4; ++j)
        if (j == (k >> 4)) a = A[j];
      if (i == k) de[k] = a.x;
      if (i >= o)
        for (int r = 0; r < EIG_CTAS; ++r) cl.map_shared_rank(x, r)[i] = a;
    }
    cl.sync();
    if (tid < 32) {
      const double2 z = make_double2(0.0, 0.0);
      const double2 xa = lane >= o && lane < B ? x[lane] : z, xb = lane + 32 >= o && lane + 32 < B ? x[lane + 32] : z;
      double s = fma(xa.x, xa.x, fma(xa.y, xa.y, fma(xb.x, xb.x, xb.y * xb.y)));
      const double2 x0 = x[o];
      const double sigma = warp_add(s), a02 = fma(x0.x, x0.x, x0.y * x0.y);
      // lane 0: |x|, other lanes: |x_0|, each with its reciprocal
      const double w = lane == 0 ? sigma : a02, r = w > 0.0 ? rsqrt(w) : 0.0, m = w * r;
      const double nx = __shfl_sync(0xffffffffu, m, 0), rx = __shfl_sync(0xffffffffu, r, 0);
      const double a0 = __shfl_sync(0xffffffffu, m, 1), ra = __shfl_sync(0xffffffffu, r, 1);
      // v_0 = x_0 - alpha = x_0 (1 + |x|/|x_0|), or |x| for x_0 = 0
      const double g = fma(nx, ra, 1.0);
      const double2 v0 = a0 > 0.0 ? make_double2(x0.x * g, x0.y * g) : make_double2(nx, 0.0);
      sv[lane] = lane == o ? v0 : xa;
      sv[lane + 32] = lane + 32 == o ? v0 : xb;
      if (lane == 0) {
        sc[0] = nx > 0.0 ? rx / (nx + a0) : 0.0;
        sc[1] = sigma;
        if (rank == 0) de[64 + k] = sigma;
      }
    }
    __syncthreads();
    if (!(sc[1] > 0.0)) continue;  // nothing below the diagonal (or not finite: reported by k_sturm); the same in every CTA
    const double tau = sc[0];
    // p = tau A v: the row's sixteen threads
    double pr = 0.0, pi = 0.0;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (16 * j + 15 >= o) {
        const double2 v = sv[sub + 16 * j];
        pr = fma(A[j].x, v.x, fma(-A[j].y, v.y, pr));
        pi = fma(A[j].x, v.y, fma(A[j].y, v.x, pi));
      }
    {  // half the lanes go on with the real parts, half with the imaginary ones
      const double give = (sub & 8) ? pr : pi, keep = (sub & 8) ? pi : pr;
      double t = keep + __shfl_xor_sync(0xffffffffu, give, 8);
      for (int q = 1; q < 8; q <<= 1) t += __shfl_xor_sync(0xffffffffu, t, q);
      t *= tau;
      const double u = __shfl_xor_sync(0xffffffffu, t, 8);
      if (sub < EIG_CTAS && i >= o && i < B)  // thread `sub` writes to CTA `sub`
        cl.map_shared_rank(sp, sub)[i] = make_double2(t, u);
    }
    cl.sync();
    if (tid < 64) {  // two warps: both form K, each its half of q
      double s = 0.0;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h;
        if (c >= o && c < B) s = fma(sv[c].x, sp[c].x, fma(sv[c].y, sp[c].y, s));
      }
      const double K = 0.5 * tau * warp_add(s);
      if (tid >= o && tid < B) sq[tid] = make_double2(fma(-K, sv[tid].x, sp[tid].x), fma(-K, sv[tid].y, sp[tid].y));
    }
    __syncthreads();
    if (i >= o && i < B) {
      const double2 vi = sv[i], qi = sq[i];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = sub + 16 * j;
        if (c >= o && c < B) {
          const double2 v = sv[c], q = sq[c];
          A[j].x = fma(-vi.x, q.x, fma(-vi.y, q.y, fma(-qi.x, v.x, fma(-qi.y, v.y, A[j].x))));
          A[j].y = fma(-vi.y, q.x, fma(vi.x, q.y, fma(-qi.y, v.x, fma(qi.x, v.y, A[j].y))));
        }
      }
    }
    __syncthreads();  // sv, sq are read before the next step's
  }
  // the last two diagonal elements and the last off-diagonal one
  if (i < B) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = sub + 16 * j;
      if (c == i && i + 2 >= B) de[i] = A[j].x;
      if (c + 1 == i && i + 1 == B) de[64 + c] = fma(A[j].x, A[j].x, A[j].y * A[j].y);
    }
  }
  cl.sync();  // no CTA leaves while its shared memory may be written
}

// Number of eigenvalues below x of T (d, squared off-diagonal e2, scaled to
// |d|, |e| <= 1): sign changes of the leading minors
// p_i = (d_i - x) p_{i-1} - e2_{i-1} p_{i-2}.  They grow by at most three a
// step; a pair that has shrunk below 2^-300 is scaled up (in the exponent
// fields: no FP64 operation, no branch), a zero counts as the sign opposite to
// its predecessor's (a pivot of -0).
__device__ __forceinline__ int sturm_count(const double* d, const double* e2, int B, double x) {
  double pm = 1.0, p = d[0] - x;
  if (p == 0.0) p = -0x1p-250;
  int cnt = __double2hiint(p) < 0;
#pragma unroll 4
  for (int i = 1; i < B; ++i) {
    double t = fma(d[i] - x, p, -(e2[i - 1] * pm));
    const int hp = __double2hiint(p);
    int ht = __double2hiint(t);
    if (((ht << 1) | __double2loint(t)) == 0) ht = (hp ^ (int)0x80000000) - (250 << 20);  // -p 2^-250, about
    const int up = max(ht & 0x7fffffff, hp & 0x7fffffff) < (1023 - 300) << 20 ? 300 << 20 : 0;
    cnt += (ht ^ hp) < 0;
    pm = __hiloint2double(hp + up, __double2loint(p));
    p = __hiloint2double(ht + up, __double2loint(t));
  }
  return cnt;
}

// Eigenvalue blockIdx.x (ascending) of T, to ev[B - 1 - blockIdx.x];
// ev[B] = 1 where T has a non-finite entry.
__global__ void __launch_bounds__(128) k_sturm(const double* __restrict__ de, int B, double* __restrict__ ev) {
  __shared__ double d[64], e2[64];
  const int tid = threadIdx.x, lane = tid & 31, idx = blockIdx.x;
  double lo = INFINITY, hi = -INFINITY;
  bool finite = true;
#pragma unroll
  for (int h = 0; h < 2; ++h) {  // every warp for itself
    const int i = lane + 32 * h;
    if (i >= B) continue;
    const double di = de[i], el = i > 0 ? de[63 + i] : 0.0, er = i + 1 < B ? de[64 + i] : 0.0;
    finite = finite && isfinite(di) && isfinite(er);
    const double r = sqrt(el) + sqrt(er);
    lo = fmin(lo, di - r);
    hi = fmax(hi, di + r);
  }
  finite = __all_sync(0xffffffffu, finite);
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if (idx == 0 && tid == 0) ev[B] = finite ? 0.0 : 1.0;
  const double span = fmax(fabs(lo), fabs(hi));
  if (!finite || !(span > 0.0)) {
    if (tid == 0) ev[B - 1 - idx] = finite ? 0.0 : NAN;
    return;
  }
  // scaled by a power of two to a span in [1, 2)
  const int k = -ilogb(span);
  if (tid < B) {
    d[tid] = ldexp(de[tid], k);
    e2[tid] = tid + 1 < B ? ldexp(ldexp(de[64 + tid], k), k) : 0.0;
  }
  double a = ldexp(lo, k) - 4.5e-16, b = ldexp(hi, k) + 4.5e-16;
  const double s1 = ldexp(span, k);
  __syncthreads();
  for (int it = 0; it < 100 && b - a > 2.2e-16 * fmax(fabs(a), fabs(b)) + 1e-19 * s1; ++it) {
    const double w = b - a, a1 = a;
    const int f = __syncthreads_count(sturm_count(d, e2, B, fma(w, (tid + 1) * (1.0 / 129.0), a1)) <= idx);
    if (f > 0) a = fma(w, f * (1.0 / 129.0), a1);           // the last point not above the eigenvalue
    if (f < 128) b = fma(w, (f + 1) * (1.0 / 129.0), a1);   // the first one above it
  }
  if (tid == 0) ev[B - 1 - idx] = ldexp(0.5 * (a + b), -k);
}

}  // namespace qc

using namespace qc;

// ------------------------------------------------------------- host ------
QC_API qc_status qc_wigner_d(int twoj, double alpha, double beta, double gamma, double* D_out) {
  clear_error();
  if (!D_out || (twoj != 1 && twoj != 3) || !std::isfinite(alpha) || !std::isfinite(beta) || !std::isfinite(gamma)) {
    set_error("qc_wigner_d: twoj must be 1 or 3, angles finite, output non-NULL");
    return QC_EINVAL;
  }
  const double c = cos(0.5 * beta), s = sin(0.5 * beta);
  const int dim = twoj + 1;
  double d[16];
  if (twoj == 1) {  // d^{1/2}(beta), m = +1/2, -1/2
    const double t[4] = {c, -s, s, c};
    for (int i = 0; i < 4; ++i) d[i] = t[i];
  } else {  // d^{3/2}(beta), m = 3/2, 1/2, -1/2, -3/2
    const double r3 = sqrt(3.0);
    const double t[16] = {c * c * c,       -r3 * c * c * s,           r3 * c * s * s,            -s * s * s,
                          r3 * c * c * s,  c * (c * c - 2.0 * s * s), -s * (2.0 * c * c - s * s), r3 * c * s * s,
                          r3 * c * s * s,  s * (2.0 * c * c - s * s), c * (c * c - 2.0 * s * s), -r3 * c * c * s,
                          s * s * s,       r3 * c * s * s,            r3 * c * c * s,            c * c * c};
    for (int i = 0; i < 16; ++i) d[i] = t[i];
  }
  for (int r = 0; r < dim; ++r)
    for (int col = 0; col < dim; ++col) {
      const double mp = 0.5 * (twoj - 2 * r), m = 0.5 * (twoj - 2 * col);
      const double ph = -(mp * alpha + m * gamma);  // e^{-i m' alpha} e^{-i m gamma}
      D_out[2 * (r * dim + col)] = d[r * dim + col] * cos(ph);
      D_out[2 * (r * dim + col) + 1] = d[r * dim + col] * sin(ph);
    }
  return QC_OK;
}

static qc_status check_batch(const void* psi, int n, qc_dtype dt, int B, const double* P, int max_n, int max_b) {
  if (!psi || !P || n < 1 || n > max_n || B < 1 || B > max_b || (dt != QC_C128 && dt != QC_C64)) {
    set_error("bad batch: psi/P NULL, n = %d (1..%d), B = %d (1..%d) or dtype %d", n, max_n, B, max_b, (int)dt);
    return QC_EINVAL;
  }
  for (int a = 0; a < B; ++a)
    if (!(P[a] >= 0.0) || !std::isfinite(P[a])) {
      set_error("weight P[%d] = %g is not a finite non-negative number", a, P[a]);
      return QC_EINVAL;
    }
  return QC_OK;
}

QC_API qc_status qc_density_matrix(const void* psi_dev, int n, qc_dtype dt, int B, const double* P_host,
                                   void* rho_dev, void* stream) {
  clear_error();
  qc_status st = check_batch(psi_dev, n, dt, B, P_host, QC_DM_MAX_QUBITS, 1 << 30);
  if (st) return st;
  if (!rho_dev) {
    set_error("rho_dev is NULL");
    return QC_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  const uint64_t N = 1ull << n;
  if (dt == QC_C128 && B <= 64) {  // tensor cores (rho_tc128.cu), unless their workspace does not fit
    st = rho_tc_c128(reinterpret_cast<const double2*>(psi_dev), n, B, P_host, reinterpret_cast<double2*>(rho_dev), s);
    if (st != QC_ENOMEM) return st;
  }
  double* P = nullptr;
  cudaError_t e = ws_alloc((void**)&P, sizeof(double) * B, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(P, P_host, sizeof(double) * B, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) {
    if (P) cudaFreeAsync(P, s);
    return cuda_fail(e, "density matrix weights");
  }
  if (dt == QC_C64 && B <= 64) {  // tensor cores (rho_tc.cu)
    cudaFreeAsync(P, s);
    return rho_tc_c64(reinterpret_cast<const float2*>(psi_dev), n, B, P_host, reinterpret_cast<float2*>(rho_dev), s);
  }
  const unsigned nt = (unsigned)((N + RHO_TILE - 1) / RHO_TILE);
  const dim3 grid(nt, nt);
  if (dt == QC_C128)
    k_rho<double2><<<grid, 256, 0, s>>>(reinterpret_cast<const double2*>(psi_dev), N, B, P,
                                         reinterpret_cast<double2*>(rho_dev));
  else
    k_rho<float2><<<grid, 256, 0, s>>>(reinterpret_cast<const float2*>(psi_dev), N, B, P,
                                        reinterpret_cast<float2*>(rho_dev));
  st = check_launch("density matrix", 1);
  cudaFreeAsync(P, s);
  return st;
}

QC_API qc_status qc_mixed_spectrum(const void* psi_dev, int n, qc_dtype dt, int B, const double* P_host,
                                   double* evals_host, double* stats_host, void* stream) {
  clear_error();
  qc_status st = check_batch(psi_dev, n, dt, B, P_host, 34, QC_SPECTRUM_MAX_UNIVERSES);
  if (st) return st;
  if (!evals_host || !stats_host) {
    set_error("NULL output");
    return QC_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  const uint64_t N = 1ull << n;
  // slices of the amplitude axis: a resident grid, each slice a multiple of GRAM_K
  const int nblk = (int)std::min<uint64_t>((N + GRAM_K - 1) / GRAM_K, (uint64_t)sm_count() * 2);
  uint64_t per = (N + nblk - 1) / nblk;
  per = (per + GRAM_K - 1) / GRAM_K * GRAM_K;
  const size_t part_b = sizeof(float4) * (size_t)nblk * B * B;
  const size_t g_b = sizeof(double2) * B * B;
  const size_t small_b = sizeof(double) * (2 * B + 1 + 128);
  char* buf = nullptr;
  cudaError_t e = ws_alloc((void**)&buf, part_b + g_b + small_b + 64, s);
  if (e != cudaSuccess) return cuda_fail(e, "spectrum workspace");
  float4* part = reinterpret_cast<float4*>(buf);
  double2* G = reinterpret_cast<double2*>(buf + part_b);
  double* sqrtP = reinterpret_cast<double*>(buf + part_b + g_b);
  double* ev = sqrtP + B;       // B eigenvalues and the flag
  double* de = ev + B + 1;      // the tridiagonal matrix
  std::vector<double> sq(B);
  for (int a = 0; a < B; ++a) sq[a] = sqrt(P_host[a]);
  e = cudaMemcpyAsync(sqrtP, sq.data(), sizeof(double) * B, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) {
    cudaFreeAsync(buf, s);
    return cuda_fail(e, "spectrum weights");
  }
  if (dt == QC_C128)
    k_gram<double2><<<nblk, 256, 0, s>>>(reinterpret_cast<const double2*>(psi_dev), N, B, per, part);
  else
    k_gram<float2><<<nblk, 256, 0, s>>>(reinterpret_cast<const float2*>(psi_dev), N, B, per, part);
  k_gram_final<<<(B * B + 31) / 32, 256, 0, s>>>(part, nblk, B, sqrtP, G);
  k_tridiag<<<EIG_CTAS, 128, 0, s>>>(G, B, de);
  k_sturm<<<B, 128, 0, s>>>(de, B, ev);
  st = check_launch("mixed spectrum", 4);
  if (!st) {
    std::vector<double> out(B + 1);
    e = cudaMemcpyAsync(out.data(), ev, sizeof(double) * (B + 1), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
      st = cuda_fail(e, "spectrum readback");
    } else {
      double tr = 0.0, p2 = 0.0, sl = 0.0;
      for (int i = 0; i < B; ++i) {
        const double l = out[i];
        evals_host[i] = l;
        tr += l;
        p2 += l * l;
        if (l > 1e-14) sl -= l * log(l);
      }
      stats_host[0] = tr;
      stats_host[1] = p2;
      stats_host[2] = sl;
      if (out[B] != 0.0) {
        set_error("mixed spectrum: the Gram matrix has a non-finite entry");
        st = QC_ECUDA;
      }
    }
  }
  cudaFreeAsync(buf, s);
  return st;
}
