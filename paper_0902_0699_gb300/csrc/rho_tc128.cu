// The ensemble density matrix of complex128 states (sec. 6.1) on the tensor
// cores: rho_tc.cu's real GEMM (rows A_i of K = 2B reals, columns Bre_j and
// Bim_j interleaved) with exact integer digits.
//
// Every amplitude index's row (its B states' sqrt(P_a) C_a) is scaled to 55-bit
// integers by the row's largest exponent and cut into seven balanced base-256
// digits (of magnitude up to 128), which bf16 holds exactly (the splitting of Ozaki, Ogita, Oishi and
// Rump, Numer. Algorithms 59, 2012).  The 28 digit products of weight 2^-8u,
// u = s + t <= 6, go to seven FP32 accumulators; a product is below 2^14, an
// accumulator sums at most 7 x 128 of them, so every sum is an exact integer
// below 2^24 and nothing is rounded until the seven are joined in 64-bit
// integers and converted to binary64 once.
//
// What is dropped (u > 6) is a fraction of the product of the two rows' scales
// (powers of two up to their largest magnitudes), about 2^-52.3 sqrt(2 B) of it.
// The double-float products of the CUDA cores (k_rho; bound at about 13 FP32
// operations a real product: 4.64 ms for 13 qubits and 64 states) are good to
// about 2^-47.6 of the terms' own sizes.  Where many states are large in both
// rows, as in an ensemble around a common state, the digits are the better
// ones; where the rows are dominated by different states (universes near
// different basis states), the others, and k_rho_fix (density.cu) replaces them.
//
// One CTA per SM works through 128 x 32 tiles on and above the block diagonal
// (off-diagonal tiles are also written mirrored).  K goes in chunks of 16: one
// MMA per digit product and chunk, 42 KiB of operands already in canonical
// layout by two bulk copies into one of four stages, three of which load while
// one is multiplied.  Seven accumulators of 64 columns take 448 of the 512
// tensor-memory columns.  One warp loads, multiplies and waits; sixteen join
// the accumulators, hand the tensor memory back (named barriers) and convert
// and store while the next tile is multiplied.  Only one thread polls an
// mbarrier: with all threads of the CTA polling for a tile's end, an MMA took
// 248 clocks instead of 57 and a bulk copy three times as long (13 qubits, 64
// states: 1.95 ms; one poller and the epilogue beside the next tile 0.79 ms,
// 1.36 TB/s of rho written).
//
// The call is stream-ordered: there is no status word.  A tile whose bounded
// wait gives up (it never has) is left to k_rho_fix, with all later ones of its
// CTA.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"
#include "fixpt.cuh"
#include "tc5.cuh"

namespace qc {

#define R8_EW 16               // epilogue warps
#define R8_T (32 * R8_EW + 32)  // and the warp that loads and multiplies
#define R8_ND 7                  // digits
#define R8_A (TC5_M * 16 * 2)    // one digit of a 128-row chunk (K = 16)
#define R8_B (TC5_N * 16 * 2)
#define R8_STAGE (R8_ND * (R8_A + R8_B))
#define R8_NST 4
#define R8_STG (R8_EW * 32 * 5 * 16)  // epilogue: each warp's 32 rows of 4 entries, padded
#define R8_SMEM (R8_NST * R8_STAGE + R8_STG + 128)
#define R8_SPIN (1u << 20)

struct Rho8Dims {
  uint64_t N;
  int B, nkc, nib, njb;  // states, K chunks of 16, 128-row blocks, 32-column blocks
};

// byte offset of (row r, k < 16) in a digit's chunk
__device__ __forceinline__ uint32_t r8_off(int r, int k8) { return (uint32_t)((r >> 3) * 256 + k8 * 128 + (r & 7) * 16); }

__device__ __forceinline__ uint64_t r8_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(256 >> 4) << 32) | (1ull << 46);
}

// One block per 32 amplitude indices: their reals through shared memory, each
// index's largest exponent, then 8 reals (one 16-byte core-matrix row per
// digit) at a time: A's row, Bre's and Bim's.  Also each row's record for
// k_rho_fix; clears redo.
__global__ void __launch_bounds__(256) k_rho8_digits(const double2* __restrict__ psi, const double* __restrict__ sqrtP,
                                                     Rho8Dims d, unsigned char* __restrict__ Aop,
                                                     unsigned char* __restrict__ Bop, int16_t* __restrict__ E,
                                                     unsigned char* __restrict__ rows, unsigned char* __restrict__ redo) {
  __shared__ double X[128][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, jb = blockIdx.x, ib = jb >> 2;
  const uint64_t i0 = (uint64_t)jb * 32;
  for (int a = w; a < d.B; a += 8) {
    double2 c = make_double2(0.0, 0.0);
    if (i0 + lane < d.N) c = psi[(uint64_t)a * d.N + i0 + lane];
    X[a][lane] = sqrtP[a] * c.x;
    X[a + d.B][lane] = sqrtP[a] * c.y;
  }
  __syncthreads();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < d.nib * d.nib; i += gridDim.x * blockDim.x) redo[i] = 0;
  for (int r = w; r < 32; r += 8) {
    int e[2];  // exponents of this lane's states
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int a = lane + 32 * h;
      e[h] = -1;  // no state, or a zero
      if (a < d.B) {
        const double x = fmax(fabs(X[a][r]), fabs(X[a + d.B][r]));
        if (!isfinite(X[a][r]) || !isfinite(X[a + d.B][r])) e[h] = 0x7FF;
        else if (x > 0.0) e[h] = (int)(__double_as_longlong(x) >> 52);
      }
    }
    const int top = __reduce_max_sync(0xffffffffu, max(e[0], e[1]));
    if (d.B <= RHO_EXACT) {
      const float sc = rho_scale(top), inv = sc > 0.f ? 1.f / sc : 0.f;
      if (lane < RHO_EXACT)
        reinterpret_cast<float*>(rows)[(i0 + r) * RHO_EXACT + lane] =
            lane < d.B ? (mag_f(X[lane][r]) + mag_f(X[lane + d.B][r])) * inv : 0.f;
      continue;
    }
    uint64_t m[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const int at = q == 4 ? 0 : max(0, top - q);
      m[q] = __ballot_sync(0xffffffffu, e[0] >= at) | (uint64_t)__ballot_sync(0xffffffffu, e[1] >= at) << 32;
      if (top == 0x7FF) m[q] = ~0ull;
    }
    if (lane == 0) reinterpret_cast<RhoBig*>(rows)[i0 + r] = RhoBig{m[0], m[1], m[2], m[3], m[4]};
  }
  const int K = 2 * d.B;
  for (int item = threadIdx.x; item < 512; item += 256) {
    const int r = item >> 4, kg = item & 15;
    double x[8];
    int em = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int k = 8 * kg + q;
      x[q] = k < K ? X[k][r] : 0.0;
      em = max(em, (int)((__double_as_longlong(x[q]) >> 52) & 0x7FF));
    }
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) em = max(em, __shfl_xor_sync(0xffffffffu, em, o));
    if (kg == 0) E[i0 + r] = (int16_t)em;
    if (kg >= 2 * d.nkc) continue;
    const int kc = kg >> 1;
    for (int form = 0; form < (jb < d.njb ? 2 : 1); ++form) {  // A and Bre, then Bim
      uint32_t out[R8_ND][4];
#pragma unroll
      for (int s = 0; s < R8_ND; ++s)
#pragma unroll
        for (int h = 0; h < 4; ++h) out[s][h] = 0;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int k = 8 * kg + q;
        double v = x[q];
        if (form) v = k >= K ? 0.0 : k < d.B ? -X[k + d.B][r] : X[k - d.B][r];
        // digits of |v|, then the sign: -v has the negated digits, and rho comes
        // out exactly Hermitian
        long long z = d2fix(fabs(v), em - 1);  // z <= 2^54
#pragma unroll
        for (int s = R8_ND - 1; s >= 0; --s) {
          const int dg = (int)(int8_t)(z & 0xff);
          z = (z - dg) >> 8;
          const __nv_bfloat16 hv = __float2bfloat16_rn(signbit(v) ? -(float)dg : (float)dg);
          out[s][q >> 1] |= (uint32_t)(*reinterpret_cast<const uint16_t*>(&hv)) << (16 * (q & 1));
        }
      }
#pragma unroll
      for (int s = 0; s < R8_ND; ++s) {
        const uint4 v = make_uint4(out[s][0], out[s][1], out[s][2], out[s][3]);
        if (form == 0)
          *reinterpret_cast<uint4*>(Aop + (((size_t)ib * d.nkc + kc) * R8_ND + s) * R8_A + r8_off((int)(i0 & 127) + r, kg & 1)) = v;
        if (jb < d.njb)
          *reinterpret_cast<uint4*>(Bop + (((size_t)jb * d.nkc + kc) * R8_ND + s) * R8_B + r8_off(2 * r + form, kg & 1)) = v;
      }
    }
  }
}

// Tiles in order of row block; row block ib has the column blocks from 4 ib.
struct R8Tile {
  int ib, jb;
  int64_t t, first;  // tile number, that of the row block's first
  __device__ void at(int64_t tile, const Rho8Dims& d) {
    t = tile;
    while (ib < d.nib && t - first >= d.njb - 4 * ib) first += d.njb - 4 * ib, ++ib;
    jb = 4 * ib + (int)(t - first);
  }
};

__global__ void __launch_bounds__(R8_T, 1) k_rho8_tc(const unsigned char* __restrict__ Aop,
                                                     const unsigned char* __restrict__ Bop,
                                                     const int16_t* __restrict__ E, Rho8Dims d, int64_t ntiles,
                                                     double2* __restrict__ rho, unsigned char* __restrict__ redo) {
  extern __shared__ __align__(1024) unsigned char rsm[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(rsm + R8_NST * R8_STAGE + R8_STG);
  __shared__ uint32_t tmem_holder;
  __shared__ int stop;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t s_base = (uint32_t)__cvta_generic_to_shared(rsm);
  // full[st]: a stage's operands are there; free[st]: the MMAs have read it; done: a tile's accumulators
  const uint32_t bar_full = (uint32_t)__cvta_generic_to_shared(bars), bar_free = bar_full + 8 * R8_NST,
                 bar_done = bar_free + 8 * R8_NST;
  if (tid == 0) {
    stop = 0;
    for (int i = 0; i < 2 * R8_NST + 1; ++i)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar_full + 8 * i));
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(
        (uint32_t)__cvta_generic_to_shared(&tmem_holder)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = tmem_holder;

  // the loading thread's next chunk, over all of this CTA's tiles
  R8Tile ld{0, 0, 0, 0}, cur{0, 0, 0, 0};
  int ld_kc = 0;
  uint32_t loaded = 0, q = 0, issued = 0;  // chunks loaded, multiplied; those whose products were issued
  ld.at(blockIdx.x, d);
  auto load = [&]() {
    if (ld.t >= ntiles) return;
    const uint32_t st = loaded % R8_NST, bar = bar_full + 8 * st, dst = s_base + st * R8_STAGE;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(R8_STAGE) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
                 "l"(Aop + ((size_t)ld.ib * d.nkc + ld_kc) * (R8_ND * R8_A)), "r"(R8_ND * R8_A), "r"(bar)
                 : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                     dst + R8_ND * R8_A),
                 "l"(Bop + ((size_t)ld.jb * d.nkc + ld_kc) * (R8_ND * R8_B)), "r"(R8_ND * R8_B), "r"(bar)
                 : "memory");
    ++loaded;
    if (++ld_kc == d.nkc) {
      ld_kc = 0;
      ld.at(ld.t + gridDim.x, d);
    }
  };
  if (warp == R8_EW) {
    // barrier 1: a tile's accumulators are complete; barrier 2: they are read
    if (lane == 0)
      for (int i = 0; i < R8_NST - 1; ++i) load();
    uint32_t ph_done = 0;
    bool ok = true;  // lane 0
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
      if (t != blockIdx.x) asm volatile("bar.sync 2, %0;\n" ::"n"(R8_T) : "memory");
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      if (lane == 0 && ok) {
        for (int kc = 0; kc < d.nkc; ++kc, ++q) {
          const uint32_t st = q % R8_NST;
          ok = tc5_mbar_wait(bar_full + 8 * st, (q / R8_NST) & 1u, R8_SPIN);
          if (!ok) break;
          const uint32_t a = s_base + st * R8_STAGE, b = a + R8_ND * R8_A;
#pragma unroll
          for (int u = 0; u < R8_ND; ++u)
#pragma unroll
            for (int s = 0; s <= u; ++s)  // digit s of A times digit u - s of B, one accumulator at a time
              tc5_mma_bf16(tmem + u * TC5_N, r8_desc(a + s * R8_A), r8_desc(b + (u - s) * R8_B),
                           kc == 0 && s == 0 ? 0u : 1u);
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                           bar_free + 8 * st)
                       : "memory");
          ++issued;
          // the chunk three ahead takes the stage of the chunk before this one
          if (q >= 1) ok = tc5_mbar_wait(bar_free + 8 * ((q - 1) % R8_NST), ((q - 1) / R8_NST) & 1u, R8_SPIN);
          if (!ok) break;
          load();
        }
        if (ok) {
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar_done)
                       : "memory");
          ok = tc5_mbar_wait(bar_done, ph_done, R8_SPIN);
          ph_done ^= 1u;
        }
        if (!ok) stop = 1;
      }
      __syncwarp();
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      asm volatile("bar.arrive 1, %0;\n" ::"n"(R8_T) : "memory");
    }
    // the last tile's arrivals at barrier 2
    asm volatile("bar.sync 2, %0;\n" ::"n"(R8_T) : "memory");
    // after a wait that gave up: what is still in flight (bounded once more)
    if (lane == 0 && !ok) {
      for (uint32_t c = q; c < loaded; ++c) tc5_mbar_wait(bar_full + 8 * (c % R8_NST), (c / R8_NST) & 1u, R8_SPIN);
      for (uint32_t c = issued >= R8_NST ? issued - R8_NST : 0; c < issued; ++c)
        tc5_mbar_wait(bar_free + 8 * (c % R8_NST), (c / R8_NST) & 1u, R8_SPIN);
    }
  } else {
    // warp w: rows 32 (w & 3) .., entries 8 (w >> 2) .. of the tile
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    const int cq = warp >> 2;
    const uint32_t lane_base = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + 16 * cq;
    double2* stg = reinterpret_cast<double2*>(rsm + R8_NST * R8_STAGE) + warp * 32 * 5;
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
      cur.at(t, d);
      const uint64_t ib0 = (uint64_t)cur.ib * TC5_M + 32 * (warp & 3), i = ib0 + lane;
      const uint64_t j0 = (uint64_t)cur.jb * 32 + 8 * cq;
      const bool mirror = cur.jb >= 4 * (cur.ib + 1);
      const int ei = E[i];
      int ej[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) ej[c] = j0 + c < d.N ? E[j0 + c] : 0;
      asm volatile("bar.sync 1, %0;\n" ::"n"(R8_T) : "memory");
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      const bool bad = *(volatile int*)&stop != 0;
      if (bad && tid == 0) redo[cur.ib * d.nib + (cur.jb >> 2)] = 1;
      // V = sum_u acc_u 2^(40 - 8u)
      long long V[16];
#pragma unroll
      for (int c = 0; c < 16; ++c) V[c] = 0;
#pragma unroll
      for (int u = 0; u < R8_ND; ++u) {
        float y[16];
        tc5_tmem_ld16(lane_base + u * TC5_N, y);
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const int z = __float2int_rn(y[c]);
          if (u < 6) V[c] += (long long)z * (1ll << (u < 6 ? 40 - 8 * u : 0));
          else V[c] += (z + 127 + (z > 0)) >> 8;  // half away from zero: conjugate entries stay conjugate
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      asm volatile("bar.arrive 2, %0;\n" ::"n"(R8_T) : "memory");
#pragma unroll
      for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int cc = 4 * h + c, F = 2096 - ei - ej[cc];
          double2 z = make_double2(fix2d(V[2 * cc], F), fix2d(V[2 * cc + 1], F));
          if (bad || ei == 0x7FF || ej[cc] == 0x7FF) z = make_double2(nan, nan);
          stg[lane * 5 + c] = z;
          if (mirror && i < d.N && j0 + cc < d.N) rho[(j0 + cc) * d.N + i] = make_double2(z.x, -z.y);
        }
        __syncwarp();
#pragma unroll
        for (int it = 0; it < 4; ++it) {  // rows of 64 bytes
          const int r = 8 * it + (lane >> 2), c = lane & 3;
          if (ib0 + r < d.N && j0 + 4 * h + c < d.N) rho[(ib0 + r) * d.N + j0 + 4 * h + c] = stg[r * 5 + c];
        }
        __syncwarp();
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
}

// rho of a complex128 batch of B <= 64 states; QC_ENOMEM (and nothing done) if
// the operand workspace does not fit.
qc_status rho_tc_c128(const double2* psi, int n, int B, const double* P_host, double2* rho, cudaStream_t s) {
  Rho8Dims d;
  d.N = 1ull << n;
  d.B = B;
  d.nkc = (2 * B + 15) / 16;
  d.nib = (int)((d.N + TC5_M - 1) / TC5_M);
  d.njb = (int)((d.N + 31) / 32);
  int64_t ntiles = 0;
  for (int ib = 0; ib < d.nib; ++ib) ntiles += d.njb - 4 * ib;
  const size_t nr = (size_t)d.nib * TC5_M, bytesA = (size_t)d.nib * d.nkc * R8_ND * R8_A,
               bytesB = (size_t)d.njb * d.nkc * R8_ND * R8_B;
  unsigned char* buf = nullptr;
  cudaError_t e = ws_alloc((void**)&buf, bytesA + bytesB + nr * (RHO_ROW + sizeof(int16_t)) +
                                             sizeof(double) * 128 + (size_t)d.nib * d.nib, s);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return QC_ENOMEM;
  }
  double* w = reinterpret_cast<double*>(buf + bytesA + bytesB);  // sqrt(P), then P
  unsigned char* rows = reinterpret_cast<unsigned char*>(w + 128);
  int16_t* E = reinterpret_cast<int16_t*>(rows + nr * RHO_ROW);
  unsigned char* redo = reinterpret_cast<unsigned char*>(E + nr);
  double host[128] = {};
  for (int a = 0; a < B; ++a) host[a] = std::sqrt(P_host[a]), host[64 + a] = P_host[a];
  int nk = put_bytes(w, host, sizeof host, s);
  k_rho8_digits<<<4 * d.nib, 256, 0, s>>>(psi, w, d, buf, buf + bytesA, E, rows, redo);
  allow_smem(k_rho8_tc, R8_SMEM);
  k_rho8_tc<<<(unsigned)std::min<int64_t>(ntiles, sm_count()), R8_T, R8_SMEM, s>>>(buf, buf + bytesA, E, d, ntiles, rho,
                                                                                  redo);
  nk += 2 + launch_rho_fix(psi, n, B, w + 64, E, rows, redo, rho, s);
  const qc_status st = check_launch("density matrix (tensor cores)", nk);
  cudaFreeAsync(buf, s);
  return st;
}

}  // namespace qc
