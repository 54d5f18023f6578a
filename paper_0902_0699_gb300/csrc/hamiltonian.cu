// One first-order step of Hamiltonian evolution (sec. 7, hbar = 1):
//   psi <- psi + sum_t A_t psi,   A_t = -i dt h_t,
// every term acting on the state as it was before the step.
//
// A term's matrix splits by the bits it flips: entry h[l][l ^ x] adds
// h[l][l ^ x] psi[j with l ^ x] to amplitude j (l = j's bits on the term's
// qubits).  Terms are grouped into passes by a tile of up to 12 index bits
// that holds their qubits: a pass stages tiles of psi in shared memory and adds,
// for each of its flips, one product per amplitude with a coefficient picked
// by one or two of j's bits; flips whose entries are all zero, and real or
// imaginary parts that are zero throughout, cost nothing.  The diagonals
// (x = 0) of all of a pass's terms depend on the tile's bits only and are
// summed once into a table of 2^kt coefficients.
//
// Passes but the last leave psi alone and accumulate in a workspace; the last
// writes psi, whose tile no other block reads.  A chain of 21 bonds and 22
// fields on 22 qubits takes three passes (eight state transfers) where one
// accumulating pass per term took 43 (129 transfers and double-float products
// of full 4x4 blocks): 3.2 -> 0.52 ms a step in complex128, 1.1 -> 0.19 ms in
// complex64, and the relative error of two steps 2.1e-14 -> 1.1e-15.
//
// complex128: products and sums of a pass in double-float, added to psi in
// FP64 (two operations an amplitude).  complex64: FP32.
#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"

namespace qc {

constexpr int HS_KT = 12;      // tile bits
constexpr int HS_PER = 8;      // amplitudes per thread
constexpr int HS_MAXENT = 96;  // flips of a pass

// One flip: partner = tile element XOR `off` (swizzled byte offset), the
// coefficient c[bit sa of j | bit sb of j << 1] (double-float re, im; complex64
// uses x and z).
struct HFlip {
  int off;
  int8_t sa, sb;  // tile positions; sb = sa for a one-qubit term
  int8_t re, im;  // whether any real / imaginary part is nonzero
  int pad[2];
  float4 c[4];
};
// One diagonal: d[bit sa | bit sb << 1]
struct HDiag {
  int8_t sa, sb, pad[6];
  double2 d[4];
};
struct HPass {
  int kt, nfix, nflip, ndiag, dre, dim;
  int first, last;
  int8_t pos[16];
  int8_t fix[40];
};

template <typename R> struct HT;
template <> struct HT<float> {
  using V = float2;
  using E = float2;  // staged amplitude
  __device__ static int at(int e) { return (e ^ ((e >> 4) & 15)) * 8; }
  __device__ static E from(V v) { return v; }
  struct Sum {
    float re = 0.f, im = 0.f;
    __device__ void mac(bool r, bool i, float4 c, E x) {
      if (r) {
        re = fmaf(c.x, x.x, re);
        im = fmaf(c.x, x.y, im);
      }
      if (i) {
        re = fmaf(-c.z, x.y, re);
        im = fmaf(c.z, x.x, im);
      }
    }
    __device__ void norm() {}
    __device__ V plus(V b) const { return make_float2(b.x + re, b.y + im); }
  };
};
template <> struct HT<double> {
  using V = double2;
  using E = float4;
  __device__ static int at(int e) { return (e ^ ((e >> 3) & 7)) * 16; }
  __device__ static E from(V v) {
    const ff a = ff_from_d(v.x), b = ff_from_d(v.y);
    return make_float4(a.hi, a.lo, b.hi, b.lo);
  }
  struct Sum {
    ffacc re{0.f, 0.f}, im{0.f, 0.f};
    __device__ void mac(bool r, bool i, float4 c, E x) {
      const ff xr = ff_make(x.x, x.y), xi = ff_make(x.z, x.w);
      if (r) {
        const ff k = ff_make(c.x, c.y);
        ffacc_add(re, k, xr);
        ffacc_add(im, k, xi);
      }
      if (i) {
        const ff k = ff_make(c.z, c.w);
        ffacc_add(re, ff_neg(k), xi);
        ffacc_add(im, k, xr);
      }
    }
    __device__ void norm() {
      ffacc_norm(re);
      ffacc_norm(im);
    }
    __device__ V plus(V b) const {
      return make_double2(b.x + ff_to_d(ffacc_result(re)), b.y + ff_to_d(ffacc_result(im)));
    }
  };
};

// The diagonals' sum for every tile element of pass blockIdx.y, in FP64,
// stored as a flip's coefficients are.
template <typename R>
__global__ void __launch_bounds__(128) k_hdiag(const HPass* __restrict__ passes, const HDiag* __restrict__ diags,
                                               const int* __restrict__ dfirst, float4* __restrict__ tab) {
  const HPass& P = passes[blockIdx.y];
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (1 << P.kt)) return;
  double2 s = make_double2(0.0, 0.0);
  const HDiag* D = diags + dfirst[blockIdx.y];
  for (int k = 0; k < P.ndiag; ++k) {
    const double2 d = D[k].d[((e >> D[k].sa) & 1) | ((e >> D[k].sb) & 1) << 1];
    s.x += d.x;
    s.y += d.y;
  }
  const ff a = ff_from_d(s.x), b = ff_from_d(s.y);
  tab[((size_t)blockIdx.y << HS_KT) + e] =
      sizeof(R) == 8 ? make_float4(a.hi, a.lo, b.hi, b.lo) : make_float4((float)s.x, 0.f, (float)s.y, 0.f);
}

template <typename R>
__global__ void __launch_bounds__(512, 2) k_hstep(typename HT<R>::V* __restrict__ psi, typename HT<R>::V* __restrict__ ws,
                                                  int ntiles, const __grid_constant__ HPass P,
                                                  const HFlip* __restrict__ flips, const float4* __restrict__ dtab) {
  using H = HT<R>;
  using E = typename H::E;
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ HFlip F[HS_MAXENT];
  const int tid = threadIdx.x, T = blockDim.x, ne = 1 << P.kt, lt = 31 - __clz(T);
  for (int i = tid; i < P.nflip * (int)(sizeof(HFlip) / 16); i += T)
    reinterpret_cast<uint4*>(F)[i] = reinterpret_cast<const uint4*>(flips)[i];
  // element e = tid + T u: offsets are the thread's part or'ed with u's
  uint64_t gT = 0, gU[3];
  int aU[3];
  for (int p = 0; p < lt && p < P.kt; ++p) gT |= (uint64_t)((tid >> p) & 1) << P.pos[p];
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    gU[x] = lt + x < P.kt ? 1ull << P.pos[lt + x] : 0;
    aU[x] = H::at(T << x);
  }
  const int aT = H::at(tid);
  auto g_of = [&](int u) { return gT | ((u & 1) ? gU[0] : 0) | ((u & 2) ? gU[1] : 0) | ((u & 4) ? gU[2] : 0); };
  auto a_of = [&](int u) { return aT ^ ((u & 1) ? aU[0] : 0) ^ ((u & 2) ? aU[1] : 0) ^ ((u & 4) ? aU[2] : 0); };
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    uint64_t base = 0;
    for (int p = 0; p < P.nfix; ++p) base |= (uint64_t)((tile >> p) & 1) << P.fix[p];
    typename H::V v[HS_PER];
#pragma unroll
    for (int u = 0; u < HS_PER; ++u)
      if (tid + T * u < ne) v[u] = psi[base | g_of(u)];
#pragma unroll
    for (int u = 0; u < HS_PER; ++u)
      if (tid + T * u < ne) *reinterpret_cast<E*>(sm + a_of(u)) = H::from(v[u]);
    __syncthreads();
#pragma unroll 1
    for (int h = 0; h < HS_PER; h += 4) {
      typename H::Sum S[4];
      if (P.ndiag) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int e = tid + T * (h + u);
          if (e < ne) S[u].mac(P.dre, P.dim, dtab[e], *reinterpret_cast<const E*>(sm + a_of(h + u)));
        }
      }
#pragma unroll 1
      for (int k = 0; k < P.nflip; ++k) {
        const HFlip& f = F[k];
        const int sa = f.sa, sb = f.sb, off = f.off;
        const bool re = f.re, im = f.im;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int e = tid + T * (h + u);
          if (e < ne)
            S[u].mac(re, im, f.c[((e >> sa) & 1) | ((e >> sb) & 1) << 1],
                     *reinterpret_cast<const E*>(sm + (a_of(h + u) ^ off)));
        }
        // at most four products since the last, and a complex diagonal's two
        // before the first (a pass's up to 194 then stay within ff.cuh's bound)
        if ((k & 1) && sizeof(R) == 8) {
#pragma unroll
          for (int u = 0; u < 4; ++u) S[u].norm();
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint64_t g = base | g_of(h + u);
        if (tid + T * (h + u) < ne) (P.last ? psi : ws)[g] = S[u].plus(P.first ? psi[g] : ws[g]);
      }
    }
    __syncthreads();
  }
}

struct HTermHost {
  int k, q[2];
  double a[32];  // -i dt h, row-major
};

// Passes for the terms: a pass starts with the first term left and takes every
// later one whose qubits fit its tile (a term that needs no new bit first).
template <typename R>
static qc_status run_hstep(qc_state* s, const std::vector<HTermHost>& terms) {
  const int n = s->n, kt = std::min(n, HS_KT), c0 = std::min(n, sizeof(R) == 8 ? 3 : 4);
  std::vector<HPass> passes;
  std::vector<HFlip> flips;
  std::vector<HDiag> diags;
  std::vector<int> ffirst, dfirst;
  std::vector<char> done(terms.size(), 0);
  size_t left = terms.size();
  while (left) {
    uint64_t tile = (1ull << c0) - 1;
    std::vector<size_t> mine;
    for (int need = 0; need <= 2; ++need) {  // new bits a term may bring
      for (size_t t = 0; t < terms.size() && (int)mine.size() < HS_MAXENT / 3; ++t) {
        if (done[t]) continue;
        uint64_t m = 0;
        for (int b = 0; b < terms[t].k; ++b) m |= 1ull << terms[t].q[b];
        if (__builtin_popcountll(m & ~tile) > need || __builtin_popcountll(tile | m) > kt) continue;
        tile |= m;
        mine.push_back(t);
        done[t] = 1;
        --left;
        if (need) need = 0, t = (size_t)-1;  // the tile grew: terms inside it first
      }
    }
    for (int q = 0; q < n && __builtin_popcountll(tile) < kt; ++q) tile |= 1ull << q;
    HPass P{};
    P.kt = kt;
    int where[64] = {};
    int np = 0;
    for (int q = 0; q < n; ++q) {
      if ((tile >> q) & 1) {
        where[q] = np;
        P.pos[np++] = (int8_t)q;
      } else {
        P.fix[P.nfix++] = (int8_t)q;
      }
    }
    ffirst.push_back((int)flips.size());
    dfirst.push_back((int)diags.size());
    for (size_t t : mine) {
      const HTermHost& H = terms[t];
      const int dim = 1 << H.k, sa = where[H.q[0]], sb = H.k == 2 ? where[H.q[1]] : sa;
      for (int x = 0; x < dim; ++x) {
        double re[4] = {}, im[4] = {};
        bool anyr = false, anyi = false;
        for (int i = 0; i < 4; ++i) {  // i = bit sa | bit sb << 1
          const int l = H.k == 2 ? i : (i & 1);
          re[i] = H.a[2 * (l * dim + (l ^ x))];
          im[i] = H.a[2 * (l * dim + (l ^ x)) + 1];
          anyr |= re[i] != 0.0;
          anyi |= im[i] != 0.0;
        }
        if (!anyr && !anyi) continue;
        if (x == 0) {
          HDiag D{};
          D.sa = (int8_t)sa;
          D.sb = (int8_t)sb;
          for (int i = 0; i < 4; ++i) D.d[i] = make_double2(re[i], im[i]);
          diags.push_back(D);
          ++P.ndiag;
          P.dre |= anyr;
          P.dim |= anyi;
        } else {
          HFlip f{};
          const int m = ((x & 1) << sa) | (H.k == 2 ? (x >> 1) << sb : 0);
          f.off = sizeof(R) == 8 ? (m ^ ((m >> 3) & 7)) * 16 : (m ^ ((m >> 4) & 15)) * 8;
          f.sa = (int8_t)sa;
          f.sb = (int8_t)sb;
          f.re = anyr;
          f.im = anyi;
          for (int i = 0; i < 4; ++i) {
            if (sizeof(R) == 8) {
              const ff a = ff_from_d(re[i]), b = ff_from_d(im[i]);
              f.c[i] = make_float4(a.hi, a.lo, b.hi, b.lo);
            } else {
              f.c[i] = make_float4((float)re[i], 0.f, (float)im[i], 0.f);
            }
          }
          flips.push_back(f);
          ++P.nflip;
        }
      }
    }
    passes.push_back(P);
  }
  const int npass = (int)passes.size();
  passes.front().first = 1;
  passes.back().last = 1;
  // one workspace: the step's partial sum (if more than one pass), tables
  using V = typename HT<R>::V;
  const size_t state = npass > 1 ? sizeof(V) << n : 0, bp = (sizeof(HPass) * npass + 15) / 16 * 16,
               bf = sizeof(HFlip) * flips.size(), bd = sizeof(HDiag) * diags.size(), bi = (4 * (size_t)npass + 15) / 16 * 16,
               bt = (sizeof(float4) << HS_KT) * npass;
  char* w = nullptr;
  cudaError_t e = ws_alloc((void**)&w, state + bt + bp + bf + bd + bi, s->stream);
  if (e != cudaSuccess) return cuda_fail(e, "Hamiltonian step workspace");
  V* acc = reinterpret_cast<V*>(w);
  float4* tab = reinterpret_cast<float4*>(w + state);
  HFlip* df = reinterpret_cast<HFlip*>(w + state + bt);
  HDiag* dd = reinterpret_cast<HDiag*>(w + state + bt + bf);
  HPass* dp = reinterpret_cast<HPass*>(w + state + bt + bf + bd);
  int* di = reinterpret_cast<int*>(w + state + bt + bf + bd + bp);
  int nk = put_bytes(df, flips.data(), bf, s->stream);
  if (!diags.empty()) {
    nk += put_bytes(dd, diags.data(), bd, s->stream) + put_bytes(dp, passes.data(), sizeof(HPass) * npass, s->stream) +
          put_bytes(di, dfirst.data(), 4 * (size_t)npass, s->stream) + 1;
    k_hdiag<R><<<dim3(std::max(1, (1 << kt) / 128), npass), 128, 0, s->stream>>>(dp, dd, di, tab);
  }
  const size_t smem = sizeof(typename HT<R>::E) << kt;
  allow_smem(k_hstep<R>, sizeof(typename HT<R>::E) << HS_KT);
  const int T = std::max(32, (1 << kt) / HS_PER), ntiles = 1 << (n - kt);
  const unsigned grid = resident_grid(k_hstep<R>, T, ntiles, 1, smem);
  // a pass is launched only after the ones before it were: the last adds what they left in the workspace to psi
  qc_status st = check_launch("Hamiltonian step setup", nk);
  for (int p = 0; p < npass && !st; ++p) {
    k_hstep<R><<<grid, T, smem, s->stream>>>(reinterpret_cast<V*>(s->data), acc, ntiles, passes[p], df + ffirst[p],
                                             tab + ((size_t)p << HS_KT));
    st = check_launch("Hamiltonian step");
  }
  cudaFreeAsync(w, s->stream);
  s->sum_valid = false;
  return st;
}

}  // namespace qc

using namespace qc;

QC_API qc_status qc_hamiltonian_step(qc_state* s, double dt, const qc_hterm* terms, int n_terms) {
  clear_error();
  qc_status st = check_state(s);
  if (st) return st;
  if (n_terms < 0 || (n_terms > 0 && !terms) || !std::isfinite(dt)) {
    set_error("qc_hamiltonian_step: bad term list or dt");
    return QC_EINVAL;
  }
  std::vector<HTermHost> H(n_terms);
  for (int t = 0; t < n_terms; ++t) {
    const qc_hterm& T = terms[t];
    if ((T.k != 1 && T.k != 2) || T.k > s->n) {
      set_error("qc_hamiltonian_step: term %d has k = %d (1 or 2 qubits)", t, T.k);
      return QC_EINVAL;
    }
    for (int b = 0; b < T.k; ++b)
      if (T.qubits[b] < 0 || T.qubits[b] >= s->n || (b == 1 && T.qubits[1] == T.qubits[0])) {
        set_error("qc_hamiltonian_step: term %d qubit %d out of range or repeated", t, T.qubits[b]);
        return QC_EINVAL;
      }
    HTermHost& A = H[t];
    A = HTermHost{T.k, {T.qubits[0], T.k == 2 ? T.qubits[1] : T.qubits[0]}, {}};
    const int dim = 1 << T.k;
    for (int e = 0; e < dim * dim; ++e) {
      const double hr = T.h[2 * e], hi = T.h[2 * e + 1];
      if (!std::isfinite(hr) || !std::isfinite(hi)) {
        set_error("qc_hamiltonian_step: term %d has a non-finite entry", t);
        return QC_EINVAL;
      }
      A.a[2 * e] = dt * hi;  // (-i dt)(hr + i hi) = dt hi - i dt hr
      A.a[2 * e + 1] = -dt * hr;
    }
  }
  if (n_terms == 0) return QC_OK;
  return s->dt == QC_C128 ? run_hstep<double>(s, H) : run_hstep<float>(s, H);
}
