// Grover search (sec. 5.1).  The Grover operator G = HALL . Inv . HALL .
// Oracle.  The oracle negates the marked amplitudes (Eq. oracle1) and
// HALL . Inv . HALL with Inv = 2|0><0| - I (Eq. inversion) equals
// 2|s><s| - I, |s> = HALL|0..0>, which maps C_i -> 2 m - C_i with m the mean
// amplitude.  So one step is one read+write pass:
//   m = (S - 2 sum_{marked} C) / N      (S = sum of all amplitudes)
//   C_i -> 2 m - C_i (unmarked),  C_i -> 2 m + C_i (marked).
// The diffusion preserves the mean, so the new amplitude sum is known
// without reading the state again: S' = N (2m - m) = N m (for complex64 the
// rounded 2m is used).  S is kept in the state's device scratch and
// recomputed by a reduction only after another operation changed the state.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "fixpt.cuh"

namespace qc {

struct MarkedList {
  int m;
  uint64_t idx[QC_MAX_MARKED];
};

// One block: m from the running sum and the marked amplitudes; saves the
// marked amplitudes and the next running sum.
template <typename R>
__global__ void k_grover_prep(const typename CT<R>::V2* __restrict__ s, uint64_t N, const MarkedList* __restrict__ ML,
                              double* __restrict__ scr) {
  __shared__ double red[2][256];
  double ar = 0.0, ai = 0.0;
  for (int i = threadIdx.x; i < ML->m; i += blockDim.x) {
    const auto v = s[ML->idx[i]];
    scr[QC_SCR_MARKED + 2 * i] = (double)v.x;
    scr[QC_SCR_MARKED + 2 * i + 1] = (double)v.y;
    ar += (double)v.x;
    ai += (double)v.y;
  }
  red[0][threadIdx.x] = ar;
  red[1][threadIdx.x] = ai;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) {
      red[0][threadIdx.x] += red[0][threadIdx.x + w];
      red[1][threadIdx.x] += red[1][threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double Nd = (double)N;
    const double mr = (scr[QC_SCR_SUM] - 2.0 * red[0][0]) / Nd;
    const double mi = (scr[QC_SCR_SUM + 1] - 2.0 * red[1][0]) / Nd;
    scr[QC_SCR_MEAN] = mr;
    scr[QC_SCR_MEAN + 1] = mi;
    const double tr = (double)(R)(2.0 * mr), ti = (double)(R)(2.0 * mi);
    scr[QC_SCR_SUM] = Nd * (tr - mr);
    scr[QC_SCR_SUM + 1] = Nd * (ti - mi);
  }
}

// C -> 2m - C over the whole state.  Real parts on the FP64 pipe, imaginary
// parts in double-float on the FP32 pipe, so that neither pipe limits the
// pass (GB300's FP64 rate allows under 2.5 operations per amplitude at HBM
// speed).
__device__ __forceinline__ double2 grover_c128(double2 a, double tr, ff ti) {
  return make_double2(tr - a.x, ff_to_d(ff_sub(ti, ff_from_d(a.y))));
}
// Four 16-byte loads in flight per thread, three blocks of 256 per SM (the
// launch caps the grid): on GB300 this streams random complex128 data at
// 0.96 of copy bandwidth, against 0.91 for two loads at eight blocks.
constexpr int GROVER_UNR = 4;
__global__ void __launch_bounds__(256, 4) k_grover_pass_c128(double2* __restrict__ s, uint64_t N, const double* __restrict__ scr) {
  const double tr = 2.0 * scr[QC_SCR_MEAN];
  const ff ti = ff_from_d(2.0 * scr[QC_SCR_MEAN + 1]);
  const uint64_t G = (uint64_t)gridDim.x * blockDim.x;
  uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (; i + (GROVER_UNR - 1) * G < N; i += GROVER_UNR * G) {
    double2 a[GROVER_UNR];
#pragma unroll
    for (int u = 0; u < GROVER_UNR; ++u) a[u] = s[i + u * G];
#pragma unroll
    for (int u = 0; u < GROVER_UNR; ++u) s[i + u * G] = grover_c128(a[u], tr, ti);
  }
  for (; i < N; i += G) s[i] = grover_c128(s[i], tr, ti);
}

__global__ void __launch_bounds__(256) k_grover_pass_c64(float4* __restrict__ s, uint64_t N2, const double* __restrict__ scr) {
  const float tr = (float)(2.0 * scr[QC_SCR_MEAN]), ti = (float)(2.0 * scr[QC_SCR_MEAN + 1]);
  const uint64_t G = (uint64_t)gridDim.x * blockDim.x;
  uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (; i + G < N2; i += 2 * G) {
    float4 a = s[i], b = s[i + G];
    s[i] = make_float4(tr - a.x, ti - a.y, tr - a.z, ti - a.w);
    s[i + G] = make_float4(tr - b.x, ti - b.y, tr - b.z, ti - b.w);
  }
  if (i < N2) {
    float4 a = s[i];
    s[i] = make_float4(tr - a.x, ti - a.y, tr - a.z, ti - a.w);
  }
}

// Marked amplitudes: 2m + C_old.
template <typename R>
__global__ void k_grover_fix(typename CT<R>::V2* __restrict__ s, const MarkedList* __restrict__ ML,
                             const double* __restrict__ scr) {
  const double mr = scr[QC_SCR_MEAN], mi = scr[QC_SCR_MEAN + 1];
  const R tr = (R)(2.0 * mr), ti = (R)(2.0 * mi);
  for (int i = threadIdx.x; i < ML->m; i += blockDim.x) {
    const R cr = (R)scr[QC_SCR_MARKED + 2 * i], ci = (R)scr[QC_SCR_MARKED + 2 * i + 1];
    s[ML->idx[i]] = CT<R>::make(tr + cr, ti + ci);
  }
}

// Device copy of the marked list, kept in the handle and re-uploaded only
// when the list changes (the upload synchronises the stream once).
static qc_status upload_marked(qc_state* s, const uint64_t* marked, int m, MarkedList** out) {
  if (!s->marked_dev) {
    cudaError_t e = cudaMalloc(&s->marked_dev, sizeof(MarkedList));
    if (e != cudaSuccess) {
      s->marked_dev = nullptr;
      return cuda_fail(e, "marked list");
    }
    s->marked_host.clear();
  }
  const bool same = (int)s->marked_host.size() == m &&
                    std::equal(s->marked_host.begin(), s->marked_host.end(), marked);
  if (!same) {
    const size_t bytes = sizeof(int) * 2 + sizeof(uint64_t) * (size_t)m;
    MarkedList* h = nullptr;
    cudaError_t e = cudaMallocHost((void**)&h, bytes);
    if (e != cudaSuccess) return cuda_fail(e, "marked list (host)");
    h->m = m;
    for (int i = 0; i < m; ++i) h->idx[i] = marked[i];
    e = cudaMemcpyAsync(s->marked_dev, h, bytes, cudaMemcpyHostToDevice, s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
    cudaFreeHost(h);
    if (e != cudaSuccess) {
      s->marked_host.clear();
      return cuda_fail(e, "marked list upload");
    }
    s->marked_host.assign(marked, marked + m);
  }
  *out = reinterpret_cast<MarkedList*>(s->marked_dev);
  return QC_OK;
}

static qc_status step_with(qc_state* s, const MarkedList* dml) {
  const uint64_t N = 1ull << s->n;
  const int T = 256;
  if (s->dt == QC_C128) {
    k_grover_prep<double><<<1, 256, 0, s->stream>>>(reinterpret_cast<const double2*>(s->data), N, dml, s->scratch);
    const unsigned g = std::min<unsigned>(resident_grid(k_grover_pass_c128, T, N, GROVER_UNR * T), 3u * (unsigned)sm_count());
    k_grover_pass_c128<<<g, T, 0, s->stream>>>(reinterpret_cast<double2*>(s->data), N, s->scratch);
    k_grover_fix<double><<<1, 256, 0, s->stream>>>(reinterpret_cast<double2*>(s->data), dml, s->scratch);
  } else {
    k_grover_prep<float><<<1, 256, 0, s->stream>>>(reinterpret_cast<const float2*>(s->data), N, dml, s->scratch);
    const uint64_t N2 = N / 2;
    if (N2 > 0)
      k_grover_pass_c64<<<resident_grid(k_grover_pass_c64, T, N2, 2 * T), T, 0, s->stream>>>(
          reinterpret_cast<float4*>(s->data), N2, s->scratch);
    k_grover_fix<float><<<1, 256, 0, s->stream>>>(reinterpret_cast<float2*>(s->data), dml, s->scratch);
  }
  return check_launch("grover step", 3);
}

qc_status launch_grover_step(qc_state* s, const uint64_t* marked, int m) {
  if (s->n < 2 && s->dt == QC_C64) {
    set_error("complex64 Grover needs n >= 2");
    return QC_EINVAL;
  }
  qc_status st = QC_OK;
  if (!s->sum_valid) {
    st = launch_sum(s);
    if (st) return st;
  }
  MarkedList* dml = nullptr;
  st = upload_marked(s, marked, m, &dml);
  if (st) return st;
  s->grover_partial_ready = false;  // the saved marked amplitudes are overwritten
  st = step_with(s, dml);
  s->sum_valid = (st == QC_OK);
  return st;
}

// ------------------------------------------ a state split over devices ----
// For a state split over several devices (one shard per device, the high
// index bits selecting the shard), the Grover mean needs the sum over all
// shards: each shard contributes P_r = S_r - 2 sum_{marked in r} C, the
// caller adds them (one scalar all-reduce) and hands back m = sum_r P_r / N.
// The pass itself is the single-device one.
template <typename R>
__global__ void k_grover_partial(const typename CT<R>::V2* __restrict__ s, const MarkedList* __restrict__ ML,
                                 double* __restrict__ scr) {
  __shared__ double red[2][256];
  double ar = 0.0, ai = 0.0;
  for (int i = threadIdx.x; i < ML->m; i += blockDim.x) {
    const auto v = s[ML->idx[i]];
    scr[QC_SCR_MARKED + 2 * i] = (double)v.x;
    scr[QC_SCR_MARKED + 2 * i + 1] = (double)v.y;
    ar += (double)v.x;
    ai += (double)v.y;
  }
  red[0][threadIdx.x] = ar;
  red[1][threadIdx.x] = ai;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) {
      red[0][threadIdx.x] += red[0][threadIdx.x + w];
      red[1][threadIdx.x] += red[1][threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {  // P_r in the misc slots
    scr[QC_SCR_MISC] = scr[QC_SCR_SUM] - 2.0 * red[0][0];
    scr[QC_SCR_MISC + 1] = scr[QC_SCR_SUM + 1] - 2.0 * red[1][0];
  }
}

// The given mean into the scratch, and the shard's next running sum
// S_r' = N_r (2m) - P_r (2m rounded as the pass rounds it).
template <typename R>
__global__ void k_grover_set_mean(double* __restrict__ scr, uint64_t N, double mr, double mi) {
  scr[QC_SCR_MEAN] = mr;
  scr[QC_SCR_MEAN + 1] = mi;
  const double tr = (double)(R)(2.0 * mr), ti = (double)(R)(2.0 * mi);
  scr[QC_SCR_SUM] = (double)N * tr - scr[QC_SCR_MISC];
  scr[QC_SCR_SUM + 1] = (double)N * ti - scr[QC_SCR_MISC + 1];
}

qc_status launch_grover_partial(qc_state* s, const uint64_t* marked, int m, double* out_host) {
  qc_status st = QC_OK;
  if (!s->sum_valid) {
    st = launch_sum(s);
    if (st) return st;
  }
  MarkedList* dml = nullptr;
  st = upload_marked(s, marked, m, &dml);
  if (st) return st;
  if (s->dt == QC_C128)
    k_grover_partial<double><<<1, 256, 0, s->stream>>>(reinterpret_cast<const double2*>(s->data), dml, s->scratch);
  else
    k_grover_partial<float><<<1, 256, 0, s->stream>>>(reinterpret_cast<const float2*>(s->data), dml, s->scratch);
  st = check_launch("grover partial sum");
  if (st) return st;
  cudaError_t e = cudaMemcpyAsync(out_host, s->scratch + QC_SCR_MISC, 2 * sizeof(double), cudaMemcpyDeviceToHost,
                                  s->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
  if (e != cudaSuccess) return cuda_fail(e, "grover partial readback");
  s->grover_partial_ready = true;
  return QC_OK;
}

qc_status launch_grover_apply(qc_state* s, const uint64_t* marked, int m, const double* mean) {
  if (!s->grover_partial_ready || !s->sum_valid || (int)s->marked_host.size() != m ||
      !std::equal(s->marked_host.begin(), s->marked_host.end(), marked)) {
    set_error("qc_grover_apply_mean: call qc_grover_partial with the same marked list first");
    return QC_EINVAL;
  }
  s->grover_partial_ready = false;
  const uint64_t N = 1ull << s->n;
  const int T = 256;
  const MarkedList* dml = reinterpret_cast<const MarkedList*>(s->marked_dev);
  if (s->dt == QC_C128) {
    k_grover_set_mean<double><<<1, 1, 0, s->stream>>>(s->scratch, N, mean[0], mean[1]);
    const unsigned g = std::min<unsigned>(resident_grid(k_grover_pass_c128, T, N, GROVER_UNR * T), 3u * (unsigned)sm_count());
    k_grover_pass_c128<<<g, T, 0, s->stream>>>(reinterpret_cast<double2*>(s->data), N, s->scratch);
    k_grover_fix<double><<<1, 256, 0, s->stream>>>(reinterpret_cast<double2*>(s->data), dml, s->scratch);
  } else {
    k_grover_set_mean<float><<<1, 1, 0, s->stream>>>(s->scratch, N, mean[0], mean[1]);
    const uint64_t N2 = N / 2;
    if (N2 > 0)
      k_grover_pass_c64<<<resident_grid(k_grover_pass_c64, T, N2, 2 * T), T, 0, s->stream>>>(
          reinterpret_cast<float4*>(s->data), N2, s->scratch);
    k_grover_fix<float><<<1, 256, 0, s->stream>>>(reinterpret_cast<float2*>(s->data), dml, s->scratch);
  }
  qc_status st = check_launch("grover pass (given mean)", 3);
  s->sum_valid = (st == QC_OK);
  return st;
}

// ---------------------------------------------------- whole small run ----
// HALL|0..0> followed by `iters` Grover steps in one block.  The start state
// and both operators are real, so the amplitudes are carried as real 64-bit
// fixed point (unit 2^-62), in registers, from the first to the last step.
// With P = sum of the amplitudes after the oracle = S - 2 sum_{marked} C, a
// step maps C -> 2m - C (unmarked), 2m + C (marked), 2m = 2 P / N, and the new
// sum is S' = N 2m - P.  Sums and differences are exact integers, P and S in
// 128 bits; the only rounding of a step is 2m to the unit, and S' follows it
// exactly, so S stays the sum of the amplitudes held.  A step is therefore the
// sum of the marked amplitudes (one thread each), one barrier and one
// subtraction an amplitude; summing all amplitudes in double-float each step
// took 1.6 us a step (10 qubits; 40 us for 25 steps), this 0.1 us.
struct I128 {
  unsigned long long lo;
  long long hi;
};
__device__ __forceinline__ I128 i128_of(__int128 v) { return I128{(unsigned long long)v, (long long)(v >> 64)}; }
__device__ __forceinline__ __int128 i128_to(I128 v) { return ((__int128)v.hi << 64) | (__int128)v.lo; }

template <typename V2, int PER>
__global__ void __launch_bounds__(1024) k_grover_small(V2* __restrict__ s, int n, const MarkedList* __restrict__ ML,
                                                       int iters) {
  __shared__ I128 part[2][32];
  const int tid = threadIdx.x, T = blockDim.x, N = 1 << n, m = ML->m;
  const int lane = tid & 31, warp = tid >> 5, nw = (m + 31) >> 5;  // warps that hold marked amplitudes
  // 2^(62 - n/2), rounded for odd n: sqrt 2 2^62 is 6521908912666391106.2
  const int h = (n + 1) >> 1;
  const long long a = (n & 1) ? (6521908912666391106ll + (1ll << (h - 1))) >> h : 1ll << (62 - h);
  long long c[PER], mk = tid < m ? a : 0;
#pragma unroll
  for (int u = 0; u < PER; ++u) c[u] = a;
  __int128 S = (__int128)a << n;
  const int steps = m > 16 ? 5 : m > 8 ? 4 : m > 4 ? 3 : m > 2 ? 2 : m > 1 ? 1 : 0;
  for (int it = 0; it < iters; ++it) {
    I128* buf = part[it & 1];
    if (warp < nw) {
      __int128 t = mk;
      for (int o = 1, k = 0; k < steps; ++k, o <<= 1) {
        const I128 v = i128_of(t);
        t += i128_to(I128{__shfl_xor_sync(0xffffffffu, v.lo, o), __shfl_xor_sync(0xffffffffu, v.hi, o)});
      }
      if (lane == 0) buf[warp] = i128_of(t);
    }
    __syncthreads();
    __int128 P = S;
    if (nw <= 4) {
      for (int w = 0; w < nw; ++w) P -= i128_to(buf[w]) * 2;
    } else {  // many marked: a partial sum a lane (32 of them one by one: 2.6 us a step, 1.3 so)
      __int128 t = lane < nw ? i128_to(buf[lane]) : 0;
      for (int o = 16; o; o >>= 1) {
        const I128 v = i128_of(t);
        t += i128_to(I128{__shfl_xor_sync(0xffffffffu, v.lo, o), __shfl_xor_sync(0xffffffffu, v.hi, o)});
      }
      P -= t * 2;
    }
    const long long t2 = (long long)((P + ((__int128)1 << (n - 1) >> 1)) >> (n - 1));
    S = ((__int128)t2 << n) - P;
#pragma unroll
    for (int u = 0; u < PER; ++u) c[u] = t2 - c[u];
    if (tid < m) mk += t2;
  }
  auto out = [](long long v) {
    if constexpr (sizeof(V2) == 16) return make_double2(fix2d(v, 62), 0.0);
    else return make_float2((float)v * 0x1p-62f, 0.f);
  };
#pragma unroll
  for (int u = 0; u < PER; ++u)
    if (tid + T * u < N) s[tid + T * u] = out(c[u]);
  __syncthreads();
  if (tid < m) s[ML->idx[tid]] = out(mk);
}

template <typename V2>
static void run_small(qc_state* s, const MarkedList* dml, int m, int iters) {
  V2* d = reinterpret_cast<V2*>(s->data);
  // eight amplitudes a thread (a step's scalar part is the same in every warp),
  // a thread for every marked item
  const int N = 1 << s->n, per = N <= 8192 ? 8 : 16, need = std::max(N / per, m);
  const int T = std::min(1024, std::max(32, (need + 31) / 32 * 32));
  if (per == 8) k_grover_small<V2, 8><<<1, T, 0, s->stream>>>(d, s->n, dml, iters);
  else k_grover_small<V2, 16><<<1, T, 0, s->stream>>>(d, s->n, dml, iters);
}

qc_status launch_grover_run(qc_state* s, const uint64_t* marked, int m, int iters) {
  MarkedList* dml = nullptr;
  qc_status st = upload_marked(s, marked, m, &dml);
  if (st) return st;
  const bool small = (s->dt == QC_C128) ? (s->n <= 13) : (s->n <= 14);
  if (small) {
    if (s->dt == QC_C128) run_small<double2>(s, dml, m, iters);
    else run_small<float2>(s, dml, m, iters);
    st = check_launch("grover run (one block)");
    s->sum_valid = false;
  } else {
    st = launch_fill_uniform(s);  // HALL|0..0>; records the amplitude sum
    for (int it = 0; it < iters && !st; ++it) st = step_with(s, dml);
    s->sum_valid = (st == QC_OK);
  }
  return st;
}

}  // namespace qc
