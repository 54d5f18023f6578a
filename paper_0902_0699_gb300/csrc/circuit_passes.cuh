// A parameterised circuit as passes over shared-memory tiles (used by
// adjoint.cu).
//
// A pass works on tiles of 2^kt amplitudes: the index bits in `pos` vary
// inside a tile, the others are fixed by the tile's number.  It applies, in
// this order, one-qubit operators on tile qubits (S), the diagonal rotations
// that come last on their qubit as one phase factor per amplitude (D), and a
// string of CNOTs whose targets are tile qubits (P).  A CNOT only moves an
// amplitude along its target bit, so P is a linear map of the tile's index
// bits plus a constant from the fixed control bits: it costs an XOR per
// address of the tile's load or store, and a ring CNOT(0,1) .. CNOT(n-1,0)
// needs no pass of its own.
//
// The builder takes gates in order and leaves out what does not fit; a gate
// may overtake left-out ones only if it shares no qubit with them.  With
// `merge` (complex64 forward) no operator overtakes a left-out operator
// either, so every amplitude sees the same roundings in the same order as
// under one pass per operator.
#pragma once

#include <algorithm>
#include <vector>

#include "common.cuh"

namespace qc {

constexpr int TP_MAXK = 13;     // largest tile: 2^13 amplitudes
constexpr int TP_MAXOP = 40;    // one-qubit operators of a pass
constexpr int TP_MAXRD = 14;    // register rounds of a pass
constexpr int TP_LOOK = 256;    // gates a pass leaves out before it looks no further

// A one-qubit operator: rotation kind ka with angle index pa, then (merged
// rotation pairs only) kb with pb.  `bit` is its register bit in its round.
struct TileOp {
  int8_t bit, ka, kb, tpos;
  int32_t pa, pb;
};
// A round: every thread holds the 2^RB amplitudes that differ in the tile
// positions r[0..RB) and applies operators [op0, op1) to them.
struct TileRound {
  uint16_t bas[4];  // swizzled byte offset of each register bit
  int8_t r[4];
  int8_t op0, op1, pad[2];
};
struct TilePass {
  int16_t kt, nreal;  // tile bits; index bits among them (nreal < kt only for states smaller than a register block)
  int16_t nfix, nround, nop, nfc, has_perm, has_diag, has_fac, pad;
  int8_t pos[TP_MAXK + 3];   // index bit of tile position p, ascending
  int8_t fix[32];            // the other index bits, ascending
  // P: the source of tile element e is the XOR of col[p] over e's set bits and
  // of fm[i] over the fixed index bits fc[i] that are 1 (as swizzled byte offsets)
  uint16_t col[TP_MAXK + 3];
  int8_t fc[32];
  uint16_t fm[32];
  int32_t dp[TP_MAXK + 3];   // D: angle index of the RZ on tile position p, or -1
  TileRound rd[TP_MAXRD];
  TileOp op[TP_MAXOP];
};

// Shared-memory swizzle of a tile index (linear over XOR): the register
// rounds then read any positions without bank conflicts.
template <typename R>
__host__ __device__ __forceinline__ int tp_swz(int e) {
  return sizeof(R) == 4 ? (e ^ ((e >> 4) & 15)) : (e ^ ((e >> 3) & 7));
}

// Byte offset in shared memory.
template <typename R>
__host__ __device__ __forceinline__ int tp_at(int e) {
  return tp_swz<R>(e) * (int)(2 * sizeof(R));
}

// Offset of tile number `tile` in the state.
__device__ __forceinline__ uint64_t tp_tile_base(const TilePass& P, uint64_t tile) {
  uint64_t o = 0;
  for (int p = 0; p < P.nfix; ++p) o |= ((tile >> p) & 1ull) << P.fix[p];
  return o;
}
// P's constant for a tile.
__device__ __forceinline__ int tp_cst(const TilePass& P, uint64_t base) {
  int s = 0;
  for (int i = 0; i < P.nfc; ++i) s ^= ((base >> P.fc[i]) & 1ull) ? P.fm[i] : 0;
  return s;
}

// A thread's share of a tile: the 2^LV 16-byte vectors w = tid + T u, u <
// 2^LV, of VE amplitudes.  Offsets are linear in the bits of w, so each is an
// XOR of the thread's part and of those of u's bits.
template <typename R, int LV>
struct TileShare {
  static constexpr int VE = sizeof(R) == 4 ? 2 : 1;
  uint64_t gT, gU[LV];  // amplitude offset in the state, from the tile's base
  int aT, aU[LV];       // byte offset in shared memory
  int sT, sU[LV], s1;   // byte offset of P's source (s1: of the vector's second amplitude)
  __device__ void init(const TilePass& P, int T) {
    const int e = (int)threadIdx.x * VE;
    gT = 0;
    sT = 0;
    const int lo = VE - 1, lt = 31 - __clz(T * VE);
    for (int p = lo; p < lt; ++p) {
      const int on = (e >> p) & 1;
      if (p < P.nreal) gT |= (uint64_t)on << P.pos[p];
      sT ^= on ? P.col[p] : 0;
    }
    aT = tp_at<R>(e);
    s1 = P.col[0];
#pragma unroll
    for (int x = 0; x < LV; ++x) {
      const int p = lt + x;
      gU[x] = p < P.nreal ? 1ull << P.pos[p] : 0;
      aU[x] = tp_at<R>(1 << p);
      sU[x] = p < P.kt ? P.col[p] : 0;
    }
  }
  __device__ __forceinline__ uint64_t g(int u) const {
    uint64_t o = gT;
#pragma unroll
    for (int x = 0; x < LV; ++x) o |= ((u >> x) & 1) ? gU[x] : 0;
    return o;
  }
  __device__ __forceinline__ int a(int u) const {
    int o = aT;
#pragma unroll
    for (int x = 0; x < LV; ++x) o ^= ((u >> x) & 1) ? aU[x] : 0;
    return o;
  }
  __device__ __forceinline__ int s(int u) const {
    int o = sT;
#pragma unroll
    for (int x = 0; x < LV; ++x) o ^= ((u >> x) & 1) ? sU[x] : 0;
    return o;
  }
};

// Byte offset of a thread's register block in a round, and of its element j.
template <typename R, int RB>
__device__ __forceinline__ int tp_round_base(const TileRound& rd) {
  int base = threadIdx.x;
#pragma unroll
  for (int x = 0; x < RB; ++x) base = ((base >> rd.r[x]) << (rd.r[x] + 1)) | (base & ((1 << rd.r[x]) - 1));
  return tp_at<R>(base);
}
template <int RB>
__device__ __forceinline__ int tp_round_at(int base, const int* bas, int j) {
#pragma unroll
  for (int x = 0; x < RB; ++x) base ^= ((j >> x) & 1) ? bas[x] : 0;
  return base;
}

// ------------------------------------------------------------- builder ---
// kmax: tile bits; c0: low index bits every tile keeps (row length); rb:
// register bits of a round; merge: two neighbouring rotations on a qubit
// become one operator and nothing goes to D; reverse: the rounds run the
// operators last to first (the backward sweep).
struct PassCfg {
  int kmax, c0, rb;
  bool merge, reverse;
  bool grow = true;  // operators behind a left-out gate may still bring new tile bits
};

template <typename R>
inline std::vector<TilePass> build_passes_as(const qc_gate* gates, int ng, int n, const PassCfg& cfg) {
  struct Item {
    bool cx;
    int q, c, ka, kb, pa, pb;
  };
  std::vector<Item> items;
  for (int i = 0; i < ng; ++i) {
    const qc_gate& g = gates[i];
    if (g.kind == QC_G_CNOT) {
      items.push_back(Item{true, g.q1, g.q0, 0, -1, 0, 0});
    } else if (cfg.merge && i + 1 < ng && g.kind <= QC_G_RZ && gates[i + 1].kind <= QC_G_RZ &&
               gates[i + 1].q0 == g.q0) {
      items.push_back(Item{false, g.q0, 0, g.kind, gates[i + 1].kind, g.param, gates[i + 1].param});
      ++i;
    } else {
      items.push_back(Item{false, g.q0, 0, g.kind, -1, g.kind <= QC_G_RZ ? g.param : -1, -1});
    }
  }
  const int kt = std::min(n, cfg.kmax);
  std::vector<TilePass> out;
  out.reserve(64);
  std::vector<char> done(items.size(), 0);
  std::vector<Item> S, keep;
  std::vector<std::pair<int, int>> cx;  // (control, target) in order
  size_t first = 0;
  while (first < items.size()) {
    uint64_t tile = (1ull << std::min(n, cfg.c0)) - 1, skip = 0, inp = 0;
    bool closed = false;  // no more operators
    int left = 0;         // gates left out
    S.clear();
    cx.clear();
    auto fits = [&](int q) {
      if ((tile >> q) & 1) return true;
      if (__builtin_popcountll(tile) >= kt || (skip && !cfg.grow)) return false;
      tile |= 1ull << q;
      return true;
    };
    // register rounds that S needs so far, in the order it is run
    auto rounds_of = [&](const std::vector<Item>& s) {
      uint64_t set = 0;
      int nr = 1;
      for (size_t k = 0; k < s.size(); ++k) {
        const uint64_t b = 1ull << s[cfg.reverse ? s.size() - 1 - k : k].q;
        if (!(set & b) && __builtin_popcountll(set) >= cfg.rb) set = 0, ++nr;
        set |= b;
      }
      return nr;
    };
    for (size_t i = first; i < items.size(); ++i) {
      if (done[i]) continue;
      const Item& it = items[i];
      const uint64_t b = 1ull << it.q;
      if (it.cx) {
        const uint64_t bc = 1ull << it.c;
        if (!(skip & (b | bc)) && cx.size() < 512 && fits(it.q)) {
          cx.push_back({it.c, it.q});
          inp |= b | bc;
          done[i] = 1;
        } else {
          skip |= b | bc;
          ++left;
        }
      } else {
        bool ok = !closed && !((skip | inp) & b) && S.size() < (size_t)TP_MAXOP && fits(it.q);
        if (ok) {
          S.push_back(it);
          if (S.size() > (size_t)TP_MAXRD && rounds_of(S) > TP_MAXRD) {
            S.pop_back();
            ok = false;
          }
        }
        if (ok) done[i] = 1;
        else skip |= b, closed = cfg.merge, ++left;
      }
      if (left >= TP_LOOK) break;  // planning stays linear in the gates (30000 on three qubits: 40 us a gate without)
      if ((__builtin_popcountll(tile) >= kt || (skip && !cfg.grow)) && (tile & ~skip) == 0) break;
    }
    while (first < items.size() && done[first]) ++first;
    for (int q = 0; q < n && __builtin_popcountll(tile) < kt; ++q) tile |= 1ull << q;

    TilePass P{};
    P.kt = (int16_t)std::max(kt, cfg.rb);
    P.nreal = (int16_t)kt;
    int where[64];
    for (int q = 0; q < n; ++q) {
      if ((tile >> q) & 1) {
        const int p = __builtin_popcountll(tile & ((1ull << q) - 1));
        where[q] = p;
        P.pos[p] = (int8_t)q;
      } else {
        where[q] = -1;
        P.fix[P.nfix++] = (int8_t)q;
      }
    }
    // D: RZ that nothing in S follows on its qubit.  Forward, one alone stays an
    // operator: four multiplications an amplitude, D's phase takes eight
    for (int p = 0; p < TP_MAXK + 3; ++p) P.dp[p] = -1;
    if (!cfg.merge) {
      uint64_t later = 0;
      keep.clear();
      for (size_t k = S.size(); k-- > 0;) {
        const uint64_t b = 1ull << S[k].q;
        if (S[k].ka == QC_G_RZ && !(later & b)) {
          P.dp[where[S[k].q]] = S[k].pa;
          P.has_diag = 1;
        } else {
          keep.push_back(S[k]);
        }
        later |= b;
      }
      std::reverse(keep.begin(), keep.end());
      if (cfg.reverse || S.size() - keep.size() >= 2) {
        S.swap(keep);
      } else {
        for (int p = 0; p < TP_MAXK + 3; ++p) P.dp[p] = -1;
        P.has_diag = 0;
      }
    }
    for (const Item& it : S) P.has_fac |= it.ka != QC_G_RZ;  // operators applied without their factor
    if (cfg.reverse) std::reverse(S.begin(), S.end());
    // register rounds; spare register bits come from the top of the tile
    P.nop = (int16_t)S.size();
    size_t k = 0;
    do {
      TileRound& rd = P.rd[P.nround++];
      rd.op0 = (int8_t)k;
      uint32_t set = 0;
      size_t e = k;
      for (; e < S.size(); ++e) {
        const uint32_t b = 1u << where[S[e].q];
        if (!(set & b) && __builtin_popcount(set) >= cfg.rb) break;
        set |= b;
      }
      rd.op1 = (int8_t)e;
      for (int p = P.kt - 1; p >= 0 && __builtin_popcount(set) < cfg.rb; --p) set |= 1u << p;
      int nr = 0;
      for (int p = 0; p < P.kt; ++p)
        if ((set >> p) & 1) rd.r[nr++] = (int8_t)p;
      for (int x = 0; x < cfg.rb; ++x) rd.bas[x] = (uint16_t)tp_at<R>(1 << rd.r[x]);
      for (; k < e; ++k) {
        const int p = where[S[k].q];
        int bit = 0;
        while (rd.r[bit] != p) ++bit;
        P.op[k] = TileOp{(int8_t)bit, (int8_t)S[k].ka, (int8_t)S[k].kb, (int8_t)p, S[k].pa, S[k].pb};
      }
    } while (k < S.size());
    // P: where the amplitude at a unit vector comes from
    auto back = [&](uint64_t v) {
      for (size_t x = cx.size(); x-- > 0;) v ^= ((v >> cx[x].first) & 1ull) << cx[x].second;
      return v;
    };
    auto tile_part = [&](uint64_t v) {
      int r = 0;
      for (v &= tile; v; v &= v - 1) r |= 1 << where[__builtin_ctzll(v)];
      return r;
    };
    P.has_perm = !cx.empty();
    for (int p = 0; p < P.kt; ++p) P.col[p] = (uint16_t)tp_at<R>(p < kt ? tile_part(back(1ull << P.pos[p])) : 1 << p);
    for (int i = 0; i < P.nfix; ++i) {
      const int m = tile_part(back(1ull << P.fix[i]));
      if (m) {
        P.fc[P.nfc] = P.fix[i];
        P.fm[P.nfc++] = (uint16_t)tp_at<R>(m);
      }
    }
    out.push_back(P);
  }
  return out;
}

// The shortest list over both ways to grow a tile and rows of 2^c0 or half as
// many amplitudes.  A tile that takes in a later layer's qubits can leave the
// passes after it out of step with the layers: 20 qubits, ten layers of
// rotations and a ring on 2^11-amplitude tiles are 41 passes grown greedily
// and 20 on 64-byte rows.
template <typename R>
inline std::vector<TilePass> build_passes(const qc_gate* gates, int ng, int n, const PassCfg& cfg) {
  std::vector<TilePass> best;
  for (int k = 0; k < 4; ++k) {
    PassCfg c = cfg;
    c.c0 -= k >> 1;
    c.grow = !(k & 1);
    std::vector<TilePass> p = build_passes_as<R>(gates, ng, n, c);
    if (k == 0 || p.size() < best.size()) best.swap(p);
    if (n <= cfg.kmax) break;  // one tile holds every qubit
  }
  return best;
}

}  // namespace qc
