// Planning time of circuits (circuit_passes.cuh, host code): ten times the
// gates may take ten times as long, not a hundred.  Gates on three of 20 qubits,
// which leave the tile unfilled and every later gate in view.
#include <chrono>
#include <cstdio>
#include <vector>

#include "../paper_0902_0699_gb300/csrc/circuit_passes.cuh"

using namespace qc;

static double us_a_gate(int count, const PassCfg& cfg) {
  std::vector<qc_gate> g;
  for (int i = 0; (int)g.size() < count; ++i) {
    g.push_back({QC_G_RX, i % 3, 0, (int)g.size()});
    g.push_back({QC_G_RY, (i + 1) % 3, 0, (int)g.size()});
    g.push_back({QC_G_CNOT, i % 2, 1 - i % 2, 0});
  }
  double best = 1e30;
  for (int rep = 0; rep < 3; ++rep) {
    const auto t = std::chrono::steady_clock::now();
    const std::vector<TilePass> p = build_passes<double>(g.data(), (int)g.size(), 20, cfg);
    const double us = std::chrono::duration<double, std::micro>(std::chrono::steady_clock::now() - t).count();
    if (p.empty()) return 1e30;
    best = us < best ? us : best;
  }
  return best / (double)g.size();
}

int main() {
  const PassCfg fwd{12, 3, 3, false, false}, bwd{11, 3, 3, false, true};
  for (const PassCfg& c : {fwd, bwd}) {
    const double a = us_a_gate(3000, c), b = us_a_gate(30000, c);
    if (b > 4 * a) {
      std::printf("%.2f us a gate for 3000 gates, %.2f for 30000\n", a, b);
      return 1;
    }
  }
  std::puts("ok");
  return 0;
}
