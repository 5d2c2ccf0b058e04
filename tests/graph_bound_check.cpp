// Checks of the bound on a handle's graphs (internal.hpp), compiled and run by
// test_graph_bound_cpu.py: however many pairs of vectors are solved for, by whatever
// methods, no more than kMaxGraphs stay.
#include <cstdio>

#include "internal.hpp"

static int drops = 0;
namespace helm {
void drop_graphs(helm_csr A) {
  A->graphs.clear();
  ++drops;
}
}  // namespace helm

int main() {
  static char buf[4096];
  helm_csr_s A;
  size_t most = 0;
  for (int k = 0; k < 1000; ++k) {
    const size_t more = k % 3 == 0 ? 2 : 1;  // mixed precision adds two at a time
    helm::bound_graphs(&A, more);
    for (size_t q = 0; q < more; ++q) A.graphs[std::make_tuple(buf + k, buf + 2 * k, static_cast<int>(2 * k + q))] = {};
    most = A.graphs.size() > most ? A.graphs.size() : most;
  }
  const bool ok = most == helm::kMaxGraphs && drops > 50 && drops < 1000;
  std::printf(ok ? "ok\n" : "FAILED: %zu graphs, %d drops\n", most, drops);
  return ok ? 0 : 1;
}
