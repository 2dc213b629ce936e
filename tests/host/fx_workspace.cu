// Host-only check of the fixed-point workspaces (csrc/lin_fx.cu, csrc/quad_fx.cu,
// from the library): for every N and rules and radial nodes from few to many,
// the bytes that a batch needs never fall as the batch grows, so a buffer
// sized for one batch serves every smaller one.  Prints "ok <cases>" or the
// first batch that needs less than the one before it.  Runs no kernel.
#include <cstdio>
#include <vector>

#include "../../paper_2503_09580_gb300/csrc/lin_fx.h"

namespace lbo {
namespace fx {
#define DECL(n) size_t q_workspace_bytes_##n(int B, int J, const QuadRule& rule);
DECL(16) DECL(24) DECL(32) DECL(48) DECL(64)
}  // namespace fx
}  // namespace lbo

using namespace lbo::fx;

int main() {
  size_t (*const bytes[])(int, int, const QuadRule&) = {q_workspace_bytes_16, q_workspace_bytes_24, q_workspace_bytes_32,
                                                        q_workspace_bytes_48, q_workspace_bytes_64};
  const int size[] = {16, 24, 32, 48, 64};
  int cases = 0;
  for (int n = 0; n < 5; ++n)
    for (int J : {1, 5, 9, 17, 32, 64, 256})
      for (int p : {1, 2, 4, 16, 32}) {
        std::vector<int> begin(1, 0);  // rings of 2 p nodes in fours, their middle pair in twos
        for (int a = 0; a < p; ++a)
          for (int left = 2 * p; left > 0; left -= 4) begin.push_back(begin.back() + (left < 4 ? left : 4));
        QuadRule rule{};
        rule.M = 2 * p * p;
        rule.class_begin = begin.data();
        rule.classes = (int)begin.size() - 1;
        size_t before = 0;
        for (int B = 1; B <= 2500; B += B < 700 ? 1 : 31) {
          const size_t now = bytes[n](B, J, rule);
          if (now < before) {
            std::printf("N = %d, J = %d, p = %d: batch %d needs %zu bytes, a smaller one %zu\n", size[n], J, p, B, now, before);
            return 1;
          }
          before = now;
          ++cases;
        }
      }
  std::printf("ok %d\n", cases);
  return 0;
}
