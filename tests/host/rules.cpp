// The host's launch rules on batches given as argv: "tail" sm_count N T count [N T count ...]
// prints whether graph mode runs one tail CTA per scenario; "threads" sm_count r128 r64 r32
// relaxed N T count [N T count ...], a group each, prints the threads per CTA.
#include "tadmm_impl.h"

#include <cstdio>
#include <cstring>

namespace tadmm {
int set_error(int code, const std::string&) { return code; }
}  // namespace tadmm

int main(int argc, char** argv) {
  const int sm = atoi(argv[2]);
  if (!strcmp(argv[1], "tail")) {
    std::vector<tadmm::ScenMeta> scen;
    for (int k = 3; k + 2 < argc; k += 3)
      for (int c = atoi(argv[k + 2]); c > 0; --c) {
        tadmm::ScenMeta m{};
        m.N = atoi(argv[k]);
        m.T = atoi(argv[k + 1]);
        m.P = m.N * (m.N - 1) / 2;
        scen.push_back(m);
      }
    printf("%d\n", (int)tadmm::tail_per_scenario(scen, sm));
  }
  if (!strcmp(argv[1], "threads")) {
    const int resident[3] = {atoi(argv[3]), atoi(argv[4]), atoi(argv[5])};
    tadmm::GroupLoad load;
    int groups = 0;
    for (int k = 7; k + 2 < argc; k += 3) {
      const int N = atoi(argv[k]), T = atoi(argv[k + 1]);
      for (int c = atoi(argv[k + 2]); c > 0; --c, ++groups) load.add(N > tadmm::kGroupMax, tadmm::group_work(T, N * (N - 1) / 2));
    }
    printf("%d\n", tadmm::default_threads(load, groups, atoi(argv[6]), sm, resident));
  }
  return 0;
}
