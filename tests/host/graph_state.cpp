// The graph mode's device blocks under failing allocations: with the n-th failing, the
// call reports it, keeps nothing, and the next call allocates all of them.  Prints the
// number of allocations.
#include "tadmm_impl.h"

#include <cstdio>

namespace tadmm {
int set_error(int code, const std::string&) { return code; }
}  // namespace tadmm

static bool all(const tadmm_handle& h, bool set) {
  void* const p[] = {h.gs_iter, h.gs_active, h.gs_fail, h.gs_rb, h.gs_sb, h.gs_on, h.gs_done, h.gs_blk};
  for (void* q : p)
    if ((q != nullptr) != set) return false;
  return true;
}

int main() {
  int n = 1;
  for (int fail = 0; fail < n; ++fail) {
    tadmm_handle h;
    h.n_scen = 3;
    h.n_gblk = 4;
    h.tot_on = 100;
    host_cta::allocations = 0;
    host_cta::fail_at = fail;
    if (tadmm::graph_state_alloc(&h) != TADMM_ENOMEM || !all(h, false) || h.gs_ready || !host_cta::blocks.empty()) return 1;
    host_cta::allocations = 0;
    host_cta::fail_at = -1;
    if (tadmm::graph_state_alloc(&h) != TADMM_OK || !all(h, true)) return 2;
    n = host_cta::allocations;
    if ((int)host_cta::blocks.size() != n) return 3;
    tadmm::graph_state_free(&h);
    if (!all(h, false) || !host_cta::blocks.empty()) return 4;
  }
  printf("%d\n", n);
  return 0;
}
