// ratio_scan on 32 host threads against ratio_test in index order, on the same
// operands: argv[1] a seed, or "near" for an input closer to its bound than float32
// can tell from 0, whose step is as small, beside one that blocks first.  Prints the
// number of agents compared; exits 1 on the first that differs.
#include "tadmm_device.cuh"

#include <cstdio>
#include <cstdlib>
#include <random>

using namespace tadmm;

constexpr int NX = 4, NU = 2, DP = 2;

struct Agent {
  Model<double, NX, NU> M{};
  std::vector<double> U, Us;
  std::vector<uint16_t> W;
  int T;
};

static EqpScan<double> fresh() {
  EqpScan<double> o{};
  o.anum = o.aden = 1;
  o.blk = -1;
  return o;
}

static AgentCtx<double, NX, NU, DP> ctx(Agent& a) {
  AgentCtx<double, NX, NU, DP> A{};
  A.M = &a.M;
  A.N = 1;
  A.T = a.T;
  A.Wm = a.W.data();
  A.U = a.U.data();
  A.Us = a.Us.data();
  return A;
}

static bool same(Agent& a, int at) {
  EqpScan<double> want = fresh(), got[32];
  for (auto& g : got) g = fresh();
  const auto A = ctx(a);
  ratio_test<double, NX, NU, DP>(A, want);
  host_cta::run(32, [&] {
    const int lane = threadIdx.x;
    ratio_scan<double, NX, NU, DP>(A, lane == 5, got[lane]);
  });
  const EqpScan<double>& g = got[5];
  const bool ok = g.blk == want.blk && (want.blk < 0 || (g.anum == want.anum && g.aden == want.aden && g.bside == want.bside));
  if (!ok)
    printf("agent %d: blocks at %d, %g / %g, side %d; in index order %d, %g / %g, side %d\n", at, g.blk, g.anum, g.aden,
           g.bside, want.blk, want.anum, want.aden, want.bside);
  return ok;
}

int main(int, char** argv) {
  if (!strcmp(argv[1], "near")) {
    int at = 0;
    for (double tiny : {1e-38, 3e-39, 1e-45, 5e-324})
      for (double step : {1.5 * tiny, 4e-38, 1e-20, 1e-9, 1e-3}) {
        Agent a;
        a.T = 3;
        for (int c = 0; c < NU; ++c) a.M.umax[c] = 1.0;   // the box [0, 1]
        a.U = {0.5, tiny, 0.25, 0.5, 0.5, 0.5};
        a.Us = {0.75, tiny - step, -0.5, 0.5, 0.5, 0.5};   // input 2 blocks at a third of the step
        a.W.assign(3, 0);
        if (!same(a, at++)) return 1;
      }
    printf("%d\n", at);
    return 0;
  }
  std::mt19937_64 rng(atoll(argv[1]));
  auto uni = [&] { return std::uniform_real_distribution<double>(0, 1)(rng); };
  const int n = 40;
  for (int at = 0; at < n; ++at) {
    Agent a;
    a.T = 1 + (int)(uni() * 130);   // below and above the 128 inputs that stay in registers
    for (int c = 0; c < NU; ++c) {
      a.M.umin[c] = uni() < 0.5 ? 0.0 : -uni();
      a.M.umax[c] = a.M.umin[c] + uni();
    }
    a.W.resize(a.T);
    a.U.resize(a.T * NU);
    a.Us.resize(a.T * NU);
    for (int t = 0; t < a.T; ++t) {
      a.W[t] = uni() < 0.2 ? 1 : (uni() < 0.1 ? 0x200 : 0);
      for (int c = 0; c < NU; ++c) {
        const double span = a.M.umax[c] - a.M.umin[c];
        // distances from a bound and steps over the whole exponent range, some equal
        const double d = uni() < 0.2 ? 0.0 : span * exp2(-(uni() < 0.5 ? 4 : 200) * uni());
        const bool low = uni() < 0.5;
        double u = low ? a.M.umin[c] + d : a.M.umax[c] - d;
        double s = uni() < 0.3 ? d : span * exp2(-(uni() < 0.5 ? 4 : 200) * uni());
        if (uni() < 0.1) s = uni() < 0.5 ? 0.0 : s * (uni() < 0.5 ? 1e19 : 1e300);
        a.U[t * NU + c] = u;
        a.Us[t * NU + c] = low ? u - s : u + s;
      }
    }
    if (!same(a, at)) return 1;
  }
  printf("%d\n", n);
  return 0;
}
