// k_bwd_polish on host threads: two agents that do not move, two steps, one pair.
// argv: what (0: a halfspace is violated, 1: a free input is outside its box, 2: an
// active halfspace has a negative multiplier), the held warp and its barrier.
// Prints the flags hmask[0..1], the working sets and pchg.
#include "tadmm_device.cuh"
#include "tadmm_adjoint.cuh"

#include <cstdio>
#include <cstdlib>

using namespace tadmm;

int main(int argc, char** argv) {
  (void)argc;
  const int what = atoi(argv[1]);
  constexpr int N = 2, T = 2, NX = 4, NU = 2, DP = 2;
  ScenMeta s{};
  s.N = N;
  s.T = T;
  s.P = 1;
  s.d = 1.0;
  s.rho = 1.0;
  // positions 2 apart, or 0.5 at the second step
  double X[N * (T + 1) * NX] = {}, U[N * T * NU] = {}, G[N * T * NU] = {}, force[N * T * DP] = {};
  for (int t = 0; t <= T; ++t) X[((T + 1) + t) * NX] = (what == 0 && t == T) ? -0.5 : -2.0;
  if (what == 1) U[(1 * T + 1) * NU] = 1.5;   // agent 1, second step, first input: above the box
  const double model[NX * NX + NX * NU + 2 * NU] = {1, 0, .1, 0, 0, 1, 0, .1, 0, 0, 1, 0, 0, 0, 0, 1,
                                                    .005, 0, 0, .005, .1, 0, 0, .1, -1, -1, 1, 1};
  const double zero[N * NX] = {}, one[N * NU] = {1, 1, 1, 1}, a[T * DP] = {1, 0, 1, 0};
  const int32_t pairs[1] = {0 | (1 << 16)};
  uint8_t hm[T] = {};
  uint16_t Wb[N * T] = {};
  int32_t act[T] = {}, pchg[1] = {-1};
  double mu[4 * T] = {};
  BwdScen bs{};
  if (what == 2) {
    bs.m = 1;
    hm[1] = 1;
    act[0] = 1;
    mu[0] = -3.0;
  }
  Dev<double> D{};
  D.meta = &s;
  D.pairs = pairs;
  D.model = model;
  D.Qd = D.Qfd = zero;   // no costates but the inputs' own
  D.Rd = one;
  D.x_ref = zero;
  D.a = a;
  BwdDev<double> B{};
  B.bs = &bs;
  B.act = act;
  B.vec = mu;
  B.force = force;
  B.Xp = X;
  B.Up = U;
  B.Wu = G;
  B.Wb = Wb;
  B.hmask = hm;
  B.pchg = pchg;
  B.kkt_tol = 1e-9;
  host_cta::hold(atoi(argv[2]), atoi(argv[3]));
  host_cta::run(128, [&] { k_bwd_polish<double, NX, NU, DP, true>(D, B); });
  printf("%d %d", hm[0], hm[1]);
  for (uint16_t w : Wb) printf(" %d", w);
  printf(" %d\n", pchg[0]);
  return 0;
}
