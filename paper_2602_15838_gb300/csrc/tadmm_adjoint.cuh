// Implicit differentiation of the converged problem (K-d).
//
// At the final active set of a solve (inputs held at a bound by the last
// x-update, and halfspaces whose projection step theta exceeds theta_eps), the
// centralized QP of Eq. (1) with linearized halfspaces reduces to an
// equality-constrained QP.  Its KKT system is differentiated implicitly
// (OptNet-style): per agent, a block-tridiagonal LQ problem solved by the
// Riccati recursion of Sec. IV.B on the global Hessian (2Q, 2Q_T, 2R, no ADMM
// penalty); the coupling through the active halfspaces G z = d is eliminated
// with the dense Schur complement S = G Psi G' of the per-agent position
// responses Psi.  The polished primal solution and the adjoint of a loss
// gradient dl/dX follow from two block solves each; the parameter gradients
// are closed forms in the polished solution and the adjoint.
//
// Active rows may be linearly dependent (several halfspaces through the same
// agents and step, or rows whose positions are fixed by inputs held at a
// bound); S is then singular and the multipliers are not unique.  S is
// factored with diagonal pivoting up to its numerical rank, and the
// multipliers are the least-squares solution of S mu = b in the factor's
// range: the polished point then satisfies the active rows with their
// right-hand side projected onto the range of the rows (exactly the rows
// when they are consistent), and the gradient is that of this solution map.
#pragma once

#include <climits>

namespace tadmm {

struct BwdScen {
  int64_t psi_off;   // per-agent responses [N][T][DP][T][DP]
  int64_t s_off;     // Schur complement [m][m], then the normal matrix [m][m]
  int64_t v_off;     // vectors [4][m]: the two multipliers, two blocks of scratch
  int32_t m;         // active halfspaces
  int32_t pad;
};

template <typename F>
struct BwdDev {
  const BwdScen* bs;
  int32_t* act;              // per scenario at ps_off: active pair-step indices q (t-major)
  int32_t* piv;              // per scenario at ps_off: pivot order of the Schur factorization
  int32_t* act_cnt;          // [n_scen]
  unsigned long long* amask; // [agents] bit t-1 set when the agent has an active halfspace at t
  F* psi;
  F* kks;                    // [agents][DP][T][NU] affine gains of the in-flight solves
  F* pos0;                   // [agent-steps][DP] base positions, then adjoint base positions
  F* force;                  // [agent-steps][DP] coupling forces G' mu on each agent
  F* S;
  F* vec;
  F* Xp;                     // polished states, caller layout [agent-state][NX]
  F* Up;                     // polished inputs, caller layout [agent-step][NU]
  F* Wx;                     // adjoint states, caller layout
  F* Wu;                     // adjoint inputs, caller layout
  const double* gX;          // dl/dX, caller layout (float64)
  double* gQ;                // [agents][NX]
  double* gQf;               // [agents][NX]
  double* gR;                // [agents][NU]
  double* gGoal;             // [agents][NX]
  int32_t* bstatus;          // [n_scen]
  int32_t* ndep;             // [n_scen] active rows found dependent (m - rank)
  uint8_t* hmask;            // [pair-steps] active halfspaces (scenario layout [T][P] at ps_off)
  uint16_t* Wb;              // [agent-steps] inputs held at a bound (layout of Wm)
  int32_t* pchg;             // [n_scen] polishing: the active set changed in this round
  int32_t adjoint;           // 0: stop after the polished primal point (polishing rounds)
  double kkt_tol;            // polishing: relative tolerance of the KKT conditions
  double theta_eps;
  double rank_tol;           // relative pivot size below which a row counts as dependent
  int64_t kk_stride;         // Tmax * NU
};

// Active set of the last solve's final iterate: halfspaces whose projection
// step theta exceeds theta_eps and the inputs the last x-update held at a
// bound (one CTA per scenario).
template <typename F, int NX, int NU, int DP>
__global__ void k_bwd_init(Dev<F> D, BwdDev<F> B) {
  const int sc = blockIdx.x;
  const ScenMeta s = D.meta[sc];
  const F* th = D.theta + (size_t)(D.cur_lvl[sc] >> 1) * D.tot_ps + s.ps_off;
  const int64_t PT = (int64_t)s.P * s.T, NT = (int64_t)s.N * s.T;
  for (int64_t q = threadIdx.x; q < PT; q += blockDim.x) B.hmask[s.ps_off + q] = double(th[q]) > B.theta_eps ? 1 : 0;
  for (int64_t e = threadIdx.x; e < NT; e += blockDim.x) B.Wb[s.as_off + e] = D.Wm[s.as_off + e];
}

constexpr int kBwdThreads = 256;  // threads of a scenario's CTA here

// Ordered compaction of the active halfspaces of one scenario (one CTA).
template <typename F, int NX, int NU, int DP>
__global__ void __launch_bounds__(kBwdThreads) k_bwd_count(Dev<F> D, BwdDev<F> B) {
  constexpr int NW = kBwdThreads / 32;
  __shared__ int part[NW];
  const int sc = blockIdx.x, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const ScenMeta s = D.meta[sc];
  const uint8_t* hm = B.hmask + s.ps_off;
  for (int i = tid; i < s.N; i += kBwdThreads) B.amask[s.agent_off + i] = 0ull;
  __syncthreads();
  const int64_t PT = (int64_t)s.P * s.T;
  int count = 0;
  for (int64_t base = 0; base < PT; base += kBwdThreads) {
    const int64_t q = base + tid;
    const bool on = q < PT && hm[q] != 0;
    const unsigned ball = __ballot_sync(0xffffffffu, on);
    if (lane == 0) part[w] = __popc(ball);
    __syncthreads();
    int pos = count + __popc(ball & ((1u << lane) - 1u));
#pragma unroll
    for (int v = 0; v < NW; ++v) {
      if (v < w) pos += part[v];
      count += part[v];
    }
    if (on) {
      B.act[s.ps_off + pos] = (int32_t)q;
      const int tm1 = (int)(q / s.P), pair = (int)(q - (int64_t)tm1 * s.P);
      const int pk = D.pairs[s.pair_off + pair];
      atomicOr(&B.amask[s.agent_off + (pk & 0xFFFF)], 1ull << tm1);
      atomicOr(&B.amask[s.agent_off + (pk >> 16)], 1ull << tm1);
    }
    __syncthreads();
  }
  if (tid == 0) B.act_cnt[sc] = count;
}

// Riccati solve of one agent's equality-constrained LQ problem with the cached
// factors of its working set: linear term lin(t, r) on x_t (t = 1..T), initial
// state x0, inputs of the working set at their bounds (at_bounds) or at zero.
// Emits every state through outx(t, x) and every input through outu(t, u).
template <typename F, int NX, int NU, class Lin, class OutX, class OutU>
__device__ void lq_solve(const Model<F, NX, NU>& Mo, const F* cache, const uint16_t* Wm, int N, int i, int T,
                         Lin lin, const F (&x0)[NX], bool at_bounds, F* kk, OutX outx, OutU outu) {
  using CL = CacheLayout<NX, NU>;
  auto C = [&](int t, int e) -> F { return cache[((size_t)t * CL::E + e) * N + i]; };
  F pn[NX];
#pragma unroll
  for (int r = 0; r < NX; ++r) pn[r] = lin(T, r);
  for (int t = T - 1; t >= 0; --t) {
    const uint16_t mask = Wm[(size_t)t * N + i];
    F Pcp[NX];
#pragma unroll
    for (int r = 0; r < NX; ++r) Pcp[r] = pn[r];
    if (mask && at_bounds) {
      F cv[NX];
#pragma unroll
      for (int r = 0; r < NX; ++r) {
        F acc = 0;
#pragma unroll
        for (int c = 0; c < NU; ++c) {
          if (mask & (1u << c)) acc = fma(Mo.B[r][c], Mo.umin[c], acc);
          else if (mask & (0x100u << c)) acc = fma(Mo.B[r][c], Mo.umax[c], acc);
        }
        cv[r] = acc;
      }
#pragma unroll
      for (int r = 0; r < NX; ++r) {
        F acc = Pcp[r];
#pragma unroll
        for (int c = 0; c < NX; ++c) acc = fma(C(t + 1, CL::P + r * NX + c), cv[c], acc);
        Pcp[r] = acc;
      }
    }
    F sv[NU], kv[NU], L[NU][NU];
#pragma unroll
    for (int a = 0; a < NU; ++a) {
      F acc = 0;
#pragma unroll
      for (int r = 0; r < NX; ++r) acc = fma(Mo.B[r][a], Pcp[r], acc);
      sv[a] = (mask & (0x101u << a)) ? F(0) : acc;
#pragma unroll
      for (int b = 0; b < NU; ++b) L[a][b] = C(t, CL::L + (b <= a ? a * NU + b : b * NU + a));
    }
    neg_sinv<F, NU>(L, sv, kv);
#pragma unroll
    for (int a = 0; a < NU; ++a) kk[t * NU + a] = kv[a];
    if (t >= 1) {
#pragma unroll
      for (int r = 0; r < NX; ++r) {
        F acc = lin(t, r);
#pragma unroll
        for (int k = 0; k < NX; ++k) acc = fma(Mo.A[k][r], Pcp[k], acc);
#pragma unroll
        for (int k = 0; k < NU; ++k) acc = fma(C(t, CL::K + k * NX + r), sv[k], acc);
        pn[r] = acc;
      }
    }
  }
  F xv[NX];
#pragma unroll
  for (int r = 0; r < NX; ++r) xv[r] = x0[r];
  outx(0, xv);
  for (int t = 0; t < T; ++t) {
    const uint16_t mask = Wm[(size_t)t * N + i];
    F uv[NU];
#pragma unroll
    for (int a = 0; a < NU; ++a) {
      if (mask & (1u << a)) uv[a] = at_bounds ? Mo.umin[a] : F(0);
      else if (mask & (0x100u << a)) uv[a] = at_bounds ? Mo.umax[a] : F(0);
      else {
        F acc = kk[t * NU + a];
#pragma unroll
        for (int c = 0; c < NX; ++c) acc = fma(C(t, CL::K + a * NX + c), xv[c], acc);
        uv[a] = acc;
      }
    }
    F xn[NX];
#pragma unroll
    for (int r = 0; r < NX; ++r) {
      F acc = 0;
#pragma unroll
      for (int c = 0; c < NX; ++c) acc = fma(Mo.A[r][c], xv[c], acc);
#pragma unroll
      for (int c = 0; c < NU; ++c) acc = fma(Mo.B[r][c], uv[c], acc);
      xn[r] = acc;
    }
    outu(t, uv);
    outx(t + 1, xn);
#pragma unroll
    for (int r = 0; r < NX; ++r) xv[r] = xn[r];
  }
}

// lq_solve for one axis of the double integrator, on the axis words of the factor
// cache (tadmm_axis.cuh): the same values without the zeros between the axes.
// The linear term starts at step tl (it is zero after it).  kk(t) is a word of
// scratch per stage; outx(t, position, velocity), outu(t, u).
template <typename F, int NX, int NU, class Lin, class Kk, class OutX, class OutU>
__device__ __forceinline__ void lq_axis(const Model<F, NX, NU>& Mo, const F* cache, const uint16_t* Wm, int N, int i,
                                        int T, int c, int tl, Lin lin, F xp, F xv, bool at_bounds, Kk kk, OutX outx,
                                        OutU outu) {
  using L = AxisCache;
  constexpr int DP = NU;
  // a11 = 1, read so that a product in the linear term stays rounded
  const F a11 = Mo.A[0][0], dt = Mo.A[0][DP], b1 = Mo.B[0][0], b2 = Mo.B[DP][0];
  auto C = [&](int t, int w) -> F { return cache[((size_t)(t * L::E + w) * DP + c) * N + i]; };
  const std::true_type pos{};   // compile-time, so that a term of the positions only joins their product
  const std::false_type vel{};
  F pp = lin(tl, c, pos), pv = lin(tl, DP + c, vel);
  for (int t = tl - 1; t >= 0; --t) {
    const uint32_t mask = Wm[(size_t)t * N + i];
    const bool hd = (mask >> c) & 0x101u;
    F qp = pp, qv = pv;  // P_{t+1} B u_held + p_{t+1}
    if (hd && at_bounds) {
      const F ub = ((mask >> c) & 1u) ? Mo.umin[c] : Mo.umax[c], cp = b1 * ub, cv = b2 * ub;
      qp = fma(C(t + 1, L::PV), cv, fma(C(t + 1, L::PP), cp, qp));
      qv = fma(C(t + 1, L::VV), cv, fma(C(t + 1, L::PV), cp, qv));
    }
    const F sv = hd ? F(0) : fma(b2, qv, b1 * qp);
    kk(t) = -(C(t, L::SI) * sv);
    if (t >= 1) {
      pp = fma(a11, qp, lin(t, c, pos));
      pv = fma(a11, qv, fma(dt, qp, lin(t, DP + c, vel)));
      if (!hd) {
        pp = fma(C(t, L::G1), sv, pp);
        pv = fma(C(t, L::G2), sv, pv);
      }
    }
  }
  outx(0, xp, xv);
  for (int t = 0; t < T; ++t) {
    const uint32_t mask = Wm[(size_t)t * N + i];
    F u = F(0);
    if (!((mask >> c) & 0x101u)) u = fma(C(t, L::G2), xv, fma(C(t, L::G1), xp, t < tl ? F(kk(t)) : F(0)));
    else if (at_bounds) u = ((mask >> c) & 1u) ? Mo.umin[c] : Mo.umax[c];
    xp = fma(b1, u, fma(dt, xv, xp));
    xv = fma(b2, u, xv);
    outu(t, u);
    outx(t + 1, xp, xv);
  }
}

// Largest value of the CTA and the lowest index it has (kBwdThreads threads).
template <typename F>
__device__ __forceinline__ void cta_argmax(F& v, int& i, F* red_v, int* red_i) {
  constexpr unsigned FULL = 0xffffffffu;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const F v2 = shfl_f(v, (threadIdx.x & 31) ^ o);
    const int i2 = __shfl_xor_sync(FULL, i, o);
    if (v2 > v || (v2 == v && i2 < i)) { v = v2; i = i2; }
  }
  if ((threadIdx.x & 31) == 0) {
    red_v[threadIdx.x >> 5] = v;
    red_i[threadIdx.x >> 5] = i;
  }
  __syncthreads();
  v = red_v[0];
  i = red_i[0];
#pragma unroll
  for (int w = 1; w < kBwdThreads / 32; ++w) {
    const F v2 = red_v[w];
    const int i2 = red_i[w];
    if (v2 > v || (v2 == v && i2 < i)) { v = v2; i = i2; }
  }
  __syncthreads();
}

// The dense algebra below keeps, for every entry, the operations and the order
// of the plain definitions (right-looking updates in step order, row sums in
// column order) and changes only who does them and from where they read.  One
// CTA works on a scenario's matrix of a few hundred rows, which is in L2 but not
// in L1, so what bounds the plain forms is the latency of one dependent load per
// multiplication: they are left-looking here, each thread with one row whose
// entries of a step's column it sums up from consecutive words.
// With the solves by axis below: 12 polishing rounds and a backward pass over 64
// scenarios of 16 agents 72.9 -> 38.2 ms, 4 rounds over 9 scenarios of 20 agents
// (several hundred rows) 489 -> 108 ms.  What is left in the former (48 to 152 active
// rows, 1.3 ms of a CTA a round): 45 % the pivoted factor, whose every step waits for
// its barriers and its sums' loads, and 30 % the substitutions, of which warp_backward
// is a chain of m^2 / 2 multiply-adds of 68 cycles.

// Rank-revealing Cholesky of the positive semidefinite m x m matrix S (full
// symmetric storage) by one CTA, with diagonal pivoting: step k takes the
// largest remaining diagonal entry (ties to the lowest position) and stops
// when it is not above rank_tol times the largest diagonal entry of S.  The
// pivot order goes to piv; column c of the factor replaces row piv[c] of S, by
// the rows' own numbers.  d [m]: scratch.  Returns the rank (same in every thread).
template <typename F>
__device__ int cta_pivoted_cholesky(F* S, int m, int* piv, F* d, F rank_tol) {
  __shared__ F red_v[kBwdThreads / 32];
  __shared__ int red_i[kBwdThreads / 32];
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int r = tid; r < m; r += nt) {
    piv[r] = r;
    d[r] = S[(size_t)r * m + r];
  }
  __syncthreads();
  F dref = F(0);
  for (int k = 0; k < m; ++k) {
    F v = F(-1);
    int j = m;
    for (int p = k + tid; p < m; p += nt) {
      const F w = d[piv[p]];
      if (w > v) { v = w; j = p; }
    }
    cta_argmax(v, j, red_v, red_i);
    if (k == 0) dref = v;
    if (j >= m || !(v > rank_tol * dref)) return k;
    const int pk = piv[j], pj = piv[k];
    const F lkk = sqrt_(v);
    F* const col = S + (size_t)pk * m;
    for (int p = k + 1 + tid; p < m; p += nt) {
      const int r = p == j ? pj : piv[p];
      F acc = col[r];
      int c = 0;
      for (; c + 4 <= k; c += 4) {
        F a[4], b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const F* const q = S + (size_t)piv[c + u] * m;
          a[u] = q[r];
          b[u] = q[pk];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) acc = fma(-a[u], b[u], acc);
      }
      for (; c < k; ++c) {
        const F* const q = S + (size_t)piv[c] * m;
        acc = fma(-q[r], q[pk], acc);
      }
      const F l = acc / lkk;
      col[r] = l;
      d[r] = fma(-l, l, d[r]);
    }
    __syncthreads();
    if (tid == 0) {
      col[pk] = lkk;
      piv[j] = pj;
      piv[k] = pk;
    }
    __syncthreads();
  }
  return m;
}

// The factor by position: Q[c m + p] = L(p, c) for p >= c, from S as
// cta_pivoted_cholesky leaves it.
template <typename F>
__device__ void cta_by_position(const F* S, int m, const int* piv, int rank, F* Q) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int c = w; c < rank; c += nw) {
    const F* const col = S + (size_t)piv[c] * m;
    for (int p = c + lane; p < m; p += 32) Q[(size_t)c * m + p] = col[piv[p]];
  }
  __syncthreads();
}

// In-place Cholesky of the n x n SPD matrix M (full symmetric storage) by one
// CTA: column c of the factor replaces row c from the diagonal on.  Sets *s_bad on
// a non-positive pivot (and goes on with 1 in its place).
template <typename F>
__device__ void cta_cholesky(F* M, int n, int* s_bad) {
  const int tid = threadIdx.x, nt = blockDim.x;
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    F* const col = M + (size_t)k * n;
    for (int r = k + tid; r < n; r += nt) {
      F acc = col[r];
      int c = 0;
      for (; c + 4 <= k; c += 4) {
        F a[4], b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          a[u] = M[(size_t)(c + u) * n + r];
          b[u] = M[(size_t)(c + u) * n + k];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) acc = fma(-a[u], b[u], acc);
      }
      for (; c < k; ++c) acc = fma(-M[(size_t)c * n + r], M[(size_t)c * n + k], acc);
      col[r] = acc;
    }
    __syncthreads();
    const F dkk = col[k];
    if (!(dkk > F(0)) && tid == 0) *s_bad = 1;
    const F lkk = sqrt_(dkk > F(0) ? dkk : F(1));
    __syncthreads();
    for (int r = k + tid; r < n; r += nt) col[r] = r == k ? lkk : col[r] / lkk;
    __syncthreads();
  }
}

// Normal matrix M = L'L (rank x rank) of a rank-deficient factor (by position)
// and its Cholesky factor, by one CTA (nothing to do when rank = m).  Sets *s_bad
// if M is not positive definite.  Tiles of 32 x 32 entries, their rows' columns
// staged 32 at a time; the entries of L above its diagonal count as zeros.
template <typename F>
__device__ void cta_ls_prepare(const F* Q, int m, int rank, F* M, int* s_bad) {
  if (rank == m || rank == 0) return;
  __shared__ F ta[32][33], tb[32][33];
  constexpr int NR = 32 / (kBwdThreads / 32);  // entries per thread
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5, ny = kBwdThreads / 32;
  for (int a0 = 0; a0 < rank; a0 += 32)
    for (int b0 = 0; b0 <= a0; b0 += 32) {
      F acc[NR];
#pragma unroll
      for (int u = 0; u < NR; ++u) acc[u] = F(0);
      for (int i0 = a0; i0 < m; i0 += 32) {
        const int i = i0 + x;
#pragma unroll
        for (int u = 0; u < NR; ++u) {
          const int a = a0 + y + u * ny, b = b0 + y + u * ny;
          ta[y + u * ny][x] = (a < rank && i < m && i >= a) ? Q[(size_t)a * m + i] : F(0);
          tb[y + u * ny][x] = (b < rank && i < m && i >= b) ? Q[(size_t)b * m + i] : F(0);
        }
        __syncthreads();
#pragma unroll 8
        for (int i2 = 0; i2 < 32; ++i2)
#pragma unroll
          for (int u = 0; u < NR; ++u) acc[u] = fma(ta[y + u * ny][i2], tb[x][i2], acc[u]);
        __syncthreads();
      }
#pragma unroll
      for (int u = 0; u < NR; ++u) {
        const int a = a0 + y + u * ny, b = b0 + x;
        if (a < rank && b <= a) {
          M[(size_t)a * rank + b] = acc[u];
          M[(size_t)b * rank + a] = acc[u];
        }
      }
    }
  cta_cholesky(M, rank, s_bad);
}

// x <- L^{-1} x for the n x n lower triangle L(r, c) = Q[c ld + r], by one warp:
// each solved entry is taken out of all later rows (the row sums' own order).
template <typename F>
__device__ void warp_forward(const F* Q, int ld, int n, F* x) {
  const int lane = threadIdx.x & 31;
  for (int k = 0; k < n; ++k) {
    const F* const col = Q + (size_t)k * ld;
    const F xk = x[k] / col[k];
    __syncwarp();
    if (lane == 0) x[k] = xk;
    for (int r = k + 1 + lane; r < n; r += 32) x[r] = fma(-col[r], xk, x[r]);
    __syncwarp();
  }
}

// x <- L^{-T} x, by one warp.  A row's sum runs over the later rows in
// increasing order, so it starts with the one that was solved last and is one
// chain of multiply-adds; the lanes load its operands 32 at a time, ahead.
template <typename F>
__device__ void warp_backward(const F* Q, int ld, int n, F* x) {
  const int lane = threadIdx.x & 31;
  for (int r = n - 1; r >= 0; --r) {
    const F* const col = Q + (size_t)r * ld;
    F v = x[r];
    F q = r + 1 + lane < n ? col[r + 1 + lane] : F(0), y = r + 1 + lane < n ? x[r + 1 + lane] : F(0);
    for (int k0 = r + 1; k0 < n; k0 += 32) {
      const F qc = q, yc = y;
      const int kn = k0 + 32 + lane;
      q = kn < n ? col[kn] : F(0);
      y = kn < n ? x[kn] : F(0);
      const int cnt = min(32, n - k0);
#pragma unroll 4
      for (int l = 0; l < cnt; ++l) v = fma(-shfl_f(qc, l), shfl_f(yc, l), v);
    }
    v = v / col[r];
    __syncwarp();
    if (lane == 0) x[r] = v;
    __syncwarp();
  }
}

// Least-squares solution of S lambda = b within the range of the pivoted factor
// Q (by position), by one CTA (b is overwritten by lambda, tmp has m entries):
// v minimizes |L v - b_p| (b_p = b in pivot order), lambda_p = [L11^{-T} v; 0].
// For rank = m this is the plain solve L11^{-T} L11^{-1} b_p.
template <typename F>
__device__ void cta_ls_apply(const F* Q, int m, const int* piv, int rank, const F* M, F* b, F* tmp) {
  const int tid = threadIdx.x, nt = blockDim.x;
  __syncthreads();
  if (rank == m) {
    for (int p = tid; p < m; p += nt) tmp[p] = b[piv[p]];
  } else {
    for (int a = tid; a < rank; a += nt) {
      F acc = 0;
      for (int i = a; i < m; ++i) acc = fma(Q[(size_t)a * m + i], b[piv[i]], acc);
      tmp[a] = acc;
    }
  }
  __syncthreads();
  if (tid < 32) {
    if (rank == m) {
      warp_forward(Q, m, m, tmp);
    } else if (rank > 0) {
      warp_forward(M, rank, rank, tmp);
      warp_backward(M, rank, rank, tmp);
    }
    warp_backward(Q, m, rank, tmp);
  }
  __syncthreads();
  for (int p = tid; p < m; p += nt) b[piv[p]] = p < rank ? tmp[p] : F(0);
  __syncthreads();
}

template <typename F, int NX, int NU, int DP, bool DI>
__global__ void __launch_bounds__(kBwdThreads) k_bwd_main(Dev<F> D, BwdDev<F> B) {
  using CL = CacheLayout<NX, NU>;
  __shared__ Model<F, NX, NU> Mo;
  __shared__ int s_bad, s_cnt;
  load_model<F, NX, NU>(Mo, D.model);
  const int sc = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
  const ScenMeta s = D.meta[sc];
  const BwdScen bs = B.bs[sc];
  const int N = s.N, T = s.T, P = s.P, m = bs.m;
  if (tid == 0) {
    s_bad = 0;
    s_cnt = 0;
  }
  __syncthreads();
  F* cache = D.cache + s.xs_off * CL::E;
  const uint16_t* Wm = B.Wb + s.as_off;
  const int32_t* act = B.act + s.ps_off;
  const F* a = D.a + s.ps_off * DP;
  const int32_t* pr = D.pairs + s.pair_off;
  F* psi = B.psi + bs.psi_off;
  F* Sm = B.S + bs.s_off;
  F* Mn = Sm + (size_t)m * m;
  int* piv = B.piv + s.ps_off;
  F* rhs = B.vec + bs.v_off;
  F* tmp = rhs + 2 * m;
  F* diag = rhs + 3 * m;
  F* pos0 = B.pos0 + s.as_off * DP;
  F* force = B.force + s.as_off * DP;
  auto Q = [&](int i, int r) { return D.Qd[(s.agent_off + i) * NX + r]; };
  auto Qf = [&](int i, int r) { return D.Qfd[(s.agent_off + i) * NX + r]; };
  auto XR = [&](int i, int r) { return D.x_ref[(s.agent_off + i) * NX + r]; };

  // Solves the LQ problem of every agent with linear term lin(i, t, r) and initial
  // state x0(i, r), and hands out states (outx(i, t, r, x)) and inputs
  // (outu(i, t, c, u)): one thread per axis of an agent for the double integrator,
  // else one per agent.
  auto solve_agents = [&](auto lin, auto x0, bool at_bounds, auto outx, auto outu) {
    if constexpr (DI) {
      for (int e = tid; e < N * DP; e += nt) {
        const int c = e / N, i = e - c * N;
        F* kk = B.kks + ((s.agent_off + i) * DP + c) * (size_t)B.kk_stride;
        lq_axis<F, NX, NU>(Mo, cache, Wm, N, i, T, c, T, [&](int t, int r, auto pos) { return lin(i, t, r, pos); }, x0(i, c),
                           x0(i, DP + c), at_bounds, [&](int t) -> F& { return kk[t]; },
                           [&](int t, F xp, F xv) {
                             outx(i, t, c, xp);
                             outx(i, t, DP + c, xv);
                           },
                           [&](int t, F u) { outu(i, t, c, u); });
      }
    } else {
      for (int i = tid; i < N; i += nt) {
        F xs[NX];
#pragma unroll
        for (int r = 0; r < NX; ++r) xs[r] = x0(i, r);
        F* kk = B.kks + ((s.agent_off + i) * DP) * (size_t)B.kk_stride;
        lq_solve<F, NX, NU>(agent_model<F, NX, NU>(D, Mo, s, i), cache, Wm, N, i, T,
                            [&](int t, int r) { return lin(i, t, r, r < DP); }, xs, at_bounds, kk,
                            [&](int t, const F (&x)[NX]) {
#pragma unroll
                              for (int r = 0; r < NX; ++r) outx(i, t, r, x[r]);
                            },
                            [&](int t, const F (&u)[NU]) {
#pragma unroll
                              for (int c = 0; c < NU; ++c) outu(i, t, c, u[c]);
                            });
      }
    }
    __syncthreads();
  };
  auto no_input = [](int, int, int, F) {};
  auto zero0 = [](int, int) { return F(0); };
  auto init0 = [&](int i, int r) { return D.x_init[(s.agent_off + i) * NX + r]; };
  // positions of every step t >= 1, the base of a right-hand side
  auto to_pos0 = [&](int i, int t, int r, F x) {
    if (t >= 1 && r < DP) pos0[((size_t)i * T + (t - 1)) * DP + r] = x;
  };

  // 1. factorization of the global per-agent Hessian with the final working set
  if constexpr (DI) {
    // one lane per axis, as many agents of a warp as fit
    using AC = AgentConst<NX, NU>;
    constexpr int NG = 32 / DP, kRun = NG * (kBwdThreads / 32);
    __shared__ F kct[AC::KC * kRun];
    const int lane = tid & 31, g = lane / DP;
    for (int i0 = 0; i0 < N; i0 += kRun) {
      const int q = (tid >> 5) * NG + g, i = i0 + q;
      const bool mine = g < NG && i < N;
      AxisView<F, NX, NU, DP, 1> V;
      V.N = N;
      V.T = T;
      V.ks = kRun;
      V.nc = 0;
      V.c0 = mine ? lane - g * DP : 0;
      V.rho = F(0);
      const int64_t ag = s.agent_off + (mine ? i : 0);
      V.cache = cache + V.c0 * N + (mine ? i : 0);
      V.Wm = B.Wb + s.as_off + (mine ? i : 0);
      V.Cm = D.Cm + s.as_off + (mine ? i : 0);
      V.Us = nullptr;
      V.Xo = nullptr;
      V.h = nullptr;
      V.xr = nullptr;
      V.xi = nullptr;
      V.qf = D.Qfd + ag * NX + V.c0;
      V.kc = kct + (mine ? q : 0) + V.c0 * kRun;
      axis_model(V, Mo);
      if (mine) {
        kct[(AC::RB + V.c0) * kRun + q] = F(2) * D.Rd[ag * NU + V.c0];
        kct[(AC::QB + V.c0) * kRun + q] = F(2) * Q(i, V.c0);
        kct[(AC::QB + DP + V.c0) * kRun + q] = F(2) * Q(i, DP + V.c0);
      }
      __syncwarp();
      if (axis_factor<false>(V, mine, T - 1, mine ? g * DP : 0)) atomicOr(&s_bad, 1);
      __syncwarp();
    }
    __syncthreads();
    // the forward factor cache no longer matches: force a refactorization on the next solve
    for (int e = tid; e < N * T; e += nt) D.Cm[s.as_off + e] = 0xFFFF;
  } else {
    for (int i = tid; i < N; i += nt) {
      F rbar[NU], qbar[NX];
#pragma unroll
      for (int c = 0; c < NU; ++c) rbar[c] = F(2) * D.Rd[(s.agent_off + i) * NU + c];
#pragma unroll
      for (int r = 0; r < NX; ++r) qbar[r] = F(2) * Q(i, r);
      F Pn[NX][NX];
#pragma unroll
      for (int r = 0; r < NX; ++r)
#pragma unroll
        for (int c = 0; c < NX; ++c) {
          Pn[r][c] = (r == c) ? F(2) * Qf(i, r) : F(0);
          cache[((size_t)T * CL::E + CL::P + r * NX + c) * N + i] = Pn[r][c];
        }
      int bad = 0;
      for (int t = T - 1; t >= 0; --t) {
        const uint16_t mask = Wm[(size_t)t * N + i];
        F Pt[NX][NX], K[NU][NX], L[NU][NU];
        auto put = [&](int r, int c, F v) {
          Pt[r][c] = v;
          Pt[c][r] = v;
        };
        auto putB = [](int, int, F) {};
        bad |= factor_stage<F, NX, NU>(agent_model<F, NX, NU>(D, Mo, s, i), Pn, mask, rbar, t >= 1 ? qbar : nullptr, 1, put, putB, K, L);
#pragma unroll
        for (int r = 0; r < NU; ++r) {
#pragma unroll
          for (int c = 0; c < NX; ++c) cache[((size_t)t * CL::E + CL::K + r * NX + c) * N + i] = K[r][c];
#pragma unroll
          for (int c = 0; c <= r; ++c) cache[((size_t)t * CL::E + CL::L + r * NU + c) * N + i] = L[r][c];
        }
        if (t >= 1) {
#pragma unroll
          for (int r = 0; r < NX; ++r)
#pragma unroll
            for (int c = 0; c < NX; ++c) {
              cache[((size_t)t * CL::E + CL::P + r * NX + c) * N + i] = Pt[r][c];
              Pn[r][c] = Pt[r][c];
            }
        }
      }
      if (bad) atomicOr(&s_bad, 1);
      // the forward factor cache no longer matches: force a refactorization on the next solve
      for (int t = 0; t < T; ++t) D.Cm[s.as_off + (size_t)t * N + i] = 0xFFFF;
    }
  }
  __syncthreads();

  // 2. position responses to unit forces at the agent's active times
  if constexpr (DI) {
    // (agent, step) of every response, listed in the force block (written later)
    int* const list = reinterpret_cast<int*>(force);
    for (int i = tid; i < N; i += nt) {
      unsigned long long msk = B.amask[s.agent_off + i];
      int at = msk ? atomicAdd(&s_cnt, __popcll(msk)) : 0;
      for (; msk; msk &= msk - 1) list[at++] = i | (__ffsll((long long)msk) - 1) << 16;
    }
    __syncthreads();
    const int nr = s_cnt;
    for (int e = tid; e < nr * DP; e += nt) {
      const int c = e / nr, i = list[e - c * nr] & 0xFFFF, tp = (list[e - c * nr] >> 16) + 1;
      // a response moves its own axis only; a word of another axis holds the gains
      F* const out = psi + (((size_t)i * T + (tp - 1)) * DP + c) * T * DP;
      const int other = c == 0 ? 1 : 0;
      lq_axis<F, NX, NU>(Mo, cache, Wm, N, i, T, c, tp,
                         [&](int t, int, auto pos) { return (pos && t == tp) ? F(-1) : F(0); }, F(0), F(0), false,
                         [&](int t) -> F& { return out[t * DP + other]; },
                         [&](int t, F xp, F) {
                           if (t >= 1) out[(t - 1) * DP + c] = xp;
                         },
                         [](int, F) {});
    }
  } else {
    const F z0[NX] = {};
    for (int task = tid; task < N * DP; task += nt) {
      const int i = task / DP, cin = task % DP;
      const unsigned long long msk = B.amask[s.agent_off + i];
      F* kk = B.kks + ((s.agent_off + i) * DP + cin) * (size_t)B.kk_stride;
      for (int tp = 1; tp <= T; ++tp) {
        if (!((msk >> (tp - 1)) & 1ull)) continue;
        auto lin = [&](int t, int r) -> F { return (t == tp && r == cin) ? F(-1) : F(0); };
        auto outx = [&](int t, const F (&x)[NX]) {
          if (t >= 1) {
#pragma unroll
            for (int c = 0; c < DP; ++c)
              psi[((((size_t)i * T + (tp - 1)) * DP + cin) * T + (t - 1)) * DP + c] = x[c];
          }
        };
        auto outu = [&](int, const F (&)[NU]) {};
        lq_solve<F, NX, NU>(agent_model<F, NX, NU>(D, Mo, s, i), cache, Wm, N, i, T, lin, z0, false, kk, outx, outu);
      }
    }
  }
  __syncthreads();
  // 3. base solution (cost terms only) for the right-hand side of S mu = d - G z0
  auto cost = [&](int i, int t, int r, auto) -> F { return (F(-2) * (t < T ? Q(i, r) : Qf(i, r))) * XR(i, r); };
  solve_agents(cost, init0, true, to_pos0, no_input);

  // 4. Schur complement S_hk = sum over shared agents of sigma sigma a_h' Psi a_k
  auto hs = [&](int h, int& i, int& j, int& tm1, int& pair) {
    const int q = act[h];
    tm1 = q / P;
    pair = q - tm1 * P;
    const int pk = pr[pair];
    i = pk & 0xFFFF;
    j = pk >> 16;
  };
  for (int e = tid; e < m * m; e += nt) {
    const int h = e / m, k = e % m;
    if (k > h) continue;
    int ih, jh, th, ph, ik, jk, tk, pk2;
    hs(h, ih, jh, th, ph);
    hs(k, ik, jk, tk, pk2);
    F acc = 0;
    const int ag[2] = {ih, jh};
    const F sg[2] = {F(1), F(-1)};
    for (int u = 0; u < 2; ++u) {
      const int ma = ag[u];
      F sk = 0;
      if (ma == ik) sk = F(1);
      else if (ma == jk) sk = F(-1);
      else continue;
      F v = 0;
#pragma unroll
      for (int cin = 0; cin < DP; ++cin) {
        const F ak = a[((size_t)tk * DP + cin) * P + pk2];
#pragma unroll
        for (int cout = 0; cout < DP; ++cout) {
          if (DI && cout != cin) continue;  // the axes do not respond to one another
          const F ah = a[((size_t)th * DP + cout) * P + ph];
          v = fma(ah * psi[((((size_t)ma * T + tk) * DP + cin) * T + th) * DP + cout], ak, v);
        }
      }
      acc = fma(sg[u] * sk, v, acc);
    }
    Sm[(size_t)h * m + k] = acc;
    Sm[(size_t)k * m + h] = acc;
  }
  for (int h = tid; h < m; h += nt) {
    int i, j, tm1, pair;
    hs(h, i, j, tm1, pair);
    F v = F(s.d);
#pragma unroll
    for (int c = 0; c < DP; ++c)
      v = fma(-a[((size_t)tm1 * DP + c) * P + pair],
              pos0[((size_t)i * T + tm1) * DP + c] - pos0[((size_t)j * T + tm1) * DP + c], v);
    rhs[h] = v;
  }
  // 5. rank-revealing factorization of S; least-squares multipliers mu
  __syncthreads();
  const int rank = m > 0 ? cta_pivoted_cholesky(Sm, m, piv, diag, F(B.rank_tol)) : 0;
  __syncthreads();
  if (m > 0) {
    // the factor by position in the second block; the normal matrix in the first
    cta_by_position(Sm, m, piv, rank, Mn);
    cta_ls_prepare(Mn, m, rank, Sm, &s_bad);
    cta_ls_apply(Mn, m, piv, rank, Sm, rhs, tmp);
  }

  // 6. coupling forces G' mu, polished primal solve
  auto forces = [&](const F* lam) {
    for (int e = tid; e < N * T * DP; e += nt) force[e] = 0;
    __syncthreads();
    // the active rows are sorted by step: one thread per step, in their order
    for (int t = tid; t < T; t += nt) {
      int lo = 0, hi = m;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (act[mid] < t * P) lo = mid + 1;
        else hi = mid;
      }
      for (int h = lo; h < m && act[h] < (t + 1) * P; ++h) {
        int i, j, tm1, pair;
        hs(h, i, j, tm1, pair);
#pragma unroll
        for (int c = 0; c < DP; ++c) {
          const F f = lam[h] * a[((size_t)tm1 * DP + c) * P + pair];
          force[((size_t)i * T + tm1) * DP + c] += f;
          force[((size_t)j * T + tm1) * DP + c] -= f;
        }
      }
    }
    __syncthreads();
  };
  forces(rhs);
  solve_agents(
      [&](int i, int t, int r, auto pos) -> F {
        F v = cost(i, t, r, pos);
        if (pos) v -= force[((size_t)i * T + (t - 1)) * DP + r];
        return v;
      },
      init0, true, [&](int i, int t, int r, F x) { B.Xp[(s.xs_off + (int64_t)i * (T + 1) + t) * NX + r] = x; },
      [&](int i, int t, int c, F u) { B.Up[(s.as_off + (int64_t)i * T + t) * NU + c] = u; });

  F* lamw = rhs + m;
  if (!B.adjoint) {
    if (tid == 0) {
      bool fin = true;
      for (int h = 0; h < m; ++h) fin = fin && finite_(rhs[h]);
      B.bstatus[sc] = (s_bad || !fin) ? ST_NUMERIC : ST_CONVERGED;
      B.ndep[sc] = m - rank;
    }
    return;
  }
  // 7. adjoint: w0 = H^{-1} dl/dz (homogeneous), S lam = -G w0, w = w0 + Psi G' lam
  auto loss = [&](int i, int t, int r, auto) -> F { return -F(B.gX[(s.xs_off + (int64_t)i * (T + 1) + t) * NX + r]); };
  solve_agents(loss, zero0, false, to_pos0, no_input);
  for (int h = tid; h < m; h += nt) {
    int i, j, tm1, pair;
    hs(h, i, j, tm1, pair);
    F v = 0;
#pragma unroll
    for (int c = 0; c < DP; ++c)
      v = fma(-a[((size_t)tm1 * DP + c) * P + pair],
              pos0[((size_t)i * T + tm1) * DP + c] - pos0[((size_t)j * T + tm1) * DP + c], v);
    lamw[h] = v;
  }
  __syncthreads();
  if (m > 0) cta_ls_apply(Mn, m, piv, rank, Sm, lamw, tmp);
  forces(lamw);
  solve_agents(
      [&](int i, int t, int r, auto pos) -> F {
        F v = loss(i, t, r, pos);
        if (pos) v -= force[((size_t)i * T + (t - 1)) * DP + r];
        return v;
      },
      zero0, false, [&](int i, int t, int r, F x) { B.Wx[(s.xs_off + (int64_t)i * (T + 1) + t) * NX + r] = x; },
      [&](int i, int t, int c, F u) { B.Wu[(s.as_off + (int64_t)i * T + t) * NU + c] = u; });

  // 8. gradients: dl/dtheta = -w' (dH/dtheta z + dg/dtheta)
  for (int i = tid; i < N; i += nt) {
    const int64_t ag = s.agent_off + i;
    const F* Xp = B.Xp + (s.xs_off + (int64_t)i * (T + 1)) * NX;
    const F* Up = B.Up + (s.as_off + (int64_t)i * T) * NU;
    const F* Wx = B.Wx + (s.xs_off + (int64_t)i * (T + 1)) * NX;
    const F* Wu = B.Wu + (s.as_off + (int64_t)i * T) * NU;
#pragma unroll
    for (int r = 0; r < NX; ++r) {
      F gq = 0, gqf = 0, gg = 0;
      for (int t = 1; t <= T; ++t) {
        const F w = Wx[(size_t)t * NX + r];
        const F e = Xp[(size_t)t * NX + r] - XR(i, r);
        if (t < T) {
          gq = fma(F(-2) * w, e, gq);
          gg = fma(F(2) * Q(i, r), w, gg);
        } else {
          gqf = fma(F(-2) * w, e, gqf);
          gg = fma(F(2) * Qf(i, r), w, gg);
        }
      }
      if (B.gQ) B.gQ[ag * NX + r] = double(gq);
      if (B.gQf) B.gQf[ag * NX + r] = double(gqf);
      if (B.gGoal) B.gGoal[ag * NX + r] = double(gg);
    }
#pragma unroll
    for (int c = 0; c < NU; ++c) {
      F gr = 0;
      for (int t = 0; t < T; ++t) gr = fma(F(-2) * Wu[(size_t)t * NU + c], Up[(size_t)t * NU + c], gr);
      if (B.gR) B.gR[ag * NU + c] = double(gr);
    }
  }
  if (tid == 0) {
    bool fin = true;
    for (int h = 0; h < m; ++h) fin = fin && finite_(rhs[h]) && finite_(lamw[h]);
    B.bstatus[sc] = (s_bad || !fin) ? ST_NUMERIC : ST_CONVERGED;
    B.ndep[sc] = m - rank;
  }
}

// One round of active-set polishing on the centralized QP (one CTA per
// scenario), after k_bwd_main (adjoint = 0) has formed the polished point of
// the current active set, its halfspace multipliers mu (in the order of the
// active list) and the coupling forces G' mu.  KKT check at that point:
//   - halfspace rows: active ones need mu >= 0, inactive ones a'(p_i - p_j) >= d;
//   - inputs: held ones need a non-negative bound multiplier, from
//     stationarity mu_lower = 2 R u_t + B' lambda_{t+1} (mu_upper its negative)
//     with the costates lambda_t = 2 Q_t (x_t - x_ref) - C' f_t + A' lambda_{t+1}
//     of the global problem (f_t the coupling force), free ones lie in the box.
// One change per round, as in a primal active-set method: the row with the
// most negative multiplier below -kkt_tol * max(1, largest |multiplier|)
// leaves the set; if there is none, the most violated row (halfspace
// violation relative to max(1, d), box violation relative to max(1, |bound|))
// beyond kkt_tol enters it (an input held at the violated bound).  Ties go to
// the lowest index (halfspace rows in active-list or pair-step order first,
// then inputs by agent, step, component).  pchg[sc] = 1 when the set changed.
template <typename F, int NX, int NU, int DP, bool DI>
__global__ void __launch_bounds__(128) k_bwd_polish(Dev<F> D, BwdDev<F> B) {
  __shared__ Model<F, NX, NU> Mo;
  // one key per search: a late warp may still read the first search's when the
  // second search writes
  __shared__ unsigned long long s_scale, s_drop, s_add;
  __shared__ long long s_idx;
  load_model<F, NX, NU>(Mo, D.model);
  const int sc = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
  const ScenMeta s = D.meta[sc];
  const BwdScen bs = B.bs[sc];
  const int N = s.N, T = s.T, P = s.P, m = bs.m;
  const int32_t* act = B.act + s.ps_off;
  const F* mu = B.vec + bs.v_off;
  const F* a = D.a + s.ps_off * DP;
  const int32_t* pr = D.pairs + s.pair_off;
  const F* force = B.force + s.as_off * DP;
  uint16_t* Wb = B.Wb + s.as_off;
  uint8_t* hm = B.hmask + s.ps_off;
  const int64_t PT = (int64_t)P * T;
  if (tid == 0) {
    s_scale = ord_bits(F(1));
    s_drop = s_add = ~0ull;
    s_idx = LLONG_MAX;
  }
  __syncthreads();
  // g = 2 R u_t + B' lambda_{t+1} of every input, from the costates backwards from
  // lambda_{T+1} = 0, kept in the adjoint's input block (unused in these rounds):
  // one thread per axis of an agent for the double integrator, else per agent
  F* const G = B.Wu + s.as_off * NU;
  if constexpr (DI) {
    constexpr int H = NU;
    const F one = Mo.A[0][0], dt = Mo.A[0][H], b1 = Mo.B[0][0], b2 = Mo.B[H][0];
    for (int e = tid; e < N * H; e += nt) {
      const int c = e / N, i = e - c * N;
      const int64_t ag = s.agent_off + i;
      const F* Xp = B.Xp + (s.xs_off + (int64_t)i * (T + 1)) * NX;
      const F* Up = B.Up + (s.as_off + (int64_t)i * T) * NU;
      F lp = F(0), lv = F(0);
      for (int t = T; t >= 1; --t) {
        const F* const w = (t < T ? D.Qd : D.Qfd) + ag * NX;
        F np = (F(2) * w[c]) * (Xp[(size_t)t * NX + c] - D.x_ref[ag * NX + c]);
        np -= force[((size_t)i * T + (t - 1)) * DP + c];
        const F nv = (F(2) * w[H + c]) * (Xp[(size_t)t * NX + H + c] - D.x_ref[ag * NX + H + c]);
        lv = fma(one, lv, fma(dt, lp, nv));
        lp = fma(one, lp, np);
        const F g = (F(2) * D.Rd[ag * NU + c]) * Up[(size_t)(t - 1) * NU + c];
        G[((size_t)i * T + (t - 1)) * NU + c] = fma(b2, lv, fma(b1, lp, g));
      }
    }
  } else {
    for (int i = tid; i < N; i += nt) {
      const Model<F, NX, NU>& Ma = agent_model<F, NX, NU>(D, Mo, s, i);
      const F* Xp = B.Xp + (s.xs_off + (int64_t)i * (T + 1)) * NX;
      const F* Up = B.Up + (s.as_off + (int64_t)i * T) * NU;
      F lam[NX];
#pragma unroll
      for (int r = 0; r < NX; ++r) lam[r] = F(0);
      for (int t = T; t >= 1; --t) {
        F ln[NX];
#pragma unroll
        for (int r = 0; r < NX; ++r) {
          const F q = t < T ? D.Qd[(s.agent_off + i) * NX + r] : D.Qfd[(s.agent_off + i) * NX + r];
          F acc = (F(2) * q) * (Xp[(size_t)t * NX + r] - D.x_ref[(s.agent_off + i) * NX + r]);
          if (r < DP) acc -= force[((size_t)i * T + (t - 1)) * DP + r];
#pragma unroll
          for (int k = 0; k < NX; ++k) acc = fma(Ma.A[k][r], lam[k], acc);
          ln[r] = acc;
        }
#pragma unroll
        for (int c = 0; c < NU; ++c) {
          F g = (F(2) * D.Rd[(s.agent_off + i) * NU + c]) * Up[(size_t)(t - 1) * NU + c];
#pragma unroll
          for (int r = 0; r < NX; ++r) g = fma(Ma.B[r][c], ln[r], g);
          G[((size_t)i * T + (t - 1)) * NU + c] = g;
        }
#pragma unroll
        for (int r = 0; r < NX; ++r) lam[r] = ln[r];
      }
    }
  }
  __syncthreads();
  // visit(index, i, t, c, working-set mask) for every input, agents, then steps, then components
  const int nin = N * T * NU;
  auto inputs = [&](auto&& visit) {
    for (int e = tid; e < nin; e += nt) {
      const int c = e % NU, it = e / NU, t = it % T, i = it / T;
      visit(e, i, t, c, Wb[(size_t)t * N + i]);
    }
  };
  auto bound_mu = [](uint16_t msk, int c, F g) -> F { return (msk & (1u << c)) ? g : -g; };
  auto held = [](uint16_t msk, int c) -> bool { return (msk & (0x101u << c)) != 0; };
  // largest |multiplier|
  {
    unsigned long long top = 0;
    inputs([&](int e, int, int, int c, uint16_t msk) {
      if (held(msk, c)) {
        const unsigned long long v = abs_bits(bound_mu(msk, c, G[e]));
        top = v > top ? v : top;
      }
    });
    for (int h = tid; h < m; h += nt) {
      const unsigned long long v = abs_bits(mu[h]);
      top = v > top ? v : top;
    }
    if (top) atomicMax(&s_scale, top);
  }
  __syncthreads();
  const F tol = F(B.kkt_tol);
  const F mtol = tol * from_bits(s_scale, F(0));
  // 1. the most negative multiplier (smallest order key), then its lowest index
  {
    unsigned long long low = ~0ull;
    for (int h = tid; h < m; h += nt)
      if (mu[h] < -mtol) low = min(low, mono_key(mu[h]));
    inputs([&](int e, int, int, int c, uint16_t msk) {
      if (held(msk, c) && bound_mu(msk, c, G[e]) < -mtol) low = min(low, mono_key(bound_mu(msk, c, G[e])));
    });
    if (low != ~0ull) atomicMin(&s_drop, low);
  }
  __syncthreads();
  const unsigned long long kdrop = s_drop;
  if (kdrop != ~0ull) {
    long long at = LLONG_MAX;
    for (int h = tid; h < m; h += nt)
      if (mono_key(mu[h]) == kdrop) at = min(at, (long long)h);
    inputs([&](int e, int, int, int c, uint16_t msk) {
      if (held(msk, c) && mono_key(bound_mu(msk, c, G[e])) == kdrop) at = min(at, (long long)m + e);
    });
    if (at != LLONG_MAX) atomicMin(&s_idx, at);
    __syncthreads();
    if (tid == 0) {
      const long long e = s_idx;
      if (e < m) {
        hm[act[e]] = 0;
      } else {
        const long long r = e - m;
        const int c = (int)(r % NU), t = (int)((r / NU) % T), i = (int)(r / ((long long)NU * T));
        Wb[(size_t)t * N + i] = (uint16_t)(Wb[(size_t)t * N + i] & ~(0x101u << c));
      }
      B.pchg[sc] = 1;
    }
    return;
  }
  // 2. the most violated row (largest relative violation), then its lowest index
  const F dscale = F(s.d) > F(1) ? F(s.d) : F(1);
  auto slack_rel = [&](int64_t q) -> F {   // a'(p_i - p_j) - d, relative to max(1, d)
    const int tm1 = (int)(q / P), pair = (int)(q - (int64_t)tm1 * P);
    const int pk = pr[pair], i = pk & 0xFFFF, j = pk >> 16;
    const F* xi = B.Xp + (s.xs_off + (int64_t)i * (T + 1) + tm1 + 1) * NX;
    const F* xj = B.Xp + (s.xs_off + (int64_t)j * (T + 1) + tm1 + 1) * NX;
    F v = -F(s.d);
#pragma unroll
    for (int c = 0; c < DP; ++c) v = fma(a[((size_t)tm1 * DP + c) * P + pair], xi[c] - xj[c], v);
    return v / dscale;
  };
  auto box_rel = [](F u, F lo, F hi) -> F {   // distance outside the box, relative; <= 0 inside
    const F sl = fabs_(lo) > F(1) ? fabs_(lo) : F(1), sh = fabs_(hi) > F(1) ? fabs_(hi) : F(1);
    const F vl = (lo - u) / sl, vh = (u - hi) / sh;
    return vl > vh ? vl : vh;
  };
  const F* const Up = B.Up + s.as_off * NU;
  auto box_of = [&](int e, int i, int c) -> F {
    const Model<F, NX, NU>& Ma = DI ? Mo : agent_model<F, NX, NU>(D, Mo, s, i);
    return box_rel(Up[e], Ma.umin[c], Ma.umax[c]);
  };
  {
    unsigned long long low = ~0ull;
    for (int64_t q = tid; q < PT; q += nt)
      if (!hm[q]) {
        const F v = -slack_rel(q);
        if (v > tol) low = min(low, ~mono_key(v));
      }
    inputs([&](int e, int i, int, int c, uint16_t msk) {
      if (!held(msk, c)) {
        const F v = box_of(e, i, c);
        if (v > tol) low = min(low, ~mono_key(v));
      }
    });
    if (low != ~0ull) atomicMin(&s_add, low);
  }
  __syncthreads();
  const unsigned long long kadd = s_add;
  if (kadd == ~0ull) {
    if (tid == 0) B.pchg[sc] = 0;   // KKT conditions hold
    return;
  }
  {
    long long at = LLONG_MAX;
    for (int64_t q = tid; q < PT; q += nt)
      if (!hm[q] && ~mono_key(-slack_rel(q)) == kadd) at = min(at, (long long)q);
    inputs([&](int e, int i, int, int c, uint16_t msk) {
      if (!held(msk, c) && ~mono_key(box_of(e, i, c)) == kadd) at = min(at, (long long)PT + e);
    });
    if (at != LLONG_MAX) atomicMin(&s_idx, at);
  }
  __syncthreads();
  if (tid == 0) {
    const long long e = s_idx;
    if (e < PT) {
      hm[e] = 1;
    } else {
      const long long r = e - PT;
      const int c = (int)(r % NU), t = (int)((r / NU) % T), i = (int)(r / ((long long)NU * T));
      const F u = B.Up[(s.as_off + (int64_t)i * T + t) * NU + c];
      const Model<F, NX, NU>& Ma = agent_model<F, NX, NU>(D, Mo, s, i);
      const uint16_t bit = (u < Ma.umin[c]) ? (uint16_t)(1u << c) : (uint16_t)(0x100u << c);
      Wb[(size_t)t * N + i] = (uint16_t)(Wb[(size_t)t * N + i] | bit);
    }
    B.pchg[sc] = 1;
  }
}

// Active set in the caller's layouts: halfspace flags [pair-step] (pair-major,
// then t) and held inputs [agent][t][nu] (0 free, 1 lower, 2 upper).
template <typename F>
__global__ void k_bwd_export_set(Dev<F> D, BwdDev<F> B, int nu, uint8_t* act_out, int8_t* W_out) {
  const int sc = blockIdx.x;
  const ScenMeta s = D.meta[sc];
  const int64_t PT = (int64_t)s.P * s.T, NT = (int64_t)s.N * s.T;
  if (act_out)
    for (int64_t q = threadIdx.x; q < PT; q += blockDim.x) {
      const int tm1 = (int)(q / s.P), pair = (int)(q - (int64_t)tm1 * s.P);
      act_out[s.ps_off + (int64_t)pair * s.T + tm1] = B.hmask[s.ps_off + q];
    }
  if (W_out)
    for (int64_t e = threadIdx.x; e < NT; e += blockDim.x) {
      const int t = (int)(e / s.N), i = (int)(e - (int64_t)t * s.N);
      const uint16_t msk = B.Wb[s.as_off + e];
      for (int c = 0; c < nu; ++c)
        W_out[(s.as_off + (int64_t)i * s.T + t) * nu + c] = (msk & (1u << c)) ? 1 : ((msk & (0x100u << c)) ? 2 : 0);
    }
}

template <typename F>
__global__ void k_bwd_export_x(const F* Xp, int64_t n, double* out) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    out[k] = double(Xp[k]);
}

}  // namespace tadmm
