// The x-update's equality-constrained solves for axis-separable models (included
// by tadmm_device.cuh, after the agent context).
//
// With A = [[I, dt I], [0, a22 I]], B = [[b1 I], [b2 I]] (the double integrator has
// a22 = 1; HET: per-agent models, each with its own dt, a22, b1, b2) and the
// diagonal weights that the problem has, every matrix of the Riccati recursion of
// Sec. IV.B couples a position component with its own velocity only: P_t, K_t, S_t and P_{t+1}B fall apart into one two-state,
// one-input recursion per axis, and the entries between axes are zeros.  The
// general products form those zeros and add them; here they are left out, and
// every other value is formed by the same operations in the same order, so the
// results have the same bits.  (The inverse of S keeps the form of the general
// code, adjugate over determinant, since its rounding is part of that.  In double-float,
// where a product by the constant 1 is a rounding of its own in the general products,
// the results differ by such roundings, at the same distance from float64.)
//
// The FP64 pipe bounds these loops: a warp issues one FP64 instruction per about
// 68 cycles, an SM one per 20, whatever the number of active lanes.  An EQP pass
// takes 14 of them per axis and stage (28 per agent in 2D, where the 4x4 products
// took 38 with no held input in the warp and up to 60 with some); a stage
// factorization about 30 and the reciprocal on one lane per axis (54 on four lanes
// per agent, 121 on one).  A round of few agents takes one lane per axis, so 14
// instructions serve up to 16 agents in 2D and 10 in 3D.  Measured, FP64: the
// 4096-scenario mixed batch over 500 iterations 769 -> 546 ms, a 512-agent 3D
// swarm 2.76 -> 1.73 ms per iteration in graph mode, a two-agent crossing
// 2.58 -> 1.49 ms; 1024 scenarios in float32 over 200 iterations 117 -> 69 ms.
// Agents of unlike mass and damping, which took the dense products on one lane
// each: 256 scenarios of 5 to 32 agents over 100 iterations 244 -> 55 ms.
#pragma once

namespace tadmm {

// Words of one axis of one stage of the factor cache.  A free input needs its
// feedback and feedforward, a held one its column of P_{t+1}B and B'p_{t+1}, so
// these share their words.
struct AxisCache {
  static constexpr int PP = 0, PV = 1, VV = 2;  // P_t: position, cross, velocity
  static constexpr int G1 = 3, G2 = 4;          // free: K_t; held: P_{t+1}B (position, velocity)
  static constexpr int SI = 5;                  // S_t^{-1}
  static constexpr int D = 6;                   // free: k_t; held: B'p_{t+1} (written by the pass)
  static constexpr int E = 7;
};

// A float near v for a test with a margin: the magnitude cut to 24 bits, by
// integer instructions (a conversion would take the FP64 pipe).  Values below
// 2^-126 give 0; values of 2^60 and above, infinities and NaN give NaN, which
// fails every comparison.
__device__ __forceinline__ float near_f32(double v) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const uint32_t mag = hi & 0x7FFFFFFFu;
  const uint32_t cut = (__funnelshift_l(lo, hi, 3) & 0x7FFFFFFFu) ^ 0x40000000u;
  uint32_t r = mag < 0x38100000u ? 0u : cut;
  r = mag >= 0x43B00000u ? 0x7FC00000u : r;
  return __uint_as_float(r | (hi & 0x80000000u));
}

__device__ __forceinline__ float near_f32(float v) {
  return fabsf(v) < 0x1p60f ? v : __uint_as_float(0x7FC00000u);
}
__device__ __forceinline__ float near_f32(df64 v) { return near_f32(v.hi); }

// Margin of such a test on a sum of a few products: of the sizes' sum (its operands' cuts
// of 2^-23 and its roundings of 2^-24 stay below 2^-20), and for what a cut to 0 leaves out.
constexpr float kNearRel = 0x1p-19f, kNearAbs = 1e-17f;

// Part of an agent's data that a lane works on: AX axes from c0 on (all of them,
// or one when the agents of a round are spread over lanes).  Pointers are those
// of the agent's first axis; word w of an axis a lies a * N further on.
template <typename F, int NX, int NU, int DP, int AX>
struct AxisView {
  using AC = AgentConst<NX, NU>;
  F* cache;
  uint16_t* Wm;
  uint16_t* Cm;
  F* Us;
  F* Xo;
  const F* h;
  const F* kc;      // agent constants, shifted to axis c0
  const F* qf;      // rows of Qf, x_ref and x_init, shifted to axis c0
  const F* xr;
  const F* xi;
  F rho, dt, a22, b1, b2, lo[AX], hi[AX];
  int N, T, ks, c0, nc;

  __device__ __forceinline__ F& C(int t, int w, int a) const { return cache[((t * AxisCache::E + w) * DP + a) * N]; }
  __device__ __forceinline__ F& us(int t, int a) const { return Us[(t * DP + a) * N]; }
  __device__ __forceinline__ F& x(int t, int r) const { return Xo[(t * NX + r) * N]; }  // r = a, or DP + a
  __device__ __forceinline__ F hv(int t, int a) const { return h[((t - 1) * DP + a) * N]; }
  __device__ __forceinline__ F k(int e) const { return kc[e * ks]; }
  // input a of this view held at a bound by mask w; its bound
  __device__ __forceinline__ bool held(uint32_t w, int a) const { return (w >> (c0 + a)) & 0x101u; }
  __device__ __forceinline__ F bound(uint32_t w, int a) const { return ((w >> (c0 + a)) & 1u) ? lo[a] : hi[a]; }
};

template <int AX, typename F, int NX, int NU, int DP>
__device__ __forceinline__ void axis_model(AxisView<F, NX, NU, DP, AX>& V, const Model<F, NX, NU>& M) {
  V.dt = M.A[0][DP];
  V.a22 = M.A[DP][DP];
  V.b1 = M.B[0][0];
  V.b2 = M.B[DP][0];
#pragma unroll
  for (int a = 0; a < AX; ++a) {
    V.lo[a] = M.umin[V.c0 + a];
    V.hi[a] = M.umax[V.c0 + a];
  }
}

// The lane's own agent with all its axes.
template <typename F, int NX, int NU, int DP>
__device__ __forceinline__ AxisView<F, NX, NU, DP, DP> axis_view(const AgentCtx<F, NX, NU, DP>& A) {
  using AC = AgentConst<NX, NU>;
  AxisView<F, NX, NU, DP, DP> V;
  V.cache = A.cache + A.i;
  V.Wm = A.Wm + A.i;
  V.Cm = A.Cm + A.i;
  V.Us = A.Us + A.i;
  V.Xo = A.Xo + A.i;
  V.h = A.h + A.i;
  V.kc = A.kc;
  V.qf = A.qf;
  V.xr = A.xr;
  V.xi = A.xi;
  V.N = A.N;
  V.T = A.T;
  V.ks = A.ks;
  V.c0 = 0;
  V.nc = A.nc;
  V.rho = A.k(AC::RHO);
  axis_model(V, *A.M);
  return V;
}

// Axis c of the agent of lane src (every lane of the warp calls this).
template <typename F, int NX, int NU, int DP>
__device__ __forceinline__ AxisView<F, NX, NU, DP, 1> axis_view_of(const AgentCtx<F, NX, NU, DP>& A, int src, int c) {
  using AC = AgentConst<NX, NU>;
  constexpr unsigned FULL = 0xffffffffu;
  auto sp = [&](auto p) { return (decltype(p))__shfl_sync(FULL, (unsigned long long)p, src); };
  AxisView<F, NX, NU, DP, 1> V;
  V.N = __shfl_sync(FULL, A.N, src);
  V.T = __shfl_sync(FULL, A.T, src);
  V.ks = __shfl_sync(FULL, A.ks, src);
  V.nc = __shfl_sync(FULL, A.nc, src);
  const int i = __shfl_sync(FULL, A.i, src), off = c * V.N + i;
  V.c0 = c;
  V.cache = sp(A.cache) + off;
  V.Wm = sp(A.Wm) + i;
  V.Cm = sp(A.Cm) + i;
  V.Us = sp(A.Us) + off;
  V.Xo = sp(A.Xo) + off;
  V.h = sp(A.h) + off;
  const F* kc = sp(A.kc);
  V.rho = kc[AC::RHO * V.ks];
  V.kc = kc + c * V.ks;
  V.qf = sp(A.qf) + c;
  V.xr = sp(A.xr) + c;
  V.xi = sp(A.xi) + c;
  axis_model(V, *sp(A.M));
  return V;
}

// Stage factorizations dirty..0 of the view's axes (Sec. IV.B restricted to the
// free inputs), the values of P kept in registers from stage to stage.
// AX == DP: the calling lane's own agent; `act` may differ between lanes.
// AX == 1: lanes gb .. gb + DP - 1 hold the axes of one agent and exchange their S;
// every lane of the warp calls this.  Returns 1 on a non-positive pivot.
template <bool HET, typename F, int NX, int NU, int DP, int AX>
__device__ __forceinline__ int axis_factor(const AxisView<F, NX, NU, DP, AX>& V, bool act, int dirty, int gb) {
  using AC = AgentConst<NX, NU>;
  using L = AxisCache;
  static_assert(AX == 1 || AX == DP, "one axis per lane, or all");
  constexpr unsigned FULL = 0xffffffffu;
  int bad = 0;
  F pp[AX], pv[AX], vv[AX];
  const int last = AX == 1 ? __reduce_max_sync(FULL, act ? dirty : -1) : (act ? dirty : -1);
#pragma unroll
  for (int a = 0; a < AX; ++a) pp[a] = pv[a] = vv[a] = F(0);
  for (int t = last; t >= 0; --t) {
    const bool on = act && t <= dirty;
    if (on && t == dirty) {
      // P_{t+1}: the terminal weights, or the stage above the changed ones
#pragma unroll
      for (int a = 0; a < AX; ++a) {
        if (t == V.T - 1) {
          pp[a] = F(2) * V.qf[a] + V.rho * F(V.nc);
          pv[a] = F(0);
          vv[a] = F(2) * V.qf[DP + a] + F(0);
          V.C(V.T, L::PP, a) = pp[a];
          V.C(V.T, L::PV, a) = pv[a];
          V.C(V.T, L::VV, a) = vv[a];
        } else {
          pp[a] = V.C(t + 1, L::PP, a);
          pv[a] = V.C(t + 1, L::PV, a);
          vv[a] = V.C(t + 1, L::VV, a);
        }
      }
    }
    const uint32_t mask = on ? V.Wm[t * V.N] : 0u;
    F pav[AX], pvv[AX], pb1[AX], pb2[AX], S[AX], mp[AX], mv[AX];
#pragma unroll
    for (int a = 0; a < AX; ++a) {
      // PA = [[pp, pav], [pv, pvv]], PB = [pb1; pb2]
      if constexpr (HET) {  // the order of the general products
        pav[a] = fma(pv[a], V.a22, pp[a] * V.dt);
        pvv[a] = fma(vv[a], V.a22, pv[a] * V.dt);
      } else {
        pav[a] = fma(pp[a], V.dt, pv[a]);
        pvv[a] = fma(pv[a], V.dt, vv[a]);
      }
      pb1[a] = fma(pv[a], V.b2, pp[a] * V.b1);
      pb2[a] = fma(vv[a], V.b2, pv[a] * V.b1);
      const bool hd = V.held(mask, a);
      F s = on ? V.k(AC::RB + a) : F(1);
      s = fma(V.b1, pb1[a], s);
      s = fma(V.b2, pb2[a], s);
      S[a] = hd ? F(1) : s;
      mp[a] = hd ? F(0) : fma(V.b2, pv[a], V.b1 * pp[a]);
      mv[a] = hd ? F(0) : fma(V.b2, pvv[a], V.b1 * pav[a]);
    }
    // S^{-1} by the adjugate of the diagonal matrix S
    F Sd[DP], si[AX];
#pragma unroll
    for (int c = 0; c < DP; ++c) {
      if constexpr (AX == 1) Sd[c] = shfl_f(S[0], gb + c);
      else Sd[c] = S[c];
    }
    if constexpr (DP == 2) {
      const F det = Sd[0] * Sd[1];
      if (on && (!(Sd[0] > F(0)) || !(det > F(0)))) bad = 1;
      const F id = F(1) / det;
      if constexpr (AX == 1) si[0] = (V.c0 == 0 ? Sd[1] : Sd[0]) * id;
      else { si[0] = Sd[1] * id; si[1] = Sd[0] * id; }
    } else {
      const F c00 = Sd[1] * Sd[2], c11 = Sd[0] * Sd[2], c22 = Sd[0] * Sd[1];
      const F det = Sd[0] * c00;
      if (on && (!(Sd[0] > F(0)) || !(c22 > F(0)) || !(det > F(0)))) bad = 1;
      const F id = F(1) / det;
      if constexpr (AX == 1) si[0] = (V.c0 == 0 ? c00 : (V.c0 == 1 ? c11 : c22)) * id;
      else { si[0] = c00 * id; si[1] = c11 * id; si[2] = c22 * id; }
    }
    if (!on) continue;
#pragma unroll
    for (int a = 0; a < AX; ++a) {
      const F k1 = -(si[a] * mp[a]), k2 = -(si[a] * mv[a]);
      const bool hd = V.held(mask, a);
      V.C(t, L::G1, a) = hd ? pb1[a] : k1;
      V.C(t, L::G2, a) = hd ? pb2[a] : k2;
      V.C(t, L::SI, a) = si[a];
      if (t >= 1) {
        // P_t = Qbar_t + A'(P A) + M'K
        const F npp = fma(mp[a], k1, V.k(AC::QB + a) + pp[a]);
        const F npv = fma(mp[a], k2, pav[a]);
        const F nvv = fma(mv[a], k2, fma(HET ? V.a22 : F(1), pvv[a], fma(V.dt, pav[a], V.k(AC::QB + DP + a))));
        pp[a] = npp;
        pv[a] = npv;
        vv[a] = nvv;
        V.C(t, L::PP, a) = npp;
        V.C(t, L::PV, a) = npv;
        V.C(t, L::VV, a) = nvv;
      }
    }
    if (V.c0 == 0) V.Cm[t * V.N] = (uint16_t)mask;
  }
  return bad;
}

// What a pass found: a free input left the box, a non-finite state, a held
// input whose multiplier is not surely positive, one that is not a number.
enum { PASS_OUT = 1, PASS_BAD = 2, PASS_MULT = 4, PASS_NAN = 8 };

// One EQP solve of the view's axes with the cached factors: backward affine
// pass, forward rollout (Sec. IV.B) writing Us and X.  Held inputs add no
// instruction to a stage: their lane puts other operands into the same ones.
// The next stage's operands are loaded one stage ahead.  The multipliers of held
// inputs decide only where one is negative, so in float64 their sign is taken
// from a float32 value with a margin over its error, and mult_scan forms them
// where that leaves a doubt.
template <bool HET, typename F, int NX, int NU, int DP, int AX>
__device__ __forceinline__ int axis_pass(const AxisView<F, NX, NU, DP, AX>& V) {
  using AC = AgentConst<NX, NU>;
  using L = AxisCache;
  const int T = V.T;
  int found = 0;
  F pn[AX], vn[AX];  // p_{t+1}: position and velocity rows
#pragma unroll
  for (int a = 0; a < AX; ++a) {
    pn[a] = lin_term(terminal_lin(V.qf[a], V.xr[a]), V.rho, V.hv(T, a));
    vn[a] = terminal_lin(V.qf[DP + a], V.xr[DP + a]);
  }
  uint32_t mask_n = V.Wm[(T - 1) * V.N];
  F g1n[AX], g2n[AX], sin_[AX], hn[AX];
#pragma unroll
  for (int a = 0; a < AX; ++a) {
    g1n[a] = V.C(T - 1, L::G1, a);
    g2n[a] = V.C(T - 1, L::G2, a);
    sin_[a] = V.C(T - 1, L::SI, a);
    hn[a] = T > 1 ? V.hv(T - 1, a) : F(0);
  }
  for (int t = T - 1; t >= 0; --t) {
    const uint32_t mask = mask_n;
    F g1[AX], g2[AX], si[AX], ht[AX];
#pragma unroll
    for (int a = 0; a < AX; ++a) {
      g1[a] = g1n[a];
      g2[a] = g2n[a];
      si[a] = sin_[a];
      ht[a] = hn[a];
    }
    if (t >= 1) {
      mask_n = V.Wm[(t - 1) * V.N];
#pragma unroll
      for (int a = 0; a < AX; ++a) {
        g1n[a] = V.C(t - 1, L::G1, a);
        g2n[a] = V.C(t - 1, L::G2, a);
        sin_[a] = V.C(t - 1, L::SI, a);
        hn[a] = t > 1 ? V.hv(t - 1, a) : F(0);
      }
    }
#pragma unroll
    for (int a = 0; a < AX; ++a) {
      const bool hd = V.held(mask, a);
      const F ub = V.bound(mask, a);
      const F bp = fma(V.b2, vn[a], V.b1 * pn[a]);  // B'p_{t+1}
      V.C(t, L::D, a) = hd ? bp : -(si[a] * bp);
      if (t >= 1) {
        // p_t = q_t + A'(p_{t+1} + P_{t+1}B u_held) + K'B'p_{t+1}; free: the last
        // term, held: the second (K = 0)
        const F qp = lin_term(V.k(AC::QL + a), V.rho, ht[a]), qv = V.k(AC::QL + DP + a);
        const F e1 = fma(hd ? g1[a] : F(1), hd ? ub : qp, pn[a]);
        const F e2 = fma(hd ? F(1) : g1[a], hd ? qp : bp, e1);
        const F f1 = fma(hd ? g2[a] : V.dt, hd ? ub : pn[a], hd ? vn[a] : qv);
        const F a22 = HET ? V.a22 : F(1);
        const F f2 = fma(hd ? V.dt : a22, hd ? e1 : vn[a], hd ? qv : f1);
        const F f3 = fma(hd ? a22 : g2[a], hd ? f1 : bp, f2);
        pn[a] = e2;
        vn[a] = f3;
      }
    }
  }

  // forward rollout
  unsigned long long kmin[AX], kmax[AX];
  F xp[AX], xv[AX], dn[AX];
  mask_n = V.Wm[0];
#pragma unroll
  for (int a = 0; a < AX; ++a) {
    kmin[a] = mono_key(V.lo[a]);
    kmax[a] = mono_key(V.hi[a]);
    xp[a] = V.xi[a];
    xv[a] = V.xi[DP + a];
    V.x(0, a) = xp[a];
    V.x(0, DP + a) = xv[a];
    g1n[a] = V.C(0, L::G1, a);
    g2n[a] = V.C(0, L::G2, a);
    dn[a] = V.C(0, L::D, a);
  }
  for (int t = 0; t < T; ++t) {
    const uint32_t mask = mask_n;
    F g1[AX], g2[AX], d[AX];
#pragma unroll
    for (int a = 0; a < AX; ++a) {
      g1[a] = g1n[a];
      g2[a] = g2n[a];
      d[a] = dn[a];
    }
    if (t + 1 < T) {
      mask_n = V.Wm[(t + 1) * V.N];
#pragma unroll
      for (int a = 0; a < AX; ++a) {
        g1n[a] = V.C(t + 1, L::G1, a);
        g2n[a] = V.C(t + 1, L::G2, a);
        dn[a] = V.C(t + 1, L::D, a);
      }
    }
#pragma unroll
    for (int a = 0; a < AX; ++a) {
      const bool hd = V.held(mask, a);
      const F uf = fma(g2[a], xv[a], fma(g1[a], xp[a], d[a]));
      const unsigned long long ku = mono_key(uf);
      if (!hd && ((ku < kmin[a]) | (ku > kmax[a]))) found |= PASS_OUT;
      const F u = hd ? V.bound(mask, a) : uf;
      xp[a] = fma(V.b1, u, fma(V.dt, xv[a], xp[a]));
      xv[a] = fma(V.b2, u, HET ? V.a22 * xv[a] : xv[a]);
      if (hd) {
        // multiplier +-(Rbar u + B'lambda_{t+1}), B'lambda_{t+1} = (P_{t+1}B)'x_{t+1} + B'p_{t+1}
        const bool low = (mask >> (V.c0 + a)) & 1u;
        if constexpr (std::is_same<F, double>::value) {
          const float a1 = near_f32(g1[a]) * near_f32(xp[a]), a2 = near_f32(g2[a]) * near_f32(xv[a]);
          const float a3 = near_f32(V.k(AC::RB + a)) * near_f32(u), a0 = near_f32(d[a]);
          const float g = (a0 + a1) + (a2 + a3);
          // each product is within 2^-22 of its own, each sum within 2^-23 of the sizes' sum
          const float size = (fabsf(a0) + fabsf(a1)) + (fabsf(a2) + fabsf(a3));
          const float tol = fmaf(size, kNearRel, kNearAbs);
          if (!((low ? g : -g) > tol)) found |= (g == g) ? PASS_MULT : (PASS_MULT | PASS_NAN);
        } else {
          const F g = fma(V.k(AC::RB + a), u, fma(g2[a], xv[a], fma(g1[a], xp[a], d[a])));
          const F mu = low ? g : -g;
          if (sign_set(mu)) found |= PASS_MULT;
          if (nan_key(abs_bits(mu), F(0))) found |= PASS_MULT | PASS_NAN;
        }
      }
      V.us(t, a) = u;
      V.x(t + 1, a) = xp[a];
      V.x(t + 1, DP + a) = xv[a];
    }
  }
#pragma unroll
  for (int a = 0; a < AX; ++a) {
    if (!(xp[a] == xp[a]) || fabs_(xp[a]) > F(1e30)) found |= PASS_BAD;
    if (!(xv[a] == xv[a]) || fabs_(xv[a]) > F(1e30)) found |= PASS_BAD;
  }
  return found;
}

// Refactorization and (PASS) EQP solve of the agents of the lanes with `go` (every
// lane of the warp calls this).  The FP64 pipe charges an instruction the same
// whatever the number of active lanes, so when the agents' axes fit the warp's
// lanes they take one lane each, and otherwise each lane takes its own agent,
// all axes.  Returns the pass's findings to the lane that owns the agent.
template <bool HET, bool PASS, typename F, int NX, int NU, int DP>
__device__ __forceinline__ int axis_round_of(const AgentCtx<F, NX, NU, DP>& A, bool go, int dirty,
                                             unsigned long long& nfact) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int NG = 32 / DP;  // agents whose axes fit a warp
  const unsigned owners = __ballot_sync(FULL, go);
  if (go && dirty >= 0) nfact += (unsigned long long)(dirty + 1);
  int found = 0;
  __syncwarp();
  constexpr bool lanes = std::is_same<F, double>::value || std::is_same<F, float>::value;
  if (lanes && A.coop && __popc(owners) <= NG) {
    const int lane = threadIdx.x & 31, g = lane / DP, gb = g * DP;
    unsigned m = owners;  // its lowest bit: the g-th owner
    for (int k = 0; k < g; ++k) m &= m - 1;
    const bool act = g < NG && m != 0;
    const int src = act ? __ffs(m) - 1 : lane;
    const AxisView<F, NX, NU, DP, 1> V = axis_view_of<F, NX, NU, DP>(A, src, act ? lane - gb : 0);
    const int od = __shfl_sync(FULL, dirty, src);
    if (axis_factor<HET>(V, act, od, act ? gb : 0)) found = PASS_BAD;
    __syncwarp();
    if constexpr (PASS) {
      if (act) found |= axis_pass<HET>(V);
      __syncwarp();
    }
    int all = 0;
    const int at = go ? __popc(owners & ((1u << lane) - 1u)) * DP : lane;
#pragma unroll
    for (int c = 0; c < DP; ++c) all |= __shfl_sync(FULL, found, go ? at + c : lane);
    found = all;
  } else if (go) {
    const AxisView<F, NX, NU, DP, DP> V = axis_view<F, NX, NU, DP>(A);
    if (axis_factor<HET>(V, true, dirty, 0)) found = PASS_BAD;
    if constexpr (PASS) found |= axis_pass<HET>(V);
  }
  __syncwarp();
  return go ? found : 0;
}

template <typename F, int NX, int NU, int DP, bool PASS = true>
__device__ __forceinline__ int axis_round(const AgentCtx<F, NX, NU, DP>& A, bool go, int dirty,
                                          unsigned long long& nfact) {
  return A.het ? axis_round_of<true, PASS>(A, go, dirty, nfact) : axis_round_of<false, PASS>(A, go, dirty, nfact);
}

// Ratio test (see ratio_test) of the agents of the lanes with `need`, into o.  The
// warp takes one agent at a time, its inputs spread over the lanes: 2 FP64
// instructions per 32 inputs and 2 per candidate, where one lane per agent takes 4
// per input of the warp's longest loop (8 per stage in 2D beside the 14 or 28 of a
// pass).  The smallest ratio comes out of the same comparisons num aden < anum den
// in index order as there, taken over the candidates alone: the inputs whose float32
// ratio is within 2^-18 of the smallest one's.  Any other ratio is larger than that
// by far more than the comparisons' rounding, so it can neither win nor stand in a
// winner's way.  A 512-agent 3D swarm over its first 20 iterations: 34.9 -> 30.2 ms,
// 200 small 3D swarms over 60: 64.4 -> 61.8 ms; the 4096-scenario batch, most of
// whose rounds do not block, is level.  Every lane of the warp calls this.
template <typename F, int NX, int NU, int DP>
__device__ void ratio_scan(const AgentCtx<F, NX, NU, DP>& A, bool need, EqpScan<F>& o) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int kKeep = 4;  // inputs per lane that stay in registers between the two passes
  const Model<F, NX, NU>& Mo = *A.M;
  const int lane = threadIdx.x & 31;
  for (unsigned rem = __ballot_sync(FULL, need); rem; rem &= rem - 1) {
    const int src = __ffs(rem) - 1;
    auto sp = [&](auto p) { return (decltype(p))__shfl_sync(FULL, (unsigned long long)p, src); };
    const uint16_t* const Wm = sp(A.Wm);
    const F* const U = sp(A.U);
    const F* const Us = sp(A.Us);
    const int N = __shfl_sync(FULL, A.N, src), n = __shfl_sync(FULL, A.T, src) * NU;
    const int i = __shfl_sync(FULL, A.i, src);
    // distance to the bound (at least 0) and size of the step of input e; false if it cannot block
    auto ratio = [&](int e, F& num, F& den, bool& lower) -> bool {
      const int t = e / NU, a = e - t * NU;
      if (e >= n || ((Wm[t * N + i] >> a) & 0x101u)) return false;
      const F cu = U[e * N + i], p = Us[e * N + i] - cu;
      const unsigned long long pb = abs_bits(p);
      if (pb == ord_bits(F(0))) return false;
      lower = sign_set(p);
      const F lo = a == 0 ? Mo.umin[0] : (a == 1 ? Mo.umin[1] : Mo.umin[NU - 1]);
      const F hi = a == 0 ? Mo.umax[0] : (a == 1 ? Mo.umax[1] : Mo.umax[NU - 1]);
      num = (lower ? cu : hi) - (lower ? lo : cu);
      if (sign_set(num)) num = F(0);
      den = from_bits(pb, F(0));
      return true;
    };
    // float32 bounds of the ratio: both operands cut to 24 bits (2^-23 each), one
    // division.  A distance that is cut to zero and is not zero has no bounds (NaN:
    // it stays a candidate and limits no other).
    auto low_of = [&](F num, F den, float& up) -> float {
      const float fn = near_f32(num);
      const bool lost = fn == 0.0f && abs_bits(num) != ord_bits(F(0));
      const float r = (lost ? __uint_as_float(0x7FC00000u) : fn) / near_f32(den);
      up = r < 1e-30f ? 1e-30f : r * (1.0f + 0x1p-19f);
      return r < 1e-30f ? 0.0f : r * (1.0f - 0x1p-19f);
    };
    F num[kKeep], den[kKeep];
    float low[kKeep];
    bool neg[kKeep], has[kKeep];
    float lim = 1.0f;
    for (int e0 = 0; e0 < n; e0 += 32 * kKeep) {
#pragma unroll
      for (int j = 0; j < kKeep; ++j) {
        has[j] = ratio(e0 + 32 * j + lane, num[j], den[j], neg[j]);
        float up = 1.0f;
        low[j] = has[j] ? low_of(num[j], den[j], up) : 0.0f;
        if (has[j] && up < lim) lim = up;
      }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) lim = fminf(lim, __shfl_xor_sync(FULL, lim, off));
    F anum = F(1), aden = F(1);
    int blk = -1, side = 0;
    for (int e0 = 0; e0 < n; e0 += 32 * kKeep) {
#pragma unroll
      for (int j = 0; j < kKeep; ++j) {
        if (n > 32 * kKeep) {
          has[j] = ratio(e0 + 32 * j + lane, num[j], den[j], neg[j]);
          float up;
          low[j] = has[j] ? low_of(num[j], den[j], up) : 0.0f;
        }
        unsigned cand = __ballot_sync(FULL, has[j] && !(low[j] > lim));
        const unsigned down = __ballot_sync(FULL, neg[j]);
        for (; cand; cand &= cand - 1) {
          const int l = __ffs(cand) - 1;
          const F cn = shfl_f(num[j], l), cd = shfl_f(den[j], l);
          if (mono_key(cn * aden) < mono_key(anum * cd)) {
            anum = cn;
            aden = cd;
            blk = e0 + 32 * j + l;
            side = (down >> l) & 1u ? 1 : 2;
          }
        }
      }
    }
    if (lane == src) {
      o.anum = anum;
      o.aden = aden;
      o.blk = blk;
      o.bside = side;
    }
  }
}

// u <- u + alpha (us - u) for the agents of the lanes with `need`, the warp taking
// one agent at a time.  Every lane of the warp calls this.
template <typename F, int NX, int NU, int DP>
__device__ void step_scan(const AgentCtx<F, NX, NU, DP>& A, bool need, F alpha) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  for (unsigned rem = __ballot_sync(FULL, need); rem; rem &= rem - 1) {
    const int src = __ffs(rem) - 1;
    auto sp = [&](auto p) { return (decltype(p))__shfl_sync(FULL, (unsigned long long)p, src); };
    F* const U = sp(A.U);
    const F* const Us = sp(A.Us);
    const int N = __shfl_sync(FULL, A.N, src), n = __shfl_sync(FULL, A.T, src) * NU;
    const int i = __shfl_sync(FULL, A.i, src);
    const F al = shfl_f(alpha, src);
    for (int e = lane; e < n; e += 32) {
      const F cu = U[e * N + i];
      U[e * N + i] = fma(al, Us[e * N + i] - cu, cu);
    }
  }
  __syncwarp();
}

// Multipliers of the held inputs of the agents of the lanes with `need`: the
// most negative one (the lowest index of equal ones), the largest magnitude and
// a NaN flag, into o.  The warp takes one agent at a time, its inputs spread
// over the lanes.  Every lane of the warp calls this.
template <typename F, int NX, int NU, int DP>
__device__ void mult_scan(const AgentCtx<F, NX, NU, DP>& A, bool need, EqpScan<F>& o) {
  using AC = AgentConst<NX, NU>;
  using L = AxisCache;
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  for (unsigned rem = __ballot_sync(FULL, need); rem; rem &= rem - 1) {
    const int src = __ffs(rem) - 1;
    auto sp = [&](auto p) { return (decltype(p))__shfl_sync(FULL, (unsigned long long)p, src); };
    const F* const cache = sp(A.cache);
    const uint16_t* const Wm = sp(A.Wm);
    const F* const Us = sp(A.Us);
    const F* const Xo = sp(A.Xo);
    const F* const kc = sp(A.kc);
    const int N = __shfl_sync(FULL, A.N, src), T = __shfl_sync(FULL, A.T, src);
    const int i = __shfl_sync(FULL, A.i, src), ks = __shfl_sync(FULL, A.ks, src);
    F worst = F(0), scale = F(1);
    int widx = -1, bad = 0;
    for (int e = lane; e < T * NU; e += 32) {
      const int t = e / NU, a = e - t * NU;
      const uint32_t mask = Wm[t * N + i];
      if (!((mask >> a) & 0x101u)) continue;
      auto C = [&](int w) { return cache[((t * L::E + w) * DP + a) * N + i]; };
      F g = C(L::D);
      g = fma(C(L::G1), Xo[((t + 1) * NX + a) * N + i], g);
      g = fma(C(L::G2), Xo[((t + 1) * NX + DP + a) * N + i], g);
      g = fma(kc[(AC::RB + a) * ks], Us[(t * NU + a) * N + i], g);
      const F mu = ((mask >> a) & 1u) ? g : -g;
      const unsigned long long ab = abs_bits(mu);
      if (ab > abs_bits(scale)) scale = from_bits(ab, F(0));
      if (mono_key(mu) < mono_key(worst)) { worst = mu; widx = e; }
      if (nan_key(ab, F(0))) bad = 1;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const F w2 = shfl_f(worst, lane ^ off), s2 = shfl_f(scale, lane ^ off);
      const int i2 = __shfl_sync(FULL, widx, lane ^ off), b2 = __shfl_sync(FULL, bad, lane ^ off);
      const unsigned long long k1 = mono_key(worst), k2 = mono_key(w2);
      if (i2 >= 0 && (widx < 0 || k2 < k1 || (k2 == k1 && i2 < widx))) {
        worst = w2;
        widx = i2;
      }
      if (abs_bits(s2) > abs_bits(scale)) scale = s2;
      bad |= b2;
    }
    if (lane == src) {
      o.worst = worst;
      o.widx = widx;
      o.scale = scale;
      o.bad |= bad;
    }
  }
}

}  // namespace tadmm
