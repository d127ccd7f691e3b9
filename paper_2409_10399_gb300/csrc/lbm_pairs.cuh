// The FP32 step of a D2Q9 or D3Q19 node with the two phases' arithmetic in
// pairs (packed float instructions).  Included by lbm_kernels.cuh, whose
// fused_step_node it stands in for there: the same method, rounded in another
// order.  Not for the stores with half planes: their rounding feeds back on
// itself, so that any other rounding of the arithmetic leaves the fields as far
// from the scalar form's as both are from the exact ones; nor for D1Q3.
// Measured (us per step; scalar and launched in order -> paired and overlapped):
// 2D box of 512 x 2048 with its inlet 80.3 -> 79.8, 256 x 1024 16.8 -> 14.5, 3D column
// of 256 x 256 x 128 1,647 -> 1,423, of 150 x 122 x 250 996 -> 839, 48 ragged 2D
// columns 1,559 -> 1,427.  2D: instructions 49.2 -> 36.5 M per launch, and
// the step waits on memory (6.2 long-scoreboard stalls per issue); more warps
// would help, but the registers of five blocks are all taken (StepBounds).
#pragma once

namespace lbm {

// A quantity of the gas and the liquid.  The two phases' schemes are relaxed by
// the same formulas with constants of their own, so the node's arithmetic is
// written on pairs, each one operand of the packed instructions (add, mul,
// fma.rn.f32x2, every component rounded as by the scalar one).  They take the
// FP32 pipe as long as two scalar instructions but one issue slot and one place
// in the code, and both count: the step is straight-line code that every warp
// runs once.  Every operation is rounded one by one, so that the interior and the
// general path give the same bits.
struct Two {
  float g, l;
};
__device__ __forceinline__ Two both(float x) { return Two{x, x}; }
struct T2 {
  typedef Two V;
  static __device__ __forceinline__ V add(V a, V b) {
    const float2 r = __fadd2_rn(make_float2(a.g, a.l), make_float2(b.g, b.l));
    return V{r.x, r.y};
  }
  static __device__ __forceinline__ V mul(V a, V b) {
    const float2 r = __fmul2_rn(make_float2(a.g, a.l), make_float2(b.g, b.l));
    return V{r.x, r.y};
  }
  static __device__ __forceinline__ V fma(V a, V b, V c) {
    const float2 r = __ffma2_rn(make_float2(a.g, a.l), make_float2(b.g, b.l), make_float2(c.g, c.l));
    return V{r.x, r.y};
  }
  // a b - c and c - a b: scalar instructions, whose operands take a sign (a
  // packed one would need the negated pair in registers)
  static __device__ __forceinline__ V fms(V a, V b, V c) { return V{__fmaf_rn(a.g, b.g, -c.g), __fmaf_rn(a.l, b.l, -c.l)}; }
  static __device__ __forceinline__ V fnma(V a, V b, V c) { return V{__fmaf_rn(-a.g, b.g, c.g), __fmaf_rn(-a.l, b.l, c.l)}; }
  // a - b, rounded once (b times -1 is exact)
  static __device__ __forceinline__ V sub(V a, V b) { return fma(b, both(-1.0f), a); }
};

// v_q . u of both phases, for a direction whose first nonzero component is
// +1 (q > opp q)
template <class L>
__device__ __forceinline__ Two vdot_two(int q, const Two u[3]) {
  Two s = both(0.0f);
  bool first = true;
#pragma unroll
  for (int d = 0; d < L::D; d++) {
    const int vd = L::v(q, d);
    if (vd == 0) continue;
    s = first ? u[d] : (vd > 0 ? T2::add(s, u[d]) : T2::sub(s, u[d]));
    first = false;
  }
  return s;
}
// v_q . u = s + e exactly: the sum of its at most two nonzero terms
// (D2Q9, D3Q19 diagonals) as a two-sum, e = 0 along the axes (false).
template <class L>
__device__ __forceinline__ bool vdot2(int q, const Two u[3], Two &s, Two &e) {
  typedef T2 O;
  Two t[2] = {both(0.0f), both(0.0f)};
  int n = 0;
  bool minus = false;
#pragma unroll
  for (int d = 0; d < L::D; d++) {
    const int vd = L::v(q, d);
    if (vd != 0 && n < 2) {
      t[n++] = u[d];
      minus = vd < 0;
    }
  }
  s = t[0];
  if (n < 2) return false;
  s = minus ? O::sub(t[0], t[1]) : O::add(t[0], t[1]);
  const Two bb = O::sub(s, t[0]), r = O::sub(t[0], O::sub(s, bb));
  e = minus ? O::sub(r, O::add(t[1], bb)) : O::add(r, O::sub(t[1], bb));
  return true;
}

// population q of the schemes of pair p: (g, l), (alpha_g, alpha_l), (beta_g, beta_l)
template <class L>
__device__ __forceinline__ Two two(const Pops<L, float, float, false> &P, int p, int q) {
  return Two{P.f[2 * p][q], P.f[2 * p + 1][q]};
}

template <class L> struct PairMoments {
  Two de;            // eps_g - 1, eps_l - 1
  Two u[3];
  Two mP[6];         // -(Pi - cs2 I), packed as in Moments
  Two a, mJ[3];      // a, and minus the first moment J, of f_alpha
  Two da;            // a - r
  float esum;        // a_g + a_l - (r_g + r_l), summed direction by direction
  Two S;             // 1 - beta
  Two al;            // alpha^B
  float dalg;        // alpha^B_g - r_g
  Two c;             // alpha^B - a
};

template <class L>
__device__ __forceinline__ void pair_sums(const Pops<L, float, float, false> &P, PairMoments<L> &m) {
  typedef T2 O;
  constexpr int D = L::D;
  m.de = two(P, 0, 0);
  m.a = two(P, 1, 0);
  m.S = two(P, 2, 0);
  m.esum = Rn<float>::add(m.a.g, m.a.l);
#pragma unroll
  for (int d = 0; d < 3; d++) m.u[d] = m.mJ[d] = both(0.0f);
#pragma unroll
  for (int k = 0; k < 6; k++) m.mP[k] = both(0.0f);
  bool u0[3] = {true, true, true};  // no term yet
#pragma unroll
  for (int q = 1; q < L::Q; q++) {
    const int qo = L::opp(q);
    if (q > qo) continue;
    const Two f0 = two(P, 0, q), g0 = two(P, 0, qo), f1 = two(P, 1, q), g1 = two(P, 1, qo);
    const Two sm = O::add(f0, g0), sa = O::add(f1, g1), sb = O::add(two(P, 2, q), two(P, 2, qo));
    // f_q - f_opp(q) and its negative
    const Two df = O::sub(f0, g0), dn = O::sub(g0, f0), ja = O::sub(f1, g1), jn = O::sub(g1, f1);
    m.de = O::add(m.de, sm);
    m.a = O::add(m.a, sa);
    m.S = O::add(m.S, sb);
    m.esum = Rn<float>::add(m.esum, Rn<float>::add(Rn<float>::add(f1.g, f1.l), Rn<float>::add(g1.g, g1.l)));
#pragma unroll
    for (int d = 0; d < D; d++) {
      const int vd = L::v(q, d);
      if (vd != 0) {
        m.u[d] = u0[d] ? (vd > 0 ? df : dn) : (vd > 0 ? O::add(m.u[d], df) : O::sub(m.u[d], df));
        m.mJ[d] = u0[d] ? (vd > 0 ? jn : ja) : (vd > 0 ? O::sub(m.mJ[d], ja) : O::add(m.mJ[d], ja));
        u0[d] = false;
      }
#pragma unroll
      for (int e = d; e < D; e++) {
        const int vv = vd * L::v(q, e), k = pidx(d, e);
        if (vv != 0) m.mP[k] = vv > 0 ? O::sub(m.mP[k], sm) : O::add(m.mP[k], sm);
      }
    }
  }
  m.S = O::mul(m.S, both(-1.0f));
}

template <class L>
__device__ __forceinline__ void pair_moments(const StepArgs &a, const Pops<L, float, float, false> &f, PairMoments<L> &m) {
  typedef T2 O;
  typedef Rn<float> N;
  const PhysT<float> &P = phys<float>(a);
  pair_sums<L>(f, m);
  m.da = m.a;
  m.a = O::add(m.a, Two{P.r_ag, P.r_al});
  m.c = both(0.0f);
  if (a.spalding == 0) {
    m.al = m.a;
    m.dalg = m.da.g;
  } else {
    // Eq. (spalding) in deviations, the renormalisation kept as a number of its
    // own (moments)
    if (m.a.g >= 0.0f && m.a.g <= 1.0f && m.a.l >= 0.0f && m.a.l <= 1.0f && N::add(m.a.g, m.a.l) > 0.0f) {
      const float e = N::add(m.esum, P.rsum1);
      const float k = e / N::add(1.0f, e);
      m.c = O::mul(m.a, both(-k));
      m.dalg = N::add(m.da.g, m.c.g);
    } else {
      float Bg = m.a.g < 0.0f ? 0.0f : (m.a.g > 1.0f ? 1.0f : m.a.g);
      float Bl = m.a.l < 0.0f ? 0.0f : (m.a.l > 1.0f ? 1.0f : m.a.l);
      float sum = N::add(Bg, Bl);
      m.dalg = N::sub(sum > 0.0f ? Bg / sum : 0.5f, P.r_ag);
      m.c.g = N::sub(m.dalg, m.da.g);
      m.c.l = N::sub(N::sub(-m.dalg, P.rsum1), m.da.l);
    }
    m.al.g = N::add(P.r_ag, m.dalg);
    m.al.l = N::add(P.r_al, N::sub(-m.dalg, P.rsum1));  // alpha^B_l = 1 - alpha^B_g
  }
}

// One node: fused_step_node's contract (S = R = float, six schemes).
template <class L, class OffT, bool IO>
__device__ __forceinline__ void paired_step_node(const StepArgs &a, Geo &g, bool active, int tid, int parity, int latch,
                                                 bool blk_xch, int gstride, float *xch) {
  typedef float R;
  typedef T2 O;
  typedef Rn<float> N;
  constexpr int D = L::D, Q = L::Q;
  const int gax = a.g_axis;
  Pops<L, float, float, false> f;
  PairMoments<L> m;
  Two c[3] = {both(0.0f), both(0.0f), both(0.0f)};
  bool interior = false;
  if (active) {
    make_geo(a, D, g);
    interior = !(g.xp[0] || g.xm[0] || g.xp[1] || g.xm[1] || g.xp[2] || g.xm[2]);
  }
  interior = __all_sync(__activemask(), interior);
  if (active) {
    if (interior) load_node<L, float, float, false, OffT, true>(a, g, parity, f);
    else load_node<L, float, float, false, OffT>(a, g, parity, f);
  }
  if (active) {
    pair_moments<L>(a, f, m);
#pragma unroll
    for (int d = 0; d < D; d++) {
      // Eq. (velocitybeta) with beta = 1: alpha_l (u_g - u_l), alpha_g (u_l - u_g)
      const R dv = N::sub(m.u[d].g, m.u[d].l);
      c[d] = O::mul(Two{m.al.l, m.al.g}, Two{dv, -dv});
    }
  }
  if (IO && blk_xch) {
    if (active) {
#pragma unroll
      for (int d = 0; d < 3; d++) {
        xch[tid * XCH + d] = m.u[d].g;
        xch[tid * XCH + 3 + d] = m.u[d].l;
        xch[tid * XCH + 8 + d] = c[d].g;
        xch[tid * XCH + 11 + d] = c[d].l;
      }
      xch[tid * XCH + 6] = m.al.g;
      xch[tid * XCH + 7] = m.al.l;
    }
    __syncthreads();
  }
  if (!active) return;

  const PhysT<R> &P = phys<R>(a);
  const R R_ = P.R_, invR = P.invR;
  // ---- sources: Eq. (lbmbetataylorzeroth5), dashpot Eqs. (lbm-cont-g1Dhat),
  //      (lbm-cont-l1Dhat) third strategy with phi*eps_l - 1 = (eps_g - 1)/R
  const Two dp = {m.de.g, N::mul(m.de.g, invR)};  // eps_g - 1, phi eps_l - 1
  Two u2 = O::mul(m.u[0], m.u[0]);
#pragma unroll
  for (int d = 1; d < D; d++) u2 = O::fma(m.u[d], m.u[d], u2);
  float *held = (float *)a.held;
  Two Spp;
  R Lam;
  if (latch) {
    Spp = O::fma(O::mul(both(-P.gamma), u2), dp, m.S);
    Lam = N::mul(N::mul(m.al.g, m.al.l), N::fma(m.al.l, R_, m.al.g));  // Eq. (Lambda)
    held[g.node] = Spp.g;
    held[a.plane + g.node] = Spp.l;
    held[2 * a.plane + g.node] = Lam;
  } else {
    Spp.g = held[g.node];
    Spp.l = held[a.plane + g.node];
    Lam = held[2 * a.plane + g.node];
  }

  // ---- grad(alpha): Eq. (gradlnalpha) times alpha, corrected by Eq. (spalding2);
  //      grad^G alpha_l = -grad^G alpha_g
  Two gG[3];
#pragma unroll
  for (int d = 0; d < D; d++) {
    const Two gr = O::mul(both(P.kgrad), O::fma(m.a, m.u[d], m.mJ[d]));
    const R v = N::mul(0.5f, N::sub(gr.g, gr.l));
    gG[d] = Two{v, -v};
  }

  // ---- stress sigma = A (Pi^eq - Pi) + B S'' I (Eq. (lbm-sigma3); D = 1:
  //      Eq. (taylor-second31Db)), Pi^eq from Eq. (secondtensoreq)
  Two sG[3];
  {
    const Two A = {P.A_g, P.A_l}, BS_ = O::mul(Two{P.B_g, P.B_l}, Spp);
    Two AN[6];
#pragma unroll
    for (int d = 0; d < D; d++)
#pragma unroll
      for (int e = d; e < D; e++) {
        const int k = pidx(d, e);
        Two n = O::fma(m.u[d], m.u[e], m.mP[k]);
        if (d == e) n = O::fma(both(1.0f / 3.0f), dp, n);
        AN[k] = O::mul(A, n);
      }
#pragma unroll
    for (int d = 0; d < D; d++) {
      sG[d] = O::mul(BS_, gG[d]);
#pragma unroll
      for (int e = 0; e < D; e++) sG[d] = O::fma(AN[pidx(d, e)], gG[e], sG[d]);
    }
  }

  // ---- drag (Eq. (interphasemomentum), CGW Eq. (CliftGraceWeber)), wall
  //      friction (Eq. (wallmomentum1D)), forces Eqs. (Gg), (Gl), (Gg1D)
  Two G[3] = {both(0.0f), both(0.0f), both(0.0f)};
  {
    R du[3], du2 = 0.0f;
#pragma unroll
    for (int d = 0; d < D; d++) {
      du[d] = N::sub(m.u[d].l, m.u[d].g);
      du2 = N::fma(du[d], du[d], du2);
    }
    const R KI = N::mul(a.cgw ? N::mul(P.kappa_I, Lam) : P.kappa_I, sqrt(du2));
    const R KW = N::mul(a.cgw ? N::mul(P.kappa_W, Lam) : P.kappa_W, sqrt(u2.l));
    const R fl = P.afloor;
    const Two inv = {1.0f / (m.al.g > fl ? m.al.g : fl), 1.0f / (m.al.l > fl ? m.al.l : fl)};
#pragma unroll
    for (int d = 0; d < D; d++) {
      const R x = N::mul(KI, du[d]);
      const Two fr = {x, N::mul(N::fma(KW, m.u[d].l, x), -invR)};
      G[d] = O::fma(O::add(sG[d], fr), inv, O::mul(Spp, m.u[d]));
      if (d == a.g_axis) G[d].g = N::add(G[d].g, P.buoy);
    }
  }

  // ---- collisions and AA store with face rules
  const Two om = {P.omega_g, P.omega_l}, om_a = both(P.omega_a);
  // f_alpha relaxes to f^eq(alpha^B, u) (Spalding mode 2) or f^eq(a, u):
  // its even part w [(alpha^B - r) + alpha^B q] is taken as
  // w [(a - r) + a q] + w c (1 + q) with c = alpha^B - a (0 unless mode 2),
  // so that c is not lost to the spacing of a - r
  const Two aeq = a.spalding == 2 ? m.al : m.a;
  const Two ceq = a.spalding == 2 ? m.c : both(0.0f);
  const R rag = P.r_ag, ral = P.r_al;
  // Eq. (eta) for the moving directions: eta_q(phi) = phi, so the offsets of
  // f_I^eq - w are eps_g - 1 (phi_g = 1) and phi eps_l - 1 = dp.l, and f_L's
  // is S psi.  The rest direction's takes what makes the zeroth moments
  // exact with the weights in use (sum w_q = 1): w_0 eta_0 = 1 - (1 - w_0)
  // phi, so its f_I^eq is the remainder of the moving directions' (taken as
  // such by the rest direction's collision below), and w_0 f_L(0) = S -
  // (1 - w_0) psi S, (1 - w_0) x formed as x - w_0 x so that no rounded
  // 1 - w_0 biases it.
  const Two psi = {P.psi_g, P.psi_l}, eLq = O::mul(Spp, psi);
  // -3/2 u.u and -3/2 c.c of the quadratic terms
  Two c2 = both(0.0f);
#pragma unroll
  for (int d = 0; d < D; d++) c2 = O::fma(c[d], c[d], c2);
  const Two qc0 = O::mul(both(-1.5f), c2), qu0 = O::mul(both(-1.5f), u2);

  // f_beta at a face, EQ(S) with c extrapolated full-way from the neighbour xn
  auto beta_ext = [&](const int qo, const R *xn) {
    R cb[3] = {0.0f, 0.0f, 0.0f}, cc[3] = {0.0f, 0.0f, 0.0f};
    Two o;
#pragma unroll
    for (int d = 0; d < D; d++) {
      cb[d] = N::fma(2.0f, c[d].g, -xn[8 + d]);
      cc[d] = N::fma(2.0f, c[d].l, -xn[11 + d]);
    }
    beta_pair<L, R>(qo, cb, cc, o.g, o.l);
    return o;
  };
  // face rules of direction q (walls, Tables 1-2) and its AA store; INTc
  // (std::true_type for interior nodes) compiles them out
  auto finish = [&](const int q, Two out[3], auto INTc) {
    constexpr bool INT = decltype(INTc)::value;
    const R w = wq<L, R>(q);
    const bool cross = !INT && crosses<L>(g, q, +1);
    if (IO && cross) {
      const int rule = face_rule<L>(a, g, q);
      const int qo = L::opp(q);
      if (rule == BC_INLET) {
        // Table 1: f_g, f_l BB(I) (Eq. (BB): -2 w v.u^B/cs2), f_alpha EQ(S)
        // Dirichlet, f_beta EQ(S) with beta and c extrapolated full-way.
        const R vq = (R)(gax == 0 ? L::v(q, 0) : (gax == 1 ? L::v(q, 1) : L::v(q, 2)));
        const R b2 = N::mul(-2.0f * aq<L, R>(q), vq);
        out[0] = O::fma(both(b2), Two{P.ugIN, P.ulIN}, out[0]);
        R uin[3], lin[3];
#pragma unroll
        for (int d = 0; d < 3; d++) {
          uin[d] = d == gax ? P.ugIN : 0.0f;
          lin[d] = d == gax ? P.ulIN : 0.0f;
        }
        out[1].g = feqS_dev<L, R>(qo, P.aIN, uin, P.ugIN * P.ugIN, rag);
        out[1].l = feqS_dev<L, R>(qo, 1.0f - P.aIN, lin, P.ulIN * P.ulIN, ral);
        out[2] = beta_ext(qo, xch + (tid + gstride) * XCH);
      } else if (rule == BC_OUTLET) {
        // Table 2: f_g, f_l ABB(I) with eps = 1 (so phi = 1) and u EX(hw);
        // f_alpha ABB(S) with alpha, u EX(hw); f_beta EQ(S) with c EX(fw).
        const R *xn = xch + (tid - gstride) * XCH;
        R ubg[3] = {0.0f, 0.0f, 0.0f}, ubl[3] = {0.0f, 0.0f, 0.0f};
        R ubg2 = 0.0f, ubl2 = 0.0f;
#pragma unroll
        for (int d = 0; d < D; d++) {
          ubg[d] = N::fma(1.5f, m.u[d].g, N::mul(-0.5f, xn[d]));
          ubl[d] = N::fma(1.5f, m.u[d].l, N::mul(-0.5f, xn[3 + d]));
          ubg2 = N::fma(ubg[d], ubg[d], ubg2);
          ubl2 = N::fma(ubl[d], ubl[d], ubl2);
        }
        const R vbg = vdot<L, R>(q, ubg), vbl = vdot<L, R>(q, ubl);
        const Two qq = {N::fma(N::mul(4.5f, vbg), vbg, N::mul(-1.5f, ubg2)),
                           N::fma(N::mul(4.5f, vbl), vbl, N::mul(-1.5f, ubl2))};
        const Two ab = {N::fma(1.5f, m.al.g, N::mul(-0.5f, xn[6])),
                           N::fma(1.5f, m.al.l, N::mul(-0.5f, xn[7]))};
        out[0] = O::sub(O::mul(both(2.0f * w), qq), out[0]);
        out[1] = O::sub(O::mul(both(2.0f * w), O::fma(ab, qq, O::sub(ab, Two{rag, ral}))), out[1]);
        out[2] = beta_ext(qo, xn);
      }
      // BC_WALL: half-way bounce-back keeps out[] as is
    }
    int pq;
    const long long idx = write_slot<L>(a, g, q, cross, parity, pq);
    const OffT off = pop_offset<L, OffT>(a, pq, idx);
#pragma unroll
    for (int p = 0; p < 3; p++) {
      Store<float>::st((float *)scheme_base<L, float>(a, 2 * p) + off, out[p].g);
      Store<float>::st((float *)scheme_base<L, float>(a, 2 * p + 1) + off, out[p].l);
    }
  };

  // Collisions: the moving directions in pairs (q, opp q), q the one whose first
  // component is +1, the rest direction last, its non-equilibrium part the
  // remainder of theirs (fused_step_node says why, and why the hi + lo forms).
  // The rest direction's four populations wait in shared memory meanwhile: four live
  // registers fewer, so fewer spills (the scalar form's 2D box 99 -> 80 us).
  constexpr int NST = StepBounds<L, float>::threads;
  __shared__ float rest_stash[4 * NST];
  volatile R *const stash = rest_stash + threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
  auto rest_f = [&](int p) -> Two {
    return Two{stash[2 * p * NST], stash[(2 * p + 1) * NST]};
  };
  auto collide_rest = [&](const Two nsum[2], auto INTc) {
    const R wu = wq<L, R>(0);
    Two out[3];
    const Two rest_L = O::sub(Spp, O::mul(psi, O::fma(both(-wu), Spp, Spp)));
    out[0] = O::add(rest_f(0), O::fnma(om, nsum[0], rest_L));
    out[1] = O::fma(om_a, O::sub(ceq, nsum[1]), rest_f(1));
    out[2] = O::mul(both(wu), qc0);  // v_0 = 0
    finish(0, out, INTc);
  };

  auto collide_all = [&](auto INTc) {
  Two nsum[2] = {both(0.0f), both(0.0f)};  // sum over the moving directions of f^eq - f
#pragma unroll
  for (int s = 0; s < 4; s++) stash[s * NST] = f.f[s][0];
#pragma unroll
  for (int qo = 1; qo < Q; qo++) {
    const int q = L::opp(qo);
    if (q > qo) {
      const Two w = both(wq<L, R>(q)), aw = both(aq<L, R>(q));
      const Two vG = vdot_two<L>(q, G);
      // v . u = vs + ve exactly (a two-sum of its at most two nonzero terms)
      Two vs, ve;
      const bool diag = vdot2<L>(q, m.u, vs, ve);
      const Two qu = O::fma(O::mul(both(4.5f), vs), vs, qu0);
      // even parts of f_I^eq - w and odd parts a_q v . u as hi + lo
      const Two X = O::mul(w, dp);
      const Two Xl = O::fma(w, qu, O::fms(w, dp, X));
      const Two Y = O::mul(aw, vs);
      Two Yl = O::fms(aw, vs, Y);
      if (diag) Yl = O::fma(aw, ve, Yl);
      const Two F = O::mul(w, eLq), Hf = O::mul(aw, vG);
      // f_alpha: alpha^B = a + c (c the renormalisation, Spalding mode 2)
      const Two Xa = O::mul(w, m.da);
      // (Two groupings of the same sum, by the lattice and the rules compiled in,
      // not by size.  D2Q9 is held to 96 registers for its five blocks: with an
      // inlet the shorter grouping's code spills where it hurts, 2D box 85.7 us a
      // step against 79.8; without, 256 x 1024 14.6 against 15.0.  To be measured
      // again when the launch bounds, the face rules or the compiler change.)
      Two Xal;
      if (IO && Q == 9) {
        Xal = O::add(O::add(O::fms(w, m.da, Xa), O::mul(w, O::mul(m.a, qu))), O::mul(w, O::mul(ceq, O::add(both(1.0f), qu))));
      } else {
        const Two al_q = O::fma(m.a, qu, O::fma(ceq, qu, ceq));  // a q + c (1 + q)
        Xal = O::fma(w, al_q, O::fms(w, m.da, Xa));
      }
      const Two Ya = O::mul(aeq, Y);
      const Two fi = two(f, 0, q), fio = two(f, 0, qo), fa = two(f, 1, q), fao = two(f, 1, qo);
      auto neq = [&](Two fv, bool minus) {  // (X - fv) + X_lo +- (Y + Y_lo), X - fv as the exact s + e
        const Two s = O::sub(X, fv), sy = minus ? O::sub(s, Y) : O::add(s, Y);
        const Two bb = O::sub(s, X);
        const Two e = O::sub(O::sub(X, O::sub(s, bb)), O::add(fv, bb));
        return O::add(sy, O::add(e, minus ? O::sub(Xl, Yl) : O::add(Xl, Yl)));
      };
      const Two ta[2] = {neq(fi, false), O::add(O::add(O::sub(Xa, fa), Xal), Ya)};
      const Two tb[2] = {neq(fio, true), O::sub(O::add(O::sub(Xa, fao), Xal), Ya)};
#pragma unroll
      for (int p = 0; p < 2; p++) nsum[p] = O::add(nsum[p], O::add(ta[p], tb[p]));
      Two oa[3], ob[3];
      oa[0] = O::add(fi, O::fma(om, ta[0], O::add(F, Hf)));
      ob[0] = O::add(fio, O::fma(om, tb[0], O::sub(F, Hf)));
      oa[1] = O::fma(om_a, ta[1], fa);
      ob[1] = O::fma(om_a, tb[1], fao);
      {
        // beta_dev of q and opp(q) from one even part (v_opp . c = -v_q . c exactly)
        const Two vc = vdot_two<L>(q, c);
        const Two x = O::mul(w, O::fma(O::mul(both(4.5f), vc), vc, qc0));
        oa[2] = O::fma(aw, vc, x);
        ob[2] = O::fnma(aw, vc, x);
      }
      // (The order of the stores, the same bits either way: D2Q9, at 96
      // registers, 79.5 us a step of the 2D box this way and 84.3 the other, D3Q19
      // FP32, at 168, 1.40 ms at 256 x 256 x 128 this way and 1.47 the other.  Like
      // the grouping above it is the register allocation's choice, to be measured
      // again when the launch bounds or the compiler change.)
      if (Q == 19) {
        finish(qo, ob, INTc);
        finish(q, oa, INTc);
      } else {
        finish(q, oa, INTc);
        finish(qo, ob, INTc);
      }
    }
  }
  collide_rest(nsum, INTc);
  };
  if (interior) collide_all(std::true_type{});
  else collide_all(std::false_type{});
}

}  // namespace lbm
