// FP64 reference path of short 1D lattices: several steps in one launch.
#pragma once
#include "lbm_ref.cuh"

namespace lbm {

// A step of a few hundred nodes is a dependent chain of FP64 operations on a
// nearly empty GPU.  One FP64 instruction of a warp takes its SM quarter 64
// cycles (76 with all four quarters busy), however many lanes are active and
// whether or not it depends on the last one, so the step's time is 64 cycles
// times the instructions a warp executes.  Hence:
//  - a node takes eight lanes: one per scheme (f_I, f_alpha, f_beta of the gas
//    and of the liquid; each holds its three populations) and two spare.  The
//    two phases' formulas are the same with phi = 1 for the gas, and the
//    schemes' collisions have one shape, f + omega (W (E +- v.u/cs2 + quad) -
//    f), so all lanes run one instruction stream on their own operands; the
//    node's six divisions run as three, each lane dividing a pair of its own.
//    About 95 FP64 instructions a step instead of 190 for a thread per node;
//  - the populations stay in registers over `steps` steps: a block of 16
//    nodes also holds the steps - 1 nodes beyond its core on either side
//    (each step makes one more of them stale) and stores its core only.  The
//    launch reads one store and writes another (pop_out, held_out), so no
//    block reads what another writes.
// The expressions and their order are those of k_step_ref, and so are the
// results, bit for bit.
// Measured (us per step; against k_step_ref, a thread per node and a launch
// per step, with the same divisions): 512 nodes between walls 6.1 against
// 12.6, 200 nodes with inlet and outlet 7.7 against 21.0; about 5.3 us a step
// plus 5 us a launch while an SM holds one block, 8.8 us with two.

// |x| = sqrt(x x): exact in radix 2 unless x x leaves the normal range (below
// 2^-300 and for all finite x from 2^500 on the formula as it stands is taken; S.
// Boldo, "Stupid is as stupid does: taking the square root of the square of
// a floating-point number", 2015)
__device__ __forceinline__ double r1_abs(double x) {
  const unsigned h = (unsigned)__double2hiint(x) & 0x7fffffffu;
  if (ref_small(x) || h - ((1023u + 500u) << 20) < (524u << 20)) return sqrt(x * x);
  return fabs(x);
}
// first + x/cs2 + quad and first - x/cs2 + quad, x = v.u of the +1 direction
__device__ __forceinline__ void r1_feq(const RefConst &k, double first, double x, double &plus, double &minus) {
  const double n = x * x - k.cs2 * (x * x);
  const bool s = ref_small(x);
  const double a = s ? x / k.cs2 : div_cs2<true>(x, k), b = s ? n / k.two_cs4 : div_two_cs4<true>(n, k);
  plus = first + a + b;
  minus = first - a + b;
}

__global__ void __launch_bounds__(8 * R1_NODES) k_steps_ref_1d(const __grid_constant__ Ref1DArgs r) {
  // what a lane's neighbours read of it, double-buffered by the step's parity:
  // its two moving populations and, for the face rules, its node's eps or
  // alpha^B, u and c
  __shared__ double move[2][2][8 * R1_NODES], rule[2][3][8 * R1_NODES];
  const StepArgs &a = r.a;
  const RefConst K{a.cs2, a.two_cs4, a.k0};
  const int tid = threadIdx.x, l8 = tid & 7, ph = l8 & 1, i = tid >> 3, N = a.n[0], H = r.steps;
  const bool liq = ph != 0, isI = l8 < 2, isA = (l8 >> 1) == 1, isB = (l8 >> 1) == 2, isX = l8 >= 6;
  const int core = r1_core(H);
  const bool per = a.bc_lo[0] == BC_PERIODIC;
  const int xl = (int)blockIdx.x * core - r.shift - (H - 1) + i;  // on the unrolled line
  const int x = per ? ((xl % N) + N) % N : xl;
  const bool in = x >= 0 && x < N && !isX;
  const bool lo = !per && x == 0, hi = !per && x == N - 1;
  const bool mine = i >= H - 1 && i < H - 1 + core && xl >= 0 && xl < N && !isX;
  // does the block hold a face node with a rule (block-uniform)?
  const int x0 = xl - i;
  const bool face = (a.has_inlet && x0 <= 0 && x0 + R1_NODES > 0) ||
                    (a.has_outlet && x0 <= N - 1 && x0 + R1_NODES > N - 1);
  const int plane0 = (2 * (l8 >> 1) + ph) * 3;
  const int xp = x + 1 >= N ? 0 : x + 1, xm = x <= 0 ? N - 1 : x - 1;  // wrapped (periodic axis)

  // populations of the own scheme (lanes without a node: a harmless state)
  double f0 = 0.5, f1 = 0.25, f2 = 0.25, Spp = 0.0, Lam = 0.0;
  if (in) {
    // odd steps read slot (x - v_q, opp q), or (x, q) behind a face
    const double *pop = (const double *)a.pop, *held = (const double *)a.held;
    const bool odd = a.parity != 0, o1 = odd && !hi, o2 = odd && !lo;
    f0 = pop[(long long)plane0 * a.plane + x];
    f1 = pop[(long long)(plane0 + (o1 ? 2 : 1)) * a.plane + (o1 ? xp : x)];
    f2 = pop[(long long)(plane0 + (o2 ? 1 : 2)) * a.plane + (o2 ? xm : x)];
    Spp = held[(long long)ph * a.plane + x];
    Lam = held[2 * a.plane + x];
  }
  constexpr double w0 = Lattice<1>::w(0), w1 = Lattice<1>::w(1);
  const double om = isI ? (liq ? a.omega_l : a.omega_g) : a.omega_a;
  const double psi = liq ? a.psi_l : a.psi_g, eta0 = liq ? a.eta0_l : a.eta0_g, nuef = liq ? a.nuef_l : a.nuef_g;
  // functions of the latched values
  double wS0, sE, C;
  auto latched = [&]() {
    wS0 = w0 * (Spp * eta0);
    sE = Spp * psi;
    C = psi * K.cs2 * Spp;
  };
  latched();
  // coefficient of the drag (f_I lanes) and of the wall friction (f_alpha)
  auto coefficient = [&]() {
    const double k = isI ? a.kappa_I : a.kappa_W;
    return a.cgw ? k * Lam : k;
  };
  double kap = coefficient();
  const unsigned m = 0xffffffffu;
  const int n8 = tid & 24;  // the node's first lane in its warp
  auto get = [&](double v, int lane8) { return __shfl_sync(m, v, n8 + lane8); };
  double o0 = 0.0, o1 = 0.0, o2 = 0.0;

  for (int k = 0; k < H; k++) {
    const double m0 = f0 + f1 + f2, m1 = -f1 + f2, m2 = f1 + f2;
    const double eps_g = get(m0, 0), eps_l = get(m0, 1), a_g = get(m0, 2), a_l = get(m0, 3);
    const double u_g = get(m1, 0), u_l = get(m1, 1);
    const double eps = liq ? eps_l : eps_g, aa = liq ? a_l : a_g, u = liq ? u_l : u_g;
    const double du = liq ? u_l - u_g : u_g - u_l;
    // first division: Eq. (spalding); (eps_g - 1)/R in the spare lanes
    const double Bg = spalB(a_g), Bl = spalB(a_l);
    const double sum = (isX ? eps_g : Bg) + (isX ? -1.0 : Bl);
    const bool some = isX || ref_above(sum, 0.0);
    const double qA = (isX ? sum : Bg) / (isX ? a.R : (some ? sum : 1.0));
    const double g = some ? qA : 0.5;
    const double one = 1.0 + (isX ? qA : -g);  // alpha^B_l; 1 + (eps_g - 1)/R in the spare lanes
    double al = liq ? one : g, al_o = liq ? g : one;
    if (a.spalding == 0) {
      al = aa;
      al_o = liq ? a_g : a_l;
    }
    if (r.latch >> k & 1u) {
      const double gg = liq ? al_o : al, ll = liq ? al : al_o;
      Lam = gg * ll * (gg + ll * a.R);  // Eq. (Lambda)
      kap = coefficient();
    }
    const double ad = ref_above(al, a.afloor) ? al : a.afloor;
    // c (f_beta lanes, Eq. (velocitybeta)); the divisors alpha, R alpha_l
    const double cden = (isB ? al_o : (liq ? a.R : 1.0)) * (isB ? du : ad);
    // second division: drag (f_I), wall friction (f_alpha, liquid), phi (spare lanes)
    const double vel = isI ? (liq ? du : -du) : u;
    const bool zero = (isA && a.kappa_W == 0.0) || isB;
    const double num = kap * r1_abs(vel) * vel;
    const double qB = (isX ? one : (zero ? 1.0 : num)) / (isX ? eps_l : (isB ? 1.0 : cden));
    const double phi_l = get(qB, 6), fric = a.kappa_W == 0.0 ? 0.0 : get(qB, 3), phi = liq ? phi_l : 1.0;
    if (r.latch >> k & 1u) {
      const double b = get(m0, 4 + ph);
      Spp = (1.0 - b) - a.gamma * (u * u) * (phi * eps - 1.0);
      latched();
    }
    // grad alpha (formed in the f_alpha lanes), stress, force
    const double gr = a.kgrad * (aa * u - m1);
    const double gr_own = get(gr, 2 + ph), gr_oth = get(gr, 3 - ph);
    const double gG = __fma_rn(-0.5, gr_own + gr_oth, gr_own);  // halving is exact
    const double uu = u * u;
    const double sG = nuef * (om * ((K.cs2 * phi * eps + uu) - m2) + C) * gG;
    const double qC = (isI ? sG : 1.0) / (isI ? ad : 1.0);
    double G = Spp * u + qC;
    G = G + (liq ? -qB : a.buoy);
    G = G + (liq ? -fric : qB);
    // collisions; v: u for f_I and f_alpha, c for f_beta
    const double v = isB ? cden : u, vv = v * v, cu = K.cs2 * vv;
    const double E0 = isI ? eps * (1.0 + K.k0 * (1.0 - phi)) : 1.0, E1 = isI ? eps * phi : 1.0;
    const double wa = isA ? (a.spalding == 2 ? al : aa) : 1.0;
    double b0, b1, av, gv;
    if (ref_small(v) || (isI && ref_small(G))) {
      b0 = (0.0 - cu) / K.two_cs4;
      b1 = (vv - cu) / K.two_cs4;
      av = v / K.cs2;
      gv = G / K.cs2;
    } else {
      b0 = div_two_cs4<true>(-cu, K);
      b1 = div_two_cs4<true>(vv - cu, K);
      av = div_cs2<true>(v, K);
      gv = div_cs2<true>(G, K);
    }
    const double r0 = w0 * wa * (E0 + b0), r1 = w1 * wa * (E1 - av + b1), r2 = w1 * wa * (E1 + av + b1);
    o0 = f0 + om * (r0 - f0);
    o1 = f1 + om * (r1 - f1);
    o2 = f2 + om * (r2 - f2);
    const double s0 = o0 + wS0, s1 = o1 + w1 * (sE - gv), s2 = o2 + w1 * (sE + gv);
    o0 = isI ? s0 : (isB ? r0 : o0);
    o1 = isI ? s1 : (isB ? r1 : o1);
    o2 = isI ? s2 : (isB ? r2 : o2);
    const int p = k & 1;
    if (face) {
      // Tables 1 and 2 (k_step_ref's rules)
      rule[p][0][tid] = isA ? al : eps;
      rule[p][1][tid] = u;
      rule[p][2][tid] = cden;
      __syncthreads();
      const int tr = tid + 8 < 8 * R1_NODES ? tid + 8 : tid, tl = tid >= 8 ? tid - 8 : tid;
      if (lo && a.has_inlet) {
        const double epsB = 1.5 * eps - 0.5 * rule[p][0][tr];
        const double epsB_g = 1.5 * eps_g - 0.5 * rule[p][0][tr - ph];
        const double phiB = isI && liq ? (1.0 + (epsB_g - 1.0) / a.R) / epsB : 1.0;
        const double uB = liq ? r.ulIN[k] : r.ugIN[k], aB = liq ? 1.0 - r.aIN[k] : r.aIN[k];
        double P, M;
        r1_feq(K, isI ? epsB * phiB : 1.0, isB ? 2.0 * cden - rule[p][2][tr] : uB, P, M);
        o1 = isI ? o1 + w1 * P - w1 * M : w1 * (isA ? aB : 1.0) * P;
      }
      if (hi && a.has_outlet) {
        const double ab = isA ? 1.5 * al - 0.5 * rule[p][0][tl] : 1.0;
        double P, M;
        r1_feq(K, 1.0, isB ? 2.0 * cden - rule[p][2][tl] : 1.5 * u - 0.5 * rule[p][1][tl], P, M);
        o2 = isB ? w1 * M : -o2 + w1 * ab * M + w1 * ab * P;
      }
    }
    if (k + 1 < H) {
      // streaming; behind a face the reflected value comes back
      move[p][0][tid] = o1;
      move[p][1][tid] = o2;
      __syncthreads();
      const int tr = tid + 8 < 8 * R1_NODES ? tid + 8 : tid, tl = tid >= 8 ? tid - 8 : tid;
      f0 = o0;
      f1 = hi ? o2 : move[p][0][tr];
      f2 = lo ? o1 : move[p][1][tl];
    }
  }
  if (!mine) return;
  // the last step's store: slot (x, opp q) on even steps and behind a face,
  // (x + v_q, q) on odd ones
  const bool odd = ((a.parity + H - 1) & 1) != 0, p1 = odd && !lo, p2 = odd && !hi;
  r.pop_out[(long long)plane0 * a.plane + x] = o0;
  r.pop_out[(long long)(plane0 + (p1 ? 1 : 2)) * a.plane + (p1 ? xm : x)] = o1;
  r.pop_out[(long long)(plane0 + (p2 ? 2 : 1)) * a.plane + (p2 ? xp : x)] = o2;
  if (isI) r.held_out[(long long)ph * a.plane + x] = Spp;
  if (l8 == 0) r.held_out[2 * a.plane + x] = Lam;
}

}  // namespace lbm
